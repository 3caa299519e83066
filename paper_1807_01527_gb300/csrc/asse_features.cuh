// Per-warp pieces of the feature rows that count ages in shared memory: the
// candidate rows (asse_candidates.cu) and the synthetic training states
// (asse_learn.cu).  The rows of a pool's ATVs have kernels of their own
// (asse_features.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/asse_learn.h"
#include "asse_device.cuh"
#include "asse_swar.cuh"

namespace asse {

// Each lane counts ages in its own column of a [64][32] histogram of 16-bit
// counters, zero on entry and left zero, so the histogram needs no atomics;
// the lanes then add up one age row each, reading the row rotated by the age so
// that no two lanes hit one bank.
constexpr uint32_t HIST_WORDS = 64 * 32 / 2;  // (a lane counts at most g/32 <= 128)

// Per-position tables of the window ending at the slice whose block 0 has ACT
// c0: desc[q] the count ranges of word q, actw[q] the ACT of each of its
// fields (AT counters; unused for aging counters).  All threads of the block.
template <int WB>
__device__ void feature_tables(const Params &P, uint32_t c0, uint32_t kp, RangeDesc *desc, uint32_t *actw)
{
    constexpr uint32_t F = 32 / WB;
    for (uint32_t q = threadIdx.x; q < P.Wd; q += blockDim.x) {
        desc[q] = count_desc<WB>(P, q, c0, kp);
        uint32_t a = 0;
        for (uint32_t j = 0; j < F; j++) {
            const uint32_t h = q * F + j;
            if (h < P.g)
                a |= act_of(P, c0, pos_block(P, h)) << (j * WB);
        }
        actw[q] = a;
    }
}

// The feature row of one ATV of cnt active ATs whose ages are counted in hist
// ([kp][32] 16-bit, a column per lane; left zero), by one warp.
__device__ __forceinline__ void write_feature_row(const Params &P, uint32_t cnt, uint32_t kp, float lp, float lup,
                                                  float lmean, uint16_t *hist, __nv_bfloat16 *row, uint32_t lane)
{
    __syncwarp();
    uint32_t bins[2] = {0, 0};
#pragma unroll
    for (uint32_t t = 0; t < 2; t++) {
        const uint32_t e = lane + 32 * t;
        if (e < kp) {
            uint16_t *hr = hist + e * 32;
            uint32_t acc = 0;
            for (uint32_t j = 0; j < 32; j++) {
                const uint32_t c = (j + e) & 31;
                acc += hr[c];
                hr[c] = 0;
            }
            bins[t] = acc;
        }
    }
    const float inv_g = 1.0f / (float)P.g;
#pragma unroll
    for (uint32_t m = 0; m < (ASSE_FEAT + 31) / 32; m++) {
        const uint32_t e = lane + 32 * m;
        // age e - 1 is held by lane (e - 1) mod 32, in bins[(e - 1) / 32]
        const uint32_t src = (e + 31) & 31;
        const uint32_t b0 = __shfl_sync(FULL_MASK, bins[0], src);
        const uint32_t b1 = __shfl_sync(FULL_MASK, bins[1], src);
        if (e >= ASSE_FEAT)
            continue;
        float v = 0.0f;
        if (e == 0)
            v = (float)cnt * inv_g;
        else if (e <= 64)
            v = (float)(e - 1 < 32 ? b0 : b1) * inv_g;
        else if (e == 65)
            v = lp;
        else if (e == 66)
            v = lup;
        else if (e == 67)
            v = lmean;
        row[e] = __float2bfloat16_rn(v);
    }
}

}  // namespace asse
