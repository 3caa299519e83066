// Feature rows of every ATV of a pool (asse_features, include/asse_learn.h).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>

#include "../../include/asse_learn.h"
#include "asse_features.cuh"

namespace asse {

namespace {

using bf16 = __nv_bfloat16;
constexpr int FEAT = ASSE_FEAT;

// BF16 bits of v (round to nearest even).
__device__ __forceinline__ uint32_t bf16_bits(float v)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v));
}

constexpr int FEAT_THREADS = 256;
constexpr int FEAT_WARPS = FEAT_THREADS / 32;

// Bit 0 of every field of a word of wb-bit fields.
constexpr uint32_t plane_mask(int wb)
{
    uint32_t m = 0;
    for (int j = 0; j < 32 / wb; j++)
        m |= 1u << (j * wb);
    return m;
}

// Feature rows from the packed words, bit-sliced.  Eight lanes share an ATV.
// A lane takes WB words at a time, ngrp words apart, and gathers their bits b
// into plane b (field j of the i-th word at bit j WB + i: 28 to 32 fields to a
// plane, two operations per word and plane).  On the planes the age of every
// field, ACT minus value mod 2k with the ACT planes of the position from a
// table, takes six operations per plane, and each age one more and a population
// count, where extracting the fields one by one and counting them in shared
// memory took about twenty operations per active field, on as many lanes as had
// one.  The counts of two ages share a word; the eight lanes end with NA / 8
// ages each and write the row.  Bound: integer issue and population counts.
// 262,144 ATVs of 512 five-bit fields, ages 0..9: 147 -> 64 us (cold caches).
//
// NA: ages counted, 16 or 64 (kp <= NA).  ctl non-null: C0 of the open slice
// comes from the device slice state (a captured graph replays the launch slice
// after slice).
template <int WB, int NA>
__global__ void __launch_bounds__(FEAT_THREADS) features_kernel(Params P, const uint32_t *pool, uint32_t c0,
                                                                const SliceCtl *ctl, uint32_t kp,
                                                                const unsigned long long *aat, bf16 *x,
                                                                uint32_t total_atv, int vec)
{
    constexpr uint32_t F = 32 / WB;
    constexpr int R = NA / 2;   // count words
    constexpr int Q = R / 8;    // of them in each lane at the end
    extern __shared__ uint32_t fsm[];
    if (ctl)
        c0 = ctl->c0;
    const uint32_t nwords = (P.g + F - 1) / F, ngrp = (nwords + WB - 1) / WB;
    uint32_t *tab = fsm;                                             // [WB + 1][ngrp]: ACT planes, fields below g
    float *ltab = reinterpret_cast<float *>(tab + (WB + 1) * ngrp);  // [(r + 2) nf]
    for (uint32_t i = threadIdx.x; i < (WB + 1) * ngrp; i += FEAT_THREADS)
        tab[i] = 0;
    // load features of every (row, frame), then UP and mean P of every frame,
    // once per block (FP64, then stored as FP32)
    const double denom = (double)P.g * (double)(P.cmask + 1);
    for (uint32_t frame = threadIdx.x; frame < P.nf; frame += FEAT_THREADS) {
        double up = 1.0, sum = 0.0;
        for (uint32_t i = 0; i < P.r; i++) {
            const double pi = (double)aat[(size_t)i * P.nf + frame] / denom;
            up *= pi;
            sum += pi;
            ltab[i * P.nf + frame] = (float)pi;
        }
        ltab[P.r * P.nf + frame] = (float)up;
        ltab[(P.r + 1) * P.nf + frame] = (float)(sum / P.r);
    }
    __syncthreads();
    for (uint32_t q = threadIdx.x; q < nwords; q += FEAT_THREADS) {
        const uint32_t i = q / ngrp, gi = q - i * ngrp;  // the i-th word of group gi
        for (uint32_t j = 0; j < F; j++) {
            const uint32_t h = q * F + j;
            if (h >= P.g)
                break;
            const uint32_t act = P.ace ? P.k : act_of(P, c0, pos_block(P, h)), bit = 1u << (j * WB + i);
            for (uint32_t b = 0; b < WB; b++)
                if ((act >> b) & 1)
                    atomicOr(&tab[b * ngrp + gi], bit);
            atomicOr(&tab[WB * ngrp + gi], bit);
        }
    }
    __syncthreads();
    // a visit age slices ago left ACT - age mod 2k, or k - age in an aging
    // counter; the inactive value is 2k, or 0
    const uint32_t wrap = P.ace ? 0u : P.k2;
    constexpr uint32_t M = plane_mask(WB);
    const uint32_t lane = threadIdx.x & 31, grp = lane >> 3, sub = lane & 7;
    const float inv_g = 1.0f / (float)P.g;
    const uint32_t warps = gridDim.x * FEAT_WARPS;
    for (uint32_t a0 = (blockIdx.x * FEAT_WARPS + (threadIdx.x >> 5)) * 4; a0 < total_atv; a0 += warps * 4) {
        const uint32_t atv = a0 + grp;
        const bool mine = atv < total_atv;
        const uint32_t *words = pool + (size_t)(mine ? atv : a0) * P.Wd;
        uint32_t acc[R];
#pragma unroll
        for (int i = 0; i < R; i++)
            acc[i] = 0;
        for (uint32_t gi = sub; gi < ngrp; gi += 8) {
            uint32_t pl[WB];
#pragma unroll
            for (int b = 0; b < WB; b++)
                pl[b] = 0;
#pragma unroll
            for (int i = 0; i < WB; i++) {
                const uint32_t q = gi + i * ngrp;
                const uint32_t w = q < nwords ? words[q] : 0u;
#pragma unroll
                for (int b = 0; b < WB; b++)
                    pl[b] |= (i >= b ? w << (i - b) : w >> (b - i)) & (M << i);
            }
            uint32_t none = ~0u, br = 0, d[WB];
#pragma unroll
            for (int b = 0; b < WB; b++) {
                const uint32_t act = tab[b * ngrp + gi], same = ~(pl[b] ^ (0u - ((wrap >> b) & 1)));
                none &= same;
                d[b] = act ^ pl[b] ^ br;
                br = (~act & pl[b]) | (~(act ^ pl[b]) & br);
            }
            const uint32_t on = mine ? tab[WB * ngrp + gi] & ~none : 0u;
            // ACT - value below 0: + 2k
            uint32_t cy = 0;
#pragma unroll
            for (int b = 0; b < WB; b++) {
                const uint32_t t = br & (0u - ((wrap >> b) & 1)), v = d[b];
                d[b] = v ^ t ^ cy;
                cy = (v & t) | (cy & (v | t));
            }
            auto bit = [&](int b) { return b < WB ? d[b < WB ? b : 0] : 0u; };
            uint32_t in = on;  // age below NA
#pragma unroll
            for (int b = NA == 64 ? 6 : 4; b < WB; b++)
                in &= ~d[b];
#pragma unroll
            for (int a16 = 0; a16 < NA; a16 += 16) {
                if ((uint32_t)a16 < kp) {
                    const uint32_t h = NA == 64 ? in & (a16 & 32 ? bit(5) : ~bit(5)) & (a16 & 16 ? bit(4) : ~bit(4)) : in;
#pragma unroll
                    for (int a4 = a16; a4 < a16 + 16; a4 += 4) {
                        if ((uint32_t)a4 < kp) {
                            const uint32_t hq = h & (a4 & 8 ? bit(3) : ~bit(3)) & (a4 & 4 ? bit(2) : ~bit(2));
#pragma unroll
                            for (int a = a4; a < a4 + 4; a++) {
                                const uint32_t m = hq & (a & 2 ? bit(1) : ~bit(1)) & (a & 1 ? bit(0) : ~bit(0));
                                acc[a / 2] += (uint32_t)__popc(m) << (16 * (a & 1));
                            }
                        }
                    }
                }
            }
        }
        // add up over the eight lanes; lane sub keeps count words Q sub ..
        auto fold = [&](auto half_c, uint32_t off) {
            constexpr int half = decltype(half_c)::value;
            const bool up = (sub & off) != 0;
#pragma unroll
            for (int i = 0; i < half; i++) {
                const uint32_t give = up ? acc[i] : acc[i + half], keep = up ? acc[i + half] : acc[i];
                acc[i] = keep + __shfl_xor_sync(FULL_MASK, give, off);
            }
        };
        fold(std::integral_constant<int, R / 2>(), 4);
        fold(std::integral_constant<int, R / 4>(), 2);
        fold(std::integral_constant<int, R / 8>(), 1);
        // its ages 2 Q sub ..; those past the window do not count
        uint32_t own = 0, e[2 * Q];
#pragma unroll
        for (int i = 0; i < 2 * Q; i++) {
            const uint32_t c = i & 1 ? acc[i / 2] >> 16 : acc[i / 2] & 0xffffu;
            const uint32_t n = 2 * Q * sub + i < kp ? c : 0u;
            own += n;
            e[i] = bf16_bits((float)n * inv_g);
        }
        uint32_t cnt = own;
        cnt += __shfl_xor_sync(FULL_MASK, cnt, 1);
        cnt += __shfl_xor_sync(FULL_MASK, cnt, 2);
        cnt += __shfl_xor_sync(FULL_MASK, cnt, 4);
        // element 0 is the count, age a element a + 1: the lane's elements start
        // with the last age of the lane before
        const uint32_t last = __shfl_up_sync(FULL_MASK, e[2 * Q - 1], 1);
        const uint32_t firste = sub == 0 ? bf16_bits((float)cnt * inv_g) : last;
        if (!mine)
            continue;
        const uint32_t row = atv >> P.E_log2, frame = (atv & ((1u << P.E_log2) - 1)) >> P.c;
        const uint32_t l65 = bf16_bits(ltab[row * P.nf + frame]) << 16;
        const uint32_t l66 = bf16_bits(ltab[P.r * P.nf + frame]) | (bf16_bits(ltab[(P.r + 1) * P.nf + frame]) << 16);
        uint32_t out[Q + 4];  // words of the row: Q sub .., then four of the words past them
        out[0] = firste | (e[0] << 16);
#pragma unroll
        for (int i = 1; i < Q; i++)
            out[i] = e[2 * i - 1] | (e[2 * i] << 16);
        // NA = 16: words 8..39 are left, four to a lane, word 8 (age 15) with lane
        // 7; NA = 64: words 32..35 (age 63 and the loads) with lane 7, 36..39 lane 6
        const uint32_t tail = NA == 16 ? (sub == 7 ? 8u : 12u + 4 * sub) : (sub == 7 ? 32u : 36u);
        const bool has_tail = NA == 16 || sub >= 6;
        out[Q] = (sub == 7 ? e[2 * Q - 1] : 0u) | (tail == 32 ? l65 : 0u);
        out[Q + 1] = tail == 32 ? l66 : 0u;
        out[Q + 2] = out[Q + 3] = 0;
        uint32_t *dst = reinterpret_cast<uint32_t *>(x + (size_t)atv * FEAT);
        if (vec) {
            if constexpr (Q == 1)
                dst[sub] = out[0];
            else
                *reinterpret_cast<uint4 *>(dst + Q * sub) = make_uint4(out[0], out[1], out[2], out[3]);
            if (has_tail)
                *reinterpret_cast<uint4 *>(dst + tail) = make_uint4(out[Q], out[Q + 1], out[Q + 2], out[Q + 3]);
        } else {
            uint16_t *d16 = reinterpret_cast<uint16_t *>(dst);
#pragma unroll
            for (int i = 0; i < Q + 4; i++) {
                if (i >= Q && !has_tail)
                    break;
                const uint32_t at = 2 * (i < Q ? Q * sub + i : tail + i - Q);
                d16[at] = (uint16_t)out[i];
                d16[at + 1] = (uint16_t)(out[i] >> 16);
            }
        }
    }
}

// Feature rows of a pool with slice counts (ASSE_COUNTER_AT_HIST): the
// active ATs of age a are the count of the slice a slices back, phase c0 - a
// (mod 2k), so a row needs the k' counts of its ATV (2 bytes each, 64
// contiguous bytes per warp and phase) instead of its words.  A thread builds
// the row of one ATV in registers and writes it as ten 16-byte stores (VEC,
// x 16-byte aligned) or 80 2-byte stores; the L2 merges the rows' sectors
// (staging a warp's rows in shared memory for fully coalesced stores took
// longer: 0.205 against 0.153 ms for the long pool, fewer resident warps).
// The values are the ones the word kernel computes: count / g and the three
// loads, rounded to BF16.
template <bool VEC>
__global__ void __launch_bounds__(256) hist_features_kernel(Params P, uint32_t c0, const SliceCtl *ctl, uint32_t kp,
                                                            const unsigned long long *aat, bf16 *x,
                                                            uint32_t total_atv)
{
    extern __shared__ uint32_t fsm[];
    if (ctl)
        c0 = ctl->c0;
    float *ltab = reinterpret_cast<float *>(fsm);  // [(r + 2) nf]
    const double denom = (double)P.g * (double)(P.cmask + 1);
    for (uint32_t frame = threadIdx.x; frame < P.nf; frame += blockDim.x) {
        double up = 1.0, sum = 0.0;
        for (uint32_t i = 0; i < P.r; i++) {
            const double pi = (double)aat[(size_t)i * P.nf + frame] / denom;
            up *= pi;
            sum += pi;
            ltab[i * P.nf + frame] = (float)pi;
        }
        ltab[P.r * P.nf + frame] = (float)up;
        ltab[(P.r + 1) * P.nf + frame] = (float)(sum / P.r);
    }
    __syncthreads();
    const float inv_g = 1.0f / (float)P.g;
    for (uint32_t atv = blockIdx.x * blockDim.x + threadIdx.x; atv < total_atv; atv += gridDim.x * blockDim.x) {
        uint32_t pk[FEAT / 2];  // element e in bits 16 (e & 1) of pk[e / 2]
#pragma unroll
        for (int j = 0; j < FEAT / 2; j++)
            pk[j] = 0;
        uint32_t cnt = 0, ph = c0;
#pragma unroll
        for (int a = 0; a < 64; a++) {
            if ((uint32_t)a < kp) {
                const uint32_t c = P.hist[(uint64_t)ph * total_atv + atv];
                cnt += c;
                pk[(1 + a) >> 1] |= bf16_bits((float)c * inv_g) << (16 * ((1 + a) & 1));
                ph = ph == 0 ? P.k2 - 1 : ph - 1;
            }
        }
        const uint32_t row = atv >> P.E_log2, frame = (atv & ((1u << P.E_log2) - 1)) >> P.c;
        pk[0] |= bf16_bits((float)cnt * inv_g);
        pk[32] |= bf16_bits(ltab[row * P.nf + frame]) << 16;                                   // 65: P
        pk[33] = bf16_bits(ltab[P.r * P.nf + frame]) | (bf16_bits(ltab[(P.r + 1) * P.nf + frame]) << 16);  // 66, 67
        bf16 *dst = x + (size_t)atv * FEAT;
        if constexpr (VEC) {
            uint4 *d4 = reinterpret_cast<uint4 *>(dst);
#pragma unroll
            for (int j = 0; j < FEAT / 8; j++)
                d4[j] = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
        } else {
            uint16_t *d = reinterpret_cast<uint16_t *>(dst);
#pragma unroll
            for (int e = 0; e < FEAT; e++)
                d[e] = (uint16_t)(pk[e >> 1] >> (16 * (e & 1)));
        }
    }
}

}  // namespace

}  // namespace asse

using namespace asse;

namespace asse {

cudaError_t launch_features(const FeatureView &v, uint16_t *x_dev)
{
    const uint32_t total = v.P.r << v.P.E_log2;
    if (v.P.hist != nullptr && v.kp <= 64) {
        // slice counts: the rows from the counts, not from the words
        const size_t smem = (size_t)(v.P.r + 2) * v.P.nf * sizeof(float);
        const bool vec = ((uintptr_t)x_dev & 15) == 0;
        auto kern = vec ? hist_features_kernel<true> : hist_features_kernel<false>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
        const uint64_t want = (total + 255) / 256;
        const uint64_t full = (uint64_t)v.sms * resident_blocks(kern, 256, smem);
        kern<<<(unsigned)(want < full ? want : full), 256, smem, v.stream>>>(
            v.P, v.c0, v.ctl, v.kp, v.aat, reinterpret_cast<bf16 *>(x_dev), total);
        *v.launches += 1;
        return cudaGetLastError();
    }
    cudaError_t e = dispatch_w(v.w, [&](auto wb) {
        constexpr int WB = decltype(wb)::value;
        constexpr uint32_t F = 32 / WB;
        const uint32_t nwords = (v.P.g + F - 1) / F, ngrp = (nwords + WB - 1) / WB;
        const size_t smem = ((size_t)(WB + 1) * ngrp + (size_t)(v.P.r + 2) * v.P.nf) * sizeof(uint32_t);
        auto kern = features_kernel<WB, 16>;
        if constexpr (WB >= 5) {  // narrower counters have windows of at most 15 slices
            if (v.kp > 16)
                kern = features_kernel<WB, 64>;
        }
        const uint64_t want = (total + 4 * FEAT_WARPS - 1) / (4 * FEAT_WARPS);
        const uint64_t full = (uint64_t)v.sms * resident_blocks(kern, FEAT_THREADS, smem);
        kern<<<(unsigned)(want < full ? want : full), FEAT_THREADS, smem, v.stream>>>(
            v.P, v.pool, v.c0, v.ctl, v.kp, v.aat, reinterpret_cast<bf16 *>(x_dev), total,
            ((uintptr_t)x_dev & 15) == 0 ? 1 : 0);
        return cudaGetLastError();
    });
    *v.launches += 1;
    return e;
}

}  // namespace asse

extern "C" {

int asse_features(asse_pool *pool, uint16_t *x_dev)
{
    if (!pool || !x_dev)
        return pool ? pool_fail(pool, ASSE_EINVAL, "x_dev is NULL") : ASSE_EINVAL;
    FeatureView v;
    if (int rc = pool_feature_view(pool, &v))
        return rc;
    if (v.kp > 64)
        return pool_fail(pool, ASSE_EINVAL, "features need k' <= 64");
    const cudaError_t e = launch_features(v, x_dev);
    if (e != cudaSuccess)
        return pool_fail(pool, ASSE_ECUDA, std::string("features launch: ") + cudaGetErrorString(e));
    return ASSE_OK;
}

}  // extern "C"
