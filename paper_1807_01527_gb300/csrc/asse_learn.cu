// Learned per-ATV cardinality model (include/asse_learn.h): feature rows of
// ATV states, synthetic training states, and the MLP (FEAT -> 256 -> 256 -> 1,
// ReLU) with its training step, all in the library's own kernels.
//
// Every matrix product of the training pass runs on the 5th-generation tensor
// cores (tcgen05, BF16 operands, FP32 accumulation in tensor memory) through
// one kernel whose operands are addressed by (row, k) strides
// (launch_tc_gemm, asse_mlp_tc.cu), so the forward products and the
// transposed ones of the weight gradients (split over the batch) are the same
// kernel with a different epilogue: bias + ReLU -> BF16, the same + dot with w3
// (the last layer fused into the second), gradient masked by the ReLU -> BF16
// with its column sums, or FP32 atomic accumulation.  A step is six launches.
// Inference has its own fused tcgen05 kernel.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/asse_learn.h"
#include "asse_device.cuh"
#include "asse_features.cuh"
#include "asse_mlp_tc.h"
#include "asse_pool_access.h"
#include "asse_synth.cuh"

using bf16 = __nv_bfloat16;

namespace asse {

namespace {

constexpr int FEAT = ASSE_FEAT;
constexpr int HID = ASSE_HID;
// offsets of the parameter blocks in the flat fp32 parameter vector
constexpr size_t OFF_W1 = 0;
constexpr size_t OFF_B1 = OFF_W1 + (size_t)HID * FEAT;
constexpr size_t OFF_W2 = OFF_B1 + HID;
constexpr size_t OFF_B2 = OFF_W2 + (size_t)HID * HID;
constexpr size_t OFF_W3 = OFF_B2 + HID;
constexpr size_t OFF_B3 = OFF_W3 + HID;
constexpr size_t NPARAMS = OFF_B3 + 1;
static_assert(NPARAMS == ASSE_MLP_NPARAMS, "parameter layout");

// est[i] = exp(max(y[i], 0)) where the ATV holds an active AT and the model
// is inside its training range (y <= max_log_n, the log of the largest
// cardinality it was trained on; a cardinality is at least 1), else the
// linear-counting estimate of Eq. 2 from the ATV's count: 0 for an empty
// ATV, and a saturated count g taken as g - 1/2.
__global__ void learned_combine_kernel(const float *y, const uint16_t *cnt, uint32_t g, float max_log_n,
                                       uint64_t n, float *est, uint32_t *n_fallback)
{
    uint32_t fb = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const float yi = y[i];
        const uint32_t c = cnt[i];
        if (c > 0 && yi <= max_log_n) {
            est[i] = expf(fmaxf(yi, 0.0f));
        } else {
            const double cc = c >= g ? (double)g - 0.5 : (double)c;
            est[i] = (float)(-(double)g * log(((double)g - cc) / (double)g));
            fb++;
        }
    }
    fb = __reduce_add_sync(FULL_MASK, fb);
    if ((threadIdx.x & 31) == 0 && fb)
        atomicAdd(n_fallback, fb);
}

// ---------------------------------------------------------------- learned report

// The host addresses of n candidate records, contiguous for the feature kernel.
__global__ void cand_aips_kernel(const asse_superpoint *c, uint64_t n, uint32_t *aips)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        aips[i] = c[i].aip;
}

// The decision of asse_report_learned for each candidate: inside the model's
// training range its estimate exp(max(y, 0)) and est >= theta, else the
// candidate's Eq. 4 estimate and decision as restored.  The reported records
// are packed into rep, each warp taking its places with one atomic.
__global__ void learned_report_kernel(const asse_superpoint *cand, const float *y, uint64_t n, float max_log_n,
                                      float theta, asse_superpoint *rep, unsigned long long *n_rep)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    // one bound per warp, so that every lane takes part in the ballot
    for (uint64_t base = blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); base < n; base += stride) {
        const uint64_t i = base + lane;
        asse_superpoint sp{};
        bool keep = false;
        if (i < n) {
            sp = cand[i];
            const float yi = y[i];
            if (yi <= max_log_n) {  // false for a NaN output: Eq. 4 stands
                sp.est = expf(fmaxf(yi, 0.0f));
                sp.flags = ASSE_SP_LEARNED | (sp.est >= theta ? ASSE_SP_REPORTED : 0u);
            }
            keep = (sp.flags & ASSE_SP_REPORTED) != 0;
        }
        const unsigned m = __ballot_sync(FULL_MASK, keep);
        unsigned long long at = 0;
        if (lane == 0 && m)
            at = atomicAdd(n_rep, (unsigned long long)__popc(m));
        at = __shfl_sync(FULL_MASK, at, 0);
        if (keep)
            rep[at + __popc(m & ((1u << lane) - 1u))] = sp;
    }
}

// ---------------------------------------------------------------- synthetic states

struct SynthArgs {
    uint64_t seed;
    uint32_t n_max_log2;
    float bg_max;
};

constexpr int SYNTH_WARPS = 8;
constexpr uint32_t SYNTH_MAX_BATCH = 32;      // states a block takes at a time
constexpr uint32_t SYNTH_TABLE_BYTES = 49152; // largest table of mixed background draw indices

// Shared memory of synth_kernel, in bytes.
__host__ __device__ inline size_t synth_smem(uint32_t k, uint32_t g, uint32_t batch, bool table)
{
    return (size_t)batch * k * sizeof(double) + (table ? (size_t)k * g * sizeof(uint64_t) : 0) +
           (size_t)SYNTH_WARPS * (g * sizeof(int) + k * 32 * sizeof(uint16_t)) +
           (size_t)batch * (k + 1) * sizeof(uint32_t);
}

// The state at the end of slice k - 1 is, for every AT, the last slice that
// set it, from two kinds of draws: the host's distinct bips, bip j in the
// slice s with end[s] <= j < end[s + 1], and the background, which sets AT h
// in slice s if its draw is below pbg.  All k slices are in the window, so
// the age of an AT is k - 1 minus that slice and the packed words are not
// needed.  What bounds it is integer issue, so the draws that cannot change
// the state are not made:
//  * the bips run from the last to the first, and once every AT is set the
//    earlier ones (of the same or earlier slices) change nothing: about
//    g ln g draws of up to 2^n_max_log2;
//  * the background of an AT runs from the last slice back to its first hit,
//    and only over slices after the bips'.  unit() < pbg is the same as the
//    53-bit draw below ceil(pbg 2^53), an integer comparison, and the inner
//    SplitMix64 of the draw index, the same for every state, comes from a
//    table of the block where k g of them fit.
// The FP64 terms (1/64 of the FP32 rate here) are computed with a lane per
// state and slice, a batch of states at a time, then one warp draws one state.
// 16,384 states of k = 10, g = 512, n up to 2^20: 2,290 us with a block a
// state and every draw made, 200 us now.
__global__ void __launch_bounds__(SYNTH_WARPS * 32) synth_kernel(Params P, SynthArgs S, uint64_t first, uint64_t n,
                                                                 uint32_t batch, int table, bf16 *x,
                                                                 float *log_n, float *lc)
{
    extern __shared__ double synth_sm[];
    const uint32_t k = P.k, g = P.g;
    double *w = synth_sm;                                              // [batch][k] shares, then their running sums
    uint64_t *tab = reinterpret_cast<uint64_t *>(w + batch * k);       // [k][g] if table
    int *last_all = reinterpret_cast<int *>(tab + (table ? k * g : 0));             // [warps][g]
    uint16_t *hist_all = reinterpret_cast<uint16_t *>(last_all + SYNTH_WARPS * g);  // [warps][k][32], zero between uses
    uint32_t *end_all = reinterpret_cast<uint32_t *>(hist_all + SYNTH_WARPS * k * 32);  // [batch][k + 1]
    __shared__ uint32_t card[SYNTH_MAX_BATCH], cnts[SYNTH_MAX_BATCH];
    __shared__ float pbg[SYNTH_MAX_BATCH];
    __shared__ uint64_t below[SYNTH_MAX_BATCH];  // ceil(pbg 2^53)
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int *last = last_all + warp * g;
    uint16_t *hist = hist_all + warp * k * 32;
    for (uint32_t i = tid; i < SYNTH_WARPS * k * 32; i += blockDim.x)
        hist_all[i] = 0;
    if (table)
        for (uint32_t i = tid; i < k * g; i += blockDim.x)
            tab[i] = splitmix(((uint64_t)(i / g) << 32) | (i % g));
    for (uint64_t b0 = (uint64_t)blockIdx.x * batch; b0 < n; b0 += (uint64_t)gridDim.x * batch) {
        const uint32_t nb = (uint32_t)(n - b0 < batch ? n - b0 : batch);
        auto state_key = [&](uint32_t q) { return splitmix(S.seed ^ splitmix(first + b0 + q + 0x51ED270B27ull)); };
        for (uint32_t e = tid; e < nb * k; e += blockDim.x)
            w[e] = -log(unit(state_key(e / k), 16 + e % k) + 1e-300);
        for (uint32_t q = tid; q < nb; q += blockDim.x) {
            const uint64_t key = state_key(q);
            const double lnmax = (double)S.n_max_log2 * 0.6931471805599453;
            const double c = floor(exp(unit(key, 1) * lnmax));
            card[q] = (uint32_t)(c < 1.0 ? 1.0 : c);
            const float pb = (float)(unit(key, 2) * (double)S.bg_max);
            pbg[q] = pb;
            below[q] = (uint64_t)ceil((double)pb * 9007199254740992.0);
        }
        __syncthreads();
        for (uint32_t q = tid; q < nb; q += blockDim.x) {
            double cum = 0.0;
            for (uint32_t s = 0; s < k; s++) {
                cum += w[q * k + s];
                w[q * k + s] = cum;
            }
        }
        __syncthreads();
        for (uint32_t e = tid; e < nb * k; e += blockDim.x) {
            const uint32_t q = e / k, s = e - q * k;
            uint32_t *end = end_all + q * (k + 1);
            end[s + 1] = s + 1 == k ? card[q] : (uint32_t)floor((double)card[q] * w[e] / w[q * k + k - 1]);
            if (s == 0)
                end[0] = 0;
        }
        __syncthreads();
        for (uint32_t q = warp; q < nb; q += SYNTH_WARPS) {
            const uint64_t key = state_key(q);
            const uint32_t base = (uint32_t)(key >> 32);
            const uint32_t *end = end_all + q * (k + 1);
            for (uint32_t h = lane; h < g; h += 32)
                last[h] = -1;
            __syncwarp();
            // bips from the last to the first, 128 at a time, while an AT is unset
            uint32_t unset = g, hi = card[q], s = k - 1;
            while (hi > 0 && unset > 0) {
                const uint32_t lo = hi > 128 ? hi - 128 : 0;
                uint32_t fresh = 0;
#pragma unroll
                for (uint32_t u = 0; u < 4; u++) {
                    if (lane + 32 * u < hi - lo) {
                        const uint32_t j = hi - 1 - lane - 32 * u;
                        while (end[s] > j)
                            s--;
                        fresh += atomicMax(&last[bip_hash(P, mix32(base + j))], (int)s) < 0 ? 1u : 0u;
                    }
                }
                unset -= __reduce_add_sync(FULL_MASK, fresh);
                hi = lo;
            }
            __syncwarp();
            // background, and the ages counted in the lane's column
            uint32_t cnt = 0;
            const uint64_t bkey = key ^ 0xB5ull, lim = below[q];
            for (uint32_t h = lane; h < g; h += 32) {
                int l = last[h];
                for (int t = (int)k - 1; t > l; t--) {
                    const uint64_t ix = table ? tab[(uint32_t)t * g + h] : splitmix(((uint64_t)t << 32) | h);
                    if ((splitmix(bkey ^ ix) >> 11) < lim)
                        l = t;
                }
                if (l >= 0) {
                    hist[(k - 1 - (uint32_t)l) * 32 + lane] += 1;
                    cnt++;
                }
            }
            cnt = __reduce_add_sync(FULL_MASK, cnt);
            const float pw = 1.0f - powf(1.0f - pbg[q], (float)k);  // background activity over the window
            write_feature_row(P, cnt, k, pw, powf(pw, (float)P.r), pw, hist, x + (b0 + q) * FEAT, lane);
            if (lane == 0)
                cnts[q] = cnt;
        }
        __syncthreads();
        for (uint32_t q = tid; q < nb; q += blockDim.x) {
            log_n[b0 + q] = (float)log((double)card[q]);
            const double c = cnts[q] >= g ? (double)g - 0.5 : (double)cnts[q];
            lc[b0 + q] = (float)(-(double)g * log(((double)g - c) / (double)g));
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- elementwise

// From the four partial sums of every output (columns 64 q .. of the second
// layer, q = 0..3; y = b3 + their sum) to the gradient of the second layer's
// outputs.  Squared error of the log: dy = 2 (y - t) / n, loss += (y - t)^2 / n.
// Squared relative error of the estimate exp(y) against exp(t): with
// e = exp(y - t), loss += (e - 1)^2 / n and dy = 2 (e - 1) e / n (y - t
// clamped at 20 so that e stays finite).  Then dZ2 = bf16(dy[m] w3[n] [H2 > 0]);
// dw3[n] += dy[m] H2[m][n]; db2[n] += dZ2; db3 += dy.
//
// A block takes 32 rows at a time: a lane of its first warp per row for dy, then
// a warp per row, a lane per eight columns (16-byte loads and stores).  The sums
// stay in registers until the block's last row, so that a column takes one
// atomic per block (n / 32 of them; with 2,048 blocks of a thread per column
// they were most of 18 us, 4,096 rows).
constexpr int OUT_ROWS = 32;
__global__ void __launch_bounds__(256) out_grad_kernel(const float *yp, const float *b3, const float *t, uint64_t n,
                                                       int kind, const bf16 *H2, const float *w3, bf16 *dZ2,
                                                       float *g_w3, float *g_b2, float *g_b3, float *loss)
{
    __shared__ float dy[OUT_ROWS];
    __shared__ float red[8][2][HID];
    let_next_start();
    wait_for_last();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float w[8], sw[8], sb[8], s3 = 0.0f, sl = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        w[i] = w3[lane * 8 + i];
        sw[i] = sb[i] = 0.0f;
    }
    for (uint64_t base = (uint64_t)blockIdx.x * OUT_ROWS; base < n; base += (uint64_t)gridDim.x * OUT_ROWS) {
        __syncthreads();  // the last rows' dy are read
        if (warp == 0) {
            const uint64_t m = base + lane;
            float g = 0.0f;
            if (m < n) {
                float y = *b3;
#pragma unroll
                for (int q = 0; q < HID / 64; q++)
                    y += yp[q * n + m];
                const float d = y - t[m];
                if (kind == ASSE_LOSS_REL_MSE) {
                    const float e = expf(fminf(d, 20.0f));
                    g = 2.0f * (e - 1.0f) * e / (float)n;
                    sl += (e - 1.0f) * (e - 1.0f) / (float)n;
                } else {
                    g = 2.0f * d / (float)n;
                    sl += d * d / (float)n;
                }
                s3 += g;
            }
            dy[lane] = g;
        }
        __syncthreads();
#pragma unroll
        for (int rr = 0; rr < OUT_ROWS; rr += 8) {
            const uint64_t m = base + rr + warp;
            if (m >= n)
                break;
            const float d = dy[rr + warp];
            const uint4 h4 = *reinterpret_cast<const uint4 *>(H2 + m * HID + lane * 8);
            uint32_t z4[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint32_t hw = u4get(h4, i);
                uint32_t zz = 0;
#pragma unroll
                for (int b = 0; b < 2; b++) {
                    const int c = 2 * i + b;
                    const float h = __uint_as_float(b ? hw & 0xffff0000u : hw << 16);
                    const bf16 z = __float2bfloat16_rn(h > 0.0f ? d * w[c] : 0.0f);
                    zz |= (uint32_t)__bfloat16_as_ushort(z) << (16 * b);
                    sw[c] += d * h;
                    sb[c] += __bfloat162float(z);
                }
                z4[i] = zz;
            }
            *reinterpret_cast<uint4 *>(dZ2 + m * HID + lane * 8) = make_uint4(z4[0], z4[1], z4[2], z4[3]);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        red[warp][0][lane * 8 + i] = sw[i];
        red[warp][1][lane * 8 + i] = sb[i];
    }
    __syncthreads();
    float a = 0.0f, b = 0.0f;
#pragma unroll
    for (int v = 0; v < 8; v++) {
        a += red[v][0][threadIdx.x];
        b += red[v][1][threadIdx.x];
    }
    atomicAdd(&g_w3[threadIdx.x], a);
    atomicAdd(&g_b2[threadIdx.x], b);
    if (warp == 0) {
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            s3 += __shfl_xor_sync(FULL_MASK, s3, off);
            sl += __shfl_xor_sync(FULL_MASK, sl, off);
        }
        if (lane == 0) {
            atomicAdd(g_b3, s3);
            atomicAdd(loss, sl);
        }
    }
}

// Adam on the fp32 parameters, refreshing the bf16 copies of W1 and W2, as
// they are and packed for the inference kernel.
__global__ void adam_kernel(float *p, const float *gr, float *m1, float *m2, uint64_t n, float lr, float b1t,
                            float b2t, bf16 *w1b, bf16 *w2b, bf16 *w1p, bf16 *w2p)
{
    let_next_start();
    wait_for_last();
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const float g = gr[i];
        const float a = 0.9f * m1[i] + 0.1f * g;
        const float b = 0.999f * m2[i] + 0.001f * g * g;
        m1[i] = a;
        m2[i] = b;
        const float v = p[i] - lr * (a / b1t) / (sqrtf(b / b2t) + 1e-8f);
        p[i] = v;
        if (i < OFF_B1) {
            const uint32_t e = (uint32_t)(i - OFF_W1);
            w1p[mlp_w1p_at(e / FEAT, e % FEAT)] = w1b[e] = __float2bfloat16_rn(v);
        } else if (i >= OFF_W2 && i < OFF_B2) {
            const uint32_t e = (uint32_t)(i - OFF_W2);
            w2p[mlp_w2p_at(e / HID, e % HID)] = w2b[e] = __float2bfloat16_rn(v);
        }
    }
}

__global__ void to_bf16_kernel(const float *p, bf16 *w1b, bf16 *w2b)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < NPARAMS;
         i += (uint64_t)gridDim.x * blockDim.x) {
        if (i < OFF_B1)
            w1b[i - OFF_W1] = __float2bfloat16_rn(p[i]);
        else if (i >= OFF_W2 && i < OFF_B2)
            w2b[i - OFF_W2] = __float2bfloat16_rn(p[i]);
    }
}

}  // namespace

}  // namespace asse

using namespace asse;

struct asse_mlp {
    cudaStream_t stream = nullptr;
    float *params = nullptr, *grads = nullptr, *m1 = nullptr, *m2 = nullptr;
    bf16 *w1b = nullptr, *w2b = nullptr;
    bf16 *w1p = nullptr, *w2p = nullptr;  // packed operand images of the tensor-core inference
    int *error = nullptr;                 // set by a kernel whose wait gave up
    uint64_t cap = 0;  // rows of the activation workspace
    bf16 *H1 = nullptr, *H2 = nullptr, *dZ2 = nullptr, *dZ1 = nullptr;
    float *y = nullptr;     // partial sums of the outputs, HID / 64 per row
    float *loss = nullptr;  // after the gradients, in their allocation
    uint64_t steps = 0;
    int loss_kind = ASSE_LOSS_LOG_MSE;
    // workspace of asse_report_learned, for rl_cap candidates
    unsigned char *rl = nullptr;
    uint64_t rl_cap = 0;
    uint64_t launches = 0;
    std::string err;
};

namespace {

int mlp_fail(asse_mlp *m, int code, const std::string &msg)
{
    if (m)
        m->err = msg;
    return code;
}

#define MCK(m, call)                                                                         \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return mlp_fail((m), ASSE_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

int ensure_workspace(asse_mlp *m, uint64_t rows)
{
    if (rows <= m->cap)
        return ASSE_OK;
    cudaStreamSynchronize(m->stream);
    cudaFree(m->H1);
    cudaFree(m->H2);
    cudaFree(m->dZ2);
    cudaFree(m->dZ1);
    cudaFree(m->y);
    m->H1 = m->H2 = m->dZ2 = m->dZ1 = nullptr;
    m->y = nullptr;
    m->cap = 0;
    const size_t act = rows * HID * sizeof(bf16);
    MCK(m, cudaMalloc(&m->H1, act));
    MCK(m, cudaMalloc(&m->H2, act));
    MCK(m, cudaMalloc(&m->dZ2, act));
    MCK(m, cudaMalloc(&m->dZ1, act));
    MCK(m, cudaMalloc(&m->y, rows * (HID / 64) * sizeof(float)));
    m->cap = rows;
    return ASSE_OK;
}

// The gradients of the mean loss of n rows: five launches.
int backward(asse_mlp *m, const bf16 *x, const float *t, uint64_t n, float *loss_dev)
{
    if (int rc = ensure_workspace(m, n))
        return rc;
    const float *P = m->params;
    float *G = m->grads;
    MCK(m, cudaGetLastError());
    const TcExtra nothing{};
    // the first launch also zeroes the gradients and the loss
    const TcProduct h1{TcOperand{x, FEAT, 1}, TcOperand{m->w1b, FEAT, 1}, (int)n, HID, FEAT, 1,
                       TcEpi{TE_BIAS_RELU, P + OFF_B1, nullptr, nullptr, m->H1, nullptr, nullptr, HID}};
    MCK(m, launch_tc_gemm(&h1, 1, TcExtra{G, (uint32_t)NPARAMS + 1, nullptr, nullptr}, m->error, m->stream,
                          &m->launches));
    const TcProduct h2{TcOperand{m->H1, HID, 1}, TcOperand{m->w2b, HID, 1}, (int)n, HID, HID, 1,
                       TcEpi{TE_BIAS_RELU_DOT, P + OFF_B2, P + OFF_W3, nullptr, m->H2, nullptr, m->y, HID}};
    MCK(m, launch_tc_gemm(&h2, 1, nothing, m->error, m->stream, &m->launches));
    const uint64_t ob = (n + OUT_ROWS - 1) / OUT_ROWS;
    MCK(m, launch_dependent(out_grad_kernel, dim3((unsigned)(ob < 608 ? ob : 608)), 256, 0, m->stream, m->y, P + OFF_B3,
                            t, n, m->loss_kind, m->H2, P + OFF_W3, m->dZ2, G + OFF_W3, G + OFF_B2, G + OFF_B3,
                            m->loss));
    m->launches++;
    // the weight-gradient products reduce over the batch: split it so that
    // enough CTAs share the work
    const int splits = (int)((n + 255) / 256);
    const TcProduct hidden[2] = {
        // dW2[o][i] = sum_m dZ2[m][o] H1[m][i]
        {TcOperand{m->dZ2, 1, HID}, TcOperand{m->H1, 1, HID}, HID, HID, (int)n, splits,
         TcEpi{TE_ATOMIC, nullptr, nullptr, nullptr, nullptr, G + OFF_W2, nullptr, HID}},
        // dZ1 = (dZ2 W2) masked by H1 > 0, db1 its column sums
        {TcOperand{m->dZ2, HID, 1}, TcOperand{m->w2b, 1, HID}, (int)n, HID, HID, 1,
         TcEpi{TE_RELU_GRAD, nullptr, nullptr, m->H1, m->dZ1, G + OFF_B1, nullptr, HID}}};
    MCK(m, launch_tc_gemm(hidden, 2, nothing, m->error, m->stream, &m->launches));
    // dW1[o][j] = sum_m dZ1[m][o] X[m][j]; this launch also hands the loss out
    // (two tiles only: split twice as far)
    const TcProduct w1{TcOperand{m->dZ1, 1, HID}, TcOperand{x, 1, FEAT}, HID, FEAT, (int)n, (int)((n + 127) / 128),
                       TcEpi{TE_ATOMIC, nullptr, nullptr, nullptr, nullptr, G + OFF_W1, nullptr, FEAT}};
    MCK(m, launch_tc_gemm(&w1, 1, TcExtra{nullptr, 0, loss_dev, m->loss}, m->error, m->stream, &m->launches));
    return ASSE_OK;
}

}  // namespace

namespace asse {

int mlp_enqueue_learned(asse_mlp *m, const FeatureView &v, float max_log_n, uint16_t *x_dev, float *est_dev,
                        uint32_t *nfb_dev, std::string *why)
{
    cudaError_t e = launch_features(v, x_dev);
    if (e != cudaSuccess) {
        *why = std::string("features launch: ") + cudaGetErrorString(e);
        return ASSE_ECUDA;
    }
    const uint64_t total = (uint64_t)v.P.r << v.P.E_log2;
    // the model's outputs go to est_dev first, then are replaced in place
    const int rc = launch_mlp_forward_tc(reinterpret_cast<const bf16 *>(x_dev), total, m->w1p, m->w2p, m->params,
                                         est_dev, m->error, v.stream, v.launches, why);
    if (rc != 0)
        return rc == 1 ? ASSE_EINVAL : ASSE_ECUDA;
    e = cudaMemsetAsync(nfb_dev, 0, sizeof(uint32_t), v.stream);
    if (e == cudaSuccess) {
        const unsigned grid = (unsigned)v.sms * 4;
        learned_combine_kernel<<<grid, 256, 0, v.stream>>>(est_dev, v.cnt, v.P.g, max_log_n, total, est_dev,
                                                           nfb_dev);
        *v.launches += 1;
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        *why = std::string("learned combine: ") + cudaGetErrorString(e);
        return ASSE_ECUDA;
    }
    return ASSE_OK;
}

}  // namespace asse

using namespace asse;

extern "C" {

int asse_estimate_learned(asse_pool *pool, asse_mlp *mlp, float max_log_n, uint16_t *x_dev, float *est_dev,
                          uint32_t *n_fallback_dev)
{
    if (!pool || !mlp || !x_dev || !est_dev || !n_fallback_dev || !(max_log_n >= 0.0f))
        return pool ? pool_fail(pool, ASSE_EINVAL, "NULL argument or negative max_log_n") : ASSE_EINVAL;
    if ((reinterpret_cast<uintptr_t>(x_dev) & 15u) != 0)
        return pool_fail(pool, ASSE_EINVAL, "x_dev must be 16-byte aligned");
    FeatureView v;
    if (int rc = pool_feature_view(pool, &v))
        return rc;
    if (mlp->stream != v.stream)
        return pool_fail(pool, ASSE_EINVAL, "the model and the pool must use the same stream");
    if (v.kp > 64)
        return pool_fail(pool, ASSE_EINVAL, "features need k' <= 64");
    std::string why;
    if (int rc = mlp_enqueue_learned(mlp, v, max_log_n, x_dev, est_dev, n_fallback_dev, &why))
        return pool_fail(pool, rc, why);
    return ASSE_OK;
}

int asse_report_learned(asse_pool *pool, asse_mlp *m, float max_log_n, asse_superpoint *out, uint64_t cap,
                        uint64_t *n_out, int where)
{
    if (!pool || !m || !n_out || !(max_log_n >= 0.0f) || (where != ASSE_HOST && where != ASSE_DEVICE))
        return pool ? pool_fail(pool, ASSE_EINVAL, "NULL argument, negative max_log_n or unknown where") : ASSE_EINVAL;
    FeatureView v;
    if (int rc = pool_feature_view(pool, &v))
        return rc;
    if (m->stream != v.stream)
        return pool_fail(pool, ASSE_EINVAL, "the model and the pool must use the same stream");
    if (v.kp > 64)
        return pool_fail(pool, ASSE_EINVAL, "features need k' <= 64");
    // workspace, in 256-byte aligned parts of rl_cap records each: feature
    // rows, candidate records, host addresses (then the model's outputs over
    // them), reported records, and the count of reported records
    auto part = [](uint64_t bytes) { return (bytes + 255) / 256 * 256; };
    const uint64_t lcap = pool_list_cap(pool);
    if (lcap > m->rl_cap) {
        cudaFree(m->rl);  // waits for work that may still use the old workspace
        m->rl = nullptr;
        m->rl_cap = 0;
        const uint64_t bytes = part(lcap * FEAT * sizeof(bf16)) + 2 * part(lcap * sizeof(asse_superpoint)) +
                               part(lcap * sizeof(float)) + 256;
        if (cudaMalloc((void **)&m->rl, bytes) != cudaSuccess) {
            cudaGetLastError();
            m->rl = nullptr;
            return pool_fail(pool, ASSE_ENOMEM, "workspace of the learned report");
        }
        m->rl_cap = lcap;
    }
    const uint64_t c = m->rl_cap;
    uint16_t *x = reinterpret_cast<uint16_t *>(m->rl);
    auto *cand = reinterpret_cast<asse_superpoint *>(m->rl + part(c * FEAT * sizeof(bf16)));
    auto *yb = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(cand) + part(c * sizeof(asse_superpoint)));
    auto *rep = reinterpret_cast<asse_superpoint *>(reinterpret_cast<unsigned char *>(yb) + part(c * sizeof(float)));
    auto *n_rep_dev =
        reinterpret_cast<unsigned long long *>(reinterpret_cast<unsigned char *>(rep) + part(c * sizeof(asse_superpoint)));
    // the candidates of the last restore (synchronises; ECAPACITY passes on an overflowed restore)
    uint64_t n = 0;
    if (int rc = asse_candidates(pool, cand, c, &n, ASSE_DEVICE)) {
        *n_out = n;
        return rc;
    }
    *n_out = 0;
    if (n == 0)
        return ASSE_OK;
    const uint64_t blocks = (n + 255) / 256, full = (uint64_t)v.sms * 4;
    const unsigned grid = (unsigned)(blocks < full ? blocks : full);
    uint32_t *aips = reinterpret_cast<uint32_t *>(yb);
    cand_aips_kernel<<<grid, 256, 0, v.stream>>>(cand, n, aips);
    *v.launches += 1;
    if (cudaError_t e = cudaGetLastError(); e != cudaSuccess)
        return pool_fail(pool, ASSE_ECUDA, std::string("candidate addresses: ") + cudaGetErrorString(e));
    if (int rc = asse_candidate_features(pool, aips, n, x))
        return rc;
    std::string why;
    if (int rc = launch_mlp_forward_tc(reinterpret_cast<const bf16 *>(x), n, m->w1p, m->w2p, m->params, yb, m->error,
                                       v.stream, v.launches, &why))
        return pool_fail(pool, rc == 1 ? ASSE_EINVAL : ASSE_ECUDA, why);
    unsigned long long n_rep = 0;
    int gave_up = 0;
    cudaError_t e = cudaMemsetAsync(n_rep_dev, 0, sizeof(unsigned long long), v.stream);
    if (e == cudaSuccess) {
        learned_report_kernel<<<grid, 256, 0, v.stream>>>(cand, yb, n, max_log_n, (float)v.P.theta, rep, n_rep_dev);
        *v.launches += 1;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&n_rep, n_rep_dev, sizeof n_rep, cudaMemcpyDeviceToHost, v.stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&gave_up, m->error, sizeof gave_up, cudaMemcpyDeviceToHost, v.stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(v.stream);
    if (e != cudaSuccess)
        return pool_fail(pool, ASSE_ECUDA, std::string("learned report: ") + cudaGetErrorString(e));
    if (gave_up)
        return pool_fail(pool, ASSE_ETIMEOUT, "the tensor-core MLP gave up waiting for its pipeline");
    *n_out = n_rep;
    const uint64_t k = n_rep < cap ? n_rep : cap;
    if (k > 0) {
        if (!out)
            return pool_fail(pool, ASSE_EINVAL, "out is NULL");
        e = cudaMemcpyAsync(out, rep, k * sizeof(asse_superpoint),
                            where == ASSE_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, v.stream);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(v.stream);
        if (e != cudaSuccess)
            return pool_fail(pool, ASSE_ECUDA, std::string("learned report copy: ") + cudaGetErrorString(e));
    }
    if (n_rep > cap)
        return pool_fail(pool, ASSE_ECAPACITY, "output capacity smaller than the learned report");
    return ASSE_OK;
}

int asse_synth_states(const asse_synth_cfg *cfg, uint64_t first, uint64_t n, uint16_t *x_dev, float *log_n_dev,
                      float *lc_dev, void *stream)
{
    if (!cfg || (n > 0 && (!x_dev || !log_n_dev || !lc_dev)))
        return ASSE_EINVAL;
    if (cfg->k < 1 || cfg->k > 64 || cfg->g < 2 * cfg->k || cfg->g > 4096 || cfg->r < 1 || cfg->n_max_log2 > 24 ||
        (cfg->bh_a & 1) == 0 || !(cfg->bg_max >= 0.0f && cfg->bg_max <= 1.0f))
        return ASSE_EINVAL;
    if (n == 0)
        return ASSE_OK;
    // an ATV of at most 928 words: 3,712 byte-wide fields
    if (cfg->g > 928 * (32 / packed_width(ASSE_COUNTER_AT, cfg->k)))
        return ASSE_EINVAL;
    Params P{};
    P.k = cfg->k;
    P.g = cfg->g;
    P.r = cfg->r;
    P.bh_a = cfg->bh_a;
    P.bh_b = cfg->bh_b;
    SynthArgs S{cfg->seed, cfg->n_max_log2, cfg->bg_max};
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // as many states a block as leave four blocks an SM, 8 to 32 of them
    const uint64_t share = n / ((uint64_t)sms * 4) / SYNTH_WARPS * SYNTH_WARPS;
    const uint32_t batch = share < SYNTH_WARPS ? SYNTH_WARPS : share > SYNTH_MAX_BATCH ? SYNTH_MAX_BATCH : (uint32_t)share;
    const bool table = (uint64_t)cfg->k * cfg->g * sizeof(uint64_t) <= SYNTH_TABLE_BYTES;
    const size_t smem = synth_smem(cfg->k, cfg->g, batch, table);
    const uint64_t blocks = (n + batch - 1) / batch;
    cudaError_t e = cudaFuncSetAttribute(synth_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) {
        synth_kernel<<<(unsigned)(blocks < (1u << 30) ? blocks : (1u << 30)), SYNTH_WARPS * 32, smem,
                       (cudaStream_t)stream>>>(P, S, first, n, batch, table ? 1 : 0,
                                               reinterpret_cast<bf16 *>(x_dev), log_n_dev, lc_dev);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? ASSE_OK : ASSE_ECUDA;
}

int asse_mlp_create(uint64_t seed, void *stream, asse_mlp **out)
{
    if (!out)
        return ASSE_EINVAL;
    *out = nullptr;
    asse_mlp *m = new (std::nothrow) asse_mlp();
    if (!m)
        return ASSE_ENOMEM;
    m->stream = (cudaStream_t)stream;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **p, size_t b) {
        if (e == cudaSuccess)
            e = cudaMalloc(p, b);
    };
    alloc((void **)&m->params, NPARAMS * sizeof(float));
    alloc((void **)&m->grads, (NPARAMS + 1) * sizeof(float));
    m->loss = m->grads + NPARAMS;
    alloc((void **)&m->m1, NPARAMS * sizeof(float));
    alloc((void **)&m->m2, NPARAMS * sizeof(float));
    alloc((void **)&m->w1b, (size_t)HID * FEAT * sizeof(bf16));
    alloc((void **)&m->w2b, (size_t)HID * HID * sizeof(bf16));
    alloc((void **)&m->w1p, (size_t)HID * FEAT * sizeof(bf16));
    alloc((void **)&m->w2p, (size_t)HID * HID * sizeof(bf16));
    alloc((void **)&m->error, sizeof(int));
    if (e == cudaSuccess)
        e = cudaMemsetAsync(m->error, 0, sizeof(int), m->stream);
    if (e != cudaSuccess) {
        asse_mlp_destroy(m);
        return e == cudaErrorMemoryAllocation ? ASSE_ENOMEM : ASSE_ECUDA;
    }
    // Kaiming-uniform weights (bound sqrt(6 / fan_in)), zero biases, drawn on
    // the host from SplitMix64 of the seed
    std::vector<float> h(NPARAMS, 0.0f);
    uint64_t state = seed * 0x9E3779B97F4A7C15ull + 1;
    auto next = [&]() {
        uint64_t z = (state += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    const double b1 = std::sqrt(6.0 / 68.0), b2 = std::sqrt(6.0 / HID), b3 = std::sqrt(6.0 / HID);
    for (size_t o = 0; o < (size_t)HID; o++)
        for (size_t j = 0; j < (size_t)FEAT; j++)
            h[OFF_W1 + o * FEAT + j] = j < 68 ? (float)((2 * next() - 1) * b1) : 0.0f;
    for (size_t i = 0; i < (size_t)HID * HID; i++)
        h[OFF_W2 + i] = (float)((2 * next() - 1) * b2);
    for (size_t i = 0; i < (size_t)HID; i++)
        h[OFF_W3 + i] = (float)((2 * next() - 1) * b3);
    int rc = asse_mlp_set_params(m, h.data());
    if (rc == ASSE_OK) {
        cudaMemsetAsync(m->m1, 0, NPARAMS * sizeof(float), m->stream);
        cudaMemsetAsync(m->m2, 0, NPARAMS * sizeof(float), m->stream);
        if (cudaStreamSynchronize(m->stream) != cudaSuccess)
            rc = ASSE_ECUDA;
    }
    if (rc != ASSE_OK) {
        asse_mlp_destroy(m);
        return rc;
    }
    *out = m;
    return ASSE_OK;
}

void asse_mlp_destroy(asse_mlp *m)
{
    if (!m)
        return;
    cudaStreamSynchronize(m->stream);
    for (void *p : {(void *)m->params, (void *)m->grads, (void *)m->m1, (void *)m->m2, (void *)m->w1b, (void *)m->w2b,
                    (void *)m->H1, (void *)m->H2, (void *)m->dZ2, (void *)m->dZ1, (void *)m->y,
                    (void *)m->w1p, (void *)m->w2p, (void *)m->error, (void *)m->rl})
        cudaFree(p);
    delete m;
}

int asse_mlp_set_stream(asse_mlp *m, void *stream)
{
    if (!m)
        return ASSE_EINVAL;
    m->stream = (cudaStream_t)stream;
    return ASSE_OK;
}

int asse_mlp_get_params(asse_mlp *m, float *host)
{
    if (!m || !host)
        return ASSE_EINVAL;
    MCK(m, cudaMemcpyAsync(host, m->params, NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    MCK(m, cudaStreamSynchronize(m->stream));
    return ASSE_OK;
}

int asse_mlp_set_params(asse_mlp *m, const float *host)
{
    if (!m || !host)
        return ASSE_EINVAL;
    MCK(m, cudaMemcpyAsync(m->params, host, NPARAMS * sizeof(float), cudaMemcpyHostToDevice, m->stream));
    to_bf16_kernel<<<64, 256, 0, m->stream>>>(m->params, m->w1b, m->w2b);
    m->launches++;
    MCK(m, cudaGetLastError());
    MCK(m, launch_mlp_pack(m->params, m->w1p, m->w2p, m->stream, &m->launches));
    MCK(m, cudaStreamSynchronize(m->stream));
    return ASSE_OK;
}

int asse_mlp_get_grads(asse_mlp *m, float *host)
{
    if (!m || !host)
        return ASSE_EINVAL;
    MCK(m, cudaMemcpyAsync(host, m->grads, NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    MCK(m, cudaStreamSynchronize(m->stream));
    return ASSE_OK;
}

int asse_mlp_forward(asse_mlp *m, const uint16_t *x_dev, uint64_t n, float *y_dev)
{
    if (!m || (n > 0 && (!x_dev || !y_dev)))
        return ASSE_EINVAL;
    if (n > 0x7fffffffull)
        return mlp_fail(m, ASSE_EINVAL, "at most 2^31-1 rows per call");
    if (n == 0)
        return ASSE_OK;
    std::string why;
    const int rc = launch_mlp_forward_tc(reinterpret_cast<const bf16 *>(x_dev), n, m->w1p, m->w2p, m->params, y_dev,
                                         m->error, m->stream, &m->launches, &why);
    if (rc == 1)
        return mlp_fail(m, ASSE_EINVAL, why);
    if (rc != 0)
        return mlp_fail(m, ASSE_ECUDA, why);
    return ASSE_OK;
}

int asse_mlp_backward(asse_mlp *m, const uint16_t *x_dev, const float *t_dev, uint64_t n, float *loss_dev)
{
    if (!m || n == 0 || !x_dev || !t_dev)
        return ASSE_EINVAL;
    if (n > 0x7fffffffull)
        return mlp_fail(m, ASSE_EINVAL, "at most 2^31-1 rows per call");
    return backward(m, reinterpret_cast<const bf16 *>(x_dev), t_dev, n, loss_dev);
}

int asse_mlp_train_step(asse_mlp *m, const uint16_t *x_dev, const float *t_dev, uint64_t n, float lr,
                        float *loss_dev)
{
    if (int rc = asse_mlp_backward(m, x_dev, t_dev, n, loss_dev))
        return rc;
    m->steps++;
    const float b1t = 1.0f - powf(0.9f, (float)m->steps), b2t = 1.0f - powf(0.999f, (float)m->steps);
    MCK(m, launch_dependent(adam_kernel, dim3((unsigned)((NPARAMS + 255) / 256)), 256, 0, m->stream, m->params, m->grads,
                            m->m1, m->m2, NPARAMS, lr, b1t, b2t, m->w1b, m->w2b, m->w1p, m->w2p));
    m->launches++;
    return ASSE_OK;
}

int asse_mlp_set_loss(asse_mlp *m, int kind)
{
    if (!m)
        return ASSE_EINVAL;
    if (kind != ASSE_LOSS_LOG_MSE && kind != ASSE_LOSS_REL_MSE)
        return mlp_fail(m, ASSE_EINVAL, "loss must be ASSE_LOSS_LOG_MSE or ASSE_LOSS_REL_MSE");
    m->loss_kind = kind;
    return ASSE_OK;
}

int asse_mlp_check(asse_mlp *m)
{
    if (!m)
        return ASSE_EINVAL;
    MCK(m, cudaStreamSynchronize(m->stream));
    int flag = 0;
    MCK(m, cudaMemcpy(&flag, m->error, sizeof(int), cudaMemcpyDeviceToHost));
    if (flag)
        return mlp_fail(m, ASSE_ETIMEOUT, "a tensor-core MLP kernel gave up waiting for its pipeline");
    return ASSE_OK;
}

const char *asse_mlp_last_error(const asse_mlp *m) { return m ? m->err.c_str() : ""; }

}  // extern "C"
