// K3: restore (Algorithm 4, Sec. 4.2) and cardinality estimation (Algorithm
// 5 and Eq. 4, Sec. 4.3), plus the estimate of caller-given hosts.
//
// restore_kernel runs one CTA per frame.  Instead of enumerating the whole
// product SA(0,j) x ... x SA(r-1,j) and testing each tuple, it joins the rows
// one at a time: a partial tuple carries the LBS bits its columns fixed and
// the positions they cover, and a column of the next row is kept only if it
// agrees on every position already covered.  Since the column windows are
// contiguous runs of positions, agreeing with all earlier rows is the same
// as the paper's check of each row against the next, so the surviving tuples
// are exactly Algorithm 4's.  Complete tuples give LBS, f = LBS.frame and
// aip = f^-1(f); NAT is the popcount of the AND of the r active masks the
// scan kept, and Eq. 4 is evaluated in FP64.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "asse_device.cuh"
#include "asse_swar.cuh"

namespace asse {

namespace {

// Eq. 4 with explicit rounding (no contraction): n = -g ln((g-NAT)/(g(1-UP))),
// +inf when NAT = g or UP = 1, 0 when the ratio is 1 or more.
__device__ __forceinline__ void eq4(uint32_t g, uint32_t theta, uint32_t nat, double up, float &est, uint32_t &flags)
{
    flags = 0;
    if (nat >= g || up >= 1.0) {
        est = INFINITY;
        flags = ASSE_SP_SATURATED | ASSE_SP_REPORTED;
        return;
    }
    const double num = (double)(g - nat);
    const double den = __dmul_rn((double)g, __dsub_rn(1.0, up));
    const double ratio = __ddiv_rn(num, den);
    double e = 0.0;
    if (ratio < 1.0)
        e = __dmul_rn(-(double)g, log(ratio));
    est = (float)e;
    if (e >= (double)theta)
        flags |= ASSE_SP_REPORTED;
}

// Eq. 4 for the candidates of one frame, in FP32 where that is provably
// within 8e-6 relative of the FP64 value above, else by eq4: FP64 on this GPU
// runs at a small fraction of the FP32 rate, and the restore's FP64 chains
// were a third of its time.  ln((g-NAT)/(g(1-UP))) = a - b with
// a = ln(1 - NAT/g) and b = ln(1 - UP).  For NAT < g/2, a = log1pf(-NAT/g):
// the rounding of NAT/g is amplified at most 1.5x, so a is within 5e-7
// relative; above, a = logf(g-NAT) - logf(g) of exact integers, within 2e-6
// absolute (1 ulp of logs below ln 4096) while |a| >= ln 2, so within 3e-6
// relative.  b = log1pf(-UP) with UP < 1/2 is within 5e-7.  When
// |a - b| >= max(|a|, |b|) / 2 the difference is within 2 x 3.5e-6, and the
// product by g and the FP32 result add 1e-7.  The FP64 path takes every
// ratio near or above 1 and every estimate within 0.1 % of theta, so the
// report decision is FP64's.
__device__ __forceinline__ void eq4_fast(uint32_t g, uint32_t theta, uint32_t nat, double up, float b_up,
                                         float &est, uint32_t &flags)
{
    if (nat < g && up < 0.5) {
        const float a = 2u * nat < g ? log1pf(-(float)nat / (float)g) : logf((float)(g - nat)) - logf((float)g);
        const float d = a - b_up;
        const float e = -(float)g * d;
        if (d < 0.0f && fabsf(d) >= 0.5f * fmaxf(fabsf(a), fabsf(b_up)) &&
            fabsf(e - (float)theta) > 1e-3f * (float)theta) {
            est = e;
            flags = e >= (float)theta ? ASSE_SP_REPORTED : 0u;
            return;
        }
    }
    eq4(g, theta, nat, up, est, flags);
}

// UP of a frame (Sec. 4.3): product over rows of |AAT(k',i,j)| / (g 2^c).
__device__ __forceinline__ double frame_up(const Params &P, const unsigned long long *aat, uint32_t frame)
{
    const double denom = __dmul_rn((double)P.g, (double)(P.cmask + 1));
    double up = 1.0;
    for (uint32_t i = 0; i < P.r; i++)
        up = __dmul_rn(up, __ddiv_rn((double)aat[(size_t)i * P.nf + frame], denom));
    return up;
}

// The candidates of a warp (one per lane, if ok) join CSIP, those that reach
// theta the report too: one atomic per list for the warp.
__device__ __forceinline__ void emit(Status *st, asse_superpoint *csip, asse_superpoint *report, uint64_t out_cap,
                                     const HostReport &host, const asse_superpoint &sp, bool ok)
{
    const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    const bool rep = ok && (sp.flags & ASSE_SP_REPORTED) != 0;
    const unsigned mc = __ballot_sync(FULL_MASK, ok), mr = __ballot_sync(FULL_MASK, rep);
    unsigned long long base = 0;
    if (lane == 0 && mc)
        base = atomicAdd(&st->n_csip, (unsigned long long)__popc(mc));
    if (lane == 1 && mr)
        base = atomicAdd(&st->n_report, (unsigned long long)__popc(mr));
    const unsigned long long p = __shfl_sync(FULL_MASK, base, 0) + __popc(mc & lt);
    const unsigned long long p2 = __shfl_sync(FULL_MASK, base, 1) + __popc(mr & lt);
    if (ok && p < out_cap)
        csip[p] = sp;
    if (rep && p2 < out_cap)
        report[p2] = sp;
    if (rep && p2 < host.cap)
        *reinterpret_cast<uint4 *>(host.report + p2) = make_uint4(sp.aip, sp.nat, __float_as_uint(sp.est), sp.flags);
}

constexpr int RESTORE_THREADS = 512;
constexpr uint32_t RESTORE_SMEM_TUPLES = 640;  // per level; the rest of a level spills to the global scratch
constexpr uint32_t RESTORE_SMEM_COLS = 512;    // columns of each row's SA list placed in shared memory

__device__ __forceinline__ void overflow(Status *st, uint32_t needed)
{
    atomicExch(&st->overflow, 1u);
    atomicMax(&st->needed, (unsigned long long)needed);
}

// Tuple a of a level: the first RESTORE_SMEM_TUPLES in shared memory, the rest
// in this frame's part of the global scratch.
__device__ __forceinline__ Tuple *tuple_at(Tuple *sm, Tuple *gl, uint32_t a)
{
    return a < RESTORE_SMEM_TUPLES ? sm + a : gl + a;
}

// The restore of frame blockIdx.x.
__device__ void restore_frame(const Params &P, const ScanOut &o, Tuple *scratch, uint32_t cap, asse_superpoint *csip,
                              asse_superpoint *report, uint64_t out_cap, const HostReport &host)
{
    __shared__ uint32_t n_sa[8];
    __shared__ double p_row[8];  // |AAT(k',i,j)| / (g 2^c) of each row (Sec. 4.3)
    __shared__ uint32_t n_next;
    __shared__ double up_s;      // UP of the frame, and ln(1 - UP) in FP32
    __shared__ float b_up_s;
    __shared__ Tuple sm_t[2][RESTORE_SMEM_TUPLES];
    __shared__ uint2 sm_x[4][RESTORE_SMEM_COLS];  // (bits, positions) of the columns of rows 0..3
    const uint32_t j = blockIdx.x;
    const uint32_t cols = P.cmask + 1;
    const int tid = threadIdx.x;
    // every row's list length and load (one division per thread), and the
    // columns of rows 0..3 placed on LBS positions, all in one pass
    if (tid < (int)P.r) {
        const uint32_t i = tid;
        n_sa[i] = o.sa_n[i * P.nf + j];
        p_row[i] = __ddiv_rn((double)o.aat[(size_t)i * P.nf + j], __dmul_rn((double)P.g, (double)(P.cmask + 1)));
    }
    for (uint32_t e = tid; e < 4 * RESTORE_SMEM_COLS; e += RESTORE_THREADS) {
        const uint32_t i = e / RESTORE_SMEM_COLS, b = e - i * RESTORE_SMEM_COLS;
        if (i < P.r && b < o.sa_n[i * P.nf + j]) {
            uint32_t v, m;
            place(P, o.sa_x[((size_t)i * P.nf + j) * cols + b], (int)i, v, m);
            sm_x[i][b] = make_uint2(v, m);
        }
    }
    if (tid == 0)
        n_next = 0;
    __syncthreads();
    for (uint32_t i = 0; i < P.r; i++)
        if (n_sa[i] == 0)
            return;
    if (tid == RESTORE_THREADS - 1) {
        // UP of the frame: the product over the rows, in row order
        double up = 1.0;
        for (uint32_t i = 0; i < P.r; i++)
            up = __dmul_rn(up, p_row[i]);
        up_s = up;
        b_up_s = log1pf(-(float)up);
    }
    Tuple *cur_g = scratch + (size_t)j * 2 * cap;
    Tuple *nxt_g = cur_g + cap;
    Tuple *cur_s = sm_t[0], *nxt_s = sm_t[1];
    uint32_t n_cur = n_sa[0];
    if (n_cur > cap) {
        if (tid == 0)
            overflow(o.status, n_cur);
        return;
    }
    // level 0: the columns of SA(0, j)
    for (uint32_t a = tid; a < n_cur; a += RESTORE_THREADS) {
        Tuple t;
        if (a < RESTORE_SMEM_COLS) {
            t.L = sm_x[0][a].x;
            t.known = sm_x[0][a].y;
        } else {
            place(P, o.sa_x[(size_t)j * cols + a], 0, t.L, t.known);
        }
        t.slot[0] = (uint16_t)a;
        *tuple_at(cur_s, cur_g, a) = t;
    }
    __syncthreads();
    // levels 1..r-1: keep a column of row i if it agrees with the tuple on
    // every position already covered
    for (uint32_t i = 1; i < P.r; i++) {
        const uint32_t ni = n_sa[i];
        const uint32_t *xs = o.sa_x + ((size_t)i * P.nf + j) * cols;
        // a warp takes one tuple at a time, its lanes the row's columns;
        // survivors are counted with one shared-memory atomic per warp round
        const int lane = tid & 31, warp = tid >> 5;
        const unsigned lt = (1u << lane) - 1u;
        for (uint32_t a = warp; a < n_cur; a += RESTORE_THREADS / 32) {
            const Tuple t = *tuple_at(cur_s, cur_g, a);
            for (uint32_t b0 = 0; b0 < ni; b0 += 32) {
                const uint32_t b = b0 + lane;
                bool keep = false;
                uint32_t v = 0, m = 0;
                if (b < ni) {
                    if (i < 4 && b < RESTORE_SMEM_COLS) {
                        const uint2 vm = sm_x[i][b];
                        v = vm.x;
                        m = vm.y;
                    } else {
                        place(P, xs[b], (int)i, v, m);
                    }
                    keep = ((t.L ^ v) & m & t.known) == 0;
                }
                const unsigned mk = __ballot_sync(FULL_MASK, keep);
                if (mk == 0)
                    continue;
                uint32_t base = 0;
                if (lane == 0)
                    base = atomicAdd(&n_next, (uint32_t)__popc(mk));
                base = __shfl_sync(FULL_MASK, base, 0);
                if (keep) {
                    const uint32_t p = base + __popc(mk & lt);
                    if (p < cap) {
                        Tuple t2 = t;
                        t2.L = t.L | v;
                        t2.known = t.known | m;
                        t2.slot[i] = (uint16_t)b;
                        *tuple_at(nxt_s, nxt_g, p) = t2;
                    }
                }
            }
        }
        __syncthreads();
        n_cur = n_next;
        if (n_cur > cap) {
            if (tid == 0)
                overflow(o.status, n_cur);
            return;
        }
        Tuple *tmp = cur_s;
        cur_s = nxt_s;
        nxt_s = tmp;
        tmp = cur_g;
        cur_g = nxt_g;
        nxt_g = tmp;
        __syncthreads();  // every thread has read n_next before it is reset
        if (tid == 0)
            n_next = 0;
        __syncthreads();
    }
    // NAT and the estimate of the complete tuples, RESTORE_THREADS at a time.
    // What bounds this is latency: the masks are read with as many lanes per
    // tuple as a mask has words (32 at most), then a lane takes a tuple through
    // the inverse mangling and Eq. 4 and a warp appends its tuples to the lists
    // with one atomic each; a warp taking one tuple at a time through all of it
    // took 13.8 us for the link workload, 11.7 now.
    uint32_t ll = 0;  // log2 lanes per tuple
    while (ll < 5 && (1u << ll) < P.mw)
        ll++;
    const uint32_t groups = RESTORE_THREADS >> ll, grp = (uint32_t)tid >> ll, sub = (uint32_t)tid & ((1u << ll) - 1);
    uint32_t *nat_s = reinterpret_cast<uint32_t *>(nxt_s);  // the other level's tuples are not needed any more
    static_assert(RESTORE_SMEM_TUPLES * sizeof(Tuple) >= RESTORE_THREADS * sizeof(uint32_t), "NATs of a round");
    const uint32_t *masks = o.sa_mask + (size_t)j * cols * P.mw;
    for (uint32_t t0 = 0; t0 < n_cur; t0 += RESTORE_THREADS) {
        const uint32_t nt = min(n_cur - t0, (uint32_t)RESTORE_THREADS);
        __syncthreads();  // the frame's UP is written, the last round's NATs are read
        for (uint32_t q0 = 0; q0 < nt; q0 += groups) {
            const uint32_t q = q0 + grp;
            uint32_t nat = 0;
            if (q < nt) {
                const Tuple *tu = tuple_at(cur_s, cur_g, t0 + q);
                for (uint32_t m = sub; m < P.mw; m += 1u << ll) {
                    uint32_t acc = FULL_MASK;
                    for (uint32_t i = 0; i < P.r; i++)
                        acc &= masks[((size_t)i * P.nf * cols + tu->slot[i]) * P.mw + m];
                    nat += __popc(acc);
                }
            }
            for (uint32_t off = 1; off < (1u << ll); off <<= 1)
                nat += __shfl_xor_sync(FULL_MASK, nat, off);
            if (sub == 0 && q < nt)
                nat_s[q] = nat;
        }
        __syncthreads();
        if ((uint32_t)(tid & ~31) < nt) {
            const bool ok = (uint32_t)tid < nt;
            asse_superpoint sp{};
            if (ok) {
                const uint32_t y = (uint32_t)(((uint64_t)tuple_at(cur_s, cur_g, t0 + tid)->L << P.u) | j);
                sp.aip = unmangle(P.Ainv, y);
                sp.nat = nat_s[tid];
                eq4_fast(P.g, P.theta, sp.nat, up_s, b_up_s, sp.est, sp.flags);
            }
            emit(o.status, csip, report, out_cap, host, sp, ok);
        }
    }
}

// One block per frame and window.  With a host report, the reported records are also
// written to pinned host memory as they are found, and the last block to finish
// writes the status there: a report then waits for this kernel alone.  Copies
// of both on a stream of their own after the restore came 13 us after its end.
__global__ void __launch_bounds__(RESTORE_THREADS) restore_kernel(Params P, const __grid_constant__ ScanWindows W,
                                                                  uint32_t cap,
                                                                  const __grid_constant__ RestoreWindows out,
                                                                  uint64_t out_cap, SliceCtl *advance)
{
    wait_for_last();
    // the scan of this close has read the slice state; open the next slice
    if (advance != nullptr && blockIdx.x == 0 && blockIdx.y == 0)
        open_next_slice(P, advance);
    const ScanOut o = W.o[blockIdx.y];
    const RestoreOut ro = out.w[blockIdx.y];
    const HostReport host = ro.host;
    restore_frame(P, o, ro.scratch, cap, ro.csip, ro.report, out_cap, host);
    if (host.status == nullptr)
        return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();  // this block's counts before its own
        if ((atomicAdd(&o.status->done, 1u) + 1) % gridDim.x == 0) {  // (of a repeated restore too)
            __threadfence();
            volatile Status *st = o.status;
            host.status->n_csip = st->n_csip;
            host.status->n_report = st->n_report;
            host.status->needed = st->needed;
            host.status->overflow = st->overflow;
        }
    }
}

constexpr int ESTIMATE_THREADS = 256;

// Sec. 4.3 for given hosts: NAT as the AND over the r rows of the active
// fields of each word, Eq. 4 with the frame's UP.
//
// A warp takes hpw hosts (4, 8, 16 or 32): lane l computes f of host l, then
// eight lanes share a host, each reading 16-byte chunks of its r ATVs (r loads
// in flight a lane) and testing them with the scan's one-range test, whose entry
// of a word position, from a table of the block, serves all r rows.  NAT needs
// no field order, so the test's bits of the rows are ANDed as they are.  Eq. 4
// stays in FP64 (1/64 of the FP32 rate here: a lane per host keeps 32 of them
// on one issue; with one lane of the warp at work it was most of the time) and
// the UP of every frame is computed once per block.
// A scan, a restore and the estimate of 100,003 hosts of a 92 MB pool (g = 512,
// r = 4): 751 -> 215 us a pass, of which this kernel took 583.
template <int WB, int R, bool BG>
__global__ void __launch_bounds__(ESTIMATE_THREADS) estimate_kernel(Params P, const uint32_t *pool, uint32_t c0,
                                                                    uint32_t kp, const unsigned long long *aat,
                                                                    const uint32_t *aips, uint64_t n, uint32_t hpw,
                                                                    asse_superpoint *out)
{
    extern __shared__ uint4 est_sm[];
    using L = CyclicLayout<WB, BG>;
    using Entry = typename L::Entry;
    Entry *ent = reinterpret_cast<Entry *>(est_sm);        // [Wd]
    double *up = reinterpret_cast<double *>(ent + P.Wd);   // [nf]
    for (uint32_t q = threadIdx.x; q < P.Wd; q += blockDim.x)
        ent[q] = cyclic_count_entry<WB, BG>(P, q, c0, kp);
    const typename L::Limit lim = L::limit(cyclic_vmax(P.ace != 0, P.k, L::W));
    for (uint32_t j = threadIdx.x; j < P.nf; j += blockDim.x)
        up[j] = frame_up(P, aat, j);
    __syncthreads();
    const int r = R ? R : (int)P.r;
    constexpr int RM = R ? R : 8;
    const uint32_t lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3;
    const uint32_t chunks = P.Wd / 4;
    const uint64_t stride = (uint64_t)gridDim.x * (ESTIMATE_THREADS / 32) * hpw;
    for (uint64_t base = ((uint64_t)blockIdx.x * (ESTIMATE_THREADS / 32) + (threadIdx.x >> 5)) * hpw; base < n;
         base += stride) {
        const bool mine = lane < hpw && base + lane < n;
        const uint32_t aip = mine ? aips[base + lane] : 0u;
        const uint32_t f = mangle(P.A, aip);
        uint32_t nat = 0;
        for (uint32_t i0 = 0; i0 < hpw; i0 += 4) {
            const uint32_t hf = __shfl_sync(FULL_MASK, f, i0 + grp);
            uint32_t c = 0;
            if (base + i0 + grp < n) {
                const uint32_t z = hf & (P.nf - 1);
                const uint64_t LL = lbs_twice(P, hf);
                const uint4 *a[RM];
#pragma unroll
                for (int i = 0; i < RM; i++)
                    if (i < r)
                        a[i] = reinterpret_cast<const uint4 *>(
                            pool + (((uint64_t)i << P.E_log2) + ((z << P.c) | column(P, LL, i))) * P.Wd);
                for (uint32_t ch = sub; ch < chunks; ch += 8) {
                    uint4 x[RM];
#pragma unroll
                    for (int i = 0; i < RM; i++)
                        if (i < r)
                            x[i] = a[i][ch];
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const Entry d = ent[4 * ch + e];
                        uint32_t m = FULL_MASK;
#pragma unroll
                        for (int i = 0; i < RM; i++)
                            if (i < r)
                                m &= L::test(u4get(x[i], e), d, lim);
                        c += __popc(m);
                    }
                }
            }
            c += __shfl_xor_sync(FULL_MASK, c, 1);
            c += __shfl_xor_sync(FULL_MASK, c, 2);
            c += __shfl_xor_sync(FULL_MASK, c, 4);
            // host i0 + g belongs to lane i0 + g
            c = __shfl_sync(FULL_MASK, c, (lane & 3) * 8);
            if ((lane & ~3u) == i0)
                nat = c;
        }
        if (mine) {
            asse_superpoint sp;
            sp.aip = aip;
            sp.nat = nat;
            eq4(P.g, P.theta, nat, up[f & (P.nf - 1)], sp.est, sp.flags);
            out[base + lane] = sp;
        }
    }
}

}  // namespace

cudaError_t launch_restores(const Params &P, const ScanWindows &W, uint32_t cap, const RestoreWindows &out,
                            uint64_t out_cap, cudaStream_t s, uint64_t *launches, SliceCtl *advance)
{
    *launches += 1;
    return launch_dependent(restore_kernel, dim3(P.nf, W.n), RESTORE_THREADS, 0, s, P, W, cap, out, out_cap, advance);
}

cudaError_t launch_restore(const Params &P, const ScanOut &o, Tuple *scratch, uint32_t cap, asse_superpoint *csip,
                           asse_superpoint *report, uint64_t out_cap, cudaStream_t s, uint64_t *launches,
                           SliceCtl *advance, const HostReport &host)
{
    ScanWindows W{};
    W.n = 1;
    W.o[0] = o;
    RestoreWindows out{};
    out.w[0] = RestoreOut{scratch, csip, report, host};
    return launch_restores(P, W, cap, out, out_cap, s, launches, advance);
}

cudaError_t launch_estimate(const Params &P, uint32_t w, const uint32_t *pool, uint32_t c0, uint32_t kp,
                            const unsigned long long *aat, const uint32_t *aips, uint64_t n, asse_superpoint *out,
                            int sms, cudaStream_t s, uint64_t *launches)
{
    if (n == 0)
        return cudaSuccess;
    // as many hosts a warp as still leave eight warps an SM
    uint32_t hpw = 32;
    while (hpw > 4 && n < (uint64_t)hpw * sms * 8)
        hpw /= 2;
    const bool bg = byte_guard(w, P.ace ? ASSE_COUNTER_ACE : ASSE_COUNTER_AT, P.k);
    *launches += 1;
    return dispatch_w(w, [&](auto wb) {
        constexpr int WB = decltype(wb)::value;
        auto kern = P.r == 4 ? estimate_kernel<WB, 4, false> : estimate_kernel<WB, 0, false>;
        if constexpr (WB == 8) {
            if (bg)
                kern = P.r == 4 ? estimate_kernel<8, 4, true> : estimate_kernel<8, 0, true>;
        }
        const size_t smem = (size_t)P.Wd * (bg ? sizeof(uint2) : sizeof(uint4)) + P.nf * sizeof(double);
        const uint64_t per = (uint64_t)hpw * (ESTIMATE_THREADS / 32);
        const uint64_t want = (n + per - 1) / per;
        const uint64_t full = (uint64_t)sms * resident_blocks(kern, ESTIMATE_THREADS, smem);
        kern<<<(unsigned)(want < full ? want : full), ESTIMATE_THREADS, smem, s>>>(P, pool, c0, kp, aat, aips, n, hpw,
                                                                                 out);
        return cudaGetLastError();
    });
}

}  // namespace asse
