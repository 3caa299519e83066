// K2: the per-slice scan of the whole pool, with the refresh fused in, and
// the standalone refresh kernels.
//
// scan_kernel is a persistent kernel whose warps work alone.  lpa lanes (eight
// for ATVs of 32 words and more) share an ATV: lane p reads its 16-byte chunks
// p, p + lpa, ... straight from global memory, so that a warp's load covers
// whole 128-byte stretches of its ATVs, and a warp takes SCAN_U ATVs per group
// of lanes at a time: SCAN_U loads in flight a lane, and one read of a word's
// range entry (the same for the four groups, one shared-memory wavefront)
// serves SCAN_U words.
//
// The activity test (Algorithm 1) and the refresh's (Algorithm 2) run on every
// field of a word at once, as one cyclic range per field with the entry of the
// word's position (asse_cyclic.h).  What bounds the scan of a pool in L2 is the
// integer pipe, which is why the test has as few operations as that: two plain
// ranges per field took 23 a word of five-bit fields, this 15.
//
// Fused scan of a 92 MB pool in L2: 39 us with tiles staged by bulk copies and
// two ranges, 38 with these loads, 31 with one range too; with aging counters
// 46 -> 28; three windows at once 79 -> 67; a 1.07 GB pool 269 -> 192 us (5.6
// TB/s, 0.82 of the measured copy rate).  A thread that kept one chunk position
// and its entries in registers, the counts of a block added up through shared
// memory, ran 50 and 242 us: its block-wide barriers cost more than the table.
//
// Per ATV the lanes form |ATV|^{k'} (Sec. 3), the row-frame loads |AAT(k',i,j)|
// (Sec. 4.3) and, for a super ATV (Sec. 4.2), its column and, from its words
// read again, its g-bit active mask.  With FUSE the warp then reads the words of
// the two refreshed blocks again (AT), or all words (aging counters), most of
// them still in its L1, and writes them back.
#include <cuda_runtime.h>

#include <cstdint>

#include "asse_device.cuh"
#include "asse_swar.cuh"

namespace asse {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_WARPS = SCAN_THREADS / 32;
constexpr uint32_t SCAN_U = 4;  // ATVs of a group of lanes per tile

// ---------------------------------------------------------------- scan kernel

// Shared memory of scan_kernel: the entries of every window and of the
// refresh, and the masks.
template <int WB, bool BG>
size_t scan_smem(uint32_t Wd, uint32_t mw, uint32_t nw)
{
    return (size_t)(nw + 1) * Wd * sizeof(typename CyclicLayout<WB, BG>::Entry) +
           (size_t)SCAN_WARPS * mw * sizeof(uint32_t);
}

// Lanes of an ATV of S 16-byte chunks: eight, or fewer where more than a fifth
// of their last chunks would lie past the ATV.
inline uint32_t scan_lanes(uint32_t S)
{
    uint32_t lpa = 8;
    while (lpa > 1 && 5 * S < 4 * ((S + lpa - 1) / lpa * lpa))
        lpa /= 2;
    return lpa;
}

// NW: the most windows this instantiation counts (1, or MAX_WINDOWS for the
// multi-window close, which runs W.n <= NW of them).  BG: byte-wide fields
// with values below 128, tested four at a time.
template <int WB, bool FUSE, int NW, bool BG>
__global__ void __launch_bounds__(SCAN_THREADS, 4)
    scan_kernel(Params P, uint32_t *pool, const ScanWindows W, const SliceCtl *ctl, uint32_t total_atv, uint32_t lpa)
{
    static_assert(!BG || WB == 8, "the in-field guard needs byte-wide fields");
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t nw = NW == 1 ? 1u : W.n;
    const uint32_t nchunk = P.Wd / 4;
    using L = CyclicLayout<WB, BG>;
    using Entry = typename L::Entry;
    // entry of word q of window m at m * Wd + (q mod 4) * Wd / 4 + q / 4: the
    // lanes of an ATV read consecutive entries
    auto didx = [&](uint32_t m, uint32_t q) { return m * P.Wd + (q & 3u) * nchunk + (q >> 2); };
    Entry *cd = reinterpret_cast<Entry *>(smem);                      // [nw][Wd]
    Entry *rd = cd + nw * P.Wd;                                       // [Wd]
    uint32_t *maskbuf = reinterpret_cast<uint32_t *>(rd + P.Wd);      // [warps][mw]

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    wait_for_last();
    const uint32_t c0 = ctl->c0;
    const Refresh &R = ctl->R;
    for (uint32_t e = tid; e < nw * P.Wd; e += SCAN_THREADS) {
        const uint32_t m = e / P.Wd, q = e - m * P.Wd;
        cd[didx(m, q)] = cyclic_count_entry<WB, BG>(P, q, c0, W.kp[m]);
        if (FUSE && m == 0 && !P.ace)
            rd[q] = cyclic_refresh_entry<WB, BG>(P, q, R.c0n);
    }
    const typename L::Limit lim = L::limit(cyclic_vmax(P.ace != 0, P.k, L::W));
    __syncthreads();

    const uint32_t groups = 32 / lpa;        // ATVs side by side in a warp
    const uint32_t grp = lane / lpa, sub = lane - grp * lpa;
    const uint32_t apt = groups * SCAN_U;    // ATVs of a tile
    const uint32_t ntiles = (total_atv + apt - 1) / apt;
    const uint32_t cols = P.cmask + 1;
    uint32_t *my_mask = maskbuf + warp * P.mw;
    // tiles are dealt round-robin over all warps of the grid: at any moment
    // the warps read one contiguous stretch of the pool
    for (uint32_t tile = blockIdx.x * SCAN_WARPS + warp; tile < ntiles; tile += gridDim.x * SCAN_WARPS) {
        const uint32_t atv0 = tile * apt;
        const uint32_t n_atv = min(apt, total_atv - atv0);
        const uint4 *src = reinterpret_cast<const uint4 *>(pool) + (size_t)(atv0 + grp) * nchunk;
        uint32_t cnt[NW][SCAN_U];
#pragma unroll
        for (int m = 0; m < NW; m++)
#pragma unroll
            for (uint32_t u = 0; u < SCAN_U; u++)
                cnt[m][u] = 0;
        for (uint32_t ch = sub; ch < nchunk; ch += lpa) {
            uint4 x[SCAN_U];
#pragma unroll
            for (uint32_t u = 0; u < SCAN_U; u++)
                x[u] = u * groups + grp < n_atv ? src[(size_t)u * groups * nchunk + ch] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int m = 0; m < NW; m++) {
                if (m < (int)nw) {
                    const Entry *tab = cd + m * P.Wd + ch;
                    uint32_t bits[SCAN_U];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const Entry d = tab[j * nchunk];
#pragma unroll
                        for (uint32_t u = 0; u < SCAN_U; u++) {
                            const uint32_t b = L::test(u4get(x[u], j), d, lim);
                            if constexpr (BG)  // the guards of the four words side by side in the bytes
                                bits[u] = j == 0 ? b : bits[u] | (b >> j);
                            else
                                cnt[m][u] += __popc(b);
                        }
                    }
                    if constexpr (BG) {
#pragma unroll
                        for (uint32_t u = 0; u < SCAN_U; u++)
                            cnt[m][u] += __popc(bits[u]);
                    }
                }
            }
        }
        // the lanes of an ATV add up, two 16-bit counts to a word; then its lane
        // u takes ATV u (lane u mod lpa, in turns, where it has fewer lanes)
#pragma unroll 1
        for (uint32_t m = 0; m < nw; m++) {
            const ScanOut &o = W.o[m];
            uint32_t c01 = 0, c23 = 0;
#pragma unroll
            for (int mm = 0; mm < NW; mm++)
                if (NW == 1 || (uint32_t)mm == m) {
                    c01 = cnt[mm][0] | (cnt[mm][1] << 16);
                    c23 = cnt[mm][2] | (cnt[mm][3] << 16);
                }
            for (uint32_t off = 1; off < lpa; off <<= 1) {
                c01 += __shfl_xor_sync(FULL_MASK, c01, off);
                c23 += __shfl_xor_sync(FULL_MASK, c23, off);
            }
            for (uint32_t u0 = 0; u0 < SCAN_U; u0 += lpa) {
                const uint32_t u = u0 + sub, i = u * groups + grp;
                const bool head = u < SCAN_U && i < n_atv;
                const uint32_t c2 = (u & 2) ? c23 : c01;
                const uint32_t c = (u & 1) ? c2 >> 16 : c2 & 0xffffu;
                const uint32_t atv = atv0 + i;
                const uint32_t sg = head ? atv >> P.c : 0xffffffffu;  // row * 2^u + frame
                if (head)
                    o.cnt[atv] = (uint16_t)c;
                // one atomic for the tile where its ATVs are of one row-frame
                if (atv0 >> P.c == (atv0 + n_atv - 1) >> P.c) {
                    const uint32_t s = __reduce_add_sync(FULL_MASK, head ? c : 0u);
                    if (lane == 0 && s)
                        atomicAdd(&o.aat[atv0 >> P.c], (unsigned long long)s);
                } else {
                    const unsigned same = __match_any_sync(FULL_MASK, sg);
                    const uint32_t s = __reduce_add_sync(same, head ? c : 0u);
                    if (head && (uint32_t)(__ffs(same) - 1) == lane && s)
                        atomicAdd(&o.aat[sg], (unsigned long long)s);
                }
                const bool sup = head && c >= P.T;
                uint32_t slot = 0;
                if (sup) {
                    slot = atomicAdd(&o.sa_n[sg], 1u);
                    o.sa_x[(size_t)sg * cols + slot] = atv & P.cmask;
                }
                unsigned sbits = __ballot_sync(FULL_MASK, sup);
                while (sbits) {
                    // the g-bit active mask of one super ATV, for Algorithm 5;
                    // all 32 lanes share its words
                    const uint32_t hl = __ffs(sbits) - 1;
                    sbits &= sbits - 1;
                    const uint32_t slot_a = __shfl_sync(FULL_MASK, slot, hl);
                    const uint32_t atv_a = __shfl_sync(FULL_MASK, atv, hl);
                    for (uint32_t k = lane; k < P.mw; k += 32)
                        my_mask[k] = 0;
                    __syncwarp();
                    {
                        constexpr uint32_t F = 32 / WB;
                        for (uint32_t q = lane; q < P.Wd; q += 32) {
                            const uint32_t word = pool[(size_t)atv_a * P.Wd + q];
                            const uint32_t am = L::compress(L::test(word, cd[didx(m, q)], lim));
                            if (am) {
                                const uint32_t pos = q * F, off = pos & 31;
                                atomicOr(&my_mask[pos >> 5], am << off);
                                if (off + F > 32 && (am >> (32 - off)))
                                    atomicOr(&my_mask[(pos >> 5) + 1], am >> (32 - off));
                            }
                        }
                    }
                    __syncwarp();
                    uint32_t *dst = o.sa_mask + ((size_t)(atv_a >> P.c) * cols + slot_a) * P.mw;
                    for (uint32_t k = lane; k < P.mw; k += 32)
                        dst[k] = my_mask[k];
                    __syncwarp();
                }
            }
        }
        // the tile's words are counted and its masks made: its words may change
        if (FUSE)
            __syncwarp();
        if (FUSE && !P.ace) {
            // Algorithm 2 for the next slice on the words of the two refreshed blocks
            for (uint32_t rr = 0; rr < R.n_ranges; rr++) {
                const uint32_t q0 = R.q_lo[rr], len = R.q_hi[rr] - q0 + 1;
                const uint32_t inv = 0xffffffffu / len + 1;  // e / len by a multiply-high, exact for e len < 2^32
                for (uint32_t e = lane; e < n_atv * len; e += 32) {
                    const uint32_t i = len == 1 ? e : __umulhi(e, inv), q = q0 + (e - i * len);
                    uint32_t *wp = pool + (size_t)(atv0 + i) * P.Wd + q;
                    const uint32_t w = *wp;
                    const uint32_t v = cyclic_refresh<WB, BG>(P, w, rd[q], lim);
                    if (v != w)
                        *wp = v;
                }
            }
        }
        if (FUSE && P.ace) {
            // every aging counter loses one
            uint4 *wp = reinterpret_cast<uint4 *>(pool) + (size_t)atv0 * nchunk;
            for (uint32_t e = lane; e < n_atv * nchunk; e += 32) {
                const uint4 v = wp[e];
                wp[e] = BG ? make_uint4(decay_bytes(v.x), decay_bytes(v.y), decay_bytes(v.z), decay_bytes(v.w))
                           : make_uint4(decay_swar<WB>(v.x), decay_swar<WB>(v.y), decay_swar<WB>(v.z),
                                        decay_swar<WB>(v.w));
            }
        }
    }
    let_next_start();
}

// ---------------------------------------------------------------- A3 alone

// Algorithm 2 on every field of a word whose new ACT is 0 or k.
template <int WB>
__device__ __forceinline__ uint32_t refresh_word(const Params &P, uint32_t word, uint32_t q, uint32_t c0n)
{
    constexpr uint32_t F = 32 / WB;
    constexpr uint32_t FM = (1u << WB) - 1;
    uint32_t out = word;
#pragma unroll
    for (uint32_t j = 0; j < F; j++) {
        const uint32_t h = q * F + j;
        if (h < P.g) {
            const uint32_t a = act_of(P, c0n, pos_block(P, h));
            const uint32_t v = (word >> (j * WB)) & FM;
            out = (out & ~(FM << (j * WB))) | (preserve(P, v, a) << (j * WB));
        }
    }
    return out;
}

// One thread per (ATV, word of the two refreshed blocks).
template <int WB>
__global__ void __launch_bounds__(256) refresh_kernel(Params P, uint32_t *pool, const SliceCtl *ctl, uint32_t total_atv)
{
    const Refresh R = ctl->R;
    const uint32_t nw0 = R.n_ranges > 0 ? R.q_hi[0] - R.q_lo[0] + 1 : 0;
    const uint32_t nw1 = R.n_ranges > 1 ? R.q_hi[1] - R.q_lo[1] + 1 : 0;
    const uint64_t nw = nw0 + nw1;
    const uint64_t total = (uint64_t)total_atv * nw;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    if (P.hist) {
        // the window sums lose the phase that leaves the window (c0 - k + 1
        // mod 2k), and the slice counts of the opening slice's phase start
        // again from zero: every AT they counted (set 2k slices ago) has been
        // cleared by now
        const uint32_t c0 = ctl->c0;
        const uint32_t leave = c0 + P.k + 1 >= P.k2 ? c0 + P.k + 1 - P.k2 : c0 + P.k + 1;
        const uint16_t *hl = P.hist + (uint64_t)leave * total_atv;
        uint16_t *hz = P.hist + (uint64_t)R.c0n * total_atv;
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total_atv; i += stride) {
            P.hsum[i] = (uint16_t)(P.hsum[i] - hl[i]);
            hz[i] = 0;
        }
    }
    for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += stride) {
        const uint64_t atv = idx / nw;
        const uint32_t kq = (uint32_t)(idx - atv * nw);
        const uint32_t q = kq < nw0 ? R.q_lo[0] + kq : R.q_lo[1] + (kq - nw0);
        uint32_t *wp = pool + atv * P.Wd + q;
        const uint32_t word = *wp;
        const uint32_t nwd = refresh_word<WB>(P, word, q, R.c0n);
        if (nwd != word)
            *wp = nwd;
    }
}

// Aging counters alone: the full-pool decrement of every slice.
template <int WB>
__global__ void __launch_bounds__(256) ace_decay_kernel(uint4 *pool, uint64_t nvec)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += stride) {
        const uint4 a = pool[v];
        const uint4 b = make_uint4(decay_swar<WB>(a.x), decay_swar<WB>(a.y), decay_swar<WB>(a.z),
                                   decay_swar<WB>(a.w));
        if (a.x != b.x || a.y != b.y || a.z != b.z || a.w != b.w)
            pool[v] = b;
    }
}

}  // namespace

namespace {

template <int NW>
cudaError_t launch_scan_nw(const Params &P, uint32_t w, uint32_t *pool, const ScanWindows &W, bool fuse,
                           const SliceCtl *ctl, int sms, cudaStream_t s)
{
    const uint32_t total = P.r << P.E_log2;
    const uint32_t lpa = scan_lanes(P.Wd / 4);
    const bool bg = byte_guard(w, P.ace ? ASSE_COUNTER_ACE : ASSE_COUNTER_AT, P.k);
    return dispatch_w(w, [&](auto wb) {
        constexpr int WB = decltype(wb)::value;
        auto kern = scan_kernel<WB, true, NW, false>;
        if constexpr (NW == 1) {
            if (!fuse)
                kern = scan_kernel<WB, false, 1, false>;
        }
        if constexpr (WB == 8) {
            if (bg) {
                kern = scan_kernel<8, true, NW, true>;
                if constexpr (NW == 1) {
                    if (!fuse)
                        kern = scan_kernel<8, false, 1, true>;
                }
            }
        }
        const size_t smem = bg ? scan_smem<8, true>(P.Wd, P.mw, W.n) : scan_smem<WB, false>(P.Wd, P.mw, W.n);
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
        const uint32_t per = 32 / lpa * SCAN_U * SCAN_WARPS;  // ATVs of a block's tiles
        const uint32_t want = (total + per - 1) / per;
        const uint32_t full = (uint32_t)sms * resident_blocks(kern, SCAN_THREADS, smem);
        return launch_dependent(kern, dim3(want < full ? want : full), SCAN_THREADS, smem, s, P, pool, W, ctl, total, lpa);
    });
}

}  // namespace

cudaError_t launch_scan(const Params &P, uint32_t w, uint32_t *pool, uint32_t kp, bool fuse, const SliceCtl *ctl,
                        const ScanOut &o, int sms, cudaStream_t s, uint64_t *launches)
{
    ScanWindows W{};
    W.n = 1;
    W.kp[0] = kp;
    W.o[0] = o;
    *launches += 1;
    return launch_scan_nw<1>(P, w, pool, W, fuse, ctl, sms, s);
}

cudaError_t launch_scan_windows(const Params &P, uint32_t w, uint32_t *pool, const ScanWindows &W,
                                const SliceCtl *ctl, int sms, cudaStream_t s, uint64_t *launches)
{
    if (W.n < 1 || W.n > (uint32_t)MAX_WINDOWS)
        return cudaErrorInvalidValue;
    *launches += 1;
    return launch_scan_nw<MAX_WINDOWS>(P, w, pool, W, true, ctl, sms, s);
}

cudaError_t launch_refresh(const Params &P, uint32_t w, uint32_t *pool, const SliceCtl *ctl, int sms, cudaStream_t s,
                           uint64_t *launches)
{
    const uint32_t total = P.r << P.E_log2;
    if (P.ace) {
        const uint64_t nvec = (uint64_t)total * P.Wd / 4;
        *launches += 1;
        return dispatch_w(w, [&](auto wb) {
            constexpr int WB = decltype(wb)::value;
            const uint64_t full = (uint64_t)sms * resident_blocks(ace_decay_kernel<WB>, 256, 0);
            const uint64_t want = (nvec + 255) / 256;
            ace_decay_kernel<WB><<<(unsigned)(want < full ? want : full), 256, 0, s>>>(
                reinterpret_cast<uint4 *>(pool), nvec);
            return cudaGetLastError();
        });
    }
    *launches += 1;
    return dispatch_w(w, [&](auto wb) {
        constexpr int WB = decltype(wb)::value;
        const unsigned grid = (unsigned)sms * resident_blocks(refresh_kernel<WB>, 256, 0);
        refresh_kernel<WB><<<grid, 256, 0, s>>>(P, pool, ctl, total);
        return cudaGetLastError();
    });
}

}  // namespace asse
