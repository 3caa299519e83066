// Host side of the ASSE C ABI (include/asse.h): parameter validation, device
// state, the slice lifecycle and the copies across the process/device
// boundary.  All device work goes through the kernel launchers declared in
// asse_internal.h (asse_ingest.cu, asse_scan.cu, asse_restore.cu, asse_probe.cu).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>

#include "asse_internal.h"
#include "asse_pool_access.h"

using namespace asse;

namespace {

thread_local std::string g_create_error;

// Host input comes in chunks of up to a staging buffer, the last one, if it has more
// than HOST_SPLIT pairs, in two parts: the second of at most HOST_TAIL pairs.  Both
// start at multiples of HOST_ALIGN pairs.
constexpr uint64_t HOST_TAIL = 1ull << 20, HOST_SPLIT = 5ull << 18, HOST_ALIGN = 1ull << 16;

uint64_t host_aligned(uint64_t pairs) { return (pairs + HOST_ALIGN - 1) / HOST_ALIGN * HOST_ALIGN; }

// Pairs of the next chunk, left pairs from the end: a buffer of stage pairs
// (even), or half of what is left where that fits in the two.
uint64_t host_chunk(uint64_t left, uint64_t stage)
{
    if (left <= stage)
        return left;
    const uint64_t half = host_aligned(left / 2);
    return left < 2 * stage && half < stage ? half : stage;
}

// Pairs of the first part of a last chunk of m pairs.
uint64_t host_first(uint64_t m)
{
    return m <= HOST_SPLIT ? m : m < 2 * HOST_TAIL ? HOST_TAIL : host_aligned(m - HOST_TAIL);
}

struct SnapHeader {
    char magic[8];
    uint32_t version;
    uint32_t header_bytes;
    asse_config cfg;
    uint64_t slice;
    uint64_t pool_words;
    uint32_t w, words;
};

}  // namespace

struct asse_pool {
    asse_config cfg{};
    Params P{};
    uint32_t w = 0, F = 0, words_used = 0, blk = 0;
    uint64_t t = 0;
    cudaStream_t stream = nullptr, copy_stream = nullptr;
    cudaEvent_t copied[2] = {nullptr, nullptr}, consumed[2] = {nullptr, nullptr};
    int sms = 0;
    uint32_t *pool = nullptr;
    uint64_t pool_words = 0;
    uint16_t *cnt = nullptr;
    unsigned long long *aat = nullptr;
    uint32_t *sa_n = nullptr, *sa_x = nullptr, *sa_mask = nullptr;
    Tuple *scratch = nullptr;
    uint32_t cap = 0;
    asse_superpoint *csip = nullptr, *report = nullptr;
    uint64_t out_cap = 0;
    Status *status = nullptr;
    Status *status_host = nullptr;
    // the restore of a close also writes the status and the head of the report
    // to pinned host memory (status_host, report_host), so that reading a short
    // report takes one wait, for the close only
    asse_superpoint *report_host = nullptr;
    uint64_t report_host_cap = 0;
    int report_host_valid = 0;
    int captured = 0;  // a graph of the caller's holds a restore of this pool
    cudaEvent_t close_done = nullptr;  // recorded after the last close
    Status *status_read = nullptr;     // pinned, for reading any other status
    // asse_set_timing: events around the scan and the restore of each close
    cudaEvent_t tev[3] = {nullptr, nullptr, nullptr};
    int timing = 0, timed = 0;
    SliceCtl *ctl = nullptr;  // device copy of the slice-dependent launch arguments
    uint32_t *stage[2] = {nullptr, nullptr};
    uint64_t stage_pairs = 0;
    uint32_t stage_next = 0;  // the staging buffer of the next chunk
    uint64_t slice_pairs = 0;   // ingested into the open slice
    uint64_t claim_pairs = ~0ull;  // so many at most go through a key table the pool could do without
    uint64_t blind_pairs = ~0ull;  // and, in a larger pool, are set without reading what they change
    uint32_t *q_aips = nullptr;
    asse_superpoint *q_out = nullptr;
    uint64_t q_cap = 0;
    // outputs of windows 1 .. MAX_WINDOWS-1 of a multi-window close (window 0
    // uses the buffers above), allocated on first use
    struct Win {
        unsigned char *block = nullptr;  // holds all of the device ones
        uint16_t *cnt = nullptr;
        unsigned long long *aat = nullptr;
        uint32_t *sa_n = nullptr, *sa_x = nullptr, *sa_mask = nullptr;
        Status *status = nullptr;
        asse_superpoint *csip = nullptr, *report = nullptr;
        Tuple *scratch = nullptr;
        Status *status_host = nullptr;
        asse_superpoint *report_host = nullptr;
    } win[MAX_WINDOWS - 1];
    int stream_changed = 0;  // asse_set_stream since the last scan, restore or close
    uint32_t n_windows = 1, sel = 0;  // windows of the last close, the one the readers return
    int scanned = 0, refreshed = 0, restored = 0, ingested = 0;
    uint32_t scan_kp = 0;
    uint64_t scan_slice = 0;
    uint64_t launches = 0;
    std::string err;
};

namespace {

int fail(asse_pool *p, int code, const std::string &msg)
{
    if (p)
        p->err = msg;
    else
        g_create_error = msg;
    return code;
}

int cuda_fail(asse_pool *p, cudaError_t e, const char *what)
{
    return fail(p, ASSE_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define CK(p, call)                                   \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess)                        \
            return cuda_fail((p), e_, #call);         \
    } while (0)

uint64_t inverse_mod(uint64_t a, uint64_t m)
{
    __int128 t0 = 0, t1 = 1, r0 = (__int128)m, r1 = (__int128)a;
    while (r1 != 0) {
        __int128 q = r0 / r1, tmp;
        tmp = r0 - q * r1; r0 = r1; r1 = tmp;
        tmp = t0 - q * t1; t0 = t1; t1 = tmp;
    }
    if (t0 < 0)
        t0 += (__int128)m;
    return (uint64_t)t0;
}

int validate(const asse_config *c, std::string &why)
{
    char buf[256];
    auto bad = [&](const char *m) { why = m; return ASSE_EINVAL; };
    if (!c)
        return bad("cfg is NULL");
    if (c->counter != ASSE_COUNTER_AT && c->counter != ASSE_COUNTER_ACE && c->counter != ASSE_COUNTER_AT_ALIGNED &&
        c->counter != ASSE_COUNTER_AT_HIST)
        return bad("counter must be ASSE_COUNTER_AT, ASSE_COUNTER_ACE, ASSE_COUNTER_AT_ALIGNED or ASSE_COUNTER_AT_HIST");
    if (c->k < 1 || c->k > 127)
        return bad("k must be in [1, 127]");
    if (c->g < 2 * c->k || c->g > 4096)
        return bad("g must be in [2k, 4096]");
    if (c->r < 2 || c->r > 8)
        return bad("r must be in [2, 8]");
    if (c->c < 1 || c->c > 16 || c->u > 8 || c->c + c->u > 24)
        return bad("need 1 <= c <= 16, u <= 8, c + u <= 24");
    const uint32_t W = 32 - c->u;
    if (c->c > W || c->s < 1 || c->s > c->c || c->s * (c->r - 1) >= W) {
        snprintf(buf, sizeof buf, "need c <= 32-u, 1 <= s <= c and s*(r-1) < 32-u (c=%u s=%u r=%u u=%u)", c->c, c->s,
                 c->r, c->u);
        why = buf;
        return ASSE_EINVAL;
    }
    if (c->c + c->s * (c->r - 1) < W)
        return bad("column windows do not cover LBS: need c + s*(r-1) >= 32-u (completeness, Sec. 4.1)");
    if (c->A < 2)
        return bad("A must be in [2, 2^32)");
    if ((c->bh_a & 1) == 0)
        return bad("bh_a must be odd");
    if (c->theta < 1)
        return bad("theta must be >= 1");
    if (c->key_table > ASSE_KEYS_OFF)
        return bad("key_table must be ASSE_KEYS_AUTO, ASSE_KEYS_ON or ASSE_KEYS_OFF");
    if (c->cluster != ASSE_CLUSTER_AUTO && c->cluster != 1 && c->cluster != 2 && c->cluster != 4 && c->cluster != 8)
        return bad("cluster must be ASSE_CLUSTER_AUTO, 1, 2, 4 or 8");
    // the scan and the estimates keep an entry per word of an ATV in shared
    // memory (of up to four windows and the refresh: 40 KB for 512 words)
    const uint32_t w = packed_width(c->counter, c->k);
    if ((c->g + 32 / w - 1) / (32 / w) > 512)
        return bad("an ATV must fit in 512 words: need g <= 512 * floor(32 / w)");
    return ASSE_OK;
}

ScanOut scan_out(asse_pool *p)
{
    ScanOut o;
    o.cnt = p->cnt;
    o.aat = p->aat;
    o.sa_n = p->sa_n;
    o.sa_x = p->sa_x;
    o.sa_mask = p->sa_mask;
    o.status = p->status;
    return o;
}

// Scan outputs, status and lists of window m of the last close.
ScanOut scan_out_w(asse_pool *p, uint32_t m)
{
    if (m == 0)
        return scan_out(p);
    const asse_pool::Win &w = p->win[m - 1];
    ScanOut o;
    o.cnt = w.cnt;
    o.aat = w.aat;
    o.sa_n = w.sa_n;
    o.sa_x = w.sa_x;
    o.sa_mask = w.sa_mask;
    o.status = w.status;
    return o;
}

asse_superpoint *list_w(asse_pool *p, uint32_t m, bool reported)
{
    if (m == 0)
        return reported ? p->report : p->csip;
    return reported ? p->win[m - 1].report : p->win[m - 1].csip;
}

__global__ void init_pool_kernel(uint32_t *pool, uint64_t nwords, uint32_t Wd, uint32_t words_used,
                                 uint32_t full_word, uint32_t last_word)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nwords; i += stride) {
        const uint32_t q = (uint32_t)(i % Wd);
        pool[i] = q + 1 < words_used ? full_word : (q + 1 == words_used ? last_word : 0u);
    }
}

// On a stream set since, work that rewrites what the last close wrote waits for
// that close.
int wait_last_close(asse_pool *p)
{
    if (p->stream_changed)
        CK(p, cudaStreamWaitEvent(p->stream, p->close_done, 0));
    p->stream_changed = 0;
    return ASSE_OK;
}

// Where the restore of window m of a close writes for the host.
HostReport host_report_w(asse_pool *p, uint32_t m)
{
    return m == 0 ? HostReport{p->status_host, p->report_host, p->report_host_cap}
                  : HostReport{p->win[m - 1].status_host, p->win[m - 1].report_host, p->report_host_cap};
}

// Whether the pool's stream is being captured.  The graph may be replayed at any
// time, also while the host reads a report, so a restore in it writes device
// memory only (HostReport()), records no event, and from then on the readers take
// status and lists from the device.
int check_capture(asse_pool *p, bool *capturing)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    CK(p, cudaStreamIsCapturing(p->stream, &st));
    *capturing = st != cudaStreamCaptureStatusNone;
    return ASSE_OK;
}

// After the restore of a close or of asse_restore is queued.
int note_restore(asse_pool *p, bool capturing)
{
    if (capturing)
        p->captured = 1;
    else
        CK(p, cudaEventRecord(p->close_done, p->stream));
    p->report_host_valid = !p->captured;
    return ASSE_OK;
}

int reset_close_state(asse_pool *p)
{
    ScanWindows W{};
    W.n = 1;
    W.o[0] = scan_out(p);
    CK(p, launch_reset(W, p->cfg.r * p->P.nf, p->stream, &p->launches));
    return ASSE_OK;
}

int check_kp(asse_pool *p, uint32_t kp)
{
    if (kp < 1 || kp > p->cfg.k)
        return fail(p, ASSE_EINVAL, "kp must be in [1, k]");
    return ASSE_OK;
}

int read_list(asse_pool *p, bool reported, asse_superpoint *out, uint64_t cap, uint64_t *n_out, int where)
{
    if (!p || !n_out)
        return fail(p, ASSE_EINVAL, "NULL argument");
    if (!p->restored)
        return fail(p, ASSE_ESTATE, "no restore since the last scan");
    const HostReport host = host_report_w(p, p->sel);
    // the close is done, on whichever stream; later work already queued (the
    // next batch) keeps running
    CK(p, cudaEventSynchronize(p->close_done));
    if (!p->report_host_valid) {
        CK(p, cudaMemcpyAsync(p->status_read, scan_out_w(p, p->sel).status, sizeof(Status), cudaMemcpyDeviceToHost,
                              p->stream));
        CK(p, cudaStreamSynchronize(p->stream));
    }
    const Status st = p->report_host_valid ? *host.status : *p->status_read;
    if (st.overflow) {
        *n_out = st.needed;
        char buf[200];
        snprintf(buf, sizeof buf, "restore needed %llu column tuples in one frame, restore_cap is %u",
                 (unsigned long long)st.needed, p->cap);
        return fail(p, ASSE_ECAPACITY, buf);
    }
    const uint64_t n = reported ? st.n_report : st.n_csip;
    *n_out = n;
    const uint64_t m = n < cap ? n : cap;
    if (m > 0 && reported && where != ASSE_DEVICE && p->report_host_valid && m <= p->report_host_cap) {
        if (!out)
            return fail(p, ASSE_EINVAL, "out is NULL");
        memcpy(out, host.report, m * sizeof(asse_superpoint));
    } else if (m > 0) {
        if (!out)
            return fail(p, ASSE_EINVAL, "out is NULL");
        CK(p, cudaMemcpyAsync(out, list_w(p, p->sel, reported), m * sizeof(asse_superpoint),
                              where == ASSE_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, p->stream));
        CK(p, cudaStreamSynchronize(p->stream));  // also of a device buffer, which any stream may read next
    }
    if (n > cap)
        return fail(p, ASSE_ECAPACITY, "output capacity smaller than the list");
    return ASSE_OK;
}

void free_all(asse_pool *p)
{
    cudaFree(p->pool);
    cudaFree(p->cnt);
    cudaFree(p->aat);
    cudaFree(p->sa_n);
    cudaFree(p->sa_x);
    cudaFree(p->sa_mask);
    cudaFree(p->scratch);
    cudaFree(p->csip);
    cudaFree(p->report);
    cudaFree(p->status);
    cudaFree(p->ctl);
    cudaFree(p->P.keys);
    cudaFree(p->P.hist);
    cudaFree(p->P.hsum);
    cudaFree(p->stage[0]);
    cudaFree(p->stage[1]);
    cudaFree(p->q_aips);
    cudaFree(p->q_out);
    for (auto &w : p->win) {
        if (w.status_host)
            cudaFreeHost(w.status_host);
        cudaFree(w.block);
    }
    if (p->status_host)
        cudaFreeHost(p->status_host);
    if (p->status_read)
        cudaFreeHost(p->status_read);
    if (p->report_host)
        cudaFreeHost(p->report_host);
    if (p->close_done)
        cudaEventDestroy(p->close_done);
    for (cudaEvent_t ev : p->tev)
        if (ev)
            cudaEventDestroy(ev);
    for (int i = 0; i < 2; i++) {
        if (p->copied[i])
            cudaEventDestroy(p->copied[i]);
        if (p->consumed[i])
            cudaEventDestroy(p->consumed[i]);
    }
    if (p->copy_stream)
        cudaStreamDestroy(p->copy_stream);
}

}  // namespace

namespace asse {

int pool_restore_view(asse_pool *p, RestoreView *v)
{
    if (!p->scanned)
        return fail(p, ASSE_ESTATE, "restore needs a scan of the open slice");
    p->report_host_valid = 0;
    v->P = p->P;
    v->o = scan_out_w(p, p->sel);
    v->stream = p->stream;
    v->launches = &p->launches;
    return ASSE_OK;
}

int pool_fail(asse_pool *p, int code, const std::string &msg) { return fail(p, code, msg); }

int pool_enqueue_close(asse_pool *p, uint32_t kp, const HostReport &host, bool timed)
{
    if (int rc = reset_close_state(p))
        return rc;
    if (timed)
        CK(p, cudaEventRecord(p->tev[0], p->stream));
    // counts from the slice counts, or from every AT; either way with the
    // refresh for the next slice fused in
    if (p->P.hist)
        CK(p, launch_hist_scan(p->P, p->w, p->pool, kp, true, p->ctl, scan_out(p), p->sms, p->stream, &p->launches));
    else
        CK(p, launch_scan(p->P, p->w, p->pool, kp, true, p->ctl, scan_out(p), p->sms, p->stream, &p->launches));
    if (timed)
        CK(p, cudaEventRecord(p->tev[1], p->stream));
    CK(p, launch_restore(p->P, scan_out(p), p->scratch, p->cap, p->csip, p->report, p->out_cap, p->stream,
                         &p->launches, p->ctl, host));
    if (timed)
        CK(p, cudaEventRecord(p->tev[2], p->stream));
    return ASSE_OK;
}

int pool_enqueue_scan(asse_pool *p, uint32_t kp)
{
    if (int rc = reset_close_state(p))
        return rc;
    if (p->P.hist)
        CK(p, launch_hist_scan(p->P, p->w, p->pool, kp, false, p->ctl, scan_out(p), p->sms, p->stream,
                               &p->launches));
    else
        CK(p, launch_scan(p->P, p->w, p->pool, kp, false, p->ctl, scan_out(p), p->sms, p->stream, &p->launches));
    return ASSE_OK;
}

int pool_enqueue_restore_refresh(asse_pool *p, const HostReport &host)
{
    CK(p, launch_restore(p->P, scan_out(p), p->scratch, p->cap, p->csip, p->report, p->out_cap, p->stream,
                         &p->launches, nullptr, host));
    CK(p, launch_refresh(p->P, p->w, p->pool, p->ctl, p->sms, p->stream, &p->launches));
    CK(p, launch_advance_ctl(p->P, p->ctl, p->stream, &p->launches));
    return ASSE_OK;
}

FeatureView pool_feature_view_device(asse_pool *p, uint32_t kp)
{
    FeatureView v{};
    v.P = p->P;
    v.w = p->w;
    v.pool = p->pool;
    v.c0 = 0;
    v.kp = kp;
    v.ctl = p->ctl;
    v.aat = p->aat;
    v.cnt = p->cnt;
    v.stream = p->stream;
    v.launches = &p->launches;
    v.sms = p->sms;
    return v;
}

void pool_after_close(asse_pool *p, uint32_t kp)
{
    p->report_host_valid = 0;
    p->n_windows = 1;
    p->sel = 0;
    p->report_host_valid = 0;
    p->scanned = 1;
    p->restored = 1;
    p->refreshed = 1;
    p->ingested = 0;
    p->scan_kp = kp;
    p->scan_slice = p->t;
    p->t += 1;
    p->slice_pairs = 0;
}

int pool_enqueue_ingest(asse_pool *p, const uint32_t *pairs_dev, const unsigned long long *n_dev)
{
    CK(p, launch_ingest(p->P, p->w, p->pool, pairs_dev, 0, n_dev, p->ctl, p->sms, p->stream, &p->launches));
    p->ingested = 1;
    return ASSE_OK;
}

uint32_t pool_restore_cap(const asse_pool *p) { return p->cap; }

// Whether a pool that fits in the L2 cache takes a key table it could do
// without (key_table AUTO): for plain timestamps and aging counters, whose
// claimed keys are then set without being read, a claim in place of the r pool
// words pays at every size measured (8.4 M pairs a slice on a 92 MB pool: 89
// against 103 us; 65,536 on 0.5 MB: 6.2 against 8.4 us).  With slice counts the
// words are read either way and the claim only adds an access (146 against 142
// us), so those pools take none.
static bool key_table_pays(const asse_config *cfg)
{
    return cfg->key_table == ASSE_KEYS_AUTO && cfg->counter != ASSE_COUNTER_AT_HIST;
}

// Pairs of a slice up to which such a table is used: two per AT of a row, four
// where the fields are bytes, whose blind set is one store.  A slice of many more
// distinct keys than fields finds most fields set, and its keys push one another
// out of the table, so that claiming each and setting it blind costs more than
// reading its words.  With / without the table, us, 8.4 M pairs of random hosts:
// 4 pairs per AT 457 / 208 (five bits, 4,096 ATVs a row), 64 per AT 517 / 132 (four
// bits, 1,024); of the workloads' Zipf hosts 102 / 88 and 113 / 68.  At one pair
// per AT it is 463 / 411 and 95 / 98, at a half 69 / 57 and 22 / 29.
static uint64_t claim_pairs(const Params &P, uint32_t w)
{
    return ((uint64_t)P.g << P.E_log2) * (w == 8 ? 4 : 2);
}

// Pairs of a slice of a pool larger than L2 up to which claimed keys are set
// blind: one per 10 ATs of a row, or 5 where the fields are bytes.  While most
// words are touched once, a set without a read spares an access; later ones find
// the word read and changed already, and a blind set of a field that holds the
// value still writes it.  Blind / read, us: 352 MB of five-bit fields, a pair per
// 30 ATs 66 / 76, 10 170 / 164, 5 319 / 303; 1 GB of bytes, 30 129 / 168, 10 361 /
// 387, 8 449 / 466; 512 MB of bytes, 5 332 / 323, 4 407 / 396.
static uint64_t blind_pairs(const Params &P, uint32_t w)
{
    return ((uint64_t)P.g << P.E_log2) / (w == 8 ? 5 : 10);
}

// log2 entries of the key table asse_create cannot do without on the current
// device (0: none).
static uint32_t needed_keys_log2(uint32_t mode, uint64_t n_atv, uint64_t pool_bytes)
{
    int dev = 0, l2 = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) != cudaSuccess)
        cudaGetLastError();
    return key_table_log2(n_atv, pool_bytes, (unsigned long long)l2, mode);
}

bool pool_needs_keys(const asse_config *cfg)
{
    const uint32_t F = 32 / packed_width(cfg->counter, cfg->k);
    const uint64_t Wd = ((cfg->g + F - 1) / F + 7) / 8 * 8;
    const uint64_t n_atv = (uint64_t)cfg->r << (cfg->c + cfg->u);
    return needed_keys_log2(cfg->key_table, n_atv, n_atv * Wd * 4) != 0;
}

// Device bytes asse_create allocates for cfg (the server's admission unit;
// a server's pools take no key table they could do without, so that its
// budget admits as many streams either way).
uint64_t pool_device_bytes(const asse_config *cfg)
{
    const uint32_t w = packed_width(cfg->counter, cfg->k);
    const uint32_t F = 32 / w;
    const uint64_t Wd = ((cfg->g + F - 1) / F + 7) / 8 * 8;
    const uint64_t n_atv = (uint64_t)cfg->r << (cfg->c + cfg->u);
    const uint64_t nf = 1ull << cfg->u, nseg = cfg->r * nf, mw = (cfg->g + 31) / 32;
    const uint64_t cap = cfg->restore_cap ? cfg->restore_cap : 4096;
    const uint64_t stage = cfg->max_batch ? (cfg->max_batch + 1) / 2 * 2 : (4ull << 20);
    const uint32_t klg = needed_keys_log2(cfg->key_table, n_atv, n_atv * Wd * 4);
    const uint64_t hist = cfg->counter == ASSE_COUNTER_AT_HIST ? ((uint64_t)2 * cfg->k + 1) * n_atv * 2 : 0;
    return hist + n_atv * Wd * 4 + n_atv * 2 + nseg * (8 + 4) + n_atv * 4 + n_atv * mw * 4 + nf * 2 * cap * sizeof(Tuple) +
           2 * cap * nf * sizeof(asse_superpoint) + sizeof(Status) + sizeof(SliceCtl) + 2 * stage * 8 +
           (klg ? sizeof(unsigned long long) << klg : 0);
}

uint64_t pool_list_cap(const asse_pool *p) { return p ? p->out_cap : 0; }

int pool_feature_view(asse_pool *p, FeatureView *v)
{
    if (!p->scanned || p->refreshed || p->ingested || p->scan_slice != p->t)
        return fail(p, ASSE_ESTATE, "features need a scan of the open slice and no refresh or ingest since");
    v->P = p->P;
    v->w = p->w;
    v->pool = p->pool;
    v->c0 = (uint32_t)(p->t % (2 * p->cfg.k));
    v->kp = p->scan_kp;
    v->ctl = nullptr;
    v->aat = p->aat;
    v->cnt = p->cnt;
    v->stream = p->stream;
    v->launches = &p->launches;
    v->sms = p->sms;
    return ASSE_OK;
}

}  // namespace asse

extern "C" {

const char *asse_strerror(int status)
{
    switch (status) {
    case ASSE_OK: return "ASSE_OK";
    case ASSE_EINVAL: return "ASSE_EINVAL";
    case ASSE_ENOMEM: return "ASSE_ENOMEM";
    case ASSE_ECAPACITY: return "ASSE_ECAPACITY";
    case ASSE_ECUDA: return "ASSE_ECUDA";
    case ASSE_ESTATE: return "ASSE_ESTATE";
    case 6: return "ASSE_EAGAIN";
    case ASSE_ETIMEOUT: return "ASSE_ETIMEOUT";
    default: return "unknown status";
    }
}

const char *asse_last_error(const asse_pool *pool)
{
    return pool ? pool->err.c_str() : g_create_error.c_str();
}

uint64_t asse_launches(const asse_pool *pool) { return pool ? pool->launches : 0; }

int asse_create(const asse_config *cfg, void *stream, asse_pool **out)
{
    if (!out)
        return fail(nullptr, ASSE_EINVAL, "out is NULL");
    *out = nullptr;
    std::string why;
    if (validate(cfg, why) != ASSE_OK)
        return fail(nullptr, ASSE_EINVAL, why);
    asse_pool *p = new (std::nothrow) asse_pool();
    if (!p)
        return fail(nullptr, ASSE_ENOMEM, "host allocation failed");
    p->cfg = *cfg;
    p->stream = (cudaStream_t)stream;
    const uint32_t k = cfg->k;
    const bool ace = cfg->counter == ASSE_COUNTER_ACE;
    p->w = packed_width(cfg->counter, k);
    p->F = 32 / p->w;
    p->words_used = (cfg->g + p->F - 1) / p->F;
    const uint32_t Wd = (p->words_used + 7) / 8 * 8;
    // the aligned variant is one block of g ATs (every AT has ACT C0)
    p->blk = cfg->counter == ASSE_COUNTER_AT_ALIGNED ? cfg->g : cfg->g / (2 * k);
    Params &P = p->P;
    P.k = k;
    P.k2 = 2 * k;
    P.g = cfg->g;
    P.r = cfg->r;
    P.c = cfg->c;
    P.u = cfg->u;
    P.W = 32 - cfg->u;
    P.E_log2 = cfg->c + cfg->u;
    P.Wd = Wd;
    P.A = cfg->A;
    P.cmask = (1u << cfg->c) - 1;
    P.theta = cfg->theta;
    const double g = (double)cfg->g;
    P.T = (uint32_t)std::ceil(g - g * std::exp(-(double)cfg->theta / g));
    P.ace = ace ? 1 : 0;
    P.nf = 1u << cfg->u;
    P.mw = (cfg->g + 31) / 32;
    P.blk = p->blk;
    P.F = p->F;
    P.blk_magic = ((1ull << 32) + p->blk - 1) / p->blk;
    // timestamps with 2k blocks keep each pair of blocks that one refresh
    // checks side by side (block_slot)
    P.paired = (cfg->counter == ASSE_COUNTER_AT || cfg->counter == ASSE_COUNTER_AT_HIST) ? 1 : 0;
    P.Ainv = inverse_mod(cfg->A, 4294967311ull);
    P.bh_a = cfg->bh_a;
    P.bh_b = cfg->bh_b;
    P.cl = cfg->cluster == ASSE_CLUSTER_AUTO ? 1u : cfg->cluster;
    P.blind = 1;
    for (uint32_t i = 0; i < 8; i++)
        P.xshift[i] = i < cfg->r ? 2 * P.W - cfg->c - cfg->s * i : 0;
    p->cap = cfg->restore_cap ? cfg->restore_cap : 4096;
    p->out_cap = (uint64_t)p->cap * P.nf;
    p->stage_pairs = cfg->max_batch ? (cfg->max_batch + 1) / 2 * 2 : (4ull << 20);

    const uint64_t n_atv = (uint64_t)cfg->r << P.E_log2;
    p->pool_words = n_atv * Wd;
    const size_t nseg = (size_t)cfg->r * P.nf;
    const size_t slots = (size_t)cfg->r << P.E_log2;  // super-ATV slots: every ATV of a row-frame
    cudaError_t e = cudaSuccess;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
        delete p;
        return cuda_fail(nullptr, e, "cudaGetDevice/cudaDeviceGetAttribute");
    }
    auto alloc = [&](void **ptr, size_t bytes) {
        if (e == cudaSuccess)
            e = cudaMalloc(ptr, bytes);
    };
    alloc((void **)&p->pool, p->pool_words * 4);
    alloc((void **)&p->cnt, n_atv * sizeof(uint16_t));
    alloc((void **)&p->aat, nseg * sizeof(unsigned long long));
    alloc((void **)&p->sa_n, nseg * sizeof(uint32_t));
    alloc((void **)&p->sa_x, slots * sizeof(uint32_t));
    alloc((void **)&p->sa_mask, slots * P.mw * sizeof(uint32_t));
    alloc((void **)&p->scratch, (size_t)P.nf * 2 * p->cap * sizeof(Tuple));
    alloc((void **)&p->csip, p->out_cap * sizeof(asse_superpoint));
    alloc((void **)&p->report, p->out_cap * sizeof(asse_superpoint));
    alloc((void **)&p->status, sizeof(Status));
    alloc((void **)&p->ctl, sizeof(SliceCtl));
    int l2 = 0;
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
    P.klg = key_table_log2(n_atv, p->pool_words * 4, (unsigned long long)l2, cfg->key_table);
    if (P.klg)
        alloc((void **)&P.keys, sizeof(unsigned long long) << P.klg);
    if (p->pool_words * 4 > (uint64_t)l2)
        p->blind_pairs = blind_pairs(P, p->w);
    if (cfg->counter == ASSE_COUNTER_AT_HIST) {
        alloc((void **)&P.hist, (size_t)2 * k * n_atv * sizeof(uint16_t));
        alloc((void **)&P.hsum, (size_t)n_atv * sizeof(uint16_t));
    }
    alloc((void **)&p->stage[0], p->stage_pairs * 8);
    alloc((void **)&p->stage[1], p->stage_pairs * 8);
    // the key table of a pool that fits in L2 only makes its ingest faster: the
    // pool does without one that cannot be allocated
    if (e == cudaSuccess && !P.klg && key_table_pays(cfg)) {
        P.klg = key_table_log2(n_atv, p->pool_words * 4, (unsigned long long)l2, ASSE_KEYS_ON);
        if (cudaMalloc((void **)&P.keys, sizeof(unsigned long long) << P.klg) != cudaSuccess) {
            cudaGetLastError();
            P.keys = nullptr;
            P.klg = 0;
        } else {
            p->claim_pairs = claim_pairs(P, p->w);
        }
    }
    if (e == cudaSuccess)
        e = cudaMallocHost((void **)&p->status_host, sizeof(Status));
    if (e == cudaSuccess)
        e = cudaMallocHost((void **)&p->status_read, sizeof(Status));
    p->report_host_cap = p->out_cap < 4096 ? p->out_cap : 4096;
    if (e == cudaSuccess)
        e = cudaMallocHost((void **)&p->report_host, p->report_host_cap * sizeof(asse_superpoint));
    if (e == cudaSuccess)
        e = cudaEventCreateWithFlags(&p->close_done, cudaEventDisableTiming);
    if (e == cudaSuccess)
        e = cudaStreamCreateWithFlags(&p->copy_stream, cudaStreamNonBlocking);
    for (int i = 0; i < 2 && e == cudaSuccess; i++) {
        e = cudaEventCreateWithFlags(&p->copied[i], cudaEventDisableTiming);
        if (e == cudaSuccess)
            e = cudaEventCreateWithFlags(&p->consumed[i], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) {
        const bool oom = e == cudaErrorMemoryAllocation;
        cudaGetLastError();
        free_all(p);
        delete p;
        return oom ? fail(nullptr, ASSE_ENOMEM, "device allocation failed")
                   : cuda_fail(nullptr, e, "asse_create");
    }
    // InitAT: every field of every ATV at its inactive value (2k, or 0 for
    // aging counters); fields past g and padding words hold 0.
    const uint32_t fill = ace ? 0u : 2 * k;
    uint32_t full_word = 0, last_word = 0;
    for (uint32_t j = 0; j < p->F; j++) {
        full_word |= fill << (j * p->w);
        if ((p->words_used - 1) * p->F + j < cfg->g)
            last_word |= fill << (j * p->w);
    }
    init_pool_kernel<<<p->sms * 4, 256, 0, p->stream>>>(p->pool, p->pool_words, Wd, p->words_used, full_word,
                                                          last_word);
    p->launches++;
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemsetAsync(p->status, 0, sizeof(Status), p->stream);
    if (e == cudaSuccess && P.keys)
        e = cudaMemsetAsync(P.keys, 0xff, sizeof(unsigned long long) << P.klg, p->stream);
    if (e == cudaSuccess && P.hist)
        e = cudaMemsetAsync(P.hist, 0, (size_t)2 * k * n_atv * sizeof(uint16_t), p->stream);
    if (e == cudaSuccess && P.hsum)
        e = cudaMemsetAsync(P.hsum, 0, (size_t)n_atv * sizeof(uint16_t), p->stream);
    const SliceCtl ctl0 = slice_ctl(P, 0);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p->ctl, &ctl0, sizeof ctl0, cudaMemcpyHostToDevice, p->stream);

    if (e == cudaSuccess)
        e = cudaStreamSynchronize(p->stream);
    if (e != cudaSuccess) {
        free_all(p);
        delete p;
        return cuda_fail(nullptr, e, "pool initialisation");
    }
    *out = p;
    return ASSE_OK;
}

void asse_destroy(asse_pool *pool)
{
    if (!pool)
        return;
    cudaStreamSynchronize(pool->stream);
    cudaStreamSynchronize(pool->copy_stream);
    cudaEventSynchronize(pool->close_done);  // of another stream, if it was changed
    free_all(pool);
    delete pool;
}

int asse_set_stream(asse_pool *pool, void *stream)
{
    if (!pool)
        return ASSE_EINVAL;
    pool->stream = (cudaStream_t)stream;
    pool->stream_changed = 1;
    return ASSE_OK;
}

int asse_ingest(asse_pool *p, const uint32_t *pairs, uint64_t n, int where)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (n == 0)
        return ASSE_OK;
    if (!pairs)
        return fail(p, ASSE_EINVAL, "pairs is NULL");
    p->ingested = 1;  // the pool no longer matches the last scan
    if (where != ASSE_HOST && where != ASSE_DEVICE)
        return fail(p, ASSE_EINVAL, "where must be ASSE_HOST or ASSE_DEVICE");
    if (where == ASSE_DEVICE && ((uintptr_t)pairs & 15) != 0)
        return fail(p, ASSE_EINVAL, "device pairs must be 16-byte aligned");
    // (a captured close opens slices that the host does not see)
    p->slice_pairs = p->captured ? n : p->slice_pairs + n;
    Params P = p->P;
    if (p->slice_pairs > p->claim_pairs)
        P.keys = nullptr;
    P.blind = p->slice_pairs <= p->blind_pairs ? 1 : 0;
    if (where == ASSE_DEVICE) {
        CK(p, launch_ingest(P, p->w, p->pool, pairs, n, nullptr, p->ctl, p->sms, p->stream, &p->launches));
        return ASSE_OK;
    }
    // Double-buffered staging (Sec. 4.4): the copy engines move chunk i+1 on
    // the copy stream while chunk i is ingested on the pool's stream, and the
    // call returns once the last chunk is copied, so the ingest and the close
    // of this slice overlap the caller's next transfer.  (The kernel could
    // read pinned memory in place over the host link, but that keeps the SMs
    // busy for the whole transfer: 19.3 against 23.1 G pairs/s end to end on
    // the link workload with the next batch queued before each report.)
    // Chunks of a whole buffer, through the two in turn, from one call to the
    // next: each boundary costs the copy engine about 2 us (chunks of 1 Mi
    // pairs, the next batch queued before each report: 23.7 against 25.3 G
    // pairs/s on the long workload, 23.1 against 23.9 on the link).  What follows
    // the last copy, though, is the ingest of what it brought, so the last chunk
    // comes in two parts (host_first; 8 Mi pairs ingested, closed and reported
    // before the next: 422 -> 399 us).
    cudaEvent_t last = nullptr;
    uint32_t part = 0;
    for (uint64_t off = 0; off < n;) {
        const uint32_t b = p->stage_next;
        const uint64_t m = host_chunk(n - off, p->stage_pairs);
        const uint64_t first = m == n - off ? host_first(m) : m;
        CK(p, cudaStreamWaitEvent(p->copy_stream, p->consumed[b], 0));
        for (uint64_t at = 0, k = first; at < m; at += k, k = m - at, part ^= 1) {
            uint32_t *dst = p->stage[b] + 2 * at;
            last = p->copied[part];
            CK(p, cudaMemcpyAsync(dst, pairs + 2 * (off + at), k * 8, cudaMemcpyHostToDevice, p->copy_stream));
            CK(p, cudaEventRecord(last, p->copy_stream));
            CK(p, cudaStreamWaitEvent(p->stream, last, 0));
            CK(p, launch_ingest(P, p->w, p->pool, dst, k, nullptr, p->ctl, p->sms, p->stream, &p->launches));
        }
        CK(p, cudaEventRecord(p->consumed[b], p->stream));
        p->stage_next = b ^ 1;
        off += m;
    }
    // the caller may reuse its host buffer once every chunk has been copied
    CK(p, cudaEventSynchronize(last));
    return ASSE_OK;
}

int asse_scan(asse_pool *p, uint32_t kp)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (int rc = check_kp(p, kp))
        return rc;
    if (int rc = wait_last_close(p))
        return rc;
    if (int rc = pool_enqueue_scan(p, kp))
        return rc;
    p->n_windows = 1;
    p->sel = 0;
    p->report_host_valid = 0;
    p->scanned = 1;
    p->refreshed = 0;
    p->restored = 0;
    p->ingested = 0;
    p->scan_kp = kp;
    p->scan_slice = p->t;
    return ASSE_OK;
}

int asse_restore(asse_pool *p)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (!p->scanned)
        return fail(p, ASSE_ESTATE, "restore needs a scan of the open slice");
    p->report_host_valid = 0;
    bool capturing = false;
    if (int rc = check_capture(p, &capturing))
        return rc;
    if (int rc = wait_last_close(p))
        return rc;
    CK(p, launch_restore(p->P, scan_out(p), p->scratch, p->cap, p->csip, p->report, p->out_cap, p->stream,
                         &p->launches, nullptr, capturing ? HostReport() : host_report_w(p, 0)));
    p->restored = 1;
    return note_restore(p, capturing);
}

int asse_advance(asse_pool *p)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    CK(p, launch_refresh(p->P, p->w, p->pool, p->ctl, p->sms, p->stream, &p->launches));
    CK(p, launch_advance_ctl(p->P, p->ctl, p->stream, &p->launches));
    p->t += 1;
    p->slice_pairs = 0;
    p->refreshed = 1;
    return ASSE_OK;
}

int asse_close_slice(asse_pool *p, uint32_t kp)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (int rc = check_kp(p, kp))
        return rc;
    bool capturing = false;
    if (int rc = check_capture(p, &capturing))
        return rc;
    if (int rc = wait_last_close(p))
        return rc;
    if (int rc = pool_enqueue_close(p, kp, capturing ? HostReport() : host_report_w(p, 0), p->timing != 0))
        return rc;
    pool_after_close(p, kp);
    p->timed = p->timing;
    return note_restore(p, capturing);
}

int asse_close_slice_multi(asse_pool *p, const uint32_t *kps, uint32_t n_windows)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (!kps || n_windows < 1 || n_windows > (uint32_t)MAX_WINDOWS)
        return fail(p, ASSE_EINVAL, "need kps and 1 <= n_windows <= ASSE_MAX_WINDOWS");
    for (uint32_t m = 0; m < n_windows; m++)
        if (int rc = check_kp(p, kps[m]))
            return rc;
    // outputs of the extra windows, on first use
    const uint64_t n_atv = (uint64_t)p->cfg.r << p->P.E_log2;
    const size_t nseg = (size_t)p->cfg.r * p->P.nf;
    for (uint32_t m = 1; m < n_windows; m++) {
        asse_pool::Win &w = p->win[m - 1];
        if (w.cnt)
            continue;
        // one allocation, in 256-byte aligned parts
        size_t bytes = 0;
        auto part = [&](size_t n) {
            const size_t at = bytes;
            bytes += (n + 255) / 256 * 256;
            return at;
        };
        const size_t cnt = part(n_atv * sizeof(uint16_t)), aat = part(nseg * sizeof(unsigned long long)),
                     sa_n = part(nseg * sizeof(uint32_t)), sa_x = part(n_atv * sizeof(uint32_t)),
                     sa_mask = part(n_atv * p->P.mw * sizeof(uint32_t)), status = part(sizeof(Status)),
                     csip = part(p->out_cap * sizeof(asse_superpoint)),
                     report = part(p->out_cap * sizeof(asse_superpoint)),
                     scratch = part((size_t)p->P.nf * 2 * p->cap * sizeof(Tuple));
        cudaError_t e = cudaMalloc((void **)&w.block, bytes);
        // the status, then the head of the report
        if (e == cudaSuccess)
            e = cudaMallocHost((void **)&w.status_host, 256 + p->report_host_cap * sizeof(asse_superpoint));
        if (e != cudaSuccess) {
            cudaGetLastError();
            cudaFree(w.block);
            w = asse_pool::Win();
            return e == cudaErrorMemoryAllocation ? fail(p, ASSE_ENOMEM, "window outputs: device allocation failed")
                                                  : cuda_fail(p, e, "window outputs");
        }
        w.report_host = reinterpret_cast<asse_superpoint *>(reinterpret_cast<char *>(w.status_host) + 256);
        w.cnt = reinterpret_cast<uint16_t *>(w.block + cnt);
        w.aat = reinterpret_cast<unsigned long long *>(w.block + aat);
        w.sa_n = reinterpret_cast<uint32_t *>(w.block + sa_n);
        w.sa_x = reinterpret_cast<uint32_t *>(w.block + sa_x);
        w.sa_mask = reinterpret_cast<uint32_t *>(w.block + sa_mask);
        w.status = reinterpret_cast<Status *>(w.block + status);
        w.csip = reinterpret_cast<asse_superpoint *>(w.block + csip);
        w.report = reinterpret_cast<asse_superpoint *>(w.block + report);
        w.scratch = reinterpret_cast<Tuple *>(w.block + scratch);
    }
    bool capturing = false;
    if (int rc = check_capture(p, &capturing))
        return rc;
    if (int rc = wait_last_close(p))
        return rc;
    ScanWindows W{};
    RestoreWindows out{};
    W.n = n_windows;
    for (uint32_t m = 0; m < n_windows; m++) {
        W.kp[m] = kps[m];
        W.o[m] = scan_out_w(p, m);
        out.w[m] = RestoreOut{m == 0 ? p->scratch : p->win[m - 1].scratch, list_w(p, m, false), list_w(p, m, true),
                              capturing ? HostReport() : host_report_w(p, m)};
    }
    CK(p, launch_reset(W, p->cfg.r * p->P.nf, p->stream, &p->launches));
    if (p->P.hist) {
        // one count pass per window over the slice counts, then the restore,
        // the refresh (with the zeroing of the next slice's counts) and the next slice
        for (uint32_t m = 0; m < n_windows; m++)
            CK(p, launch_hist_scan(p->P, p->w, p->pool, kps[m], false, p->ctl, W.o[m], p->sms, p->stream,
                                   &p->launches));
        CK(p, launch_restores(p->P, W, p->cap, out, p->out_cap, p->stream, &p->launches));
        CK(p, launch_refresh(p->P, p->w, p->pool, p->ctl, p->sms, p->stream, &p->launches));
        CK(p, launch_advance_ctl(p->P, p->ctl, p->stream, &p->launches));
    } else {
        CK(p, launch_scan_windows(p->P, p->w, p->pool, W, p->ctl, p->sms, p->stream, &p->launches));
        CK(p, launch_restores(p->P, W, p->cap, out, p->out_cap, p->stream, &p->launches, p->ctl));
    }
    pool_after_close(p, kps[0]);
    p->n_windows = n_windows;
    return note_restore(p, capturing);
}

int asse_set_timing(asse_pool *p, int on)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    for (int i = 0; i < 3 && on; i++)
        if (!p->tev[i])
            CK(p, cudaEventCreate(&p->tev[i]));
    p->timing = on ? 1 : 0;
    p->timed = 0;
    return ASSE_OK;
}

int asse_close_timing(asse_pool *p, float *ms)
{
    if (!p || !ms)
        return fail(p, ASSE_EINVAL, "pool and ms must not be NULL");
    if (!p->timed)
        return fail(p, ASSE_ESTATE, "no close since asse_set_timing(pool, 1)");
    CK(p, cudaEventSynchronize(p->tev[2]));
    CK(p, cudaEventElapsedTime(&ms[0], p->tev[0], p->tev[1]));
    CK(p, cudaEventElapsedTime(&ms[1], p->tev[1], p->tev[2]));
    return ASSE_OK;
}

int asse_select_window(asse_pool *p, uint32_t window)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (window >= p->n_windows)
        return fail(p, ASSE_EINVAL, "window index beyond the windows of the last close");
    p->sel = window;
    return ASSE_OK;
}

int asse_estimate(asse_pool *p, const uint32_t *aips, uint64_t n, asse_superpoint *out, int where)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (!p->scanned || p->refreshed || p->ingested || p->scan_slice != p->t)
        return fail(p, ASSE_ESTATE, "estimate needs a scan of the open slice and no refresh since");
    if (n == 0)
        return ASSE_OK;
    if (!aips || !out)
        return fail(p, ASSE_EINVAL, "NULL argument");
    const uint32_t c0 = (uint32_t)(p->t % (2 * p->cfg.k));
    if (where == ASSE_DEVICE) {
        CK(p, launch_estimate(p->P, p->w, p->pool, c0, p->scan_kp, p->aat, aips, n, out, p->sms, p->stream,
                              &p->launches));
        return ASSE_OK;
    }
    if (n > p->q_cap) {
        cudaFree(p->q_aips);
        cudaFree(p->q_out);
        p->q_aips = nullptr;
        p->q_out = nullptr;
        p->q_cap = 0;
        CK(p, cudaMalloc((void **)&p->q_aips, n * sizeof(uint32_t)));
        CK(p, cudaMalloc((void **)&p->q_out, n * sizeof(asse_superpoint)));
        p->q_cap = n;
    }
    CK(p, cudaMemcpyAsync(p->q_aips, aips, n * sizeof(uint32_t), cudaMemcpyHostToDevice, p->stream));
    CK(p, launch_estimate(p->P, p->w, p->pool, c0, p->scan_kp, p->aat, p->q_aips, n, p->q_out, p->sms, p->stream,
                          &p->launches));
    CK(p, cudaMemcpyAsync(out, p->q_out, n * sizeof(asse_superpoint), cudaMemcpyDeviceToHost, p->stream));
    CK(p, cudaStreamSynchronize(p->stream));
    return ASSE_OK;
}

int asse_report(asse_pool *p, asse_superpoint *out, uint64_t cap, uint64_t *n_out, int where)
{
    return read_list(p, true, out, cap, n_out, where);
}

int asse_candidates(asse_pool *p, asse_superpoint *out, uint64_t cap, uint64_t *n_out, int where)
{
    return read_list(p, false, out, cap, n_out, where);
}

int asse_counts(asse_pool *p, uint16_t *out, int where)
{
    if (!p || !out)
        return fail(p, ASSE_EINVAL, "NULL argument");
    if (!p->scanned)
        return fail(p, ASSE_ESTATE, "no scan");
    const size_t bytes = ((size_t)p->cfg.r << p->P.E_log2) * sizeof(uint16_t);
    CK(p, cudaMemcpyAsync(out, scan_out_w(p, p->sel).cnt, bytes,
                          where == ASSE_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, p->stream));
    if (where != ASSE_DEVICE)
        CK(p, cudaStreamSynchronize(p->stream));
    return ASSE_OK;
}

int asse_loads(asse_pool *p, uint64_t *out)
{
    if (!p || !out)
        return fail(p, ASSE_EINVAL, "NULL argument");
    if (!p->scanned)
        return fail(p, ASSE_ESTATE, "no scan");
    CK(p, cudaMemcpyAsync(out, scan_out_w(p, p->sel).aat, (size_t)p->cfg.r * p->P.nf * sizeof(uint64_t),
                          cudaMemcpyDeviceToHost, p->stream));
    CK(p, cudaStreamSynchronize(p->stream));
    return ASSE_OK;
}

int asse_info(const asse_pool *p, asse_pool_info *out)
{
    if (!p || !out)
        return ASSE_EINVAL;
    out->w = p->w;
    out->fields = p->F;
    out->words = p->P.Wd;
    out->E = 1u << p->P.E_log2;
    out->threshold = p->P.T;
    out->block = p->blk;
    out->k = p->P.k;
    out->paired = p->P.paired;
    out->slice = p->t;
    out->pool_words = p->pool_words;
    out->pool = p->pool;
    return ASSE_OK;
}

int asse_read_pool(asse_pool *p, uint32_t *out, int where)
{
    if (!p || !out)
        return fail(p, ASSE_EINVAL, "NULL argument");
    CK(p, cudaMemcpyAsync(out, p->pool, p->pool_words * 4,
                          where == ASSE_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, p->stream));
    if (where != ASSE_DEVICE)
        CK(p, cudaStreamSynchronize(p->stream));
    return ASSE_OK;
}

int asse_snapshot(asse_pool *p, void *dst, uint64_t cap, uint64_t *n_out)
{
    if (!p || !n_out)
        return fail(p, ASSE_EINVAL, "NULL argument");
    const uint64_t need = sizeof(SnapHeader) + p->pool_words * 4;
    *n_out = need;
    if (!dst)
        return ASSE_OK;
    if (cap < need)
        return fail(p, ASSE_ECAPACITY, "snapshot buffer too small");
    SnapHeader h;
    memset(&h, 0, sizeof h);
    memcpy(h.magic, "ASSEPOOL", 8);
    h.version = 1;
    h.header_bytes = sizeof(SnapHeader);
    h.cfg = p->cfg;
    h.slice = p->t;
    h.pool_words = p->pool_words;
    h.w = p->w;
    h.words = p->P.Wd;
    memcpy(dst, &h, sizeof h);
    CK(p, cudaMemcpyAsync((char *)dst + sizeof h, p->pool, p->pool_words * 4, cudaMemcpyDeviceToHost, p->stream));
    CK(p, cudaStreamSynchronize(p->stream));
    return ASSE_OK;
}

int asse_probe_random_reads(asse_pool *p, uint64_t n_reads, uint64_t *n_issued)
{
    if (!p)
        return fail(nullptr, ASSE_EINVAL, "pool is NULL");
    if (n_reads > (1ull << 34))
        return fail(p, ASSE_EINVAL, "n_reads must be at most 2^34");
    uint64_t issued = 0;
    if (n_reads > 0)
        CK(p, launch_random_reads(p->pool, p->pool_words, n_reads, p->sms, p->stream, &p->launches, &issued));
    if (n_issued)
        *n_issued = issued;
    return ASSE_OK;
}

int asse_load(asse_pool *p, const void *src, uint64_t n)
{
    if (!p || !src)
        return fail(p, ASSE_EINVAL, "NULL argument");
    p->report_host_valid = 0;
    SnapHeader h;
    if (n < sizeof h)
        return fail(p, ASSE_EINVAL, "image too small");
    memcpy(&h, src, sizeof h);
    if (memcmp(h.magic, "ASSEPOOL", 8) != 0 || h.version != 1 || h.header_bytes != sizeof h)
        return fail(p, ASSE_EINVAL, "not an ASSE pool image");
    const asse_config &a = h.cfg, &b = p->cfg;
    if (a.k != b.k || a.theta != b.theta || a.g != b.g || a.r != b.r || a.c != b.c || a.u != b.u || a.s != b.s ||
        a.A != b.A || a.bh_a != b.bh_a || a.bh_b != b.bh_b || a.counter != b.counter ||
        h.pool_words != p->pool_words || h.w != p->w || h.words != p->P.Wd)
        return fail(p, ASSE_EINVAL, "image was written by a pool with another configuration");
    if (n < sizeof h + p->pool_words * 4)
        return fail(p, ASSE_EINVAL, "image truncated");
    CK(p, cudaMemcpyAsync(p->pool, (const char *)src + sizeof h, p->pool_words * 4, cudaMemcpyHostToDevice,
                          p->stream));
    const SliceCtl c = slice_ctl(p->P, h.slice);
    CK(p, cudaMemcpyAsync(p->ctl, &c, sizeof c, cudaMemcpyHostToDevice, p->stream));
    // the key table describes the replaced state
    if (p->P.keys)
        CK(p, cudaMemsetAsync(p->P.keys, 0xff, sizeof(unsigned long long) << p->P.klg, p->stream));
    // slice counts of a histogram pool, counted again from the loaded words
    if (p->P.hist)
        CK(p, launch_hist_rebuild(p->P, p->w, p->pool, p->ctl, p->sms, p->stream, &p->launches));
    CK(p, cudaStreamSynchronize(p->stream));
    p->t = h.slice;
    p->slice_pairs = 0;
    p->scanned = p->restored = p->refreshed = 0;
    return ASSE_OK;
}

}  // extern "C"
