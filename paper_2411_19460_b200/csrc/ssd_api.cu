// Host side of libssd: argument validation, workspace layout, and the segment driver that runs
// Algorithm 1 (forward, storing the state at every segment boundary) and Algorithm 2 (backward,
// segments right to left: recompute from the stored state, back-propagate, hand dh to the left)
// for one SSD layer.  Checkpoint memory is set by the segment length: the scratch holds the chunk
// states of ONE segment, the boundary buffer one state per segment.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <vector>

#include "ssd_internal.h"
#include "ssd_sm100.cuh"

namespace ssd {

static thread_local int g_last_cuda = 0;

// ---- optional instrumentation: launch counter and per-kernel-kind CUDA-event timing ----
static std::atomic<long long> g_launches{0};
struct ProfEvent { int kind; cudaEvent_t a, b; };
static bool g_prof_on = false;
static std::vector<ProfEvent> g_prof_pool;
static size_t g_prof_used = 0;

static const char *const kKindNames[KIND_COUNT] = {
    "chunk_state", "state_pass_fwd", "chunk_scan_fwd", "dstate_contrib",
    "state_pass_bwd", "bwd_dx", "bwd_dC", "bwd_dB", "bwd_finish", "final_dAdD", "glue", "decode_step", "bwd_dBdC", "conv1d", "gated_norm"};

static ProfEvent *prof_begin(int kind, cudaStream_t st) {
    if (!g_prof_on) return nullptr;
    if (g_prof_used == g_prof_pool.size()) {
        ProfEvent ev;
        ev.kind = kind;
        if (cudaEventCreate(&ev.a) != cudaSuccess || cudaEventCreate(&ev.b) != cudaSuccess) return nullptr;
        g_prof_pool.push_back(ev);
    }
    ProfEvent *ev = &g_prof_pool[g_prof_used++];
    ev->kind = kind;
    cudaEventRecord(ev->a, st);
    return ev;
}
static void prof_end(ProfEvent *ev, cudaStream_t st) {
    if (ev) cudaEventRecord(ev->b, st);
}

// Scratch regions of one call.  What the kernels of neighbouring segments touch at the same time exists more than once on the
// tensor-core path: the records and states that the forward chain leaves three times, so that it runs two segments ahead (with
// two copies it waited for the large kernels two segments back: 24 heads, 2048-token segments, 52 us a segment instead of 36),
// the rest twice; where they are small, once more each (chain_copies).
static const int kChainCopies = 4, kGradCopies = 3;      // at most
struct Layout {
    size_t status, hcarry, Gst, gcarry, dAp, dDp;
    size_t rec[kChainCopies], Hbf[kChainCopies], cs[2], dtT[2], Hst[2], cbt[2];
    size_t Gbf[kGradCopies], ghdot[kGradCopies], ddt_dir[kGradCopies], rho[kGradCopies], rho2[kGradCopies], psi[kGradCopies], psi2[kGradCopies],
        pB[kGradCopies], pC[kGradCopies];
    size_t total;
};

// All the copies of the per-segment scratch pay only when there are segments enough to pipeline; two or three long segments get
// a second copy of the forward chain's output and one of the rest.
static const int kMinSegmentsForTwins = 4;

struct Plan {
    int B, L, H, P, N, G, Q, seg, nseg, ncs, nct, hpg, nsl, dtype;   // Q: steps per chunk (split path) or block (tensor cores)
    bool use_tc, serial;
    bool keep_cb;          // split path: the scratch holds C B^T (always, except in the built-in one)
    int64_t x_bs, dt_bs, bc_bs;
    size_t esz;
};

// Head ranges per group for the dB/dC kernel, whose CTAs are (block, head range).  The launches of two neighbouring segments run
// at the same time, beside the other kernels, so what counts is the time on the SMs, (CTAs) x (eight head-times of set-up and
// output plus the heads of the range), once three launches of 32 blocks (or the whole sequence, if it is shorter) make a wave;
// below that the time of one CTA.  A function of the sequence alone, so that the summation order of dB/dC does not depend on the
// segment length, and therefore the best for one segment length, 4096.  The backward of 32768 steps, us, with a wave out of one
// launch of 32 blocks, of two, three and six:
//   80 heads, seg 1024: 1580 1735 2052 3008   2048: 1317 1249 1330 1762   4096: 1182 1192 1107 1227   8192: 1244 1186 1146 1097
//   24 heads             853  988  986 1289          759  658  658  809          685  588  595  566          650  639  640  580
// (8 groups of 10 heads: the same within 2 %.)
static const int kBcBlocks = 96;
static int bc_head_split(int blocks, int groups, int hpg) {
    int best = 1;
    double best_t = -1;
    const int max_split = hpg >= 4 ? hpg / 4 : 1;
    for (int ns = 1; ns <= max_split; ++ns) {
        const int hps = (hpg + ns - 1) / ns;
        if ((hpg + hps - 1) / hps != ns) continue;      // would leave an empty range
        const double waves = (double)(blocks < kBcBlocks ? blocks : kBcBlocks) * groups * ns / kNumSMs;
        // a short sequence is one launch or two, whose last wave takes as long as a full one
        const double t = (blocks < kBcBlocks ? ceil(waves) : waves > 1 ? waves : 1) * (8 + hps);
        if (best_t < 0 || t < best_t) { best_t = t; best = ns; }
    }
    return best;
}

// The same for the kernel of the split path, whose ranges have Q/64 + 3 slots each and as many CTAs as the chunk has tile pairs and
// twice its tiles.  A range costs its CTAs the last products and the slices, some four heads' worth, so ranges of eight heads where
// 1024 steps (the choice may not depend on the segments) then have 200 CTAs, of four or two below that, of one where two leave next to
// none.  Backward, us, with ranges of one, two, four, eight heads (CTAs of 1024 steps with eight):
//   fp32, 2 x 4096 steps of 24 heads, chunk 256 (432)       -  934  813  752       4096 of 24, chunk 256 (216)    -  537  468  444
//   bf16, 2 x 8192 of 32 heads, chunk 128 (448)             -  842  800  750       4096 of 24, chunk 128, segments of 512 (168)  -  245  238  300
//   4096 of 8 heads, chunk 256, one segment (72)          230  185  165    -       1024 of 4, chunk 64 (48)      70   78   98    -
// Long sequences (64 chunks and more, counted per group): no more slots than two per head, what a slice for each head would take (2 x
// 8192 steps of 8 heads 711 -> 618 us, 8192 of 80 heads in 8 groups 2852 -> 2332 us and 985 -> 381 MB of scratch).
static int simt_head_ranges(const Plan &pl) {
    const int nrt = pl.Q / 64, slots = nrt + 3, roles = nrt * (nrt + 1) / 2 + 2 * nrt;
    const int chunks = pl.nct < 1024 / pl.Q ? pl.nct : 1024 / pl.Q;
    auto ctas = [&](int per) { return (long long)pl.B * chunks * pl.G * roles * ((pl.hpg + per - 1) / per); };
    int per = 8;
    while (per > 2 && ctas(per) < 200) per /= 2;
    if (per == 2 && ctas(2) < 150) per = 1;
    int n = (pl.hpg + per - 1) / per;
    if (pl.B * pl.nct * pl.G >= 64 && n * slots > 2 * pl.hpg) n = 2 * pl.hpg >= slots ? 2 * pl.hpg / slots : 1;
    const int hps = (pl.hpg + n - 1) / n;
    return (pl.hpg + hps - 1) / hps;                    // no empty range
}

static int make_plan(const ssd_shape_t *s, Plan &pl) {
    if (!s) return SSD_EINVAL;
    if (s->B <= 0 || s->L <= 0 || s->H <= 0 || s->P <= 0 || s->N <= 0 || s->G <= 0 || s->chunk <= 0 ||
        s->seg < 0)
        return SSD_EINVAL;
    if (s->H % s->G) return SSD_EINVAL;
    if (s->dtype != SSD_DTYPE_F32 && s->dtype != SSD_DTYPE_BF16) return SSD_EUNSUPPORTED;
    if (s->P != 64) return SSD_EUNSUPPORTED;
    if (s->N != 64 && s->N != 128) return SSD_EUNSUPPORTED;
    if (s->chunk != 64 && s->chunk != 128 && s->chunk != 256) return SSD_EUNSUPPORTED;
    if (s->L % s->chunk) return SSD_EINVAL;
    const int seg = s->seg == 0 ? s->L : (s->seg > s->L ? s->L : s->seg);
    if (seg % s->chunk) return SSD_EINVAL;
    if (s->x_bstride < 0 || s->dt_bstride < 0 || s->bc_bstride < 0) return SSD_EINVAL;
    pl.B = s->B; pl.L = s->L; pl.H = s->H; pl.P = s->P; pl.N = s->N; pl.G = s->G;
    pl.use_tc = tc_supported(s->dtype, s->flags, s->P, s->N, s->chunk, s->H / s->G);
    pl.Q = pl.use_tc ? kTcBlock : s->chunk;
    pl.seg = seg;
    pl.nseg = (s->L + seg - 1) / seg;
    pl.ncs = seg / pl.Q;
    pl.nct = s->L / pl.Q;
    pl.hpg = s->H / s->G;
    pl.dtype = s->dtype;
    pl.esz = s->dtype == SSD_DTYPE_BF16 ? 2 : 4;
    pl.x_bs = s->x_bstride ? s->x_bstride : (int64_t)s->L * s->H * s->P;
    pl.dt_bs = s->dt_bstride ? s->dt_bstride : (int64_t)s->L * s->H;
    pl.bc_bs = s->bc_bstride ? s->bc_bstride : (int64_t)s->L * s->G * s->N;
    if (pl.x_bs < (int64_t)s->L * s->H * s->P || pl.dt_bs < (int64_t)s->L * s->H ||
        pl.bc_bs < (int64_t)s->L * s->G * s->N)
        return SSD_EINVAL;
    if (((size_t)s->H * s->P * pl.esz) % 16 || ((size_t)s->G * s->N * pl.esz) % 16 ||
        ((size_t)pl.x_bs * pl.esz) % 16 || ((size_t)pl.bc_bs * pl.esz) % 16)
        return SSD_EALIGN;
    pl.serial = (s->flags & SSD_FLAG_SERIAL) != 0;
    pl.keep_cb = true;
    // Partial slices of the dB/dC head sums: one per CTA head range
    pl.nsl = pl.use_tc ? bc_head_split(pl.B * pl.nct, pl.G, pl.hpg) : simt_head_ranges(pl) * (pl.Q / 64 + 3);
    return SSD_OK;
}

// split path: whether the sums of a segment ride in a launch of its neighbour.  In the forward that takes second copies of states
// and C B^T, up to 64 MiB of them: in four segments, fp32, N = 128, chunk 256, they are worth 12 % at 8 MiB (24 heads, 2048 steps, 324 ->
// 286 us), 6 % at 24 MiB (80 heads, 2048 steps, 854 -> 800), 4 % at 46 MiB (4096 steps, 1628 -> 1558).
static bool simt_overlap(const Plan &pl, bool bwd) {
    const size_t copy = ((size_t)pl.B * pl.H * (pl.ncs + 1) * pl.P * pl.N + (size_t)pl.B * pl.ncs * pl.G * pl.Q * pl.Q) * sizeof(float);
    return pl.nseg > 1 && (bwd || copy <= (size_t)64 << 20);
}

// split path: whether the readers of a state make it from the sums of the segment's other chunks.  That saves a launch per segment and
// direction, some 6 us, and reads 16 KB tiles that a state pass would have added up.  Forward + backward, us, with passes and without,
// by the number of those tiles a launch of y: 24 (1024 steps of 4 heads) 146 and 129, 288 (4096 of 24 heads) 526 and 453, 768 (2 x 4096 of
// 8, N = 128) 550 and 540, 896 316 and 282, 1344 (8192 of 24 heads) 1287 and 1387, 2304 1112 and 1133.
static bool simt_readers(const Plan &pl) {
    const long long tiles = (long long)pl.ncs * (pl.ncs - 1) / 2 * (pl.Q / 64) * pl.B * pl.H * (pl.N / 64);
    return !pl.use_tc && pl.ncs <= kReaderChunks && tiles <= 1024;
}

// Copies of what the forward chain leaves, and of what the gradient chain and the large kernels leave (tensor-core path).  A copy comes
// back when its segment's tail is done: chain, dB/dC beside dx, tail and the hand-overs take 77 us of 24 heads and 2048 steps, so with
// two copies a segment can start every 38 us, while the gradient chain alone takes 28; the recompute likewise with three.  Where
// the copies are small that latency is the bound, and there is one more of each: backward of 8 segments of that size 352 -> 316 us,
// 16 of 1024 steps 513 -> 437 us (64 heads: 915 -> 716, 80: 1055 -> 820); 64 heads, 8 of 2048 (16 MiB) 602 -> 527 us;
// with 80 heads and 4096 steps, where SM time is the bound, 8 segments take the same with and without.
static const size_t kSmallStates = (size_t)16 << 20;
static bool small_states(const Plan &pl) { return (size_t)pl.B * pl.H * pl.ncs * pl.P * pl.N * 2 <= kSmallStates; }
static int chain_copies(const Plan &pl, bool bwd) {
    return pl.nseg >= kMinSegmentsForTwins ? (bwd && small_states(pl) ? 4 : 3) : pl.nseg > 1 ? 2 : 1;
}
static int grad_copies(const Plan &pl) { return pl.nseg >= kMinSegmentsForTwins ? (small_states(pl) ? 3 : 2) : 1; }

// `twins`: whether the second and third copies may exist at all (not for callers that keep every kernel in order on one
// stream: SSD_FLAG_SERIAL and the built-in scratch of ssd_fwd_static_ws).
static void make_layout(const Plan &pl, int op, Layout &lo, bool twins) {
    const size_t PN = (size_t)pl.P * pl.N, BH = (size_t)pl.B * pl.H;
    const size_t vec = BH * pl.ncs * pl.Q * sizeof(float);
    const size_t st = BH * (pl.ncs + 1) * PN * sizeof(float), stb = BH * pl.ncs * PN * 2;
    const bool bwd = (op == SSD_OP_BWD_SEG);
    const int ncp = twins ? chain_copies(pl, bwd) : 1, ngc = twins && pl.use_tc ? grad_copies(pl) : 1;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    auto take2 = [&](size_t (&r)[2], size_t bytes, bool two) {
        r[0] = take(bytes);
        r[1] = two ? take(bytes) : r[0];
    };
    auto take_n = [&](auto &r, size_t bytes, int copies) {
        for (int i = 0; i < (int)(sizeof(r) / sizeof(r[0])); ++i) r[i] = i < copies ? take(bytes) : r[i % copies];
    };
    memset(&lo, 0, sizeof(lo));
    lo.status = take(256);
    const int vcopies = bwd && small_states(pl) ? 3 : 2;      // of the vectors; of the records one more
    if (!bwd) lo.hcarry = take(BH * PN * sizeof(float));      // the backward starts every segment from `boundary`
    // the vectors and records (a fraction of the states) exist as often for any number of segments
    if (pl.use_tc) {
        take_n(lo.rec, BH * pl.ncs * REC_FLOATS * sizeof(float), twins ? vcopies + 1 : 1);
        take_n(lo.Hbf, stb, ncp);
    } else {
        // two copies where a launch works on two neighbouring segments: y beside the next segment's sums, and in the backward,
        // where only the step sizes meet, the finishing steps beside them
        const bool two = twins && simt_overlap(pl, bwd);
        take2(lo.cs, vec, two && !bwd);
        take2(lo.dtT, vec, two);
        take2(lo.Hst, st, two && !bwd);
        if (pl.keep_cb) take2(lo.cbt, (size_t)pl.B * pl.ncs * pl.G * pl.Q * pl.Q * sizeof(float), two && !bwd);
    }
    if (bwd) {
        lo.gcarry = take(BH * PN * sizeof(float));
        if (pl.use_tc) take_n(lo.Gbf, stb, ngc);
        else lo.Gst = take(st);
        take_n(lo.ghdot, BH * pl.ncs * 16 * sizeof(float), ngc);
        const int vn = twins && pl.use_tc ? vcopies : 1;
        take_n(lo.ddt_dir, vec, vn);
        const size_t vec_tiles = pl.use_tc ? vec : vec * (pl.Q / 64);
        take_n(lo.rho, vec_tiles, vn);
        take_n(lo.rho2, vec, vn);
        take_n(lo.psi, vec_tiles, vn);
        take_n(lo.psi2, vec, vn);
        const size_t part = (size_t)pl.B * pl.seg * pl.G * pl.nsl * pl.N * sizeof(float);
        take_n(lo.pC, part, ngc);
        if (pl.use_tc) take_n(lo.pB, part, ngc);
        lo.dAp = take(BH * pl.nct * sizeof(float));
        lo.dDp = take(BH * pl.nct * 4 * sizeof(float));
    }
    lo.total = o;
}

// Layout of the built-in scratch: in order on one stream, so no second copies, and C B^T only if there is room for it.  What fits
// is then what fitted when every tile of y made its own part of C B^T: 8 bytes a step and head, and the states.
static void make_static_layout(Plan &pl, Layout &lo) {
    make_layout(pl, SSD_OP_FWD, lo, false);
    if (lo.total <= (size_t)SSD_STATIC_WS_BYTES || pl.use_tc) return;
    pl.keep_cb = false;
    make_layout(pl, SSD_OP_FWD, lo, false);
}

// Whether two buffers of n and m floats (null: none) have a byte in common
static bool overlap_of(const float *a, size_t n, const float *b, size_t m) { return a && b && a < b + m && b < a + n; }

static bool misaligned(const void *p) { return ((uintptr_t)p & 15u) != 0; }

static int check_device() {
    static thread_local int cached_dev = -1;
    static thread_local int cached_ok = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) { g_last_cuda = (int)e; return SSD_ECUDA; }
    if (dev != cached_dev) {
        int major = 0;
        e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (e != cudaSuccess) { g_last_cuda = (int)e; return SSD_ECUDA; }
        cached_dev = dev;
        cached_ok = (major == 10);
    }
    return cached_ok ? SSD_OK : SSD_EDEVICE;
}

// Helper streams per (host thread, device) with the events that fork them off the caller's stream and join them
// back: s[4] recomputes a segment's chunk states (in the forward: the whole state chain is on s[0], y of odd segments on s[1]), s[0] runs the
// state-gradient part of the chain, s[1] / s[3] the dB/dC kernel of even / odd segments beside dx on the caller's
// stream, s[2] a segment's finishing kernel.  Created on first use, never
// destroyed (they hold no device memory); the caller's stream stays the only one the caller has to order
// against.  A wait refers to the last record before it, so an event that is waited for before it is recorded again serves every
// segment; those that are waited for some segments later go round with the copies of the scratch regions.
struct SideStreams {
    int dev = -1;
    cudaStream_t s[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // gradient chain | dB/dC, even | tails | dB/dC, odd | recompute
    cudaEvent_t start = nullptr;
    cudaEvent_t chain_done = nullptr, big_done[kChainCopies] = {}, tail_done[kChainCopies] = {}, rec_done = nullptr, join = nullptr, dx_done = nullptr;
};
static SideStreams *side_streams() {
    static thread_local std::vector<SideStreams> all;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    for (auto &a : all)
        if (a.dev == dev) return &a;
    SideStreams a;
    a.dev = dev;
    for (int i = 0; i < 5; ++i)
        if (cudaStreamCreateWithFlags(&a.s[i], cudaStreamNonBlocking) != cudaSuccess) return nullptr;
    std::vector<cudaEvent_t *> evs = {&a.start, &a.chain_done, &a.rec_done, &a.join, &a.dx_done};
    for (int i = 0; i < kChainCopies; ++i) {
        evs.push_back(&a.big_done[i]);
        evs.push_back(&a.tail_done[i]);
    }
    for (cudaEvent_t *ev : evs)
        if (cudaEventCreateWithFlags(ev, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    all.push_back(a);
    return &all.back();
}

#define SSD_TRY(expr)                                   \
    do {                                                \
        cudaError_t e__ = (expr);                       \
        if (e__ != cudaSuccess) {                       \
            g_last_cuda = (int)e__;                     \
            return SSD_ECUDA;                           \
        }                                               \
    } while (0)

// one kernel launch of kind `kind` on stream `st`
#define SSD_LAUNCH(kind, expr)                          \
    do {                                                \
        ProfEvent *pe__ = prof_begin(kind, st);         \
        cudaError_t e__ = (expr);                       \
        prof_end(pe__, st);                             \
        g_launches.fetch_add(1, std::memory_order_relaxed); \
        if (e__ != cudaSuccess) {                       \
            g_last_cuda = (int)e__;                     \
            return SSD_ECUDA;                           \
        }                                               \
    } while (0)

// Points the kernels at copy kc of the regions that the forward chain writes and copy k of the others.
static void select_copy(const Layout &lo, void *ws, int kc, int k, SegParams &sp) {
    char *w = (char *)ws;
    auto at = [&](size_t r) { return r ? (float *)(w + r) : nullptr; };
    auto f = [&](const auto &r) { return at(r[k < (int)(sizeof(r) / sizeof(r[0])) ? k : 0]); };
    sp.rec = at(lo.rec[kc]);
    sp.cs = f(lo.cs);
    sp.dtT = sp.rec ? sp.rec + REC_DT : f(lo.dtT);
    sp.dt_stride = sp.rec ? (int)REC_FLOATS : sp.Q;
    sp.Hbf = (__nv_bfloat16 *)at(lo.Hbf[kc]);
    sp.Hst = f(lo.Hst);
    sp.cbt = f(lo.cbt);
    sp.Gbf = (__nv_bfloat16 *)f(lo.Gbf);
    sp.ghdot = f(lo.ghdot);
    sp.ddt_dir = f(lo.ddt_dir);
    sp.rho = f(lo.rho);
    sp.rho2 = f(lo.rho2);
    sp.psi = f(lo.psi);
    sp.psi2 = f(lo.psi2);
    sp.pB = f(lo.pB);
    sp.pC = f(lo.pC);
}

static void fill_params(const Plan &pl, const Layout &lo, void *ws, SegParams &sp) {
    memset(&sp, 0, sizeof(sp));
    sp.B = pl.B; sp.L = pl.L; sp.H = pl.H; sp.P = pl.P; sp.N = pl.N; sp.G = pl.G; sp.Q = pl.Q;
    sp.inv_H = inverse_of(pl.H);
    sp.hpg = pl.hpg; sp.ncs = pl.ncs; sp.nct = pl.nct; sp.nsl = pl.nsl;
    sp.ndd = pl.use_tc ? 4 : pl.Q / 64;
    sp.scan_ctas = kNumSMs;
    sp.chain_heads = 1;
    sp.ngh = pl.use_tc ? 8 : pl.P * pl.N / kStatePassElems;
    sp.x_bs = pl.x_bs; sp.dt_bs = pl.dt_bs; sp.bc_bs = pl.bc_bs;
    char *w = (char *)ws;
    sp.status = (unsigned int *)(w + lo.status);
    sp.tiles = pl.use_tc ? 0 : pl.Q / 64;
    sp.hcarry = lo.hcarry ? (float *)(w + lo.hcarry) : nullptr;
    sp.Gst = (float *)(w + lo.Gst);
    sp.gcarry = (float *)(w + lo.gcarry);
    sp.dAp = (float *)(w + lo.dAp);
    sp.dDp = (float *)(w + lo.dDp);
    select_copy(lo, ws, 0, 0, sp);
}

static void set_segment(const Plan &pl, int k, SegParams &sp) {
    sp.t0 = k * pl.seg;
    const int len = (pl.L - sp.t0 < pl.seg) ? pl.L - sp.t0 : pl.seg;
    sp.nc = len / pl.Q;
    sp.inv_nc = inverse_of(sp.nc);
    sp.c0 = sp.t0 / pl.Q;
}

// Heads per CTA of the forward chain.  Two where a CTA per head would not fit one wave, and in a pipelined backward with heads
// enough: the other kernels of a segment take longer than the chain there, so that its SM time counts and not its latency
// (4096 steps of 80 heads: 60 us on 40 SMs against 38 on 80; in the forward, where only y is beside it, 63 us a segment
// against 57).  Backward of 65536 steps, us, one head and two per CTA: 64 heads, seg 4096 1820 and 1877, seg 8192 1720 and 1844;
// 80 heads the same within 1 %, in 8 groups 2659 and 2604; 96 heads 2650 and 2594.  2 x 64 heads: 1 to 3 % for one.
static int chain_heads(const Plan &pl, bool pipelined_bwd) {
    const int ctas = pl.B * pl.H;
    return pl.hpg % 2 == 0 && (ctas > kNumSMs || (pipelined_bwd && ctas > kNumSMs / 2)) ? 2 : 1;
}

// CTAs of the y / dx kernel (its results do not depend on them).  It takes the whole GPU unless the segments are pipelined and
// small: then the kernels that run beside it (chain kernels, one CTA per head; dB/dC) get SMs of their own, because a chain
// that waits for the large kernel to finish makes the segments serial (24 heads, 2048-token segments: a chain kernel takes 15
// us on 24 SMs, y 8 us on all of them).  Not where less than a quarter of the GPU would be left for it.
static int scan_ctas(const SegParams &sp, bool pipelined, bool bwd) {
    if (!pipelined) return kNumSMs;
    const int beside = sp.B * sp.H / sp.chain_heads + (bwd ? sp.B * sp.H : 0) + (bwd ? sp.nc * sp.nsl * sp.G * sp.B : 0);
    return kNumSMs - beside >= kNumSMs / 4 ? kNumSMs - beside : kNumSMs;
}

// The tensor maps of copies 0 .. nh-1 of the forward chain's output and 0 .. ng-1 of the gradients.
static bool state_maps(const Layout &lo, void *ws, const SegParams &sp0, TcMaps *mh, int nh, TcMaps *mg, int ng) {
    SegParams sp = sp0;
    for (int i = 0; i < nh || i < ng; ++i) {
        select_copy(lo, ws, i < nh ? i : 0, i < ng ? i : 0, sp);
        SegParams one = sp;
        one.Gbf = nullptr;
        if (i < nh && !tc_state_maps(one, mh[i])) return false;
        one = sp;
        one.Hbf = nullptr;
        if (i < ng && !tc_state_maps(one, mg[i])) return false;
    }
    return true;
}

static int forward_impl(const ssd_shape_t *shape, const void *x, const float *dt, const float *A,
                        const void *Bm, const void *Cm, const float *D, const float *h0, void *y,
                        float *h_final, float *boundary, bool need_boundary, void *ws,
                        size_t ws_bytes, void *stream, bool built_in_ws = false) {
    Plan pl;
    int rc = make_plan(shape, pl);
    if (rc) return rc;
    if (!x || !dt || !A || !Bm || !Cm || !D || !y || !ws) return SSD_EINVAL;
    if (need_boundary && !boundary) return SSD_EINVAL;
    if (misaligned(x) || misaligned(dt) || misaligned(A) || misaligned(Bm) || misaligned(Cm) ||
        misaligned(D) || misaligned(y) || (h0 && misaligned(h0)) || (h_final && misaligned(h_final)) ||
        (boundary && misaligned(boundary)))
        return SSD_EALIGN;
    Layout lo;
    const bool beside = !built_in_ws && !pl.serial;       // work of neighbouring segments side by side
    if (built_in_ws) make_static_layout(pl, lo);
    else make_layout(pl, need_boundary ? SSD_OP_FWD_SEG : SSD_OP_FWD, lo, beside);
    if (((uintptr_t)ws & 255u) || ws_bytes < lo.total) return SSD_EWORKSPACE;
    rc = check_device();
    if (rc) return rc;

    cudaStream_t st = (cudaStream_t)stream;
    SegParams sp;
    fill_params(pl, lo, ws, sp);
    sp.x = x; sp.dt = dt; sp.A = A; sp.Bm = Bm; sp.Cm = Cm; sp.D = D; sp.y = y;
    sp.first = 1;       // the status word is cleared by the first launch
    TcMaps maps;
    if (pl.use_tc && !tc_make_maps(sp, maps)) return SSD_ECUDA;
    const long long PN = (long long)pl.P * pl.N;
    if (pl.use_tc && pl.nseg >= kMinSegmentsForTwins && beside && !g_prof_on) {
        // Algorithm 1 with the state chain ahead: it runs on a helper stream, up to as many segments ahead of y on the caller's
        // stream as there are copies of what both touch (records, bf16 states), and fills what y leaves idle.  The carried state
        // belongs to the chain alone.
        SideStreams *side = side_streams();
        if (!side) { g_last_cuda = (int)cudaGetLastError(); return SSD_ECUDA; }
        const int ncp = chain_copies(pl, false);
        TcMaps mk[kChainCopies] = {maps, maps, maps, maps};
        if (!state_maps(lo, ws, sp, mk, ncp, nullptr, 0)) return SSD_ECUDA;
        cudaStream_t chain = side->s[0];
        sp.chain_heads = chain_heads(pl, false);
        SSD_TRY(cudaEventRecord(side->start, st));
        SSD_TRY(cudaStreamWaitEvent(chain, side->start, 0));
        for (int k = 0; k < pl.nseg; ++k) {
            const int cp = k % ncp;
            set_segment(pl, k, sp);
            sp.first = k == 0;
            select_copy(lo, ws, cp, 0, sp);
            if (k >= ncp) SSD_TRY(cudaStreamWaitEvent(chain, side->big_done[cp], 0));   // y of segment k - ncp has read this copy
            {
                cudaStream_t st = chain;
                const float *init = (k == 0) ? h0 : sp.hcarry;
                float *bnd = boundary ? boundary + (size_t)k * pl.H * PN : nullptr;
                SSD_LAUNCH(KIND_CHUNK_STATE, launch_chain_fwd(sp, mk[cp], init, (long long)pl.H * PN, bnd, (long long)pl.nseg * pl.H * PN,
                                                              (k == pl.nseg - 1) ? h_final : nullptr, st));
                SSD_TRY(cudaEventRecord(side->chain_done, st));
            }
            // y of a segment waits for its chain alone: on two streams in turn its CTAs take the SMs of the one before as they come free,
            // where in one stream the next launch began some 6 us after the end (80 heads, 4096 steps: a segment 54 -> 49 us; dx of
            // neighbouring segments on two streams: no change there, 24 heads 2 % slower)
            cudaStream_t ys = k & 1 ? side->s[1] : st;
            SSD_TRY(cudaStreamWaitEvent(ys, side->chain_done, 0));
            sp.scan_ctas = scan_ctas(sp, k + 1 < pl.nseg, false);
            {
                cudaStream_t st = ys;
                SSD_LAUNCH(KIND_SCAN_FWD, launch_scan_tc(sp, mk[cp], SC_FWD, st));
                if (k + ncp < pl.nseg) SSD_TRY(cudaEventRecord(side->big_done[cp], st));
                if ((k & 1) && k + 2 >= pl.nseg) SSD_TRY(cudaEventRecord(side->join, st));
            }
        }
        SSD_TRY(cudaStreamWaitEvent(st, side->join, 0));        // the last one on the helper stream
        return SSD_OK;
    }
    sp.chain_heads = chain_heads(pl, false);
    const bool overlap = beside && simt_overlap(pl, false);
    // Readers only where a segment's exit state has the next one's copy to go to, and not where it or the boundary state goes to h0 itself:
    // its CTAs would store what the tiles of y in the same launch still read.  (A state pass reads and stores an element in one thread.)
    const size_t nh = (size_t)pl.B * pl.H * PN;
    const bool in_place = (pl.nseg == 1 && overlap_of(h0, nh, h_final, nh)) || overlap_of(h0, nh, boundary, nh * pl.nseg);
    const bool readers = beside && simt_readers(pl) && (overlap || pl.nseg == 1) && !in_place;
    SegParams next;
    for (int k = 0; k < pl.nseg; ++k) {
        set_segment(pl, k, sp);
        sp.first = k == 0;
        const float *init = (k == 0) ? h0 : sp.hcarry;
        float *bnd = boundary ? boundary + (size_t)k * pl.H * PN : nullptr, *fin = (k == pl.nseg - 1) ? h_final : nullptr;
        if (pl.use_tc) {
            SSD_LAUNCH(KIND_CHUNK_STATE, launch_chain_fwd(sp, maps, init, (long long)pl.H * PN, bnd, (long long)pl.nseg * pl.H * PN, fin, st));
            SSD_LAUNCH(KIND_SCAN_FWD, launch_scan_tc(sp, maps, SC_FWD, st));
            continue;
        }
        select_copy(lo, ws, 0, k & 1, sp);
        if (k == 0 || !overlap) SSD_LAUNCH(KIND_CHUNK_STATE, launch_simt(sp, nullptr, nullptr, pl.dtype, SIMT_SUMS, st));
        StatePass pass = {bnd, nullptr, fin, (int64_t)pl.nseg * pl.H * PN, 0};
        if (readers) {
            sp.hinit = k == 0 ? h0 : sp.Hst;
            sp.hinit_bs = k == 0 ? pl.H * PN : (pl.ncs + 1) * pl.H * PN;
        } else {
            SSD_LAUNCH(KIND_STATE_PASS_FWD, launch_state_pass_fwd(sp, init, (long long)pl.H * PN, bnd, (long long)pl.nseg * pl.H * PN, fin, st));
        }
        const bool ahead = overlap && k + 1 < pl.nseg;      // the next segment's sums in the launch of y
        if (ahead) {
            next = sp;
            set_segment(pl, k + 1, next);
            select_copy(lo, ws, 0, (k + 1) & 1, next);
            pass.leave = next.Hst;                          // slot 0 of the next segment's copy
            pass.leave_bs = (pl.ncs + 1) * pl.H * PN;
        }
        SSD_LAUNCH(KIND_SCAN_FWD, launch_simt(sp, ahead ? &next : nullptr, readers ? &pass : nullptr, pl.dtype, SIMT_Y, st));
    }
    return SSD_OK;
}

// ---- self-test of the bounded device-side wait: a barrier that nothing ever arrives on
// One warp waits on it with the given limit, gives up, records that in the status word and returns normally: the
// same mbar_wait path, status word and host read-back that every kernel of the library relies on, with no copy in
// flight and no tensor memory held, so that giving up is harmless here.
__global__ void k_selftest_wait(unsigned int *status, long long limit_clk, long long *waited_clk) {
    __shared__ uint64_t bar;
    __shared__ uint32_t abort_flag;
    if (threadIdx.x == 0) {
        sm100::mbar_init(&bar, 1);
        abort_flag = 0;
        sm100::fence_barrier_init();
    }
    __syncthreads();
    const long long t0 = clock64();
    const bool done = sm100::mbar_wait_limited(&bar, 0, &abort_flag, status, limit_clk);
    if (threadIdx.x == 0 && waited_clk) *waited_clk = done ? -1 : clock64() - t0;
}

// ---- built-in scratch for ssd_fwd_static_ws (callers that cannot allocate) ----
// Lives in the device image of this library: one copy per GPU that loads it, for the life of the
// process.  In host code `g_static_ws` is only a handle for cudaGetSymbolAddress, never a pointer.
static __device__ __align__(256) unsigned char g_static_ws[SSD_STATIC_WS_BYTES];

static const int kMaxDevices = 64;
static std::mutex g_static_mu;
static void *g_static_addr[kMaxDevices] = {nullptr};

// Device address of g_static_ws on the current device, looked up once per device.
static int static_ws_address(void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) { g_last_cuda = (int)e; return SSD_ECUDA; }
    if (dev < 0 || dev >= kMaxDevices) return SSD_EDEVICE;
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_addr[dev]) {
        void *ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_static_ws);
        if (e != cudaSuccess || !ptr) { g_last_cuda = (int)e; return SSD_ECUDA; }
        g_static_addr[dev] = ptr;
    }
    *out = g_static_addr[dev];
    return SSD_OK;
}

}  // namespace ssd

using namespace ssd;

extern "C" {

size_t ssd_workspace_bytes(const ssd_shape_t *shape, int op) {
    Plan pl;
    if (make_plan(shape, pl)) return 0;
    if (op != SSD_OP_FWD && op != SSD_OP_FWD_SEG && op != SSD_OP_BWD_SEG) return 0;
    Layout lo;
    make_layout(pl, op, lo, !pl.serial);
    return lo.total;
}

size_t ssd_boundary_bytes(const ssd_shape_t *shape) {
    Plan pl;
    if (make_plan(shape, pl)) return 0;
    return (size_t)pl.B * pl.nseg * pl.H * pl.P * pl.N * sizeof(float);
}

int ssd_fwd(const ssd_shape_t *shape, const void *x, const float *dt, const float *A, const void *Bm,
            const void *Cm, const float *D, const float *h0, void *y, float *h_final, void *ws,
            size_t ws_bytes, void *stream) {
    return forward_impl(shape, x, dt, A, Bm, Cm, D, h0, y, h_final, nullptr, false, ws, ws_bytes, stream);
}

int ssd_fwd_static_ws(const ssd_shape_t *shape, const void *x, const float *dt, const float *A,
                      const void *Bm, const void *Cm, const float *D, const float *h0, void *y,
                      float *h_final, void *stream) {
    Plan pl;
    int rc = make_plan(shape, pl);
    if (rc) return rc;
    Layout lo;
    make_static_layout(pl, lo);
    if (lo.total > (size_t)SSD_STATIC_WS_BYTES) return SSD_ETOOLARGE;
    if (!x || !dt || !A || !Bm || !Cm || !D || !y) return SSD_EINVAL;
    rc = check_device();
    if (rc) return rc;
    void *ws = nullptr;
    rc = static_ws_address(&ws);
    if (rc) return rc;
    // forward_impl zeroes the status word on the stream and writes every other scratch region
    // before reading it, so stale contents of the shared array cannot leak into the outputs.
    return forward_impl(shape, x, dt, A, Bm, Cm, D, h0, y, h_final, nullptr, false, ws,
                        (size_t)SSD_STATIC_WS_BYTES, stream, true);
}

int ssd_fwd_segmented(const ssd_shape_t *shape, const void *x, const float *dt, const float *A,
                      const void *Bm, const void *Cm, const float *D, const float *h0, void *y,
                      float *h_final, float *boundary, void *ws, size_t ws_bytes, void *stream) {
    return forward_impl(shape, x, dt, A, Bm, Cm, D, h0, y, h_final, boundary, true, ws, ws_bytes, stream);
}

int ssd_bwd_segmented(const ssd_shape_t *shape, const void *x, const float *dt, const float *A,
                      const void *Bm, const void *Cm, const float *D, const float *boundary,
                      const void *dy, const float *dh_final, void *dx, float *ddt, float *dA, void *dB,
                      void *dC, float *dD, float *dh0, void *ws, size_t ws_bytes, void *stream) {
    Plan pl;
    int rc = make_plan(shape, pl);
    if (rc) return rc;
    if (!x || !dt || !A || !Bm || !Cm || !D || !boundary || !dy || !dx || !ddt || !dA || !dB || !dC ||
        !dD || !ws)
        return SSD_EINVAL;
    if (misaligned(x) || misaligned(dt) || misaligned(A) || misaligned(Bm) || misaligned(Cm) ||
        misaligned(D) || misaligned(boundary) || misaligned(dy) || (dh_final && misaligned(dh_final)) ||
        misaligned(dx) || misaligned(ddt) || misaligned(dA) || misaligned(dB) || misaligned(dC) ||
        misaligned(dD) || (dh0 && misaligned(dh0)))
        return SSD_EALIGN;
    Layout lo;
    make_layout(pl, SSD_OP_BWD_SEG, lo, !pl.serial);
    if (((uintptr_t)ws & 255u) || ws_bytes < lo.total) return SSD_EWORKSPACE;
    rc = check_device();
    if (rc) return rc;

    cudaStream_t st = (cudaStream_t)stream;
    SegParams sp;
    fill_params(pl, lo, ws, sp);
    sp.x = x; sp.dt = dt; sp.A = A; sp.Bm = Bm; sp.Cm = Cm; sp.D = D; sp.dy = dy;
    sp.dx = dx; sp.ddt = ddt; sp.dB = dB; sp.dC = dC;
    sp.dx_skip = (shape->flags & SSD_FLAG_SKIP_GRAD) ? 1.f : 0.f;
    sp.first = 1;       // the status word is cleared by the first launch
    TcMaps maps;
    if (pl.use_tc && !tc_make_maps(sp, maps)) return SSD_ECUDA;
    const long long PN = (long long)pl.P * pl.N;
    const bool split_bc = (shape->flags & SSD_FLAG_SPLIT_BC) != 0;
    SideStreams *side = nullptr;
    if (pl.use_tc && !(shape->flags & SSD_FLAG_SERIAL) && !g_prof_on) {
        side = side_streams();
        if (!side) { g_last_cuda = (int)cudaGetLastError(); return SSD_ECUDA; }
    }
    if (side) {
        // Algorithm 2 as three pipelines that meet through events.  Segment k (right to left) needs
        //   chain(k): Recompute_Forward (chunk states, forward state pass), the state-gradient contributions and
        //             the backward state pass -- all it takes from segment k+1 is the state gradient handed left;
        //   big(k)  : dx on the caller's stream beside dB/dC on a second one -- they read what chain(k) left;
        //   tail(k) : the finishing kernel.
        // chain(k-1) runs on its own stream while big(k) is busy and fills the SMs that big(k)'s last, partly
        // idle wave leaves free; tail(k) runs under big(k-1)'s predecessors likewise.  What chain(k-1) writes and
        // big(k) / tail(k) read exists more than once and goes round with the segments; the carried gradient belongs to the
        // chain alone.
        const bool twin = pl.nseg >= kMinSegmentsForTwins;    // else one copy of what the gradient chain writes
        const int ncp = chain_copies(pl, true), npar = grad_copies(pl);
        sp.chain_heads = chain_heads(pl, pl.nseg > 1);
        TcMaps cmaps[kChainCopies] = {maps, maps, maps, maps}, gmaps[kGradCopies];
        if (!state_maps(lo, ws, sp, cmaps, ncp, gmaps, npar)) return SSD_ECUDA;
        cudaStream_t grads = side->s[0], recomp = side->s[4], tails = side->s[2];
        SSD_TRY(cudaEventRecord(side->start, st));
        SSD_TRY(cudaStreamWaitEvent(recomp, side->start, 0));
        SSD_TRY(cudaStreamWaitEvent(grads, side->start, 0));
        for (int k = pl.nseg - 1; k >= 0; --k) {
            const int i = pl.nseg - 1 - k, par = i % npar, cp = i % ncp;
            set_segment(pl, k, sp);
            sp.first = i == 0;
            select_copy(lo, ws, cp, par, sp);
            TcMaps mk = cmaps[cp];
            mk.G = gmaps[par].G;
            mk.Gst = gmaps[par].Gst;
            // ---- chain(k), first half: Recompute_Forward.  Its copy was last read by big(k + ncp) and tail(k + ncp).
            if (i >= ncp) SSD_TRY(cudaStreamWaitEvent(recomp, side->tail_done[(i - ncp) % kChainCopies], 0));
            {
                cudaStream_t st = recomp;
                SSD_LAUNCH(KIND_CHUNK_STATE, launch_chain_fwd(sp, mk, boundary + (size_t)k * pl.H * PN, (long long)pl.nseg * pl.H * PN,
                                                              nullptr, 0, nullptr, st));
                SSD_TRY(cudaEventRecord(side->rec_done, st));
            }
            // ---- chain(k), second half: the state gradients, which alone wait for segment k+1 (stream order: the
            // gradient handed left)
            // What it writes was last read by big and tail of the segment npar before.
            SSD_TRY(cudaStreamWaitEvent(grads, side->rec_done, 0));
            if (i >= npar) SSD_TRY(cudaStreamWaitEvent(grads, side->tail_done[(i - npar) % kChainCopies], 0));
            {
                cudaStream_t st = grads;
                const float *ginit = (k == pl.nseg - 1) ? dh_final : sp.gcarry;
                float *gleft = (k == 0 && dh0) ? dh0 : sp.gcarry;
                SSD_LAUNCH(KIND_DSTATE, launch_chain_bwd(sp, mk, ginit, gleft, st));
                SSD_TRY(cudaEventRecord(side->chain_done, st));
            }
            // ---- big(k); what it leaves for tail(k) (direct ddt, rho, psi, partial dB/dC slices) alternates too, and
            // chain(k) has already waited for the last reader of this copy.  The dB/dC kernels of
            // neighbouring segments are on different streams: with short segments one alone does not fill the GPU.
            cudaStream_t bcs = side->s[i & 1 ? 3 : 1];
            SSD_TRY(cudaStreamWaitEvent(st, side->chain_done, 0));
            SSD_TRY(cudaStreamWaitEvent(bcs, side->chain_done, 0));
            {
                cudaStream_t st = bcs;
                if (!split_bc) {
                    SSD_LAUNCH(KIND_BWD_DBDC, launch_grad_bc(sp, mk, BC_DC | BC_DB, st));
                } else {
                    SSD_LAUNCH(KIND_BWD_DC, launch_grad_bc(sp, mk, BC_DC, st));
                    SSD_LAUNCH(KIND_BWD_DB, launch_grad_bc(sp, mk, BC_DB, st));
                }
                SSD_TRY(cudaEventRecord(side->join, st));
            }
            sp.scan_ctas = scan_ctas(sp, twin, true);
            SSD_LAUNCH(KIND_BWD_DX, launch_scan_tc(sp, mk, SC_DX, st));
            SSD_TRY(cudaEventRecord(side->dx_done, st));
            // ---- tail(k), after both
            SSD_TRY(cudaStreamWaitEvent(tails, side->dx_done, 0));
            SSD_TRY(cudaStreamWaitEvent(tails, side->join, 0));
            {
                cudaStream_t st = tails;
                SSD_LAUNCH(KIND_BWD_FINISH, launch_bwd_tail(sp, pl.dtype, st));
                SSD_TRY(cudaEventRecord(side->tail_done[i % kChainCopies], st));
            }
        }
        SSD_TRY(cudaStreamWaitEvent(st, side->tail_done[(pl.nseg - 1) % kChainCopies], 0));   // the finishing stream is in order: this covers every segment
    } else {
        sp.chain_heads = chain_heads(pl, false);
        // no readers where dh0 goes to what they read beside it: the first segment's state, or the gradient that enters the only segment
        const size_t nh = (size_t)pl.B * pl.H * PN;
        const bool in_place = (pl.nseg == 1 && overlap_of(dh0, nh, dh_final, nh)) || overlap_of(dh0, nh, boundary, nh * pl.nseg);
        const bool readers = !pl.serial && simt_readers(pl) && !in_place;
        for (int k = pl.nseg - 1; k >= 0; --k) {
            set_segment(pl, k, sp);
            sp.first = k == pl.nseg - 1;
            // Recompute_Forward: chunk-entry states of segment k from the stored boundary state; then backward through the
            // segment: dh enters from the right, leaves to the left
            const float *hin = boundary + (size_t)k * pl.H * PN, *ginit = (k == pl.nseg - 1) ? dh_final : sp.gcarry;
            float *gleft = (k == 0 && dh0) ? dh0 : sp.gcarry;
            if (pl.use_tc) {
                SSD_LAUNCH(KIND_CHUNK_STATE, launch_chain_fwd(sp, maps, hin, (long long)pl.nseg * pl.H * PN, nullptr, 0, nullptr, st));
                SSD_LAUNCH(KIND_DSTATE, launch_chain_bwd(sp, maps, ginit, gleft, st));
                SSD_LAUNCH(KIND_BWD_DX, launch_scan_tc(sp, maps, SC_DX, st));
                if (!split_bc) {
                    SSD_LAUNCH(KIND_BWD_DBDC, launch_grad_bc(sp, maps, BC_DC | BC_DB, st));
                } else {
                    SSD_LAUNCH(KIND_BWD_DC, launch_grad_bc(sp, maps, BC_DC, st));
                    SSD_LAUNCH(KIND_BWD_DB, launch_grad_bc(sp, maps, BC_DB, st));
                }
            } else {
                select_copy(lo, ws, 0, k & 1, sp);
                if (k == pl.nseg - 1 || pl.serial) SSD_LAUNCH(KIND_CHUNK_STATE, launch_simt(sp, nullptr, nullptr, pl.dtype, SIMT_SUMS_GRAD, st));
                if (readers) {
                    // the gradient handed left is written while the one from the right is read: in gcarry and the last slot of Gst in turn
                    const int64_t own = pl.H * PN, slots = (pl.ncs + 1) * pl.H * PN;
                    float *const turn[2] = {sp.gcarry, sp.Gst + (size_t)pl.ncs * pl.H * PN};
                    const int i = pl.nseg - 1 - k;
                    sp.hinit = hin;
                    sp.hinit_bs = pl.nseg * pl.H * PN;
                    sp.ginit = i == 0 ? dh_final : turn[i & 1];
                    sp.ginit_bs = i == 0 || !(i & 1) ? own : slots;
                    StatePass pass = {};
                    pass.leave = k == 0 && dh0 ? dh0 : turn[(i + 1) & 1];
                    pass.leave_bs = (k == 0 && dh0) || !((i + 1) & 1) ? own : slots;
                    SSD_LAUNCH(KIND_BWD_DX, launch_simt(sp, nullptr, &pass, pl.dtype, SIMT_BWD, st));
                } else {
                    SSD_LAUNCH(KIND_STATE_PASS_BWD, launch_state_pass_bwd(sp, hin, (long long)pl.nseg * pl.H * PN, ginit, gleft, st));
                    SSD_LAUNCH(KIND_BWD_DX, launch_simt(sp, nullptr, nullptr, pl.dtype, SIMT_BWD, st));
                }
                if (k > 0 && !pl.serial) {
                    SegParams next = sp;
                    set_segment(pl, k - 1, next);
                    select_copy(lo, ws, 0, (k - 1) & 1, next);
                    SSD_LAUNCH(KIND_BWD_FINISH, launch_simt(sp, &next, nullptr, pl.dtype, SIMT_TAIL, st));
                    continue;
                }
            }
            SSD_LAUNCH(KIND_BWD_FINISH, launch_bwd_tail(sp, pl.dtype, st));
        }
    }
    SSD_LAUNCH(KIND_FINAL, launch_final_dAdD(sp, dA, dD, (shape->flags & SSD_FLAG_ACCUM_PARAM_GRADS) != 0, st));
    return SSD_OK;
}

static int glue_check(const ssd_shape_t *s, const void *a, const void *b, size_t &esz, long long &bs) {
    if (!s || !a || !b) return SSD_EINVAL;
    if (s->B <= 0 || s->L <= 0 || s->H <= 0) return SSD_EINVAL;
    if (s->P != 64) return SSD_EUNSUPPORTED;
    if (s->dtype != SSD_DTYPE_F32 && s->dtype != SSD_DTYPE_BF16) return SSD_EUNSUPPORTED;
    esz = s->dtype == SSD_DTYPE_BF16 ? 2 : 4;
    bs = s->x_bstride ? s->x_bstride : (long long)s->L * s->H * s->P;
    if (bs < (long long)s->L * s->H * s->P) return SSD_EINVAL;
    if (misaligned(a) || misaligned(b) || ((size_t)bs * esz) % 16) return SSD_EALIGN;
    return SSD_OK;
}

int ssd_glue_fwd(const ssd_shape_t *shape, const void *x, const void *y, const float *W, void *x_next, void *stream) {
    size_t esz; long long bs;
    int rc = glue_check(shape, x, y, esz, bs);
    if (rc) return rc;
    if (!W || !x_next) return SSD_EINVAL;
    if (misaligned(W) || misaligned(x_next)) return SSD_EALIGN;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_GLUE, launch_glue(shape->dtype, false, x, y, W, x_next, (long long)shape->L * shape->H, bs, shape->B, st));
    return SSD_OK;
}

int ssd_glue_bwd(const ssd_shape_t *shape, const void *g_next, const float *W, void *dz, void *stream) {
    size_t esz; long long bs;
    int rc = glue_check(shape, g_next, dz, esz, bs);
    if (rc) return rc;
    if (!W) return SSD_EINVAL;
    if (misaligned(W)) return SSD_EALIGN;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_GLUE, launch_glue(shape->dtype, true, g_next, nullptr, W, dz, (long long)shape->L * shape->H, bs, shape->B, st));
    return SSD_OK;
}

int ssd_glue_residual(const ssd_shape_t *shape, void *dx, const void *dz, void *stream) {
    size_t esz; long long bs;
    int rc = glue_check(shape, dx, dz, esz, bs);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_GLUE, launch_residual(shape->dtype, dx, dz, (long long)shape->L * shape->H * shape->P, bs, shape->B, st));
    return SSD_OK;
}

int ssd_decode_step(const ssd_shape_t *s, const void *x, const float *dt, const float *A, const void *Bm,
                    const void *Cm, const float *D, float *h, void *y, void *stream) {
    if (!s || !x || !dt || !A || !Bm || !Cm || !D || !h || !y) return SSD_EINVAL;
    if (s->B <= 0 || s->L != 1 || s->H <= 0 || s->P <= 0 || s->G <= 0 || s->H % s->G) return SSD_EINVAL;
    if (s->N != 64 && s->N != 128) return SSD_EUNSUPPORTED;
    if (s->dtype != SSD_DTYPE_F32 && s->dtype != SSD_DTYPE_BF16) return SSD_EUNSUPPORTED;
    const long long x_bs = s->x_bstride ? s->x_bstride : (long long)s->H * s->P;
    const long long dt_bs = s->dt_bstride ? s->dt_bstride : (long long)s->H;
    const long long bc_bs = s->bc_bstride ? s->bc_bstride : (long long)s->G * s->N;
    if (x_bs < (long long)s->H * s->P || dt_bs < s->H || bc_bs < (long long)s->G * s->N) return SSD_EINVAL;
    if (misaligned(x) || misaligned(dt) || misaligned(A) || misaligned(Bm) || misaligned(Cm) || misaligned(D) ||
        misaligned(h) || misaligned(y))
        return SSD_EALIGN;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_DECODE, launch_decode_step(s->dtype, s->N, x, dt, A, Bm, Cm, D, h, y, s->B, s->H, s->P, s->G,
                                               x_bs, dt_bs, bc_bs, st));
    return SSD_OK;
}

static int conv_check(int B, int L, int C, int dtype, long long &bs, long long u_bstride) {
    if (B <= 0 || L < 3 || C <= 0 || (C % 8)) return SSD_EINVAL;
    if (dtype != SSD_DTYPE_F32 && dtype != SSD_DTYPE_BF16) return SSD_EUNSUPPORTED;
    bs = u_bstride ? u_bstride : (long long)L * C;
    if (bs < (long long)L * C) return SSD_EINVAL;
    if (((size_t)bs * (dtype == SSD_DTYPE_BF16 ? 2 : 4)) % 16) return SSD_EALIGN;
    return SSD_OK;
}

size_t ssd_conv_workspace_bytes(int B, int L, int C) {
    if (B <= 0 || L <= 0 || C <= 0) return 0;
    return (size_t)B * conv_tiles(L) * 5 * C * sizeof(float);
}

int ssd_conv_fwd(int B, int L, int C, int dtype, const void *u, long long u_bstride, const float *w, const float *bias,
                 const void *state_in, void *out, void *state_out, void *stream) {
    long long bs;
    int rc = conv_check(B, L, C, dtype, bs, u_bstride);
    if (rc) return rc;
    if (!u || !w || !bias || !out) return SSD_EINVAL;
    if (misaligned(u) || misaligned(w) || misaligned(bias) || misaligned(out) || (state_in && misaligned(state_in)) ||
        (state_out && misaligned(state_out)))
        return SSD_EALIGN;
    rc = check_device();
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_CONV, launch_conv_fwd(dtype, u, bs, w, bias, state_in, out, state_out, B, L, C, st));
    return SSD_OK;
}

int ssd_conv_bwd(int B, int L, int C, int dtype, const void *u, long long u_bstride, const float *w, const float *bias,
                 const void *state_in, const void *dout, const float *dtail, void *du, float *dstate, float *dw,
                 float *dbias, int accumulate, void *ws, size_t ws_bytes, void *stream) {
    long long bs;
    int rc = conv_check(B, L, C, dtype, bs, u_bstride);
    if (rc) return rc;
    if (!u || !w || !bias || !dout || !du || !dw || !dbias || !ws) return SSD_EINVAL;
    if (misaligned(u) || misaligned(w) || misaligned(bias) || misaligned(dout) || misaligned(du) || misaligned(dw) ||
        misaligned(dbias) || (state_in && misaligned(state_in)) || (dtail && misaligned(dtail)) ||
        (dstate && misaligned(dstate)))
        return SSD_EALIGN;
    if (((uintptr_t)ws & 255u) || ws_bytes < ssd_conv_workspace_bytes(B, L, C)) return SSD_EWORKSPACE;
    rc = check_device();
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_CONV, launch_conv_bwd(dtype, u, bs, w, bias, state_in, dout, dtail, du, dstate, dw, dbias,
                                          accumulate ? 1 : 0, (float *)ws, B, L, C, st));
    return SSD_OK;
}

static int norm_check(long long rows, int D, int group, int dtype) {
    if (rows <= 0 || D <= 0 || group <= 0 || (D % group) || (group % 4)) return SSD_EINVAL;
    if (group > gated_norm_max_group() || gated_norm_tiles(rows) > 2147483647ll || D / group > 65535) return SSD_EUNSUPPORTED;
    if (dtype != SSD_DTYPE_F32 && dtype != SSD_DTYPE_BF16) return SSD_EUNSUPPORTED;
    if (((size_t)D * (dtype == SSD_DTYPE_BF16 ? 2 : 4)) % 16) return SSD_EALIGN;
    return SSD_OK;
}

size_t ssd_gated_norm_workspace_bytes(long long rows, int D) {
    if (rows <= 0 || D <= 0) return 0;
    return (size_t)gated_norm_tiles(rows) * D * sizeof(float);
}

int ssd_gated_norm_fwd(long long rows, int D, int group, int dtype, const void *y, const void *z, const float *gamma, float eps,
                       void *out, void *stream) {
    int rc = norm_check(rows, D, group, dtype);
    if (rc) return rc;
    if (!y || !z || !gamma || !out) return SSD_EINVAL;
    if (misaligned(y) || misaligned(z) || misaligned(gamma) || misaligned(out)) return SSD_EALIGN;
    rc = check_device();
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_NORM, launch_gated_norm_fwd(dtype, y, z, gamma, eps, out, rows, D, group, st));
    return SSD_OK;
}

int ssd_gated_norm_bwd(long long rows, int D, int group, int dtype, const void *y, const void *z, const float *gamma, float eps,
                       const void *dout, void *dy, void *dz, float *dgamma, int accumulate, void *ws, size_t ws_bytes,
                       void *stream) {
    int rc = norm_check(rows, D, group, dtype);
    if (rc) return rc;
    if (!y || !z || !gamma || !dout || !dy || !dz || !dgamma || !ws) return SSD_EINVAL;
    if (misaligned(y) || misaligned(z) || misaligned(gamma) || misaligned(dout) || misaligned(dy) || misaligned(dz) ||
        misaligned(dgamma))
        return SSD_EALIGN;
    if (((uintptr_t)ws & 255u) || ws_bytes < ssd_gated_norm_workspace_bytes(rows, D)) return SSD_EWORKSPACE;
    rc = check_device();
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_LAUNCH(KIND_NORM, launch_gated_norm_bwd(dtype, y, z, gamma, eps, dout, dy, dz, dgamma, accumulate ? 1 : 0, (float *)ws,
                                                rows, D, group, st));
    return SSD_OK;
}

int ssd_selftest_wait_timeout(void *ws, size_t ws_bytes, long long limit_cycles, void *stream) {
    if (!ws || limit_cycles < 0) return SSD_EINVAL;
    if (((uintptr_t)ws & 255u) || ws_bytes < 512) return SSD_EWORKSPACE;
    int rc = check_device();
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    SSD_TRY(cudaMemsetAsync(ws, 0, 512, st));
    k_selftest_wait<<<1, 32, 0, st>>>((unsigned int *)ws, limit_cycles, (long long *)((char *)ws + 256));
    SSD_TRY(cudaGetLastError());
    return SSD_OK;
}

int ssd_poll_status(void *ws) {
    if (!ws) return SSD_EINVAL;
    unsigned int word = 0;
    cudaError_t e = cudaMemcpy(&word, ws, sizeof(word), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) { g_last_cuda = (int)e; return SSD_ECUDA; }
    return word ? SSD_ETIMEOUT : SSD_OK;
}

const char *ssd_strerror(int code) {
    switch (code) {
        case SSD_OK: return "ok";
        case SSD_EINVAL: return "invalid argument (null pointer, bad size, H % G, L % chunk or seg % chunk)";
        case SSD_EUNSUPPORTED: return "unsupported shape or dtype (P=64, N in {64,128}, chunk in {64,128,256})";
        case SSD_EALIGN: return "pointer or stride not 16-byte aligned";
        case SSD_EWORKSPACE: return "workspace too small or not 256-byte aligned";
        case SSD_EDEVICE: return "current device is not compute capability 10.x";
        case SSD_ECUDA: return "CUDA call failed (see ssd_last_cuda_error)";
        case SSD_ETIMEOUT: return "a bounded device-side wait expired";
        case SSD_ETOOLARGE: return "shape needs more scratch than the built-in static buffer (SSD_STATIC_WS_BYTES); reduce seg or pass your own workspace to ssd_fwd";
        default: return "unknown error";
    }
}

int ssd_version(void) { return SSD_VERSION; }

long long ssd_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int ssd_kernel_kinds(void) { return KIND_COUNT; }

const char *ssd_kernel_name(int kind) {
    return (kind >= 0 && kind < KIND_COUNT) ? kKindNames[kind] : "";
}

int ssd_profile(int enable) {
    g_prof_on = enable != 0;
    g_prof_used = 0;
    return SSD_OK;
}

int ssd_profile_read(double *ms, long long *launches, int n) {
    if (!ms || !launches || n < KIND_COUNT) return SSD_EINVAL;
    for (int i = 0; i < n; ++i) { ms[i] = 0.0; launches[i] = 0; }
    for (size_t i = 0; i < g_prof_used; ++i) {
        ProfEvent &ev = g_prof_pool[i];
        cudaError_t e = cudaEventSynchronize(ev.b);
        float t = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t, ev.a, ev.b);
        if (e != cudaSuccess) { g_last_cuda = (int)e; return SSD_ECUDA; }
        ms[ev.kind] += (double)t;
        launches[ev.kind] += 1;
    }
    g_prof_used = 0;
    return SSD_OK;
}

int ssd_last_cuda_error(void) { return g_last_cuda; }

}  // extern "C"
