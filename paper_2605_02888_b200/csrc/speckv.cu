// Host side of libspeckv: argument checks, workspace plan and kernel launches behind the
// C ABI declared in include/speckv.h.  No allocation, no synchronisation.  The only state the
// library keeps between calls is one per-device constant (the address of the built-in scratch array), published with
// release/acquire atomics; it does not survive cudaDeviceReset.
#include "speckv.h"
#include "speckv_internal.h"

#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdint>

#include "speckv_kernels.cuh"
#include "speckv_sweep.cuh"
#include "speckv_shard.cuh"
#include "speckv_sample.cuh"

namespace {

using namespace speckv;

constexpr int kSliceBytes = 262144;  // bytes of one logit row that one sweep CTA streams
// Draft sampling has no row epilogue and no draw behind it, so its slices are cut for balance.  fp32 rows: half as long, since the
// last round of CTAs weighs more when fewer of them share an SM (V = 84,032, slices of 256 / 128 KB: 120 rows of 5 59.9 -> 45.1 us,
// 500 of 3 110.6 -> 91.1, 1,000 of 4 178.5 -> 143.5; V = 151,936, 64 of 8 69.8 -> 59.3; with a persistent share of chunks per CTA,
// the way before, 54.4 / 100.8 / 157.3 / 71.2).  Rows below 64 KB are cut only where that does not start a second round: 64 rows of
// 8 positions, V = 3,000, fp32 13.8 -> 8.7 us, V = 6,000, bf16 13.6 -> 9.1.
constexpr int kSampleF32SliceBytes = 131072, kSampleWholeBytes = 65536;
constexpr size_t kAlign = 256;

inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct Plan {
    int J_full;      // logit rows per batch row with verification: 2*G + 1
    size_t off_pos, off_tick, off_info, off_part, off_tokl, off_spans, off_dsum, off_list, total;
    size_t total_signals;  // what the signals alone use
};

inline int esize(speckv_dtype dt) { return dt == SPECKV_BF16 ? 2 : 4; }

// Bounds-checked build: the extents a call's kernels may touch, registered on the call's stream before
// its first kernel.  Range 0: draft logits, 1: target logits, 2: workspace, 3..: further caller arrays.
struct DbgExtra { const void* p; size_t bytes; };
cudaError_t dbg_register(cudaStream_t cs, const speckv_batch* bt, bool target, const void* ws, size_t ws_bytes,
                         const DbgExtra* extra = nullptr, int n_extra = 0) {
#ifdef SPECKV_DEBUG
    DbgRanges r{};
    auto span = [&](const void* base, int64_t sb, int64_t sp, int n_pos) -> unsigned long long {
        const long long last = static_cast<long long>(bt->B - 1) * sb + static_cast<long long>(n_pos - 1) * sp + bt->V;
        return reinterpret_cast<unsigned long long>(base) + static_cast<unsigned long long>(last) * esize(bt->dtype);
    };
    if (bt->B > 0 && bt->draft_logits) {
        r.lo[0] = reinterpret_cast<unsigned long long>(bt->draft_logits);
        r.hi[0] = span(bt->draft_logits, bt->draft_stride_b, bt->draft_stride_pos, bt->gamma_max);
    }
    if (bt->B > 0 && target && bt->target_logits) {
        r.lo[1] = reinterpret_cast<unsigned long long>(bt->target_logits);
        r.hi[1] = span(bt->target_logits, bt->target_stride_b, bt->target_stride_pos, bt->gamma_max + 1);
    }
    r.lo[2] = reinterpret_cast<unsigned long long>(ws);
    r.hi[2] = r.lo[2] + ws_bytes;
    for (int k = 0; k < n_extra && 3 + k < kDbgRanges; ++k) {
        r.lo[3 + k] = reinterpret_cast<unsigned long long>(extra[k].p);
        r.hi[3 + k] = r.lo[3 + k] + extra[k].bytes;
    }
    return cudaMemcpyToSymbolAsync(g_dbg_ranges, &r, sizeof r, 0, cudaMemcpyHostToDevice, cs);
#else
    (void)cs; (void)bt; (void)target; (void)ws; (void)ws_bytes; (void)extra; (void)n_extra;
    return cudaSuccess;
#endif
}

// CTA slots of the chip for a sweep of this type (148 SMs).
int cta_slots(speckv_dtype dt) { return 148 * (dt == SPECKV_BF16 ? SweepShape<__nv_bfloat16>::kCtas : SweepShape<float>::kCtas); }

// Vocabulary slices per logit row for a sweep over J logit rows per batch row, one CTA each, and the granules that one
// warp takes of a slice: P.nsplit, P.per_warp.  aligned: every row starts on the 16-byte grid.  sample: draft sampling.  most: what
// the partials of a row have room for, or its epilogue time for.
void choose_slices(KParams& P, speckv_dtype dt, bool aligned, bool sample = false, int most = kMaxSplit) {
    const int E = 16 / esize(dt);
    const int ng = (P.V + E - 1 + (aligned ? 0 : E - 1)) / E;  // granules a row can touch
    const bool whole = sample && 16LL * ng < kSampleWholeBytes;  // not more CTAs than slots
    int ns = static_cast<int>(std::lround(16.0 * ng / static_cast<double>(sample && dt == SPECKV_F32 ? kSampleF32SliceBytes : kSliceBytes)));
    if (ns < 1) ns = 1;
    // Small batches: enough CTAs to fill the slots of the chip once.  Aiming at more starts a second
    // round of short CTAs: with 1,184 instead of 740 (bf16), step of 64 bf16 rows, V = 32,000, 37.7 us instead of 33.1, of 37 rows,
    // V = 50,257, 32.6 instead of 31.1; one row the same.
    const long long rows = static_cast<long long>(P.B) * P.J;
    const int slots = cta_slots(dt);
    const long long want = (slots + (whole ? 0 : rows - 1)) / (rows > 0 ? rows : 1);
    if (want > ns) ns = static_cast<int>(want > most ? most : want);
    if (ns > most) ns = most;
    // At least one granule per lane, and whole steps of the warp: one with idle lanes costs as much as a full one, and lanes
    // that differ in their number of steps part in the last round of the loop (ranges of 128-byte lines before: step of 64 bf16
    // rows, V = 32,000, 30.2 us, this way 29.3; of 256 fp32 rows, V = 128,256, 226.5 / 222.8; draft sampling of those 113.2 / 110.9).
    // Rounding down makes more slices: only where they still fit the small-batch count (500 rows of V = 3,000, bf16, gamma 4, when
    // the sweep took them: 52 us with one slice per logit row, 68 us with two).
    int pw = (ng + ns * kWarps - 1) / (ns * kWarps);
    const int near = (pw + 16) / 32 * 32 < 32 ? 32 : (pw + 16) / 32 * 32;
    const int step = 32 * (kVec / E);
    if (pw >= 256) pw = (pw + step - 1) / step * step;
    else if (((ng + near * kWarps - 1) / (near * kWarps)) * rows <= slots + (whole ? 0 : rows)) pw = near;
    else pw = (pw + 31) / 32 * 32;
    while ((ng + pw * kWarps - 1) / (pw * kWarps) > most) pw += 32;
    P.per_warp = pw;
    P.nsplit = (ng + pw * kWarps - 1) / (pw * kWarps);
}

// CTAs per draw and granules per warp: P.R, P.draw_pw.  16,384 elements per CTA; a small batch spreads over the CTA slots
// (1.6 times), and many rows (of which about a third draw) share 4,096 CTAs rather than pay a CTA's start and end for every
// 16,384 elements.  (V = 128,256, bf16, 4 / 8 / 16 / 32 CTAs per draw: step of 1,024 rows 399 / 408 / 427 / 462 us, of 256
// rows 141 / 138 / 138 / 141.)
constexpr int kDrawElems = 16384, kDrawSmallCtas = 1184, kDrawMostCtas = 4096;
void choose_draw(KParams& P, speckv_dtype dt, bool aligned) {
    const int E = 16 / esize(dt);
    const int ng = (P.V + E - 1 + (aligned ? 0 : E - 1)) / E;
    int R = (P.V + kDrawElems - 1) / kDrawElems;
    const int want = (kDrawSmallCtas + P.B - 1) / P.B, cap = (ng + 32 * kWarps - 1) / (32 * kWarps);  // one granule per lane at least
    const int most = kDrawMostCtas / P.B, least = (P.V + 4 * kDrawElems - 1) / (4 * kDrawElems);
    if (want > R) R = want < cap ? want : cap > R ? cap : R;
    else if (R > most) R = most > least ? most : least;
    if (R > kMaxShares) R = kMaxShares;
    P.draw_pw = ((ng + R * kWarps - 1) / (R * kWarps) + 7) / 8 * 8;
    P.R = (ng + P.draw_pw * kWarps - 1) / (P.draw_pw * kWarps);
}

// Short rows: one CTA per batch row (batch_row_kernel) with P.nsplit warps per logit row, as many as leave none without work.
// The limits lie where the CTA's time, which grows with the length and the number of its rows, meets that of a CTA per logit
// row, which grows with their number in the batch.  Sweep -> this way (gamma fixed at its largest):
//   step, bf16 / fp32: 64 rows, gamma 8, V = 4,000, 24.4 -> 19.9 / 24.5 -> 21.5 us; 256 rows, gamma 8, V = 8,000, 55 -> 38 / 63 -> 48;
//   1,000 rows, gamma 8, V = 3,000, 112 -> 63 / 129 -> 62
//   few rows of many positions, fp32: step of 4 rows, V = 4,000, gamma 8 17.9 -> 20.5, gamma 16 19.4 -> 30.0, gamma 16, V = 2,000
//   19.0 -> 22.9 (ragged, where half of the positions are used, 15.4 -> 12.6); signals of 16 rows, V = 4,000, gamma 12 14.0 -> 14.4,
//   gamma 16 11.4 -> 14.8, gamma 8 10.9 -> 9.9; of 40 rows, gamma 16 (bf16) 16.4 -> 12.6
//   1,024 rows, gamma 4, V = 14,528: step, bf16 132 -> 114, fp32 equal
//   large batches, fp32: 1,100 rows, gamma 4, V = 12,000, signals 62.3 -> 48.5, step 153.5 -> 133.9; 4,000 rows, gamma 4, V = 14,528,
//   signals 157.7 -> 132.1; 12,000 rows, gamma 2, signals V = 20,000 402 -> 328 (gamma 1, V = 14,528 215 -> 209), step V = 14,528
//   equal, V = 20,000 8 % more.  300 rows, gamma 4, V = 12,000: step 53.7 -> 54.7.
bool short_rows(const KParams& P) {
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const long long rows = static_cast<long long>(P.B) * P.J, work = static_cast<long long>(P.J) * P.V;  // work: elements of one CTA
    if (P.B >= 2048 && !verify) return P.V <= (P.J > 1 ? 20480 : 12288);
    if (P.B >= 1024) return P.V <= 15360;
    if (P.B >= 256) return P.V <= 8192;
    if (P.V > 4096) return false;
    if (verify) return rows > 160 || work <= 98304;
    return rows > 256 || work <= (rows > 160 ? 45056 : 36864);
}
bool choose_batch_rows(KParams& P, speckv_dtype dt, bool aligned) {
    if (!short_rows(P)) return false;
    const int E = 16 / esize(dt);
    const int ng = (P.V + E - 1 + (aligned ? 0 : E - 1)) / E;
    P.nsplit = 1;
    while (P.J * P.nsplit * 2 <= kWarps) P.nsplit *= 2;
    P.n_spans = P.nsplit;
    P.per_warp = (ng + P.nsplit - 1) / P.nsplit;
    P.R = 1;
    P.draw_pw = (ng + kWarps - 1) / kWarps;
    return true;
}

// Does the call write one of its outputs over its gamma or its temperatures?
bool overwrites_rows(const KParams& P) {
    auto in = [&](const void* out, size_t words, const void* rows) {
        const uintptr_t o = reinterpret_cast<uintptr_t>(out), r = reinterpret_cast<uintptr_t>(rows);
        return out && rows && o < r + 4 * static_cast<size_t>(P.B) && r < o + 4 * words;
    };
    const size_t B = static_cast<size_t>(P.B), G = static_cast<size_t>(P.G);
    const struct { const void* p; size_t words; } outs[] = {{P.gamma_next, B}, {P.n_acc, B}, {P.status, B}, {P.out_tok, B * (G + 1)},
        {P.H, B * G}, {P.C, B * G}, {P.feat, 4 * B}, {P.scores, B * static_cast<size_t>(P.n_out)}};
    for (const auto& o : outs)
        if (in(o.p, o.words, P.gamma) || in(o.p, o.words, P.temp)) return true;
    return false;
}

// A small batch whose sweep has no generations: its CTAs find their work themselves (a thread per batch row), and its draws belong
// to batch rows.  Not where the call writes over gamma or the temperatures (the next gamma in the place of this step's): every CTA reads
// those of all rows, the later ones while the epilogues of the first rows write; a list is complete before the sweep starts.
// CTAs per draw: 64 granules per warp, two loads a lane, as far as the span sums' places and the CTA slots go (1.6
// times, as choose_draw).
void choose_direct(KParams& P, speckv_dtype dt, bool aligned) {
    if (P.B > kDirectMostB || P.n_tests || overwrites_rows(P)) return;
    P.direct = 1;
    if (!(P.mode & MODE_VERIFY)) return;
    const int E = 16 / esize(dt);
    const int ng = (P.V + E - 1 + (aligned ? 0 : E - 1)) / E;
    int R = (ng + kWarps * 64 - 1) / (kWarps * 64);
    const int most = kDirectSums / kWarps, fit = kDrawSmallCtas / P.B;
    if (R > most) R = most;
    if (R > fit) R = fit < 1 ? 1 : fit;
    P.draw_pw = ((ng + R * kWarps - 1) / (R * kWarps) + 7) / 8 * 8;
    P.R = (ng + P.draw_pw * kWarps - 1) / (P.draw_pw * kWarps);
}

// Order of the sweep and its early tests (verification, large batches): position 0 of every batch row first and the later target rows
// position by position, so that a position's acceptance test is in before the CTAs of the later target rows start.  Without tests the
// order is the same; batch row by batch row is as fast there (verification of 300 bf16 rows of 2, V = 20,000 / 50,257, 33.9 / 53.5 us and
// 34.6 / 52.8 that way, a rank's four calls, 256 rows, V = 128,256 over 3 / 2 ranks, 95.0 / 114.3 and 96.3 / 114.8).
constexpr int kBriefSlice = 131072;  // bytes of a slice from which on the test of a position beyond the second pays
void choose_tests(KParams& P, speckv_dtype dt) {
    // ... where the grid has that many CTAs: the third generation has to start after the first one's tests, that is
    // one and a half rounds of CTA slots behind it (one row, V = 32,000: taking the tests for nothing cost 4 us of 20)
    const long long ahead = static_cast<long long>(P.B) * P.nsplit * (P.G + 1);
    if (2 * ahead < 3 * cta_slots(dt)) return;
    P.pos_bits = P.nsplit <= 7 ? 4 : 8;  // twice nsplit arrivals at most
    // Position by position the tests of one are in before the next one's CTAs start, where a position has a round of CTAs or its
    // CTAs are short; else batch rows that complete one after the other are worth more (position by position: 256 bf16 rows,
    // V = 128,256, 131.9 -> 133.3 us, 96 greedy fp32 rows 85.1 -> 86.3; 512 fp32 rows, V = 151,936, 495 -> 475).  A test keeps a CTA
    // slot for 2.5 us: of short slices only the first two positions (all of them: 1,000 fp32 rows, V = 20,000, 173 -> 184 us,
    // 600 bf16 rows of 4, V = 14,000, 69.7 -> 76.4), and no more where the rows go one by one.
    const bool brief = P.per_warp * kWarps * 16 < kBriefSlice;
    P.rows_major = !brief && static_cast<long long>(P.B) * P.nsplit < cta_slots(dt);
    P.n_tests = brief || P.rows_major ? 2 : 64 / P.pos_bits;
}

Plan make_plan(const speckv_batch* bt) {
    Plan p;
    const size_t B = static_cast<size_t>(bt->B);
    p.J_full = 2 * bt->gamma_max + 1;
    size_t off = 0;
    p.off_pos = off; off += 2 * B * sizeof(int);  // positions' tickets
    p.off_tick = off; off = align_up(off + (4 * B + 4) * sizeof(int));  // tickets, counters, draw queue, early stops
    p.off_info = off; off = align_up(off + B * sizeof(RowInfo));
    p.off_part = off; off = align_up(off + B * p.J_full * kMaxSplit * sizeof(float4));
    p.off_tokl = off; off = align_up(off + B * static_cast<size_t>(bt->gamma_max) * sizeof(float2));
    p.total_signals = off < kAlign ? kAlign : off;
    p.off_spans = off; off = align_up(off + B * kMaxSplit * kWarps * sizeof(float2));
    p.off_dsum = off; off = align_up(off + B * kMaxShares * kWarps * sizeof(double));
    p.off_list = off; off = align_up(off + B * p.J_full * sizeof(int2));
    p.total = off < kAlign ? kAlign : off;
    return p;
}

// what the caller must provide
size_t workspace_total(const speckv_batch* bt) { return make_plan(bt).total; }

// What is held against the scratch array of speckv_signals_static: the signals' scratch and a word per 256 columns of every batch
// row, which it once had.  More than is used, so that the batches that are refused stay the same.
size_t static_figure(const speckv_batch* bt) {
    return make_plan(bt).total_signals + align_up(static_cast<size_t>(bt->B) * ((static_cast<size_t>(bt->V) + 255) / 256) * sizeof(float));
}

// polls a waiting CTA spends before it gives a row up (SPECKV_ROW_TIMEOUT); lowered by tests only
std::atomic<int> g_wait_limit{1 << 20};

speckv_status check_batch(const speckv_batch* bt, bool need_target) {
    if (!bt) return SPECKV_ERR_INVALID_ARG;
    if (bt->B < 0 || bt->gamma_max < 1 || bt->V < 1) return SPECKV_ERR_INVALID_ARG;
    if (bt->dtype != SPECKV_F32 && bt->dtype != SPECKV_BF16) return SPECKV_ERR_UNSUPPORTED;
    if (bt->gamma_max > SPECKV_MAX_GAMMA) return SPECKV_ERR_UNSUPPORTED;
    if (bt->V > (1 << 30) || bt->B > (1 << 24)) return SPECKV_ERR_UNSUPPORTED;
    if (bt->B == 0) return SPECKV_OK;
    if (!bt->draft_logits) return SPECKV_ERR_INVALID_ARG;
    // a stride of 0 broadcasts one row; anything else must step over whole rows
    auto stride_ok = [&](int64_t s) { return s == 0 || s >= bt->V; };
    if (!stride_ok(bt->draft_stride_b) || !stride_ok(bt->draft_stride_pos)) return SPECKV_ERR_INVALID_ARG;
    if (need_target) {
        if (!bt->target_logits || !bt->draft_tokens || !bt->uniforms) return SPECKV_ERR_INVALID_ARG;
        if (!stride_ok(bt->target_stride_b) || !stride_ok(bt->target_stride_pos)) return SPECKV_ERR_INVALID_ARG;
    }
    if (!(bt->temperature) && !(bt->temperature_scalar >= 0.f)) return SPECKV_ERR_INVALID_ARG;
    if (bt->flags & ~(SPECKV_READ_ALL_TARGET_ROWS | SPECKV_SCHEDULE_SLICED)) return SPECKV_ERR_INVALID_ARG;
    return SPECKV_OK;
}

speckv_status check_mlp(const speckv_mlp* m) {
    if (!m || !m->W2 || !m->b2) return SPECKV_ERR_INVALID_ARG;
    if (m->feature_layout < 0 || m->feature_layout > 2) return SPECKV_ERR_INVALID_ARG;
    const int min_hidden = m->feature_layout == 2 ? 0 : 1;  // the paper-form predictor may be linear
    if (m->n_hidden < min_hidden || m->n_out < 1 || m->n_in < 1) return SPECKV_ERR_INVALID_ARG;
    if (m->n_hidden > 0 && (!m->W1 || !m->b1)) return SPECKV_ERR_INVALID_ARG;
    if (m->n_hidden > SPECKV_MAX_HIDDEN || m->n_out > 8 || m->n_in > 8) return SPECKV_ERR_UNSUPPORTED;
    if (m->score_transform != 0 && m->score_transform != 1) return SPECKV_ERR_INVALID_ARG;
    if (m->n_in < (m->feature_layout == 0 ? 3 : m->feature_layout == 1 ? 4 : 5)) return SPECKV_ERR_INVALID_ARG;
    return SPECKV_OK;
}

bool rows_aligned(const void* base, int64_t sb, int64_t sp, int es) {
    return (reinterpret_cast<uintptr_t>(base) % 16 == 0) && ((sb * es) % 16 == 0) && ((sp * es) % 16 == 0);
}

void fill_mlp(KParams& P, const speckv_mlp* m, const float* comp) {
    P.n_in = m->n_in; P.n_hidden = m->n_hidden; P.n_out = m->n_out;
    P.layout = m->feature_layout; P.transform = m->score_transform;
    P.n_comp = m->n_in - (m->feature_layout == 0 ? 3 : m->feature_layout == 1 ? 4 : 5);
    P.W1 = m->W1; P.b1 = m->b1; P.W2 = m->W2; P.b2 = m->b2; P.comp = comp;
    for (int j = 0; j < 8; ++j) P.gch[j] = m->gamma_choices[j];
}

struct Events {  // optional timing events around the kernels of a step
    cudaEvent_t before_sweep = nullptr, after_sweep = nullptr, after_resample = nullptr;
};

// Launches CTAs as a programmatic dependent of what is in front of it in the stream (wait_for_predecessors), so
// that the launch itself is over when that ends.  Calls one after the other in a stream: step of 1 fp32 row, V = 32,000, 19.5 ->
// 17.9 us, of 64 bf16 rows 34.2 -> 32.3, signals and controller of 128, V = 128,256, 52.6 -> 49.2, a rank's four calls 66.4 -> 61.2.
template <class... Params, class... Args>
cudaError_t launch_threads(void (*kernel)(Params...), unsigned grid, unsigned threads, cudaStream_t st, const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <class... Params, class... Args>
cudaError_t launch(void (*kernel)(Params...), unsigned grid, cudaStream_t st, const Args&... args) {
    return launch_threads(kernel, grid, kThreads, st, args...);
}

constexpr int kPrepRows = 32;  // batch rows per CTA of the preparing kernel at least; 64 CTAs at most

// The sliced sweep: list and cleared counters, then the sweep with n_draw CTAs behind it.
template <typename T>
cudaError_t launch_sliced(KParams P, long long n_draw, cudaStream_t st, cudaEvent_t before_sweep) {
    P.n_draw = static_cast<int>(n_draw);
    const unsigned grid = static_cast<unsigned>(static_cast<long long>(P.B) * P.J * P.nsplit + n_draw);
    if (P.direct) {
        const int words = P.rdone ? P.B * P.R * kWarps : P.B;
        cudaError_t e = launch(prep_direct_kernel, static_cast<unsigned>((words + kThreads - 1) / kThreads), st, P);
        if (e != cudaSuccess) return e;
        if (before_sweep) cudaEventRecord(before_sweep, st);
        return launch(sweep_kernel<T, true>, grid, st, P);
    }
    int seg = (P.B + 63) / 64;
    seg = seg < kPrepRows ? kPrepRows : (seg + 31) / 32 * 32;
    cudaError_t e = launch(prep_kernel, static_cast<unsigned>((P.B + seg - 1) / seg), st, P, seg);
    if (e != cudaSuccess) return e;
    if (before_sweep) cudaEventRecord(before_sweep, st);
    return launch(sweep_kernel<T, false>, grid, st, P);
}

template <typename T>
cudaError_t launch_all(const KParams& P, cudaStream_t st, const Events& ev) {
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const long long n_draw = verify ? static_cast<long long>(P.B) * P.R : 0;
    const bool merged = static_cast<long long>(P.B) * P.J * P.nsplit + n_draw <= 0x7fffffffLL;
    cudaError_t e = launch_sliced<T>(P, merged ? n_draw : 0, st, ev.before_sweep);
    if (e != cudaSuccess) return e;
    if (ev.after_sweep) cudaEventRecord(ev.after_sweep, st);
    if (!merged) {  // more CTAs than a grid holds: the draws' part as a launch of its own
        resample_kernel<T><<<static_cast<unsigned>(n_draw), kThreads, 0, st>>>(P);
        e = cudaGetLastError();
    }
    if (ev.after_resample) cudaEventRecord(ev.after_resample, st);
    return e;
}

// A short row's batch in one launch.
template <typename T>
cudaError_t launch_rows(const KParams& P, cudaStream_t st, const Events& ev) {
    if (ev.before_sweep) cudaEventRecord(ev.before_sweep, st);
    const cudaError_t e = launch(batch_row_kernel<T>, static_cast<unsigned>(P.B), st, P);
    if (ev.after_sweep) cudaEventRecord(ev.after_sweep, st);
    if (ev.after_resample) cudaEventRecord(ev.after_resample, st);
    return e;
}

// Does every logit row of the call start on the 16-byte grid?
bool call_aligned(const speckv_batch* bt, bool verify) {
    const int es = esize(bt->dtype);
    return rows_aligned(bt->draft_logits, bt->draft_stride_b, bt->draft_stride_pos, es) &&
           (!verify || rows_aligned(bt->target_logits, bt->target_stride_b, bt->target_stride_pos, es));
}

// How a call of signals / verify / step is cut: sizes, slices, order and draws.  Returns whether it takes a CTA per batch row.  The
// outputs and the rows' parameters are in P already.
bool plan_call(KParams& P, const speckv_batch* bt, int mode) {
    const bool verify = (mode & MODE_VERIFY) != 0;
    P.B = bt->B; P.G = bt->gamma_max; P.V = bt->V;
    P.J = verify ? 2 * bt->gamma_max + 1 : bt->gamma_max;
    P.mode = mode;
    const bool aligned = call_aligned(bt, verify);
    choose_slices(P, bt->dtype, aligned);
    choose_draw(P, bt->dtype, aligned);
    P.n_spans = P.nsplit * kWarps;
    if (choose_batch_rows(P, bt->dtype, aligned)) return true;
    if (verify) choose_tests(P, bt->dtype);
    choose_direct(P, bt->dtype, aligned);
    return false;
}

// Shared driver of signals / verify / step.
speckv_status run(const speckv_batch* bt, int mode, const float* comp, const speckv_mlp* mlp, float* H,
                  float* C, float* feat, float* scores, int32_t* gamma_next, int32_t* n_accepted,
                  int32_t* out_tokens, int32_t* row_status, void* ws, size_t ws_bytes, void* stream,
                  const Events& ev = Events()) {
    const bool verify = (mode & MODE_VERIFY) != 0;
    speckv_status st = check_batch(bt, verify);
    if (st != SPECKV_OK) return st;
    if (mode & MODE_MLP) {
        st = check_mlp(mlp);
        if (st != SPECKV_OK) return st;
        if (!gamma_next || !feat) return SPECKV_ERR_INVALID_ARG;
    }
    if (verify && (!n_accepted || !out_tokens)) return SPECKV_ERR_INVALID_ARG;
    if (bt->B == 0) return SPECKV_OK;
    const Plan pl = make_plan(bt);
    if (!ws || reinterpret_cast<uintptr_t>(ws) % kAlign != 0) return SPECKV_ERR_INVALID_ARG;
    if (ws_bytes < (verify ? pl.total : pl.total_signals)) return SPECKV_ERR_WORKSPACE;

    KParams P{};
    P.bits = bt->entropy_in_bits ? 1 : 0;
    P.wait_limit = g_wait_limit.load(std::memory_order_relaxed);
    P.d = bt->draft_logits; P.dsb = bt->draft_stride_b; P.dsp = bt->draft_stride_pos;
    P.t = bt->target_logits; P.tsb = bt->target_stride_b; P.tsp = bt->target_stride_pos;
    P.tok = bt->draft_tokens; P.gamma = bt->gamma; P.temp = bt->temperature;
    P.temp_scalar = bt->temperature_scalar; P.u = bt->uniforms;
    if (mode & MODE_MLP) fill_mlp(P, mlp, comp);
    P.H = H; P.C = C; P.feat = feat; P.scores = scores; P.gamma_next = gamma_next;
    P.n_acc = n_accepted; P.out_tok = out_tokens; P.status = row_status;
    const bool by_row = plan_call(P, bt, mode);
    char* w = static_cast<char*>(ws);
    P.tick1 = reinterpret_cast<int*>(w + pl.off_tick);
    P.tick2 = P.tick1 + P.B;
    P.n_list = P.tick1 + 2 * P.B;
    P.q_front = P.n_list + 1;
    P.q_back = P.n_list + 2;
    P.info = reinterpret_cast<RowInfo*>(w + pl.off_info);
    P.part = reinterpret_cast<float4*>(w + pl.off_part);
    P.dsum = reinterpret_cast<double*>(w + pl.off_dsum);

    if (static_cast<long long>(P.B) * P.J * P.nsplit > 0x7fffffffLL) return SPECKV_ERR_UNSUPPORTED;

    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (dbg_register(cs, bt, verify, ws, ws_bytes) != cudaSuccess) return SPECKV_ERR_CUDA;
    // signals: behind their partials, which take a third of that region; verification: a region of its own
    P.list = reinterpret_cast<int2*>(verify ? w + pl.off_list : reinterpret_cast<char*>(P.part + static_cast<size_t>(P.B) * P.J * P.nsplit));
    if (by_row) {
        P.tokl = reinterpret_cast<float2*>(w + pl.off_tokl);
        P.spans = verify ? reinterpret_cast<float2*>(w + pl.off_spans) : nullptr;
        const cudaError_t e = bt->dtype == SPECKV_BF16 ? launch_rows<__nv_bfloat16>(P, cs, ev) : launch_rows<float>(P, cs, ev);
        return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
    }
    if (verify) {
        P.rdone = P.n_list + 4;
        P.tokl = reinterpret_cast<float2*>(w + pl.off_tokl);
        P.spans = reinterpret_cast<float2*>(w + pl.off_spans);
        P.read_all = (bt->flags & SPECKV_READ_ALL_TARGET_ROWS) ? 1 : 0;
        if (P.n_tests) {
            P.early = P.rdone + P.B;
            P.tick_pos = reinterpret_cast<unsigned long long*>(w + pl.off_pos);
        }
    }
    const cudaError_t e = bt->dtype == SPECKV_BF16 ? launch_all<__nv_bfloat16>(P, cs, ev) : launch_all<float>(P, cs, ev);
    return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

// Draft-side sampling: its own workspace plan (one draw per drafted position).  A position has a span for every warp that a row of
// this length can keep busy with a granule per lane, wherever it sits on the 16-byte grid.
struct SamplePlan {
    size_t off_tick, off_spans, total;
    int most_spans;
};
SamplePlan make_sample_plan(const speckv_batch* bt) {
    SamplePlan p;
    const size_t B = static_cast<size_t>(bt->B), G = static_cast<size_t>(bt->gamma_max);
    size_t off = 0;
    p.off_tick = off; off = align_up(off + (B * G + 2 * B) * sizeof(int));  // tickets per position and per row, row status
    const int E = 16 / esize(bt->dtype), ng = (bt->V + 2 * (E - 1)) / E, warps = (ng + 31) / 32;
    p.most_spans = warps < kMaxSplit * kWarps ? warps : kMaxSplit * kWarps;
    p.off_spans = off; off = align_up(off + B * G * p.most_spans * sizeof(float2));
    p.total = off < kAlign ? kAlign : off;
    return p;
}

void plan_sample(KParams& P, const speckv_batch* bt, const SamplePlan& pl) {
    P.B = bt->B; P.G = bt->gamma_max; P.V = bt->V;
    P.J = bt->gamma_max;
    choose_slices(P, bt->dtype, rows_aligned(bt->draft_logits, bt->draft_stride_b, bt->draft_stride_pos, esize(bt->dtype)), true);
    // Pieces of a warp's range: none (one) where the CTA reads the whole range again at once, a granule per thread; else pieces of that
    // length, whole groups of steps, and not more of them than there is room for.  Piece sums for all rows: 24 fp32 rows of 4,
    // V = 32,000, 12.3 -> 12.7 us, 293 bf16 rows of 8, V = 1,553, 17.8 -> 18.7; for none: 256 bf16 rows of 8, V = 128,256, 70.8 instead
    // of 65, 182 fp32 rows of 2, V = 15,936, 13.4 instead of 11.6.
    const int steps = bt->dtype == SPECKV_BF16 ? SweepShape<__nv_bfloat16>::kSteps : SweepShape<float>::kSteps;
    const int group = steps * 32 * (kVec * esize(bt->dtype) / 16), groups = (P.per_warp + group - 1) / group;
    P.fine = (P.per_warp + kThreads - 1) / kThreads;
    if (P.fine > groups) P.fine = groups;
    if (P.fine > kMostFine) P.fine = kMostFine;
    while (P.fine > 1 && P.nsplit * kWarps * P.fine > pl.most_spans) --P.fine;
    P.fine_groups = (groups + P.fine - 1) / P.fine;
    // (per_warp is 32 at least, so a warp behind the last span has no granule)
    P.n_spans = P.nsplit * kWarps * P.fine < pl.most_spans ? P.nsplit * kWarps * P.fine : pl.most_spans;
}

speckv_status run_sample(const speckv_batch* bt, const float* uniforms, int32_t* tokens, int32_t* row_status,
                         void* ws, size_t ws_bytes, void* stream) {
    speckv_status st = check_batch(bt, false);
    if (st != SPECKV_OK) return st;
    if (bt->B == 0) return SPECKV_OK;
    if (!uniforms || !tokens) return SPECKV_ERR_INVALID_ARG;
    if (static_cast<long long>(bt->B) * bt->gamma_max > (1 << 24)) return SPECKV_ERR_UNSUPPORTED;
    const SamplePlan pl = make_sample_plan(bt);
    if (!ws || reinterpret_cast<uintptr_t>(ws) % kAlign != 0) return SPECKV_ERR_INVALID_ARG;
    if (ws_bytes < pl.total) return SPECKV_ERR_WORKSPACE;

    KParams P{};
    plan_sample(P, bt, pl);
    P.d = bt->draft_logits; P.dsb = bt->draft_stride_b; P.dsp = bt->draft_stride_pos;
    P.gamma = bt->gamma; P.temp = bt->temperature; P.temp_scalar = bt->temperature_scalar;
    P.u = uniforms;
    P.out_tok = tokens; P.status = row_status;
    char* w = static_cast<char*>(ws);
    P.tick1 = reinterpret_cast<int*>(w + pl.off_tick);
    P.tick2 = P.tick1 + static_cast<size_t>(P.B) * P.G;
    P.rdone = P.tick2 + P.B;
    P.spans = reinterpret_cast<float2*>(w + pl.off_spans);
    if (static_cast<long long>(P.B) * P.J * P.nsplit > 0x7fffffffLL) return SPECKV_ERR_UNSUPPORTED;

    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (dbg_register(cs, bt, false, ws, ws_bytes) != cudaSuccess) return SPECKV_ERR_CUDA;
    const int n_tick = P.B * (2 + P.G);
    const unsigned n_clear = static_cast<unsigned>(n_tick < 64 * kThreads ? (n_tick + kThreads - 1) / kThreads : 64);
    cudaError_t e = launch(clear_kernel, n_clear, cs, P.tick1, n_tick);
    if (e != cudaSuccess) return SPECKV_ERR_CUDA;
    const unsigned grid = static_cast<unsigned>(P.B) * P.G * P.nsplit;
    if (P.fine > 1) e = bt->dtype == SPECKV_BF16 ? launch(sample_kernel<__nv_bfloat16, true>, grid, cs, P) : launch(sample_kernel<float, true>, grid, cs, P);
    else e = bt->dtype == SPECKV_BF16 ? launch(sample_kernel<__nv_bfloat16, false>, grid, cs, P) : launch(sample_kernel<float, false>, grid, cs, P);
    return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

// Scratch for speckv_signals_static: lives in the library image, one copy per device that loads it.
static __device__ __align__(256) unsigned char g_static_scratch[SPECKV_STATIC_SCRATCH_BYTES];

// Device address of g_static_scratch on the current device.  In host code the array's name only
// stands for the symbol; the address a kernel can use has to be asked for, once per device.
cudaError_t static_scratch_address(void** out) {
    static std::atomic<void*> cached[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool slot = dev >= 0 && dev < 64;
    void* p = slot ? cached[dev].load(std::memory_order_acquire) : nullptr;
    if (!p) {
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return e;
        if (slot) cached[dev].store(p, std::memory_order_release);
    }
    *out = p;
    return cudaSuccess;
}

// ---- vocabulary-sharded verification (speckv_shard.cuh) ----
struct ShardPlan {
    size_t off_tick, off_part, off_dsum, off_dsum2, off_list, total;
};
ShardPlan make_shard_plan(const speckv_batch* bt) {
    ShardPlan p;
    const size_t B = static_cast<size_t>(bt->B), J = 2 * static_cast<size_t>(bt->gamma_max) + 1;
    size_t off = 0;
    p.off_tick = off; off = align_up(off + (3 * B + 4) * sizeof(int));  // sweep tickets, draw tickets, counters, row queue
    p.off_part = off; off = align_up(off + B * J * kMaxSplit * sizeof(float4));
    p.off_dsum = off; off = align_up(off + B * kMaxShares * kWarps * sizeof(double));
    p.off_dsum2 = off; off = align_up(off + B * kMaxShares * kWarps * sizeof(double));
    p.off_list = off; off = align_up(off + B * J * sizeof(int2));
    p.total = off < kAlign ? kAlign : off;
    return p;
}

// A slice row short enough for one CTA in a batch that fills the SMs with one CTA per row: no ticket, nothing to clear first.
constexpr int kShardOneCtaRows = 128, kShardOneCtaGran = 4096;
// Slices of a wide slice row at most: one lane of export_epilogue merges a logit row's partials one after the other (one row,
// gamma 2, V = 31,680, fp32: this call 20.8 us with up to 32 slices, 16.6 with 16, as many as it had before the sweep aimed at whole steps).
constexpr int kExportSplit = 16;
// Batches with more rows than the chip has slots for CTAs of 256 threads: two warps per row (finish of 8,000 rows, gamma 2 / 8 / 16,
// 57.5 / 61.7 / 78.0 -> 31.3 / 46.7 / 64.6 us; of 500 rows, gamma 16, the four calls 35.9 -> 40.5, so below that eight).
constexpr int kShardManyRows = 741;
// Slice rows of a step or two per lane, one warp each: two steps in flight beside 5 CTAs per SM (8,000 rows, gamma 16, V = 128,
// fp32, 188 -> 163 us; 1,024 rows, bf16, 25.9 -> 22.3).
constexpr int kShardTinyRowBytes = 2048;
constexpr int kShardWarpRowBytes = 65536;  // slice rows up to this size are swept by one warp each

// what every shard call needs from the local batch
speckv_status shard_params(const speckv_batch* bt, void* ws, size_t ws_bytes, KParams& P, ShardPlan& pl) {
    speckv_status st = check_batch(bt, true);
    if (st != SPECKV_OK) return st;
    pl = make_shard_plan(bt);
    if (bt->B == 0) return SPECKV_OK;
    if (!ws || reinterpret_cast<uintptr_t>(ws) % kAlign != 0) return SPECKV_ERR_INVALID_ARG;
    if (ws_bytes < pl.total) return SPECKV_ERR_WORKSPACE;
    P.B = bt->B; P.G = bt->gamma_max; P.V = bt->V; P.J = 2 * bt->gamma_max + 1;
    const int es = esize(bt->dtype);
    choose_draw(P, bt->dtype, rows_aligned(bt->draft_logits, bt->draft_stride_b, bt->draft_stride_pos, es) &&
                                  rows_aligned(bt->target_logits, bt->target_stride_b, bt->target_stride_pos, es));
    if (P.B >= kShardOneCtaRows && P.draw_pw * P.R * kWarps <= kShardOneCtaGran) {
        P.draw_pw *= P.R;
        P.R = 1;
    }
    P.mode = MODE_VERIFY; P.bits = bt->entropy_in_bits ? 1 : 0;
    P.d = bt->draft_logits; P.dsb = bt->draft_stride_b; P.dsp = bt->draft_stride_pos;
    P.t = bt->target_logits; P.tsb = bt->target_stride_b; P.tsp = bt->target_stride_pos;
    P.tok = bt->draft_tokens; P.gamma = bt->gamma; P.temp = bt->temperature;
    P.temp_scalar = bt->temperature_scalar; P.u = bt->uniforms;
    char* w = static_cast<char*>(ws);
    P.tick1 = reinterpret_cast<int*>(w + pl.off_tick);
    P.tick2 = P.tick1 + P.B;
    P.n_list = P.tick1 + 2 * P.B;
    P.q_front = P.n_list + 1;
    P.q_back = P.n_list + 2;
    P.part = reinterpret_cast<float4*>(w + pl.off_part);
    P.dsum = reinterpret_cast<double*>(w + pl.off_dsum);
    P.dsum2 = reinterpret_cast<double*>(w + pl.off_dsum2);
    P.list = reinterpret_cast<int2*>(w + pl.off_list);
    return SPECKV_OK;
}
bool shard_aligned(const speckv_batch* bt) {
    const int es = esize(bt->dtype);
    return rows_aligned(bt->draft_logits, bt->draft_stride_b, bt->draft_stride_pos, es) &&
           rows_aligned(bt->target_logits, bt->target_stride_b, bt->target_stride_pos, es);
}

// Kernels of speckv_internal_wait_probe: arbitrary status words and empty token slots before the draw
// kernel runs, and afterwards a row epilogue that arrives late and raises each row's completion flag.
__global__ void wait_probe_fill(KParams P) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= P.B) return;
    P.status[b] = 0x5a5a;
    P.out_tok[2 * b] = -1;
    P.out_tok[2 * b + 1] = -1;
}
__global__ void wait_probe_late_epilogue(KParams P) {
    const int b = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (b >= P.B) return;
    if ((threadIdx.x & 31) == 0) P.status[b] = 0;
    __syncwarp();
    row_done_signal(P, b, row_done_slot(P, RS_BONUS), RS_BONUS, 1);
}

}  // namespace

extern "C" {

speckv_status speckv_workspace_size(const speckv_batch* batch, size_t* bytes) {
    if (!bytes) return SPECKV_ERR_INVALID_ARG;
    if (!batch || batch->B < 0 || batch->gamma_max < 1 || batch->V < 1) return SPECKV_ERR_INVALID_ARG;
    if (batch->gamma_max > SPECKV_MAX_GAMMA || batch->V > (1 << 30) || batch->B > (1 << 24))
        return SPECKV_ERR_UNSUPPORTED;
    *bytes = workspace_total(batch);
    return SPECKV_OK;
}

speckv_status speckv_signals(const speckv_batch* batch, float* H, float* C, float* feat,
                             int32_t* row_status, void* workspace, size_t workspace_bytes,
                             void* cuda_stream) {
    return run(batch, MODE_SIGNALS, nullptr, nullptr, H, C, feat, nullptr, nullptr, nullptr, nullptr,
               row_status, workspace, workspace_bytes, cuda_stream);
}

speckv_status speckv_signals_static(const speckv_batch* batch, float* H, float* C, float* feat,
                                    int32_t* row_status, void* cuda_stream) {
    speckv_status st = check_batch(batch, false);
    if (st != SPECKV_OK) return st;
    if (batch->B == 0) return SPECKV_OK;
    if (static_figure(batch) > SPECKV_STATIC_SCRATCH_BYTES) return SPECKV_ERR_STATIC_LIMIT;
    void* scratch = nullptr;
    if (static_scratch_address(&scratch) != cudaSuccess || !scratch) return SPECKV_ERR_CUDA;
    // run() clears the ticket counters on the caller's stream; nothing else needs a known start
    return run(batch, MODE_SIGNALS, nullptr, nullptr, H, C, feat, nullptr, nullptr, nullptr, nullptr,
               row_status, scratch, SPECKV_STATIC_SCRATCH_BYTES, cuda_stream);
}

speckv_status speckv_sample_workspace_size(const speckv_batch* batch, size_t* bytes) {
    if (!bytes) return SPECKV_ERR_INVALID_ARG;
    if (!batch || batch->B < 0 || batch->gamma_max < 1 || batch->V < 1) return SPECKV_ERR_INVALID_ARG;
    if (batch->gamma_max > SPECKV_MAX_GAMMA || batch->V > (1 << 30) || batch->B > (1 << 24))
        return SPECKV_ERR_UNSUPPORTED;
    *bytes = make_sample_plan(batch).total;
    return SPECKV_OK;
}

speckv_status speckv_sample_draft(const speckv_batch* batch, const float* uniforms, int32_t* tokens,
                                  int32_t* row_status, void* workspace, size_t workspace_bytes,
                                  void* cuda_stream) {
    return run_sample(batch, uniforms, tokens, row_status, workspace, workspace_bytes, cuda_stream);
}

speckv_status speckv_select_gamma(int32_t B, const float* feat, const float* comp,
                                  const speckv_mlp* mlp, float* scores, int32_t* gamma_next,
                                  void* cuda_stream) {
    if (B < 0) return SPECKV_ERR_INVALID_ARG;
    speckv_status st = check_mlp(mlp);
    if (st != SPECKV_OK) return st;
    if (B == 0) return SPECKV_OK;
    if (!feat || !gamma_next) return SPECKV_ERR_INVALID_ARG;
    KParams P{};
    P.B = B;
    fill_mlp(P, mlp, comp);
    P.scores = scores; P.gamma_next = gamma_next;
    const int grid = (B + kWarps - 1) / kWarps;
    return launch(select_gamma_kernel, grid, static_cast<cudaStream_t>(cuda_stream), P, feat) == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

speckv_status speckv_verify(const speckv_batch* batch, int32_t* n_accepted, int32_t* out_tokens,
                            int32_t* row_status, void* workspace, size_t workspace_bytes,
                            void* cuda_stream) {
    return run(batch, MODE_VERIFY, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
               n_accepted, out_tokens, row_status, workspace, workspace_bytes, cuda_stream);
}

speckv_status speckv_step(const speckv_batch* batch, const float* comp, const speckv_mlp* mlp,
                          float* H, float* C, float* feat, float* scores, int32_t* gamma_next,
                          int32_t* n_accepted, int32_t* out_tokens, int32_t* row_status,
                          void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return run(batch, MODE_SIGNALS | MODE_VERIFY | MODE_MLP, comp, mlp, H, C, feat, scores, gamma_next,
               n_accepted, out_tokens, row_status, workspace, workspace_bytes, cuda_stream);
}

speckv_status speckv_step_profiled(const speckv_batch* batch, const float* comp, const speckv_mlp* mlp,
                                   float* H, float* C, float* feat, float* scores,
                                   int32_t* gamma_next, int32_t* n_accepted, int32_t* out_tokens,
                                   int32_t* row_status, void* workspace, size_t workspace_bytes,
                                   void* cuda_stream, void* ev_before_sweep, void* ev_after_sweep,
                                   void* ev_after_resample) {
    Events ev;
    ev.before_sweep = static_cast<cudaEvent_t>(ev_before_sweep);
    ev.after_sweep = static_cast<cudaEvent_t>(ev_after_sweep);
    ev.after_resample = static_cast<cudaEvent_t>(ev_after_resample);
    return run(batch, MODE_SIGNALS | MODE_VERIFY | MODE_MLP, comp, mlp, H, C, feat, scores, gamma_next,
               n_accepted, out_tokens, row_status, workspace, workspace_bytes, cuda_stream, ev);
}

#ifdef SPECKV_DEBUG
namespace {
__global__ void dbg_selftest_kernel() {
    // addresses that no call has registered: looked at, never dereferenced
    dbg_ok(reinterpret_cast<const void*>(0x10ull), 16, DBG_LOGIT16);
    dbg_ok(reinterpret_cast<const void*>(0x20ull), 4, DBG_WS_STORE);
}
}  // namespace
#endif

speckv_status speckv_internal_debug_report(unsigned long long* out4, int reset, int selftest) {
#ifdef SPECKV_DEBUG
    if (!out4) return SPECKV_ERR_INVALID_ARG;
    if (selftest) dbg_selftest_kernel<<<1, 1>>>();
    if (cudaDeviceSynchronize() != cudaSuccess) return SPECKV_ERR_CUDA;
    if (cudaMemcpyFromSymbol(out4, g_dbg_report, sizeof(unsigned long long) * 4) != cudaSuccess) return SPECKV_ERR_CUDA;
    if (reset) {
        const unsigned long long zero[4] = {0, 0, 0, 0};
        if (cudaMemcpyToSymbol(g_dbg_report, zero, sizeof zero) != cudaSuccess) return SPECKV_ERR_CUDA;
    }
    return SPECKV_OK;
#else
    (void)out4; (void)reset; (void)selftest;
    return SPECKV_ERR_UNSUPPORTED;
#endif
}

int speckv_internal_set_wait_limit(int polls) {
    if (polls < 1) polls = 1;
    return g_wait_limit.exchange(polls);
}

speckv_status speckv_internal_plan(const speckv_batch* batch, int call, int32_t* plan) {
    if (!plan || call < 0 || call > 3) return SPECKV_ERR_INVALID_ARG;
    const bool verify = call == 1 || call == 3;
    const speckv_status st = check_batch(batch, verify);
    if (st != SPECKV_OK) return st;
    if (batch->B == 0) return SPECKV_ERR_INVALID_ARG;
    KParams P{};
    P.gamma = batch->gamma; P.temp = batch->temperature;
    if (call == 3) P.gamma_next = const_cast<int32_t*>(batch->gamma);
    bool by_row = false;
    if (call == 2) plan_sample(P, batch, make_sample_plan(batch));
    else by_row = plan_call(P, batch, verify ? MODE_SIGNALS | MODE_VERIFY : MODE_SIGNALS);
    const int steps = batch->dtype == SPECKV_BF16 ? SweepShape<__nv_bfloat16>::kSteps : SweepShape<float>::kSteps;
    plan[0] = by_row; plan[1] = P.nsplit; plan[2] = P.per_warp; plan[3] = P.n_spans; plan[4] = P.R; plan[5] = P.draw_pw;
    plan[6] = P.direct;
    plan[7] = call == 2 ? P.fine : 1;
    plan[8] = call == 2 ? P.fine_groups * steps * 32 * (kVec * esize(batch->dtype) / 16) : P.per_warp;
    plan[9] = P.n_tests; plan[10] = P.pos_bits; plan[11] = P.rows_major;
    return SPECKV_OK;
}

speckv_status speckv_internal_wait_probe(int32_t B, int32_t* row_status, int32_t* out_tokens, void* workspace,
                                         size_t workspace_bytes, void* cuda_stream) {
    if (B < 1 || B > 4096 || !row_status || !out_tokens || !workspace) return SPECKV_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(workspace) % kAlign != 0 || workspace_bytes < 2 * static_cast<size_t>(B) * sizeof(int))
        return SPECKV_ERR_WORKSPACE;
    // the draw kernel on its own, one CTA per batch row, with completion flags that nothing raises
    KParams P{};
    P.B = B; P.G = 1; P.V = 256; P.J = 3; P.R = 1; P.draw_pw = 8;
    P.mode = MODE_VERIFY;
    P.wait_limit = g_wait_limit.load(std::memory_order_relaxed);
    P.status = row_status; P.out_tok = out_tokens;
    P.rdone = static_cast<int*>(workspace);
    P.tick2 = P.rdone + B;
    P.q_front = P.q_back = P.tick2;  // the draws' tickets are not reached
    cudaStream_t cs = static_cast<cudaStream_t>(cuda_stream);
    {
        speckv_batch none{};
        if (dbg_register(cs, &none, false, workspace, workspace_bytes) != cudaSuccess) return SPECKV_ERR_CUDA;
    }
    if (cudaMemsetAsync(workspace, 0, 2 * static_cast<size_t>(B) * sizeof(int), cs) != cudaSuccess) return SPECKV_ERR_CUDA;
    wait_probe_fill<<<(B + 255) / 256, 256, 0, cs>>>(P);
    resample_kernel<float><<<static_cast<unsigned>(B), kThreads, 0, cs>>>(P);
    wait_probe_late_epilogue<<<(B + kWarps - 1) / kWarps, kThreads, 0, cs>>>(P);
    return cudaGetLastError() == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

speckv_status speckv_shard_workspace_size(const speckv_batch* local, size_t* bytes) {
    if (!bytes) return SPECKV_ERR_INVALID_ARG;
    if (!local || local->B < 0 || local->gamma_max < 1 || local->V < 1) return SPECKV_ERR_INVALID_ARG;
    if (local->gamma_max > SPECKV_MAX_GAMMA || local->V > (1 << 30) || local->B > (1 << 24))
        return SPECKV_ERR_UNSUPPORTED;
    *bytes = make_shard_plan(local).total;
    return SPECKV_OK;
}

speckv_status speckv_shard_sweep(const speckv_batch* local, int64_t v_begin, float* shard_state, float* shard_tokl,
                                 void* workspace, size_t workspace_bytes, void* cuda_stream) {
    KParams P{};
    ShardPlan pl;
    speckv_status st = shard_params(local, workspace, workspace_bytes, P, pl);
    if (st != SPECKV_OK || local->B == 0) return st;
    if (!shard_state || !shard_tokl || v_begin < 0 || v_begin > (1LL << 30)) return SPECKV_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(shard_state) % 16 != 0 || reinterpret_cast<uintptr_t>(shard_tokl) % 8 != 0) return SPECKV_ERR_INVALID_ARG;
    const bool al = shard_aligned(local);
    choose_slices(P, local->dtype, al, false, kExportSplit);
    if (static_cast<long long>(P.B) * P.J * P.nsplit > 0x7fffffffLL) return SPECKV_ERR_UNSUPPORTED;
    P.v_begin = static_cast<int>(v_begin);
    P.export_state = 1;
    P.state = reinterpret_cast<float4*>(shard_state);
    P.tokl = reinterpret_cast<float2*>(shard_tokl);
    cudaStream_t cs = static_cast<cudaStream_t>(cuda_stream);
    {
        const DbgExtra ex[2] = {{shard_state, static_cast<size_t>(P.B) * P.J * sizeof(float4)},
                                {shard_tokl, static_cast<size_t>(P.B) * P.G * sizeof(float2)}};
        if (dbg_register(cs, local, true, workspace, workspace_bytes, ex, 2) != cudaSuccess) return SPECKV_ERR_CUDA;
    }
    // A slice row is short (V / n_shards columns) and one CTA per short row is mostly overhead, so rows of up to 64 KB are
    // swept by a few warps each, as many as fill the SMs with a granule or two per lane left; wider slices take the
    // CTA-per-slice sweep.
    const long long row_bytes = static_cast<long long>(P.V) * esize(local->dtype), rows = static_cast<long long>(P.B) * P.J;
    if (row_bytes <= kShardWarpRowBytes) {
        int rw = 1;
        while (rw < kWarps && rows * rw < 148 * 4 * kWarps && row_bytes >= 2048LL * rw) rw *= 2;
        const unsigned g2 = static_cast<unsigned>((rows * rw + kWarps - 1) / kWarps);
        const bool bf16 = local->dtype == SPECKV_BF16;
        cudaError_t e;
        if (rw == 1 && row_bytes <= kShardTinyRowBytes)
            e = bf16 ? launch(shard_rows_kernel<__nv_bfloat16, 2, 5>, g2, cs, P, rw) : launch(shard_rows_kernel<float, 2, 5>, g2, cs, P, rw);
        else
            e = bf16 ? launch(shard_rows_kernel<__nv_bfloat16, 5, 4>, g2, cs, P, rw) : launch(shard_rows_kernel<float, 4, 4>, g2, cs, P, rw);
        return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
    }
    if (cudaMemsetAsync(shard_tokl, 0, static_cast<size_t>(P.B) * P.G * sizeof(float2), cs) != cudaSuccess)
        return SPECKV_ERR_CUDA;
    const cudaError_t e = local->dtype == SPECKV_BF16 ? launch_sliced<__nv_bfloat16>(P, 0, cs, nullptr) : launch_sliced<float>(P, 0, cs, nullptr);
    return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

speckv_status speckv_shard_finish(const speckv_batch* local, int32_t n_shards, int32_t shard_width, int32_t V_total,
                                  const float* all_state, const float* all_tokl, const float* comp,
                                  const speckv_mlp* mlp, float* H, float* C, float* feat, float* scores,
                                  int32_t* gamma_next, int32_t* n_accepted, int32_t* out_tokens, int32_t* row_status,
                                  void* row_info, void* cuda_stream) {
    speckv_status st = check_batch(local, true);
    if (st != SPECKV_OK) return st;
    if (n_shards < 1 || n_shards > 32 || shard_width < 1 || V_total < 1) return SPECKV_ERR_INVALID_ARG;
    if (static_cast<long long>(shard_width) * (n_shards - 1) >= V_total) return SPECKV_ERR_INVALID_ARG;
    if (local->B == 0) return SPECKV_OK;
    if (!all_state || !all_tokl || !n_accepted || !out_tokens || !row_info) return SPECKV_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(row_info) % 16 != 0 || reinterpret_cast<uintptr_t>(all_state) % 16 != 0 ||
        reinterpret_cast<uintptr_t>(all_tokl) % 8 != 0)
        return SPECKV_ERR_INVALID_ARG;
    KParams P{};
    P.B = local->B; P.G = local->gamma_max; P.V = V_total; P.J = 2 * local->gamma_max + 1;
    P.mode = MODE_SIGNALS | MODE_VERIFY; P.bits = local->entropy_in_bits ? 1 : 0;
    if (mlp) {
        st = check_mlp(mlp);
        if (st != SPECKV_OK) return st;
        if (!gamma_next || !feat) return SPECKV_ERR_INVALID_ARG;
        P.mode |= MODE_MLP;
        fill_mlp(P, mlp, comp);
    }
    P.tok = local->draft_tokens; P.gamma = local->gamma; P.temp = local->temperature;
    P.temp_scalar = local->temperature_scalar; P.u = local->uniforms;
    P.H = H; P.C = C; P.feat = feat; P.scores = scores; P.gamma_next = gamma_next;
    P.n_acc = n_accepted; P.out_tok = out_tokens; P.status = row_status;
    P.part = const_cast<float4*>(reinterpret_cast<const float4*>(all_state));
    P.part_stride = P.B * P.J;
    P.nsplit = n_shards;
    P.n_shards = n_shards; P.shard_width = shard_width;
    P.tokl = const_cast<float2*>(reinterpret_cast<const float2*>(all_tokl));
    P.tokl_stride = static_cast<long long>(P.B) * P.G;
    P.info = static_cast<RowInfo*>(row_info);
    if (static_cast<long long>(P.B) * P.J > 0x7fffffffLL) return SPECKV_ERR_UNSUPPORTED;
    const unsigned grid = static_cast<unsigned>(P.B);
    {
        speckv_batch none{};  // this call reads no logits: only the gathered arrays and the row records
        const DbgExtra ex[3] = {{all_state, static_cast<size_t>(n_shards) * P.B * P.J * sizeof(float4)},
                                {all_tokl, static_cast<size_t>(n_shards) * P.B * P.G * sizeof(float2)},
                                {row_info, static_cast<size_t>(P.B) * sizeof(RowInfo)}};
        if (dbg_register(static_cast<cudaStream_t>(cuda_stream), &none, false, nullptr, 0, ex, 3) != cudaSuccess) return SPECKV_ERR_CUDA;
    }
    const unsigned threads = P.B >= kShardManyRows ? 64 : kThreads;
    return launch_threads(shard_finish_kernel, grid, threads, static_cast<cudaStream_t>(cuda_stream), P) == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

speckv_status speckv_shard_draw_sums(const speckv_batch* local, const void* row_info, double* shard_weight,
                                     void* workspace, size_t workspace_bytes, void* cuda_stream) {
    KParams P{};
    ShardPlan pl;
    speckv_status st = shard_params(local, workspace, workspace_bytes, P, pl);
    if (st != SPECKV_OK || local->B == 0) return st;
    if (!row_info || !shard_weight || reinterpret_cast<uintptr_t>(row_info) % 16 != 0) return SPECKV_ERR_INVALID_ARG;
    P.info = static_cast<RowInfo*>(const_cast<void*>(row_info));
    P.weight = shard_weight;
    cudaStream_t cs = static_cast<cudaStream_t>(cuda_stream);
    {
        const DbgExtra ex[1] = {{row_info, static_cast<size_t>(P.B) * sizeof(RowInfo)}};
        if (dbg_register(cs, local, true, workspace, workspace_bytes, ex, 1) != cudaSuccess) return SPECKV_ERR_CUDA;
    }
    if (P.R > 1 && cudaMemsetAsync(P.tick2, 0, static_cast<size_t>(P.B) * sizeof(int), cs) != cudaSuccess) return SPECKV_ERR_CUDA;
    if (static_cast<long long>(P.B) * P.R > 0x7fffffffLL) return SPECKV_ERR_UNSUPPORTED;
    const unsigned grid = static_cast<unsigned>(P.B) * static_cast<unsigned>(P.R);
    const cudaError_t e = local->dtype == SPECKV_BF16 ? launch(shard_sums_kernel<__nv_bfloat16>, grid, cs, P)
                                                      : launch(shard_sums_kernel<float>, grid, cs, P);
    return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

speckv_status speckv_shard_draw_pick(const speckv_batch* local, int64_t v_begin, int32_t rank, int32_t n_shards,
                                     const void* row_info, const double* all_weight, int32_t* out_tokens,
                                     void* workspace, size_t workspace_bytes, void* cuda_stream) {
    KParams P{};
    ShardPlan pl;
    speckv_status st = shard_params(local, workspace, workspace_bytes, P, pl);
    if (st != SPECKV_OK || local->B == 0) return st;
    if (!row_info || !all_weight || !out_tokens || reinterpret_cast<uintptr_t>(row_info) % 16 != 0) return SPECKV_ERR_INVALID_ARG;
    if (n_shards < 1 || n_shards > 32 || rank < 0 || rank >= n_shards || v_begin < 0 || v_begin > (1LL << 30))
        return SPECKV_ERR_INVALID_ARG;
    P.info = static_cast<RowInfo*>(const_cast<void*>(row_info));
    P.all_weight = all_weight;
    P.out_tok = out_tokens;
    P.rank = rank; P.n_shards = n_shards; P.v_begin = static_cast<int>(v_begin);
    cudaStream_t cs = static_cast<cudaStream_t>(cuda_stream);
    {
        const DbgExtra ex[1] = {{row_info, static_cast<size_t>(P.B) * sizeof(RowInfo)}};
        if (dbg_register(cs, local, true, workspace, workspace_bytes, ex, 1) != cudaSuccess) return SPECKV_ERR_CUDA;
    }
    const unsigned grid = static_cast<unsigned>(P.B);
    // as many warps as a span has parts of one granule per lane (8,000 rows, V = 128 and 2,000: 45 and 51 -> 11 and 12 us)
    unsigned threads = 32;
    while (threads < kThreads && threads < static_cast<unsigned>(P.draw_pw)) threads *= 2;
    const cudaError_t e = local->dtype == SPECKV_BF16 ? launch_threads(shard_pick_kernel<__nv_bfloat16>, grid, threads, cs, P)
                                                      : launch_threads(shard_pick_kernel<float>, grid, threads, cs, P);
    return e == cudaSuccess ? SPECKV_OK : SPECKV_ERR_CUDA;
}

const char* speckv_status_string(speckv_status s) {
    switch (s) {
        case SPECKV_OK: return "ok";
        case SPECKV_ERR_INVALID_ARG: return "invalid argument";
        case SPECKV_ERR_UNSUPPORTED: return "unsupported size or type";
        case SPECKV_ERR_WORKSPACE: return "workspace too small";
        case SPECKV_ERR_CUDA: return "CUDA launch failed";
        case SPECKV_ERR_STATIC_LIMIT: return "batch needs more scratch than the built-in array holds";
    }
    return "unknown status";
}

int speckv_version(void) { return 100; }

}  // extern "C"
