// Device code of libspeckv: the streaming sweep over vocabulary-sized logit rows and the per-row epilogue (signals,
// acceptance, controller); the draws are in speckv_draw.cuh, the kernels of a step in speckv_sweep.cuh.
//
// Scheme (sm_100a, CUDA cores only -- the work is a streaming reduction, not a contraction):
//   prep kernel     clears the counters and lists the logit rows in use in the order of the sweep's grid.
//   sweep kernel    one CTA per (row b, logit row j, vocabulary slice s).  Each thread keeps
//                   an online-softmax state over 16-byte vector loads, the CTA merges the
//                   256 states and stores one partial.  The last CTA of a batch row to finish
//                   (found with a ticket counter, nobody waits) merges that row's partials,
//                   decides the acceptances, puts the row into the draw queue, writes
//                   the signals and the controller outputs and draws a bonus token.
//   draws           R CTAs per rejected row sum the residual weights of the stop position's two rows,
//                   and the last of them
//                   locates the inverse-CDF threshold and writes the fresh token.  These CTAs
//                   sit behind the sweep CTAs in the sweep kernel's own grid and wait (bounded)
//                   for a row of the queue.
//   direct grid     small batches: prep_direct_kernel clears counters, records and sums; the sweep's CTAs find their logit row from
//                   gamma and the temperatures themselves (direct_entry), and each batch row has drawing CTAs of its own, which wait
//                   (bounded) for the row's record and for one another's sums; the last of them in the grid picks (direct_draw).
//   short rows      one CTA per batch row does all of that in one launch (batch_row_kernel).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace speckv {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kVec = 8;                 // elements per lane per step
constexpr int kMaxShares = 32;          // CTAs that share one draw at most
constexpr int kMaxSplit = 32;
constexpr int kMaxGamma = 16;           // SPECKV_MAX_GAMMA
// Loads in flight per thread (steps of kVec elements: 16 bytes of bf16, 32 of fp32) and CTAs per SM the sweep is compiled for.
// Step of 256 / 1,024 bf16 rows, V = 128,256, and draft sampling of 256: 5 CTAs x 4 steps 141 / 418 / 81 us, 5 x 3 144 / 430 / 83,
// 4 x 4 142 / 437 / 87, 6 x 3 146 / 430 / 88 (the GPU's time, one box).  fp32 needs twice the bytes in flight and fewer
// instructions for them, so fewer warps with more registers: step of 512 rows, V = 151,936, verification of 96 greedy rows,
// and step of 256 rows, V = 128,256: 4 CTAs x 4 steps 502 / 90 / 224 us, 5 x 2 512 / 94.5 / 235, 4 x 3 508 / 91 / 227,
// 5 x 3 (spills) 680 / 111 / 306.
template <typename T> struct SweepShape;
template <> struct SweepShape<__nv_bfloat16> { static constexpr int kSteps = 4, kCtas = 5; };
template <> struct SweepShape<float> { static constexpr int kSteps = 4, kCtas = 4; };
// Every kernel is launched so that its CTAs may be placed as soon as all CTAs of the kernel in front of it in the stream have
// called dependents_may_start() or ended.  It writes memory only behind wait_for_predecessors(), that is when that kernel has
// ended and its writes are visible, and lets its own successor in after that, so what holds for one holds for the whole chain.
// It reads behind it too, but for a direct grid's sweep and draft sampling: the kernel in front of them (prep_direct_kernel,
// clear_kernel) writes nothing but the workspace and has waited for everything in front of it before it let them start, so gamma, the
// temperatures and the logits are complete in L2 and are read from there, past L1 (ldg_early, __ldcg).  That holds for what no CTA of
// the same grid writes: a step that writes the next gamma over this one's takes no direct grid (overwrites_rows() in speckv.cu).
// A kernel is therefore already running while its inputs are written (the drafted tokens, the next gamma and the logits come from
// the call in front of it), so none of them is read through the non-coherent path (__ldg, ld.global.nc), which is for data that
// nobody writes while the kernel runs.  Plain loads cost nothing here: all cases within 0.3 %.
__device__ __forceinline__ void wait_for_predecessors() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
constexpr float kFloor = -1.2676506002282294e30f;  // -2^100: logits below count as -inf
constexpr uint32_t kFloorBf16x2 = 0xF180F180u;     // -2^100 as two bf16
constexpr double kLn2 = 0.6931471805599453094;
constexpr double kLog2e = 1.4426950408889634074;

// ---- bounds-checked build (-DSPECKV_DEBUG) ---------------------------------------------------------
// Every global-memory access whose address comes out of index arithmetic (the logit loads of every
// kernel, the reads and writes of the workspace, the reads of the caller's state arrays in the sharded
// step) is first compared with the extents the host registered for the call.  An access outside them
// is counted, its address kept, and NOT performed: loads give a neutral value, stores are dropped.
// Nothing traps.  In the ordinary build the check is the constant true.
constexpr int kDbgRanges = 8;
struct DbgRanges { unsigned long long lo[kDbgRanges], hi[kDbgRanges]; };
#ifdef SPECKV_DEBUG
__device__ DbgRanges g_dbg_ranges;
__device__ unsigned long long g_dbg_report[4];  // violations, first offending address, its size, the kind of access
__device__ __forceinline__ bool dbg_ok(const void* p, unsigned bytes, int kind) {
    const unsigned long long a = reinterpret_cast<unsigned long long>(p);
#pragma unroll
    for (int k = 0; k < kDbgRanges; ++k)
        if (a >= g_dbg_ranges.lo[k] && a + bytes <= g_dbg_ranges.hi[k]) return true;
    if (atomicAdd(&g_dbg_report[0], 1ull) == 0ull) {
        g_dbg_report[1] = a;
        g_dbg_report[2] = bytes;
        g_dbg_report[3] = static_cast<unsigned long long>(kind);
    }
    return false;
}
#else
__device__ __forceinline__ bool dbg_ok(const void*, unsigned, int) { return true; }
#endif
enum : int { DBG_LOGIT16 = 1, DBG_LOGIT1 = 2, DBG_WS_LOAD = 3, DBG_WS_STORE = 4 };

enum : int { MODE_SIGNALS = 1, MODE_VERIFY = 2, MODE_MLP = 4 };
enum : int { PATH_DRAFT = 0, PATH_TARGET = 1, PATH_ARGMAX = 2 };
enum : int { RS_NONE = 0, RS_RESIDUAL = 1, RS_BONUS = 2 };

struct RowInfo {  // written by the sweep kernel's row epilogue, read by the resample kernel
    int mode;     // RS_*
    int n;        // stop position
    float u2;     // uniform for the resample / bonus draw
    float scale;  // log2(e) / T as used by the sweep
    double lse2_p;  // log2-sum-exp2 of the target row at n
    double lse2_q;  // same for the draft row (residual only)
};

static_assert(sizeof(RowInfo) == 32, "the resample kernel reads a RowInfo as two 16-byte words");

struct KParams {
    int B, G, V, J, nsplit, R, mode, bits;
    int per_warp;  // sweep kernel: 16-byte granules of a logit row that one warp folds; a slice is kWarps times that
    int n_spans;    // spans per batch row (verification) or position (draft sampling)
    int fine, fine_groups;  // draft sampling: spans per warp range, and groups of steps in each (the last one has what is left)
    int2* list;     // sliced sweep: one entry per logit row to sweep, in the order of the grid (prep_kernel)
    int* n_list;    //   and how many there are; CTAs behind the last one draw
    int n_draw;     // sliced sweep: CTAs that may draw (R per batch row), 0 = none
    int direct;  // sweep kernel: a small batch, whose CTAs find their work from gamma and the temperatures themselves, without a list,
                 // and whose draws belong to batch rows, without a queue
    int draw_pw;  // draw: granules of the stop position that one warp sums; R CTAs of kWarps warps per batch row
    int *q_front, *q_back;  // draw queue: rows with a residual draw fill rdone from the front, the others from the back
    int wait_limit;  // polls a resample CTA spends on its row's completion flag before it gives the row up
    // Order of the sweep (verification): first the draft and target row of position 0 of every batch row, then the other draft rows,
    // last the other target rows, position by position (rows_major: batch row by batch row), which are left unread where the walk is
    // already known to have stopped in front of them (early != nullptr).
    int read_all;
    int* early;       // [B] the lowest position + 1 at which a test has ended the walk so far
    unsigned long long* tick_pos;  // [B] arrivals of each position's draft and target slices, pos_bits bits each
    int pos_bits, n_tests;  // positions from n_tests on are not tested
    int rows_major;
    const void* d; long long dsb, dsp;
    const void* t; long long tsb, tsp;
    const int* tok; const int* gamma; const float* temp; float temp_scalar; const float* u;
    // controller
    int n_in, n_hidden, n_out, layout, transform, n_comp;
    const float *W1, *b1, *W2, *b2, *comp;
    int gch[8];
    // outputs
    float *H, *C, *feat, *scores;
    int *gamma_next, *n_acc, *out_tok, *status;
    // workspace
    int *tick1, *tick2;
    float2* tokl;  // [B, G] (draft logit, target logit) at the draft token, left by the register-staged sweep; may be NULL
    int* rdone;  // verification: the draw queue's slots, one per batch row (row_done_signal); draft-side sampling: row status
    RowInfo* info;
    float4* part;
    float2* spans;  // (reference, sum) of every warp's range of the row a plain draw may need: verification [B, nsplit * kWarps]
                    // (target position gamma_b), draft-side sampling [B * G, n_spans]
    double* dsum;   // draw: [B, kMaxShares * kWarps] span weights of the stop position
    double* dsum2;  // shard draw: the same of p beside the residual's
    // vocabulary-sharded verification (speckv_shard.cuh); all zero otherwise
    int part_stride;   // row epilogue: float4s between successive partials of one logit row (0 = adjacent)
    int n_shards;      // row epilogue: tokl holds one [B, G] table per shard, tokl_stride float2s apart
    int shard_width;   //   and the shard owning token x is min(x / shard_width, n_shards - 1)
    long long tokl_stride;
    int v_begin;       // sweep: first vocabulary index of this shard's slice (the batch's V is the slice width)
    int export_state;  // sweep: 1 = the row's last CTA writes the merged per-logit-row states instead of the row epilogue
    float4* state;     // [B, J] merged states of this shard (export)
    double* weight;    // shard draw: [B, 2] (residual mass, p mass) of this shard
    const double* all_weight;  // [n_shards, B, 2]
    int rank;
};

// ----------------------------------------------------------------------------------------
// small helpers
// ----------------------------------------------------------------------------------------
// A kernel's parameters for the functions that are not inlined: handed a reference to the parameter itself they fetch every field
// as global memory, a miss each the first time, and a row epilogue is a chain of cold fields.  With these copied while the tickets
// travel and one scan less per pick (speckv_draw.cuh): step of 16 bf16 rows, V = 128,256, 33.4 -> 30.7 us, of 64, V = 32,000,
// 30.8 -> 27.5, of 4, V = 70,528, 16.5 -> 13.7.  Thread first + k copies word k; the
// caller has a barrier before the first use.
__device__ __forceinline__ void params_to_shared(const KParams& P, KParams* sh, int first) {
    for (int k = static_cast<int>(threadIdx.x) - first; k >= 0 && k < static_cast<int>(sizeof(KParams) / 4); k += static_cast<int>(blockDim.x) - first)
        reinterpret_cast<int*>(sh)[k] = reinterpret_cast<const int*>(&P)[k];
}
__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Packed pairs of fp32 (sm_100 f32x2 arithmetic): one instruction works on two elements.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 ex2_2(f2 a) {
    float x, y;
    unpack2(a, x, y);
    return pack2(ex2f(x), ex2f(y));
}
__device__ __forceinline__ float hsum2(f2 a) {
    float x, y;
    unpack2(a, x, y);
    return x + y;
}

__device__ __forceinline__ float max_nan(float a, float b) {  // NaN-propagating max
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
    uint4 v;
    if (!dbg_ok(p, 16, DBG_LOGIT16)) return make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
// The same for a kernel that reads before its griddepcontrol.wait: straight from L2, since a line that L1 still holds of an
// earlier kernel's read may be older than what has been written since.
__device__ __forceinline__ uint4 ldg_early(const void* p) {
    uint4 v;
    if (!dbg_ok(p, 16, DBG_LOGIT16)) return make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
    asm volatile("ld.relaxed.gpu.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ __nv_bfloat162 as_bf2(uint32_t u) {
    return *reinterpret_cast<__nv_bfloat162*>(&u);
}
__device__ __forceinline__ uint32_t as_u32(__nv_bfloat162 h) {
    return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// Raw register image of kVec consecutive elements.
template <typename T> struct Raw;
template <> struct Raw<__nv_bfloat16> { uint4 a; };
template <> struct Raw<float> { uint4 a, b; };

template <typename T> __device__ __forceinline__ Raw<T> raw_fill(float v);
template <> __device__ __forceinline__ Raw<__nv_bfloat16> raw_fill<__nv_bfloat16>(float v) {
    uint32_t h = __float_as_uint(v) >> 16;  // callers pass bf16-representable values
    h |= h << 16;
    Raw<__nv_bfloat16> r; r.a = make_uint4(h, h, h, h); return r;
}
template <> __device__ __forceinline__ Raw<float> raw_fill<float>(float v) {
    uint32_t w = __float_as_uint(v);
    Raw<float> r; r.a = make_uint4(w, w, w, w); r.b = r.a; return r;
}

template <typename T> __device__ __forceinline__ void unpack(const Raw<T>& r, float (&x)[kVec]);
template <> __device__ __forceinline__ void unpack<__nv_bfloat16>(const Raw<__nv_bfloat16>& r, float (&x)[kVec]) {
    x[0] = bf_lo(r.a.x); x[1] = bf_hi(r.a.x); x[2] = bf_lo(r.a.y); x[3] = bf_hi(r.a.y);
    x[4] = bf_lo(r.a.z); x[5] = bf_hi(r.a.z); x[6] = bf_lo(r.a.w); x[7] = bf_hi(r.a.w);
}
template <> __device__ __forceinline__ void unpack<float>(const Raw<float>& r, float (&x)[kVec]) {
    x[0] = __uint_as_float(r.a.x); x[1] = __uint_as_float(r.a.y);
    x[2] = __uint_as_float(r.a.z); x[3] = __uint_as_float(r.a.w);
    x[4] = __uint_as_float(r.b.x); x[5] = __uint_as_float(r.b.y);
    x[6] = __uint_as_float(r.b.z); x[7] = __uint_as_float(r.b.w);
}

// the same kVec elements as four packed pairs
__device__ __forceinline__ void unpack_pairs(const Raw<__nv_bfloat16>& r, f2 (&x)[4]) {
    x[0] = pack2(bf_lo(r.a.x), bf_hi(r.a.x)); x[1] = pack2(bf_lo(r.a.y), bf_hi(r.a.y));
    x[2] = pack2(bf_lo(r.a.z), bf_hi(r.a.z)); x[3] = pack2(bf_lo(r.a.w), bf_hi(r.a.w));
}
__device__ __forceinline__ void unpack_pairs(const Raw<float>& r, f2 (&x)[4]) {
    x[0] = pack2(__uint_as_float(r.a.x), __uint_as_float(r.a.y));
    x[1] = pack2(__uint_as_float(r.a.z), __uint_as_float(r.a.w));
    x[2] = pack2(__uint_as_float(r.b.x), __uint_as_float(r.b.y));
    x[3] = pack2(__uint_as_float(r.b.z), __uint_as_float(r.b.w));
}

__device__ __forceinline__ float elem_to_float(const __nv_bfloat16* p, long long i) {
    if (!dbg_ok(p + i, 2, DBG_LOGIT1)) return 0.f;
    return __uint_as_float(static_cast<uint32_t>(reinterpret_cast<const unsigned short*>(p)[i]) << 16);
}
__device__ __forceinline__ float elem_to_float(const float* p, long long i) {
    if (!dbg_ok(p + i, 4, DBG_LOGIT1)) return 0.f;
    return p[i];
}

// NaN-propagating maximum of the kVec raw elements.
__device__ __forceinline__ float raw_max(const Raw<__nv_bfloat16>& r) {
    __nv_bfloat162 m = __hmax2_nan(__hmax2_nan(as_bf2(r.a.x), as_bf2(r.a.y)),
                                   __hmax2_nan(as_bf2(r.a.z), as_bf2(r.a.w)));
    uint32_t u = as_u32(m);
    return max_nan(bf_lo(u), bf_hi(u));
}
__device__ __forceinline__ float raw_max(const Raw<float>& r) {
    float a = max_nan(max_nan(__uint_as_float(r.a.x), __uint_as_float(r.a.y)),
                      max_nan(__uint_as_float(r.a.z), __uint_as_float(r.a.w)));
    float b = max_nan(max_nan(__uint_as_float(r.b.x), __uint_as_float(r.b.y)),
                      max_nan(__uint_as_float(r.b.z), __uint_as_float(r.b.w)));
    return max_nan(a, b);
}

// Is any raw element >= m (or a NaN)?  For bf16 the test runs on packed pairs; m must be bf16-representable there.
__device__ __forceinline__ bool raw_exceeds(const Raw<__nv_bfloat16>& r, float m) {
    __nv_bfloat162 mx = __hmax2_nan(__hmax2_nan(as_bf2(r.a.x), as_bf2(r.a.y)),
                                    __hmax2_nan(as_bf2(r.a.z), as_bf2(r.a.w)));
    uint32_t mb = __float_as_uint(m) >> 16;
    return !__hblt2(mx, as_bf2(mb | (mb << 16)));
}
__device__ __forceinline__ bool raw_exceeds(const Raw<float>& r, float m) { return !(raw_max(r) < m); }
// The same for two at once.
__device__ __forceinline__ bool raw_exceeds2(const Raw<__nv_bfloat16>& r, const Raw<__nv_bfloat16>& s, float m) {
    const __nv_bfloat162 a = __hmax2_nan(__hmax2_nan(as_bf2(r.a.x), as_bf2(r.a.y)), __hmax2_nan(as_bf2(r.a.z), as_bf2(r.a.w)));
    const __nv_bfloat162 b = __hmax2_nan(__hmax2_nan(as_bf2(s.a.x), as_bf2(s.a.y)), __hmax2_nan(as_bf2(s.a.z), as_bf2(s.a.w)));
    const uint32_t u = as_u32(__hmax2_nan(a, b));
    return !(max_nan(bf_lo(u), bf_hi(u)) < m);
}
__device__ __forceinline__ bool raw_exceeds2(const Raw<float>& r, const Raw<float>& s, float m) {
    return !(max_nan(raw_max(r), raw_max(s)) < m);
}

// How many raw elements equal m; they become -inf.
__device__ __forceinline__ float raw_take_equal(Raw<__nv_bfloat16>& r, float m) {  // m is bf16-representable
    float n = 0.f;
    auto take = [&](uint32_t& w) {  // by value, so that the two zeros are equal
        if (bf_lo(w) == m) { w = (w & 0xFFFF0000u) | 0xFF80u; n += 1.f; }
        if (bf_hi(w) == m) { w = (w & 0x0000FFFFu) | 0xFF800000u; n += 1.f; }
    };
    take(r.a.x); take(r.a.y); take(r.a.z); take(r.a.w);
    return n;
}
__device__ __forceinline__ float raw_take_equal(Raw<float>& r, float m) {
    float n = 0.f;
    auto take = [&](uint32_t& w) {
        if (__uint_as_float(w) == m) { w = 0xFF800000u; n += 1.f; }
    };
    take(r.a.x); take(r.a.y); take(r.a.z); take(r.a.w);
    take(r.b.x); take(r.b.y); take(r.b.z); take(r.b.w);
    return n;
}
// Clamp the raw elements from below at kFloor (NaN becomes kFloor as well).
__device__ __forceinline__ void raw_floor(Raw<__nv_bfloat16>& r) {
    const __nv_bfloat162 f = as_bf2(kFloorBf16x2);
    r.a.x = as_u32(__hmax2(as_bf2(r.a.x), f));
    r.a.y = as_u32(__hmax2(as_bf2(r.a.y), f));
    r.a.z = as_u32(__hmax2(as_bf2(r.a.z), f));
    r.a.w = as_u32(__hmax2(as_bf2(r.a.w), f));
}
__device__ __forceinline__ void raw_floor(Raw<float>& r) {
    r.a.x = __float_as_uint(fmaxf(__uint_as_float(r.a.x), kFloor));
    r.a.y = __float_as_uint(fmaxf(__uint_as_float(r.a.y), kFloor));
    r.a.z = __float_as_uint(fmaxf(__uint_as_float(r.a.z), kFloor));
    r.a.w = __float_as_uint(fmaxf(__uint_as_float(r.a.w), kFloor));
    r.b.x = __float_as_uint(fmaxf(__uint_as_float(r.b.x), kFloor));
    r.b.y = __float_as_uint(fmaxf(__uint_as_float(r.b.y), kFloor));
    r.b.z = __float_as_uint(fmaxf(__uint_as_float(r.b.z), kFloor));
    r.b.w = __float_as_uint(fmaxf(__uint_as_float(r.b.w), kFloor));
}

// ----------------------------------------------------------------------------------------
// Sums and maxima over the warp
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_maxf(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ----------------------------------------------------------------------------------------
// Per-thread sweep states.  All three share the shape (a, b, c, d) of a float4 partial.
//
// DRAFT   a = m (running max, logit units), b = cnt (elements equal to m that are kept out of
//         the sum so that a dominant token never absorbs the tail), c = Zx = sum over the other
//         elements of 2^((x-m)*scale), d = S = sum of 2^((x-m)*scale) * (x-m).
//         Z = cnt + Zx; entropy (nats) = ln Z - ln2*scale*S/Z; confidence = 1/Z  (Sec. 4.2).
//         cnt = NaN marks a NaN / +inf input.
//         While it sweeps, a thread keeps its sums against r = fl(m * scale), so that an element's exponent is one
//         fused multiply-add; partial() moves them to m itself.  That needs r close to m * scale: where it is not (far(): the
//         rounding of |r| > 2^28 is up to 2^5 and more, or kFloor * scale overflows or is next to 0) the warp's range is folded
//         again by draft_far(), from differences of logits.
// TARGET  a = r (reference, log2 units), b = Z = sum 2^(x*scale - r); c,d unused.  Any r serves that keeps the sum in
//         range; it is not the maximum.  NaN / +inf inputs surface as a non-finite Z.
// ARGMAX  a = best value, b = index (bit pattern), c = bad flag (non-zero: NaN / +inf seen).
// ----------------------------------------------------------------------------------------
struct DraftState {
    float m, r, cnt;
    f2 za, sa;  // two running sums each of Zx and of 2^y * y, y = x * scale - r
    bool bad;
    __device__ __forceinline__ void init(float m0, float scale) {
        m = m0; r = __fmul_rn(m0, scale); cnt = 0.f; bad = false;
        za = sa = pack2(0.f, 0.f);
    }
    __device__ __forceinline__ float zsum() const { return hsum2(za); }
    __device__ __forceinline__ float ssum() const { return hsum2(sa); }

    // The warp's maximum m is the same in all lanes, and a step in which any lane holds an element >= m (or a NaN) is taken by all
    // of them here: the new maximum is the warp's, so that from then on only a still larger element comes this way.
    // (A maximum per lane left each of the elements above the first reference to come here by itself, about as many as the range is
    // longer than what the reference was taken from, at 200 instructions each; the range takes 45 a step.)
    __device__ __forceinline__ void raise(float v, float scale) {  // everything gathered so far moves below the new maximum v > m
        const float rn = __fmul_rn(v, scale), dr = __fsub_rn(r, rn), f = ex2f(dr);
        const float y = fmaf(m, scale, -r), zc = cnt * ex2f(y);  // the elements equal to the old maximum join the sums
        const float z = zsum();
        float sv = fmaf(dr, zc + z, fmaf(zc, y, ssum())) * f;
        if (f == 0.f) sv = 0.f;  // a product with dr, which behind masked elements is about 2^100 * scale, may be infinite
        za = pack2((zc + z) * f, 0.f);
        sa = pack2(sv, 0.f);
        cnt = 0.f;
        m = v;
        r = rn;
    }
    // the lane's largest finite element; notes a NaN / +inf
    template <typename T>
    __device__ __forceinline__ float finite_max(const Raw<T>& raw) {
        const float v = raw_max(raw);
        if (v < __int_as_float(0x7f800000)) return v;
        bad = true;
        return kFloor;
    }
    // counts the elements equal to m and takes them out of the step
    template <typename T>
    __device__ __forceinline__ void take_top(Raw<T>& raw) {
        cnt += raw_take_equal(raw, m);
    }

    template <typename T>
    __device__ __forceinline__ void add(Raw<T> raw, float scale) {  // all elements below m
        raw_floor(raw);
        f2 x[4];
        unpack_pairs(raw, x);
        const f2 sc2 = pack2(scale, scale), nr2 = pack2(-r, -r);
        const f2 y0 = fma2(x[0], sc2, nr2), y1 = fma2(x[1], sc2, nr2), y2 = fma2(x[2], sc2, nr2), y3 = fma2(x[3], sc2, nr2);
        const f2 e0 = ex2_2(y0), e1 = ex2_2(y1), e2 = ex2_2(y2), e3 = ex2_2(y3);
        za = add2(za, add2(add2(e0, e1), add2(e2, e3)));
        sa = add2(sa, fma2(e0, y0, fma2(e1, y1, fma2(e2, y2, mul2(e3, y3)))));
    }
    template <typename T>
    __device__ __forceinline__ void step(const Raw<T>& raw, float scale) {
        Raw<T> v = raw;
        if (__any_sync(0xffffffffu, raw_exceeds(raw, m))) {  // rare after the warm start
            const float top = warp_maxf(finite_max<T>(v));
            if (top > m) raise(top, scale);
            take_top<T>(v);
        }
        add<T>(v, scale);
    }
    // two steps with one test for both (for four the registers run out: signals of 128 bf16 rows, V = 128,256, 53 us; 48 this
    // way; 50 with a test for each)
    template <typename T>
    __device__ __forceinline__ void step2(Raw<T>& a, Raw<T>& b, float scale) {
        if (__any_sync(0xffffffffu, raw_exceeds2(a, b, m))) {
            const float top = warp_maxf(fmaxf(finite_max<T>(a), finite_max<T>(b)));
            if (top > m) raise(top, scale);
            take_top<T>(a);
            take_top<T>(b);
        }
        add<T>(a, scale);
        add<T>(b, scale);
    }
    // Sums that are not to be used: see above.  A maximum far below zero that was left behind shows in what it did to them.  (Below
    // 2^-93 the exponent of kFloor is above -128, and an element that only stands for none has weight.)
    __device__ __forceinline__ bool far(const float4& part, float scale) const {
        return !bad && (scale > 0x1p27f || scale < 0x1p-93f || (m > kFloor && !(fabsf(r) <= 0x1p28f)) || !(fabsf(part.z) + fabsf(part.w) < __int_as_float(0x7f800000)));
    }
    __device__ __forceinline__ float4 partial(float scale) const {
        const float d = fmaf(m, scale, -r), f = ex2f(-d), z = zsum();  // y against m itself is smaller by d, a rounding
        return make_float4(m, bad ? __int_as_float(0x7fc00000) : cnt, z * f, fmaf(-d, z, ssum()) * f / scale);
    }
};

// (m, cnt, Zx, S) merge; `scale` converts logit units to log2 units.
__device__ __forceinline__ float4 merge_draft(float4 a, float4 b, float scale) {
    float m = fmaxf(a.x, b.x);
    float da = a.x - m, db = b.x - m;
    float fa = ex2f(da * scale), fb = ex2f(db * scale);
    float za = a.y + a.z, zb = b.y + b.z;
    float4 r;
    r.x = m;
    r.y = (a.x == m ? a.y : 0.f) + (b.x == m ? b.y : 0.f);
    r.z = (a.x == m ? a.z : za * fa) + (b.x == m ? b.z : zb * fb);
    r.w = (a.x == m ? a.w : fmaf(da, za, a.w) * fa) + (b.x == m ? b.w : fmaf(db, zb, b.w) * fb);
    // a NaN count must survive even when its side is scaled away
    if (a.y != a.y || b.y != b.y) r.y = __int_as_float(0x7fc00000);
    return r;
}

constexpr float kBigSum = 1.1529215e18f;  // 2^60

// The sums of a group of steps are gathered apart and looked at once: an element far above the reference shows as a sum
// beyond 2^60 (or an overflow, or a NaN), and only then is the group read again and the reference raised.  No element
// is compared with anything: 24 instructions per 8 bf16 elements instead of 30 (with the draft's exponent in one
// fused multiply-add and four loads in flight: draft sampling of 256 rows, V = 128,256, 83 -> 81 us, step 142.5 -> 141).
struct TargetState {
    float r, z;
    // (finite also where masked elements stand in front, m0 = kFloor, and the temperature is so low that kFloor * scale overflows)
    __device__ __forceinline__ void init(float m0, float scale) { r = fmaxf(__fmul_rn(m0, scale), -3.0e38f); z = 0.f; }
    template <typename T>
    __device__ __forceinline__ void add(const Raw<T>& raw, float scale, f2& ga, f2& gb) const {
        f2 x[4];
        unpack_pairs(raw, x);
        const f2 sc2 = pack2(scale, scale), nr2 = pack2(-r, -r);
        const f2 e0 = ex2_2(fma2(x[0], sc2, nr2)), e1 = ex2_2(fma2(x[1], sc2, nr2));
        const f2 e2 = ex2_2(fma2(x[2], sc2, nr2)), e3 = ex2_2(fma2(x[3], sc2, nr2));
        ga = add2(ga, e0); gb = add2(gb, e1);
        ga = add2(ga, e2); gb = add2(gb, e3);
    }
    // one step with its maximum taken first; returns what the sum gathered so far was multiplied by
    template <typename T>
    __device__ __forceinline__ float careful(const Raw<T>& raw, float scale) {
        const float v = raw_max(raw), rn = __fmul_rn(v, scale);
        if (!(v < __int_as_float(0x7f800000))) { z = __int_as_float(0x7fc00000); return 1.f; }
        float f = 1.f;
        if (rn > r) { f = ex2f(__fsub_rn(r, rn)); z *= f; r = rn; }
        f2 ga = pack2(0.f, 0.f), gb = ga;
        add(raw, scale, ga, gb);
        z += hsum2(add2(ga, gb));
        return f;
    }
    __device__ __forceinline__ float4 partial() const { return make_float4(r, z, 0.f, 0.f); }
};

__device__ __forceinline__ float4 merge_target(float4 a, float4 b) {
    float r = fmaxf(a.x, b.x);
    float4 o;
    o.x = r;
    o.y = a.y * ex2f(a.x - r) + b.y * ex2f(b.x - r);
    if (a.y != a.y || b.y != b.y) o.y = __int_as_float(0x7fc00000);
    o.z = o.w = 0.f;
    return o;
}

struct ArgmaxState {
    float best; int idx; bool bad;
    __device__ __forceinline__ void init(float m0) { best = m0; idx = 0x7fffffff; bad = false; }
    // the two halves of kVec/2 elements start at vocabulary index ea and eb
    template <typename T>
    __device__ __forceinline__ void step(const Raw<T>& raw, int ea, int eb) {
        if (!raw_exceeds(raw, best)) return;
        float x[kVec];
        unpack<T>(raw, x);
#pragma unroll
        for (int j = 0; j < kVec; ++j) {
            const int idx_j = (j < kVec / 2) ? ea + j : eb + j - kVec / 2;
            bad |= (x[j] != x[j]) || (x[j] == __int_as_float(0x7f800000));
            if (x[j] > best || (x[j] == best && idx_j < idx)) { best = x[j]; idx = idx_j; }
        }
    }
    __device__ __forceinline__ float4 partial() const {
        return make_float4(best, __int_as_float(idx), bad ? 1.f : 0.f, 0.f);
    }
};

__device__ __forceinline__ float4 merge_argmax(float4 a, float4 b) {
    int ia = __float_as_int(a.y), ib = __float_as_int(b.y);
    bool take_b = (b.x > a.x) || (b.x == a.x && ib < ia);
    float4 o = take_b ? b : a;
    o.z = a.z + b.z;
    return o;
}

__device__ __forceinline__ float4 shfl_xor4(float4 v, int mask) {
    v.x = __shfl_xor_sync(0xffffffffu, v.x, mask);
    v.y = __shfl_xor_sync(0xffffffffu, v.y, mask);
    v.z = __shfl_xor_sync(0xffffffffu, v.z, mask);
    v.w = __shfl_xor_sync(0xffffffffu, v.w, mask);
    return v;
}

// ----------------------------------------------------------------------------------------
// Warp-level merge of the 32 per-thread partials (result valid in every lane).
// DRAFT / TARGET: bring every lane to the warp-wide reference, then plain sums.
// ----------------------------------------------------------------------------------------
template <int PATH>
__device__ __forceinline__ float4 warp_merge(float4 p, float scale) {
    if constexpr (PATH == PATH_DRAFT) {
        const float M = warp_maxf(p.x);
        if (p.x != M) {  // this lane's maximum is not the warp's: its count joins the scaled sum
            const float dm = p.x - M, f = ex2f(dm * scale), za = p.y + p.z;
            p.w = fmaf(dm, za, p.w) * f;
            p.z = za * f;
            p.y = 0.f;
        }
        return make_float4(M, warp_sumf(p.y), warp_sumf(p.z), warp_sumf(p.w));
    } else if constexpr (PATH == PATH_TARGET) {
        const float R = warp_maxf(p.x);
        return make_float4(R, warp_sumf(p.y * ex2f(p.x - R)), 0.f, 0.f);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) p = merge_argmax(p, shfl_xor4(p, o));
        return p;
    }
}

// ----------------------------------------------------------------------------------------
// A logit row as 16-byte granules of the address space.  A row may start and end inside a granule (an odd vocabulary
// size shifts every row against the 16-byte grid): the sums do not care in which lane an element is folded, so whole
// granules are loaded wherever the row sits and only the first and the last one, where they are shared with a
// neighbouring row, are fetched element by element.  (Element by element throughout, an unaligned row was bound by its
// load instructions: signals of 700 fp32 rows, gamma 4, V = 30,001: 92.8 us, this way 57.2; step of 300 bf16 rows, gamma up
// to 6, V = 50,257: 132.9 -> 90.1 us.)
// ----------------------------------------------------------------------------------------
struct GranRow {
    const uint4* base;  // the row's first granule (its address rounded down to 16 bytes)
    int ng;             // granules that hold elements of the row
    int meta;           // bits 0-3: elements of the first granule in front of the row; 4-7: elements of the last granule
                        // that are the row's (0: all)
    __device__ __forceinline__ int shift() const { return meta & 15; }
    __device__ __forceinline__ int tail() const { return meta >> 4; }
    __device__ __forceinline__ int whole_lo() const { return shift() ? 1 : 0; }        // whole granules: [whole_lo, whole_hi)
    __device__ __forceinline__ int whole_hi() const { return ng - (tail() ? 1 : 0); }
};
template <typename T>
__device__ __forceinline__ GranRow make_row(const T* p, int V) {
    constexpr int E = 16 / sizeof(T);
    GranRow r;
    const unsigned long long a = reinterpret_cast<unsigned long long>(p);
    const int shift = static_cast<int>(a & 15) / static_cast<int>(sizeof(T));
    r.base = reinterpret_cast<const uint4*>(a & ~15ull);
    r.ng = (shift + V + E - 1) / E;
    r.meta = shift | (((shift + V) % E) << 4);
    return r;
}
template <typename T>
__device__ __forceinline__ uint4 gran_fill(float v) {  // bf16: v is representable
    uint32_t h = __float_as_uint(v);
    if constexpr (sizeof(T) == 2) h = (h >> 16) | (h & 0xFFFF0000u);
    return make_uint4(h, h, h, h);
}
// A first or last granule that is only partly the row's; the rest of it reads as `pad`.
template <typename T>
__device__ __noinline__ uint4 gran_edge(const GranRow r, int g, float pad) {
    constexpr int E = 16 / sizeof(T);
    const T* p = reinterpret_cast<const T*>(r.base + g);
    const int lo = g == 0 ? r.shift() : 0;
    const int hi = (g == r.ng - 1 && r.tail()) ? r.tail() : E;
    float x[E];
#pragma unroll
    for (int j = 0; j < E; ++j) x[j] = (j >= lo && j < hi) ? elem_to_float(p, j) : pad;
    uint4 o;
    if constexpr (sizeof(T) == 2) {
        o.x = (__float_as_uint(x[0]) >> 16) | (__float_as_uint(x[1]) & 0xFFFF0000u);
        o.y = (__float_as_uint(x[2]) >> 16) | (__float_as_uint(x[3]) & 0xFFFF0000u);
        o.z = (__float_as_uint(x[4]) >> 16) | (__float_as_uint(x[5]) & 0xFFFF0000u);
        o.w = (__float_as_uint(x[6]) >> 16) | (__float_as_uint(x[7]) & 0xFFFF0000u);
    } else {
        o = make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
    }
    return o;
}

// Any granule, whole or not.
template <typename T>
__device__ __forceinline__ uint4 gran_any(const GranRow& r, int g) {  // outside the row: -inf, that is weight 0
    const float ninf = __int_as_float(0xff800000);
    if (g < 0 || g >= r.ng) return gran_fill<T>(ninf);
    if (g < r.whole_lo() || g >= r.whole_hi()) return gran_edge<T>(r, g, ninf);
    return ldg_stream(r.base + g);
}

// One warp: the draft partial of granules [lo, hi) for logits and temperatures of any size (DraftState::far), every exponent
// (x - m) * scale from a difference of logits.  Plain rather than fast: a row takes it from |logit| / T of 2e8 on, or from T of 1.4e28.
template <typename T>
__device__ __noinline__ float4 draft_far(const T* p, int V, int lo, int hi, float scale) {
    constexpr int E = 16 / sizeof(T);
    const GranRow row = make_row(p, V);
    float m = kFloor, cnt = 0.f, z = 0.f, s = 0.f;  // s: of 2^y * y
    bool bad = false;
    for (int g = lo + (threadIdx.x & 31); g < min(hi, row.ng); g += 32) {
        const uint4 v = gran_any<T>(row, g);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < E; ++j) {
            float x = sizeof(T) == 4 ? __uint_as_float(w[j % 4]) : (j & 1) ? bf_hi(w[j / 2]) : bf_lo(w[j / 2]);
            bad |= x != x || x == __int_as_float(0x7f800000);
            if (!(x > kFloor)) continue;  // no weight at any temperature
            const float y = -fabsf(x - m) * scale, e = ex2f(y);  // y may be infinite (and at scale = inf not a number where x = m)
            if (x > m) {
                s = e > 0.f ? fmaf(y, cnt + z, s) * e : 0.f;
                z = (cnt + z) * e;
                cnt = 1.f;
                m = x;
            } else if (x == m) {
                cnt += 1.f;
            } else if (e > 0.f) {
                z += e;
                s = fmaf(e, y, s);
            }
        }
    }
    return warp_merge<PATH_DRAFT>(make_float4(m, bad ? __int_as_float(0x7fc00000) : cnt, z, s / scale), scale);
}

constexpr int kFineStride = kThreads + 4;  // floats between the sums of a lane's pieces, so that 4 lanes each can read one piece
constexpr int kMostFine = 8;
// ----------------------------------------------------------------------------------------
// One WARP sweeps granules [lo, hi) of one logit row.  Lane l owns
// granules l, l+32, ... of the range; a step folds kVec elements per lane (bf16: one granule, fp32: two granules 32
// apart, so that every load of the warp covers 512 contiguous bytes), U steps are in flight.  Warps of a CTA take
// adjacent ranges and never wait for one another once the loop runs.
//   start   requests the first U steps: all it takes is the row's address
//   warm    the reference the sums start from: the largest element of the first steps, over the warp, or over the CTA whose
//           warps sweep ranges of the same row (one barrier, every warp must call)
//   run     folds the range and returns the merged partial in every lane
// ----------------------------------------------------------------------------------------
template <typename T, int U>
struct WarpSweep {
    static constexpr int E = 16 / sizeof(T);
    static constexpr int GS = kVec / E;  // granules per lane and step
    const uint4* p;
    int a, left, n_main, meta, ng;
    bool first_edge, last_edge;
    Raw<T> buf[U];

    template <bool EARLY = false>
    __device__ __forceinline__ Raw<T> load(int k) const {
        auto ld = [](const uint4* q) { return EARLY ? ldg_early(q) : ldg_stream(q); };
        Raw<T> r;
        r.a = ld(p + 32 * GS * k);
        if constexpr (GS == 2) r.b = (left > 64 * k + 32) ? ld(p + 64 * k + 32) : gran_fill<T>(__int_as_float(0xff800000));
        return r;
    }
    // incomplete granules: lane 0 the row's first, lane 1 its last
    __device__ __forceinline__ Raw<T> edge() const {
        const int lane = threadIdx.x & 31;
        GranRow row;
        row.base = p - a - lane; row.ng = ng; row.meta = meta;
        Raw<T> e = raw_fill<T>(__int_as_float(0xff800000));
        if (first_edge && lane == 0) e.a = gran_edge<T>(row, 0, __int_as_float(0xff800000));
        if (last_edge && lane == 1) e.a = gran_edge<T>(row, ng - 1, __int_as_float(0xff800000));
        return e;
    }
    template <bool EARLY = false>  // in front of the kernel's griddepcontrol.wait
    __device__ __forceinline__ void start(const GranRow& row, int lo, int hi) {
        const int lane = threadIdx.x & 31;
        a = max(lo, row.whole_lo());
        left = min(hi, row.whole_hi()) - a - lane;  // whole granules from this lane's first one on
        n_main = left > 0 ? (left + 32 * GS - 1) / (32 * GS) : 0;
        p = row.base + a + lane;
        meta = row.meta;
        ng = row.ng;
        first_edge = row.shift() != 0 && lo == 0 && hi > 0;
        last_edge = row.tail() != 0 && row.ng - 1 >= lo && row.ng - 1 < hi && !(row.shift() != 0 && row.ng == 1);
#pragma unroll
        for (int k = 0; k < U; ++k) {
            buf[k] = raw_fill<T>(__int_as_float(0xff800000));
            if (k < n_main) buf[k] = load<EARLY>(k);
        }
    }
    // A step holding NaN / +inf / only -inf contributes the floor; its owner meets the offending element again
    // in its own state and flags it there.
    template <bool CTA>
    __device__ __forceinline__ float warm(volatile float* sh_m0) const {
        float m0 = kFloor;
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const float v = raw_max(buf[k]);
            if (v >= kFloor && v < __int_as_float(0x7f800000)) m0 = fmaxf(m0, v);
        }
        m0 = warp_maxf(m0);
        if (CTA) {
            if ((threadIdx.x & 31) == 0) sh_m0[threadIdx.x >> 5] = m0;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < kWarps; ++w) m0 = fmaxf(m0, sh_m0[w]);
        }
        return m0;
    }
    // The spans that a warp leaves of a row which is to be drawn from: its range in n pieces of `groups` times U steps each, piece k's
    // sum in the lane's sh[k * kFineStride].
    struct Fine {
        float* sh;
        int n, groups;
    };
    // PATH_DRAFT: through draft() only.  FINE: the pieces' sums are in shared memory, relative to the warp's reference.
    template <int PATH, bool FINE = false>
    __device__ __forceinline__ float4 run(float m0, float scale, bool* far = nullptr, const Fine fine = Fine()) {
        const int lane = threadIdx.x & 31;
        DraftState ds; TargetState ts; ArgmaxState as;
        if constexpr (PATH == PATH_DRAFT) ds.init(m0, scale);
        else if constexpr (PATH == PATH_TARGET) ts.init(m0, scale);
        else as.init(m0);
        if constexpr (PATH == PATH_TARGET) {
            if (first_edge || last_edge) ts.template careful<T>(edge(), scale);
            // FINE: ts.z is the present piece's sum, `behind` what lane 1 has of the row's last granule
            float behind = 0.f;
            int piece = 0, left_groups = fine.groups;
            if (FINE && lane == 1) { behind = ts.z; ts.z = 0.f; }
            // steps i .. i+n-1 went into ga, gb
            auto close = [&](f2 ga, f2 gb, int i, int n) {
                const float g = hsum2(add2(ga, gb));
                if (g < kBigSum) {
                    ts.z += g;
                } else {
#pragma unroll 1
                    for (int k = i; k < i + n; ++k) {
                        const float f = ts.template careful<T>(load(k), scale);
                        if (FINE && f != 1.f) {
                            behind *= f;
                            for (int q = 0; q < piece; ++q) fine.sh[q * kFineStride] *= f;
                        }
                    }
                }
            };
            int i = 0;
            for (; i + U <= n_main; i += U) {
                f2 ga = pack2(0.f, 0.f), gb = ga;
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const Raw<T> cur = buf[k];
                    const int nx = i + U + k;
                    if (nx < n_main) buf[k] = load(nx);
                    ts.template add<T>(cur, scale, ga, gb);
                }
                close(ga, gb, i, U);
                if (FINE && --left_groups == 0) {  // (a lane has fine.n * fine.groups whole groups at most)
                    fine.sh[piece * kFineStride] = ts.z;
                    ts.z = 0.f;
                    ++piece;
                    left_groups = fine.groups;
                }
            }
            f2 ga = pack2(0.f, 0.f), gb = ga;
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (i + k < n_main) ts.template add<T>(buf[k], scale, ga, gb);
            close(ga, gb, i, n_main - i);
            if (FINE) {
                const float R = warp_maxf(ts.r), f = ex2f(ts.r - R);
                if (piece < fine.n) fine.sh[piece++ * kFineStride] = ts.z;
                else fine.sh[(fine.n - 1) * kFineStride] += ts.z;
                for (; piece < fine.n; ++piece) fine.sh[piece * kFineStride] = 0.f;
                if (last_edge && lane == 1) fine.sh[min((ng - 1 - a) / (fine.groups * U * 32 * GS), fine.n - 1) * kFineStride] += behind;
                if (f != 1.f)
                    for (int q = 0; q < fine.n; ++q) fine.sh[q * kFineStride] *= f;
                return make_float4(R, 0.f, 0.f, 0.f);
            }
        } else {
            const int shift = meta & 15;
            auto process = [&](const Raw<T>& v, int g) {  // g: granule of the first half
                if constexpr (PATH == PATH_DRAFT) ds.template step<T>(v, scale);
                else as.template step<T>(v, g * E - shift, GS == 2 ? (g + 32) * E - shift : g * E - shift + kVec / 2);
            };
            if (first_edge || last_edge) process(edge(), lane == 0 ? 0 : ng - 1);
            // The lanes' votes on a draft step need all of them: the loop ends with the last step that all lanes have, and one without the
            // last step folds nothing.
            const int n_all = PATH == PATH_DRAFT ? __shfl_sync(0xffffffffu, n_main, 31) : n_main;
            int i = 0;
            // A step's registers are loaded again when it has been folded, not before: a copy of it to fold from is four registers
            // more, and the 48 there are spilled (b256 and b1024 as above 137 / 432 us, this way with pairs of draft steps 134 / 414).
            for (; i + U <= n_all; i += U) {
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    if constexpr (PATH == PATH_DRAFT && U % 2 == 0) {
                        if (k % 2) continue;
                        ds.template step2<T>(buf[k], buf[k + 1], scale);
                        if (i + U + k + 1 < n_main) buf[k + 1] = load(i + U + k + 1);
                    } else {
                        process(buf[k], a + lane + 32 * GS * (i + k));
                    }
                    if (i + U + k < n_main) buf[k] = load(i + U + k);
                }
            }
            const int n_any = PATH == PATH_DRAFT ? __shfl_sync(0xffffffffu, n_main, 0) : n_main;
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (i + k >= n_any) continue;
                if (PATH == PATH_DRAFT && i + k >= n_main) buf[k] = raw_fill<T>(__int_as_float(0xff800000));
                process(buf[k], a + lane + 32 * GS * (i + k));
            }
        }
        float4 part;
        if constexpr (PATH == PATH_DRAFT) {
            part = ds.partial(scale);
            *far = __any_sync(0xffffffffu, ds.far(part, scale));
        }
        else if constexpr (PATH == PATH_TARGET) part = ts.partial();
        else part = as.partial();
        return warp_merge<PATH>(part, scale);
    }
    // a draft row's range [lo, hi)
    __device__ __forceinline__ float4 draft(float m0, float scale, const T* row, int V, int lo, int hi) {
        bool far;
        const float4 part = run<PATH_DRAFT>(m0, scale, &far);
        return far ? draft_far<T>(row, V, lo, hi, scale) : part;
    }
};

// ----------------------------------------------------------------------------------------
// Row epilogue helpers (one warp, double precision; a few dozen values per row)
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ float4 ldcg4(const float4* p) {
    if (!dbg_ok(p, 16, DBG_WS_LOAD)) return make_float4(0.f, 0.f, 0.f, 0.f);
    return __ldcg(p);
}
// a store into the workspace (or a caller's state array) at an index that was computed
#define SPECKV_ST(lvalue, value) do { if (dbg_ok(&(lvalue), sizeof(lvalue), DBG_WS_STORE)) (lvalue) = (value); } while (0)

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Controller (Sec. 4.3, Eq. 1) for one row, executed by a full warp.  The parameters are fetched
// first, all at once (ctl_load), so that their memory latency overlaps whatever comes between
// the load and the evaluation.  Lane k holds hidden unit k's weights, b2[k] and comp[k].
struct CtlRegs {
    float w1[8], w2[8];
    float b1, b2k, compk;
};
__device__ __forceinline__ CtlRegs ctl_load(const KParams& P, int b, int lane) {
    CtlRegs c;
    const bool hid = lane < P.n_hidden;
#pragma unroll
    for (int f = 0; f < 8; ++f) c.w1[f] = (hid && f < P.n_in) ? P.W1[lane * P.n_in + f] : 0.f;
    if (P.layout == 2) {
        // the paper's f(x, gamma): one output head; without hidden units W2 weighs the inputs directly
#pragma unroll
        for (int j = 1; j < 8; ++j) c.w2[j] = 0.f;
        c.w2[0] = (P.n_hidden > 0 ? hid : lane < P.n_in) ? P.W2[lane] : 0.f;
        c.b2k = lane == 0 ? P.b2[0] : 0.f;
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) c.w2[j] = (hid && j < P.n_out) ? P.W2[j * P.n_hidden + lane] : 0.f;
        c.b2k = lane < P.n_out ? P.b2[lane] : 0.f;
    }
    c.b1 = hid ? P.b1[lane] : 0.f;
    c.compk = (P.comp && lane < P.n_comp) ? P.comp[static_cast<long long>(b) * P.n_comp + lane] : 0.f;
    return c;
}
// f4 = Hbar, cbar, Hmax, cmin.  fp32 throughout: 164 multiply-adds on values of order one.  All outputs' reductions run
// together, output by output only the last comparison: five shuffle steps instead of five per output, and a third of the
// code (a row epilogue is one pass over cold instructions; the controller was 2.0 to 3.6 us of it).
__device__ __forceinline__ void ctl_eval(const KParams& P, const CtlRegs& c, const float (&f4)[4],
                                         float* scores_row, int* gamma_next) {
    const int lane = threadIdx.x & 31;
    // inputs x[0..n_in) in the layout's order: four signals (layout 0: three, without Hmax), then the compression features;
    // layout 2 has the candidate gamma as its last input
    const int n_sig = P.layout == 0 ? 3 : 4;
    const int n_x = P.layout == 2 ? P.n_in - 1 : P.n_in;
    float h = c.b1, wg = 0.f, xl = 0.f;  // hidden pre-activation (without gamma); gamma's weight; x[lane]
#pragma unroll
    for (int f = 0; f < 8; ++f) {
        const float cv = __shfl_sync(0xffffffffu, c.compk, (f - n_sig) & 31);
        const float sig = f == 0 ? f4[0] : f == 1 ? f4[1] : f == 2 ? (P.layout == 0 ? f4[3] : f4[2]) : f4[3];
        const float x = f < n_sig ? sig : cv;
        if (f < n_x) h = fmaf(c.w1[f], x, h);
        if (P.layout == 2 && f == n_x) wg = c.w1[f];
        if (f == lane && f < n_x) xl = x;
    }
    float t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float g = static_cast<float>(P.gch[j]);
        if (P.layout == 2 && P.n_hidden == 0) {  // Sec. 4.3 as printed, linear
            t[j] = lane < n_x ? c.w2[0] * xl : (lane == n_x ? c.w2[0] * g : 0.f);
        } else {
            const float hj = P.layout == 2 ? fmaf(wg, g, h) : h;
            t[j] = (lane < P.n_hidden && hj > 0.f) ? (P.layout == 2 ? c.w2[0] : c.w2[j]) * hj : 0.f;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int j = 0; j < 8; ++j) t[j] += __shfl_xor_sync(0xffffffffu, t[j], o);
    }
    // lane j: output j
    float v = t[0];
#pragma unroll
    for (int j = 1; j < 8; ++j) v = lane == j ? t[j] : v;
    const float b2 = P.layout == 2 ? __shfl_sync(0xffffffffu, c.b2k, 0) : c.b2k;
    const int g = P.gch[lane & 7];
    const float o = v + b2;
    const float e = (P.transform == 0) ? fmaf(o, static_cast<float>(g), 1.f) : o;
    if (scores_row && lane < P.n_out) scores_row[lane] = e;
    // the lowest index with the largest score; a NaN never wins against what stands before it
    float best = __shfl_sync(0xffffffffu, e, 0);
    int best_j = 0;
#pragma unroll
    for (int j = 1; j < 8; ++j) {
        const float ej = __shfl_sync(0xffffffffu, e, j);
        if (j < P.n_out && ej > best) { best = ej; best_j = j; }
    }
    if (gamma_next && lane == 0) *gamma_next = P.gch[best_j];
}

// log2 of a positive finite number in double: it enters the normalisers of p and q, and the residual
// max(0, p - q) sees the difference of their errors magnified by 1 / (its own mass); a few dozen calls
// per batch row, so the cost does not show
__device__ __forceinline__ double log2_split(double z) { return log2(z); }

// End of a row epilogue (whole warp): everything the warp wrote for batch row b becomes visible, then the row takes a slot
// of the draw queue: rows with a residual draw from the front in the order in which they complete, all others from the
// back, so that every slot is filled once all rows are done.  Group g of the CTAs that draw waits for slot g, not for a
// batch row: it starts on the first finished row whatever its number, and the groups that find nothing to draw come last
// (by batch row, 1,024 rows of which a third draw spent 9 us of all CTA slots on groups with nothing to do).
constexpr int kSlotDone = 1 << 30, kSlotTimeout = 1 << 31;  // bits 0-23: batch row, 24: a residual draw, 25-28: stop position
__device__ __forceinline__ int row_done_slot(const KParams& P, int mode) {  // whole warp; lane 0 has the answer
    if (!P.rdone || (threadIdx.x & 31) != 0) return 0;
    return mode == RS_RESIDUAL ? atomicAdd(P.q_front, 1) : P.B - 1 - atomicAdd(P.q_back, 1);
}
__device__ __forceinline__ void row_done_signal(const KParams& P, int b, int slot, int mode, int n) {  // (direct grid: slot b)
    if (!P.rdone) return;
    __threadfence();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        const int old = atomicOr(P.rdone + slot, kSlotDone | b | (mode == RS_RESIDUAL ? 1 << 24 | n << 25 : 0));
        // a group whose bounded wait ran out before this point left its mark here: the row's fresh
        // token will never be drawn, and the status written above must say so
        if ((old & kSlotTimeout) && (!P.direct || mode == RS_RESIDUAL)) {
            if (P.status) atomicOr(P.status + b, 16);
            if (P.direct) P.out_tok[static_cast<long long>(b) * (P.G + 1) + n] = -1;
        }
    }
}

// A row's record as the drawing CTAs of a direct grid wait for it: two 16-byte words, each stored at once, each of which tells
// whether it has been stored (prep_direct_kernel leaves all bits set; neither a mode nor a normaliser looks like that).  No
// fence and no counter between the decision and the draw: with them (a slot of the queue taken, the record, a fence, the flag)
// the drawing CTAs went on 2 us later.
__device__ __forceinline__ void row_info_publish(RowInfo* p, const RowInfo& ri) {
    if (!dbg_ok(p, sizeof(RowInfo), DBG_WS_STORE)) return;
    asm volatile("{ .reg .b128 v; .reg .b64 lo, hi; mov.b64 lo, {%1, %2}; mov.b64 hi, {%3, %4}; mov.b128 v, {lo, hi}; st.relaxed.gpu.global.b128 [%0], v; }"
                 :: "l"(p), "r"(ri.mode), "r"(ri.n), "r"(__float_as_int(ri.u2)), "r"(__float_as_int(ri.scale)) : "memory");
    asm volatile("{ .reg .b128 v; mov.b128 v, {%1, %2}; st.relaxed.gpu.global.b128 [%0], v; }"
                 :: "l"(reinterpret_cast<char*>(p) + 16), "l"(__double_as_longlong(ri.lse2_p)), "l"(__double_as_longlong(ri.lse2_q)) : "memory");
}
// A span's sum, as one word that tells whether it has been stored.
__device__ __forceinline__ void span_publish(double2* p, double w) {
    if (!dbg_ok(p, sizeof(double2), DBG_WS_STORE)) return;
    asm volatile("{ .reg .b128 v; mov.b128 v, {%1, %2}; st.relaxed.gpu.global.b128 [%0], v; }" :: "l"(p), "l"(__double_as_longlong(w)), "l"(0ll) : "memory");
}
__device__ __forceinline__ bool span_read(const double2* p, double* w) {
    long long a = 0, b = 0;
    if (dbg_ok(p, sizeof(double2), DBG_WS_LOAD))
        asm volatile("{ .reg .b128 v; ld.relaxed.gpu.global.b128 v, [%2]; mov.b128 {%0, %1}, v; }" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    *w = __longlong_as_double(a);
    return b == 0;
}
// One thread; false when the bound ran out.
__device__ __forceinline__ bool row_info_wait(const RowInfo* p, int limit, RowInfo* out) {
    for (int it = 0; it < limit; ++it) {
        long long a, b, c, d;
        asm volatile("{ .reg .b128 v; ld.relaxed.gpu.global.b128 v, [%2]; mov.b128 {%0, %1}, v; }" : "=l"(a), "=l"(b) : "l"(p) : "memory");
        asm volatile("{ .reg .b128 v; ld.relaxed.gpu.global.b128 v, [%2]; mov.b128 {%0, %1}, v; }" : "=l"(c), "=l"(d) : "l"(reinterpret_cast<const char*>(p) + 16) : "memory");
        if (static_cast<int>(a) != -1 && c != -1) {
            out->mode = static_cast<int>(a);
            out->n = static_cast<int>(a >> 32);
            out->u2 = __int_as_float(static_cast<int>(b));
            out->scale = __int_as_float(static_cast<int>(b >> 32));
            out->lse2_p = __longlong_as_double(c);
            out->lse2_q = __longlong_as_double(d);
            return true;
        }
        __nanosleep(it < 256 ? 100 : 1000);
    }
    return false;
}

// Bounded wait for a slot of the draw queue (one thread polls).  The slot's value, 0 when the bound ran out.
__device__ __forceinline__ int row_done_wait(const int* flag, int limit) {
    for (int it = 0; it < limit; ++it) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v & kSlotDone) return v;
        __nanosleep(it < 64 ? 100 : 1000);
    }
    return 0;
}

// What one lane of a row's epilogue learns about its position (lane i: draft position i, target position i).
struct RowDecide {
    int x;            // draft token (-1 where the lane has none)
    float u_res;      // second uniform of the position
    float Hi, ci;     // entropy (nats) and confidence of the draft distribution
    double lse2_q, lse2_p;  // log2-normalisers of draft and target
    int amax;         // greedy rows: argmax of the target row
    bool dbad, tbad;  // non-finite draft row / target row at this position
    bool badtok, accept;
};

// The per-position part of a row epilogue, by the warps of a CTA: a group of 32 lanes (16 where a logit row has at most 16 partials)
// decides one position, the lower half gathering the draft row's partials and the upper half the target row's, so that
// they cost one memory round trip and a few shuffle steps instead of a chain of them, and one double-precision log2 serves
// draft row, target row and uniform.
// Latency-bound: one batch row in 15 slices (fp32, V = 32,000, gamma 4), with a lane per position the prefix and the row
// epilogue each walked a chain of 11 dependent round trips and the step took 45.1 us; this way 23.0 us.  256 rows of
// bf16, V = 128,256: 150.5 -> 145.6 us (the chain is also the end of a large step).  The test of a position and the row
// epilogue call this one compiled body, so that both reach the same bits.
// Decides positions first, first + 1 (16 lanes each) or first alone.  A logit row has nsplit partials: its slices', adjacent in
// P.part, or (part_stride) the states of as many vocabulary shards, part_stride apart.
template <typename T>
__device__ __noinline__ void decide_positions(const KParams& P, int b, int gam, bool greedy, float scale, int first, int n_pos,
                                              RowDecide* out) {
    const int lane = threadIdx.x & 31, n = P.nsplit;
    const int half = n <= 16 ? 8 : 16;  // lanes per logit row, at most two partials each
    const int k = lane & (half - 1), lead = lane & ~(2 * half - 1);  // lane within the row, first lane of the group
    const bool tgt_half = (lane & half) != 0;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const int i = first + (lane >= 2 * half ? 1 : 0);
    const bool in = i < n_pos;
    const bool dr_on = in && i < gam, tok_on = dr_on && verify;

    // ---- one round trip ----
    const bool on = tgt_half ? in && verify : dr_on;
    const long long jrow = static_cast<long long>(b) * P.J + (tgt_half || !verify ? i : P.G + 1 + i);
    const long long ps = P.part_stride > 0 ? P.part_stride : 1;
    const float4* src = P.part + (P.part_stride > 0 ? jrow : jrow * n);
    const float4 none = tgt_half && greedy ? make_float4(kFloor, __int_as_float(0x7fffffff), 0.f, 0.f)
                                           : make_float4(tgt_half ? -3.0e38f : kFloor, 0.f, 0.f, 0.f);
    float4 a = none, a2 = none;
    if (on && k < n) a = ldcg4(src + k * ps);
    if (on && k + half < n) a2 = ldcg4(src + (k + half) * ps);
    int x = -1;
    float u_acc = 0.f, u_res = 0.f;
    float2 tl = make_float2(0.f, 0.f);
    {
        const long long at = static_cast<long long>(b) * P.G + i;
        const long long urow = (static_cast<long long>(b) * (P.G + 1) + i) * 2;
        if (tok_on) {
            x = P.tok[at];
            u_acc = P.u[urow];
            // left by the sweep CTA of the draft position; with shards, in the table of the one whose slice holds the token
            if (P.shard_width > 0) {
                const long long shard = x > 0 ? min(x / P.shard_width, P.n_shards - 1) : 0;
                if (!greedy) tl = __ldcg(P.tokl + at + shard * P.tokl_stride);
            } else if (!greedy) {
                tl = __ldcg(P.tokl + at);  // without waiting for x
            }
        }
        if (in && verify) u_res = P.u[urow + 1];
    }

    int amax = -1;
    bool tbad = false;
    if (greedy && verify) {  // uniform across the warp; the draft lanes go along and are not looked at
        float4 g = merge_argmax(a, a2);
        for (int m = half >> 1; m > 0; m >>= 1) g = merge_argmax(g, shfl_xor4(g, m));
        amax = __shfl_sync(0xffffffffu, __float_as_int(g.y), lead + half);
        const float best = __shfl_sync(0xffffffffu, g.x, lead + half), bad = __shfl_sync(0xffffffffu, g.z, lead + half);
        tbad = bad != 0.f || amax == 0x7fffffff || !(best > kFloor);
    }
    // draft partial: (m, cnt, Zx, S); target partial (r, Z): both as (reference, cnt, Z, S) with the reference in log2 units
    // for the target lanes
    const float sc = tgt_half ? 1.f : scale;
    if (tgt_half) {
        a.z = a.y; a.y = 0.f; a.w = 0.f;
        a2.z = a2.y; a2.y = 0.f; a2.w = 0.f;
    }
    float M = fmaxf(a.x, a2.x);
    for (int m = half >> 1; m > 0; m >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, m));
    float cnt = 0.f, Z = 0.f, S = 0.f;
    auto add = [&](const float4& v) {
        const float dm = v.x - M, f = ex2f(dm * sc), za = v.y + v.z;
        const bool top = v.x == M;  // below the maximum a count joins the scaled sum
        cnt += top ? v.y : 0.f;
        Z += top ? v.z : za * f;
        S += top ? v.w : fmaf(dm, za, v.w) * f;
    };
    add(a);
    add(a2);
    for (int m = half >> 1; m > 0; m >>= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, m);
        Z += __shfl_xor_sync(0xffffffffu, Z, m);
        S += __shfl_xor_sync(0xffffffffu, S, m);
    }
    // the group's first lane: draft normaliser, first target lane: target normaliser, a lane between them: accept uniform
    const int u_lane = lead + (half >> 1);
    const double arg = lane == u_lane ? static_cast<double>(u_acc) : static_cast<double>(cnt) + static_cast<double>(Z);
    const double l2 = log2_split(arg);
    const double l2_p = __shfl_sync(0xffffffffu, l2, lead + half), l2_u = __shfl_sync(0xffffffffu, l2, u_lane);
    const float Rp = __shfl_sync(0xffffffffu, M, lead + half), Zp = __shfl_sync(0xffffffffu, Z, lead + half);
    if (lane != lead || !in) return;

    float Hi = 0.f, ci = 0.f;
    double lse2_q = 0.0, lse2_p = 0.0;
    bool dbad = false, accept = true;
    if (dr_on) {
        const float Zall = cnt + Z;
        if (!(cnt >= 1.f) || !(Zall < 3e38f) || !(M > kFloor)) {
            dbad = true;
        } else {
            const float lnZ = (cnt == 1.f) ? log1pf(Z) : logf(cnt) + log1pf(Z / cnt);
            const float rZ = 1.f / Zall;
            Hi = fmaxf(lnZ - static_cast<float>(kLn2) * scale * S * rZ, 0.f);
            ci = rZ;
            lse2_q = static_cast<double>(M) * static_cast<double>(scale) + l2;
        }
    }
    if (verify && !greedy) {
        if (!(Zp > 0.f) || !(Zp < 3e38f)) tbad = true;
        else lse2_p = static_cast<double>(Rp) + l2_p;
    }
    const bool badtok = tok_on && (x < 0 || x >= P.V);
    if (tok_on && !dbad && !badtok && !tbad) {
        if (greedy) {
            accept = (x == amax);
        } else {
            const double sd = static_cast<double>(scale);
            const double lq = static_cast<double>(tl.x) * sd - lse2_q, lp = static_cast<double>(tl.y) * sd - lse2_p;
            accept = (l2_u + lq) < lp;  // u * q(x) < p(x); u = 0: log2 is -inf
        }
    }
    RowDecide& o = out[i];
    o.x = x; o.u_res = u_res; o.Hi = Hi; o.ci = ci; o.lse2_q = lse2_q; o.lse2_p = lse2_p; o.amax = amax;
    o.dbad = dbad; o.tbad = tbad; o.badtok = badtok; o.accept = accept;
}
// Positions 0..n_pos-1 by all warps of the CTA; the caller synchronises.  Warp 0 has the fewest.
template <typename T>
__device__ __forceinline__ void decide_all(const KParams& P, int b, int gam, bool greedy, float scale, int n_pos, RowDecide* pos) {
    const int per = P.nsplit <= 16 ? 2 : 1, nw = static_cast<int>(blockDim.x >> 5);
    for (int i = (nw - 1 - static_cast<int>(threadIdx.x >> 5)) * per; i < n_pos; i += nw * per)
        decide_positions<T>(P, b, gam, greedy, scale, i, n_pos, pos);
}

// The acceptance test of one position (one warp), run when the partials of its draft and target row are in, while the rest of the
// batch row is still being swept.  A position that ends the walk is noted, so that CTAs which have not started yet can leave
// the target rows behind it unread.
template <typename T>
__device__ __noinline__ void test_position(const KParams& P, int b, int gam, bool greedy, float scale, int i, RowDecide* pos) {
    decide_positions<T>(P, b, gam, greedy, scale, i, i + 1, pos);
    __syncwarp();
    const RowDecide& d = pos[i];
    if ((threadIdx.x & 31) == 0 && (d.tbad || d.dbad || d.badtok || !d.accept)) atomicMin(P.early + b, i + 1);
}

// log2(e) / T, the factor of every exponent of a row (greedy rows: T = 1).
__device__ __forceinline__ float row_scale(float Tf) {
    return static_cast<float>(kLog2e / static_cast<double>(Tf == 0.f ? 1.f : Tf));
}
// Status bits a row's gamma and temperature give by themselves.
__device__ __forceinline__ int row_status0(const KParams& P, int gam, float Tf) {
    return (gam < 1 || gam > P.G ? 1 : 0) | (!(Tf >= 0.f) || Tf == __int_as_float(0x7f800000) ? 8 : 0);
}

// The walk over the positions (one warp, lane i holding position i's decision): where it ends, and the row's status.
//
// The positions are walked in order; the walk ends at the first one whose target row is non-finite
// (which flags the row), whose draft token is out of range, or whose token is rejected.  Target rows
// behind that position are not part of the step (Sec. 3.1 discards what follows the first mismatch):
// whatever they hold flags nothing.  A non-finite draft row flags the row wherever it is.
__device__ __forceinline__ int row_walk(const KParams& P, int gam, float Tf, const RowDecide& dec, int* stop_at) {
    const int lane = threadIdx.x & 31;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    int status = row_status0(P, gam, Tf);
    const bool tg_on = !status && verify && lane <= gam;
    const unsigned stop = __ballot_sync(0xffffffffu, tg_on && (dec.tbad || (lane < gam && (dec.badtok || !dec.accept))));
    const int first = stop ? (__ffs(stop) - 1) : gam;
    const bool tbad_first = __shfl_sync(0xffffffffu, dec.tbad ? 1 : 0, first & 31) != 0;
    const bool any_dbad = __any_sync(0xffffffffu, dec.dbad), any_badtok = __any_sync(0xffffffffu, dec.badtok);
    if (status == 0) status = (any_dbad || (verify && tbad_first) ? 4 : 0) | (any_badtok ? 2 : 0);
    *stop_at = (status == 0 && verify) ? first : 0;
    return status;
}

// What the walk decides (one warp): status, accepted count, tokens except a drawn one, the record a draw needs and the
// row's completion flag.  own_bonus: a bonus token is drawn by the caller (from the sweep's spans), not by the CTAs
// that wait for the flag.
__device__ __noinline__ void finish_verify(const KParams& P, int b, int gam, float Tf, float scale, const RowDecide& dec, bool own_bonus) {
    const int lane = threadIdx.x & 31;
    const int G = P.G;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const bool greedy = (Tf == 0.f);
    int n;
    const int status = row_walk(P, gam, Tf, dec, &n);
    const int rs_mode = (verify && status == 0 && !greedy) ? (n < gam ? RS_RESIDUAL : RS_BONUS) : RS_NONE;
    const bool direct = P.direct != 0;
    const int slot = direct ? b : row_done_slot(P, rs_mode);  // travels while the outputs are written
    if (verify) {
        // fresh token: known here for greedy rows, drawn by the resample step otherwise
        const int amax_n = __shfl_sync(0xffffffffu, dec.amax, n);
        const double lp_n = __shfl_sync(0xffffffffu, dec.lse2_p, n);
        const double lq_n = __shfl_sync(0xffffffffu, dec.lse2_q, n < gam ? n : 0);
        const float u2_n = __shfl_sync(0xffffffffu, dec.u_res, n);
        RowInfo ri;
        ri.mode = rs_mode;
        ri.n = n;
        ri.u2 = (status == 0 && !greedy) ? u2_n : 0.f;
        ri.scale = scale;
        ri.lse2_p = lp_n;
        ri.lse2_q = lq_n;
        if (direct && lane == 0) row_info_publish(P.info + b, ri);
        // (a direct grid's draw may be done before this: its place is left alone)
        if (lane <= G && !(own_bonus && rs_mode == RS_BONUS && lane == n) && !(direct && rs_mode == RS_RESIDUAL && lane == n)) {
            int v = -1;
            if (status == 0) {
                if (lane < n) v = dec.x;
                else if (lane == n && greedy) v = amax_n;
            }
            P.out_tok[static_cast<long long>(b) * (G + 1) + lane] = v;
        }
        if (lane == 0) {
            P.n_acc[b] = n;
            if (!direct) SPECKV_ST(P.info[b], ri);
        }
    }
    if (P.status && lane == 0) P.status[b] = status;
    row_done_signal(P, b, slot, rs_mode, n);
}

// The signals and the controller's outputs (one warp); ctl: the controller's parameters, fetched beforehand.
__device__ __noinline__ void finish_signals(const KParams& P, int b, int gam, float Tf, const RowDecide& dec, const CtlRegs& ctl) {
    const int lane = threadIdx.x & 31;
    const int G = P.G;
    int n;
    const int status = row_walk(P, gam, Tf, dec, &n);
    const float in_bits = P.bits ? static_cast<float>(kLog2e) : 1.f;
    const float Hout = (status == 0 && lane < gam) ? dec.Hi * in_bits : 0.f;
    const float Cout = (status == 0 && lane < gam) ? dec.ci : 0.f;
    float f4[4] = {Hout, Cout, Hout, (status == 0 && lane < gam) ? -Cout : -2.f};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        f4[0] += __shfl_xor_sync(0xffffffffu, f4[0], o);
        f4[1] += __shfl_xor_sync(0xffffffffu, f4[1], o);
        f4[2] = fmaxf(f4[2], __shfl_xor_sync(0xffffffffu, f4[2], o));
        f4[3] = fmaxf(f4[3], __shfl_xor_sync(0xffffffffu, f4[3], o));
    }
    f4[0] = status == 0 ? f4[0] / static_cast<float>(gam) : 0.f;
    f4[1] = status == 0 ? f4[1] / static_cast<float>(gam) : 0.f;
    f4[3] = status == 0 ? -f4[3] : 0.f;
    if (lane < G) {
        if (P.H) P.H[static_cast<long long>(b) * G + lane] = Hout;
        if (P.C) P.C[static_cast<long long>(b) * G + lane] = Cout;
    }
    if (P.feat && lane < 4)
        P.feat[static_cast<long long>(b) * 4 + lane] = lane == 0 ? f4[0] : lane == 1 ? f4[1] : lane == 2 ? f4[2] : f4[3];
    if (P.mode & MODE_MLP) {
        if (status == 0) {
            ctl_eval(P, ctl, f4, P.scores ? P.scores + static_cast<long long>(b) * P.n_out : nullptr, P.gamma_next + b);
        } else {
            if (P.scores && lane < P.n_out) P.scores[static_cast<long long>(b) * P.n_out + lane] = 0.f;
            if (lane == 0) P.gamma_next[b] = 0;
        }
    }
}

// Epilogue of a vocabulary shard's sweep (one warp per batch row): lane i merges this shard's nd
// partials of draft position i and nt partials of target position i (the counts may differ from lane
// to lane) and writes the two merged states; the row epilogue proper runs later on the states of all
// shards.  An argmax index becomes a global vocabulary index.
__device__ __noinline__ void export_epilogue(const KParams& P, int b, int gam, float Tf, const float4* pd, int nd,
                                             const float4* pt, int nt) {
    const int lane = threadIdx.x & 31;
    const int G = P.G;
    const bool ok = (gam >= 1 && gam <= G) && (Tf >= 0.f) && (Tf != __int_as_float(0x7f800000));
    const bool greedy = (Tf == 0.f);
    const float scale = static_cast<float>(kLog2e / static_cast<double>(greedy ? 1.f : Tf));
    float4* out = P.state + static_cast<long long>(b) * P.J;
    if (lane < G) {
        float4 ad = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok && lane < gam && nd > 0) {
            ad = ldcg4(pd);
            for (int k = 1; k < nd; ++k) ad = merge_draft(ad, ldcg4(pd + k), scale);
        }
        SPECKV_ST(out[G + 1 + lane], ad);
    }
    if (lane <= G) {
        float4 at = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok && lane <= gam && nt > 0) {
            at = ldcg4(pt);
            for (int k = 1; k < nt; ++k) at = greedy ? merge_argmax(at, ldcg4(pt + k)) : merge_target(at, ldcg4(pt + k));
            if (greedy) {
                const int idx = __float_as_int(at.y);
                if (idx != 0x7fffffff) at.y = __int_as_float(idx + P.v_begin);
            }
        }
        SPECKV_ST(out[lane], at);
    }
}

// ----------------------------------------------------------------------------------------
// Stand-alone controller: one warp per row.
// ----------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) select_gamma_kernel(const __grid_constant__ KParams P, const float* feat_in) {
    wait_for_predecessors();
    dependents_may_start();
    const int b = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (b >= P.B) return;
    float f4[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) f4[k] = feat_in[static_cast<long long>(b) * 4 + k];
    const CtlRegs ctl = ctl_load(P, b, threadIdx.x & 31);
    ctl_eval(P, ctl, f4, P.scores ? P.scores + static_cast<long long>(b) * P.n_out : nullptr, P.gamma_next + b);
}

}  // namespace speckv
