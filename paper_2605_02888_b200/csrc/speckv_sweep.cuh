// The register-staged sweep: one CTA per slice of a logit row, row epilogues by the CTA that completes a row, draws of
// rejected rows by further CTAs of the same grid.
#pragma once

#include "speckv_draw.cuh"

namespace speckv {

// Row epilogue of the sliced sweep: a whole CTA.  A warp per position decides; then, side by side, warp 0 walks the positions
// and raises the row's flag, warp 1 writes the signals and runs the controller, and warps 2.. draw a bonus token from the sums
// that the sweep left of the target row at position gamma.  Latency-bound (cold instructions and dependent round trips): one
// after the other in one warp this took 6.6 us behind the last partial of a lone row, this way 4 us less.
constexpr int kDrawWarp0 = 2;
template <typename T>
__device__ __noinline__ void row_epilogue_cta(const KParams& P, int b, int gam, float Tf, float scale, RowDecide* pos, double* sh_sum,
                                              DrawSrc* sh_src) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const int n_pos = row_status0(P, gam, Tf) ? 0 : verify ? gam + 1 : gam;
    // the parameters travel while the positions are decided; warps 0 and 1 take the last turns
    CtlRegs ctl;
    if (warp == 1 && (P.mode & MODE_MLP) && n_pos) ctl = ctl_load(P, b, lane);
    decide_all<T>(P, b, gam, Tf == 0.f, scale, n_pos, pos);
    __syncthreads();
    if (warp >= kDrawWarp0) {
        // a bonus draw: every position accepted, nothing flagged (a sharded step draws in calls of its own)
        if (!P.spans || !n_pos || Tf == 0.f) return;
        bool ends = false;
        if (lane < n_pos) ends = pos[lane].dbad || pos[lane].tbad || pos[lane].badtok || !pos[lane].accept;
        if (__any_sync(0xffffffffu, ends)) return;
        const T* row = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(gam) * P.tsp;
        const int n = P.n_spans;
        const int tok = draw_from_spans<T>(row, P.V, scale, P.spans + static_cast<long long>(b) * n, n, P.per_warp, pos[gam].u_res,
                                           warp - kDrawWarp0, kWarps - kDrawWarp0, 1, sh_sum, sh_src);
        if (tok != kNotMine && lane == 0) P.out_tok[static_cast<long long>(b) * (P.G + 1) + gam] = max(tok, 0);
        return;
    }
    RowDecide dec;
    dec.x = -1; dec.u_res = 0.f; dec.Hi = dec.ci = 0.f; dec.lse2_q = dec.lse2_p = 0.0; dec.amax = -1;
    dec.dbad = dec.tbad = dec.badtok = false; dec.accept = true;
    if (lane < n_pos) dec = pos[lane];
    if (warp == 0) finish_verify(P, b, gam, Tf, scale, dec, P.spans != nullptr);
    else if (P.mode & MODE_SIGNALS) finish_signals(P, b, gam, Tf, dec, ctl);
}

// ----------------------------------------------------------------------------------------
// What the sweep has to know before it starts: cleared counters and the list of the logit rows to sweep in grid order.  The
// grid has CTAs for every position up to gamma_max, and gamma lives in device memory; with the list the CTAs that have work
// come first and the surplus goes to the draws.  (One CTA per stored position, leaving again when gamma said so, cost
// 1.8 us of a CTA slot each: 20 us of a step of 1,024 rows that use half of their positions.)
// Grid: a segment of batch rows per CTA; every CTA reads all rows' gamma and temperature for the prefix.
// ----------------------------------------------------------------------------------------
enum : int { ENTRY_FLAGGED = 256 };  // entry: (batch row, row index j | generation << 6 | ENTRY_FLAGGED | gamma << 16)
__global__ void __launch_bounds__(kThreads) prep_kernel(const __grid_constant__ KParams P, int seg) {
    // rows of each gamma (and, last, flagged ones) in front of this CTA's segment and in all
    constexpr int kFlagged = kMaxGamma + 1, kBins = kMaxGamma + 2;
    __shared__ int sh[2][kBins];
    if (threadIdx.x < 2 * kBins) sh[threadIdx.x / kBins][threadIdx.x % kBins] = 0;
    __syncthreads();
    wait_for_predecessors();
    dependents_may_start();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b0 = blockIdx.x * seg, b1 = min(P.B, b0 + seg);
    for (int b = b0 + threadIdx.x; b < b1; b += kThreads) {
        P.tick1[b] = 0;
        if (P.rdone) { P.tick2[b] = 0; P.rdone[b] = 0; }
        if (P.early) { P.tick_pos[b] = 0; P.early[b] = 0x7fffffff; }
    }
    for (int b = threadIdx.x; b < P.B; b += kThreads) {
        const int gam = P.gamma ? P.gamma[b] : P.G;
        const int bin = row_status0(P, gam, P.temp ? P.temp[b] : P.temp_scalar) ? kFlagged : gam;
        atomicAdd(&sh[1][bin], 1);
        if (b < b0) atomicAdd(&sh[0][bin], 1);
    }
    __syncthreads();
    if (warp != 0) return;
    // lane p: rows that have a draft row at position p - 1, that is a target row at position p (gamma >= p)
    int before = lane >= 1 && lane <= kMaxGamma ? sh[0][lane] : 0, total = lane >= 1 && lane <= kMaxGamma ? sh[1][lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_down_sync(0xffffffffu, before, o), y = __shfl_down_sync(0xffffffffu, total, o);
        if (lane + o < 32) { before += x; total += y; }
    }
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    // First generation: position 0 of every row (one entry for a flagged one); second: the other draft rows, batch row by batch row;
    // third: the other target rows, position by position or batch row by batch row.
    const int ok_before = __shfl_sync(0xffffffffu, before, 1), ok_total = __shfl_sync(0xffffffffu, total, 1);
    const int per0 = verify ? 2 : 1;
    int at_a = per0 * ok_before + sh[0][kFlagged];
    const int n_a = per0 * ok_total + sh[1][kFlagged];
    int at_b = n_a, n_b = 0, at_r = ok_before;
    for (int p = 2; p <= P.G; ++p) {
        at_b += __shfl_sync(0xffffffffu, before, p);
        at_r += __shfl_sync(0xffffffffu, before, p);
        n_b += __shfl_sync(0xffffffffu, total, p);
    }
    int scan = lane >= 1 ? total : 0;  // rows of the third generation in front of position `lane`
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, scan, o);
        if (lane >= o) scan += x;
    }
    int at_c = n_a + n_b + scan - total + before;  // lane p: where the segment's next row of position p goes
    at_r += n_a + n_b;  // rows_major: where the segment's next row's entries of the third generation go
    const int n_c = verify ? __shfl_sync(0xffffffffu, scan, 31) : 0;
    if (blockIdx.x == 0 && lane == 0) {
        *P.n_list = n_a + n_b + n_c;
        *P.q_front = 0;
        *P.q_back = 0;
    }
    const unsigned below = (1u << lane) - 1;
    const int jd = verify ? P.G + 1 : 0;  // row index of draft position 0
    for (int r0 = b0; r0 < b1; r0 += 32) {
        const int b = r0 + lane;
        int gam = 0;
        bool flagged = false;
        if (b < b1) {
            gam = P.gamma ? P.gamma[b] : P.G;
            flagged = row_status0(P, gam, P.temp ? P.temp[b] : P.temp_scalar) != 0;
            if (flagged) gam = 0;
        }
        auto put = [&](int i, int j, int gen) { SPECKV_ST(P.list[i], make_int2(b, j | gen << 6 | (gam & 31) << 16)); };
        const unsigned ok = __ballot_sync(0xffffffffu, gam > 0), bad = __ballot_sync(0xffffffffu, flagged);
        const int a = at_a + per0 * __popc(ok & below) + __popc(bad & below);
        if (flagged) SPECKV_ST(P.list[a], make_int2(b, ENTRY_FLAGGED));
        if (gam > 0) {
            put(a, jd, 0);
            if (verify) put(a + 1, 0, 0);
        }
        at_a += per0 * __popc(ok) + __popc(bad);
        int more = max(gam - 1, 0), incl = more;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        for (int p = 1; p < gam; ++p) put(at_b + incl - more + p - 1, jd + p, 1);
        at_b += __shfl_sync(0xffffffffu, incl, 31);
        if (!verify) continue;
        if (P.rows_major) {
            int all = gam;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, all, o);
                if (lane >= o) all += x;
            }
            for (int p = 1; p <= gam; ++p) put(at_r + all - gam + p - 1, p, 2);
            at_r += __shfl_sync(0xffffffffu, all, 31);
            continue;
        }
        for (int p = 1; p <= P.G; ++p) {
            const unsigned has = __ballot_sync(0xffffffffu, gam >= p);
            const int c = __shfl_sync(0xffffffffu, at_c, p);
            if (gam >= p) put(c + __popc(has & below), p, 2);
            if (lane == p) at_c += __popc(has);
        }
    }
}

// Small batches are latency-bound: 42 MB stream in 7 us, and the step around them took 33 us.  A direct grid (choose_direct() in
// speckv.cu) takes from that chain what is not work: its CTAs ask for their first logits 2.5 us earlier, since they need no list, and
// a row's draw starts and ends on words that it waits for (direct_draw).  Step of 16 bf16 rows, V = 128,256, 30.7 -> 25.2 us; of 64,
// V = 32,000, 27.5 -> 24.4; of 37, V = 50,257, 27.1 -> 22.9; of one fp32 row, V = 32,000, 13.4 -> 11.1; signals of 128 bf16 rows,
// V = 128,256, 48.7 -> 45.9.
//
// A direct grid needs cleared counters, empty records and empty sums, and nothing of that before its CTAs have folded their slices:
// this kernel lets them start at once, and they wait for its end behind their first loads.
__global__ void __launch_bounds__(kThreads) prep_direct_kernel(const __grid_constant__ KParams P) {
    wait_for_predecessors();
    dependents_may_start();
    const int k = blockIdx.x * kThreads + threadIdx.x;
    if (k < P.B) {
        P.tick1[k] = 0;
        if (P.rdone) {
            P.rdone[k] = 0;
            int4* info = reinterpret_cast<int4*>(P.info + k);
            info[0] = info[1] = make_int4(-1, -1, -1, -1);
        }
    }
    const int n = P.R * kWarps;
    if (P.rdone && k < P.B * n)
        SPECKV_ST(reinterpret_cast<int4*>(P.dsum)[k / n * kDirectSums + k % n], make_int4(-1, -1, -1, -1));
}
// What CTA `entry` of a direct grid sweeps, by the whole CTA: the batch rows' logit rows follow one another (a flagged batch row has
// one entry), targets in front of drafts.  prep_direct_kernel has waited for everything in front of it before it let this kernel
// start, so gamma and the temperatures are complete in L2 although this kernel has not waited yet.  Returns the number of entries.
struct DirectEntry { int2 entry; float temp; };
constexpr int kDirectMostB = kThreads;
__device__ __forceinline__ int direct_entry(const KParams& P, int i, DirectEntry* sh, int* sh_scan) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = threadIdx.x;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    int cnt = 0, gam = 0;
    float Tf = 0.f;
    bool flagged = false;
    if (b < P.B) {
        gam = P.gamma ? __ldcg(P.gamma + b) : P.G;
        Tf = P.temp ? __ldcg(P.temp + b) : P.temp_scalar;
        flagged = row_status0(P, gam, Tf) != 0;
        cnt = flagged ? 1 : verify ? 2 * gam + 1 : gam;
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) sh_scan[warp] = incl;
    __syncthreads();
    int at = incl - cnt, total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const int v = sh_scan[w];
        at += w < warp ? v : 0;
        total += v;
    }
    const int q = i - at;
    if (q >= 0 && q < cnt) {
        const int j = !verify || q <= gam ? q : P.G + 1 + q - (gam + 1);
        sh->entry = make_int2(b, flagged ? ENTRY_FLAGGED : (j | 1 << 6 | (gam & 31) << 16));
        sh->temp = Tf;
    }
    __syncthreads();
    return total;
}

// ----------------------------------------------------------------------------------------
// Sweep kernel.  CTA i sweeps slice i % nsplit of the logit row in list entry i / nsplit (direct grid: of the i / nsplit-th logit row
// in use).  With verification the
// grid carries more CTAs behind them that draw the fresh tokens of rejected rows in the same launch:
// CTAs start in index order, so these start exactly when the sweep runs out of slices, wait (with
// a bound) for a row of the draw queue and fill the SMs that the sweep's last CTAs
// leave one by one.  A second launch, even a programmatic dependent one, starts microseconds
// after the last sweep CTA has started and leaves most of the drain unused.
// Bound by memory: a CTA streams its 256 KB in 22 us beside 4 others per SM, 6.3 TB/s over the chip while about 530 of the
// 740 resident CTAs stream; the others are starting (2.8 us) or merging and taking tickets (3 us).  It is the one sweep for
// all types and all rows but short ones (batch_row_kernel): a persistent ring of bulk copies, which fp32 batches of 384 to 1,024 rows took before, streamed at
// 6.7 TB/s but drew its tokens in a launch of its own and could leave no row unread (step of 512 fp32 rows, V = 151,936:
// 578 us with the ring, 523 this way; 384 rows 440 / 394; 1,000 rows, V = 60,000, 535 / 418).
// A direct grid is a kernel of its own: one body with both ways of finding the work and both ways of drawing spilled 216 / 324
// bytes (stores / loads) of bf16 and 52 / 44 of fp32 in all batches.  Apart, 32 / 32 and 20 / 16 with the list, 180 / 284 and 20 / 16
// direct: step of 1,000 bf16 rows of 6, V = 20,000, 128.6 -> 126.3 us, of 1,024, V = 128,256, 388.5 -> 386.1, of 16 23.9 -> 23.4, of 37,
// V = 50,257, 22.4 -> 21.9, of one fp32 row, V = 32,000, 11.3 -> 10.9, signals of 700 fp32 rows of 4, V = 30,001, 59.0 -> 57.9.  (The
// direct grid's spills are its draw's, behind a wait: out of line, 20 / 20 bytes, signals of 128 bf16 rows, V = 128,256, take 43.1 us,
// this way 42.5.)
// ----------------------------------------------------------------------------------------
template <typename T, bool DIRECT>
__global__ void __launch_bounds__(kThreads, SweepShape<T>::kCtas) sweep_kernel(const __grid_constant__ KParams P) {
    __shared__ float4 sh_part[kWarps];
    __shared__ RowDecide sh_pos[kMaxGamma + 1];
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    __shared__ int sh_last;
    __shared__ int sh_early;
    __shared__ float sh_m0[kWarps];
    __shared__ __align__(16) KParams sh_P;
    __shared__ DirectEntry sh_entry;  // DIRECT only, as the next one
    __shared__ int sh_scan[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const int i = static_cast<int>(blockIdx.x) / P.nsplit, s = static_cast<int>(blockIdx.x) - i * P.nsplit;
    int2 entry = make_int2(0, 0);
    int n_list;
    if constexpr (DIRECT) {
        n_list = direct_entry(P, i, &sh_entry, sh_scan);
        entry = sh_entry.entry;
    } else {
        wait_for_predecessors();  // the list and the cleared counters
        dependents_may_start();
        if (i < P.B * P.J && dbg_ok(P.list + i, 8, DBG_WS_LOAD)) entry = __ldcg(P.list + i);
        n_list = __ldcg(P.n_list);
    }
    if (i >= n_list) {
        const int d = static_cast<int>(blockIdx.x) - n_list * P.nsplit;
        if constexpr (DIRECT) {
            wait_for_predecessors();
            dependents_may_start();
            if (d < P.n_draw) direct_draw<T>(P, d, &sh_src, sh_sum);
        } else if (d < P.n_draw) {
            resample_body<T>(P, d);
        }
        return;
    }
    const int b = entry.x, j = entry.y & 63, gen = (entry.y >> 6) & 3;
    const bool row_ok = !(entry.y & ENTRY_FLAGGED);
    const bool is_target = verify && j <= P.G;  // target positions come first in a batch row's numbering
    const int pos = is_target ? j : (verify ? j - (P.G + 1) : j);
    int gam = entry.y >> 16;
    float Tf, scale = 0.f;
    if (row_ok) {
        // the first logits are requested before anything else about the row is known
        const T* row = is_target ? static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp
                                 : static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(pos) * P.dsp;
        const int lo = (s * kWarps + warp) * P.per_warp;  // this warp's granules: the CTA's slice is cut into one contiguous range per warp
        WarpSweep<T, SweepShape<T>::kSteps> ws;
        if constexpr (DIRECT) {
            ws.template start<true>(make_row(row, P.V), lo, lo + P.per_warp);
            wait_for_predecessors();
            dependents_may_start();
            Tf = sh_entry.temp;
        } else {
            ws.start(make_row(row, P.V), lo, lo + P.per_warp);
            Tf = P.temp ? P.temp[b] : P.temp_scalar;
        }
        if (!DIRECT && threadIdx.x == 0) {
            // one thread reads what is known of the row's stop position, so that the whole CTA takes one decision
            int e = 0x7fffffff;
            if (P.early && gen == 2 && !P.read_all)
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(e) : "l"(P.early + b) : "memory");
            sh_early = e;
        }
        const float m0 = ws.template warm<true>(sh_m0);
        const bool greedy = (Tf == 0.f);
        scale = row_scale(Tf);
        const long long pidx = (static_cast<long long>(b) * P.J + j) * P.nsplit + s;  // this CTA's partial
        if (!DIRECT && gen == 2 && sh_early <= pos) {
            // The walk stopped at a position before this one: the row epilogue never looks here, the partial only has to
            // be finite.
            if (threadIdx.x == 0)
                SPECKV_ST(P.part[pidx], greedy ? make_float4(kFloor, __int_as_float(0x7fffffff), 0.f, 0.f)
                                               : make_float4(kFloor, 0.f, 0.f, 0.f));
        } else {
            float4 part;
            int path;
            if (!is_target) {
                if (verify && P.tokl && s == 0 && threadIdx.x == 0 && !greedy) {
                    // the acceptance test of this position needs both logits at the draft token: fetch them
                    // now, while the sweep hides the latency, and leave them for the row epilogue
                    const int x = P.tok[static_cast<long long>(b) * P.G + pos] - P.v_begin;  // index in this slice
                    if (x >= 0 && x < P.V) {
                        const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb +
                                        static_cast<long long>(pos) * P.tsp;
                        SPECKV_ST(P.tokl[static_cast<long long>(b) * P.G + pos], make_float2(elem_to_float(row, x), elem_to_float(trow, x)));
                    }
                }
                part = ws.draft(m0, scale, row, P.V, lo, lo + P.per_warp);
                path = PATH_DRAFT;
            } else if (greedy) {
                part = ws.template run<PATH_ARGMAX>(m0, scale);
                path = PATH_ARGMAX;
            } else {
                part = ws.template run<PATH_TARGET>(m0, scale);
                path = PATH_TARGET;
                // the position a bonus token would be drawn from: this warp's sum is a span of that draw
                if (P.spans && pos == gam && lane == 0)
                    SPECKV_ST(P.spans[(static_cast<long long>(b) * P.nsplit + s) * kWarps + warp], make_float2(part.x, part.y));
            }
            if (lane == 0) sh_part[warp] = part;
            __syncthreads();
            if (warp == 0) {
                const float4 none = (path == PATH_ARGMAX) ? make_float4(kFloor, __int_as_float(0x7fffffff), 0.f, 0.f)
                                  : make_float4(path == PATH_TARGET ? -3.0e38f : kFloor, 0.f, 0.f, 0.f);
                const float4 w = lane < kWarps ? sh_part[lane] : none;
                const float4 acc = (path == PATH_DRAFT) ? warp_merge<PATH_DRAFT>(w, scale)
                                 : (path == PATH_TARGET) ? warp_merge<PATH_TARGET>(w, scale) : warp_merge<PATH_ARGMAX>(w, scale);
                if (lane == 0) SPECKV_ST(P.part[pidx], acc);
            }
        }
    } else {
        if constexpr (DIRECT) {
            wait_for_predecessors();
            dependents_may_start();
        }
        if (s != 0) return;  // a flagged row has one CTA, for the epilogue
        gam = P.gamma ? P.gamma[b] : P.G;
        Tf = P.temp ? P.temp[b] : P.temp_scalar;
    }

    // tickets: the last of a position's CTAs takes its acceptance test, the last of all of the row's CTAs runs the row epilogue;
    // nobody waits
    if (threadIdx.x == 0) {
        const int n_rows = verify ? 2 * gam + 1 : gam;
        const int n_tickets = row_ok ? n_rows * P.nsplit : 1;
        __threadfence();
        int l = 0;
        if (!DIRECT && P.early && row_ok && pos < gam && pos < P.n_tests) {
            const int sh = pos * P.pos_bits;
            const unsigned long long old = atomicAdd(P.tick_pos + b, 1ull << sh);
            l = static_cast<int>(old >> sh & ((1ull << P.pos_bits) - 1)) == 2 * P.nsplit - 1 ? 1 : 0;
        }
        if (atomicAdd(P.tick1 + b, 1) == n_tickets - 1) l = 2;  // (the whole row's epilogue: no test before it)
        if (l) __threadfence();
        sh_last = l;
    }
    params_to_shared(P, &sh_P, 32);  // while the tickets travel
    __syncthreads();
    const int last = sh_last;
    if (!DIRECT && (last & 1)) {
        if (warp == 0) test_position<T>(sh_P, b, gam, Tf == 0.f, scale, pos, sh_pos);
        return;
    }
    if (!(last & 2)) return;
    if (!DIRECT && P.export_state) {
        const long long row0 = static_cast<long long>(b) * P.J;
        if (warp == 0)
            export_epilogue(sh_P, b, gam, Tf, P.part + (row0 + P.G + 1 + lane) * P.nsplit, P.nsplit,
                            P.part + (row0 + lane) * P.nsplit, P.nsplit);
        return;
    }
    row_epilogue_cta<T>(sh_P, b, gam, Tf, scale, sh_pos, sh_sum, &sh_src);
}

// ----------------------------------------------------------------------------------------
// Short rows: a whole batch row by one CTA, in one launch without a list, tickets or a queue.  P.nsplit neighbouring warps
// fold a logit row, each a contiguous range whose partial is also a span of a bonus draw; the row epilogue and the residual
// draw follow in the same CTA.  Latency-bound: a CTA's life is a chain of about 10 us behind its loads, so what counts is that
// a batch row has one such chain and one CTA, not one CTA's start, merge and ticket (6 us) for every logit row (step of 500
// rows, V = 3,000, gamma up to 8: bf16 64.8 -> 36.5 us, fp32 72.4 -> 37.0; of 8 to 16 rows about 20 -> 17).  Which batches: short_rows()
// in speckv.cu.
// ----------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kThreads, 4) batch_row_kernel(const __grid_constant__ KParams P) {
    __shared__ RowDecide sh_pos[kMaxGamma + 1];
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    __shared__ __align__(16) KParams sh_P;
    params_to_shared(P, &sh_P, 0);
    wait_for_predecessors();
    dependents_may_start();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const int gam = P.gamma ? P.gamma[b] : P.G;
    const float Tf = P.temp ? P.temp[b] : P.temp_scalar, scale = row_scale(Tf);
    const bool greedy = (Tf == 0.f);
    if (!row_status0(P, gam, Tf)) {
        const int n_rows = verify ? 2 * gam + 1 : gam, sub = warp % P.nsplit;
        for (int q = warp / P.nsplit; q < n_rows; q += kWarps / P.nsplit) {
            const bool is_target = verify && q <= gam;
            const int pos = is_target || !verify ? q : q - (gam + 1), j = is_target || !verify ? pos : P.G + 1 + pos;
            const T* row = is_target ? static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp
                                     : static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(pos) * P.dsp;
            WarpSweep<T, 4> ws;
            ws.start(make_row(row, P.V), sub * P.per_warp, sub * P.per_warp + P.per_warp);
            if (verify && !is_target && !greedy && lane == 0 && sub == 0) {  // both logits at the draft token
                const long long at = static_cast<long long>(b) * P.G + pos;
                const int x = P.tok[at];
                if (x >= 0 && x < P.V) {
                    const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp;
                    SPECKV_ST(P.tokl[at], make_float2(elem_to_float(row, x), elem_to_float(trow, x)));
                }
            }
            const float m0 = ws.template warm<false>(nullptr);
            float4 part;
            if (!is_target) part = ws.draft(m0, scale, row, P.V, sub * P.per_warp, sub * P.per_warp + P.per_warp);
            else if (greedy) part = ws.template run<PATH_ARGMAX>(m0, scale);
            else part = ws.template run<PATH_TARGET>(m0, scale);
            if (lane == 0) {
                SPECKV_ST(P.part[(static_cast<long long>(b) * P.J + j) * P.nsplit + sub], part);
                if (is_target && pos == gam && !greedy)
                    SPECKV_ST(P.spans[static_cast<long long>(b) * P.nsplit + sub], make_float2(part.x, part.y));
            }
        }
    }
    __syncthreads();
    row_epilogue_cta<T>(sh_P, b, gam, Tf, scale, sh_pos, sh_sum, &sh_src);
    if (!verify) return;
    __syncthreads();
    const RowInfo ri = row_info_load(P.info + b);
    if (ri.mode == RS_RESIDUAL) resample_row<T>(P, b, ri.n, 0);
}

}  // namespace speckv
