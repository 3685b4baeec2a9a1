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
__device__ __noinline__ void row_epilogue_cta(const KParams& P, int b, int gam, float Tf, RowDecide* pos, double* sh_sum,
                                              DrawSrc* sh_src) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    const long long row0 = static_cast<long long>(b) * P.J;
    const int n_pos = row_status0(P, gam, Tf) ? 0 : verify ? gam + 1 : gam;
    // the parameters travel while the positions are decided; warps 0 and 1 take the last turns
    CtlRegs ctl;
    if (warp == 1 && (P.mode & MODE_MLP) && n_pos) ctl = ctl_load(P, b, lane);
    for (int i = kWarps - 1 - warp; i < n_pos; i += kWarps)
        decide_position<T>(P, b, gam, Tf, i, P.part + (row0 + (verify ? P.G + 1 + i : i)) * P.nsplit, P.part + (row0 + i) * P.nsplit,
                           P.nsplit, pos[i]);
    __syncthreads();
    if (warp >= kDrawWarp0) {
        // a bonus draw: every position accepted, nothing flagged
        if (!verify || !n_pos || Tf == 0.f) return;
        bool ends = false;
        if (lane < n_pos) ends = pos[lane].dbad || pos[lane].tbad || pos[lane].badtok || !pos[lane].accept;
        if (__any_sync(0xffffffffu, ends)) return;
        const T* row = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(gam) * P.tsp;
        const float scale = static_cast<float>(kLog2e / static_cast<double>(Tf));
        const int n = P.nsplit * kWarps;
        const int tok = draw_from_spans<T>(row, P.V, scale, P.spans + static_cast<long long>(b) * n, n, P.per_warp, pos[gam].u_res,
                                           warp - kDrawWarp0, kWarps - kDrawWarp0, 1, sh_sum, sh_src);
        if (tok != kNotMine && lane == 0) P.out_tok[static_cast<long long>(b) * (P.G + 1) + gam] = max(tok, 0);
        return;
    }
    RowDecide dec;
    dec.x = -1; dec.u_res = 0.f; dec.Hi = dec.ci = 0.f; dec.lse2_q = dec.lse2_p = 0.0; dec.amax = -1;
    dec.dbad = dec.tbad = dec.badtok = false; dec.accept = true;
    if (lane < n_pos) dec = pos[lane];
    if (warp == 0) finish_verify(P, b, gam, Tf, dec, true);
    else if (P.mode & MODE_SIGNALS) finish_signals(P, b, gam, Tf, dec, ctl);
}

// ----------------------------------------------------------------------------------------
// Sweep kernel.  CTAs 0 .. n_sweep-1 sweep one slice of one logit row each.  With verification the
// grid may carry B*R more CTAs behind them that draw the fresh tokens of rejected rows in the same launch:
// CTAs start in index order, so these start exactly when the sweep runs out of slices, wait (with
// a bound) for their batch row's completion flag and fill the SMs that the sweep's last CTAs
// leave one by one.  A second launch, even a programmatic dependent one, starts microseconds
// after the last sweep CTA has started and leaves most of the drain unused.
// ----------------------------------------------------------------------------------------
template <typename T, int U>
__global__ void __launch_bounds__(kThreads, kSweepCtasPerSm) sweep_kernel(const __grid_constant__ KParams P) {
    if (static_cast<int>(blockIdx.x) >= P.n_sweep) {
        resample_body<T>(P, static_cast<int>(blockIdx.x) - P.n_sweep);
        return;
    }
    __shared__ float4 sh_part[kWarps];
    __shared__ RowDecide sh_pos[kMaxGamma + 1];
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    __shared__ int sh_last;
    __shared__ int sh_early;
    __shared__ float sh_m0[kWarps];
    asm volatile("griddepcontrol.launch_dependents;");  // a dependent resample kernel may be scheduled as SMs free up
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    int b, j, s, gen = 0;
    if (P.early) {
        // generation order: CTAs start in index order, so a later generation starts when the earlier ones
        // are all under way and, for all but the smallest batches, long after the first one has finished
        const int ns = P.nsplit, k1 = P.k_early + 1;
        const int nA = k1 * P.B * 2 * ns, nB = (P.G - k1) * P.B * ns;
        int i = blockIdx.x, p, is_draft;
        if (i < nA) {
            p = i / (2 * P.B * ns); i -= p * (2 * P.B * ns);
            b = i / (2 * ns); i -= b * (2 * ns);
            is_draft = i / ns; s = i - is_draft * ns;
        } else {
            // the later generations go batch row by batch row, so that the rows complete one after another
            gen = (i < nA + nB) ? 1 : 2;
            i -= (gen == 1) ? nA : nA + nB;
            const int per_b = (gen == 1 ? P.G - k1 : P.G + 1 - k1) * ns;
            b = i / per_b; i -= b * per_b;
            p = i / ns; s = i - p * ns;
            p += k1;
            is_draft = (gen == 1);
        }
        j = is_draft ? P.G + 1 + p : p;
    } else {
        const int per_row = P.J * P.nsplit;
        b = blockIdx.x / per_row;
        const int r = blockIdx.x - b * per_row;
        j = r / P.nsplit;
        s = r - j * P.nsplit;
    }
    // the row's gamma and temperature travel together with the one thing a CTA of the last generation has
    // to learn first: one memory round trip before the CTA knows whether it has work
    int gam = P.gamma ? P.gamma[b] : P.G;
    float Tf = P.temp ? P.temp[b] : P.temp_scalar;
    if (threadIdx.x == 0) {
        // one thread reads what is known of the row's stop position, so that the whole CTA takes one decision
        int e = 0;
        if (gen == 2 && !P.read_all)
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(e) : "l"(P.early + b) : "memory");
        sh_early = e;
    }
    if (threadIdx.x < kWarps) sh_m0[threadIdx.x] = kFloor;
    __syncthreads();  // before any load is issued
    const int rem = j * P.nsplit + s;

    const bool row_ok = (gam >= 1 && gam <= P.G) && (Tf >= 0.f) && (Tf != __int_as_float(0x7f800000));
    const bool greedy = (Tf == 0.f);
    const float scale = static_cast<float>(kLog2e / static_cast<double>(greedy ? 1.f : Tf));

    // logit row handled by this CTA: with verification, j <= G are target positions and the
    // rest draft positions; signals alone sweep draft positions only
    const bool is_target = verify && j <= P.G;
    const int pos = is_target ? j : (verify ? j - (P.G + 1) : j);
    const bool active = row_ok && (is_target ? pos <= gam : pos < gam);
    const long long pidx = (static_cast<long long>(b) * P.J + j) * P.nsplit + s;  // this CTA's partial

    // the walk stopped at a position before this one
    const bool skipped = active && gen == 2 && sh_early != 0 && sh_early <= P.k_early + 1;
    if (skipped) {
        // the row epilogue never looks behind the stop position; the partial only has to be finite
        if (threadIdx.x == 0)
            SPECKV_ST(P.part[pidx], greedy ? make_float4(kFloor, __int_as_float(0x7fffffff), 0.f, 0.f)
                                           : make_float4(kFloor, 0.f, 0.f, 0.f));
    } else if (active) {
        // this warp's granules: the CTA's slice is cut into one contiguous range per warp
        const int lo = (s * kWarps + warp) * P.per_warp, hi = lo + P.per_warp;
        float4 part;
        int path;
        if (is_target) {
            const T* row = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb +
                           static_cast<long long>(pos) * P.tsp;
            if (greedy) { part = sweep_warp<T, PATH_ARGMAX, U>(make_row(row, P.V), lo, hi, scale, sh_m0); path = PATH_ARGMAX; }
            else { part = sweep_warp<T, PATH_TARGET, U>(make_row(row, P.V), lo, hi, scale, sh_m0); path = PATH_TARGET; }
            // the position a bonus token would be drawn from: this warp's sum is a span of that draw
            if (P.spans && pos == gam && !greedy && lane == 0)
                SPECKV_ST(P.spans[(static_cast<long long>(b) * P.nsplit + s) * kWarps + warp], make_float2(part.x, part.y));
        } else {
            const T* row = static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb +
                           static_cast<long long>(pos) * P.dsp;
            if (verify && P.tokl && s == 0 && threadIdx.x == 0 && !greedy) {
                // the acceptance test of this position needs both logits at the draft token: fetch them
                // now, while the sweep hides the latency, and leave them for the row epilogue
                const int x = __ldg(P.tok + static_cast<long long>(b) * P.G + pos) - P.v_begin;  // index in this slice
                if (x >= 0 && x < P.V) {
                    const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb +
                                    static_cast<long long>(pos) * P.tsp;
                    SPECKV_ST(P.tokl[static_cast<long long>(b) * P.G + pos], make_float2(elem_to_float(row, x), elem_to_float(trow, x)));
                }
            }
            part = sweep_warp<T, PATH_DRAFT, U>(make_row(row, P.V), lo, hi, scale, sh_m0);
            path = PATH_DRAFT;
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
    } else if (row_ok || rem != 0) {
        return;  // unused position: nothing to count; a flagged row keeps its first CTA for the epilogue
    }

    // tickets: the last of the row's CTAs of positions 0..k_early takes their acceptance tests, the last of all its active
    // CTAs runs the row epilogue; nobody waits
    if (threadIdx.x == 0) {
        const int n_rows = verify ? 2 * gam + 1 : gam;
        const int n_tickets = row_ok ? n_rows * P.nsplit : 1;
        const int n_pre = (min(P.k_early, gam) + 1 + min(P.k_early + 1, gam)) * P.nsplit;
        __threadfence();
        int pre = -1;
        if (P.early && active && gen == 0) pre = atomicAdd(P.tick_early + b, 1);
        const int all = atomicAdd(P.tick1 + b, 1);
        const int l = (all == n_tickets - 1 ? 2 : 0) | (pre == n_pre - 1 ? 1 : 0);
        if (l) __threadfence();
        sh_last = l;
    }
    __syncthreads();
    const int last = sh_last;
    if (last & 1) prefix_epilogue<T>(P, b, gam, Tf, sh_pos);
    if (!(last & 2)) return;
    if (P.export_state) {
        const long long row0 = static_cast<long long>(b) * P.J;
        if (warp == 0)
            export_epilogue(P, b, gam, Tf, P.part + (row0 + P.G + 1 + lane) * P.nsplit, P.nsplit,
                            P.part + (row0 + lane) * P.nsplit, P.nsplit);
        return;
    }
    row_epilogue_cta<T>(P, b, gam, Tf, sh_pos, sh_sum, &sh_src);
}

}  // namespace speckv
