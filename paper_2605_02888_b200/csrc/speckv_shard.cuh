// Vocabulary-sharded verification: every rank holds the columns [v_begin, v_begin + V_local) of all
// logit rows (a tensor-parallel output projection leaves them like that) and the full-vocabulary
// logits are never gathered.  What crosses the ranks is small:
//   1. sweep of the local slice          -> one merged state per logit row and shard (16 bytes each)
//   2. row epilogue on all shards' states -> signals, controller, acceptance, stop position (every
//      rank computes the same, from the same gathered bytes)
//   3. weight of the stop position's residual (or target) distribution over the local slice
//      -> two doubles per batch row and shard
//   4. the shard whose slice holds the threshold u * W draws the token.
// The statistics are those of the unsharded path: the online-softmax states merge associatively
// (Sec. 3.1 fixes only the distributions, not how their normalisers are summed), and the inverse
// CDF runs over the vocabulary in index order, shard after shard.
#pragma once

#include "speckv_sweep.cuh"

namespace speckv {

// Phase 1 for short slice rows: row_warps (1, 2, 4 or 8) neighbouring warps per (batch row, logit row), each on a contiguous
// range with U loads of 16 bytes in flight per lane; their merged state is the shard's state of that row.
// No partials, no tickets.  (Wider slices use sweep_kernel with export_state set.)  Latency-bound: one warp folds a 32 KB row in
// 16 rounds of loads, and 256 rows of 17 are fewer warps than the SMs hold (64 rows of 4 shards, V = 32,000: 18.4 us, several warps per row 16.4).
// (Steps in flight: 5 of bf16, 4 of fp32 beside 4 CTAs per SM; one rank of 8 of 256 bf16 rows 54.3 us, with the sweep's shape 57.4.)
template <typename T, int U, int CTAS>
__global__ void __launch_bounds__(kThreads, CTAS) shard_rows_kernel(const __grid_constant__ KParams P, const int row_warps) {
    __shared__ float4 sh_part[kWarps];
    wait_for_predecessors();
    dependents_may_start();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long w = (static_cast<long long>(blockIdx.x) * kWarps + warp) / row_warps;
    const int sub = warp % row_warps;
    const bool in = w < static_cast<long long>(P.B) * P.J;
    const int b = in ? static_cast<int>(w / P.J) : 0, j = in ? static_cast<int>(w - static_cast<long long>(b) * P.J) : 0;
    const int gam = P.gamma ? P.gamma[b] : P.G;
    const float Tf = P.temp ? P.temp[b] : P.temp_scalar;
    const bool row_ok = row_status0(P, gam, Tf) == 0;
    const bool greedy = (Tf == 0.f);
    const float scale = row_scale(Tf);
    const bool is_target = j <= P.G;
    const int pos = is_target ? j : j - (P.G + 1);
    const bool active = in && row_ok && (is_target ? pos <= gam : pos < gam);
    float4 st = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 tl = make_float2(0.f, 0.f);
    if (active) {
        const T* row = is_target ? static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp
                                 : static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(pos) * P.dsp;
        const GranRow gr = make_row(row, P.V);
        const int per = (gr.ng + row_warps - 1) / row_warps;
        WarpSweep<T, U> ws;
        ws.start(gr, sub * per, sub * per + per);
        if (!is_target && lane == 0 && sub == 0 && !greedy) {
            // both logits at the draft token, if it falls into this slice
            const int x = P.tok[static_cast<long long>(b) * P.G + pos] - P.v_begin;
            if (x >= 0 && x < P.V) {
                const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp;
                tl = make_float2(elem_to_float(row, x), elem_to_float(trow, x));
            }
        }
        const float m0 = ws.template warm<false>(nullptr);
        if (!is_target) {
            st = ws.draft(m0, scale, row, P.V, sub * per, sub * per + per);
        } else if (greedy) {
            st = ws.template run<PATH_ARGMAX>(m0, scale);
            const int idx = __float_as_int(st.y);
            if (idx != 0x7fffffff) st.y = __int_as_float(idx + P.v_begin);
        } else {
            st = ws.template run<PATH_TARGET>(m0, scale);
        }
    }
    if (row_warps > 1) {
        if (lane == 0) sh_part[warp] = st;
        __syncthreads();
        if (sub == 0 && active)
            for (int k = 1; k < row_warps; ++k) {
                const float4 o = sh_part[warp + k];
                st = !is_target ? merge_draft(st, o, scale) : greedy ? merge_argmax(st, o) : merge_target(st, o);
            }
    }
    if (lane == 0 && sub == 0 && in) {
        P.state[static_cast<long long>(b) * P.J + j] = st;
        if (!is_target) SPECKV_ST(P.tokl[static_cast<long long>(b) * P.G + pos], tl);
    }
}

// Phase 2: one CTA (of two warps at least) per batch row, the row epilogue of the sweep on the n_shards gathered states of each logit row
// (nsplit = n_shards, part_stride apart).  Latency-bound: with a warp per row, a lane per position and a chain of n_shards
// dependent loads in each, the four calls of 256 rows and 8 shards took 12 us more (with the changes to phases 1 and 3).
__global__ void __launch_bounds__(kThreads) shard_finish_kernel(const __grid_constant__ KParams P) {
    __shared__ RowDecide sh_pos[kMaxGamma + 1];
    __shared__ __align__(16) KParams sh_P;
    params_to_shared(P, &sh_P, 0);
    __syncthreads();
    wait_for_predecessors();
    dependents_may_start();
    const int b = blockIdx.x;
    const int gam = P.gamma ? P.gamma[b] : P.G;
    const float Tf = P.temp ? P.temp[b] : P.temp_scalar;
    row_epilogue_cta<float>(sh_P, b, gam, Tf, row_scale(Tf), sh_pos, nullptr, nullptr);
}

// Phase 3: grid B * R.  Span weights of the stop position over the local slice: of the row's own
// weights and, for a residual draw, of p as well, from the same pass (the draw falls back to p when the residual is
// numerically empty, and whether it is shows only once all shards' masses are known).  The last
// CTA of a row adds them up; with R = 1 there is no ticket.
template <typename T>
__global__ void __launch_bounds__(kThreads, 4) shard_sums_kernel(const __grid_constant__ KParams P) {
    __shared__ int sh_flag;
    wait_for_predecessors();
    dependents_may_start();
    const int b = blockIdx.x / P.R;
    const int share = blockIdx.x - b * P.R;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const RowInfo ri = P.info[b];
    if (ri.mode == RS_NONE) {
        if (share == 0 && threadIdx.x < 2) P.weight[2 * static_cast<long long>(b) + threadIdx.x] = 0.0;
        return;
    }
    const bool res = ri.mode == RS_RESIDUAL;
    const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(ri.n) * P.tsp;
    const T* drow = static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(ri.n) * P.dsp;
    const DrawSrc src = make_draw<T>(trow, res ? drow : nullptr, P.V);
    double* dr = P.dsum + static_cast<long long>(b) * (kMaxShares * kWarps);
    double* dp = P.dsum2 + static_cast<long long>(b) * (kMaxShares * kWarps);
    const int span = share * kWarps + warp, g0 = span * P.draw_pw, g1 = min(src.t.ng, g0 + P.draw_pw);
    const double2 w = res ? warp_weights<T, true, true>(src, g0, g1, NormOfRecord{P.info + b})
                           : warp_weights<T, false, true>(src, g0, g1, NormOfRecord{P.info + b});
    if (lane == 0) {
        SPECKV_ST(dr[span], w.x);
        SPECKV_ST(dp[span], w.y);
    }
    __syncthreads();
    if (P.R > 1) {
        if (threadIdx.x == 0) {
            __threadfence();
            const bool last = atomicAdd(P.tick2 + b, 1) == P.R - 1;
            if (last) __threadfence();
            sh_flag = last;
        }
        __syncthreads();
        if (!sh_flag) return;
    }
    if (warp != 0) return;
    double tr = 0.0, tp = 0.0;
    for (int k = lane; k < P.R * kWarps; k += 32)
        if (dbg_ok(dr + k, 8, DBG_WS_LOAD) && dbg_ok(dp + k, 8, DBG_WS_LOAD)) {
            tr += __ldcg(dr + k);
            tp += __ldcg(dp + k);
        }
    tr = warp_sum(tr);
    tp = warp_sum(tp);
    if (lane == 0) {
        P.weight[2 * static_cast<long long>(b)] = res ? tr : 0.0;  // a bonus row has no residual
        P.weight[2 * static_cast<long long>(b) + 1] = tp;
    }
}

// Phase 4: one CTA per batch row.  Every rank finds the owning shard from the gathered masses; the
// owner searches its own spans and writes the token into out_tokens[b, n]; the others leave the
// -1 that the row epilogue put there, so an element-wise maximum over the ranks completes the row.
template <typename T>
__global__ void __launch_bounds__(kThreads) shard_pick_kernel(const __grid_constant__ KParams P) {
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    __shared__ int sh_go;
    __shared__ int sh_mode;
    __shared__ double sh_tau;
    wait_for_predecessors();
    dependents_may_start();
    const int b = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const RowInfo ri = P.info[b];
    if (ri.mode == RS_NONE) return;
    if (warp == 0) {
        // lane r holds shard r's masses (n_shards <= 32)
        double wr = 0.0, wp = 0.0;
        if (lane < P.n_shards) {
            const double* w = P.all_weight + (static_cast<long long>(lane) * P.B + b) * 2;
            wr = w[0];
            wp = w[1];
        }
        // shards are added in index order on every rank, so all ranks see the same totals
        double tot_r = 0.0, tot_p = 0.0;
        for (int r = 0; r < P.n_shards; ++r) {
            tot_r += __shfl_sync(0xffffffffu, wr, r);
            tot_p += __shfl_sync(0xffffffffu, wp, r);
        }
        const bool use_res = (ri.mode == RS_RESIDUAL) && (tot_r > 1e-6);
        const double tot = use_res ? tot_r : tot_p;
        const double tau = static_cast<double>(ri.u2) * tot;
        double run = 0.0, before = 0.0;
        int owner = -1, last_pos = -1;
        double last_before = 0.0;
        for (int r = 0; r < P.n_shards; ++r) {
            const double w = __shfl_sync(0xffffffffu, use_res ? wr : wp, r);
            if (w > 0.0) { last_pos = r; last_before = run; }
            if (owner < 0 && w > 0.0 && run + w > tau) { owner = r; before = run; }
            run += w;
        }
        if (owner < 0) { owner = last_pos; before = last_before; }
        if (lane == 0) {
            sh_go = (owner == P.rank);
            sh_mode = use_res ? RS_RESIDUAL : RS_BONUS;
            sh_tau = tau - before;
            // no shard has any mass: cannot happen for a finite row; same answer as the unsharded path
            if (owner < 0 && P.rank == 0) P.out_tok[static_cast<long long>(b) * (P.G + 1) + ri.n] = 0;
        }
    }
    __syncthreads();
    if (!sh_go) return;
    const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(ri.n) * P.tsp;
    const T* drow = static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(ri.n) * P.dsp;
    const bool res = sh_mode == RS_RESIDUAL;
    if (threadIdx.x == 0) {
        DrawSrc src = make_draw<T>(trow, res ? drow : nullptr, P.V);
        set_norm(src, ri.scale, ri.lse2_p, ri.lse2_q);
        sh_src = src;
    }
    const double* dsum = (res ? P.dsum : P.dsum2) + static_cast<long long>(b) * (kMaxShares * kWarps);
    double before = 0.0, total, tau;
    const int own = pick_many<false, 8>(P.R * kWarps, [&](int k) { return dbg_ok(dsum + k, 8, DBG_WS_LOAD) ? __ldcg(dsum + k) : 0.0; },
                                     sh_tau, &before, &total, &tau);
    __syncthreads();
    if (own < 0) return;
    const int g0 = own * P.draw_pw, g1 = min(sh_src.t.ng, g0 + P.draw_pw);
    const int tok = res ? find_token<T, true>(sh_src, g0, g1, tau - before, false, warp, blockDim.x >> 5, 1, sh_sum)
                        : find_token<T, false>(sh_src, g0, g1, tau - before, false, warp, blockDim.x >> 5, 1, sh_sum);
    if (lane == 0 && tok >= 0) P.out_tok[static_cast<long long>(b) * (P.G + 1) + ri.n] = tok + P.v_begin;
}

}  // namespace speckv
