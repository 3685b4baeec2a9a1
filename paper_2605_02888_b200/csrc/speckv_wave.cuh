// The sweep of batches that the chip holds at once: every warp takes an equal share of all logit rows in use, wherever that
// share begins and ends.
#pragma once

#include "speckv_sweep.cuh"

namespace speckv {

#ifndef WAVE_CTAS
#define WAVE_CTAS(T) SweepShape<T>::kCtas
#endif
constexpr int kWaveMaxB = 1024;  // batch rows whose prefix a CTA keeps
constexpr int kWaveMostSums = kMaxShares * kWarps / 2;  // span sums of a draw, 16 bytes each in the place of the other kernels' 8

// How `total` rows of at most ng granules are cut for nw warps.  Few rows: each into the same number of whole units, so that
// no warp has parts of two rows.  Otherwise the rows follow one another and a unit begins where the one before it ends.
// step: granules of a warp's step.  A row is part of kMaxSplit units at most.
__host__ __device__ inline void wave_cut(int total, int ng, int nw, int step, int* len, int* chunk) {
    if (total < 1) total = 1;
    if (total <= nw / 6) {
        int k = nw / total;
        const int most = (ng + step - 1) / step;
        if (k > most) k = most;
        if (k > kMaxSplit) k = kMaxSplit;
        const int c = ((ng + k - 1) / k + step - 1) / step * step;
        *chunk = c;
        *len = (ng + c - 1) / c * c;
    } else {
        const int l = (ng + 31) / 32 * 32;
        const long long all = static_cast<long long>(total) * l;
        *len = l;
        *chunk = static_cast<int>(((all + nw - 1) / nw + 31) / 32 * 32);
    }
}

// Clears what the wave kernel counts in and leaves the rows' records and the draws' sums empty.
__global__ void __launch_bounds__(kThreads) prep_wave_kernel(const __grid_constant__ KParams P) {
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
        SPECKV_ST(reinterpret_cast<int4*>(P.dsum)[k / n * kWaveMostSums + k % n], make_int4(-1, -1, -1, -1));
}

// The CTAs of one batch row's draw from a residual.  All wait for the row's record and sum their spans; the last one in the grid, which
// waits for CTAs in front of it only, picks the span and finds the token.  (As resample_row, with the record and the sums passed on
// as words that tell by themselves that they are there: no counter, no fence, nothing read twice.)
template <typename T>
__device__ __forceinline__ void wave_draw(const KParams& P, const int d, DrawSrc* sh_src, double* sh_sum) {
    __shared__ int sh_go;
    __shared__ RowInfo sh_info;
    const int b = d / P.R, share = d - b * P.R, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Gave up: the mark goes where the row epilogue, should it come after all, finds it (finish_verify); if it has been there, the
    // row is marked here.
    auto give_up = [&]() {
        const int old = atomicOr(P.rdone + b, kSlotTimeout);
        if (old & kSlotDone) {
            if (P.status) atomicOr(P.status + b, 16);
            if ((old >> 24) & 1) P.out_tok[static_cast<long long>(b) * (P.G + 1) + ((old >> 25) & 15)] = -1;
        }
    };
    if (threadIdx.x == 0) {
        RowInfo ri;
        ri.mode = RS_NONE;
        if (!row_info_wait(P.info + b, P.wait_limit, &ri)) give_up();
        if (ri.mode == RS_RESIDUAL) {
            DrawSrc s = make_draw<T>(static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(ri.n) * P.tsp,
                                     static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(ri.n) * P.dsp, P.V);
            set_norm(s, ri.scale, ri.lse2_p, ri.lse2_q);
            *sh_src = s;
        }
        sh_info = ri;
    }
    __syncthreads();
    if (sh_info.mode != RS_RESIDUAL) return;
    double2* sums = reinterpret_cast<double2*>(P.dsum) + static_cast<long long>(b) * kWaveMostSums;
    {
        const int span = share * kWarps + warp, g0 = span * P.draw_pw;
        const double w = warp_weights<T, true, false>(*sh_src, g0, min(sh_src->t.ng, g0 + P.draw_pw), NormReady{sh_src}).x;
        if (lane == 0) span_publish(sums + span, w);
    }
    if (share != P.R - 1) return;
    if (warp == 0) {
        constexpr int MOST = kWaveMostSums / 32;
        const int n = P.R * kWarps, per = (n + 31) >> 5;
        double v[MOST];
        bool got[MOST], all = false;
#pragma unroll
        for (int i = 0; i < MOST; ++i) { v[i] = 0.0; got[i] = i >= per || lane * per + i >= n; }
        for (int it = 0; it < P.wait_limit && !all; ++it) {
            bool mine = true;
#pragma unroll
            for (int i = 0; i < MOST; ++i) {
                if (!got[i]) got[i] = span_read(sums + lane * per + i, &v[i]);
                mine = mine && got[i];
            }
            all = __all_sync(0xffffffffu, mine);
            if (!all && it >= 64) __nanosleep(1000);
        }
        double before = 0.0, total = 0.0, tau = 0.0;
        const int own = pick_many<true, MOST>(n, [&](int k) {
            double x = v[0];
#pragma unroll
            for (int i = 1; i < MOST; ++i) if (k - lane * per == i) x = v[i];
            return x;
        }, static_cast<double>(sh_info.u2), &before, &total, &tau);
        if (lane == 0) {
            if (!all) give_up();
            sh_go = !all ? -1 : total > 1e-6 ? 1 : 0;
            sh_src->r0 = own * P.draw_pw;
            sh_src->r1 = min(sh_src->t.ng, (own + 1) * P.draw_pw);
            sh_src->tau = tau - before;
        }
    }
    __syncthreads();
    const int go = sh_go;
    if (go < 0) return;
    int tok;
    if (go) tok = find_token<T, true>(*sh_src, sh_src->r0, sh_src->r1, sh_src->tau, false, warp, kWarps, 1, sh_sum);
    else tok = find_token<T, false>(*sh_src, 0, sh_src->t.ng, static_cast<double>(sh_info.u2), true, warp, kWarps, 1, sh_sum);
    if (tok != kNotMine && lane == 0) P.out_tok[static_cast<long long>(b) * (P.G + 1) + sh_info.n] = max(tok, 0);
}

template <typename T>
__global__ void __launch_bounds__(kThreads, WAVE_CTAS(T)) wave_kernel(const __grid_constant__ KParams P) {
    constexpr int E = 16 / static_cast<int>(sizeof(T));
    __shared__ int sh_prefix[kWaveMaxB + 1];
    __shared__ float sh_temp[kWaveMaxB];
    __shared__ float sh_m0[kWarps];
    __shared__ int sh_row[kWarps];
    __shared__ int sh_scan[kWarps];
    __shared__ int sh_list[kThreads];
    __shared__ int sh_n_list;
    __shared__ RowDecide sh_pos[kMaxGamma + 1];
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    __shared__ __align__(16) KParams sh_P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = static_cast<int>(blockIdx.x);
    const bool verify = (P.mode & MODE_VERIFY) != 0;
    if (c >= P.n_stream) {
        wait_for_predecessors();
        dependents_may_start();
        wave_draw<T>(P, c - P.n_stream, &sh_src, sh_sum);
        return;
    }
    // Logit rows in front of each batch row.  prep_wave_kernel lets this kernel start when it has itself waited for everything in
    // front of it, so gamma, the temperatures and the logits are complete in L2 although this kernel has not waited yet.
    {
        const int per = (P.B + kThreads - 1) / kThreads, b0 = threadIdx.x * per;
        int cnt[kWaveMaxB / kThreads], sum = 0;
#pragma unroll
        for (int k = 0; k < kWaveMaxB / kThreads; ++k) {
            cnt[k] = 0;
            if (k < per && b0 + k < P.B) {
                const int gam = P.gamma ? __ldcg(P.gamma + b0 + k) : P.G;
                const float Tf = P.temp ? __ldcg(P.temp + b0 + k) : P.temp_scalar;
                if (!row_status0(P, gam, Tf)) cnt[k] = verify ? 2 * gam + 1 : gam;
                sh_temp[b0 + k] = Tf;
            }
        }
#pragma unroll
        for (int k = 0; k < kWaveMaxB / kThreads; ++k) sum += cnt[k];
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) sh_scan[warp] = incl;
        if (threadIdx.x == 0) sh_n_list = 0;
        __syncthreads();
        int at = incl - sum;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) at += w < warp ? sh_scan[w] : 0;
#pragma unroll
        for (int k = 0; k < kWaveMaxB / kThreads; ++k)
            if (k < per && b0 + k < P.B) {
                sh_prefix[b0 + k] = at;
                at += cnt[k];
                if (b0 + k == P.B - 1) sh_prefix[P.B] = at;
            }
        __syncthreads();
    }
    const int total = sh_prefix[P.B];
    RowParts rp;
    wave_cut(total, P.wave_ng, P.n_stream * kWarps, 32 * (kVec / E), &rp.len, &rp.chunk);
    const int end = total * rp.len;
    int g = min((c * kWarps + warp) * rp.chunk, end);  // (c * kWarps * chunk < 2^31: at most one unit per row more than the rows have)
    const int g_end = min(g + rp.chunk, end);
    // batch row of logit row r: the last one with prefix <= r (those without rows share their successor's prefix)
    auto batch_row = [&](int r) {
        int lo = 0, hi = P.B;  // prefix[lo] <= r < prefix[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (sh_prefix[mid] <= r) lo = mid; else hi = mid;
        }
        return lo;
    };
    for (bool first = true; first || g < g_end; first = false) {
        if (g >= g_end) {  // nothing for this warp, but the CTA's barrier
            wait_for_predecessors();
            dependents_may_start();
            params_to_shared(P, &sh_P);
            if (lane == 0) sh_row[warp] = -1;
            __syncthreads();
            break;
        }
        const int r = static_cast<int>(static_cast<unsigned>(g) / static_cast<unsigned>(rp.len)), b = batch_row(r), q = r - sh_prefix[b];
        const int cnt = sh_prefix[b + 1] - sh_prefix[b], gam = verify ? (cnt - 1) >> 1 : cnt;
        const bool is_target = verify && q <= gam;
        const int pos = is_target || !verify ? q : q - (gam + 1), j = is_target || !verify ? pos : P.G + 1 + pos;
        const T* row = is_target ? static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp
                                 : static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(pos) * P.dsp;
        const int lo = g - r * rp.len, hi = min(rp.len, lo + (g_end - g));
        WarpSweep<T, SweepShape<T>::kSteps> ws;
        ws.template start<true>(make_row(row, P.V), lo, hi);
        if (first) {  // behind the first loads: the counters are clear, the records empty
            wait_for_predecessors();
            dependents_may_start();
        }
        if (first) params_to_shared(P, &sh_P);
        const float Tf = sh_temp[b];
        const bool greedy = (Tf == 0.f);
        if (verify && !is_target && !greedy && lane == 0 && lo == 0) {  // both logits at the draft token
            const long long at = static_cast<long long>(b) * P.G + pos;
            const int x = P.tok[at];
            if (x >= 0 && x < P.V) {
                const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(pos) * P.tsp;
                SPECKV_ST(P.tokl[at], make_float2(elem_to_float(row, x), elem_to_float(trow, x)));
            }
        }
        const float scale = row_scale(Tf);
        // The largest element of the first steps, over the warps of the CTA that begin in the same row: a draft row's range has as many
        // elements above its reference, each of which takes a path of its own, as the range is longer than what the reference was taken from.
        float m0 = ws.template warm<false>(nullptr);
        if (first) {
            if (lane == 0) { sh_m0[warp] = m0; sh_row[warp] = r; }
            __syncthreads();
        }
#pragma unroll
        for (int w = 0; w < kWarps; ++w)
            if (sh_row[w] == r) m0 = fmaxf(m0, sh_m0[w]);
        float4 part;
        if (!is_target) part = ws.draft(m0, scale, row, P.V, lo, hi);
        else if (greedy) part = ws.template run<PATH_ARGMAX>(m0, scale);
        else part = ws.template run<PATH_TARGET>(m0, scale);
        if (lane == 0) SPECKV_ST(P.part[(static_cast<long long>(b) * P.J + j) * kMaxSplit + (c * kWarps + warp - rp.first(r))], part);
        g = r * rp.len + hi;
    }
    __syncthreads();
    // Tickets: the last of the CTAs that have a part of a batch row runs its epilogue; nobody waits.
    {
        const int cta = kWarps * rp.chunk, c0 = min(c * cta, end), c1 = min(c0 + cta, end);
        if (c0 < c1) {
            const int first = batch_row(static_cast<int>(static_cast<unsigned>(c0) / static_cast<unsigned>(rp.len)));
            const int last = batch_row(static_cast<int>(static_cast<unsigned>(c1 - 1) / static_cast<unsigned>(rp.len)));
            for (int b = first + threadIdx.x; b <= last; b += kThreads) {
                const int s = sh_prefix[b] * rp.len, e = sh_prefix[b + 1] * rp.len;
                if (s == e) continue;
                __threadfence();
                if (atomicAdd(P.tick1 + b, 1) == (e - 1) / cta - s / cta) {
                    __threadfence();
                    sh_list[atomicAdd(&sh_n_list, 1)] = b;
                }
            }
        }
        // batch rows without a logit row in use (a flagged gamma or temperature)
        if (threadIdx.x < 32)
            for (int b = c + P.n_stream * static_cast<int>(threadIdx.x); b < P.B; b += 32 * P.n_stream)
                if (sh_prefix[b] == sh_prefix[b + 1]) sh_list[atomicAdd(&sh_n_list, 1)] = b;
    }
    __syncthreads();
    const int n_list = sh_n_list;
    for (int k = 0; k < n_list; ++k) {
        const int b = sh_list[k];
        rp.row = sh_prefix[b];
        const int cnt = sh_prefix[b + 1] - rp.row;
        const int gam = cnt > 0 ? (verify ? (cnt - 1) >> 1 : cnt) : P.gamma ? __ldcg(P.gamma + b) : P.G;
        const float Tf = sh_temp[b];
        row_epilogue_cta<T>(sh_P, b, gam, Tf, row_scale(Tf), sh_pos, sh_sum, &sh_src, rp);
        __syncthreads();
    }
}

}  // namespace speckv
