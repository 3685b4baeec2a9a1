// Draft-side sampling in one pass over the logits (tokens[b,i] ~ softmax(d_i / T_b) by inverse CDF,
// argmax for T_b = 0; the drafting step of Sec. 3.1).
//
// A drafted position is one logit row, swept like a target row: each warp leaves the sum of its contiguous range, and
// these sums are the spans of a plain draw (speckv_draw.cuh), so the CTA that completes the row reads one warp range again
// and nothing else.  Of a long range it leaves the sums of up to eight pieces, so that what is read again is a granule per thread, one
// round trip: every row is drawn from, and the ranges read again were an eighth of the traffic (256 bf16 rows of 8, V = 128,256, 70.8 ->
// 65 us; 287 fp32 rows of 6, V = 29,184, 31.3 -> 27.9).
#pragma once

#include "speckv_draw.cuh"

namespace speckv {

// grid: B * G * nsplit CTAs, one per (batch row, position, vocabulary slice).  P.spans holds [B*G, n_spans]
// (reference, sum) pairs, one per warp that can have granules, for greedy rows (best value or NaN, index); P.tick1 one counter per position, P.tick2 one per
// batch row, P.rdone (here: a per-row status word), all zeroed by clear_kernel.
// (A kernel, since nothing can be launched ahead of the end of a memset: sampling of 24 fp32 rows, V = 32,000, 14.4 us with
// that, 10.7 this way; of one bf16 row, V = 128,256, 12.4 / 8.8.)
__global__ void __launch_bounds__(kThreads) clear_kernel(int* p, int n) {
    wait_for_predecessors();
    dependents_may_start();
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) SPECKV_ST(p[i], 0);
}

// FINE: ranges in pieces (P.fine > 1).  A kernel of its own: in one with the other the short ranges paid 12 / 4 bytes of spills (fp32; bf16
// 60 / 44) and 8 KB of shared memory, apart neither spills (293 bf16 rows of 8, V = 1,553, 24.7 -> 23.9 us; 256 rows, V = 128,256, 65.8 ->
// 64.9).
template <typename T, bool FINE>
__global__ void __launch_bounds__(kThreads, SweepShape<T>::kCtas) sample_kernel(const __grid_constant__ KParams P) {
    __shared__ int sh_last;
    __shared__ float sh_m0[kWarps];
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = blockIdx.x / P.nsplit;  // draw: batch row b, drafted position i
    const int s = blockIdx.x - r * P.nsplit;
    const int b = r / P.G, i = r - b * P.G;
    // clear_kernel has waited for everything in front of it before it let this kernel start: what this one reads is complete in L2
    // although it has not waited yet, and it writes nothing before it has.
    const int gam = P.gamma ? __ldcg(P.gamma + b) : P.G;
    const float Tf = P.temp ? __ldcg(P.temp + b) : P.temp_scalar;
    const int bits = row_status0(P, gam, Tf);
    if (bits || i >= gam) {  // nothing to draw at this position
        wait_for_predecessors();
        dependents_may_start();
        if (s == 0 && threadIdx.x == 0) {
            P.out_tok[r] = -1;
            if (i == 0 && bits && P.status) P.status[b] = bits;
        }
        return;
    }
    const bool greedy = (Tf == 0.f);
    const float scale = static_cast<float>(kLog2e / static_cast<double>(greedy ? 1.f : Tf));
    const T* row = static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(i) * P.dsp;
    const int n = P.n_spans, fine = FINE ? P.fine : 1;
    float2* spans = P.spans + static_cast<long long>(r) * n;
    {
        const int lo = (s * kWarps + warp) * P.per_warp;
        WarpSweep<T, SweepShape<T>::kSteps> ws;
        ws.template start<true>(make_row(row, P.V), lo, lo + P.per_warp);
        wait_for_predecessors();
        dependents_may_start();
        const float m0 = ws.template warm<true>(sh_m0);
        const int at = s * kWarps + warp;
        if (greedy) {
            const float4 p = ws.template run<PATH_ARGMAX>(m0, scale);
            if (lane == 0 && at * fine < n) SPECKV_ST(spans[at * fine], make_float2(p.z != 0.f ? __int_as_float(0x7fc00000) : p.x, p.y));
        } else if constexpr (!FINE) {
            const float4 p = ws.template run<PATH_TARGET>(m0, scale);
            if (lane == 0 && at < n) SPECKV_ST(spans[at], make_float2(p.x, p.y));
        } else {
            __shared__ float sh_fine[kMostFine * kFineStride];
            const float4 p = ws.template run<PATH_TARGET, true>(m0, scale, nullptr, {sh_fine + threadIdx.x, fine, P.fine_groups});
            __syncwarp();
            // four lanes add up a piece
            const int k = lane >> 2;
            double sum = 0.0;
            if (k < fine) {
                const float* x = sh_fine + k * kFineStride + warp * 32 + (lane & 3) * 8;
#pragma unroll
                for (int q = 0; q < 8; ++q) sum += static_cast<double>(x[q]);
            }
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            if (k < fine && (lane & 3) == 0 && at * fine + k < n) SPECKV_ST(spans[at * fine + k], make_float2(p.x, static_cast<float>(sum)));
        }
    }
    __syncthreads();
    if (P.nsplit > 1) {  // else this CTA is the row's last: no ticket (256 bf16 rows, V = 128,256: 73.4 us with it, 71.3 without)
        if (threadIdx.x == 0) {
            __threadfence();
            const bool last = atomicAdd(P.tick1 + r, 1) == P.nsplit - 1;
            if (last) __threadfence();
            sh_last = last;
        }
        __syncthreads();
        if (!sh_last) return;
    }

    // ---- the row's last CTA ----
    int tok = -1;
    bool bad = false;
    if (greedy) {
        float4 g = make_float4(kFloor, __int_as_float(0x7fffffff), 0.f, 0.f);
        for (int k = lane * fine; k < n; k += 32 * fine) {
            const float2 v = dbg_ok(spans + k, 8, DBG_WS_LOAD) ? __ldcg(spans + k) : make_float2(kFloor, 0.f);
            g = merge_argmax(g, make_float4(v.x, v.y, v.x != v.x ? 1.f : 0.f, 0.f));
        }
        g = warp_merge<PATH_ARGMAX>(g, scale);
        bad = g.z != 0.f || !(g.x > kFloor);
        tok = __float_as_int(g.y);
    } else {
        tok = draw_from_spans<T>(row, P.V, scale, spans, n, P.per_warp, P.u[r], warp, kWarps, 1, sh_sum, &sh_src, fine,
                                 FINE ? P.fine_groups * SweepShape<T>::kSteps * 32 * (kVec * static_cast<int>(sizeof(T)) / 16) : 0);
        if (tok == kNotMine) return;
        bad = tok < 0;
    }
    if (greedy && warp != 0) return;
    // per-row bookkeeping: the row's status is the OR over its positions; a flagged row gives -1 everywhere
    int last = 0;
    if (lane == 0) {
        P.out_tok[r] = bad ? -1 : tok;
        if (bad) atomicOr(P.rdone + b, 4);
        __threadfence();
        last = (atomicAdd(P.tick2 + b, 1) == gam - 1);
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last) return;
    __threadfence();
    const int st = __ldcg(P.rdone + b);
    if (st && lane < P.G) P.out_tok[static_cast<long long>(b) * P.G + lane] = -1;
    if (lane == 0 && P.status) P.status[b] = st;
}

}  // namespace speckv
