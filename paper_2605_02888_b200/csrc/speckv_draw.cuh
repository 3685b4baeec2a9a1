// Drawing a token by inverse CDF in vocabulary order (Sec. 3.1: the fresh token of a step, the tokens of a draft).
//   residual  w_v = max(0, p_v - q_v)     a rejected position
//   plain     w_v = p_v                   the bonus position, a drafted position
// Weights are fp32, everything above one lane's granule is summed in double.  A draw knows the weight of a few ranges
// ("spans", one per warp that summed it), takes the span that holds the threshold and narrows it down: a CTA sums up to 64
// parts of the range at once, picks one, until 32 granules are left, which one warp scans.  A plain draw gets its spans
// from the sweep itself (the sums a warp leaves of its range are the span weights), so beyond one span it never reads the
// row again; a residual needs both normalisers first, so its spans are summed by CTAs of their own.
#pragma once

#include "speckv_kernels.cuh"

namespace speckv {

// A row's record, as the two 16-byte words it consists of
__device__ __forceinline__ RowInfo row_info_load(const RowInfo* p) {
    const int4 lo = __ldcg(reinterpret_cast<const int4*>(p)), hi = __ldcg(reinterpret_cast<const int4*>(p) + 1);
    RowInfo ri;
    ri.mode = lo.x; ri.n = lo.y; ri.u2 = __int_as_float(lo.z); ri.scale = __int_as_float(lo.w);
    ri.lse2_p = __hiloint2double(hi.y, hi.x);
    ri.lse2_q = __hiloint2double(hi.w, hi.z);
    return ri;
}

struct DrawSrc {
    GranRow t, d;        // target row, draft row (residual only)
    int dg, off;         // granule g of t covers the elements of d from granule g + dg, element off, on
    int in_lo, in_hi;    // granules of t for which all granules involved are whole ones of their rows
    float scale, lp, lq, c;  // log2(e) / T, the log2-normalisers rounded to fp32, and what the rounding took from them:
                             // p - q = (2^(x_t * scale - lp) - c * 2^(x_d * scale - lq)) * 2^(lp - lse_p), c = 2^((lq - lse_q) - (lp - lse_p));
                             // the last factor is common to all weights and left out
    bool wide;               // normalisers so large that their rounding is not small: the weights take it exactly
    float plo, qlo;          // wide: lse_p - lp and lse_q - lq
    int r0, r1;              // draw_from_spans: the chosen span (r1 <= r0: there is none)
    double tau;
};

// The rows of a draw; the constants follow by set_norm, so that loads can go out while those are still on their way.
template <typename T>
__device__ __forceinline__ DrawSrc make_draw(const T* trow, const T* drow, int V) {
    constexpr int E = 16 / sizeof(T);
    DrawSrc s;
    s.t = make_row(trow, V);
    s.d = drow ? make_row(drow, V) : s.t;
    s.off = s.d.shift() - s.t.shift();
    s.dg = 0;
    if (s.off < 0) { s.off += E; s.dg = -1; }
    s.in_lo = max(s.t.whole_lo(), s.d.whole_lo() - s.dg);
    s.in_hi = min(s.t.whole_hi(), s.d.whole_hi() - s.dg - (s.off ? 1 : 0));
    return s;
}
__device__ __forceinline__ void set_norm(DrawSrc& s, float scale, double lse_p, double lse_q) {
    s.scale = scale;
    s.lp = static_cast<float>(lse_p);
    s.lq = static_cast<float>(lse_q);
    s.plo = static_cast<float>(lse_p - static_cast<double>(s.lp));
    s.qlo = static_cast<float>(lse_q - static_cast<double>(s.lq));
    s.c = ex2f(static_cast<float>((static_cast<double>(s.lq) - lse_q) - (static_cast<double>(s.lp) - lse_p)));
    // Left out, the common factor is within 2^(1/64) of one (normalisers below 2^19); the two masses that are compared with a
    // constant (1e-6) and with each other over shards need no more.  At 2^28, the logits of a few hundred at T = 1e-6 or 2e8
    // at T = 1, it would be 2^16 and a residual of any mass could pass for empty.
    s.wide = fmaxf(fabsf(s.plo), fabsf(s.qlo)) > 0x1p-6f;
}

// ---- weights of one granule ------------------------------------------------------------------------------
__device__ __forceinline__ void gran_pairs(const uint4& g, f2 (&x)[4]) {
    x[0] = pack2(bf_lo(g.x), bf_hi(g.x)); x[1] = pack2(bf_lo(g.y), bf_hi(g.y));
    x[2] = pack2(bf_lo(g.z), bf_hi(g.z)); x[3] = pack2(bf_lo(g.w), bf_hi(g.w));
}
__device__ __forceinline__ void gran_pairs(const uint4& g, f2 (&x)[2]) {
    x[0] = pack2(__uint_as_float(g.x), __uint_as_float(g.y));
    x[1] = pack2(__uint_as_float(g.z), __uint_as_float(g.w));
}
template <typename T, bool RES>
__device__ __forceinline__ void gran_weights(float scale, float lp, float lq, float c, const uint4& t, const uint4& d,
                                             float (&w)[16 / sizeof(T)], float* sum_p = nullptr) {
    constexpr int NP = 8 / sizeof(T);
    const f2 sc2 = pack2(scale, scale), p2 = pack2(-lp, -lp);
    f2 xt[NP];
    gran_pairs(t, xt);
    if constexpr (!RES) {
#pragma unroll
        for (int i = 0; i < NP; ++i) unpack2(ex2_2(fma2(xt[i], sc2, p2)), w[2 * i], w[2 * i + 1]);
    } else {
        const f2 q2 = pack2(-lq, -lq), c2 = pack2(-c, -c);
        f2 xd[NP];
        gran_pairs(d, xd);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const f2 p = ex2_2(fma2(xt[i], sc2, p2)), q = ex2_2(fma2(xd[i], sc2, q2));
            if (sum_p) *sum_p += hsum2(p);  // (known at compile time)
            float lo, hi;
            unpack2(fma2(q, c2, p), lo, hi);
            w[2 * i] = fmaxf(lo, 0.f);
            w[2 * i + 1] = fmaxf(hi, 0.f);
        }
    }
}
// The same for normalisers of any size.  Rarely taken, and out of line so that a draw, a chain of cold code, does not fetch it.
template <typename T> struct GranW { float w[16 / sizeof(T)], p; };  // p: sum of p
template <typename T, bool RES>
__device__ __noinline__ GranW<T> gran_weights_wide(float scale, float lp, float plo, float lq, float qlo, uint4 t, uint4 d) {
    constexpr int NP = 8 / sizeof(T);
    const f2 sc2 = pack2(scale, scale), ph = pack2(-lp, -lp), pl = pack2(plo, plo), qh = pack2(-lq, -lq), ql = pack2(qlo, qlo);
    f2 xt[NP], xd[NP];
    gran_pairs(t, xt);
    if (RES) gran_pairs(d, xd);
    GranW<T> o;
    o.p = 0.f;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const f2 p = ex2_2(sub2(fma2(xt[i], sc2, ph), pl));
        o.p += hsum2(p);
        unpack2(RES ? sub2(p, ex2_2(sub2(fma2(xd[i], sc2, qh), ql))) : p, o.w[2 * i], o.w[2 * i + 1]);
        o.w[2 * i] = fmaxf(o.w[2 * i], 0.f);
        o.w[2 * i + 1] = fmaxf(o.w[2 * i + 1], 0.f);
    }
    return o;
}
template <typename T, bool RES>
__device__ __forceinline__ float gran_weight(float scale, float lp, float lq, float c, const uint4& t, const uint4& d,
                                             float* sum_p = nullptr) {
    float w[16 / sizeof(T)];
    gran_weights<T, RES>(scale, lp, lq, c, t, d, w, sum_p);
    float a = 0.f;
#pragma unroll
    for (int j = 0; j < static_cast<int>(16 / sizeof(T)); ++j) a += w[j];
    return a;
}

// ---- granules that are not whole, and rows that sit differently on the 16-byte grid -------------------------
// elements off, off + 1, ... of the 2 * E elements in a and b
template <typename T>
__device__ __forceinline__ uint4 gran_shift(const uint4& a, const uint4& b, int off) {
    constexpr int EW = 4 / sizeof(T);  // elements per 32-bit word
    uint32_t w[7] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z};
    uint32_t top = b.w;
    const int wo = off / EW;
    uint32_t v[8] = {w[0], w[1], w[2], w[3], w[4], w[5], w[6], top};
    if (wo & 2) {
#pragma unroll
        for (int i = 0; i < 6; ++i) v[i] = v[i + 2];
    }
    if (wo & 1) {
#pragma unroll
        for (int i = 0; i < 5; ++i) v[i] = v[i + 1];
    }
    if (EW == 2 && (off & 1)) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __funnelshift_r(v[i], v[i + 1], 16);
    }
    return make_uint4(v[0], v[1], v[2], v[3]);
}
template <typename T>
__device__ __forceinline__ uint4 draft_any(const DrawSrc& s, int g) {  // the draft's elements of t's granule g
    const uint4 a = gran_any<T>(s.d, g + s.dg);
    return s.off ? gran_shift<T>(a, gran_any<T>(s.d, g + s.dg + 1), s.off) : a;
}
// The lane's granule g of both rows; those at or behind g1 have no weight.  WIDE: normalisers of any size (s.wide).
template <typename T, bool RES, bool WIDE = true>
__device__ __forceinline__ void load_weights(const DrawSrc& s, int g, int g1, float (&w)[16 / sizeof(T)]) {
    uint4 t = gran_fill<T>(__int_as_float(0xff800000)), d = t;
    if (g < g1) {
        if (g >= s.in_lo && g < s.in_hi) {
            t = ldg_stream(s.t.base + g);
            if (RES) d = ldg_stream(s.d.base + g + s.dg);
            if (RES && s.off) d = gran_shift<T>(d, ldg_stream(s.d.base + g + s.dg + 1), s.off);
        } else {
            t = gran_any<T>(s.t, g);
            if (RES) d = draft_any<T>(s, g);
        }
    }
    if (WIDE && s.wide) {
        const GranW<T> o = gran_weights_wide<T, RES>(s.scale, s.lp, s.plo, s.lq, s.qlo, t, d);
#pragma unroll
        for (int j = 0; j < static_cast<int>(16 / sizeof(T)); ++j) w[j] = o.w[j];
    } else {
        gran_weights<T, RES>(s.scale, s.lp, s.lq, s.c, t, d, w);
    }
}
template <typename T, bool RES>
__device__ __noinline__ double gran_weight_any(const DrawSrc s, int g) {
    float w[16 / sizeof(T)];
    load_weights<T, RES>(s, g, 0x7fffffff, w);
    double a = 0.0;
#pragma unroll
    for (int j = 0; j < static_cast<int>(16 / sizeof(T)); ++j) a += static_cast<double>(w[j]);
    return a;
}

// ---- sums ----------------------------------------------------------------------------------------------------
// Sum over whole granules pt[0], pt[32], ... (n left from this lane's first one on) of the weights that the row record says.
// Two loads per row are in flight (four where the record is known) and none is requested ahead: the other warps of the SM, not this one, hide the latency, and
// the loop, compiled by itself, does without the spills that the kernel around it has at 48 registers (step of 1,024 bf16 rows,
// V = 128,256, 430 us; two requested ahead 9 us more, four in flight 5 us more).  The record is fetched behind the first loads.
// WITH_P: the sum of p as well (.y).
struct NormOfRecord {  // the row's record in global memory
    static constexpr int kInFlight = 2;
    const RowInfo* info;
    __device__ __forceinline__ DrawSrc get() const {
        const RowInfo ri = row_info_load(info);
        DrawSrc s;
        set_norm(s, ri.scale, ri.lse2_p, ri.lse2_q);
        return s;
    }
};
struct NormReady {  // in shared memory
    static constexpr int kInFlight = 4;
    const DrawSrc* src;
    __device__ __forceinline__ DrawSrc get() const {
        DrawSrc s;
        s.scale = src->scale; s.lp = src->lp; s.lq = src->lq; s.c = src->c; s.wide = src->wide; s.plo = src->plo; s.qlo = src->qlo;
        return s;
    }
};
template <typename T, bool RES, bool SHIFTED, bool WITH_P, class Norm>
__device__ __noinline__ double2 span_weight(const uint4* pt, const uint4* pd, int n, int off, const Norm norm) {
    constexpr int KU = SHIFTED ? 1 : Norm::kInFlight;
    uint4 t[KU], d[KU], d1[KU];
    auto load = [&]() {
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            t[u] = gran_fill<T>(__int_as_float(0xff800000));
            if (RES) d[u] = t[u];
            if (RES && SHIFTED) d1[u] = t[u];
            if (32 * u < n) {
                t[u] = ldg_stream(pt + 32 * u);
                if (RES) d[u] = ldg_stream(pd + 32 * u);
                if (RES && SHIFTED) d1[u] = ldg_stream(pd + 32 * u + 1);
            }
        }
        pt += 32 * KU;
        pd += 32 * KU;
        n -= 32 * KU;
    };
    load();
    const DrawSrc s = norm.get();
    double2 acc = make_double2(0.0, 0.0);
    if (s.wide) {  // from the start again, a granule at a time
        n += 32 * KU;
        pt -= 32 * KU;
        pd -= 32 * KU;
        for (; n > 0; n -= 32, pt += 32, pd += 32) {
            const uint4 a = ldg_stream(pt);
            uint4 b = a;
            if (RES) b = ldg_stream(pd);
            if (RES && SHIFTED) b = gran_shift<T>(b, ldg_stream(pd + 1), off);
            const GranW<T> o = gran_weights_wide<T, RES>(s.scale, s.lp, s.plo, s.lq, s.qlo, a, b);
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < static_cast<int>(16 / sizeof(T)); ++j) sum += o.w[j];
            acc.x += static_cast<double>(sum);
            if (WITH_P) acc.y += static_cast<double>(o.p);
        }
        return acc;
    }
    for (;;) {
        float w = 0.f, wp = 0.f;
#pragma unroll
        for (int u = 0; u < KU; ++u)
            w += gran_weight<T, RES>(s.scale, s.lp, s.lq, s.c, t[u], RES ? (SHIFTED ? gran_shift<T>(d[u], d1[u], off) : d[u]) : t[u],
                                     RES && WITH_P ? &wp : nullptr);
        acc.x += static_cast<double>(w);
        if (WITH_P) acc.y += static_cast<double>(RES ? wp : w);
        if (n <= 0) return acc;
        load();
    }
}
// Weight of granules [g0, g1), one warp, the same in every lane (.x; WITH_P: of p in .y).  Of s only the rows are needed.
template <typename T, bool RES, bool WITH_P, class Norm>
__device__ __forceinline__ double2 warp_weights(const DrawSrc& s, int g0, int g1, const Norm norm) {
    const int lane = threadIdx.x & 31;
    const int a = min(max(g0, s.in_lo), g1), e = max(min(g1, s.in_hi), a);
    double2 acc = make_double2(0.0, 0.0);
    if (e - a - lane > 0) {
        const uint4 *pt = s.t.base + a + lane, *pd = s.d.base + s.dg + a + lane;
        acc = (RES && s.off) ? span_weight<T, RES, RES, WITH_P>(pt, pd, e - a - lane, s.off, norm)
                             : span_weight<T, RES, false, WITH_P>(pt, pd, e - a - lane, 0, norm);
    }
    __syncwarp();
    // incomplete granules in front of and behind [a, e): a handful at most, one per lane
    const int nl = a - g0, nr = g1 - e;
    if (nl + nr > 0) {
        DrawSrc c = norm.get();
        c.t = s.t; c.d = s.d; c.dg = s.dg; c.off = s.off; c.in_lo = s.in_lo; c.in_hi = s.in_hi;
        for (int k = lane; k < nl + nr; k += 32) {
            const int g = k < nl ? g0 + k : e + (k - nl);
            acc.x += gran_weight_any<T, RES>(c, g);
            if (WITH_P) acc.y += gran_weight_any<T, false>(c, g);
        }
    }
    acc.x = warp_sum(acc.x);
    if (WITH_P) acc.y = warp_sum(acc.y);
    return acc;
}

// ---- picking -------------------------------------------------------------------------------------------------
// Which of n <= 32 * MOST weights get(0..n-1) holds tau (u itself, or u * total where FRACTION is set): the first at which the
// running sum exceeds it, else the last with weight; *before: the sum in front of it, *total: of all.  -1: none has weight.
// One scan over the lanes, each of which walks its own weights behind it: 0.4 us less than a scan for the lane and one for its
// weights, in a chain that a draw goes through two or three times.
template <bool FRACTION, int MOST, class F>
__device__ __forceinline__ int pick_many(int n, F get, double u, double* before, double* total, double* tau_out) {
    const int lane = threadIdx.x & 31;
    const int per = (n + 31) >> 5;  // lane k takes weights k * per ...
    double v[MOST], w = 0.0;
#pragma unroll
    for (int i = 0; i < MOST; ++i) {
        v[i] = (i < per && lane * per + i < n) ? get(lane * per + i) : 0.0;
        w += v[i];
    }
    double incl = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    *total = __shfl_sync(0xffffffffu, incl, 31);
    const double tau = FRACTION ? u * *total : u;
    *tau_out = tau;
    const unsigned hit = __ballot_sync(0xffffffffu, incl > tau && w > 0.0);
    const unsigned pos = __ballot_sync(0xffffffffu, w > 0.0);
    if (!pos) return -1;
    const int own = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
    double run = incl - w, at = 0.0;
    int sub = 0;
    bool found = false;
#pragma unroll
    for (int i = 0; i < MOST; ++i) {
        if (v[i] > 0.0 && !found) {
            sub = i;
            at = run;
            found = run + v[i] > tau;
        }
        run += v[i];
    }
    *before = __shfl_sync(0xffffffffu, at, own);
    return own * per + __shfl_sync(0xffffffffu, sub, own);
}

// One warp: the token among 32 consecutive granules whose weights its lanes hold (lane 0 granule g0).
template <typename T>
__device__ __forceinline__ int scan_weights(const DrawSrc& s, int g0, const float (&w)[16 / sizeof(T)], double tau) {
    constexpr int E = 16 / sizeof(T);
    const int lane = threadIdx.x & 31;
    double tot = 0.0;
#pragma unroll
    for (int j = 0; j < E; ++j) tot += static_cast<double>(w[j]);
    double incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    double run = incl - tot;
    int found = 0x7fffffff, last = -1;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        run += static_cast<double>(w[j]);
        if (w[j] > 0.f) {
            last = (g0 + lane) * E - s.t.shift() + j;
            if (run > tau && found == 0x7fffffff) found = last;
        }
    }
    const int f = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(found)));
    return f != 0x7fffffff ? f : __reduce_max_sync(0xffffffffu, last);
}

constexpr int kNotMine = -2;

// nw warps (this one is wi) that share named barrier `bar`: the token within granules [g0, g1) at tau (`fraction`: at tau times
// the range's own weight).  Exactly one warp gets the answer (-1: nothing in the range has weight), the others kNotMine.
// sh: 64 doubles of shared memory.
template <typename T, bool RES>
__device__ __noinline__ int find_token(const DrawSrc& s, int g0, int g1, double tau, bool fraction, int wi, int nw, int bar, double* sh) {
    constexpr int E = 16 / sizeof(T);
    const int lane = threadIdx.x & 31;
    for (;;) {
        const int n = g1 - g0;
        const int sub = ((n + 63) / 64 + 31) / 32 * 32, cnt = (n + sub - 1) / sub;
        const bool leaf = cnt <= nw && sub == 32;  // one granule per lane: the warp that holds the token has its weights at hand
        float w[E];
        if (leaf) {
            load_weights<T, RES>(s, g0 + wi * 32 + lane, g1, w);
            double a = 0.0;
#pragma unroll
            for (int j = 0; j < E; ++j) a += static_cast<double>(w[j]);
            a = warp_sum(a);
            if (lane == 0 && wi < cnt) sh[wi] = a;
        } else if (!RES && sub == 32 && !s.wide) {  // four parts at a time: one round trip for them
            for (int k = wi; k < cnt; k += 4 * nw) {
                uint4 t[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int g = g0 + (k + u * nw) * 32 + lane;
                    t[u] = gran_fill<T>(__int_as_float(0xff800000));
                    if (g < g1) t[u] = gran_any<T>(s.t, g);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const double a = warp_sum(static_cast<double>(gran_weight<T, false>(s.scale, s.lp, 0.f, 0.f, t[u], t[u])));
                    if (lane == 0 && k + u * nw < cnt) sh[k + u * nw] = a;
                }
            }
        } else {
            for (int k = wi; k < cnt; k += nw) {
                double a = 0.0;
                for (int g = g0 + k * sub; g < min(g1, g0 + (k + 1) * sub); g += 32) {
                    load_weights<T, RES>(s, g + lane, min(g1, g0 + (k + 1) * sub), w);
#pragma unroll
                    for (int j = 0; j < E; ++j) a += static_cast<double>(w[j]);
                }
                a = warp_sum(a);
                if (lane == 0) sh[k] = a;
            }
        }
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nw * 32) : "memory");
        double before = 0.0, total, t;
        int own;
        if (fraction) own = pick_many<true, 2>(cnt, [&](int i) { return sh[i]; }, tau, &before, &total, &t);
        else own = pick_many<false, 2>(cnt, [&](int i) { return sh[i]; }, tau, &before, &total, &t);
        if (own < 0) return wi == 0 ? -1 : kNotMine;
        fraction = false;
        tau = t - before;
        if (leaf) return wi == own ? scan_weights<T>(s, g0 + own * 32, w, tau) : kNotMine;
        g0 += own * sub;
        g1 = min(g1, g0 + sub);
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nw * 32) : "memory");  // sh is written again
    }
}

// Sums of eight values over the warp with nine shuffles: on return lane 4 * k holds (in v[0]) the sum of the k-th.
__device__ __forceinline__ double warp_sum8(double (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 4, o = 16; w > 0; w >>= 1, o >>= 1) {
#pragma unroll
        for (int k = 0; k < w; ++k) {  // the lower half of the lanes goes on with the lower half of the values
            const bool up = (lane & o) != 0;
            const double give = up ? v[k] : v[k + w];
            v[k] = (up ? v[k + w] : v[k]) + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// A plain draw from the sums that the sweep's warps have left of a row (spans: reference in log2 units and sum, one per
// warp range, or of F pieces of it that are `piece` granules long): nw warps of a CTA, one of which gets the token (find_token).  -1: the row holds a NaN / +inf or has no weight.
// The first warp picks the span and, once all have summed its parts, the part and the token: picking in all warps was 40 % of
// the instructions of draft sampling, where every row is drawn from (256 bf16 rows, V = 128,256: 81 us, this way 73).
template <typename T>
__device__ __forceinline__ int draw_from_spans(const T* row, int V, float scale, const float2* spans, int n, int per_warp, float u,
                                               int wi, int nw, int bar, double* sh, DrawSrc* sh_src, int F = 1, int piece = 0) {
    const int lane = threadIdx.x & 31;
    if (wi == 0) {
        const int per = (n + 31) >> 5;
        float2 v[8];
        float R = -3.0e38f;
        bool bad = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = lane * per + i;
            v[i] = make_float2(-3.0e38f, 0.f);
            if (i < per && k < n && dbg_ok(spans + k, 8, DBG_WS_LOAD)) v[i] = __ldcg(spans + k);
            R = fmaxf(R, v[i].x);
            bad |= !(v[i].y < 3e38f);
        }
        R = warp_maxf(R);
        double before = 0.0, total, tau;
        const int own = pick_many<true, 8>(n, [&](int k) {
            const int i = k - lane * per;
            float2 x = v[0];
#pragma unroll
            for (int q = 1; q < 8; ++q) if (i == q) x = v[q];
            // The reference is the row's largest exponent but for its rounding, 2^6 at most below 2^31.  A span of less than 2^-100 then
            // has less than 2^-36 of the total and counts as empty: its elements, below 2^-126 each, may read as 0, so that a threshold
            // of 0 would find nothing in it.  From 2^31 on the reference may lie so far above the row that this is all the row has.
            const float f = ex2f(x.x - R), y = fabsf(x.x) < 0x1p31f && x.y * f < 0x1p-100f ? 0.f : x.y;
            return static_cast<double>(y) * static_cast<double>(f);
        }, static_cast<double>(u), &before, &total, &tau);
        const bool none = __any_sync(0xffffffffu, bad) || own < 0;
        if (lane == 0) {
            DrawSrc s = make_draw<T>(row, nullptr, V);
            set_norm(s, scale, static_cast<double>(R), 0.0);  // an fp32 value: exact whatever its size
            const int w = own / F, k = own - w * F, lo = w * per_warp, a = max(lo, s.t.whole_lo());
            s.r0 = none ? 0 : k > 0 ? a + k * piece : lo;
            s.r1 = none ? 0 : min(s.t.ng, k < F - 1 ? min(a + (k + 1) * piece, lo + per_warp) : lo + per_warp);
            s.tau = tau - before;
            *sh_src = s;
        }
    }
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nw * 32) : "memory");
    const int g0 = sh_src->r0, g1 = sh_src->r1;
    if (g1 <= g0) return wi == 0 ? -1 : kNotMine;
    if (g1 - g0 > 64 * 32) return find_token<T, false>(*sh_src, g0, g1, sh_src->tau, false, wi, nw, bar, sh);
    const int cnt = (g1 - g0 + 31) >> 5;  // parts of one granule per lane
    float w[16 / sizeof(T)];
    if (cnt <= nw) {  // one per warp: the warp that holds the token has its weights at hand
        load_weights<T, false, false>(*sh_src, g0 + wi * 32 + lane, g1, w);
        double a = 0.0;
#pragma unroll
        for (int j = 0; j < static_cast<int>(16 / sizeof(T)); ++j) a += static_cast<double>(w[j]);
        a = warp_sum(a);
        if (lane == 0) sh[wi] = a;
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nw * 32) : "memory");
        const double tau = sh_src->tau;
        double run = 0.0, before = 0.0;
        int own = -1;
        bool hit = false;
        for (int k = 0; k < cnt; ++k) {
            const double x = sh[k];
            if (x > 0.0 && !hit) {
                own = k;
                before = run;
                hit = run + x > tau;
            }
            run += x;
        }
        if (own < 0) return wi == 0 ? -1 : kNotMine;
        return wi == own ? scan_weights<T>(*sh_src, g0 + own * 32, w, tau - before) : kNotMine;
    }
    // part k by warp k % nw, eight at a time
    const float sc = sh_src->scale, lp = sh_src->lp;
    for (int k0 = wi; k0 < cnt; k0 += 8 * nw) {
        double a[8];
#pragma unroll
        for (int h = 0; h < 8; h += 4) {  // four loads in flight
            uint4 t[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int g = g0 + (k0 + (h + q) * nw) * 32 + lane;
                t[q] = gran_fill<T>(__int_as_float(0xff800000));
                if (g < g1) t[q] = gran_any<T>(sh_src->t, g);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) a[h + q] = static_cast<double>(gran_weight<T, false>(sc, lp, 0.f, 0.f, t[q], t[q]));
        }
        const double sum = warp_sum8(a);
        const int k = k0 + (lane >> 2) * nw;
        if ((lane & 3) == 0 && k < cnt) sh[k] = sum;
    }
    if (wi != 0) {
        asm volatile("bar.arrive %0, %1;" ::"r"(bar), "r"(nw * 32) : "memory");
        return kNotMine;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nw * 32) : "memory");
    double before = 0.0, total, tau;
    const int own = pick_many<false, 2>(cnt, [&](int i) { return sh[i]; }, sh_src->tau, &before, &total, &tau);
    if (own < 0) return -1;
    load_weights<T, false, false>(*sh_src, g0 + own * 32 + lane, g1, w);
    return scan_weights<T>(*sh_src, g0 + own * 32, w, tau - before);
}

// ----------------------------------------------------------------------------------------
// One CTA's share of the draw from the residual of batch row b at stop position n.
// The last of the row's CTAs to arrive locates the token.  A residual whose total mass is below 1e-6 cannot be told from
// rounding noise and is treated as empty (p == q at the stop position): the token is then drawn from p.
// ----------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void resample_row(const KParams& P, const int b, const int n, const int share) {
    __shared__ int sh_flag;
    __shared__ DrawSrc sh_src;
    __shared__ double sh_sum[64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T* trow = static_cast<const T*>(P.t) + static_cast<long long>(b) * P.tsb + static_cast<long long>(n) * P.tsp;
    const T* drow = static_cast<const T*>(P.d) + static_cast<long long>(b) * P.dsb + static_cast<long long>(n) * P.dsp;
    const DrawSrc src = make_draw<T>(trow, drow, P.V);
    double* dsum = P.dsum + static_cast<long long>(b) * (kMaxShares * kWarps);
    const int span = share * kWarps + warp;
    {
        const int g0 = span * P.draw_pw;
        const double w = warp_weights<T, true, false>(src, g0, min(src.t.ng, g0 + P.draw_pw), NormOfRecord{P.info + b}).x;
        if (lane == 0) SPECKV_ST(dsum[span], w);
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

    // ---- last CTA of the row: locate the threshold (every warp picks the span, redundantly) ----
    const RowInfo ri = row_info_load(P.info + b);
    if (threadIdx.x == 0) {
        DrawSrc c = make_draw<T>(trow, drow, P.V);
        set_norm(c, ri.scale, ri.lse2_p, ri.lse2_q);
        sh_src = c;
    }
    double before = 0.0, total, tau;
    const int own = pick_many<true, 8>(P.R * kWarps, [&](int k) { return dbg_ok(dsum + k, 8, DBG_WS_LOAD) ? __ldcg(dsum + k) : 0.0; },
                                       static_cast<double>(ri.u2), &before, &total, &tau);
    __syncthreads();
    const int ng = sh_src.t.ng;
    int tok;
    if (total > 1e-6)
        tok = find_token<T, true>(sh_src, own * P.draw_pw, min(ng, (own + 1) * P.draw_pw), tau - before, false, warp, kWarps, 1, sh_sum);
    else
        tok = find_token<T, false>(sh_src, 0, ng, static_cast<double>(ri.u2), true, warp, kWarps, 1, sh_sum);
    if (tok != kNotMine && lane == 0) P.out_tok[static_cast<long long>(b) * (P.G + 1) + n] = max(tok, 0);
}

constexpr int kDirectSums = kMaxShares * kWarps / 2;  // span sums of a direct grid's draw, 16 bytes each in the place of the other draws' 8
// The CTAs of one batch row's draw from a residual.  All wait for the row's record and sum their spans; the last one in the grid, which
// waits for CTAs in front of it only, picks the span and finds the token.  (As resample_row, with the record and the sums passed on
// as words that tell by themselves that they are there: no counter, no fence, nothing read twice.  From the record to the token
// 6.6 -> 4.9 us, 16 bf16 rows, V = 128,256.)
template <typename T>
__device__ __forceinline__ void direct_draw(const KParams& P, const int d, DrawSrc* sh_src, double* sh_sum) {
    __shared__ int sh_go;
    __shared__ RowInfo sh_info;
    const int b = d / P.R, share = d - b * P.R, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Gave up: the mark goes where the row epilogue, should it come after all, finds it (finish_verify); if it has been there, the
    // row is marked here.
    auto give_up = [&]() {
        const int old = atomicOr(P.rdone + b, kSlotTimeout);
        if ((old & kSlotDone) && ((old >> 24) & 1)) {
            if (P.status) atomicOr(P.status + b, 16);
            P.out_tok[static_cast<long long>(b) * (P.G + 1) + ((old >> 25) & 15)] = -1;
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
    double2* sums = reinterpret_cast<double2*>(P.dsum) + static_cast<long long>(b) * kDirectSums;
    {
        const int span = share * kWarps + warp, g0 = span * P.draw_pw;
        const double w = warp_weights<T, true, false>(*sh_src, g0, min(sh_src->t.ng, g0 + P.draw_pw), NormReady{sh_src}).x;
        if (lane == 0) span_publish(sums + span, w);
    }
    if (share != P.R - 1) return;
    if (warp == 0) {
        constexpr int MOST = kDirectSums / 32;
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
__device__ __forceinline__ void resample_body(const KParams& P, const int bid) {
    __shared__ int sh_wait;
    // one-dimensional grid, R consecutive CTAs per draw
    const int g = bid / P.R, share = bid - g * P.R;
    // Group g takes the row in slot g of the draw queue.  Every sweep CTA is resident or done before the first CTA that
    // draws starts, so all slots get filled and the wait ends; it is bounded all the same.
    if (threadIdx.x == 0) sh_wait = row_done_wait(P.rdone + g, P.wait_limit);
    __syncthreads();
    const int v = sh_wait;
    if (!v) {
        // Gave up.  The mark goes on the slot: if the row epilogue has already written the
        // status (the slot was filled just after the last poll) the bit is added here, otherwise the
        // epilogue finds the mark when it takes the slot and adds the bit itself.
        if (threadIdx.x == 0 && share == 0) {
            const int old = atomicOr(P.rdone + g, kSlotTimeout);
            if ((old & kSlotDone) && P.status) atomicOr(P.status + (old & 0xffffff), 16);
        }
        return;
    }
    if ((v >> 24) & 1) resample_row<T>(P, v & 0xffffff, (v >> 25) & 15, share);  // else: nothing to draw for that row
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 4) resample_kernel(const __grid_constant__ KParams P) {
    resample_body<T>(P, static_cast<int>(blockIdx.x));
}

}  // namespace speckv
