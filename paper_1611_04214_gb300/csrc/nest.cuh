// Two line inverses in a row along one axis, H_c H_c, with the line held on the chip between them
// (registers and shared memory), so that a pass of the 2D iteration reads and writes every field
// once.  A thread owns a chunk of K consecutive nodes; chunks are scanned as in
// sweep_common.cuh (zero-start segments, FP64 boundary solve per line, second pass from the
// carries).
//
// Lines whose length is not a multiple of K are cut into chunks of K and K - 1 nodes (the K-node ones
// first).
#pragma once

#include "nest_shape.h"
#include "sweep_common.cuh"

namespace molt {

// ---- a register value: two FP32 lines (or half lines) packed, or one scalar ----
template <typename T, int W> struct NestVec;
template <> struct NestVec<float, 2> : Lanes<2> {
    using T = float;
    static constexpr int W = 2;
    static __device__ __forceinline__ V mul(V a, V b) {
        V r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
        return r;
    }
    static __device__ __forceinline__ V sub(V a, V b) { return fma(b, splat(-1.0f), a); }
    static __device__ __forceinline__ V pair(float lo, float hi) { return pack(lo, hi); }
    static __device__ __forceinline__ V swap(V a) { return pack(get(a, 1), get(a, 0)); }
    // halves chosen by a mask: bit 0 = low, bit 1 = high half taken from b
    static __device__ __forceinline__ V blend(V a, V b, int mask) {
        return pack((mask & 1) ? get(b, 0) : get(a, 0), (mask & 2) ? get(b, 1) : get(a, 1));
    }
};
template <typename S> struct NestVec<S, 1> {
    using T = S;
    using V = S;
    static constexpr int W = 1;
    static __device__ __forceinline__ V splat(T a) { return a; }
    static __device__ __forceinline__ V zero() { return T(0); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return ::fma(a, b, c); }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
    static __device__ __forceinline__ V sub(V a, V b) { return a - b; }
    static __device__ __forceinline__ T get(V a, int) { return a; }
    static __device__ __forceinline__ V pair(T lo, T) { return lo; }
    static __device__ __forceinline__ V swap(V a) { return a; }
    static __device__ __forceinline__ V blend(V a, V b, int mask) { return (mask & 1) ? b : a; }
};

// Coefficients of one inverse in the form the chunks are evaluated.  With x the window of a chunk
// (x[i] = node start - M/2 + i), wl the interior stencil of J^L (J^R is its mirror image),
//   alpha = sum_o wl_o d^o,  beta_i = sum_{o >= i} wl_o d^(o-i),  gamma_m = beta_m + beta_{M-m} (beta_0 := 0 here),
// the recurrences of Eq. IL / IR give
//   P^L_k = Q_k + sum_{i=1..M} beta_i x[k+i],        Q_k = d Q_{k-1} + alpha x[k],
//   P^R_k = R_k + sum_{i=1..M} beta_i x[k+M-i],      R_k = d R_{k+1} + alpha x[k+M],
//   out_k = Q_k + R_k + sum_m gamma_m x[k+m]         (gamma symmetric):
// two one-term recurrences and one symmetric stencil instead of two full stencils.
template <typename V>
struct NestCoef {
    V alpha, beta[kMaxM + 1], gamma[kMaxM / 2 + 1];
};
// Ghost values of the M/2 nodes beyond a wall: the polynomial of degree M through the first M + 1
// nodes of the line.  Every centred stencil near the wall then interpolates that polynomial, which is
// the shifted wall stencil (Sec. 3.2 reading).
template <int M>
__host__ __device__ constexpr double nest_ghost_weight(int g, int o) {
    double c = 1.0;
    for (int k = 0; k <= M; ++k)
        if (k != o) c = c * (-g - k) / (o - k);
    return c;
}

// What a thread's chunk is along its line.
struct NestChunk {
    int cnt;        // nodes (0: none)
    int mA, mB;     // halves at the left / right wall (0 away from walls and on periodic lines)
};

template <class N, int M, int CNT, int KM>
__device__ __forceinline__ void nest_ghosts(const NestChunk& c, typename N::V (&x)[KM]) {
    using V = typename N::V;
    using T = typename N::T;
    constexpr int H = M / 2;
    if (c.mA) {
#pragma unroll
        for (int g = 1; g <= H; ++g) {
            V e = N::mul(N::splat(T(nest_ghost_weight<M>(g, 0))), x[H]);
#pragma unroll
            for (int o = 1; o <= M; ++o) e = N::fma(N::splat(T(nest_ghost_weight<M>(g, o))), x[H + o], e);
            x[H - g] = N::blend(x[H - g], e, c.mA);
        }
    }
    if (c.mB) {
#pragma unroll
        for (int g = 1; g <= H; ++g) {
            V e = N::mul(N::splat(T(nest_ghost_weight<M>(g, 0))), x[H + CNT - 1]);
#pragma unroll
            for (int o = 1; o <= M; ++o) e = N::fma(N::splat(T(nest_ghost_weight<M>(g, o))), x[H + CNT - 1 - o], e);
            x[H + CNT - 1 + g] = N::blend(x[H + CNT - 1 + g], e, c.mB);
        }
    }
}

// R_k + sum_m gamma_m x[k+m]; Q_k is added last, so that the sum rounds at the size of one half of the output (Q and R
// are about half of it each) and not of all of it.
template <class N, int M, int KM>
__device__ __forceinline__ typename N::V nest_stencil(const NestCoef<typename N::V>& w, const typename N::V (&x)[KM], int k,
                                                      typename N::V r) {
    constexpr int H = M / 2;
#pragma unroll
    for (int m = 0; m < H; ++m) r = N::fma(w.gamma[m], N::add(x[k + m], x[k + M - m]), r);
    return N::fma(w.gamma[H], x[k + H], r);
}

// Zero-start aggregates of a chunk of CNT nodes: P^L at its last node and P^R at its first one with
// nothing entering (I^L_0 = 0 and I^R_N = 0 at walls).  pw = d^(CNT-1).
template <class N, int M, int CNT, int KM>
__device__ __forceinline__ void nest_agg(const NestCoef<typename N::V>& w, typename N::T d, typename N::T pw,
                                         const NestChunk& c, const typename N::V (&x)[KM], typename N::V& aL,
                                         typename N::V& aR) {
    using V = typename N::V;
    const V dv = N::splat(d), nd = N::splat(-d), pv = N::splat(pw);
    V s = x[0], r = x[CNT - 1 + M];
#pragma unroll
    for (int k = 1; k < CNT; ++k) {
        s = N::fma(dv, s, x[k]);
        r = N::fma(dv, r, x[CNT - 1 - k + M]);
    }
    // (the large term last: the sums before it round at the size of the weights)
    V a = N::mul(w.beta[1], x[CNT]), b = N::mul(w.beta[1], x[M - 1]);
    V ka = N::mul(w.beta[1], x[0]), kb = N::mul(w.beta[1], x[CNT - 1 + M]);
#pragma unroll
    for (int i = 2; i <= M; ++i) {
        a = N::fma(w.beta[i], x[CNT - 1 + i], a);
        b = N::fma(w.beta[i], x[M - i], b);
        ka = N::fma(w.beta[i], x[i - 1], ka);
        kb = N::fma(w.beta[i], x[CNT - i + M], kb);
    }
    a = N::fma(w.alpha, s, a);
    b = N::fma(w.alpha, r, b);
    ka = N::mul(nd, ka);
    kb = N::mul(nd, kb);
    if (c.mA | c.mB) {
        V wa = N::mul(w.alpha, x[0]), wb = N::mul(w.alpha, x[CNT - 1 + M]);
#pragma unroll
        for (int i = 1; i <= M; ++i) {
            wa = N::fma(w.beta[i], x[i], wa);
            wb = N::fma(w.beta[i], x[CNT - 1 + M - i], wb);
        }
        ka = N::blend(ka, N::sub(N::zero(), wa), c.mA);
        kb = N::blend(kb, N::sub(N::zero(), wb), c.mB);
    }
    aL = N::fma(pv, ka, a);
    aR = N::fma(pv, kb, b);
}

// Outputs of a chunk of CNT nodes from the carries entering it; at a wall P^L_0 = end(0) = B_a and
// P^R_N = end(1) = B_b instead.
template <class N, int K, int M, int CNT, int KM, class End>
__device__ __forceinline__ void nest_finish(const NestCoef<typename N::V>& w, typename N::T d, const NestChunk& c,
                                            const typename N::V (&x)[KM], typename N::V cL, typename N::V cR,
                                            End end, typename N::V (&out)[K]) {
    using V = typename N::V;
    constexpr int H = M / 2;
    const V dv = N::splat(d), m1 = N::splat(typename N::T(-1));
    V ka = N::mul(w.beta[1], x[0]), kb = N::mul(w.beta[1], x[CNT - 1 + M]);
#pragma unroll
    for (int i = 2; i <= M; ++i) {
        ka = N::fma(w.beta[i], x[i - 1], ka);
        kb = N::fma(w.beta[i], x[CNT - i + M], kb);
    }
    V q = N::fma(dv, N::fma(m1, ka, cL), N::mul(w.alpha, x[0]));
    V r = N::fma(dv, N::fma(m1, kb, cR), N::mul(w.alpha, x[CNT - 1 + M]));
    if (c.mA | c.mB) {
        V wa = end(0), wb = end(1);
#pragma unroll
        for (int i = 1; i <= M; ++i) {
            wa = N::fma(N::mul(m1, w.beta[i]), x[i], wa);
            wb = N::fma(N::mul(m1, w.beta[i]), x[CNT - 1 + M - i], wb);
        }
        q = N::blend(q, wa, c.mA);
        r = N::blend(r, wb, c.mB);
    }
    out[CNT - 1] = r;
#pragma unroll
    for (int k = CNT - 2; k >= 0; --k) {
        r = N::fma(dv, r, N::mul(w.alpha, x[k + M]));
        out[k] = r;
    }
#pragma unroll
    for (int k = 0; k < CNT; ++k) {
        if (k > 0) q = N::fma(dv, q, N::mul(w.alpha, x[k]));
        out[k] = N::add(nest_stencil<N, M>(w, x, k, out[k]), q);
    }
}

// The same with the shifted wall stencils themselves (chunks of CNT > M nodes): the local integrals of the M/2 nodes
// next to a wall are formed directly (wlA .. wrB) and the two-recurrence form starts behind them, where
// no stencil leaves the line.
template <class N, int M, int CNT, int KM>
struct NestWall {
    using V = typename N::V;
    using T = typename N::T;
    static constexpr int H = M / 2;
    const LineParams<T>& lp;
    const NestCoef<V>& w;
    const V (&x)[KM];
    __device__ __forceinline__ V sum(const T (&c)[kMaxStencil], int first) const {
        V a = N::mul(N::splat(c[0]), x[first]);
#pragma unroll
        for (int o = 1; o <= M; ++o) a = N::fma(N::splat(c[o]), x[first + o], a);
        return a;
    }
    // left wall: J^L_k (k = 1..H-1), J^R_k (k = 0..H-1); right wall: of node CNT-H+j
    __device__ __forceinline__ V jla(int k) const { return sum(lp.wlA[k - 1], H); }
    __device__ __forceinline__ V jra(int k) const { return sum(lp.wrA[k], H); }
    __device__ __forceinline__ V jlb(int j) const { return sum(lp.wlB[j], H + CNT - 1 - M); }
    __device__ __forceinline__ V jrb(int j) const { return sum(lp.wrB[j], H + CNT - 1 - M); }
    // P^L_k - Q_k and P^R_k - R_k
    __device__ __forceinline__ V bl(int k) const {
        V a = N::mul(w.beta[1], x[k + 1]);
#pragma unroll
        for (int i = 2; i <= M; ++i) a = N::fma(w.beta[i], x[k + i], a);
        return a;
    }
    __device__ __forceinline__ V br(int k) const {
        V a = N::mul(w.beta[1], x[k + M - 1]);
#pragma unroll
        for (int i = 2; i <= M; ++i) a = N::fma(w.beta[i], x[k + M - i], a);
        return a;
    }
};

// As nest_agg, walls by their shifted stencils.
template <class N, int M, int CNT, int KM>
__device__ __forceinline__ void nest_agg_wall(const LineParams<typename N::T>& lp, const NestCoef<typename N::V>& w,
                                         typename N::T pw, const NestChunk& c, const typename N::V (&x)[KM],
                                         typename N::V& aL, typename N::V& aR) {
    using V = typename N::V;
    constexpr int H = M / 2;
    const V dv = N::splat(lp.d), nd = N::splat(-lp.d), pv = N::splat(pw);
    V s = x[0], r = x[CNT - 1 + M];
#pragma unroll
    for (int k = 1; k < CNT; ++k) {
        s = N::fma(dv, s, x[k]);
        r = N::fma(dv, r, x[CNT - 1 - k + M]);
    }
    // (the large term last: the sums before it round at the size of the weights)
    V a = N::mul(w.beta[1], x[CNT]), b = N::mul(w.beta[1], x[M - 1]);
    V ka = N::mul(w.beta[1], x[0]), kb = N::mul(w.beta[1], x[CNT - 1 + M]);
#pragma unroll
    for (int i = 2; i <= M; ++i) {
        a = N::fma(w.beta[i], x[CNT - 1 + i], a);
        b = N::fma(w.beta[i], x[M - i], b);
        ka = N::fma(w.beta[i], x[i - 1], ka);
        kb = N::fma(w.beta[i], x[CNT - i + M], kb);
    }
    a = N::fma(w.alpha, s, a);
    b = N::fma(w.alpha, r, b);
    aL = N::fma(pv, N::mul(nd, ka), a);
    aR = N::fma(pv, N::mul(nd, kb), b);
    if (c.mA | c.mB) {
        const NestWall<N, M, CNT, KM> wl{lp, w, x};
        const V m1 = N::splat(typename N::T(-1));
        if (c.mA) {
            V p = N::zero(), q = N::mul(nd, kb);   // kb: R just past the chunk is -kb
#pragma unroll
            for (int k = 1; k < H; ++k) p = N::fma(dv, p, wl.jla(k));
            p = N::fma(m1, wl.bl(H - 1), p);
#pragma unroll
            for (int k = H; k < CNT; ++k) p = N::fma(dv, p, N::mul(w.alpha, x[k]));
            q = N::add(q, N::mul(w.alpha, x[CNT - 1 + M]));
#pragma unroll
            for (int k = CNT - 2; k >= H; --k) q = N::fma(dv, q, N::mul(w.alpha, x[k + M]));
            q = N::add(q, wl.br(H));
#pragma unroll
            for (int k = H - 1; k >= 0; --k) q = N::fma(dv, q, wl.jra(k));
            aL = N::blend(aL, N::add(p, wl.bl(CNT - 1)), c.mA);
            aR = N::blend(aR, q, c.mA);
        }
        if (c.mB) {
            V p = N::mul(nd, ka), q = N::zero();   // Q just before the chunk is -ka
#pragma unroll
            for (int k = CNT - 2; k >= CNT - H; --k) q = N::fma(dv, q, wl.jrb(k - (CNT - H)));
            q = N::fma(m1, wl.br(CNT - H), q);
#pragma unroll
            for (int k = CNT - H - 1; k >= 0; --k) q = N::fma(dv, q, N::mul(w.alpha, x[k + M]));
            p = N::add(p, N::mul(w.alpha, x[0]));
#pragma unroll
            for (int k = 1; k < CNT - H; ++k) p = N::fma(dv, p, N::mul(w.alpha, x[k]));
            p = N::add(p, wl.bl(CNT - 1 - H));
#pragma unroll
            for (int k = CNT - H; k < CNT; ++k) p = N::fma(dv, p, wl.jlb(k - (CNT - H)));
            aL = N::blend(aL, p, c.mB);
            aR = N::blend(aR, N::add(q, wl.br(0)), c.mB);
        }
    }
}

// As nest_finish, walls by their shifted stencils.
template <class N, int K, int M, int CNT, int KM, class End>
__device__ __forceinline__ void nest_finish_wall(const LineParams<typename N::T>& lp, const NestCoef<typename N::V>& w,
                                            const NestChunk& c, const typename N::V (&x)[KM], typename N::V cL,
                                            typename N::V cR, End end, typename N::V (&out)[K]) {
    using V = typename N::V;
    constexpr int H = M / 2;
    static_assert(H > 1, "(the right wall's start is a node before the last)");
    const V dv = N::splat(lp.d), m1 = N::splat(typename N::T(-1));
    const NestWall<N, M, CNT, KM> wl{lp, w, x};
    V ka = N::mul(w.beta[1], x[0]), kb = N::mul(w.beta[1], x[CNT - 1 + M]);
#pragma unroll
    for (int i = 2; i <= M; ++i) {
        ka = N::fma(w.beta[i], x[i - 1], ka);
        kb = N::fma(w.beta[i], x[CNT - i + M], kb);
    }
    V q = N::fma(dv, N::fma(m1, ka, cL), N::mul(w.alpha, x[0]));
    V r = N::fma(dv, N::fma(m1, kb, cR), N::mul(w.alpha, x[CNT - 1 + M]));
    V pb[H];                      // right wall: P^R of the last H nodes
#pragma unroll
    for (int j = 0; j < H; ++j) pb[j] = N::zero();
    V rs = N::zero();             // ... and R of node CNT - H
    if (c.mB) {
        pb[H - 1] = end(1);
#pragma unroll
        for (int j = H - 2; j >= 0; --j) pb[j] = N::fma(dv, pb[j + 1], wl.jrb(j));
        rs = N::fma(m1, wl.br(CNT - H), pb[0]);
    }
    out[CNT - 1] = r;
#pragma unroll
    for (int k = CNT - 2; k >= 0; --k) {
        r = N::fma(dv, r, N::mul(w.alpha, x[k + M]));
        if (k == CNT - H && c.mB) r = N::blend(r, rs, c.mB);
        out[k] = r;
    }
    V pa[H], qs = N::zero();      // left wall: the first H outputs, Q of node H - 1
#pragma unroll
    for (int j = 0; j < H; ++j) pa[j] = N::zero();
    if (c.mA) {
        V p = N::add(out[H], wl.br(H));
#pragma unroll
        for (int k = H - 1; k >= 0; --k) {
            p = N::fma(dv, p, wl.jra(k));
            pa[k] = p;
        }
        p = end(0);
        pa[0] = N::add(pa[0], p);
#pragma unroll
        for (int k = 1; k < H; ++k) {
            p = N::fma(dv, p, wl.jla(k));
            pa[k] = N::add(pa[k], p);
        }
        qs = N::fma(m1, wl.bl(H - 1), p);
    }
    V ql = N::zero();             // Q of node CNT - 1 - H
#pragma unroll
    for (int k = 0; k < CNT; ++k) {
        if (k > 0) q = N::fma(dv, q, N::mul(w.alpha, x[k]));
        if (k == H - 1 && c.mA) q = N::blend(q, qs, c.mA);
        if (k == CNT - 1 - H) ql = q;
        out[k] = N::add(nest_stencil<N, M>(w, x, k, out[k]), q);
    }
    if (c.mA) {
#pragma unroll
        for (int k = 0; k < H; ++k) out[k] = N::blend(out[k], pa[k], c.mA);
    }
    if (c.mB) {
        V p = N::add(ql, wl.bl(CNT - 1 - H));
#pragma unroll
        for (int j = 0; j < H; ++j) {
            p = N::fma(dv, p, wl.jlb(j));
            out[CNT - H + j] = N::blend(out[CNT - H + j], N::add(pb[j], p), c.mB);
        }
    }
}

// Walls by ghost values or by shifted stencils.  Sixth order's ghosts weigh the first nodes by up to 140, which on rough data
// costs FP32 two bits of the nodes beside a wall (1024^2 Neumann, two solves: largest error 3.5e-6 of the field's largest value
// with ghosts, 7.1e-7 with the stencils, 8.0e-7 by single sweeps); fourth order's (up to 10) cost nothing
// measurable (6.8e-7, 6.5e-7, 7.3e-7), and in FP64 neither does (256^2, M = 6: 5.8e-14, 5.3e-14, 5.4e-14).  The stencils are
// work for the warps that hold a wall, which are all of them on short FP64 lines: 256^2 FP64, M = 6, 135 us an
// iteration, with ghosts 102.
template <class N, int M> inline constexpr bool kNestGhosts = M <= 4 || sizeof(typename N::T) == 8;

// The powers d^(K-1) and d^(K-2): what a value decays by over a chunk of K or K - 1 nodes, one node less.
template <typename T> struct NestPow { T full, less; };

template <class N, int K, int M, bool RAG, int KM>
__device__ __forceinline__ void nest_chunk_agg(const LineParams<typename N::T>& lp, const NestCoef<typename N::V>& w,
                                               const NestPow<typename N::T>& p, const NestChunk& c,
                                               typename N::V (&x)[KM], typename N::V& aL, typename N::V& aR) {
    if constexpr (kNestGhosts<N, M>) {
        if (!RAG || c.cnt == K) {
            nest_ghosts<N, M, K>(c, x);
            nest_agg<N, M, K>(w, lp.d, p.full, c, x, aL, aR);
        } else {
            nest_ghosts<N, M, K - 1>(c, x);
            nest_agg<N, M, K - 1>(w, lp.d, p.less, c, x, aL, aR);
        }
    } else {
        if (!RAG || c.cnt == K) nest_agg_wall<N, M, K>(lp, w, p.full, c, x, aL, aR);
        else nest_agg_wall<N, M, K - 1>(lp, w, p.less, c, x, aL, aR);
    }
    if (c.cnt == 0) aL = aR = N::zero();
}

// end(0), end(1): the boundary values of the line, asked for at walls only.
template <class N, int K, int M, bool RAG, int KM, class End>
__device__ __forceinline__ void nest_chunk_finish(const LineParams<typename N::T>& lp, const NestCoef<typename N::V>& w,
                                                  const NestChunk& c, const typename N::V (&x)[KM], typename N::V cL,
                                                  typename N::V cR, End end, typename N::V (&out)[K]) {
    if constexpr (kNestGhosts<N, M>) {
        if (!RAG || c.cnt == K) nest_finish<N, K, M, K>(w, lp.d, c, x, cL, cR, end, out);
        else nest_finish<N, K, M, K - 1>(w, lp.d, c, x, cL, cR, end, out);
    } else {
        if (!RAG || c.cnt == K) nest_finish_wall<N, K, M, K>(lp, w, c, x, cL, cR, end, out);
        else nest_finish_wall<N, K, M, K - 1>(lp, w, c, x, cL, cR, end, out);
    }
}

// Halo values hl (before the chunk) and hr (after it) into the window x.
template <class N, int K, int M, bool RAG, int KM>
__device__ __forceinline__ void nest_set_halo(int cnt, const typename N::V (&hl)[M / 2], const typename N::V (&hr)[M / 2],
                                              typename N::V (&x)[KM]) {
    constexpr int H = M / 2;
#pragma unroll
    for (int h = 0; h < H; ++h) x[h] = hl[h];
    if (!RAG || cnt == K) {
#pragma unroll
        for (int h = 0; h < H; ++h) x[H + K + h] = hr[h];
    } else {
#pragma unroll
        for (int h = 0; h < H; ++h) x[H + K - 1 + h] = hr[h];
    }
}

template <class N>
__device__ __forceinline__ typename N::V shfl_up_v(typename N::V v, int delta, int width = 32) {
    return __shfl_up_sync(kFull, v, delta, width);
}
template <class N>
__device__ __forceinline__ typename N::V shfl_down_v(typename N::V v, int delta, int width = 32) {
    return __shfl_down_sync(kFull, v, delta, width);
}

// B_a, B_b (walls) or the carries X (periodic) of one line from I_0 = I^R_0 and I_N = I^L_N, in FP64.
template <typename T>
__device__ __forceinline__ void nest_boundary(const LineParams<T>& lp, T I0, T IN, T& xl, T& xr) {
    const double i0 = static_cast<double>(I0), in = static_cast<double>(IN);
    if (lp.bc == BC_PERIODIC) {
        xl = static_cast<T>(in * lp.inv1mmu);
        xr = static_cast<T>(i0 * lp.inv1mmu);
    } else {
        xl = static_cast<T>(lp.bAA * i0 + lp.bAB * in);
        xr = static_cast<T>(lp.bBA * i0 + lp.bBB * in);
    }
}

// ---- thread-block clusters ----
__device__ __forceinline__ void nest_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The 8-byte value at the address of `local` in the shared memory of block `rank` of the cluster.
__device__ __forceinline__ unsigned long long nest_ld_cluster(const void* local, int rank) {
    unsigned remote;
    unsigned long long v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote)
                 : "r"(static_cast<unsigned>(__cvta_generic_to_shared(local))), "r"(rank));
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(remote) : "memory");
    return v;
}
__device__ __forceinline__ double nest_from_bits(unsigned long long b, double) { return __longlong_as_double(static_cast<long long>(b)); }
__device__ __forceinline__ unsigned long long nest_from_bits(unsigned long long b, unsigned long long) { return b; }

// =========================================================================================
// Columns.  A block owns `slots` chunks of 2^lcp column values (8 bytes each: two FP32 columns or one FP64
// column), thread = slot * values + value; the blocks of a strip of columns form a cluster along y and
// exchange their segments and chunk edges through distributed shared memory.
//   scalar / vector pass:  s = H w, b = H G, t = H s, a = H b (G = the lagged term),
//       A = beta (2a - b) - w + 2s - t,  B = -beta a - 2 (s - t),  E = Y - t,
//     the y part of the iteration whose x part is w + E + H (B + H A) (solver.cpp);
//   3D z pass:  outputs a3 = t, b3 = -2s + 4t - beta a, c3 = -w + 4s - 4t + beta (3a - b);
//   copy: out = H H in, or H in.
// Bound: issue slots and the latency of the scan's barriers (1.5 to 1.9 of 4 instructions a cycle, 16 warps a SM), not
// memory: 4096^2 Neumann FP32 198 us = 1700 GB/s of its 20 B a point, the row pass 80 us.  Two blocks a SM with 128
// registers, chunks of K = 8: 4096^2 Neumann FP32 276 us an iteration, vector model 593, 2048^2 78, 1001 x 777 37;
// three blocks at 80 registers spill and take 300, 674, 87 and 40 (M = 6, 4096^2: 298 against 337).  The copy of up
// to fourth order fits 80 registers: its three blocks give 250 us for the right side against 267.  K = 16 needs
// 121 KB a block for the arrays below, one block a SM.  32-byte row segments (4 values) let one block hold 512 nodes.
template <typename T>
struct NestColArgs {
    const T* in0;
    const T* in1;     // vector model: the second component; 3D y pass: b
    const T* in2;     // 3D y pass: c
    const T* Y;
    const T* U;       // sixth-order pass: u
    T* o0;
    T* o1;
    T* o2;
    int ld;           // distance of two nodes of a column
    long long slab;   // distance of two slabs of columns
    int ncols;        // columns of a slab
    int lcp;          // log2 of the values per strip (2..4)
    int slots;        // chunks per block
    int C;            // blocks per cluster
    NestCut cut;
    T g1, beta, vs;
    int comp;
    int single;       // copy: one inverse only
    NestPow<T> pw;
    int exact;        // the boundary solve is needed (see nest_col_scan)
};

// Shared words of the column scan.  Stream = (field, value, direction): stream 2 (q cp + value) + dir.
template <class N, int NF>
struct NestColShared {
    using V = typename N::V;
    using T = typename N::T;
    V tot[2][NF * 32];   // this block's total of each stream, per inverse (read by the cluster)
    V E[NF * 32];        // segment entering this block
    V X[NF * 32];        // line totals, then the boundary values
    T bd[16];            // decay of each block of the cluster
};

// What the column scan needs of a thread.
template <typename V, typename T>
struct NestColScan {
    int lcp, cpi, slot, slots, C, rank;
    int live;       // chunks of this block
    int full;       // ... of which the first `full` have K nodes
    T Df, Dl;       // decay of a chunk of K / K - 1 nodes
    V* ex;          // [stream][slots + 4]: chunk aggregates, then the segment entering each chunk
    const T* dec;   // per thread, nt apart: decay from the line's ends, and from this block's ends
    int nt;
    int exact;      // the boundary values need the FP64 solve (else e^{-nu N} is below any rounding)
};

// Carries entering every chunk (of the whole column) from the chunks' zero-start aggregates.  Every
// stream is scanned by 16 lanes (up to 4 chunks each); the totals of the cluster's blocks are read and scanned
// by the same lanes; one warp solves the boundary systems in FP64, skipped where mu = e^{-nu N} is so
// small (2^-64) that the solve only copies the totals.
// UNI: every chunk of the block has K nodes and 16 lanes hold equal numbers of them.
template <class N, int NF, bool UNI>
__device__ __forceinline__ void nest_col_scan(const LineParams<typename N::T>& lp,
                                              const NestColScan<typename N::V, typename N::T>& c,
                                              NestColShared<N, NF>& sh, int level) {
    using V = typename N::V;
    using T = typename N::T;
    __syncthreads();
    const int streams = (2 * NF) << c.lcp, pitch = c.slots + 4;
    const int p = threadIdx.x & 15;
    const int per = (c.slots + 15) >> 4;   // chunks per lane, 1..4
#pragma unroll 1
    for (int st = threadIdx.x >> 4; st < streams; st += c.nt >> 4) {
        const int dir = st & 1;
        // this lane's chunks in the order of the recurrence
        V* ex = c.ex + st * pitch + (dir ? c.slots - 1 - p * per : p * per);
        const int step = dir ? -1 : 1;
        V v[4];
        V e = N::zero();
        T D = T(1);
        auto decay = [&](int k) {
            if constexpr (UNI) return c.Df;
            const int i = p * per + k, sl = dir ? c.slots - 1 - i : i;
            return sl >= c.live ? T(1) : sl < c.full ? c.Df : c.Dl;
        };
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k < per && (UNI || p * per + k < c.slots)) {
                v[k] = ex[k * step];
                const T dk = decay(k);
                e = N::fma(e, N::splat(dk), v[k]);
                D *= dk;
            }
        }
        // inclusive scan over the 16 lanes, then the segment entering this lane
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const V u = shfl_up_v<N>(e, o, 16);
            if constexpr (UNI) {
                if (p >= o) e = N::fma(u, N::splat(D), e);
                D *= D;
            } else {
                const T du = __shfl_up_sync(kFull, D, o, 16);
                if (p >= o) {
                    e = N::fma(u, N::splat(D), e);
                    D *= du;
                }
            }
        }
        V in = shfl_up_v<N>(e, 1, 16);
        if (p == 0) in = N::zero();
        if (p == 15) {
            sh.tot[level][st] = e;
            sh.X[st] = e;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k < per && (UNI || p * per + k < c.slots)) {
                ex[k * step] = in;
                in = N::fma(in, N::splat(decay(k)), v[k]);
            }
        }
    }
    if (c.C > 1) {
        nest_cluster_sync();
#pragma unroll 1
        for (int st = threadIdx.x >> 4; st < streams; st += c.nt >> 4) {
            const int dir = st & 1, r = dir ? c.C - 1 - p : p;
            V e = N::zero();
            T D = T(1);
            if (p < c.C) {
                e = nest_from_bits(nest_ld_cluster(&sh.tot[level][st], r), V());
                D = sh.bd[r];
            }
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                const V u = shfl_up_v<N>(e, o, 16);
                const T du = __shfl_up_sync(kFull, D, o, 16);
                if (p >= o) {
                    e = N::fma(u, N::splat(D), e);
                    D *= du;
                }
            }
            V in = shfl_up_v<N>(e, 1, 16);
            if (p == 0) in = N::zero();
            if (r == c.rank) sh.E[st] = in;
            if (p == 15) sh.X[st] = e;
        }
    }
    __syncthreads();
    if (c.exact) {
        if (threadIdx.x < 32) {
            for (int t = threadIdx.x; t < (NF << c.lcp); t += 32) {
                const V in = sh.X[2 * t], i0 = sh.X[2 * t + 1];
                T xl[2], xr[2];
                nest_boundary<T>(lp, N::get(i0, 0), N::get(in, 0), xl[0], xr[0]);
                if constexpr (N::W == 2) nest_boundary<T>(lp, N::get(i0, 1), N::get(in, 1), xl[1], xr[1]);
                else xl[1] = xr[1] = T(0);
                sh.X[2 * t] = N::pair(xl[0], xl[1]);
                sh.X[2 * t + 1] = N::pair(xr[0], xr[1]);
            }
        }
        __syncthreads();
    }
}

// Boundary value (dir 0: B_a or the carry at the start, dir 1: B_b or the carry at the end) of a column.
template <class N, int NF>
__device__ __forceinline__ typename N::V nest_col_end(const LineParams<typename N::T>& lp,
                                                      const NestColScan<typename N::V, typename N::T>& c,
                                                      const NestColShared<N, NF>& sh, int q, int dir) {
    using T = typename N::T;
    const int t = 2 * ((q << c.lcp) + c.cpi);
    if (c.exact || lp.bc == BC_PERIODIC) return sh.X[t + dir];
    // walls with mu = 0: B_a = +- I_0, B_b = +- I_N
    return N::mul(N::splat(lp.bc == BC_DIRICHLET ? T(-1) : T(1)), sh.X[t + 1 - dir]);
}

// The carry entering this thread's chunk of field q from the start (dir 0) or the end (dir 1).
template <class N, int NF>
__device__ __forceinline__ typename N::V nest_col_carry(const LineParams<typename N::T>& lp,
                                                        const NestColScan<typename N::V, typename N::T>& c,
                                                        const NestColShared<N, NF>& sh, int q, int dir) {
    using V = typename N::V;
    const int st = 2 * ((q << c.lcp) + c.cpi) + dir;
    V e = N::fma(N::splat(c.dec[dir * c.nt]), nest_col_end<N, NF>(lp, c, sh, q, dir), c.ex[st * (c.slots + 4) + c.slot]);
    if (c.C > 1) e = N::fma(N::splat(c.dec[(2 + dir) * c.nt]), sh.E[st], e);
    return e;
}

// Geometry of a thread of the column kernels.
struct NestColGeo {
    int nt, cpi, slot, rank, ci, start;
    bool live;       // the chunk has nodes
    bool on;         // ... and its columns exist
    long long base;  // offset of node 0 of the (first) column
    bool both;       // the second column of the pair exists
};

template <class N, int K, bool RAG>
__device__ __forceinline__ NestColGeo nest_col_geo(const LineParams<typename N::T>& lp,
                                                   const NestColArgs<typename N::T>& a, NestChunk& ck) {
    NestColGeo g;
    const int tid = threadIdx.x;
    g.nt = blockDim.x;
    g.cpi = tid & ((1 << a.lcp) - 1);
    g.slot = tid >> a.lcp;
    g.rank = blockIdx.y;   // a cluster is the blocks of one strip
    g.ci = g.rank * a.slots + g.slot;
    g.live = g.slot < a.slots && g.ci < a.cut.nc;
    if (!g.live) g.ci = 0;
    ck.cnt = !g.live ? 0 : (!RAG || g.ci < a.cut.rem) ? K : K - 1;
    g.start = RAG ? g.ci * (K - 1) + min(g.ci, a.cut.rem) : g.ci * K;
    const int col = ((blockIdx.x << a.lcp) + g.cpi) * N::W;
    g.on = g.live && col < a.ncols;
    g.both = col + 1 < a.ncols;
    g.base = a.slab * blockIdx.z + (col < a.ncols ? col : 0);
    const bool walls = lp.bc != BC_PERIODIC;
    ck.mA = g.live && walls && g.ci == 0 ? (1 << N::W) - 1 : 0;
    ck.mB = g.live && walls && g.ci == a.cut.nc - 1 ? (1 << N::W) - 1 : 0;
    return g;
}

template <class N, int K, bool RAG, class SH>
__device__ __forceinline__ NestColScan<typename N::V, typename N::T> nest_col_scan_setup(
    const LineParams<typename N::T>& lp, const NestColArgs<typename N::T>& a, const NestColGeo& g, const NestChunk& ck,
    typename N::V* ex, typename N::T* dec, SH& sh) {
    using T = typename N::T;
    const int m = lp.bc == BC_PERIODIC ? 0 : 1;   // a wall's value starts one node later
    // first node of block r of the cluster
    auto first = [&](int r) {
        const int ch = min(r * a.slots, a.cut.nc);
        return RAG ? ch * (K - 1) + min(ch, a.cut.rem) : ch * K;
    };
    dec[0] = dev_exp(-lp.nu * T(max(g.start - m, 0)));
    dec[g.nt] = dev_exp(-lp.nu * T(max(lp.n - g.start - ck.cnt - m, 0)));
    if (a.C > 1) {
        dec[2 * g.nt] = dev_exp(-lp.nu * T(g.start - first(g.rank)));
        dec[3 * g.nt] = dev_exp(-lp.nu * T(first(g.rank + 1) - g.start - ck.cnt));
        if (threadIdx.x < a.C) sh.bd[threadIdx.x] = dev_exp(-lp.nu * T(first(threadIdx.x + 1) - first(threadIdx.x)));
    }
    const int c0 = g.rank * a.slots;
    return {a.lcp, g.cpi, g.slot, a.slots, a.C, g.rank, min(a.slots, a.cut.nc - c0), RAG ? a.cut.rem - c0 : a.slots,
            a.pw.full * lp.d, a.pw.less * lp.d, ex, dec, g.nt, a.exact};
}

// The column value (or pair) at offset i of a field; WIDE: column pairs are 8-byte aligned.
template <class N, bool WIDE>
__device__ __forceinline__ typename N::V nest_load(const typename N::T* p, bool both) {
    if constexpr (N::W == 2) {
        if constexpr (WIDE) return *reinterpret_cast<const unsigned long long*>(p);
        else return N::pair(p[0], both ? p[1] : 0.0f);
    } else {
        return *p;
    }
}
template <class N, bool WIDE>
__device__ __forceinline__ void nest_store(typename N::T* p, typename N::V v, bool both) {
    if constexpr (N::W == 2) {
        if constexpr (WIDE) {
            *reinterpret_cast<unsigned long long*>(p) = v;
        } else {
            p[0] = N::get(v, 0);
            if (both) p[1] = N::get(v, 1);
        }
    } else {
        *p = v;
    }
}

template <class N>
__device__ __forceinline__ typename N::V nest_cubic(typename N::V x, typename N::V g1) {
    return N::mul(x, N::fma(x, x, g1));
}
template <class N>
__device__ __forceinline__ typename N::V nest_vch(typename N::V x1, typename N::V x2, int comp, typename N::T s) {
    using T = typename N::T;
    const T lo = vch_lag<T>(N::get(x1, 0), N::get(x2, 0), comp, s);
    if constexpr (N::W == 2) return N::pair(lo, vch_lag<T>(N::get(x1, 1), N::get(x2, 1), comp, s));
    else return lo;
}

__device__ __forceinline__ void nest_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Window of a field's column chunk from global memory: rows wrapped on periodic columns, clamped at walls
// (ghosts replace those values, or no stencil uses them).
template <class N, int K, int M, bool RAG, bool WIDE, int KM>
__device__ __forceinline__ void nest_col_window(const typename N::T* f, const NestColGeo& g, int n, bool periodic, int ld,
                                                typename N::V (&x)[KM]) {
    constexpr int H = M / 2, SAFE = RAG ? K - 1 : K;   // rows that certainly belong to the chunk
    const typename N::T* base = f + g.base;
    auto far = [&](int p) {
        int r = p;
        if (p < 0) r = periodic ? p + n : 0;
        if (p >= n) r = periodic ? p - n : n - 1;
        return nest_load<N, WIDE>(base + static_cast<long long>(r) * ld, g.both);
    };
    const typename N::T* q = base + static_cast<long long>(g.start) * ld;
#pragma unroll
    for (int k = 0; k < SAFE; ++k) x[H + k] = nest_load<N, WIDE>(q + static_cast<long long>(ld) * k, g.both);
#pragma unroll
    for (int h = 0; h < H; ++h) x[h] = far(g.start - H + h);
#pragma unroll
    for (int k = SAFE; k < K + H; ++k) x[H + k] = far(g.start + k);
}

// Values a thread keeps in shared memory: NA arrays of K nodes and the ends of the second field's
// window, an odd number of 8-byte words (the lanes of a half warp then hit 16 different bank pairs).
template <int K, int M, int NA>
__host__ __device__ constexpr int nest_col_pitch() {
    return NA == 1 ? K + 1 : NA * K + M + 1;
}

template <int K, int M>
__host__ __device__ constexpr int nest_col3_pitch() { return 3 * K + 2 * M + 1; }

// FORM 0: every chunk of every block has K nodes and the blocks' chunks come in multiples of 16; 1: chunks
// of K nodes; 2: chunks of K and K - 1 nodes.
template <class N, int M, int FORM, bool WIDE, int MODE>
__global__ void __launch_bounds__(256, MODE == NEST_COPY && M <= 4 ? 3 : 2)
nest_cols_kernel(const __grid_constant__ LineParams<typename N::T> lp,
                 const __grid_constant__ NestCoef<typename N::V> w,
                 const __grid_constant__ NestColArgs<typename N::T> a) {
    using V = typename N::V;
    using T = typename N::T;
    constexpr bool RAG = FORM == 2;
    constexpr int K = kNestColK, H = M / 2, NF = MODE == NEST_COPY ? 1 : 2;
    // per thread in shared memory: arrays 0 = field 0 (w, then s), 1 = field 1 (G, then b), 2 = w, then
    // the ends of field 1's window
    extern __shared__ __align__(16) unsigned char nest_sm[];
    __shared__ NestColShared<N, NF> sh;
    NestChunk ck;
    const NestColGeo g = nest_col_geo<N, K, RAG>(lp, a, ck);
    const int nt = g.nt;
    const V* all = reinterpret_cast<const V*>(nest_sm);
    constexpr int NA = MODE == NEST_COPY ? 1 : 3, PITCH = nest_col_pitch<K, M, NA>();
    V* own = reinterpret_cast<V*>(nest_sm) + threadIdx.x * PITCH;
    auto arr = [&](int f, int k) -> V& { return own[f * K + k]; };
    auto end1 = [&](int h) -> V& { return own[NA * K + h]; };
    V x[K + M], hl[H], hr[H];   // hl, hr: the window's ends of field 0
    // ---- windows of the fields: nodes to shared memory, ends to hl / hr ----
    auto keep = [&](int q) {
#pragma unroll
        for (int k = 0; k < K; ++k) arr(q, k) = x[H + k];
    };
    auto keep_ends = [&](int q) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if (q == 0) {
                hl[h] = x[h];
                hr[h] = x[H + K + h];
            } else {
                end1(h) = x[h];
                end1(H + h) = x[H + K + h];
            }
        }
    };
    {
        const bool periodic = lp.bc == BC_PERIODIC;
        nest_col_window<N, K, M, RAG, WIDE>(a.in0, g, lp.n, periodic, a.ld, x);
        if constexpr (MODE == NEST_VCH) {
            V y[K + M];
            nest_col_window<N, K, M, RAG, WIDE>(a.in1, g, lp.n, periodic, a.ld, y);
#pragma unroll
            for (int i = 0; i < K + M; ++i) {
                const V gg = nest_vch<N>(x[i], y[i], a.comp, a.vs);
                if (a.comp) x[i] = y[i];
                y[i] = gg;
            }
            keep(0);
            keep_ends(0);
#pragma unroll
            for (int k = 0; k < K; ++k) arr(2, k) = x[H + k];
#pragma unroll
            for (int i = 0; i < K + M; ++i) x[i] = y[i];
            keep(1);
            keep_ends(1);
        } else {
            keep(0);
            keep_ends(0);
            if constexpr (NF == 2) {
                const V g1 = N::splat(a.g1);
#pragma unroll
                for (int k = 0; k < K; ++k) arr(2, k) = x[H + k];
#pragma unroll
                for (int i = 0; i < K + M; ++i) x[i] = nest_cubic<N>(x[i], g1);
                keep(1);
                keep_ends(1);
            }
        }
    }
    V* ex = reinterpret_cast<V*>(nest_sm) + PITCH * nt;
    T* dec = reinterpret_cast<T*>(ex + ((2 * NF) << a.lcp) * (a.slots + 4)) + threadIdx.x;
    const NestColScan<V, T> c = nest_col_scan_setup<N, K, RAG>(lp, a, g, ck, ex, dec, sh);

#pragma unroll 1
    for (int level = MODE == NEST_COPY && a.single ? 1 : 0; level < 2; ++level) {
        if (level == 1 && !(MODE == NEST_COPY && a.single)) {
            // edges of the chunks before and after this one (wrapped on periodic columns)
            if (a.C > 1) nest_cluster_sync();
            else __syncthreads();
            const int nc = a.cut.nc, last = (nc - 1) - a.slots * (a.C - 1);   // slot of the column's last chunk
            const bool pin = g.slot > 0, fin = g.slot < a.slots - 1 && g.ci < nc - 1;   // within this block
            // (threads without a chunk read this block's own memory)
            const int pr = pin || !g.live ? g.rank : g.rank > 0 ? g.rank - 1 : a.C - 1;
            const int fr = fin || !g.live ? g.rank : g.ci < nc - 1 ? g.rank + 1 : 0;
            const int ps = pin ? g.slot - 1 : g.rank > 0 ? a.slots - 1 : last, fs = fin ? g.slot + 1 : 0;
            const int pcnt = (!RAG || (g.ci > 0 ? g.ci - 1 : nc - 1) < a.cut.rem) ? K : K - 1;
            const V* pe = all + ((ps << a.lcp) + g.cpi) * PITCH + (pcnt - H);
            const V* fe = all + ((fs << a.lcp) + g.cpi) * PITCH;
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                V l[H], r[H];
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const V *lp_ = pe + q * K + h, *rp = fe + q * K + h;
                    l[h] = pr == g.rank ? *lp_ : nest_from_bits(nest_ld_cluster(lp_, pr), V());
                    r[h] = fr == g.rank ? *rp : nest_from_bits(nest_ld_cluster(rp, fr), V());
                }
                if (RAG && ck.cnt == K - 1) {
                    arr(q, K - 1) = r[0];
#pragma unroll
                    for (int h = 0; h + 1 < H; ++h) r[h] = r[h + 1];
                }
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    if (q == 0) {
                        hl[h] = l[h];
                        hr[h] = r[h];
                    } else {
                        end1(h) = l[h];
                        end1(H + h) = r[h];
                    }
                }
            }
        }
        auto window = [&](int q) {
#pragma unroll
            for (int k = 0; k < K; ++k) x[H + k] = arr(q, k);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                x[h] = q == 0 ? hl[h] : end1(h);
                x[H + K + h] = q == 0 ? hr[h] : end1(H + h);
            }
        };
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            window(q);
            V aL, aR;
            nest_chunk_agg<N, K, M, RAG>(lp, w, a.pw, ck, x, aL, aR);
            if (g.slot < a.slots) {
                V* e = ex + 2 * ((q << a.lcp) + g.cpi) * (a.slots + 4) + g.slot;
                e[0] = aL;
                e[a.slots + 4] = aR;
            }
            if (kNestGhosts<N, M> && (ck.mA | ck.mB)) {   // the ghosts
                keep_ends(q);
                if (RAG) arr(q, K - 1) = x[H + K - 1];
            }
        }
        // offset of the chunk in the fields (opaque: its addresses are not to be kept through the loop)
        long long o0 = g.base + static_cast<long long>(g.start) * a.ld;
        asm volatile("" : "+l"(o0));
        if constexpr (MODE == NEST_SCALAR || MODE == NEST_VCH) {
            // the right side is wanted right after the scan: fetch it into L2 meanwhile
            if (level == 1 && g.on && (g.cpi & 3) == 0) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (!RAG || k < K - 1 || ck.cnt == K)
                        nest_prefetch(a.Y + o0 + static_cast<long long>(a.ld) * k);
            }
        }
        nest_col_scan<N, NF, FORM == 0>(lp, c, sh, level);
        // no block leaves while another may still read its shared memory
        if (level == 1 && a.C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        V out[K];
        // the chunk's values to a field
        auto put = [&](T* f, auto value) {
            if (g.on) {
                T* p = f + o0;
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (!RAG || k < K - 1 || ck.cnt == K)
                        nest_store<N, WIDE>(p + static_cast<long long>(a.ld) * k, value(k), g.both);
            }
        };
        auto finish = [&](int q) {
            nest_chunk_finish<N, K, M, RAG>(lp, w, ck, x, nest_col_carry<N, NF>(lp, c, sh, q, 0),
                                               nest_col_carry<N, NF>(lp, c, sh, q, 1),
                                               [&](int dir) { return nest_col_end<N, NF>(lp, c, sh, q, dir); }, out);
        };
        window(0);
        finish(0);
        if (level == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) arr(0, k) = out[k];
        } else if constexpr (MODE == NEST_COPY) {
            put(a.o0, [&](int k) { return out[k]; });
        } else {
            const V m1 = N::splat(T(-1));
            if constexpr (MODE == NEST_Z3) put(a.o0, [&](int k) { return out[k]; });
            else if (g.on) {
                V y[K];
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (!RAG || k < K - 1 || ck.cnt == K)
                        y[k] = nest_load<N, WIDE>(a.Y + o0 + static_cast<long long>(a.ld) * k, g.both);
                put(a.o2, [&](int k) { return N::fma(m1, out[k], y[k]); });
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const V s = x[H + k], t = out[k];
                const V u = N::fma(m1, t, s);                          // s - t
                const V z = N::fma(m1, arr(2, k), s);                  // s - w
                if constexpr (MODE == NEST_Z3) {
                    arr(0, k) = N::mul(N::splat(T(2)), N::fma(m1, u, t));                 // -2s + 4t
                    arr(2, k) = N::fma(N::splat(T(3)), u, N::fma(m1, t, z));              // -w + 4s - 4t
                } else {
                    arr(0, k) = u;
                    arr(2, k) = N::add(z, u);                          // 2s - w - t
                }
            }
        }
        if constexpr (NF == 2) {
            window(1);
            finish(1);
            if (level == 0) {
#pragma unroll
                for (int k = 0; k < K; ++k) arr(1, k) = out[k];
            } else {
                const V be = N::splat(a.beta), nb = N::splat(-a.beta), m1 = N::splat(T(-1));
                const V m = N::splat(MODE == NEST_Z3 ? T(3) : T(2));
                put(MODE == NEST_Z3 ? a.o2 : a.o0,
                    [&](int k) { return N::fma(be, N::fma(m, out[k], N::mul(m1, x[H + k])), arr(2, k)); });
                put(a.o1, [&](int k) {
                    return N::fma(nb, out[k], MODE == NEST_Z3 ? arr(0, k) : N::mul(N::splat(T(-2)), arr(0, k)));
                });
            }
        }
    }
    if (a.C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// =========================================================================================
// 3D y pass (solver3d.cpp): from the z pass's a, b, c of one slab's columns
//   E = Y - H H a,   B = H (-2a + H b),   A = -a + H (b + H c),
// the data of the x pass w + E + H (B + H A).  Three fields through the two inverses of the kernel above; bound
// like it by issue slots and barriers (1.75 of 4 instructions a cycle): 256^3 FP32 182 us = 2580 GB/s of its 28 B a
// point; the z pass (16 B) 120 us, the x pass (20 B) 69 us.  The iteration takes 378 us; fifteen separate sweeps took 1817.
// Sixth-order model (fch2d.cpp), the same kernel with the fields p, q, r, u and z of nest_fch2_kernel:
//   E = z + H (u + H p),   B = u + H (2p - u + H q),   A = p + H (q + H r):
// 2048^2 FP32, M = 6: 97 us = 1380 GB/s of its 32 B a point, 1.07 of 4 instructions a cycle (clusters of four blocks).
// =========================================================================================
template <class N, int M, int FORM, bool WIDE, int MODE>
__global__ void __launch_bounds__(256, 2)
nest_cols3_kernel(const __grid_constant__ LineParams<typename N::T> lp,
                  const __grid_constant__ NestCoef<typename N::V> w,
                  const __grid_constant__ NestColArgs<typename N::T> a) {
    using V = typename N::V;
    using T = typename N::T;
    constexpr bool RAG = FORM == 2;
    constexpr int K = kNestColK, H = M / 2, NF = 3, PITCH = nest_col3_pitch<K, M>();
    // per thread: three arrays of the chunk's nodes, then the ends of the windows of fields 1 and 2
    extern __shared__ __align__(16) unsigned char nest_sm[];
    __shared__ NestColShared<N, NF> sh;
    NestChunk ck;
    const NestColGeo g = nest_col_geo<N, K, RAG>(lp, a, ck);
    const V* all = reinterpret_cast<const V*>(nest_sm);
    V* own = reinterpret_cast<V*>(nest_sm) + threadIdx.x * PITCH;
    auto arr = [&](int f, int k) -> V& { return own[f * K + k]; };
    auto end = [&](int q, int h) -> V& { return own[NF * K + (q - 1) * M + h]; };
    V x[K + M], hl[H], hr[H];   // hl, hr: the window's ends of field 0
    auto keep_ends = [&](int q, const V (&l)[H], const V (&r)[H]) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if (q == 0) {
                hl[h] = l[h];
                hr[h] = r[h];
            } else {
                end(q, h) = l[h];
                end(q, H + h) = r[h];
            }
        }
    };
    auto window_ends = [&](int q) {
        V l[H], r[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            l[h] = x[h];
            r[h] = x[H + K + h];
        }
        keep_ends(q, l, r);
    };
    auto window = [&](int q) {
#pragma unroll
        for (int k = 0; k < K; ++k) x[H + k] = arr(q, k);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            x[h] = q == 0 ? hl[h] : end(q, h);
            x[H + K + h] = q == 0 ? hr[h] : end(q, H + h);
        }
    };
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        nest_col_window<N, K, M, RAG, WIDE>(q == 0 ? a.in0 : q == 1 ? a.in1 : a.in2, g, lp.n, lp.bc == BC_PERIODIC, a.ld, x);
#pragma unroll
        for (int k = 0; k < K; ++k) arr(q, k) = x[H + k];
        window_ends(q);
    }
    V* ex = reinterpret_cast<V*>(nest_sm) + PITCH * g.nt;
    T* dec = reinterpret_cast<T*>(ex + ((2 * NF) << a.lcp) * (a.slots + 4)) + threadIdx.x;
    const NestColScan<V, T> c = nest_col_scan_setup<N, K, RAG>(lp, a, g, ck, ex, dec, sh);

#pragma unroll 1
    for (int level = 0; level < 2; ++level) {
        if (level == 1) {
            // edges of the chunks before and after this one (wrapped on periodic columns); as nest_cols_kernel
            if (a.C > 1) nest_cluster_sync();
            else __syncthreads();
            const int nc = a.cut.nc, last = (nc - 1) - a.slots * (a.C - 1);
            const bool pin = g.slot > 0, fin = g.slot < a.slots - 1 && g.ci < nc - 1;
            const int pr = pin || !g.live ? g.rank : g.rank > 0 ? g.rank - 1 : a.C - 1;
            const int fr = fin || !g.live ? g.rank : g.ci < nc - 1 ? g.rank + 1 : 0;
            const int ps = pin ? g.slot - 1 : g.rank > 0 ? a.slots - 1 : last, fs = fin ? g.slot + 1 : 0;
            const int pcnt = (!RAG || (g.ci > 0 ? g.ci - 1 : nc - 1) < a.cut.rem) ? K : K - 1;
            const V* pe = all + ((ps << a.lcp) + g.cpi) * PITCH + (pcnt - H);
            const V* fe = all + ((fs << a.lcp) + g.cpi) * PITCH;
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                V l[H], r[H];
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const V *lq = pe + q * K + h, *rq = fe + q * K + h;
                    l[h] = pr == g.rank ? *lq : nest_from_bits(nest_ld_cluster(lq, pr), V());
                    r[h] = fr == g.rank ? *rq : nest_from_bits(nest_ld_cluster(rq, fr), V());
                }
                if (RAG && ck.cnt == K - 1) {
                    arr(q, K - 1) = r[0];
#pragma unroll
                    for (int h = 0; h + 1 < H; ++h) r[h] = r[h + 1];
                }
                keep_ends(q, l, r);
            }
        }
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            window(q);
            V aL, aR;
            nest_chunk_agg<N, K, M, RAG>(lp, w, a.pw, ck, x, aL, aR);
            if (g.slot < a.slots) {
                V* e = ex + 2 * ((q << a.lcp) + g.cpi) * (a.slots + 4) + g.slot;
                e[0] = aL;
                e[a.slots + 4] = aR;
            }
            if (kNestGhosts<N, M> && (ck.mA | ck.mB)) {   // the ghosts
                window_ends(q);
                if (RAG) arr(q, K - 1) = x[H + K - 1];
            }
        }
        // offset of the chunk in the fields (opaque: its addresses are not to be kept through the loop)
        long long o0 = g.base + static_cast<long long>(g.start) * a.ld;
        asm volatile("" : "+l"(o0));
        nest_col_scan<N, NF, FORM == 0>(lp, c, sh, level);
        // no block leaves while another may still read its shared memory
        if (level == 1 && a.C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        V out[K];
        auto finish = [&](int q) {
            window(q);
            nest_chunk_finish<N, K, M, RAG>(lp, w, ck, x, nest_col_carry<N, NF>(lp, c, sh, q, 0),
                                               nest_col_carry<N, NF>(lp, c, sh, q, 1),
                                               [&](int dir) { return nest_col_end<N, NF>(lp, c, sh, q, dir); }, out);
        };
        const V m1 = N::splat(T(-1)), m2 = N::splat(T(-2));
        if (level == 0) {
            constexpr bool SIX = MODE == NEST_FCH2;
            auto u = [&](int k) {   // (a register array of it would spill)
                return g.on && (!RAG || k < K - 1 || ck.cnt == K)
                           ? nest_load<N, WIDE>(a.U + o0 + static_cast<long long>(a.ld) * k, g.both) : N::zero();
            };
            finish(2);
#pragma unroll
            for (int k = 0; k < K; ++k) arr(2, k) = N::add(out[k], arr(1, k));              // b + H c
            finish(1);
#pragma unroll
            for (int k = 0; k < K; ++k)                                                     // -2a + H b
                arr(1, k) = SIX ? N::fma(N::splat(T(2)), arr(0, k), N::fma(m1, u(k), out[k])) : N::fma(m2, arr(0, k), out[k]);
            finish(0);
#pragma unroll
            for (int k = 0; k < K; ++k) arr(0, k) = SIX ? N::add(u(k), out[k]) : out[k];
        } else {
            // out -> field f, or (other) other + s out
            auto put = [&](T* f, const T* other, V so, V sf) {
                if (!g.on) return;
                V y[K];
                if (other) {
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (!RAG || k < K - 1 || ck.cnt == K)
                            y[k] = nest_load<N, WIDE>(other + o0 + static_cast<long long>(a.ld) * k, g.both);
                }
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (!RAG || k < K - 1 || ck.cnt == K)
                        nest_store<N, WIDE>(f + o0 + static_cast<long long>(a.ld) * k,
                                            other ? N::fma(sf, y[k], N::mul(so, out[k])) : out[k], g.both);
            };
            const V one = N::splat(T(1));
            finish(0);
            put(a.o2, a.Y, MODE == NEST_FCH2 ? one : m1, one);
            finish(1);
            put(a.o1, MODE == NEST_FCH2 ? a.U : nullptr, one, one);
            finish(2);
            put(a.o0, a.in0, one, MODE == NEST_FCH2 ? one : m1);
        }
    }
    if (a.C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace molt
