// Launch layer of the nested passes (nest.cuh, nest_rows.cuh), one quadrature order per translation
// unit and precision (nest_f32_m2.cu to nest_f64_m6.cu).
#pragma once

#include <cmath>
#include <cstring>

#include "launch.cuh"
#include "nest.cuh"
#include "nest_rows.cuh"
#include "nest_shape.h"

namespace molt {
namespace detail {

inline bool aligned8(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7) == 0; }

// A coefficient as the register values hold it.
inline void nest_put(unsigned long long* o, double v) {
    const float f = static_cast<float>(v);
    unsigned b;
    std::memcpy(&b, &f, 4);
    *o = (static_cast<unsigned long long>(b) << 32) | b;
}
template <typename T>
void nest_put(T* o, double v) { *o = static_cast<T>(v); }

// Coefficients of an inverse (NestCoef) of nest_line_params, the quadrature weights in FP64.
template <typename V, int M, typename T>
NestCoef<V> nest_coef(const LineParams<T>& lp) {
    NestCoef<V> c;
    std::memset(&c, 0, sizeof(c));
    const double d = static_cast<double>(lp.d);
    const double nu = nest_nu(lp);
    int offs[M + 1];
    double w[M + 1], beta[M + 1];
    for (int o = 0; o <= M; ++o) offs[o] = o - M / 2;
    quadrature_weights(nu, M, offs, 0, w);
    double acc = 0.0;
    for (int i = M; i >= 0; --i) beta[i] = acc = w[i] + d * acc;
    nest_put(&c.alpha, beta[0]);
    for (int i = 1; i <= M; ++i) nest_put(&c.beta[i], beta[i]);
    beta[0] = 0.0;
    for (int m = 0; m <= M / 2; ++m) nest_put(&c.gamma[m], beta[m] + beta[M - m]);
    return c;
}
template <typename T>
NestPow<T> nest_pow(const LineParams<T>& lp, int K) {
    const double d = static_cast<double>(lp.d);
    return {static_cast<T>(std::pow(d, K - 1)), static_cast<T>(std::pow(d, K - 2))};
}

// One column kernel, F::kern(); F::kPitch values per thread, F::kNF fields.
template <class F, int M, typename T>
cudaError_t nest_cols_run(const LineParams<T>& lp, const NestCols<T>& p, cudaStream_t st, Prof* prof) {
    using N = NestVec<T, sizeof(T) == 4 ? 2 : 1>;
    NestColArgs<T> a{};
    a.in0 = p.in0, a.in1 = p.in1, a.in2 = p.in2, a.Y = p.Y, a.U = p.U, a.single = p.single, a.o0 = p.o0, a.o1 = p.o1, a.o2 = p.o2;
    a.ld = static_cast<int>(p.ld), a.slab = p.slab, a.ncols = p.ncols;
    a.g1 = p.g1, a.beta = p.beta, a.vs = p.vs, a.comp = p.comp;
    int strips;
    if (!nest_col_shape<N::W>(lp.n, p.ncols, p.nslabs, &a.cut, &a.lcp, &a.C, &a.slots, &strips) || p.ld > 0x7fffffffLL ||
        p.nslabs > 65535)
        return cudaErrorInvalidValue;
    a.pw = nest_pow(lp, kNestColK);
    a.exact = static_cast<double>(lp.nu) * lp.N < 45.0;   // e^-45 < 2^-64
    const int nt = ((a.slots << a.lcp) + 31) / 32 * 32;
    const size_t smem = static_cast<size_t>(nt) * (F::kPitch * sizeof(typename N::V) + 4 * sizeof(T)) +
                        (static_cast<size_t>(2 * F::kNF * (a.slots + 4)) << a.lcp) * sizeof(typename N::V);
    auto kern = F::kern();
    static PerDevice limits;
    const int limit = limits.get([&] {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return -1;
        return smem_optin(kern);
    });
    if (limit < 0 || smem > static_cast<size_t>(limit)) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = a.C;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(strips, a.C, p.nslabs);
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = a.C > 1 ? 1 : 0;
    const NestCoef<typename N::V> w = nest_coef<typename N::V, M>(lp);
    prof_begin(prof, F::kSlot, st);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, lp, w, a);
    prof_end(prof, st);
    return e;
}

template <typename T, int M, int FORM, bool WIDE, int MODE> struct NestColsPass {
    static constexpr int kPitch = nest_col_pitch<kNestColK, M, MODE == NEST_COPY ? 1 : 3>();
    static constexpr int kNF = MODE == NEST_COPY ? 1 : 2, kSlot = MODE == NEST_COPY ? kProfNestColsRhs : kProfNestCols;
    static auto kern() { return nest_cols_kernel<NestVec<T, sizeof(T) == 4 ? 2 : 1>, M, FORM, WIDE, MODE>; }
};
template <typename T, int M, int FORM, bool WIDE, int MODE> struct NestCols3Pass {
    static constexpr int kPitch = nest_col3_pitch<kNestColK, M>(), kNF = 3, kSlot = kProfNestCols;
    static auto kern() { return nest_cols3_kernel<NestVec<T, sizeof(T) == 4 ? 2 : 1>, M, FORM, WIDE, MODE>; }
};
template <typename T, int M, int FORM, bool WIDE>
struct NestColsPass<T, M, FORM, WIDE, NEST_Y3> : NestCols3Pass<T, M, FORM, WIDE, NEST_Y3> {};
template <typename T, int M, int FORM, bool WIDE>
struct NestColsPass<T, M, FORM, WIDE, NEST_FCH2> : NestCols3Pass<T, M, FORM, WIDE, NEST_FCH2> {};

// One row kernel, F::kern(); args has the layout but for `ahead`.
template <class F, class N, int M, bool WARP, class Args>
cudaError_t nest_rows_launch(const LineParams<typename N::T>& lp, Args a, cudaStream_t st, Prof* prof, int slot) {
    const int block = WARP ? 128 : a.TL;
    const int per = WARP ? block / a.TL : 1;
    const size_t smem = WARP ? 0 : static_cast<size_t>(2 * M) * a.TL * sizeof(typename N::V);
    static PerDevice limits;
    const int limit = limits.get([&] { return smem_optin(F::kern()); });
    if (limit < 0 || smem > static_cast<size_t>(limit)) return cudaErrorInvalidValue;
    const NestCoef<typename N::V> w = nest_coef<typename N::V, M>(lp);
    // two blocks a SM (the kernel's launch bounds); short lines are on their way before they are wanted
    a.ahead = WARP ? 0 : 2 * 152;
    prof_begin(prof, slot, st);
    F::kern()<<<(a.nlines + per - 1) / per, block, smem, st>>>(lp, w, a);
    prof_end(prof, st);
    return cudaGetLastError();
}

// Lines cut into chunks of one length or two (RAG), teams within a warp or of a block.  F<N, M, RAG, WARP>::kern()
// is the kernel.
template <class N, int M, template <class, int, bool, bool> class F, class Args>
cudaError_t nest_rows_team(const LineParams<typename N::T>& lp, Args a, cudaStream_t st, Prof* prof, int slot) {
    const int nc = a.cut.nc;
    const bool warp = nc <= 32, rag = N::W == 1 && a.cut.rem != nc;
    a.TL = (nc + 31) / 32 * 32;
    if (warp)
        for (a.TL = 1; a.TL < nc;) a.TL *= 2;
    if constexpr (N::W == 1) {
        if (rag)
            return warp ? nest_rows_launch<F<N, M, true, true>, N, M, true>(lp, a, st, prof, slot)
                        : nest_rows_launch<F<N, M, true, false>, N, M, false>(lp, a, st, prof, slot);
    }
    return warp ? nest_rows_launch<F<N, M, false, true>, N, M, true>(lp, a, st, prof, slot)
                : nest_rows_launch<F<N, M, false, false>, N, M, false>(lp, a, st, prof, slot);
}
template <class N, int M, bool RAG, bool WARP> struct NestRowPass {
    static auto kern() { return nest_rows_kernel<N, M, RAG, WARP, NEST_ROW_PASS>; }
};
template <class N, int M, bool RAG, bool WARP> struct NestRowCopy {
    static auto kern() { return nest_rows_kernel<N, M, RAG, WARP, NEST_ROW_COPY>; }
};
template <class N, int M, bool RAG, bool WARP> struct NestFchPass {
    static auto kern() { return nest_fch_kernel<N, M, RAG, WARP>; }
};

template <class N, int M, bool RAG, bool WARP> struct NestFch2Pass {
    static auto kern() { return nest_fch2_kernel<N, M, RAG, WARP>; }
};

template <typename T, int M, template <class, int, bool, bool> class F, class Args>
cudaError_t nest_rows_run(const LineParams<T>& lp, Args a, int nlines, bool aligned, cudaStream_t st, Prof* prof, int slot) {
    int W;
    if (!nest_row_shape<T>(lp.n, &W, &a.cut) || (W == 2 && !aligned)) return cudaErrorInvalidValue;
    a.nlines = nlines;
    a.half = lp.n / W;
    a.pw = nest_pow(lp, kNestRowK);
    if constexpr (sizeof(T) == 4) {
        if (W == 2) return nest_rows_team<NestVec<float, 2>, M, F>(lp, a, st, prof, slot);
    }
    return nest_rows_team<NestVec<T, 1>, M, F>(lp, a, st, prof, slot);
}

}  // namespace detail

namespace detail {
// Column pairs by 8-byte accesses where every row starts on 8 bytes; FP32 grids with an odd number of
// columns take the two columns one by one.
template <typename T, int M, int MODE>
cudaError_t nest_cols_mode(const LineParams<T>& lp, const NestCols<T>& p, cudaStream_t st, Prof* prof) {
    bool wide = p.ncols % 2 == 0 && p.ld % 2 == 0 && p.slab % 2 == 0;
    const T* fields[] = {p.in0, p.in1, p.in2, p.Y, p.U, p.o0, p.o1, p.o2};
    for (const T* f : fields) wide = wide && aligned8(f);
    const int nc = lp.n / kNestColK, C = (nc + 63) / 64;
    const int form = lp.n % kNestColK != 0 ? 2 : nc % (16 * C) != 0 ? 1 : 0;
    if constexpr (sizeof(T) == 4) {
        if (!wide)
            return form == 2 ? nest_cols_run<NestColsPass<T, M, 2, false, MODE>, M>(lp, p, st, prof)
                             : nest_cols_run<NestColsPass<T, M, 1, false, MODE>, M>(lp, p, st, prof);
    }
    return form == 2   ? nest_cols_run<NestColsPass<T, M, 2, true, MODE>, M>(lp, p, st, prof)
           : form == 1 ? nest_cols_run<NestColsPass<T, M, 1, true, MODE>, M>(lp, p, st, prof)
                       : nest_cols_run<NestColsPass<T, M, 0, true, MODE>, M>(lp, p, st, prof);
}
}  // namespace detail

template <int M, typename T>
cudaError_t nest_cols_m(const LineParams<T>& lp, int mode, const NestCols<T>& p, cudaStream_t st, Prof* prof) {
    using namespace detail;
    switch (mode) {
        case NEST_SCALAR: return nest_cols_mode<T, M, NEST_SCALAR>(lp, p, st, prof);
        case NEST_VCH: return nest_cols_mode<T, M, NEST_VCH>(lp, p, st, prof);
        case NEST_COPY: return nest_cols_mode<T, M, NEST_COPY>(lp, p, st, prof);
        case NEST_FCH2: return nest_cols_mode<T, M, NEST_FCH2>(lp, p, st, prof);
    }
    if constexpr (sizeof(T) == 4) {   // 3D runs in FP32
        if (mode == NEST_Z3) return nest_cols_mode<T, M, NEST_Z3>(lp, p, st, prof);
        if (mode == NEST_Y3) return nest_cols_mode<T, M, NEST_Y3>(lp, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

template <int M, typename T>
cudaError_t nest_rows_m(const LineParams<T>& lp, int mode, const NestRows<T>& p, cudaStream_t st, Prof* prof) {
    using namespace detail;
    NestRowArgs<T> a{};
    a.A = p.A, a.B = p.B, a.E = p.E, a.w = p.w, a.fix = p.fix, a.wall = p.wall, a.red = p.red;
    const bool al = aligned16(p.A) && aligned16(p.B) && aligned16(p.E) && aligned16(p.w);
    return mode == NEST_ROW_PASS ? nest_rows_run<T, M, NestRowPass>(lp, a, p.nlines, al, st, prof, kProfNestRows)
                                 : nest_rows_run<T, M, NestRowCopy>(lp, a, p.nlines, al, st, prof, kProfNestRowsRhs);
}

template <int M, typename T>
cudaError_t nest_fch_m(const LineParams<T>& lp, const NestFch<T>& p, cudaStream_t st) {
    using namespace detail;
    NestFchArgs<T> a{};
    a.v = p.v, a.lap = p.lap, a.h2 = p.h2, a.red = p.red;
    static_cast<FchCoef<T>&>(a) = fch_coef<T>(p);
    const bool al = aligned16(p.v) && aligned16(p.lap) && aligned16(p.h2);
    return nest_rows_run<T, M, NestFchPass>(lp, a, p.nlines, al, st, nullptr, 0);
}

template <int M, typename T>
cudaError_t nest_fch2_m(const LineParams<T>& lp, const NestFch2<T>& p, cudaStream_t st) {
    using namespace detail;
    NestFch2Args<T> a{};
    a.W = p.W, a.hy = p.hy, a.m2 = p.m2, a.v = p.v, a.p = p.p, a.q = p.q, a.r = p.r, a.u = p.u, a.z = p.z, a.red = p.red;
    static_cast<FchCoef<T>&>(a) = fch_coef<T>(p);
    bool al = true;
    const T* fields[] = {p.W, p.hy, p.m2, p.v, p.p, p.q, p.r, p.u, p.z};
    for (const T* f : fields) al = al && aligned16(f);
    return nest_rows_run<T, M, NestFch2Pass>(lp, a, p.nlines, al, st, nullptr, 0);
}

#define MOLT_INSTANTIATE_NEST(M, T)                                                                                  \
    template cudaError_t molt::nest_cols_m<M, T>(const molt::LineParams<T>&, int, const molt::NestCols<T>&, cudaStream_t, \
                                                 molt::Prof*);                                                       \
    template cudaError_t molt::nest_rows_m<M, T>(const molt::LineParams<T>&, int, const molt::NestRows<T>&, cudaStream_t, \
                                                 molt::Prof*);                                                       \
    template cudaError_t molt::nest_fch_m<M, T>(const molt::LineParams<T>&, const molt::NestFch<T>&, cudaStream_t);      \
    template cudaError_t molt::nest_fch2_m<M, T>(const molt::LineParams<T>&, const molt::NestFch2<T>&, cudaStream_t);

}  // namespace molt
