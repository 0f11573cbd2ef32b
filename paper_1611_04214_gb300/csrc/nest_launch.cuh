// Launch layer of the nested passes (nest.cuh, nest_rows.cuh), one quadrature order per translation
// unit (nest_m2.cu, nest_m4.cu, nest_m6.cu).
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

// Coefficients of an inverse (NestCoef).  The quadrature weights are those of nu' = -ln d for the
// decay d as the kernel holds it: the recurrence and the weights then belong to one operator (H 1 = 1
// holds with a rounded d too).
template <typename V, int M, typename T>
NestCoef<V> nest_coef(const LineParams<T>& lp) {
    NestCoef<V> c;
    std::memset(&c, 0, sizeof(c));
    const double d = static_cast<double>(lp.d);
    const double nu = d > 0.0 && d < 1.0 ? -std::log(d) : static_cast<double>(lp.nu);
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

template <typename T, int M, int FORM, bool WIDE, int MODE>
cudaError_t nest_cols_run(const LineParams<T>& lp, const NestCols<T>& p, cudaStream_t st, Prof* prof) {
    using N = NestVec<T, sizeof(T) == 4 ? 2 : 1>;
    NestColArgs<T> a{};
    a.in0 = p.in0, a.in1 = p.in1, a.Y = p.Y, a.o0 = p.o0, a.o1 = p.o1, a.o2 = p.o2;
    a.ld = static_cast<int>(p.ld), a.slab = p.slab, a.ncols = p.ncols;
    a.g1 = p.g1, a.beta = p.beta, a.vs = p.vs, a.comp = p.comp;
    int strips;
    if (!nest_col_shape<N::W>(lp.n, p.ncols, p.nslabs, &a.cut, &a.lcp, &a.C, &a.slots, &strips) || p.ld > 0x7fffffffLL ||
        p.nslabs > 65535)
        return cudaErrorInvalidValue;
    a.pw = nest_pow(lp, kNestColK);
    a.exact = static_cast<double>(lp.nu) * lp.N < 45.0;   // e^-45 < 2^-64
    const int nt = ((a.slots << a.lcp) + 31) / 32 * 32;
    constexpr int NA = MODE == NEST_COPY ? 1 : 3, NF = MODE == NEST_COPY ? 1 : 2;
    const size_t smem = static_cast<size_t>(nt) * (nest_col_pitch<kNestColK, M, NA>() * sizeof(typename N::V) + 4 * sizeof(T)) +
                        (static_cast<size_t>(2 * NF * (a.slots + 4)) << a.lcp) * sizeof(typename N::V);
    auto kern = nest_cols_kernel<N, M, FORM, WIDE, MODE>;
    static int limit = [&] {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return -1;
        return smem_optin(kern);
    }();
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
    prof_begin(prof, MODE == NEST_COPY ? kProfNestColsRhs : kProfNestCols, st);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, lp, w, a);
    prof_end(prof, st);
    return e;
}

template <class N, int M, bool RAG, bool WARP, int MODE>
cudaError_t nest_rows_launch(const LineParams<typename N::T>& lp, const NestRowArgs<typename N::T>& a_in, cudaStream_t st,
                             Prof* prof) {
    auto kern = nest_rows_kernel<N, M, RAG, WARP, MODE>;
    const int block = WARP ? 128 : a_in.TL;
    const int per = WARP ? block / a_in.TL : 1;
    const size_t smem = WARP ? 0 : static_cast<size_t>(2 * M) * a_in.TL * sizeof(typename N::V);
    static int limit = smem_optin(kern);
    if (limit < 0 || smem > static_cast<size_t>(limit)) return cudaErrorInvalidValue;
    const NestCoef<typename N::V> w = nest_coef<typename N::V, M>(lp);
    NestRowArgs<typename N::T> a = a_in;
    // two blocks a SM (the kernel's launch bounds); lines that stay in L2 anyway need no fetching ahead
    a.ahead = WARP ? 0 : 2 * 152;
    prof_begin(prof, MODE == NEST_ROW_COPY ? kProfNestRowsRhs : kProfNestRows, st);
    kern<<<(a.nlines + per - 1) / per, block, smem, st>>>(lp, w, a);
    prof_end(prof, st);
    return cudaGetLastError();
}

template <class N, int M, int MODE>
cudaError_t nest_rows_team(const LineParams<typename N::T>& lp, NestRowArgs<typename N::T>& a, bool rag, cudaStream_t st,
                           Prof* prof) {
    const int nc = a.cut.nc;
    if (nc <= 32) {
        a.TL = 1;
        while (a.TL < nc) a.TL *= 2;
        if constexpr (N::W == 1)
            if (rag) return nest_rows_launch<N, M, true, true, MODE>(lp, a, st, prof);
        return nest_rows_launch<N, M, false, true, MODE>(lp, a, st, prof);
    }
    a.TL = (nc + 31) / 32 * 32;
    if constexpr (N::W == 1)
        if (rag) return nest_rows_launch<N, M, true, false, MODE>(lp, a, st, prof);
    return nest_rows_launch<N, M, false, false, MODE>(lp, a, st, prof);
}

template <typename T, int M, int MODE>
cudaError_t nest_rows_run(const LineParams<T>& lp, const NestRows<T>& p, cudaStream_t st, Prof* prof) {
    NestRowArgs<T> a{};
    a.A = p.A, a.B = p.B, a.E = p.E, a.w = p.w, a.nlines = p.nlines, a.fix = p.fix, a.wall = p.wall, a.red = p.red;
    int W;
    if (!nest_row_shape<T>(lp.n, &W, &a.cut)) return cudaErrorInvalidValue;
    const T* fields[] = {p.A, p.B, p.E, p.w};
    for (const T* f : fields)
        if (W == 2 && !aligned16(f)) return cudaErrorInvalidValue;
    a.half = lp.n / W;
    a.pw = nest_pow(lp, kNestRowK);
    const bool rag = a.cut.rem != a.cut.nc;
    if constexpr (sizeof(T) == 4) {
        if (W == 2) return nest_rows_team<NestVec<float, 2>, M, MODE>(lp, a, rag, st, prof);
    }
    return nest_rows_team<NestVec<T, 1>, M, MODE>(lp, a, rag, st, prof);
}

}  // namespace detail

namespace detail {
// Column pairs by 8-byte accesses where every row starts on 8 bytes; FP32 grids with an odd number of
// columns take the two columns one by one.
template <typename T, int M, int MODE>
cudaError_t nest_cols_mode(const LineParams<T>& lp, const NestCols<T>& p, cudaStream_t st, Prof* prof) {
    bool wide = p.ncols % 2 == 0 && p.ld % 2 == 0 && p.slab % 2 == 0;
    const T* fields[] = {p.in0, p.in1, p.Y, p.o0, p.o1, p.o2};
    for (const T* f : fields) wide = wide && aligned8(f);
    const int nc = lp.n / kNestColK, C = (nc + 63) / 64;
    const int form = lp.n % kNestColK != 0 ? 2 : nc % (16 * C) != 0 ? 1 : 0;
    if constexpr (sizeof(T) == 4) {
        if (!wide)
            return form == 2 ? nest_cols_run<T, M, 2, false, MODE>(lp, p, st, prof)
                             : nest_cols_run<T, M, 1, false, MODE>(lp, p, st, prof);
    }
    return form == 2   ? nest_cols_run<T, M, 2, true, MODE>(lp, p, st, prof)
           : form == 1 ? nest_cols_run<T, M, 1, true, MODE>(lp, p, st, prof)
                       : nest_cols_run<T, M, 0, true, MODE>(lp, p, st, prof);
}
}  // namespace detail

template <int M, typename T>
cudaError_t nest_cols_m(const LineParams<T>& lp, int mode, const NestCols<T>& p, cudaStream_t st, Prof* prof) {
    using namespace detail;
    switch (mode) {
        case NEST_SCALAR: return nest_cols_mode<T, M, NEST_SCALAR>(lp, p, st, prof);
        case NEST_VCH: return nest_cols_mode<T, M, NEST_VCH>(lp, p, st, prof);
        case NEST_COPY: return nest_cols_mode<T, M, NEST_COPY>(lp, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

template <int M, typename T>
cudaError_t nest_rows_m(const LineParams<T>& lp, int mode, const NestRows<T>& p, cudaStream_t st, Prof* prof) {
    using namespace detail;
    return mode == NEST_ROW_PASS ? nest_rows_run<T, M, NEST_ROW_PASS>(lp, p, st, prof)
                                 : nest_rows_run<T, M, NEST_ROW_COPY>(lp, p, st, prof);
}

#define MOLT_INSTANTIATE_NEST(M, T)                                                                                  \
    template cudaError_t molt::nest_cols_m<M, T>(const molt::LineParams<T>&, int, const molt::NestCols<T>&, cudaStream_t, \
                                                 molt::Prof*);                                                       \
    template cudaError_t molt::nest_rows_m<M, T>(const molt::LineParams<T>&, int, const molt::NestRows<T>&, cudaStream_t, \
                                                 molt::Prof*);

}  // namespace molt
