// Entry of the nested passes: eligibility and the dispatch on the quadrature order.
#include "nest_shape.h"

namespace molt {

template <typename T>
bool nest_rows_ok(int n) {
    int W;
    NestCut cut;
    return detail::nest_row_shape<T>(n, &W, &cut);
}

template <typename T>
bool nest_cols_ok(int n) {
    NestCut cut;
    int lcp, C, slots, strips;
    return detail::nest_col_shape<1>(n, 1, 1, &cut, &lcp, &C, &slots, &strips) && cut.nc >= 2;
}

template <typename T>
cudaError_t nest_cols(const LineParams<T>& lp, int mode, const NestCols<T>& p, cudaStream_t st, long long* launches,
                      Prof* prof) {
    if (launches) *launches += 1;
    const LineParams<T> q = nest_line_params(lp);
    switch (lp.M) {
        case 2: return nest_cols_m<2, T>(q, mode, p, st, prof);
        case 4: return nest_cols_m<4, T>(q, mode, p, st, prof);
        case 6: return nest_cols_m<6, T>(q, mode, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t nest_rows(const LineParams<T>& lp, int mode, const NestRows<T>& p, cudaStream_t st, long long* launches,
                      Prof* prof) {
    if (launches) *launches += 1;
    const LineParams<T> q = nest_line_params(lp);
    switch (lp.M) {
        case 2: return nest_rows_m<2, T>(q, mode, p, st, prof);
        case 4: return nest_rows_m<4, T>(q, mode, p, st, prof);
        case 6: return nest_rows_m<6, T>(q, mode, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t nest_fch(const LineParams<T>& lp, const NestFch<T>& p, cudaStream_t st, long long* launches) {
    if (launches) *launches += 1;
    const LineParams<T> q = nest_line_params(lp);
    switch (lp.M) {
        case 2: return nest_fch_m<2, T>(q, p, st);
        case 4: return nest_fch_m<4, T>(q, p, st);
        case 6: return nest_fch_m<6, T>(q, p, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t nest_fch2(const LineParams<T>& lp, const NestFch2<T>& p, cudaStream_t st, long long* launches) {
    if (launches) *launches += 1;
    const LineParams<T> q = nest_line_params(lp);
    switch (lp.M) {
        case 2: return nest_fch2_m<2, T>(q, p, st);
        case 4: return nest_fch2_m<4, T>(q, p, st);
        case 6: return nest_fch2_m<6, T>(q, p, st);
    }
    return cudaErrorInvalidValue;
}

#define MOLT_NEST_ENTRY(T)                                                                                            \
    template bool nest_rows_ok<T>(int);                                                                              \
    template bool nest_cols_ok<T>(int);                                                                              \
    template cudaError_t nest_cols<T>(const LineParams<T>&, int, const NestCols<T>&, cudaStream_t, long long*, Prof*); \
    template cudaError_t nest_rows<T>(const LineParams<T>&, int, const NestRows<T>&, cudaStream_t, long long*, Prof*);    \
    template cudaError_t nest_fch<T>(const LineParams<T>&, const NestFch<T>&, cudaStream_t, long long*);                  \
    template cudaError_t nest_fch2<T>(const LineParams<T>&, const NestFch2<T>&, cudaStream_t, long long*);
MOLT_NEST_ENTRY(float)
MOLT_NEST_ENTRY(double)

}  // namespace molt
