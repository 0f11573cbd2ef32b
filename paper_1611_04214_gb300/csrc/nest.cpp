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
    switch (lp.M) {
        case 2: return nest_cols_m<2, T>(lp, mode, p, st, prof);
        case 4: return nest_cols_m<4, T>(lp, mode, p, st, prof);
        case 6: return nest_cols_m<6, T>(lp, mode, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t nest_rows(const LineParams<T>& lp, int mode, const NestRows<T>& p, cudaStream_t st, long long* launches,
                      Prof* prof) {
    if (launches) *launches += 1;
    switch (lp.M) {
        case 2: return nest_rows_m<2, T>(lp, mode, p, st, prof);
        case 4: return nest_rows_m<4, T>(lp, mode, p, st, prof);
        case 6: return nest_rows_m<6, T>(lp, mode, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

#define MOLT_NEST_ENTRY(T)                                                                                            \
    template bool nest_rows_ok<T>(int);                                                                              \
    template bool nest_cols_ok<T>(int);                                                                              \
    template cudaError_t nest_cols<T>(const LineParams<T>&, int, const NestCols<T>&, cudaStream_t, long long*, Prof*); \
    template cudaError_t nest_rows<T>(const LineParams<T>&, int, const NestRows<T>&, cudaStream_t, long long*, Prof*);
MOLT_NEST_ENTRY(float)
MOLT_NEST_ENTRY(double)

}  // namespace molt
