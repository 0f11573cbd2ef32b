// How the nested passes cut lines into chunks and blocks (host).
#pragma once

#include "molt_internal.h"

namespace molt {

// nodes of a full chunk (one thread's share of a line)
constexpr int kNestColK = 8, kNestRowK = 16;

// How a line of n nodes is cut into chunks: nc chunks, the first `rem` of K nodes, the others of K - 1.
struct NestCut {
    int nc, rem;
};

namespace detail {

inline bool nest_cut(int n, int K, NestCut* cut) {
    if (n < 1) return false;
    const int nc = (n + K - 1) / K;
    if ((K - 1) * nc > n) return false;
    cut->nc = nc;
    cut->rem = n - (K - 1) * nc;
    return true;
}

// Column geometry: a block holds at most 256 values.  Strips of 4 values (32-byte row segments) keep a
// column of up to 512 nodes in one block and of up to 8192 nodes in a cluster of 16; shorter columns take
// wider strips while there are enough of them for two blocks on each of the 152 SMs.
template <int W>
bool nest_col_shape(int n, int ncols, int nslabs, NestCut* cut, int* lcp, int* C, int* slots, int* strips) {
    if (!nest_cut(n, kNestColK, cut)) return false;
    *C = (cut->nc + 63) / 64;
    if (*C > 16) return false;
    *slots = (cut->nc + *C - 1) / *C;
    *lcp = *slots <= 16 ? 4 : *slots <= 32 ? 3 : 2;
    for (;;) {
        *strips = (ncols + (W << *lcp) - 1) / (W << *lcp);
        if (*lcp == 2 || static_cast<long long>(*strips) * nslabs * *C >= 2 * 152) break;
        *lcp -= 1;
    }
    return true;
}

// Packed FP32 halves need half lines of whole chunks; other FP32 lines and FP64 run one value per register.
// At most 256 (packed) or 512 threads per line.
template <typename T>
bool nest_row_shape(int n, int* W, NestCut* cut) {
    if (sizeof(T) == 4 && n % (2 * kNestRowK) == 0 && n >= 4 * kNestRowK && nest_cut(n / 2, kNestRowK, cut)) {
        *W = 2;
        return cut->nc <= 256;
    }
    *W = 1;
    return nest_cut(n, kNestRowK, cut) && cut->nc >= 2 && cut->nc <= 512;
}

}  // namespace detail
}  // namespace molt
