// The single-line loop (nest_line.cuh): both precisions, every quadrature order.
#include "nest_launch.cuh"
#include "nest_line.cuh"

namespace molt {
namespace detail {

constexpr int kLineThreads = 512;

// Nodes a thread: the fewest that keep the line within 512 threads.
inline int line_k(int n) {
    for (int K = 2; K <= 8; K *= 2)
        if (n <= K * kLineThreads) return K;
    return 0;
}

template <typename T, int M, int K, bool RAG>
cudaError_t line_run(const LineParams<T>& li, const LineParams<T>& lo, const NestLine<T>& p, const NestCut& cut,
                     cudaStream_t st, Prof* prof) {
    using N = NestVec<T, 1>;
    NestLineArgs<T> a{};
    a.nlines = 1, a.half = li.n, a.TL = (cut.nc + 31) / 32 * 32, a.cut = cut;
    a.pw = nest_pow(li, K), a.pwo = nest_pow(lo, K);
    a.w = p.w, a.Y = p.Y, a.r = p.r, a.Yout = p.Yout, a.g2 = p.g2, a.g1 = p.g1, a.beta = p.beta, a.fix = p.fix, a.wall = p.wall;
    a.tol = p.tol, a.max_iter = p.max_iter, a.fp32 = sizeof(T) == 4, a.ls = p.ls, a.red = p.red;
    auto kern = nest_line_kernel<N, K, M, RAG>;
    static PerDevice limits;
    const int limit = limits.get([&] { return smem_optin(kern); });
    const size_t smem = 2 * static_cast<size_t>(li.n) * sizeof(T);
    if (limit < 0 || smem > static_cast<size_t>(limit)) return cudaErrorInvalidValue;
    prof_begin(prof, p.Yout ? kProfLineRhs : kProfLine, st);
    kern<<<1, a.TL, smem, st>>>(li, lo, a);
    prof_end(prof, st);
    return cudaGetLastError();
}

template <typename T, int M>
cudaError_t line_order(const LineParams<T>& li, const LineParams<T>& lo, const NestLine<T>& p, cudaStream_t st, Prof* prof) {
    NestCut cut;
    const int K = line_k(li.n);
    if (K == 0 || !nest_cut(li.n, K, &cut)) return cudaErrorInvalidValue;
    const bool rag = cut.rem != cut.nc;
    switch (K) {
        case 2: return rag ? line_run<T, M, 2, true>(li, lo, p, cut, st, prof) : line_run<T, M, 2, false>(li, lo, p, cut, st, prof);
        case 4: return rag ? line_run<T, M, 4, true>(li, lo, p, cut, st, prof) : line_run<T, M, 4, false>(li, lo, p, cut, st, prof);
        default: return rag ? line_run<T, M, 8, true>(li, lo, p, cut, st, prof) : line_run<T, M, 8, false>(li, lo, p, cut, st, prof);
    }
}

}  // namespace detail

// Lines of 32 nodes (every thread's window then lies within one wrap of the line) to 4096.  Longer ones run over the whole chip.
// Neumann, M = 4, us an iteration, one block against the sweeps: 256 nodes FP32 3.8 against 15.1, FP64 11.2 against 32;
// 4096 FP32 6.2 against 12.9, FP64 61 against 87; 8192 (16 nodes a thread) FP32 18 against 16.
template <typename T>
bool nest_line_ok(int n) {
    NestCut cut;
    const int K = detail::line_k(n);
    return n >= 32 && K != 0 && detail::nest_cut(n, K, &cut);
}

template <typename T>
cudaError_t nest_line(const LineParams<T>& li, const LineParams<T>& lo, const NestLine<T>& p, cudaStream_t st,
                      long long* launches, Prof* prof) {
    if (launches) *launches += 1;
    const LineParams<T> ai = nest_line_params(li), ao = nest_line_params(lo);
    switch (li.M) {
        case 2: return detail::line_order<T, 2>(ai, ao, p, st, prof);
        case 4: return detail::line_order<T, 4>(ai, ao, p, st, prof);
        case 6: return detail::line_order<T, 6>(ai, ao, p, st, prof);
    }
    return cudaErrorInvalidValue;
}

template bool nest_line_ok<float>(int);
template bool nest_line_ok<double>(int);
template cudaError_t nest_line<float>(const LineParams<float>&, const LineParams<float>&, const NestLine<float>&,
                                      cudaStream_t, long long*, Prof*);
template cudaError_t nest_line<double>(const LineParams<double>&, const LineParams<double>&, const NestLine<double>&,
                                       cudaStream_t, long long*, Prof*);

}  // namespace molt
