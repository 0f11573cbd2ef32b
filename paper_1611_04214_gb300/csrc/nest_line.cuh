// A single 1D line: the whole fixed-point loop of a stage in one block (solver.cpp).  The iterate and the
// right side stay in registers, the swept values pass through shared memory, and thread 0 applies the
// stopping rule, so an iteration
//   E = H_i [beta G(w)] - beta G(w),   w <- Y + H_o E
// costs two on-chip inverses instead of three launches.  K nodes a thread: as few as 512 threads allow, so that the
// four schedulers of the SM share the FP64 work (two multiply-adds a cycle and SM on this part).
// Bound: the chain of an iteration (two scans, four block barriers each) in FP32, 256 nodes 3.8 us against 15.1 of three launches;
// the FP64 units of one SM in FP64, 4096 nodes 61 us against 87.
#pragma once

#include "nest_rows.cuh"

namespace molt {

template <typename T>
struct NestLineArgs : NestRowLayout<T> {
    T* w;             // the iterate: first guess in, last iterate out
    const T* Y;       // the stage's right side, or
    const T* r;       // ... r, from which Y = H_o H_i r (Y null)
    T* Yout;          // only compute Y from r, into here
    T g2, g1, beta;
    int fix;          // Dirichlet lines: the walls hold `wall` after every iteration
    T wall;
    double tol;
    int max_iter, fp32;
    LoopState* ls;
    unsigned long long* red;   // the last iteration's maxima (may be null)
    NestPow<T> pwo;   // as pw, for the outer inverse
};

// One inverse of the line in shared memory xs (n values): out = H xs of this thread's chunk.  With few nodes a
// thread the local integrals themselves are the cheaper form (no corrections per chunk), and any node may
// have a wall stencil.
template <class N, int K, int M>
__device__ __forceinline__ void nest_line_inverse(const LineParams<typename N::T>& lp,
                                                  const NestRowThread<N>& g, const NestRowScan<typename N::T>& c,
                                                  NestRowShared<N>& sh, const typename N::V* xs, typename N::V (&out)[K]) {
    using T = typename N::T;
    constexpr int H = M / 2;
    const int n = lp.n, cnt = g.on ? g.ck.cnt : 0, start = g.start;
    const bool periodic = lp.bc == BC_PERIODIC;
    T jl[K], jr[K];
    {
        T x[K + M];
#pragma unroll
        for (int i = 0; i < K + M; ++i) {
            int p = start - H + i;
            if (p < 0) p = periodic ? p + n : 0;
            if (p >= n) p = periodic ? p - n : n - 1;
            x[i] = g.on ? xs[p] : T(0);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            T a = T(0), b = T(0);
#pragma unroll
            for (int o = 0; o <= M; ++o) {
                a = ::fma(lp.wl[o], x[k + o], a);
                b = ::fma(lp.wr[o], x[k + o], b);
            }
            jl[k] = a;
            jr[k] = b;
        }
    }
    if (!periodic && cnt > 0 && (start < H || start + cnt > n - H)) {
        // the shifted wall stencils (as local_integrals), J^L_0 = 0 and J^R_N = 0
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = start + k, e = j - (n - H);
            if (k < cnt && (j < H || e >= 0)) {
                T a = T(0), b = T(0);
                for (int o = 0; o <= M; ++o) {
                    const T v = xs[j < H ? o : n - 1 - M + o];
                    if (j >= 1) a = ::fma(j < H ? lp.wlA[j - 1][o] : lp.wlB[e][o], v, a);
                    if (j < n - 1) b = ::fma(j < H ? lp.wrA[j][o] : lp.wrB[e][o], v, b);
                }
                jl[k] = a;
                jr[k] = b;
            }
        }
    }
    T aL, aR, cL, cR, XL, XR;
    chunk_aggregates<T, K>(lp.d, cnt, jl, jr, aL, aR);
    nest_row_scan<N, false>(lp, c, sh, aL, aR, cL, cR, XL, XR);
    if (!periodic) {
        if (start == 0 && cnt > 0) {
            jl[0] += XL;
            cL = T(0);
        }
        if (start + cnt == n && cnt > 0) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k == cnt - 1) jr[k] += XR;
            cR = T(0);
        }
    }
    chunk_finish<T, K>(lp.d, cnt, cL, cR, jl, jr);
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = jr[k];
}

template <class N, int K, int M, bool RAG>
__global__ void __launch_bounds__(512, 1)
nest_line_kernel(const __grid_constant__ LineParams<typename N::T> li, const __grid_constant__ LineParams<typename N::T> lo,
                 const __grid_constant__ NestLineArgs<typename N::T> a) {
    using V = typename N::V;
    using T = typename N::T;
    extern __shared__ __align__(16) unsigned char nest_line_sm[];
    V* xs = reinterpret_cast<V*>(nest_line_sm);
    V* xe = xs + li.n;
    __shared__ NestRowShared<N> shi, sho;
    __shared__ T s_max[2][16];
    __shared__ int s_stop;
    NestRowThread<N> g = nest_row_thread<N, K, RAG, false>(li, a);
    nest_row_scan_setup<N, K, RAG, false>(li, a, g, shi);
    NestRowThread<N> go = g;
    {
        NestRowLayout<T> b = a;
        b.pw = a.pwo;
        nest_row_scan_setup<N, K, RAG, false>(lo, b, go, sho);
    }
    const int n = li.n, start = g.start, cnt = g.on ? g.ck.cnt : 0;
    V w[K], y[K], out[K];
    auto put = [&](V* s, const V (&v)[K]) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < cnt) s[start + k] = v[k];
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        w[k] = k < cnt ? a.w[start + k] : T(0);
        y[k] = k < cnt ? (a.Y ? a.Y : a.r)[start + k] : T(0);
    }
    if (!a.Y) {
        put(xs, y);
        __syncthreads();
        nest_line_inverse<N, K, M>(li, g, g.c, shi, xs, out);
        put(xe, out);
        __syncthreads();
        nest_line_inverse<N, K, M>(lo, g, go.c, sho, xe, y);
        if (a.Yout) {
            put(a.Yout, y);
            return;
        }
    }
    // state of the stopping rule (thread 0)
    double best = __longlong_as_double(0x7ff0000000000000LL), res = best, vmax = 0.0, tol_used = 0.0;
    int stall = 0, conv = 0, k_it = 0, bad = 0;
    for (;;) {
        V gl[K];
#pragma unroll
        for (int k = 0; k < K; ++k) gl[k] = a.beta * g_lag(w[k], a.g2, a.g1);
        put(xs, gl);
        __syncthreads();
        nest_line_inverse<N, K, M>(li, g, g.c, shi, xs, out);
#pragma unroll
        for (int k = 0; k < K; ++k) out[k] -= gl[k];
        put(xe, out);
        __syncthreads();
        nest_line_inverse<N, K, M>(lo, g, go.c, sho, xe, out);
        T dm = T(0), vm = T(0);
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < cnt) {
                const T nw = y[k] + out[k];
                dm = abs_max(dm, fabs(nw - w[k]));
                vm = abs_max(vm, fabs(nw));
                w[k] = a.fix && (start + k == 0 || start + k == n - 1) ? a.wall : nw;
            }
        const bool nan_here = vm != vm || dm != dm;   // (the line is NaN throughout then: nest_reduce)
        dm = nest_warp_max(nan_here ? T(0) : dm);
        vm = nest_warp_max(nan_here ? T(0) : vm);
        if (g.c.lane == 0) {
            s_max[0][g.c.warp] = dm;
            s_max[1][g.c.warp] = vm;
        }
        bad = __syncthreads_or(nan_here);
        if (threadIdx.x == 0) {
            // as loop_check: tolerance, FP32 floor of 2 ulp of max|w|, stall at the FP32 noise floor, cap, NaN
            T d = T(0), v = T(0);
            for (int q = 0; q < g.c.nwarps; ++q) {
                d = abs_max(d, s_max[0][q]);
                v = abs_max(v, s_max[1][q]);
            }
            res = static_cast<double>(d);
            vmax = static_cast<double>(v);
            const double ulp = vmax * 5.9604644775390625e-08;
            tol_used = a.fp32 ? fmax(a.tol, 2.0 * ulp) : a.tol;
            ++k_it;
            bool stop = false;
            if (!isfinite(res)) {
                stop = true;
            } else if (res < tol_used) {
                conv = 1;
            } else if (res < best) {
                best = res;
                stall = 0;
            } else if (a.fp32 && res < 64.0 * ulp && ++stall >= 6) {
                conv = 1;
                tol_used = res;
            }
            s_stop = stop || conv || k_it >= a.max_iter;
            if (bad) conv = 0;
        }
        __syncthreads();
        if (s_stop) break;
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (k < cnt) a.w[start + k] = w[k];
    if (threadIdx.x == 0) {
        LoopState s;
        s.k = k_it;
        s.stall = stall;
        s.done = 1;
        s.converged = conv;
        s.best = best;
        s.res = bad ? nan("") : res;
        s.tol_used = tol_used;
        *a.ls = s;
        if (a.red) {
            a.red[0] = static_cast<unsigned long long>(__double_as_longlong(res));
            a.red[1] = static_cast<unsigned long long>(__double_as_longlong(vmax));
            a.red[2] = bad ? 1ull : 0ull;
        }
    }
}

}  // namespace molt
