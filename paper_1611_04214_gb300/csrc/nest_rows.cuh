// Two line inverses in a row along x (rows), the line in registers between them (see nest.cuh).
// A team of TL threads owns a line: thread t holds chunk t, and in packed FP32 chunk t of the
// line's first half in the low and of its second half in the high half of each register pair.  Teams of
// up to 32 threads are parts of a warp (no block barrier anywhere), longer lines take a block.
//   pass:  w <- w + (E + H (B + H A)), with the residual of the iteration (E = Y - H_y H_y w);
//   copy:  out = H H in.
// Bound: the latency of a line's chain (load, two scans, loads of B, E and w) at two lines a SM: 8192^2 FP32 285 us
// = 4700 GB/s of its 20 B a point (0.69 of the copy rate) for two inverses, against 306 + 237 us of passes 2 and 4; the
// fetches into L2 ahead of use give 5% of it.
#pragma once

#include "nest.cuh"

namespace molt {

// How the lines are laid over threads.
template <typename T>
struct NestRowLayout {
    int nlines;
    int half;        // nodes of a register half (n or n / 2)
    int TL;          // threads per line
    NestCut cut;     // of a half
    NestPow<T> pw;   // d^(cnt-1) of the two chunk lengths
    int ahead;       // lines resident at a time (0: nothing is fetched ahead)
};

template <typename T>
struct NestRowArgs : NestRowLayout<T> {
    const T* A;
    const T* B;
    const T* E;
    T* w;            // pass: the iterate, in place; copy: the output
    int fix;         // Dirichlet grids: write `wall` to the wall nodes
    T wall;
    unsigned long long* red;
};

template <class N>
struct NestRowShared {
    using V = typename N::V;
    using T = typename N::T;
    V tot[2][16];
    V ex[2][16];
    V X[2];
    T wd[16], wdf[16], wdb[16];
};

template <typename T>
struct NestRowScan {
    int lane, warp, nwarps, tl, width;
    T df[5], db[5];
    T Dxf, Dxb;      // decay of the scan group's chunks before / after this one
    T Dh;            // decay over a half
    T pl[2], pr[2];  // decay from the line's ends, per half
};

// Totals of the halves -> carries entering the halves (E) and line totals.
template <class N>
__device__ __forceinline__ void nest_halves(typename N::V f, typename N::V b, typename N::T Dh, typename N::V& Ef,
                                            typename N::V& Eb, typename N::T& IN, typename N::T& I0) {
    using T = typename N::T;
    if constexpr (N::W == 2) {
        Ef = N::pair(T(0), N::get(f, 0));
        Eb = N::pair(N::get(b, 1), T(0));
        IN = ::fma(N::get(f, 0), Dh, N::get(f, 1));
        I0 = ::fma(N::get(b, 1), Dh, N::get(b, 0));
    } else {
        Ef = Eb = N::zero();
        IN = f;
        I0 = b;
    }
}

template <class N, bool WARP>
__device__ __forceinline__ void nest_row_scan(const LineParams<typename N::T>& lp, const NestRowScan<typename N::T>& c,
                                              NestRowShared<N>& sh, typename N::V aL, typename N::V aR,
                                              typename N::V& cL, typename N::V& cR, typename N::V& XL,
                                              typename N::V& XR) {
    using V = typename N::V;
    using T = typename N::T;
    V a = aL, b = aR;
    const int width = WARP ? c.width : 32, li = c.lane & (width - 1);
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int o = 1 << s;
        if (o < width) {
            const V u = shfl_up_v<N>(a, o, width), v = shfl_down_v<N>(b, o, width);
            if (li >= o) a = N::fma(u, N::splat(c.df[s]), a);
            if (li + o < width) b = N::fma(v, N::splat(c.db[s]), b);
        }
    }
    V ax = shfl_up_v<N>(a, 1, width), bx = shfl_down_v<N>(b, 1, width);
    if (li == 0) ax = N::zero();
    if (li == width - 1) bx = N::zero();
    V Ef, Eb;
    T IN, I0, xl, xr;
    if constexpr (WARP) {
        const V f = __shfl_sync(kFull, a, width - 1, width), g = __shfl_sync(kFull, b, 0, width);
        nest_halves<N>(f, g, c.Dh, Ef, Eb, IN, I0);
        nest_boundary<T>(lp, I0, IN, xl, xr);
        XL = N::splat(xl);
        XR = N::splat(xr);
    } else {
        if (c.lane == 31) sh.tot[0][c.warp] = a;
        if (c.lane == 0) sh.tot[1][c.warp] = b;
        __syncthreads();
        if (c.warp == 0) {
            // scan of the warps' totals, one warp per lane
            const bool has = c.lane < c.nwarps;
            V f = has ? sh.tot[0][c.lane] : N::zero(), g = has ? sh.tot[1][c.lane] : N::zero();
            T fd = has ? sh.wd[c.lane] : T(1), gd = fd;
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                const V u = shfl_up_v<N>(f, o), v = shfl_down_v<N>(g, o);
                const T ud = __shfl_up_sync(kFull, fd, o), vd = __shfl_down_sync(kFull, gd, o);
                if (c.lane >= o) {
                    f = N::fma(u, N::splat(fd), f);
                    fd *= ud;
                }
                if (c.lane + o < 32) {
                    g = N::fma(v, N::splat(gd), g);
                    gd *= vd;
                }
            }
            const V tf = __shfl_sync(kFull, f, c.nwarps - 1), tg = __shfl_sync(kFull, g, 0);
            V fx = shfl_up_v<N>(f, 1), gx = shfl_down_v<N>(g, 1);
            if (c.lane == 0) fx = N::zero();
            if (c.lane >= c.nwarps - 1) gx = N::zero();
            nest_halves<N>(tf, tg, c.Dh, Ef, Eb, IN, I0);
            nest_boundary<T>(lp, I0, IN, xl, xr);
            if (has) {
                sh.ex[0][c.lane] = N::fma(Ef, N::splat(sh.wdf[c.lane]), fx);
                sh.ex[1][c.lane] = N::fma(Eb, N::splat(sh.wdb[c.lane]), gx);
            }
            if (c.lane == 0) {
                sh.X[0] = N::splat(xl);
                sh.X[1] = N::splat(xr);
            }
        }
        __syncthreads();
        Ef = sh.ex[0][c.warp];
        Eb = sh.ex[1][c.warp];
        XL = sh.X[0];
        XR = sh.X[1];
    }
    const V pl = N::pair(c.pl[0], c.pl[1]), pr = N::pair(c.pr[0], c.pr[1]);
    cL = N::fma(pl, XL, N::fma(Ef, N::splat(c.Dxf), ax));
    cR = N::fma(pr, XR, N::fma(Eb, N::splat(c.Dxb), bx));
}

// Edge values of the neighbouring chunks of the line (wrapped; a low half continues in the high half).
template <class N, int K, int M, bool RAG, bool WARP, int KM>
__device__ __forceinline__ void nest_row_halo(const NestRowScan<typename N::T>& c, int nc, int cnt,
                                              typename N::V* edge, int TL, typename N::V (&x)[KM]) {
    using V = typename N::V;
    constexpr int H = M / 2;
    V l[H], r[H];
    const int tl = c.tl;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        V e = x[H + K - H + h];
        if (RAG && cnt != K) e = x[H + K - 1 - H + h];
        if constexpr (WARP) {
            const int base = c.lane - tl;
            const int pl = base + (tl > 0 ? tl - 1 : nc - 1), fl = base + (tl < nc - 1 ? tl + 1 : 0);
            l[h] = __shfl_sync(kFull, e, pl);
            r[h] = __shfl_sync(kFull, x[H + h], fl);
        } else {
            edge[h * TL + tl] = e;
            edge[(H + h) * TL + tl] = x[H + h];
        }
    }
    if constexpr (!WARP) {
        __syncthreads();
        const int pl = tl > 0 ? tl - 1 : nc - 1, fl = tl < nc - 1 ? tl + 1 : 0;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            l[h] = edge[h * TL + pl];
            r[h] = edge[(H + h) * TL + fl];
        }
    }
    if constexpr (N::W == 2) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if (tl == 0) l[h] = N::swap(l[h]);
            if (tl == nc - 1) r[h] = N::swap(r[h]);
        }
    }
    nest_set_halo<N, K, M, RAG>(cnt, l, r, x);
}

// Nodes p.. of one half line (float4 chunks), or of a scalar line.
template <class N, int K, bool RAG, int OFF, int KM>
__device__ __forceinline__ void nest_row_load(const typename N::T* f, int half, int start, int cnt, bool on,
                                              typename N::V (&x)[KM]) {
    using T = typename N::T;
    if constexpr (N::W == 2) {
#pragma unroll
        for (int j = 0; j < K / 4; ++j) {
            float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
            if (on && (!RAG || 4 * j < cnt)) {
                lo = *reinterpret_cast<const float4*>(f + start + 4 * j);
                hi = *reinterpret_cast<const float4*>(f + half + start + 4 * j);
            }
            x[OFF + 4 * j] = N::pair(lo.x, hi.x);
            x[OFF + 4 * j + 1] = N::pair(lo.y, hi.y);
            x[OFF + 4 * j + 2] = N::pair(lo.z, hi.z);
            x[OFF + 4 * j + 3] = N::pair(lo.w, hi.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) x[OFF + k] = on && (!RAG || k < cnt) ? f[start + k] : T(0);
    }
}

// Block maximum of the residual values into the FP64 slots; blocks that would not raise a slot leave
// it alone (the slots only grow, so a stale read costs an atomic at most).  A NaN marks the third slot, as in
// block_reduce_store; a thread's nodes belong to one line, which is NaN throughout then, so the thread's whole share is
// left out.
template <typename T>
__device__ __forceinline__ T nest_warp_max(T v) {
    if constexpr (sizeof(T) == 4) {
        // non-negative floats order like their bits
        return __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(v)));
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = abs_max(v, __shfl_xor_sync(kFull, v, o));
        return v;
    }
}
template <typename T>
__device__ __forceinline__ void nest_reduce(RedAcc<T> r, unsigned long long* slots) {
    __shared__ T s_max[2][16];
    const bool bad = r.vmax != r.vmax || r.dmax != r.dmax;
    const T dm = nest_warp_max(bad ? T(0) : r.dmax), vm = nest_warp_max(bad ? T(0) : r.vmax);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (__any_sync(kFull, bad) && lane == 0) atomicMax(slots + 2, 1ull);
    if (lane == 0) {
        s_max[0][warp] = dm;
        s_max[1][warp] = vm;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        T m = T(0);
        for (int w = 0; w < nw; ++w) m = abs_max(m, s_max[threadIdx.x][w]);
        const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(static_cast<double>(m)));
        if (b > *static_cast<volatile unsigned long long*>(slots + threadIdx.x)) atomicMax(slots + threadIdx.x, b);
    }
}

// A thread's place: its line, chunk and the constants of the scans.
template <class N>
struct NestRowThread {
    using T = typename N::T;
    NestRowScan<T> c;
    NestChunk ck;
    int line, start;
    bool on;          // the thread has nodes of a line
    size_t row;       // offset of the line
};

template <class N, int K, bool RAG, bool WARP>
__device__ __forceinline__ NestRowThread<N> nest_row_thread(const LineParams<typename N::T>& lp,
                                                            const NestRowLayout<typename N::T>& a) {
    using T = typename N::T;
    NestRowThread<N> g;
    NestRowScan<T>& c = g.c;
    c.lane = threadIdx.x & 31;
    c.warp = threadIdx.x >> 5;
    c.nwarps = blockDim.x >> 5;
    c.width = a.TL < 32 ? a.TL : 32;
    if constexpr (WARP) {
        c.tl = c.lane & (a.TL - 1);
        g.line = (blockIdx.x * c.nwarps + c.warp) * (32 / a.TL) + c.lane / a.TL;
    } else {
        c.tl = threadIdx.x;
        g.line = blockIdx.x;
    }
    const bool live = c.tl < a.cut.nc;
    g.on = live && g.line < a.nlines;
    const int ci = live ? c.tl : 0;
    g.ck.cnt = !live ? 0 : (!RAG || ci < a.cut.rem) ? K : K - 1;
    g.start = RAG ? ci * (K - 1) + min(ci, a.cut.rem) : ci * K;
    const bool periodic = lp.bc == BC_PERIODIC;
    g.ck.mA = live && !periodic && ci == 0 ? 1 : 0;
    g.ck.mB = live && !periodic && ci == a.cut.nc - 1 ? N::W : 0;
    g.row = static_cast<size_t>(g.on ? g.line : 0) * lp.n;
    return g;
}

// The scans' constants of a thread (after the first loads have been issued).
template <class N, int K, bool RAG, bool WARP>
__device__ __forceinline__ void nest_row_scan_setup(const LineParams<typename N::T>& lp,
                                                    const NestRowLayout<typename N::T>& a, NestRowThread<N>& g,
                                                    NestRowShared<N>& sh) {
    using T = typename N::T;
    NestRowScan<T>& c = g.c;
    const int cnt = g.ck.cnt;
    const T D = cnt == 0 ? T(1) : (!RAG || cnt == K) ? a.pw.full * lp.d : a.pw.less * lp.d;
    T f = D, b = D;
    const int li = c.lane & (c.width - 1);
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int o = 1 << s;
        c.df[s] = f;
        c.db[s] = b;
        if (o < c.width) {
            const T u = __shfl_up_sync(kFull, f, o, c.width), v = __shfl_down_sync(kFull, b, o, c.width);
            if (li >= o) f *= u;
            if (li + o < c.width) b *= v;
        }
    }
    c.Dxf = __shfl_up_sync(kFull, f, 1, c.width);
    c.Dxb = __shfl_down_sync(kFull, b, 1, c.width);
    if (li == 0) c.Dxf = T(1);
    if (li == c.width - 1) c.Dxb = T(1);
    c.Dh = dev_exp(-lp.nu * T(a.half));
    const int last = g.start + cnt;
#pragma unroll
    for (int q = 0; q < N::W; ++q) {
        const int p = q * a.half, m = lp.bc == BC_PERIODIC ? 0 : 1;   // a wall's value starts one node later
        c.pl[q] = dev_exp(-lp.nu * T(max(p + g.start - m, 0)));
        c.pr[q] = dev_exp(-lp.nu * T(max(lp.n - p - last - m, 0)));
    }
    if constexpr (N::W == 1) c.pl[1] = c.pr[1] = T(0);
    if constexpr (!WARP) {
        if (c.lane == 31) sh.wd[c.warp] = f;
        __syncthreads();
        if (threadIdx.x == 0) {
            T p = T(1);
            for (int w = 0; w < c.nwarps; ++w) {
                sh.wdf[w] = p;
                p *= sh.wd[w];
            }
            p = T(1);
            for (int w = c.nwarps - 1; w >= 0; --w) {
                sh.wdb[w] = p;
                p *= sh.wd[w];
            }
        }
    }
}

// x (the window's own nodes set) <- H x: the outputs in out, the window's ends completed.
template <class N, int K, int M, bool RAG, bool WARP, int KM>
__device__ __forceinline__ void nest_row_inverse(const LineParams<typename N::T>& lp,
                                                 const NestCoef<typename N::V>& w,
                                                 const NestRowLayout<typename N::T>& a, const NestRowThread<N>& g,
                                                 NestRowShared<N>& sh, typename N::V* edge, typename N::V (&x)[KM],
                                                 typename N::V (&out)[K]) {
    using V = typename N::V;
    V aL, aR, cL, cR, XL, XR;
    nest_row_halo<N, K, M, RAG, WARP>(g.c, a.cut.nc, g.ck.cnt, edge, a.TL, x);
    nest_chunk_agg<N, K, M, RAG>(lp, w, a.pw, g.ck, x, aL, aR);
    nest_row_scan<N, WARP>(lp, g.c, sh, aL, aR, cL, cR, XL, XR);
    nest_chunk_finish<N, K, M, RAG>(lp, w, g.ck, x, cL, cR, [&](int dir) { return dir ? XR : XL; }, out);
}

// value(k), the thread's k-th node, to a field.
template <class N, int K, bool RAG, class F>
__device__ __forceinline__ void nest_row_store(typename N::T* f, int half, int start, int cnt, F value) {
    using T = typename N::T;
    if constexpr (N::W == 2) {
#pragma unroll
        for (int j = 0; j < K / 4; ++j) {
            const typename N::V a = value(4 * j), b = value(4 * j + 1), c = value(4 * j + 2), d = value(4 * j + 3);
#pragma unroll
            for (int q = 0; q < 2; ++q)
                *reinterpret_cast<float4*>(f + q * half + start + 4 * j) =
                    make_float4(N::get(a, q), N::get(b, q), N::get(c, q), N::get(d, q));
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (!RAG || k < cnt) f[start + k] = value(k);
    }
}

template <class N, int M, bool RAG, bool WARP, int MODE>
__global__ void __launch_bounds__(N::W == 2 ? 256 : 512, N::W == 2 ? 2 : 1)
nest_rows_kernel(const __grid_constant__ LineParams<typename N::T> lp,
                 const __grid_constant__ NestCoef<typename N::V> w,
                 const __grid_constant__ NestRowArgs<typename N::T> a) {
    using V = typename N::V;
    using T = typename N::T;
    constexpr int K = kNestRowK, H = M / 2;
    extern __shared__ __align__(16) unsigned char nest_row_sm[];
    V* edge = reinterpret_cast<V*>(nest_row_sm);      // two sets of 2 H values per thread (block teams)
    __shared__ NestRowShared<N> sh;
    NestRowThread<N> g = nest_row_thread<N, K, RAG, WARP>(lp, a);
    const int start = g.start, cnt = g.ck.cnt, line = g.line;
    const size_t row = g.row;

    V x[K + M], out[K];
    nest_row_load<N, K, RAG, H>(a.A + row, a.half, start, cnt, g.on, x);
    if (a.ahead) {
        // the fields that this line needs later, and the first one of the line after the resident ones, into L2
        const int step = 128 / sizeof(T);
        const size_t next = static_cast<size_t>(line + a.ahead < a.nlines ? line + a.ahead : a.nlines - 1) * lp.n;
        for (int p = g.c.tl * step; p < lp.n; p += a.TL * step) {
            if constexpr (MODE == NEST_ROW_PASS) {
                nest_prefetch(a.B + row + p);
                nest_prefetch(a.E + row + p);
                nest_prefetch(a.w + row + p);
            }
            nest_prefetch(a.A + next + p);
        }
    }
    nest_row_scan_setup<N, K, RAG, WARP>(lp, a, g, sh);

    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge, x, out);
    if constexpr (MODE == NEST_ROW_PASS) nest_row_load<N, K, RAG, H>(a.B + row, a.half, start, cnt, g.on, x);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if constexpr (MODE == NEST_ROW_PASS) x[H + k] = N::add(x[H + k], out[k]);
        else x[H + k] = out[k];
    }
    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge + 2 * H * a.TL, x, out);

    if constexpr (MODE == NEST_ROW_COPY) {
        if (g.on) nest_row_store<N, K, RAG>(a.w + row, a.half, start, cnt, [&](int k) { return out[k]; });
    } else {
        RedAcc<T> red{T(0), T(0)};
        const bool wall_row = a.fix && (line == 0 || line == a.nlines - 1);
        auto put = [&](T h, T e, T o, int p) {
            const T nw = o + (e + h);
            red.dmax = abs_max(red.dmax, fabs(nw - o));
            red.vmax = abs_max(red.vmax, fabs(nw));
            return a.fix && (wall_row || p == 0 || p == lp.n - 1) ? a.wall : nw;
        };
        if constexpr (N::W == 2) {
#pragma unroll
            for (int j = 0; j < K / 4; ++j)
                if (g.on) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int p = q * a.half + start + 4 * j;
                        const float4 e = *reinterpret_cast<const float4*>(a.E + row + p);
                        float4* dst = reinterpret_cast<float4*>(a.w + row + p);
                        const float4 o = *dst;
                        float4 v;
                        v.x = put(N::get(out[4 * j], q), e.x, o.x, p);
                        v.y = put(N::get(out[4 * j + 1], q), e.y, o.y, p + 1);
                        v.z = put(N::get(out[4 * j + 2], q), e.z, o.z, p + 2);
                        v.w = put(N::get(out[4 * j + 3], q), e.w, o.w, p + 3);
                        *dst = v;
                    }
                }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (g.on && (!RAG || k < cnt)) {
                    const size_t i = row + start + k;
                    a.w[i] = put(out[k], a.E[i], a.w[i], start + k);
                }
        }
        nest_reduce<T>(red, a.red);
    }
}

// Sixth-order model on independent lines: one whole iteration (fch1d.cpp).  With f = f(v), p the pointwise
// lagged product (fch_pointwise), G = c_eta v - c_f f + c_p p and A = (3 + c_eta) v - c_f f, the terms collect by
// linearity of H into
//   q = H G - A,   z = H^2 v^n + H q - q,   v <- H z,   Lap v <- (v - z) / a,
// three inverses with the line in registers; v and Lap v are written once, H^2 v^n is read once, v is read again
// (from L2) where holding it would spill.
// Bound: latency at 16 warps a SM (1.5 of 4 instructions a cycle; loads and the shuffles of three scans): 16384 lines of
// 1024 nodes, FP32, M = 6: 107 us an iteration = 3100 GB/s of the 20 B a point, fourteen kernels took 606; FP64, 4096
// lines: 670 us, FP64 units, against 1856.
template <typename T>
struct NestFchArgs : NestRowLayout<T>, FchCoef<T> {
    T* v;
    T* lap;
    const T* h2;
    unsigned long long* red;
};

template <class N, int M, bool RAG, bool WARP>
__global__ void __launch_bounds__(N::W == 2 ? 256 : 512, N::W == 2 ? 2 : 1)
nest_fch_kernel(const __grid_constant__ LineParams<typename N::T> lp,
                const __grid_constant__ NestCoef<typename N::V> w,
                const __grid_constant__ NestFchArgs<typename N::T> a) {
    using V = typename N::V;
    using T = typename N::T;
    constexpr int K = kNestRowK, H = M / 2;
    extern __shared__ __align__(16) unsigned char nest_row_sm[];
    V* edge = reinterpret_cast<V*>(nest_row_sm);
    __shared__ NestRowShared<N> sh;
    NestRowThread<N> g = nest_row_thread<N, K, RAG, WARP>(lp, a);
    const int start = g.start, cnt = g.ck.cnt;
    const size_t row = g.row;
    const V m1 = N::splat(T(-1)), c3 = N::splat(a.c3), nf = N::splat(-a.c_f);
    auto cube = [&](V x) { return N::mul(x, N::fma(x, N::add(x, N::splat(T(-3))), N::splat(T(2)))); };   // f(v)

    V x[K + M], out[K];
    nest_row_load<N, K, RAG, H>(a.v + row, a.half, start, cnt, g.on, x);
    {
        V l[K];
        nest_row_load<N, K, RAG, 0>(a.lap + row, a.half, start, cnt, g.on, l);
        const V e2 = N::splat(a.eps2), ee = N::splat(a.eta_eps2), ce = N::splat(a.c_eta), cp = N::splat(a.c_p);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const V v = x[H + k], f = cube(v);
            const V fp = N::fma(v, N::fma(N::splat(T(3)), v, N::splat(T(-6))), N::splat(T(2)));
            const V p = N::fma(f, fp, N::mul(m1, N::fma(N::mul(e2, fp), l[k], N::mul(ee, f))));
            x[H + k] = N::fma(cp, p, N::fma(nf, f, N::mul(ce, v)));
        }
    }
    nest_row_scan_setup<N, K, RAG, WARP>(lp, a, g, sh);
    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge, x, out);
    nest_row_load<N, K, RAG, H>(a.v + row, a.half, start, cnt, g.on, x);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const V v = x[H + k];
        x[H + k] = N::fma(m1, N::fma(nf, cube(v), N::mul(c3, v)), out[k]);           // q
    }
    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge + 2 * H * a.TL, x, out);
    {
        V h2[K];
        nest_row_load<N, K, RAG, 0>(a.h2 + row, a.half, start, cnt, g.on, h2);
#pragma unroll
        for (int k = 0; k < K; ++k) x[H + k] = N::add(h2[k], N::fma(m1, x[H + k], out[k]));   // z
    }
    // (the first set of edges is free again: every thread has passed the second inverse's barriers)
    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge, x, out);
    RedAcc<T> red{T(0), T(0)};
    if (g.on) {
        const V ia = N::splat(a.inv_a);
        nest_row_store<N, K, RAG>(a.lap + row, a.half, start, cnt,
                                  [&](int k) { return N::mul(ia, N::fma(m1, x[H + k], out[k])); });
        nest_row_load<N, K, RAG, H>(a.v + row, a.half, start, cnt, true, x);
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (!RAG || k < cnt) {
                const V e = N::fma(m1, x[H + k], out[k]);
#pragma unroll
                for (int q = 0; q < N::W; ++q) {
                    red.dmax = abs_max(red.dmax, fabs(N::get(e, q)));
                    red.vmax = abs_max(red.vmax, fabs(N::get(out[k], q)));
                }
            }
        nest_row_store<N, K, RAG>(a.v + row, a.half, start, cnt, [&](int k) { return out[k]; });
    }
    nest_reduce<T>(red, a.red);
}

// Four nodes 4j .. 4j + 3 of a thread's chunk.
template <class N, bool RAG>
__device__ __forceinline__ void nest_row_load4(const typename N::T* f, int half, int start, int cnt, int j,
                                               typename N::V (&x)[4]) {
    using T = typename N::T;
    if constexpr (N::W == 2) {
        const float4 lo = *reinterpret_cast<const float4*>(f + start + 4 * j);
        const float4 hi = *reinterpret_cast<const float4*>(f + half + start + 4 * j);
        x[0] = N::pair(lo.x, hi.x), x[1] = N::pair(lo.y, hi.y), x[2] = N::pair(lo.z, hi.z), x[3] = N::pair(lo.w, hi.w);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = !RAG || 4 * j + i < cnt ? f[start + 4 * j + i] : T(0);
    }
}
template <class N, bool RAG>
__device__ __forceinline__ void nest_row_store4(typename N::T* f, int half, int start, int cnt, int j,
                                                const typename N::V (&x)[4]) {
    if constexpr (N::W == 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            *reinterpret_cast<float4*>(f + q * half + start + 4 * j) =
                make_float4(N::get(x[0], q), N::get(x[1], q), N::get(x[2], q), N::get(x[3], q));
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (!RAG || 4 * j + i < cnt) f[start + 4 * j + i] = x[i];
    }
}

// Sixth-order model in 2D, the x pass that opens an iteration (fch2d.cpp): from W and H_y W
//   v = H_x H_y W,  X W = v - H_x W - H_y W + W,  a Lap v = 2v - H_x W - H_y W,
// and from these, point by point, the fields of the y pass
//   p = A + E,  q = -(s1 + 2p),  r = 2 s1 + E,  u = -E - X W,  z = M^{-2} v^n + X W - W
// with s1 = 2A + B.  v goes out before the second inverse and is read again after it, so that one inverse's
// registers are live at a time.
// Bound: latency of two line chains at 16 warps a SM and 40 B a point: 2048^2 FP32, M = 6: 60 us = 2800 GB/s.  The whole
// iteration (y pass 97, x pass 28, H_y W 22, this 60 us) takes 210 us; fourteen sweeps and twelve other kernels took 455.
template <typename T>
struct NestFch2Args : NestRowLayout<T>, FchCoef<T> {
    const T *W, *hy, *m2;
    T *v, *p, *q, *r, *u, *z;
    unsigned long long* red;
};

template <class N, int M, bool RAG, bool WARP>
__global__ void __launch_bounds__(N::W == 2 ? 256 : 512, N::W == 2 ? 2 : 1)
nest_fch2_kernel(const __grid_constant__ LineParams<typename N::T> lp,
                 const __grid_constant__ NestCoef<typename N::V> w,
                 const __grid_constant__ NestFch2Args<typename N::T> a) {
    using V = typename N::V;
    using T = typename N::T;
    constexpr int K = kNestRowK, H = M / 2;
    extern __shared__ __align__(16) unsigned char nest_row_sm[];
    V* edge = reinterpret_cast<V*>(nest_row_sm);
    __shared__ NestRowShared<N> sh;
    NestRowThread<N> g = nest_row_thread<N, K, RAG, WARP>(lp, a);
    const int start = g.start, cnt = g.ck.cnt;
    const size_t row = g.row;
    const V m1 = N::splat(T(-1)), two = N::splat(T(2)), three = N::splat(T(3));
    V x[K + M], out[K];
    RedAcc<T> red{T(0), T(0)};
    nest_row_load<N, K, RAG, H>(a.hy + row, a.half, start, cnt, g.on, x);
    nest_row_scan_setup<N, K, RAG, WARP>(lp, a, g, sh);
    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge, x, out);
    if (g.on) {
#pragma unroll
        for (int j = 0; j < K / 4; ++j) {
            V o[4];
            nest_row_load4<N, RAG>(a.v + row, a.half, start, cnt, j, o);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (!RAG || 4 * j + i < cnt) {
                    const V e = N::fma(m1, o[i], out[4 * j + i]);
#pragma unroll
                    for (int q = 0; q < N::W; ++q) {
                        red.dmax = abs_max(red.dmax, fabs(N::get(e, q)));
                        red.vmax = abs_max(red.vmax, fabs(N::get(out[4 * j + i], q)));
                    }
                }
        }
        nest_row_store<N, K, RAG>(a.v + row, a.half, start, cnt, [&](int k) { return out[k]; });
    }
    nest_row_load<N, K, RAG, H>(a.W + row, a.half, start, cnt, g.on, x);
    nest_row_inverse<N, K, M, RAG, WARP>(lp, w, a, g, sh, edge + 2 * H * a.TL, x, out);
    if (g.on) {
        const V e2 = N::splat(a.eps2), ee = N::splat(a.eta_eps2), cp = N::splat(a.c_p), nf = N::splat(-a.c_f);
        const V c3 = N::splat(a.c3), c32 = N::splat(a.c32), nf2 = N::splat(T(-2) * a.c_f);
        const V ia = N::splat(a.inv_a);
#pragma unroll
        for (int j = 0; j < K / 4; ++j) {
            V v[4], hy[4], m2[4], P[4], Q[4], R[4], U[4];
            nest_row_load4<N, RAG>(a.v + row, a.half, start, cnt, j, v);
            nest_row_load4<N, RAG>(a.hy + row, a.half, start, cnt, j, hy);
            nest_row_load4<N, RAG>(a.m2 + row, a.half, start, cnt, j, m2);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const V W = x[H + 4 * j + i], t = v[i];
                const V h = N::add(out[4 * j + i], hy[i]);                              // H_x W + H_y W
                const V lap = N::mul(ia, N::fma(two, t, N::mul(m1, h)));
                const V xw = N::add(N::fma(m1, h, t), W);
                const V E = N::fma(N::mul(m1, three), W, xw);
                const V f = N::mul(t, N::fma(t, N::add(t, N::splat(T(-3))), two));
                const V fp = N::fma(t, N::fma(three, t, N::splat(T(-6))), two);
                const V pp = N::fma(f, fp, N::mul(m1, N::fma(N::mul(e2, fp), lap, N::mul(ee, f))));
                const V s1 = N::fma(cp, pp, N::fma(nf2, f, N::mul(c32, t)));
                P[i] = N::add(N::fma(nf, f, N::mul(c3, t)), E);
                Q[i] = N::mul(m1, N::fma(two, P[i], s1));
                R[i] = N::fma(two, s1, E);
                U[i] = N::mul(m1, N::add(E, xw));
                m2[i] = N::add(m2[i], N::fma(m1, W, xw));
            }
            nest_row_store4<N, RAG>(a.p + row, a.half, start, cnt, j, P);
            nest_row_store4<N, RAG>(a.q + row, a.half, start, cnt, j, Q);
            nest_row_store4<N, RAG>(a.r + row, a.half, start, cnt, j, R);
            nest_row_store4<N, RAG>(a.u + row, a.half, start, cnt, j, U);
            nest_row_store4<N, RAG>(a.z + row, a.half, start, cnt, j, m2);
        }
    }
    nest_reduce<T>(red, a.red);
}

}  // namespace molt
