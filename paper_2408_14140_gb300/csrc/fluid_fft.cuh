// The spectral solves of the fluid step: a real field of n0 x n1 x n2 values
// as its half spectrum in x, n2 planes of n1 rows of n0/2 complex points, and
// the points kx = n0/2 beside it (n2 rows of n1).  Five passes over these:
//   x forward (from the real field), y forward,
//   z: forward, the operator's inverse symbol, inverse -- in one kernel,
//   y inverse, x inverse (to the real field).
// Every pass reads and writes each point once, so a field moves 10 times its
// bytes, half of what a complex field with a zero imaginary part would.
//
// x forward takes two rows (planes 2z', 2z'+1) as the real and the imaginary
// part of one complex line Z and separates their spectra A, B by
// A(k) = (Z(k) + conj Z(n0-k))/2, B(k) = (Z(k) - conj Z(n0-k))/2i; x inverse
// puts Z = A + iB together again.
//
// Two denser packings measured worse errors in FP32 and were not kept: planes
// packed through all passes (the symbols of kz and kz + n2/2 applied to the
// packed spectrum) gave 1.2 to 1.5 times the projection's error of u, and
// kx = 0 and n0/2 sharing a point up to 4 times its error of p, since the
// rounding of the large modes then reaches the nearly checkerboard ones, which
// the pressure solve amplifies by up to 1e5.
#pragma once

#include "fft_core.cuh"

namespace gbib {

// Operators diagonal in Fourier space.
enum { kSolveHelmholtz = 0, kSolveDivGrad = 1 };
struct SymbolArgs {
    int kind;
    double scale;  // 1 / (points of the transform) and, for div grad, the constant factor
    double g;      // Helmholtz: 4 coef / h^2
    float scale32, g32;
    SymbolArgs(int k, double s, double c) : kind(k), scale(s), g(c), scale32((float)s), g32((float)c) {}
    __device__ __forceinline__ void get(double &s, double &c) const { s = scale, c = g; }
    __device__ __forceinline__ void get(float &s, float &c) const { s = scale32, c = g32; }
};

// The half spectrum of one field: `c` the points kx < n0/2, `ny` those of
// kx = n0/2, one a row; fields follow one another in both.  The points of
// 2^logg adjacent rows (or of any number, if nylog is 0) lie side by side, a
// group every 2^(logg + nylog).  The projection keeps them at the start of the
// right-hand side's rows that the same CTA of the x pass reads, so that it needs
// no memory beyond two scalar fields (a point in each row instead cost the z pass
// of 64x64x128 in FP32 2 us of 35 a call).
template <class A> struct Spectrum {
    typename A::Mem *c, *ny;
    int logg, nylog;
};
// The place of point i of 2^logg side by side, 2^(logg + step) a group.
__device__ __forceinline__ long long grouped(long long i, int logg, int step) {
    return ((i >> logg) << (logg + step)) + (i & ((1LL << logg) - 1));
}
// Lines (row pairs) of one CTA of the x passes.
template <class A> __host__ __device__ constexpr int x_lines(int logN) {
    return (1 << logN) / A::points(logN) >= 128 ? 1 : 128 / ((1 << logN) / A::points(logN));
}

// The launches (one field, or ncomp fields one after another in memory).
template <class A>
struct FftGrid {
    int n[3], log2n[3];
    const typename A::W *tw;                    // [kTwiddles]
    const typename A::Mem *trig;                // [kRoots] (cos, sin)(2 pi k / kRoots)
};

// The scale of a line from its threads' points: mag[] the larger component's
// magnitude of each point.  FAST_T: the line's threads are neighbours in the
// CTA; else `lanes` lines interleave.  slot[0], slot[1]: the lines' words for
// the maximum and the sum, zero before (unused with FAST_T up to a warp).
template <class A, int LOGN, bool PAIR, int M, int TPL, bool FAST_T>
__device__ __forceinline__ LineScale points_scale(const int (&mag)[M], int *max_slot, int *sum_slot, int line, int lanes) {
    using R = typename A::Real;
    int h = 0;
#pragma unroll
    for (int m = 0; m < M; ++m) h = max(h, mag[m]);
    if (FAST_T) {
#pragma unroll
        for (int o = (TPL < 32 ? TPL : 32) / 2; o > 0; o >>= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    } else {
        for (int o = lanes; o < 32; o <<= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    }
    const bool shared = !FAST_T || TPL > 32, first = FAST_T ? (threadIdx.x & 31) == 0 : (int)(threadIdx.x & 31) < lanes;
    if (shared) {
        if (first) atomicMax(max_slot + line, h);
        __syncthreads();
        h = max_slot[line];
    }
    const int emax = exponent_of<R>(h);
    unsigned s = 0;
#pragma unroll
    for (int m = 0; m < M; ++m) s += bound_of<R>(mag[m], emax);
    if (FAST_T) {
#pragma unroll
        for (int o = (TPL < 32 ? TPL : 32) / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    } else {
        for (int o = lanes; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (shared) {
        if (first) atomicAdd((unsigned *)sum_slot + line, s);
        __syncthreads();
        s = (unsigned)sum_slot[line];
    }
    return line_scale<A, LOGN, PAIR>(emax, s);
}

// A thread's points of a line to the transform's arithmetic and back; returns
// the line's scale.
template <class A, int LOGN, int E, int TPL, bool FAST_T>
__device__ __forceinline__ LineScale points_in(const typename A::Mem (&z)[E], typename A::C (&v)[E], int *max_slot,
                                         int *sum_slot, int line, int lanes) {
    if constexpr (A::kFixed) {
        int mag[E];
#pragma unroll
        for (int m = 0; m < E; ++m) mag[m] = max(magnitude(z[m].x), magnitude(z[m].y));
        const LineScale sc = points_scale<A, LOGN, false, E, TPL, FAST_T>(mag, max_slot, sum_slot, line, lanes);
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = typename A::C{to_fixed(z[m].x, sc.first), to_fixed(z[m].y, sc.first)};
        return sc;
    } else {
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = typename A::C{z[m].x, z[m].y};
        return {0, 0, 0};
    }
}
template <class A> __device__ __forceinline__ typename A::Mem point_out(typename A::C v, int unit) {
    typename A::Mem z;
    if constexpr (A::kFixed) {
        from_fixed(v.x, unit, z.x);
        from_fixed(v.y, unit, z.y);
    } else {
        z.x = v.x;
        z.y = v.y;
    }
    return z;
}

// ---- x: the real field's row pairs <-> the half spectrum ----------------------
enum { kXForward = 0, kXField = 1, kXPressure = 2 };

template <class A, int LOGN> struct XShape {
    static constexpr int N = 1 << LOGN, E = A::points(LOGN), TPL = N / E;
    static constexpr int LPC = x_lines<A>(LOGN);
    static constexpr int T = TPL * LPC;
    static constexpr int PITCH = N + N / E;                 // one point of padding per E: conflict-free writes
    static constexpr size_t smem = (size_t)LPC * PITCH * sizeof(typename A::C);
};

// kXField writes the field; kXPressure writes p' over the old pressure and
// beside it, for FP64 fields, the difference p_old - p', whose gradient is all
// the projection needs, and the difference's largest magnitude (high word) in
// *maxold; for FP32 fields p_old itself, since the difference's rounding would
// show in u.
template <class A, int LOGN, int MODE>
__global__ void __launch_bounds__(XShape<A, LOGN>::T)
k_fft_x(const typename A::Real *src, Spectrum<A> sp, typename A::Real *__restrict__ dst, typename A::Real *old, int *__restrict__ maxold, int log1, int log2, const typename A::W *__restrict__ tw) {
    using S = XShape<A, LOGN>;
    using C = typename A::C;
    using R = typename A::Real;
    using Mem = typename A::Mem;
    constexpr int N = S::N, E = S::E, TPL = S::TPL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_line[2][S::LPC];
    C *sm = (C *)smem_raw;
    const int t = threadIdx.x % TPL, l = threadIdx.x / TPL;
    const long long line = (long long)blockIdx.x * S::LPC + l;  // z' n1 + y
    const long long n1 = 1LL << log1, plane = n1 << LOGN;
    const long long row = ((line >> log1) * 2 * n1 + (line & (n1 - 1))) << LOGN;  // of plane 2z'
    const long long comp = (long long)blockIdx.y << (LOGN + log1 + log2);
    Mem *ca = sp.c + ((comp + row) >> 1), *cb = ca + (plane >> 1);  // the two rows' half spectra
    Mem *na = sp.ny + grouped((comp + row) >> LOGN, sp.logg, sp.nylog), *nb = na + (n1 << sp.nylog);  // and their points n0/2
    if (A::kFixed && TPL > 32) {
        if (threadIdx.x < 2 * S::LPC) (&s_line[0][0])[threadIdx.x] = 0;
        __syncthreads();
    }
    auto at = [l](int p) { return l * S::PITCH + p + p / E; };
    grid_dep_wait();
    C v[E];
    LineScale sc = {0, 0, 0};
    constexpr bool kPair = MODE != kXForward;
    if constexpr (MODE == kXForward) {
        Mem z[E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const R *r = src + comp + row + t + TPL * m;
            z[m] = Mem{r[0], r[plane]};
        }
        sc = points_in<A, LOGN, E, TPL, true>(z, v, s_line[0], s_line[1], l, 0);
    } else {
        // Z(k) = A(k) + i B(k), Z(n0 - k) = conj A(k) + i conj B(k); real points
        // at 0 and n0/2.  The sums are formed in the transform's arithmetic.
        Mem a[E], b[E];
        C va[E], vb[E];
        int mag[2 * E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int p = t + TPL * m, k = m >= E / 2 ? (N - p) & (N / 2 - 1) : p;
            const bool mid = m == E / 2 && t == 0;
            a[m] = *(mid ? na : ca + k), b[m] = *(mid ? nb : cb + k);
            if (mid || p == 0) a[m].y = b[m].y = 0;
            mag[2 * m] = max(magnitude(a[m].x), magnitude(a[m].y));
            mag[2 * m + 1] = max(magnitude(b[m].x), magnitude(b[m].y));
        }
        if constexpr (A::kFixed) sc = points_scale<A, LOGN, kPair, 2 * E, TPL, true>(mag, s_line[0], s_line[1], l, 0);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            if constexpr (A::kFixed) {
                va[m] = C{to_fixed(a[m].x, sc.first), to_fixed(a[m].y, sc.first)};
                vb[m] = C{to_fixed(b[m].x, sc.first), to_fixed(b[m].y, sc.first)};
            } else {
                va[m] = C{a[m].x, a[m].y};
                vb[m] = C{b[m].x, b[m].y};
            }
            v[m] = m >= E / 2 ? C{va[m].x + vb[m].y, vb[m].x - va[m].y} : C{va[m].x - vb[m].y, va[m].y + vb[m].x};
        }
    }
    fft_line<A, LOGN, MODE != kXForward, kPair>(v, t, sm, at, tw, sc.sum);
    const int unit = sc.last;
    grid_dep_launch();
    if constexpr (MODE == kXForward) {
        // separation: the thread's lower points k < n0/2 and their mirrors from
        // shared memory; twice A or B comes in (one more bit of the integers)
        const int half = unit == kUnitNan ? unit : unit - 1;
        auto put = [&](Mem *at, decltype(v[0].x) x, decltype(v[0].x) y) {
            const Mem z = point_out<A>(C{x, y}, half);
            *at = A::kFixed ? z : Mem{(R)0.5 * z.x, (R)0.5 * z.y};
        };
        __syncthreads();
#pragma unroll
        for (int m = 0; m < E; ++m)
            if (m >= E / 2 || m == 0) sm[at(t + TPL * m)] = v[m];
        __syncthreads();
#pragma unroll
        for (int m = 0; m < E / 2; ++m) {
            const int k = t + TPL * m;
            const C n = sm[at((N - k) & (N - 1))];
            put(ca + k, v[m].x + n.x, v[m].y - n.y);
            put(cb + k, v[m].y + n.y, n.x - v[m].x);
        }
        if (t == 0) {
            const C n = v[E / 2];
            put(na, n.x + n.x, n.x - n.x);
            put(nb, n.y + n.y, n.y - n.y);
        }
    } else {
        int big = 0;
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const Mem z = point_out<A>(v[m], unit);
            const long long i0 = comp + row + t + TPL * m, i1 = i0 + plane;
            if (MODE == kXPressure) {
                const R a = dst[i0], b = dst[i1];
                const R c = sizeof(R) == 8 ? a - z.x : a, e = sizeof(R) == 8 ? b - z.y : b;
                old[i0] = c;
                old[i1] = e;
                if (sizeof(R) == 8) big = max(big, max(magnitude(c), magnitude(e)));
            }
            dst[i0] = z.x;
            dst[i1] = z.y;
        }
        if (MODE == kXPressure && sizeof(R) == 8) {
            big = __reduce_max_sync(0xffffffffu, big);
            if ((threadIdx.x & 31) == 0 && big > *(volatile int *)maxold) atomicMax(maxold, big);
        }
    }
}

// ---- y: lines of stride n0/2 = 2^logr points, adjacent lines in adjacent threads
template <class A, int LOGN> struct YShape {
    static constexpr int N = 1 << LOGN, E = A::points(LOGN), TPL = N / E;
    static constexpr int L0 = A::lanes(LOGN), LANES = L0 * TPL >= 128 ? L0 : 128 / TPL;
    static constexpr int T = TPL * LANES;
    static constexpr size_t smem = (size_t)LANES * N * sizeof(typename A::C);
};

template <class A, int LOGN, bool INV>
__global__ void __launch_bounds__(YShape<A, LOGN>::T)
k_fft_y(Spectrum<A> sp, int logr, int log2, const typename A::W *__restrict__ tw) {
    using S = YShape<A, LOGN>;
    using C = typename A::C;
    constexpr int E = S::E, TPL = S::TPL, LANES = S::LANES;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_line[2][LANES];
    C *sm = (C *)smem_raw;
    const int t = threadIdx.x / LANES, l = threadIdx.x % LANES;
    // LANES lines in (z, kx) order, after them the n2 lines of kx = n0/2
    const int regular = (1 << (logr + log2)) / LANES;
    const bool last = (int)blockIdx.x >= regular;
    const int q = (last ? (int)blockIdx.x - regular : (int)blockIdx.x) * LANES + l;
    const bool active = !last || q < 1 << log2;
    const int step = last ? sp.nylog : logr;  // log2 of the points' stride (grouped in the last lines)
    typename A::Mem *cl = last ? sp.ny + ((((long long)blockIdx.y << log2) + q) << (LOGN + sp.nylog))
                               : sp.c + ((long long)blockIdx.y << (LOGN + logr + log2)) +
                                     ((long long)(q >> logr) << (LOGN + logr)) + (q & ((1 << logr) - 1));
    if (A::kFixed) {
        for (int i = threadIdx.x; i < 2 * LANES; i += S::T) (&s_line[0][0])[i] = 0;
        __syncthreads();
    }
    grid_dep_wait();
    typename A::Mem z[E];
#pragma unroll
    for (int m = 0; m < E; ++m) z[m] = last ? typename A::Mem{0, 0} : cl[(long long)(t + TPL * m) << step];
    if (last && active)
#pragma unroll
        for (int m = 0; m < E; ++m) z[m] = cl[grouped(t + TPL * m, sp.logg, step)];
    C v[E];
    const LineScale sc = points_in<A, LOGN, E, TPL, false>(z, v, s_line[0], s_line[1], l, LANES);
    auto at = [l](int p) { return p * LANES + l; };
    fft_line<A, LOGN, INV>(v, t, sm, at, tw, sc.sum);
    grid_dep_launch();
#pragma unroll
    for (int m = 0; m < E; ++m) {
        z[m] = point_out<A>(v[m], sc.last);
        if (!last) cl[(long long)(t + TPL * m) << step] = z[m];
    }
    if (last && active)
#pragma unroll
        for (int m = 0; m < E; ++m) cl[grouped(t + TPL * m, sp.logg, step)] = z[m];
}

// ---- z: forward, symbol, inverse --------------------------------------------
template <class A, int LOGN> struct ZShape {
    static constexpr int N = 1 << LOGN, E = A::points(LOGN), TPL = N / E;
    static constexpr int L0 = A::lanes(LOGN), LANES = L0 * TPL >= 128 ? L0 : 128 / TPL;
    static constexpr int T = TPL * LANES;
    static constexpr int MINB = (A::kFixed ? 896 : 768) / T;  // 28 warps (24) an SM: 72 registers (80)
    static constexpr size_t points = (size_t)LANES * N * sizeof(typename A::C);
    static constexpr size_t smem = points + (size_t)(N / 2 + 1) * LANES * sizeof(typename A::Real);
};

// The operator along a line (kx, ky), in the squared sine and cosine sz, cz of
// kz's half angle: Helmholtz 1 + g (sx + sy + sz); D G over -4/h^2,
// (sx cy + sy cx) cz + (cx cy) sz, as p cz + q sz.  inverse(): the scale over
// it, 0 on D G's null modes.
template <typename R> struct LineSymbol {
    R p, q, scale;
    bool helmholtz;
    __device__ __forceinline__ LineSymbol(const SymbolArgs &sy, R sx, R cx, R sy2, R cy) {
        R g;
        sy.get(scale, g);
        helmholtz = sy.kind == kSolveHelmholtz;
        p = helmholtz ? fma(g, sx + sy2, (R)1) : sx * cy + sy2 * cx;
        q = helmholtz ? g : cx * cy;
    }
    __device__ __forceinline__ R inverse(R sz, R cz) const {
        const R d = helmholtz ? fma(q, sz, p) : fma(p, cz, q * sz);
        if (!helmholtz && d <= (R)3e-13) return (R)0;
        return scale / d;
    }
};

template <class A, int LOGN>
__global__ void __launch_bounds__(ZShape<A, LOGN>::T, ZShape<A, LOGN>::MINB)
k_fft_z(Spectrum<A> sp, int logr, int log1, SymbolArgs sy, const typename A::W *__restrict__ tw,
        const typename A::Mem *__restrict__ trig) {
    using S = ZShape<A, LOGN>;
    using C = typename A::C;
    using R = typename A::Real;
    using Mem = typename A::Mem;
    constexpr int N = S::N, E = S::E, TPL = S::TPL, LANES = S::LANES;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_line[4][LANES];
    C *sm = (C *)smem_raw;
    R *fs = (R *)(smem_raw + S::points);  // [N/2 + 1][LANES] inverse symbols (even in kz)
    const int l = threadIdx.x % LANES, t = threadIdx.x / LANES;
    // LANES lines in (ky, kx) order, after them the n1 lines of kx = n0/2
    const int regular = (1 << (logr + log1)) / LANES;
    const bool last = (int)blockIdx.x >= regular;
    const int q = (last ? (int)blockIdx.x - regular : (int)blockIdx.x) * LANES + l;
    const bool active = !last || q < 1 << log1;
    const int kx = last ? 1 << logr : q & ((1 << logr) - 1), ky = last ? q & ((1 << log1) - 1) : q >> logr;
    const int shift = last ? log1 + sp.nylog : logr + log1;  // log2 of the points' stride
    Mem *cl = (last ? sp.ny + grouped(q, sp.logg, sp.nylog) : sp.c + q) + ((long long)blockIdx.y << (LOGN + shift));
    if (A::kFixed)
        for (int i = threadIdx.x; i < 4 * LANES; i += S::T) (&s_line[0][0])[i] = 0;
    {
        // the thread's lane's symbol at kz = t, t + TPL, ... <= n2/2
        const Mem hx = __ldg(trig + kx * (kRoots / 4 >> logr)), hy = __ldg(trig + ky * (kRoots / 2 >> log1));
        const LineSymbol<R> sym(sy, hx.y * hx.y, hx.x * hx.x, hy.y * hy.y, hy.x * hy.x);
        for (int kz = t; kz <= N / 2; kz += TPL) {
            const Mem hz = __ldg(trig + kz * (kRoots / 2 / N));
            fs[kz * LANES + l] = sym.inverse(hz.y * hz.y, hz.x * hz.x);
        }
    }
    if (A::kFixed) __syncthreads();
    grid_dep_wait();
    Mem z[E];
#pragma unroll
    for (int m = 0; m < E; ++m) z[m] = active ? cl[(long long)(t + TPL * m) << shift] : Mem{0, 0};
    C v[E];
    LineScale sc = points_in<A, LOGN, E, TPL, false>(z, v, s_line[0], s_line[1], l, LANES);
    auto at = [l](int p) { return p * LANES + l; };
    fft_line<A, LOGN, false>(v, t, sm, at, tw, sc.sum);
#pragma unroll
    for (int m = 0; m < E; ++m) {
        z[m] = point_out<A>(v[m], sc.last);
    }
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = t + TPL * m;
        const R f = fs[(k <= N / 2 ? k : N - k) * LANES + l];
        z[m] = Mem{f * z[m].x, f * z[m].y};
    }
    sc = points_in<A, LOGN, E, TPL, false>(z, v, s_line[2], s_line[3], l, LANES);
    fft_line<A, LOGN, true>(v, t, sm, at, tw, sc.sum);
    grid_dep_launch();
    if (active) {
#pragma unroll
        for (int m = 0; m < E; ++m) {
            z[m] = point_out<A>(v[m], sc.last);
            cl[(long long)(t + TPL * m) << shift] = z[m];
        }
    }
}

// ---- launches (defined per arithmetic in their own translation units) --------
template <class A> cudaError_t fft_x(int mode, const FftGrid<A> &g, int ncomp, const typename A::Real *src,
                                     Spectrum<A> sp, typename A::Real *dst, typename A::Real *old, int *maxold, cudaStream_t s);
template <class A> cudaError_t fft_y(bool inverse, const FftGrid<A> &g, int ncomp, Spectrum<A> sp, cudaStream_t s);
template <class A> cudaError_t fft_z(const FftGrid<A> &g, int ncomp, Spectrum<A> sp, const SymbolArgs &sy,
                                     cudaStream_t s);

template <typename Kern, typename... Args>
inline cudaError_t launch_fft(Kern kern, dim3 grid, int threads, size_t smem, cudaStream_t s, Args... args) {
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_pdl(kern, grid, dim3(threads), smem, s, args...);
}

template <class A, int LOGN>
cudaError_t launch_x(int mode, const FftGrid<A> &g, int ncomp, const typename A::Real *src, Spectrum<A> sp,
                     typename A::Real *dst, typename A::Real *old, int *maxold, cudaStream_t s) {
    using S = XShape<A, LOGN>;
    const dim3 grid(g.n[1] * (g.n[2] / 2) / S::LPC, ncomp);
    auto k = mode == kXForward ? k_fft_x<A, LOGN, kXForward>
                               : (mode == kXField ? k_fft_x<A, LOGN, kXField> : k_fft_x<A, LOGN, kXPressure>);
    return launch_fft(k, grid, S::T, S::smem, s, src, sp, dst, old, maxold, g.log2n[1], g.log2n[2], g.tw);
}
template <class A, int LOGN>
cudaError_t launch_y(bool inverse, const FftGrid<A> &g, int ncomp, Spectrum<A> sp, cudaStream_t s) {
    using S = YShape<A, LOGN>;
    const dim3 grid(g.n[0] / 2 * g.n[2] / S::LANES + (g.n[2] + S::LANES - 1) / S::LANES, ncomp);
    auto k = inverse ? k_fft_y<A, LOGN, true> : k_fft_y<A, LOGN, false>;
    return launch_fft(k, grid, S::T, S::smem, s, sp, g.log2n[0] - 1, g.log2n[2], g.tw);
}
template <class A, int LOGN>
cudaError_t launch_z(const FftGrid<A> &g, int ncomp, Spectrum<A> sp, const SymbolArgs &sy, cudaStream_t s) {
    using S = ZShape<A, LOGN>;
    const dim3 grid(g.n[0] / 2 * g.n[1] / S::LANES + (g.n[1] + S::LANES - 1) / S::LANES, ncomp);
    return launch_fft(k_fft_z<A, LOGN>, grid, S::T, S::smem, s, sp, g.log2n[0] - 1, g.log2n[1], sy, g.tw, g.trig);
}

}  // namespace gbib
