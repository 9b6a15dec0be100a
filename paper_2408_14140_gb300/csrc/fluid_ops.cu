// The fluid step around the IB forcing on one uniform periodic level
// (arXiv 2408.14140, Sec. 3.1): Step 1, the momentum predictor (Eq. 31), and
// Step 3, the level projection (Eqs. ns_lp1-ns_lp3).
//
// Grid (semi-staggered, Sec. 3.1): velocity at cell centres, [3][n2][n1][n0]
// (x fastest); pressure at nodes, [n2][n1][n0], node (i, j, k) the lower
// corner of cell (i, j, k).
//   G p  (cells)  = along x, (1/4h) sum over the cell's four x-edges of p(i+1) - p(i)
//   D V  (nodes)  = the negative adjoint of G, so the projection's Laplacian is D G
//   L_c u (cells) = 7-point Laplacian per component
// The implicit solves -- (I - nu dt/2 L_c) for Crank-Nicolson viscosity and
// D G for the pressure -- are diagonal in Fourier space on a periodic grid
// and are done exactly with FFTs (fluid_fft.cuh), so every grid axis must be
// a power of two.  Convection div(u u)^{n+1/2} is a second-order
// Godunov edge extrapolation: per face, states from both neighbours by a
// Taylor step along monotonized-central limited slopes, the normal velocity
// from the Burgers Riemann solution of the two normal states, the state
// upwinded by it, and the flux difference over the cell.
//
// The stencil kernels march along z: a thread owns a column (i, j) of a chunk
// of planes, keeps what the next plane needs again in registers and reads the
// in-plane neighbours through L1.  All sizes are powers of two, so periodic
// indices are masks.
#include "fluid_fft.cuh"

namespace gbib {

struct LevelDims {
    int n0, n1, n2, zc;  // zc: planes of one CTA's chunk
};

// The thread's column and its chunk of planes.
struct Column {
    int i, j, k0, k1;
    __device__ __forceinline__ Column(const LevelDims &d)
        : i(blockIdx.x * blockDim.x + threadIdx.x), j(blockIdx.y * blockDim.y + threadIdx.y), k0(blockIdx.z * d.zc),
          k1(blockIdx.z * d.zc + d.zc) {}
};

// Half the monotonized-central slope from the differences a (below) and b
// (above) and their sum s: min(|a|, |b|, |s|/4) with their sign, 0 at extrema.
__device__ __forceinline__ float half_slope(float a, float b, float s) {
    const float m = fminf(fminf(fabsf(a), fabsf(b)), 0.25f * fabsf(s));
    return a * b > 0.0f ? copysignf(m, s) : 0.0f;
}
// For FP64 the comparisons run on the integer pipe: the order of non-negative
// doubles is that of their bits.
__device__ __forceinline__ double half_slope(double a, double b, double s) {
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b), is = __double_as_longlong(0.25 * s);
    constexpr long long mag = 0x7fffffffffffffffLL;
    const long long m = min(min(ia & mag, ib & mag), is & mag);
    return (ia ^ ib) < 0 ? 0.0 : __longlong_as_double(m | (ia & ~mag));
}
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool negative(float x) { return x < 0.0f; }
__device__ __forceinline__ bool negative(double x) { return 2 * __double_as_longlong(x) != 0 && __double_as_longlong(x) < 0; }

// Fluxes of all three components through a face with states l and r, the
// normal component being a (Burgers Riemann solution, upwinded).
template <typename T>
__device__ __forceinline__ void upwind_flux(const T l[3], const T r[3], int a, T flux[3]) {
    const T s = l[a] + r[a];
    const bool up = positive(s) && positive(l[a]), down = negative(s) && negative(r[a]);
    const T un = up ? l[a] : (down ? r[a] : (T)0);
#pragma unroll
    for (int c = 0; c < 3; ++c) flux[c] = un * (up ? l[c] : r[c]);
}

// Flux difference and second difference of the three components along axis a
// at the middle of five cells v.  k = dt / h.
template <typename T>
__device__ __forceinline__ void axis_terms(const T v[5][3], int a, T k, T conv[3], T lap[3]) {
    T lm[3], rm[3], lp[3], rp[3];  // states at the faces -1/2 and +1/2
    const T cl0 = fma(-k, v[1][a], (T)1), cr1 = fma(k, v[2][a], (T)1), cl1 = fma(-k, v[2][a], (T)1),
            cr2 = fma(k, v[3][a], (T)1);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const T d0 = v[1][c] - v[0][c], d1 = v[2][c] - v[1][c], d2 = v[3][c] - v[2][c], d3 = v[4][c] - v[3][c];
        const T s0 = half_slope(d0, d1, d0 + d1), s1 = half_slope(d1, d2, d1 + d2), s2 = half_slope(d2, d3, d2 + d3);
        lm[c] = fma(cl0, s0, v[1][c]);
        rm[c] = fma(-cr1, s1, v[2][c]);
        lp[c] = fma(cl1, s1, v[2][c]);
        rp[c] = fma(-cr2, s2, v[3][c]);
        lap[c] += d2 - d1;
    }
    T fm[3], fp[3];
    upwind_flux(lm, rm, a, fm);
    upwind_flux(lp, rp, a, fp);
#pragma unroll
    for (int c = 0; c < 3; ++c) conv[c] += fp[c] - fm[c];
}

// A cell's gradient sums from its corners on one node plane: x and y
// differences, and the corners themselves for the z differences.  Differences
// are taken before anything is added: a sum of pressures would leave its
// rounding in the gradient.
template <typename T>
__device__ __forceinline__ void plane_corners(T p00, T p10, T p01, T p11, T &gx, T &gy, T s[4]) {
    gx = (p10 - p00) + (p11 - p01);
    gy = (p01 - p00) + (p11 - p10);
    s[0] = p00, s[1] = p10, s[2] = p01, s[3] = p11;
}
// The z sum between two node planes; s0 becomes s1.
template <typename T> __device__ __forceinline__ T z_corners(T s0[4], const T s1[4]) {
    const T r = ((s1[0] - s0[0]) + (s1[1] - s0[1])) + ((s1[2] - s0[2]) + (s1[3] - s0[3]));
#pragma unroll
    for (int o = 0; o < 4; ++o) s0[o] = s1[o];
    return r;
}

// Right-hand side of the predictor at every cell,
//   u^n + dt (-div(u u) - G p / rho + (nu / 2) L_c u^n + g).
// Along z the five cells, the lower face's flux and the middle cell's states
// stay in registers from plane to plane.
struct RhsArgs {
    double k;            // dt / h
    double cc, cg, cl;   // -dt / h, -dt / (4 h rho), nu dt / (2 h^2)
    double dg[3];        // dt g
};
constexpr int kStencilThreads = 256;
template <typename T>
__global__ void __launch_bounds__(kStencilThreads) k_predictor_rhs(LevelDims d, const T *__restrict__ u,
                                                                   const T *__restrict__ p, RhsArgs a,
                                                                   T *__restrict__ out) {
    const Column q(d);
    const int m0 = d.n0 - 1, m1 = d.n1 - 1, m2 = d.n2 - 1;
    const size_t plane = (size_t)d.n0 * d.n1, N = plane * d.n2;
    const T k = (T)a.k, cc = (T)a.cc, cg = (T)a.cg, cl = (T)a.cl;
    const int row = q.j * d.n0, i0 = row + q.i;
    int ix[4], iy[4];  // in-plane neighbours -2, -1, +1, +2
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const int s = o < 2 ? o - 2 : o - 1;
        ix[o] = row + ((q.i + s) & m0);
        iy[o] = ((q.j + s) & m1) * d.n0 + q.i;
    }
    const int px = row + ((q.i + 1) & m0), py = ((q.j + 1) & m1) * d.n0 + q.i, pxy = ((q.j + 1) & m1) * d.n0 + ((q.i + 1) & m0);
    auto corners = [&](int kk, T &gx, T &gy, T s[4]) {
        const T *pk = p + (size_t)kk * plane;
        plane_corners(pk[i0], pk[px], pk[py], pk[pxy], gx, gy, s);
    };
    grid_dep_wait();
    T z[5][3];
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int c = 0; c < 3; ++c) z[o][c] = u[c * N + (size_t)((q.k0 + o - 2) & m2) * plane + i0];
    // the lower face's flux and the middle cell's left states, as the loop carries them
    T fm[3], left[3], gx0, gy0, s0[4];
    {
        const T cl0 = fma(-k, z[1][2], (T)1), cr1 = fma(k, z[2][2], (T)1), cl1 = fma(-k, z[2][2], (T)1);
        T l[3], r[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T d0 = z[1][c] - z[0][c], d1 = z[2][c] - z[1][c], d2 = z[3][c] - z[2][c];
            const T s1 = half_slope(d1, d2, d1 + d2);
            l[c] = fma(cl0, half_slope(d0, d1, d0 + d1), z[1][c]);
            r[c] = fma(-cr1, s1, z[2][c]);
            left[c] = fma(cl1, s1, z[2][c]);
        }
        upwind_flux(l, r, 2, fm);
    }
    corners(q.k0, gx0, gy0, s0);
    for (int kk = q.k0; kk < q.k1; ++kk) {
        const size_t base = (size_t)kk * plane;
#pragma unroll
        for (int c = 0; c < 3; ++c) z[4][c] = u[c * N + (size_t)((kk + 2) & m2) * plane + i0];
        T conv[3] = {0, 0, 0}, lap[3] = {0, 0, 0};
        T v[5][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[2][c] = z[2][c];
#pragma unroll
            for (int o = 0; o < 4; ++o) v[o < 2 ? o : o + 1][c] = u[c * N + base + ix[o]];
        }
        axis_terms(v, 0, k, conv, lap);
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int o = 0; o < 4; ++o) v[o < 2 ? o : o + 1][c] = u[c * N + base + iy[o]];
        axis_terms(v, 1, k, conv, lap);
        {
            const T cr = fma(k, z[3][2], (T)1), cn = fma(-k, z[3][2], (T)1);
            T r[3], next[3], fp[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T d1 = z[2][c] - z[1][c], d2 = z[3][c] - z[2][c], d3 = z[4][c] - z[3][c];
                const T s = half_slope(d2, d3, d2 + d3);
                r[c] = fma(-cr, s, z[3][c]);
                next[c] = fma(cn, s, z[3][c]);
                lap[c] += d2 - d1;
            }
            upwind_flux(left, r, 2, fp);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                conv[c] += fp[c] - fm[c];
                fm[c] = fp[c];
                left[c] = next[c];
            }
        }
        T gx1, gy1, s1[4];
        corners((kk + 1) & m2, gx1, gy1, s1);
        const T gp[3] = {gx0 + gx1, gy0 + gy1, z_corners(s0, s1)};
        gx0 = gx1, gy0 = gy1;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            out[c * N + base + i0] = fma(cl, lap[c], fma(cc, conv[c], fma(cg, gp[c], z[2][c] + (T)a.dg[c])));
#pragma unroll
            for (int o = 0; o < 4; ++o) z[o][c] = z[o + 1][c];
        }
    }
}

// A sum of differences.  FP32: compensated (Knuth's TwoSum of every
// difference and every addition), since the solve amplifies the rounding of
// the nearly checkerboard modes most, up to 1e5 times at 256^3, and a plain
// sum leaves there what a difference of single-precision velocities does not.
template <typename T> struct DiffSum {
    T s;
    __device__ __forceinline__ void clear() { s = 0; }
    __device__ __forceinline__ void add(T a, T b) { s += a - b; }
    __device__ __forceinline__ void add(const DiffSum &o) { s += o.s; }
    __device__ __forceinline__ T value() const { return s; }
};
template <> struct DiffSum<float> {
    float s, e;
    __device__ __forceinline__ void clear() { s = e = 0.0f; }
    __device__ __forceinline__ float two_sum(float a, float b, float &err) const {
        const float t = __fadd_rn(a, b), bb = __fsub_rn(t, a);
        err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bb)), __fsub_rn(b, bb));
        return t;
    }
    __device__ __forceinline__ void add(float a, float b) {
        float e0, e1;
        const float d = two_sum(a, -b, e0);
        s = two_sum(s, d, e1);
        e = __fadd_rn(e, __fadd_rn(e0, e1));
    }
    __device__ __forceinline__ void add(const DiffSum &o) {
        float e1;
        s = two_sum(s, o.s, e1);
        e = __fadd_rn(e, __fadd_rn(o.e, e1));
    }
    __device__ __forceinline__ float value() const { return __fadd_rn(s, e); }
};

// D V at every node, V = u*/dt + G p_old / rho_f (Eq. ns_lp1).  D u is the sum
// over the planes k - 1 and k of the in-plane differences; D G p is the
// 27-point operator formed from in-plane second differences (so a constant
// pressure cancels exactly): with r the second x difference of a row, y that
// of the column along y and z along z,
//   16 h^2 D G p = (3 r- + 2 r0 + 3 r+ + 8 y)(k-1) + the same (k+1)
//                  + 2 (r- - 2 r0 + r+)(k) + 16 z.
template <typename T>
__global__ void __launch_bounds__(kStencilThreads) k_projection_div(LevelDims d, const T *__restrict__ u,
                                                                    const T *__restrict__ p, double cu, double cp,
                                                                    T *__restrict__ out) {
    const Column q(d);
    const int m0 = d.n0 - 1, m1 = d.n1 - 1, m2 = d.n2 - 1;
    const size_t plane = (size_t)d.n0 * d.n1, N = plane * d.n2;
    const int xm = (q.i - 1) & m0, xp = (q.i + 1) & m0, x0 = q.i;
    const int ym = ((q.j - 1) & m1) * d.n0, yp = ((q.j + 1) & m1) * d.n0, y0 = q.j * d.n0;
    auto pressure = [&](int kk, T &a, T &b, T &c) {
        const T *pk = p + (size_t)kk * plane;
        c = pk[y0 + x0];
        const T cm = pk[ym + x0], cp1 = pk[yp + x0];
        const T r0 = (pk[y0 + xp] - c) - (c - pk[y0 + xm]);
        const T rm = (pk[ym + xp] - cm) - (cm - pk[ym + xm]);
        const T rp = (pk[yp + xp] - cp1) - (cp1 - pk[yp + xm]);
        const T yy = (cp1 - c) - (c - cm), s = rm + rp;
        a = fma((T)3, s, fma((T)2, r0, (T)8 * yy));
        b = fma((T)-2, r0, s);
    };
    // differences of u around the node: x and y parts in the plane, and the z
    // component's four values, whose differences between planes are taken
    // before they are added
    auto velocity = [&](int kk, DiffSum<T> &xy, T w[4]) {
        const T *uk = u + (size_t)kk * plane;
        const T *vk = uk + N, *wk = vk + N;
        xy.clear();
        xy.add(uk[y0 + x0], uk[y0 + xm]);
        xy.add(uk[ym + x0], uk[ym + xm]);
        xy.add(vk[y0 + x0], vk[ym + x0]);
        xy.add(vk[y0 + xm], vk[ym + xm]);
        w[0] = wk[y0 + x0], w[1] = wk[y0 + xm], w[2] = wk[ym + x0], w[3] = wk[ym + xm];
    };
    grid_dep_wait();
    T am, bm, cm, a0, b0, c0, wm[4];
    DiffSum<T> xym;
    pressure((q.k0 - 1) & m2, am, bm, cm);
    pressure(q.k0, a0, b0, c0);
    T dzm = c0 - cm;
    velocity((q.k0 - 1) & m2, xym, wm);
    for (int kk = q.k0; kk < q.k1; ++kk) {
        T a1, b1, c1, w[4];
        DiffSum<T> xy;
        pressure((kk + 1) & m2, a1, b1, c1);
        velocity(kk, xy, w);
        const T dz = c1 - c0;
        const T dgp = fma((T)16, dz - dzm, fma((T)2, b0, am + a1));
        xym.add(xy);
#pragma unroll
        for (int o = 0; o < 4; ++o) xym.add(w[o], wm[o]);
        out[(size_t)kk * plane + y0 + x0] = fma((T)cp, dgp, (T)cu * xym.value());
        am = a0, a0 = a1, b0 = b1, c0 = c1, dzm = dz, xym = xy;
#pragma unroll
        for (int o = 0; o < 4; ++o) wm[o] = w[o];
    }
}

// u^{n+1} = dt (V - G p_new / rho_f) = u* + (dt / rho_f) G (p_old - p_new)
// (Eq. ns_lp3).  FP64: q holds p_old - p_new; FP32: q holds p_old and p p_new
// (fluid_fft.cuh, kXPressure).
template <typename T>
__global__ void __launch_bounds__(kStencilThreads) k_projection_update(LevelDims d, T *__restrict__ u,
                                                                       const T *__restrict__ q,
                                                                       const T *__restrict__ p, double cg) {
    constexpr bool kTwo = sizeof(T) == 4;
    const Column o(d);
    const int m0 = d.n0 - 1, m1 = d.n1 - 1, m2 = d.n2 - 1;
    const size_t plane = (size_t)d.n0 * d.n1, N = plane * d.n2;
    const int i0 = o.j * d.n0 + o.i, px = o.j * d.n0 + ((o.i + 1) & m0), py = ((o.j + 1) & m1) * d.n0 + o.i,
              pxy = ((o.j + 1) & m1) * d.n0 + ((o.i + 1) & m0);
    auto corners = [&](const T *f, int kk, T &gx, T &gy, T s[4]) {
        const T *pk = f + (size_t)kk * plane;
        plane_corners(pk[i0], pk[px], pk[py], pk[pxy], gx, gy, s);
    };
    grid_dep_wait();
    T gx0, gy0, s0[4], hx0 = 0, hy0 = 0, r0[4];
    corners(q, o.k0, gx0, gy0, s0);
    if (kTwo) corners(p, o.k0, hx0, hy0, r0);
    for (int kk = o.k0; kk < o.k1; ++kk) {
        T gx1, gy1, s1[4], hx1, hy1, r1[4];
        corners(q, (kk + 1) & m2, gx1, gy1, s1);
        T *uk = u + (size_t)kk * plane + i0;
        const T u0 = uk[0], u1 = uk[N], u2 = uk[2 * N];
        T g[3] = {gx0 + gx1, gy0 + gy1, z_corners(s0, s1)};
        if (kTwo) {
            corners(p, (kk + 1) & m2, hx1, hy1, r1);
            g[0] -= hx0 + hx1, g[1] -= hy0 + hy1, g[2] -= z_corners(r0, r1);
            hx0 = hx1, hy0 = hy1;
        }
        uk[0] = fma((T)cg, g[0], u0);
        uk[N] = fma((T)cg, g[1], u1);
        uk[2 * N] = fma((T)cg, g[2], u2);
        gx0 = gx1, gy0 = gy1;
    }
}

static int ilog2_exact(int n) {
    int l = 0;
    while ((1 << l) < n) ++l;
    return (1 << l) == n ? l : -1;
}

static int check_fluid_grid(const ib_grid *grid) {
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    for (int a = 0; a < 3; ++a) {
        const int l = ilog2_exact(grid->n[a]);
        if (l < 4 || l > 10)
            return set_error(IB_ERR_UNSUPPORTED, "fluid step: n[%d] = %d must be a power of two in [16, 1024]", a,
                             grid->n[a]);
    }
    return IB_OK;
}

// Launch shape of the stencil kernels: 32 x 8 columns (16 x 16 on the smallest
// grids) and chunks of planes, at most 32 and at least 4, that give each SM
// several CTAs.
struct StencilGrid {
    LevelDims d;
    dim3 grid, block;
    StencilGrid(ib_ctx *ctx, const int n[3]) : d{n[0], n[1], n[2], 32} {
        block = dim3(n[0] < 32 ? 16 : 32, n[0] < 32 ? 16 : 8, 1);
        const long long tiles = (long long)(n[0] / block.x) * (n[1] / block.y);
        if (d.zc > n[2]) d.zc = n[2];
        while (d.zc > 4 && tiles * (n[2] / d.zc) < 6LL * ctx->sm_count) d.zc /= 2;
        grid = dim3(n[0] / block.x, n[1] / block.y, n[2] / d.zc);
    }
};

template <class A> static FftGrid<A> fft_grid(ib_ctx *ctx, const int n[3]) {
    FftGrid<A> g;
    for (int a = 0; a < 3; ++a) g.n[a] = n[a], g.log2n[a] = ilog2_exact(n[a]);
    if constexpr (A::kFixed) g.roots = ctx->fft_tab->roots_fx;
    else g.roots = ctx->fft_tab->roots32;
    if constexpr (sizeof(typename A::Real) == 8) g.trig = ctx->fft_tab->trig64;
    else g.trig = ctx->fft_tab->trig32;
    return g;
}

// The spectral solve of ncomp fields from `src` to `dst`: x passes in the
// arithmetic X, the others in A.
template <class X, class A>
static cudaError_t solve(ib_ctx *ctx, const int n[3], int ncomp, const typename A::Real *src, Spectrum<A> c,
                         const SymbolArgs &sy, int out, typename A::Real *dst, typename A::Real *old, cudaStream_t s) {
    const FftGrid<X> gx = fft_grid<X>(ctx, n);
    const FftGrid<A> g = fft_grid<A>(ctx, n);
    const Spectrum<X> cx = {c.c, c.ny};
    cudaError_t e = fft_x<X>(kXForward, gx, ncomp, src, cx, nullptr, nullptr, s);
    if (e == cudaSuccess) e = fft_y<A>(false, g, ncomp, c, s);
    if (e == cudaSuccess) e = fft_z<A>(g, ncomp, c, sy, s);
    if (e == cudaSuccess) e = fft_y<A>(true, g, ncomp, c, s);
    if (e == cudaSuccess) e = fft_x<X>(out, gx, ncomp, nullptr, cx, dst, old, s);
    return e;
}

template <class A>
static int run_predictor(ib_ctx *ctx, const ib_grid *grid, const void *u, const void *p, double rho_f, double mu,
                         const double g[3], double dt, void *u_star, cudaStream_t s) {
    using T = typename A::Real;
    const size_t N = (size_t)grid->n[0] * grid->n[1] * grid->n[2];
    const double h = grid->h, nu = mu / rho_f;
    Arena ar(ctx);
    const size_t ny = (size_t)grid->n[1] * grid->n[2];
    Spectrum<A> c;
    c.c = ar.take<typename A::Mem>(3 * (N / 2));
    c.ny = ar.take<typename A::Mem>(3 * ny);
    if (!ar.ok()) return oom_error(ar.used, ar.cap);
    const StencilGrid sg(ctx, grid->n);
    const RhsArgs a = {dt / h, -dt / h, -dt / (4.0 * h * rho_f), 0.5 * nu * dt / (h * h), {dt * g[0], dt * g[1], dt * g[2]}};
    const double points = (double)N;  // the transforms are unscaled
    const SymbolArgs sy = {kSolveHelmholtz, 1.0 / points, 0.5 * nu * dt * 4.0 / (h * h)};
    PhaseTimer tm(ctx, IB_PHASE_FLUID_PREDICTOR, s);
    // the right-hand side in u_star, the point buffers in the workspace
    cudaError_t e = launch_pdl(k_predictor_rhs<T>, sg.grid, sg.block, 0, s, sg.d, (const T *)u, (const T *)p, a, (T *)u_star);
    if (e == cudaSuccess) e = solve<A, A>(ctx, grid->n, 3, (const T *)u_star, c, sy, kXField, (T *)u_star, nullptr, s);
    if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "fluid_predictor: %s", cudaGetErrorString(e));
    return check_launch("fluid_predictor");
}

template <class A>
static int run_projection(ib_ctx *ctx, const ib_grid *grid, void *u, void *p, double rho_f, double dt,
                          cudaStream_t s) {
    using T = typename A::Real;
    const size_t N = (size_t)grid->n[0] * grid->n[1] * grid->n[2];
    const double h = grid->h;
    Arena ar(ctx);
    Spectrum<A> c;
    c.c = ar.take<typename A::Mem>(N / 2);
    c.ny = ar.take<typename A::Mem>((size_t)grid->n[1] * grid->n[2]);
    T *q = ar.take<T>(N);
    if (!ar.ok()) return oom_error(ar.used, ar.cap);
    const StencilGrid sg(ctx, grid->n);
    // p_new = rho_f (D G)^-1 D V   (Eq. ns_lp2 with L p = div((1/rho_f) grad p))
    const SymbolArgs sy = {kSolveDivGrad, -rho_f * h * h / 4.0 / (double)N, 0.0};
    PhaseTimer tm(ctx, IB_PHASE_FLUID_PROJECTION, s);
    cudaError_t e = launch_pdl(k_projection_div<T>, sg.grid, sg.block, 0, s, sg.d, (const T *)u, (const T *)p,
                               0.25 / (h * dt), 0.0625 / (h * h * rho_f), q);
    if (e == cudaSuccess) e = solve<typename A::Pressure, A>(ctx, grid->n, 1, q, c, sy, kXPressure, (T *)p, q, s);
    if (e == cudaSuccess)
        e = launch_pdl(k_projection_update<T>, sg.grid, sg.block, 0, s, sg.d, (T *)u, (const T *)q,
                       (const T *)p, dt / (4.0 * h * rho_f));
    if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "level_projection: %s", cudaGetErrorString(e));
    return check_launch("level_projection");
}

}  // namespace gbib

using namespace gbib;

extern "C" {

int fluid_predictor(ib_ctx *ctx, const ib_grid *grid, const void *u, const void *p, double rho_f, double mu,
                    const double *g, double dt, void *u_star, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    int rc = check_fluid_grid(grid);
    if (rc) return rc;
    if (!u || !p || !u_star || !g) return set_error(IB_ERR_INVALID, "NULL array");
    if (!(rho_f > 0.0) || !(mu >= 0.0) || !isfinite(mu) || !(dt > 0.0) || !isfinite(dt) || !isfinite(g[0]) ||
        !isfinite(g[1]) || !isfinite(g[2]))
        return set_error(IB_ERR_INVALID, "rho_f > 0, mu >= 0, dt > 0 and g must be finite");
    if (grid->prec == IB_F64)
        return run_predictor<Fx64>(ctx, grid, u, p, rho_f, mu, g, dt, u_star, (cudaStream_t)stream);
    return run_predictor<Fp32>(ctx, grid, u, p, rho_f, mu, g, dt, u_star, (cudaStream_t)stream);
}

int level_projection(ib_ctx *ctx, const ib_grid *grid, void *u, void *p, double rho_f, double dt, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    int rc = check_fluid_grid(grid);
    if (rc) return rc;
    if (!u || !p) return set_error(IB_ERR_INVALID, "NULL array");
    if (!(rho_f > 0.0) || !(dt > 0.0) || !isfinite(dt)) return set_error(IB_ERR_INVALID, "rho_f > 0 and dt > 0");
    if (grid->prec == IB_F64) return run_projection<Fx64>(ctx, grid, u, p, rho_f, dt, (cudaStream_t)stream);
    return run_projection<Fp32>(ctx, grid, u, p, rho_f, dt, (cudaStream_t)stream);
}

}  // extern "C"
