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

constexpr int kStencilThreads = 256;
// The thread's column and its chunk of planes.
struct Column {
    int i, j, k0, k1;
    __device__ __forceinline__ Column(const LevelDims &d)
        : i(blockIdx.x * blockDim.x + threadIdx.x), j(blockIdx.y * blockDim.y + threadIdx.y), k0(blockIdx.z * d.zc),
          k1(blockIdx.z * d.zc + d.zc) {}
};

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

// ---- the predictor's right-hand side in three arithmetics --------------------
struct RhsArgs {
    double k;            // dt / h
    double cc, cg, cl;   // -dt / h, -dt / (4 h rho), nu dt / (2 h^2)
    double dg[3];        // dt g
};

// The words of the fields' largest magnitudes (high words): each velocity
// component's, the pressure's and (projection) p_old - p's.
enum { kMaxU = 0, kMaxP = 3, kMaxOld = 4, kMaxima = 5 };
static_assert(kMaxima <= FftTables::kWords, "a fluid call's words");

// FP32 and FP64 as they stand.  kc: a cell's dt/h u_a; up / down: its states
// towards the faces above and below, v +- (1 -+ c) m; half_slope: half the
// monotonized-central slope from the differences a (below) and b (above),
// min(|a|, |b|, |a + b| / 4) with their sign, 0 at extrema; normal: a face's
// normal velocity u_a as product takes it; result: the increment is formed first
// and u0 takes one rounding, by the varying sum (dt g alone added to u0 rounds the
// same way in every cell of a binade: the mean velocity then drifts by up to half
// its last bit a step).  Arguments a and k name the component.
template <typename R> struct PlainNum {
    using T = R;
    using V = R;
    static constexpr bool kExact = true;  // u() loses nothing
    R k, cc, cg, cl, dg[3];
    __device__ PlainNum(const RhsArgs &a, const int *)
        : k((R)a.k), cc((R)a.cc), cg((R)a.cg), cl((R)a.cl), dg{(R)a.dg[0], (R)a.dg[1], (R)a.dg[2]} {}
    __device__ __forceinline__ V u(T x, int) const { return x; }
    __device__ __forceinline__ V p(T x) const { return x; }
    __device__ __forceinline__ V kc(V v, int) const { return k * v; }
    __device__ __forceinline__ V up(V v, V c, V m) const { return fma((R)1 - c, m, v); }
    __device__ __forceinline__ V down(V v, V c, V m) const { return fma((R)-1 - c, m, v); }
    __device__ __forceinline__ V half_slope(V a, V b) const {
        if constexpr (sizeof(R) == 8) {
            // comparisons on the integer pipe: the order of non-negative doubles is that of their bits
            constexpr long long mag = 0x7fffffffffffffffLL;
            const long long x = __double_as_longlong(a), y = __double_as_longlong(b),
                            z = __double_as_longlong(0.25 * (a + b));
            const long long m = min(min(x & mag, y & mag), z & mag);
            return (x ^ y) < 0 ? 0.0 : __longlong_as_double(m | (x & ~mag));
        } else {
            const R s = a + b, m = fmin(fmin(fabs(a), fabs(b)), (R)0.25 * fabs(s));
            return a * b > (R)0 ? copysign(m, s) : (R)0;
        }
    }
    __device__ __forceinline__ bool positive(V x) const { return x > (R)0; }
    __device__ __forceinline__ bool negative(V x) const { return x < (R)0; }
    __device__ __forceinline__ V normal(V un, int) const { return un; }
    __device__ __forceinline__ V product(V un, V s) const { return un * s; }
    __device__ __forceinline__ T result(T u0, V lap, V conv, V gp, int k) const {
        return u0 + fma(cl, lap, fma(cc, conv, fma(cg, gp, dg[k])));
    }
};

// FP64 fields in 64-bit fixed point: each velocity component and p in a unit of
// its own, in which its largest value has 59 bits (one unit for all three left a component 10^-8 times the largest one's size an error of 2e-9
// of its values).  Differences and sums are then exact, and what a small value
// loses in its conversion is 2^-60 of its component's largest one.  A flux is the
// state in its component's unit times the normal velocity in the largest
// component's, so that the three axes' fluxes add up.  A product is off by half a
// unit and the low halves' product that it leaves out: at most 0.75 units in
// mul<64>, 1.5 in mul<62>, 2.5 in mul<61>.  The FP64 pipe (a warp instruction in
// 16 clocks of an SM) forms only the final sum.  The CTA keeps it in shared
// memory: in registers it spilled more.
struct FixedNum {
    using T = double;
    using V = long long;
    static constexpr bool kExact = false;
    static constexpr int kBits = 59;
    int unit[3], punit;    // to_fixed's
    int shift[3];          // from a component's unit to the largest one's,
    long long half[3];     // and what rounds that
    Halves kk[3];          // dt/h in units: c = kk v / 2^62 in Q58
    double cc[3], cl[3], cg;  // with the units' powers of two
    double dg[3];
    // the largest component's and a component's exponent (a component of zeros
    // takes the largest one's unit)
    __device__ static int largest(const int *m) { return exponent_of<double>(max(max(m[0], m[1]), m[2])); }
    __device__ static int exponent(const int *m, int k) { return m[k] ? exponent_of<double>(m[k]) : largest(m); }
    // the ranges in which no sum overflows: the largest |p| and each component's
    // largest value within 2^(+-400) (or zero), and a Courant number dt/h max|u| (of
    // the power of two above the maximum) up to 2
    __device__ static bool fits(const RhsArgs &a, const int *m) {
        bool in = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) in = in && abs(exponent(m + kMaxU, k) - 1023) <= 400;
        const int f = exponent_of<double>(m[kMaxP]);
        return in && (f <= 1 || abs(f - 1023) <= 400) && a.k * pow2(largest(m + kMaxU) - 1022) <= 2.0;
    }
    __device__ static double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }
    __device__ FixedNum(const RhsArgs &a, const int *m) {
        const int most = largest(m + kMaxU);
        const int ep = exponent_of<double>(m[kMaxP]);
        punit = ep - kBits;
        cg = ep > 1 ? a.cg * pow2(ep - 1022 - kBits) : 0.0;  // a pressure of 0 (or below 2^-1022)
        for (int k = 0; k < 3; ++k) {
            const int e = exponent(m + kMaxU, k), su = e - 1022 - kBits;
            unit[k] = e - kBits;
            shift[k] = min(most - e, 62);
            half[k] = (1LL << shift[k]) >> 1;
            kk[k] = halves(__double2ll_rn(a.k * pow2(su) * pow2(58 + 62)));
            cc[k] = a.cc * pow2(su + (most - 1022 - kBits) + 63);
            cl[k] = a.cl * pow2(su);
            dg[k] = a.dg[k];
        }
    }
    __device__ __forceinline__ V u(T x, int k) const { return to_fixed(x, unit[k]); }
    __device__ __forceinline__ V p(T x) const { return to_fixed(x, punit); }
    // a b / 2^SH, rounded
    template <int SH> __device__ __forceinline__ static V mul(Halves x, Halves y) {
        const long long s = (long long)x.hi * y.hi;
        const long long t = (long long)x.hi * y.lo + ((long long)x.lo * y.hi + (1LL << (SH - 33)));
        return SH == 64 ? s + (t >> 32) : (long long)((unsigned long long)s << (64 - SH)) + (t >> (SH - 32));
    }
    // Q61: the Q58 product shifted (its rounding counts against a slope only)
    __device__ __forceinline__ V kc(V v, int a) const { return mul<62>(halves(v), kk[a]) << 3; }
    __device__ __forceinline__ V up(V v, V c, V m) const { return v + mul<61>(halves((1LL << 61) - c), halves(m)); }
    __device__ __forceinline__ V down(V v, V c, V m) const { return v - mul<61>(halves((1LL << 61) + c), halves(m)); }
    __device__ __forceinline__ V half_slope(V a, V b) const {
        const V s = a >> 63, x = (a ^ s) - s, y = (b ^ s) - s;  // |a|, |b| where the signs agree
        V m = x < y ? x : y;
        const V q = (x + y) >> 2;
        m = m < q ? m : q;
        return (a ^ b) < 0 ? 0 : (m ^ s) - s;
    }
    __device__ __forceinline__ bool positive(V x) const { return x > 0; }
    __device__ __forceinline__ bool negative(V x) const { return x < 0; }
    __device__ __forceinline__ V normal(V un, int a) const { return (un + half[a]) >> shift[a]; }
    __device__ __forceinline__ V product(V un, V s) const { return mul<64>(halves(un << 1), halves(s)); }
    __device__ __forceinline__ T result(T u0, V lap, V conv, V gp, int k) const {
        return u0 + fma(cl[k], (double)lap, fma(cc[k], (double)conv, fma(cg, (double)gp, dg[k])));
    }
};

// Fluxes of all three components through a face with states l and r, the
// normal component being a (Burgers Riemann solution, upwinded).
template <class Q>
__device__ __forceinline__ void upwind_flux(const Q &q, const typename Q::V l[3], const typename Q::V r[3], int a,
                                            typename Q::V flux[3]) {
    const typename Q::V s = l[a] + r[a];
    const bool up = q.positive(s) && q.positive(l[a]), down = q.negative(s) && q.negative(r[a]);
    const typename Q::V un = q.normal(up ? l[a] : (down ? r[a] : 0), a);
#pragma unroll
    for (int c = 0; c < 3; ++c) flux[c] = q.product(un, up ? l[c] : r[c]);
}

// Right-hand side of the predictor at every cell,
//   u^n + dt (-div(u u) - G p / rho + (nu / 2) L_c u^n + g),
// every slope, state and flux formed once.  A CTA marches a TX x TY tile of
// columns along z: 256 threads own a column each and keep its five cells, the
// lower z face's flux and the z states in registers; the plane's cells are in
// shared memory with a halo of two.  A cell's two states along x and y come
// from its slope; the face above takes the neighbour's lower state (x: the next
// lane's by a shuffle, y: through shared memory) and passes its flux on the
// same way.  Three more warps own the halo: they load and convert it and form
// the tile's outer states and fluxes.
template <int TX> struct RhsTile {
    static constexpr int TY = 256 / TX, CELLS = 256, HALO = 96, T = CELLS + HALO;
    static constexpr int UX = TX + 4, UY = TY + 4, ITEMS = 4 * TX + 4 * TY;  // halo cells of one component
    static constexpr int PER = (3 * ITEMS + HALO - 1) / HALO;
};
template <class V, int TX> struct RhsShared {
    using S = RhsTile<TX>;
    V u[3][S::UY][S::UX];
    V p[S::TY + 1][TX + 1];
    V ry[3][S::TY + 1][TX], fy[3][S::TY + 1][TX];  // lower y states, lower y faces' fluxes
    V rx[3][S::TY], fx[3][S::TY];                  // the states above and the fluxes below the tile in x
};

// A cell's slope terms along one axis (stride of the shared plane): the
// state towards the upper face and the lower one.
template <class Q>
__device__ __forceinline__ typename Q::V states(const Q &q, typename Q::V vm, typename Q::V v0, typename Q::V vp,
                                                typename Q::V c, typename Q::V &up, typename Q::V &down) {
    const typename Q::V a = v0 - vm, b = vp - v0, m = q.half_slope(a, b);
    up = q.up(v0, c, m);
    down = q.down(v0, c, m);
    return b - a;
}

template <class Q, int TX>
__device__ __forceinline__ void rhs_tile(const Q &q, const LevelDims &d, const typename Q::T *__restrict__ u,
                                         const typename Q::T *__restrict__ p, const RhsArgs &a,
                                         typename Q::T *__restrict__ out, RhsShared<typename Q::V, TX> &s) {
    using S = RhsTile<TX>;
    using T = typename Q::T;
    using V = typename Q::V;
    constexpr int TY = S::TY;
    const int m0 = d.n0 - 1, m1 = d.n1 - 1, m2 = d.n2 - 1, tid = threadIdx.x;
    const size_t plane = (size_t)d.n0 * d.n1, N = plane * d.n2;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, k0 = blockIdx.z * d.zc, k1 = k0 + d.zc;
    if (tid >= S::CELLS) {
        // ---- the halo's warps ----
        const int h = tid - S::CELLS;
        int off[S::PER], at[S::PER];
        T raw[S::PER];
        V *const flat = &s.u[0][0][0];
#pragma unroll
        for (int r = 0; r < S::PER; ++r) {
            const int e = h + r * S::HALO, c = e / S::ITEMS, i = e % S::ITEMS;
            int x, y;
            if (i < 4 * TY) y = i >> 2, x = (i & 3) < 2 ? (i & 3) - 2 : TX + (i & 3) - 2;
            else x = (i - 4 * TY) % TX, y = (i - 4 * TY) / TX, y = y < 2 ? y - 2 : TY + y - 2;
            at[r] = e < 3 * S::ITEMS ? (c * S::UY + y + 2) * S::UX + x + 2 : -1;
            off[r] = ((y0 + y) & m1) * d.n0 + ((x0 + x) & m0);
            if (at[r] >= 0) raw[r] = u[c * N + (size_t)k0 * plane + off[r]];
        }
        // pressure nodes above the tile in x and y
        const bool edge = h < TX + TY + 1;
        const int ex = h < TX ? h : TX, ey = h < TX ? TY : h - TX;  // (TX, TY) is the last one's
        const int eo = ((y0 + ey) & m1) * d.n0 + ((x0 + ex) & m0);
        T praw = 0;
        if (edge) {
            s.p[ey][ex] = q.p(p[(size_t)k0 * plane + eo]);
            praw = p[(size_t)((k0 + 1) & m2) * plane + eo];
        }
        __syncthreads();  // the first plane's nodes there
        __syncthreads();  // and read
        // the tile's outer faces: lower ones (their flux), then upper ones (the state above)
        const bool low = h < TX + TY, face = h < 2 * (TX + TY);
        const int f = low ? h : h - (TX + TY);
        const bool ax = f < TY;               // an x face of row f, or a y face of column f - TY
        const int fi = ax ? f : f - TY;
        const V *b = ax ? &s.u[0][fi + 2][low ? 1 : TX + 2] : &s.u[0][low ? 1 : TY + 2][fi + 2];  // the outer cell
        const int st = ax ? 1 : S::UX;
        constexpr int CS = S::UX * S::UY;
        for (int kk = k0; kk < k1; ++kk) {
#pragma unroll
            for (int r = 0; r < S::PER; ++r)
                if (at[r] >= 0) flat[at[r]] = q.u(raw[r], (h + r * S::HALO) / S::ITEMS);
            if (edge) s.p[ey][ex] = q.p(praw);
            __syncthreads();  // A
            if (kk + 1 < k1) {
#pragma unroll
                for (int r = 0; r < S::PER; ++r)
                    if (at[r] >= 0)
                        raw[r] = u[(h + r * S::HALO) / S::ITEMS * N + (size_t)(kk + 1) * plane + off[r]];
                if (edge) praw = p[(size_t)((kk + 2) & m2) * plane + eo];
            }
            if (face) {
                const V vn = b[(ax ? 0 : 1) * CS];
                V up[3], down[3];
                const V c = q.kc(vn, ax ? 0 : 1);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const V *e = b + k * CS;
                    states(q, e[-st], e[0], e[st], c, up[k], down[k]);
                }
                if (low) {
                    V u1[3], d1[3], fl[3];
                    const V c1 = q.kc(b[(ax ? 0 : 1) * CS + st], ax ? 0 : 1);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const V *e = b + k * CS + st;
                        states(q, e[-st], e[0], e[st], c1, u1[k], d1[k]);
                    }
                    if (ax) upwind_flux(q, up, d1, 0, fl);
                    else upwind_flux(q, up, d1, 1, fl);
#pragma unroll
                    for (int k = 0; k < 3; ++k) (ax ? s.fx[k][fi] : s.fy[k][0][fi]) = fl[k];
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) (ax ? s.rx[k][fi] : s.ry[k][TY][fi]) = down[k];
                }
            }
            __syncthreads();  // B
            __syncthreads();  // C
        }
        return;
    }
    // ---- the cells' threads ----
    const int tx = tid % TX, ty = tid / TX, i0 = (y0 + ty) * d.n0 + x0 + tx;
    const unsigned mask = 0xffffffffu;
    V z[5][3], left[3], fm[3], s0[4];
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int c = 0; c < 3; ++c) z[o][c] = q.u(u[c * N + (size_t)((k0 + o - 2) & m2) * plane + i0], c);
    s.p[ty][tx] = q.p(p[(size_t)k0 * plane + i0]);
    {
        V l[3], r[3], x;
        const V cl = q.kc(z[1][2], 2), cn = q.kc(z[2][2], 2);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            states(q, z[0][c], z[1][c], z[2][c], cl, l[c], x);
            states(q, z[1][c], z[2][c], z[3][c], cn, left[c], r[c]);
        }
        upwind_flux(q, l, r, 2, fm);
    }
    __syncthreads();  // the first plane's nodes there
    V gx0, gy0;
    plane_corners(s.p[ty][tx], s.p[ty][tx + 1], s.p[ty + 1][tx], s.p[ty + 1][tx + 1], gx0, gy0, s0);
    __syncthreads();  // and read
    T praw = p[(size_t)((k0 + 1) & m2) * plane + i0];
    for (int kk = k0; kk < k1; ++kk) {
        T far[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            far[c] = u[c * N + (size_t)((kk + 2) & m2) * plane + i0];
            s.u[c][ty + 2][tx + 2] = z[2][c];
        }
        s.p[ty][tx] = q.p(praw);
        __syncthreads();  // A
        if (kk + 1 < k1) praw = p[(size_t)((kk + 2) & m2) * plane + i0];
        V lap[3], conv[3], ly[3];
        {
            const V c = q.kc(z[2][1], 1);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                V r;
                lap[k] = states(q, s.u[k][ty + 1][tx + 2], z[2][k], s.u[k][ty + 3][tx + 2], c, ly[k], r);
                s.ry[k][ty][tx] = r;
            }
        }
        V lx[3], rx[3];
        {
            const V c = q.kc(z[2][0], 0);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                lap[k] += states(q, s.u[k][ty + 2][tx + 1], z[2][k], s.u[k][ty + 2][tx + 3], c, lx[k], rx[k]);
        }
        V gx1, gy1, s1[4];
        plane_corners(s.p[ty][tx], s.p[ty][tx + 1], s.p[ty + 1][tx], s.p[ty + 1][tx + 1], gx1, gy1, s1);
        const V gp[3] = {gx0 + gx1, gy0 + gy1, z_corners(s0, s1)};
        gx0 = gx1, gy0 = gy1;
        __syncthreads();  // B
        T mid[3];  // the cell's own values (fixed point: read again, the conversion may have rounded them)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if constexpr (!Q::kExact) mid[k] = u[k * N + (size_t)kk * plane + i0];
            else mid[k] = z[2][k];
        }
        V fy[3];
        {
            V r[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) r[k] = s.ry[k][ty + 1][tx];
            upwind_flux(q, ly, r, 1, fy);
#pragma unroll
            for (int k = 0; k < 3; ++k) s.fy[k][ty + 1][tx] = fy[k];
        }
        {
            V r[3], f[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                r[k] = __shfl_down_sync(mask, rx[k], 1, TX);
                if (tx == TX - 1) r[k] = s.rx[k][ty];
            }
            upwind_flux(q, lx, r, 0, f);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                V b = __shfl_up_sync(mask, f[k], 1, TX);
                if (tx == 0) b = s.fx[k][ty];
                conv[k] = f[k] - b;
            }
        }
        {
            V r[3], f[3], next[3];
            const V c = q.kc(z[3][2], 2);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                z[4][k] = q.u(far[k], k);
                states(q, z[2][k], z[3][k], z[4][k], c, next[k], r[k]);
                lap[k] += (z[3][k] - z[2][k]) - (z[2][k] - z[1][k]);
            }
            upwind_flux(q, left, r, 2, f);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                conv[k] += f[k] - fm[k];
                fm[k] = f[k];
                left[k] = next[k];
            }
        }
        __syncthreads();  // C
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            conv[k] += fy[k] - s.fy[k][ty][tx];
            out[k * N + (size_t)kk * plane + i0] = q.result(mid[k], lap[k], conv[k], gp[k], k);
#pragma unroll
            for (int o = 0; o < 4; ++o) z[o][k] = z[o + 1][k];
        }
    }
}

// FP64 fields: the fixed-point kernel where the field's maxima fit it, else (a
// NaN, an infinity, a Courant number above 2) the plain one, each returning at
// once where the other serves.  (Both paths in one kernel took its registers
// for both: the plain one spilled, 2.0 ms at 128^3 against 0.6.)
template <class Q, int TX, int MINB>
__global__ void __launch_bounds__(RhsTile<TX>::T, MINB)
k_predictor_rhs(LevelDims d, const typename Q::T *__restrict__ u, const typename Q::T *__restrict__ p, RhsArgs a,
                const int *__restrict__ maxima, typename Q::T *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto &sh = *(RhsShared<typename Q::V, TX> *)smem_raw;
    grid_dep_wait();
    if constexpr (sizeof(typename Q::T) == 8) {
        if (FixedNum::fits(a, maxima) == Q::kExact) return;
    }
    if constexpr (Q::kExact) {
        rhs_tile<Q, TX>(Q(a, maxima), d, u, p, a, out, sh);
    } else {
        __shared__ __align__(8) unsigned char s_num[sizeof(Q)];
        if (threadIdx.x == 0) *(Q *)s_num = Q(a, maxima);
        __syncthreads();
        rhs_tile<Q, TX>(*(const Q *)s_num, d, u, p, a, out, sh);
    }
}

// The largest magnitudes (high words) of an FP64 velocity field and a nodal
// field, into words that are zero before.  16-byte loads (V double2) where both
// fields start on 16 bytes; a caller's view that starts on 8 takes V double.
constexpr int kMaxThreads = 512;
__device__ __forceinline__ int largest(double v) { return magnitude(v); }
__device__ __forceinline__ int largest(double2 v) { return max(magnitude(v.x), magnitude(v.y)); }
template <typename V>
__global__ void __launch_bounds__(kMaxThreads) k_field_maxima(long long N, const V *__restrict__ u, const V *__restrict__ p,
                                                              int *__restrict__ maxima) {
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    // blockIdx.y: a velocity component or the pressure
    const long long step = (long long)gridDim.x * kMaxThreads, n = N * (long long)sizeof(double) / (long long)sizeof(V);
    const V *const v = blockIdx.y < 3 ? u + blockIdx.y * n : p;
    int x = 0;
#pragma unroll 8
    for (long long i = (long long)blockIdx.x * kMaxThreads + threadIdx.x; i < n; i += step) x = max(x, largest(v[i]));
    x = __reduce_max_sync(0xffffffffu, x);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, x);
    __syncthreads();
    static_assert(kMaxU == 0 && kMaxP == 3, "the maxima's order");
    if (threadIdx.x == 0) atomicMax(maxima + blockIdx.y, s_max);
}

// The largest |u|'s high word (the linear stencils have one unit for u: their
// sums mix the components).
__device__ __forceinline__ int largest_u(const int *maxima) {
    return max(max(maxima[kMaxU], maxima[kMaxU + 1]), maxima[kMaxU + 2]);
}
// Maxima (high words) that the linear stencils' fixed point takes: their unit
// is a normal double, the values finite; or 0.
__device__ __forceinline__ bool fixed_range(int a, int b) {
    const int e = a >> 20, f = b >> 20;
    return (a == 0 || (e >= 64 && e <= 2000)) && (b == 0 || (f >= 64 && f <= 2000));
}
// F units, on the integer pipe (the conversion instruction holds the FP64 pipe
// for 16 clocks of an SM).  Only for units of fixed_range: no subnormals.
__device__ __forceinline__ double fixed_value(long long F, int unit) {
    const unsigned long long u = F < 0 ? 0ull - (unsigned long long)F : (unsigned long long)F;
    const int lz = __clzll((long long)u);
    const unsigned long long n = u << (lz & 63);
    const unsigned long long r = ((unsigned long long)(unsigned)(63 - lz + unit) << 52) + ((n >> 11) + ((n >> 10) & 1ull));
    return __longlong_as_double((long long)((u ? r : 0ull) | ((unsigned long long)F & 0x8000000000000000ull)));
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
                                                                    const int *__restrict__ maxima,
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
    if (sizeof(T) == 8 && fixed_range(largest_u(maxima), maxima[kMaxP])) return;  // k_projection_div_fixed
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
                                                                       const T *__restrict__ p, double cg,
                                                                       const int *__restrict__ maxima) {
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
    if (sizeof(T) == 8 && fixed_range(maxima[kMaxOld], 0)) return;  // k_projection_update_fixed
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

// The two projection stencils of FP64 fields in 64-bit fixed point, units of
// the field's largest value: the sums are exact in any order, so they are
// formed from a plane's corner and edge sums in shared memory, and the FP64
// pipe, which bound the plain kernels (705 and 306 us at 512x128x128), only
// scales the result.  u has 58 bits (24 terms), p 56 (coefficients up to 96 in
// all), p_old - p_new 59 (8 terms).
template <int TX> struct PlaneTile {
    static constexpr int TY = kStencilThreads / TX;
};

// Per step k: the cells' plane k and the nodes' plane k + 1 in shared memory,
// double buffered; out at the nodes' plane k.
template <int TX>
__global__ void __launch_bounds__(kStencilThreads, 4)
k_projection_div_fixed(LevelDims d, const double *__restrict__ u, const double *__restrict__ p, double cu, double cp,
                       const int *__restrict__ maxima, double *__restrict__ out) {
    constexpr int TY = PlaneTile<TX>::TY, BU = 58, BP = 56;
    constexpr int UH = TX + TY + 1, PH = 2 * (TX + 2) + 2 * TY;  // halo values of a component, of the nodes
    static_assert(3 * UH + PH <= kStencilThreads, "one halo value a thread");
    __shared__ long long su[2][3][TY + 1][TX + 1], sp[2][TY + 2][TX + 2];
    const int m0 = d.n0 - 1, m1 = d.n1 - 1, m2 = d.n2 - 1, tid = threadIdx.x;
    const size_t plane = (size_t)d.n0 * d.n1, N = plane * d.n2;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, k0 = blockIdx.z * d.zc, k1 = k0 + d.zc;
    const int tx = tid % TX, ty = tid / TX, i0 = (y0 + ty) * d.n0 + x0 + tx;
    // the thread's halo value: a cell below the tile (component hc) or a node around it (hc = 3)
    int hc = tid < 3 * UH ? tid / UH : (tid < 3 * UH + PH ? 3 : 4), hx, hy;
    if (hc < 3) {
        const int i = tid % UH;  // column -1 from row -1, then row -1
        hx = i <= TY ? -1 : i - TY - 1;
        hy = i <= TY ? i - 1 : -1;
    } else {
        const int i = tid - 3 * UH;  // rows -1 and TY, then columns -1 and TX
        if (i < 2 * (TX + 2)) hx = i % (TX + 2) - 1, hy = i < TX + 2 ? -1 : TY;
        else hx = (i & 1) ? TX : -1, hy = (i - 2 * (TX + 2)) >> 1;
    }
    const int ho = ((y0 + hy) & m1) * d.n0 + ((x0 + hx) & m0);
    const double *hsrc = (hc < 3 ? u + hc * N : p) + ho;
    grid_dep_wait();
    const int mu = largest_u(maxima), mp = maxima[kMaxP];
    if (!fixed_range(mu, mp)) return;  // k_projection_div
    const int eu = exponent_of<double>(mu), ep = exponent_of<double>(mp);
    // with the units (a field of zeros has none); the conversions of the two
    // sums stay on the FP64 pipe, which this kernel leaves idle (116 us against
    // 109 with them on the integer pipe)
    cu *= mu ? __hiloint2double((eu + 1 - BU) << 20, 0) : 0.0;
    cp *= mp ? __hiloint2double((ep + 1 - BP) << 20, 0) : 0.0;
    double ru[3], rp, rh = 0;
    auto load = [&](int k) {
        const size_t uk = (size_t)(k & m2) * plane, pk = (size_t)((k + 1) & m2) * plane;
#pragma unroll
        for (int c = 0; c < 3; ++c) ru[c] = u[c * N + uk + i0];
        rp = p[pk + i0];
        if (hc < 4) rh = hsrc[hc < 3 ? uk : pk];
    };
    load(k0 - 2);
    long long xy0 = 0, w0 = 0, am = 0, a0 = 0, b0 = 0;
    for (int k = k0 - 2; k < k1; ++k) {
        const int b = k & 1;
#pragma unroll
        for (int c = 0; c < 3; ++c) su[b][c][ty + 1][tx + 1] = to_fixed(ru[c], eu - BU);
        sp[b][ty + 1][tx + 1] = to_fixed(rp, ep - BP);
        if (hc < 3) su[b][hc][hy + 1][hx + 1] = to_fixed(rh, eu - BU);
        else if (hc == 3) sp[b][hy + 1][hx + 1] = to_fixed(rh, ep - BP);
        if (k + 1 < k1) load(k + 1);
        __syncthreads();
        const long long(*U)[TX + 1] = su[b][0], (*V)[TX + 1] = su[b][1], (*W)[TX + 1] = su[b][2];
        const long long(*P)[TX + 2] = sp[b];
        const int i = tx + 1, j = ty + 1;
        const long long xy = (U[j][i] - U[j][i - 1]) + (U[j - 1][i] - U[j - 1][i - 1]) + (V[j][i] - V[j - 1][i]) +
                             (V[j][i - 1] - V[j - 1][i - 1]);
        const long long w = (W[j][i] + W[j][i - 1]) + (W[j - 1][i] + W[j - 1][i - 1]);
        const long long c = (P[j - 1][i - 1] + P[j - 1][i + 1]) + (P[j + 1][i - 1] + P[j + 1][i + 1]);
        const long long e = (P[j - 1][i] + P[j + 1][i]) + (P[j][i - 1] + P[j][i + 1]), m = P[j][i];
        // 16 h^2 D G p = (3c + 2e - 4m)(k-1) + (2c - 4e - 24m)(k) + (3c + 2e - 4m)(k+1)
        const long long a1 = 3 * c + 2 * (e - 2 * m), b1 = 2 * (c - 2 * e - 12 * m);
        if (k >= k0) {
            const long long du = (xy0 + xy) + (w - w0), dg = am + b0 + a1;
            out[(size_t)k * plane + i0] = fma(cp, (double)dg, cu * (double)du);
        }
        xy0 = xy, w0 = w, am = a0, a0 = a1, b0 = b1;
    }
}

template <int TX>
__global__ void __launch_bounds__(kStencilThreads, 4)
k_projection_update_fixed(LevelDims d, double *__restrict__ u, const double *__restrict__ q, double cg,
                          const int *__restrict__ maxima) {
    constexpr int TY = PlaneTile<TX>::TY, B = 59, QH = TX + TY + 1;
    __shared__ long long sq[2][TY + 1][TX + 1];
    const int m0 = d.n0 - 1, m1 = d.n1 - 1, m2 = d.n2 - 1, tid = threadIdx.x;
    const size_t plane = (size_t)d.n0 * d.n1, N = plane * d.n2;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, k0 = blockIdx.z * d.zc, k1 = k0 + d.zc;
    const int tx = tid % TX, ty = tid / TX, i0 = (y0 + ty) * d.n0 + x0 + tx;
    // halo nodes: column TX up to row TY, then row TY
    const int hx = tid <= TY ? TX : tid - TY - 1, hy = tid <= TY ? tid : TY;
    const int ho = ((y0 + hy) & m1) * d.n0 + ((x0 + hx) & m0);
    grid_dep_wait();
    const int mq = maxima[kMaxOld];
    if (!fixed_range(mq, 0)) return;  // k_projection_update
    const int eq = exponent_of<double>(mq);
    double rq, rh = 0, v[3];
    auto load = [&](int k) {  // nodes' plane k + 1, cells' plane k
        const size_t qk = (size_t)((k + 1) & m2) * plane;
        rq = q[qk + i0];
        if (tid < QH) rh = q[qk + ho];
    };
    load(k0 - 1);
    long long gx0 = 0, gy0 = 0, s0 = 0;
    for (int k = k0 - 1; k < k1; ++k) {
        const int b = k & 1;
        sq[b][ty][tx] = to_fixed(rq, eq - B);
        if (tid < QH) sq[b][hy][hx] = to_fixed(rh, eq - B);
        if (k + 1 < k1) load(k + 1);
        double *uk = u + (size_t)k * plane + i0;
        if (k >= k0)
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = uk[c * N];
        __syncthreads();
        const long long q00 = sq[b][ty][tx], q10 = sq[b][ty][tx + 1], q01 = sq[b][ty + 1][tx], q11 = sq[b][ty + 1][tx + 1];
        const long long gx = (q10 + q11) - (q00 + q01), gy = (q01 + q11) - (q00 + q10), s = (q00 + q10) + (q01 + q11);
        if (k >= k0) {
            uk[0] = fma(cg, fixed_value(gx0 + gx, eq - B), v[0]);
            uk[N] = fma(cg, fixed_value(gy0 + gy, eq - B), v[1]);
            uk[2 * N] = fma(cg, fixed_value(s - s0, eq - B), v[2]);
        }
        gx0 = gx, gy0 = gy, s0 = s;
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
    if constexpr (A::kFixed) g.tw = ctx->fft_tab->tw_fx;
    else g.tw = ctx->fft_tab->tw32;
    if constexpr (sizeof(typename A::Real) == 8) g.trig = ctx->fft_tab->trig64;
    else g.trig = ctx->fft_tab->trig32;
    return g;
}

// The spectral solve of ncomp fields from `src` to `dst`: x passes in the
// arithmetic X, the others in A.
template <class X, class A>
static cudaError_t solve(ib_ctx *ctx, const int n[3], int ncomp, const typename A::Real *src, Spectrum<A> c,
                         const SymbolArgs &sy, int out, typename A::Real *dst, typename A::Real *old, int *maxima,
                         cudaStream_t s) {
    const FftGrid<X> gx = fft_grid<X>(ctx, n);
    const FftGrid<A> g = fft_grid<A>(ctx, n);
    const Spectrum<X> cx = {c.c, c.ny, c.logg, c.nylog};
    cudaError_t e = fft_x<X>(kXForward, gx, ncomp, src, cx, nullptr, nullptr, nullptr, s);
    if (e == cudaSuccess) e = fft_y<A>(false, g, ncomp, c, s);
    if (e == cudaSuccess) e = fft_z<A>(g, ncomp, c, sy, s);
    if (e == cudaSuccess) e = fft_y<A>(true, g, ncomp, c, s);
    if (e == cudaSuccess) e = fft_x<X>(out, gx, ncomp, nullptr, cx, dst, old, maxima, s);
    return e;
}

// Maxima of u and p into their words, the others zero.
static cudaError_t field_maxima(ib_ctx *ctx, size_t N, const double *u, const double *p, int *maxima, cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(maxima, 0, kMaxima * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const dim3 grid((ctx->sm_count + 1) / 2, 4);
    if ((((uintptr_t)u | (uintptr_t)p) & 15) == 0)
        k_field_maxima<<<grid, kMaxThreads, 0, s>>>((long long)N, (const double2 *)u, (const double2 *)p, maxima);
    else
        k_field_maxima<<<grid, kMaxThreads, 0, s>>>((long long)N, u, p, maxima);
    return cudaGetLastError();
}

template <class Q, int TX, int MINB>
static cudaError_t launch_rhs(ib_ctx *ctx, LevelDims d, const void *u, const void *p, const RhsArgs &a,
                              const int *maxima, void *out, cudaStream_t s) {
    using S = RhsTile<TX>;
    using T = typename Q::T;
    const size_t smem = sizeof(RhsShared<typename Q::V, TX>);
    auto k = k_predictor_rhs<Q, TX, MINB>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)(d.n0 / TX) * (d.n1 / S::TY);
    d.zc = d.n2 < 32 ? d.n2 : 32;
    while (d.zc > 4 && tiles * (d.n2 / d.zc) < 4LL * ctx->sm_count) d.zc /= 2;
    return launch_pdl(k, dim3(d.n0 / TX, d.n1 / S::TY, d.n2 / d.zc), dim3(S::T), smem, s, d, (const T *)u, (const T *)p,
                      a, maxima, (T *)out);
}
// CTAs per SM: FP32 three (56 registers), fixed point two (80, some spilled: 22
// warps hide more than 11 without), plain FP64 one.
template <int TX>
static cudaError_t predictor_rhs(ib_ctx *ctx, const LevelDims &d, const float *u, const float *p, const RhsArgs &a, int *,
                                 float *out, cudaStream_t s) {
    return launch_rhs<PlainNum<float>, TX, 3>(ctx, d, u, p, a, nullptr, out, s);
}
template <int TX>
static cudaError_t predictor_rhs(ib_ctx *ctx, const LevelDims &d, const double *u, const double *p, const RhsArgs &a,
                                 int *maxima, double *out, cudaStream_t s) {
    cudaError_t e = field_maxima(ctx, (size_t)d.n0 * d.n1 * d.n2, u, p, maxima, s);
    if (e == cudaSuccess) e = launch_rhs<FixedNum, TX, 2>(ctx, d, u, p, a, maxima, out, s);
    if (e == cudaSuccess) e = launch_rhs<PlainNum<double>, TX, 1>(ctx, d, u, p, a, maxima, out, s);
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
    c.logg = c.nylog = 0;
    int *const maxima = ctx->fft_tab->words;
    if (!ar.ok()) return oom_error(ar.used, ar.cap);
    const StencilGrid sg(ctx, grid->n);
    const RhsArgs a = {dt / h, -dt / h, -dt / (4.0 * h * rho_f), 0.5 * nu * dt / (h * h), {dt * g[0], dt * g[1], dt * g[2]}};
    const double points = (double)N;  // the transforms are unscaled
    const SymbolArgs sy(kSolveHelmholtz, 1.0 / points, 0.5 * nu * dt * 4.0 / (h * h));
    PhaseTimer tm(ctx, IB_PHASE_FLUID_PREDICTOR, s);
    // the right-hand side in u_star, the point buffers in the workspace
    cudaError_t e = sg.d.n0 >= 32 ? predictor_rhs<32>(ctx, sg.d, (const T *)u, (const T *)p, a, maxima, (T *)u_star, s)
                                  : predictor_rhs<16>(ctx, sg.d, (const T *)u, (const T *)p, a, maxima, (T *)u_star, s);
    if (e == cudaSuccess) e = solve<A, A>(ctx, grid->n, 3, (const T *)u_star, c, sy, kXField, (T *)u_star, nullptr, nullptr, s);
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
    T *q = ar.take<T>(N);
    c.ny = (typename A::Mem *)q;  // (see Spectrum)
    c.nylog = ilog2_exact(grid->n[0]) - 1;
    const int lines = x_lines<typename A::Pressure>(c.nylog + 1);
    c.logg = ilog2_exact(lines < grid->n[1] ? lines : grid->n[1]);
    int *const maxima = ctx->fft_tab->words;
    if (!ar.ok()) return oom_error(ar.used, ar.cap);
    const StencilGrid sg(ctx, grid->n);
    // p_new = rho_f (D G)^-1 D V   (Eq. ns_lp2 with L p = div((1/rho_f) grad p))
    const SymbolArgs sy(kSolveDivGrad, -rho_f * h * h / 4.0 / (double)N, 0.0);
    PhaseTimer tm(ctx, IB_PHASE_FLUID_PROJECTION, s);
    cudaError_t e = cudaSuccess;
    const double cu = 0.25 / (h * dt), cp = 0.0625 / (h * h * rho_f), cg = dt / (4.0 * h * rho_f);
    const dim3 block1(kStencilThreads);
    if constexpr (sizeof(T) == 8) {
        e = field_maxima(ctx, N, (const double *)u, (const double *)p, maxima, s);
        auto k = sg.d.n0 >= 32 ? k_projection_div_fixed<32> : k_projection_div_fixed<16>;
        if (e == cudaSuccess)
            e = launch_pdl(k, sg.grid, block1, 0, s, sg.d, (const double *)u, (const double *)p, cu, cp, maxima, (double *)q);
    }
    if (e == cudaSuccess)
        e = launch_pdl(k_projection_div<T>, sg.grid, sg.block, 0, s, sg.d, (const T *)u, (const T *)p, cu, cp, maxima, q);
    if (e == cudaSuccess)
        e = solve<typename A::Pressure, A>(ctx, grid->n, 1, q, c, sy, kXPressure, (T *)p, q, maxima + kMaxOld, s);
    if constexpr (sizeof(T) == 8) {
        auto k = sg.d.n0 >= 32 ? k_projection_update_fixed<32> : k_projection_update_fixed<16>;
        if (e == cudaSuccess) e = launch_pdl(k, sg.grid, block1, 0, s, sg.d, (double *)u, (const double *)q, cg, maxima);
    }
    if (e == cudaSuccess)
        e = launch_pdl(k_projection_update<T>, sg.grid, sg.block, 0, s, sg.d, (T *)u, (const T *)q, (const T *)p, cg, maxima);
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
