// Velocity interpolation, force spreading and Algorithm 1 (multidirect
// forcing) of arXiv 2408.14140, Sec. 3.1 Step 2.
//
// Data path on the device
// -----------------------
//  1. Marker preparation: position X_l = X_r + R_l, desired velocity
//     U^d_l = U_r + W_r x R_l (Eq. pr1), the first stencil cell ("anchor",
//     wrapped) and the per-axis kernel weights, computed once per call.
//  2. Binning: every marker is listed in each spreading tile (8^3 cells) its
//     stencil touches.  Tiles are global grid tiles (simultaneous order and
//     ib_spread) or tiles of each particle's own bounding box (sequential
//     order).  Each tile's list is sorted by (anchor row, marker index) once,
//     which fixes the summation order of every cell: spreading is a
//     deterministic gather over marker bins, with no floating-point atomics.
//  3. Passes: per wavefront of non-conflicting particles and per forcing pass
//     m, an interpolation over markers (U, F += (U^d - U)/dt) and a gather over
//     the tiles' cells (u += S (U^d - U) dV / h^3, the increment of Algorithm
//     1's correction), a kernel each; wavefronts beyond the count of the call
//     before run in one persistent cooperative kernel, whose phases are
//     separated by grid-wide barriers with bounded waits.
//
// The correction is applied incrementally, u(m) = u(m-1) + dt S(F^m - F^{m-1}),
// which equals the paper's u(m) = u(0) + dt S F^m in exact arithmetic and
// needs no copy of u(0).
#include <float.h>

#include "ib_device.cuh"

namespace gbib {

// A position along an axis in cells from the first cell's centre (rounded the same
// wherever it is formed).
__device__ __forceinline__ double cell_position(double X, double org, double inv_h) {
    return __fma_rn(__dsub_rn(X, org), inv_h, -0.5);
}

// A marker's wrapped anchor and its per-axis weights in the pass storage
// form (FP32, or double-float pairs for FP64 fields).
template <typename T, int KER>
__device__ __forceinline__ uint64_t marker_weights(const DevGrid &g, const double X[3],
                                                   PS<T> w[12], int first[3]) {
    int a[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double s = cell_position(X[d], g.org[d], g.inv_h);
        const FirstCell f = axis_weights<KER>(s, g.n[d], w + 4 * d);
        first[d] = f.cell;
        a[d] = f.wrapped;
    }
    return pack_anchor(a[0], a[1], a[2]);
}

// A marker's weights to the workspace, 16 bytes a store.
__device__ __forceinline__ void store_weights(float *dst, const float w[12]) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
        ((float4 *)dst)[k] = make_float4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
}
__device__ __forceinline__ void store_weights(float2 *dst, const float2 w[12]) {
#pragma unroll
    for (int k = 0; k < 6; ++k)
        ((float4 *)dst)[k] = make_float4(w[2 * k].x, w[2 * k].y, w[2 * k + 1].x, w[2 * k + 1].y);
}

// ---------------------------------------------------------------------------
// ib_interpolate
// ---------------------------------------------------------------------------
template <typename T, int KER>
__global__ void __launch_bounds__(256) k_interpolate(DevGrid g, const T *__restrict__ u, int M,
                                                     const double *__restrict__ X,
                                                     double *__restrict__ U, DevStatus *st) {
    constexpr int KW = Kernel<KER>::W;
    long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < M; l += gridDim.x * blockDim.x) {
        double x[3] = {X[3 * l], X[3 * l + 1], X[3 * l + 2]};
        if (!finite3(x)) {
            raise_status(st, IB_ERR_NONFINITE, l);
            U[3 * l] = U[3 * l + 1] = U[3 * l + 2] = 0.0;
            continue;
        }
        PS<T> ws[12];
        int first[3];
        uint64_t anc = marker_weights<T, KER>(g, x, ws, first);
        T o[3];
        interp_marker<T, KW>(u, g, N, anc, ws, o);
        U[3 * l] = (double)o[0];
        U[3 * l + 1] = (double)o[1];
        U[3 * l + 2] = (double)o[2];
    }
}

// ---------------------------------------------------------------------------
// marker preparation
// ---------------------------------------------------------------------------
// Standalone spreading: positions X given, source A = F dV / h^3.
template <typename T, int KER>
__global__ void k_prep_spread(DevGrid g, int M, const double *__restrict__ X,
                              const double *__restrict__ F, const double *__restrict__ dV,
                              MarkerState<T> ms, DevStatus *st) {
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < M; l += gridDim.x * blockDim.x) {
        double x[3] = {X[3 * l], X[3 * l + 1], X[3 * l + 2]};
        double f[3] = {F[3 * l], F[3 * l + 1], F[3 * l + 2]};
        double dv = dV[l];
        bool ok = finite3(x) && finite3(f) && isfinite(dv);
        if (!ok) {
            raise_status(st, IB_ERR_NONFINITE, l);
            x[0] = g.org[0];
            x[1] = g.org[1];
            x[2] = g.org[2];
            f[0] = f[1] = f[2] = 0.0;
            dv = 0.0;
        }
        PS<T> w[12];
        int first[3];
        ms.anchor[l] = marker_weights<T, KER>(g, x, w, first);
        store_weights(ms.wts + 12 * (size_t)l, w);
        double q = dv * g.inv_h3;
        ms.A[4 * l + 0] = to_store((T)(f[0] * q));
        ms.A[4 * l + 1] = to_store((T)(f[1] * q));
        ms.A[4 * l + 2] = to_store((T)(f[2] * q));
        ms.A[4 * l + 3] = to_store(T(0));
    }
}

// The marker radius of each particle, rho_p = max_l |R_l| (one CTA per
// particle; a marker with a non-finite input, or any marker of a particle
// with a non-finite state, counts as R_l = 0, as in the marker preparation,
// which reports it).  It reads only the call's inputs, so the conflict lists
// and the wavefront levels, which need rho, run on the context's second
// stream beside the marker preparation.  rho only widens the FP32 conflict
// test (whose margin is h/16), so it is formed in FP32 from the components'
// leading 24 bits (split on the integer pipe, each at most |R_l|) and then
// enlarged by a relative 2^-18, which keeps it an upper bound of max |R_l|
// above the FP32 roundings; no FP64 operation runs per marker.
constexpr int kRadiusThreads = 1024;  // a particle's ~2k markers: two loads in flight per thread
__global__ void __launch_bounds__(kRadiusThreads) k_marker_radius(int P, const double *__restrict__ Xr,
                                                       const double *__restrict__ Ur,
                                                       const double *__restrict__ Wr,
                                                       const int *__restrict__ moff, const double *__restrict__ R,
                                                       const double *__restrict__ dV, double *__restrict__ rho) {
    __shared__ float s_max[kRadiusThreads / 32];
    const int p = blockIdx.x;
    if (p >= P) return;
    const bool pok = finite3(Xr + 3 * p) && finite3(Ur + 3 * p) && finite3(Wr + 3 * p);
    float rmax = 0.0f;  // squared; the root is taken once below
    const int m1 = moff[p + 1];
#pragma unroll 4
    for (int l = moff[p] + threadIdx.x; l < m1; l += blockDim.x) {
        const double r[3] = {R[3 * l], R[3 * l + 1], R[3 * l + 2]};
        if (pok && finite3(r) && finite_bits(dV[l])) {
            const float x = df_split(r[0]).x, y = df_split(r[1]).x, z = df_split(r[2]).x;
            rmax = fmaxf(rmax, fmaf(z, z, fmaf(y, y, x * x)));
        }
    }
    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_down_sync(0xffffffffu, rmax, o));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = rmax;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) rmax = fmaxf(rmax, s_max[w]);
        rho[p] = (double)sqrtf(rmax) * (1.0 + 0x1p-18);
    }
}

// Per particle (kPrepSplit CTAs): marker positions, desired velocities,
// anchors, weights, and the particle's unwrapped stencil box.  Scratch of the
// cross-CTA reductions: per particle the stencil box bounds (lo starts at a
// huge value, hi at a very negative one) and a
// completion count (0).
//
// Bound by the FP64 pipe: FP64 is kept for the position, the first stencil cell
// and the desired velocity; roundings to FP32 run on the integer pipe, a warp
// reduces its box bounds before the atomics, and the weights leave in 16-byte
// stores.  512 spheres of 800 markers, FP32 fields: 76 -> 51 us (20 us for 64
// spheres of 1800 in FP64, as before: few warps, bound by their latency).
struct PrepScratch {
    int *lo, *hi;                // [P][3], from the particle's centre cell
    unsigned int *done;          // [P]
};
constexpr int kPrepSplit = 4;    // CTAs per particle

// A particle's box bounds are counted in 32 bits from about its centre's cell.  Of
// a centre 2^27 cells or more from the origin that cell, and the markers' first
// cells along the axis, take 64 bits: by these calls, after the markers' loop (in
// it, and with the loop's arithmetic modulo 2^32 instead, the kernel took 57 to 60
// us, not 51: other registers, fewer CTAs).  A marker kFar cells or more from its
// centre makes the box too wide.
constexpr int kFar = 1 << 28;
static __device__ __noinline__ long long far_cell(double x, double org, double inv_h) {
    return (long long)floor((x - org) * inv_h);
}
template <int KER>
static __device__ __noinline__ int2 far_bounds(const double *R, const double *dV, int l0, int l1, int d, double xc, double org,
                                               double inv_h) {
    const long long cell = far_cell(xc, org, inv_h);
    int2 b = make_int2(INT_MAX, INT_MIN);
    for (int l = l0; l < l1; l += blockDim.x) {
        const double r = finite3(R + 3 * l) && finite_bits(dV[l]) ? R[3 * l + d] : 0.0;
        const double s = cell_position(xc + r, org, inv_h);
        const long long off = (long long)floor(KER == IB_DELTA_ROMA3 ? s + 0.5 : s) - 1 - cell;
        const bool near = off > -kFar && off < kFar;
        b.x = min(b.x, near ? (int)off : -2 * kFar);
        b.y = max(b.y, near ? (int)off + Kernel<KER>::W - 1 : 2 * kFar);
    }
    return b;
}

template <typename T, int KER>
__global__ void __launch_bounds__(256) k_prep_particles(
    CaseTab ct, int P, const double *__restrict__ Xr, const double *__restrict__ Ur,
    const double *__restrict__ Wr, const int *__restrict__ moff, const double *__restrict__ R,
    const double *__restrict__ dV, MarkerState<T> ms, double *__restrict__ F,
    int4 *__restrict__ box_lo, int4 *__restrict__ box_dim,
    int *__restrict__ part_of, PrepScratch ps, DevStatus *st) {
    constexpr int KW = Kernel<KER>::W;
    __shared__ int s_lo[3], s_hi[3];
    __shared__ int s_last;
    const int p = blockIdx.x / kPrepSplit, part = blockIdx.x % kPrepSplit;
    if (p >= P) return;
    const DevGrid g = ct.of_particle(p).g;
    if (threadIdx.x < 3) {
        s_lo[threadIdx.x] = INT_MAX;
        s_hi[threadIdx.x] = INT_MIN;
    }
    __syncthreads();
    double xc[3] = {Xr[3 * p], Xr[3 * p + 1], Xr[3 * p + 2]};
    double uc[3] = {Ur[3 * p], Ur[3 * p + 1], Ur[3 * p + 2]};
    double wc[3] = {Wr[3 * p], Wr[3 * p + 1], Wr[3 * p + 2]};
    bool pok = finite3(xc) && finite3(uc) && finite3(wc);
    if (!pok && threadIdx.x == 0 && part == 0) raise_status(st, IB_ERR_NONFINITE, p);
    const int m0 = moff[p], m1 = moff[p + 1];
    const int nm = m1 - m0;
    const int l0 = m0 + (int)((long long)part * nm / kPrepSplit), l1 = m0 + (int)((long long)(part + 1) * nm / kPrepSplit);
    int cell[3];  // the bounds' base, the same in all of the particle's CTAs
    bool far = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float c = pok ? (df_round(xc[d]) - df_round(g.org[d])) * df_round(g.inv_h) : 0.0f;
        far = far || !(fabsf(c) < 0x1p27f);
        cell[d] = max(-kFar, min(kFar, __float2int_rd(c)));
    }
    int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
    for (int l = l0 + threadIdx.x; l < l1; l += blockDim.x) {
        double r[3] = {R[3 * l], R[3 * l + 1], R[3 * l + 2]};
        double dv = dV[l];
        if (!pok || !finite3(r) || !finite_bits(dv)) {
            raise_status(st, IB_ERR_NONFINITE, l);
            r[0] = r[1] = r[2] = 0.0;
        }
        double x[3] = {xc[0] + r[0], xc[1] + r[1], xc[2] + r[2]};
        if (!pok) x[0] = g.org[0], x[1] = g.org[1], x[2] = g.org[2];
        PS<T> w[12];
        int first[3];
        ms.anchor[l] = marker_weights<T, KER>(g, x, w, first);
        store_weights(ms.wts + 12 * (size_t)l, w);
        const double ud[3] = {uc[0] + (wc[1] * r[2] - wc[2] * r[1]), uc[1] + (wc[2] * r[0] - wc[0] * r[2]),
                              uc[2] + (wc[0] * r[1] - wc[1] * r[0])};
        if constexpr (sizeof(T) == 4) {
            const float2 a = df_round_pair(ud[0]), b = df_round_pair(ud[1]), c = df_round_pair(ud[2]);
            ((float4 *)(ms.Ud32 + 8 * (size_t)l))[0] = make_float4(a.x, b.x, c.x, df_round(dv * g.inv_h3));
            ((float4 *)(ms.Ud32 + 8 * (size_t)l))[1] = make_float4(a.y, b.y, c.y, 0.f);
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) ms.Ud[3 * l + c] = ud[c];
        }
        F[3 * l] = F[3 * l + 1] = F[3 * l + 2] = 0.0;
        part_of[l] = p;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int off = max(-kFar, min(kFar, first[d] - cell[d]));
            lo[d] = min(lo[d], off);
            hi[d] = max(hi[d], off + KW - 1);
        }
    }
    const bool wide = min(min(lo[0], lo[1]), lo[2]) <= -kFar || max(max(hi[0], hi[1]), hi[2]) >= kFar;
    if (far || wide) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int2 b = far ? far_bounds<KER>(R, dV, l0 + threadIdx.x, l1, d, xc[d], g.org[d], g.inv_h)
                               : make_int2(-2 * kFar, 2 * kFar);
            lo[d] = b.x, hi[d] = b.y;
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        lo[d] = __reduce_min_sync(0xffffffffu, lo[d]);
        hi[d] = __reduce_max_sync(0xffffffffu, hi[d]);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&s_lo[d], lo[d]);
            atomicMax(&s_hi[d], hi[d]);
        }
    }
    __syncthreads();
    // combine the particle's CTAs; the last one to finish writes the results
    if (threadIdx.x == 0) {
        for (int d = 0; d < 3; ++d) {
            atomicMin(&ps.lo[3 * p + d], s_lo[d]);
            atomicMax(&ps.hi[3 * p + d], s_hi[d]);
        }
        __threadfence();
        s_last = atomicAdd(&ps.done[p], 1u) == kPrepSplit - 1;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_last) {
        long long blo[3];
        int dims[3];
        for (int d = 0; d < 3; ++d) {
            const int l = atomicAdd(&ps.lo[3 * p + d], 0), h = atomicAdd(&ps.hi[3 * p + d], 0);
            blo[d] = (far ? far_cell(xc[d], g.org[d], g.inv_h) : cell[d]) + l;
            dims[d] = h - l + 1;
        }
        if (m1 > m0) {
            box_lo[p] = make_int4(wrap_int(blo[0], g.n[0]), wrap_int(blo[1], g.n[1]), wrap_int(blo[2], g.n[2]), 0);
            box_dim[p] = make_int4(dims[0], dims[1], dims[2], 0);
            for (int d = 0; d < 3; ++d)
                if (dims[d] > kMaxBox || dims[d] > g.n[d]) raise_status(st, IB_ERR_UNSUPPORTED, p);
        } else {
            box_lo[p] = make_int4(0, 0, 0, 0);
            box_dim[p] = make_int4(0, 0, 0, 0);
        }
    }
}

// ---------------------------------------------------------------------------
// wavefront levels (sequential order).  One CTA.
// Particles p and q conflict when their marker stencils may share a cell:
// nearest-image centre distance < rho_p + rho_q + sqrt(3) * W * h.  level(p)
// = 1 + max level(q) over conflicting q < p; a level's particles have
// pairwise disjoint stencil supports, so running a level at once equals
// running its particles one after another.
// ---------------------------------------------------------------------------
struct LevelOut {
    int *level;       // [P]
    int *rank;        // [P] position of p in level-major order
    int *mbase;       // [P] first slot of p's markers in the level-major marker list
    int *lev_pbeg;    // [P+1] first level-major rank of each level
    int *lev_mbeg;    // [P+1] first level-major marker of each level
    int *nlev;        // [1]
};


// Conflict lists: for every p, the q < p whose stencils may share a cell
// (count -1 = more than kMaxNbr, scanned again when levels are assigned).
// The test runs in FP32 against a limit widened by h/16, far above FP32
// rounding of unit-scale positions, so no true conflict is ever missed (an
// extra conflict only serialises two particles).
__global__ void k_conflicts(CaseTab ct, int P, int KW, const double *__restrict__ Xr,
                            const double *__restrict__ rho, int *__restrict__ nbr_cnt,
                            int *__restrict__ nbr) {
    grid_dep_wait();
    // one warp per particle p; lanes test q = p0 + lane, p0 + 32 + lane, ...
    // and the hits are appended in ascending q (ballot order)
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < P; p += nw) {
        const DevCase cd = ct.of_particle(p);
        const DevGrid &g = cd.g;
        const float L[3] = {(float)(g.n[0] * g.h), (float)(g.n[1] * g.h), (float)(g.n[2] * g.h)};
        const float iL[3] = {1.0f / L[0], 1.0f / L[1], 1.0f / L[2]};
        const float halo = (float)(1.7320508075688772 * KW * g.h + 0.0625 * g.h);
        const float xp[3] = {(float)Xr[3 * p], (float)Xr[3 * p + 1], (float)Xr[3 * p + 2]};
        const float rp = (float)rho[p] + halo;
        int cnt = 0;
        for (int q0 = cd.p0; q0 < p; q0 += 32) {  // particles of other cases never conflict
            const int q = q0 + lane;
            bool hit = false;
            if (q < p) {
                float d2 = 0.0f;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    float d = (float)Xr[3 * q + a] - xp[a];
                    d -= L[a] * rintf(d * iL[a]);
                    d2 += d * d;
                }
                const float lim = rp + (float)rho[q];
                hit = d2 < lim * lim;
            }
            const unsigned b = __ballot_sync(0xffffffffu, hit);
            const int pos = cnt + __popc(b & ((1u << lane) - 1u));
            if (hit && pos < kMaxNbr) nbr[(size_t)p * kMaxNbr + pos] = q;
            cnt += __popc(b);
        }
        if (lane == 0) nbr_cnt[p] = cnt <= kMaxNbr ? cnt : -1;
    }
}

// Levels by a sweep over each case's particles in index order (level(p)
// needs only the q < p of its own case; cases are independent and swept in
// parallel, one thread each), then a parallel counting sort of the particles
// by level and the level-major marker offsets.  The sweep's dependent reads
// stay on chip: levels in shared memory (up to kLevOnchipP particles) and the
// conflict lists too when they fit (kLevNbrP).  The order of particles inside
// a level is the order their atomic increments land in; it does not affect
// any result (a level's particles have disjoint stencil supports).
constexpr int kLevOnchipP = 8192;
constexpr int kLevNbrP = 1024;
constexpr size_t kLevSmem = (size_t)kLevOnchipP * 4 + (size_t)kLevNbrP * (2 + 2 * kMaxNbr);

// Exclusive scan of f(0..n-1) by one CTA (chunks of blockDim.x), calling
// out(i, prefix) for every i and returning the total (all threads).
template <typename F, typename O>
__device__ __forceinline__ int block_scan_chunked(int n, F f, O out) {
    __shared__ int s_w[32];
    __shared__ int s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < n; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const int v = i < n ? f(i) : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        int wpre = 0;
        for (int w = 0; w < warp; ++w) wpre += s_w[w];
        const int carry = s_carry;
        if (i < n) out(i, carry + wpre + x - v);
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
            for (int w = 0; w < nw; ++w) t += s_w[w];
            s_carry = carry + t;
        }
        __syncthreads();
    }
    return s_carry;
}

constexpr int kLevSweeps = 64;  // parallel relaxation sweeps before the ordered sweep
// threads of the one k_levels CTA: 512 (24k registers) fit on an SM beside a
// marker-preparation CTA, so the levels need not wait for that kernel's tail
constexpr int kLevThreads = 512;

__global__ void __launch_bounds__(kLevThreads) k_levels(CaseTab ct, int P, int order, int KW,
                                                 const double *__restrict__ Xr,
                                                 const double *__restrict__ rho,
                                                 const int *__restrict__ moff,
                                                 const int *__restrict__ nbr_cnt,
                                                 const int *__restrict__ nbr, LevelOut lo,
                                                 int *__restrict__ by_rank, int *__restrict__ lev_cur) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char lsm[];
    __shared__ int s_nl;
    const bool lev_on = P <= kLevOnchipP;
    const bool nbr_on = P <= kLevNbrP && order == IB_ORDER_SEQUENTIAL;
    int *lev = lev_on ? (int *)lsm : lo.level;
    short *s_cnt = (short *)(lsm + (size_t)kLevOnchipP * 4);
    unsigned short *s_nbr = (unsigned short *)(s_cnt + kLevNbrP);
    if (threadIdx.x == 0) s_nl = 0;
    for (int i = threadIdx.x; i <= P; i += blockDim.x) {
        lo.lev_pbeg[i] = 0;
        lev_cur[i] = 0;
    }
    if (nbr_on)
        for (int p = threadIdx.x; p < P; p += blockDim.x) {
            const int c = nbr_cnt[p];
            s_cnt[p] = (short)c;
            for (int k = 0; k < c; ++k) s_nbr[p * kMaxNbr + k] = (unsigned short)nbr[(size_t)p * kMaxNbr + k];
        }
    __threadfence();  // the zeroed counters reach L2 before the atomics below
    __syncthreads();
    int mymax = 0;
    // ---- parallel levels: lev(p) = 1 + max lev(q) over conflicting q < p (0
    // without), the longest path to p in the conflict DAG, relaxed for all
    // particles at once until nothing changes.  Values only grow and never
    // pass the fixed point, so reading a neighbour's value mid-sweep is
    // harmless; a conflict chain of length c takes c + 1 sweeps.  Full
    // conflict lists, or chains longer than kLevSweeps, fall back to the
    // sweep in particle order below (which recomputes every level).
    __shared__ int s_flag;
    bool levels_done = false;
    if (order == IB_ORDER_SEQUENTIAL) {
        volatile int *vlev = lev;
        if (threadIdx.x == 0) s_flag = 0;
        __syncthreads();
        for (int p = threadIdx.x; p < P; p += blockDim.x) {
            if ((nbr_on ? s_cnt[p] : nbr_cnt[p]) < 0) s_flag = 1;
            vlev[p] = 0;
        }
        __syncthreads();
        const bool any_full = s_flag != 0;
        __syncthreads();
        for (int it = 0; !any_full && it < kLevSweeps; ++it) {
            if (threadIdx.x == 0) s_flag = 0;
            __syncthreads();
            for (int p = threadIdx.x; p < P; p += blockDim.x) {
                const int cn = nbr_on ? s_cnt[p] : nbr_cnt[p];
                int best = 0;
                for (int k = 0; k < cn; ++k)
                    best = max(best, vlev[nbr_on ? s_nbr[p * kMaxNbr + k] : nbr[(size_t)p * kMaxNbr + k]] + 1);
                if (best != vlev[p]) {
                    vlev[p] = best;
                    s_flag = 1;
                }
            }
            __syncthreads();
            const bool changed = s_flag != 0;
            __syncthreads();
            if (!changed) {
                levels_done = true;
                break;
            }
        }
        if (levels_done)
            for (int p = threadIdx.x; p < P; p += blockDim.x) mymax = max(mymax, vlev[p] + 1);
    }
    // ---- sweep in particle order, one thread per case
    const int ncases = ct.arr ? ct.ncases : 1;
    for (int c = threadIdx.x; !levels_done && c < ncases; c += blockDim.x) {
        const DevCase cd = ct.get(c);
        for (int p = cd.p0; p < cd.p1; ++p) {
            int best = 0;
            if (order == IB_ORDER_SEQUENTIAL) {
                const int cn = nbr_on ? s_cnt[p] : nbr_cnt[p];
                if (cn >= 0) {
                    for (int k = 0; k < cn; ++k)
                        best = max(best, lev[nbr_on ? s_nbr[p * kMaxNbr + k] : nbr[(size_t)p * kMaxNbr + k]] + 1);
                } else {
                    const DevGrid &g = cd.g;
                    const double L[3] = {g.n[0] * g.h, g.n[1] * g.h, g.n[2] * g.h};
                    const double iL[3] = {1.0 / L[0], 1.0 / L[1], 1.0 / L[2]};
                    const double halo = 1.7320508075688772 * KW * g.h;
                    for (int q = cd.p0; q < p; ++q) {
                        float d2 = 0.0f;
                        for (int a = 0; a < 3; ++a) {
                            float d = (float)Xr[3 * q + a] - (float)Xr[3 * p + a];
                            d -= (float)L[a] * rintf(d * (float)iL[a]);
                            d2 += d * d;
                        }
                        const float lim = (float)(rho[p] + rho[q] + halo + 0.0625 * g.h);
                        if (d2 < lim * lim) best = max(best, lev[q] + 1);
                    }
                }
            }
            lev[p] = best;
            mymax = max(mymax, best + 1);
        }
    }
    atomicMax(&s_nl, mymax);
    __syncthreads();
    const int nl = s_nl;
    // ---- counting sort by level
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        if (lev_on) lo.level[p] = lev[p];
        atomicAdd(&lo.lev_pbeg[lev[p]], 1);
    }
    __syncthreads();
    // counts -> exclusive offsets, in place (read through atomics: written by atomics above)
    block_scan_chunked(nl, [&](int l) { return atomicAdd(&lo.lev_pbeg[l], 0); },
                       [&](int l, int pre) { atomicExch(&lev_cur[l], pre); });
    __syncthreads();
    // (values shared through L2 are written and read with atomics throughout)
    for (int l = threadIdx.x; l < nl; l += blockDim.x) atomicExch(&lo.lev_pbeg[l], atomicAdd(&lev_cur[l], 0));
    if (threadIdx.x == 0) {
        lo.lev_pbeg[nl] = P;
        *lo.nlev = nl;
    }
    __syncthreads();
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        const int r = atomicAdd(&lev_cur[lev[p]], 1);
        lo.rank[p] = r;
        atomicExch(&by_rank[r], p);
    }
    __syncthreads();
    // ---- level-major marker offsets: exclusive scan of marker counts by rank
    const int M = block_scan_chunked(
        P, [&](int r) { const int p = atomicAdd(&by_rank[r], 0); return moff[p + 1] - moff[p]; },
        [&](int r, int pre) { atomicExch(&lo.mbase[atomicAdd(&by_rank[r], 0)], pre); });
    __syncthreads();
    for (int l = threadIdx.x; l < nl; l += blockDim.x) {
        const int r = atomicAdd(&lo.lev_pbeg[l], 0);
        lo.lev_mbeg[l] = atomicAdd(&lo.mbase[atomicAdd(&by_rank[r], 0)], 0);
    }
    if (threadIdx.x == 0) lo.lev_mbeg[nl] = M;
}

// ---------------------------------------------------------------------------
// slot counting and filling
// ---------------------------------------------------------------------------
// Tiles a marker's stencil touches along one axis: distinct tile indices of
// the KW cells from `first`.  Global tiles use wrapped cells; local tiles use
// cells relative to the particle box (no wrap, box <= grid).
template <int KW>
__device__ __forceinline__ int axis_tiles_global(int first, int n, int t[3]) {
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const int tt = wrap_add(first, k, n) / kTile;
        int j = 0;
        while (j < cnt && t[j] != tt) ++j;
        if (j == cnt && cnt < 3) t[cnt++] = tt;
    }
    return cnt;
}

template <int KW>
__device__ __forceinline__ int axis_tiles_local(int first_rel, int t[3]) {
    t[0] = first_rel / kTile;
    t[1] = (first_rel + KW - 1) / kTile;
    return t[1] != t[0] ? 2 : 1;
}

struct SlotGeom {
    int mode;              // 0 global tiles (per case), 1 particle-local tiles
    const int *part_of;    // [M], nullptr: every marker in case 0
    const int *rank;       // [P]
    const int4 *box_lo;    // [P]
    const int4 *box_dim;   // [P]
};

// Enumerate the dense slots of marker l and call f(slot).
template <int KW, typename Fn>
__device__ __forceinline__ void for_marker_slots(const CaseTab &ct, const SlotGeom &sg, int l,
                                                 uint64_t anc, Fn f) {
    int tx[3], ty[3], tz[3], nx, ny, nz;
    uint32_t base = 0;
    const DevCase &cd = ct.get(sg.part_of ? ct.case_of(sg.part_of[l]) : 0);
    const DevGrid &g = cd.g;
    if (sg.mode == 0) {
        nx = axis_tiles_global<KW>(anchor_x(anc), g.n[0], tx);
        ny = axis_tiles_global<KW>(anchor_y(anc), g.n[1], ty);
        nz = axis_tiles_global<KW>(anchor_z(anc), g.n[2], tz);
    } else {
        int p = sg.part_of[l];
        int4 blo = sg.box_lo[p];
        // relative first cell: (anchor - box_lo) mod n, < box dims
        // box_lo is wrapped by the preparation kernel: [0, n)
        const int rx = wrap_diff(anchor_x(anc), blo.x, g.n[0]);
        const int ry = wrap_diff(anchor_y(anc), blo.y, g.n[1]);
        const int rz = wrap_diff(anchor_z(anc), blo.z, g.n[2]);
        nx = axis_tiles_local<KW>(rx, tx);
        ny = axis_tiles_local<KW>(ry, ty);
        nz = axis_tiles_local<KW>(rz, tz);
        // a box wider than kMaxBox is reported by the preparation kernel;
        // keep every slot id in range regardless
        if (tx[nx - 1] >= kLocalTiles || ty[ny - 1] >= kLocalTiles || tz[nz - 1] >= kLocalTiles) return;
        base = (uint32_t)sg.rank[p] * kLocalSlots;
    }
    for (int k = 0; k < nz; ++k)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                uint32_t s;
                if (sg.mode == 0)
                    s = cd.tile_off + ((uint32_t)tz[k] * cd.tiles[1] + ty[j]) * cd.tiles[0] + tx[i];
                else
                    s = base + ((uint32_t)tz[k] * kLocalTiles + ty[j]) * kLocalTiles + tx[i];
                f(s);
            }
}

template <int KW>
__global__ void k_slot_count(CaseTab ct, int M, SlotGeom sg, const uint64_t *__restrict__ anchor,
                             uint32_t *__restrict__ count) {
    grid_dep_wait();
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < M; l += gridDim.x * blockDim.x)
        for_marker_slots<KW>(ct, sg, l, anchor[l], [&](uint32_t s) { atomicAdd(count + s, 1u); });
}

template <int KW>
__global__ void k_slot_fill(CaseTab ct, int M, SlotGeom sg, const uint64_t *__restrict__ anchor,
                            const uint32_t *__restrict__ start, uint32_t *__restrict__ cursor,
                            uint32_t *__restrict__ cand) {
    grid_dep_wait();
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < M; l += gridDim.x * blockDim.x)
        for_marker_slots<KW>(ct, sg, l, anchor[l], [&](uint32_t s) {
            cand[start[s] + atomicAdd(cursor + s, 1u)] = (uint32_t)l;
        });
}

// ---------------------------------------------------------------------------
// single-pass exclusive scans (decoupled look-back, Merrill & Garland 2016):
// each CTA takes the next tile of kLbTile elements from a ticket counter,
// publishes its tile sum, then -- walking back over the tiles before it
// until one has published its inclusive prefix -- its own inclusive prefix,
// and scans the tile from that base.  A tile waits only for tiles taken
// earlier by CTAs already running, so every wait ends; each is bounded all
// the same (IB_ERR_TIMEOUT).  Tile words pack a 2-bit state (0 none,
// 1 tile sum, 2 inclusive prefix) above a 62-bit value; the words and the
// ticket are zeroed before the call's kernel chain.
// ---------------------------------------------------------------------------
constexpr int kLbThreads = 256, kLbItems = 8, kLbTile = kLbThreads * kLbItems;
constexpr unsigned long long kLbVal = (1ull << 62) - 1;

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Exclusive scan of one value per thread over the CTA (64-bit, fixed order).
__device__ __forceinline__ unsigned long long lb_block_scan(unsigned long long v, unsigned long long *total) {
    __shared__ unsigned long long s_w[kLbThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    unsigned long long wbase = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kLbThreads / 32; ++w) {
        if (w < warp) wbase += s_w[w];
        tot += s_w[w];
    }
    *total = tot;
    return wbase + x - v;
}

// The tile's exclusive base: warp 0 publishes the tile sum, then reads the
// words of the 32 tiles before it at once (lane l: tile - 1 - l), waiting for
// each to be published, and adds the sums up to the nearest inclusive prefix;
// without one it moves 32 tiles further back.  Positions before tile 0 count
// as an inclusive prefix of 0.  Every thread gets the base.  false: a wait
// gave up.
__device__ __forceinline__ bool lb_tile_base(int tile, unsigned long long tot, unsigned long long *tstat,
                                             DevStatus *st, unsigned long long &base) {
    __shared__ unsigned long long s_base;
    __shared__ int s_ok;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        unsigned long long pre = 0;
        bool ok = true;
        if (tile > 0) {
            if (lane == 0) st_release64(tstat + tile, (1ull << 62) | tot);
            for (int hi = tile - 1;; hi -= 32) {
                const int j = hi - lane;
                unsigned long long w = j >= 0 ? ld_acquire64(tstat + j) : (2ull << 62);
                if ((w >> 62) == 0) {
                    const long long t0 = clock64();
                    do {
                        if (clock64() - t0 > kSpinCycles) {
                            raise_status(st, IB_ERR_TIMEOUT, -2);
                            w = 2ull << 62;  // give up: stop here
                            ok = false;
                            break;
                        }
                        w = ld_acquire64(tstat + j);
                    } while ((w >> 62) == 0);
                }
                __syncwarp();
                const unsigned incl = __ballot_sync(0xffffffffu, (w >> 62) == 2);
                const int first = incl ? __ffs(incl) - 1 : 31;
                unsigned long long v = (lane <= first && j >= 0) ? (w & kLbVal) : 0ull;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                pre += v;
                if (incl) break;
            }
            ok = __all_sync(0xffffffffu, ok);
        }
        if (lane == 0) {
            st_release64(tstat + tile, (2ull << 62) | ((pre + tot) & kLbVal));
            s_base = pre;
            s_ok = ok ? 1 : 0;
        }
    }
    __syncthreads();
    base = s_base;
    return s_ok != 0;
}

// The dense slots: start = exclusive scan of the counts, flag_scan =
// exclusive scan of (count > 0), and dense_of[flag_scan[i]] = i for every
// non-empty slot i -- one pass over the counts (the two sums packed in one
// 64-bit word: counts below, flags from bit 32).
__global__ void __launch_bounds__(kLbThreads) k_slot_scan(const uint32_t *__restrict__ count, int n,
                                                          uint32_t *__restrict__ start,
                                                          uint32_t *__restrict__ flag_scan,
                                                          uint32_t *__restrict__ dense_of,
                                                          unsigned long long *tstat, unsigned int *ticket,
                                                          DevStatus *st) {
    __shared__ int s_tile;
    grid_dep_wait();
    if (threadIdx.x == 0) s_tile = (int)atomicAdd(ticket, 1u);
    __syncthreads();
    const int tile = s_tile;
    const int i0 = tile * kLbTile + threadIdx.x * kLbItems;
    uint32_t c[kLbItems];
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < kLbItems; ++k) {
        c[k] = i0 + k < n ? count[i0 + k] : 0u;
        sum += (unsigned long long)c[k] | ((unsigned long long)(c[k] != 0u) << 32);
    }
    unsigned long long tot, base;
    const unsigned long long ex = lb_block_scan(sum, &tot);
    if (!lb_tile_base(tile, tot, tstat, st, base)) return;
    unsigned long long run = base + ex;
#pragma unroll
    for (int k = 0; k < kLbItems; ++k) {
        const int i = i0 + k;
        if (i < n) {
            start[i] = (uint32_t)run;
            flag_scan[i] = (uint32_t)(run >> 32);
            if (c[k]) dense_of[run >> 32] = (uint32_t)i;
        }
        run += (unsigned long long)c[k] | ((unsigned long long)(c[k] != 0u) << 32);
    }
    if (i0 <= n && n < i0 + kLbItems) {  // the thread holding position n writes the totals
        start[n] = (uint32_t)run;
        flag_scan[n] = (uint32_t)(run >> 32);
    }
}

// Per wavefront, the slices of its tiles, longest first (a counting sort by
// their rows; equal ones in any order): one warp of the wavefront gather takes
// a slice, and the last round of warps then has the shortest.  Only the order
// of work changes.  Wavefront L's list starts at lev_slice[L].x, taken from the
// cursor in whatever order the wavefronts come, and has lev_slice[L].y entries
// {tile, slice, first pair of the tile, cells}.  A wavefront's tiles are consecutive:
// global tiles form one, a particle's local tiles follow its rank.
constexpr int kSliceOrderThreads = 1024;
__global__ void __launch_bounds__(kSliceOrderThreads) k_level_slices(int mode, const int *__restrict__ nlev_p,
                                                                     const int *__restrict__ lev_pbeg, int ndense,
                                                                     Slots sl, unsigned int *__restrict__ cursor,
                                                                     int2 *__restrict__ lev_slice,
                                                                     int4 *__restrict__ slices) {
    grid_dep_wait();
    __shared__ int s_hist[256], s_base;
    const int nl = *nlev_p;
    auto first_tile = [&](int L) {
        if (mode == 0) return L == 0 ? 0 : (int)sl.flag_scan[ndense];
        const long long d = (long long)lev_pbeg[L] * kLocalSlots;
        return (int)sl.flag_scan[d < ndense ? d : ndense];
    };
    for (int L = blockIdx.x; L < nl; L += gridDim.x) {  // one CTA per wavefront
        const int s0 = first_tile(L), s1 = first_tile(L + 1);
        int base = 0;
        for (int k = threadIdx.x; k < 256; k += blockDim.x) s_hist[k] = 0;
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {
            for (int t = s0 + threadIdx.x; t < s1; t += blockDim.x) {
                const int4 ti = sl.tinfo[t];
                const uint4 l4 = sl.slen[t];
                const unsigned lw[4] = {l4.x, l4.y, l4.z, l4.w};
                const int ns = (ti.z + 31) >> 5;
#pragma unroll
                for (int s = 0; s < 16; ++s)
                    if (s < ns) {
                        const int j = atomicAdd(&s_hist[255 - ((lw[s >> 2] >> (8 * (s & 3))) & 255u)], 1);
                        if (pass) slices[base + j] = make_int4(t, s, ti.x, ti.z);
                    }
            }
            __syncthreads();
            if (pass == 0) {
                const int total =
                    block_scan_chunked(256, [&](int k) { return s_hist[k]; }, [&](int k, int pre) { s_hist[k] = pre; });
                if (threadIdx.x == 0) {
                    s_base = (int)atomicAdd(cursor, (unsigned)total);
                    lev_slice[L] = make_int2(s_base, total);
                }
                __syncthreads();
                base = s_base;
            }
        }
        __syncthreads();
    }
}

// Level-major marker list: the markers of the particle of rank r follow
// those of the particles of lower rank, each particle's in index order (the
// Fibonacci lattice index already walks the sphere band by band in z; a
// spatial sort of each particle's markers measured slower end to end).
__global__ void k_marker_order(int P, const int *__restrict__ moff, const int *__restrict__ mbase,
                               int *__restrict__ mperm) {
    grid_dep_wait();
    for (int p = blockIdx.x; p < P; p += gridDim.x) {
        const int m0 = moff[p], n = moff[p + 1] - m0, base = mbase[p];
        for (int i = threadIdx.x; i < n; i += blockDim.x) mperm[base + i] = m0 + i;
    }
}

// Case of dense global-tile slot d: the last case whose tile_off <= d.
__device__ __forceinline__ int case_of_tile(const CaseTab &ct, uint32_t d) {
    if (!ct.arr) return 0;
    int a = 0, b = ct.ncases - 1;
    while (a < b) {
        const int mid = (a + b + 1) >> 1;
        if (ct.arr[mid].tile_off <= d) a = mid;
        else b = mid - 1;
    }
    return a;
}

__device__ __forceinline__ int slot_geometry(const CaseTab &ct, int mode, const SlotGeom &sg, const Slots &sl,
                                             const int *level, uint32_t d, uint32_t b, int lo[3], int dim[3],
                                             int &lev) {
    lev = 0;
    if (mode == 0) {
        const int c = case_of_tile(ct, d);
        const DevCase &cd = ct.get(c);
        const DevGrid &g = cd.g;
        d -= cd.tile_off;
        const int t[3] = {(int)(d % cd.tiles[0]), (int)((d / cd.tiles[0]) % cd.tiles[1]),
                          (int)(d / ((uint32_t)cd.tiles[0] * cd.tiles[1]))};
        for (int a = 0; a < 3; ++a) {
            lo[a] = t[a] * kTile;
            dim[a] = min(kTile, g.n[a] - lo[a]);
        }
        return c;
    } else {
        const int p = sg.part_of[sl.cand[b]];  // every candidate of a local tile has the same particle
        const DevGrid &g = ct.of_particle(p).g;
        const int lt = (int)(d % kLocalSlots);
        const int t[3] = {lt % kLocalTiles, (lt / kLocalTiles) % kLocalTiles, lt / (kLocalTiles * kLocalTiles)};
        const int4 blo = sg.box_lo[p], bd = sg.box_dim[p];
        const int bl[3] = {blo.x, blo.y, blo.z}, bdm[3] = {bd.x, bd.y, bd.z};
        for (int a = 0; a < 3; ++a) {
            lo[a] = wrap_int((long long)bl[a] + t[a] * kTile, g.n[a]);
            dim[a] = min(kTile, bdm[a] - t[a] * kTile);
        }
        lev = level[p];
        return ct.case_of(p);
    }
}

// v mod n for v in [-n, 2n)
__device__ __forceinline__ int wrap_once(int v, int n) {
    v += v < 0 ? n : 0;
    return v >= n ? v - n : v;
}

__device__ __forceinline__ unsigned long long slot_key(const DevGrid &g, const uint64_t *anchor, uint32_t m,
                                                       const int lo[3]) {
    const uint64_t anc = anchor[m];
    // anchor and lo lie in [0, n): one conditional add or subtract wraps
    const int rz = wrap_once(anchor_z(anc) - lo[2] + 3, g.n[2]);
    const int ry = wrap_once(anchor_y(anc) - lo[1] + 3, g.n[1]);
    const int v = wrap_once(anchor_x(anc) - lo[0] + 3, g.n[0]);
    const int bin = (rz < kRow && ry < kRow && v < kRow) ? (rz * kRow + ry) * kBinsPerRow + v
                                                         : kBins - 1;  // never read
    return ((unsigned long long)bin << 32) | m;
}

// The bins' starts of slot cs (only the particle-resident form reads them):
// bin_of(i) the bin of sorted candidate i; `lane`/`nl` split the work.
template <class Bin>
__device__ __forceinline__ void slot_bins(int nc, int cs, const Slots &sl, int lane, int nl, Bin bin_of) {
    uint16_t *bs = sl.bins + (size_t)cs * kBins;
    for (int r = lane; r < kBins; r += nl) {
        // first index whose bin >= r
        int a = 0, e = nc;
        while (a < e) {
            const int mid = (a + e) >> 1;
            if (bin_of(mid) < r) a = mid + 1;
            else e = mid;
        }
        bs[r] = (uint16_t)(r == kBins - 1 ? nc : a);
    }
}

// ---------------------------------------------------------------------------
// sorted candidates and per-cell gather lists.  A cell's contributions are the
// candidates whose stencil covers it.  The bin walk of gather_cell visits a
// tile's bins in ascending (anchor z, y, x) order and a bin's candidates in
// index order -- in ascending candidate index, the order the tile's candidates
// are sorted in -- so listing every cell's candidates in ascending index
// reproduces its summation order.
//
// A stencil is a product of three ranges, so cell (x, y, z)'s candidates are
// the intersection of three bit sets over the candidates: those covering
// column x, row y and plane z of the tile.  The 24 bit sets come from warp
// ballots, 32 candidates at a time; a cell's pair count is the population of
// its intersection, and its list the set bits in ascending order -- no
// ranking, no atomics and no walk over the candidates.  Only the cells with a
// list (about a third of the tile's) get a thread for the emission, and the
// list goes through shared memory, so that pair words and weights leave in
// coalesced rows.
//
// A tile has about 70 candidates and 950 pairs: a CTA of four warps takes one,
// ten CTAs an SM (eight warps a tile idled in barriers; one warp a tile was
// bound by its own latency).  It sorts by rank: every thread counts the keys
// below its own, 32 bits wide, the bin and the marker's distance from the
// tile's first one (64 where that does not fit).  Tiles of more than kListCand
// candidates go to a second kernel, whose CTAs sort them by a bitonic network.
// ---------------------------------------------------------------------------
// The lists' layout.  The wavefront gather takes 32 cells a warp (a slice), so
// a tile's cells are ordered by list length, longest first, and a slice's
// pairs lie row by row: row k holds the k-th pair of every cell that has one,
// in lane order, with no padding (jagged diagonal storage; a lane's place in a
// row is its rank among the lanes with more than k pairs).  A pair is its
// marker and its weight.  The group kernels walk a cell's pairs alone: for
// them each list is contiguous and a pair is candidate | offset << 16.
constexpr int kListThreads = 128;
constexpr int kListCtas = 10;              // CTAs of an SM
constexpr int kSpreadCtas = 6;             // of the summing form (5 and 8: 90 and 99 us)
constexpr int kListCand = 512;
constexpr int kPairThreads = 256;          // the large tiles' CTAs
constexpr int kPairWords = kMaxCand / 32;  // words of a bit set
constexpr int kMarkBits = 21;
constexpr int kSlices = kTileCells / 32;   // slices of a tile
constexpr int kLenBins = 128;              // list lengths told apart in the order (longer: any order)
static_assert(kTileCells == 4 * kListThreads && kTileCells == 2 * kPairThreads && kBins <= 1 << (32 - kMarkBits) &&
                  kSlices == 16,
              "tile lists");

struct ListShared {
    int hist[kLenBins];
    int sum[kSlices];                      // pairs of each slice
    uint16_t cell[kTileCells], cnt[kTileCells];
    // rows of each slice (at most 255 told), read as one 16-byte word
    alignas(16) unsigned char len[kSlices];
    int nb;                                // band cells
    int np;                                // pairs of the tile
    uint32_t base;                         // its first pair
};
static_assert(offsetof(ListShared, len) % 16 == 0 && alignof(ListShared) == 16, "16-byte read");
struct CtaLists {
    unsigned long long keys[kMaxCand];
    unsigned set[3 * kTile][kPairWords + 1];
    short first[kMaxCand];
    ListShared ls;
};

// Tile coordinates + 3 of a bin's anchor (past the tile for the last bin).
__device__ __forceinline__ int3 bin_anchor(int bin) {
    const int row = bin / kBinsPerRow;
    return make_int3(bin - row * kBinsPerRow, row % kRow, row / kRow);
}

// One 32-candidate word of the tile's 24 bit sets, lane l < 24 returning set l's
// word: columns, rows, planes covered by the lane's candidate, whose anchor is
// at r - 3.
template <int KW>
__device__ __forceinline__ unsigned cover_word(int3 r, const int dim[3], int lane) {
    unsigned mine = 0;
#pragma unroll
    for (int x = 0; x < kTile; ++x) {
        const unsigned vx = __ballot_sync(0xffffffffu, (unsigned)(x + 3 - r.x) < (unsigned)KW && x < dim[0]);
        const unsigned vy = __ballot_sync(0xffffffffu, (unsigned)(x + 3 - r.y) < (unsigned)KW && x < dim[1]);
        const unsigned vz = __ballot_sync(0xffffffffu, (unsigned)(x + 3 - r.z) < (unsigned)KW && x < dim[2]);
        if (lane == x) mine = vx;
        if (lane == kTile + x) mine = vy;
        if (lane == 2 * kTile + x) mine = vz;
    }
    return mine;
}

// a marker's spread source
__device__ __forceinline__ void load_source(const float *A, uint32_t m, float a[3]) {
    const float4 v = ((const float4 *)A)[m];
    a[0] = v.x, a[1] = v.y, a[2] = v.z;
}
__device__ __forceinline__ void load_source(const float2 *A, uint32_t m, float2 a[3]) {
    const float4 v = ((const float4 *)A)[2 * (size_t)m];
    a[0] = make_float2(v.x, v.y), a[1] = make_float2(v.z, v.w);
    a[2] = A[4 * (size_t)m + 2];
}

// Standalone spreading sums a tile's cells where the lists would be written: its
// lists are read once, so writing and reading them cost more than the sums (64
// spheres of 1800 markers, FP64: lists and gather 63 + 53 us, 84 us together).
template <typename T>
struct SpreadSum {
    const PS<T> *A;  // [M][4] sources
    T *f;            // null: write the lists
    DevGrid g;
    int lo[3];
};

// A tile's lists from its bit sets of nw words (set(i, w): columns, rows, planes
// for i from 0, 8, 16), by a CTA of NT threads.  The caller has zeroed ls.hist,
// ls.np and ls.len before a barrier.  The tile takes its share of the pair arrays
// from a cursor, so no scan of the candidates' pair counts is needed (5 to 16 us a
// call); where it lies changes no sum.
// With SUM every cell's sum is added to the field instead (a lane a cell, the
// pairs in the same order).
template <typename T, int NT, bool SUM, class Set, class First, class Mark>
__device__ __forceinline__ void build_lists(const Slots &sl, int cs, int nc, int nw, bool jagged,
                                            const PS<T> *__restrict__ wts, ListShared &ls, Set set, First first,
                                            Mark mark, const SpreadSum<T> &sp) {
    constexpr int C = kTileCells / NT;  // cells a thread, neighbours along x
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int t[C], r[C];
    {
        const int x = (C * tid) & 7, y = ((C * tid) >> 3) & 7, z = (C * tid) >> 6;
#pragma unroll
        for (int k = 0; k < C; ++k) t[k] = 0;
        for (int w = 0; w < nw; ++w) {
            const unsigned yz = set(kTile + y, w) & set(2 * kTile + z, w);
#pragma unroll
            for (int k = 0; k < C; ++k) t[k] += __popc(yz & set(x + k, w));
        }
    }
    // counting sort of the cells by list length
    auto bucket = [](int n) { return kLenBins - 1 - min(n, kLenBins - 1); };
#pragma unroll
    for (int k = 0; k < C; ++k) r[k] = t[k] > 0 ? atomicAdd(&ls.hist[bucket(t[k])], 1) : 0;
    if constexpr (!SUM) {
        int sum = 0;
#pragma unroll
        for (int k = 0; k < C; ++k) sum += t[k];
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0) atomicAdd(&ls.np, sum);
    }
    __syncthreads();
    if (!SUM && tid == 32) ls.base = atomicAdd(sl.pair_cursor, (unsigned)ls.np);
    if (warp == 0) {
        int h[kLenBins / 32], s = 0;
#pragma unroll
        for (int k = 0; k < kLenBins / 32; ++k) {
            h[k] = ls.hist[kLenBins / 32 * lane + k];
            s += h[k];
        }
        int inc = s;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        int run = inc - s;
#pragma unroll
        for (int k = 0; k < kLenBins / 32; ++k) {
            ls.hist[kLenBins / 32 * lane + k] = run;
            run += h[k];
        }
        if (lane == 31) ls.nb = inc;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < C; ++k)
        if (t[k] > 0) {
            const int q = ls.hist[bucket(t[k])] + r[k];
            ls.cell[q] = (uint16_t)(C * tid + k);
            ls.cnt[q] = (uint16_t)t[k];
        }
    __syncthreads();
    const int nb = ls.nb, ns = (nb + 31) >> 5;
    for (int s = warp; s < ns; s += NT / 32) {
        const int n = 32 * s + lane < nb ? ls.cnt[32 * s + lane] : 0;
        const int sum = __reduce_add_sync(0xffffffffu, n), len = __reduce_max_sync(0xffffffffu, n);
        if (lane == 0) ls.sum[s] = sum, ls.len[s] = (unsigned char)min(len, 255);
    }
    __syncthreads();
    if constexpr (SUM) {
        const DevGrid &g = sp.g;
        const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
        for (int s = warp; s < ns; s += NT / 32) {
            const int q = 32 * s + lane;
            const int c = q < nb ? ls.cell[q] : 0, n = q < nb ? ls.cnt[q] : 0;
            const int x = c & 7, y = (c >> 3) & 7, z = c >> 6, code = x + 4 * y + 16 * z;
            T *const f = sp.f +
                         ((long long)wrap_add(sp.lo[2], z, g.n[2]) * g.n[1] + wrap_add(sp.lo[1], y, g.n[1])) * g.n[0] +
                         wrap_add(sp.lo[0], x, g.n[0]);
            T v[3] = {T(0), T(0), T(0)};
            if (n > 0) v[0] = f[0], v[1] = f[N], v[2] = f[2 * N];
            const int rows = __reduce_max_sync(0xffffffffu, n);
            SumAcc<T> acc[3];
            int w = -1;
            unsigned m = 0;
            constexpr int kU = 4;  // rows whose loads are in flight together
            for (int k0 = 0; k0 < rows; k0 += kU) {
                PS<T> wx[kU], wy[kU], wz[kU], a[kU][3];
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (k0 + u < n) {
                        while (!m) {
                            ++w;
                            m = set(x, w) & set(kTile + y, w) & set(2 * kTile + z, w);
                        }
                        const int i = 32 * w + __ffs((int)m) - 1, oc = code - first(i);
                        m &= m - 1;
                        const uint32_t mk = mark(i);
                        const PS<T> *wm = wts + 12 * (size_t)mk;
                        wx[u] = wm[oc & 3];
                        wy[u] = wm[4 + ((oc >> 2) & 3)];
                        wz[u] = wm[8 + (oc >> 4)];
                        load_source(sp.A, mk, a[u]);
                    }
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (k0 + u < n) {
                        const PS<T> wt = pair_weight3(wx[u], wy[u], wz[u]);
                        acc[0].add(wt, a[u][0]);
                        acc[1].add(wt, a[u][1]);
                        acc[2].add(wt, a[u][2]);
                    }
            }
            if (n > 0) {
                f[0] = v[0] + acc[0].value();
                f[N] = v[1] + acc[1].value();
                f[2 * N] = v[2] + acc[2].value();
            }
        }
        return;
    }
    const uint32_t pb = ls.base;
    // (more pairs than the arrays hold only with a box wider than its grid, which is
    // reported: such a tile is left empty)
    const bool fits = (unsigned long long)pb + ls.np <= sl.pair_cap;
    uint32_t *const pairs = sl.pairs + pb;
    PS<T> *const pw = (PS<T> *)sl.pw + pb;
    int2 *const band = sl.band + pb;
    for (int s = fits ? warp : ns; s < ns; s += NT / 32) {
        const int q = 32 * s + lane;
        const int c = q < nb ? ls.cell[q] : 0, n = q < nb ? ls.cnt[q] : 0;
        int base = 0;
        for (int j = 0; j < s; ++j) base += ls.sum[j];
        int own = n;  // the list's first pair where lists are contiguous
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, own, o);
            if (lane >= o) own += v;
        }
        own += base - n;
        if (q < nb) band[q] = make_int2(c | (n << 16), jagged ? base : own);
        const int x = c & 7, y = (c >> 3) & 7, z = c >> 6, code = x + 4 * y + 16 * z;
        const int rows = __reduce_max_sync(0xffffffffu, n);
        int w = -1, off = base;
        unsigned m = 0;
        constexpr int kU = 4;  // rows whose loads are in flight together
        for (int k0 = 0; k0 < rows; k0 += kU) {
            int i[kU], pos[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const bool act = k0 + u < n;
                const unsigned a = __ballot_sync(0xffffffffu, act);
                pos[u] = act ? (jagged ? off + __popc(a & ((1u << lane) - 1u)) : own + k0 + u) : -1;
                off += __popc(a);
                i[u] = 0;
                if (act) {
                    while (!m) {
                        ++w;
                        m = set(x, w) & set(kTile + y, w) & set(2 * kTile + z, w);
                    }
                    i[u] = 32 * w + __ffs((int)m) - 1;
                    m &= m - 1;
                }
            }
            uint32_t mk[kU];
            int oc[kU];
            PS<T> wx[kU], wy[kU], wz[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                mk[u] = mark(i[u]);
                oc[u] = pos[u] >= 0 ? code - first(i[u]) : 0;
                const PS<T> *wm = wts + 12 * (size_t)mk[u];
                wx[u] = wm[oc[u] & 3];
                wy[u] = wm[4 + ((oc[u] >> 2) & 3)];
                wz[u] = wm[8 + (oc[u] >> 4)];
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (pos[u] >= 0) {
                    pairs[pos[u]] = jagged ? mk[u] : (uint32_t)i[u] | ((uint32_t)oc[u] << 16);
                    pw[pos[u]] = pair_weight3(wx[u], wy[u], wz[u]);
                }
        }
    }
    if (tid == 0) {
        sl.nband[cs] = fits ? nb : 0;
        sl.tinfo[cs] = make_int4((int)pb, fits ? ls.np : 0, fits ? nb : 0, nc);
        sl.slen[cs] = *(const uint4 *)ls.len;
    }
}

template <typename T, int KW, bool SUM>
__global__ void __launch_bounds__(kListThreads, SUM ? kSpreadCtas : kListCtas) k_tile_lists(
    CaseTab ct, int mode, int ncompact_cap, const int *__restrict__ ncompact_p, SlotGeom sg,
    const uint32_t *__restrict__ dense_of, const uint32_t *__restrict__ start, const uint64_t *__restrict__ anchor,
    const int *__restrict__ level, Slots sl, const PS<T> *__restrict__ wts, int jagged, int *__restrict__ big,
    int *__restrict__ nbig, SpreadSum<T> sp) {
    constexpr int kSetPitch = kListCand / 32 + 1;  // odd: no bank conflicts
    __shared__ __align__(16) unsigned long long s_keys[kListCand];  // or 32-bit keys
    __shared__ uint32_t s_mark[kListCand];
    __shared__ unsigned s_set[3 * kTile][kSetPitch];
    __shared__ short s_first[kListCand];
    __shared__ uint16_t s_rel[kListCand];  // anchor + 3, 4 bits an axis
    __shared__ uint32_t s_min[kListThreads / 32], s_max[kListThreads / 32];
    __shared__ __align__(16) ListShared s_ls;
    grid_dep_wait();
    const int ncompact = min(*ncompact_p, ncompact_cap);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kE = kListCand / kListThreads;  // candidates a thread
    for (int cs = blockIdx.x; cs < ncompact; cs += gridDim.x) {
        const uint32_t d = dense_of[cs];
        const uint32_t b = start[d];
        const int nc = (int)(start[d + 1] - b);
        if (nc > kListCand) {
            if (tid == 0) big[atomicAdd(nbig, 1)] = cs;
            continue;
        }
        int lo[3], dim[3], lev;
        const int cse = slot_geometry(ct, mode, sg, sl, level, d, b, lo, dim, lev);
        const DevGrid &g = ct.get(cse).g;
        uint32_t m[kE], mn = ~0u, mx = 0;
        int bin[kE];
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            const int i = tid + e * kListThreads;
            m[e] = 0;
            bin[e] = 0;
            if (i < nc) {
                m[e] = sl.cand[b + i];
                bin[e] = (int)(slot_key(g, anchor, m[e], lo) >> 32);
                mn = min(mn, m[e]), mx = max(mx, m[e]);
            }
        }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) s_min[warp] = mn, s_max[warp] = mx;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kListThreads / 32; ++w) mn = min(mn, s_min[w]), mx = max(mx, s_max[w]);
        // ranks: keys padded with maxima to a multiple of the vector loads
        int rank[kE];
#pragma unroll
        for (int e = 0; e < kE; ++e) rank[e] = 0;
        const int ne = (nc + kListThreads - 1) / kListThreads;
        if (mx - mn < (1u << kMarkBits)) {
            uint32_t *keys = (uint32_t *)s_keys, key[kE];
#pragma unroll
            for (int e = 0; e < kE; ++e) {
                const int i = tid + e * kListThreads;
                key[e] = i < nc ? ((uint32_t)bin[e] << kMarkBits) | (m[e] - mn) : ~0u;
                if (e < ne) keys[i] = key[e];
            }
            __syncthreads();
            for (int j = 0; j < nc; j += 4) {
                const uint4 q = *(const uint4 *)(keys + j);
#pragma unroll
                for (int e = 0; e < kE; ++e)
                    if (e < ne) rank[e] += (q.x < key[e]) + (q.y < key[e]) + (q.z < key[e]) + (q.w < key[e]);
            }
        } else {
            unsigned long long key[kE];
#pragma unroll
            for (int e = 0; e < kE; ++e) {
                const int i = tid + e * kListThreads;
                key[e] = i < nc ? ((unsigned long long)bin[e] << 32) | m[e] : ~0ull;
                if (e < ne) s_keys[i] = key[e];
            }
            __syncthreads();
            for (int j = 0; j < nc; ++j) {
                const unsigned long long q = s_keys[j];
#pragma unroll
                for (int e = 0; e < kE; ++e)
                    if (e < ne) rank[e] += q < key[e];
            }
        }
#pragma unroll
        for (int e = 0; e < kE; ++e)
            if (tid + e * kListThreads < nc) {
                const int3 q = bin_anchor(bin[e]);
                const int r = rank[e];
                s_mark[r] = m[e];
                if (!SUM) sl.cand[b + r] = m[e];
                s_rel[r] = (uint16_t)(q.x | (q.y << 4) | (q.z << 8));
                s_first[r] = (short)((q.x - 3) + 4 * (q.y - 3) + 16 * (q.z - 3));
            }
        __syncthreads();
        if (sl.bins)
            slot_bins(nc, cs, sl, tid, kListThreads, [&](int i) {
                const int q = s_rel[i];
                return ((q >> 8) * kRow + ((q >> 4) & 15)) * kBinsPerRow + (q & 15);
            });
        const int nw = (nc + 31) >> 5;
        for (int w = warp; w < nw; w += kListThreads / 32) {
            const int i = 32 * w + lane, q = i < nc ? s_rel[i] : 0xfff;  // past the tile
            const unsigned mine = cover_word<KW>(make_int3(q & 15, (q >> 4) & 15, q >> 8), dim, lane);
            if (lane < 3 * kTile) s_set[lane][w] = mine;
        }
        s_ls.hist[tid] = 0;
        if (tid == 0) s_ls.np = 0;
        if (tid < kSlices) s_ls.len[tid] = 0;
        __syncthreads();
        if (SUM) sp.lo[0] = lo[0], sp.lo[1] = lo[1], sp.lo[2] = lo[2], sp.g = g;
        build_lists<T, kListThreads, SUM>(sl, cs, nc, nw, jagged != 0, wts, s_ls,
                                          [&](int i, int w) { return s_set[i][w]; }, [&](int i) { return s_first[i]; },
                                          [&](int i) { return s_mark[i]; }, sp);
        if (!SUM && tid == 0) {
            sl.geo_lo[cs] = make_int4(lo[0], lo[1], lo[2], lev);
            sl.geo_dim[cs] = make_int4(dim[0], dim[1], dim[2], (int)b);
            sl.geo_case[cs] = cse;
        }
        __syncthreads();  // the next tile overwrites the shared lists
    }
}

// The tiles of more than kListCand candidates, one CTA each.
template <typename T, int KW, bool SUM>
__global__ void __launch_bounds__(kPairThreads) k_tile_lists_large(
    CaseTab ct, int mode, SlotGeom sg, const uint32_t *__restrict__ dense_of, const uint32_t *__restrict__ start,
    const uint64_t *__restrict__ anchor, const int *__restrict__ level, Slots sl, const PS<T> *__restrict__ wts,
    int jagged, const int *__restrict__ big, const int *__restrict__ nbig_p, DevStatus *st, SpreadSum<T> sp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_dep_wait();
    const int nbig = *nbig_p, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    CtaLists &sh = *(CtaLists *)smem_raw;
    {
        for (int q = blockIdx.x; q < nbig; q += gridDim.x) {
            const int cs = big[q];
            const uint32_t d = dense_of[cs];
            const uint32_t b = start[d];
            int nc = (int)(start[d + 1] - b);
            int lo[3], dim[3], lev;
            const int cse = slot_geometry(ct, mode, sg, sl, level, d, b, lo, dim, lev);
            const DevGrid &g = ct.get(cse).g;
            if (nc > kMaxCand) {
                // report, and leave an empty tile (no bins, no cells)
                if (tid == 0) raise_status(st, IB_ERR_UNSUPPORTED, nc);
                nc = 0;
                dim[0] = dim[1] = dim[2] = 0;
            }
            int np2 = 1;
            while (np2 < nc) np2 <<= 1;
            for (int i = tid; i < np2; i += kPairThreads)
                sh.keys[i] = i < nc ? slot_key(g, anchor, sl.cand[b + i], lo) : ~0ull;
            __syncthreads();
            for (int k = 2; k <= np2; k <<= 1)
                for (int j = k >> 1; j > 0; j >>= 1) {
                    for (int i = tid; i < np2; i += kPairThreads) {
                        const int ixj = i ^ j;
                        if (ixj > i) {
                            const unsigned long long x = sh.keys[i], y = sh.keys[ixj];
                            if ((x > y) == ((i & k) == 0)) {
                                sh.keys[i] = y;
                                sh.keys[ixj] = x;
                            }
                        }
                    }
                    __syncthreads();
                }
            if (sl.bins) slot_bins(nc, cs, sl, tid, kPairThreads, [&](int i) { return (int)(sh.keys[i] >> 32); });
            // sorted candidates and the bit sets, one word per warp and step
            const int nw = (nc + 31) >> 5;
            for (int w = warp; w < nw; w += kPairThreads / 32) {
                const int i = 32 * w + lane;
                int3 r = make_int3(15, 15, 15);
                if (i < nc) {
                    r = bin_anchor((int)(sh.keys[i] >> 32));
                    if (!SUM) sl.cand[b + i] = (uint32_t)(sh.keys[i] & 0xffffffffu);
                    sh.first[i] = (short)((r.x - 3) + 4 * (r.y - 3) + 16 * (r.z - 3));
                }
                const unsigned mine = cover_word<KW>(r, dim, lane);
                if (lane < 3 * kTile) sh.set[lane][w] = mine;
            }
            if (tid < kLenBins) sh.ls.hist[tid] = 0;
            if (tid == 0) sh.ls.np = 0;
            if (tid < kSlices) sh.ls.len[tid] = 0;
            __syncthreads();
            if (SUM) sp.lo[0] = lo[0], sp.lo[1] = lo[1], sp.lo[2] = lo[2], sp.g = g;
            build_lists<T, kPairThreads, SUM>(sl, cs, nc, nw, jagged != 0, wts, sh.ls,
                                              [&](int i, int w) { return sh.set[i][w]; },
                                              [&](int i) { return sh.first[i]; },
                                              [&](int i) { return (uint32_t)(sh.keys[i] & 0xffffffffu); }, sp);
            if (!SUM && tid == 0) {
                sl.geo_lo[cs] = make_int4(lo[0], lo[1], lo[2], lev);
                sl.geo_dim[cs] = make_int4(dim[0], dim[1], dim[2], (int)b);
                sl.geo_case[cs] = cse;
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// Spreading (ib_spread) with warp-aggregated atomics: one lane per marker,
// weights formed on the fly, no binning.
template <typename T, int KER>
__global__ void __launch_bounds__(256) k_spread_atomic(DevGrid g, int M, const double *__restrict__ X,
                                                       const double *__restrict__ F, const double *__restrict__ dV,
                                                       T *__restrict__ f, DevStatus *st) {
    constexpr int KW = Kernel<KER>::W;
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    const int lane = threadIdx.x & 31;
    const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
    // warp-uniform loop: every lane takes part in the matching
    for (long long base = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < M;
         base += nwarps * 32) {
        const long long l = base + lane;
        bool valid = l < M;
        double x[3] = {0, 0, 0}, fv[3] = {0, 0, 0}, dv = 0.0;
        if (valid) {
            x[0] = X[3 * l], x[1] = X[3 * l + 1], x[2] = X[3 * l + 2];
            fv[0] = F[3 * l], fv[1] = F[3 * l + 1], fv[2] = F[3 * l + 2];
            dv = dV[l];
            if (!(finite3(x) && finite3(fv) && isfinite(dv))) {
                raise_status(st, IB_ERR_NONFINITE, (int)l);
                valid = false;
            }
        }
        if (!valid) x[0] = g.org[0], x[1] = g.org[1], x[2] = g.org[2];
        PS<T> ws[12], A[3];
        int first[3];
        const uint64_t anc = marker_weights<T, KER>(g, x, ws, first);
        const double q = dv * g.inv_h3;
#pragma unroll
        for (int c = 0; c < 3; ++c) A[c] = to_store((T)(fv[c] * q));
        scatter_marker<T, KW>(f, (T *)nullptr, g, N, anc, ws, A, valid, 0.0);
    }
}

// ---------------------------------------------------------------------------
// grid barrier with a bounded wait
// ---------------------------------------------------------------------------
struct Barrier {
    unsigned int *count;
    unsigned int *gen;
};


// Sense-free generation barrier over all CTAs of a cooperative launch.  The
// waiting thread polls the generation word without sleeping (a sleep's wake-up
// latency dominated the phases) and gives up after kSpinCycles SM cycles,
// raising IB_ERR_TIMEOUT; every CTA then returns.

__device__ __forceinline__ bool grid_sync(Barrier b, DevStatus *st) {
    __syncthreads();
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        const unsigned int g0 = ld_acquire(b.gen);
        __threadfence();
        const unsigned int arrived = atomicAdd(b.count, 1u);
        int ok = 1;
        if (arrived == gridDim.x - 1) {
            atomicExch(b.count, 0u);
            __threadfence();
            atomicAdd(b.gen, 1u);
        } else {
            const long long t0 = clock64();
            while (ld_acquire(b.gen) == g0) {
                if (clock64() - t0 > kSpinCycles) {
                    raise_status(st, IB_ERR_TIMEOUT, (int)blockIdx.x);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        s_ok = ok && (*(volatile int *)&st->code != IB_ERR_TIMEOUT);
    }
    __syncthreads();
    return s_ok;
}

// ---------------------------------------------------------------------------
// persistent multidirect-forcing passes (cooperative launch)
// ---------------------------------------------------------------------------
constexpr int kInterpThreads = 256;  // level interpolation CTA

template <typename T>
struct PassArgs {
    CaseTab ct;        // cases: grid, u, accumulated force field (nullable)
    const int *part_of;  // [M] particle of each marker
    double *F;
    const double *dV;
    MarkerState<T> ms;
    Slots sl;
    const int *mperm;
    const int *lev_mbeg;
    const int2 *lev_slice;  // per wavefront, its slices' first entry and number
    const int4 *slices;     // (k_level_slices)
    const int *nlev;
    int Ns;
    int L0;  // first wavefront the persistent kernel processes
    int atomic;  // spread with warp-aggregated atomics instead of the tile gather
    double dt, inv_dt;  // inv_dt = 1 / dt, formed on the host
    Barrier bar;
    DevStatus *st;
};

// ---------------------------------------------------------------------------
// one wavefront pass as two ordinary kernels (the form CUDA-graph replay runs
// back to back): interpolation over the wavefront's markers, then a gather
// with one warp per slice of 32 cells, many warps per SM hiding latency.
//
// Every level kernel but the first of a call is launched as a programmatic
// dependent of the one before it: it starts while its predecessor finishes,
// loads what the predecessor does not write (marker weights, anchors, desired
// velocities, forces; the slice's record, field values and first pairs), then waits for the predecessor and reads what it wrote (the
// field for an interpolation, the spread sources for a gather).  Every CTA
// waits before it exits, so a level kernel completes only after its
// predecessor.  An interpolation lets its gather start right after its own
// wait (the gather's warps load theirs meanwhile); for FP32 fields a
// gather lets the next interpolation start only as its CTAs exit, so that
// interpolation's CTAs land on idle SMs (measured faster than an early start),
// and for FP64 fields once each of its CTAs has waited and reached a last slice.
// ---------------------------------------------------------------------------
template <typename T, int KER>
__global__ void __launch_bounds__(kInterpThreads) k_interp_level(PassArgs<T> a, int L) {
    constexpr int KW = Kernel<KER>::W;
    // all 81 loads of a Roma-kernel marker in flight at once for FP32 fields
    constexpr bool kAll = KW == 3 && sizeof(T) == 4;
    const int nl = *a.nlev;
    const int m0 = L < nl ? a.lev_mbeg[L] : 0, m1 = L < nl ? a.lev_mbeg[L + 1] : 0;
    const int stride = gridDim.x * blockDim.x;
    int i = m0 + blockIdx.x * blockDim.x + threadIdx.x;
    // one marker's data but the field (loaded before the wait for the first)
    int l = 0;
    uint64_t anc = 0;
    PS<T> w[12];
    PassMarker<T> pm;
    double F[3];
    auto load = [&]() {
        l = a.mperm[i];
        anc = a.ms.anchor[l];
        if (kAll)
#pragma unroll
            for (int k = 0; k < 12; ++k) w[k] = __ldg(a.ms.wts + 12 * (size_t)l + k);
        pm.load(a.ms, a.dV, a.ct.of_particle(a.part_of[l]).g.inv_h3, l);
#pragma unroll
        for (int c = 0; c < 3; ++c) F[c] = a.F[3 * l + c];
    };
    if (i < m1) load();
    grid_dep_wait();
    grid_dep_launch();
    for (bool first = true; i < m1; i += stride, first = false) {
        if (!first) load();
        const DevCase cd = a.ct.of_particle(a.part_of[l]);
        const DevGrid &g = cd.g;
        const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
        T U[3];
        // the field was written by the predecessor: plain loads
        // (weights from registers when every tap is unrolled, else from memory)
        interp_marker<T, KW, true, kAll>((const T *)cd.u, g, N, anc, kAll ? w : a.ms.wts + 12 * (size_t)l, U);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T e = pm.err(c, U[c]);
            a.F[3 * l + c] = PassMarker<T>::force(F[c], e, a.inv_dt);
            a.ms.A[4 * l + c] = pm.source(e);
        }
    }
}

// FP64 fields: one thread per marker component, three per marker.  Each sums
// its component's taps in the order of interp_marker (planes z, rows y,
// columns x; the same double-float products and additions), so the result
// is bitwise the one-thread form's; three times the threads hide the latency
// of the double-float chains and of the field loads.
constexpr bool kInterpSplit = true;  // FP64 level interpolation by component
constexpr bool kInterpSplitAll = true;  // every tap of a component in flight at once

template <int KW, bool ALL>
__device__ __forceinline__ double interp_component(const double *__restrict__ uc, const DevGrid &g, uint64_t anc,
                                                   const float2 *w) {
    int ix[KW], iy[KW], iz[KW];
    const int ax = anchor_x(anc), ay = anchor_y(anc), az = anchor_z(anc);
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        ix[k] = wrap_add(ax, k, g.n[0]);
        iy[k] = wrap_add(ay, k, g.n[1]);
        iz[k] = wrap_add(az, k, g.n[2]);
    }
    SumAcc<double> acc;
    auto plane = [&](int kz) {
        double v[KW][KW];
#pragma unroll
        for (int ky = 0; ky < KW; ++ky) {
            const long long row = ((long long)iz[kz] * g.n[1] + iy[ky]) * g.n[0];
#pragma unroll
            for (int kx = 0; kx < KW; ++kx) v[ky][kx] = uc[row + ix[kx]];
        }
#pragma unroll
        for (int ky = 0; ky < KW; ++ky) {
            const float2 wyz = df_mul(w[8 + kz], w[4 + ky]);
#pragma unroll
            for (int kx = 0; kx < KW; ++kx) acc.add(df_mul(wyz, w[kx]), df_split(v[ky][kx]));
        }
    };
    if (ALL) {
#pragma unroll
        for (int kz = 0; kz < KW; ++kz) plane(kz);
    } else {
#pragma unroll 1
        for (int kz = 0; kz < KW; ++kz) plane(kz);
    }
    return acc.value();
}

template <typename T, int KER>
__global__ void __launch_bounds__(kInterpThreads) k_interp_level_c3(PassArgs<T> a, int L) {
    static_assert(sizeof(T) == 8, "component split serves FP64 fields");
    constexpr int KW = Kernel<KER>::W;
    const int nl = *a.nlev;
    const int m0 = L < nl ? a.lev_mbeg[L] : 0, m1 = L < nl ? a.lev_mbeg[L + 1] : 0;
    const int n3 = 3 * (m1 - m0);
    const int stride = gridDim.x * blockDim.x;
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    // one item's data but the field (loaded before the wait for the first)
    int l = 0, c = 0;
    uint64_t anc = 0;
    float2 w[12];
    double ud = 0.0, q = 0.0, F = 0.0;
    auto load = [&]() {
        l = a.mperm[m0 + t / 3];
        c = t % 3;
        anc = a.ms.anchor[l];
#pragma unroll
        for (int k = 0; k < 12; ++k) w[k] = __ldg(a.ms.wts + 12 * (size_t)l + k);
        ud = __ldg(a.ms.Ud + 3 * l + c);
        q = a.dV[l] * a.ct.of_particle(a.part_of[l]).g.inv_h3;
        F = a.F[3 * l + c];
    };
    if (t < n3) load();
    grid_dep_wait();
    grid_dep_launch();
    for (bool first = true; t < n3; t += stride, first = false) {
        if (!first) load();
        const DevCase cd = a.ct.of_particle(a.part_of[l]);
        const DevGrid &g = cd.g;
        const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
        const double U = interp_component<KW, kInterpSplitAll>((const double *)cd.u + c * N, g, anc, w);
        const double e = ud - U;
        a.F[3 * l + c] = fma(e, a.inv_dt, F);
        a.ms.A[4 * l + c] = to_store(e * q);
    }
}

// The wavefront gather: one warp per slice of 32 band cells, a lane per cell,
// over the slices' jagged rows.  Pair words and weights come in coalesced rows
// straight from memory (they stay in L2 through a wavefront's passes), the
// sources from L2 and L1 (a marker's is read by the 27 cells of its stencil);
// no shared memory, no barrier, and kSliceRows rows in flight a warp.  A tile
// per CTA with its lists staged in shared memory spent most of its time in
// staging round trips and barriers: 17.0 us a launch on the 256^3 cluster in
// FP64 (50 on its first wavefront).
//
// Before the wait (nothing here is written by the interpolation): the slice's
// record and cells, the cells' field values and the first rows.  Each cell's
// pairs are added in ascending candidate order, as in the bin walk.
constexpr int kSliceThreads = 128;
template <typename T> constexpr int kSliceCtas = sizeof(T) == 4 ? 8 : 6;  // CTAs of an SM
constexpr int kSliceRows = 4;

template <typename T, class Wait>
__device__ __forceinline__ void gather_slice(const CaseTab &ct, int4 rec, const Slots &sl, const PS<T> *A, double inv_dt,
                                             Wait wait) {
    using S = PS<T>;
    constexpr int U = kSliceRows;
    const int lane = threadIdx.x & 31, q = 32 * rec.y + lane, cs = rec.x;
    const uint32_t pb = (uint32_t)rec.z;
    const bool has = q < rec.w;
    const int2 e = has ? sl.band[pb + q] : make_int2(0, 0);
    const int4 lo = sl.geo_lo[cs];
    const DevCase cd = ct.get(sl.geo_case[cs]);
    const DevGrid &g = cd.g;
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    T *const u = (T *)cd.u;
    const int cnt = e.x >> 16, cell = e.x & 0xffff;
    const long long c = ((long long)wrap_add(lo.z, cell >> 6, g.n[2]) * g.n[1] + wrap_add(lo.y, (cell >> 3) & 7, g.n[1])) *
                            g.n[0] +
                        wrap_add(lo.x, cell & 7, g.n[0]);
    T v[3] = {T(0), T(0), T(0)};
    if (has) v[0] = u[c], v[1] = u[N + c], v[2] = u[2 * N + c];
    const uint32_t *const pairs = sl.pairs + pb;
    const S *const pw = (const S *)sl.pw + pb;
    int off = __shfl_sync(0xffffffffu, e.y, 0);
    const int rows = __reduce_max_sync(0xffffffffu, cnt);
    uint32_t mk[U];
    S wt[U];
    auto load_rows = [&](int k0) {
#pragma unroll
        for (int r = 0; r < U; ++r) {
            const bool act = k0 + r < cnt;
            const unsigned a = __ballot_sync(0xffffffffu, act);
            const int pos = off + __popc(a & ((1u << lane) - 1u));
            off += __popc(a);
            mk[r] = act ? __ldg(pairs + pos) : 0u;
            wt[r] = act ? __ldg(pw + pos) : S();
        }
    };
    load_rows(0);
    wait();
    SumAcc<T> acc[3];
    for (int k0 = 0; k0 < rows; k0 += U) {
        S a[U][3], w[U];
#pragma unroll
        for (int r = 0; r < U; ++r) {
            w[r] = wt[r];
            a[r][0] = a[r][1] = a[r][2] = S();
            if (k0 + r < cnt) load_source(A, mk[r], a[r]);
        }
        if (k0 + U < rows) load_rows(k0 + U);
#pragma unroll
        for (int r = 0; r < U; ++r)
            if (k0 + r < cnt) {
                acc[0].add(w[r], a[r][0]);
                acc[1].add(w[r], a[r][1]);
                acc[2].add(w[r], a[r][2]);
            }
    }
    if (has) {
        T *const f_out = (T *)cd.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T s = acc[k].value();
            u[k * N + c] = v[k] + s;
            if (f_out) f_out[k * N + c] += (T)(s * inv_dt);
        }
    }
}

template <typename T, int KER>
__global__ void __launch_bounds__(kSliceThreads, kSliceCtas<T>) k_gather_level(PassArgs<T> a, int L) {
    const int nl = *a.nlev;
    const int2 ls = L < nl ? a.lev_slice[L] : make_int2(0, 0);
    const int step = gridDim.x * (kSliceThreads / 32);
    for (int j = blockIdx.x * (kSliceThreads / 32) + (threadIdx.x >> 5); j < ls.y; j += step) {
        // FP64 fields: at its last slice a warp lets the next interpolation be
        // scheduled, so its CTAs load their marker data while the last slices
        // sum (after the wait: that data includes the forces that the
        // interpolation before this kernel wrote)
        gather_slice<T>(a.ct, a.slices[ls.x + j], a.sl, a.ms.A, a.inv_dt, [&] {
            grid_dep_wait();
            if (sizeof(T) == 8 && j + step >= ls.y) grid_dep_launch();
        });
    }
    grid_dep_wait();  // every CTA waits before it exits
}

// The atomic form of a wavefront's spreading (ib_ctx_set_spread_mode):
// every marker of the wavefront adds S A to the field with warp-aggregated
// atomics.  Its position data are loaded before the wait; the sources after.
template <typename T, int KER>
__global__ void __launch_bounds__(256) k_scatter_level(PassArgs<T> a, int L) {
    constexpr int KW = Kernel<KER>::W;
    const int nl = *a.nlev;
    const int m0 = L < nl ? a.lev_mbeg[L] : 0, m1 = L < nl ? a.lev_mbeg[L + 1] : 0;
    const int lane = threadIdx.x & 31;
    const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
    bool waited = false;
    for (long long base = m0 + ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < m1;
         base += nwarps * 32) {
        const long long i = base + lane;
        const bool valid = i < m1;
        const int l = valid ? a.mperm[i] : a.mperm[m0];
        const uint64_t anc = a.ms.anchor[l];
        PS<T> w[12], A[3];
#pragma unroll
        for (int k = 0; k < 12; ++k) w[k] = __ldg(a.ms.wts + 12 * (size_t)l + k);
        const DevCase cd = a.ct.of_particle(a.part_of[l]);
        if (!waited) {
            grid_dep_wait();
            waited = true;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) A[c] = a.ms.A[4 * (size_t)l + c];
        const long long N = (long long)cd.g.n[0] * cd.g.n[1] * cd.g.n[2];
        scatter_marker<T, KW>((T *)cd.u, (T *)cd.f, cd.g, N, anc, w, A, valid, a.inv_dt);
    }
    if (!waited) grid_dep_wait();
}

template <typename T, int KER>
__global__ void __launch_bounds__(256) k_mdf_passes(PassArgs<T> a) {
    constexpr int KW = Kernel<KER>::W;
    const int nl = *a.nlev;
    const double inv_dt = a.inv_dt;
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const int gsz = gridDim.x * blockDim.x;
    for (int L = a.L0; L < nl; ++L) {
        const int m0 = a.lev_mbeg[L], m1 = a.lev_mbeg[L + 1];
        const int2 ls = a.atomic ? make_int2(0, 0) : a.lev_slice[L];
        for (int m = 0; m < a.Ns; ++m) {
            // interpolation phase: U = J u, F += (U^d - U)/dt, A = (U^d - U) dV / h^3
            for (int i = m0 + gtid; i < m1; i += gsz) {
                const int l = a.mperm[i];
                const DevCase cd = a.ct.of_particle(a.part_of[l]);
                const DevGrid &g = cd.g;
                const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
                T U[3];
                interp_marker<T, KW, true>((const T *)cd.u, g, N, a.ms.anchor[l], a.ms.wts + 12 * (size_t)l, U);
                PassMarker<T> pm;
                pm.load(a.ms, a.dV, g.inv_h3, l);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const T e = pm.err(c, U[c]);
                    a.F[3 * l + c] = PassMarker<T>::force(a.F[3 * l + c], e, inv_dt);
                    a.ms.A[4 * l + c] = pm.source(e);
                }
            }
            if (!grid_sync(a.bar, a.st)) return;
            if (a.atomic) {
                // atomic spreading of the wavefront's markers (warp-uniform loop)
                const int lane = threadIdx.x & 31;
                const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
                for (long long base = m0 + ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32;
                     base < m1; base += nwarps * 32) {
                    const long long i = base + lane;
                    const bool valid = i < m1;
                    const int l = valid ? a.mperm[i] : a.mperm[m0];
                    const DevCase cd = a.ct.of_particle(a.part_of[l]);
                    const long long N = (long long)cd.g.n[0] * cd.g.n[1] * cd.g.n[2];
                    PS<T> w[12], A[3];
#pragma unroll
                    for (int k = 0; k < 12; ++k) w[k] = a.ms.wts[12 * (size_t)l + k];
#pragma unroll
                    for (int c = 0; c < 3; ++c) A[c] = a.ms.A[4 * (size_t)l + c];
                    scatter_marker<T, KW>((T *)cd.u, (T *)cd.f, cd.g, N, a.ms.anchor[l], w, A, valid, inv_dt);
                }
            } else {
                // gather phase over the wavefront's slices
                for (int j = gtid >> 5; j < ls.y; j += gsz >> 5)
                    gather_slice<T>(a.ct, a.slices[ls.x + j], a.sl, a.ms.A, inv_dt, [] {});
            }
            if (!grid_sync(a.bar, a.st)) return;
        }
    }
    // non-finite result check of the forces (cheap, once)
    for (int l = gtid; l < a.lev_mbeg[nl]; l += gsz) {
        int m = a.mperm[l];
        double fv[3] = {a.F[3 * m], a.F[3 * m + 1], a.F[3 * m + 2]};
        if (!finite3(fv)) raise_status(a.st, IB_ERR_NONFINITE, m);
    }
}

// ---------------------------------------------------------------------------
// host helpers
// ---------------------------------------------------------------------------
static int grid_blocks(long long work, int threads, int sm) {
    long long b = (work + threads - 1) / threads;
    long long cap = (long long)sm * 8;
    if (b < 1) b = 1;
    return (int)(b < cap ? b : cap);
}

template <typename T>
static bool take_markers(Arena &ar, int M, MarkerState<T> &ms) {
    ms.anchor = ar.take<uint64_t>(M > 0 ? M : 1);
    ms.wts = ar.take<PS<T>>((size_t)12 * (M > 0 ? M : 1));
    ms.A = ar.take<PS<T>>((size_t)4 * (M > 0 ? M : 1));
    ms.Ud = sizeof(T) == 8 ? ar.take<double>((size_t)3 * (M > 0 ? M : 1)) : nullptr;
    ms.Ud32 = sizeof(T) == 4 ? ar.take<float>((size_t)8 * (M > 0 ? M : 1)) : nullptr;
    return ar.ok();
}

// A call's counters and cursors set in one launch: four memsets of a few words to
// a megabyte each were four more steps of the preparation's chain.
struct Fill {
    unsigned *p[4];
    unsigned n[4], value[4];  // 32-bit words
};
__global__ void __launch_bounds__(256) k_fill(Fill f) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
        for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < f.n[a]; i += gridDim.x * blockDim.x)
            f.p[a][i] = f.value[a];
}
static void launch_fill(ib_ctx *ctx, const Fill &f, cudaStream_t s) {
    unsigned most = 0;
    for (int a = 0; a < 4; ++a) most = f.n[a] > most ? f.n[a] : most;
    k_fill<<<grid_blocks(most, 256, ctx->sm_count), 256, 0, s>>>(f);
}

// Slot lists for `M` prepared markers over ndense dense slots, in two steps
// so that a call issues every memset before its kernel chain (the chain's
// kernels are programmatic dependents of one another; a memset in between
// would break it).
struct SlotScratch {
    size_t cand_cap;
    int ncompact_cap;
    int lb_tiles;                 // look-back tiles of the slot scan
    unsigned long long *lb_stat;  // [lb_tiles] tile words
    // [4] the scan's ticket, the cursors of the pairs and of the slices, the number
    // of large tiles
    unsigned int *words;
    int *big;                     // [ncompact_cap] large tiles
};

// Workspace of the slot lists, and the zeroing they need.
template <typename T, int KW>
static int slots_alloc(ib_ctx *ctx, Arena &ar, int M, int ndense, int mode, Slots &sl, SlotScratch &sc, cudaStream_t s,
                       bool with_pairs, bool with_bins) {
    const size_t per = mode == 0 ? 27 : 8;
    sc.cand_cap = (size_t)M * per + 1;
    sc.ncompact_cap = (int)((size_t)M * per < (size_t)ndense ? (size_t)M * per : (size_t)ndense);
    if (sc.ncompact_cap < 1) sc.ncompact_cap = 1;
    const int ncap = sc.ncompact_cap;
    sl.count = ar.take<uint32_t>(ndense);
    sl.start = ar.take<uint32_t>(ndense + 1);
    sl.cursor = ar.take<uint32_t>(ndense);
    sl.flag_scan = ar.take<uint32_t>(ndense + 1);
    sc.lb_tiles = ndense / kLbTile + 1;
    sc.lb_stat = ar.take<unsigned long long>(sc.lb_tiles);
    sc.words = ar.take<unsigned int>(4);
    sc.big = ar.take<int>(ncap);
    sl.dense_of = ar.take<uint32_t>(ncap);
    sl.cand = ar.take<uint32_t>(sc.cand_cap);
    // bin tables: only the particle-resident form walks them
    sl.bins = with_bins ? ar.take<uint16_t>((size_t)ncap * kBins) : nullptr;
    sl.geo_lo = ar.take<int4>(ncap);
    sl.geo_dim = ar.take<int4>(ncap);
    sl.geo_case = ar.take<int>(ncap);
    constexpr int KW3 = KW * KW * KW;
    if (with_pairs) {
        // every stencil cell of every marker is one pair: KW^3 M in total
        sl.pair_cursor = sc.words + 1;
        sl.pair_cap = (unsigned long long)KW3 * M;
        sl.band = ar.take<int2>((size_t)KW3 * M);
        sl.pairs = ar.take<uint32_t>((size_t)KW3 * M);
        sl.pw = ar.take<PS<T>>((size_t)KW3 * M);
        sl.nband = ar.take<int>(ncap);
        sl.tinfo = ar.take<int4>(ncap);
        sl.slen = ar.take<uint4>(ncap);
    } else {
        sl.pair_cursor = nullptr;
        sl.pair_cap = 0;
        sl.band = nullptr;
        sl.pairs = nullptr;
        sl.nband = nullptr;
        sl.tinfo = nullptr;
        sl.slen = nullptr;
        sl.pw = nullptr;
    }
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    launch_fill(ctx, Fill{{sl.count, sl.cursor, (unsigned *)sc.lb_stat, sc.words},
                          {(unsigned)ndense, (unsigned)ndense, 2u * (unsigned)sc.lb_tiles, 4u}, {0, 0, 0, 0}}, s);
    return IB_OK;
}

// The kernel chain: count, scan and compact, fill, sort and per-cell lists -- or,
// given a field to spread into (sp.f), the cells' sums.
template <typename T, int KW>
static int slots_build(ib_ctx *ctx, const CaseTab &ct, int M, int ndense, SlotGeom sg, const uint64_t *anchor,
                       const PS<T> *wts, const int *level, Slots &sl, const SlotScratch &sc, int *&ncompact_dev,
                       cudaStream_t s, bool jagged, bool pdl_first = true, SpreadSum<T> sp = {}) {
    const int nb = grid_blocks(M, 256, ctx->sm_count);
    launch_dep(pdl_first, k_slot_count<KW>, dim3(nb), dim3(256), 0, s, ct, M, sg, anchor, sl.count);
    launch_pdl(k_slot_scan, dim3(sc.lb_tiles), dim3(kLbThreads), 0, s, (const uint32_t *)sl.count, ndense,
               sl.start, sl.flag_scan, sl.dense_of, sc.lb_stat, sc.words, ctx->status);
    launch_pdl(k_slot_fill<KW>, dim3(nb), dim3(256), 0, s, ct, M, sg, anchor, (const uint32_t *)sl.start,
               sl.cursor, sl.cand);
    ncompact_dev = (int *)(sl.flag_scan + ndense);
    auto lists = [&](auto small, auto large, int ctas) {
        launch_pdl(small, dim3(ctx->sm_count * ctas), dim3(kListThreads), 0, s, ct, sg.mode, sc.ncompact_cap,
                   (const int *)ncompact_dev, sg, (const uint32_t *)sl.dense_of, (const uint32_t *)sl.start, anchor,
                   level, sl, wts, jagged ? 1 : 0, sc.big, (int *)sc.words + 3, sp);
        resident_ctas(ctx, (const void *)large, kPairThreads, sizeof(CtaLists));  // (its shared memory limit)
        launch_pdl(large, dim3(ctx->sm_count), dim3(kPairThreads), sizeof(CtaLists), s, ct, sg.mode, sg,
                   (const uint32_t *)sl.dense_of, (const uint32_t *)sl.start, anchor, level, sl, wts, jagged ? 1 : 0,
                   (const int *)sc.big, (const int *)sc.words + 3, ctx->status, sp);
    };
    if (sp.f) lists(k_tile_lists<T, KW, true>, k_tile_lists_large<T, KW, true>, kSpreadCtas);
    else lists(k_tile_lists<T, KW, false>, k_tile_lists_large<T, KW, false>, kListCtas);
    return check_launch("slot lists");
}

template <typename T, int KER>
static int run_interpolate(ib_ctx *ctx, const DevGrid &g, const void *u, int M, const double *X,
                           double *U, cudaStream_t s) {
    int nb = grid_blocks(M, 256, ctx->sm_count);
    PhaseTimer tm(ctx, IB_PHASE_INTERP, s);
    k_interpolate<T, KER><<<nb, 256, 0, s>>>(g, (const T *)u, M, X, U, ctx->status);
    return check_launch("ib_interpolate");
}

template <typename T, int KER>
static int run_spread(ib_ctx *ctx, const ib_grid *grid, int M, const double *X, const double *F,
                      const double *dV, void *f, cudaStream_t s) {
    constexpr int KW = Kernel<KER>::W;
    if (ctx->spread_mode == IB_SPREAD_ATOMIC) {
        PhaseTimer tm(ctx, IB_PHASE_SPREAD, s);
        const DevGrid g = make_dev_grid(grid);
        k_spread_atomic<T, KER><<<grid_blocks(M, 256, ctx->sm_count), 256, 0, s>>>(g, M, X, F, dV, (T *)f,
                                                                                 ctx->status);
        return check_launch("ib_spread");
    }
    Arena ar(ctx);
    MarkerState<T> ms;
    take_markers<T>(ar, M, ms);
    const CaseTab ct = single_case(grid, f, nullptr, 0);  // spread into the case's u slot
    const DevGrid &g = ct.one.g;
    SlotGeom sg{};
    sg.mode = 0;
    const long long ndense = ct.ntiles;
    if (ndense > (1LL << 30)) return set_error(IB_ERR_UNSUPPORTED, "grid has too many tiles");
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    int nb = grid_blocks(M, 256, ctx->sm_count);
    Slots sl;
    SlotScratch sc;
    int *ncompact = nullptr;
    int rc = slots_alloc<T, KW>(ctx, ar, M, (int)ndense, sg.mode, sl, sc, s, false, false);
    if (rc) return rc;
    PhaseTimer tm(ctx, IB_PHASE_SPREAD, s);
    k_prep_spread<T, KER><<<nb, 256, 0, s>>>(g, M, X, F, dV, ms, ctx->status);
    rc = slots_build<T, KW>(ctx, ct, M, (int)ndense, sg, ms.anchor, (const PS<T> *)ms.wts, nullptr, sl, sc, ncompact, s,
                            true, true, SpreadSum<T>{ms.A, (T *)f});
    if (rc) return rc;
    return check_launch("ib_spread");
}

template <typename T, int KER>
static int run_mdf(ib_ctx *ctx, Arena &ar, const CaseTab &ct, const ib_particles *pp, const ib_markers *mk,
                   int Ns, double dt, int order, double *F_out, cudaStream_t s) {
    constexpr int KW = Kernel<KER>::W;
    int P = pp->P, M = mk->M;
    MarkerState<T> ms;
    take_markers<T>(ar, M, ms);
    double *rho = ar.take<double>(P);
    int4 *box_lo = ar.take<int4>(P);
    int4 *box_dim = ar.take<int4>(P);
    int *part_of = ar.take<int>(M > 0 ? M : 1);
    PrepScratch prep_ps;
    prep_ps.lo = ar.take<int>((size_t)3 * P);
    prep_ps.hi = ar.take<int>((size_t)3 * P);
    prep_ps.done = ar.take<unsigned int>(P);
    LevelOut lo;
    lo.level = ar.take<int>(P);
    lo.rank = ar.take<int>(P);
    lo.mbase = ar.take<int>(P);
    lo.lev_pbeg = ar.take<int>(P + 1);
    lo.lev_mbeg = ar.take<int>(P + 1);
    lo.nlev = ar.take<int>(1);
    int *lev_work = ar.take<int>(P + 1);  // the particle of each rank
    int *lev_cur = ar.take<int>(P + 1);
    int *nbr_cnt = ar.take<int>(P);
    int *nbr = ar.take<int>((size_t)P * kMaxNbr);
    int *mperm = ar.take<int>(M > 0 ? M : 1);
    unsigned int *sched = ar.take<unsigned int>(P + 1);  // done counters + ticket
    Barrier bar;
    bar.count = ar.take<unsigned int>(2);
    bar.gen = bar.count + 1;
    SlotGeom sg{};
    sg.mode = order == IB_ORDER_SEQUENTIAL ? 1 : 0;
    const long long ndense = sg.mode == 0 ? ct.ntiles : (long long)P * kLocalSlots;
    if (ndense > (1LL << 30)) return set_error(IB_ERR_UNSUPPORTED, "too many tiles");
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    // the particle-resident and particle-group forms serve FP32 fields; FP64
    // fields always run the wavefront form (double-float pass sums)
    const int pass_kernels = sizeof(T) == 4 ? ctx->pass_kernels : IB_PASSES_WAVEFRONT;
    const bool resident = order == IB_ORDER_SEQUENTIAL && pass_kernels == IB_PASSES_RESIDENT;
    // atomic spreading (wavefront form): no tile lists at all
    const bool wavefront = order == IB_ORDER_SIMULTANEOUS || pass_kernels == IB_PASSES_AUTO ||
                           pass_kernels == IB_PASSES_WAVEFRONT;
    const bool atomic = wavefront && ctx->spread_mode == IB_SPREAD_ATOMIC;
    Slots sl{};
    SlotScratch sc{};
    int rc = IB_OK;
    int2 *lev_slice = nullptr;
    int4 *slices = nullptr;
    if (!atomic) {
        rc = slots_alloc<T, KW>(ctx, ar, M, (int)ndense, sg.mode, sl, sc, s, true, resident);
        if (rc) return rc;
        lev_slice = ar.take<int2>(P + 1);
        // a tile of p pairs has at most p / 32 + 1 slices
        slices = ar.take<int4>((size_t)KW * KW * KW * M / 32 + sc.ncompact_cap + 1);
    }
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    PassArgs<T> a;
    a.ct = ct;
    a.part_of = part_of;
    a.F = F_out;
    a.dV = mk->dV;
    a.ms = ms;
    a.sl = sl;
    a.mperm = mperm;
    a.lev_mbeg = lo.lev_mbeg;
    a.lev_slice = lev_slice;
    a.slices = slices;
    a.nlev = lo.nlev;
    a.Ns = Ns;
    a.dt = dt;
    a.inv_dt = 1.0 / dt;
    a.bar = bar;
    a.st = ctx->status;
    a.atomic = atomic ? 1 : 0;
    // wavefronts enqueued as separate kernels: the count the last call on this
    // context copied to a pinned host word (read without synchronising: an
    // aligned 4-byte word is either the old or the new count; a short count
    // only leaves more wavefronts to the persistent kernel)
    ctx->nlev_hint = *(volatile int *)ctx->h_nlev;
    const int Lenq = ctx->nlev_hint < P ? ctx->nlev_hint : P;
    a.L0 = Lenq;
    // the level kernels' launch shapes; the first interpolation runs on the
    // context's second stream beside the slot-list kernels (it reads only the
    // field and the prepared markers), and the first gather joins it
    const bool level_path = !(sizeof(T) == 4 && order == IB_ORDER_SEQUENTIAL &&
                              (pass_kernels == IB_PASSES_RESIDENT || pass_kernels == IB_PASSES_GROUPS));
    const bool fork = level_path && Lenq >= 1;
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t ci = {};
    ci.gridDim = dim3(sizeof(T) == 8 && kInterpSplit ? grid_blocks(3LL * M, kInterpThreads, ctx->sm_count)
                                                     : grid_blocks(M, kInterpThreads, ctx->sm_count));
    ci.blockDim = dim3(kInterpThreads);
    ci.stream = s;
    ci.attrs = pdl;
    auto launch_interp = [&](int L, cudaStream_t st, bool dep) {
        ci.stream = st;
        ci.numAttrs = dep ? 1 : 0;
        if constexpr (sizeof(T) == 8 && kInterpSplit)
            cudaLaunchKernelEx(&ci, k_interp_level_c3<T, KER>, a, L);
        else
            cudaLaunchKernelEx(&ci, k_interp_level<T, KER>, a, L);
        ci.stream = s;
    };
    PhaseTimer tprep(ctx, IB_PHASE_MDF_PREP, s);
    // the marker radii, conflict lists, levels and level-major marker order
    // on the second stream, beside the marker preparation (after everything
    // already enqueued on the call's stream, whose earlier work may still use
    // this workspace)
    cudaStream_t fs = ctx->fork_stream;
    cudaEventRecord(ctx->fork_ev[0], s);
    cudaStreamWaitEvent(fs, ctx->fork_ev[0], 0);
    k_marker_radius<<<P, kRadiusThreads, 0, fs>>>(P, pp->Xr, pp->Ur, pp->Wr, pp->marker_offset, mk->R, mk->dV, rho);
    if (order == IB_ORDER_SEQUENTIAL)
        launch_pdl(k_conflicts, dim3(grid_blocks(32 * P, 256, ctx->sm_count)), dim3(256), 0, fs, ct, P, KW,
                   (const double *)pp->Xr, (const double *)rho, nbr_cnt, nbr);
    resident_ctas(ctx, (const void *)k_levels, kLevThreads, kLevSmem);  // (its shared memory limit)
    launch_pdl(k_levels, dim3(1), dim3(kLevThreads), kLevSmem, fs, ct, P, order, KW, (const double *)pp->Xr,
               (const double *)rho, (const int *)pp->marker_offset, (const int *)nbr_cnt, (const int *)nbr, lo,
               lev_work, lev_cur);
    launch_pdl(k_marker_order, dim3(P < ctx->sm_count * 4 ? P : ctx->sm_count * 4), dim3(256), 0, fs, P,
               (const int *)pp->marker_offset, (const int *)lo.mbase, mperm);
    cudaEventRecord(ctx->fork_ev[3], fs);
    // (box bounds far above and far below any cell)
    launch_fill(ctx, Fill{{bar.count, (unsigned *)prep_ps.lo, (unsigned *)prep_ps.hi, prep_ps.done},
                          {2u, 3u * (unsigned)P, 3u * (unsigned)P, (unsigned)P},
                          {0u, 0x7f7f7f7fu, 0x80808080u, 0u}}, s);
    k_prep_particles<T, KER><<<P * kPrepSplit, 256, 0, s>>>(ct, P, pp->Xr, pp->Ur, pp->Wr, pp->marker_offset, mk->R,
                                                 mk->dV, ms, F_out, box_lo, box_dim, part_of, prep_ps,
                                                 ctx->status);
    // the first interpolation (second stream) needs the prepared markers and
    // the marker order; the slot lists (this stream) need the levels' ranks
    cudaEventRecord(ctx->fork_ev[2], s);
    if (fork) {
        cudaStreamWaitEvent(fs, ctx->fork_ev[2], 0);
        if (ctx->field_wait) cudaStreamWaitEvent(fs, (cudaEvent_t)ctx->field_wait, 0);
        launch_interp(0, fs, false);
        cudaEventRecord(ctx->fork_ev[1], fs);
    }
    cudaStreamWaitEvent(s, ctx->fork_ev[3], 0);
    sg.part_of = part_of;
    sg.rank = lo.rank;
    sg.box_lo = box_lo;
    sg.box_dim = box_dim;
    int *ncompact = nullptr;
    if (!atomic) {
        rc = slots_build<T, KW>(ctx, ct, M, (int)ndense, sg, ms.anchor, (const PS<T> *)ms.wts, lo.level, sl, sc,
                                ncompact, s, level_path, false);
        if (rc) return rc;
        a.sl = sl;
    }
    if constexpr (sizeof(T) == 4) {
    if (order == IB_ORDER_SEQUENTIAL &&
        (pass_kernels == IB_PASSES_RESIDENT || pass_kernels == IB_PASSES_GROUPS)) {
        const bool groups = pass_kernels == IB_PASSES_GROUPS;
        const int ngroups = groups ? mdf_groups_count<T, KER>(ctx) : 0;
        if (groups && ngroups < 1) return set_error(IB_ERR_CUDA, "group kernel: no resident group");
        unsigned int *gwords = groups ? ar.take<unsigned int>((size_t)4 * ngroups) : nullptr;
        if (!ar.ok()) return oom_error(ar.used, ar.cap);
        // particle-resident passes: one cluster per particle, scheduled by rank
        ResidentArgs<T> ra;
        ra.ct = ct;
        ra.F = F_out;
        ra.dV = mk->dV;
        ra.ms = ms;
        ra.sl = sl;
        ra.mperm = mperm;
        ra.mbase = lo.mbase;
        ra.moff = pp->marker_offset;
        ra.by_rank = lev_work;  // k_levels leaves the particle of each rank there
        ra.rank = lo.rank;
        ra.level = lo.level;
        ra.box_lo = box_lo;
        ra.nbr_cnt = nbr_cnt;
        ra.nbr = nbr;
        ra.done = sched;
        ra.ticket = sched + P;
        ra.gwords = gwords;
        ra.P = P;
        ra.Ns = Ns;
        ra.dt = dt;
        ra.inv_dt = 1.0 / dt;
        ra.st = ctx->status;
        cudaMemsetAsync(sched, 0, sizeof(unsigned int) * (P + 1), s);
        if (groups) cudaMemsetAsync(gwords, 0, sizeof(unsigned int) * 4 * ngroups, s);
        tprep.stop();
        if (ctx->field_wait) cudaStreamWaitEvent(s, (cudaEvent_t)ctx->field_wait, 0);
        PhaseTimer tpass(ctx, IB_PHASE_MDF_PASSES, s);
        rc = groups ? launch_mdf_groups<T, KER>(ctx, ra, s) : launch_mdf_resident<T, KER>(ctx, ra, s);
        if (rc) return rc;
        tpass.stop();
        return check_launch("ib_multidirect_forcing");
    }
    }
    if (!atomic) {
        launch_pdl(k_level_slices, dim3(P < 64 ? P : 64), dim3(kSliceOrderThreads), 0, s, sg.mode,
                   (const int *)lo.nlev, (const int *)lo.lev_pbeg, (int)ndense, sl, sc.words + 2, lev_slice, slices);
    }
    tprep.stop();
    // (the field is first read and written by the pass kernels below)
    if (ctx->field_wait) cudaStreamWaitEvent(s, (cudaEvent_t)ctx->field_wait, 0);
    // one timed phase: the wavefront kernels and the persistent remainder
    PhaseTimer tpass(ctx, IB_PHASE_MDF_PASSES, s);
    {
        // one resident wave of gather CTAs (grid-stride over the wavefront's slices)
        int gper = kSliceCtas<T>;
        if (ctx->gather_ctas > 0 && ctx->gather_ctas < gper) gper = ctx->gather_ctas;
        // every level kernel after the first is a programmatic dependent of
        // the one before it (see k_interp_level); the first gather instead
        // waits for the interpolation on the second stream
        cudaLaunchConfig_t cg = {};
        cg.gridDim = dim3(ctx->sm_count * gper);
        cg.blockDim = dim3(kSliceThreads);
        cg.stream = s;
        cg.attrs = pdl;
        // the atomic form: one lane per marker of the largest wavefront at most
        cudaLaunchConfig_t cs = cg;
        cs.gridDim = dim3(grid_blocks(M, 256, ctx->sm_count));
        cs.blockDim = dim3(256);
        if (fork) cudaStreamWaitEvent(s, ctx->fork_ev[1], 0);
        for (int L = 0; L < Lenq; ++L)
            for (int m = 0; m < Ns; ++m) {
                const bool first = L == 0 && m == 0;
                if (!first || !fork) {
                    PhaseTimer ti(ctx, IB_PHASE_MDF_INTERP, s);
                    launch_interp(L, s, !first);
                }
                PhaseTimer tg(ctx, IB_PHASE_MDF_GATHER, s);
                cg.numAttrs = cs.numAttrs = first && fork ? 0 : 1;
                if (atomic)
                    cudaLaunchKernelEx(&cs, k_scatter_level<T, KER>, a, L);
                else
                    cudaLaunchKernelEx(&cg, k_gather_level<T, KER>, a, L);
            }
    }
    const int per_sm = resident_ctas(ctx, (const void *)k_mdf_passes<T, KER>, 256, 0);
    if (per_sm < 1) return set_error(IB_ERR_CUDA, "mdf kernel cannot be resident");
    int nblocks = per_sm * ctx->sm_count;
    void *args[] = {&a};
    cudaError_t e =
        cudaLaunchCooperativeKernel((const void *)k_mdf_passes<T, KER>, nblocks, 256, args, 0, s);
    if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "mdf launch: %s", cudaGetErrorString(e));
    tpass.stop();
    cudaMemcpyAsync(ctx->h_nlev, lo.nlev, sizeof(int), cudaMemcpyDeviceToHost, s);
    return check_launch("ib_multidirect_forcing");
}

}  // namespace gbib

using namespace gbib;

#define DISPATCH(prec, delta, FN, ...)                                                            \
    ((prec) == IB_F64 ? ((delta) == IB_DELTA_ROMA3 ? FN<double, IB_DELTA_ROMA3>(__VA_ARGS__)      \
                                                   : FN<double, IB_DELTA_PESKIN4>(__VA_ARGS__))   \
                      : ((delta) == IB_DELTA_ROMA3 ? FN<float, IB_DELTA_ROMA3>(__VA_ARGS__)       \
                                                   : FN<float, IB_DELTA_PESKIN4>(__VA_ARGS__)))

extern "C" {

int ib_interpolate(ib_ctx *ctx, const ib_grid *grid, const void *u, int M, const double *X, int delta,
                   double *U, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (delta != IB_DELTA_ROMA3 && delta != IB_DELTA_PESKIN4) return set_error(IB_ERR_INVALID, "bad delta");
    if (M < 0) return set_error(IB_ERR_INVALID, "M < 0");
    if (M == 0) return IB_OK;
    if (!u || !X || !U) return set_error(IB_ERR_INVALID, "NULL array");
    DevGrid g = make_dev_grid(grid);
    return DISPATCH(grid->prec, delta, run_interpolate, ctx, g, u, M, X, U, (cudaStream_t)stream);
}

int ib_spread(ib_ctx *ctx, const ib_grid *grid, int M, const double *X, const double *F, const double *dV,
              int delta, void *f, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (delta != IB_DELTA_ROMA3 && delta != IB_DELTA_PESKIN4) return set_error(IB_ERR_INVALID, "bad delta");
    if (M < 0) return set_error(IB_ERR_INVALID, "M < 0");
    if (M == 0) return IB_OK;
    if (!X || !F || !dV || !f) return set_error(IB_ERR_INVALID, "NULL array");
    return DISPATCH(grid->prec, delta, run_spread, ctx, grid, M, X, F, dV, f, (cudaStream_t)stream);
}

// Arguments shared by the single-case and batch forms; 1 = nothing to do.
static int check_mdf_args(ib_ctx *ctx, const ib_particles *parts, const ib_markers *marks, int Ns, double dt,
                          int delta, int order, const double *F_out) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    if (!parts || !marks) return set_error(IB_ERR_INVALID, "particles/markers NULL");
    if (delta != IB_DELTA_ROMA3 && delta != IB_DELTA_PESKIN4) return set_error(IB_ERR_INVALID, "bad delta");
    if (order != IB_ORDER_SEQUENTIAL && order != IB_ORDER_SIMULTANEOUS)
        return set_error(IB_ERR_INVALID, "bad order");
    if (Ns < 1) return set_error(IB_ERR_INVALID, "Ns must be >= 1");
    if (!(dt > 0.0) || !isfinite(dt)) return set_error(IB_ERR_INVALID, "dt must be finite and > 0");
    if (parts->P < 0 || marks->M < 0) return set_error(IB_ERR_INVALID, "negative P or M");
    if (parts->P == 0 || marks->M == 0) return 1;
    if (!parts->Xr || !parts->Ur || !parts->Wr || !parts->marker_offset || !marks->R || !marks->dV || !F_out)
        return set_error(IB_ERR_INVALID, "NULL array");
    return IB_OK;
}

int ib_multidirect_forcing(ib_ctx *ctx, const ib_grid *grid, void *u, const ib_particles *parts,
                           const ib_markers *marks, int Ns, double dt, int delta, int order, double *F_out,
                           void *f_out, void *stream) {
    int rc = check_mdf_args(ctx, parts, marks, Ns, dt, delta, order, F_out);
    if (rc) return rc == 1 ? IB_OK : rc;
    rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (!u) return set_error(IB_ERR_INVALID, "NULL array");
    const CaseTab ct = single_case(grid, u, f_out, parts->P);
    Arena ar(ctx);
    return DISPATCH(grid->prec, delta, run_mdf, ctx, ar, ct, parts, marks, Ns, dt, order, F_out,
                    (cudaStream_t)stream);
}

int ib_batch_table_multidirect_forcing(ib_ctx *ctx, const ib_batch_table *table, const ib_particles *parts,
                                       const ib_markers *marks, int Ns, double dt, int delta, int order,
                                       double *F_out, void *stream) {
    int rc = check_mdf_args(ctx, parts, marks, Ns, dt, delta, order, F_out);
    if (rc) return rc == 1 ? IB_OK : rc;
    CaseTab ct;
    rc = table_cases(table, parts->P, ct);
    if (rc) return rc;
    Arena ar(ctx);
    return DISPATCH(table->prec, delta, run_mdf, ctx, ar, ct, parts, marks, Ns, dt, order, F_out,
                    (cudaStream_t)stream);
}

int ib_batch_multidirect_forcing(ib_ctx *ctx, int ncases, const ib_case *cases, const ib_particles *parts,
                                 const ib_markers *marks, int Ns, double dt, int delta, int order, double *F_out,
                                 void *stream) {
    int rc = check_mdf_args(ctx, parts, marks, Ns, dt, delta, order, F_out);
    if (rc) return rc == 1 ? IB_OK : rc;
    for (int c = 0; c < ncases && cases; ++c)
        if (!cases[c].u) return set_error(IB_ERR_INVALID, "case %d: NULL field", c);
    Arena ar(ctx);
    CaseTab ct;
    rc = build_case_table(ctx, ar, ncases, cases, parts->P, 1, ct, (cudaStream_t)stream);
    if (rc) return rc;
    return DISPATCH(cases[0].grid.prec, delta, run_mdf, ctx, ar, ct, parts, marks, Ns, dt, order, F_out,
                    (cudaStream_t)stream);
}

}  // extern "C"
