// Per-particle reductions and updates around Algorithm 1 (arXiv 2408.14140):
//   * PVF volume integrals (Sec. 4.1, Eqs. level-set function / Heaviside;
//     the flow-unsteadiness terms of Eqs. particle1/particle2),
//   * marker force and torque (first terms of Eqs. particle1/particle2),
//   * repulsive-potential collision (Eq. DKT_model) + Newton-Euler update
//     (Eqs. particle1, particle2) + centroid update (Eq. pr2).
// All sums run in a fixed order (per-thread partials, then fixed warp, CTA
// and cross-CTA orders), so results are bitwise reproducible.  The volume
// integrals' per-cell sums are double-float (FP32 pipes, about 44 significant
// bits) in both field precisions; the force, torque, collision and update
// arithmetic is FP64.
#include <climits>
#include <mutex>
#include <new>

#include "df.cuh"
#include "gbib_internal.cuh"

namespace gbib {

constexpr double kPi = 3.14159265358979323846;

// Fixed-order sum of NV doubles over a CTA of NT threads (NT / 32 >= NV
// warps); result valid in thread 0.  The values go through shared memory and
// warp k sums quantity k (each lane NT / 32 entries, then a shuffle tree):
// NV (NT / 32 + 5) FP64 warp instructions, against NV * 5 per warp for a
// shuffle tree in every warp -- FP64 issue is scarce on this part.
template <int NV, int NT>
__device__ __forceinline__ void block_sum(double v[NV]) {
    static_assert(NT / 32 >= NV, "one warp per quantity");
    __shared__ double red[NV][NT];
#pragma unroll
    for (int k = 0; k < NV; ++k) red[k][threadIdx.x] = v[k];
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < NV) {
        double x = 0.0;
#pragma unroll
        for (int m = 0; m < NT / 32; ++m) x += red[wid][lane + 32 * m];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[wid][0] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = red[k][0];
}

// ---------------------------------------------------------------------------
// volume integrals.  Grid = P * nsplit CTAs; CTA (p, s) walks a slab of
// cell planes of particle p's box.  Cells whose centre lies deeper than
// R - 0.8661 h have all corners inside (alpha = 1) and are summed by columns;
// those within R + 0.8661 h form alpha from their eight corner values, the level
// set phi = |x - X_r|/R - 1, evaluated once per node (only for nodes within
// 1.75 h of the surface: the corners of every such cell) into two rolling node
// planes in shared memory.  The last CTA of a particle (completion counter)
// adds the nsplit partial sums in slab order.
// ---------------------------------------------------------------------------
constexpr int kVolSplit = 8;       // CTAs per particle of the allocation-free entry point
constexpr int kVolMaxSplit = 32;
constexpr int kVolThreads = 256;   // 8 warps
constexpr int kVolMaxBox = 40;     // cells per axis of one particle's box (tabulated path)
constexpr int kVolAx = kVolMaxBox + 1;
constexpr int kVolWarps = kVolThreads / 32;
// What the interior sums read: grid offsets of rows and planes, the cells'
// offsets from X_r as float pairs and their squares in FP32, per axis.
struct VolTables {
    long long row_off[kVolAx], plane_off[kVolAx];
    float2 tbf[3][kVolAx];
    float tcf[3][kVolAx];
};
struct VolShared {
    float4 phi[2][kVolAx * kVolAx];  // node planes: (max(-phi, 0), max(phi, 0)) as float pairs
    VolTables tb;
    float2 tsq[3][kVolAx];           // squares of the nodes' offsets as float pairs
    int count[2][kVolWarps];         // entries of the warps' lists: near nodes, cut cells
    uint16_t list[2][kVolWarps][(kVolAx + kVolWarps - 1) / kVolWarps * kVolAx];
};
constexpr size_t kVolSmem = sizeof(VolShared);
static_assert(kVolSmem >= 10 * kVolThreads * sizeof(double), "the CTA sums reuse the dynamic shared memory");

// Double-float accumulation: a sum kept as the unevaluated pair hi + lo of two
// floats -- Knuth's TwoSum for the addition error and the fused multiply-add
// for the exact product error (Dekker 1971) -- about 44 significant bits on
// the FP32 pipes, which run 64 times faster than FP64 on GB300.  Used for the
// level set, alpha and the field sums of both field precisions; the per-CTA
// tables and the CTA reduction stay FP64.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ void df_add2(DF &a, float bh, float bl) {
    const float s = a.hi + bh;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (bh - bb);
    a.hi = s;
    a.lo += e + bl;
}
// a += (rh + rl) (wh + wl), keeping the product's rounding error and the
// first-order cross terms
__device__ __forceinline__ void df_add_prod(DF &a, float rh, float rl, float wh, float wl) {
    const float pr = rh * wh;
    const float pe = fmaf(rh, wh, -pr) + fmaf(rh, wl, rl * wh);
    df_add2(a, pr, pe);
}
// hi + lo of every lane added over the warp (fixed shuffle order); result in lane 0
__device__ __forceinline__ void df_warp_sum(DF &a) {
    for (int o = 16; o > 0; o >>= 1) {
        const float bh = __shfl_down_sync(0xffffffffu, a.hi, o), bl = __shfl_down_sync(0xffffffffu, a.lo, o);
        const float lo = a.lo;
        a.lo = 0.f;
        df_add2(a, bh, bl + lo);
    }
}
__device__ __forceinline__ float2 df_split_rn(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}
// A field value as a float pair: an FP32 value exactly (lo = 0), an FP64 value
// split on the integer pipe (within 2^-47 of the double; no FP64 operation)
__device__ __forceinline__ float2 field_pair(float x) { return make_float2(x, 0.0f); }
__device__ __forceinline__ float2 field_pair(double x) { return df_split(x); }
// a + b, both double-float, renormalised (TwoSum on the high parts)
__device__ __forceinline__ DF df_sum(DF a, DF b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb);
    const float l = e + (a.lo + b.lo);
    const float h = s + l;
    return DF{h, l - (h - s)};
}
// phi = sqrt(x2) * iR - 1 in double-float, x2 > 0: the square root by one
// Newton step from the FP32 reciprocal square root (Heron's iteration; the
// start's relative error below 2^-22 leaves about 2^-45), then the product
// with 1/R and the subtraction.
__device__ __forceinline__ DF df_phi(DF x2, float2 iR) {
    const float rs = rsqrtf(x2.hi);
    const float r = x2.hi * rs;
    const float p = r * r;
    const float pe = fmaf(r, r, -p);
    const float corr = (((x2.hi - p) - pe) + x2.lo) * (0.5f * rs);
    const float q = r * iR.x;
    const float qe = fmaf(r, iR.x, -q) + fmaf(r, iR.y, corr * iR.x);
    return df_sum(DF{q, qe}, DF{-1.0f, 0.0f});
}

// A thread's double-float sums of w = alpha u, of the six products ry w2,
// rz w1, rz w0, rx w2, rx w1, ry w0 (r x w = (ry w2 - rz w1, rz w0 - rx w2,
// rx w1 - ry w0)), of the cut cells' alpha, and its number of cells of alpha 1.
struct VolSums {
    DF W[3] = {}, Pm[6] = {}, V = {};
    unsigned inside = 0;
};
// one cell's share: its alpha, field values and centre offsets as float pairs
template <typename T>
__device__ __forceinline__ void add_cut_cell(VolSums &s, float2 a2, const float2 v[3], float2 fx, float2 fy, float2 fz) {
    df_add2(s.V, a2.x, a2.y);
    float wh[3], wl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        // alpha u with the product's rounding error and the cross terms
        wh[c] = a2.x * v[c].x;
        wl[c] = fmaf(a2.x, v[c].x, -wh[c]) + a2.y * v[c].x;
        if constexpr (sizeof(T) == 8) wl[c] = fmaf(a2.x, v[c].y, wl[c]);
        df_add2(s.W[c], wh[c], wl[c]);
    }
    df_add_prod(s.Pm[0], fy.x, fy.y, wh[2], wl[2]);
    df_add_prod(s.Pm[1], fz.x, fz.y, wh[1], wl[1]);
    df_add_prod(s.Pm[2], fz.x, fz.y, wh[0], wl[0]);
    df_add_prod(s.Pm[3], fx.x, fx.y, wh[2], wl[2]);
    df_add_prod(s.Pm[4], fx.x, fx.y, wh[1], wl[1]);
    df_add_prod(s.Pm[5], fy.x, fy.y, wh[0], wl[0]);
}

// The tables of a box (its first cell lo, centre c), by warps 0 to 5.
__device__ __forceinline__ void volume_tables(VolTables &tb, const DevGrid &g, const int lo[3], const int dims[3],
                                              const double c[3]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 3) {
        for (int i = lane; i < dims[warp]; i += 32) {
            const double xc = g.org[warp] + ((double)(lo[warp] + i) + 0.5) * g.h - c[warp];
            tb.tbf[warp][i] = df_split_rn(xc);
            tb.tcf[warp][i] = (float)(xc * xc);
        }
    } else if (warp == 3) {
        for (int j = lane; j < dims[1]; j += 32) tb.row_off[j] = (long long)wrap_int(lo[1] + j, g.n[1]) * g.n[0];
    } else if (warp == 4) {
        for (int k = lane; k < dims[2]; k += 32)
            tb.plane_off[k] = (long long)wrap_int(lo[2] + k, g.n[2]) * g.n[1] * g.n[0];
    }
}
// The square of the distance R + off h from a particle's centre, or below = -1
// (lower bounds) or 0 (upper ones) where that is not positive; and the FP32 bound
// of squares from it, with a relative margin far above their rounding (lower
// bounds below, upper ones above).  k_volume and k_volume_plan both tell the cells
// of alpha 1 apart by the first: the roundings are explicit, so that a cell is
// inside for both or for neither.
constexpr double kInside = -0.8661, kOutside = 0.8661;  // in h: past a cell's half diagonal
__device__ __forceinline__ double bound_sq(double R, double off, double h, double below) {
    const double b = __fma_rn(off, h, R);
    return b > 0.0 ? __dmul_rn(b, b) : below;
}
__device__ __forceinline__ float lower_bound32(double sq) { return sq < 0.0 ? -1.0f : __fmul_rn((float)sq, 1.0f - 1e-5f); }
__device__ __forceinline__ float upper_bound32(double sq) { return __fmul_rn((float)sq, 1.0f + 1e-5f); }

// squared distance of a cell's centre from X_r in FP32 (one order everywhere)
__device__ __forceinline__ float centre_sq(float xy, float z) { return __fadd_rn(xy, z); }

// The cells of alpha 1 (squared distance below rin2) in planes [z0, z1): a thread
// takes columns of the slab, so that a cell costs three sums and the two
// products with its z offset; those with x and y are taken once a column.
// DEPTH planes' field values are loaded together (two of an FP64 field where four
// would not fit the registers of k_volume: 41 against 38 us).
template <int DEPTH, typename T>
__device__ __forceinline__ void interior_columns(VolSums &s, const T *__restrict__ u, const DevGrid &g, const VolTables &tb,
                                                 int lo0w, const int dims[3], int z0, int z1, float rin2) {
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    for (int q = threadIdx.x; q < dims[0] * dims[1]; q += kVolThreads) {
        const int j = q / dims[0], i = q - j * dims[0];
        const float xy = __fadd_rn(tb.tcf[0][i], tb.tcf[1][j]);
        if (!(xy < rin2)) continue;
        const T *const col = u + tb.row_off[j] + wrap_add(lo0w, i, g.n[0]);
        DF S[3] = {}, Z0 = {}, Z1 = {};
        unsigned n = 0;
        for (int k0 = z0; k0 < z1; k0 += DEPTH) {
            bool in[DEPTH];
            T v[DEPTH][3];
#pragma unroll
            for (int r = 0; r < DEPTH; ++r) {
                in[r] = k0 + r < z1 && centre_sq(xy, tb.tcf[2][k0 + r]) < rin2;
                if (in[r])
#pragma unroll
                    for (int c = 0; c < 3; ++c) v[r][c] = col[c * N + tb.plane_off[k0 + r]];
            }
#pragma unroll
            for (int r = 0; r < DEPTH; ++r) {
                if (!in[r]) continue;
                const float2 fz = tb.tbf[2][k0 + r];
                const float2 v0 = field_pair(v[r][0]), v1 = field_pair(v[r][1]), v2 = field_pair(v[r][2]);
                df_add2(S[0], v0.x, v0.y);
                df_add2(S[1], v1.x, v1.y);
                df_add2(S[2], v2.x, v2.y);
                df_add_prod(Z0, fz.x, fz.y, v0.x, v0.y);
                df_add_prod(Z1, fz.x, fz.y, v1.x, v1.y);
                ++n;
            }
        }
        if (n == 0) continue;
        const float2 fx = tb.tbf[0][i], fy = tb.tbf[1][j];
#pragma unroll
        for (int c = 0; c < 3; ++c) df_add2(s.W[c], S[c].hi, S[c].lo);
        df_add_prod(s.Pm[0], fy.x, fy.y, S[2].hi, S[2].lo);
        df_add2(s.Pm[1], Z1.hi, Z1.lo);
        df_add2(s.Pm[2], Z0.hi, Z0.lo);
        df_add_prod(s.Pm[3], fx.x, fx.y, S[2].hi, S[2].lo);
        df_add_prod(s.Pm[4], fx.x, fx.y, S[1].hi, S[1].lo);
        df_add_prod(s.Pm[5], fy.x, fy.y, S[0].hi, S[0].lo);
        s.inside += n;
    }
}

// End of a CTA of the double-float sums: the CTA's sums in double-float, one
// conversion to FP64 per quantity, and the particle's nsplit CTA sums in FP64, in
// order, by the last CTA of the particle to finish (FP64 issue is scarce on this
// part: no FP64 operation per warp).  The threads' sums go through shared memory
// (s_sum, free again once every thread is here): a warp adds a quantity, its
// lanes kVolWarps entries each before the shuffles, a third of the instructions of
// shuffle trees in every warp.
struct VolFinish {
    float2 sum[10][kVolThreads];
};
__device__ __forceinline__ void volume_finish_df(VolSums &s, double h, int p, int split, int nsplit,
                                                 double *__restrict__ partial, unsigned int *__restrict__ done,
                                                 double *Iu, double *Irxu, double *vol, VolFinish &f) {
    __shared__ unsigned s_ncell[kVolWarps];
    __shared__ double s_q[10];
    __shared__ int s_last_df;
    const unsigned ncell = __reduce_add_sync(0xffffffffu, s.inside);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) s_ncell[wid] = ncell;
    __syncthreads();  // every thread is done with the shared memory reused here
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        const DF x = q < 3 ? s.W[q] : q < 9 ? s.Pm[q < 3 || q > 8 ? 0 : q - 3] : s.V;
        f.sum[q][threadIdx.x] = make_float2(x.hi, x.lo);
    }
    __syncthreads();
    for (int q = wid; q < 10; q += kVolWarps) {
        DF x = {0.f, 0.f};
#pragma unroll
        for (int m = 0; m < kVolWarps; ++m) {
            const float2 y = f.sum[q][lane + 32 * m];
            df_add2(x, y.x, y.y);
        }
        df_warp_sum(x);
        if (lane == 0) s_q[q] = df_to_double(make_float2(x.hi, x.lo));
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        const int k = threadIdx.x;
        double x;
        if (k < 3) {
            x = s_q[k];
        } else if (k < 6) {
            x = s_q[3 + 2 * (k - 3)] - s_q[4 + 2 * (k - 3)];  // (ry w2 - rz w1, rz w0 - rx w2, rx w1 - ry w0)
        } else {
            unsigned n = 0;
            for (int w = 0; w < kVolWarps; ++w) n += s_ncell[w];
            x = (double)n + s_q[9];
        }
        const double h3 = h * h * h;
        partial[((size_t)p * nsplit + split) * 7 + k] = x * h3;
        __threadfence();  // release: partials before the count
    }
    __syncwarp();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last_df = atomicAdd(done + p, 1u) == (unsigned int)nsplit - 1;
        __threadfence();  // acquire: the count before the other partials
    }
    __syncthreads();
    if (s_last_df && threadIdx.x < 7) {
        const int k = threadIdx.x;
        double x = 0.0;
        for (int sp = 0; sp < nsplit; ++sp) x += __ldcg(partial + ((size_t)p * nsplit + sp) * 7 + k);
        if (k < 3) {
            if (Iu) Iu[3 * p + k] = x;
        } else if (k < 6) {
            if (Irxu) Irxu[3 * p + k - 3] = x;
        } else if (vol) {
            vol[p] = x;
        }
        if (k == 0) done[p] = 0;  // ready for the next call
    }
}

// Exclusive scan of cnt[0..n) into pre[0..n] by warp 0 (n may exceed 32).
__device__ __forceinline__ void warp0_scan(const int *cnt, int *pre, int n) {
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    int carry = 0;
    for (int base = 0; base < n; base += 32) {
        const int v = base + lane < n ? cnt[base + lane] : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (base + lane < n) pre[base + lane] = carry + x - v;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) pre[n] = carry;
}

// Row of flat index t: largest r with pre[r] <= t (pre ascending, pre[0] = 0).
__device__ __forceinline__ int find_row(const int *pre, int nrows, int t) {
    int a = 0, b = nrows - 1;
    while (a < b) {
        const int mid = (a + b + 1) >> 1;
        if (pre[mid] <= t) a = mid;
        else b = mid - 1;
    }
    return a;
}

// End of a volume-integral CTA: the fixed-order CTA sum of the 7 partial
// sums, scaled by h^3, is stored as slab `split` of particle p; the last slab
// of the particle to finish (completion counter) adds the nsplit slabs in
// order and writes the particle's integrals.
// s_acc: shared scratch of 7 * kVolThreads doubles (the kernel's dynamic shared
// memory, free again once the CTA's sums are done).
__device__ void volume_finish(double acc[7], double h, int p, int split, int nsplit, double *__restrict__ partial,
                              unsigned int *__restrict__ done, double *Iu, double *Irxu, double *vol, double *s_acc) {
    __shared__ int s_last;
    // fixed-order CTA sum of the 7 partials through shared memory: 7 warps,
    // one per quantity, each lane adding 8 entries then a shuffle tree (FP64
    // adds are scarce on this part: a shuffle tree over all 256 threads would
    // cost more FP64 work than a thin slab's cells)
    {
        __syncthreads();  // every thread is done with the shared memory reused here
#pragma unroll
        for (int k = 0; k < 7; ++k) s_acc[k * kVolThreads + threadIdx.x] = acc[k];
        __syncthreads();
        const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
        if (wq < 7) {
            double x = 0.0;
#pragma unroll
            for (int m = 0; m < kVolThreads / 32; ++m) x += s_acc[wq * kVolThreads + lane + 32 * m];
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (lane == 0) s_acc[wq * kVolThreads] = x;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const double h3 = h * h * h;
#pragma unroll
            for (int k = 0; k < 7; ++k) acc[k] = s_acc[k * kVolThreads] * h3;
        }
    }
    __shared__ double s_part[kVolMaxSplit * 7];
    if (threadIdx.x == 0) {
        double *dst = partial + ((size_t)p * nsplit + split) * 7;
        for (int k = 0; k < 7; ++k) dst[k] = acc[k];
        __threadfence();  // release: partials before the count
        s_last = atomicAdd(done + p, 1u) == (unsigned int)nsplit - 1;
        __threadfence();  // acquire: the count before the other partials
    }
    __syncthreads();
    if (s_last) {
        // the last CTA of the particle adds the partials in slab order
        for (int i = threadIdx.x; i < nsplit * 7; i += blockDim.x) s_part[i] = partial[(size_t)p * nsplit * 7 + i];
        __syncthreads();
    }
    if (s_last && threadIdx.x == 0) {
        double sum[7] = {0, 0, 0, 0, 0, 0, 0};
        for (int sp = 0; sp < nsplit; ++sp)
            for (int k = 0; k < 7; ++k) sum[k] += s_part[sp * 7 + k];
        if (Iu)
            for (int a = 0; a < 3; ++a) Iu[3 * p + a] = sum[a];
        if (Irxu)
            for (int a = 0; a < 3; ++a) Irxu[3 * p + a] = sum[3 + a];
        if (vol) vol[p] = sum[6];
        done[p] = 0;  // ready for the next call
    }
}

// Per plane the CTA lists the near nodes and the cut cells (a list a warp, from
// ballots over its rows, tested on FP32 squares of the tables) and runs the
// lists end to end, a thread an entry, two barriers a plane; everything per
// node and cell is double-float on the FP32 pipes.  64 spheres of 24 cells in an
// FP64 field: 39 us; 57 us with per-row index ranges, row scans and a row search
// per entry (five barriers a plane) and the interior cells listed as well.
//
// A kept volume plan (particle_volume_integrals_keep / _plan): per particle,
// the cut cells plane by plane in visiting order, with their alpha or a skip
// mark, so that a second call at the same particle positions sums another field
// over the same cells with the same alpha without evaluating a level set (the
// cells of alpha 1 follow from the positions).  Capacity `cap` entries per
// particle; a keeping CTA's slab starts at dims0 dims1 z0, and each plane's
// header gives its list's count and first entry.
struct PvfPlanDev {
    int cap;
    int2 *hdr;        // [P][kVolAx] per plane: cut cells, first entry
    unsigned *bent;   // [P][cap] cut cell i | j << 8, or kPvfSkip
    float2 *balpha;   // [P][cap] its alpha as a float pair
    double *pos;      // [P][4] X_r and R the plan was kept for
};
constexpr unsigned kPvfSkip = 0x80000000u;

// MODE 0: plain; 1: also keep the plan (k_volume_plan sums from it).
template <typename T, int MODE = 0>
__global__ void __launch_bounds__(kVolThreads, 3) k_volume(CaseTab ct, int P, int nsplit,
                                                        const double *__restrict__ Xr,
                                                        const double *__restrict__ radius,
                                                        double *__restrict__ partial,
                                                        unsigned int *__restrict__ done, double *Iu,
                                                        double *Irxu, double *vol, DevStatus *st,
                                                        PvfPlanDev pl = PvfPlanDev{}) {
    extern __shared__ __align__(16) double s_vol[];
    VolShared &s = *(VolShared *)s_vol;
    const int p = blockIdx.x / nsplit, split = blockIdx.x % nsplit;
    if (p >= P) return;
    const DevCase &cd = ct.of_particle(p);
    const DevGrid g = cd.g;
    const T *__restrict__ u = (const T *)cd.u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the particle's scalars, formed once by warp 0 (FP64 is scarce here: 256
    // threads each forming them cost more than a slab's cells)
    __shared__ double s_c[3], s_sq[4], s_iR;
    __shared__ float s_fsq[4];
    __shared__ float2 s_iRf;
    __shared__ int s_box[7];
    if (warp == 0) {
        const double cc[3] = {Xr[3 * p], Xr[3 * p + 1], Xr[3 * p + 2]};
        const double R0 = radius[p];
        bool okk = finite3(cc) && isfinite(R0) && R0 > 0.0;
        if (!okk && lane == 0 && split == 0) raise_status(st, IB_ERR_NONFINITE, p);
        if (okk) {
            // a lane an axis
            const int a = lane < 3 ? lane : 0;
            const double ca = a == 0 ? cc[0] : a == 1 ? cc[1] : cc[2];
            const long long l = (long long)floor((ca - R0 - g.org[a]) * g.inv_h) - 1;
            const long long hgh = (long long)floor((ca + R0 - g.org[a]) * g.inv_h) + 1;
            const int d = (int)(hgh - l + 1);
            if (lane < 3) {
                s_box[a] = (int)l;
                s_box[3 + a] = d;
            }
            okk = __all_sync(0xffffffffu, !(d > g.n[a] || l < INT_MIN / 2 || l > INT_MAX / 2));
            if (!okk && lane == 0 && split == 0) raise_status(st, IB_ERR_UNSUPPORTED, p);
            if constexpr (MODE != 0) {
                const bool tabbed = __all_sync(0xffffffffu, d <= kVolMaxBox);
                __syncwarp();
                if (okk && (!tabbed || (long long)s_box[3] * s_box[4] * s_box[5] > pl.cap)) {
                    if (lane == 0 && split == 0) raise_status(st, IB_ERR_UNSUPPORTED, p);
                    okk = false;
                }
            }
            // squares of the bounds: cells surely inside, cells of alpha 0, the
            // node shell (a lane a bound)
            const double off = lane == 0 ? kInside : lane == 1 ? kOutside : lane == 2 ? -1.75 : 1.75;
            if (lane < 4) {
                // (the nodes and cells that matter lie 0.01 h inside the node shell and
                // 8e-5 h inside the cell bounds; cells in the FP32 margin take the corner
                // formula, exact for them too)
                const double sq = bound_sq(R0, off, g.h, lane == 0 ? -1.0 : 0.0);
                s_sq[lane] = sq;
                s_fsq[lane] = lane & 1 ? upper_bound32(sq) : lower_bound32(sq);
            }
            const double ir = 1.0 / R0;
            if (lane == 0) s_iR = ir, s_iRf = df_split_rn(ir);
        }
        if (lane < 3) s_c[lane] = lane == 0 ? cc[0] : lane == 1 ? cc[1] : cc[2];
        if (MODE != 0 && split == 0 && lane == 0) {
            pl.pos[4 * p] = cc[0], pl.pos[4 * p + 1] = cc[1], pl.pos[4 * p + 2] = cc[2];
            pl.pos[4 * p + 3] = R0;
        }
        if (lane == 0) s_box[6] = okk;
    }
    __syncthreads();
    const double c[3] = {s_c[0], s_c[1], s_c[2]};
    const bool ok = s_box[6] != 0;
    const int lo[3] = {ok ? s_box[0] : 0, ok ? s_box[1] : 0, ok ? s_box[2] : 0};
    const int dims[3] = {ok ? s_box[3] : 0, ok ? s_box[4] : 0, ok ? s_box[5] : 0};
    const int t = (dims[2] + nsplit - 1) / nsplit;
    const int z0 = split * t, z1 = min(dims[2], z0 + t);
    const int lo0w = ok ? wrap_int(lo[0], g.n[0]) : 0;
    if (dims[0] <= kVolMaxBox && dims[1] <= kVolMaxBox && dims[2] <= kVolMaxBox) {
        VolSums sums;
        if (ok && z0 < z1) {
            const int nx = dims[0] + 1, ny = dims[1] + 1;
            volume_tables(s.tb, g, lo, dims, c);
            if (warp >= 5) {  // (warps 0 to 4 fill the other tables)
                const int a = warp - 5;
                for (int i = lane; i <= dims[a]; i += 32) {
                    const double xn = g.org[a] + (double)(lo[a] + i) * g.h - c[a];
                    s.tsq[a][i] = df_split_rn(xn * xn);
                }
            }
            const float rin2 = s_fsq[0], rout2 = s_fsq[1], sl2 = s_fsq[2], sh2 = s_fsq[3];
            const float2 iRf = s_iRf;
            __syncthreads();
            auto push = [&](uint16_t *list, int &cnt, bool flag, int code) {
                const unsigned b = __ballot_sync(0xffffffffu, flag);
                if (flag) list[cnt + __popc(b & ((1u << lane) - 1u))] = (uint16_t)code;
                cnt += __popc(b);
            };
            // run(entry's place, i, j) over the warps' lists end to end
            auto run_lists = [&](int which, auto &&run) {
                int start = 0, w = 0, n = s.count[which][0];
                for (int e = threadIdx.x;; e += kVolThreads) {
                    while (w < kVolWarps && e >= start + n) {
                        start += n;
                        ++w;
                        n = w < kVolWarps ? s.count[which][w] : 0;
                    }
                    if (w == kVolWarps) break;
                    const int code = s.list[which][w][e - start];
                    run(e, code & 255, code >> 8);
                }
            };
            auto list_nodes = [&](int kn) {
                const float z2 = s.tsq[2][kn].x;
                int cnt = 0;
                for (int i0 = 0; i0 < nx; i0 += 32) {
                    const int i = i0 + lane;
                    const float xz = i < nx ? s.tsq[0][i].x + z2 : 0.0f;
                    for (int j = warp; j < ny; j += kVolWarps) {
                        const float q = xz + s.tsq[1][j].x;
                        push(s.list[0][warp], cnt, i < nx && q >= sl2 && q <= sh2, j << 8 | i);
                    }
                }
                if (lane == 0) s.count[0][warp] = cnt;
            };
            // a listed node's level set value in double-float
            auto eval_nodes = [&](int kn) {
                float4 *const buf = s.phi[kn & 1];
                const DF z2 = {s.tsq[2][kn].x, s.tsq[2][kn].y};
                run_lists(0, [&](int, int i, int j) {
                    const DF x2 = df_sum(DF{s.tsq[0][i].x, s.tsq[0][i].y},
                                         df_sum(DF{s.tsq[1][j].x, s.tsq[1][j].y}, z2));
                    const DF ph = x2.hi > 0.0f ? df_phi(x2, iRf) : DF{-1.0f, 0.0f};
                    buf[j * nx + i] = ph.hi < 0.0f ? make_float4(-ph.hi, -ph.lo, 0.f, 0.f)
                                                   : make_float4(0.f, 0.f, ph.hi, ph.lo);
                });
            };
            auto list_cells = [&](int kz) {
                const float z2 = s.tb.tcf[2][kz];
                int cnt = 0;
                for (int i0 = 0; i0 < dims[0]; i0 += 32) {
                    const int i = i0 + lane;
                    const bool cell = i < dims[0];
                    const float x2 = cell ? s.tb.tcf[0][i] : 0.0f;
                    for (int j = warp; j < dims[1]; j += kVolWarps) {
                        const float q = centre_sq(__fadd_rn(x2, s.tb.tcf[1][j]), z2);
                        push(s.list[1][warp], cnt, cell && !(q < rin2) && q <= rout2, j << 8 | i);
                    }
                }
                if (lane == 0) s.count[1][warp] = cnt;
            };
            list_nodes(z0);
            __syncthreads();
            eval_nodes(z0);
            __syncthreads();
            list_nodes(z0 + 1);
            interior_columns<sizeof(T) == 8 ? 2 : 4>(sums, u, g, s.tb, lo0w, dims, z0, z1, rin2);
            // the CTA's entries in the plan: from dims0 dims1 z0 on, plane by plane
            const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
            long long pb = (long long)p * pl.cap + (long long)dims[0] * dims[1] * z0;
            for (int kz = z0; kz < z1; ++kz) {
                __syncthreads();
                eval_nodes(kz + 1);
                list_cells(kz);
                __syncthreads();
                int ncut = 0;
                if constexpr (MODE == 1) {
                    for (int w = 0; w < kVolWarps; ++w) ncut += s.count[1][w];
                    if (threadIdx.x == 0) pl.hdr[p * kVolAx + kz] = make_int2(ncut, (int)(pb - (long long)p * pl.cap));
                }
                const float4 *const f0 = s.phi[kz & 1], *const f1 = s.phi[(kz + 1) & 1];
                const float2 fz = s.tb.tbf[2][kz];
                const T *const up = u + s.tb.plane_off[kz];
                // alpha = sum of max(-phi, 0) / sum |phi| over the corners, in double-float
                run_lists(1, [&](int e, int i, int j) {
                    if (MODE == 1) pl.bent[pb + e] = kPvfSkip;  // until the cell counts
                    // (loaded before alpha is known: its latency overlaps the sums)
                    const T *const uc = up + s.tb.row_off[j] + wrap_add(lo0w, i, g.n[0]);
                    const T u3[3] = {uc[0], uc[N], uc[2 * N]};
                    const int qn = j * nx + i;
                    const float4 cn[8] = {f0[qn], f0[qn + 1], f0[qn + nx], f0[qn + nx + 1],
                                          f1[qn], f1[qn + 1], f1[qn + nx], f1[qn + nx + 1]};
                    DF num = {0.f, 0.f}, neg = {0.f, 0.f};
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        df_add2(num, cn[m].x, cn[m].y);
                        df_add2(neg, cn[m].z, cn[m].w);
                    }
                    num = df_sum(num, DF{0.f, 0.f});
                    neg = df_sum(neg, DF{0.f, 0.f});
                    if (num.hi == 0.0f && neg.hi > 0.0f) return;  // alpha = 0
                    float2 a2 = make_float2(1.f, 0.f);
                    const DF den = df_sum(num, neg);
                    if (den.hi == 0.0f) {
                        a2 = make_float2(0.5f, 0.f);
                    } else if (neg.hi != 0.0f) {
                        if (den.hi < 1e-30f) {
                            a2 = df_split_rn(((double)num.hi + num.lo) / ((double)den.hi + den.lo));
                        } else {
                            // num / den: a quotient and one remainder correction
                            const float rd = __frcp_rn(den.hi);
                            const float q1 = num.hi * rd;
                            const float pr = q1 * den.hi;
                            const float pe = fmaf(q1, den.hi, -pr);
                            const float rr = ((num.hi - pr) - pe) + fmaf(-q1, den.lo, num.lo);
                            a2 = make_float2(q1, rr * rd);
                        }
                    }
                    if constexpr (MODE == 1) {
                        pl.bent[pb + e] = (unsigned)i | ((unsigned)j << 8);
                        pl.balpha[pb + e] = a2;
                    }
                    const float2 v[3] = {field_pair(u3[0]), field_pair(u3[1]), field_pair(u3[2])};
                    add_cut_cell<T>(sums, a2, v, s.tb.tbf[0][i], s.tb.tbf[1][j], fz);
                });
                pb += ncut;
                if (kz + 1 < z1) list_nodes(kz + 2);
            }
        }
        volume_finish_df(sums, g.h, p, split, nsplit, partial, done, Iu, Irxu, vol, *(VolFinish *)s_vol);
        return;
    }
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    {
        const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
        const double h = g.h, iR = s_iR, rin2 = s_sq[0], rout2 = s_sq[1];
        {
            // boxes wider than kVolMaxBox: every cell of the slab, corners evaluated directly
            for (int kz = z0; kz < z1; ++kz) {
                const int k = lo[2] + kz;
                const double rz = g.org[2] + ((double)k + 0.5) * h - c[2];
                const long long plane_off = (long long)wrap_int(k, g.n[2]) * g.n[1];
                for (int q = threadIdx.x; q < dims[0] * dims[1]; q += blockDim.x) {
                    const int j = q / dims[0], i = q - j * dims[0];
                    const double rx = g.org[0] + ((double)(lo[0] + i) + 0.5) * h - c[0];
                    const double ry = g.org[1] + ((double)(lo[1] + j) + 0.5) * h - c[1];
                    const double d2 = rx * rx + ry * ry + rz * rz;
                    if (d2 > rout2) continue;
                    double al = 1.0;
                    if (!(d2 < rin2)) {
                        double num = 0.0, den = 0.0;
#pragma unroll
                        for (int m = 0; m < 8; ++m) {
                            const double x = g.org[0] + (double)(lo[0] + i + (m & 1)) * h - c[0];
                            const double y = g.org[1] + (double)(lo[1] + j + ((m >> 1) & 1)) * h - c[1];
                            const double z = g.org[2] + (double)(k + ((m >> 2) & 1)) * h - c[2];
                            const double ph = sqrt(x * x + y * y + z * z) * iR - 1.0;
                            if (-ph > 0.0) num += -ph;
                            den += fabs(ph);
                        }
                        al = den > 0.0 ? num / den : 0.5;
                        if (al == 0.0) continue;
                    }
                    const long long cc = (plane_off + wrap_int(lo[1] + j, g.n[1])) * g.n[0] + wrap_add(lo0w, i, g.n[0]);
                    const double u0 = (double)u[cc], u1 = (double)u[N + cc], u2 = (double)u[2 * N + cc];
                    acc[0] += al * u0;
                    acc[1] += al * u1;
                    acc[2] += al * u2;
                    acc[3] += al * (ry * u2 - rz * u1);
                    acc[4] += al * (rz * u0 - rx * u2);
                    acc[5] += al * (rx * u1 - ry * u0);
                    acc[6] += al;
                }
            }
        }
    }
    volume_finish(acc, g.h, p, split, nsplit, partial, done, Iu, Irxu, vol, s_vol);
}

// ---------------------------------------------------------------------------
// Volume integrals from a kept plan: the cells of alpha 1 by columns of a slab of
// planes, as in k_volume, and the particle's kept cut cells with their alpha, one
// list per particle (the planes' lists in plane order), split evenly over nsplit
// CTAs, each taking a contiguous range, kPlanUnroll cells at a time with their
// list entries and field values loaded together.  The same cells, alpha and
// per-cell arithmetic as k_volume, in another summation order.  64 spheres of 24
// cells in an FP64 field: 27 us; 32 us with the interior cells read from a list.
// ---------------------------------------------------------------------------
constexpr int kPlanUnroll = 4;

template <typename T>
__global__ void __launch_bounds__(kVolThreads, 2) k_volume_plan(CaseTab ct, int P, int nsplit,
                                                              const double *__restrict__ Xr,
                                                              const double *__restrict__ radius,
                                                              double *__restrict__ partial,
                                                              unsigned int *__restrict__ done, double *Iu,
                                                              double *Irxu, double *vol, DevStatus *st,
                                                              PvfPlanDev pl) {
    __shared__ VolTables tb;
    __shared__ VolFinish fin;
    __shared__ int c_cut[kVolAx], b_cut[kVolAx], p_cut[kVolAx + 1];
    __shared__ double s_c[3];
    __shared__ float s_rin2;
    __shared__ int s_box[7];
    const int p = blockIdx.x / nsplit, split = blockIdx.x % nsplit;
    if (p >= P) return;
    const DevCase &cd = ct.of_particle(p);
    const DevGrid g = cd.g;
    const T *__restrict__ u = (const T *)cd.u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the plan's plane headers, loaded beside the particle's scalars (every
    // particle has kVolAx header slots; only the box's planes are read)
    if (warp > 0)
        for (int k = threadIdx.x - 32; k < kVolAx; k += kVolThreads - 32) {
            const int2 hc = pl.hdr[p * kVolAx + k];
            c_cut[k] = hc.x;
            b_cut[k] = hc.y;
        }
    else {
        // the particle's box as the keeping call formed it, once the plan is
        // known to be this particle's; a lane an axis
        const double cc[3] = {Xr[3 * p], Xr[3 * p + 1], Xr[3 * p + 2]};
        const double R0 = radius[p];
        const double *q = pl.pos + 4 * p;
        bool okk = q[0] == cc[0] && q[1] == cc[1] && q[2] == cc[2] && q[3] == R0;
        if (!okk && lane == 0 && split == 0) raise_status(st, IB_ERR_INVALID, p);  // not the plan's particle
        okk = okk && finite3(cc) && isfinite(R0) && R0 > 0.0;
        if (okk) {
            const int a = lane < 3 ? lane : 0;
            const double ca = a == 0 ? cc[0] : a == 1 ? cc[1] : cc[2];
            const long long l = (long long)floor((ca - R0 - g.org[a]) * g.inv_h) - 1;
            const long long hgh = (long long)floor((ca + R0 - g.org[a]) * g.inv_h) + 1;
            const int d = (int)(hgh - l + 1);
            if (lane < 3) {
                s_box[a] = (int)l;
                s_box[3 + a] = d;
                s_c[a] = ca;
            }
            // the keeping call kept only boxes of the tabulated size
            okk = __all_sync(0xffffffffu, !(d > g.n[a] || d > kVolMaxBox || l < INT_MIN / 2 || l > INT_MAX / 2));
            __syncwarp();
            if (okk && (long long)s_box[3] * s_box[4] * s_box[5] > pl.cap) okk = false;  // not kept (reported then)
            if (lane == 0) s_rin2 = lower_bound32(bound_sq(R0, kInside, g.h, -1.0));
        }
        if (lane == 0) s_box[6] = okk;
    }
    __syncthreads();
    VolSums sums;
    if (s_box[6]) {
        const int lo[3] = {s_box[0], s_box[1], s_box[2]}, dims[3] = {s_box[3], s_box[4], s_box[5]};
        const double c[3] = {s_c[0], s_c[1], s_c[2]};
        const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
        const int lo0w = wrap_int(lo[0], g.n[0]);
        volume_tables(tb, g, lo, dims, c);
        warp0_scan(c_cut, p_cut, dims[2]);
        __syncthreads();
        const int t = (dims[2] + nsplit - 1) / nsplit;
        interior_columns<4>(sums, u, g, tb, lo0w, dims, min(dims[2], split * t), min(dims[2], (split + 1) * t), s_rin2);
        // cut cells: the kept alpha (entries of cells with alpha = 0 are marked)
        const long long base = (long long)p * pl.cap;
        const int NB = p_cut[dims[2]];
        const int j0 = (int)((long long)NB * split / nsplit), j1 = (int)((long long)NB * (split + 1) / nsplit);
        // a thread's entries ascend, so its plane only moves forward
        int kzb = j0 + (int)threadIdx.x < j1 ? find_row(p_cut, dims[2], j0 + threadIdx.x) : 0;
        for (int e0 = j0 + threadIdx.x; e0 < j1; e0 += kPlanUnroll * kVolThreads) {
            int kz[kPlanUnroll];
            unsigned ent[kPlanUnroll];
            float2 al[kPlanUnroll];
#pragma unroll
            for (int t = 0; t < kPlanUnroll; ++t) {
                const int e = e0 + t * kVolThreads;
                if (e < j1)
                    while (p_cut[kzb + 1] <= e) ++kzb;
                kz[t] = kzb;
                const long long at = base + b_cut[kz[t]] + (e - p_cut[kz[t]]);
                ent[t] = e < j1 ? pl.bent[at] : kPvfSkip;
                al[t] = e < j1 ? pl.balpha[at] : make_float2(0.f, 0.f);
            }
            float2 v[kPlanUnroll][3];
#pragma unroll
            for (int t = 0; t < kPlanUnroll; ++t) {
                if (ent[t] == kPvfSkip) continue;
                const int i = (int)(ent[t] & 255u), j = (int)(ent[t] >> 8);
                const long long cc = tb.plane_off[kz[t]] + tb.row_off[j] + wrap_add(lo0w, i, g.n[0]);
#pragma unroll
                for (int c = 0; c < 3; ++c) v[t][c] = field_pair(u[c * N + cc]);
            }
#pragma unroll
            for (int t = 0; t < kPlanUnroll; ++t) {
                if (ent[t] == kPvfSkip) continue;
                const int i = (int)(ent[t] & 255u), j = (int)(ent[t] >> 8);
                add_cut_cell<T>(sums, al[t], v[t], tb.tbf[0][i], tb.tbf[1][j], tb.tbf[2][kz[t]]);
            }
        }
    }
    volume_finish_df(sums, g.h, p, split, nsplit, partial, done, Iu, Irxu, vol, fin);
}

// ---------------------------------------------------------------------------
// Volume integrals of axis-aligned ellipsoids (semi-axes a, b, c), through
// the level set of Eq. (level-set function of spheroidal geometries).  Grid =
// P * nsplit CTAs, CTA (p, s) walks a slab of cell planes of particle p's
// box.  The kernel is bound by the FP64 pipe (2 operations per clock and SM), so
// FP64 is kept for what needs it: FP32 squares of the scaled cell centres tell
// the cells with every corner inside (alpha = 1: five FP64 operations) and
// outside (none) from those the surface may cut, and the level set is evaluated
// only at nodes near the surface, once per node into two rolling node planes in
// shared memory.  An FP64 instruction costs the same for one lane as for 32:
// the CTA lists a plane's near nodes and cut cells (a list a warp, in the order
// of its rows) and runs the lists end to end, and what is the same for the CTA
// or a plane is computed by one warp.  48 ellipsoids of FP32 fields in boxes of
// up to 28 cells an axis: 64 us; 167 us with the level set at every node and
// alpha for every cell, 99 us with each warp running its own rows' lists.
// Boxes wider than kEllAx - 1 cells in x or y evaluate the corners per cell.
// The same sums as the oracle, grouped per lane, CTA and slab.
// ---------------------------------------------------------------------------
constexpr int kEllAx = 65;
constexpr int kEllWarps = kVolThreads / 32;
struct EllBox {
    double c[3], ia[3];  // centre, inverse semi-axes
    int lo[3], dims[3];  // first cell and cells per axis
    bool ok;
};
struct EllShared {
    double plane[2][kEllAx * kEllAx];
    double sq[3][kEllAx];                  // squares of the nodes' scaled coordinates
    double r[3][kEllAx];                   // the cells' distances from the centre
    float nsq[3][kEllAx], csq[3][kEllAx];  // FP32 squares: nodes, cell centres
    int off[3][kEllAx];                    // the cells' wrapped grid indices
    EllBox box;
    int count[2][kEllWarps];  // entries of the warps' lists: near nodes, cut cells
    uint16_t list[2][kEllWarps][(kEllAx + kEllWarps - 1) / kEllWarps * kEllAx];
};
constexpr size_t kEllSmem = sizeof(EllShared);
static_assert(kEllSmem >= 7 * kVolThreads * sizeof(double), "the CTA sum reuses the dynamic shared memory");

__device__ __forceinline__ double pvf_alpha8(const double ph[8]) {
    double num = 0.0, den = 0.0;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        // max(-phi, 0) and |phi| by the sign bit
        const double mag = fabs(ph[m]);
        num += __double_as_longlong(ph[m]) < 0 ? mag : 0.0;
        den += mag;
    }
    return den > 0.0 ? num / den : 0.5;
}
// an FP32 field value, exact, widened on the integer pipe (which takes subnormals as 0)
__device__ __forceinline__ double widened(float x) {
    return (__float_as_uint(x) << 1) - 1u < 0xffffffu ? (double)x : df_widen(x);
}
__device__ __forceinline__ double widened(double x) { return x; }

template <typename T>
__global__ void __launch_bounds__(kVolThreads) k_volume_ellipsoid(CaseTab ct, int P, int nsplit,
                                                                  const double *__restrict__ Xr,
                                                                  const double *__restrict__ axes,
                                                                  double *__restrict__ partial,
                                                                  unsigned int *__restrict__ done, double *Iu,
                                                                  double *Irxu, double *vol, DevStatus *st) {
    extern __shared__ __align__(16) double s_phi[];
    EllShared &s = *(EllShared *)s_phi;
    const int p = blockIdx.x / nsplit, split = blockIdx.x % nsplit;
    if (p >= P) return;
    const DevCase cd = ct.of_particle(p);
    const DevGrid g = cd.g;
    const T *__restrict__ u = (const T *)cd.u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {
        const double ctr[3] = {Xr[3 * p], Xr[3 * p + 1], Xr[3 * p + 2]};
        const double ax[3] = {axes[3 * p], axes[3 * p + 1], axes[3 * p + 2]};
        bool ok = finite3(ctr) && finite3(ax) && ax[0] > 0.0 && ax[1] > 0.0 && ax[2] > 0.0;
        if (!ok && lane == 0 && split == 0) raise_status(st, IB_ERR_NONFINITE, p);
        if (ok) {
            bool fits = true;
            for (int a = 0; a < 3; ++a) {
                const long long l = (long long)floor((ctr[a] - ax[a] - g.org[a]) * g.inv_h) - 1;
                const long long hg = (long long)floor((ctr[a] + ax[a] - g.org[a]) * g.inv_h) + 1;
                const int d = (int)(hg - l + 1);
                if (d > g.n[a] || l < INT_MIN / 2 || l > INT_MAX / 2) fits = false;
                if (lane == 0) {
                    s.box.c[a] = ctr[a];
                    s.box.ia[a] = 1.0 / ax[a];
                    s.box.lo[a] = (int)l;
                    s.box.dims[a] = d;
                }
            }
            if (!fits && lane == 0 && split == 0) raise_status(st, IB_ERR_UNSUPPORTED, p);
            ok = fits;
        }
        if (lane == 0) s.box.ok = ok;
    }
    __syncthreads();
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    const EllBox &bx = s.box;
    const bool ok = bx.ok;
    const int lo[3] = {ok ? bx.lo[0] : 0, ok ? bx.lo[1] : 0, ok ? bx.lo[2] : 0};
    const int dims[3] = {ok ? bx.dims[0] : 0, ok ? bx.dims[1] : 0, ok ? bx.dims[2] : 0};
    const int t = (dims[2] + nsplit - 1) / nsplit;
    const int z0 = split * t, z1 = min(dims[2], z0 + t);
    if (ok && z0 < z1) {
        const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
        const double h = g.h;
        const int nx = dims[0] + 1, ny = dims[1] + 1;
        if (nx <= kEllAx && ny <= kEllAx) {
            // axis a's entries of nodes and cells first, first + 1, ... (at most
            // kEllAx, none beyond the box)
            auto table = [&](int a, int first) {
                const double ia = bx.ia[a], ca = bx.c[a];
                for (int i = lane; i < kEllAx && first + i <= dims[a]; i += 32) {
                    const double x = (g.org[a] + (double)(lo[a] + first + i) * h - ca) * ia;
                    const double r = g.org[a] + ((double)(lo[a] + first + i) + 0.5) * h - ca;
                    s.sq[a][i] = x * x;
                    s.nsq[a][i] = (float)(x * x);
                    s.r[a][i] = r;
                    s.csq[a][i] = (float)(r * ia * (r * ia));
                    s.off[a][i] = wrap_int(lo[a] + first + i, g.n[a]);
                }
            };
            // a corner lies within del of its cell's centre in scaled
            // coordinates; the margin is far above the FP32 squares' rounding
            const float fa[3] = {(float)h * (float)bx.ia[0], (float)h * (float)bx.ia[1], (float)h * (float)bx.ia[2]};
            const float del = 0.5f * sqrtf(fa[0] * fa[0] + fa[1] * fa[1] + fa[2] * fa[2]) * 1.0001f + 1e-5f;
            const float in = 1.0f - del, out = 1.0f + del, nin = 1.0f - 2.0f * del, nout = 1.0f + 2.0f * del;
            const float in2 = in > 0.0f ? in * in * 0.9999f : -1.0f, out2 = out * out * 1.0001f;
            const float nin2 = nin > 0.0f ? nin * nin * 0.9999f : -1.0f, nout2 = nout * nout * 1.0001f;
            // append the lanes' flagged entries to the warp's list
            auto push = [&](uint16_t *list, int &cnt, bool flag, int code) {
                const unsigned b = __ballot_sync(0xffffffffu, flag);
                if (flag) list[cnt + __popc(b & ((1u << lane) - 1u))] = (uint16_t)code;
                cnt += __popc(b);
            };
            // run(entry) over the warps' lists end to end, 32 entries a warp
            auto run_lists = [&](int which, auto &&run) {
                int start = 0, w = 0, n = s.count[which][0];
                for (int e = threadIdx.x;; e += kVolThreads) {
                    while (w < kEllWarps && e >= start + n) {
                        start += n;
                        ++w;
                        n = w < kEllWarps ? s.count[which][w] : 0;
                    }
                    if (w == kEllWarps) break;
                    const int code = s.list[which][w][e - start];
                    run(code & 255, code >> 8);
                }
            };
            // the tables hold the z planes zt, ..., zt + kEllAx - 1
            int zt = z0;
            auto list_nodes = [&](int kn) {
                const float z2 = s.nsq[2][kn - zt];
                int cnt = 0;
                for (int i0 = 0; i0 < nx; i0 += 32) {
                    const int i = i0 + lane;
                    const float x2 = i < nx ? s.nsq[0][i] + z2 : -1.0f;
                    for (int j = warp; j < ny; j += kEllWarps) {
                        const float q = x2 + s.nsq[1][j];
                        push(s.list[0][warp], cnt, x2 >= 0.0f && q >= nin2 && q <= nout2, j << 8 | i);
                    }
                }
                if (lane == 0) s.count[0][warp] = cnt;
            };
            auto eval_nodes = [&](int kn) {
                double *const buf = s.plane[kn & 1];
                const double zz = s.sq[2][kn - zt];
                run_lists(0, [&](int i, int j) { buf[j * nx + i] = sqrt(s.sq[0][i] + s.sq[1][j] + zz) - 1.0; });
            };
            if (warp < 3) table(warp, warp == 2 ? z0 : 0);
            __syncthreads();
            list_nodes(z0);
            __syncthreads();
            eval_nodes(z0);
            __syncthreads();
            list_nodes(z0 + 1);
            __syncthreads();
            int inside = 0;  // cells of alpha 1
            for (int kz = z0; kz < z1; ++kz) {
                eval_nodes(kz + 1);
                const float z2 = s.csq[2][kz - zt];
                const double rz = s.r[2][kz - zt];
                const long long zrow = (long long)s.off[2][kz - zt] * g.n[1];
                // list the cut cells; sum a lane's cells of alpha 1 per column step
                int cuts = 0;
                for (int i0 = 0; i0 < dims[0]; i0 += 32) {
                    const int i = i0 + lane;
                    const bool cell = i < dims[0];
                    const float x2 = cell ? s.csq[0][i] + z2 : 0.0f;
                    const int ox = cell ? s.off[0][i] : 0;
                    double pu[3] = {0, 0, 0}, yu0 = 0.0, yu2 = 0.0;
                    const int before = inside;
                    for (int j = warp; j < dims[1]; j += kEllWarps) {
                        const float q = x2 + s.csq[1][j];
                        if (cell && q < in2) {
                            const long long cc = (zrow + s.off[1][j]) * g.n[0] + ox;
                            const double u0 = widened(u[cc]), u1 = widened(u[N + cc]), u2 = widened(u[2 * N + cc]);
                            const double ry = s.r[1][j];
                            pu[0] += u0, pu[1] += u1, pu[2] += u2;
                            yu0 = fma(ry, u0, yu0);
                            yu2 = fma(ry, u2, yu2);
                            ++inside;
                        }
                        push(s.list[1][warp], cuts, cell && q >= in2 && q <= out2, j << 8 | i);
                    }
                    if (inside != before) {
                        const double rx = s.r[0][i];
                        acc[0] += pu[0];
                        acc[1] += pu[1];
                        acc[2] += pu[2];
                        acc[3] += fma(-rz, pu[1], yu2);
                        acc[4] = fma(rz, pu[0], fma(-rx, pu[2], acc[4]));
                        acc[5] += fma(rx, pu[1], -yu0);
                    }
                }
                if (lane == 0) s.count[1][warp] = cuts;
                __syncthreads();
                const double *b0 = s.plane[kz & 1], *b1 = s.plane[(kz + 1) & 1];
                run_lists(1, [&](int i, int j) {
                    const int qn = j * nx + i;
                    const double ph[8] = {b0[qn], b0[qn + 1], b0[qn + nx], b0[qn + nx + 1],
                                          b1[qn], b1[qn + 1], b1[qn + nx], b1[qn + nx + 1]};
                    const double al = pvf_alpha8(ph);
                    if (al == 0.0) return;
                    const long long cc = (zrow + s.off[1][j]) * g.n[0] + s.off[0][i];
                    const double u0 = al * widened(u[cc]), u1 = al * widened(u[N + cc]),
                                 u2 = al * widened(u[2 * N + cc]);
                    const double rx = s.r[0][i], ry = s.r[1][j];
                    acc[0] += u0;
                    acc[1] += u1;
                    acc[2] += u2;
                    acc[3] = fma(ry, u2, fma(-rz, u1, acc[3]));
                    acc[4] = fma(rz, u0, fma(-rx, u2, acc[4]));
                    acc[5] = fma(rx, u1, fma(-ry, u0, acc[5]));
                    acc[6] += al;
                });
                if (kz + 1 < z1) {
                    if (kz + 2 - zt == kEllAx) {  // the next planes' table
                        __syncthreads();
                        zt = kz + 1;
                        if (warp == 2) table(2, zt);
                        __syncthreads();
                    }
                    list_nodes(kz + 2);
                }
                __syncthreads();
            }
            acc[6] += (double)inside;
        } else {
            const double c[3] = {bx.c[0], bx.c[1], bx.c[2]}, ia[3] = {bx.ia[0], bx.ia[1], bx.ia[2]};
            auto level = [&](int i, int j, int k) {  // node (lo + (i, j, k)): x_node = org + index h
                const double x = (g.org[0] + (double)(lo[0] + i) * h - c[0]) * ia[0];
                const double y = (g.org[1] + (double)(lo[1] + j) * h - c[1]) * ia[1];
                const double z = (g.org[2] + (double)(lo[2] + k) * h - c[2]) * ia[2];
                return sqrt(x * x + y * y + z * z) - 1.0;
            };
            for (int kz = z0; kz < z1; ++kz)
                for (int q = threadIdx.x; q < dims[0] * dims[1]; q += blockDim.x) {
                    const int j = q / dims[0], i = q - j * dims[0];
                    double ph[8];
#pragma unroll
                    for (int m = 0; m < 8; ++m) ph[m] = level(i + (m & 1), j + ((m >> 1) & 1), kz + ((m >> 2) & 1));
                    const double al = pvf_alpha8(ph);
                    if (al == 0.0) continue;
                    const long long cc = ((long long)wrap_int(lo[2] + kz, g.n[2]) * g.n[1] + wrap_int(lo[1] + j, g.n[1])) *
                                             g.n[0] + wrap_int(lo[0] + i, g.n[0]);
                    const double r[3] = {g.org[0] + ((double)(lo[0] + i) + 0.5) * h - c[0],
                                         g.org[1] + ((double)(lo[1] + j) + 0.5) * h - c[1],
                                         g.org[2] + ((double)(lo[2] + kz) + 0.5) * h - c[2]};
                    const double u0 = (double)u[cc], u1 = (double)u[N + cc], u2 = (double)u[2 * N + cc];
                    acc[0] += al * u0;
                    acc[1] += al * u1;
                    acc[2] += al * u2;
                    acc[3] += al * (r[1] * u2 - r[2] * u1);
                    acc[4] += al * (r[2] * u0 - r[0] * u2);
                    acc[5] += al * (r[0] * u1 - r[1] * u0);
                    acc[6] += al;
                }
        }
    }
    volume_finish(acc, g.h, p, split, nsplit, partial, done, Iu, Irxu, vol, s_phi);
}

// Drag diagnostic of Eq. FD: F_D = F_ib + rho_f (Iu^{n+1} - Iu^n) / dt.
__global__ void k_drag(int P, const double *__restrict__ Fib, const double *__restrict__ Iu_new,
                       const double *__restrict__ Iu_old, double rho_f, double dt, double *__restrict__ FD) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < 3 * P; q += gridDim.x * blockDim.x)
        FD[q] = Fib[q] + rho_f * (Iu_new[q] - Iu_old[q]) / dt;
}

// ---------------------------------------------------------------------------
// force and torque (Sec. 3.2.2): nsplit CTAs per particle, each summing a
// contiguous range of the particle's markers in FP64; with nsplit > 1 the
// particle's last CTA adds the CTAs' partial sums in CTA order (deterministic).
// FP64 issue (two operations per clock per SM) bounds these sums, so each
// particle's markers are spread over kFtSplit CTAs.  The split is a constant:
// a particle's sums do not depend on the other particles of the call (a
// request served alone equals the same request in a batch, bit for bit).
// ---------------------------------------------------------------------------
constexpr int kFtThreads = 256;
constexpr int kFtSplit = 4;
__global__ void __launch_bounds__(kFtThreads) k_force_torque(int P, int nsplit, const int *__restrict__ moff,
                                                             const double *__restrict__ R,
                                                             const double *__restrict__ dV,
                                                             const double *__restrict__ F, double rho_f,
                                                             double *__restrict__ partial,
                                                             unsigned int *__restrict__ done,
                                                             double *__restrict__ Fib, double *__restrict__ Tib) {
    const int p = blockIdx.x / nsplit, part = blockIdx.x % nsplit;
    if (p >= P) return;
    const int m0 = moff[p], nm = moff[p + 1] - m0;
    const int l0 = m0 + (int)((long long)part * nm / nsplit), l1 = m0 + (int)((long long)(part + 1) * nm / nsplit);
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int l = l0 + threadIdx.x; l < l1; l += blockDim.x) {
        double gx = F[3 * l] * dV[l], gy = F[3 * l + 1] * dV[l], gz = F[3 * l + 2] * dV[l];
        double rx = R[3 * l], ry = R[3 * l + 1], rz = R[3 * l + 2];
        acc[0] += gx;
        acc[1] += gy;
        acc[2] += gz;
        acc[3] += ry * gz - rz * gy;
        acc[4] += rz * gx - rx * gz;
        acc[5] += rx * gy - ry * gx;
    }
    block_sum<6, kFtThreads>(acc);
    if (threadIdx.x != 0) return;
    if (nsplit > 1) {
        // the particle's last CTA adds the partial sums in CTA order
        double *dst = partial + ((size_t)p * nsplit + part) * 6;
        for (int a = 0; a < 6; ++a) dst[a] = acc[a];
        __threadfence();  // release: partials before the count
        const bool last = atomicAdd(done + p, 1u) == (unsigned int)nsplit - 1;
        __threadfence();  // acquire: the count before the other partials
        if (!last) return;
        for (int a = 0; a < 6; ++a) acc[a] = 0.0;
        for (int k = 0; k < nsplit; ++k)
            for (int a = 0; a < 6; ++a) acc[a] += __ldcg(partial + ((size_t)p * nsplit + k) * 6 + a);
    }
    for (int a = 0; a < 3; ++a) {
        Fib[3 * p + a] = -rho_f * acc[a];
        Tib[3 * p + a] = -rho_f * acc[3 + a];
    }
}

// ---------------------------------------------------------------------------
// collision + Newton-Euler: one thread per particle, pairs in index order
// ---------------------------------------------------------------------------
struct CollideArgs {
    int P;
    CaseTab ct;  // pairs are taken within a case, in the case's periodic box
    double *Xr, *Ur, *Wr;
    const double *radius, *rho_p;
    double dt, inv_dt;  // inv_dt = 1 / dt, formed on the host
    const double *Fib, *Tib, *Iu_new, *Iu_old, *Ir_new, *Ir_old;
    double *Fc_out;
    double *Xnew;  // [P][3] scratch: positions are read by every thread
};

// One warp per particle i; lane k takes j = k, k + 32, ...; the lane partial
// sums are combined by a fixed shuffle tree (deterministic).
__global__ void k_collide_forces(CollideArgs a, double *__restrict__ Fc) {
    const int lane = threadIdx.x & 31;
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= a.P) return;
    const DevCase &cd = a.ct.of_particle(i);
    const ib_phys &ph = cd.phys;
    const double L[3] = {cd.g.n[0] * cd.g.h, cd.g.n[1] * cd.g.h, cd.g.n[2] * cd.g.h};
    const double iL[3] = {1.0 / L[0], 1.0 / L[1], 1.0 / L[2]};
    const double xi[3] = {a.Xr[3 * i], a.Xr[3 * i + 1], a.Xr[3 * i + 2]};
    const double Ri = a.radius[i];
    const double mi = a.rho_p[i] * 4.0 / 3.0 * kPi * Ri * Ri * Ri;
    const double idc = 1.0 / ph.d_c;
    const double gscale = 0.5 * ph.g_coll / ph.eps_c;
    double f[3] = {0, 0, 0};
    for (int j = cd.p0 + lane; j < cd.p1; j += 32) {
        if (j == i) continue;
        double del[3], d2 = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double dd = a.Xr[3 * j + k] - xi[k];
            del[k] = dd - L[k] * rint(dd * iL[k]);
            d2 += del[k] * del[k];
        }
        const double Rj = a.radius[j];
        const double Dc = Ri + Rj + ph.d_c;
        if (d2 < Dc * Dc && d2 > 0.0) {
            const double d = sqrt(d2);
            const double mj = a.rho_p[j] * 4.0 / 3.0 * kPi * Rj * Rj * Rj;
            const double q = (d - Dc) * idc;
            const double coef = -((mi + mj) * gscale) * q * q / d;
#pragma unroll
            for (int k = 0; k < 3; ++k) f[k] += coef * del[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
        for (int o = 16; o > 0; o >>= 1) f[k] += __shfl_down_sync(0xffffffffu, f[k], o);
    if (lane == 0)
        for (int k = 0; k < 3; ++k) Fc[3 * i + k] = f[k];
}

__global__ void k_newton_euler(CollideArgs a, const double *__restrict__ Fc, DevStatus *st) {
    grid_dep_wait();  // a programmatic dependent of the collision forces
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.P) return;
    const DevCase &cd = a.ct.of_particle(p);
    const ib_phys &ph = cd.phys;
    double Rp = a.radius[p];
    double V = 4.0 / 3.0 * kPi * Rp * Rp * Rp;
    double m = a.rho_p[p] * V;
    double I = 0.4 * m * Rp * Rp;
    // FP64 divisions are long instruction sequences on a part with two FP64
    // operations per clock per SM: 1/dt comes from the host, dt/m and dt/I
    // are formed once
    const double dtm = a.dt / m, dtI = a.dt / I;
    bool ok = true;
    for (int k = 0; k < 3; ++k) {
        double Un = a.Ur[3 * p + k];
        double rhs = a.Fib[3 * p + k] + ph.rho_f * (a.Iu_new[3 * p + k] - a.Iu_old[3 * p + k]) * a.inv_dt +
                     (a.rho_p[p] - ph.rho_f) * V * ph.g[k] + Fc[3 * p + k];
        double Unew = Un + dtm * rhs;
        double trq = a.Tib[3 * p + k] + ph.rho_f * (a.Ir_new[3 * p + k] - a.Ir_old[3 * p + k]) * a.inv_dt;
        double Wnew = a.Wr[3 * p + k] + dtI * trq;
        double Xnew = a.Xr[3 * p + k] + 0.5 * a.dt * (Unew + Un);
        ok = ok && isfinite(Unew) && isfinite(Wnew) && isfinite(Xnew);
        a.Ur[3 * p + k] = Unew;
        a.Wr[3 * p + k] = Wnew;
        a.Xr[3 * p + k] = Xnew;
        if (a.Fc_out) a.Fc_out[3 * p + k] = Fc[3 * p + k];
    }
    if (!ok) raise_status(st, IB_ERR_NONFINITE, p);
}

// CTAs per particle: the context's choice, or (0) as many as fill one resident
// wave of `kern` for P particles, within [1, kVolMaxSplit].
static int volume_split(ib_ctx *ctx, const void *kern, size_t smem, int P) {
    if (ctx->vol_split > 0) {
        resident_ctas(ctx, kern, kVolThreads, smem);  // (raises its shared memory limit)
        return ctx->vol_split;
    }
    const int per_sm = resident_ctas(ctx, kern, kVolThreads, smem);
    const long long n = (long long)(per_sm < 1 ? 1 : per_sm) * ctx->sm_count / (P > 0 ? P : 1);
    return (int)(n < 1 ? 1 : (n > kVolMaxSplit ? kVolMaxSplit : n));
}

template <typename T>
static int run_volume(ib_ctx *ctx, Arena &ar, const CaseTab &ct, const ib_particles *pp, double *Iu,
                      double *Irxu, double *vol, cudaStream_t s) {
    const int nsplit = volume_split(ctx, (const void *)k_volume<T>, kVolSmem, pp->P);
    double *partial = ar.take<double>((size_t)pp->P * nsplit * 7);
    unsigned int *done = ar.take<unsigned int>(pp->P);
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    PhaseTimer tm(ctx, IB_PHASE_VOLUME, s);
    cudaMemsetAsync(done, 0, sizeof(unsigned int) * pp->P, s);
    k_volume<T><<<pp->P * nsplit, kVolThreads, kVolSmem, s>>>(ct, pp->P, nsplit, pp->Xr, pp->radius, partial,
                                                               done, Iu, Irxu, vol, ctx->status);
    return check_launch("particle_volume_integrals");
}

// ---- allocation-free variant: scratch in a fixed device array -------------
// kVolSplit * 7 partial sums per particle for up to IB_STATIC_VOLUME_MAX_P
// particles (2048 * 8 * 7 doubles = 896 KiB).  Host code must not pass the
// array's name to a kernel (that is a host-side stand-in); the device address
// is looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) double g_volume_scratch[(size_t)IB_STATIC_VOLUME_MAX_P * kVolSplit * 7];
static __device__ DevStatus g_volume_status;
// completion counters of the final reduction; zero at load, reset by each call
static __device__ unsigned int g_volume_done[IB_STATIC_VOLUME_MAX_P];

constexpr int kMaxDevices = 64;
static std::mutex g_scratch_mu;
static double *g_scratch_ptr[kMaxDevices] = {};
static DevStatus *g_status_ptr[kMaxDevices] = {};
static unsigned int *g_done_ptr[kMaxDevices] = {};

static int static_scratch(double **scratch, DevStatus **status, unsigned int **done) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return set_error(IB_ERR_CUDA, "no current CUDA device");
    if (dev < 0 || dev >= kMaxDevices) return set_error(IB_ERR_UNSUPPORTED, "device id %d too large", dev);
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr, *q = nullptr, *r = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_volume_scratch);
        if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
        e = cudaGetSymbolAddress(&q, g_volume_status);
        if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "cudaGetSymbolAddress(status): %s", cudaGetErrorString(e));
        e = cudaGetSymbolAddress(&r, g_volume_done);
        if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "cudaGetSymbolAddress(done): %s", cudaGetErrorString(e));
        e = cudaFuncSetAttribute(k_volume<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVolSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_volume<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVolSmem);
        if (e != cudaSuccess) return set_error(IB_ERR_CUDA, "volume kernel attribute: %s", cudaGetErrorString(e));
        g_scratch_ptr[dev] = (double *)p;
        g_status_ptr[dev] = (DevStatus *)q;
        g_done_ptr[dev] = (unsigned int *)r;
    }
    *scratch = g_scratch_ptr[dev];
    *status = g_status_ptr[dev];
    *done = g_done_ptr[dev];
    return IB_OK;
}

template <typename T>
static int run_volume_static(const CaseTab &ct, const ib_particles *pp, double *Iu,
                             double *Irxu, double *vol, cudaStream_t s) {
    double *partial = nullptr;
    DevStatus *st = nullptr;
    unsigned int *done = nullptr;
    int rc = static_scratch(&partial, &st, &done);
    if (rc) return rc;
    k_volume<T><<<pp->P * kVolSplit, kVolThreads, kVolSmem, s>>>(ct, pp->P, kVolSplit, pp->Xr, pp->radius,
                                                                 partial, done, Iu, Irxu, vol, st);
    return check_launch("particle_volume_integrals_static");
}

template <typename T, int MODE>
static int run_volume_plan(ib_ctx *ctx, Arena &ar, const CaseTab &ct, const ib_particles *pp, int nsplit,
                           const PvfPlanDev &pl, double *Iu, double *Irxu, double *vol, cudaStream_t s) {
    double *partial = ar.take<double>((size_t)pp->P * nsplit * 7);
    unsigned int *done = ar.take<unsigned int>(pp->P);
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    PhaseTimer tm(ctx, IB_PHASE_VOLUME, s);
    cudaMemsetAsync(done, 0, sizeof(unsigned int) * pp->P, s);
    k_volume<T, MODE><<<pp->P * nsplit, kVolThreads, kVolSmem, s>>>(ct, pp->P, nsplit, pp->Xr, pp->radius, partial,
                                                                    done, Iu, Irxu, vol, ctx->status, pl);
    return check_launch("particle_volume_integrals_keep");
}

template <typename T>
static int run_plan_sums(ib_ctx *ctx, Arena &ar, const CaseTab &ct, const ib_particles *pp, const PvfPlanDev &pl,
                         double *Iu, double *Irxu, double *vol, cudaStream_t s) {
    const int nsplit = volume_split(ctx, (const void *)k_volume_plan<T>, 0, pp->P);
    double *partial = ar.take<double>((size_t)pp->P * nsplit * 7);
    unsigned int *done = ar.take<unsigned int>(pp->P);
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    PhaseTimer tm(ctx, IB_PHASE_VOLUME, s);
    cudaMemsetAsync(done, 0, sizeof(unsigned int) * pp->P, s);
    k_volume_plan<T><<<pp->P * nsplit, kVolThreads, 0, s>>>(ct, pp->P, nsplit, pp->Xr, pp->radius, partial,
                                                                    done, Iu, Irxu, vol, ctx->status, pl);
    return check_launch("particle_volume_integrals_plan");
}

}  // namespace gbib

using namespace gbib;

// The kept volume plan: device lists and the call it was kept for.
struct ib_pvf_plan {
    int device;
    int P, cap;
    int nsplit;     // CTAs per particle of the keeping call (0: not kept yet)
    ib_grid grid;   // the keeping call's grid
    void *mem;
    PvfPlanDev dev;
};

static bool same_grid(const ib_grid &a, const ib_grid &b) {
    return a.n[0] == b.n[0] && a.n[1] == b.n[1] && a.n[2] == b.n[2] && a.h == b.h && a.origin[0] == b.origin[0] &&
           a.origin[1] == b.origin[1] && a.origin[2] == b.origin[2] && a.prec == b.prec;
}

extern "C" {

int ib_pvf_plan_create(ib_ctx *ctx, int P, int max_box_cells, ib_pvf_plan **plan) {
    if (!ctx || !plan) return set_error(IB_ERR_INVALID, "NULL argument");
    *plan = nullptr;
    if (P < 1 || max_box_cells < 1 || max_box_cells > kVolMaxBox * kVolMaxBox * kVolMaxBox)
        return set_error(IB_ERR_INVALID, "bad plan size (P %d, max_box_cells %d)", P, max_box_cells);
    const size_t cap = (size_t)max_box_cells;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_hdr = up(sizeof(int2) * (size_t)P * kVolAx), b_bent = up(sizeof(unsigned) * P * cap),
                 b_alpha = up(sizeof(float2) * P * cap), b_pos = up(sizeof(double) * 4 * (size_t)P);
    ib_pvf_plan *pl = new (std::nothrow) ib_pvf_plan();
    if (!pl) return set_error(IB_ERR_OOM, "plan object");
    pl->device = ctx->device;
    pl->P = P;
    pl->cap = max_box_cells;
    pl->nsplit = 0;
    if (cudaMalloc(&pl->mem, b_hdr + b_bent + b_alpha + b_pos) != cudaSuccess) {
        cudaGetLastError();
        delete pl;
        return set_error(IB_ERR_OOM, "plan of %zu bytes", b_hdr + b_bent + b_alpha + b_pos);
    }
    char *m = (char *)pl->mem;
    pl->dev.cap = max_box_cells;
    pl->dev.hdr = (int2 *)m;
    pl->dev.bent = (unsigned *)(m + b_hdr);
    pl->dev.balpha = (float2 *)(m + b_hdr + b_bent);
    pl->dev.pos = (double *)(m + b_hdr + b_bent + b_alpha);
    *plan = pl;
    return IB_OK;
}

int ib_pvf_plan_destroy(ib_pvf_plan *plan) {
    if (!plan) return IB_OK;
    cudaDeviceSynchronize();
    cudaFree(plan->mem);
    delete plan;
    return IB_OK;
}

int particle_volume_integrals_keep(ib_ctx *ctx, const ib_grid *grid, const void *u, const ib_particles *parts,
                                   ib_pvf_plan *plan, double *Iu, double *Irxu, double *vol, void *stream) {
    if (!ctx || !plan) return set_error(IB_ERR_INVALID, "NULL argument");
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (!parts || parts->P < 0) return set_error(IB_ERR_INVALID, "bad particles");
    if (parts->P != plan->P) return set_error(IB_ERR_INVALID, "plan made for %d particles, not %d", plan->P, parts->P);
    if (!u || !parts->Xr || !parts->radius) return set_error(IB_ERR_INVALID, "NULL array");
    const CaseTab ct = single_case(grid, (void *)u, nullptr, parts->P);
    Arena ar(ctx);
    int nsplit;
    if (grid->prec == IB_F64)
        nsplit = volume_split(ctx, (const void *)k_volume<double, 1>, kVolSmem, parts->P);
    else
        nsplit = volume_split(ctx, (const void *)k_volume<float, 1>, kVolSmem, parts->P);
    plan->nsplit = nsplit;
    plan->grid = *grid;
    if (grid->prec == IB_F64)
        return run_volume_plan<double, 1>(ctx, ar, ct, parts, nsplit, plan->dev, Iu, Irxu, vol, (cudaStream_t)stream);
    return run_volume_plan<float, 1>(ctx, ar, ct, parts, nsplit, plan->dev, Iu, Irxu, vol, (cudaStream_t)stream);
}

int particle_volume_integrals_plan(ib_ctx *ctx, const ib_grid *grid, const void *u, const ib_particles *parts,
                                   const ib_pvf_plan *plan, double *Iu, double *Irxu, double *vol, void *stream) {
    if (!ctx || !plan) return set_error(IB_ERR_INVALID, "NULL argument");
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (!parts || parts->P != plan->P) return set_error(IB_ERR_INVALID, "plan made for %d particles", plan->P);
    if (plan->nsplit < 1) return set_error(IB_ERR_INVALID, "plan not kept yet");
    if (!same_grid(*grid, plan->grid)) return set_error(IB_ERR_INVALID, "grid differs from the plan's");
    if (!u || !parts->Xr || !parts->radius) return set_error(IB_ERR_INVALID, "NULL array");
    const CaseTab ct = single_case(grid, (void *)u, nullptr, parts->P);
    Arena ar(ctx);
    // any split: the plan holds each particle's cells
    if (grid->prec == IB_F64)
        return run_plan_sums<double>(ctx, ar, ct, parts, plan->dev, Iu, Irxu, vol, (cudaStream_t)stream);
    return run_plan_sums<float>(ctx, ar, ct, parts, plan->dev, Iu, Irxu, vol, (cudaStream_t)stream);
}

int particle_volume_integrals(ib_ctx *ctx, const ib_grid *grid, const void *u, const ib_particles *parts,
                              double *Iu, double *Irxu, double *vol, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (!parts || parts->P < 0) return set_error(IB_ERR_INVALID, "bad particles");
    if (parts->P == 0) return IB_OK;
    if (!u || !parts->Xr || !parts->radius) return set_error(IB_ERR_INVALID, "NULL array");
    if ((long long)parts->P * kVolMaxSplit > (1LL << 31) - 1) return set_error(IB_ERR_UNSUPPORTED, "too many particles");
    const CaseTab ct = single_case(grid, (void *)u, nullptr, parts->P);
    Arena ar(ctx);
    if (grid->prec == IB_F64)
        return run_volume<double>(ctx, ar, ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
    return run_volume<float>(ctx, ar, ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
}

int ib_batch_volume_integrals(ib_ctx *ctx, int ncases, const ib_case *cases, const ib_particles *parts,
                              double *Iu, double *Irxu, double *vol, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    if (!parts || parts->P < 0) return set_error(IB_ERR_INVALID, "bad particles");
    if (parts->P == 0) return IB_OK;
    if (!parts->Xr || !parts->radius || !Iu || !Irxu || !vol) return set_error(IB_ERR_INVALID, "NULL array");
    for (int c = 0; c < ncases && cases; ++c)
        if (!cases[c].u) return set_error(IB_ERR_INVALID, "case %d: NULL field", c);
    if ((long long)parts->P * kVolMaxSplit > (1LL << 31) - 1) return set_error(IB_ERR_UNSUPPORTED, "too many particles");
    Arena ar(ctx);
    CaseTab ct;
    int rc = build_case_table(ctx, ar, ncases, cases, parts->P, 1, ct, (cudaStream_t)stream);
    if (rc) return rc;
    if (cases[0].grid.prec == IB_F64)
        return run_volume<double>(ctx, ar, ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
    return run_volume<float>(ctx, ar, ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
}

int particle_volume_integrals_static(const ib_grid *grid, const void *u, const ib_particles *parts,
                                     double *Iu, double *Irxu, double *vol, void *stream) {
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (!parts || parts->P < 0) return set_error(IB_ERR_INVALID, "bad particles");
    if (parts->P > IB_STATIC_VOLUME_MAX_P)
        return set_error(IB_ERR_INVALID, "particle_volume_integrals_static: P = %d exceeds the fixed maximum %d",
                         parts->P, IB_STATIC_VOLUME_MAX_P);
    if (parts->P == 0) return IB_OK;
    if (!u || !parts->Xr || !parts->radius) return set_error(IB_ERR_INVALID, "NULL array");
    const CaseTab ct = single_case(grid, (void *)u, nullptr, parts->P);
    if (grid->prec == IB_F64)
        return run_volume_static<double>(ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
    return run_volume_static<float>(ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
}

int particle_volume_integrals_ellipsoid(ib_ctx *ctx, const ib_grid *grid, const void *u, int P, const double *Xr,
                                        const double *axes, double *Iu, double *Irxu, double *vol, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    int rc = validate_grid(grid, 1);
    if (rc) return rc;
    if (P < 0) return set_error(IB_ERR_INVALID, "P < 0");
    if (P == 0) return IB_OK;
    if (!u || !Xr || !axes || !Iu || !Irxu || !vol) return set_error(IB_ERR_INVALID, "NULL array");
    if ((long long)P * kVolMaxSplit > (1LL << 31) - 1) return set_error(IB_ERR_UNSUPPORTED, "too many particles");
    const CaseTab ct = single_case(grid, (void *)u, nullptr, P);
    Arena ar(ctx);
    const void *ek = grid->prec == IB_F64 ? (const void *)k_volume_ellipsoid<double> : (const void *)k_volume_ellipsoid<float>;
    const int nsplit = volume_split(ctx, ek, kEllSmem, P);
    double *partial = ar.take<double>((size_t)P * nsplit * 7);
    unsigned int *done = ar.take<unsigned int>(P);
    if (!ar.ok()) return oom_error(ar.used, ar.cap);
    cudaStream_t s = (cudaStream_t)stream;
    PhaseTimer tm(ctx, IB_PHASE_VOLUME, s);
    cudaMemsetAsync(done, 0, sizeof(unsigned int) * P, s);
    if (grid->prec == IB_F64) {
        k_volume_ellipsoid<double><<<P * nsplit, kVolThreads, kEllSmem, s>>>(ct, P, nsplit, Xr, axes, partial, done,
                                                                             Iu, Irxu, vol, ctx->status);
    } else {
        k_volume_ellipsoid<float><<<P * nsplit, kVolThreads, kEllSmem, s>>>(ct, P, nsplit, Xr, axes, partial, done,
                                                                            Iu, Irxu, vol, ctx->status);
    }
    return check_launch("particle_volume_integrals_ellipsoid");
}

int particle_drag_force(ib_ctx *ctx, int P, const double *F_ib, const double *Iu_new, const double *Iu_old,
                        double rho_f, double dt, double *F_D, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    if (P < 0) return set_error(IB_ERR_INVALID, "P < 0");
    if (!(dt > 0.0) || !isfinite(dt) || !isfinite(rho_f)) return set_error(IB_ERR_INVALID, "dt or rho_f invalid");
    if (P == 0) return IB_OK;
    if (!F_ib || !Iu_new || !Iu_old || !F_D) return set_error(IB_ERR_INVALID, "NULL array");
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (3 * P + 255) / 256;
    k_drag<<<nb < 1024 ? nb : 1024, 256, 0, s>>>(P, F_ib, Iu_new, Iu_old, rho_f, dt, F_D);
    return check_launch("particle_drag_force");
}

int particle_force_torque(ib_ctx *ctx, const ib_particles *parts, const ib_markers *marks, const double *F,
                          double rho_f, double *F_ib, double *T_ib, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    if (!parts || !marks || parts->P < 0 || marks->M < 0) return set_error(IB_ERR_INVALID, "bad arguments");
    if (!isfinite(rho_f)) return set_error(IB_ERR_INVALID, "rho_f not finite");
    if (parts->P == 0) return IB_OK;
    if (!parts->marker_offset || !F_ib || !T_ib || (marks->M > 0 && (!marks->R || !marks->dV || !F)))
        return set_error(IB_ERR_INVALID, "NULL array");
    const int P = parts->P, nsplit = kFtSplit;
    cudaStream_t s = (cudaStream_t)stream;
    Arena ar(ctx);
    double *partial = nsplit > 1 ? ar.take<double>((size_t)P * nsplit * 6) : nullptr;
    unsigned int *done = nsplit > 1 ? ar.take<unsigned int>(P) : nullptr;
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    PhaseTimer tm(ctx, IB_PHASE_FORCE, s);
    if (done) cudaMemsetAsync(done, 0, sizeof(unsigned int) * P, s);
    k_force_torque<<<P * nsplit, kFtThreads, 0, s>>>(P, nsplit, parts->marker_offset, marks->R, marks->dV, F, rho_f,
                                                   partial, done, F_ib, T_ib);
    return check_launch("particle_force_torque");
}

// Arguments shared by the single-case and batch forms; 1 = nothing to do.
static int check_collide_args(ib_ctx *ctx, const ib_particles *parts, const ib_phys *phys, double dt,
                              const double *F_ib, const double *T_ib, const double *Iu_new, const double *Iu_old,
                              const double *Irxu_new, const double *Irxu_old) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    if (!parts || !phys || parts->P < 0) return set_error(IB_ERR_INVALID, "bad arguments");
    if (!(dt > 0.0) || !isfinite(dt)) return set_error(IB_ERR_INVALID, "dt must be finite and > 0");
    if (!(phys->eps_c > 0.0) || !(phys->d_c > 0.0)) return set_error(IB_ERR_INVALID, "eps_c and d_c must be > 0");
    if (parts->P == 0) return 1;
    if (!parts->Xr || !parts->Ur || !parts->Wr || !parts->radius || !parts->rho_p || !F_ib || !T_ib ||
        !Iu_new || !Iu_old || !Irxu_new || !Irxu_old)
        return set_error(IB_ERR_INVALID, "NULL array");
    return IB_OK;
}

static int run_collide(ib_ctx *ctx, Arena &ar, const CaseTab &ct, ib_particles *parts,
                       double dt, const double *F_ib, const double *T_ib, const double *Iu_new,
                       const double *Iu_old, const double *Irxu_new, const double *Irxu_old, double *Fc_out,
                       cudaStream_t s) {
    double *Fc = ar.take<double>((size_t)3 * parts->P);
    if (!ar.ok())
        return oom_error(ar.used, ar.cap);
    CollideArgs a;
    a.P = parts->P;
    a.ct = ct;
    a.Xr = parts->Xr;
    a.Ur = parts->Ur;
    a.Wr = parts->Wr;
    a.radius = parts->radius;
    a.rho_p = parts->rho_p;
    a.dt = dt;
    a.inv_dt = 1.0 / dt;
    a.Fib = F_ib;
    a.Tib = T_ib;
    a.Iu_new = Iu_new;
    a.Iu_old = Iu_old;
    a.Ir_new = Irxu_new;
    a.Ir_old = Irxu_old;
    a.Fc_out = Fc_out;
    a.Xnew = nullptr;
    // one warp per CTA: both kernels are FP64-issue bound (two operations per
    // clock per SM), so the particles' warps are spread over as many SMs
    PhaseTimer tm(ctx, IB_PHASE_COLLIDE, s);
    k_collide_forces<<<parts->P, 32, 0, s>>>(a, Fc);
    launch_pdl(k_newton_euler, dim3((parts->P + 31) / 32), dim3(32), 0, s, a, (const double *)Fc, ctx->status);
    return check_launch("particle_collide_update");
}

int particle_collide_update(ib_ctx *ctx, ib_particles *parts, const ib_grid *grid, const ib_phys *phys,
                            double dt, const double *F_ib, const double *T_ib, const double *Iu_new,
                            const double *Iu_old, const double *Irxu_new, const double *Irxu_old,
                            double *Fc_out, void *stream) {
    int rc = check_collide_args(ctx, parts, phys, dt, F_ib, T_ib, Iu_new, Iu_old, Irxu_new, Irxu_old);
    if (rc) return rc == 1 ? IB_OK : rc;
    rc = validate_grid(grid, 0);
    if (rc) return rc;
    CaseTab ct = single_case(grid, nullptr, nullptr, parts->P);
    ct.one.phys = *phys;
    Arena ar(ctx);
    return run_collide(ctx, ar, ct, parts, dt, F_ib, T_ib, Iu_new, Iu_old, Irxu_new, Irxu_old, Fc_out,
                       (cudaStream_t)stream);
}

int ib_batch_table_volume_integrals(ib_ctx *ctx, const ib_batch_table *table, const ib_particles *parts,
                                    double *Iu, double *Irxu, double *vol, void *stream) {
    if (!ctx) return set_error(IB_ERR_INVALID, "ctx is NULL");
    if (!parts || parts->P < 0) return set_error(IB_ERR_INVALID, "bad particles");
    CaseTab ct;
    int rc = table_cases(table, parts->P, ct);
    if (rc) return rc;
    if (parts->P == 0) return IB_OK;
    if (!parts->Xr || !parts->radius || !Iu || !Irxu || !vol) return set_error(IB_ERR_INVALID, "NULL array");
    if ((long long)parts->P * kVolMaxSplit > (1LL << 31) - 1) return set_error(IB_ERR_UNSUPPORTED, "too many particles");
    Arena ar(ctx);
    if (table->prec == IB_F64) return run_volume<double>(ctx, ar, ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
    return run_volume<float>(ctx, ar, ct, parts, Iu, Irxu, vol, (cudaStream_t)stream);
}

int ib_batch_table_collide_update(ib_ctx *ctx, const ib_batch_table *table, ib_particles *parts, double dt,
                                  const double *F_ib, const double *T_ib, const double *Iu_new,
                                  const double *Iu_old, const double *Irxu_new, const double *Irxu_old,
                                  double *Fc_out, void *stream) {
    if (table && !table->has_phys) return set_error(IB_ERR_INVALID, "the table was created without physical parameters");
    const ib_phys *ph = table ? &table->ct.one.phys : nullptr;
    int rc = check_collide_args(ctx, parts, ph, dt, F_ib, T_ib, Iu_new, Iu_old, Irxu_new, Irxu_old);
    if (rc) return rc == 1 ? IB_OK : rc;
    CaseTab ct;
    rc = table_cases(table, parts->P, ct);
    if (rc) return rc;
    Arena ar(ctx);
    return run_collide(ctx, ar, ct, parts, dt, F_ib, T_ib, Iu_new, Iu_old, Irxu_new, Irxu_old, Fc_out,
                       (cudaStream_t)stream);
}

int ib_batch_collide_update(ib_ctx *ctx, int ncases, const ib_case *cases, ib_particles *parts,
                            const ib_phys *phys, double dt, const double *F_ib, const double *T_ib,
                            const double *Iu_new, const double *Iu_old, const double *Irxu_new,
                            const double *Irxu_old, double *Fc_out, void *stream) {
    int rc = check_collide_args(ctx, parts, phys, dt, F_ib, T_ib, Iu_new, Iu_old, Irxu_new, Irxu_old);
    if (rc) return rc == 1 ? IB_OK : rc;
    Arena ar(ctx);
    CaseTab ct;
    for (int c = 0; c < ncases && cases; ++c)
        if (!(phys[c].eps_c > 0.0) || !(phys[c].d_c > 0.0))
            return set_error(IB_ERR_INVALID, "case %d: eps_c and d_c must be > 0", c);
    rc = build_case_table(ctx, ar, ncases, cases, parts->P, 0, ct, (cudaStream_t)stream, phys);
    if (rc) return rc;
    return run_collide(ctx, ar, ct, parts, dt, F_ib, T_ib, Iu_new, Iu_old, Irxu_new, Irxu_old, Fc_out,
                       (cudaStream_t)stream);
}

}  // extern "C"
