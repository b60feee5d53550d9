// vp_fused.cu -- one-pass step: [Lambda_p^{-1}] + push + deposit + [Lambda_x^{-1}].
//
// Sec. III update w_fin = Lambda^{-1} Delta^T w_in with Lambda = Lambda_x (x) Lambda_p
// (tent basis). In cubic B-spline Galerkin mode the library keeps, between
// steps, s = Lambda_x^{-1} r where r = Delta^T w is the deposit; one step is then
//   w  = Lambda_p^{-1} s         (per column, on the source side)
//   r' = Delta^T w               (push every node, deposit with the B3 kernel)
//   s' = Lambda_x^{-1} r'        (per row, on the destination side)
// so each step reads and writes the mesh once. With the tent deposit or the
// lumped projection there is no solve and the state is w itself.
//
// One CTA owns one destination tile [X0, X0+TX) x [P0, P0+TP). It keeps a
// shared-memory window: the tile widened by the x-solve halo D and a guard
// band G. It bounds the source nodes whose pushed B3 footprint reaches the
// widened tile. FP32: each thread takes a pair of adjacent source columns through a segment
// of those rows in packed arithmetic (vp_walk.cuh). FP64: each thread takes one column:
//   * Galerkin: the p solve is the Thomas algorithm for tridiag(1/6, 2/3, 1/6)
//     (exact pivots near row 0), walked downwards in chunks of rows: the
//     forward sweep of a chunk starts kHalo rows below it (truncation
//     |z|^kHalo, z = sqrt(3) - 2) and is kept in a shared-memory column buffer;
//     the back substitution carries on from the chunk above;
//   * every node is pushed (displacement tables, vp_internal.h) and its N x N
//     taps accumulate in an N x N register ring that follows the node's base
//     row; when the ring moves one row, the row that leaves it is added to the
//     window with N shared-memory atomics.
// Contributions outside the window belong to other tiles, except rows beyond
// an open momentum edge, which are counted as lost by the tile that owns the edge
// row in that column. Finally each warp takes window rows, solves Lambda_x along them
// (first-order recurrences over per-lane chunks; a lane's carry comes from the chunks
// next to it, in FP64 rows of other lengths from a warp scan), and the
// tile is stored once.
#include <math.h>

#include "vp_fel.cuh"
#include "vp_internal.h"
#include "vp_sum.cuh"
#include "vp_walk.cuh"
#include "vp_walk64.cuh"

namespace vp {
namespace {

// look-ahead / x-solve halo: |z|^16 = 7e-10 (FP32; also keeps stores 16-byte aligned),
// |z|^28 = 1e-16 (FP64)
template <typename T>
struct Halo {
    static constexpr int value = sizeof(T) == 4 ? 16 : 28;
};
constexpr int kMaxGroups = 16;      // groups of 64 source columns whose rows are bounded on their own
constexpr int kSumWarps = 8;        // virtual warps of the per-tile FEL column sums
constexpr int kMinSegRows = 8;      // shortest row segment of the FP32 walk (each restarts its rings)
// elements of the per-thread column buffer: one chunk of rows; FP32 threads walk two columns
template <typename T>
struct GRows {
    static constexpr int value = sizeof(T) == 4 ? 2 * kC32 : kC64;
};
constexpr int kXBig = kFusedMaxRow / 32;   // elements per lane for rows up to kFusedMaxRow
constexpr int kXBig32 = 20;                // FP32: whole-period rows of kFusedMaxRow with the halo on both sides

__device__ __forceinline__ int imod(int a, int n)
{
    int r = a % n;
    return r < 0 ? r + n : r;
}

// z^n for the pole z = sqrt(3) - 2 < 0
template <typename T>
__device__ __forceinline__ T zpow(int n);

template <>
__device__ __forceinline__ float zpow<float>(int n)
{
    // log2|z| = log2(2 - sqrt(3))
    const float m = exp2f((float)n * -1.8999686269529425f);
    return (n & 1) ? -m : m;
}

template <>
__device__ __forceinline__ double zpow<double>(int n)
{
    const double m = exp2((double)n * -1.8999686269529425);
    return (n & 1) ? -m : m;
}

// range of sin over [lo, hi] in FP32 (|lo|, |hi| < 1e3), widened by 1e-4
__device__ void sin_range32(float lo, float hi, float &smin, float &smax)
{
    const float twopi = 6.28318530717958647692f;
    if (hi - lo >= twopi - 1e-4f) {
        smin = -1.f;
        smax = 1.f;
        return;
    }
    const float k = floorf(lo / twopi);
    const float a = lo - k * twopi, b = hi - k * twopi;
    const float sa = sinf(a), sb = sinf(b);
    smin = fminf(sa, sb) - 1e-4f;
    smax = fmaxf(sa, sb) + 1e-4f;
    const float h1 = 1.57079632679f, h3 = 4.71238898038f;
    if ((a <= h1 + 1e-4f && h1 - 1e-4f <= b) || (a <= h1 + twopi + 1e-4f && h1 + twopi - 1e-4f <= b))
        smax = 1.f;
    if ((a <= h3 + 1e-4f && h3 - 1e-4f <= b) || (a <= h3 + twopi + 1e-4f && h3 + twopi - 1e-4f <= b))
        smin = -1.f;
}

// Window cells. FP32: fixed-point integers at a per-tile scale, so that the deposit uses
// native integer shared-memory atomics (a float atomicAdd on shared memory is a
// compare-and-swap loop) and the sums do not depend on the order of the additions: the
// FP32 step is bit-reproducible. FP64: doubles.
// raw cell value (in the tile's scaled units)
__device__ __forceinline__ double wraw(const float *p) { return (double)*reinterpret_cast<const int *>(p); }
__device__ __forceinline__ double wraw(const double *p) { return *p; }
// cell value in weight units
__device__ __forceinline__ float wget(const float *p, float iq)
{
    return (float)*reinterpret_cast<const int *>(p) * iq;
}
__device__ __forceinline__ double wget(const double *p, double) { return *p; }
__device__ __forceinline__ void wfold(float *d, const float *s)
{
    *reinterpret_cast<int *>(d) += *reinterpret_cast<const int *>(s);
}
__device__ __forceinline__ void wfold(double *d, const double *s) { *d += *s; }

struct WinGeom {
    int WW, WH, ws;      // window width, height, row stride (elements)
    int WX0, WP0;        // grid column (unwrapped) and row of window cell (0, 0)
    int own_c0, own_c1;  // the tile's own columns, window coordinates [c0, c1)
    int np, nx;
    bool full;           // the tile spans the whole period
};

constexpr double kXScale64 = -6.0 * -0.26794919243112270647;   // -6 z, after the two recursions
// padded staging layout of a row: element c at c + c / 8, so that lanes reading
// contiguous chunks of 8 hit distinct shared-memory banks
__device__ __forceinline__ int padc(int c) { return c + (c >> 3); }

// FP64 Lambda_x^{-1} (T x = row, T = tridiag(1/6, 2/3, 1/6)) of one row of length L held in
// shared memory, by one warp. Returns each lane's elements base .. base + per - 1 in v.
// cyclic: the row is one whole period; else the row is padded by the halo on both
// sides and the recurrences start from zero at its ends (truncation |z|^halo).
template <int kXMax>
__device__ void solve_row_x(const double *row, int L, bool cyclic, int lane, double *v, int &per, int &base, bool padded)
{
    per = (L + 31) / 32;
    base = lane * per;
    const double z = -0.26794919243112270647;
#pragma unroll
    for (int k = 0; k < kXMax; ++k)
        v[k] = (k < per && base + k < L) ? row[padded ? padc(base + k) : base + k] : 0.0;
    const double zper = zpow<double>(per);
    // causal y_i = x_i + z y_{i-1}: lane-local sweep, then carries by a warp scan
    double y = 0.0;
#pragma unroll
    for (int k = 0; k < kXMax; ++k)
        if (k < per) {
            y = v[k] + z * y;
            v[k] = y;
        }
    double endv = y;
    double zp = zper;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, endv, off);
        if (lane >= off) endv += zp * o;
        zp *= zp;
    }
    double carry = __shfl_up_sync(0xffffffffu, endv, 1);
    if (lane == 0) carry = 0.0;
    {
        double zk = z;
#pragma unroll
        for (int k = 0; k < kXMax; ++k)
            if (k < per) {
                v[k] += zk * carry;
                zk *= z;
            }
    }
    if (cyclic) {
        // y_{-1} = y_{L-1}: with E the zero-start value at L-1, y_{-1} = E / (1 - z^L)
        const int ll = (L - 1) / per, kl = (L - 1) - ll * per;
        double mine = 0.0;
#pragma unroll
        for (int k = 0; k < kXMax; ++k)
            if (k == kl) mine = v[k];
        const double E = __shfl_sync(0xffffffffu, mine, ll);
        const double yprev = E / (1.0 - zpow<double>(L));
        double zk = zpow<double>(base + 1);
#pragma unroll
        for (int k = 0; k < kXMax; ++k)
            if (k < per) {
                v[k] += zk * yprev;
                zk *= z;
            }
    }
    // anticausal u_i = y_i + z u_{i+1}
    int last = per - 1;
    if (base + last >= L) last = L - 1 - base;   // may be negative for idle lanes
    double u = 0.0;
#pragma unroll
    for (int k = kXMax - 1; k >= 0; --k)
        if (k <= last) {
            u = v[k] + z * u;
            v[k] = u;
        }
    double startv = u;
    zp = zper;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = __shfl_down_sync(0xffffffffu, startv, off);
        if (lane + off < 32) startv += zp * o;
        zp *= zp;
    }
    double carry2 = __shfl_down_sync(0xffffffffu, startv, 1);
    if (lane == 31) carry2 = 0.0;
    {
        double zk = z;
#pragma unroll
        for (int k = kXMax - 1; k >= 0; --k)
            if (k <= last) {
                v[k] += zk * carry2;
                zk *= z;
            }
    }
    if (cyclic) {
        // u_L = u_0: with S the zero-end value at 0, u_L = S / (1 - z^L)
        const double S = __shfl_sync(0xffffffffu, v[0], 0);
        const double unext = S / (1.0 - zpow<double>(L));
        // element i gets z^{L - i} u_L
#pragma unroll
        for (int k = 0; k < kXMax; ++k)
            if (k <= last) v[k] += zpow<double>(L - (base + k)) * unext;
    }
#pragma unroll
    for (int k = 0; k < kXMax; ++k) v[k] *= kXScale64;
}

// z^n for the pole z = sqrt(3) - 2, at compile time
constexpr double zconst(int n)
{
    double r = 1.0;
    for (int k = 0; k < n; ++k) r *= -0.26794919243112270647;
    return r;
}

// Lambda_x^{-1} of one window row of exactly 32 KX elements (the common case of the
// windowed tiles): the recurrences start from zero at both row ends and every power of z
// the lane sweeps and the carries need is a compile-time constant. row == nullptr: v
// already holds the lane's KX elements.
// A lane's carry is the recurrence value at the end of the chunks next to it. Where the
// halo spans at most three chunks it sums only those chunks' zero-start end values (two
// or three shuffles, no scan): what it leaves out is weighted by |z|^halo or less, the
// truncation the recurrences already have at the window ends.
template <typename T, int KX>
__device__ __forceinline__ void solve_row_x_exact(const T *row, int lane, T *v, bool padded, T sh,
                                                  T sl)
{
    const int base = lane * KX;
    const T z = (T)zconst(1);
    if (row)
#pragma unroll
        for (int k = 0; k < KX; ++k) v[k] = row[padded ? padc(base + k) : base + k];
    // causal y_i = x_i + z y_{i-1}: lane-local, then the carry of the lanes below
    T y = T(0);
#pragma unroll
    for (int k = 0; k < KX; ++k) {
        y = v[k] + z * y;
        v[k] = y;
    }
    T endv = y;
    T carry = T(0);
    constexpr int NCH = (Halo<T>::value + KX - 1) / KX;
    if constexpr (NCH <= 3) {
#pragma unroll
        for (int c = 1; c <= NCH; ++c) {
            const T o = __shfl_up_sync(0xffffffffu, endv, c);
            if (lane >= c) carry += (T)zconst((c - 1) * KX) * o;
        }
    } else {
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            const T o = __shfl_up_sync(0xffffffffu, endv, 1 << s);
            if (lane >= (1 << s)) endv += (T)zconst(KX << s) * o;
        }
        carry = __shfl_up_sync(0xffffffffu, endv, 1);
        if (lane == 0) carry = T(0);
    }
#pragma unroll
    for (int k = 0; k < KX; ++k) v[k] += (T)zconst(k + 1) * carry;
    // anticausal u_i = y_i + z u_{i+1}
    T u = T(0);
#pragma unroll
    for (int k = KX - 1; k >= 0; --k) {
        u = v[k] + z * u;
        v[k] = u;
    }
    T startv = u;
    T carry2 = T(0);
    if constexpr (NCH <= 3) {
#pragma unroll
        for (int c = 1; c <= NCH; ++c) {
            const T o = __shfl_down_sync(0xffffffffu, startv, c);
            if (lane + c < 32) carry2 += (T)zconst((c - 1) * KX) * o;
        }
    } else {
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            const T o = __shfl_down_sync(0xffffffffu, startv, 1 << s);
            if (lane + (1 << s) < 32) startv += (T)zconst(KX << s) * o;
        }
        carry2 = __shfl_down_sync(0xffffffffu, startv, 1);
        if (lane == 31) carry2 = T(0);
    }
#pragma unroll
    for (int k = 0; k < KX; ++k) v[k] += (T)zconst(KX - k) * carry2;
#pragma unroll
    for (int k = 0; k < KX; ++k) v[k] = sizeof(T) == 4 ? v[k] * sh + v[k] * sl : v[k] * sh;
}

}  // namespace

// The window's own cells in weight units into the destination rows: one warp per row, FP32 rows
// with 16-byte loads of the fixed-point cells and 16-byte stores where the destination row allows.
// MAX: track max|value| in om (the stored state's per-tile maximum) and flag non-finite values
// (FP64 cells; FP32 cells are integers times a finite scale).
template <typename T, bool MAX>
__device__ __forceinline__ void store_window_rows(const T *win, const WinGeom &W, T *dst, int nx, int P0,
                                                  int X0, int TXe, int TPe, int G, int Gp, T iq, int warp,
                                                  int nwarps, int lane, float &om, bool &bad)
{
    for (int rr = warp; rr < TPe; rr += nwarps) {
        const T *row = win + (size_t)(rr + Gp) * W.ws + G;
        T *drow = dst + (size_t)(P0 + rr) * nx + X0;
        int c0 = 0;
        if constexpr (sizeof(T) == 4) {
            if ((reinterpret_cast<uintptr_t>(drow) & 15) == 0) {
                const int n4 = TXe >> 2;
                const int4 *r4 = reinterpret_cast<const int4 *>(row);
                float4 *d4 = reinterpret_cast<float4 *>(drow);
                for (int c4 = lane; c4 < n4; c4 += 32) {
                    const int4 q = r4[c4];
                    const float4 o = make_float4((float)q.x * iq, (float)q.y * iq, (float)q.z * iq, (float)q.w * iq);
                    d4[c4] = o;
                    if (MAX) om = fmaxf(om, fmaxf(fmaxf(fabsf(o.x), fabsf(o.y)), fmaxf(fabsf(o.z), fabsf(o.w))));
                }
                c0 = n4 << 2;
            }
        }
        for (int c = c0 + lane; c < TXe; c += 32) {
            const T v = wget(row + c, iq);
            drow[c] = v;
            if (MAX) {
                om = fmaxf(om, fabsf((float)v));
                bad |= !isfinite(v);
            }
        }
    }
}

// FP64: Lambda_x solve of the tile's window rows (one warp per row) and the tile store.
template <int KX>
__device__ __forceinline__ void solve_rows_f64(double *win, const WinGeom &W, double *dst, int L, bool full, int D, int G,
                                               int Gp, int TXe, int TPe, int P0, int X0, int nx, bool want_part, int warp,
                                               int nwarps, int lane, bool &bad, double *stage_all, int stage_len)
{
    // per-warp padded copy of the row (conflict-free reads of contiguous chunks)
    const int plen = padc(L) + 8;
    const bool use_stage = (size_t)nwarps * plen <= (size_t)stage_len;
    double *stage = stage_all + (size_t)warp * plen;
    for (int rr = warp; rr < TPe; rr += nwarps) {
        double *row = win + (size_t)(rr + Gp) * W.ws + G;
        double *dst_row = dst + (size_t)(P0 + rr) * nx + X0 - D;
        double v[KX];
        int per, base;
        const bool exact = !full && L == 32 * KX;
        if (use_stage)
            for (int c = lane; c < L; c += 32) stage[padc(c)] = row[c];
        __syncwarp();
        const double *from = use_stage ? stage : row;
        if (exact) {
            solve_row_x_exact<double, KX>(from, lane, v, use_stage, kXScale64, 0.0);
            per = KX;
            base = lane * KX;
        } else {
            solve_row_x<KX>(from, L, full, lane, v, per, base, use_stage);
        }
        __syncwarp();
        double chk = 0.0;   // v * 0 is 0 for finite values and NaN otherwise
        if (!(exact && (base + KX <= D || base >= D + TXe))) {
            // (lanes whose chunk lies in the halo store nothing)
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                const int c = base + k;
                if (k < per && c >= D && c < D + TXe) {
                    dst_row[c] = v[k];
                    chk = fma(v[k], 0.0, chk);
                    if (want_part) row[c] = v[k];   // keep s for the column sums
                }
            }
        }
        bad |= chk != 0.0;
    }
}

// FP32: Lambda_x solve of the tile's window rows and the tile store, one warp per row, always as a row of
// 32 KX elements (every power of z a compile-time constant): the tile's own columns with at least the halo
// on both sides. Window columns beyond the widened tile hold partial deposits or zeros; what they change in
// the own columns weighs |z|^17 or less, the truncation of the halo. Whole-period rows take their halo from
// the period's other end. (A row of another length through run-time chunk lengths cost 2700 cycles against
// about 300.)
template <int KX>
__device__ __forceinline__ void solve_rows_f32(float *win, const WinGeom &W, float *dst, bool full, int G, int Gp, int TXe,
                                               int TPe, int P0, int X0, int nx, bool want_part, int warp,
                                               int nwarps, int lane, float sh, float sl, float iq, float &om, bool &bad)
{
    constexpr int D = Halo<float>::value;
    static_assert(KX % 4 == 0, "chunks are read 16 bytes at a time");
    // element e of the row is window column e + o; the own columns start at element s
    const int o = full ? 0 : (W.own_c0 + TXe + D <= 32 * KX ? 0 : W.own_c0 - D);
    const int s = full ? D : W.own_c0 - o;
    const int base = lane * KX;
    int w0 = base - D;   // whole period: first column of the lane's chunk, wrapped
    if (full) w0 = imod(w0, nx);
    for (int rr = warp; rr < TPe; rr += nwarps) {
        float *row = win + (size_t)(rr + Gp) * W.ws;
        float v[KX];
        if (full) {
            const int *cell = reinterpret_cast<const int *>(row + G);
            int c = w0;
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                v[k] = base + k < nx + 2 * D ? (float)cell[c] * iq : 0.f;
                if (++c == nx) c = 0;
            }
        } else {
            const int4 *r4 = reinterpret_cast<const int4 *>(row + o + base);
#pragma unroll
            for (int k4 = 0; k4 < KX / 4; ++k4) {
                const int4 q = base + o + 4 * k4 < W.ws ? r4[k4] : make_int4(0, 0, 0, 0);
                v[4 * k4 + 0] = (float)q.x * iq;
                v[4 * k4 + 1] = (float)q.y * iq;
                v[4 * k4 + 2] = (float)q.z * iq;
                v[4 * k4 + 3] = (float)q.w * iq;
            }
        }
        if (want_part) __syncwarp();   // the row is read before any of it is overwritten below
        solve_row_x_exact<float, KX>(nullptr, lane, v, false, sh, sl);
        float *dp = dst + (size_t)(P0 + rr) * nx + X0 + base - s;
        float *keep = row + (full ? G + base - s : o + base);
        if (base >= s && base + KX <= s + TXe && (reinterpret_cast<uintptr_t>(dp) & 15) == 0) {
#pragma unroll
            for (int k = 0; k < KX; k += 4) {
                const float4 q = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
                *reinterpret_cast<float4 *>(dp + k) = q;
                om = fmaxf(om, fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
            }
            // keep s for the column sums
            if (want_part)
#pragma unroll
                for (int k = 0; k < KX; ++k) keep[k] = v[k];
        } else if (base < s + TXe && base + KX > s) {
#pragma unroll
            for (int k = 0; k < KX; ++k)
                if (base + k >= s && base + k < s + TXe) {
                    dp[k] = v[k];
                    om = fmaxf(om, fabsf(v[k]));
                    if (want_part) keep[k] = v[k];
                }
        }
        float chk = 0.f;   // v * 0 is 0 for finite values and NaN otherwise
#pragma unroll
        for (int k = 0; k < KX; ++k) chk = fmaf(v[k], 0.f, chk);
        bad |= chk != 0.f;
    }
}

// Rows of [ja, jb] from which the columns c0 .. c1 (unwrapped, up to nx of them) can reach the widened tile, by one
// warp: the bounds of the tile's source rectangle for these columns alone. Called where the rectangle is much
// taller than the tile: strong shear along p, or columns across the period of a force that is not periodic. period: the
// tile walks one whole period of columns, each for all its images.
template <typename T>
__device__ __forceinline__ int2 rows_of_columns(const FusedArgs<T> &A, int c0, int c1, int ja, int jb, int X0, int TXe, int P0,
                                             int TPe, int D, int R, float Mf, float phif, bool period)
{
    const Geometry &g = A.g;
    const float SL = 0.05f;
    const float EU = fabsf((float)g.KU) * Mf, EV = fabsf((float)g.KV) * Mf, KVM = (float)g.KV * Mf;
    const float acc_lo = P0 == 0 ? -1e30f : (float)(P0 - R), acc_hi = P0 + TPe == g.np ? 1e30f : (float)(P0 + TPe - 1 + R);
    const int lane = threadIdx.x & 31;
    float vcl = 1e30f, vch = -1e30f;
    for (int c = c0 + lane; c <= c1; c += 32) {
        const float2 vb = A.vcbf[imod(c, g.nx) / kColBlock];
        vcl = fminf(vcl, vb.x);
        vch = fmaxf(vch, vb.y);
    }
    for (int o = 16; o > 0; o >>= 1) {
        vcl = fminf(vcl, __shfl_xor_sync(0xffffffffu, vcl, o));
        vch = fmaxf(vch, __shfl_xor_sync(0xffffffffu, vch, o));
    }
    int lo = 0x7fffffff, hi = -0x7fffffff;
    for (int j = ja + lane; j <= jb; j += 32) {
        const float4 rb = A.rowbf[j];   // u, v, y
        float tlo = 0.f, thi = 0.f;
        if (EV > 0.f) {
            float smin, smax;
            const float x0f = (float)g.x0, hxf = (float)g.hx, padf = (float)g.a_pad;
            sin_range32(x0f + c0 * hxf - padf + rb.z + phif, x0f + c1 * hxf + padf + rb.z + phif, smin, smax);
            tlo = fminf(KVM * smin, KVM * smax);
            thi = fmaxf(KVM * smin, KVM * smax);
        }
        const float vlo = (float)j + rb.y + vcl + tlo - SL, vhi = (float)j + rb.y + vch + thi + SL;
        const int ia = (int)floorf((float)(X0 - D - R) - rb.x - EU - (float)g.uc_max - SL);
        const int ib = (int)ceilf((float)(X0 + TXe + D - 1 + R) - rb.x + EU - (float)g.uc_min + SL);
        bool reach = A.full_row || (c0 <= ib && c1 >= ia);
        if (period && !reach)   // an image of c0 in [ia, ib], or one of ia in [c0, c1]
            reach = ib - ia + 1 >= g.nx || imod(c0 - ia, g.nx) <= ib - ia || imod(ia - c0, g.nx) <= c1 - c0;
        if (vhi > acc_lo && vlo < acc_hi && reach) {
            lo = min(lo, j);
            hi = max(hi, j);
        }
    }
    return make_int2(__reduce_min_sync(0xffffffffu, lo), __reduce_max_sync(0xffffffffu, hi));
}

// Programmatic dependent launch: a step's CTAs may start, and clear their windows, while the launch before them
// in the stream ends; here they wait until it has completed and its writes are visible, then let the launch after
// them start in turn (it waits at the same place). Without the launch attribute both are no-ops. What it hides is
// the launch and its first microsecond: a step of 357 x 300 nodes 22.9 -> 21.2 us, of 2048 x 2048 46.5 -> 45.3.
__device__ __forceinline__ void after_previous_launch()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// One destination tile of one simulation (A may live in shared or global memory).
template <typename T, int BASIS, bool GAL, bool UTERM>
__device__ __forceinline__ void fused_tile(const FusedArgs<T> &A, const int tile,
                                           unsigned char *smem_raw)
{
    constexpr int R = (BASIS == VP_BASIS_TENT) ? 1 : 2;
    T *win = reinterpret_cast<T *>(smem_raw);
    T *gcol = win + (size_t)A.ws * (A.tp + 2 * A.Gp);   // [GRows][blockDim] column buffer (Galerkin)
    // row cache: the tile's rows ja .. jb of the push's row table (when they fit)
    RowEntry<T> *rowc = reinterpret_cast<RowEntry<T> *>(gcol + (size_t)GRows<T>::value * blockDim.x);
    __shared__ int s_ia, s_ib, s_ja, s_jb, s_omax;
    __shared__ double s_part[3][kSumWarps], s_lost[kFusedThreads / 32];
    // Thomas pivots of tridiag(1/6, 2/3, 1/6) in T: entry kPivots holds the limit
    constexpr int kPv = sizeof(T) == 4 ? kPiv32 : kPivots;
    __shared__ T piv_cp[kPivots + 1], piv_ib[kPivots + 1];
    __shared__ float2 piv32[kPiv32 + 1];
    __shared__ WalkWin s_win;
    __shared__ int2 s_rows[kMaxGroups];
    __shared__ T sig_s[kFusedMaxTileP];   // column-sum weights of Lambda_p^{-1} for the tile rows

    const Geometry &g = A.g;
    const int nx = g.nx, np = g.np;
    const int tix = tile % A.ntx, tip = tile / A.ntx;
    const int X0 = tix * A.tx, P0 = tip * A.tp;
    const int TXe = min(A.tx, nx - X0), TPe = min(A.tp, np - P0);
    const bool full = A.full_row != 0;
    constexpr int kHalo = Halo<T>::value;
    // x halo of the in-tile x solve (none for whole-period tiles and for a separate x pass)
    const int D = (GAL && !full && !A.xpass) ? kHalo : 0;
    const int G = A.G, Gp = A.Gp;   // guard bands: columns, rows
    WinGeom W;
    W.WW = full ? nx + 2 * G : TXe + 2 * D + 2 * G;
    W.WH = TPe + 2 * Gp;
    W.ws = A.ws;
    W.WX0 = X0 - D - G;
    W.WP0 = P0 - Gp;
    W.own_c0 = G + D;
    W.own_c1 = G + D + TXe;
    W.np = np;
    W.nx = nx;
    W.full = full;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;

    {
        const int nvec = (int)(((size_t)W.WH * W.ws * sizeof(T)) / 16);
        uint4 *w4 = reinterpret_cast<uint4 *>(win);
        for (int k = tid; k < nvec; k += blockDim.x) w4[k] = make_uint4(0, 0, 0, 0);
        for (int k = nvec * (16 / (int)sizeof(T)) + tid; k < W.WH * W.ws; k += blockDim.x) win[k] = T(0);
    }
    // everything below reads or writes what the launch before this one may still be writing
    after_previous_launch();
    // the tile's source rectangle, when an earlier step has left it (asked for first: all that follows
    // depends on it)
    const int4 known = A.tile_src ? A.tile_src[tile] : make_int4(kTileSrcUnset, 0, 0, 0);
    const bool cached = known.x != kTileSrcUnset;
    for (int k = tid; GAL && k <= kPv; k += blockDim.x) {
        // FP32: rows from kPiv32 on take the limit
        const int e = k == kPv ? kPivots : k;
        if (sizeof(T) == 4) {
            piv32[k] = make_float2((float)A.piv[2 * e + 1], (float)A.piv[2 * e]);
        } else {
            piv_cp[k] = (T)A.piv[2 * e];
            piv_ib[k] = (T)A.piv[2 * e + 1];
        }
    }
    if (GAL && A.fel_partials)
        for (int k = tid; k < TPe; k += blockDim.x) sig_s[k] = (T)A.sigma[P0 + k];
    if (tid == 0) {
        s_ia = s_ja = 0x7fffffff;
        s_ib = s_jb = -0x7fffffff;
        s_omax = 0;
        {
            s_win.WW = W.WW;
            s_win.own_c0 = full ? 0 : W.own_c0;
            s_win.own_c1 = full ? W.WW : W.own_c1;
            s_win.nx = nx;
        }
    }
    double al = g.alpha0, be = g.beta0, M = g.m0, phi = g.phi0;
    if (g.kind == VP_PUSH_FEL_DKD) {
        al = -A.state[ST_K_IM];
        be = A.state[ST_K_RE];
        M = A.state[ST_M];
        phi = A.state[ST_PHI];
    }

    // ---- bound the source nodes whose footprint can reach the widened tile (FP32 with
    //      slack: every magnitude here is below 1e5 cells, where FP32 is exact to 1e-2);
    //      a push that does not change between steps gives the same bounds every step
    int ia = known.x, ib = known.y, ja = known.z, jb = known.w;
    if (!cached) {
        __syncthreads();
        const float SL = 0.05f;
        const float Mf = (float)M, phif = (float)phi;
        const float EU = fabsf((float)g.KU) * Mf, EV = fabsf((float)g.KV) * Mf;
        const float KVM = (float)g.KV * Mf;
        const float vcmin = (float)g.vc_min, vcmax = (float)g.vc_max;
        const float ucmin = (float)g.uc_min, ucmax = (float)g.uc_max;
        const float vd_min = vcmin + (float)g.vr_min - EV, vd_max = vcmax + (float)g.vr_max + EV;
        const float x0f = (float)g.x0, hxf = (float)g.hx, padf = (float)g.a_pad;
        const bool edge_lo = P0 == 0, edge_hi = P0 + TPe == np;
        const int jlo = edge_lo ? 0 : max(0, (int)floorf((float)(P0 - R) - vd_max - SL));
        const int jhi = edge_hi ? np - 1 : min(np - 1, (int)ceilf((float)(P0 + TPe - 1 + R) - vd_min + SL));
        const float acc_lo = edge_lo ? -1e30f : (float)(P0 - R);
        const float acc_hi = edge_hi ? 1e30f : (float)(P0 + TPe - 1 + R);
        int my_ia = 0x7fffffff, my_ib = -0x7fffffff, my_ja = 0x7fffffff, my_jb = -0x7fffffff;
        for (int j = jlo + tid; j <= jhi; j += blockDim.x) {
            const float4 rb = A.rowbf[j];   // u, v, y
            int ia, ib;
            float vcl = vcmin, vch = vcmax;
            float smin = -1.f, smax = 1.f;
            if (full) {
                ia = 0;
                ib = nx - 1;
            } else {
                ia = (int)floorf((float)(X0 - D - R) - rb.x - EU - ucmax - SL);
                ib = (int)ceilf((float)(X0 + TXe + D - 1 + R) - rb.x + EU - ucmin + SL);
                const int width = ib - ia + 1;
                if (width < nx - 2 * kColBlock) {
                    vcl = 1e30f;
                    vch = -1e30f;
                    const int start = imod(ia, nx);
                    int seg_lo[2], seg_hi[2], nseg = 1;
                    if (start + width <= nx) {
                        seg_lo[0] = start;
                        seg_hi[0] = start + width - 1;
                    } else {
                        seg_lo[0] = start;
                        seg_hi[0] = nx - 1;
                        seg_lo[1] = 0;
                        seg_hi[1] = start + width - 1 - nx;
                        nseg = 2;
                    }
                    for (int sg = 0; sg < nseg; ++sg)
                        for (int bq = seg_lo[sg] / kColBlock; bq <= seg_hi[sg] / kColBlock; ++bq) {
                            const float2 vb = A.vcbf[bq];
                            vcl = fminf(vcl, vb.x);
                            vch = fmaxf(vch, vb.y);
                        }
                    if (EV > 0.f)
                        sin_range32(x0f + ia * hxf - padf + rb.z + phif, x0f + ib * hxf + padf + rb.z + phif,
                                    smin, smax);
                }
            }
            float tlo = 0.f, thi = 0.f;
            if (EV > 0.f) {
                tlo = fminf(KVM * smin, KVM * smax);
                thi = fmaxf(KVM * smin, KVM * smax);
            }
            const float vlo = (float)j + rb.y + vcl + tlo - SL;
            const float vhi = (float)j + rb.y + vch + thi + SL;
            if (vhi > acc_lo && vlo < acc_hi) {
                my_ia = min(my_ia, ia);
                my_ib = max(my_ib, ib);
                my_ja = min(my_ja, j);
                my_jb = max(my_jb, j);
            }
        }
        if (my_jb >= my_ja) {
            atomicMin(&s_ia, my_ia);
            atomicMax(&s_ib, my_ib);
            atomicMin(&s_ja, my_ja);
            atomicMax(&s_jb, my_jb);
        }
        __syncthreads();
        ia = s_ia;
        ib = s_ib;
        ja = s_ja;
        jb = s_jb;
        // Strong shear along x: the rows' source columns together span more than a period. Each column is then walked
        // once, and its nodes land at their images in the window (a column that counted for one of its images alone
        // left out the others: 28% of the weight of 640 x 512 turned by 1 rad). The period is centred on the tile,
        // from an even column on (pairs in 8-byte loads)
        if (!full && jb >= ja && (unsigned)ib - (unsigned)ia >= (unsigned)nx) {
            ia = (X0 + (TXe - nx) / 2) & ~1;
            ib = ia + nx - 1;
        }
        if (A.tile_src && tid == 0) A.tile_src[tile] = make_int4(ia, ib, ja, jb);
    }
    const bool period = !full && jb >= ja && ib - ia + 1 == nx;
    if (tid == 0) s_win.wrap = full ? G : (period ? 0 : -1);
    double lost = 0.0;   // in the window's scaled units until the end of the tile

    // ---- the row table of the source rows into shared memory, when it fits: every node of a
    //      row reads that row's entry, and a shared-memory load is shorter than an L1 hit
    const bool rows_cached = jb >= ja && jb - ja + 1 <= A.rowcache;
    if (rows_cached) {
        constexpr int kVec = (int)(sizeof(RowEntry<T>) / 16);
        const float4 *from = reinterpret_cast<const float4 *>(A.row + ja);
        float4 *to = reinterpret_cast<float4 *>(rowc);
        for (int k = tid; k < kVec * (jb - ja + 1); k += blockDim.x) to[k] = __ldg(from + k);
    }
    const RowEntry<T> *srow = rowc - ja;   // srow[j]: row j (rows_cached only)

    // ---- FP32: fixed-point scale of the window from max|s| over the rows the walk reads, taken
    //      from the per-tile maxima the previous step (or vp_set_f) recorded for the state.
    //      The truncated Thomas solve keeps |w| <= 3 max|s| (forward gain 1/(beta - 1/6) <= 2.2,
    //      back substitution 1/(1 - c') <= 1.37); a cell sums the B3 taps of the nodes pushed near
    //      it, about one for an area-preserving flow: 8 times that bound fits in int32.
    T qs = T(1), iq = T(1);
    if (sizeof(T) == 4) {
        // every warp for itself: no exchange between warps
        unsigned mx = 0u;   // bits of a non-negative float: ordered as the float
        const unsigned *map = reinterpret_cast<const unsigned *>(A.smax_in);
        if (jb >= ja) {
            const int r0 = GAL ? max(0, ja - kHalo) : ja, r1 = GAL ? min(np - 1, jb + kHalo) : jb;
            const int c0 = imod(ia, nx), c1 = c0 + min(ib - ia + 1, nx) - 1;
            // tile columns the source columns c0 .. c1 (wrapped) lie in
            const int t0 = c0 / A.tx, nt = (c1 < nx ? c1 / A.tx : A.ntx + (c1 - nx) / A.tx) - t0 + 1;
            const int q0 = r0 / A.tp, nq = r1 / A.tp - q0 + 1;
            for (int k = lane; k < nt * nq; k += 32) {
                const int q = k / nt;
                int tc = t0 + k - q * nt;
                if (tc >= A.ntx) tc -= A.ntx;
                mx = max(mx, map[(q0 + q) * A.ntx + tc]);
            }
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (!(__uint_as_float(mx) <= 3.0e38f)) {
            qs = T(0);   // a non-finite state, reported when it was written: its deposit is dropped
            iq = T(0);
        } else {
            // the scale is a power of two, so that iq = 1 / qs is exact (a rounded iq scales the
            // tile's weights by 1 +- 6e-8, a gain that repeats over the steps while the tile's
            // maximum stays put): qs = 2^(32 - e) with m = f 2^e, f in [0.5, 1), i.e. qs m in
            // [2^31, 2^32): a cell reaches 2^31 only at 4 to 8 times the largest weight (16 to 32
            // times with the Thomas gain bound), against about one for an area-preserving flow
            // (a floor of 1e-28 keeps qs finite where the state is zero)
            const float m = fmaxf(__uint_as_float(mx), 1e-28f) * (GAL ? 3.1f : 1.f) * 8.f;
            int e2;
            frexpf(m, &e2);
            qs = (T)ldexpf(1.f, 32 - e2);
            iq = (T)ldexpf(1.f, e2 - 32);
        }
    }
    // FP32: a thread walks a pair of adjacent columns. The first column of every pair is even where the mesh
    // allows, so that a pair's source values are one 8-byte load
    const int ia2 = (nx & 1) == 0 && ib - ia + 2 <= nx ? ia - (ia & 1) : ia;
    const int wsrc = jb >= ja ? min(ib - ia2 + 1, nx) : 0;
    const int npair = (wsrc + 1) >> 1, nwp = (npair + 31) >> 5;
    // a rectangle much taller than the tile: the rows of every warp's columns alone
    const bool loose = sizeof(T) == 4 && jb - ja + 1 > 2 * TPe + 24 && nwp <= kMaxGroups;
    if (loose)
        for (int wi = warp; wi < nwp; wi += nwarps) {
            const int c0 = ia2 + 64 * wi;
            int2 r = rows_of_columns<T>(A, c0, min(c0 + 63, ia2 + wsrc - 1), ja, jb, X0, TXe, P0, TPe, D, R, (float)M,
                                        (float)phi, period);
            if (r.x > r.y) r = make_int2(1, 0);
            if (lane == 0) s_rows[wi] = r;
        }
    __syncthreads();   // the zeroed window, the row table, the pivots, the groups' rows

    const int edge = (P0 == 0 ? 1 : 0) | (P0 + TPe == np ? 2 : 0);   // the open edges the tile owns: below, above

    // ---- walk the source columns
    if constexpr (sizeof(T) == 4) {
        // FP32: items of (pair of adjacent columns, segment of rows)
        const int rows = jb - ja + 1, nseg = min(A.nseg, max(1, rows / kMinSegRows)), len = (rows + nseg - 1) / nseg;
        Walk32 K;
        K.src = A.src;
        K.nx = nx;
        K.np = np;
        K.row = A.row;
        K.rowc = smem_addr(rowc) - (unsigned)ja * (unsigned)sizeof(RowEntry<float>);
        K.piv = piv32;
        K.W = &s_win;
        K.win = smem_addr(win);
        K.ws4 = W.ws * 4;
        K.lim = W.WH * W.ws * 4;
        K.WW = W.WW;
        K.WP0 = W.WP0;
        K.edge = edge;
        // kept in registers: rebuilt from the arguments at every use they cost 20 of 200 instructions a row
        K.ws4 = opaque(K.ws4);
        K.lim = opaque(K.lim);
        K.edge = opaque(K.edge);
        const unsigned gc = smem_addr(gcol) + 8u * tid, gs = 8u * blockDim.x;
        // a warp's lanes share their segment (a warp over two segments runs both, one after the other)
        for (int wi = warp; wi < nwp * nseg; wi += nwarps) {
            const int sg = wi / nwp, q = (wi - sg * nwp) * 32 + lane, ic = ia2 + 2 * q;
            int r_lo = ja + sg * len, r_hi = min(jb, r_lo + len - 1);
            if (loose) {
                const int2 r = s_rows[wi - sg * nwp];   // none: (1, 0)
                const int l = (r.y - r.x + nseg) / nseg;
                r_lo = r.x + sg * l;
                r_hi = min(r.y, r_lo + l - 1);
            }
            if (q >= npair || r_lo > r_hi) continue;
            const int imA = imod(ic, nx), imB = imA + 1 < nx ? imA + 1 : 0;
            // a last pair of one column: its second column takes the weight 0
            const bool two = ic + 1 - ia2 < wsrc;
            const f2_t q2 = f2_pack(qs, two ? qs : 0.f);
            if (rows_cached)
                walk_pair<BASIS, GAL, UTERM, true>(K, A.col[imA], A.col[imB], imA, imB, ic - W.WX0, r_lo, r_hi, q2,
                                                   (float)al, (float)be, (float)g.KU, (float)g.KV, gc, gs, lost);
            else
                walk_pair<BASIS, GAL, UTERM, false>(K, A.col[imA], A.col[imB], imA, imB, ic - W.WX0, r_lo, r_hi, q2,
                                                    (float)al, (float)be, (float)g.KU, (float)g.KV, gc, gs, lost);
        }
    } else if (jb >= ja) {
        // FP64: items of (column, segment of rows)
        const int wcol = min(ib - ia + 1, nx);
        const int rows = jb - ja + 1, nseg = min(A.nseg, max(1, rows / kMinSegRows)), len = (rows + nseg - 1) / nseg;
        Walk64 K;
        K.src = A.src;
        K.nx = nx;
        K.np = np;
        K.row = A.row;
        K.rowc = srow;
        K.piv_ib = piv_ib;
        K.piv_cp = piv_cp;
        K.W = &s_win;
        K.win = win;
        K.ws = W.ws;
        K.lim = W.WH * W.ws;
        K.WW = W.WW;
        K.WP0 = W.WP0;
        K.edge = edge;
        const int nw = (wcol + 31) >> 5;
        for (int wi = warp; wi < nw * nseg; wi += nwarps) {
            const int sg = wi / nw, q = (wi - sg * nw) * 32 + lane, ic = ia + q;
            const int r_lo = ja + sg * len, r_hi = min(jb, r_lo + len - 1);
            if (q >= wcol || r_lo > r_hi) continue;
            const int im = imod(ic, nx);
            if (rows_cached)
                walk_col64<BASIS, GAL, UTERM, true>(K, A.col[im], im, ic - W.WX0, r_lo, r_hi, al, be, g.KU, g.KV,
                                                    gcol + tid, (int)blockDim.x, lost);
            else
                walk_col64<BASIS, GAL, UTERM, false>(K, A.col[im], im, ic - W.WX0, r_lo, r_hi, al, be, g.KU, g.KV,
                                                     gcol + tid, (int)blockDim.x, lost);
        }
    }
    __syncthreads();

    // ---- guard rows beyond an open momentum edge that the tile owns: lost weight of the own columns. Where tiles are
    // lower than the guard, other tiles' windows reach past the mesh too; what lands there is the owner's to count.
    // (Loops over these rows alone, not unrolled: a test in a loop over all guard rows of every tile cost the whole
    // step 2%, 8192 x 8192 491 us for 480, by the registers it took)
    if (edge) {
        const int c0 = full ? 0 : W.own_c0, c1 = full ? W.WW : W.own_c1;
#pragma unroll 1
        for (int k = edge & 1 ? 0 : Gp; k < (edge & 2 ? 2 * Gp : Gp); ++k) {   // below the tile, then above it
            const T *row = win + (size_t)(k < Gp ? k : TPe + k) * W.ws;
#pragma unroll 1
            for (int c = c0 + tid; c < c1; c += blockDim.x) lost += wraw(row + c);
        }
    }
    if (full) {
        // fold the guard columns onto the period: [-G, 0) -> [nx - G, nx), [nx, nx + G) -> [0, G)
        __syncthreads();
        if (nx >= G) {
            for (int k = tid; k < TPe * G; k += blockDim.x) {
                const int rr = k / G + Gp, c = k - (k / G) * G;
                T *row = win + (size_t)rr * W.ws;
                wfold(row + nx + c, row + c);
                wfold(row + G + c, row + G + nx + c);
            }
        } else {
            // a band longer than the period: several of its columns have the same image
            for (int rr = tid; rr < TPe; rr += blockDim.x) {
                T *row = win + (size_t)(rr + Gp) * W.ws;
                for (int c = 0; c < G; ++c) {
                    wfold(row + G + imod(c - G, nx), row + c);
                    wfold(row + G + c % nx, row + G + nx + c);
                }
            }
        }
    }
    __syncthreads();

    // ---- store the tile (Galerkin: after the Lambda_x solve); FEL column sums
    const bool want_part = A.fel_partials != 0;
    bool bad = false;
    float om = 0.f;   // FP32: max|s'| of the stored outputs
    double pw = 0.0, pc = 0.0, ps = 0.0;
    if (GAL && A.xpass) {
        // separate x pass: store the deposit r = Delta^T w of the own columns in weight units; the
        // row pass solves Lambda_x, records max|s'| per tile and checks the outputs
        store_window_rows<T, false>(win, W, A.dst, nx, P0, X0, TXe, TPe, G, Gp, iq, warp, nwarps, lane, om, bad);
    } else if (GAL) {
        if constexpr (sizeof(T) == 4) {
            const float sh = (float)A.piv[kPivXsFused], sl = (float)A.piv[kPivXsFused + 1];
            if ((full ? nx : A.tx) + 2 * kHalo <= 256)
                solve_rows_f32<8>(win, W, A.dst, full, G, Gp, TXe, TPe, P0, X0, nx, want_part, warp, nwarps, lane, sh,
                                  sl, iq, om, bad);
            else
                solve_rows_f32<kXBig32>(win, W, A.dst, full, G, Gp, TXe, TPe, P0, X0, nx, want_part, warp, nwarps, lane,
                                        sh, sl, iq, om, bad);
        } else {
            const int L = full ? nx : TXe + 2 * D;
            if (L <= 256)
                solve_rows_f64<8>(win, W, A.dst, L, full, D, G, Gp, TXe, TPe, P0, X0, nx, want_part, warp, nwarps, lane,
                                  bad, gcol, GRows<T>::value * blockDim.x);
            else
                solve_rows_f64<kXBig>(win, W, A.dst, L, full, D, G, Gp, TXe, TPe, P0, X0, nx, want_part, warp, nwarps,
                                      lane, bad, gcol, GRows<T>::value * blockDim.x);
        }
    } else {
        // no solve: the deposit is the new state (its max|w| sets the next step's window scale)
        store_window_rows<T, true>(win, W, A.dst, nx, P0, X0, TXe, TPe, G, Gp, iq, warp, nwarps, lane, om, bad);
    }
    if (want_part) {
        // FEL: column sums of w over the tile (Galerkin: sum_j w_ij = sum_j sigma_j s_ij; with a
        // separate x pass the window keeps the deposit r, and bunch_x turns its cos/sin sums into
        // those of s')
        __syncthreads();
        const bool sums_of_s = GAL && !A.xpass;
        // columns go to kSumWarps virtual warps whatever the block size, so that a simulation's sums are
        // formed in the same order alone and in a batch
        for (int vw = warp; vw < kSumWarps; vw += nwarps) {
        pw = pc = ps = 0.0;
        for (int c = vw * 32 + lane; c < TXe; c += 32 * kSumWarps) {
            // four interleaved compensated sums (rows rr = q mod 4), added in a fixed order at the
            // end: four independent chains of shared-memory loads and error-free steps instead of one
            DSum<T> acc[4];
            const T *cell = win + (size_t)Gp * W.ws + G + D + c;
            int rr = 0;
            for (; rr + 4 <= TPe; rr += 4, cell += 4 * W.ws) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    // in-tile x solve: the epilogue left s in the own columns; else the cells hold
                    // the deposit
                    const T v = sums_of_s ? cell[q * W.ws] : wget(cell + q * W.ws, iq);
                    if (GAL) acc[q].add_prod(sig_s[rr + q], v);
                    else acc[q].add(v);
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (rr + q < TPe) {
                    const T v = sums_of_s ? cell[q * W.ws] : wget(cell + q * W.ws, iq);
                    if (GAL) acc[q].add_prod(sig_s[rr + q], v);
                    else acc[q].add(v);
                }
            const double sum = (acc[0].value() + acc[1].value()) + (acc[2].value() + acc[3].value());
            const double2 t = A.csx[X0 + c];
            pw += sum;
            pc += sum * t.x;
            ps += sum * t.y;
        }
        pc *= A.bunch_x;
        ps *= A.bunch_x;
        for (int o = 16; o > 0; o >>= 1) {
            pw += __shfl_down_sync(0xffffffffu, pw, o);
            pc += __shfl_down_sync(0xffffffffu, pc, o);
            ps += __shfl_down_sync(0xffffffffu, ps, o);
        }
        if (lane == 0) {
            s_part[0][vw] = pw;
            s_part[1][vw] = pc;
            s_part[2][vw] = ps;
        }
        }
    }
    if (bad) atomicOr(A.err, ERRF_NONFINITE);

    // ---- per-tile reductions in a fixed order (FP64 work only where there is weight to sum)
    // FP32: record max|s'| of the tile for the next step's window scale
    if (sizeof(T) == 4 && om > 0.f) atomicMax(&s_omax, __float_as_int(om));
    const bool any_lost = __syncthreads_or(lost != 0.0);
    if (sizeof(T) == 4 && tid == 0) A.smax_out[tile] = __int_as_float(s_omax);
    if (want_part && tid < 3) {
        double t = 0.0;
        for (int w = 0; w < kSumWarps; ++w) t += s_part[tid][w];
        A.tile_part[3 * tile + tid] = t;
        __threadfence();   // visible before thread 0 takes the step's ticket
    }
    if (any_lost) {
        // back to weight units: iq = 1 / qs exactly (a power of two; 0 for a dropped deposit)
        double v = lost * (double)iq;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) s_lost[warp] = v;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < nwarps; ++w) t += s_lost[w];
            A.tile_lost[tile] += t;
        }
    }
}

// The end of a simulation's step, in the same launch: each CTA takes a ticket once its tile's partial sums
// are visible device-wide (they are written and fenced before); the CTA that draws the simulation's last ticket
// sees every partial and finishes the step: the FEL field update from all tile partials in the fixed order of
// fel_finalize_core (the window's shared memory, no longer needed, is its scratch), else the step count. It then
// resets the counter for the next launch. No CTA waits on another. Returns whether this CTA was the last.
template <typename T>
__device__ __forceinline__ bool finish_step(const FusedArgs<T> &A, unsigned char *smem_raw)
{
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(A.ticket, 1) == A.ntx * A.ntp - 1;
    }
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    double *state = const_cast<double *>(A.state);
    if (A.fel_partials) {
        fel_finalize_core(A.tile_part, A.ntx * A.ntp, state, A.hist, A.hist_cap, A.g.dt, 0, 0, false,
                          reinterpret_cast<double *>(smem_raw));
    } else if (threadIdx.x == 0) {
        const double st = state[ST_STEP] + 1.0;
        state[ST_STEP] = st;
        state[ST_TAU] = st * A.g.dt;
    }
    if (threadIdx.x == 0) *A.ticket = 0;
    return true;
}

template <typename T, int BASIS, bool GAL, bool UTERM>
__global__ void __launch_bounds__(kFusedThreads, 2)
    step_fused_kernel(const FusedArgs<T> A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fused_tile<T, BASIS, GAL, UTERM>(A, blockIdx.x, smem_raw);
    finish_step<T>(A, smem_raw);
}

// Batched step: CTA b takes the (instance, tile) item b of the work list (largest tiles first;
// the hardware hands out CTAs in index order as slots free up); instance k uses
// args[2 k + parity[k]] (parity = which buffer holds its current state) and its tile is skipped
// once the instance has taken its steps (left[k] == 0). One CTA per item rather than a persistent
// loop over an atomic counter: inside a loop the compiler kept the arguments of every item live
// and spilled 400 bytes per thread. The CTA that ends an instance's step (every CTA of it has read
// parity and left by then) also flips its parity and counts it down: as a launch of its own that took 5 to 8 us a
// step, against 40 us for the tiles of a dozen served requests.
template <typename T, int BASIS, bool GAL, bool UTERM>
__global__ void __launch_bounds__(kFusedThreads, 2)
    step_fused_batch_kernel(const FusedArgs<T> *__restrict__ args, int *parity, int *left,
                            const int2 *__restrict__ items, int nitems)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) FusedArgs<T> sA;
    if ((int)blockIdx.x >= nitems) return;
    const int2 e = items[blockIdx.x];
    if (left[e.x] <= 0) return;   // this simulation takes no more steps in this call
    const FusedArgs<T> *src = args + 2 * e.x + parity[e.x];
    constexpr int nwords = sizeof(FusedArgs<T>) / 4;
    for (int k = threadIdx.x; k < nwords; k += blockDim.x)
        reinterpret_cast<int *>(&sA)[k] = reinterpret_cast<const int *>(src)[k];
    __syncthreads();
    fused_tile<T, BASIS, GAL, UTERM>(sA, e.y, smem_raw);
    if (finish_step<T>(sA, smem_raw) && threadIdx.x == 0) {
        parity[e.x] ^= 1;
        left[e.x] -= 1;
    }
}

template <typename T>
size_t fused_smem_bytes(int ws, int wh, int threads, int rowcache)
{
    return (size_t)ws * wh * sizeof(T) + (size_t)GRows<T>::value * threads * sizeof(T) +
           (size_t)rowcache * sizeof(RowEntry<T>);
}

int fused_rowcache_rows(int precision, size_t base_bytes, int ctas)
{
    // shared memory of an SM, reserved per CTA, and the larger static shared memory of the step
    // kernels (the batched one holds its FusedArgs there); defaults if no device answers
    int dev = 0, per_sm = 233472, reserved = 1024;
    size_t stat = 4096;
    if (cudaGetDevice(&dev) == cudaSuccess) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess) per_sm = v;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrReservedSharedMemoryPerBlock, dev) == cudaSuccess) reserved = v;
        cudaFuncAttributes fa;
        const void *k = precision == VP_FP64
                            ? reinterpret_cast<const void *>(step_fused_kernel<double, VP_BASIS_CUBIC_BSPLINE, true, true>)
                            : reinterpret_cast<const void *>(step_fused_batch_kernel<float, VP_BASIS_CUBIC_BSPLINE, true, true>);
        if (cudaFuncGetAttributes(&fa, k) == cudaSuccess) stat = fa.sharedSizeBytes + 256;
        cudaGetLastError();
    }
    const long budget = (long)per_sm / (ctas < 1 ? 1 : ctas) - reserved - (long)stat - (long)base_bytes;
    const size_t row = precision == VP_FP64 ? sizeof(RowEntry<double>) : sizeof(RowEntry<float>);
    long rows = budget > 0 ? budget / (long)row : 0;
    if (rows > 256) rows = 256;
    return rows >= 32 ? (int)rows : 0;
}

// k<<<grid, threads, smem, s>>>(args...), ahead: as a programmatic dependent launch
template <typename... KA, typename... A>
static cudaError_t launch_ahead(void (*k)(KA...), int grid, int threads, size_t smem, cudaStream_t s, bool ahead, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = ahead ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, KA(args)...);
}

template <typename T>
cudaError_t launch_step_fused(const FusedArgs<T> &a, int threads, bool ahead, cudaStream_t s)
{
    const int wh = a.tp + 2 * a.Gp;
    // the last CTA's field update uses the window memory as its scratch
    const size_t smem_tile = fused_smem_bytes<T>(a.ws, wh, threads, a.rowcache);
    const size_t smem = smem_tile > kFinSmem ? smem_tile : kFinSmem;
    const int grid = a.ntx * a.ntp;
    const bool gal = a.g.basis == VP_BASIS_CUBIC_BSPLINE && a.g.projection == VP_PROJ_GALERKIN;
    const bool uterm = a.g.kind == VP_PUSH_FEL_DKD;
#define VP_LAUNCH_FUSED(B, GL, UT)                                                            \
    do {                                                                                      \
        auto k = step_fused_kernel<T, B, GL, UT>;                                             \
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                             (int)smem);                                      \
        if (e != cudaSuccess) return e;                                                       \
        return launch_ahead(k, grid, threads, smem, s, ahead, a);                             \
    } while (0)
    if (a.g.basis == VP_BASIS_TENT) {
        if (uterm) VP_LAUNCH_FUSED(VP_BASIS_TENT, false, true);
        else VP_LAUNCH_FUSED(VP_BASIS_TENT, false, false);
    } else if (!gal) {
        if (uterm) VP_LAUNCH_FUSED(VP_BASIS_CUBIC_BSPLINE, false, true);
        else VP_LAUNCH_FUSED(VP_BASIS_CUBIC_BSPLINE, false, false);
    } else {
        if (uterm) VP_LAUNCH_FUSED(VP_BASIS_CUBIC_BSPLINE, true, true);
        else VP_LAUNCH_FUSED(VP_BASIS_CUBIC_BSPLINE, true, false);
    }
#undef VP_LAUNCH_FUSED
}

// s = Lambda_p w along columns (tridiag(1/6, 2/3, 1/6), zero beyond the open edges). Each thread
// walks one column through a chunk of rows, so every input row is read once (plus a halo
// row at either end of the chunk): w may be host memory the device reads in place.
// MAX: also max|s| over each tx x tp tile into the zeroed map[][ntx] (infinity, and the error flag, where a
// value is not finite), which as a pass of its own read the state once more (0.137 ms for 8192 x 8192).
constexpr int kMulCols = 256;

// m (bits of a non-negative float) of the columns of one warp into their tiles of one tile row
__device__ __forceinline__ void max_to_map(unsigned m, int col, int nx, int tx, unsigned *map_row)
{
    const int t0 = __shfl_sync(0xffffffffu, col, 0) / tx, t = min(col, nx - 1) / tx;
    if (__all_sync(0xffffffffu, t == t0)) {
        m = __reduce_max_sync(0xffffffffu, m);
        if ((threadIdx.x & 31) == 0 && m != 0u) atomicMax(map_row + t0, m);
    } else if (m != 0u) {
        atomicMax(map_row + t, m);
    }
}

template <typename T, bool MAX>
__global__ void __launch_bounds__(kMulCols)
    lambda_p_mul_kernel(const T *__restrict__ w, T *__restrict__ s, int nx, int np, int rows, unsigned *map, int tx,
                        int tp, int ntx, unsigned *err)
{
    const int col = blockIdx.x * kMulCols + threadIdx.x;
    if (!MAX && col >= nx) return;
    const bool in = col < nx;
    const int j0 = blockIdx.y * rows, j1 = min(j0 + rows, np);
    T lo = in && j0 > 0 ? w[(size_t)(j0 - 1) * nx + col] : T(0);
    T c = in ? w[(size_t)j0 * nx + col] : T(0);
    for (int ja = j0; ja < j1;) {   // rows of one tile row at a time
        const int jb = MAX ? min(j1, (ja / tp + 1) * tp) : j1;
        float m = 0.f, chk = 0.f;
#pragma unroll 8
        for (int j = ja; j < jb; ++j) {
            const T hi = in && j + 1 < np ? w[(size_t)(j + 1) * nx + col] : T(0);
            const T v = (lo + hi) * (T(1) / T(6)) + c * (T(2) / T(3));
            if (in) s[(size_t)j * nx + col] = v;
            if (MAX) {
                m = fmaxf(m, fabsf((float)v));
                chk = fmaf((float)v, 0.f, chk);   // 0, or NaN once a value is not finite
            }
            lo = c;
            c = hi;
        }
        if (MAX) {
            if (chk != 0.f) {
                m = __int_as_float(0x7f800000);
                atomicOr(err, ERRF_NONFINITE);
            }
            max_to_map(__float_as_uint(m), col, nx, tx, map + (size_t)(ja / tp) * ntx);
        }
        ja = jb;
    }
}

// max|s| per tile of a state that is there already (no solve, so nothing else passes over it), into the zeroed
// map: a warp takes 32 columns of a chunk of rows, as above
__global__ void __launch_bounds__(kMulCols)
    tile_max_kernel(const float *__restrict__ s, unsigned *map, int nx, int np, int rows, int tx, int tp, int ntx,
                    unsigned *err)
{
    const int col = blockIdx.x * kMulCols + threadIdx.x;
    const bool in = col < nx;
    const int j0 = blockIdx.y * rows, j1 = min(j0 + rows, np);
    for (int ja = j0; ja < j1;) {
        const int jb = min(j1, (ja / tp + 1) * tp);
        float m = 0.f, chk = 0.f;
#pragma unroll 16
        for (int j = ja; j < jb; ++j) {
            const float v = in ? s[(size_t)j * nx + col] : 0.f;
            m = fmaxf(m, fabsf(v));
            chk = fmaf(v, 0.f, chk);
        }
        if (chk != 0.f) {
            m = __int_as_float(0x7f800000);
            atomicOr(err, ERRF_NONFINITE);
        }
        max_to_map(__float_as_uint(m), col, nx, tx, map + (size_t)(ja / tp) * ntx);
        ja = jb;
    }
}

// rows per block of the two kernels above: 64, or 16 where 64 would leave most SMs without a block
static int column_rows(int nx, int np)
{
    const long blocks = (long)((nx + kMulCols - 1) / kMulCols) * ((np + 63) / 64);
    int rows = blocks < 152 * 4 ? 16 : 64;
    while ((np + rows - 1) / rows > 65535) rows *= 2;
    return rows;
}

cudaError_t launch_tile_max(const float *s, float *map, int nx, int np, int tx, int tp, int ntx, unsigned *err, cudaStream_t st)
{
    const int rows = column_rows(nx, np);
    const dim3 grid((nx + kMulCols - 1) / kMulCols, (np + rows - 1) / rows);
    tile_max_kernel<<<grid, kMulCols, 0, st>>>(s, reinterpret_cast<unsigned *>(map), nx, np, rows, tx, tp, ntx, err);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lambda_p_mul(const T *w, T *s, int nx, int np, float *map, int tx, int tp, int ntx,
                                unsigned *err, cudaStream_t st)
{
    const int rows = column_rows(nx, np);
    const dim3 grid((nx + kMulCols - 1) / kMulCols, (np + rows - 1) / rows);
    if ((np + 63) / 64 > 65535) return cudaErrorInvalidConfiguration;
    if (map) {
        lambda_p_mul_kernel<T, true><<<grid, kMulCols, 0, st>>>(w, s, nx, np, rows, reinterpret_cast<unsigned *>(map), tx,
                                                                tp, ntx, err);
    } else {
        lambda_p_mul_kernel<T, false><<<grid, kMulCols, 0, st>>>(w, s, nx, np, rows, nullptr, 1, 1, 1, err);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_step_fused_batch(const FusedArgs<T> *args, int *parity, int *left,
                                    const int2 *items, int nitems, int basis, int projection,
                                    size_t smem, int threads, int grid, cudaStream_t s)
{
    const bool gal = basis == VP_BASIS_CUBIC_BSPLINE && projection == VP_PROJ_GALERKIN;
#define VP_LAUNCH_BATCH(B, GL)                                                                \
    do {                                                                                      \
        auto k = step_fused_batch_kernel<T, B, GL, true>;                                     \
        if (grid <= 0) /* set-up call: shared-memory attribute only (not capturable) */       \
            return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,        \
                                        (int)smem);                                           \
        k<<<grid, threads, smem, s>>>(args, parity, left, items, nitems);                     \
    } while (0)
    if (basis == VP_BASIS_TENT) VP_LAUNCH_BATCH(VP_BASIS_TENT, false);
    else if (!gal) VP_LAUNCH_BATCH(VP_BASIS_CUBIC_BSPLINE, false);
    else VP_LAUNCH_BATCH(VP_BASIS_CUBIC_BSPLINE, true);
#undef VP_LAUNCH_BATCH
    return cudaGetLastError();
}

// CTAs of the batched step kernel that fit on one SM with this dynamic shared memory and block
// size (sets the kernel's shared-memory attribute first); 0 if the query fails
int fused_batch_blocks_per_sm(int basis, int projection, size_t smem, int threads)
{
    const bool gal = basis == VP_BASIS_CUBIC_BSPLINE && projection == VP_PROJ_GALERKIN;
    const void *k = (const void *)step_fused_batch_kernel<float, VP_BASIS_CUBIC_BSPLINE, true, true>;
    if (basis == VP_BASIS_TENT) k = (const void *)step_fused_batch_kernel<float, VP_BASIS_TENT, false, true>;
    else if (!gal) k = (const void *)step_fused_batch_kernel<float, VP_BASIS_CUBIC_BSPLINE, false, true>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// ---------------------------------------------------------------------------
// Lambda_x^{-1} of whole rows, for plans with a separate x pass (Sec. III: Lambda = Lambda_x (x)
// Lambda_p, with Lambda_x the cyclic tridiag(1/6, 2/3, 1/6) of the periodic coordinate).
// Thread t of a row's CTA holds the elements t K .. t K + K - 1 in registers (K = 32 FP32, 16
// FP64; only the last chunk of a row may be shorter). The causal recurrence y_i = r_i + z y_{i-1}
// and the anticausal u_i = y_i + z u_{i+1} (z = sqrt(3) - 2) run chunk-locally from zero; a
// block-wide scan of the pairs (z^len, zero-start end value) gives each chunk its exact carry,
// and the periodic closure adds z^{i+1} y_{-1} with y_{-1} = E / (1 - z^L), E the zero-start
// value at L - 1 (anticausal: z^{L-i} u_L with u_L = S / (1 - z^L)), as FP64 whole-period tiles
// do within a warp. Nothing is truncated. A whole chunk takes its carry and closure as one term,
// z^{k+1} (carry + z^base y_{-1}), with the powers of z as compile-time constants.
// The row sits in shared memory with element c at c + V (c / (32 V)), V the elements of 16
// bytes: the coalesced 16-byte copies and the 16-byte chunk reads of a quarter warp then hit
// distinct banks. Rows are taken from the last one down: the step kernel wrote the high rows
// last (still in L2), and the next step reads the low rows first.
template <typename T>
__device__ __forceinline__ int xrow_idx(int c)
{
    constexpr int V = 16 / (int)sizeof(T), SH = sizeof(T) == 4 ? 5 : 4;
    return c + V * (c >> SH);
}

// 16 bytes of shared memory to and from V consecutive register elements
__device__ __forceinline__ void xload16(const float *p, float *v)
{
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}
__device__ __forceinline__ void xload16(const double *p, double *v)
{
    const double2 q = *reinterpret_cast<const double2 *>(p);
    v[0] = q.x;
    v[1] = q.y;
}
__device__ __forceinline__ void xstore16(float *p, const float *v)
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void xstore16(double *p, const double *v)
{
    *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
}

__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

template <typename T>
__device__ __forceinline__ void xscan_combine(T &A, T &b, T Ao, T bo)
{
    // (A, b) after (Ao, bo) along the recurrence: b + A bo, A Ao
    b = fma(A, bo, b);
    A *= Ao;
}

// asynchronous copies from global into shared memory (cp.async): the thread goes on while the
// copies land in the padded row layout; cp.async.wait_all waits for the thread's own copies
__device__ __forceinline__ void cp_async_16(void *dst, const void *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
template <int B>
__device__ __forceinline__ void cp_async_elem(void *dst, const void *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(B) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// start copying one mesh row into a padded shared-memory row buffer (16-byte copies when every
// row starts 16-byte aligned, else one element per copy)
template <typename T>
__device__ __forceinline__ void xrow_fetch(T *buf, const T *rin, int nx, bool vec)
{
    constexpr int V = 16 / (int)sizeof(T);
    if (vec)
        for (int q = threadIdx.x; q < nx / V; q += blockDim.x)
            cp_async_16(buf + xrow_idx<T>(q * V), rin + (size_t)q * V);
    else
        for (int c = threadIdx.x; c < nx; c += blockDim.x)
            cp_async_elem<(int)sizeof(T)>(buf + xrow_idx<T>(c), rin + c);
    cp_async_commit();
}

// Block-wide exclusive scan of the chunk pairs (A, b) of one recurrence direction: returns the
// value the recurrence carries into this thread's chunk, and in total the value at the row's far
// end (zero start). DOWN: the anticausal direction (from the last chunk down). One barrier: every
// warp combines the per-warp totals itself; each direction has its own sA, sB.
template <typename T, bool DOWN>
__device__ __forceinline__ T xrow_carry(T A, T b, T *sA, T *sB, T &total)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const T Ao = DOWN ? __shfl_down_sync(0xffffffffu, A, off) : __shfl_up_sync(0xffffffffu, A, off);
        const T bo = DOWN ? __shfl_down_sync(0xffffffffu, b, off) : __shfl_up_sync(0xffffffffu, b, off);
        if (DOWN ? lane + off < 32 : lane >= off) xscan_combine(A, b, Ao, bo);
    }
    if (lane == (DOWN ? 0 : 31)) {
        sA[warp] = A;
        sB[warp] = b;
    }
    T Ae = DOWN ? __shfl_down_sync(0xffffffffu, A, 1) : __shfl_up_sync(0xffffffffu, A, 1);
    T be = DOWN ? __shfl_down_sync(0xffffffffu, b, 1) : __shfl_up_sync(0xffffffffu, b, 1);
    if (lane == (DOWN ? 31 : 0)) {
        Ae = T(1);
        be = T(0);
    }
    __syncthreads();
    T c = T(0), cw = T(0);
    for (int k = 0; k < nwarps; ++k) {
        const int w = DOWN ? nwarps - 1 - k : k;
        if (w == warp) cw = c;
        c = fma(sA[w], c, sB[w]);
    }
    total = c;
    return fma(Ae, cw, be);
}

// Lambda_x^{-1} (times -1/(6z)) of one row whose elements base .. base + len - 1 this thread
// holds in v (len == K: a whole chunk), the threads of the block holding the row in order.
// sA, sB: [2][warps], one pair of arrays per direction (a row's causal scan and the next row's
// are separated by the anticausal scan's barrier and the row's store barrier).
template <typename T, int K>
__device__ __forceinline__ void xsolve_row_regs(T *v, const int len, const T zbase, const T zend, const T closure,
                                                T (*sA)[kXRowMaxThreads / 32], T (*sB)[kXRowMaxThreads / 32])
{
    const T z = (T)zconst(1);
    const bool whole = len == K;
    // causal sweep from zero, then the carry and the periodic closure
    T y = T(0), A = T(1);
    if (whole) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            y = fma(z, y, v[k]);
            v[k] = y;
        }
        A = (T)zconst(K);
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < len) {
                y = fma(z, y, v[k]);
                v[k] = y;
                A *= z;
            }
    }
    {
        T E;
        const T carry = xrow_carry<T, false>(A, y, sA[0], sB[0], E);
        const T yprev = E * closure;             // y_{-1} = y_{L-1}
        const T cin = fma(zbase, yprev, carry);  // element base + k: z^{k+1} cin
        if (whole) {
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = fma((T)zconst(k + 1), cin, v[k]);
        } else {
            T zk = z;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < len) {
                    v[k] = fma(zk, cin, v[k]);
                    zk *= z;
                }
        }
    }
    // anticausal sweep from zero at the chunk end, then the carry and the periodic closure
    T u = T(0);
    A = T(1);
    if (whole) {
#pragma unroll
        for (int k = K - 1; k >= 0; --k) {
            u = fma(z, u, v[k]);
            v[k] = u;
        }
        A = (T)zconst(K);
    } else {
#pragma unroll
        for (int k = K - 1; k >= 0; --k)
            if (k < len) {
                u = fma(z, u, v[k]);
                v[k] = u;
                A *= z;
            }
    }
    {
        T S;
        const T carry = xrow_carry<T, true>(A, u, sA[1], sB[1], S);
        const T unext = S * closure;   // u_L = u_0
        // element base + k: z^{len - k} (carry + z^{L - base - len} u_L)
        const T cin = len > 0 ? fma(zend, unext, carry) : T(0);
        if (whole) {
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = fma((T)zconst(K - k), cin, v[k]);
        } else {
            T zk = z;
#pragma unroll
            for (int k = K - 1; k >= 0; --k)
                if (k < len) {
                    v[k] = fma(zk, cin, v[k]);
                    zk *= z;
                }
        }
    }
}

// Persistent: each CTA takes rows np - 1 - blockIdx.x, then gridDim.x further down, and copies
// the next row into its second buffer while it solves the current one.
template <typename T, int K, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 3 : 1)
    xsolve_rows_kernel(const T *r, T *out, int nx, int np,   // r == out: in place
                       const double *__restrict__ scale, int tx, int tp, int ntx,
                       float *__restrict__ smax_out, unsigned *__restrict__ err, int row_stride, int nbuf)
{
    extern __shared__ __align__(16) unsigned char xs_raw[];
    T *buf0 = reinterpret_cast<T *>(xs_raw);
    int *tmax = reinterpret_cast<int *>(buf0 + (size_t)nbuf * row_stride);
    __shared__ T sA[2][kXRowMaxThreads / 32], sB[2][kXRowMaxThreads / 32];
    constexpr int V = 16 / (int)sizeof(T);
    const int tid = threadIdx.x;
    const bool vec = (nx % V) == 0;   // every row starts 16-byte aligned
    const T sh = sizeof(T) == 4 ? (T)scale[0] : T(-6) * (T)zconst(1);
    const T sl = sizeof(T) == 4 ? (T)scale[1] : T(0);
    const int base = tid * K;
    const int len = max(0, min(K, nx - base));
    // z^base, z^(nx - base - len) and 1 / (1 - z^nx) of the periodic closure, the same in every row. |z|^128 =
    // 6e-74: past that a power changes nothing it is added to (as FP64 powers in every row they were half of an
    // FP64 row's operations)
    const T zbase = base < 128 ? zpow<T>(base) : T(0), zend = nx - base - len < 128 ? zpow<T>(nx - base - len) : T(0);
    const T closure = nx < 128 ? T(1) / (T(1) - zpow<T>(nx)) : T(1);
    // A chunk lies in one tile when the tile width is a multiple of the chunk, as the planner's 224 is; for other widths
    // the maxima are found element by element (240: 38 instructions a node for 28, 0.112 ms for 0.095, 8192 x 8192)
    const bool one_tile = tx % K == 0;

    // zeros past the row end in every buffer (read with the last chunks, never stored)
    for (int b = 0; b < nbuf; ++b)
        for (int c = nx + tid; c < (int)blockDim.x * K; c += blockDim.x)
            buf0[(size_t)b * row_stride + xrow_idx<T>(c)] = T(0);
    if (sizeof(T) == 4)
        for (int k = tid; k < ntx; k += blockDim.x) tmax[k] = 0;
    after_previous_launch();
    int i = blockIdx.x;
    if (i < np) xrow_fetch(buf0, r + (size_t)(np - 1 - i) * nx, nx, vec);
    bool bad = false;
    for (int it = 0; i < np; i += gridDim.x, ++it) {
        const int row = np - 1 - i;
        T *cur = buf0 + (size_t)(nbuf == 2 ? (it & 1) : 0) * row_stride;
        cp_async_wait_all();
        __syncthreads();   // the row is in cur; the stores of the other buffer's row have read it
        const int inext = i + gridDim.x;
        if (nbuf == 2 && inext < np)
            xrow_fetch(buf0 + (size_t)((it + 1) & 1) * row_stride, r + (size_t)(np - 1 - inext) * nx, nx, vec);

        T v[K];
#pragma unroll
        for (int j = 0; j < K / V; ++j) xload16(cur + xrow_idx<T>(base + j * V), &v[j * V]);
        xsolve_row_regs<T, K>(v, len, zbase, zend, closure, sA, sB);

        // the scale -6z (FP32: the step's unit-DC-gain pair sh + sl), checks, per-tile max|s'|
        T chk = T(0);
        float m = 0.f;
        if (len == K) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                v[k] = sizeof(T) == 4 ? fma(v[k], sl, v[k] * sh) : v[k] * sh;
                if constexpr (sizeof(T) == 8) {
                    bad |= not_finite(v[k]);   // integer operations
                } else {
                    chk = fma(v[k], T(0), chk);
                    m = fmaxf(m, fabsf((float)v[k]));
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < len) {
                    v[k] = sizeof(T) == 4 ? fma(v[k], sl, v[k] * sh) : v[k] * sh;
                    chk = fma(v[k], T(0), chk);
                    m = fmaxf(m, fabsf((float)v[k]));
                }
        }
        bad |= chk != T(0);
        if (sizeof(T) == 4 && smax_out && len > 0) {
            if (one_tile) {
                if (m > 0.f) atomicMax(&tmax[base / tx], __float_as_int(m));
            } else {
                int tc = base / tx, nb = (tc + 1) * tx;
                m = 0.f;
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < len) {
                        if (base + k >= nb) {
                            if (m > 0.f) atomicMax(&tmax[tc], __float_as_int(m));
                            m = 0.f;
                            ++tc;
                            nb += tx;
                        }
                        m = fmaxf(m, fabsf((float)v[k]));
                    }
                if (m > 0.f) atomicMax(&tmax[tc], __float_as_int(m));
            }
        }
#pragma unroll
        for (int j = 0; j < K / V; ++j) xstore16(cur + xrow_idx<T>(base + j * V), &v[j * V]);
        __syncthreads();

        T *rout = out + (size_t)row * nx;
        if (vec) {
            int4 *o4 = reinterpret_cast<int4 *>(rout);
            for (int q = tid; q < nx / V; q += blockDim.x)
                o4[q] = *reinterpret_cast<const int4 *>(cur + xrow_idx<T>(q * V));
        } else {
            for (int c = tid; c < nx; c += blockDim.x) rout[c] = cur[xrow_idx<T>(c)];
        }
        if (sizeof(T) == 4 && smax_out) {
            int *mo = reinterpret_cast<int *>(smax_out) + (size_t)(row / tp) * ntx;
            for (int k = tid; k < ntx; k += blockDim.x) {
                const int mk = tmax[k];
                if (mk != 0) {
                    atomicMax(mo + k, mk);
                    tmax[k] = 0;
                }
            }
        }
        if (nbuf == 1 && inext < np) {
            __syncthreads();
            xrow_fetch(cur, r + (size_t)(np - 1 - inext) * nx, nx, vec);
        }
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(err, ERRF_NONFINITE);
}

void xrow_shape(int precision, int nx, int *threads, int *per)
{
    const int K = xrow_max_per(precision);
    *threads = 0;
    *per = 0;
    if (nx < 1 || (long)nx > (long)kXRowMaxThreads * K) return;
    *threads = ((nx + K - 1) / K + 31) / 32 * 32;
    *per = K;
}

// bytes of one padded row buffer (a multiple of 16): every chunk of every thread, with the pads
static size_t xrow_row_bytes(int precision, int nx)
{
    int t = 0, p = 0;
    xrow_shape(precision, nx, &t, &p);
    if (t == 0) return 0;
    const int V = precision == VP_FP64 ? 2 : 4, line = precision == VP_FP64 ? 16 : 32;
    const size_t sz = precision == VP_FP64 ? 8 : 4;
    const size_t n = (size_t)t * p;
    return ((n + V * (n / line) + V) * sz + 15) & ~(size_t)15;
}

// two row buffers (the next row is copied in while the current one is solved) when they fit
int xrow_buffers(int precision, int nx, int ntx)
{
    const size_t tm = precision == VP_FP64 ? 0 : (size_t)ntx * sizeof(int);
    return 2 * xrow_row_bytes(precision, nx) + tm <= (size_t)200 * 1024 ? 2 : 1;
}

size_t xrow_smem_bytes(int precision, int nx, int ntx)
{
    const size_t row = xrow_row_bytes(precision, nx);
    if (row == 0) return 0;
    return (size_t)xrow_buffers(precision, nx, ntx) * row +
           (precision == VP_FP64 ? 0 : (size_t)ntx * sizeof(int));
}

// block-size bound of the instantiation: rows up to 256 chunks (FP32 8192 nodes) keep their
// chunks in registers at two CTAs per SM; the larger forms serve longer rows
template <typename T>
static auto xrow_kernel(int threads)
{
    constexpr int K = sizeof(T) == 8 ? 16 : 32;
    return threads <= 256 ? xsolve_rows_kernel<T, K, 256>
                          : (threads <= 512 ? xsolve_rows_kernel<T, K, 512> : xsolve_rows_kernel<T, K, 1024>);
}

template <typename T>
static int xrow_grid_of(int nx, int np, int ntx)
{
    const int prec = sizeof(T) == 8 ? VP_FP64 : VP_FP32;
    int threads = 0, per = 0;
    xrow_shape(prec, nx, &threads, &per);
    if (threads == 0) return 0;
    const size_t smem = xrow_smem_bytes(prec, nx, ntx);
    auto k = xrow_kernel<T>(threads);
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return np;   // one CTA per row
    }
    const long g = (long)sms * (per_sm > 0 ? per_sm : 1);
    return (int)(g < np ? g : np);
}

int xrow_grid_size(int precision, int nx, int np, int ntx)
{
    return precision == VP_FP64 ? xrow_grid_of<double>(nx, np, ntx) : xrow_grid_of<float>(nx, np, ntx);
}

template <typename T>
cudaError_t launch_xsolve_rows(const T *r, T *out, int nx, int np, const double *scale, int tx, int tp,
                               int ntx, float *smax_out, unsigned *err, int grid, bool ahead, cudaStream_t s)
{
    const int prec = sizeof(T) == 8 ? VP_FP64 : VP_FP32;
    int threads = 0, per = 0;
    xrow_shape(prec, nx, &threads, &per);
    if (threads == 0) return cudaErrorInvalidValue;
    const size_t smem = xrow_smem_bytes(prec, nx, ntx);
    const int nbuf = xrow_buffers(prec, nx, ntx);
    const int stride = (int)(xrow_row_bytes(prec, nx) / sizeof(T));
    auto k = xrow_kernel<T>(threads);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    if (grid <= 0 || grid > np) grid = np;
    return launch_ahead(k, grid, threads, smem, s, ahead, r, out, nx, np, scale, tx, tp, ntx, smax_out, err, stride,
                        nbuf);
}

template cudaError_t launch_xsolve_rows<float>(const float *, float *, int, int, const double *, int, int,
                                               int, float *, unsigned *, int, bool, cudaStream_t);
template cudaError_t launch_xsolve_rows<double>(const double *, double *, int, int, const double *, int,
                                                int, int, float *, unsigned *, int, bool, cudaStream_t);

template cudaError_t launch_step_fused_batch<float>(const FusedArgs<float> *, int *, int *,
                                                    const int2 *, int, int, int, size_t, int, int,
                                                    cudaStream_t);
template size_t fused_smem_bytes<float>(int, int, int, int);
template size_t fused_smem_bytes<double>(int, int, int, int);
template cudaError_t launch_step_fused<float>(const FusedArgs<float> &, int, bool, cudaStream_t);
template cudaError_t launch_step_fused<double>(const FusedArgs<double> &, int, bool, cudaStream_t);
template cudaError_t launch_lambda_p_mul<float>(const float *, float *, int, int, float *, int, int, int,
                                                unsigned *, cudaStream_t);
template cudaError_t launch_lambda_p_mul<double>(const double *, double *, int, int, float *, int, int, int,
                                                 unsigned *, cudaStream_t);

}  // namespace vp
