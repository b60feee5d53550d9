// vp_walk64.cuh -- FP64 source walk of the one-pass kernel: [Lambda_p^{-1}] + push + deposit of one source
// column per thread, through a segment of the tile's rows.
//
// Bound by the FP64 pipe (2 operations per clock and SM on this GPU: a warp's instruction holds it for 16
// clocks), so what counts is FP64 operations per node and how many nodes a tile walks beside its own. Same
// form as the FP32 walk (vp_walk.cuh): rows downwards, an N x N ring of accumulators that follows the node,
// restarted where the next node is not one row further down in the same columns; integer keys decide, and
// floors cost one addition less than a compare and a correction would.
#pragma once

#include "vp_walk.cuh"

namespace vp {
namespace {

constexpr int kC64 = 24;      // rows per chunk of the p solve: one chunk serves a third of 64 rows and the B3 reach
constexpr int kHalo64 = 28;   // |z|^28 = 1e-16

struct Walk64 {
    const double *src;
    int nx, np;
    const RowEntry<double> *row, *rowc;   // the push's row table; the tile's copy in shared memory (row 0 of both)
    const double *piv_ib, *piv_cp;        // Thomas pivots of rows 0 .. kPivots, the last one the limit
    const WalkWin *W;
    double *win;
    int ws, lim;                          // window row stride and size in cells
    int WW, WP0, edge;
};

// floor of x and its fraction: adding 1.5 2^52 rounds to an integer in the low mantissa bits; the sign of what
// is left (an integer test) says whether it was rounded up. Valid for |x| < 2^31.
__device__ __forceinline__ int split64(double x, double &frac)
{
    const double magic = 6755399441055744.0;
    const double t = x + magic;
    const double r = x - (t - magic);
    const bool up = __double2hiint(r) < 0;   // rounded up (x - x is +0)
    frac = r + (up ? 1.0 : 0.0);
    return __double2loint(t) - (up ? 1 : 0);
}

template <int N, int BASIS>
__device__ __forceinline__ void weights64(double t, double *w)
{
    if (BASIS == VP_BASIS_TENT) {
        w[0] = 1.0 - t;
        w[1] = t;
    } else {
        // cubic B-spline at offsets 1 + t, t, 1 - t, 2 - t in ten operations: w[0] + w[3] = 1/6 + (t^2 - t) / 2, and
        // w[1] = 2/3 - t^2 + 3 w[3]; the third from the sum of one
        const double t2 = t * t;
        const double h = fma(0.5, fma(t, t, -t), 1.0 / 6.0);
        w[3] = t2 * (t * (1.0 / 6.0));
        w[0] = h - w[3];
        if (__double2hiint(w[0]) < 0) w[0] = 0.0;   // rounding at t near 1: the taps stay non-negative
        w[1] = fma(3.0, w[3], 2.0 / 3.0 - t2);
        w[2] = (1.0 - h) - w[1];
    }
}

// the row that leaves the ring, into the window at cell offset off
template <int N>
__device__ __forceinline__ void leave_row64(const Walk64 &K, const double *a, int off, double &lost)
{
    if ((unsigned)off < (unsigned)K.lim) {
        double *p = K.win + off;
#pragma unroll
        for (int q = 0; q < N; ++q) atomicAdd(p + q, a[q]);
    } else if (K.edge & (off < 0 ? 1 : 2)) {
        int c = off % K.ws;
        if (c < 0) c += K.ws;
#pragma unroll
        for (int q = 0; q < N; ++q)
            if (c + q >= K.W->own_c0 && c + q < K.W->own_c1) lost += a[q];
    }
}

// Walk rows r_hi .. r_lo (downwards) of source column im (window column colrel before the push). gc: the thread's
// column buffer (kC64 entries, nth apart).
template <int BASIS, bool GAL, bool UTERM, bool SROW>
__device__ __forceinline__ void walk_col64(const Walk64 &K, const ColEntry<double> e, int im, int colrel, int r_lo,
                                           int r_hi, double al, double be, double KU, double KV, double *gc, int nth,
                                           double &lost)
{
    constexpr int N = BASIS == VP_BASIS_TENT ? 2 : 4;
    constexpr int LO = BASIS == VP_BASIS_TENT ? 0 : -1;
    // sine term: al sin(a + y) + be cos(a + y) = cy (al sa + be ca) + sy (al ca - be sa)
    const double Pc = al * e.sa + be * e.ca, Qc = al * e.ca - be * e.sa;
    const double cv1 = KV * Pc, cv2 = KV * Qc, cu1 = KU * Pc, cu2 = KU * Qc;
    const int bu = colrel + e.ui + LO, bv = e.vi + LO - K.WP0;
    const double *src = K.src + im;
    const size_t pitch = (size_t)K.nx;
    double acc[N][N];
#pragma unroll
    for (int b = 0; b < N; ++b)
#pragma unroll
        for (int a = 0; a < N; ++a) acc[b][a] = 0.0;
    int ku = kRingDead, kv = 0, off = 0;
    const double sixth = 1.0 / 6.0;
    double uv = 0.0;
    bool first = true;
    const int nrows = r_hi - r_lo + 1, nch = (nrows + kC64 - 1) / kC64, per = (nrows + nch - 1) / nch;
    for (int c_hi = r_hi; c_hi >= r_lo;) {
        const int c_lo = max(r_lo, c_hi - per + 1), cn = c_hi - c_lo + 1;
        if (GAL) {
            // forward sweep from kHalo64 rows below the chunk (or from row 0), eight rows' loads at a time; in the
            // first chunk also over kHalo64 rows above it, where what the back substitution brings from there is
            // summed on the way up: sum_k prod(-c') g
            const int top = first ? min(K.np - 1, c_hi + kHalo64) : c_hi;
            const int r0 = max(0, c_lo - kHalo64);
            double gv = 0.0, c = 1.0, x[8];
            const double *p = src + (size_t)r0 * pitch;
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = r0 + k <= top ? __ldg(p + k * pitch) : 0.0;
            for (int rr = r0; rr <= top; rr += 8) {
                p += 8 * pitch;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int row = rr + k;
                    const double xk = x[k];
                    x[k] = row + 8 <= top ? __ldg(p + k * pitch) : 0.0;
                    if (row <= top) {
                        const int pr = min(row, kPivots);
                        gv = (xk - sixth * gv) * K.piv_ib[pr];
                        if (row >= c_lo && row <= c_hi) gc[(row - c_lo) * nth] = gv;
                        if (row > c_hi) {
                            uv = fma(c, gv, uv);
                            c *= -K.piv_cp[pr];
                        }
                    }
                }
            }
            first = false;
        } else {
            const double *p = src + (size_t)c_lo * pitch;
#pragma unroll
            for (int k = 0; k < kC64; ++k)
                if (k < cn) gc[k * nth] = __ldg(p + k * pitch);
        }
        const double *gp = gc + (cn - 1) * nth;
#pragma unroll 1
        for (int r = c_hi; r >= c_lo; --r, gp -= nth) {
            double w = *gp;
            if (GAL) w = uv = w - K.piv_cp[min(r, kPivots)] * uv;   // back substitution w_j = g_j - c'_j w_{j+1}
            const RowEntry<double> q = SROW ? K.rowc[r] : K.row[r];
            double fu = e.uf + q.uf, fv = e.vf + q.vf, tu, tv, wx[N], wy[N];
            if (UTERM) fu += cu1 * q.cy + cu2 * q.sy;
            fv = fv + cv1 * q.cy + cv2 * q.sy;
            const int nku = split64(fu, tu) + q.ui, nkv = split64(fv, tv) + q.vi;
            weights64<N, BASIS>(tu, wx);
            weights64<N, BASIS>(tv, wy);
#pragma unroll
            for (int b = 0; b < N; ++b) wy[b] *= w;
            if (nku != ku || nkv != kv) {
                if (ku != kRingDead) {
#pragma unroll
                    for (int b = N - 1; b >= 0; --b) leave_row64<N>(K, acc[b], off - (N - 1 - b) * K.ws, lost);
#pragma unroll
                    for (int b = 0; b < N; ++b)
#pragma unroll
                        for (int a = 0; a < N; ++a) acc[b][a] = 0.0;
                }
                ku = nku;
                kv = nkv;
                int m = nku + bu;
                if ((unsigned)m > (unsigned)(K.WW - N)) m = fold_col<N>(K.W, m);
                off = (r + nkv + bv + N) * K.ws + m;
            } else {
                leave_row64<N>(K, acc[N - 1], off, lost);
            }
            off -= K.ws;
#pragma unroll
            for (int b = N - 1; b > 0; --b)
#pragma unroll
                for (int a = 0; a < N; ++a) acc[b][a] = fma(wy[b], wx[a], acc[b - 1][a]);
#pragma unroll
            for (int a = 0; a < N; ++a) acc[0][a] = wy[0] * wx[a];
        }
        c_hi = c_lo - 1;
    }
#pragma unroll
    for (int b = N - 1; b >= 0; --b) leave_row64<N>(K, acc[b], off - (N - 1 - b) * K.ws, lost);
}

}  // namespace
}  // namespace vp
