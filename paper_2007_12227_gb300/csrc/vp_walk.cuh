// vp_walk.cuh -- FP32 source walk of the one-pass kernel: [Lambda_p^{-1}] + push + deposit of two
// adjacent source columns per thread in packed f32x2 arithmetic.
//
// What bounds the walk is instruction issue: the N x N taps, their weights and the push of every node,
// against 8 bytes of mesh traffic. Each thread therefore takes a PAIR of adjacent columns, column A in
// the low and column B in the high half of every 64-bit register, so that each FADD2 / FMUL2 / FFMA2
// does both nodes of a row: the p-solve recurrences, the push, the tap weights and the N x N taps, and the
// row's push entry, the loop and the test for the common case are paid once for two nodes. Two CTAs of 8
// warps share an SM (4 warps a sub-partition, 128 registers a thread). Measured on the 4096 x 4096
// pendulum step without its x solve: 61 M warp instructions and 0.123 ms, against 94 M and 0.150 ms for one
// column per thread with the (x, p) halves of a node packed; 8192 x 8192 with the deposit alone 0.357 ms
// against 0.473, in one pass with both solves 0.479 against 0.632 (0.395 and 0.512 while steps were not launched
// ahead and lost weight was added cell by cell in FP64).
//
// What mattered beside the packing, in instructions of the row loop: no function call in it (the calling
// convention cost moves and spills), no copy of the 32 accumulators between the common path and the restart
// (one path sets them; a restart only empties them first), no predicate on a shared-memory reduction (it
// becomes a branch around it), column entries by value (a reference was read again in every row), and the
// tile's constants kept in registers.
//
// A pair walks its rows downwards (the direction of the back substitution). The taps accumulate in an
// N x N ring per column, acc[b][a] = window row n + b, column m + a; when both nodes land one row
// further down in the same columns (the common case) the top row leaves the ring for the window.
// Anything else (first node, a column shift, a jump) adds the ring's rows to the window and restarts
// it.
#pragma once

#include "vp_internal.h"
#include "vp_sum.cuh"

namespace vp {
namespace {

// FP32 pairs in one 64-bit register, for packed FADD2 / FMUL2 / FFMA2
typedef unsigned long long f2_t;
__device__ __forceinline__ float2 f2_f(f2_t a) { return *reinterpret_cast<float2 *>(&a); }
__device__ __forceinline__ f2_t f2_u(float2 a) { return *reinterpret_cast<f2_t *>(&a); }
__device__ __forceinline__ f2_t f2_pack(float a, float b) { return f2_u(make_float2(a, b)); }
__device__ __forceinline__ f2_t f2_dup(float a) { return f2_pack(a, a); }
__device__ __forceinline__ float f2_lo(f2_t a) { return f2_f(a).x; }
__device__ __forceinline__ float f2_hi(f2_t a) { return f2_f(a).y; }
__device__ __forceinline__ void f2_unpack(f2_t r, float &a, float &b)
{
    a = f2_lo(r);
    b = f2_hi(r);
}
__device__ __forceinline__ f2_t f2_add(f2_t a, f2_t b)
{
    return f2_u(__fadd2_rn(f2_f(a), f2_f(b)));
}
__device__ __forceinline__ f2_t f2_sub(f2_t a, f2_t b)
{
    f2_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2_t f2_mul(f2_t a, f2_t b)
{
    return f2_u(__fmul2_rn(f2_f(a), f2_f(b)));
}
__device__ __forceinline__ f2_t f2_fma(f2_t a, f2_t b, f2_t c)
{
    return f2_u(__ffma2_rn(f2_f(a), f2_f(b), f2_f(c)));
}

// Shared memory by 32-bit address. (Through generic pointers the compiler rebuilt the window's base
// address in every turn of the row loop.) volatile keeps the accesses in order; the barriers around the
// walk are the usual ones.
__device__ __forceinline__ unsigned smem_addr(const void *p)
{
    unsigned a;
    asm volatile("mov.u32 %0, %1;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)));
    return a;
}
// a value the compiler does not rebuild from its inputs at every use
__device__ __forceinline__ int opaque(int x)
{
    asm volatile("mov.u32 %0, %0;" : "+r"(x));
    return x;
}
__device__ __forceinline__ void win_add(unsigned a, float v)
{
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(a), "r"(__float2int_rn(v)));
}
__device__ __forceinline__ f2_t lds_f2(unsigned a)
{
    f2_t r;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(r) : "r"(a));
    return r;
}
__device__ __forceinline__ void sts_f2(unsigned a, f2_t v)
{
    asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(v));
}
__device__ __forceinline__ float4 lds_f4(unsigned a)
{
    float4 r;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
                 : "r"(a)
                );
    return r;
}

// the tile's window as the walk's rare paths need it (in shared memory: no registers in the common path)
struct WalkWin {
    int WW;                  // window width
    int own_c0, own_c1;      // the columns whose lost weight the tile counts
    int nx;
    int wrap;                // the tile walks a whole period of source columns: first window column of the images that
                             // their nodes land at; else -1
};

// Weight of a row's cells a (window columns ca ..) and b (cb ..) that the tile counts as lost, countA, countB: the
// rows that are. Error-free sums of both columns in packed FP32 (the row's total to 2^-48), so that FP64, which
// runs at a 64th of the rate, is left with one addition a row: with the cells converted and added one by one,
// tiles beyond whose edge many rows land took 7000 cycles a source row (640 x 512 rotated by pi / 10: 240 us a step, 170
// so; the shorter code also helps meshes that lose nothing, 8192 x 8192 0.490 -> 0.479 ms).
template <int N>
__device__ __forceinline__ void lose_row(const WalkWin *W, const f2_t *acc, bool countA, int ca, bool countB, int cb,
                                         double &lost)
{
    const int o0 = W->own_c0, o1 = W->own_c1;
    f2_t hi = 0ull, lo = 0ull;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const f2_t x = f2_pack(countA && ca + q >= o0 && ca + q < o1 ? f2_lo(acc[q]) : 0.f,
                               countB && cb + q >= o0 && cb + q < o1 ? f2_hi(acc[q]) : 0.f);
        const f2_t t = f2_add(hi, x), y = f2_sub(t, hi);
        lo = f2_add(lo, f2_add(f2_sub(hi, f2_sub(t, y)), f2_sub(x, y)));
        hi = t;
    }
    DSum<float> s;
    s.add(f2_lo(hi));
    s.add(f2_hi(hi));
    s.lo += f2_lo(lo) + f2_hi(lo);
    if (s.hi != 0.f || s.lo != 0.f) lost += s.value();
}

// Window column of a node's first tap, m, where it lies outside [0, WW - N]. Where the tile walks a whole period of
// source columns, the node lands at its image: in a whole-period tile (from the first own column on) the N cells end in
// the right guard band at the latest, which is folded; a narrower window (from its first column on) holds one image
// of a column at most. What is still outside belongs to other tiles or to the guard band, at least N wide, which
// nobody reads: it is moved into the band.
template <int N>
__device__ __forceinline__ int fold_col(const WalkWin *W, int m)
{
    if (W->wrap >= 0) {
        m = (m - W->wrap) % W->nx;
        m += W->wrap + (m < 0 ? W->nx : 0);
    }
    return max(0, min(m, W->WW - N));
}

// One pair's state. The integer displacement of a node is the low mantissa bits of (fraction + 1.5 2^23)
// plus the row's integer part; ku, kv hold that sum for the ring's nodes, so an unchanged set of keys in
// the next row down means: same columns, one row further down.
template <int N>
struct PairRing {
    f2_t acc[N][N];    // [row b][column a]
    int kuA, kuB, kvA, kvB;
    int off;           // window offset (bytes) of column A's leaving row at the next row
    int dBA;           // offset (bytes) of B's cells relative to A's
    int cA, cB;        // window offset (bytes) of their first columns in window row 0
};
constexpr int kRingDead = (int)0x80000000;   // a key no node has

// Lambda_p^{-1} of FP32: Thomas pivots from this row on equal their limits in FP32 (the difference
// falls as |z|^(2 r): |z|^24 = 2e-14)
constexpr int kPiv32 = 12;
// rows per chunk of the p solve: two chunks serve a segment of half the default tile (64 rows, the B3
// reach and the spread of the displacements), each after kHalo32 warm-up rows
constexpr int kC32 = 18;
constexpr int kHalo32 = 16;   // |z|^16 = 7e-10

struct Walk32 {
    const float *src;      // the state read
    int nx, np;
    const RowEntry<float> *row;   // the push's row table (global memory)
    unsigned rowc;         // shared-memory address of entry 0 of the tile's copy
    const float2 *piv;     // (1 / beta, c') of rows 0 .. kPiv32, the last one the limit (shared memory)
    const WalkWin *W;
    unsigned win;
    int ws4, lim;          // bytes of a window row, of the window
    int WW, WP0;
    int edge;              // the open edges the tile owns (1: the first mesh row, 2: the last): it counts the weight lost there
};

// One row of a pair's rings into the window. Rows outside the window belong to other tiles: they are clamped
// into the window's guard rows (a predicate on a shared-memory reduction becomes a branch around it), in their own
// columns (one common place for them all serialised the warp's additions: 3900 cycles a row where strong shear carries
// most rows outside). Guard rows are read only in a tile that owns an open edge, and on that edge's side: there the
// rows beyond count as lost here, and zeros are added in their place.
template <int N>
__device__ __forceinline__ void leave_row(const Walk32 &K, const f2_t *acc, int off, int dBA, int cA, int cB, double &lost)
{
    float a[N], b[N];
#pragma unroll
    for (int q = 0; q < N; ++q) f2_unpack(acc[q], a[q], b[q]);
    if (K.edge) {
        const bool inA = (unsigned)off < (unsigned)K.lim, inB = (unsigned)(off + dBA) < (unsigned)K.lim;
        if (!(inA && inB)) {
            lose_row<N>(K.W, acc, !inA && (K.edge & (off < 0 ? 1 : 2)), cA >> 2,
                        !inB && (K.edge & (off + dBA < 0 ? 1 : 2)), cB >> 2, lost);
#pragma unroll
            for (int q = 0; q < N; ++q) {
                a[q] = inA ? a[q] : 0.f;
                b[q] = inB ? b[q] : 0.f;
            }
        }
    }
    const int top = K.lim - K.ws4;
    const unsigned pA = K.win + (unsigned)max(cA, min(off, top + cA)),
                   pB = K.win + (unsigned)max(cB, min(off + dBA, top + cB));
#pragma unroll
    for (int q = 0; q < N; ++q) win_add(pA + 4 * q, a[q]);
#pragma unroll
    for (int q = 0; q < N; ++q) win_add(pB + 4 * q, b[q]);
}

// The whole ring, top row first (off: its offset), which leaves it empty.
template <int N>
__device__ __forceinline__ void leave_ring(const Walk32 &K, f2_t (&acc)[N][N], int off, int dBA, int cA, int cB, double &lost)
{
#pragma unroll
    for (int k = 0; k < N; ++k, off -= K.ws4) {
        leave_row<N>(K, acc[N - 1], off, dBA, cA, cB, lost);
#pragma unroll
        for (int b = N - 1; b > 0; --b)
#pragma unroll
            for (int a = 0; a < N; ++a) acc[b][a] = acc[b - 1][a];
#pragma unroll
        for (int a = 0; a < N; ++a) acc[0][a] = 0ull;
    }
}

template <int N, int BASIS>
__device__ __forceinline__ void pair_weights(f2_t F, f2_t &bits, f2_t *w)
{
    // base cell round(x - 1/2), so that the fraction t lies in [0, 1] (t = 1 at an exact node gives the
    // same deposit as t = 0 one cell further: the B3 and tent kernels are continuous)
    const f2_t ONE = f2_dup(1.f), MAG = f2_dup(12582912.f);   // 1, 1.5 * 2^23
    bits = f2_add(f2_add(F, f2_dup(-0.5f)), MAG);
    const f2_t T = f2_sub(F, f2_sub(bits, MAG));
    const f2_t S = f2_sub(ONE, T);
    if (BASIS == VP_BASIS_TENT) {
        w[0] = S;
        w[1] = T;
    } else {
        // three weights rounded to multiples of 2^-23 ((x + 1) - 1), the fourth 1 minus them: every step
        // of that is exact and the four sum to exactly one, so the step keeps the mass up to unbiased
        // rounding whatever the fractions (a node pushed by whole cells would otherwise lose 2^-26 of
        // its weight per axis and step)
        const f2_t T2 = f2_mul(T, T), S2 = f2_mul(S, S);
        const f2_t SIX = f2_dup(1.f / 6.f);
        const f2_t S3 = f2_mul(S2, S), T3 = f2_mul(T2, T);
        w[0] = f2_sub(f2_fma(S3, SIX, ONE), ONE);
        w[3] = f2_sub(f2_fma(T3, SIX, ONE), ONE);
        const f2_t H = f2_fma(T, f2_dup(0.5f), f2_dup(-1.f));
        w[1] = f2_sub(f2_add(f2_fma(T2, H, f2_dup(2.f / 3.f)), ONE), ONE);
        w[2] = f2_sub(f2_sub(f2_sub(ONE, w[0]), w[3]), w[1]);
    }
}

// the source values of row k of a chunk; VEC: one 8-byte load (the pair is aligned and does not wrap).
// volatile: the two forms stay apart (merged, both were issued under predicates)
template <bool VEC>
__device__ __forceinline__ f2_t load_pair(const char *pA, const char *pB, unsigned pitch, unsigned k)
{
    const size_t o = (size_t)k * pitch;   // 32 x 32 -> 64 bits
    f2_t v;
    if (VEC) {
        asm volatile("ld.global.nc.b64 %0, [%1];" : "=l"(v) : "l"(pA + o));
    } else {
        float a, b;
        asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(a) : "l"(pA + o));
        asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(b) : "l"(pB + o));
        v = f2_pack(a, b);
    }
    return v;
}

// forward sweep g_j = (s_j - g_{j-1} / 6) / beta_j with the limit pivots over kHalo32 + kC32 rows from
// pA, pB on; the last kC32 rows go to the column buffer. FIRST: na more rows above them start the back
// substitution: uv = sum_k (-c')^k g_{j + k} of the rows j = top + 1, ... (what lies beyond kHalo32 rows weighs
// |z|^kHalo32), summed on the way up, so that they need no room. kFly rows' loads are always in flight ahead of
// the recurrence.
template <bool VEC, bool FIRST>
__device__ __forceinline__ void forward_far(const char *pA, const char *pB, unsigned pitch, f2_t IBq, f2_t NIB6,
                                            float ncp, int na, unsigned gc, unsigned gs, f2_t &uv)
{
    constexpr int kFly = 16, kRows = kHalo32 + kC32;
    static_assert(kHalo32 <= kFly, "the loads of the look-ahead above the top row fit those in flight");
    f2_t x[kFly], gv = 0ull;
#pragma unroll
    for (int k = 0; k < kFly; ++k) x[k] = load_pair<VEC>(pA, pB, pitch, k);
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        gv = f2_fma(NIB6, gv, f2_mul(x[k % kFly], IBq));
        if (k + kFly < kRows) x[k % kFly] = load_pair<VEC>(pA, pB, pitch, k + kFly);
        else if (FIRST && k + kFly - kRows < na) x[k % kFly] = load_pair<VEC>(pA, pB, pitch, k + kFly);
        if (k >= kHalo32) sts_f2(gc + (k - kHalo32) * gs, gv);
    }
    if (FIRST) {
        float c = 1.f;
#pragma unroll
        for (int k = 0; k < kFly; ++k)
            if (k < na) {
                gv = f2_fma(NIB6, gv, f2_mul(x[(kRows + k) % kFly], IBq));
                uv = f2_fma(f2_dup(c), gv, uv);
                c *= ncp;
            }
    }
}

// Walk rows r_hi .. r_lo (downwards) of the source columns imA, imB (window columns colrel, colrel + 1
// before the push). gc: shared-memory address of the thread's column buffer (kC32 entries, gs bytes
// apart). q2: the window scale per column (0 for a column that is not there). SROW: the row table is in
// shared memory.
template <int BASIS, bool GAL, bool UTERM, bool SROW>
__device__ __forceinline__ void walk_pair(const Walk32 &K, const ColEntry<float> eA, const ColEntry<float> eB,
                                          int imA, int imB, int colrel, int r_lo, int r_hi, f2_t q2, float al,
                                          float be, float KU, float KV, unsigned gc, unsigned gs, double &lost)
{
    constexpr int N = BASIS == VP_BASIS_TENT ? 2 : 4;
    constexpr int LO = BASIS == VP_BASIS_TENT ? 0 : -1;
    constexpr int kBias = 0x4B400000;   // bits of 1.5 * 2^23
    // sine term: al sin(a + y) + be cos(a + y) = cy (al sa + be ca) + sy (al ca - be sa)
    const float PA = al * eA.sa + be * eA.ca, QA = al * eA.ca - be * eA.sa;
    const float PB = al * eB.sa + be * eB.ca, QB = al * eB.ca - be * eB.sa;
    const f2_t cv1 = f2_pack(KV * PA, KV * PB), cv2 = f2_pack(KV * QA, KV * QB);
    // KU s from KV s: both are multiples of the same step. (The quotient's rounding, 6e-8 of the kick along x, is
    // of the size of KU's own in FP32; it saves two pairs of column constants)
    const f2_t KR = f2_dup(KV != 0.f ? KU / KV : 0.f);
    // window column / row of the first tap = key + base (+ the row index)
    const int buA = colrel + eA.ui - kBias + LO, buB = colrel + 1 + eB.ui - kBias + LO;
    const int bvA = eA.vi - kBias + LO - K.WP0, bvB = eB.vi - kBias + LO - K.WP0;
    const bool vec = imB == imA + 1 && ((imA | K.nx) & 1) == 0;
    const unsigned pitch = (unsigned)K.nx * 4u;
    const char *sA = reinterpret_cast<const char *>(K.src + imA), *sB = reinterpret_cast<const char *>(K.src + imB);

    PairRing<N> g;
    g.kuA = kRingDead;
    g.kuB = g.kvA = g.kvB = 0;
    g.off = g.dBA = g.cA = g.cB = 0;
#pragma unroll
    for (int b = 0; b < N; ++b)
#pragma unroll
        for (int a = 0; a < N; ++a) g.acc[b][a] = 0ull;

    const float sixth = 1.f / 6.f;
    const float2 pinf = GAL ? K.piv[kPiv32] : make_float2(0.f, 0.f);
    const f2_t IBq = f2_mul(f2_dup(pinf.x), q2);      // the window scale (a power of two) rides on the solve
    const f2_t NIB6 = f2_dup(-(sixth * pinf.x));
    f2_t NCP = f2_dup(-pinf.y);
    f2_t uv = 0ull;

    const int nrows = r_hi - r_lo + 1, nch = (nrows + kC32 - 1) / kC32, per = (nrows + nch - 1) / nch;
    bool first = true;
    for (int c_hi = r_hi; c_hi >= r_lo;) {
        const int c_lo = max(r_lo, c_hi - per + 1);
        const int b0 = c_hi - kC32 + 1;   // the row of column buffer entry 0
        if (GAL) {
            const int na = min(K.np - 1, r_hi + kHalo32) - r_hi;   // rows of the look-ahead above the top row
            if (b0 - kHalo32 >= kPiv32) {
                const size_t o = (size_t)(b0 - kHalo32) * pitch;
                if (vec) {
                    if (first) forward_far<true, true>(sA + o, sB + o, pitch, IBq, NIB6, -pinf.y, na, gc, gs, uv);
                    else forward_far<true, false>(sA + o, sB + o, pitch, IBq, NIB6, -pinf.y, 0, gc, gs, uv);
                } else {
                    if (first) forward_far<false, true>(sA + o, sB + o, pitch, IBq, NIB6, -pinf.y, na, gc, gs, uv);
                    else forward_far<false, false>(sA + o, sB + o, pitch, IBq, NIB6, -pinf.y, 0, gc, gs, uv);
                }
                NCP = f2_dup(-pinf.y);
            } else {
                // near the first row: exact pivots, eight rows' loads at a time, and the back substitution
                // with its own factors, so that the column buffer holds the weights
                f2_t gv = 0ull;
                const int top = first ? c_hi + na : c_hi;
                float c = 1.f;
                for (int rr = max(0, c_lo - kHalo32); rr <= top; rr += 8) {
                    f2_t x[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const size_t o = (size_t)min(rr + k, top) * pitch;
                        x[k] = vec ? load_pair<true>(sA + o, sB + o, pitch, 0) : load_pair<false>(sA + o, sB + o, pitch, 0);
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int row = rr + k;
                        if (row <= top) {
                            const float2 pv = K.piv[min(row, kPiv32)];
                            gv = f2_mul(f2_fma(f2_dup(-sixth), gv, f2_mul(x[k], q2)), f2_dup(pv.x));
                            if (row >= c_lo && row <= c_hi) sts_f2(gc + (row - b0) * gs, gv);
                            if (row > c_hi) {
                                uv = f2_fma(f2_dup(c), gv, uv);
                                c *= -pv.y;
                            }
                        }
                    }
                }
                f2_t u = uv;
                for (int r = c_hi; r >= c_lo; --r) {
                    u = f2_fma(f2_dup(-K.piv[min(r, kPiv32)].y), u, lds_f2(gc + (r - b0) * gs));
                    sts_f2(gc + (r - b0) * gs, u);
                }
                NCP = 0ull;
            }
            first = false;
        } else {
            // the deposit alone: the chunk's loads are issued together, kept in the column buffer
            const size_t o = (size_t)c_lo * pitch;
            const int cn = c_hi - c_lo + 1, k0 = c_lo - b0;
            if (vec) {
#pragma unroll
                for (int k = 0; k < kC32; ++k)
                    if (k < cn) sts_f2(gc + (k0 + k) * gs, f2_mul(load_pair<true>(sA + o, sB + o, pitch, k), q2));
            } else {
#pragma unroll
                for (int k = 0; k < kC32; ++k)
                    if (k < cn) sts_f2(gc + (k0 + k) * gs, f2_mul(load_pair<false>(sA + o, sB + o, pitch, k), q2));
            }
        }

        unsigned gp = gc + (kC32 - 1) * gs;
        unsigned rs = K.rowc + (unsigned)c_hi * (unsigned)sizeof(RowEntry<float>);
        const float4 *rp = reinterpret_cast<const float4 *>(K.row + c_hi);
#pragma unroll 1
        for (int r = c_hi; r >= c_lo; --r) {
            f2_t w2 = lds_f2(gp);
            if (GAL) w2 = uv = f2_fma(NCP, uv, w2);   // back substitution w_j = g_j - c' w_{j+1}
            // ui, vi, uf, vf; cy, cy, sy, sy
            const float4 q0 = SROW ? lds_f4(rs) : __ldg(rp), q1 = SROW ? lds_f4(rs + 16) : __ldg(rp + 1);
            gp -= gs;
            rs -= (unsigned)sizeof(RowEntry<float>);
            rp -= 2;
            const f2_t CY = f2_pack(q1.x, q1.y), SY = f2_pack(q1.z, q1.w);
            f2_t Fu = f2_pack(eA.uf + q0.z, eB.uf + q0.z);
            f2_t Fv = f2_pack(eA.vf + q0.w, eB.vf + q0.w);
            // (with UTERM and KU = 0, as a pendulum in a batch, the same bits as without)
            if (UTERM) Fu = f2_fma(KR, f2_fma(cv2, SY, f2_mul(cv1, CY)), Fu);
            Fv = f2_fma(cv2, SY, f2_fma(cv1, CY, Fv));
            f2_t bu, bv, wx[N], wy[N];
            pair_weights<N, BASIS>(Fu, bu, wx);
            pair_weights<N, BASIS>(Fv, bv, wy);
            const int ri = __float_as_int(q0.x), rj = __float_as_int(q0.y);
            const int kuA = __float_as_int(f2_lo(bu)) + ri, kuB = __float_as_int(f2_hi(bu)) + ri;
            const int kvA = __float_as_int(f2_lo(bv)) + rj, kvB = __float_as_int(f2_hi(bv)) + rj;
#pragma unroll
            for (int b = 0; b < N; ++b) wy[b] = f2_mul(wy[b], w2);
            const int diff = (kuA ^ g.kuA) | (kuB ^ g.kuB) | (kvA ^ g.kvA) | (kvB ^ g.kvB);
            if (diff != 0) {
                // not one row further down in the same columns: the ring goes to the window and starts
                // again (empty, so that the common path below sets it to this node)
                if (g.kuA != kRingDead) leave_ring<N>(K, g.acc, g.off, g.dBA, g.cA, g.cB, lost);
                int mA = kuA + buA, mB = kuB + buB;
                const unsigned cmax = (unsigned)(K.WW - N);
                if ((unsigned)mA > cmax) mA = fold_col<N>(K.W, mA);
                if ((unsigned)mB > cmax) mB = fold_col<N>(K.W, mB);
                g.kuA = kuA;
                g.kuB = kuB;
                g.kvA = kvA;
                g.kvB = kvB;
                g.cA = 4 * mA;
                g.cB = 4 * mB;
                g.off = (r + kvA + bvA + N) * K.ws4 + g.cA;
                g.dBA = (r + kvB + bvB + N) * K.ws4 + g.cB - g.off;
            }
            // the top row leaves, the others move up
            leave_row<N>(K, g.acc[N - 1], g.off, g.dBA, g.cA, g.cB, lost);
            g.off -= K.ws4;
#pragma unroll
            for (int b = N - 1; b > 0; --b)
#pragma unroll
                for (int a = 0; a < N; ++a) g.acc[b][a] = f2_fma(wy[b], wx[a], g.acc[b - 1][a]);
#pragma unroll
            for (int a = 0; a < N; ++a) g.acc[0][a] = f2_mul(wy[0], wx[a]);
        }
        c_hi = c_lo - 1;
    }
    leave_ring<N>(K, g.acc, g.off, g.dBA, g.cA, g.cB, lost);
}

}  // namespace
}  // namespace vp
