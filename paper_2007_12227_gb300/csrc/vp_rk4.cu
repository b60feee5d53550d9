// vp_rk4.cu -- the FEL step with the classical fourth-order Runge-Kutta integrator (Sec. IV.B:
// the paper integrates its FEL equations with RK4).
//
// Every mesh node is a particle of d theta/dz = delta + eta, d eta/dz = -(K e^{i theta} + c.c.)
// with K = A + i sigma2 <e^{-i theta}>; A moves by dA/dz = <e^{-i theta}>. The four stages
// need the bunching b_s of all particles at their stage-s phases,
//   theta_1 = theta                      f_s = -2 Re(K_s e^{i theta_s})
//   theta_2 = theta + h/2 (delta + p)    (half drift of the row)
//   theta_3 = theta_2 + h^2/4 f_1        (f_1 depends on the column only)
//   theta_4 = theta + h (delta + p) + h^2/2 f_2
// so, with (rc, rs)_j = e^{i h/2 (delta + p_j)} tabulated per row:
//   b_1 is the bunching of the mesh weights, which the last field update left;
//   b_2 and b_3 both come from the column sums of w rc and w rs: e^{i theta_2} and e^{i theta_3} are a
//   factor of the column times (rc, rs), and theta_3 needs K_1 only: one pass over the weights;
//   b_4 takes a second pass (f_2 mixes row and column), then comes the deposit of every node at
//   theta + h (delta + p) + h^2/6 (f_1 + f_2 + f_3), p + h/6 (f_1 + 2 f_2 + 2 f_3 + f_4),
//   and A' = A + h/6 (b_1 + 2 b_2 + 2 b_3 + b_4), kept in the state for the field update.
// Bound by the FP64 pipe (2 operations per clock and SM): the phases are rotations of tabulated ones, and
// the one angle left per node, h^2/2 f_2, is small and takes a short series (four sums with up to three
// sincos a node each, and 16 blocks for 512 x 256, took 0.51 ms a step there). The push is evaluated in
// FP64 as increments from the node whatever the precision of the weights, so the FP32 path keeps sub-cell
// positions. This path is the paper's integrator for validation; the one-pass drift-kick-drift kernel is
// the fast path.
#include <math.h>

#include "vp_internal.h"

namespace vp {
namespace {

constexpr int kThreads = 128;
constexpr int kWarpRows = 8;                             // rows a warp takes of its 32 columns
constexpr int kRows = kWarpRows * (kThreads / 32);       // rows of a block
constexpr int kAmp = 256;                                // threads of the amplitude kernels

// e^{i x}: its series for the small angles of the fourth stage (below 2^-6 the first term left out is under
// 2^-70), else sincos
__device__ __forceinline__ void phase(double x, double &c, double &s)
{
    if (fabs(x) < 0.015625) {
        const double q = x * x;
        s = x * fma(q, fma(q, fma(q, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), 1.0);
        c = fma(q, fma(q, fma(q, fma(q, 1.0 / 40320.0, -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
    } else {
        sincos(x, &s, &c);
    }
}
__device__ __forceinline__ void rotate(double &c, double &s, double rc, double rs)
{
    const double t = c * rc - s * rs;
    s = s * rc + c * rs;
    c = t;
}
__device__ __forceinline__ double force(const double *K, double c, double s) { return -2.0 * (K[0] * c - K[1] * s); }

// K_1 = A + i sigma2 b_1
__device__ __forceinline__ void first_amp(const double *state, double sigma2, double *K)
{
    K[0] = state[ST_A_RE] - sigma2 * state[ST_B_IM];
    K[1] = state[ST_A_IM] + sigma2 * state[ST_B_RE];
}

// sums of NV values over the block (fixed order) into part[NV blockIdx]
template <int NV>
__device__ __forceinline__ void block_sums(const double *v, double *part)
{
    __shared__ double s_red[NV][kThreads / 32];
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double t = v[q];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) s_red[q][wy] = t;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int k = 0; k < kThreads / 32; ++k) t += s_red[threadIdx.x][k];
        part[(size_t)NV * blockIdx.x + threadIdx.x] = t;
    }
}

// stages 2 and 3: sum w, then (sum w cos, sum w sin) of theta_2 and of theta_3
template <typename T>
__global__ void __launch_bounds__(kThreads)
    rk4_mid_kernel(const T *__restrict__ w, Geometry g, const double2 *__restrict__ csx, const double *__restrict__ rt,
                   const double *__restrict__ state, double *part)
{
    const int strips = (g.nx + 31) / 32, lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int col = (int)(blockIdx.x % strips) * 32 + lane;
    const int r0 = (int)(blockIdx.x / strips) * kRows + wy * kWarpRows, r1 = min(r0 + kWarpRows, g.np);
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (col < g.nx) {
        T x[kWarpRows];
#pragma unroll
        for (int k = 0; k < kWarpRows; ++k) x[k] = r0 + k < r1 ? w[(size_t)(r0 + k) * g.nx + col] : T(0);
        double m = 0.0, C = 0.0, S = 0.0;
#pragma unroll
        for (int k = 0; k < kWarpRows; ++k)
            if (r0 + k < r1) {
                const double ww = (double)x[k];
                m += ww;
                C = fma(ww, rt[r0 + k], C);
                S = fma(ww, rt[g.np + r0 + k], S);
            }
        double K1[2];
        first_amp(state, g.sigma2, K1);
        double2 e = csx[col];
        v[0] = m;
        v[1] = e.x * C - e.y * S;
        v[2] = e.y * C + e.x * S;
        double c, s;
        phase(0.25 * g.dt * g.dt * force(K1, e.x, e.y), c, s);
        rotate(e.x, e.y, c, s);
        v[3] = e.x * C - e.y * S;
        v[4] = e.y * C + e.x * S;
    }
    block_sums<5>(v, part);
}

// stage 4: sum w, sum w cos theta_4, sum w sin theta_4
template <typename T>
__global__ void __launch_bounds__(kThreads)
    rk4_last_kernel(const T *__restrict__ w, Geometry g, const double2 *__restrict__ csx, const double *__restrict__ rt,
                    const double *__restrict__ state, double *part)
{
    const int strips = (g.nx + 31) / 32, lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int col = (int)(blockIdx.x % strips) * 32 + lane;
    const int r0 = (int)(blockIdx.x / strips) * kRows + wy * kWarpRows, r1 = min(r0 + kWarpRows, g.np);
    double v[3] = {0.0, 0.0, 0.0};
    if (col < g.nx) {
        const double K2[2] = {state[ST_RK_K + 2], state[ST_RK_K + 3]};
        const double2 e = csx[col];
        T x[kWarpRows];
#pragma unroll
        for (int k = 0; k < kWarpRows; ++k) x[k] = r0 + k < r1 ? w[(size_t)(r0 + k) * g.nx + col] : T(0);
#pragma unroll
        for (int k = 0; k < kWarpRows; ++k) {
            const double ww = (double)x[k];
            if (ww == 0.0) continue;
            const double rc = rt[r0 + k], rs = rt[g.np + r0 + k];
            double c = e.x, s = e.y, ec, es;
            rotate(c, s, rc, rs);
            phase(0.5 * g.dt * g.dt * force(K2, c, s), ec, es);
            rotate(c, s, rc, rs);
            rotate(c, s, ec, es);
            v[0] += ww;
            v[1] = fma(ww, c, v[1]);
            v[2] = fma(ww, s, v[2]);
        }
    }
    block_sums<3>(v, part);
}

// bunchings from the partial sums (fixed order) and the stage amplitudes K_s = A_s + i sigma2 b_s. last = 0: b_2, b_3
// (with b_1 from the state); last = 1: b_4, and A' = A + h/6 (b_1 + 2 b_2 + 2 b_3 + b_4) into ST_AH (the field update
// stores it)
__global__ void rk4_amp_kernel(const double *__restrict__ part, int nparts, double *state, int last, double dt,
                               double sigma2)
{
    __shared__ double s[5][kAmp];
    const int nv = last ? 3 : 5;
    double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int k = threadIdx.x; k < nparts; k += blockDim.x)
#pragma unroll
        for (int q = 0; q < 5; ++q)
            if (q < nv) a[q] += part[(size_t)nv * k + q];
#pragma unroll
    for (int q = 0; q < 5; ++q) s[q][threadIdx.x] = a[q];
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int q = 0; q < nv; ++q) s[q][threadIdx.x] += s[q][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    double *b = state + ST_RK_B, *K = state + ST_RK_K;
    const double ar = state[ST_A_RE], ai = state[ST_A_IM];
    if (!last) {
        b[0] = state[ST_B_RE];
        b[1] = state[ST_B_IM];
        first_amp(state, sigma2, K);
        for (int st = 1; st < 3; ++st) {
            b[2 * st] = s[2 * st - 1][0] / s[0][0];
            b[2 * st + 1] = -s[2 * st][0] / s[0][0];
            K[2 * st] = ar + 0.5 * dt * b[2 * st - 2] - sigma2 * b[2 * st + 1];
            K[2 * st + 1] = ai + 0.5 * dt * b[2 * st - 1] + sigma2 * b[2 * st];
        }
    } else {
        b[6] = s[1][0] / s[0][0];
        b[7] = -s[2][0] / s[0][0];
        K[6] = ar + dt * b[4] - sigma2 * b[7];
        K[7] = ai + dt * b[5] + sigma2 * b[6];
        state[ST_AH_RE] = ar + dt / 6.0 * (b[0] + 2.0 * b[2] + 2.0 * b[4] + b[6]);
        state[ST_AH_IM] = ai + dt / 6.0 * (b[1] + 2.0 * b[3] + 2.0 * b[5] + b[7]);
    }
}

template <typename T, int BASIS>
struct RkTaps;
template <typename T>
struct RkTaps<T, VP_BASIS_TENT> {
    static constexpr int N = 2, LO = 0;
    __device__ static void weights(T t, T *w)
    {
        w[0] = T(1) - t;
        w[1] = t;
    }
};
template <typename T>
struct RkTaps<T, VP_BASIS_SEPTIC_BSPLINE> {
    static constexpr int N = 8, LO = -3;
    __device__ static void weights(T t, T *w) { septic_weights<T>(t, w); }
};
template <typename T>
struct RkTaps<T, VP_BASIS_CUBIC_BSPLINE> {
    static constexpr int N = 4, LO = -1;
    __device__ static void weights(T t, T *w)
    {
        const T s = T(1) - t, t2 = t * t, t3 = t2 * t;
        const T sixth = T(1) / T(6);   // a product: a division is a dozen FP64 operations
        w[0] = s * s * s * sixth;
        w[3] = t3 * sixth;
        w[1] = T(2) / T(3) - t2 + T(0.5) * t3;
        w[2] = (T(1) - (w[0] + w[3])) - w[1];
    }
};

// Deposit of every node at its RK4 end point into a zeroed destination. A warp walks 32 columns upwards through
// kWarpRows rows; the taps of a column gather in an N x N ring of registers that follows the node (tent and cubic
// deposits), so that a row's cells go out once as the ring leaves it instead of N times.
template <typename T, int BASIS>
__global__ void __launch_bounds__(kThreads)
    rk4_deposit_kernel(const T *__restrict__ src, T *__restrict__ dst, Geometry g, const double2 *__restrict__ csx,
                       const double *__restrict__ rt, const double *__restrict__ state, double *lost_acc)
{
    using TP = RkTaps<T, BASIS>;
    constexpr int N = TP::N;
    constexpr bool RING = N <= 4;
    constexpr int NR = RING ? N : 1;
    __shared__ double s_red[kThreads / 32];
    const int nx = g.nx, np = g.np;
    const int strips = (nx + 31) / 32, lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int col = (int)(blockIdx.x % strips) * 32 + lane;
    const int r0 = (int)(blockIdx.x / strips) * kRows + wy * kWarpRows, r1 = min(r0 + kWarpRows, np);
    double lost = 0.0;
    // cells a .. of row rr at column base m (0 <= m < nx)
    auto put = [&](const T *v, int m, long rr) {
        if (rr < 0 || rr >= np) {
#pragma unroll
            for (int a = 0; a < N; ++a) lost += (double)v[a];
            return;
        }
        T *d = dst + (size_t)rr * nx;
        int c = m;
#pragma unroll
        for (int a = 0; a < N; ++a) {
            atomicAdd(d + c, v[a]);
            if (++c == nx) c = 0;
        }
    };
    if (col < nx) {
        double K[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) K[q] = state[ST_RK_K + q];
        const double h = g.dt, ihx = 1.0 / g.hx, ihp = 1.0 / g.hp;
        const double2 e = csx[col];
        const double f1 = force(K, e.x, e.y);
        double c3, s3, pc, ps;   // e^{i (theta + h^2/4 f_1)}
        phase(0.25 * h * h * f1, pc, ps);
        c3 = e.x;
        s3 = e.y;
        rotate(c3, s3, pc, ps);
        T x[kWarpRows], acc[NR][NR];
#pragma unroll
        for (int b = 0; b < NR; ++b)
#pragma unroll
            for (int a = 0; a < NR; ++a) acc[b][a] = T(0);
        long mb = 0, nb = 0;
        int mi = 0;
        bool live = false;
#pragma unroll
        for (int k = 0; k < kWarpRows; ++k) x[k] = r0 + k < r1 ? src[(size_t)(r0 + k) * nx + col] : T(0);
#pragma unroll 1
        for (int k = 0; k < kWarpRows; ++k) {
            T w = x[0];
#pragma unroll
            for (int q = 0; q + 1 < kWarpRows; ++q) x[q] = x[q + 1];
            if (w == T(0)) continue;
            const int j = r0 + k;
            const double rc = rt[j], rs = rt[np + j];
            double c = e.x, s = e.y;
            rotate(c, s, rc, rs);
            const double f2 = force(K + 2, c, s);
            double c2 = c3, s2 = s3;
            rotate(c2, s2, rc, rs);
            const double f3 = force(K + 4, c2, s2);
            phase(0.5 * h * h * f2, pc, ps);
            rotate(c, s, rc, rs);
            rotate(c, s, pc, ps);
            const double f4 = force(K + 6, c, s);
            // end point in cells, as node index + displacement
            const double du = (h * (g.delta + (g.p0 + j * g.hp)) + h * h / 6.0 * (f1 + f2 + f3)) * ihx;
            const double dv = h / 6.0 * (f1 + 2.0 * f2 + 2.0 * f3 + f4) * ihp;
            const double fu = floor(du), fv = floor(dv);
            T wx[N], wyt[N];
            TP::weights((T)(du - fu), wx);
            TP::weights((T)(dv - fv), wyt);
#pragma unroll
            for (int b = 0; b < N; ++b) wyt[b] *= w;
            const long m = (long)col + (long)fu + TP::LO, n = (long)j + (long)fv + TP::LO;
            if constexpr (RING) {
                if (live && m == mb && n == nb + 1) {
                    put(acc[0], mi, nb);
#pragma unroll
                    for (int b = 0; b < N - 1; ++b)
#pragma unroll
                        for (int a = 0; a < N; ++a) acc[b][a] = acc[b + 1][a] + wyt[b] * wx[a];
#pragma unroll
                    for (int a = 0; a < N; ++a) acc[N - 1][a] = wyt[N - 1] * wx[a];
                } else {
                    if (live)
#pragma unroll 1
                        for (int b = 0; b < N; ++b) {
                            put(acc[0], mi, nb + b);
#pragma unroll
                            for (int q = 0; q + 1 < N; ++q)
#pragma unroll
                                for (int a = 0; a < N; ++a) acc[q][a] = acc[q + 1][a];
                        }
                    mb = m;
                    mi = (int)(m % nx);
                    if (mi < 0) mi += nx;
                    live = true;
#pragma unroll
                    for (int b = 0; b < N; ++b)
#pragma unroll
                        for (int a = 0; a < N; ++a) acc[b][a] = wyt[b] * wx[a];
                }
                nb = n;
            } else {
                mi = (int)(m % nx);
                if (mi < 0) mi += nx;
#pragma unroll
                for (int b = 0; b < N; ++b) {
                    T v[N];
#pragma unroll
                    for (int a = 0; a < N; ++a) v[a] = wyt[b] * wx[a];
                    put(v, mi, n + b);
                }
            }
        }
        if constexpr (RING) {
            if (live)
#pragma unroll
                for (int b = 0; b < N; ++b) put(acc[b], mi, nb + b);
        }
    }
    for (int o = 16; o > 0; o >>= 1) lost += __shfl_down_sync(0xffffffffu, lost, o);
    if (lane == 0) s_red[wy] = lost;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tl = 0.0;
        for (int k = 0; k < kThreads / 32; ++k) tl += s_red[k];
        if (tl != 0.0) atomicAdd(lost_acc, tl);
    }
}

}  // namespace

int rk4_stage_blocks(int nx, int np) { return ((nx + 31) / 32) * ((np + kRows - 1) / kRows); }

template <typename T>
cudaError_t launch_rk4_stages(const T *w, const Geometry &g, const double2 *csx, const double *rt, double *state,
                              double *part, cudaStream_t s)
{
    const int blocks = rk4_stage_blocks(g.nx, g.np);
    rk4_mid_kernel<T><<<blocks, kThreads, 0, s>>>(w, g, csx, rt, state, part);
    rk4_amp_kernel<<<1, kAmp, 0, s>>>(part, blocks, state, 0, g.dt, g.sigma2);
    rk4_last_kernel<T><<<blocks, kThreads, 0, s>>>(w, g, csx, rt, state, part);
    rk4_amp_kernel<<<1, kAmp, 0, s>>>(part, blocks, state, 1, g.dt, g.sigma2);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_rk4_deposit(const T *src, T *dst, const Geometry &g, const double2 *csx, const double *rt,
                               const double *state, double *lost_acc, cudaStream_t s)
{
    const int grid = rk4_stage_blocks(g.nx, g.np);
    if (g.basis == VP_BASIS_TENT)
        rk4_deposit_kernel<T, VP_BASIS_TENT><<<grid, kThreads, 0, s>>>(src, dst, g, csx, rt, state, lost_acc);
    else if (g.basis == VP_BASIS_SEPTIC_BSPLINE)
        rk4_deposit_kernel<T, VP_BASIS_SEPTIC_BSPLINE><<<grid, kThreads, 0, s>>>(src, dst, g, csx, rt, state, lost_acc);
    else
        rk4_deposit_kernel<T, VP_BASIS_CUBIC_BSPLINE><<<grid, kThreads, 0, s>>>(src, dst, g, csx, rt, state, lost_acc);
    return cudaGetLastError();
}

#define VP_RK4_INST(T)                                                                                              \
    template cudaError_t launch_rk4_stages<T>(const T *, const Geometry &, const double2 *, const double *, double *, \
                                              double *, cudaStream_t);                                              \
    template cudaError_t launch_rk4_deposit<T>(const T *, T *, const Geometry &, const double2 *, const double *,      \
                                               const double *, double *, cudaStream_t);
VP_RK4_INST(float)
VP_RK4_INST(double)
#undef VP_RK4_INST

}  // namespace vp
