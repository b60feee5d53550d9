// vp_reduce.cu -- FP64 reductions over the weights.
//
// FEL field (Sec. IV.B, dA/dz = <exp(-i Phi)>, detuning and space charge zero),
// drift-kick-drift in time:
//   A^{n+1/2} = A^n + h/2 b^n,  push with A^{n+1/2},  b^{n+1} = <exp(-i theta)>
//   of the new weights,  A^{n+1} = A^{n+1/2} + h/2 b^{n+1}.
// The bunching comes from per-block partial sums (sum w, sum w cos theta,
// sum w sin theta), reduced here in a fixed order so that results do not
// depend on scheduling.
//
// Moments (Sec. IV diagnostics: sum of weights, entropy): FP64 accumulation per
// thread, per-block partials, fixed-order final sum.
#include <math.h>

#include "vp_internal.h"
#include "vp_fel.cuh"
#include "vp_sum.cuh"

namespace vp {
namespace {

constexpr int kRedThreads = 256;
static_assert(kRedThreads == kFinThreads, "the finalize kernels run one block of kFinThreads threads");

// one block per 32-column strip x row chunk: column sums (compensated) then x cos/sin
constexpr int kFelRows = 256;

template <typename T>
__global__ void fel_partials_kernel(const T *__restrict__ w, int nx, int np,
                                    const double2 *__restrict__ csx, double *part)
{
    __shared__ double s_red[3][kRedThreads / 32];
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int col = blockIdx.x * 32 + lane;
    const int r0 = blockIdx.y * kFelRows;
    const int r1 = min(r0 + kFelRows, np);
    DSum<T> acc;
    if (col < nx)
        for (int r = r0 + wy; r < r1; r += kRedThreads / 32) acc.add(w[(size_t)r * nx + col]);
    double pw = acc.value(), pc = 0.0, ps = 0.0;
    if (col < nx) {
        const double2 t = csx[col];
        pc = pw * t.x;
        ps = pw * t.y;
    }
    double v[3] = {pw, pc, ps};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
        if (lane == 0) s_red[q][wy] = v[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const size_t b = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
        for (int q = 0; q < 3; ++q) {
            double t = 0.0;
            for (int k = 0; k < kRedThreads / 32; ++k) t += s_red[q][k];
            part[3 * b + q] = t;
        }
    }
}

// FEL space charge: per block (32 columns x kFelRows rows) the sums of the state against the
// mass weights and against the half-drift phase factors e^{-i (theta_i + phi_j)}:
// per column C = sum_j s_ij rc_j, S = sum_j s_ij rs_j, then Re += cos(th) C - sin(th) S and
// Im -= sin(th) C + cos(th) S (rc, rs already carry Lambda_p^{-1} for the state s = Lambda_p w)
template <typename T>
__global__ void fel_tilde_kernel(const T *__restrict__ st, int nx, int np, const double2 *__restrict__ csx,
                                 const double *__restrict__ rc, const double *__restrict__ rs,
                                 const double *__restrict__ sig, double *part)
{
    __shared__ double s_red[3][kRedThreads / 32];
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int col = blockIdx.x * 32 + lane;
    const int r0 = blockIdx.y * kFelRows;
    const int r1 = min(r0 + kFelRows, np);
    double m = 0.0, c = 0.0, sn = 0.0;
    if (col < nx)
        for (int r = r0 + wy; r < r1; r += kRedThreads / 32) {
            const double v = (double)st[(size_t)r * nx + col];
            m += v * (sig ? sig[r] : 1.0);
            c += v * rc[r];
            sn += v * rs[r];
        }
    double v3[3] = {m, 0.0, 0.0};
    if (col < nx) {
        const double2 t = csx[col];
        v3[1] = t.x * c - t.y * sn;
        v3[2] = -(t.y * c + t.x * sn);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        for (int o = 16; o > 0; o >>= 1) v3[q] += __shfl_down_sync(0xffffffffu, v3[q], o);
        if (lane == 0) s_red[q][wy] = v3[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const size_t b = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
        for (int q = 0; q < 3; ++q) {
            double t = 0.0;
            for (int k = 0; k < kRedThreads / 32; ++k) t += s_red[q][k];
            part[3 * b + q] = t;
        }
    }
}

// K = A^{n+1/2} + i sigma2 bt, bt = <e^{-i theta~}> from the tilde partial sums (one block)
__global__ void fel_kick_kernel(const double *__restrict__ part, int nparts, double *state, double sigma2,
                                bool exact_bounds)
{
    __shared__ double s[3][kRedThreads];
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int k = threadIdx.x; k < nparts; k += blockDim.x) {
        a0 += part[3 * k];
        a1 += part[3 * k + 1];
        a2 += part[3 * k + 2];
    }
    s[0][threadIdx.x] = a0;
    s[1][threadIdx.x] = a1;
    s[2][threadIdx.x] = a2;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int q = 0; q < 3; ++q) s[q][threadIdx.x] += s[q][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    const double bt_re = s[1][0] / s[0][0], bt_im = s[2][0] / s[0][0];
    const double kr = state[ST_AH_RE] - sigma2 * bt_im, ki = state[ST_AH_IM] + sigma2 * bt_re;
    state[ST_K_RE] = kr;
    state[ST_K_IM] = ki;
    store_kick_bounds(state, exact_bounds);
}

// FEL field update from per-block partial sums (run by one block of kFinThreads threads)
__global__ void fel_finalize_kernel(const double *__restrict__ part, int nparts, double *state, double *hist,
                                    int hist_cap, double dt, int init, int rk4, bool exact_bounds)
{
    __shared__ double s[3 * kFinThreads];
    fel_finalize_core(part, nparts, state, hist, hist_cap, dt, init, rk4, exact_bounds, s);
}

// plain step counter for non-FEL sims
__global__ void count_step_kernel(double *state, double dt)
{
    const double st = state[ST_STEP] + 1.0;
    state[ST_STEP] = st;
    state[ST_TAU] = st * dt;
}

// Moments. Bound by the FP64 pipe (2 operations per clock and SM on this GPU), not by memory: 62 FP64
// operations a node took 0.45 ms for 2048 x 2048 (0.19 ms now, the final sums 6 us against 153 in one thread
// each). A warp therefore walks 32 columns through a chunk of rows and
// keeps per column only the sums over p (w, w p, w p^2: everything else of a node's moments is a factor of its
// column), the entropy, and the negative and the trapped weight: about a dozen.
//
// w ln w of FP32 weights: with w = 2^e m and c the centre of m's 512th of [1, 2), u = m / c - 1 (|u| < 2^-10),
// ln w = (e ln 2 + ln c) + ln(1 + u), the series of ln(1 + u) cut after u^5 / 5 (the next term is below 2^-62). 1 / c
// is rounded, so ln c in the table is minus the log of that rounded value: u carries one rounding, of order 2^-53.
constexpr int kLnBits = 9, kLnTab = 1 << kLnBits;
struct alignas(16) LnTable {
    double2 c[kLnTab];   // rounded 1 / c, and -ln of it
    double e[256];       // (e - 127) ln 2
};

static_assert(sizeof(LnTable) == kLnTableBytes, "room for the table in the workspace");

__global__ void ln_table_kernel(LnTable *t)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kLnTab) {
        const double ic = 1.0 / (1.0 + (k + 0.5) / kLnTab);
        t->c[k] = make_double2(ic, -log(ic));
    }
    if (k < 256) t->e[k] = (k - 127) * 0.693147180559945309417;
}

// conversion by integer operations where it can be (a conversion instruction runs at the FP64 rate)
__device__ __forceinline__ double wide_of(float w)
{
    const unsigned b = __float_as_uint(w), e = (b >> 23) & 255u;
    if (e == 0u || e == 255u) return (double)w;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double wide_of(double w) { return w; }

__device__ __forceinline__ double ln_of(float w, const LnTable &t)
{
    const unsigned b = __float_as_uint(w);
    const int e = (int)(b >> 23);
    if (e == 0 || e == 255) return log((double)w);   // denormal or not finite
    const unsigned man = b & 0x7fffffu;
    const double m = __hiloint2double((int)(0x3ff00000u | (man >> 3)), (int)(man << 29));
    const double2 q = t.c[man >> (23 - kLnBits)];
    const double u = fma(m, q.x, -1.0);
    double s = fma(u, 0.2, -0.25);
    s = fma(u, s, 1.0 / 3.0);
    s = fma(u, s, -0.5);
    s = fma(u, s, 1.0);
    return fma(u, s, t.e[e] + q.y);
}
__device__ __forceinline__ double ln_of(double w, const LnTable &) { return log(w); }

// H < hsep as FP64 gives it; a call, so that it runs only where it is asked for
__device__ __noinline__ bool below_separatrix(double p, double V, double hsep) { return 0.5 * p * p + V < hsep; }

// rows of a warp's chunk and the chunks of a column (the same on the host and in the kernel)
__host__ __device__ __forceinline__ int moment_rows(int nx, int np)
{
    // as many warps as the chip holds (16 an SM); at least 8 rows, over which a column's factors and the block's
    // final sums are spread
    const long long strips = (nx + 31) / 32, want = 152LL * 16;
    const long long chunks = want / strips < 1 ? 1 : want / strips;
    const long long rows = (np + chunks - 1) / chunks;
    return rows < 8 ? 8 : (int)rows;
}

template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    moments_kernel(const T *__restrict__ w, Geometry g, const double2 *__restrict__ csx, const void *ln, double *part)
{
    __shared__ double s_red[kNumMoments][kRedThreads / 32];
    __shared__ LnTable s_ln;
    if (sizeof(T) == 4)
        for (int k = threadIdx.x; k < (int)(sizeof(LnTable) / 16); k += kRedThreads)
            reinterpret_cast<int4 *>(&s_ln)[k] = __ldg(static_cast<const int4 *>(ln) + k);
    __syncthreads();
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    double acc[kNumMoments];
#pragma unroll
    for (int q = 0; q < kNumMoments; ++q) acc[q] = 0.0;
    const double hsep = fabs(g.v_sign);
    const bool pend = (g.kind == VP_PUSH_LEAPFROG_KDK && g.potential == VP_POT_PENDULUM);
    const int rows = moment_rows(g.nx, g.np);
    const long long strips = (g.nx + 31) / 32, chunks = (g.np + rows - 1) / rows, ntask = strips * chunks;
    for (long long task = (long long)blockIdx.x * (kRedThreads / 32) + wy; task < ntask;
         task += (long long)gridDim.x * (kRedThreads / 32)) {
        const int i0 = (int)(task % strips) * 32 + lane, i = min(i0, g.nx - 1);
        const bool in = i0 < g.nx;
        const int r0 = (int)(task / strips) * rows, r1 = min(r0 + rows, g.np);
        const double x = g.x0 + i * g.hx;
        const double2 cs = csx[i];
        double V = 0.0;
        if (g.potential == VP_POT_PENDULUM) V = -g.v_sign * cs.x;
        else if (g.potential == VP_POT_HARMONIC) V = 0.5 * g.omega * g.omega * x * x;
        // sums over the column's chunk. s0 collects the weight of the present side of the separatrix, t0 that of
        // the other: they change places where the column crosses it
        double s0 = 0.0, t0 = 0.0, s1 = 0.0, s2 = 0.0, ent = 0.0, neg = 0.0, mx = 0.0;
        bool inside = false;
        float mxf = 0.f;
        const T *src = w + (size_t)r0 * g.nx + i;
        constexpr int F = 8;   // loads in flight
        T v[F];
        auto load = [&](int r) -> T { return in && r < r1 ? __ldg(src + (size_t)(r - r0) * g.nx) : T(0); };
#pragma unroll
        for (int k = 0; k < F; ++k) v[k] = load(r0 + k);
        const float vf = (float)(V - hsep), tol = 4.f * (float)hsep;
        double p_of = 0.0, p2_of = 0.0;   // lane l: the momentum of row rb + l (and its square), for 32 rows at a time
        float pf_of = 0.f;
        for (int rb = r0; rb < r1; rb += F) {
            const int ph = (rb - r0) & 31;
            if (ph == 0) {
                p_of = g.p0 + (rb + lane) * g.hp;
                p2_of = p_of * p_of;
                pf_of = (float)p_of;
            }
#pragma unroll
            for (int k = 0; k < F; ++k) {
                const int r = rb + k;
                const T wt = v[k];
                v[k] = load(r + F);
                const double p = __shfl_sync(0xffffffffu, p_of, ph + k), p2 = __shfl_sync(0xffffffffu, p2_of, ph + k);
                const float pf = __shfl_sync(0xffffffffu, pf_of, ph + k);
                if (wt == T(0)) continue;   // also rows past the chunk and columns past the mesh
                const double ww = wide_of(wt);
                if (pend) {
                    // H < hsep as FP64 gives it; FP32 decides where it is not close
                    const float hf = 0.5f * pf * pf + vf;
                    bool now = hf < 0.f;
                    if (fabsf(hf) <= 1e-5f * (pf * pf + tol)) now = below_separatrix(p, V, hsep);
                    if (now != inside) {
                        const double o = s0;
                        s0 = t0;
                        t0 = o;
                        inside = now;
                    }
                }
                s0 += ww;
                s1 = fma(ww, p, s1);
                s2 = fma(ww, p2, s2);
                if (wt > T(0)) ent = fma(-ww, ln_of(wt, s_ln), ent);
                else neg += ww;
                if (sizeof(T) == 4) mxf = fmaxf(mxf, fabsf((float)wt));
                else mx = fmax(mx, fabs(ww));
            }
        }
        const double sw = s0 + t0;
        acc[0] += sw;
        acc[1] = fma(sw, x, acc[1]);
        acc[2] += s1;
        acc[3] = fma(sw * x, x, acc[3]);
        acc[4] += s2;
        acc[5] = fma(s1, x, acc[5]);
        acc[6] += fma(sw, V, 0.5 * s2);
        acc[7] += inside ? s0 : (pend ? t0 : 0.0);
        acc[8] += ent;
        acc[9] += neg;
        acc[10] = fma(sw, cs.x, acc[10]);
        acc[11] = fma(sw, cs.y, acc[11]);
        acc[12] = fmax(acc[12], sizeof(T) == 4 ? (double)mxf : mx);
    }
#pragma unroll
    for (int q = 0; q < kNumMoments; ++q) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_down_sync(0xffffffffu, v, o);
            v = (q == 12) ? fmax(v, u) : v + u;
        }
        if (lane == 0) s_red[q][wy] = v;
    }
    __syncthreads();
    if (threadIdx.x < kNumMoments) {
        const int q = threadIdx.x;
        double t = 0.0;
        for (int k = 0; k < kRedThreads / 32; ++k) t = (q == 12) ? fmax(t, s_red[q][k]) : t + s_red[q][k];
        part[(size_t)q * gridDim.x + blockIdx.x] = t;
    }
}

// one warp per sum (a strided pass, then a tree: a fixed order), the last one the lost weight and the copies
__global__ void __launch_bounds__(32 * (kNumMoments + 1))
    moments_finalize_kernel(const double *__restrict__ part, int nblocks, const double *__restrict__ lost, int nlost,
                            double *out, const double *__restrict__ state, const unsigned *__restrict__ err)
{
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double *v = q < kNumMoments ? part + (size_t)q * nblocks : lost;
    const int n = q < kNumMoments ? nblocks : nlost;
    double t = 0.0;
#pragma unroll 8
    for (int b = lane; b < n; b += 32) t = (q == 12) ? fmax(t, v[b]) : t + v[b];
    for (int o = 16; o > 0; o >>= 1) {
        const double u = __shfl_down_sync(0xffffffffu, t, o);
        t = (q == 12) ? fmax(t, u) : t + u;
    }
    if (lane == 0) out[q] = t;
    if (q == kNumMoments) {
        for (int k = lane; k < ST_NSTATE; k += 32) out[kMoutState + k] = state[k];
        if (lane == 0) out[kMoutState + ST_NSTATE] = (double)*err;
    }
}

template <typename Tin, typename Tout>
__global__ void convert_kernel(const Tin *__restrict__ in, Tout *__restrict__ out, size_t n)
{
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x)
        out[k] = (Tout)in[k];
}

}  // namespace

int fel_partial_blocks(int nx, int np)
{
    return ((nx + 31) / 32) * ((np + kFelRows - 1) / kFelRows);
}

template <typename T>
cudaError_t launch_fel_tilde(const T *state, int nx, int np, const double2 *csx, const double *rc,
                             const double *rs, const double *sig, double *part, cudaStream_t s)
{
    dim3 grid((nx + 31) / 32, (np + kFelRows - 1) / kFelRows);
    fel_tilde_kernel<T><<<grid, kRedThreads, 0, s>>>(state, nx, np, csx, rc, rs, sig, part);
    return cudaGetLastError();
}
template cudaError_t launch_fel_tilde<float>(const float *, int, int, const double2 *, const double *,
                                             const double *, const double *, double *, cudaStream_t);
template cudaError_t launch_fel_tilde<double>(const double *, int, int, const double2 *, const double *,
                                              const double *, const double *, double *, cudaStream_t);

cudaError_t launch_fel_kick(const double *part, int nparts, double *state, double sigma2, bool exact_bounds,
                            cudaStream_t s)
{
    fel_kick_kernel<<<1, kRedThreads, 0, s>>>(part, nparts, state, sigma2, exact_bounds);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fel_partials(const T *w, int nx, int np, const double2 *csx, double *part,
                                cudaStream_t s)
{
    dim3 grid((nx + 31) / 32, (np + kFelRows - 1) / kFelRows);
    fel_partials_kernel<T><<<grid, kRedThreads, 0, s>>>(w, nx, np, csx, part);
    return cudaGetLastError();
}

cudaError_t launch_fel_finalize(const double *part, int nparts, double *state, double *hist,
                                int hist_cap, double dt, int init, bool exact_bounds, cudaStream_t s, int rk4)
{
    fel_finalize_kernel<<<1, kRedThreads, 0, s>>>(part, nparts, state, hist, hist_cap, dt, init, rk4, exact_bounds);
    return cudaGetLastError();
}

cudaError_t launch_count_step(double *state, double dt, cudaStream_t s)
{
    count_step_kernel<<<1, 1, 0, s>>>(state, dt);
    return cudaGetLastError();
}

int moment_blocks(int nx, int np)
{
    const int rows = moment_rows(nx, np);
    const long long tasks = (long long)((nx + 31) / 32) * ((np + rows - 1) / rows);
    const long long b = (tasks + kRedThreads / 32 - 1) / (kRedThreads / 32);
    return (int)(b < 152 * 8 ? b : 152 * 8);
}

template <typename T>
cudaError_t launch_moments(const T *w, const Geometry &g, const double2 *csx, const void *ln, double *part,
                           int nblocks, cudaStream_t s)
{
    moments_kernel<T><<<nblocks, kRedThreads, 0, s>>>(w, g, csx, ln, part);
    return cudaGetLastError();
}

cudaError_t build_ln_table(void *ln, cudaStream_t s)
{
    ln_table_kernel<<<(kLnTab + 127) / 128, 128, 0, s>>>(static_cast<LnTable *>(ln));
    return cudaGetLastError();
}

cudaError_t launch_moments_finalize(const double *part, int nblocks, const double *lost, int nlost,
                                    double *out, const double *state, const unsigned *err, cudaStream_t s)
{
    moments_finalize_kernel<<<1, 32 * (kNumMoments + 1), 0, s>>>(part, nblocks, lost, nlost, out, state, err);
    return cudaGetLastError();
}

template <typename Tin, typename Tout>
cudaError_t launch_convert(const Tin *in, Tout *out, size_t n, cudaStream_t s)
{
    size_t b = (n + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    convert_kernel<Tin, Tout><<<(int)b, 256, 0, s>>>(in, out, n);
    return cudaGetLastError();
}

template cudaError_t launch_fel_partials<float>(const float *, int, int, const double2 *, double *,
                                                cudaStream_t);
template cudaError_t launch_fel_partials<double>(const double *, int, int, const double2 *,
                                                 double *, cudaStream_t);
template cudaError_t launch_moments<float>(const float *, const Geometry &, const double2 *, const void *,
                                           double *, int, cudaStream_t);
template cudaError_t launch_moments<double>(const double *, const Geometry &, const double2 *, const void *,
                                            double *, int, cudaStream_t);
template cudaError_t launch_convert<float, double>(const float *, double *, size_t, cudaStream_t);
template cudaError_t launch_convert<double, float>(const double *, float *, size_t, cudaStream_t);

}  // namespace vp
