// rsv_simple.cu -- stand-alone S(h), dS/dh and momentum draws (FP64).
//
// S(h) and dS/dh of the RSV model (arXiv:1603.08114, Sec. 3 with eqs. (1)-(3)).
// Both read 24 B per site (dS/dh writes 8 more) and are bound by the FP64 pipe (2
// lanes per cycle and SM): S takes 9 of its instructions per site and dS/dh 10,
// with the exponential on the integer units (exp_neg), its factor 1/2 in the
// exponent and a thread's run of R sites sharing their x = h - mu (30 each
// with CUDA's exp and every neighbour recomputed: 2^22 sites 277 -> 95 us and
// 282 -> 96 us).  R is 4 for long series; short ones take a site per thread in
// small blocks, spread over the SMs.
// With leverage (th.rho != 0, the RSV model with corr(eps_t, eta_t) = rho of
// the RSV reference cited in Sec. 2) the AR term of site t is
// d_t^2 / (2 s_eta^2 (1 - rho^2)), d_t = x_{t+1} - phi x_t - rho s_eta y_t e^{-h_t/2}.
#include <cmath>

#include "rsv_device.cuh"
#include "rsv_simple.cuh"

namespace rsv {

namespace {

constexpr int kRun = 4;  // sites of a thread's run on long series

// theta and what follows from it, formed on the host (three divisions and a
// square root in every thread cost as much as four of its sites).
struct ThetaC {
    double phi, mu, xi, ie, iu, rs, B, pp, st;
};
ThetaC constants(const ThetaD& th)
{
    ThetaC c;
    c.phi = th.phi;
    c.mu = th.mu;
    c.xi = th.xi;
    c.ie = 1.0 / th.se2;
    c.iu = 1.0 / th.su2;
    c.rs = th.rho * std::sqrt(th.se2);
    c.B = 1.0 / (th.se2 * (1.0 - th.rho * th.rho));
    c.pp = 1.0 + th.phi * th.phi;
    c.st = 1.0 - th.phi * th.phi;
    return c;
}

template <bool LEV, int R>
__global__ void __launch_bounds__(256) k_force(const double* __restrict__ h,
                                               const double* __restrict__ y,
                                               const double* __restrict__ lnrv, int64_t T,
                                               ThetaC th, double* __restrict__ F)
{
    constexpr bool SMALL = R == 1;
    __shared__ u64 tab[SMALL ? 64 : kExpN];
    if (SMALL) exp_table_small(tab);
    else exp_table(tab);
    const double phi = th.phi, mu = th.mu, ie = th.ie, iu = th.iu, rs = th.rs, B = th.B;
    const double pp = th.pp, st = th.st;
    __syncthreads();
    for (int64_t t0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * R; t0 < T;
         t0 += (int64_t)gridDim.x * blockDim.x * R) {
        double hv[R + 2], yv[R], lr[R];  // h of sites t0 - 1 .. t0 + R
#pragma unroll
        for (int i = 0; i < R + 2; ++i) {
            const int64_t t = t0 - 1 + i;
            hv[i] = t >= 0 && t < T ? h[t] : mu;
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            yv[i] = t0 + i < T ? y[t0 + i] : 0.0;
            lr[i] = t0 + i < T ? lnrv[t0 + i] : 0.0;
        }
        double xl = hv[0] - mu, x = hv[1] - mu;  // (0 beyond the ends)
        double dl = 0.0;                         // leverage: d_{t-1}
        if (LEV && t0 > 0)
            dl = fma(-phi, xl, x) - rs * (y[t0 - 1] * exp_neg<1, 0, SMALL>(hv[0], tab));
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int64_t t = t0 + i;
            const double ht = hv[i + 1], xr = hv[i + 2] - mu;
            double f = fma(-iu, (lr[i] - th.xi) - ht, 0.5);
            if (LEV) {
                // derivative of the terms of s_t and s_{t-1} that hold h_t
                const double eps = yv[i] * exp_neg<1, 0, SMALL>(ht, tab);
                const double d = t + 1 < T ? fma(-phi, x, xr) - rs * eps : 0.0;
                double g = fma(d, fma(0.5 * rs, eps, -phi), dl);
                f = fma(B, g, f);
                if (t == 0) f = fma(st * ie, x, f);
                f = fma(-0.5 * eps, eps, f);
                dl = d;
            } else {
                const bool in = t > 0 && t + 1 < T;
                const double c = in ? pp : T == 1 ? st : 1.0;
                f = fma(ie, fma(c, x, -phi * (xl + xr)), f);
                f = fma(-(yv[i] * yv[i]), exp_neg<0, 1, SMALL>(ht, tab), f);
            }
            if (t < T) F[t] = f;
            xl = x;
            x = xr;
        }
    }
}

// Per-site action s_t summed per block; the last block adds the block sums in
// block order.
template <bool LEV, int R>
__global__ void __launch_bounds__(256) k_action(const double* __restrict__ h,
                                                const double* __restrict__ y,
                                                const double* __restrict__ lnrv, int64_t T,
                                                ThetaC th, double* __restrict__ partials,
                                                unsigned* __restrict__ counter,
                                                double* __restrict__ S_out)
{
    constexpr bool SMALL = R == 1;
    __shared__ u64 tab[SMALL ? 64 : kExpN];
    __shared__ double red[32];
    __shared__ int s_last;
    if (SMALL) exp_table_small(tab);
    else exp_table(tab);
    const double phi = th.phi, mu = th.mu, ie = th.ie, iu = th.iu, rs = th.rs;
    const double B = LEV ? th.B : ie;
    __syncthreads();
    // sums of h, r^2, d^2 and (y^2/2) e^{-h}
    double sh = 0.0, sr = 0.0, sd = 0.0, se = 0.0, s0 = 0.0;
    for (int64_t t0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * R; t0 < T;
         t0 += (int64_t)gridDim.x * blockDim.x * R) {
        double hv[R + 1], yv[R], lr[R];
#pragma unroll
        for (int i = 0; i < R + 1; ++i) hv[i] = t0 + i < T ? h[t0 + i] : mu;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            yv[i] = t0 + i < T ? y[t0 + i] : 0.0;
            lr[i] = t0 + i < T ? lnrv[t0 + i] : 0.0;
        }
        double x = hv[0] - mu;
        if (t0 == 0) s0 = 0.5 * ie * th.st * x * x;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const double xn = hv[i + 1] - mu;
            if (t0 + i < T) {
                const double r = (lr[i] - th.xi) - hv[i];
                sh += hv[i];
                sr = fma(r, r, sr);
                double d = fma(-phi, x, xn);
                if (LEV) {
                    const double eps = yv[i] * exp_neg<1, 0, SMALL>(hv[i], tab);
                    d = fma(-rs, eps, d);
                    se = fma(0.5 * eps, eps, se);
                } else {
                    se = fma(yv[i] * yv[i], exp_neg<0, 1, SMALL>(hv[i], tab), se);
                }
                if (t0 + i + 1 < T) sd = fma(d, d, sd);
            }
            x = xn;
        }
    }
    const double b = block_sum(fma(0.5, sh, fma(0.5 * iu, sr, fma(0.5 * B, sd, se))) + s0, red);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = b;
        __threadfence();
        s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) v += __ldcg(partials + i);
    const double S = block_sum(v, red);
    if (threadIdx.x == 0) {
        *S_out = S;
        *counter = 0u;
    }
}

// Momenta exactly as the trajectory kernels draw them: one Philox block per
// group of four sites, Box-Muller on 53-bit (FP64) or 23-bit (FP32) uniforms.
__global__ void k_draw_momenta(uint64_t seed, uint64_t series, uint64_t traj, int64_t T,
                               const float* __restrict__ minv, int bits, double* __restrict__ p)
{
    const int64_t nq = (T + 3) / 4;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nq;
         q += (int64_t)gridDim.x * blockDim.x) {
        const u64x4 r = philox_block(seed, series, traj, STREAM_MOM, (uint64_t)q);
        double z[4];
        if (bits == 53) {
            box_muller(u01_53(r.w[0]), u01_53(r.w[1]), z[0], z[1]);
            box_muller(u01_53(r.w[2]), u01_53(r.w[3]), z[2], z[3]);
        } else {
            float f[4];
            box_muller_f(u01_23(r.w[0]), u01_23(r.w[1]), f[0], f[1]);
            box_muller_f(u01_23(r.w[2]), u01_23(r.w[3]), f[2], f[3]);
            for (int i = 0; i < 4; ++i) z[i] = f[i];
        }
        for (int i = 0; i < 4; ++i) {
            const int64_t t = 4 * q + i;
            if (t >= T) break;
            if (minv) {
                if (bits == 53) z[i] = z[i] / sqrt((double)minv[t]);
                else z[i] = (double)((float)z[i] / sqrtf(minv[t]));
            }
            p[t] = z[i];
        }
    }
}

int grid_stream(int64_t n)
{
    int64_t g = (n + 255) / 256;
    if (g > 152 * 8) g = 152 * 8;
    if (g < 1) g = 1;
    return (int)g;
}

// Series of up to 152 x 256 sites: a site per thread, blocks of 64 threads (a
// block's own latency, not the FP64 pipe, is then what a call waits for).
bool short_series(int64_t T) { return T <= 152 * 256; }
int run_grid(int64_t T)
{
    return short_series(T) ? (int)((T + 63) / 64) : grid_stream((T + kRun - 1) / kRun);
}

}  // namespace

int action_grid(int64_t T) { return run_grid(T); }

cudaError_t launch_force(const double* h, const double* y, const double* lnrv, int64_t T,
                         ThetaD th, double* F, cudaStream_t st)
{
    const int g = run_grid(T), nt = short_series(T) ? 64 : 256;
    auto k = short_series(T) ? (th.rho != 0.0 ? k_force<true, 1> : k_force<false, 1>)
                             : (th.rho != 0.0 ? k_force<true, kRun> : k_force<false, kRun>);
    k<<<g, nt, 0, st>>>(h, y, lnrv, T, constants(th), F);
    return cudaGetLastError();
}

cudaError_t launch_action(const double* h, const double* y, const double* lnrv, int64_t T,
                          ThetaD th, double* partials, unsigned* counter, double* S_out,
                          cudaStream_t st)
{
    const int g = run_grid(T), nt = short_series(T) ? 64 : 256;
    auto k = short_series(T) ? (th.rho != 0.0 ? k_action<true, 1> : k_action<false, 1>)
                             : (th.rho != 0.0 ? k_action<true, kRun> : k_action<false, kRun>);
    k<<<g, nt, 0, st>>>(h, y, lnrv, T, constants(th), partials, counter, S_out);
    return cudaGetLastError();
}

cudaError_t launch_draw_momenta(uint64_t seed, uint64_t series, uint64_t traj, int64_t T,
                                const float* minv, int bits, double* p, cudaStream_t st)
{
    k_draw_momenta<<<grid_stream((T + 3) / 4), 256, 0, st>>>(seed, series, traj, T, minv, bits, p);
    return cudaGetLastError();
}

}  // namespace rsv
