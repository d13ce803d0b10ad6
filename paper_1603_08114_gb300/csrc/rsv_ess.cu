// rsv_ess.cu -- effective sample size per site of a chain of snapshots.
//
// Geyer's initial monotone sequence estimator (C. J. Geyer, Statistical
// Science 7, 1992): normalised autocorrelations rho_k from the plain sums
// gamma_k = (1/n) sum_t (x_t - m)(x_{t+k} - m); pair sums
// Gamma_m = rho_{2m} + rho_{2m+1} taken while positive and made
// non-increasing; tau = -1 + 2 sum Gamma_m, floored at 1/log10(n) (so ESS
// <= n log10 n); ESS = n / tau; a constant column (zero variance) gets 0.
// The snapshot matrix is [n][T] FP32, sample-major.  A warp takes 32 sites and
// kLags lags in one pass over the samples: each sample read serves all of
// them from a window of the last kLags older ones in registers, and the
// compensated sums are kLags independent chains.  A block of eight warps holds
// C sites: it starts with kLags lags for each 32 of them, drops the sites whose
// sum has ended after every pass (the longest of 32 sites needs several times
// the lags of the mean one) and gives the warps this frees the next lags of
// the remaining ones.  Bound by the FP32 instructions, about 40 per sample and
// pass.  1000 x 2^17 samples: 29.3 ms with a thread per site and a pass per lag
// (two reads and one chain of four dependent instructions per sample), 3.86 ms
// with kLags lags a pass, 1.22 ms with the sites compacted.
#include <cmath>

#include "rsv_ess.cuh"

namespace rsv {

namespace {

constexpr int kLags = 8, kWarps = 8;

template <int C>
__global__ void __launch_bounds__(32 * kWarps) k_ess(const float* __restrict__ x, int64_t n,
                                                     int64_t T, float* __restrict__ ess)
{
    __shared__ float gam[kLags][32 * kWarps];  // [lag][site slot], the lag groups side by side
    __shared__ float s_m[C];
    __shared__ int s_list[C], s_cnt[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t site = blockIdx.x * (int64_t)C + tid;  // (threads below C)
    const bool own = tid < C && site < T;
    if (own) {  // mean with compensation
        const float* xt = x + site;
        float s = 0.f, c = 0.f;
        auto add = [&](float r) {
            const float v = r - c;
            const float q = s + v;
            c = (q - s) - v;
            s = q;
        };
        int64_t k = 0;
        for (; k + 8 <= n; k += 8, xt += 8 * T) {
            float r[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = xt[u * T];
#pragma unroll
            for (int u = 0; u < 8; ++u) add(r[u]);
        }
        for (; k < n; ++k, xt += T) add(*xt);
        s_m[tid] = s / (float)n;
    }
    const int64_t left = T - blockIdx.x * (int64_t)C;
    int count = left < C ? (int)left : C;  // sites still summed, s_list[0 .. count)
    if (tid < C) s_list[tid] = tid;
    __syncthreads();
    // thread i < count keeps the state of site s_list[i]
    int mine = tid;
    float g0 = 0.f, tau_sum = 0.f, prev = INFINITY;
    for (int64_t first = 0; count > 0;) {
        const int cw = (count + 31) >> 5, G = kWarps / cw;  // site groups, lag groups
        const int sg = warp % cw, lg = warp / cw;
        if (lg < G) {
            const int slot = sg * 32 + lane;
            const int col = s_list[slot < count ? slot : 0];
            const float m = s_m[col];
            // gamma_{L+b} = sum_j d_j d_{j-L-b} over j ascending, d = x - m; at
            // sample j of a run of kLags the older value of lag L + b is w[(u - b) mod kLags]
            const int64_t L = first + lg * kLags;
            const float* pc = x + blockIdx.x * (int64_t)C + col + L * T;
            const float* po = pc - L * T;
            float a[kLags], ca[kLags], w[kLags];
#pragma unroll
            for (int b = 0; b < kLags; ++b) a[b] = ca[b] = w[b] = 0.f;
            auto sample = [&](int u, float cur, float old) {
                w[u] = old - m;
                const float d = cur - m;
#pragma unroll
                for (int b = 0; b < kLags; ++b) {
                    const float v = fmaf(w[(u - b) & (kLags - 1)], d, -ca[b]);
                    const float q = a[b] + v;
                    ca[b] = (q - a[b]) - v;
                    a[b] = q;
                }
            };
            int64_t j = L;
            for (; j + kLags <= n; j += kLags, pc += kLags * T, po += kLags * T) {
                float cur[kLags], old[kLags];
#pragma unroll
                for (int u = 0; u < kLags; ++u) cur[u] = pc[u * T];
                if (L == 0) {
#pragma unroll
                    for (int u = 0; u < kLags; ++u) old[u] = cur[u];
                } else {
#pragma unroll
                    for (int u = 0; u < kLags; ++u) old[u] = po[u * T];
                }
#pragma unroll
                for (int u = 0; u < kLags; ++u) sample(u, cur[u], old[u]);
            }
#pragma unroll
            for (int u = 0; u < kLags - 1; ++u)
                if (j + u < n) sample(u, pc[u * T], po[u * T]);
#pragma unroll
            for (int b = 0; b < kLags; ++b) gam[b][lg * cw * 32 + slot] = a[b] / (float)n;
        }
        __syncthreads();
        bool more = false;
        if (tid < count) {
            more = true;
            if (first == 0) g0 = gam[0][tid];
            if (!(g0 > 0.f)) more = false;  // the chain never moved at this site
            for (int p = 0; p < G * kLags / 2 && more; ++p) {
                const int64_t mm = first / 2 + p;
                const int o = (p / (kLags / 2)) * cw * 32 + tid, b = 2 * (p % (kLags / 2));
                const float G2 = (mm == 0 ? 1.0f : gam[b][o] / g0) + gam[b + 1][o] / g0;
                if (2 * mm + 1 >= n || !(G2 > 0.f)) {
                    more = false;
                } else {
                    const float Gm = fminf(G2, prev);
                    tau_sum += Gm;
                    prev = Gm;
                }
            }
            if (!more) {
                float tau = -1.f + 2.f * tau_sum;
                const float nn = (float)(n > 10 ? n : 10);
                tau = fmaxf(tau, 1.f / log10f(nn));
                ess[blockIdx.x * (int64_t)C + mine] = g0 > 0.f ? (float)n / tau : 0.f;
            }
        }
        // the remaining sites, in order, with their state
        const unsigned vote = __ballot_sync(0xffffffffu, more);
        if (lane == 0) s_cnt[warp] = __popc(vote);
        __syncthreads();
        int at = __popc(vote & ((1u << lane) - 1u)), all = 0;
#pragma unroll
        for (int v = 0; v < kWarps; ++v) {
            if (v < warp) at += s_cnt[v];
            all += s_cnt[v];
        }
        if (more) {
            s_list[at] = mine;
            gam[0][at] = g0;
            gam[1][at] = tau_sum;
            gam[2][at] = prev;
        }
        __syncthreads();
        count = all;
        first += G * kLags;
        if (tid < count) {
            mine = s_list[tid];
            g0 = gam[0][tid];
            tau_sum = gam[1][tid];
            prev = gam[2][tid];
        }
        __syncthreads();
    }
}

// A thread per site and a pass per lag, for chains of fewer samples than a pass
// of k_ess pays for: its blocks' barriers and lags beyond the chain cost more than
// reading a few samples again (2^20 sites: 2 samples 17 us against 46, 8 samples 48
// against 70; from 12 on k_ess is no slower, 16 samples 83 against 103).
constexpr int kFewSamples = 12;
__global__ void __launch_bounds__(256) k_ess_few(const float* __restrict__ x, int n, int64_t T,
                                                 float* __restrict__ ess)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= T) return;
    float s = 0.f, c = 0.f;
    for (int k = 0; k < n; ++k) {
        const float v = x[k * T + t] - c;
        const float q = s + v;
        c = (q - s) - v;
        s = q;
    }
    const float m = s / (float)n;
    auto gamma = [&](int lag) {
        float a = 0.f, ca = 0.f;
        for (int k = 0; k + lag < n; ++k) {
            const float v = fmaf(x[k * T + t] - m, x[(k + lag) * T + t] - m, -ca);
            const float q = a + v;
            ca = (q - a) - v;
            a = q;
        }
        return a / (float)n;
    };
    const float g0 = gamma(0);
    float tau_sum = 0.f, prev = INFINITY;
    for (int mm = 0; g0 > 0.f && 2 * mm + 1 < n; ++mm) {
        const float G = (mm == 0 ? 1.0f : gamma(2 * mm) / g0) + gamma(2 * mm + 1) / g0;
        if (!(G > 0.f)) break;
        prev = fminf(G, prev);
        tau_sum += prev;
    }
    const float tau = fmaxf(-1.f + 2.f * tau_sum, 1.f / log10f((float)(n > 10 ? n : 10)));
    ess[t] = g0 > 0.f ? (float)n / tau : 0.f;
}

}  // namespace

cudaError_t launch_ess(const float* x, int64_t n, int64_t T, float* ess, cudaStream_t st)
{
    // as many sites a block as keep the SMs in work (1000 samples: 2^17 sites 256
    // a block 1.22 ms, 32 a block 2.16; 2^15 sites 128 a block 0.49, 256 0.63), and
    // fewer where the sites are few, for more lags at once (500 sites 32 a block
    // 0.15 ms, 256 a block 0.30)
    auto blocks = [&](int c) { return (unsigned)((T + c - 1) / c); };
    if (n < kFewSamples) k_ess_few<<<blocks(256), 256, 0, st>>>(x, (int)n, T, ess);
    else if (blocks(256) >= 200) k_ess<256><<<blocks(256), 32 * kWarps, 0, st>>>(x, n, T, ess);
    else if (blocks(128) >= 200) k_ess<128><<<blocks(128), 32 * kWarps, 0, st>>>(x, n, T, ess);
    else if (blocks(64) >= 200) k_ess<64><<<blocks(64), 32 * kWarps, 0, st>>>(x, n, T, ess);
    else k_ess<32><<<blocks(32), 32 * kWarps, 0, st>>>(x, n, T, ess);
    return cudaGetLastError();
}

}  // namespace rsv
