// rsv_mlp.cu -- the learned diagonal mass: sampler moments, features, a BF16
// MLP trained by Adam, and mass inference.
//
// Not part of the paper (which has no learned component): this library adds a
// per-site mass m_t = s (softplus(z_t) + eps) for HMC, where z_t is a 20 -> 32 ->
// 32 -> 1 MLP (tanh hidden units) on 20 features of site t computed from a
// FROZEN state (the posterior mean hbar of a plain sampler), so the mass never
// depends on the current h and HMC stays exact.  The network is trained on
// log(1 / Var(h_t)) with the squared error in log space.  s is a fixed output
// scale, the geometric mean of the target precisions: it keeps softplus near
// its unit-slope range so that the tanh layers need not saturate to reach
// precisions of O(30).
//
// Tensor cores: the matmuls (layer 1 and 2 forward, the back-propagation
// through layer 2 and the weight gradients of layers 1 and 2) run as
// mma.sync m16n8k16 BF16 tiles with FP32 accumulation; a warp owns 16 sites.
// These GEMMs are 16 x 32 x 32 per warp; tcgen05's 128-row tiles and TMEM
// staging would idle on them, so the warp-level MMA is the right size here.
//
// Parameter vector (FP32, 1761): W1[32][20] b1[32] W2[32][32] b2[32] W3[32] b3.
#include <cmath>

#include <cuda_bf16.h>

#include "rsv_device.cuh"
#include "rsv_mlp.cuh"

namespace rsv {

namespace {

constexpr int NF = 20, NH = 32, KP = 32;  // features, hidden, padded K of layer 1
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NF, OFF_W2 = OFF_B1 + NH,
              OFF_B2 = OFF_W2 + NH * NH, OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH,
              NPARAM = OFF_B3 + 1;
static_assert(NPARAM == 1761, "parameter layout");
constexpr float EPS_M = 1e-3f;
constexpr int EDGE = 16;       // the edge proximity 2^-d is not standardised
constexpr float CLIP = 8.0f;   // standardised features are clipped to [-8, 8]
constexpr int SITES_PER_BLOCK = 64;  // 4 warps x 16 sites

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const uint32_t a = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
    const uint32_t b = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
    return a | (b << 16);
}
// D = A(16x16, row) * B(16x8, col) + C, BF16 inputs, FP32 accumulate.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float softplus_f(float z)
{
    return z > 20.f ? z : log1pf(expf(z));
}
__device__ __forceinline__ float sigmoid_f(float z) { return 1.f / (1.f + expf(-z)); }

// Shared parameter copies of one block.  The BF16 matrices have rows of LD
// entries (80 bytes): the eight rows of a fragment start in different banks and
// each row on a 16-byte boundary, as ldmatrix wants.
constexpr int LD = 40;
struct __align__(16) SParams {
    __nv_bfloat16 w1[NH * LD];   // W1[n][k], K padded with zeros
    __nv_bfloat16 w2[NH * LD];   // W2[n][k]
    __nv_bfloat16 w2t[NH * LD];  // W2[n][k] at [k][n], for the back-propagation
    float b1[NH], b2[NH], w3[NH];
    float b3;
};

// The block's copy of the parameters (through L2: the training kernel's blocks
// update them during the launch); all loads of a thread are issued together.
template <int THREADS>
__device__ __forceinline__ void load_params(const float* __restrict__ P, SParams& s)
{
    constexpr int N = (NPARAM + THREADS - 1) / THREADS;
    float v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int e = threadIdx.x + i * THREADS;
        v[i] = e < NPARAM ? __ldcg(P + e) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int e = threadIdx.x + i * THREADS;
        if (e < OFF_B1) {
            s.w1[(e / NF) * LD + e % NF] = __float2bfloat16_rn(v[i]);
        } else if (e < OFF_W2) {
            s.b1[e - OFF_B1] = v[i];
        } else if (e < OFF_B2) {
            const int n = (e - OFF_W2) / NH, k = (e - OFF_W2) % NH;
            s.w2[n * LD + k] = s.w2t[k * LD + n] = __float2bfloat16_rn(v[i]);
        } else if (e < OFF_W3) {
            s.b2[e - OFF_B2] = v[i];
        } else if (e < OFF_B3) {
            s.w3[e - OFF_W3] = v[i];
        } else if (e < NPARAM) {
            s.b3 = v[i];
        }
    }
}
// zero the padding columns of w1 (once per block)
template <int THREADS>
__device__ __forceinline__ void pad_params(SParams& s)
{
    for (int i = threadIdx.x; i < NH * (KP - NF); i += THREADS)
        s.w1[(i / (KP - NF)) * LD + NF + i % (KP - NF)] = __float2bfloat16_rn(0.f);
}

// B fragment (16 x 8, "col") of a matrix stored as M[n][k] (row n, K
// consecutive): element (k, n) = M[n0 + n][k0 + k].
__device__ __forceinline__ void b_frag_nk(const __nv_bfloat16* M, int n0, int k0, uint32_t& b0,
                                          uint32_t& b1)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const uint32_t* r = reinterpret_cast<const uint32_t*>(M + (n0 + g) * LD + k0);
    b0 = r[t];
    b1 = r[t + 4];
}
// A fragment (16 x 16, row) of a matrix stored as M[m][k]: (m, k) = M[m][k0 + k].
__device__ __forceinline__ void a_frag_mk(const __nv_bfloat16* M, int k0, uint32_t (&a)[4])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const uint32_t* r0 = reinterpret_cast<const uint32_t*>(M + g * LD + k0);
    const uint32_t* r1 = reinterpret_cast<const uint32_t*>(M + (g + 8) * LD + k0);
    a[0] = r0[t];
    a[1] = r1[t];
    a[2] = r0[t + 4];
    a[3] = r1[t + 4];
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&d)[4], const __nv_bfloat16* row)
{
    const uint32_t p = (uint32_t)__cvta_generic_to_shared(row);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(p)
                 : "memory");
}
// A fragment (16 x 16) of the TRANSPOSE of M[k][m], 16 rows k: (m, k) = M[k][m0 + m].
__device__ __forceinline__ void a_frag_t(const __nv_bfloat16* M, int m0, uint32_t (&a)[4])
{
    const int lane = threadIdx.x & 31, tile = lane >> 3, r = lane & 7;
    ldmatrix_x4_trans(a, M + ((tile >> 1) * 8 + r) * LD + m0 + (tile & 1) * 8);
}
// B fragments (16 x 8 each) of columns n0 .. n0+7 (b[0], b[1]) and n0+8 ..
// n0+15 (b[2], b[3]) of a matrix stored as M[k][n], 16 rows k.
__device__ __forceinline__ void b_frag_kn2(const __nv_bfloat16* M, int n0, uint32_t (&b)[4])
{
    const int lane = threadIdx.x & 31, tile = lane >> 3, r = lane & 7;
    ldmatrix_x4_trans(b, M + ((tile & 1) * 8 + r) * LD + n0 + (tile >> 1) * 8);
}
// A fragment of a 16 x 32 activation held as C fragments c[ntile][4] (k-step kk).
__device__ __forceinline__ void a_from_c(const float (&c)[4][4], int kk, uint32_t (&a)[4])
{
    a[0] = pack_bf16(c[2 * kk][0], c[2 * kk][1]);
    a[1] = pack_bf16(c[2 * kk][2], c[2 * kk][3]);
    a[2] = pack_bf16(c[2 * kk + 1][0], c[2 * kk + 1][1]);
    a[3] = pack_bf16(c[2 * kk + 1][2], c[2 * kk + 1][3]);
}
// C fragments of a 16 x 32 activation into M[s][n] (BF16 pairs).
__device__ __forceinline__ void store_c(const float (&c)[4][4], __nv_bfloat16* M)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        *reinterpret_cast<uint32_t*>(M + g * LD + 8 * nt + 2 * t) = pack_bf16(c[nt][0], c[nt][1]);
        *reinterpret_cast<uint32_t*>(M + (g + 8) * LD + 8 * nt + 2 * t) =
            pack_bf16(c[nt][2], c[nt][3]);
    }
}

// Site index of minibatch entry k of Adam step `step`: word k%4 of Philox
// block k/4 (counter {k/4, step, 3, 0}, key {seed, 0}), floor(hi32(w) T / 2^32).
__device__ __forceinline__ int64_t batch_site(uint64_t seed, uint64_t step, int64_t k, int64_t T)
{
    const u64x4 w = philox_block(seed, 0, step, 3, (uint64_t)(k >> 2));
    const uint64_t hi = w.w[k & 3] >> 32;
    return (int64_t)((hi * (uint64_t)T) >> 32);
}

// Forward of the 16 sites of this warp.  fs: [16][LD] features in BF16
// (shared).  Outputs: a1, a2 in C-fragment form, z3 for rows g and g+8.
__device__ __forceinline__ void mlp_forward(const SParams& sp, const __nv_bfloat16* fs, float (&a1)[4][4],
                                            float (&a2)[4][4], float& z3g, float& z3g8)
{
    const int lane = threadIdx.x & 31, t = lane & 3;
    float z1[4][4] = {};
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
        uint32_t a[4];
        a_frag_mk(fs, 16 * kk, a);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            uint32_t b0, b1;
            b_frag_nk(sp.w1, 8 * nt, 16 * kk, b0, b1);
            mma_bf16(z1[nt], a, b0, b1);
        }
    }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int n0 = 8 * nt + 2 * t;
        a1[nt][0] = tanhf(z1[nt][0] + sp.b1[n0]);
        a1[nt][1] = tanhf(z1[nt][1] + sp.b1[n0 + 1]);
        a1[nt][2] = tanhf(z1[nt][2] + sp.b1[n0]);
        a1[nt][3] = tanhf(z1[nt][3] + sp.b1[n0 + 1]);
    }
    float z2[4][4] = {};
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
        uint32_t a[4];
        a_from_c(a1, kk, a);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            uint32_t b0, b1;
            b_frag_nk(sp.w2, 8 * nt, 16 * kk, b0, b1);
            mma_bf16(z2[nt], a, b0, b1);
        }
    }
    float pg = 0.f, pg8 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int n0 = 8 * nt + 2 * t;
        a2[nt][0] = tanhf(z2[nt][0] + sp.b2[n0]);
        a2[nt][1] = tanhf(z2[nt][1] + sp.b2[n0 + 1]);
        a2[nt][2] = tanhf(z2[nt][2] + sp.b2[n0]);
        a2[nt][3] = tanhf(z2[nt][3] + sp.b2[n0 + 1]);
        pg = fmaf(a2[nt][0], sp.w3[n0], fmaf(a2[nt][1], sp.w3[n0 + 1], pg));
        pg8 = fmaf(a2[nt][2], sp.w3[n0], fmaf(a2[nt][3], sp.w3[n0 + 1], pg8));
    }
    // the 4 lanes of a group hold the 32 columns of rows g and g+8
    pg += __shfl_xor_sync(0xffffffffu, pg, 1);
    pg += __shfl_xor_sync(0xffffffffu, pg, 2);
    pg8 += __shfl_xor_sync(0xffffffffu, pg8, 1);
    pg8 += __shfl_xor_sync(0xffffffffu, pg8, 2);
    z3g = pg + sp.b3;
    z3g8 = pg8 + sp.b3;
}

struct StepArgs {
    const float* feat;    // [T][NF] standardised features
    const float* target;  // [T]
    int64_t T;
    float* params;        // [NPARAM] FP32 master, updated in place
    float* adam_m;
    float* adam_v;
    float* grad_out;      // optional: the gradient of this batch [NPARAM]
    float* partials;      // [batch / 64][NPARAM + 1]
    unsigned* counter;    // arrival counter (step kernel) or grid barrier (training kernel)
    uint64_t seed, step;  // minibatch of Adam step `step`
    int64_t adam_t;       // 1-based Adam time of this step
    float lr, b1, b2, eps;
    int batch;
    int update;
    float* loss_out;      // optional
    const float* log_scale;  // optional device scalar: log s
    // training kernel: steps of this launch, the barrier's wait limit (clock
    // cycles) and the status word that tells of a wait that ran out
    int n_steps;
    long long wait_limit;
    int* status;
};

// The features and targets of a warp's 16 sites of one minibatch, fetched into
// registers: lane l holds elements l, l + 32, ... of the 16 x NF features, and
// the site index and target of entry l & 15.
struct Fetch {
    float f[16 * NF / 32];
    float y;
};
static_assert(16 * NF % 32 == 0, "whole lanes");
__device__ __forceinline__ void fetch_sites(const StepArgs& A, uint64_t step, int64_t k0, Fetch& q)
{
    const int lane = threadIdx.x & 31;
    const int64_t site = batch_site(A.seed, step, k0 + (lane & 15), A.T);
    q.y = A.target[site];
#pragma unroll
    for (int i = 0; i < 16 * NF / 32; ++i) {
        const int e = lane + 32 * i;
        q.f[i] = A.feat[__shfl_sync(0xffffffffu, site, e / NF) * NF + e % NF];
    }
}

// The block's working memory (dynamic shared memory).
struct __align__(16) StepSmem {
    SParams sp;
    __nv_bfloat16 fs[4][16 * LD];  // features of the warp's sites
    __nv_bfloat16 a1[4][16 * LD];  // a1, for dW2
    __nv_bfloat16 d[4][16 * LD];   // dz2, then dz1
    float grad[4][NPARAM + 1];     // each warp's gradient (and loss, the last slot)
};
__device__ __forceinline__ void pad_features(StepSmem& S)
{
    for (int i = threadIdx.x; i < 4 * 16 * (KP - NF); i += blockDim.x)
        S.fs[0][(i / (KP - NF)) * LD + NF + i % (KP - NF)] = __float2bfloat16_rn(0.f);
}

// Loss and gradient of one group of 64 minibatch sites (16 per warp) by a
// block of 128 threads, into part[NPARAM + 1]: the warps' sums added in warp
// order.  The parameters are in S.sp, the warp's sites in q; ends with the
// block's stores to part issued (no barrier).
__device__ __forceinline__ void mlp_group(StepSmem& S, const Fetch& q, const StepArgs& A, float ls,
                                          float* __restrict__ part)
{
    const SParams& sp = S.sp;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    __nv_bfloat16* fs = S.fs[warp];
    __nv_bfloat16* st_a1 = S.a1[warp];
    __nv_bfloat16* st_d = S.d[warp];
    float* gr = S.grad[warp];
#pragma unroll
    for (int i = 0; i < 16 * NF / 32; ++i) {
        const int e = lane + 32 * i;
        fs[(e / NF) * LD + e % NF] = __float2bfloat16_rn(q.f[i]);
    }
    __syncwarp();
    float a1[4][4], a2[4][4], z3g, z3g8;
    mlp_forward(sp, fs, a1, a2, z3g, z3g8);
    // loss gradient at rows g and g+8
    const float yg = __shfl_sync(0xffffffffu, q.y, g), yg8 = __shfl_sync(0xffffffffu, q.y, g + 8);
    const float mg = softplus_f(z3g) + EPS_M, mg8 = softplus_f(z3g8) + EPS_M;
    const float lg = logf(mg) + ls - yg, lg8 = logf(mg8) + ls - yg8;
    const float invB = 1.f / (float)A.batch;
    const float g3g = 2.f * lg * invB * sigmoid_f(z3g) / mg;
    const float g3g8 = 2.f * lg8 * invB * sigmoid_f(z3g8) / mg8;
    // dz2 = g3 W3 (1 - a2^2); dW3 = sum g3 a2; db2 = sum dz2
    float dz2[4][4];
    float pw3[4][2], pb2[4][2];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int n0 = 8 * nt + 2 * t;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float w = sp.w3[n0 + c];
            dz2[nt][c] = g3g * w * (1.f - a2[nt][c] * a2[nt][c]);
            dz2[nt][2 + c] = g3g8 * w * (1.f - a2[nt][2 + c] * a2[nt][2 + c]);
            pw3[nt][c] = g3g * a2[nt][c] + g3g8 * a2[nt][2 + c];
            pb2[nt][c] = dz2[nt][c] + dz2[nt][2 + c];
        }
    }
    // stage a1 and dz2 for the weight gradient of layer 2
    store_c(a1, st_a1);
    store_c(dz2, st_d);
    __syncwarp();
    // dW2[n][k] = sum_s dz2[s][n] a1[s][k]: M = n (2 tiles), N = k (4 tiles), K = 16 sites
    uint32_t b1f[2][4];
    b_frag_kn2(st_a1, 0, b1f[0]);
    b_frag_kn2(st_a1, 16, b1f[1]);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        uint32_t a[4];
        a_frag_t(st_d, 16 * mt, a);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            float gw[4] = {};
            mma_bf16(gw, a, b1f[nt >> 1][2 * (nt & 1)], b1f[nt >> 1][2 * (nt & 1) + 1]);
            const int n = 16 * mt + g, k = 8 * nt + 2 * t;
            gr[OFF_W2 + n * NH + k] = gw[0];
            gr[OFF_W2 + n * NH + k + 1] = gw[1];
            gr[OFF_W2 + (n + 8) * NH + k] = gw[2];
            gr[OFF_W2 + (n + 8) * NH + k + 1] = gw[3];
        }
    }
    // da1 = dz2 W2 (A = dz2 rows = sites; B(k=n, n=j) = W2[n][j])
    float da1[4][4] = {};
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
        uint32_t a[4];
        a_from_c(dz2, kk, a);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            uint32_t b0, b1;
            b_frag_nk(sp.w2t, 8 * nt, 16 * kk, b0, b1);
            mma_bf16(da1[nt], a, b0, b1);
        }
    }
    // dz1 = da1 (1 - a1^2); db1 = sum dz1; stage dz1 for dW1
    float pb1[4][2];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
        for (int c = 0; c < 4; ++c) da1[nt][c] = da1[nt][c] * (1.f - a1[nt][c] * a1[nt][c]);
        pb1[nt][0] = da1[nt][0] + da1[nt][2];
        pb1[nt][1] = da1[nt][1] + da1[nt][3];
    }
    __syncwarp();
    store_c(da1, st_d);
    // sum over the 8 groups of the warp (rows), then one lane per column keeps it
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                pw3[nt][c] += __shfl_xor_sync(0xffffffffu, pw3[nt][c], o);
                pb2[nt][c] += __shfl_xor_sync(0xffffffffu, pb2[nt][c], o);
                pb1[nt][c] += __shfl_xor_sync(0xffffffffu, pb1[nt][c], o);
            }
    __syncwarp();
    // dW1[n][f] = sum_s dz1[s][n] F[s][f]: M = n (2 tiles), N = f (3 tiles hold all features)
    b_frag_kn2(fs, 0, b1f[0]);
    b_frag_kn2(fs, 16, b1f[1]);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        uint32_t a[4];
        a_frag_t(st_d, 16 * mt, a);
#pragma unroll
        for (int nt = 0; nt < 3; ++nt) {
            float gw[4] = {};
            mma_bf16(gw, a, b1f[nt >> 1][2 * (nt & 1)], b1f[nt >> 1][2 * (nt & 1) + 1]);
            const int n = 16 * mt + g, k = 8 * nt + 2 * t;
            if (k < NF) {
                gr[OFF_W1 + n * NF + k] = gw[0];
                gr[OFF_W1 + (n + 8) * NF + k] = gw[2];
            }
            if (k + 1 < NF) {
                gr[OFF_W1 + n * NF + k + 1] = gw[1];
                gr[OFF_W1 + (n + 8) * NF + k + 1] = gw[3];
            }
        }
    }
    // loss of the warp's sites
    float lsum = (t == 0) ? (lg * lg + lg8 * lg8) : 0.f;
    float g3sum = (t == 0) ? (g3g + g3g8) : 0.f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        g3sum += __shfl_xor_sync(0xffffffffu, g3sum, o);
    }
    if (g == 0) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int n = 8 * nt + 2 * t + c;
                gr[OFF_W3 + n] = pw3[nt][c];
                gr[OFF_B2 + n] = pb2[nt][c];
                gr[OFF_B1 + n] = pb1[nt][c];
            }
    }
    if (lane == 0) {
        gr[OFF_B3] = g3sum;
        gr[NPARAM] = lsum;
    }
    __syncthreads();
    for (int i = tid; i < NPARAM + 1; i += blockDim.x)
        part[i] = ((S.grad[0][i] + S.grad[1][i]) + S.grad[2][i]) + S.grad[3][i];
}

// Adam (Kingma & Ba 2015) of parameter i with gradient g, FP32; c1 = 1 - b1^t
// and c2 = 1 - b2^t of the step's time t.
struct AdamState {
    float m, v, p;
};
__device__ __forceinline__ AdamState adam_load(const StepArgs& A, int i)
{
    return AdamState{__ldcg(A.adam_m + i), __ldcg(A.adam_v + i), __ldcg(A.params + i)};
}
__device__ __forceinline__ void adam_step(const StepArgs& A, int i, float g, float c1, float c2,
                                          const AdamState& q)
{
    const float m = A.b1 * q.m + (1.f - A.b1) * g;
    const float v = A.b2 * q.v + (1.f - A.b2) * g * g;
    A.adam_m[i] = m;
    A.adam_v[i] = v;
    const float mh = m / c1;
    const float vh = v / c2;
    A.params[i] = q.p - A.lr * mh / (sqrtf(vh) + A.eps);
}
__device__ __forceinline__ void adam_corrections(const StepArgs& A, int64_t t, float& c1, float& c2)
{
    c1 = 1.f - powf(A.b1, (float)t);
    c2 = 1.f - powf(A.b2, (float)t);
}

// One minibatch in one launch, a block per group of 64 sites: loss and
// gradient partials of this block; the last block to arrive sums the partials
// in block order and (update != 0) takes an Adam step of the FP32 master
// parameters.  For a gradient alone, for training under stream capture and for
// batches whose blocks are not all resident (see k_mlp_train).
__global__ void __launch_bounds__(128) k_mlp_step(const StepArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepSmem& S = *reinterpret_cast<StepSmem*>(smem_raw);
    __shared__ int s_last;
    const int tid = threadIdx.x, warp = tid >> 5;
    Fetch q;
    fetch_sites(A, A.step, (int64_t)blockIdx.x * SITES_PER_BLOCK + warp * 16, q);
    load_params<128>(A.params, S.sp);
    pad_params<128>(S.sp);
    pad_features(S);
    __syncthreads();
    mlp_group(S, q, A, A.log_scale ? *A.log_scale : 0.f,
              A.partials + (int64_t)blockIdx.x * (NPARAM + 1));
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(A.counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    float c1 = 1.f, c2 = 1.f;
    if (A.update) adam_corrections(A, A.adam_t, c1, c2);
    for (int i = tid; i < NPARAM + 1; i += blockDim.x) {
        float s = 0.f;
#pragma unroll 16
        for (int b = 0; b < (int)gridDim.x; ++b)
            s += __ldcg(A.partials + (int64_t)b * (NPARAM + 1) + i);
        if (i == NPARAM) {
            if (A.loss_out) *A.loss_out = s / (float)A.batch;
            continue;
        }
        if (A.grad_out) A.grad_out[i] = s;
        if (A.update) adam_step(A, i, s, c1, c2, adam_load(A, i));
    }
    if (tid == 0) *A.counter = 0u;
}

// n_steps Adam steps in one cooperative launch.  A step of 64 blocks is a few
// microseconds of work between two points where every block needs all others:
// as launches it took 53 us (a launch, then one block of 128 threads adding 64
// partials for 14 parameters a thread).  Here the blocks stay: each takes its
// group's gradient, a grid barrier, then each adds the partials of its own
// slice of the parameters (block order, as the step kernel) and takes their
// Adam step, a second barrier.  The next minibatch's sites are fetched while
// the first barrier is waited for.  Batch 4096: 53 -> 7.9 us a step, batch 64 (one
// block) 27 -> 10.
struct GridBarrier {
    unsigned* bar;
    unsigned target;
    // this block's arrival (every thread's writes before it)
    __device__ __forceinline__ void arrive(unsigned blocks)
    {
        target += blocks;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(bar, 1u);
    }
    // all blocks' arrivals; false in every thread of the block when the wait
    // exceeds `limit` clock cycles (ST_TIMEOUT is then set)
    __device__ __forceinline__ bool wait(long long limit, int* status, int* s_ok)
    {
        if (threadIdx.x == 0) {
            const long long t0 = clock64();
            int ok = 1;
            unsigned v;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
                if (v >= target) break;
                if (clock64() - t0 > limit) {
                    ok = 0;
                    atomicOr(status, ST_TIMEOUT);
                    break;
                }
            }
            __threadfence();
            *s_ok = ok;
        }
        __syncthreads();
        return *s_ok != 0;
    }
};
constexpr int kRedRows = 128;  // partials staged at a time (of 32 parameters each)
__global__ void __launch_bounds__(128) k_mlp_train(const StepArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepSmem& S = *reinterpret_cast<StepSmem*>(smem_raw);
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nb = (int)gridDim.x;
    float* red = &S.grad[0][0];  // [kRedRows][32]
    static_assert(sizeof(S.grad) >= kRedRows * 32 * sizeof(float), "staging space");
    const int per = (NPARAM + 1 + nb - 1) / nb;  // parameters of a block's slice
    const int lo = min(blockIdx.x * per, NPARAM + 1), hi = min(lo + per, NPARAM + 1);
    const int64_t k0 = (int64_t)blockIdx.x * SITES_PER_BLOCK + warp * 16;
    const float ls = A.log_scale ? *A.log_scale : 0.f;
    pad_params<128>(S.sp);
    pad_features(S);
    Fetch q;
    fetch_sites(A, A.step, k0, q);
    GridBarrier gb{A.counter, 0u};
    for (int n = 0; n < A.n_steps; ++n) {
        load_params<128>(A.params, S.sp);
        __syncthreads();
        mlp_group(S, q, A, ls, A.partials + (int64_t)blockIdx.x * (NPARAM + 1));
        gb.arrive(nb);
        if (n + 1 < A.n_steps) fetch_sites(A, A.step + n + 1, k0, q);
        if (!gb.wait(A.wait_limit, A.status, &s_ok)) return;
        float c1, c2;
        adam_corrections(A, A.adam_t + n, c1, c2);
        if (per <= 32) {
            // one parameter a lane: four warps stage the rows, one adds them
            const int i = lo + lane;
            AdamState q{0.f, 0.f, 0.f};
            if (warp == 0 && i < hi && i < NPARAM) q = adam_load(A, i);
            float s = 0.f;
            for (int r0 = 0; r0 < nb; r0 += kRedRows) {
                const int rows = min(kRedRows, nb - r0);
                __syncthreads();  // the staged rows are free
#pragma unroll 16
                for (int r = warp; r < rows; r += 4)
                    red[r * 32 + lane] =
                        i < hi ? __ldcg(A.partials + (int64_t)(r0 + r) * (NPARAM + 1) + i) : 0.f;
                __syncthreads();
                if (warp == 0) {
#pragma unroll 16
                    for (int r = 0; r < rows; ++r) s += red[r * 32 + lane];
                }
            }
            if (warp == 0 && i < hi) {
                if (i < NPARAM) adam_step(A, i, s, c1, c2, q);
                else if (A.loss_out) A.loss_out[n] = s / (float)A.batch;
            }
        } else if (per <= 128) {
            // one parameter a thread
            const int i = lo + tid;
            if (i < hi) {
                AdamState q{0.f, 0.f, 0.f};
                if (i < NPARAM) q = adam_load(A, i);
                float s = 0.f;
#pragma unroll 16
                for (int r = 0; r < nb; ++r)
                    s += __ldcg(A.partials + (int64_t)r * (NPARAM + 1) + i);
                if (i < NPARAM) adam_step(A, i, s, c1, c2, q);
                else if (A.loss_out) A.loss_out[n] = s / (float)A.batch;
            }
        } else {
            // few blocks, many parameters each: kU a thread at a time over few rows
            constexpr int kU = 7;
            for (int i0 = lo + tid; i0 < hi; i0 += 128 * kU) {
                float s[kU];
                AdamState q[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int i = i0 + 128 * u;
                    s[u] = 0.f;
                    if (i < hi && i < NPARAM) q[u] = adam_load(A, i);
                }
                for (int r = 0; r < nb; ++r)
#pragma unroll
                    for (int u = 0; u < kU; ++u)
                        if (i0 + 128 * u < hi)
                            s[u] += __ldcg(A.partials + (int64_t)r * (NPARAM + 1) + i0 + 128 * u);
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int i = i0 + 128 * u;
                    if (i >= hi) continue;
                    if (i < NPARAM) adam_step(A, i, s[u], c1, c2, q[u]);
                    else if (A.loss_out) A.loss_out[n] = s[u] / (float)A.batch;
                }
            }
        }
        if (n + 1 == A.n_steps) return;
        gb.arrive(nb);
        if (!gb.wait(A.wait_limit, A.status, &s_ok)) return;
    }
}

// m_t for every site, clamped to [1/s_u^2, diagonal of the Hessian of S at
// hbar] = [1/s_u^2, A_t/s_eta^2 + 1/s_u^2 + (y_t^2/2) e^{-hbar_t}], A_t = 1 +
// phi^2 inside, 1 at the ends, 1 - phi^2 when T = 1; writes 1/m_t (and m_t if
// m_out).  A warp takes 32 sites: two tiles through the network, then one site
// per lane for the output and its clamp, whose FP64 instructions cost the same
// for one active lane as for 32 (taken by 8 lanes a tile they were most of the
// kernel).  2^20 sites: 305 -> 81 us.
__global__ void __launch_bounds__(128) k_mlp_mass(const float* __restrict__ feat, int64_t T,
                                                  const float* __restrict__ P,
                                                  const double* __restrict__ y,
                                                  const double* __restrict__ hbar, ThetaD th,
                                                  const float* __restrict__ log_scale,
                                                  const int* __restrict__ status,
                                                  float* __restrict__ minv, float* __restrict__ m_out)
{
    __shared__ SParams sp;
    __shared__ __align__(16) __nv_bfloat16 fs[4][32 * LD];
    __shared__ u64 s_exp[kExpN];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float scale = log_scale ? expf(*log_scale) : 1.f;
    load_params<128>(P, sp);
    pad_params<128>(sp);
    exp_table(s_exp);
    for (int i = tid; i < 4 * 32 * (KP - NF); i += 128)
        fs[0][(i / (KP - NF)) * LD + NF + i % (KP - NF)] = __float2bfloat16_rn(0.f);
    __syncthreads();
    const double lo = 1.0 / th.su2;
    const double in = (1.0 + th.phi * th.phi) / th.se2 + lo;
    const double end = (T == 1 ? 1.0 - th.phi * th.phi : 1.0) / th.se2 + lo;
    const float lof = (float)lo;
    // parameters of a training that ended early give no mass
    const float valid = (*status & ST_TIMEOUT) ? NAN : 1.f;
    for (int64_t base = ((int64_t)blockIdx.x * 4 + warp) * 32; base < T;
         base += (int64_t)gridDim.x * 128) {
        const int64_t s = base + lane;
        const bool act = s < T;
        const double yv = act ? y[s] : 0.0, hv = act ? hbar[s] : 0.0;
        const int64_t nf = (T - base < 32 ? T - base : 32) * NF;
        float v[NF];  // the warp's 32 x NF features with consecutive lanes
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            const int e = lane + 32 * i;
            v[i] = e < nf ? feat[base * NF + e] : 0.f;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            const int e = lane + 32 * i;
            fs[warp][(e / NF) * LD + e % NF] = __float2bfloat16_rn(v[i]);
        }
        __syncwarp();
        float z = 0.f;
#pragma unroll 1
        for (int tile = 0; tile < 2; ++tile) {
            float a1[4][4], a2[4][4], zg, zg8;
            mlp_forward(sp, fs[warp] + tile * 16 * LD, a1, a2, zg, zg8);
            // lane r of the tile's 16 takes row r (held by the lanes of group r & 7)
            const float u = __shfl_sync(0xffffffffu, zg, (lane & 7) * 4);
            const float w = __shfl_sync(0xffffffffu, zg8, (lane & 7) * 4);
            if ((lane >> 4) == tile) z = (lane & 8) ? w : u;
        }
        if (act) {
            const double hi = (s == 0 || s == T - 1 ? end : in) + 0.5 * yv * yv * exp_neg(hv, s_exp);
            const float m = fminf(fmaxf(scale * (softplus_f(z) + EPS_M), lof), (float)hi);
            minv[s] = valid / m;
            if (m_out) m_out[s] = valid * m;
        }
    }
}

// Fold n snapshot rows of x ([n][T] FP32) into running (count, mean, M2) by
// Welford's recurrence, row by row.  Bound by the FP64 pipe: the recurrence's
// seven instructions a value.  The widening of x is done on integers, and the
// division by the row's count n_k is q = d y, q + (d - q n_k) y with y = 1/n_k
// rounded to nearest: d - q n_k is exact (a multiple of ulp(q) below 2 n_k of
// them), so the sum differs from d/n_k by less than 2^-51 ulp, while an FP64
// quotient by an integer n_k lies at least 1/(2 n_k) ulp from every midpoint;
// the result is the correctly rounded quotient for n_k < 2^48, the value a
// division gives.  (Outside the exponents where these hold, a division.)
// 100 rows of 2^20 sites: 2.83 -> 1.31 ms, the same bits.
constexpr int kWelRows = 256;  // rows whose counts a block holds at a time
static __device__ __noinline__ double div_slow(double d, double n) { return d / n; }
__device__ __forceinline__ double div_count(double d, double n, double y)
{
    const unsigned h = (unsigned)__double2hiint(d), e = (h >> 20) & 0x7ffu;
    if (e - 64u > 1900u)
        return ((h << 1) | (unsigned)__double2loint(d)) == 0u ? d : div_slow(d, n);
    const double q = d * y;
    return fma(fma(-q, n, d), y, q);
}
__global__ void __launch_bounds__(256) k_welford(const float* __restrict__ x, int64_t n, int64_t T,
                                                 int64_t count, double* __restrict__ mean,
                                                 double* __restrict__ m2)
{
    __shared__ double2 s_n[kWelRows];  // (n_k, 1/n_k)
    const bool small = count + n < (int64_t(1) << 48);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t rounds = (T + stride - 1) / stride;  // the same for every thread
    for (int64_t i = 0; i < rounds; ++i) {
        const int64_t t = i * stride + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        const bool act = t < T;
        double m = act && count ? mean[t] : 0.0, s = act && count ? m2[t] : 0.0;
        for (int64_t k0 = 0; k0 < n; k0 += kWelRows) {
            const int rows = (int)(n - k0 < kWelRows ? n - k0 : kWelRows);
            __syncthreads();
            for (int r = threadIdx.x; r < rows; r += blockDim.x) {
                const double nk = (double)(count + k0 + r + 1);
                s_n[r] = make_double2(nk, 1.0 / nk);
            }
            __syncthreads();
            if (!act) continue;
            const float* xp = x + k0 * T + t;
            auto row = [&](float xv, int r) {
                const double v = f32_to_f64(xv);
                const double d = v - m;
                m += small ? div_count(d, s_n[r].x, s_n[r].y) : div_slow(d, s_n[r].x);
                s += d * (v - m);
            };
            constexpr int U = 8;  // rows in flight
            int r = 0;
            for (; r + U <= rows; r += U) {
                float v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = xp[(r + u) * T];
#pragma unroll
                for (int u = 0; u < U; ++u) row(v[u], r + u);
            }
            for (; r < rows; ++r) row(xp[r * T], r);
        }
        if (act) {
            mean[t] = m;
            m2[t] = s;
        }
    }
}

// Sums of one value per block, for a last-block finish: true in every thread
// of the last block to arrive.
__device__ __forceinline__ bool last_block(unsigned* counter, int* s_last)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!*s_last) return false;
    __threadfence();
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

// target_t = log(1 / Var(h_t)) = log((count - 1) / M2_t); hbar_t = mean_t; and
// log s = the mean over the sites of the target (FP64, fixed order), if asked
// for (one block over all sites took 0.59 ms for it at 2^20 sites).
__global__ void __launch_bounds__(256) k_welford_target(
    const double* __restrict__ mean, const double* __restrict__ m2, int64_t T, int64_t count,
    double* __restrict__ hbar, float* __restrict__ target, float* __restrict__ log_scale,
    double* __restrict__ partials, unsigned* __restrict__ counter)
{
    __shared__ double red[32];
    __shared__ int s_last;
    const double nk = (double)(count - 1), inv = 1.0 / nk;
    const bool small = count < (int64_t(1) << 48);
    double sum = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < T;
         t += (int64_t)gridDim.x * blockDim.x) {
        if (hbar) hbar[t] = mean[t];
        const double var = small ? div_count(m2[t], nk, inv) : m2[t] / nk;
        const float v = (float)log(1.0 / fmax(var, 1e-300));
        target[t] = v;
        if (log_scale) sum += f32_to_f64(v);
    }
    if (!log_scale) return;
    sum = block_sum(sum, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = sum;
    if (!last_block(counter, &s_last)) return;
    sum = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) sum += __ldcg(partials + i);
    sum = block_sum(sum, red);
    if (threadIdx.x == 0) *log_scale = (float)(sum / (double)T);
}

// The raw features of a site that depend on it (FP32): y^2, lnRV, hbar and
// (y^2/2) e^{-hbar}.  The other features are hbar of the eight sites around it
// (0 past the ends), constants of theta, and the edge proximity.
struct SiteFeat {
    float y2, lr, hb, ey;
};
__device__ __forceinline__ SiteFeat site_features(double y, double lr, double hb, const u64* s_exp)
{
    return SiteFeat{(float)(y * y), (float)lr, (float)hb, (float)(0.5 * y * y * exp_neg(hb, s_exp))};
}
__device__ __forceinline__ float const_feature(int f, const ThetaD& th)
{
    switch (f) {
        case 11: return (float)th.phi;
        case 12: return (float)th.mu;
        case 13: return (float)th.xi;
        case 14: return (float)th.se2;
        case 15: return (float)th.su2;
        case 17: return (float)((1.0 + th.phi * th.phi) / th.se2);
        default: return (float)(1.0 / th.su2);  // 18
    }
}

// Mean and 1/sd of every feature over the sites, stats = [mean(20), inv_sd(20)]:
// one pass over the inputs (24 B a site), sums in FP64 of the four site
// features about centres near their means, so that the squares keep the
// accuracy of a second pass: the mean of up to 256 sites spread over the
// series, which every block takes for itself.  (That mean is within sd
// sqrt(T / 256) of the mean, which costs the variance at most T / 256 ulp.)  The
// nine hbar columns are the same values but for the four sites at either end,
// which some columns leave out: hbar is summed without them and each column
// adds its own; constants are exact.  (The features were written out, 80 B a
// site, read back twice for the statistics and once to be standardised in
// place: 640 us at 2^20 sites, 110 now.)
constexpr int kFeatSums = 8, kFeatThreads = 256, kWing = 4;
__global__ void __launch_bounds__(kFeatThreads) k_feat_stats(
    const double* __restrict__ y, const double* __restrict__ lnrv, const double* __restrict__ hbar,
    int64_t T, ThetaD th, double* __restrict__ partials, unsigned* __restrict__ counter,
    float* __restrict__ stats)
{
    __shared__ double red[32], tot[kFeatSums], s_cf[4], s_end[2 * kWing], buf[4][kFeatThreads];
    __shared__ u64 s_exp[kExpN];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    exp_table(s_exp);
    __syncthreads();
    double cf[4];  // the centres (any finite value serves)
    {
        const int64_t m = T < kFeatThreads ? T : kFeatThreads, t = tid * T / m + T / (2 * m);
        const bool act = tid < m, in = act && t >= kWing && t < T - kWing;
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (act) {
            const SiteFeat q = site_features(y[t], lnrv[t], hbar[t], s_exp);
            v[0] = q.y2;
            v[1] = q.lr;
            v[2] = in ? q.hb : 0.f;
            v[3] = q.ey;
        }
        if (tid < 2 * kWing && T > 2 * kWing)  // the sites at the ends, for the finish
            s_end[tid] = (double)(float)hbar[tid < kWing ? tid : T - 2 * kWing + tid];
        const int n_in = __syncthreads_count(in);
        block_sum_many<4, kFeatThreads>(v, buf, tot);
        if (tid < 4) {
            const double c = tot[tid] / (tid == 2 ? (double)(n_in > 0 ? n_in : 1) : (double)m);
            s_cf[tid] = isfinite(c) ? c : 0.0;
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) cf[i] = s_cf[i];
    double sum[kFeatSums];
#pragma unroll
    for (int i = 0; i < kFeatSums; ++i) sum[i] = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + tid; t < T;
         t += (int64_t)gridDim.x * blockDim.x) {
        const SiteFeat q = site_features(y[t], lnrv[t], hbar[t], s_exp);
        const float v[4] = {q.y2, q.lr, q.hb, q.ey};
        const bool in = t >= kWing && t < T - kWing;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i == 2 && !in) continue;
            const double d = f32_to_f64(v[i]) - cf[i];
            sum[2 * i] += d;
            sum[2 * i + 1] = fma(d, d, sum[2 * i + 1]);
        }
    }
#pragma unroll
    for (int i = 0; i < kFeatSums; ++i) {
        const double b = block_sum(sum[i], red);
        if (tid == 0) partials[(int64_t)blockIdx.x * kFeatSums + i] = b;
    }
    if (!last_block(counter, &s_last)) return;
    {   // warp i adds sum i over the blocks
        const int i = tid >> 5, lane = tid & 31;
        static_assert(kFeatSums * 32 == kFeatThreads, "one warp per sum");
        double v = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32)
            v += __ldcg(partials + (int64_t)b * kFeatSums + i);
        v = warp_sum(v);
        if (lane == 0) tot[i] = v;
    }
    __syncthreads();
    const int f = tid;
    if (f >= NF) return;
    double s1 = 0.0, s2 = 0.0, cen = 0.0;
    if (f == 0 || f == 1 || f == 19) {
        const int i = f == 19 ? 3 : f;
        cen = cf[i];
        s1 = tot[2 * i];
        s2 = tot[2 * i + 1];
    } else if (f >= 2 && f <= 10) {
        // the column of hbar_{t+k}: sites j = max(k, 0) .. min(T, T + k) - 1, |k| zeros
        const int64_t k = f - 6, lo = k > 0 ? k : 0, hi = k < 0 ? T + k : T;
        if (T <= 2 * kWing) {  // no site between the ends: two passes over the column
            for (int64_t j = lo; j < hi; ++j) s1 += (double)(float)hbar[j];
            cen = s1 / (double)T;
            s1 = 0.0;
            for (int64_t t = 0; t < T; ++t) {
                const int64_t j = t + k;
                const double d = (j >= 0 && j < T ? (double)(float)hbar[j] : 0.0) - cen;
                s2 = fma(d, d, s2);
            }
        } else {
            const double nz = (double)(k < 0 ? -k : k);
            cen = cf[2];
            s1 = fma(-nz, cen, tot[4]);
            s2 = fma(nz * cen, cen, tot[5]);
            for (int e = 0; e < 2 * kWing; ++e) {
                const int64_t j = e < kWing ? e : T - 2 * kWing + e;
                if (j < lo || j >= hi) continue;
                const double d = s_end[e] - cen;
                s1 += d;
                s2 = fma(d, d, s2);
            }
        }
    } else if (f != EDGE) {
        cen = (double)const_feature(f, th);
    }
    const double dm = s1 / (double)T, m = cen + dm;
    const double sd = sqrt(fmax(s2 / (double)T - dm * dm, 0.0));
    stats[f] = f == EDGE ? 0.f : (float)m;
    stats[NF + f] = f == EDGE ? 1.f : (sd > 1e-12 * fmax(1.0, fabs(m))) ? (float)(1.0 / sd) : 0.f;
}

// The standardised, clipped features, 256 sites a block, staged in shared
// memory and written with consecutive lanes.
__global__ void __launch_bounds__(256) k_feat_write(const double* __restrict__ y,
                                                    const double* __restrict__ lnrv,
                                                    const double* __restrict__ hbar, int64_t T,
                                                    ThetaD th, const float* __restrict__ stats,
                                                    float* __restrict__ F)
{
    __shared__ float s_f[256 * NF], s_hb[256 + 8], s_m[NF], s_i[NF], s_c[NF];
    __shared__ u64 s_exp[kExpN];
    const int tid = threadIdx.x;
    exp_table(s_exp);
    if (tid < NF) {
        s_m[tid] = stats[tid];
        s_i[tid] = stats[NF + tid];
        s_c[tid] = const_feature(tid, th);
    }
    for (int64_t t0 = (int64_t)blockIdx.x * 256; t0 < T; t0 += (int64_t)gridDim.x * 256) {
        __syncthreads();
        const int64_t t = t0 + tid;
        const bool act = t < T;
        const SiteFeat q = site_features(act ? y[t] : 0.0, act ? lnrv[t] : 0.0, act ? hbar[t] : 0.0,
                                         s_exp);
        s_hb[tid + 4] = act ? q.hb : 0.f;
        if (tid < 8) {
            const int64_t s = tid < 4 ? t0 - 4 + tid : t0 + 256 + (tid - 4);
            s_hb[tid < 4 ? tid : 256 + tid] = (s >= 0 && s < T) ? (float)hbar[s] : 0.f;
        }
        __syncthreads();
        auto put = [&](int f, float v) {
            s_f[tid * NF + f] = fminf(fmaxf((v - s_m[f]) * s_i[f], -CLIP), CLIP);
        };
        const int64_t d = t < T - 1 - t ? t : T - 1 - t;  // distance to the nearer end
        put(0, q.y2);
        put(1, q.lr);
#pragma unroll
        for (int k = 0; k < 9; ++k) put(2 + k, s_hb[tid + k]);
#pragma unroll
        for (int f = 11; f < 16; ++f) put(f, s_c[f]);
        put(16, ldexpf(1.f, -(int)(d < 64 ? d : 64)));
        put(17, s_c[17]);
        put(18, s_c[18]);
        put(19, q.ey);
        __syncthreads();
        const int n = (int)(T - t0 < 256 ? T - t0 : 256) * NF;
        for (int i = tid; i < n; i += 256) F[t0 * NF + i] = s_f[i];
    }
}

constexpr int kGrid1Max = 152 * 8;
int grid1(int64_t n)
{
    int64_t g = (n + 255) / 256;
    if (g > kGrid1Max) g = kGrid1Max;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

int mlp_nparam() { return NPARAM; }
int mlp_sites_per_block() { return SITES_PER_BLOCK; }

cudaError_t launch_mlp_step(const float* feat, const float* target, int64_t T, float* params,
                            float* grad_out, float* partials, unsigned* counter, uint64_t seed,
                            uint64_t step, int batch, float* loss_out, const float* log_scale,
                            cudaStream_t st)
{
    StepArgs a{};
    a.feat = feat;
    a.target = target;
    a.T = T;
    a.params = params;
    a.grad_out = grad_out;
    a.partials = partials;
    a.counter = counter;
    a.seed = seed;
    a.step = step;
    a.batch = batch;
    a.loss_out = loss_out;
    a.log_scale = log_scale;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_step, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(StepSmem));
    if (e != cudaSuccess) return e;
    k_mlp_step<<<batch / SITES_PER_BLOCK, 128, sizeof(StepSmem), st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_mlp_train(const float* feat, const float* target, int64_t T, float* params,
                             float* adam_m, float* adam_v, float* partials, unsigned* counter,
                             unsigned* barrier, uint64_t seed, int64_t step0, int n_steps, float lr,
                             int batch, float* loss_out, const float* log_scale, bool capturing,
                             int num_sms, long long wait_limit, int* status, int64_t* launches,
                             cudaStream_t st)
{
    StepArgs a{};
    a.feat = feat;
    a.target = target;
    a.T = T;
    a.params = params;
    a.adam_m = adam_m;
    a.adam_v = adam_v;
    a.partials = partials;
    a.seed = seed;
    a.lr = lr;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.batch = batch;
    a.update = 1;
    a.log_scale = log_scale;
    a.wait_limit = wait_limit;
    a.status = status;
    const int nb = batch / SITES_PER_BLOCK;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(StepSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_step, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(StepSmem));
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mlp_train, 128,
                                                          sizeof(StepSmem));
    if (e != cudaSuccess) return e;
    // one launch for all steps when every block can be resident (the barrier
    // waits for all of them); its counter takes 2 nb per step, < 2^32
    const bool coop = !capturing && n_steps > 1 && nb <= per_sm * num_sms;
    const int most = coop ? 1 << 20 : 1;
    for (int i = 0; i < n_steps; i += most) {
        a.step = (uint64_t)(step0 + i);
        a.adam_t = step0 + i + 1;
        a.loss_out = loss_out ? loss_out + i : nullptr;
        ++*launches;
        if (coop) {
            a.n_steps = n_steps - i < most ? n_steps - i : most;
            a.counter = barrier;
            if ((e = cudaMemsetAsync(barrier, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
            void* args[] = {&a};
            e = cudaLaunchCooperativeKernel((const void*)k_mlp_train, dim3(nb), dim3(128), args,
                                            sizeof(StepSmem), st);
        } else {
            a.n_steps = 1;
            a.counter = counter;
            k_mlp_step<<<nb, 128, sizeof(StepSmem), st>>>(a);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_mlp_mass(const float* feat, int64_t T, const float* params, const double* y,
                            const double* hbar, ThetaD th, const float* log_scale,
                            const int* status, float* minv, float* m_out, cudaStream_t st)
{
    int64_t g = (T + 127) / 128;
    if (g > 152 * 8) g = 152 * 8;
    k_mlp_mass<<<(int)(g < 1 ? 1 : g), 128, 0, st>>>(feat, T, params, y, hbar, th, log_scale,
                                                      status, minv, m_out);
    return cudaGetLastError();
}

cudaError_t launch_welford(const float* x, int64_t n, int64_t T, int64_t count, double* mean,
                           double* m2, cudaStream_t st)
{
    const int64_t g = (T + 255) / 256;
    k_welford<<<(unsigned)(g < 65536 ? g : 65536), 256, 0, st>>>(x, n, T, count, mean, m2);
    return cudaGetLastError();
}

cudaError_t launch_welford_target(const double* mean, const double* m2, int64_t T, int64_t count,
                                  double* hbar, float* target, float* log_scale, double* partials,
                                  unsigned* counter, cudaStream_t st)
{
    k_welford_target<<<grid1(T), 256, 0, st>>>(mean, m2, T, count, hbar, target, log_scale,
                                               partials, counter);
    return cudaGetLastError();
}

size_t target_blocks() { return kGrid1Max; }
int feat_grid(int64_t T) { return grid1(T); }

cudaError_t launch_features(const double* y, const double* lnrv, const double* hbar, int64_t T,
                            ThetaD th, float* F, float* stats, double* partials, unsigned* counter,
                            cudaStream_t st)
{
    // two blocks per SM: a block's FP64 reductions cost as much as a few hundred sites
    const int g = grid1(T);
    k_feat_stats<<<g < 304 ? g : 304, kFeatThreads, 0, st>>>(y, lnrv, hbar, T, th, partials, counter, stats);
    k_feat_write<<<g, 256, 0, st>>>(y, lnrv, hbar, T, th, stats, F);
    return cudaGetLastError();
}

}  // namespace rsv
