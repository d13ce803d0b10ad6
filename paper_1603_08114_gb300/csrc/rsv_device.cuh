// rsv_device.cuh -- device helpers of librsv (sm_103a).
//
// Counter-based generator, Box-Muller, double-float error-free transforms and
// fixed-order reductions shared by the kernels of this library.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace rsv {

// Status bits written by kernels into the context status word.
enum : int { ST_NONFINITE = 1, ST_TIMEOUT = 2 };

// Philox counter streams (counter word 2).
enum : uint64_t { STREAM_MOM = 0, STREAM_MH = 1, STREAM_THETA = 2 };

// ---------------------------------------------------------------------------
// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11).  Each round maps
// (c0, c1, c2, c3) to (hi(B*c2) ^ c1 ^ k0, lo(B*c2), hi(A*c0) ^ c3 ^ k1, lo(A*c0))
// with A = 0xD2E7470EE14C6C93, B = 0xCA5A826395121157; between rounds the key
// advances by the Weyl increments 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B.
// ---------------------------------------------------------------------------
struct u64x4 { uint64_t w[4]; };

__device__ __forceinline__ u64x4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2,
                                               uint64_t c3, uint64_t k0, uint64_t k1)
{
    const uint64_t A = 0xD2E7470EE14C6C93ULL, B = 0xCA5A826395121157ULL;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B97F4A7C15ULL;
            k1 += 0xBB67AE8584CAA73BULL;
        }
        const uint64_t hiA = __umul64hi(A, c0), loA = A * c0;
        const uint64_t hiB = __umul64hi(B, c2), loB = B * c2;
        const uint64_t n0 = hiB ^ c1 ^ k0, n2 = hiA ^ c3 ^ k1;
        c0 = n0;
        c1 = loB;
        c2 = n2;
        c3 = loA;
    }
    u64x4 o;
    o.w[0] = c0; o.w[1] = c1; o.w[2] = c2; o.w[3] = c3;
    return o;
}

// Philox block `blk` of stream `stream` for trajectory `traj` of series `series`.
__device__ __forceinline__ u64x4 philox_block(uint64_t seed, uint64_t series, uint64_t traj,
                                             uint64_t stream, uint64_t blk)
{
    return philox4x64_10(blk, traj, stream, series, seed, 0ULL);
}

// (double)x without the FP64 pipe, on which float conversions run: the
// exponent re-biased and the mantissa shifted; zeros, subnormals, infinities and
// NaN take the conversion, out of line: inlined it would be predicated into
// every warp, and a predicated FP64 instruction occupies the pipe all the same.
static __device__ __noinline__ double f32_to_f64_slow(float x) { return (double)x; }
__device__ __forceinline__ double f32_to_f64(float x)
{
    const unsigned b = __float_as_uint(x);
    if ((b << 1) - 0x01000000u >= 0xfe000000u) return f32_to_f64_slow(x);
    return __hiloint2double((int)((b & 0x80000000u) | (((b >> 3) & 0x0fffffffu) + 0x38000000u)),
                            (int)(b << 29));
}

// Uniform in (0,1): (k + 1/2) 2^-53 from the top 53 bits.
__device__ __forceinline__ double u01_53(uint64_t w)
{
    return ((double)(w >> 11) + 0.5) * 0x1.0p-53;
}
// Uniform in (0,1) exactly representable in FP32: (k + 1/2) 2^-23, k = top 23
// bits.  Built from the bits (1 + k 2^-23 has k as its mantissa) so that no
// integer-to-float conversion runs: conversions share this GPU's slow FP64
// pipe.  Every step is exact: (1 + k 2^-23) - 1 = k 2^-23, + 2^-24 fits 24 bits.
__device__ __forceinline__ float u01_23(uint64_t w)
{
    const uint32_t k = (uint32_t)(w >> 41);
    return (__uint_as_float(0x3F800000u | k) - 1.0f) + 0x1.0p-24f;
}

// Box-Muller: r = sqrt(-2 ln u1); (r cos 2 pi u2, r sin 2 pi u2).
__device__ __forceinline__ void box_muller(double u1, double u2, double& z0, double& z1)
{
    const double r = sqrt(-2.0 * log(u1));
    double s, c;
    sincospi(2.0 * u2, &s, &c);
    z0 = r * c;
    z1 = r * s;
}
__device__ __forceinline__ void box_muller_f(float u1, float u2, float& z0, float& z1)
{
    const float r = sqrtf(-2.0f * logf(u1));
    float s, c;
    sincospif(2.0f * u2, &s, &c);
    z0 = r * c;
    z1 = r * s;
}

// ---------------------------------------------------------------------------
// Double-float arithmetic: a value is hi + lo with |lo| <= ulp(hi)/2.
// two_sum (Knuth), fast_two_sum (Dekker, |a| >= |b|), two_prod by FMA.
// Every add, subtract and multiply is an explicitly rounded intrinsic: the
// error-free transformations need s = fl(a + b) exactly, and the compiler
// would otherwise fuse a product feeding an add into an FMA (a different
// rounding of s).
// ---------------------------------------------------------------------------
struct ff { float hi, lo; };

__device__ __forceinline__ ff two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ ff fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    ff s = two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff{-b.hi, -b.lo}); }
__device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    ff p = two_prod(a.hi, b.hi);
    p.lo = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
    return fast_two_sum(p.hi, p.lo);
}
__device__ __forceinline__ ff ff_mul_f(ff a, float b)
{
    ff p = two_prod(a.hi, b);
    p.lo = __fmaf_rn(a.lo, b, p.lo);
    return fast_two_sum(p.hi, p.lo);
}
// Accumulate a double-float into a double-float (no renormalisation of the
// small part until read).
__device__ __forceinline__ void ff_acc(ff& acc, ff v)
{
    ff s = two_sum(acc.hi, v.hi);
    acc.hi = s.hi;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, v.lo));
}
__host__ __device__ __forceinline__ ff ff_from_double(double d)
{
    const float h = (float)d;
    return {h, (float)(d - (double)h)};
}
__device__ __forceinline__ double ff_to_double(ff a) { return (double)a.hi + (double)a.lo; }
// (float)d for kernels over many sites: the rounding to nearest even on the
// integer units (conversions run on the FP64 pipe, 2 lanes per cycle and SM).
// 2^-73 <= |d| < 2^127; others convert (out of line, see f32_to_f64).
static __device__ __noinline__ float f64_to_f32_slow(double d) { return (float)d; }
static __device__ __noinline__ ff ff_split_slow(double d) { return ff_from_double(d); }
__device__ __forceinline__ float f64_to_f32(double d)
{
    const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
    const unsigned E = (h >> 20) & 0x7ffu;
    if (E - 950u > 199u) return f64_to_f32_slow(d);
    unsigned fb = __funnelshift_l(l, h, 3) - 0xc0000000u;  // exponent re-biased, top 23 mantissa bits
    fb += ((l & 0x1fffffffu) + 0x0fffffffu + (fb & 1u)) >> 29;
    return __uint_as_float(fb | (h & 0x80000000u));
}
// ff_from_double likewise, the same bits: the 29 mantissa bits below the float
// (signed, after its rounding) become the small part, exactly converted in two
// pieces and rounded once.
__device__ __forceinline__ ff ff_split(double d)
{
    const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
    const unsigned E = (h >> 20) & 0x7ffu, sign = h & 0x80000000u;
    if (E - 950u > 199u) return ff_split_slow(d);
    unsigned fb = __funnelshift_l(l, h, 3) - 0xc0000000u;
    const unsigned r = l & 0x1fffffffu, up = (r + 0x0fffffffu + (fb & 1u)) >> 29;
    fb += up;
    const int D = (int)r - (int)(up << 29);  // |D| <= 2^28, in units of 2^(E - 1075)
    const float Dh = __fsub_rn(__uint_as_float((unsigned)(0x4b400000 + (D >> 8))), 12582912.0f);
    const float Dl = __fsub_rn(__uint_as_float(0x4b000000u | (unsigned)(D & 0xff)), 8388608.0f);
    const float m = __fmul_rn(__fmaf_rn(Dh, 256.0f, Dl), __uint_as_float((E - 948u) << 23));
    return {__uint_as_float(fb | sign), __fadd_rn(__uint_as_float(__float_as_uint(m) ^ sign), 0.0f)};
}

// Table of 2^(j/32), j = 0..31, as double-float pairs (filled by ff_exp_table).
__device__ __forceinline__ void ff_exp_table(float2* tab)
{
    for (int j = threadIdx.x; j < 32; j += blockDim.x) {
        const ff v = ff_from_double(exp2((double)j / 32.0));
        tab[j] = make_float2(v.hi, v.lo);
    }
}

// e^t in double-float (relative error ~1e-12 for |t| < 80, the caller's
// range), table-driven:
// t = k ln2/32 + r with k = rint(32 t / ln2), |r| <= ln2/64; e^t =
// 2^(k div 32) 2^((k mod 32)/32) e^r, e^r = 1 + r + q with the tail
// q = r^2 (1/2 + r/6 + r^2/24 + r^3/120) in FP32 (|q| < 6e-5, so its FP32
// rounding is below 1e-11 of the result).  ln2/32 is split into a 24-bit
// head and a tail so that k * head is exact through two_prod.
// k = rint(32 t / ln2) is taken by adding 1.5 2^23 (the FP32 sum then holds k
// in its low mantissa bits, rounded to nearest even, for |k| < 2^22), which
// needs no float-to-integer conversion.
__device__ __forceinline__ ff ff_exp(ff t, const float2* tab)
{
    const float C_hi = 0x1.62e43p-6f, C_lo = -0x1.05c61p-34f;  // ln2/32
    const float kr = __fmaf_rn(t.hi, 46.166241308446828f, 0x1.8p23f);  // 32/ln2
    const int k = __float_as_int(kr) - 0x4B400000;
    const float kf = __fsub_rn(kr, 0x1.8p23f);
    ff kc = two_prod(kf, C_hi);
    kc.lo = __fmaf_rn(kf, C_lo, kc.lo);
    const ff r = ff_sub(t, kc);
    const float x = r.hi;
    const float q = __fmul_rn(
        __fmul_rn(x, x),
        __fmaf_rn(x, __fmaf_rn(x, __fmaf_rn(x, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f), 0.5f));
    ff s = two_sum(x, q);
    s.lo = __fadd_rn(s.lo, r.lo);
    ff e = two_sum(1.0f, s.hi);
    e.lo = __fadd_rn(e.lo, s.lo);
    e = fast_two_sum(e.hi, e.lo);
    const float2 tv = tab[k & 31];
    ff res = ff_mul(ff{tv.x, tv.y}, e);
    // 2^(k div 32) as an exact power of two (|t| < 80 keeps it normal)
    const float sc = __int_as_float(((k >> 5) + 127) << 23);
    return ff{__fmul_rn(res.hi, sc), __fmul_rn(res.lo, sc)};
}

// ---------------------------------------------------------------------------
// e^{-x} in FP64 without the FP64 pipe.  That pipe issues 2 lanes per cycle and
// SM here (0.62 T instructions/s), the integer units 64, and the FP64 kernels
// are bound by it, so the exponential is evaluated in 64-bit fixed point on the
// integer units.  Table-driven after P. T. P. Tang ("Table-driven
// implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15, 1989): with a = -x in units of 2^-56 (|a| < 128),
//   a = k ln2/1024 + r, 0 <= r < ln2/1024 (k floored from the top bits of a;
//   r in units of 2^-66, ln2/1024 to 98 bits),
//   e^a = 2^(k div 1024) T (1 + p),  T = 2^((k mod 1024)/1024) to 63 bits,
//   p = r + r^2/2 + r^3 (1/6 + r/24)   (remainder r^5/120 < 2^-59),
// the product rounded once, to nearest, into the result's mantissa: within
// 0.65 ulp of e^a (the rounding 0.5, the truncation of a to 2^-56 up to 0.125 just
// below a power of two, the series' remainder 0.016, the truncations of p and T
// 0.004; largest seen 0.622, 0.51 away from x = 0), against ~1.1 ulp of the form on
// FP64 instructions with a 64-entry table that it replaced.  About 55 integer
// instructions and no FP64 ones, where that form took 10 of the 18 FP64
// instructions of a leapfrog step's site.  |x| >= 128, NaN, and the few arguments
// in a million whose floor or last carry is ambiguous take CUDA's exp.
// The table is the products of two 32-entry ones, 2^(i/32) and 2^(j/1024) in
// units of 2^-63 (rounded from 60 decimal digits).
// ---------------------------------------------------------------------------
constexpr int kExpN = 1024;
typedef unsigned long long u64;
static __constant__ u64 kExpHi[32] = {
    0x8000000000000000ull, 0x82cd8698ac2ba1d7ull, 0x85aac367cc487b15ull, 0x88980e8092da8527ull,
    0x8b95c1e3ea8bd6e7ull, 0x8ea4398b45cd53c0ull, 0x91c3d373ab11c336ull, 0x94f4efa8fef70961ull,
    0x9837f0518db8a96full, 0x9b8d39b9d54e5539ull, 0x9ef5326091a111aeull, 0xa27043030c496819ull,
    0xa5fed6a9b15138eaull, 0xa9a15ab4ea7c0ef8ull, 0xad583eea42a14ac6ull, 0xb123f581d2ac2590ull,
    0xb504f333f9de6484ull, 0xb8fbaf4762fb9ee9ull, 0xbd08a39f580c36bfull, 0xc12c4cca66709456ull,
    0xc5672a115506daddull, 0xc9b9bd866e2f27a3ull, 0xce248c151f8480e4ull, 0xd2a81d91f12ae45aull,
    0xd744fccad69d6af4ull, 0xdbfbb797daf23755ull, 0xe0ccdeec2a94e111ull, 0xe5b906e77c8348a8ull,
    0xeac0c6e7dd24392full, 0xefe4b99bdcdaf5cbull, 0xf5257d152486cc2cull, 0xfa83b2db722a033aull,
};
static __constant__ u64 kExpLo[32] = {
    0x8000000000000000ull, 0x8016302f17467628ull, 0x802c6436d0e04f51ull, 0x80429c17d77c18edull,
    0x8058d7d2d5e5f6b1ull, 0x806f17687707a7b0ull, 0x80855ad965e88b84ull, 0x809ba2264dada76aull,
    0x80b1ed4fd999ab6cull, 0x80c83c56b50cf780ull, 0x80de8f3b8b85a0afull, 0x80f4e5ff089f763full,
    0x810b40a1d81406d4ull, 0x81219f24a5baa59dull, 0x813801881d886f7cull, 0x814e67cceb90502dull,
    0x8164d1f3bc030773ull, 0x817b3ffd3b2f2e47ull, 0x8191b1ea15813bfdull, 0x81a827baf7838b78ull,
    0x81bea1708dde6056ull, 0x81d51f0b8557ec1dull, 0x81eba08c8ad45370ull, 0x820225f44b55b33cull,
    0x8218af4373fc25ecull, 0x822f3c7ab205c89bull, 0x8245cd9ab2cec048ull, 0x825c62a423d13f0cull,
    0x8272fb97b2a5894cull, 0x828998760d01faf3ull, 0x82a0393fe0bb0ca8ull, 0x82b6ddf5dbc35907ull,
};
// Fill tab[kExpN] (shared memory, the whole block; the caller synchronises).
__device__ __forceinline__ void exp_table(u64* tab)
{
    for (int i = threadIdx.x; i < kExpN; i += blockDim.x) {
        const u64 a = kExpHi[i >> 5], b = kExpLo[i & 31];
        const u64 hi = __umul64hi(a, b), lo = a * b;
        tab[i] = (hi << 1) + (lo >> 63) + ((lo >> 62) & 1);  // the product in units of 2^-63, rounded
    }
}
// The two small tables alone, for launches too short to be worth kExpN products:
// exp_neg<.., .., true> multiplies their entries at each evaluation.
__device__ __forceinline__ void exp_table_small(u64* tab)
{
    for (int i = threadIdx.x; i < 64; i += blockDim.x) tab[i] = i < 32 ? kExpHi[i] : kExpLo[i - 32];
}
static __device__ __noinline__ double exp_slow(double a) { return exp(a); }
// e^{-x / 2^SH} / 2^HALF (SH, HALF = 0 or 1; both halvings are exact)
template <int SH = 0, int HALF = 0, bool SMALL = false>
__device__ __forceinline__ double exp_neg(double x, const u64* tab)
{
    const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
    // |a| = M 2^(6 - sh - 62), M the 53-bit significand at bit 62
    const int sh = 1029 + SH - (int)((xh >> 20) & 0x7ffu);  // < 0: |a| >= 128, inf, NaN
    const u64 M = (((u64)((xh & 0xfffffu) | 0x100000u) << 32) | xl) << 10;
    const unsigned s63 = (unsigned)sh < 63u ? (unsigned)sh : 63u;
    const u64 m56 = M >> s63;
    const u64 A = (int)xh < 0 ? m56 : 0ull - m56;  // a in units of 2^-56
    // k = floor(a 1024/ln2) from the top 32 bits of a and 1024/ln2 in units of 2^-20
    const int k = __mulhi((int)(A >> 32), 0x5c551d94) >> 12;
    // ln2/1024 = (0xb17217f7d1cf7a - 0x54361c4c 2^-32) 2^-66
    const u64 R = (A << 10) - (u64)((long long)k * 0xb17217f7d1cf7aLL) +
                  (u64)(long long)__mulhi(k, 0x54361c4c);
    const unsigned rr = (unsigned)(R >> 24);  // r in units of 2^-42
    const u64 r2 = (u64)rr * rr;              // r^2 in units of 2^-84
    const unsigned c = __umulhi((unsigned)(r2 >> 32), rr);         // r^3, 2^-62
    const unsigned w = __umulhi(rr, 174763u) + 0x2aaaaaabu;        // 1/6 + r/24, 2^-32
    const u64 P = R + (r2 >> 19) + (__umulhi(rr, (unsigned)R << 8) >> 18) +
                  ((u64)__umulhi(c, w) << 4);                      // p, 2^-66
    u64 T;
    if (SMALL) {
        const u64 a = tab[(k >> 5) & 31], b = tab[32 + (k & 31)];
        const u64 hi = __umul64hi(a, b), lo = a * b;
        T = (hi << 1) + (lo >> 63) + ((lo >> 62) & 1);
    } else {
        T = tab[k & (kExpN - 1)];
    }
    const unsigned Th = (unsigned)(T >> 32), Tl = (unsigned)T;
    const unsigned Ph = (unsigned)(P >> 32), Pl = (unsigned)P;
    const u64 tp = (u64)Th * Ph + __umulhi(Th, Pl) + __umulhi(Tl, Ph);  // T p, 2^-65
    const u64 m = T + (tp >> 2);
    // a negative r, a carry out of m (bit 63 is set otherwise) or |a| >= 128
    if (((int)(R >> 32) | (int)~(unsigned)(m >> 32) | sh) < 0)
        return (HALF ? 0.5 : 1.0) * exp_slow(SH ? -0.5 * x : -x);
    const u64 v = (m >> 11) + ((m >> 10) & 1);
    return __longlong_as_double((long long)(v + ((u64)(unsigned)((k >> 10) + 1022 - HALF) << 52)));
}

// ---------------------------------------------------------------------------
// Reductions in a fixed order (deterministic): xor-butterfly inside a warp,
// then warp 0 over the per-warp values in warp order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ ff warp_sum_ff(ff v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ff w;
        w.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
        w.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
        v = ff_add(v, w);
    }
    return v;
}
// Block sum; `red` needs blockDim.x/32 doubles.  Result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (warp == 0) {
        for (int i = lane; i < nw; i += 32) s += red[i];
        s = warp_sum(s);
    }
    return s;
}

// A sum of FP64 terms that does not depend on their order, so that a series'
// dH is the same bits whatever block shape or tiles its sites are spread over:
// terms below 2^8 rounded to a multiple of 2^-50 (their own rounding is as coarse
// from 4 on) and added as 64-bit integers per thread (fix_term), larger ones cut
// to a multiple of 2^-64 and added, as the threads' sums are, in 128 bits.  Terms
// of 2^28 or more, infinities and NaN go to an FP64 sum beside it (|S| < 2^63 for
// 2^35 terms below that), whose order is that of the shape.  Integer work on a few
// terms a trajectory: 2^20 sites, 100 steps 1474 -> 1482 us, 4 steps 227 -> 231;
// T = 2000, 50 steps as before (49.7).
struct FixSum {
    unsigned long long lo;
    long long hi;
    double big;
};
__device__ __forceinline__ void fix_merge(FixSum& s, unsigned long long lo, long long hi, double big)
{
    s.lo += lo;
    s.hi += hi + (long long)(s.lo < lo);
    if (big != 0.0) s.big += big;  // (an FP64 addition waits on its pipe; almost never needed)
}
// A term of 2^8 or more (out of line: rare, and 28 of them a thread otherwise).
static __device__ __noinline__ FixSum fix_large(FixSum s, double v)
{
    const unsigned h = (unsigned)__double2hiint(v), E = (h >> 20) & 0x7ffu;
    if (E >= 1051u) {
        s.big += v;
        return s;
    }
    const unsigned long long M = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32) |
                                 (unsigned)__double2loint(v);
    const int sh = (int)E - 1011;  // |v| 2^64 = M 2^sh, 20 <= sh < 40
    unsigned long long lo = M << sh;
    long long hi = (long long)(M >> (64 - sh));
    if ((int)h < 0) {
        lo = 0ull - lo;
        hi = ~hi + (long long)(lo == 0ull);
    }
    s.lo += lo;
    s.hi += hi + (long long)(s.lo < lo);
    return s;
}
// +v (or -v) into a thread's sum t (units of 2^-50, up to 32 terms) or, if large, s.
__device__ __forceinline__ void fix_term(FixSum& s, long long& t, double v, bool minus)
{
    const int h = __double2hiint(v);
    if ((h & 0x7fffffff) < 0x40700000) {  // |v| < 2^8
        const long long q = __double2ll_rn(__hiloint2double(h + (50 << 20), __double2loint(v)));
        t += minus ? -q : q;
    } else {
        s = fix_large(s, minus ? -v : v);
    }
}
__device__ __forceinline__ FixSum fix_warp_sum(FixSum s)
{
    if (__any_sync(0xffffffffu, s.big != 0.0)) s.big = warp_sum(s.big);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long lo = __shfl_xor_sync(0xffffffffu, s.lo, o);
        const long long hi = __shfl_xor_sync(0xffffffffu, s.hi, o);
        fix_merge(s, lo, hi, 0.0);
    }
    return s;
}
__device__ __forceinline__ double fix_to_double(const FixSum& s)
{
    const bool neg = s.hi < 0;
    const unsigned long long lo = neg ? 0ull - s.lo : s.lo;
    const long long hi = neg ? ~s.hi + (long long)(lo == 0ull) : s.hi;
    const double d = fma((double)lo, 0x1p-64, (double)hi);
    return (neg ? -d : d) + s.big;
}

// Block sums of N values (blockDim.x = NT threads, NT / 32 >= N warps): warp i
// adds value i over the threads, lane l those of l, l + 32, ... in order, then
// a butterfly (a butterfly per warp and value first would take five of the FP64
// pipe's instructions for each one that this takes).  tot[i] is valid in every
// thread after the call.
template <int N, int NT>
__device__ __forceinline__ void block_sum_many(const double (&v)[N], double (*buf)[NT], double* tot)
{
    static_assert(NT / 32 >= N, "one warp per value");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) buf[i][threadIdx.x] = v[i];
    __syncthreads();
    if (warp < N) {
        double s = buf[warp][lane];
#pragma unroll
        for (int k = 1; k < NT / 32; ++k) s += buf[warp][lane + 32 * k];
        s = warp_sum(s);
        if (lane == 0) tot[warp] = s;
    }
    __syncthreads();
}

// Theta as stored on the device: (phi, mu, xi, sigma_eta^2, sigma_u^2), and
// the leverage rho = corr(eps_t, eta_t) of the RSV model with leverage (a
// context setting, not stored with theta; 0 is the model of eqs. (1)-(3)).
struct ThetaD {
    double phi, mu, xi, se2, su2;
    double rho = 0.0;
};
__device__ __forceinline__ ThetaD load_theta(const double* th, double rho = 0.0)
{
    return {th[0], th[1], th[2], th[3], th[4], rho};
}

}  // namespace rsv
