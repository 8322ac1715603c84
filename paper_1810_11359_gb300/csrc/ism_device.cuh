// ism_device.cuh -- device helpers shared by the libism kernels.
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

#include "ism_internal.h"

// ---------------------------------------------------------------------------
// Job lookup: the kernels of a launch set enumerate their CTAs across the
// jobs of the table; job j owns CTAs [base_j, base_{j+1}).  Bases never
// decrease; a job without CTAs of a kind shares its base with the next one,
// so the owner is the last job whose base is <= cta (binary search).
// ---------------------------------------------------------------------------
template <typename F>
__device__ __forceinline__ int ism_find_job(const JobTable& t, long long cta, F base_of)
{
    int lo = 0, hi = t.n_jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (base_of(t.j[mid]) <= cta) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// A kernel's dynamic shared-memory limit is process-wide, so a limit set to
// each launch's own need could be lowered by another host thread launching
// the same kernel between this thread's set and its launch (which would then
// fail).  Instead the limit is raised once per device to the device's opt-in
// maximum less the kernel's static shared memory; `done` holds one bit per
// device (one flag per kernel).
inline int ism_open_smem(const void* kernel, std::atomic<unsigned long long>* done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done->load(std::memory_order_acquire) & bit) return 0;
    int mx = 0;
    if ((e = cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return (int)e;
    cudaFuncAttributes fa{};
    if ((e = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return (int)e;   // static + dynamic <= opt-in
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  mx - (int)fa.sharedSizeBytes)) != cudaSuccess)
        return (int)e;
    done->fetch_or(bit, std::memory_order_release);
    return 0;
}

// Reflection coefficient w of a job: from device memory when the caller keeps
// the coefficients there, else from the job table.
__device__ __forceinline__ float ism_job_beta(const JobDev& J, int w) { return J.beta_dev ? J.beta_dev[w] : J.beta[w]; }

// g2 = 6 log2(10) / (f_s T60), the log2 of the power decay per sample of the
// diffuse tail (eq. (7)-(8)).  For coefficients in device memory T60 comes
// from the Sabine formula evaluated here with the host's FP64 operations in
// the host's order, each rounded on its own (no contraction), so the value is
// bitwise the one the host computes from the same coefficients.
__device__ __forceinline__ double ism_job_g2_fp64(const JobDev& J)
{
    const double L0 = J.L[0], L1 = J.L[1], L2 = J.L[2];
    const double S[6] = {__dmul_rn(L1, L2), __dmul_rn(L1, L2), __dmul_rn(L0, L2),
                         __dmul_rn(L0, L2), __dmul_rn(L0, L1), __dmul_rn(L0, L1)};
    double den = 0.0;
    for (int i = 0; i < 6; ++i) {
        const double b = (double)J.beta_dev[i];
        den = __dadd_rn(den, __dmul_rn(S[i], __dsub_rn(1.0, __dmul_rn(b, b))));
    }
    if (!(den > 0.0)) return 0.0;
    const double T60 = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(0.161, L0), L1), L2), den);
    if (!(T60 < 1.0e300)) return 0.0;
    return __ddiv_rn(J.g2_c, __dmul_rn((double)J.fs, T60));
}

// ---------------------------------------------------------------------------
// Float-float (unevaluated sum hi + lo) arithmetic on correctly rounded FP32
// operations (Dekker / Knuth two-sum).  Intrinsics keep the compiler from
// contracting or reordering the error terms.
// ---------------------------------------------------------------------------
struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    float s = __fadd_rn(a.hi, b.hi);
    float bb = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    float hi = __fadd_rn(s, e);
    float lo = __fsub_rn(e, __fsub_rn(hi, s));
    return {hi, lo};
}

// g2 of the job as a float-float pair (hi + lo is its FP64 value to ~2^-48).
__device__ __forceinline__ ff ism_job_g2(const JobDev& J)
{
    if (!J.beta_dev) return {J.g2, J.g2_lo};
    const double g = ism_job_g2_fp64(J);
    const float hi = (float)g;
    return {hi, (float)(g - (double)hi)};
}

// 2^(-g i) for a float-float rate g >= 0 and an integer 0 <= i < 2^24: the
// product x = g i keeps its rounding error (one FMA) and the low part of g,
// x is split into its nearest integer n and a remainder r in [-1/2, 1/2]
// (p - n is exact: Sterbenz), and 2^-x = 2^-n 2^-r.  The result carries
// exp2f's own error (2 ulp) and nothing from the size of x.
__device__ __forceinline__ float ism_exp2_neg(ff g, int i)
{
    const float fi = (float)i;
    const float p = __fmul_rn(g.hi, fi);
    if (!(p < 256.0f)) return 0.0f;   // below 2^-255: zero in FP32 (also catches an infinite rate)
    const float pe = __fmaf_rn(g.lo, fi, __fmaf_rn(g.hi, fi, -p));
    const float t = __fadd_rn(p, 12582912.0f);   // 1.5 2^23 + n, its bits hold n
    const float r = __fadd_rn(__fsub_rn(p, __fsub_rn(t, 12582912.0f)), pe);
    const int n = __float_as_int(t) - 0x4B400000;
    const float e = exp2f(-r);
    return n <= 125 ? __int_as_float(__float_as_int(e) - (n << 23)) : ldexpf(e, -n);
}

// Approximate reciprocal and reciprocal square root on the special-function
// unit (max error ~1-2 ulp).
__device__ __forceinline__ float ism_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float ism_rsqrt(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// sqrt of a positive float-float: r = a.hi / sqrt(a.hi) from the approximate
// reciprocal root, then one Newton correction from the exact residual
// a - r^2 (FMA) of the full float-float value: lo = (a - r^2) / (2 r).  The
// pair r + lo is accurate to ~2^-44 relative although r itself is not
// correctly rounded.
__device__ __forceinline__ ff ff_sqrt(ff a)
{
    float rs = ism_rsqrt(a.hi);
    float r = __fmul_rn(a.hi, rs);
    float res = __fadd_rn(__fmaf_rn(-r, r, a.hi), a.lo);
    float lo = __fmul_rn(__fmul_rn(res, 0.5f), rs);
    return {r, lo};
}

// Integer value of a float that holds an integer in [-2^22, 2^22): adding
// 1.5 * 2^23 moves it to the low mantissa bits (no rounding happens, the
// value being integral), avoiding a conversion instruction.
__device__ __forceinline__ int ism_int_of_integral(float b)
{
    return __float_as_int(__fadd_rn(b, 12582912.0f)) - 0x4B400000;
}

// Nearest integer of x for |x| < 2^22 (ties to even), same trick.
__device__ __forceinline__ int ism_round_int(float x)
{
    return __float_as_int(__fadd_rn(x, 12582912.0f)) - 0x4B400000;
}

// sin(pi f) for f in [0, 1]: g = min(f, 1 - f) in [0, 1/2] (1 - f is exact
// for f >= 1/2) and the Taylor series of sin(pi g) through (pi g)^11, whose
// remainder is below (pi/2)^13 / 13! = 5.7e-8 on [0, 1/2].
__device__ __forceinline__ float ism_sinpi01(float f)
{
    const double PI = 3.141592653589793238462643383279502884;
    const float c1 = (float)PI;
    const float c3 = (float)(-PI * PI * PI / 6.0);
    const float c5 = (float)(PI * PI * PI * PI * PI / 120.0);
    const float c7 = (float)(-PI * PI * PI * PI * PI * PI * PI / 5040.0);
    const float c9 = (float)(PI * PI * PI * PI * PI * PI * PI * PI * PI / 362880.0);
    const float c11 = (float)(-PI * PI * PI * PI * PI * PI * PI * PI * PI * PI * PI / 39916800.0);
    float g = fminf(f, __fsub_rn(1.0f, f));
    float g2 = g * g;
    float p = fmaf(g2, c11, c9);
    p = fmaf(g2, p, c7);
    p = fmaf(g2, p, c5);
    p = fmaf(g2, p, c3);
    p = fmaf(g2, p, c1);
    return p * g;
}

// cos(a), sin(a) for |a| <= pi/8 by their Taylor series through a^8 and a^9
// (remainders below a^10/10! = 2.5e-11 and a^11/11! = 7e-13).
__device__ __forceinline__ void ism_sincos_small(float a, float* s, float* c)
{
    float a2 = a * a;
    float pc = fmaf(a2, 1.0f / 40320.0f, -1.0f / 720.0f);
    pc = fmaf(a2, pc, 1.0f / 24.0f);
    pc = fmaf(a2, pc, -0.5f);
    *c = fmaf(a2, pc, 1.0f);
    float ps = fmaf(a2, 1.0f / 362880.0f, -1.0f / 5040.0f);
    ps = fmaf(a2, ps, 1.0f / 120.0f);
    ps = fmaf(a2, ps, -1.0f / 6.0f);
    *s = fmaf(a2 * a, ps, a);
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds, each two
// 32x32 -> 64-bit products of counter words 0 and 2 with M0, M1, mixed with
// words 1, 3 and the key; the key is bumped by the Weyl constants W0, W1
// between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 ism_philox(uint4 c, uint32_t k0, uint32_t k1)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        uint4 n;
        n.x = hi1 ^ c.y ^ k0;
        n.y = lo1;
        n.z = hi0 ^ c.w ^ k1;
        n.w = lo0;
        c = n;
        k0 += W0;
        k1 += W1;
    }
    return c;
}

// The FP32 noise transform, one correctly rounded operation at a time, in
// the order of its written specification (uniform, ratio, ln, scale):
//   u = ((x >> 9) + 1/2) 2^-23                      exact in FP32
//   r = u / (1 - u)                                 (1 - u exact)
//   ln r: r = m 2^e, m in (sqrt(1/2), sqrt(2)]; t = (m - 1)/(m + 1);
//         ln m = 2t + t^3 (2/3 + t^2 (2/5 + t^2 (2/7 + t^2 (2/9 + t^2 2/11))))
//         ln r = e ln2_hi + (e ln2_lo + ln m)
//   z = (sqrt(3)/pi) ln r                           unit-variance logistic
// Two FP32 values in one 64-bit register pair, and the packed FP32 operations of
// sm_100-class GPUs on them (both halves rounded as the scalar operations are).
__device__ __forceinline__ unsigned long long pk_pack(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void pk_unpack(unsigned long long r, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long pk_fma(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long pk_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long pk_add(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long pk_all(float a) { return pk_pack(a, a); }

// -(a / b), correctly rounded, for quotients far from the ends of the FP32 range:
// Markstein's sequence (IBM J. Res. Dev. 34, 1990) -- a reciprocal refined once, the
// quotient and its exact remainder by FMAs -- with every sign turned, so that no
// negation is an instruction.  Checked against / for every argument that the
// noise gives it (all 2^23 uniforms, in either half: test_noise_all_uniforms_gpu.py).
__device__ __forceinline__ unsigned long long pk_neg_div(unsigned long long a, unsigned long long b)
{
    float b0, b1;
    pk_unpack(b, b0, b1);
    unsigned long long ny = pk_pack(ism_rcp(-b0), ism_rcp(-b1));   // -1 / b, one ulp
    ny = pk_fma(ny, pk_fma(b, ny, pk_all(1.0f)), ny);
    const unsigned long long nq = pk_mul(a, ny);
    return pk_fma(pk_fma(b, nq, a), ny, nq);
}

// The transform of two words: its operations in its order, each rounded on its own, two
// at a time.  (The uniform and the exponents come from additions to 2^23 and
// 1.5 2^23 whose results are exact, not from the conversion unit.)  Tail of 512 RIRs of
// 43,200 samples: 72 us one at a time with the compiler's division, two at a time so 55.
__device__ __forceinline__ float2 ism_logistic2(uint32_t x0, uint32_t x1)
{
    // u = (n + 1/2) 2^-23 = (2^23 + n) 2^-23 - (1 - 2^-24), n = x >> 9
    const unsigned long long f = pk_pack(__uint_as_float((x0 >> 9) | 0x4B000000u), __uint_as_float((x1 >> 9) | 0x4B000000u));
    const unsigned long long u = pk_fma(f, pk_all(0x1p-23f), pk_all(-(1.0f - 0x1p-24f)));
    float r0, r1;   // -u / (1 - u)
    pk_unpack(pk_neg_div(u, pk_fma(u, pk_all(-1.0f), pk_all(1.0f))), r0, r1);
    // |r| = m 2^e, m in (sqrt(1/2), sqrt(2)]: a carry out of the mantissa above that of sqrt(2)
    const uint32_t i0 = __float_as_uint(r0), i1 = __float_as_uint(r1);
    const uint32_t c0 = i0 + 0x4AFB0Cu, c1 = i1 + 0x4AFB0Cu;
    const unsigned long long m = pk_pack(__uint_as_float(i0 - (c0 & 0xFF800000u) + 0x3F800000u),
                                         __uint_as_float(i1 - (c1 & 0xFF800000u) + 0x3F800000u));
    // 1.5 2^23 + e (the shifted word is 256 + 127 + e), then -e
    const unsigned long long eb = pk_pack(__uint_as_float((c0 >> 23) + (0x4B400000u - 383u)),
                                          __uint_as_float((c1 >> 23) + (0x4B400000u - 383u)));
    const unsigned long long ne = pk_fma(eb, pk_all(-1.0f), pk_all(12582912.0f));
    const unsigned long long nt = pk_neg_div(pk_add(m, pk_all(-1.0f)), pk_add(m, pk_all(1.0f)));   // -(m - 1) / (m + 1)
    const unsigned long long t2 = pk_mul(nt, nt);
    unsigned long long p = pk_fma(t2, pk_all(2.0f / 11.0f), pk_all(2.0f / 9.0f));
    p = pk_fma(t2, p, pk_all(2.0f / 7.0f));
    p = pk_fma(t2, p, pk_all(2.0f / 5.0f));
    p = pk_fma(t2, p, pk_all(2.0f / 3.0f));
    const unsigned long long nln = pk_fma(pk_mul(nt, t2), p, pk_mul(pk_all(2.0f), nt));   // -ln m
    const unsigned long long nl =
        pk_fma(ne, pk_all(0.693145751953125f), pk_fma(ne, pk_all(1.428606765330187e-06f), nln));
    float z0, z1;
    pk_unpack(pk_mul(pk_all(-0.5513288974761963f), nl), z0, z1);
    return make_float2(z0, z1);
}

// Noise of sample k of RIR `rir`: word k mod 4 of Philox(counter (k/4, rir,
// 0, 0), key (seed lo, seed hi)).  Returns the four logistic values of the
// counter block k/4.
__device__ __forceinline__ float4 ism_noise_block(uint64_t seed, uint32_t rir, uint32_t blk)
{
    uint4 w = ism_philox(make_uint4(blk, rir, 0u, 0u), (uint32_t)seed, (uint32_t)(seed >> 32));
    const float2 a = ism_logistic2(w.x, w.y), b = ism_logistic2(w.z, w.w);
    return make_float4(a.x, a.y, b.x, b.y);
}
