// cls_device.cuh -- device side of the CLS random walk (paper Sec. 4, "Algorithm A").
//
// One history: sample the source (paper Sec. 4.3 for the box: y, z uniform on
// the x = 0 face, cosine-law direction; rod: x = 0 moving +x), sample the
// material label from p_0, then repeat: draw the collision distance
// l_c = -ln(1-u)/Sigma_m and the interface distance l_i = -Lambda_m ln(1-u),
// compute the boundary distance l_b, and take the smallest.  Boundary: leak
// through an x face (R or T) or reflect specularly on a lateral face.
// Collision: scatter isotropically with probability c_m, else absorb.
// Interface: switch the label.  Every flight is scored by the track-length
// estimator on the uniform x mesh.
//
// Ties: boundary wins over collision and interface, collision over interface;
// an x face wins over a lateral face; equal lateral distances reflect both.
// The collision draw is consumed even when Sigma_m = 0.
#pragma once

#include <atomic>
#include <type_traits>
#include <cstdint>
#include <cuda_runtime.h>

#include "cls_fixed.h"
#include "cls_internal.h"
#include "cls_intmath.h"

namespace cls {

#define CLS_FULL_MASK 0xffffffffu

// Blocks per SM of a kernel at a given dynamic shared memory.  The opt-in for
// more than 48 KB is set first: without it the occupancy query reports zero
// blocks for such sizes.
template <typename K>
__host__ cudaError_t occupancy_with_smem(int *blocks_per_sm, K kernel, int block, size_t smem) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, block, smem);
}

// The opt-in to 200 KB of dynamic shared memory, set once per device and
// kernel (`done` holds one bit per device index below 64, set after a
// successful call; two threads racing on it only repeat the call).
template <typename K>
__host__ cudaError_t ensure_smem_optin(K kernel, std::atomic<unsigned long long> &done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// ------------------------------------------------- FP64 logarithm, sine/cosine
// The FP64 walk takes its logarithms and its sine/cosine pairs straight from
// the 53-bit integer k of a draw (u = k 2^-53), in integer arithmetic
// (cls_intmath.h), through tables that every FP64 kernel copies into shared
// memory when it starts (load_math_tables): the FP64 pipe, the walk's
// bottleneck, sees neither.
__shared__ uint16_t cls_logn_tab[CLS_LOG_TABLE_N];
__shared__ __align__(16) uint64_t cls_logt_tab[CLS_LOG_TABLE_N][2];
__shared__ __align__(16) int64_t cls_sincos_tab[CLS_SINCOS_TABLE_N][2];

template <typename P>
__device__ __forceinline__ void load_math_tables(int tid, int nthreads) {
    if constexpr (sizeof(P) == 8) {
        for (int i = tid; i < CLS_LOG_TABLE_N; i += nthreads) {
            cls_logn_tab[i] = cls_log_n_init[i];
            cls_logt_tab[i][0] = cls_log_t_init[i][0];
            cls_logt_tab[i][1] = cls_log_t_init[i][1];
        }
        for (int i = tid; i < CLS_SINCOS_TABLE_N; i += nthreads) {
            cls_sincos_tab[i][0] = cls_sincos_q62_init[i][0];
            cls_sincos_tab[i][1] = cls_sincos_q62_init[i][1];
        }
    }
}

// -ln(1 - u) for u = k 2^-53, from the shared-memory tables
__device__ __forceinline__ double exp_variate_shared(unsigned long long k) {
    return exp_variate(k, IntLogTables{cls_logn_tab, cls_logt_tab});
}

// the integer E as a double, exactly (|E| < 2^51), by the 1.5 2^52 shift
__device__ __forceinline__ double small_int_to_double(long long e) {
    return __longlong_as_double(0x4338000000000000ll + e) - 0x1.8p52;
}

// ------------------------------------------------------------------ Philox
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64 multiplies mixed with the other two words and the round key; the
// key advances by the Weyl increments between rounds.  The round keys come
// precomputed (RoundKeys, cls_internal.h): all threads of a launch share them.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const RoundKeys &rk) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ rk.k[2 * r], lo1, hi0 ^ c.w ^ rk.k[2 * r + 1], lo0);
    }
    return c;
}

// The part of the counter (j/2, h_lo, h_hi, case) that a history's blocks share,
// as the first two rounds leave it: of their four products two depend on the
// history alone.  Round one is (x, y, z, w) = (hi(M1 h_hi) ^ h_lo ^ k0,
// lo(M1 h_hi), hi(M0 b) ^ case ^ k1, lo(M0 b)) for block b, and round two takes
// the product M0 x.  Two of a block's 20 wide products less (each takes a
// warp's multiplier for 4 cycles; all blocks together took 37% of the FP32 box
// kernel's time): the box L = 10 in FP32, 1e8 histories, 98.0 -> 95.1 ms.
struct HistoryKey {
    uint32_t x_hi, x_lo;  // M0 x
    uint32_t y;           // lo(M1 h_hi)
    uint32_t cid;         // the case
};

__device__ __forceinline__ HistoryKey history_key(uint64_t h, uint32_t cid, const RoundKeys &rk) {
    const uint32_t h_hi = (uint32_t)(h >> 32);
    const uint32_t x = __umulhi(0xCD9E8D57u, h_hi) ^ (uint32_t)h ^ rk.k[0];
    return HistoryKey{__umulhi(0xD2511F53u, x), 0xD2511F53u * x, 0xCD9E8D57u * h_hi, cid};
}

// The history's id (the multipliers' inverses modulo 2^32).
__device__ __forceinline__ uint64_t history_id(const HistoryKey &key, const RoundKeys &rk) {
    const uint32_t h_hi = 0x6d7cae67u * key.y;
    const uint32_t h_lo = (0x991a7cdbu * key.x_lo) ^ __umulhi(0xCD9E8D57u, h_hi) ^ rk.k[0];
    return ((uint64_t)h_hi << 32) | h_lo;
}

// philox4x32_10 of block b of a history
__device__ __forceinline__ uint4 philox_block(uint32_t b, const HistoryKey &key, const RoundKeys &rk) {
    const uint32_t z = __umulhi(0xD2511F53u, b) ^ key.cid ^ rk.k[1], w = 0xD2511F53u * b;  // round one
    uint4 c = make_uint4(__umulhi(0xCD9E8D57u, z) ^ key.y ^ rk.k[2], 0xCD9E8D57u * z, key.x_hi ^ w ^ rk.k[3], key.x_lo);
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ rk.k[2 * r], lo1, hi0 ^ c.w ^ rk.k[2 * r + 1], lo0);
    }
    return c;
}

// ------------------------------------------------------- precision traits
template <typename P>
struct Real;

// The parameters of a case that step reads, held in registers: the narrow walk,
// whose chain of events is serial, would wait for a load at every use.
template <typename P>
struct CaseRegs {
    P sigma0, sigma1, inv_sigma0, inv_sigma1, lambda0, lambda1, L, dx, inv_dx;
    unsigned long long c53_0, c53_1;
    uint32_t c24_0, c24_1;
    int d, nbins;
};


// FP64 walk: every quantity in double; shared-memory tally bins in fixed point.
// Comparisons of distances (non-negative after clamping) and sign tests run on
// the IEEE bit patterns in the integer pipes, which order non-negative doubles
// like the numbers they encode; the FP64 pipe is left to the arithmetic.
template <>
struct Real<double> {
    static __device__ __forceinline__ unsigned long long k53(uint32_t hi, uint32_t lo) {
        return (((unsigned long long)hi << 32) | (unsigned long long)lo) >> 11;
    }
    // m 2^e, exactly, for |m| < 2^53: the bit pattern is assembled in the
    // integer pipes (leading-zero count, shift), keeping the conversion off
    // the FP64 pipe
    static __device__ __forceinline__ double scaled_int(long long m, int e) {
        const unsigned long long sgn = m < 0 ? (1ull << 63) : 0ull;
        const unsigned long long a = (unsigned long long)(m < 0 ? -m : m);
        const int p = 63 - __clzll((long long)(a | 1ull));  // leading bit
        const unsigned long long bits =
            sgn | ((unsigned long long)(p + e + 1023) << 52) | ((a << (52 - p)) & 0xFFFFFFFFFFFFFull);
        return a == 0ull ? 0.0 : __longlong_as_double((long long)bits);
    }
    // 53-bit uniform u = k 2^-53 in [0, 1) from the (hi, lo) output words
    static __device__ __forceinline__ double uniform(uint32_t hi, uint32_t lo) {
        return scaled_int((long long)k53(hi, lo), -53);
    }
    // 2u - 1 = (k - 2^52) 2^-52, exactly
    static __device__ __forceinline__ double two_u_minus_one(uint32_t hi, uint32_t lo) {
        return scaled_int((long long)k53(hi, lo) - (1ll << 52), -52);
    }
    // sqrt(u) = sqrt(2k 2^-54), in integer arithmetic
    static __device__ __forceinline__ double sqrt_uniform(uint32_t hi, uint32_t lo) {
        return sqrt_int(U128{k53(hi, lo) << 1, 0ull}, 54);
    }
    // A new direction from the draws u of mu and v of phi = 2 pi v: cosine law
    // mu = sqrt(u), st = sqrt(1 - u); isotropic mu = 2u - 1, st = sqrt(4 u (1 -
    // u)), with 1 - u and 4 u (1 - u) exact integers; a = st cos phi, b = st sin
    // phi multiplied in integers before their one rounding (an FP64 product
    // costs 64 cycles of its warp, an integer one 16).
    static __device__ __forceinline__ void direction(uint32_t hi, uint32_t lo, uint32_t phi_hi, uint32_t phi_lo,
                                                     bool cosine, double *mu, double *a, double *b) {
        const unsigned long long k = k53(hi, lo), n = (1ull << 53) - k;
        // sqrt(u) (the cosine law only: a lane starts the loop at t = 1
        // otherwise), then st, through one copy of sqrt_q61
        const U128 x1 = cosine ? U128{n << 1, 0ull} : U128{(k * n) << 2, (umulhi64(k, n) << 2) | ((k * n) >> 62)};
        const int s1 = cosine ? 54 : 106;
        U128 x = cosine ? U128{k << 1, 0ull} : x1;
        int scale = s1, e0 = 0, e1 = 0;
        uint64_t q0 = 0, q1 = 0;
#pragma unroll 1
        for (int t = cosine ? 0 : 1; t < 2; ++t) {
            q0 = q1;
            e0 = e1;
            q1 = sqrt_q61(x, scale, &e1);
            x = x1;
            scale = s1;
        }
        *mu = cosine ? fixed_to_double((int64_t)q0, e0 - 61) : two_u_minus_one(hi, lo);
        int64_t sn, cs;
        sincos_2pi_q62(k53(phi_hi, phi_lo), cls_sincos_tab, &sn, &cs);
        int64_t v = cs;
        double r0 = 0.0, r1 = 0.0;
#pragma unroll 1
        for (int t = 0; t < 2; ++t) {
            r0 = r1;
            r1 = sqrt_times_q62(q1, e1, v);
            v = sn;
        }
        *a = r0;
        *b = r1;
    }
    // 1 - u, exactly: (2^53 - k) 2^-53
    static __device__ __forceinline__ double one_minus(uint32_t hi, uint32_t lo) {
        return (double)((1ull << 53) - k53(hi, lo)) * 0x1p-53;
    }
    // u < v for the threshold ceil(v 2^53)
    static __device__ __forceinline__ bool below(uint32_t hi, uint32_t lo, unsigned long long thr53, uint32_t) {
        return k53(hi, lo) < thr53;
    }
    static __device__ __forceinline__ double inf() { return __longlong_as_double(0x7ff0000000000000ll); }
    static __device__ __forceinline__ bool pos(double w) { return __double_as_longlong(w) > 0; }
    static __device__ __forceinline__ bool neg(double w) {
        const long long b = __double_as_longlong(w);
        return b < 0 && (b << 1) != 0;
    }
    // negative values and -0 become +0
    static __device__ __forceinline__ double nonneg(double x) { return __double_as_longlong(x) < 0 ? 0.0 : x; }
    static __device__ __forceinline__ bool le(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }
    static __device__ __forceinline__ bool lt(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
    static __device__ __forceinline__ bool eq(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }
    static __device__ __forceinline__ double sigma(const CaseParams &c, int m) { return c.sigma[m]; }
    static __device__ __forceinline__ double sigma(const CaseRegs<double> &c, int m) { return m == 0 ? c.sigma0 : c.sigma1; }
    static __device__ __forceinline__ unsigned long long thr_c53(const CaseParams &c, int m) { return c.thr_c53[m]; }
    static __device__ __forceinline__ uint32_t thr_c24(const CaseParams &c, int m) { return c.thr_c24[m]; }
    static __device__ __forceinline__ unsigned long long thr_c53(const CaseRegs<double> &c, int m) { return m == 0 ? c.c53_0 : c.c53_1; }
    static __device__ __forceinline__ uint32_t thr_c24(const CaseRegs<double> &c, int m) { return m == 0 ? c.c24_0 : c.c24_1; }
    static __device__ __forceinline__ double L(const CaseParams &c) { return c.L; }
    static __device__ __forceinline__ double L(const CaseRegs<double> &c) { return c.L; }
    static __device__ __forceinline__ double dx(const CaseParams &c) { return c.dx; }
    static __device__ __forceinline__ double dx(const CaseRegs<double> &c) { return c.dx; }
    static __device__ __forceinline__ double inv_dx(const CaseParams &c) { return c.inv_dx; }
    static __device__ __forceinline__ double inv_dx(const CaseRegs<double> &c) { return c.inv_dx; }
    static __device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
    // |x| and -x on the bit pattern (integer pipes)
    static __device__ __forceinline__ double abs(double x) {
        return __longlong_as_double(__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll);
    }
    static __device__ __forceinline__ double flip(double x) {
        return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
    }
    // min(floor(t), cap) for finite t >= 0, from the bit pattern
    static __device__ __forceinline__ int floor_index(double t, int cap) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(t);
        const int e = (int)(b >> 52) - 1023;
        const int sh = min(max(52 - e, 0), 63);
        const unsigned long long v = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) >> sh;
        return (int)min(v, (unsigned long long)cap);
    }
    // t - k for finite t >= 0 and k = floor_index(t, cap) <= floor(t): the bits
    // below the binary point, plus floor(t) - k (non-zero beyond the last
    // bin), re-assembled in the integer pipes
    static __device__ __forceinline__ double frac(double t, int k) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(t);
        const int e = (int)(b >> 52) - 1023;
        if (e > 30) return t - small_int_to_double(k);
        const int sh = 52 - max(e, 0);
        const unsigned long long M = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
        const unsigned long long m = (((M >> sh) - (unsigned long long)k) << sh) + (M & ((1ull << sh) - 1ull));
        return e < 0 ? t : scaled_int((long long)m, -sh);
    }
    static __device__ __forceinline__ double inv_sigma(const CaseParams &c, int m) { return c.inv_sigma[m]; }
    static __device__ __forceinline__ double inv_sigma(const CaseRegs<double> &c, int m) { return m == 0 ? c.inv_sigma0 : c.inv_sigma1; }
    static __device__ __forceinline__ double lambda(const CaseParams &c, int m) { return c.lambda[m]; }
    static __device__ __forceinline__ double lambda(const CaseRegs<double> &c, int m) { return m == 0 ? c.lambda0 : c.lambda1; }
    // -ln(1 - u) of two draws through one copy of the evaluation (the loop is
    // kept rolled: the instruction cache is one of the walk's limits)
    static __device__ __forceinline__ void exp_variates(uint32_t hi0, uint32_t lo0, uint32_t hi1, uint32_t lo1,
                                                        double *e0, double *e1) {
        unsigned long long ka = k53(hi0, lo0), kb = k53(hi1, lo1);
        double a = 0.0, b = 0.0;
#pragma unroll 1
        for (int t = 0; t < 2; ++t) {
            a = b;
            b = exp_variate_shared(ka);
            ka = kb;
        }
        *e0 = a;
        *e1 = b;
    }
    // 1/a in integer arithmetic (Newton-Raphson, cls_intmath.h)
    static __device__ __forceinline__ double recip(double a) { return recip_int(a); }
};

// FP32 tracking: position, direction and distances in float; the flights'
// deposits are summed exactly in a fixed-point difference array and the
// per-history statistics in FP64 (the tally regions below).
template <>
struct Real<float> {
    // the same draw truncated to its top 24 bits: u = k 2^-24
    static __device__ __forceinline__ float uniform(uint32_t hi, uint32_t) { return (float)(hi >> 8) * 0x1p-24f; }
    static __device__ __forceinline__ float two_u_minus_one(uint32_t hi, uint32_t lo) { return 2.0f * uniform(hi, lo) - 1.0f; }
    // FP32 tracking takes the hardware's approximate square root, reciprocal and
    // sine/cosine (a few FP32 ulps, below the FP32 walk's own rounding noise)
    static __device__ __forceinline__ float fast_sqrt(float x) {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ float sqrt_uniform(uint32_t hi, uint32_t lo) { return fast_sqrt(uniform(hi, lo)); }
    static __device__ __forceinline__ float one_minus(uint32_t hi, uint32_t) {
        return (float)((1u << 24) - (hi >> 8)) * 0x1p-24f;
    }
    static __device__ __forceinline__ bool below(uint32_t hi, uint32_t, unsigned long long, uint32_t thr24) {
        return (hi >> 8) < thr24;
    }
    static __device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }
    static __device__ __forceinline__ bool pos(float w) { return w > 0.0f; }
    static __device__ __forceinline__ bool neg(float w) { return w < 0.0f; }
    static __device__ __forceinline__ float nonneg(float x) { return x > 0.0f ? x : 0.0f; }
    static __device__ __forceinline__ bool le(float a, float b) { return a <= b; }
    static __device__ __forceinline__ bool lt(float a, float b) { return a < b; }
    static __device__ __forceinline__ bool eq(float a, float b) { return a == b; }
    static __device__ __forceinline__ float sigma(const CaseParams &c, int m) { return c.sigma_f[m]; }
    static __device__ __forceinline__ float sigma(const CaseRegs<float> &c, int m) { return m == 0 ? c.sigma0 : c.sigma1; }
    static __device__ __forceinline__ unsigned long long thr_c53(const CaseParams &c, int m) { return c.thr_c53[m]; }
    static __device__ __forceinline__ uint32_t thr_c24(const CaseParams &c, int m) { return c.thr_c24[m]; }
    static __device__ __forceinline__ unsigned long long thr_c53(const CaseRegs<float> &c, int m) { return m == 0 ? c.c53_0 : c.c53_1; }
    static __device__ __forceinline__ uint32_t thr_c24(const CaseRegs<float> &c, int m) { return m == 0 ? c.c24_0 : c.c24_1; }
    static __device__ __forceinline__ float L(const CaseParams &c) { return c.L_f; }
    static __device__ __forceinline__ float L(const CaseRegs<float> &c) { return c.L; }
    static __device__ __forceinline__ float dx(const CaseParams &c) { return c.dx_f; }
    static __device__ __forceinline__ float dx(const CaseRegs<float> &c) { return c.dx; }
    static __device__ __forceinline__ float inv_dx(const CaseParams &c) { return c.inv_dx_f; }
    static __device__ __forceinline__ float inv_dx(const CaseRegs<float> &c) { return c.inv_dx; }
    static __device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
    static __device__ __forceinline__ float abs(float x) { return fabsf(x); }
    static __device__ __forceinline__ float flip(float x) { return -x; }
    static __device__ __forceinline__ int floor_index(float t, int cap) { return min((int)t, cap); }
    static __device__ __forceinline__ float frac(float t, int k) { return t - (float)k; }
    static __device__ __forceinline__ float exp_variate(uint32_t hi, uint32_t lo) { return -__logf(one_minus(hi, lo)); }
    static __device__ __forceinline__ float inv_sigma(const CaseParams &c, int m) { return c.inv_sigma_f[m]; }
    static __device__ __forceinline__ float inv_sigma(const CaseRegs<float> &c, int m) { return m == 0 ? c.inv_sigma0 : c.inv_sigma1; }
    static __device__ __forceinline__ float lambda(const CaseParams &c, int m) { return c.lambda_f[m]; }
    static __device__ __forceinline__ float lambda(const CaseRegs<float> &c, int m) { return m == 0 ? c.lambda0 : c.lambda1; }
    static __device__ __forceinline__ void exp_variates(uint32_t hi0, uint32_t lo0, uint32_t hi1, uint32_t lo1, float *e0,
                                                        float *e1) {
        *e0 = -__logf(one_minus(hi0, lo0));
        *e1 = -__logf(one_minus(hi1, lo1));
    }
    static __device__ __forceinline__ float recip(float a) {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
        return r;
    }
    // (sin, cos)(2 pi u) = -(sin, cos)(2 pi (u - 1/2)), the argument in [-pi, pi)
    static __device__ __forceinline__ void direction(uint32_t hi, uint32_t lo, uint32_t phi_hi, uint32_t phi_lo,
                                                     bool cosine, float *mu, float *a, float *b) {
        *mu = cosine ? sqrt_uniform(hi, lo) : two_u_minus_one(hi, lo);
        const float st = fast_sqrt(1.0f - *mu * *mu);
        float sn, cs;
        __sincosf(6.28318530717958647692f * (uniform(phi_hi, phi_lo) - 0.5f), &sn, &cs);
        *a = st * -cs;
        *b = st * -sn;
    }
};

// ----------------------------------------------------------- history state
// The mesh coordinate of a history's position: its bin, and the fraction of the
// bin width with 64 bits (all ones at x = L).  Carried by the FP64 walk, where
// the end of a flight is the start of the next; the FP32 walk forms both anew.
template <typename P>
struct MeshPoint {};
template <>
struct MeshPoint<double> {
    uint32_t k;
    unsigned long long F;
};

template <typename P>
struct History {
    P r[3];
    P w[3];
    P iw[3];          // 1 / w (infinite when the component is 0); [1] and [2] in the FP64 narrow walk only
    int m;
    uint32_t j;       // per-history draw index
    uint32_t c2, c3;  // words 2, 3 of the last Philox block (odd draws)
    HistoryKey key;   // its Philox counter words
    uint32_t events, n_coll, n_int, n_refl;
    uint32_t pend;    // direction still to draw (DIR_*), 3D and extruded geometries
    P track0, track1; // per-history track length in material 0 / 1
    MeshPoint<P> at;  // where r[0] lies on the mesh (not in the narrow walk)
};

// A new direction of the 3D or extruded walk is drawn by resolve_direction,
// which the history tracker runs once per step for every lane that needs one:
// the lanes born this step and those that scattered in the last one share one
// pass through the sqrt, sine/cosine and reciprocal arithmetic.
enum : uint32_t { DIR_NONE = 0, DIR_SCATTER = 1, DIR_SOURCE_COSINE = 2, DIR_SOURCE_ISOTROPIC = 3 };

// One flight's contribution to the mesh: a0 into bin k0, a1 into bin k1
// (k1 > k0) and c into each interior bin k0 < k < k1.  Empty when k1 < k0.
template <typename P>
struct Flight {
    int k0, k1;
    P a0, a1, c;
};

// FP64 walk: the same in fixed point, units of 2^-fix_bits bin widths
// (cls_fixed.h), formed in integer arithmetic (plan_flight).  A flight that
// scores straight into the global bins (`real`) holds the bit patterns of the
// doubles instead, in the low words.
template <>
struct Flight<double> {
    int k0, k1;
    Fix96 a0, a1, c;
    bool real;
};

__device__ __forceinline__ double flight_real(const Fix96 &a) { return __hiloint2double((int)a.w1, (int)a.w0); }
__device__ __forceinline__ Fix96 flight_bits(double v) {
    return Fix96{(uint32_t)__double2loint(v), (uint32_t)__double2hiint(v), 0u};
}
__device__ __forceinline__ double flight_real(float a) { return (double)a; }

// whether the flight scores straight into the global bins (a lane whose region
// was handed to a newer key; FP64 also flights too long for the fixed point)
__device__ __forceinline__ bool scores_global(const Flight<float> &, int lreg) { return lreg == 2; }
__device__ __forceinline__ bool scores_global(const Flight<double> &f, int) { return f.real; }

// Output words (hi, lo) of draw j = s.j of the history; advances j.  Even
// draws compute a Philox block and keep its words 2, 3 for the odd draw.
template <typename P>
__device__ __forceinline__ void draw_words(History<P> &s, const RoundKeys &key, uint32_t &hi, uint32_t &lo) {
    if ((s.j & 1u) == 0u) {
        const uint4 o = philox_block(s.j >> 1, s.key, key);
        hi = o.x;
        lo = o.y;
        s.c2 = o.z;
        s.c3 = o.w;
    } else {
        hi = s.c2;
        lo = s.c3;
    }
    ++s.j;
}

// Output words of draws j and j + 1 (j = s.j); advances j by 2.  The pair
// always needs exactly one Philox block -- words (0,1), (2,3) of block j/2 for
// even j; the cached words of the last block and words (0,1) of block
// (j+1)/2 for odd j -- so a warp computes it once, whatever its lanes' parities.
template <typename P>
__device__ __forceinline__ void draw_pair(History<P> &s, const RoundKeys &key, uint32_t &hi0, uint32_t &lo0,
                                          uint32_t &hi1, uint32_t &lo1) {
    const bool odd = (s.j & 1u) != 0u;
    const uint4 o = philox_block((s.j + 1u) >> 1, s.key, key);
    hi0 = odd ? s.c2 : o.x;
    lo0 = odd ? s.c3 : o.y;
    hi1 = odd ? o.x : o.z;
    lo1 = odd ? o.y : o.w;
    s.c2 = o.z;  // read by draw j + 2 when it is odd
    s.c3 = o.w;
    s.j += 2u;
}

template <typename P>
__device__ __forceinline__ P draw(History<P> &s, const RoundKeys &key) {
    uint32_t hi, lo;
    draw_words(s, key, hi, lo);
    return Real<P>::uniform(hi, lo);
}

// 2u - 1 for the next draw u (isotropic direction cosine)
template <typename P>
__device__ __forceinline__ P draw_iso(History<P> &s, const RoundKeys &key) {
    uint32_t hi, lo;
    draw_words(s, key, hi, lo);
    return Real<P>::two_u_minus_one(hi, lo);
}

// whether the next draw is below the value whose thresholds are given
template <typename P>
__device__ __forceinline__ bool draw_below(History<P> &s, const RoundKeys &key, unsigned long long thr53, uint32_t thr24) {
    uint32_t hi, lo;
    draw_words(s, key, hi, lo);
    return Real<P>::below(hi, lo, thr53, thr24);
}


// Geometry of a case: G is a compile-time geometry code (1, 2, 3, 11, 13) for
// launches whose cases share one geometry, 0 to read it from the case.  A
// fixed G folds every geometry branch of the walk away.
template <int G, typename Case>
__device__ __forceinline__ int geometry(const Case &cp) {
    return G != 0 ? G : cp.d;
}

template <typename P>
__device__ __forceinline__ CaseRegs<P> load_case(const CaseParams &c) {
    using R = Real<P>;
    CaseRegs<P> r;
    r.sigma0 = R::sigma(c, 0);
    r.sigma1 = R::sigma(c, 1);
    r.inv_sigma0 = R::inv_sigma(c, 0);
    r.inv_sigma1 = R::inv_sigma(c, 1);
    r.lambda0 = R::lambda(c, 0);
    r.lambda1 = R::lambda(c, 1);
    r.L = R::L(c);
    r.dx = R::dx(c);
    r.inv_dx = R::inv_dx(c);
    r.c53_0 = c.thr_c53[0];
    r.c53_1 = c.thr_c53[1];
    r.c24_0 = c.thr_c24[0];
    r.c24_1 = c.thr_c24[1];
    r.d = c.d;
    r.nbins = c.nbins;
    return r;
}

template <typename P>
__device__ __forceinline__ P recip_or_inf(P w) {
    return Real<P>::is_zero(w) ? Real<P>::inf() : Real<P>::recip(w);
}

template <typename P>
__device__ __forceinline__ void set_direction(History<P> &s, P wx, P wy, P wz) {
    s.w[0] = wx;
    s.w[1] = wy;
    s.w[2] = wz;
    s.iw[0] = recip_or_inf(wx);
}

// Direction (wx, 0, 0) of the slab and the x-projected box
template <typename P>
__device__ __forceinline__ void set_direction_x(History<P> &s, P wx) {
    s.w[0] = wx;
    s.w[1] = P(0);
    s.w[2] = P(0);
    s.iw[0] = recip_or_inf(wx);
}

// Draw the pending direction of a 3D or extruded walk: mu, then the azimuth
// phi, then (at the source) the material label, in the order of the serial
// walk.  Cosine-law incidence (paper Sec. 4.3): mu = sqrt(xi) about +x,
// omega = (mu, st cos phi, st sin phi); isotropic (scattering, volume source):
// mu = 2 xi - 1, omega = (st cos phi, st sin phi, mu); st = sqrt(1 - mu^2).
template <typename P, int G = 0>
__device__ __forceinline__ void resolve_direction(History<P> &s, const CaseParams &cp, const RoundKeys &key) {
    if constexpr (G != 0 && G != 2 && G != 3) return;  // no pending directions in these geometries
    if (s.pend == DIR_NONE) return;
    const bool cosine = s.pend == DIR_SOURCE_COSINE;
    uint32_t hi, lo, phi_hi, phi_lo;
    draw_pair(s, key, hi, lo, phi_hi, phi_lo);  // mu, then phi
    P mu, a, b;
    Real<P>::direction(hi, lo, phi_hi, phi_lo, cosine, &mu, &a, &b);
    set_direction(s, cosine ? mu : a, cosine ? a : b, cosine ? b : mu);
    if (s.pend != DIR_SCATTER) s.m = draw_below(s, key, cp.thr_p053, cp.thr_p024) ? 0 : 1;
    s.pend = DIR_NONE;
}

template <typename Case>
__device__ __forceinline__ void set_mesh_point(History<double> &s, const Case &cp);
template <typename Case>
__device__ __forceinline__ void set_mesh_point(History<float> &s, const Case &cp);

// Source: position and direction first, then the material label.  With
// DEFER, a 3D or extruded source leaves its direction and label pending for
// the caller's resolve_direction.
template <typename P, int G = 0, bool DEFER = false>
__device__ __forceinline__ void source(History<P> &s, const CaseParams &cp, const RoundKeys &key, uint64_t h) {
    using R = Real<P>;
    const int gd = geometry<G>(cp);
    s.key = history_key(h, cp.case_id, key);
    s.j = 0;
    s.events = s.n_coll = s.n_int = s.n_refl = 0;
    s.pend = DIR_NONE;
    s.track0 = s.track1 = P(0);
    s.r[0] = P(0);
    s.r[1] = P(0);
    s.r[2] = P(0);
    if constexpr (sizeof(P) == 8) s.at = MeshPoint<P>{0u, 0ull};
    const P L = R::L(cp);
    if (gd == 3 || gd == 2) {
        if (cp.source == 1) {  // suite II: uniform position, isotropic direction
            s.r[0] = L * draw(s, key);
            set_mesh_point(s, cp);
        }
        if (gd == 3) {  // y, then z
            uint32_t yh, yl, zh, zl;
            draw_pair(s, key, yh, yl, zh, zl);
            s.r[1] = L * R::uniform(yh, yl);
            s.r[2] = L * R::uniform(zh, zl);
        } else {
            s.r[1] = L * draw(s, key);
        }
        s.pend = (cp.source == 1) ? DIR_SOURCE_ISOTROPIC : DIR_SOURCE_COSINE;
        if (!DEFER) resolve_direction<P, G>(s, cp, key);
        return;
    }
    if (cp.source == 1) {
        s.r[0] = L * draw(s, key);
        set_mesh_point(s, cp);
        if (gd == 11 || gd == 13) {
            set_direction_x(s, draw_iso(s, key));
        } else {
            uint32_t hi, lo;
            draw_words(s, key, hi, lo);
            const P w = (hi >> 31) == 0u ? P(1) : P(-1);  // u < 1/2
            s.w[0] = w;
            s.w[1] = P(0);
            s.w[2] = P(0);
            s.iw[0] = w;
        }
    } else if (gd == 11 || gd == 13) {
        uint32_t hi, lo;  // slab, projected box: mu = sqrt(xi)
        draw_words(s, key, hi, lo);
        set_direction_x(s, R::sqrt_uniform(hi, lo));
    } else {
        s.w[0] = P(1);
        s.w[1] = P(0);
        s.w[2] = P(0);
        s.iw[0] = P(1);
    }
    s.m = draw_below(s, key, cp.thr_p053, cp.thr_p024) ? 0 : 1;
}

// Trace sink (only instantiated by the trace kernel).
struct TraceSink {
    double *rows;
    int cap;
    int n;
};

template <typename P, bool TRACE>
__device__ __forceinline__ void trace_row(TraceSink *tr, int ev, const History<P> &s, double l) {
    if constexpr (TRACE) {
        if (tr->n < tr->cap) {
            double *row = tr->rows + 10 * (size_t)tr->n;
            row[0] = ev;
            row[1] = (double)s.j;
            row[2] = (double)s.r[0];
            row[3] = (double)s.r[1];
            row[4] = (double)s.r[2];
            row[5] = (double)s.w[0];
            row[6] = (double)s.w[1];
            row[7] = (double)s.w[2];
            row[8] = (double)s.m;
            row[9] = l;
        }
        tr->n++;
    }
}

// Track-length estimator: the flight x0 -> x1 (length l, direction cosine wx)
// scores in bin k the path length inside e_k <= x < e_k+1, the x-overlap times
// 1/|wx|; interior bins receive dx/|wx| each.  A flight inside one bin scores
// its length l itself, which stays exact for grazing flights (|wx| -> 0).  A
// flight with wx == 0 scores its whole length in the bin that contains x0.
template <typename P>
__device__ __forceinline__ void add_track(History<P> &s, P l, int m) {
    const P t = (m == 0 ? s.track0 : s.track1) + l;  // one add, the sum selected
    s.track0 = (m == 0) ? t : s.track0;
    s.track1 = (m == 0) ? s.track1 : t;
}

template <typename Case>
__device__ __forceinline__ void plan_flight(Flight<float> &f, const Case &cp, float x0, float x1, float l, float wx,
                                            float iwx, bool) {
    using R = Real<float>;
    f.k0 = 0;
    f.k1 = -1;
    if (!R::pos(l)) return;
    const int nb = cp.nbins;
    const float inv_dx = R::inv_dx(cp);
    // the x-extent clipped to [0, L]
    const float a = R::nonneg(x0), b = R::nonneg(x1);
    if (R::is_zero(wx)) {
        const int k = R::floor_index(a * inv_dx, nb - 1);
        f.k0 = f.k1 = k;
        f.a0 = l;
        return;
    }
    const float L = R::L(cp);
    const float lo = R::lt(a, b) ? a : b;
    float hi = R::lt(a, b) ? b : a;
    hi = R::lt(L, hi) ? L : hi;
    // bin coordinates x / dx: bin index = integer part; the end bins receive
    // (1 - frac) dx / |wx| and frac dx / |wx|
    const float ulo = lo * inv_dx, uhi = hi * inv_dx;
    const int k0 = R::floor_index(ulo, nb - 1);
    const int k1 = R::floor_index(uhi, nb - 1);
    f.k0 = k0;
    f.k1 = k1;
    if (k0 == k1) {  // the flight lies inside one bin: its length itself
        f.a0 = l;
        return;
    }
    const float c = R::dx(cp) * R::abs(iwx);
    f.a0 = R::nonneg(fmaf(-R::frac(ulo, k0), c, c));
    f.a1 = R::frac(uhi, k1) * c;
    f.c = c;
}

// The mesh coordinate of x, clipped to [0, L], from u = x / dx (below 2^12).
template <typename Case>
__device__ __forceinline__ MeshPoint<double> mesh_point(const Case &cp, double x) {
    using R = Real<double>;
    const double L = R::L(cp), c = R::nonneg(x);
    const double u = (R::lt(L, c) ? L : c) * R::inv_dx(cp);
    const unsigned long long b = (unsigned long long)__double_as_longlong(u);
    const int e = (int)(b >> 52) - 1023;
    const unsigned long long M = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    MeshPoint<double> p;
    p.k = e >= 0 ? (uint32_t)(M >> (52 - e)) : 0u;
    p.F = e >= -12 ? M << (12 + e) : M >> min(-12 - e, 63);
    const uint32_t last = (uint32_t)cp.nbins - 1u;
    if (p.k > last) {  // x = L: the whole of the last bin
        p.k = last;
        p.F = ~0ull;
    }
    return p;
}

// The flight in FP64, for the global bins: bit patterns of a0, a1 and c.
__device__ __forceinline__ void plan_flight_real(Flight<double> &f, double ulo, double uhi, double l, double c) {
    using R = Real<double>;
    f.real = true;
    if (f.k0 == f.k1) {
        f.a0 = flight_bits(l);
        return;
    }
    f.a0 = flight_bits(R::nonneg(fma(-R::frac(ulo, f.k0), c, c)));
    f.a1 = flight_bits(R::frac(uhi, f.k1) * c);
    f.c = flight_bits(c);
}

template <typename Case>
__device__ __forceinline__ void plan_flight(Flight<double> &f, const Case &cp, const MeshPoint<double> &from,
                                            const MeshPoint<double> &to, double x0, double x1, double l, double iwx,
                                            bool global) {
    using R = Real<double>;
    f.k0 = 0;
    f.k1 = -1;
    f.real = global;
    if (!R::pos(l)) return;
    const bool up = R::lt(R::nonneg(x0), R::nonneg(x1));
    const int k0 = (int)(up ? from.k : to.k), k1 = (int)(up ? to.k : from.k);
    f.k0 = k0;
    f.k1 = k1;
    // in bin widths: a flight inside one bin scores its length itself, else
    // 1/|wx| in a whole bin
    const double v = k0 == k1 ? l * R::inv_dx(cp) : R::abs(iwx);
    const int F = cp.fix_bits;
    if (global || (__double2hiint(v) >> 20) >= 1023 + kFixedDepositBits - F) {
        const double a = up ? x0 : x1, b = up ? x1 : x0, L = R::L(cp);
        plan_flight_real(f, R::nonneg(a) * R::inv_dx(cp), (R::lt(L, R::nonneg(b)) ? L : R::nonneg(b)) * R::inv_dx(cp), l,
                         R::dx(cp) * R::abs(iwx));
        return;
    }
    const Fix96 q = fixed96(v, F);
    const bool multi = k0 != k1;  // else a0 = q, a1 = 0
    f.a0 = sub96(q, fraction96(multi ? (up ? from.F : to.F) : 0ull, q));
    f.a1 = fraction96(multi ? (up ? to.F : from.F) : 0ull, q);
    f.c = q;
}

// A flight by its ends alone.
template <typename Case>
__device__ __forceinline__ void plan_flight(Flight<double> &f, const Case &cp, double x0, double x1, double l, double,
                                            double iwx, bool global) {
    plan_flight(f, cp, mesh_point(cp, x0), mesh_point(cp, x1), x0, x1, l, iwx, global);
}

// Where a history's position lies on the mesh, when it has been set.
template <typename Case>
__device__ __forceinline__ void set_mesh_point(History<double> &s, const Case &cp) {
    s.at = mesh_point(cp, s.r[0]);
}
template <typename Case>
__device__ __forceinline__ void set_mesh_point(History<float> &, const Case &) {}

// Distance along the flight to the face ahead on one axis: (L - r)/omega
// moving up, (0 - r)/omega moving down, clamped at 0; infinite when omega is
// +-0.  One multiply on every lane, no branch.
template <typename P>
__device__ __forceinline__ P face_distance(P r, P w, P iw, P L) {
    using R = Real<P>;
    const P target = R::pos(w) ? L : P(0);
    const P d = R::nonneg((target - r) * iw);
    return R::is_zero(w) ? R::inf() : d;
}

// The next event: the flight's length and what ends it.
template <typename P>
struct Choice {
    P l;
    bool bnd, coll;   // boundary, collision; else interface
    int face;         // 0: x = 0, 1: x = L, 2: lateral
    bool on_y, on_z;  // reflection on a y and / or z face
};

// The smallest of the collision, interface and boundary distances: x faces,
// then the lateral faces of the box; boundary, else collision, else interface.
template <typename P, int G, typename Case>
__device__ __forceinline__ Choice<P> choose_event(const History<P> &s, const Case &cp, P l_c, P l_i, P iy, P iz) {
    using R = Real<P>;
    const int gd = geometry<G>(cp);
    const P INF = R::inf(), L = R::L(cp);
    Choice<P> c;
    c.face = R::pos(s.w[0]) ? 1 : 0;
    P l_b = face_distance(s.r[0], s.w[0], s.iw[0], L);
    P l_y = INF, l_z = INF;
    if (gd == 3 || gd == 2) {  // lateral faces: y (and z in the box; the extruded geometry has none)
        l_y = face_distance(s.r[1], s.w[1], iy, L);
        if (R::lt(l_y, l_b)) {
            l_b = l_y;
            c.face = 2;
        }
        if (gd == 3) {
            l_z = face_distance(s.r[2], s.w[2], iz, L);
            if (R::lt(l_z, l_b)) {
                l_b = l_z;
                c.face = 2;
            }
        }
    }
    c.bnd = R::le(l_b, l_c) && R::le(l_b, l_i);
    c.coll = !c.bnd && R::le(l_c, l_i);
    c.l = c.bnd ? l_b : (c.coll ? l_c : l_i);
    c.on_y = c.bnd && c.face == 2 && R::eq(l_y, l_b);
    c.on_z = c.bnd && c.face == 2 && R::eq(l_z, l_b);
    return c;
}

// l_c from -ln(1 - u) of its draw
template <typename P, typename Case>
__device__ __forceinline__ P collision_distance(const Case &cp, int m, P e_c) {
    using R = Real<P>;
    return R::pos(R::sigma(cp, m)) ? R::nonneg(e_c * R::inv_sigma(cp, m)) : R::inf();
}

// l_i from -ln(1 - u) of its draw
template <typename P, int G, typename Case>
__device__ __forceinline__ P interface_distance(const History<P> &s, const Case &cp, int m, P e_i) {
    using R = Real<P>;
    const int gd = geometry<G>(cp);
    P l_i = R::lambda(cp, m) * e_i;
    if (gd == 11) l_i *= R::abs(s.iw[0]);  // slab: the chord projected on x, Lambda/|mu|
    else if (gd == 2) l_i /= sqrt(P(1) - s.w[2] * s.w[2]);  // extruded: in-plane chord along the flight
    return R::nonneg(l_i);
}

// |x| in float, truncated to 21 bits, for 0 or 2^-126 <= |x| < 2^128 (smaller: 0)
__device__ __forceinline__ float coarse(double x) {
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
    return h < (897u << 20) ? 0.0f : __uint_as_float((h << 3) + 0x40000000u);
}

// The event of the FP64 walk with one exact distance instead of five.  The
// five are first bounded in FP32 (a filtered predicate in the sense of Fortune
// and Van Wyk, Proc. 9th ACM Symp. Computational Geometry, 1993), and where
// the nearest is certain only its distance is evaluated in FP64: one logarithm
// instead of two, at most one reciprocal (of a lateral face's direction), one
// product.  Bounds: positions and directions lose 2^-20 of their values, so a
// boundary distance lies within L 2^-18/|w| of (target - r)/|w| in FP32;
// -ln(1 - u), at most 11.1 here, from the draw's high word (within 2^-32 of u, so
// 2^-16 of 1 - u > 2^-16) and the hardware's log2 (2^-22 relative) lies within
// 2^-14, the parameters' and 1/|w|'s relative roundings (2^-23 and 2^-19.6)
// included.  The
// rest, about 2 draws in 10^4, and cases of extreme magnitudes (filter) take
// all five exactly.  Results are the exact comparison's.  FP64 instructions
// take 64 cycles per warp and scheduler here, FP32 ones one or two.  Measured
// (FP64): the box L = 10, 1e7 histories, 45.7 -> 41.1 ms; extruded 3e5 1457 ->
// 1237 us; warp instructions per event of the box 76 -> 60.
template <int G, typename Case>
__device__ __forceinline__ Choice<double> choose_filtered(const History<double> &s, const Case &cp, int m, uint32_t hi,
                                                          uint32_t lo, uint32_t ihi, uint32_t ilo) {
    using R = Real<double>;
    const int gd = geometry<G>(cp);
    const bool box = gd == 3, lateral = box || gd == 2;
    const float L = cp.L_f, err = L * 0x1p-18f;
    // the nearest so far and its bounds, and the least lower bound of the others
    int which = 0;  // 0, 1, 2: x, y, z face; 3: collision; 4: interface
    float low = 0.0f, high = 0.0f, rest = __int_as_float(0x7f800000);
    auto face = [&](int axis, float *a, float *b) {
        const float r = coarse(s.r[axis]), iw = Real<float>::recip(coarse(s.w[axis]));
        const float d = __double2hiint(s.w[axis]) >= 0 ? L - r : r;
        *a = (d - err) * iw;
        *b = (d + err) * iw;
    };
    auto consider = [&](int q, float a, float b) {
        const bool nearer = b < high;
        rest = fminf(rest, nearer ? low : a);
        low = nearer ? a : low;
        high = nearer ? b : high;
        which = nearer ? q : which;
    };
    face(0, &low, &high);
    float fa, fb;
    if (lateral) {
        face(1, &fa, &fb);
        consider(1, fa, fb);
        if (box) {
            face(2, &fa, &fb);
            consider(2, fa, fb);
        }
    }
    const float kErr = 0x1p-14f, kLn2 = 0.693147180559945f;
    const float e_c = -kLn2 * __log2f((float)~hi * 0x1p-32f), e_i = -kLn2 * __log2f((float)~ihi * 0x1p-32f);
    if (cp.sigma_f[m] > 0.0f) consider(3, (e_c - kErr) * cp.inv_sigma_f[m], (e_c + kErr) * cp.inv_sigma_f[m]);
    float la = cp.lambda_f[m], lb = la;
    if (gd == 11) {
        la *= Real<float>::recip(coarse(s.w[0]));
        lb = la;
    } else if (gd == 2) {  // 1 - wz^2 within 2^-18
        const float wz = coarse(s.w[2]), q = fmaf(-wz, wz, 1.0f);
        la *= rsqrtf(q + 0x1p-18f);
        lb *= rsqrtf(q - 0x1p-18f);
    }
    consider(4, (e_i - kErr) * la, (e_i + kErr) * lb);
    // (a certain face is never one of direction 0, whose bounds are infinite)
    const bool sure = high < rest && cp.filter && hi < 0xFFFF0000u && ihi < 0xFFFF0000u;

    Choice<double> c;
    if (sure) {
        c.bnd = which < 3;
        c.coll = which == 3;
        c.face = which == 0 ? (R::pos(s.w[0]) ? 1 : 0) : 2;
        c.on_y = which == 1;
        c.on_z = which == 2;
        // the two factors of the distance, one product for all lanes
        double a, b;
        if (c.bnd) {
            const double r = which == 0 ? s.r[0] : which == 1 ? s.r[1] : s.r[2];
            const double w = which == 0 ? s.w[0] : which == 1 ? s.w[1] : s.w[2];
            a = (R::pos(w) ? R::L(cp) : 0.0) - r;
            b = which == 0 ? s.iw[0] : R::recip(w);
        } else {
            a = exp_variate_shared(c.coll ? R::k53(hi, lo) : R::k53(ihi, ilo));
            b = c.coll ? R::inv_sigma(cp, m) : R::lambda(cp, m);
        }
        double l = a * b;
        if (which == 4) {
            if (gd == 11) l *= R::abs(s.iw[0]);
            else if (gd == 2) l /= sqrt(1.0 - s.w[2] * s.w[2]);
        }
        c.l = R::nonneg(l);
    } else {
        double x_c, x_i;
        R::exp_variates(hi, lo, ihi, ilo, &x_c, &x_i);
        c = choose_event<double, G>(s, cp, collision_distance<double>(cp, m, x_c),
                                    interface_distance<double, G>(s, cp, m, x_i), recip_or_inf(s.w[1]),
                                    recip_or_inf(s.w[2]));
    }
    return c;
}

// Where step takes its random numbers from.  PhiloxDraws: the lane's own
// Philox blocks, computed as they are needed; with DEFER a 3D or extruded
// scatter leaves its direction pending for the caller's resolve_direction.
template <typename P, int G, bool DEFER>
struct PhiloxDraws {
    const RoundKeys &key;

    // The event, from the draws of the collision, then the interface distance.
    // One Philox block serves both draws (draw_pair), except in the FP32
    // x-projected walk, where holding the pair spills registers (measured 10%
    // slower there, 4-7% faster elsewhere).
    template <typename Case>
    __device__ __forceinline__ Choice<P> choose(History<P> &s, const Case &cp, int m) {
        uint32_t hi, lo, ihi, ilo;
        if constexpr (sizeof(P) == 8) {
            draw_pair(s, key, hi, lo, ihi, ilo);
            return choose_filtered<G>(s, cp, m, hi, lo, ihi, ilo);
        } else {
            P e_c, e_i;
            if constexpr (G == 13) {
                draw_words(s, key, hi, lo);
                e_c = Real<P>::exp_variate(hi, lo);
                draw_words(s, key, ihi, ilo);
                e_i = Real<P>::exp_variate(ihi, ilo);
            } else {
                draw_pair(s, key, hi, lo, ihi, ilo);
                Real<P>::exp_variates(hi, lo, ihi, ilo, &e_c, &e_i);
            }
            return choose_event<P, G>(s, cp, collision_distance<P>(cp, m, e_c), interface_distance<P, G>(s, cp, m, e_i),
                                      Real<P>::recip(s.w[1]), Real<P>::recip(s.w[2]));
        }
    }
    template <typename Case>
    __device__ __forceinline__ void score(Flight<P> &f, History<P> &s, const Case &cp, P x1, P l, bool global) {
        if constexpr (sizeof(P) == 8) {
            const MeshPoint<P> to = mesh_point(cp, x1);
            plan_flight(f, cp, s.at, to, s.r[0], x1, l, s.iw[0], global);
            s.at = to;
        } else {
            plan_flight(f, cp, s.r[0], x1, l, s.w[0], s.iw[0], global);
        }
    }
    __device__ __forceinline__ bool below(History<P> &s, unsigned long long thr53, uint32_t thr24) {
        return draw_below(s, key, thr53, thr24);
    }
    __device__ __forceinline__ bool up(History<P> &s) {  // u < 1/2: the top bit of the draw is clear
        uint32_t hi, lo;
        draw_words(s, key, hi, lo);
        return (hi >> 31) == 0u;
    }
    __device__ __forceinline__ void scatter_x(History<P> &s) { set_direction_x(s, draw_iso(s, key)); }
    __device__ __forceinline__ void scatter(History<P> &s, const CaseParams &cp) {
        s.pend = DIR_SCATTER;
        if (!DEFER) resolve_direction<P, G>(s, cp, key);
    }
};

// NarrowDraws: draws computed ahead by the lanes of a warp (narrow_kernel).
// The buffer holds, for every draw of its range, the output words, the
// exponential variate, and the direction of a scatter whose mu is this draw
// and whose phi is the next (w[2] = mu alone for the one-dimensional walks).
template <typename P>
struct DrawBuffer {
    static constexpr int kDraws = 64;  // two for each lane of the warp
    float4 w[kDraws];                  // w[0], w[1], w[2], -
    float e[kDraws];
    uint32_t hi[kDraws];
};
template <>
struct DrawBuffer<double> {
    static constexpr int kDraws = 64;
    double2 w01[kDraws], w2i0[kDraws], i12[kDraws];  // (w[0], w[1]), (w[2], 1/w[0]), (1/w[1], 1/w[2])
    double e[kDraws];
    uint2 word[kDraws];                              // (hi, lo)
};

template <typename P, int G>
struct NarrowDraws {
    // the draws of one event: j, j + 1 (distances), j + 2 (scatter or absorb), j + 3, j + 4 (direction)
    P e_c, e_i, wx, wy, wz, ix, iy, iz;
    uint32_t t_hi, t_lo, x_hi;

    P x0, x1, l, fw, fiw;  // the flight made: its x, length, direction cosine and its reciprocal

    __device__ __forceinline__ void fetch(const DrawBuffer<P> &b, int slot) {
        e_c = b.e[slot];
        e_i = b.e[slot + 1];
        if constexpr (sizeof(P) == 8) {
            const uint2 t = b.word[slot + 2];
            t_hi = t.x;
            t_lo = t.y;
            if constexpr (G == 0 || G == 1) x_hi = b.word[slot + 3].x;
            if constexpr (G != 1) {
                const double2 w2i0 = b.w2i0[slot + 3];
                wz = w2i0.x;
                ix = w2i0.y;
            }
            if constexpr (G != 1 && G != 11 && G != 13) {
                const double2 w01 = b.w01[slot + 3], i12 = b.i12[slot + 3];
                wx = w01.x;
                wy = w01.y;
                iy = i12.x;
                iz = i12.y;
            }
        } else {
            t_hi = b.hi[slot + 2];
            t_lo = 0;
            if constexpr (G == 0 || G == 1) x_hi = b.hi[slot + 3];
            if constexpr (G != 1) {
                const float4 w = b.w[slot + 3];
                wx = w.x;
                wy = w.y;
                wz = w.z;
            }
        }
    }
    template <typename Case>
    __device__ __forceinline__ void score(Flight<P> &, const History<P> &s, const Case &, P x, P length, bool) {
        x0 = s.r[0];
        x1 = x;
        l = length;
        fw = s.w[0];
        fiw = s.iw[0];
    }
    template <typename Case>
    __device__ __forceinline__ Choice<P> choose(History<P> &s, const Case &cp, int m) {
        s.j += 2u;
        P i1, i2;
        if constexpr (sizeof(P) == 8) {
            i1 = s.iw[1];
            i2 = s.iw[2];
        } else {
            i1 = Real<P>::recip(s.w[1]);
            i2 = Real<P>::recip(s.w[2]);
        }
        return choose_event<P, G>(s, cp, collision_distance<P>(cp, m, e_c), interface_distance<P, G>(s, cp, m, e_i), i1, i2);
    }
    __device__ __forceinline__ bool below(History<P> &s, unsigned long long thr53, uint32_t thr24) {
        ++s.j;
        return Real<P>::below(t_hi, t_lo, thr53, thr24);
    }
    __device__ __forceinline__ bool up(History<P> &s) {
        ++s.j;
        return (x_hi >> 31) == 0u;
    }
    __device__ __forceinline__ void scatter_x(History<P> &s) {
        ++s.j;
        if constexpr (sizeof(P) == 8) {
            s.w[0] = wz;
            s.iw[0] = G == 0 ? iz : ix;
        } else {
            set_direction_x(s, wz);
        }
    }
    template <typename Case>
    __device__ __forceinline__ void scatter(History<P> &s, const Case &) {
        s.j += 2u;
        if constexpr (sizeof(P) == 8) {
            s.w[0] = wx;
            s.w[1] = wy;
            s.w[2] = wz;
            s.iw[0] = ix;
            s.iw[1] = iy;
            s.iw[2] = iz;
        } else {
            set_direction(s, wx, wy, wz);
        }
    }
};

// One event of Algorithm A.  Fills the flight to score and returns -1 while
// the history continues, else the terminating event (EV_LEAK_X0, EV_LEAK_XL,
// EV_ABSORB, EV_CAPPED).  global: the lane scores into the global bins.
template <typename P, bool TRACE, int G, typename Draws, typename Case>
__device__ __forceinline__ int step(History<P> &s, const Case &cp, Draws &draws, uint32_t max_events,
                                    Flight<P> &f, TraceSink *tr, bool global = false) {
    using R = Real<P>;
    const int gd = geometry<G>(cp);
    f.k0 = 0;
    f.k1 = -1;
    if (s.events == max_events) {
        trace_row<P, TRACE>(tr, EV_CAPPED, s, 0.0);
        return EV_CAPPED;
    }
    ++s.events;
    const int m = s.m;
    const P L = R::L(cp);

    // Every lane moves and scores its flight on one converged path.
    const Choice<P> c = draws.choose(s, cp, m);
    const bool bnd = c.bnd, coll = c.coll, leak = bnd && c.face != 2;
    const P l = c.l;
    const P x1 = leak ? ((c.face == 0) ? P(0) : L) : s.r[0] + l * s.w[0];
    add_track(s, l, m);
    draws.score(f, s, cp, x1, l, global);
    s.r[0] = x1;
    if (gd == 3 || gd == 2) {
        if (c.on_y) {  // specular reflection on a y face
            s.r[1] = R::pos(s.w[1]) ? L : P(0);
            s.w[1] = R::flip(s.w[1]);
            s.iw[1] = R::flip(s.iw[1]);
        } else {
            s.r[1] += l * s.w[1];
        }
    }
    if (gd == 3) {
        if (c.on_z) {  // and/or on a z face
            s.r[2] = R::pos(s.w[2]) ? L : P(0);
            s.w[2] = R::flip(s.w[2]);
            s.iw[2] = R::flip(s.iw[2]);
        } else {
            s.r[2] += l * s.w[2];
        }
    }
    if (leak) {
        const int ev = (c.face == 0) ? EV_LEAK_X0 : EV_LEAK_XL;
        trace_row<P, TRACE>(tr, ev, s, (double)l);
        return ev;
    }
    if (bnd) {
        ++s.n_refl;
        trace_row<P, TRACE>(tr, EV_REFLECT, s, (double)l);
        return -1;
    }
    if (coll) {
        ++s.n_coll;
        if (draws.below(s, R::thr_c53(cp, m), R::thr_c24(cp, m))) {
            if (gd == 1) {
                const P w = draws.up(s) ? P(1) : P(-1);
                s.w[0] = w;
                s.iw[0] = w;
            } else if (gd == 11 || gd == 13) {
                draws.scatter_x(s);  // mu = 2 xi - 1
            } else {
                draws.scatter(s, cp);  // mu = 2 xi - 1, then phi
            }
            trace_row<P, TRACE>(tr, EV_SCATTER, s, (double)l);
            return -1;
        }
        trace_row<P, TRACE>(tr, EV_ABSORB, s, (double)l);
        return EV_ABSORB;
    }
    s.m = 1 - m;
    ++s.n_int;
    trace_row<P, TRACE>(tr, EV_INTERFACE, s, (double)l);
    return -1;
}

// ------------------------------------------------------- tally regions
// A warp-private shared-memory region (layout: region_bytes() in
// cls_internal.h): the bins, FP64 statistics, counters and the lanes' own
// copies of the per-history statistics.  The bins are a fixed-point difference
// array, prefix-summed exactly at the flush: the FP32 walk's with 32 fraction
// bits of track length, the FP64 walk's in 96 bits with fix_bits of a bin width
// (cls_fixed.h).
//
// 64-bit additions in shared memory go through 32-bit halves: the low half's
// atomic returns the old value, whose carry joins the high half.  Every wrap
// of a low half is seen by exactly one addition, so the pair holds the sum
// modulo 2^64 whatever the order.  Measured at full occupancy on random
// entries of 200: 14 cycles per warp and scheduler, against 62 for a 64-bit
// integer atomic and 94 for a double (both are compare-and-swap loops, and
// slow down further where lanes meet: 90 and 250 on 20 entries; the halves
// stay at 14).  The high half is added even where it is zero: the walk is short
// of integer instructions, not of shared-memory ones (testing it first: box L =
// 10, FP32, 1e8 histories 93.5 ms, adding it always 91.9).
__device__ __forceinline__ void add_halves(uint32_t *lo, uint32_t *hi, unsigned long long x) {
    const uint32_t xl = (uint32_t)x;
    const uint32_t old = atomicAdd(lo, xl);
    uint32_t h;  // the high half and the carry of old + xl
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %3, 0;\n\t}"
        : "=r"(h)
        : "r"(old), "r"(xl), "r"((uint32_t)(x >> 32)));
    atomicAdd(hi, h);
}

template <typename P>
constexpr bool kFixedStats = sizeof(P) == 4;

// difference array entry k (k <= nbs)
__device__ __forceinline__ void add_entry(unsigned char *region, int nbs, int k, unsigned long long x) {
    uint32_t *lo = reinterpret_cast<uint32_t *>(region) + k;
    add_halves(lo, lo + nbs + 1, x);
}

template <typename P>
__device__ __forceinline__ uint32_t *region_counters(unsigned char *region, int nbs) {
    return reinterpret_cast<uint32_t *>(region + region_bins_bytes(sizeof(P) == 8, nbs) + 8 * S_NUM);
}

// counter c of the region += x (C_MAXEV: maximum, below 2^32)
__device__ __forceinline__ void add_count(uint32_t *ct, int c, unsigned long long x) {
    add_halves(ct + c, ct + C_NUM + c, x);
}

// round(c 2^32), ties to even, for 0 <= c < 2^32, in two 32-bit halves: the
// integer part of c, and the fraction c - floor(c) (exact in float) scaled by
// 2^32 (exact) and rounded to the nearest integer, below 2^32 because a
// fraction of a float is at most 1 - 2^-24.  The halves add up to the one
// rounding of c 2^32, since its integer part shifts the rounded value by a
// multiple of 2^32.  Two 32-bit conversions instead of one to 64 bits: those
// run on the FP64 pipe, which the walk's history-end statistics already use
// (measured 1% faster on the sweep and the 3D box).
__device__ __forceinline__ unsigned long long fixed32(float c) {
    const uint32_t hi = __float2uint_rz(c);
    const float frac = c - __uint2float_rz(hi);
    return ((unsigned long long)hi << 32) | __float2uint_rn(frac * 0x1p32f);
}

// The lanes' own copies of the per-history statistics: FP64 in FP64 regions;
// in FP32 regions u64 fixed point -- t0, t1 with 32 fraction bits, t^2 with
// 24; the slot of t stays unused, its sum being that of t0 and t1 -- so that
// the FP32 walk sums them exactly.
template <typename P>
using LaneStat = typename std::conditional<kFixedStats<P>, unsigned long long, double>::type;

template <typename P>
__device__ __forceinline__ LaneStat<P> *region_lane_stats(unsigned char *region, int nbs) {
    return reinterpret_cast<LaneStat<P> *>(region + region_lane_stats_offset(sizeof(P) == 8, nbs));
}

// A history longer than this (in track length) keeps its statistics out of the
// fixed-point lane copies: t <= 2^13 is below 2^45 with 32 fraction bits and
// t^2 below 2^50 with 24, so a lane's sums stay below 2^64 for up to 2^13
// histories between flushes (FP32 regions flush every 1024).
constexpr float kFixedTrackMax = 8192.0f;

template <typename P>
__device__ __forceinline__ double *region_stats(unsigned char *region, int nbs) {
    return reinterpret_cast<double *>(region + region_bins_bytes(sizeof(P) == 8, nbs));
}

// The history's track length t and t^2 into this lane's own copy of the
// region's statistics (no atomics).  FP64 walk: in FP64.  FP32 walk: the
// history's float sums per material, t0 and t1, are rounded once to 32
// fraction bits and added exactly, t = t0 + t1 from those; t^2 is the square
// of the float t, rounded to 24 fraction bits.  Returns false, with nothing
// added, for a history the fixed-point copies cannot hold (track length
// beyond kFixedTrackMax): the caller adds it to the global FP64 statistics.
template <typename P>
__device__ __forceinline__ bool finish_history(unsigned char *region, int nbs, const History<P> &s, int lane) {
    LaneStat<P> *ls = region_lane_stats<P>(region, nbs) + lane;
    if constexpr (kFixedStats<P>) {
        const float t = s.track0 + s.track1;
        if (!(t <= kFixedTrackMax)) return false;
        const unsigned long long q0 = fixed32(s.track0), q1 = fixed32(s.track1);
        // the sum of t is that of t0 plus that of t1: the flush forms it
        ls[32 * S_T2] += __float2ull_rn(t * t * 0x1p24f);
        ls[32 * S_TRACK0] += q0;
        ls[32 * S_TRACK1] += q1;
    } else {
        const double t0 = (double)s.track0;
        const double t1 = (double)s.track1;
        const double t = t0 + t1;
        ls[32 * S_T] += t;
        ls[32 * S_T2] += t * t;
        ls[32 * S_TRACK0] += t0;
        ls[32 * S_TRACK1] += t1;
    }
    return true;
}

// Draws that the source takes.
template <int G>
__device__ __forceinline__ uint32_t source_draws(const CaseParams &cp) {
    const int gd = geometry<G>(cp);
    const uint32_t volume = cp.source == 1;
    return gd == 3 ? 5u + volume : gd == 2 ? 4u + volume : gd == 1 ? 1u + 2u * volume : 2u + volume;
}

// A finished history's collisions and reflections since its draw index was
// base_j, from that and its other counters since then (the walk need not count
// them): every event takes two draws, every collision one and every scatter one
// more (a direction cosine) or two (mu and phi); and every event is a
// collision, an interface crossing, a reflection or the final leak.
template <typename P, int G>
__device__ __forceinline__ void derive_counts(const History<P> &s, const CaseParams &cp, int outcome, uint32_t base_j,
                                              uint32_t events, uint32_t *n_coll, uint32_t *n_refl) {
    const int gd = geometry<G>(cp);
    const uint32_t absorbed = outcome == EV_ABSORB, leaked = outcome == EV_LEAK_X0 || outcome == EV_LEAK_XL;
    const uint32_t extra = s.j - base_j - 2u * events;  // of collisions and scatters
    *n_coll = gd == 3 || gd == 2 ? (extra + 2u * absorbed) / 3u : (extra + absorbed) / 2u;
    *n_refl = events - *n_coll - s.n_int - leaked;
}

// Outcome and event counters of a finished history.
__device__ __forceinline__ void count_one(uint32_t *ct, int outcome, uint32_t n_coll, uint32_t n_int, uint32_t n_refl,
                                          uint32_t events, uint32_t longest) {
    const int c = (outcome == EV_LEAK_X0) ? C_R : (outcome == EV_LEAK_XL) ? C_T : (outcome == EV_ABSORB) ? C_A : C_CAPPED;
    add_count(ct, c, 1ull);
    if (n_coll) add_count(ct, C_COLL, n_coll);
    if (n_int) add_count(ct, C_INT, n_int);
    if (n_refl) add_count(ct, C_REFL, n_refl);
    add_count(ct, C_EVENTS, events);
    atomicMax(&ct[C_MAXEV], longest);
}

// The interior bins of the flights that score into the global bins, spread
// evenly over the 32 lanes: lane t of each round scores interior task base +
// t, found by a 5-step shuffle search over the warp's inclusive prefix sum of
// the interior counts ni.
__device__ __forceinline__ void spread_interior(double *gflux, uint64_t goff, int k0, double c, int ni, int lane) {
    int incl = ni;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(CLS_FULL_MASK, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(CLS_FULL_MASK, incl, 31);
    const int base_bin = k0 + 1 - (incl - ni);  // interior task t of this lane goes to base_bin + t
    for (int base = 0; base < total; base += 32) {
        const int t = base + lane;
        int o = 0;
#pragma unroll
        for (int sft = 16; sft >= 1; sft >>= 1) {
            const int v = __shfl_sync(CLS_FULL_MASK, incl, o + sft - 1);
            if (v <= t) o += sft;
        }
        const int ob = __shfl_sync(CLS_FULL_MASK, base_bin, o);
        const double oc = __shfl_sync(CLS_FULL_MASK, c, o);
        const uint64_t ogoff = __shfl_sync(CLS_FULL_MASK, goff, o);
        if (t < total) atomicAdd(&gflux[ogoff + ob + t], oc);
    }
}

// The global bins of (case, batch), as an offset into the flux array.
__device__ __forceinline__ uint64_t bins_offset(const Tallies &t, int lcase, uint32_t lbatch) {
    return ((uint64_t)lcase * (uint64_t)t.nbatch + lbatch) * (uint64_t)t.nbins_stride;
}

// Bound on a region's bins between two flushes (FP64 walk): each lane sums the
// high words of its flights' largest deposits, rounded up, at most 2^26 each, and
// the warp flushes once a lane's sum has reached 2^26: no lane's passes 2^27, so
// no bin of the warp reaches 2^96 units.  (For F = 64 that is 2^26 bin widths: in
// practice only key changes flush.)  FP32 regions are flushed by the histories fed
// into them.
constexpr uint32_t kDepositBound = 1u << (kFixedDepositBits - 64);
static_assert(32ull * 2 * kDepositBound <= 1ull << 32, "a bin's sum stays below 2^96 units");

// A flight's entries in the difference array D (bin k = D[0] + ... + D[k]): its
// bins are a0 in k0, c in each interior bin k0 < k < k1 and a1 in k1, each
// rounded once to fixed point (q0, qc, q1; zero where the flight has no such
// bin), so D[k0] += q0, D[k0+1] += d1 = qc - q0 (or q1 - q0 when k1 = k0 + 1),
// D[k1] += d2 = q1 - qc (with interior bins), D[k1+1] += d3 = -q1 (beyond one
// bin), modulo 2^64 (2^96 in the FP64 walk): the flush's prefix sum returns
// exactly the rounded deposits, whatever the order of the additions.
struct FixedFlight {
    bool multi, inter;
    unsigned long long q0, d1, d2, d3;
    __device__ __forceinline__ explicit FixedFlight(const Flight<float> &f) : multi(f.k1 > f.k0), inter(f.k1 > f.k0 + 1) {
        q0 = fixed32(f.a0);
        const unsigned long long q1 = fixed32(multi ? f.a1 : 0.0f), qc = fixed32(inter ? f.c : 0.0f);
        d1 = (inter ? qc : q1) - q0;
        d2 = q1 - qc;
        d3 = 0ull - q1;
    }
};

// The flight's entries added to the difference array; returns its share of
// kDepositBound.
__device__ __forceinline__ uint32_t deposit_flight(unsigned char *region, int nbs, const Flight<float> &f) {
    const FixedFlight q(f);
    add_entry(region, nbs, f.k0, q.q0);
    add_entry(region, nbs, f.k0 + 1, q.d1);
    if (q.inter) add_entry(region, nbs, f.k1, q.d2);
    if (q.multi) add_entry(region, nbs, f.k1 + 1, q.d3);
    return 0u;
}

// 96-bit entry k: as with 64 bits (add_halves) each word's atomic returns the old
// value, whose carry joins the next word.
__device__ __forceinline__ void add_entry(unsigned char *region, int nbs, int k, Fix96 x) {
    uint32_t *const p = reinterpret_cast<uint32_t *>(region) + k;
    uint32_t old = atomicAdd(p, x.w0);
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.cc.u32 %0, %0, 0;\n\taddc.u32 %1, %1, 0;\n\t}"
        : "+r"(x.w1), "+r"(x.w2)
        : "r"(old), "r"(x.w0));
    old = atomicAdd(p + nbs + 1, x.w1);
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %0, 0;\n\t}"
        : "+r"(x.w2)
        : "r"(old), "r"(x.w1));
    atomicAdd(p + 2 * (nbs + 1), x.w2);
}

// FP64 walk.  Entry by entry: the four entries' words sent out together, to wait
// for shared memory twice instead of eight times, take more instructions and were
// slower (1e6 histories: rod 369 against 361 us, slab 515 / 498).
__device__ __forceinline__ uint32_t deposit_flight(unsigned char *region, int nbs, const Flight<double> &f) {
    const bool multi = f.k1 > f.k0, inter = f.k1 > f.k0 + 1;
    add_entry(region, nbs, f.k0, f.a0);
    add_entry(region, nbs, f.k0 + 1, sub96(inter ? f.c : f.a1, f.a0));  // (a1 = 0 in a flight of one bin)
    if (inter) add_entry(region, nbs, f.k1, sub96(f.a1, f.c));
    if (multi) add_entry(region, nbs, f.k1 + 1, sub96(Fix96{0u, 0u, 0u}, f.a1));
    return f.c.w2 + 1u;
}

// Score the warp's flights.
//   Region lanes: the difference array's entries (FixedFlight), two integer
//   additions for a flight inside one bin, three when it spans two, four
//   otherwise.
//   Lanes that score globally (scores_global) add FP64 values to the bins of
//   their (case, batch), interior bins spread over the warp.
// Returns the lane's share of DepositBound.
template <typename P>
__device__ __forceinline__ uint32_t warp_deposit(unsigned char *regions, int rbytes, const Tallies &t, int lreg, int lcase,
                                                 uint32_t lbatch, const Flight<P> &f, int lane) {
    const int nbs = t.nbins_stride;
    const bool has = f.k1 >= f.k0, global = scores_global(f, lreg);
    uint32_t bound = 0;
    if (has) {
        if (!global) {
            // predicated, not branched: every lane with a flight runs the same code
            bound = deposit_flight(regions + lreg * rbytes, nbs, f);
        } else {
            double *gbins = t.flux + bins_offset(t, lcase, lbatch);
            atomicAdd(&gbins[f.k0], flight_real(f.a0));
            if (f.k1 > f.k0) atomicAdd(&gbins[f.k1], flight_real(f.a1));
        }
    }
    const int ni = (has && global) ? max(f.k1 - f.k0 - 1, 0) : 0;
    // one vote instead of the scan when no lane has any
    if (__any_sync(CLS_FULL_MASK, ni > 0))
        spread_interior(t.flux, bins_offset(t, lcase, lbatch), f.k0, flight_real(f.c), ni, lane);
    return bound;
}

// A finished history's outcome into the caller's record, when one is bound
// (OutcomeRecord): 0 reflected (left through x = 0), 1 transmitted (x = L),
// 2 absorbed, 3 capped.  One byte per history; the host has checked that the
// record holds the run's cases x histories.
__device__ __forceinline__ void record_outcome(const LaunchArgs &a, int case_index, const HistoryKey &key, int outcome) {
    if (a.outcomes == nullptr) return;
    const OutcomeRecord r = *a.outcomes;
    if (r.codes == nullptr) return;
    const uint64_t h = history_id(key, a.rk);
    const uint8_t code = outcome == EV_LEAK_X0 ? 0 : outcome == EV_LEAK_XL ? 1 : outcome == EV_ABSORB ? 2 : 3;
    r.codes[(uint64_t)case_index * r.stride + (h - r.first)] = code;
}

// This warp's copy of a case's global statistics.  All warps of a launch work
// on the same case or two at a time, and an FP64 addition to one address of
// global memory takes 16 ns, whoever asks (0.7 ns for integers): with one copy
// per case a sweep's flushes queued on it (38 ns per flush; 256 cases x 1e6 in
// chunks of 256 histories ran at that rate, 38 ms).
__device__ __forceinline__ double *global_stats(const Tallies &t, int case_index) {
    const unsigned w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    return t.stats + ((size_t)case_index * t.stats_copies + w % (unsigned)t.stats_copies) * S_NUM;
}

// A history's track-length statistics added straight to the case's global
// FP64 tally block.
template <typename P>
__device__ __forceinline__ void add_history_stats_global(const LaunchArgs &a, int case_index, const History<P> &s) {
    double *st = global_stats(a.t, case_index);
    const double t0 = (double)s.track0;
    const double t1 = (double)s.track1;
    const double t = t0 + t1;
    atomicAdd(&st[S_T], t);
    atomicAdd(&st[S_T2], t * t);
    if (__double_as_longlong(t0) != 0) atomicAdd(&st[S_TRACK0], t0);
    if (__double_as_longlong(t1) != 0) atomicAdd(&st[S_TRACK1], t1);
}

// History end for a lane that scores into global memory: the same statistics
// and counters as finish_history, added to the case's global tally block.
template <typename P>
__device__ __forceinline__ void finish_history_global(const LaunchArgs &a, int case_index, const History<P> &s,
                                                      int outcome, bool with_event_counts, uint32_t n_coll = 0,
                                                      uint32_t n_refl = 0, uint32_t events = 0) {
    add_history_stats_global<P>(a, case_index, s);
    unsigned long long *ct = a.t.counters + (size_t)case_index * C_NUM;
    const int c = (outcome == EV_LEAK_X0) ? C_R : (outcome == EV_LEAK_XL) ? C_T : (outcome == EV_ABSORB) ? C_A : C_CAPPED;
    atomicAdd(&ct[c], 1ull);
    if (with_event_counts) {
        if (n_coll) atomicAdd(&ct[C_COLL], (unsigned long long)n_coll);
        if (s.n_int) atomicAdd(&ct[C_INT], (unsigned long long)s.n_int);
        if (n_refl) atomicAdd(&ct[C_REFL], (unsigned long long)n_refl);
        atomicAdd(&ct[C_EVENTS], (unsigned long long)events);
    }
    atomicMax(&ct[C_MAXEV], (unsigned long long)s.events);
}

// Flush a warp region into the global tally block of (case, batch): one global
// FP64 atomic per non-zero bin and, with `ends`, per statistic and counter
// (these belong to the case: a region that moves on to another batch of the
// same case keeps them); what is flushed is zeroed.
template <typename P>
__device__ __forceinline__ void flush_region(unsigned char *region, const LaunchArgs &a, int case_index,
                                             uint32_t batch, int lane, bool ends = true) {
    const int nbs = a.t.nbins_stride;
    const int nb = a.cases[case_index].nbins;
    double *g = a.t.flux + ((size_t)case_index * a.t.nbatch + batch) * (size_t)nbs;
    // the exact prefix sum of the fixed-point difference array, 32 bins at a
    // time; its entry nb (past the last bin) sums to zero and is cleared
    uint32_t *lo = reinterpret_cast<uint32_t *>(region), *hi = lo + nbs + 1;
    if constexpr (sizeof(P) == 4) {
        unsigned long long carry = 0ull;
        for (int base = 0; base <= nb; base += 32) {
            const int k = base + lane;
            unsigned long long d = (k <= nb) ? (unsigned long long)hi[k] << 32 | lo[k] : 0ull;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long v = __shfl_up_sync(CLS_FULL_MASK, d, o);
                if (lane >= o) d += v;
            }
            const long long q = (long long)(carry + d);  // the bin's deposits, in units
            carry += __shfl_sync(CLS_FULL_MASK, d, 31);
            if (k < nb && q != 0) atomicAdd(&g[k], (double)q * 0x1p-32);
            if (k <= nb) lo[k] = hi[k] = 0u;
        }
    } else {
        const double unit = a.cases[case_index].fix_unit;
        uint32_t *top = hi + nbs + 1;
        Fix96 carry{0u, 0u, 0u};
        for (int base = 0; base <= nb; base += 32) {
            const int k = base + lane;
            Fix96 d = (k <= nb) ? Fix96{lo[k], hi[k], top[k]} : Fix96{0u, 0u, 0u};
#pragma unroll 1
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t w0 = __shfl_up_sync(CLS_FULL_MASK, d.w0, o), w1 = __shfl_up_sync(CLS_FULL_MASK, d.w1, o),
                               w2 = __shfl_up_sync(CLS_FULL_MASK, d.w2, o);
                if (lane >= o) d = add96(d, Fix96{w0, w1, w2});
            }
            const Fix96 q = add96(carry, d);  // the bin's deposits, in units
            carry = Fix96{__shfl_sync(CLS_FULL_MASK, q.w0, 31), __shfl_sync(CLS_FULL_MASK, q.w1, 31),
                          __shfl_sync(CLS_FULL_MASK, q.w2, 31)};
            if (k < nb && (q.w0 | q.w1 | q.w2) != 0u) atomicAdd(&g[k], fix96_to_double(q) * unit);
            if (k <= nb) lo[k] = hi[k] = top[k] = 0u;
        }
    }
    if (!ends) {
        __syncwarp();
        return;
    }
    // the lanes' own copies of the per-history statistics, summed over the warp
    double *gst = global_stats(a.t, case_index);
    LaneStat<P> *ls = region_lane_stats<P>(region, nbs);
#pragma unroll
    for (int q = 0; q < S_NUM; ++q) {
        double v;
        if constexpr (kFixedStats<P>)
            v = (q == S_T) ? (double)(ls[32 * S_TRACK0 + lane] + ls[32 * S_TRACK1 + lane]) * 0x1p-32
                           : (double)ls[32 * q + lane] * (q == S_T2 ? 0x1p-24 : 0x1p-32);
        else v = ls[32 * q + lane];
        ls[32 * q + lane] = 0;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(CLS_FULL_MASK, v, o);
        if (lane == 0 && __double_as_longlong(v) != 0) atomicAdd(&gst[q], v);
    }
    double *st = region_stats<P>(region, nbs);
    if (lane < S_NUM) {
        const double v = st[lane];
        if (v != 0.0) {
            atomicAdd(&gst[lane], v);
            st[lane] = 0.0;
        }
    } else if (lane < S_NUM + C_NUM) {
        const int c = lane - S_NUM;
        uint32_t *ct = region_counters<P>(region, nbs);
        const unsigned long long v = (unsigned long long)ct[C_NUM + c] << 32 | ct[c];
        if (v != 0ull) {
            unsigned long long *gc = &a.t.counters[(size_t)case_index * C_NUM + c];
            if (c == C_MAXEV) atomicMax(gc, v);
            else atomicAdd(gc, v);
            ct[c] = ct[C_NUM + c] = 0u;
        }
    }
    __syncwarp();
}

// Global chunk index -> run entry (runs are in chunk order).
__device__ __forceinline__ int find_run(const LaunchArgs &a, uint64_t ch) {
    int lo = 0, hi = a.nruns - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.runs[mid].chunk_begin <= ch) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// A warp's feeding state in the history tracker: the ids being fed, its claim
// still to be fed (positions in its run entry), its piece and the histories
// known to be claimed of it (piece < 0: none yet), the regions' keys (run entry
// and batch; run < 0: none) and the histories fed into each since its last full
// flush, and the region, run entry and batch being fed.
struct WarpFeed {
    uint64_t cursor, end;
    uint64_t pos, pos_end;
    uint64_t known;
    int run[2];
    uint32_t batch[2];
    uint32_t fed[2];
    int piece;
    int reg, cur_run;
    uint32_t cur_batch;
    int stealing;
};
static_assert(sizeof(WarpFeed) <= kWarpFeedBytes, "WarpFeed outgrew its shared memory");

// Lane states beside the terminating events (>= 0).
constexpr int kWalking = -1, kEmpty = -2;


__device__ __forceinline__ uint64_t piece_size(const LaunchArgs &a, uint32_t piece) {
    const RunCase &rc = a.runs[piece / a.pieces_per_run];
    return min(a.piece_len, rc.n - (piece % a.pieces_per_run) * a.piece_len);
}

// A piece with unclaimed histories, the one with the most among the first 128
// from this warp's starting point that have any; -1 if there is none.
__device__ __forceinline__ int find_piece(const LaunchArgs &a, int lane) {
    const uint32_t np = (uint32_t)a.nruns * a.pieces_per_run;
    const uint32_t start = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 128u % np;
    for (uint32_t o = 0; o < np; o += 128) {
        uint32_t most = 0, best = 0;
#pragma unroll 4
        for (uint32_t i = 0; i < 4; ++i) {
            const uint32_t q = o + 32 * i + lane;
            if (q >= np) break;
            const uint32_t p = (start + q) % np;
            const uint64_t size = piece_size(a, p), used = __ldcg(&a.claimed[p]);
            const uint32_t left = used < size ? (uint32_t)min(size - used, (uint64_t)0xFFFFFFFFu) : 0u;
            if (left > most) {
                most = left;
                best = p;
            }
        }
        const uint32_t top = __reduce_max_sync(CLS_FULL_MASK, most);
        if (top > 0) {
            const unsigned who = __ballot_sync(CLS_FULL_MASK, most == top);
            return __shfl_sync(CLS_FULL_MASK, (int)best, __ffs(who) - 1);
        }
    }
    return -1;
}

// The warp's next claim, into feed->pos .. pos_end of piece feed->piece;
// false when nothing is left to claim.
//
// Pieces are handed out in the order of the work list, each to `team` warps in
// turn; a warp stays with its piece until all of it is claimed, and when all
// pieces are handed out it helps with those that have histories left.  So a
// warp's histories mostly lie in one statistics batch (it flushes its bins
// seldom, and histories seldom outlive their region), and the warps work on
// many batches at a time: a bin in global memory takes an FP64 addition only
// every 16 ns, and chunks dealt out one by one sent all warps' flushes to the
// same batch (1e7 rod histories in FP32: chunks of 32 8.9 ms, of 256 1.6 ms;
// pieces 1.25 ms).  A claim takes half of the team's even share of what the warp
// last knew to be left of the piece (all of it, when it comes to one), so that
// claims shrink as it ends, within claim_bits.
__device__ __forceinline__ bool claim(WarpFeed *feed, const LaunchArgs &a, int lane) {
    const uint32_t np = (uint32_t)a.nruns * a.pieces_per_run;
    int piece = feed->piece;
    uint64_t known = feed->known;
    bool stealing = feed->stealing != 0;
    while (true) {
        if (piece >= 0) {
            const uint64_t size = piece_size(a, piece);
            const RunCase &rc = a.runs[piece / a.pieces_per_run];
            const uint64_t share = (known < size ? size - known : 0ull) / (stealing ? max(2 * a.team, 64u) : 2 * a.team);
            const uint64_t k = max(min(share, (uint64_t)a.chunk << rc.claim_bits), (uint64_t)a.chunk);
            unsigned long long got;
            if (lane == 0) got = atomicAdd(&a.claimed[piece], (unsigned long long)k);
            got = __shfl_sync(CLS_FULL_MASK, got, 0);
            if (got < size) {
                if (lane == 0) {
                    const uint64_t base = (piece % a.pieces_per_run) * a.piece_len;
                    feed->pos = base + got;
                    feed->pos_end = base + min((uint64_t)got + k, size);
                    feed->known = got + k;
                    feed->piece = piece;
                    feed->stealing = stealing;
                }
                __syncwarp();
                return true;
            }
        }
        known = 0;
        if (!stealing) {
            unsigned long long t;
            if (lane == 0) t = atomicAdd(a.chunk_counter, 1ull);
            t = __shfl_sync(CLS_FULL_MASK, t, 0);
            stealing = t >= (unsigned long long)np * a.team;
            piece = stealing ? -1 : (int)(t / a.team);
        }
        if (stealing) {
            piece = find_piece(a, lane);
            if (piece < 0) return false;
        }
    }
}

// Empty lanes take the next histories of the warp's claims, in lane order.
// Returns whether the launch has no histories left to claim; wait: the run
// entry's refill_min.
template <typename P, int G>
__device__ __forceinline__ bool refill(unsigned char *regions, int rb, WarpFeed *feed, const LaunchArgs &a,
                                       History<P> &s, int &out, int &lreg, int &lcase, uint32_t &lbatch, int &wait,
                                       int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    unsigned need = __ballot_sync(CLS_FULL_MASK, out == kEmpty);
    while (need != 0u) {
        uint64_t cursor = feed->cursor, end = feed->end;
        int reg = feed->reg;
        if (cursor == end) {
            if (feed->pos == feed->pos_end && !claim(feed, a, lane)) return true;
            const int run = feed->piece / a.pieces_per_run;
            const RunCase &rc = a.runs[run];
            const uint64_t pos = feed->pos;
            const uint32_t batch = (uint32_t)(pos / rc.batch_len);
            // the claim's histories of this batch
            const uint64_t stop = min(feed->pos_end, (uint64_t)(batch + 1ull) * rc.batch_len);
            int r = -1;
            if (feed->run[0] == run && feed->batch[0] == batch) r = 0;
            else if (feed->run[1] == run && feed->batch[1] == batch) r = 1;
            if (r < 0) {
                const bool live0 = __any_sync(CLS_FULL_MASK, out == kWalking && lreg == 0);
                const bool live1 = __any_sync(CLS_FULL_MASK, out == kWalking && lreg == 1);
                const int other = reg ^ 1;
                if (!(other ? live1 : live0)) r = other;
                else if (!(reg ? live1 : live0)) r = reg;
                else r = other;  // both referenced: evict the older region
                const int old_run = feed->run[r];
                if (old_run >= 0) {
                    flush_region<P>(regions + r * rb, a, a.runs[old_run].case_index, feed->batch[r], lane, old_run != run);
                    // lanes still walking a history of the old key go on in global memory
                    if (out == kWalking && lreg == r) lreg = 2;
                }
                __syncwarp();
                if (lane == 0) {
                    if (old_run != run) feed->fed[r] = 0;
                    feed->run[r] = run;
                    feed->batch[r] = batch;
                }
            }
            reg = r;
            cursor = rc.first + pos;
            end = rc.first + stop;
            __syncwarp();
            if (lane == 0) {
                feed->pos = stop;
                feed->end = end;
                feed->reg = reg;
                feed->cur_run = run;
                feed->cur_batch = batch;
            }
            __syncwarp();
        }
        const uint64_t avail = end - cursor;
        const uint32_t nneed = __popc(need);
        const uint32_t take = (avail < nneed) ? (uint32_t)avail : nneed;
        const uint32_t rank = __popc(need & lt_mask);
        if (((need >> lane) & 1u) && rank < take) {
            lcase = a.runs[feed->cur_run].case_index;
            lreg = reg;
            lbatch = feed->cur_batch;
            source<P, G, true>(s, a.cases[lcase], a.rk, cursor + rank);
            out = kWalking;
        }
        const uint32_t fed = feed->fed[reg] + take;
        __syncwarp();
        // FP32 regions flush before a bin's sum can outgrow its 64 bits
        const bool full = sizeof(P) == 4 && fed >= a.flush_every;
        if (full) flush_region<P>(regions + reg * rb, a, a.runs[feed->cur_run].case_index, feed->cur_batch, lane);
        if (lane == 0) {
            feed->cursor = cursor + take;
            feed->fed[reg] = full ? 0u : fed;
        }
        __syncwarp();
        need = __ballot_sync(CLS_FULL_MASK, out == kEmpty);
    }
    wait = a.runs[feed->cur_run].refill_min;
    return false;
}

// ------------------------------------------------- history-based tracker
// Persistent kernel.  Each warp claims ranges of consecutive histories (claim);
// lanes whose histories have ended take the next histories of the warp's claim
// (ballot + prefix popcount), several lanes at a time, so lanes stay busy across
// history and claim boundaries.  Bound by issue (FP32) and by instruction supply
// and the FP64 pipe (FP64).  Before fixed-point bins in 32-bit words, claims
// from pieces, batched ends and births, events chosen by FP32 bounds and the
// shorter integer routines / now: box L = 10 in FP64 1e7 histories 56.7 / 34.5
// ms, in FP32 1e8 109.3 / 90.8 ms; 256-case sweep in FP32 at 1e6 a case 54.3 /
// 37.4 ms.  Each warp owns two shared-memory tally
// regions keyed by (case, batch); a region is flushed to global memory when
// its key changes, after flush_every histories (FP32) or kDepositBound (FP64),
// or when the warp retires.
// When a new key arrives while both regions still serve live histories, the
// older region is flushed and re-keyed, and its remaining histories score
// straight into the FP64 global tallies: the warp never waits for a straggler
// of a heavy-tailed history-length distribution.
// Launch bounds: FP32 blocks of 256 threads, 4 per SM (64 registers); the 3D
// box takes 4 blocks of 224 threads (history_threads_fp32: 72 registers hold
// its state without spills).  FP64 blocks of at most kHistoryBlockFp64 = 128
// threads, 5 per SM (102 registers, 20 warps), 6 (85 registers, 24 warps) for
// the one-dimensional walks (rod, slab, x-projected box), whose state fits:
// the FP64 walk is latency-bound, and more resident warps hide its
// integer-arithmetic and shared-memory latencies (measured: 5% faster for the
// x-projected box at 6; for the 3D and mixed walks 6 blocks gain 1% on the box
// at 1e7 histories, 41.1 -> 40.6 ms then, and lose 3-5% on smaller runs).
template <typename P, int G>
struct HistoryBounds {
    static constexpr int threads = kHistoryBlockFp64, blocks = (G == 1 || G == 11 || G == 13) ? 6 : 5;
};
template <int G>
struct HistoryBounds<float, G> {
    static constexpr int threads = history_threads_fp32(G), blocks = 4;
};

// The end of a lane's history: outcome record, statistics and counters (those
// since its draw index was base_j and its events base_events).
template <typename P, int G>
__device__ __forceinline__ void end_history(unsigned char *regions, const LaunchArgs &a, const History<P> &s, int out,
                                            int lreg, int lcase, uint32_t base_j, uint32_t base_events, int lane) {
    const uint32_t events = s.events - base_events;
    uint32_t n_coll, n_refl;
    derive_counts<P, G>(s, a.cases[lcase], out, base_j, events, &n_coll, &n_refl);
    record_outcome(a, lcase, s.key, out);
    if (lreg < 2) {
        unsigned char *region = regions + lreg * a.region_bytes;
        if (!finish_history<P>(region, a.t.nbins_stride, s, lane)) add_history_stats_global<P>(a, lcase, s);
        count_one(region_counters<P>(region, a.t.nbins_stride), out, n_coll, s.n_int, n_refl, events, s.events);
    } else {
        finish_history_global<P>(a, lcase, s, out, true, n_coll, n_refl, events);
    }
}

// A history handed from a tracker to the narrow walk, with the draw index and
// events up to which its collisions, crossings and reflections are counted.
template <typename P>
struct Straggler {
    P r[3], w[3], iw, track0, track1;
    HistoryKey key;
    uint32_t j, events, n_int, m, lcase, lbatch, base_j, base_events;
};
static_assert(sizeof(Straggler<float>) <= kStragglerBytes && sizeof(Straggler<double>) <= kStragglerBytes,
              "the host sizes the hand-over buffer");

// Once nothing is left to claim, a warp whose last few histories (at most
// LaunchArgs::hand_over) would walk on alone hands them over to the narrow walk (narrow_kernel); returns whether the
// lane's history was taken (all but those beyond the buffer's capacity).
template <typename P>
__device__ __forceinline__ bool hand_over(const LaunchArgs &a, const History<P> &s, int lcase, uint32_t lbatch,
                                          uint32_t base_j, uint32_t base_events, unsigned live, int lane) {
    unsigned slot = 0;
    if (lane == 0) slot = (unsigned)atomicAdd(a.handed, (unsigned long long)__popc(live));
    slot = __shfl_sync(CLS_FULL_MASK, slot, 0) + __popc(live & ((1u << lane) - 1u));
    if (!((live >> lane) & 1u) || slot >= a.straggler_cap) return false;
    Straggler<P> t;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        t.r[i] = s.r[i];
        t.w[i] = s.w[i];
    }
    t.iw = s.iw[0];
    t.track0 = s.track0;
    t.track1 = s.track1;
    t.key = s.key;
    t.j = s.j;
    t.events = s.events;
    t.n_int = s.n_int;
    t.m = (uint32_t)s.m;
    t.lcase = (uint32_t)lcase;
    t.lbatch = lbatch;
    t.base_j = base_j;
    t.base_events = base_events;
    *reinterpret_cast<Straggler<P> *>(a.stragglers + (size_t)slot * kStragglerBytes) = t;
    return true;
}

template <typename P, int G>
__global__ void __launch_bounds__(HistoryBounds<P, G>::threads, HistoryBounds<P, G>::blocks) history_kernel(const LaunchArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int rb = a.region_bytes;
    unsigned char *regions = smem + (size_t)warp * 2 * rb;
    for (int i = lane; i < 2 * rb / 8; i += 32) reinterpret_cast<unsigned long long *>(regions)[i] = 0ull;
    load_math_tables<P>(threadIdx.x, blockDim.x);
    if constexpr (sizeof(P) == 8) __syncthreads();
    __syncwarp();

    // warp-uniform feeding state, in shared memory: it is needed where lanes
    // take new histories only, and would hold a dozen registers of every lane
    WarpFeed *feed = reinterpret_cast<WarpFeed *>(smem + (size_t)(blockDim.x >> 5) * 2 * rb + (size_t)warp * kWarpFeedBytes);
    if (lane == 0) *feed = WarpFeed{0, 0, 0, 0, 0, {-1, -1}, {0, 0}, {0, 0}, -1, 0, 0, 0, 0};
    __syncwarp();

    // lane state: `out` is kWalking, kEmpty or the terminating event of a
    // history still to be counted; lreg is the lane's tally region, or 2 once
    // that region was handed to a newer key (the lane then scores into global
    // memory)
    History<P> s;
    Flight<P> f;
    int out = kEmpty;
    bool exhausted = false;
    int lreg = 0, lcase = 0;
    uint32_t lbatch = 0;
    uint32_t deposited = 0;  // FP64 walk: this lane's share of kDepositBound
    const RoundKeys &key = a.rk;

    PhiloxDraws<P, G, true> draws{key};
    int wait = 1;  // lanes that wait before histories end and start
    while (true) {
        const unsigned idle = __ballot_sync(CLS_FULL_MASK, out != kWalking);
        // History ends and births, together, once several lanes wait for them:
        // both are long stretches of code for the few lanes concerned.
        if (__popc(idle) >= wait) {
            if (out >= 0)
                end_history<P, G>(regions, a, s, out, lreg, lcase, source_draws<G>(a.cases[lcase]), 0u, lane);
            out = out >= 0 ? kEmpty : out;
            if (!exhausted) {
                exhausted = refill<P, G>(regions, rb, feed, a, s, out, lreg, lcase, lbatch, wait, lane);
                if (exhausted) wait = 32 - a.hand_over;
            } else {
                wait = 32;  // fewer than kHandOver histories were left, beyond the hand-over's capacity
            }
            const unsigned live = __ballot_sync(CLS_FULL_MASK, out == kWalking);
            if (exhausted && live != 0u && __popc(live) <= a.hand_over) {
                if (out == kWalking) resolve_direction<P, G>(s, a.cases[lcase], key);
                if (hand_over<P>(a, s, lcase, lbatch, source_draws<G>(a.cases[lcase]), 0u, live, lane)) out = kEmpty;
            }
            if (__all_sync(CLS_FULL_MASK, out != kWalking)) break;
        }
        f.k0 = 0;
        f.k1 = -1;
        if (out == kWalking) {
            // directions of the lanes born in this step and of those that scattered in the last
            resolve_direction<P, G>(s, a.cases[lcase], key);
            const int ev = step<P, false, G>(s, a.cases[lcase], draws, a.max_events, f, nullptr, lreg == 2);
            out = ev < 0 ? kWalking : ev;
        }
        deposited += warp_deposit<P>(regions, rb, a.t, lreg, lcase, lbatch, f, lane);
        if constexpr (sizeof(P) == 8) {  // before a bin's sum can outgrow its 64 bits
            if (__any_sync(CLS_FULL_MASK, deposited >= kDepositBound)) {
                __syncwarp();
#pragma unroll 1
                for (int r = 0; r < 2; ++r)
                    if (feed->run[r] >= 0)
                        flush_region<P>(regions + r * rb, a, a.runs[feed->run[r]].case_index, feed->batch[r], lane, false);
                deposited = 0;
            }
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int r = 0; r < 2; ++r)
        if (feed->run[r] >= 0)
            flush_region<P>(regions + r * rb, a, a.runs[feed->run[r]].case_index, feed->batch[r], lane);
}

// ------------------------------------------------------- narrow walk
// One history per warp: the last histories of the history tracker's warps
// (Straggler), and whole runs too small to occupy it (LaunchArgs::narrow).
// Both are bound by the serial chain of a history's events, 1.05 us each in
// FP32 and 3.1 us in FP64 when a lone lane computes everything.  But the
// random numbers depend on their position alone: the warp's lanes compute the
// history's next 64 draws at once -- Philox blocks, exponential variates, and
// the direction a scatter at each draw would take, with its reciprocals -- and
// only distances, the event and the move are left on the chain, which every
// lane follows; the case's parameters stay in registers, and the flights are
// scored 32 at a time, one by each lane.  The arithmetic is step's
// on the same draws, so results do not change.  Measured: 1000 histories of
// the 3D box in FP64 753 us by the tracker, 483 us here; the diffusive box,
// 1e6 histories in FP32, 20.4 ms without the hand-over, 12.8 ms with it.  An
// event of a lone history takes 0.23 us in FP32 and, in FP64, 0.47 us on the rod,
// 1.2 us in the box and 1.6 us in the extruded geometry.

// The two draws of a lane's Philox block into the buffer, at `at` and at + 1.
template <typename P, int G>
__device__ __forceinline__ void fill_draws(DrawBuffer<P> &b, int at, uint32_t block, const History<P> &s,
                                           const RoundKeys &key) {
    using R = Real<P>;
    const uint4 o = philox_block(block, s.key, key);
    // the next block's first draw: phi of a direction whose mu is this block's second
    const uint32_t n_hi = __shfl_down_sync(CLS_FULL_MASK, o.x, 1), n_lo = __shfl_down_sync(CLS_FULL_MASK, o.y, 1);
    P e0, e1;
    R::exp_variates(o.x, o.y, o.z, o.w, &e0, &e1);
    b.e[at] = e0;
    b.e[at + 1] = e1;
    if constexpr (sizeof(P) == 8) {
        b.word[at] = make_uint2(o.x, o.y);
        b.word[at + 1] = make_uint2(o.z, o.w);
    } else {
        b.hi[at] = o.x;
        b.hi[at + 1] = o.z;
    }
    if constexpr (G == 1) return;
    uint32_t mu_hi = o.x, mu_lo = o.y, phi_hi = o.z, phi_lo = o.w;
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
        if constexpr (G == 11 || G == 13) {
            const P mu = R::two_u_minus_one(mu_hi, mu_lo);
            if constexpr (sizeof(P) == 8) b.w2i0[at + t] = make_double2(mu, recip_or_inf(mu));
            else b.w[at + t] = make_float4(0.0f, 0.0f, mu, 0.0f);
        } else {
            P mu, wx, wy;
            R::direction(mu_hi, mu_lo, phi_hi, phi_lo, false, &mu, &wx, &wy);
            if constexpr (sizeof(P) == 8) {
                double v = wx, r0 = 0.0, r1 = 0.0, r2 = 0.0;
#pragma unroll 1
                for (int q = 0; q < 3; ++q) {  // one copy of the reciprocal
                    r0 = r1;
                    r1 = r2;
                    r2 = recip_or_inf(v);
                    v = q == 0 ? wy : mu;
                }
                b.w01[at + t] = make_double2(wx, wy);
                b.w2i0[at + t] = make_double2(mu, r0);
                b.i12[at + t] = make_double2(r1, r2);
            } else {
                b.w[at + t] = make_float4(wx, wy, mu, 0.0f);
            }
        }
        mu_hi = o.z;
        mu_lo = o.w;
        phi_hi = n_hi;
        phi_lo = n_lo;
    }
}

template <typename P>
struct NarrowMemory {  // dynamic shared memory of a warp, followed by its tally region
    DrawBuffer<P> draws;
    WarpFeed feed;
};
static_assert(sizeof(NarrowMemory<float>) <= narrow_memory_bytes(false) &&
                  sizeof(NarrowMemory<double>) <= narrow_memory_bytes(true) && narrow_memory_bytes(false) % 16 == 0 &&
                  narrow_memory_bytes(true) % 16 == 0,
              "the host sizes the narrow walk's shared memory");

template <typename P, int G>
__global__ void __launch_bounds__(kNarrowBlock, kNarrowBlocks) narrow_kernel(const LaunchArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    unsigned long long count = 0;
    if (!a.narrow) {
        count = min(*a.handed, (unsigned long long)a.straggler_cap);
        if (blockIdx.x * (blockDim.x >> 5) >= count) return;
    }
    unsigned char *mine = smem + (size_t)(threadIdx.x >> 5) * (narrow_memory_bytes(sizeof(P) == 8) + a.region_bytes);
    NarrowMemory<P> &mem = *reinterpret_cast<NarrowMemory<P> *>(mine);
    unsigned char *region = mine + narrow_memory_bytes(sizeof(P) == 8);
    WarpFeed *feed = &mem.feed;
    for (int i = lane; i < a.region_bytes / 8; i += 32) reinterpret_cast<unsigned long long *>(region)[i] = 0ull;
    if (lane == 0) *feed = WarpFeed{0, 0, 0, 0, 0, {-1, -1}, {0, 0}, {0, 0}, -1, 0, 0, 0, 0};
    load_math_tables<P>(threadIdx.x, blockDim.x);
    if constexpr (sizeof(P) == 8) __syncthreads();
    __syncwarp();

    int key_case = -1;  // the region's (case, batch)
    uint32_t key_batch = 0, fed = 0, deposited = 0;
    // flights still to be scored, one in each lane below `held`
    P x0 = P(0), x1 = P(0), l = P(0), fw = P(0), fiw = P(0);
    int held = 0;
    auto score_held = [&]() {
        Flight<P> f;
        f.k0 = 0;
        f.k1 = -1;
        if (lane < held) plan_flight(f, a.cases[key_case], x0, x1, l, fw, fiw, false);
        deposited += warp_deposit<P>(region, a.region_bytes, a.t, 0, key_case, key_batch, f, lane);
        held = 0;
        if constexpr (sizeof(P) == 8) {  // before a bin's sum can outgrow its 64 bits
            if (__any_sync(CLS_FULL_MASK, deposited >= kDepositBound)) {
                __syncwarp();
                flush_region<P>(region, a, key_case, key_batch, lane, false);
                deposited = 0;
            }
        }
    };
    while (true) {
        // the next history: all lanes hold its state
        History<P> s;
        int lcase;
        uint32_t lbatch, base_j, base_events;
        if (a.narrow) {
            if (feed->pos == feed->pos_end && !claim(feed, a, lane)) break;
            const RunCase &rc = a.runs[feed->piece / a.pieces_per_run];
            const uint64_t pos = feed->pos;
            __syncwarp();
            if (lane == 0) feed->pos = pos + 1;
            __syncwarp();
            lcase = rc.case_index;
            lbatch = (uint32_t)(pos / rc.batch_len);
            source<P, G>(s, a.cases[lcase], a.rk, rc.first + pos);
            base_j = s.j;
            base_events = 0;
        } else {
            unsigned long long i;
            if (lane == 0) i = atomicAdd(a.taken, 1ull);
            i = __shfl_sync(CLS_FULL_MASK, i, 0);
            if (i >= count) break;
            const Straggler<P> &t = *reinterpret_cast<const Straggler<P> *>(a.stragglers + (size_t)i * kStragglerBytes);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                s.r[q] = t.r[q];
                s.w[q] = t.w[q];
            }
            s.iw[0] = t.iw;
            s.track0 = t.track0;
            s.track1 = t.track1;
            s.key = t.key;
            s.j = t.j;
            s.events = t.events;
            s.n_int = t.n_int;
            s.m = (int)t.m;
            lcase = (int)t.lcase;
            lbatch = t.lbatch;
            base_j = t.base_j;
            base_events = t.base_events;
        }
        if constexpr (sizeof(P) == 8) {
            s.iw[1] = recip_or_inf(s.w[1]);
            s.iw[2] = recip_or_inf(s.w[2]);
        }
        if (key_case != lcase || key_batch != lbatch) {
            if (held > 0) score_held();
            __syncwarp();
            if (key_case >= 0) flush_region<P>(region, a, key_case, key_batch, lane, key_case != lcase);
            key_case = lcase;
            key_batch = lbatch;
        }
        const CaseRegs<P> cp = load_case<P>(a.cases[lcase]);
        uint32_t base = s.j & ~1u, top = 0;  // draws base .. top - 1 are in the buffer
        int ev = -1;
        while (ev < 0) {
            if (s.j + 5u > top) {  // an event takes up to five draws
                base = s.j & ~1u;
                top = base + 64u;
                __syncwarp();
                fill_draws<P, G>(mem.draws, 2 * lane, (base >> 1) + lane, s, a.rk);
                __syncwarp();
            }
            NarrowDraws<P, G> draws;
            draws.fetch(mem.draws, (int)(s.j - base));
            Flight<P> f;
            draws.l = P(0);
            ev = step<P, false, G>(s, cp, draws, a.max_events, f, nullptr, false);
            // the flight waits in one lane's registers until 32 are scored together
            if (lane == held) {
                x0 = draws.x0;
                x1 = draws.x1;
                l = draws.l;
                fw = draws.fw;
                fiw = draws.fiw;
            }
            if (++held == 32) score_held();
        }
        // the event tracker's regions sum t^2 in FP64: so its stragglers', in FP32,
        // go straight to the FP64 statistics
        if (lane == 0)
            end_history<P, G>(region, a, s, ev, sizeof(P) == 4 && a.bank != nullptr ? 2 : 0, lcase, base_j, base_events, lane);
        __syncwarp();
        if (sizeof(P) == 4 && ++fed >= a.flush_every) {  // FP32: before a bin's sum can outgrow its 64 bits
            if (held > 0) score_held();
            __syncwarp();
            flush_region<P>(region, a, key_case, key_batch, lane);
            fed = 0;
        }
    }
    if (held > 0) score_held();
    __syncwarp();
    if (key_case >= 0) flush_region<P>(region, a, key_case, key_batch, lane);
}

// ------------------------------------------------------------ trace kernel
template <typename P>
__global__ void trace_kernel(const TraceArgs a) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const CaseParams &cp = a.cases[a.case_index];
    const RoundKeys key = make_round_keys(a.seed);
    load_math_tables<P>(0, 1);
    History<P> s;
    Flight<P> f;
    source<P>(s, cp, key, a.history);
    TraceSink tr{a.rows, a.cap, 0};
    PhiloxDraws<P, 0, false> draws{key};
    while (step<P, true, 0>(s, cp, draws, a.max_events, f, &tr) < 0) {
    }
    *a.n_rows = tr.n;
}

}  // namespace cls
