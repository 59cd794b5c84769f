// field.cuh -- device arithmetic in F_p, p = 2^61 - 1 (Sec. 6.1 of the paper:
// a Mersenne prime, so reduction is shifts and masks; Sec. 5.1.4: a product
// costs a few machine multiplies).  Every value handled here is canonical,
// i.e. in [0, p).
#pragma once
#include <stdint.h>

typedef uint64_t u64;
typedef unsigned int u32;

#define FP_P 0x1FFFFFFFFFFFFFFFull

__host__ __device__ __forceinline__ u64 f_add(u64 a, u64 b)
{
    u64 s = a + b;  // < 2^62, no wrap
    return s >= FP_P ? s - FP_P : s;
}

__host__ __device__ __forceinline__ u64 f_sub(u64 a, u64 b)
{
    return a >= b ? a - b : a + (FP_P - b);
}

__host__ __device__ __forceinline__ u64 f_neg(u64 a) { return a ? FP_P - a : 0; }

// 2a - b, the value at t = 2 of the line through (0, b) and (1, a).
__host__ __device__ __forceinline__ u64 f_ext2(u64 a1, u64 a0) { return f_sub(f_add(a1, a1), a0); }

// Product with 32-bit limbs.  a = a1 2^32 + a0 with a1, b1 < 2^29 (canonical
// inputs), so
//   a b = a1 b1 2^64 + (a1 b0 + a0 b1) 2^32 + a0 b0,   mid = a1 b0 + a0 b1 < 2^62.
// Using 2^61 = 1 and 2^64 = 8 (mod p):
//   mid 2^32 = (mid >> 29) 2^61 + (mid mod 2^29) 2^32 = (mid >> 29) + (mid mod 2^29) 2^32,
//   a0 b0    = (a0 b0 mod 2^61) + (a0 b0 >> 61).
// The five terms sum to less than 3 2^61 + 2^34 < 2^63; one more fold leaves
// a value below p + 4, and one conditional subtraction makes it canonical.
__device__ __forceinline__ u64 f_mul(u64 a, u64 b)
{
    const u32 a0 = (u32)a, a1 = (u32)(a >> 32);
    const u32 b0 = (u32)b, b1 = (u32)(b >> 32);
    const u64 lo = (u64)a0 * b0;
    const u64 mid = (u64)a1 * b0 + (u64)a0 * b1;
    const u64 hi = (u64)a1 * b1;
    u64 s = (hi << 3) + (mid >> 29) + ((mid & 0x1FFFFFFFull) << 32) + (lo & FP_P) + (lo >> 61);
    s = (s & FP_P) + (s >> 61);
    return s >= FP_P ? s - FP_P : s;
}

// Product with a full 64x64 -> 128 multiply and one Mersenne fold:
// a b = hi 2^64 + lo, (a b) mod 2^61 = lo & p, (a b) >> 61 = (hi << 3) | (lo >> 61);
// both parts are below p because a b <= (p-1)^2 < p 2^61, so one conditional
// subtraction suffices.
__device__ __forceinline__ u64 f_mul_wide(u64 a, u64 b)
{
    const u64 lo = a * b;
    const u64 hi = __umul64hi(a, b);
    u64 s = (lo & FP_P) + ((lo >> 61) | (hi << 3));
    return s >= FP_P ? s - FP_P : s;
}

// Host-side product for plan-time constants (never on the proof path).
static inline u64 h_mul(u64 a, u64 b)
{
    unsigned __int128 x = (unsigned __int128)a * b;
    u64 s = (u64)(x & FP_P) + (u64)(x >> 61);
    return s >= FP_P ? s - FP_P : s;
}

// Sum of a and b where both are canonical: lazy-free add used in reductions.
__device__ __forceinline__ u64 f_add3(u64 a, u64 b, u64 c) { return f_add(f_add(a, b), c); }

// Fermat inverse a^(p-2) (a != 0): p - 2 = 4 (2^59 - 1) + 1, with a^(2^59 - 1)
// by the addition chain 1, 2, 3, 6, 7, 14, 28, 29, 58, 59 on the exponents'
// lengths: 60 squarings and 10 products one after another, where
// square-and-multiply takes 120 (almost every bit of p - 2 is set).
__device__ __forceinline__ u64 f_sqn(u64 x, int n)
{
#pragma unroll 1
    for (int k = 0; k < n; k++) x = f_mul_wide(x, x);
    return x;
}

__device__ __forceinline__ u64 f_inv(u64 a)
{
    const u64 x2 = f_mul_wide(f_sqn(a, 1), a), x3 = f_mul_wide(f_sqn(x2, 1), a);
    const u64 x6 = f_mul_wide(f_sqn(x3, 3), x3), x7 = f_mul_wide(f_sqn(x6, 1), a);
    const u64 x14 = f_mul_wide(f_sqn(x7, 7), x7), x28 = f_mul_wide(f_sqn(x14, 14), x14);
    const u64 x29 = f_mul_wide(f_sqn(x28, 1), a), x58 = f_mul_wide(f_sqn(x29, 29), x29);
    const u64 x59 = f_mul_wide(f_sqn(x58, 1), a);
    return f_mul_wide(f_sqn(x59, 2), a);
}

// 1/2 = 2^60 mod p, since 2 * 2^60 = 2^61 = 1.
#define FP_INV2 0x1000000000000000ull

// splitmix64 (Steele, Lea, Flood 2014): output number k (k >= 1) of the
// generator started at `seed` is mix(seed + k * gamma).
__device__ __forceinline__ u64 splitmix64_at(u64 seed, u64 k)
{
    u64 z = seed + k * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Warp-wide field sum (all 32 lanes participate).
__device__ __forceinline__ u64 warp_sum(u64 v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = f_add(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ---- Lazy arithmetic: values in W = [0, 2^61 + 8) ("weakly reduced"). -------
// Canonical values are in W; only transcript entries must be canonical.

// Any 64-bit x -> W, congruent mod p (2^61 = 1).
__device__ __forceinline__ u64 wred(u64 x) { return (x & FP_P) + (x >> 61); }

// W -> canonical.
__device__ __forceinline__ u64 wcanon(u64 w) { return w >= FP_P ? w - FP_P : w; }

// 128-bit accumulator of products of W values (at most 64 products).
struct acc128 {
    u64 lo, hi;
};

__device__ __forceinline__ void acc_zero(acc128 &a) { a.lo = 0; a.hi = 0; }

// a += x y (exact 128-bit multiply-add).  Left to the compiler as one 128-bit
// expression it shares the four 32x32 products between the halves: 26.5
// cycles a warp and scheduler against 32.9 for a 64-bit mad.lo / madc.hi pair.
__device__ __forceinline__ void mac(acc128 &a, u64 x, u64 y)
{
    const unsigned __int128 s = (((unsigned __int128)a.hi << 64) | a.lo) + (unsigned __int128)x * y;
    a.lo = (u64)s;
    a.hi = (u64)(s >> 64);
}

// a += x (x < 2^64).
__device__ __forceinline__ void acc_add(acc128 &a, u64 x)
{
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, 0;" : "+l"(a.lo), "+l"(a.hi) : "l"(x));
}

// hi 2^64 + lo -> W: 2^64 = 8 (mod p), and 8 hi = (hi >> 58) 2^61 + (8 hi mod 2^61).
__device__ __forceinline__ u64 acc_red(const acc128 &a)
{
    const u64 t = (a.lo & FP_P) + (a.lo >> 61) + ((a.hi << 3) & FP_P) + (a.hi >> 58);
    return wred(t);
}

// The same for a below 7 * 2^122 (six products of W values and a 64-bit
// term): a = (a div 2^61) 2^61 + (a mod 2^61), and the quotient, below
// 7 * 2^61, is one funnel shift: half of acc_red's instructions.
__device__ __forceinline__ u64 acc_red7(const acc128 &a)
{
    return wred((a.lo & FP_P) + ((a.hi << 3) | (a.lo >> 61)));
}

// Product of two values whose product is below 7 * 2^122 (W values, or
// one below 2^63 and one canonical), result in W.
__device__ __forceinline__ u64 wmul(u64 x, u64 y)
{
    acc128 a;
    a.lo = x * y;
    a.hi = __umul64hi(x, y);
    return acc_red7(a);
}

// u0 + a d for u0 in W, d < 1.5 2^62 (a lazy difference u1 + 2p - u0 of W
// values) and canonical a.  The exact product is below 1.5 2^123, so u0, its
// remainder and its quotient add up below 2^64 and are reduced once.  (In 31-
// and 30-bit limbs the same took half as many instructions again.)
__device__ __forceinline__ u64 wlin1(u64 u0, u64 d, u64 a)
{
    const unsigned __int128 t = (unsigned __int128)a * d;
    const u64 lo = (u64)t, hi = (u64)(t >> 64);
    return wred(u0 + (lo & FP_P) + ((hi << 3) | (lo >> 61)));
}

// u0 + r (u1 - u0) for u0, u1 in W and canonical r.
__device__ __forceinline__ u64 wfold(u64 u0, u64 u1, u64 r) { return wlin1(u0, u1 + (2 * FP_P) - u0, r); }

// u0 + a d + b e (d, e < 1.5 2^62; a, b canonical): below 3 2^123 + 2^62.
__device__ __forceinline__ u64 wlin2(u64 u0, u64 d, u64 e, u64 a, u64 b)
{
    acc128 t;
    t.lo = u0;
    t.hi = 0;
    mac(t, a, d);
    mac(t, b, e);
    return acc_red7(t);
}

// Inclusive product scan over the warp (lane l gets prod_{j<=l} x_j).
__device__ __forceinline__ u64 warp_scan_mul(u64 x)
{
    const u32 lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (u32)o) x = f_mul(x, y);
    }
    return x;
}

// Inclusive suffix product scan (lane l gets prod_{j>=l} x_j).
__device__ __forceinline__ u64 warp_rscan_mul(u64 x)
{
    const u32 lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 y = __shfl_down_sync(0xffffffffu, x, o);
        if (lane + o < 32) x = f_mul(x, y);
    }
    return x;
}

// Product over the warp of one canonical value per lane.
__device__ __forceinline__ u64 warp_prod(u64 x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = f_mul(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// Warp-wide sum of one W value per lane -> W (a sum of four W values stays
// below 2^64, so reduce every two steps).
__device__ __forceinline__ u64 warp_wsum(u64 x)
{
    x += __shfl_xor_sync(0xffffffffu, x, 16);
    x += __shfl_xor_sync(0xffffffffu, x, 8);
    x = wred(x);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x = wred(x);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return wred(x);
}

// Warp-wide sums of n records of NV values in W (record q at part[q NV ..]):
// the lanes take every 32nd record, FN_U records' loads in flight per lane
// before any is added (the reductions over hundreds of per-CTA partials are
// load-latency bound).  h[t] (t < NV) = the canonical total of value t, in every lane.
#define FN_U 8
static_assert(FN_U == 8, "warp_record_sums adds its loads in two quarter-sums of four");
template <int NV>
__device__ __forceinline__ void warp_record_sums(const u64 *__restrict__ part, u32 n, u32 lane, u64 *h)
{
    u64 acc[NV];
#pragma unroll
    for (int t = 0; t < NV; t++) acc[t] = 0;
    for (u32 q0 = lane; q0 < n; q0 += 32 * FN_U) {
        u64 x[FN_U][NV];
#pragma unroll
        for (int u = 0; u < FN_U; u++) {
            const u32 q = q0 + 32 * u;
#pragma unroll
            for (int t = 0; t < NV; t++) x[u][t] = q < n ? part[(u64)q * NV + t] : 0;
        }
#pragma unroll
        for (int t = 0; t < NV; t++) {
            // four W values sum below 2^64; wred brings each quarter-sum back to W
            const u64 lo = wred(x[0][t] + x[1][t] + x[2][t] + x[3][t]);
            const u64 hi = wred(x[4][t] + x[5][t] + x[6][t] + x[7][t]);
            acc[t] = wred(acc[t] + lo + hi);
        }
    }
#pragma unroll
    for (int t = 0; t < NV; t++) h[t] = wcanon(warp_wsum(acc[t]));
}

