// coins.cuh -- the verifier's coins as functions of the seed, for any CTA
// that needs some (Sec. 3.1: the verifier's challenges are random field
// elements; here challenge c is the (c+1)-th accepted draw of splitmix64
// seeded with the proof seed, a draw equal to p being rejected).
#pragma once
#include "plan.h"

// Any rejected draw among the circuit's first nchal draws.  Draw k is p when
// the generator's output mix(seed + k gamma) has p in its upper 61 bits: one
// of eight outputs.  mix is a bijection, so each comes from one state z
// (mix(z) = 8 p + i) and from one k = (z - seed) / gamma mod 2^64: eight
// products instead of a pass over all the draws (3,200 for F0 over 2^16
// inputs), which every CTA that needs a coin would repeat.
__device__ __forceinline__ bool draws_rejected(const Globals &G)
{
    constexpr u64 z[8] = {0xF4FF78D94E358EDEull, 0x5337A8FA26C3E7E1ull, 0x0FD7855AD0F929D7ull, 0xF27A2DEE32FF7CD7ull,
                          0x02EF6E7444219FC4ull, 0x926590AA01CA8B12ull, 0xED4850B928DC8E2Cull, 0xCF9A04AFFA6BADC0ull};
    bool r = false;
#pragma unroll
    for (int i = 0; i < 8; i++) r |= (z[i] - G.seed) * 0xF1DE83E19937733Dull - 1 < (u64)G.nchal;
    return r;
}

// Challenge c when a draw was rejected, by walking the stream (kept out of
// line: the coin kernels are short enough for instruction fetches to count).
static __device__ __noinline__ u64 chal_slow(u64 seed, u32 c)
{
    u64 k = 1;
    for (u32 got = 0;;) {
        const u64 x = splitmix64_at(seed, k++) >> 3;
        if (x == FP_P) continue;
        if (got == c) return x;
        got++;
    }
}

// Challenge c: the (c+1)-th accepted draw.
__device__ __forceinline__ u64 chal_of(const Globals &G, bool rej, u32 c)
{
    if (!rej) return splitmix64_at(G.seed, (u64)c + 1) >> 3;
    return chal_slow(G.seed, c);
}

// Coordinate k of z_layer: z_0 = the first s_0 challenges; z_{i+1} =
// r1 + tau (r2 - r1) of layer i's line (r1, r2: its phase-2/3 challenges).
__device__ __forceinline__ u64 zcoord(const Globals &G, bool rej, u32 layer, u32 k)
{
    if (layer == 0) return chal_of(G, rej, k);
    const LayerDev &L = G.layers[layer - 1];
    const u32 co = L.chal_off, s = L.s, sn = L.sn;
    const u64 tau = chal_of(G, rej, co + s + 2 * sn);
    const u64 r1 = chal_of(G, rej, co + s + k), r2 = chal_of(G, rej, co + s + sn + k);
    return f_add(r1, f_mul(tau, f_sub(r2, r1)));
}

