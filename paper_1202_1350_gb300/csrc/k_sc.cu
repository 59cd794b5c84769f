// k_sc.cu -- sum-check waves of the prover (Sec. 4.1.1 of the paper: every
// message is a field sum of independent per-gate contributions; Sec. 3.1:
// messages are degree-2 polynomials given by their values at 0, 1, 2).
//
// Each sum-check instance (SCI) sums P(x) V(x) + B(x) over n variables bound
// low bit first.  Two kinds of instance:
//
//  * product-weighted (PROD): P(x) = sigma prod_m L_m(x_m) with linear factors
//    L_m(b) = c0_m (1-b) + c1_m b, B = gamma-multiple of P.  Folding P keeps the
//    product form, so P is never stored: round j's message is
//      g_j(t) = kappa_j L_j(t) h_j(t),  h_j(t) = sum_y E_j(y) V_j(t, y),
//    with kappa_j = sigma prod_{m<j} L_m(r_m), E_j(y) = prod_{m>j} L_m(y_m) and
//    V_j the value table folded with r_0..r_{j-1}; h_j is linear in t, so only
//    h_j(0), h_j(1) are summed.  Used for phase 1 of every layer (P = eq(z_i,
//    .)), phase 2 of TREE layers and phase 3 of every structured kind.
//  * general (GEN): P, V, B are tables folded every round; the message needs
//    P(t)V(t) + B(t) at t = 0, 1, 2.  Chunks sum the values at 0 and 1 and the
//    leading coefficient (P1 - P0)(V1 - V0) of each pair, which shares its
//    differences with the folds; k_final turns the three sums into the value
//    at 2.  The first wave forms P and B from the wiring on the fly (phase 2 of
//    SQUARE, F0 and MATMULT layers) or reads tables built by k_build23.
//
// Arithmetic is lazy: table values stay in W = [0, 2^61 + 8), products
// accumulate exactly in 128 bits and are reduced once per round per thread;
// only transcript entries are made canonical.
#include <cuda_runtime.h>

#include <algorithm>

#include "plan.h"

// --------------------------------------------------------------------------------
// Shared helpers
// --------------------------------------------------------------------------------

// Sum over the warp of 16 values per lane: afterwards lane l holds the total of
// value index l >> 1.  Inputs in W; sums are brought back to W every two
// halving steps (a sum of four W values is below 2^64).
__device__ __forceinline__ u64 warp_sum16(u64 (&v)[16])
{
    const u32 lane = threadIdx.x & 31;
#pragma unroll
    for (int step = 0; step < 4; step++) {
        const int o = 16 >> step, half = 8 >> step;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; i++) {
            const u64 send = up ? v[i] : v[i + half];
            const u64 keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            if (step & 1) v[i] = wred(v[i]);
        }
    }
    u64 r = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
    return wred(r);
}

// (The per-wave weight tables of the PROD waves are built with the coins, in
// k_coins.cu.)


// --------------------------------------------------------------------------------
// One persistent launch for the waves of every instance: CTAs of WV_NT threads
// take tasks (one chunk of one line, PROD or GEN wave) from a shared counter,
// so the whole device stays busy until the last task; a wave whose successor
// is a single chunk runs that successor in the CTA that finishes the wave's
// last chunk (no CTA ever waits for another).
// --------------------------------------------------------------------------------

#define WV_NT 128

#ifndef PR_RING
#define PR_RING 4  // rows per thread in flight
#endif

struct ProdSmem {
    union {
        ulonglong2 ring[PR_RING][4][WV_NT];  // each thread's entries of its next rows (its own copies)
        u64 u[8][1 << PR_C];                 // row groups' column sums
    };
    u64 f[8][(1 << PR_R) + 1];   // column groups' row sums
    u64 rw[1 << PR_R];
    u64 U[1 << PR_C], F[1 << PR_R];
};

struct GenSmem {
    u64 r[32];
    u64 lvl[3];
    u64 w[WV_NT / 32][16];  // per-warp sums of the in-register rounds
    u64 hs[9][WV_NT];       // per-thread sums of in-register rounds 2..4 (kept out of registers)
    u64 pend[9][WV_NT];     // triples waiting for their partner in rounds 2..4
    u64 x[3][WV_NT];        // the threads' folded triples
    u64 c[3][WV_NT + 4];    // cross rounds' pair terms: round kk's at 2 (64 - (64 >> kk)) ..
};

struct LineSmem {
    u64 a[8], b[8];          // a_k and b_k of the coordinates folded in registers
    // the threads' polynomials, coefficient c in row c, then their products'
    // (a row length that spreads the sum's reads over the banks)
    u64 part[32][WV_NT + 4];
    u64 res[32];
};

union WaveSmem {
    ProdSmem prod;
    GenSmem gen;
    LineSmem line;
};

extern __shared__ __align__(16) unsigned char wv_dyn[];  // a WaveSmem

// Load of a wave's input.  A first wave's input (layer values, or tables built
// by an earlier launch) is read-only for the whole launch and goes through
// L1, where the prefetch of the next run lands; a later wave's input is
// written by other CTAs of this launch and is read through L2.
__device__ __forceinline__ ulonglong2 ld_in(const ulonglong2 *p, bool ext) { return ext ? __ldg(p) : __ldcg(p); }
__device__ __forceinline__ u64 ld_in(const u64 *p, bool ext) { return ext ? __ldg(p) : __ldcg(p); }

// Four entries of a first wave's values, a whole sector in one load (p 32-byte
// aligned: a layer's values are, and runs are multiples of four): half the load
// instructions (F2 2^22 212 -> 210 us).
__device__ __forceinline__ void ldg4(const u64 *p, u64 &a, u64 &b, u64 &c, u64 &d)
{
    asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
}

// Asynchronous copies to shared memory: 16 bytes through L2 (also what other
// CTAs of this launch wrote), or 8 bytes through L1 (a first wave's input).
__device__ __forceinline__ void cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((u32)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
// The same through L1, for values in host memory: copies that bypass it took
// every sector across the link twice (F2 2^20: 4.19 M sectors read by the wave
// launch, 2.91 M needed; 915 us a proof, so 740).
__device__ __forceinline__ void cp16_l1(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((u32)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((u32)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Bring the line holding p into L1 ahead of its load (no register cost).
__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// The next task of the CTA (thread 0; ctr NULL: the CTA keeps the one it has).
__device__ __forceinline__ int claim_task(u32 *ctr)
{
    return (ctr && threadIdx.x == 0) ? (int)(gridDim.x + atomicAdd(ctr, 1u)) : 0;
}

// ---- PROD -----------------------------------------------------------------------
//
// Every message sum and the fold of a product-weighted chunk are linear in
// its entries, with weights that are products over the coordinates.  So a
// chunk of 2^kr rows of 2^7 columns is read once, with two multiply-adds
// per entry: U[x] = sum_row roww[row] V[row, x] holds all that the rounds of
// the column coordinates need (their sums over the rows are weighted alike),
// F[row] = sum_x colw[x] V[row, x] is the table folded by those rounds, on
// which the row coordinates' rounds run.  The rounds of either vector are
// then independent sums too (vec_rounds), one step instead of a chain of
// folds.  Folding round by round took three products an entry, a reduction
// and a fold per pair, and a chain of up to 13 dependent rounds.

// The sums of every round of a vector of 2^kk entries in shared memory (kk <=
// 7): thread 16 j + p takes round j's pairs p, p + 16, ..; w: its weights.
// Afterwards lanes p = 0..7 hold the round's sum at 0 and lanes 8..15 that at 1.
__device__ __forceinline__ u64 vec_rounds(const u64 *v, u32 kk, const u64 (&w)[4])
{
    const u32 j = threadIdx.x >> 4, p = threadIdx.x & 15;
    acc128 a0, a1;
    acc_zero(a0);
    acc_zero(a1);
    if (j < kk) {
        const u32 half = 1u << (kk - 1), bit = 1u << j;
#pragma unroll
        for (u32 i = 0; i < 4; i++) {
            const u32 y = p + 16 * i;
            if (y < half) {
                const u32 x = ((y & ~(bit - 1)) << 1) | (y & (bit - 1));
                mac(a0, w[i], v[x]);
                mac(a1, w[i], v[x | bit]);
            }
        }
    }
    // sixteen lanes' sums; the lanes' halves part after the first exchange
    const bool up = (p & 8) != 0;
    const u64 h0 = acc_red7(a0), h1 = acc_red7(a1);
    u64 h = (up ? h1 : h0) + __shfl_xor_sync(0xffffffffu, up ? h0 : h1, 8);
    h += __shfl_xor_sync(0xffffffffu, h, 4);
    h = wred(h);
    h += __shfl_xor_sync(0xffffffffu, h, 2);
    h += __shfl_xor_sync(0xffffffffu, h, 1);
    return wred(h);
}

// A thread's weights for vec_rounds.
__device__ __forceinline__ void vec_weights(const u64 *T, u32 kk, bool use, u64 (&w)[4])
{
#pragma unroll
    for (u32 i = 0; i < 4; i++)
        w[i] = (use && threadIdx.x < 16 * kk && i < vec_slots(kk)) ? __ldg(T + i * 16 * kk + threadIdx.x) : 0;
}

// One chunk of a PROD wave (each kind is a function of its own: its registers
// are allocated without those of the others, and there is one copy of its code).
__device__ __noinline__ int prod_chunk(const ProdWave &W, u32 chunk, u32 *ctr)
{
    ProdSmem &sm = reinterpret_cast<WaveSmem *>(wv_dyn)->prod;
    const u32 tid = threadIdx.x;
    const u32 nr = W.nr, kc = W.kc, kr = W.kr, nchunks = W.nchunks;
    const bool ext = W.r0 == 0, odd = (W.flags & WF_ODD) != 0;
    const u64 *blk = W.wblk;
    const u64 *in = W.in + ((u64)chunk << (odd ? nr + 1 : nr));
    // columns 2c + 32 q, + 1 of rows rg, rg + 8, .., each thread's next
    // PR_RING rows on their way into shared memory while it works: an L2 load
    // takes about two rows' products
    const u32 c = tid & 15, rg = tid >> 4, nrow = kr ? 1u << kr : 0u;
    auto fetch = [&](u32 row) {
        if (row < nrow) {
            ulonglong2 *dst = &sm.ring[(row >> 3) & (PR_RING - 1)][0][tid];
            const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(in);
            if (odd) {
                src += 2 * (row * 64 + c);
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    cp8(&dst[q * WV_NT].x, &src[32 * q].y);
                    cp8(&dst[q * WV_NT].y, &src[32 * q + 1].y);
                }
            } else if (W.flags & WF_HOST) {
                src += row * 64 + c;
#pragma unroll
                for (int q = 0; q < 4; q++) cp16_l1(&dst[q * WV_NT], &src[16 * q]);
            } else {
                src += row * 64 + c;
#pragma unroll
                for (int q = 0; q < 4; q++) cp16(&dst[q * WV_NT], &src[16 * q]);
            }
        }
        cp_commit();
    };
    if (kr) {
#pragma unroll
        for (u32 i = 0; i < PR_RING; i++) fetch(rg + 8 * i);
        if (tid < nrow) sm.rw[tid] = __ldg(blk + pw_roww(kr) + tid);
    }
    u64 wc[4], wr[4];
    vec_weights(blk + pw_tcol(kr), kc, true, wc);
    vec_weights(blk + pw_trow(kc, kr), kr, kr != 0, wr);
    const u64 *olo = blk + pw_outer(kc, kr);  // weight of the coordinates beyond the chunk
    const u64 ea = __ldg(olo + (chunk & ((1u << W.ho) - 1))), eb = __ldg(olo + (1u << W.ho) + (chunk >> W.ho));
    // fold factor of the last coordinate
    const u64 el = __ldg(blk + pw_last(kc, kr) + (kr ? 2 : 0) + ((tid >> 3) & 1));
    if (kr == 0) {
        if (tid < (1u << kc)) sm.U[tid] = ld_in(in + (odd ? 2 * tid + 1 : tid), ext);
        __syncthreads();
    } else {
        ulonglong2 cw[4];
#pragma unroll
        for (int q = 0; q < 4; q++) cw[q] = __ldg(reinterpret_cast<const ulonglong2 *>(blk) + c + 16 * q);
        acc128 u[8];
#pragma unroll
        for (int q = 0; q < 8; q++) acc_zero(u[q]);
        __syncthreads();  // sm.rw
#pragma unroll 1
        for (u32 row = rg; row < nrow; row += 8) {
            cp_wait<PR_RING - 1>();
            const ulonglong2 *src = &sm.ring[(row >> 3) & (PR_RING - 1)][0][tid];
            ulonglong2 v[4];
#pragma unroll
            for (int q = 0; q < 4; q++) v[q] = src[q * WV_NT];
            const u64 rw = sm.rw[row];
            fetch(row + 8 * PR_RING);
            acc128 f0, f1;
            acc_zero(f0);
            acc_zero(f1);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                mac(f0, cw[q].x, v[q].x);
                mac(f1, cw[q].y, v[q].y);
                mac(u[2 * q], rw, v[q].x);
                mac(u[2 * q + 1], rw, v[q].y);
            }
            u64 f = wred(acc_red7(f0) + acc_red7(f1));
            f = wred(f + __shfl_xor_sync(0xFFFFu << (tid & 16), f, 1));  // (half a warp has the same rows)
            if (!(c & 1)) sm.f[c >> 1][row] = f;
        }
        cp_wait<0>();
        __syncthreads();  // the ring's memory becomes sm.u
#pragma unroll
        for (int q = 0; q < 4; q++)
            *reinterpret_cast<ulonglong2 *>(&sm.u[rg][2 * c + 32 * q]) =
                make_ulonglong2(acc_red(u[2 * q]), acc_red(u[2 * q + 1]));
        __syncthreads();
        {
            const u64 a = wred(sm.u[0][tid] + sm.u[1][tid] + sm.u[2][tid] + sm.u[3][tid]);
            const u64 b = wred(sm.u[4][tid] + sm.u[5][tid] + sm.u[6][tid] + sm.u[7][tid]);
            sm.U[tid] = wred(a + b);
            const u32 g = (tid & 1) * 4;  // a row's eight sums, four a thread
#pragma unroll 1
            for (u32 row = tid >> 1; row < ((nrow + 63) & ~63u); row += WV_NT / 2) {
                u64 f = 0;
                if (row < nrow) f = wred(sm.f[g][row] + sm.f[g + 1][row] + sm.f[g + 2][row] + sm.f[g + 3][row]);
                f = wred(f + __shfl_xor_sync(0xffffffffu, f, 1));
                if ((tid & 1) == 0 && row < nrow) sm.F[row] = f;
            }
        }
        __syncthreads();
    }
    const int next = claim_task(ctr);
    const u32 j = tid >> 4, t = (tid >> 3) & 1;
    const bool writer = (tid & 7) == 0;
    const u64 ech = f_mul(ea, eb);
    u64 h = vec_rounds(sm.U, kc, wc);
    if (writer && j < kc) W.part[((u64)j * nchunks + chunk) * 2 + t] = wmul(h, ech);
    if (kr) {
        h = vec_rounds(sm.F, kr, wr);
        if (writer && j < kr) W.part[((u64)(kc + j) * nchunks + chunk) * 2 + t] = wmul(h, ech);
    }
    if (!(W.flags & WF_LAST)) {
        // the chunk's value for the next wave: the last round's sums, folded
        const u64 x = wmul(h, el), y = wred(x + __shfl_xor_sync(0xffffffffu, x, 8));
        if (tid == 16 * ((kr ? kr : kc) - 1)) W.out[chunk] = y;
    }
    return next;
}

// ---- GEN ------------------------------------------------------------------------

// N consecutive entries of a GEN wave's P, V, B tables at x0 (tables built
// by k_build23, or the previous wave's outputs; first waves whose tables follow
// from the wiring form P and B themselves: gen_source, bil_run).
template <int N>
__device__ __forceinline__ void gen_load(const GenWave &W, u64 x0, bool hasB, u64 (&p)[N], u64 (&v)[N], u64 (&b)[N])
{
    const bool ext = W.r0 == 0;
    const ulonglong2 *sv = reinterpret_cast<const ulonglong2 *>(W.inV + x0);
#pragma unroll
    for (int q = 0; q < N / 2; q++) {
        const ulonglong2 t = ld_in(sv + q, ext);
        v[2 * q] = t.x;
        v[2 * q + 1] = t.y;
    }
    const ulonglong2 *sp = reinterpret_cast<const ulonglong2 *>(W.inP + x0);
#pragma unroll
    for (int q = 0; q < N / 2; q++) {
        const ulonglong2 t = ld_in(sp + q, ext);
        p[2 * q] = t.x;
        p[2 * q + 1] = t.y;
    }
    if (hasB) {
        const ulonglong2 *sb = reinterpret_cast<const ulonglong2 *>(W.inB + x0);
#pragma unroll
        for (int q = 0; q < N / 2; q++) {
            const ulonglong2 t = ld_in(sb + q, ext);
            b[2 * q] = t.x;
            b[2 * q + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; q++) b[q] = 0;
    }
}

// One general pair: the message's values at t = 0, 1 (c0, c1) and its
// leading coefficient c2 = (P1 - P0)(V1 - V0), from which the value at 2 is
// 2 c1 - c0 + 2 c2 (B is linear in t); then the folds, which share the
// differences P1 - P0, V1 - V0 (lazy, below 1.5 2^62).  B is zero without hasB
// (uniform).
__device__ __forceinline__ void gen_pair(bool hasB, u64 p0, u64 p1, u64 v0, u64 v1, u64 b0, u64 b1, u64 r, u64 &c0, u64 &c1,
                                         u64 &c2, u64 &pn, u64 &vn, u64 &bn)
{
    const u64 dp = p1 + (2 * FP_P) - p0, dv = v1 + (2 * FP_P) - v0;
    c0 = wmul(p0, v0);
    c1 = wmul(p1, v1);
    c2 = wmul(wred(dp), wred(dv));
    pn = wlin1(p0, dp, r);
    vn = wlin1(v0, dv, r);
    if (hasB) {
        c0 = wred(c0 + b0);
        c1 = wred(c1 + b1);
        bn = wfold(b0, b1, r);
    }
}

// Round k on two folded triples held by one thread, summed into the
// thread's shared-memory slots hs[3j..3j+2].
__device__ __forceinline__ void gen_pair_acc(bool hasB, u64 p0, u64 p1, u64 v0, u64 v1, u64 b0, u64 b1, u64 r, GenSmem &sm,
                                             u32 j, u64 &pn, u64 &vn, u64 &bn)
{
    u64 c0, c1, c2;
    gen_pair(hasB, p0, p1, v0, v1, b0, b1, r, c0, c1, c2, pn, vn, bn);
    const u32 t = threadIdx.x;
    sm.hs[3 * j][t] = wred(sm.hs[3 * j][t] + c0);
    sm.hs[3 * j + 1][t] = wred(sm.hs[3 * j + 1][t] + c1);
    sm.hs[3 * j + 2][t] = wred(sm.hs[3 * j + 2][t] + c2);
}

// A pair of a run, its message sums into the exact accumulators a[0..2] (a
// thread's runs add at most 16 products to each, so they are reduced once at
// the end and not in every run); the folds to p, v.
__device__ __forceinline__ void gen_pair_run(u64 p0, u64 p1, u64 v0, u64 v1, u64 r, acc128 *a, u64 &p, u64 &v)
{
    const u64 dp = p1 + (2 * FP_P) - p0, dv = v1 + (2 * FP_P) - v0;
    mac(a[0], p0, v0);
    mac(a[1], p1, v1);
    mac(a[2], wred(dp), wred(dv));  // leading coefficient (see gen_pair)
    p = wlin1(p0, dp, r);
    v = wlin1(v0, dv, r);
}

// Rounds 0 and 1 of 4 entries held by one thread: sums into a[0..2], a[3..5],
// the folded values to pn, vn, bn (HASB: with B's terms).
template <bool HASB>
__device__ __forceinline__ void gen_run(const u64 (&p)[4], const u64 (&v)[4], const u64 (&b)[4], const GenSmem &sm,
                                        acc128 (&a)[6], u64 &pn, u64 &vn, u64 &bn)
{
    const u64 r0 = sm.r[0], r1 = sm.r[1];
    u64 q0, q1, u0, u1;
    gen_pair_run(p[0], p[1], v[0], v[1], r0, a, q0, u0);
    gen_pair_run(p[2], p[3], v[2], v[3], r0, a, q1, u1);
    gen_pair_run(q0, q1, u0, u1, r1, a + 3, pn, vn);
    if (HASB) {
        acc_add(a[0], b[0] + b[2]);
        acc_add(a[1], b[1] + b[3]);
        const u64 c0 = wfold(b[0], b[1], r0), c1 = wfold(b[2], b[3], r0);
        acc_add(a[3], c0);
        acc_add(a[4], c1);
        bn = wfold(c0, c1, r1);
    }
}

// First waves whose B follows from the wiring too.
__device__ __forceinline__ bool source_b(u32 src) { return src == GS_FIRST2 || src == GS_TREE2; }

// P (and B, for FIRST2 and TREE2) of one entry x of a first wave whose tables
// follow from the wiring (GS_*); v = V[x], vn = V[x with bit 0 cleared] (PAIR2)
// or set (TREE2) (.x: P, .y: B).  The factors come from the wave's own split
// table, whose pointers are there with the descriptor: through the layer's
// they were two more loads, one after another.
__device__ __noinline__ ulonglong2 gen_source(const GenWave &W, u64 x, u64 v, u64 vn)
{
    const u32 src = W.src, th = W.th;
    const bool half = src == GS_FINAL2 || src == GS_TREE2;
    const u64 *lo = W.inP, *hi = W.inB;
    const u64 t = half ? x >> 1 : src == GS_FIRST2 ? 2 * x : x;
    const u64 i = t & ((1ull << th) - 1);
    const u64 h = __ldg(hi + (t >> th));
    u64 p = wmul(__ldg(lo + i), h), b = 0;
    switch (src) {
    case GS_MM2: break;  // (the table ends with n zeros: no weight past the first matrix)
    case GS_SQ2: p = wmul(p, v); break;
    case GS_PAIR2: p = wmul(p, vn); break;
    case GS_FINAL2: p = (x & 1) ? wmul(p, v) : 0; break;
    case GS_TREE2:
        p = (x & 1) ? 0 : p;
        b = wmul(p, vn);
        break;
    default: {  // GS_FIRST2
        const u64 wa = wmul(__ldg(lo + i + 1), h);
        b = wmul(wa, v);
        p = wred(wmul(p, v) + wa);
        break;
    }
    }
    return make_ulonglong2(p, b);
}

// Rounds 0 and 1 of the first wave of a phase-2 instance of an F0_PAIR or
// F0_FINAL layer on two pairs (va, vb) of entries.  With A = w V[2q] (PAIR; w =
// eq(r_P, .) without its coordinate 0, whose value is a = (r_P)_0) or w V[2q+1]
// (FINAL), P[2q + b] is A times a factor of b alone, so round 0's message
// follows from sum A V[2q] and sum A V[2q+1] (a[0], a[1]), and its fold is A
// times a constant, left out here and applied to the later rounds by k_final:
// three products a pair besides w instead of seven.
__device__ __forceinline__ void bil_run(u64 Aa, u64 Ab, ulonglong2 va, ulonglong2 vb, const GenSmem &sm,
                                        acc128 (&a)[6], u64 &pn, u64 &vn)
{
    mac(a[0], Aa, va.x);
    mac(a[0], Ab, vb.x);
    mac(a[1], Aa, va.y);
    mac(a[1], Ab, vb.y);
    const u64 r = sm.r[0];
    gen_pair_run(Aa, Ab, wfold(va.x, va.y, r), wfold(vb.x, vb.y, r), sm.r[1], a + 3, pn, vn);
}

// In-register rounds for e in 2..5: runs of 4 entries (rounds 0, 1), then
// rounds 2.. on the runs' folded triples, combined like a binary counter.  A
// first wave's P (and B) carries a factor lo hi of a split table, and the
// thread's entries share one hi (2^e entries, within one block of the table),
// so they are formed with lo alone and hi multiplies the thread's sums and
// its folded P and B once.
__device__ __forceinline__ void gen_regs_runs(const GenWave &W, u64 x0, u32 e, bool hasB, GenSmem &sm, u64 (&h)[15],
                                              u64 &pv, u64 &vv, u64 &bv)
{
    const u32 nruns = 1u << (e - 2), src = W.src;
    const bool b_run = hasB || source_b(src), half = src == GS_FINAL2 || src == GS_TREE2;
#pragma unroll
    for (int j = 0; j < 9; j++) sm.hs[j][threadIdx.x] = 0;
    acc128 a[6];
#pragma unroll
    for (int j = 0; j < 6; j++) acc_zero(a[j]);
    const u64 *lo = nullptr;
    u64 hi = 1;
    if (src != GS_NONE) {
        const u64 x = half ? x0 >> 1 : src == GS_FIRST2 ? 2 * x0 : x0;
        lo = W.inP + (x & ((1ull << W.th) - 1));
        hi = W.inB[x >> W.th];
    }
    // the second line of each of the thread's tables (32 entries are two)
    // comes while the first is used
    if (nruns > 4) {
        prefetch_l1(W.inV + x0 + 16);
        if (src != GS_NONE) {
            prefetch_l1(lo + (half ? 8 : 16));
        } else {
            prefetch_l1(W.inP + x0 + 16);
            if (hasB) prefetch_l1(W.inB + x0 + 16);
        }
    }
    u64 tp = 0, tv = 0, tb = 0;
    // a rolled loop keeps the kernel small (instruction-cache bound when unrolled)
#pragma unroll 1
    for (u32 sub = 0; sub < nruns; sub++) {
        if (src == GS_PAIR2 || src == GS_FINAL2) {
            u64 w4[4];
            ldg4(W.inV + x0 + 4 * sub, w4[0], w4[1], w4[2], w4[3]);
            const ulonglong2 va = make_ulonglong2(w4[0], w4[1]), vb = make_ulonglong2(w4[2], w4[3]);
            const ulonglong2 *sl = reinterpret_cast<const ulonglong2 *>(lo) + (src == GS_PAIR2 ? 2 * sub : sub);
            ulonglong2 l = __ldg(sl);
            if (src == GS_PAIR2) {
                const ulonglong2 l2 = __ldg(sl + 1);
                l = make_ulonglong2(wmul(l.x + l.y, va.x), wmul(l2.x + l2.y, vb.x));
            } else {
                l = make_ulonglong2(wmul(l.x, va.y), wmul(l.y, vb.y));
            }
            bil_run(l.x, l.y, va, vb, sm, a, tp, tv);
        } else {
            u64 p[4], v[4], b[4];
            if (src == GS_NONE) {
                gen_load<4>(W, x0 + 4 * sub, hasB, p, v, b);
            } else {
                ldg4(W.inV + x0 + 4 * sub, v[0], v[1], v[2], v[3]);
                const ulonglong2 *sl = reinterpret_cast<const ulonglong2 *>(lo) + (src == GS_FIRST2 ? 4 * sub : half ? sub : 2 * sub);
                if (src == GS_FIRST2) {
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const ulonglong2 l = __ldg(sl + q);
                        p[q] = wred(wmul(l.x, v[q]) + l.y);
                        b[q] = wmul(l.y, v[q]);
                    }
                } else if (src == GS_TREE2) {
                    const ulonglong2 l = __ldg(sl);
                    p[0] = l.x, p[1] = 0, p[2] = l.y, p[3] = 0;
                    b[0] = wmul(l.x, v[1]), b[1] = 0, b[2] = wmul(l.y, v[3]), b[3] = 0;
                } else {
                    const ulonglong2 l = __ldg(sl), l2 = __ldg(sl + 1);
                    p[0] = l.x, p[1] = l.y, p[2] = l2.x, p[3] = l2.y;
                    if (src == GS_SQ2) {
#pragma unroll
                        for (int q = 0; q < 4; q++) p[q] = wmul(p[q], v[q]);
                    }
                }
            }
            if (b_run)
                gen_run<true>(p, v, b, sm, a, tp, tv, tb);
            else
                gen_run<false>(p, v, b, sm, a, tp, tv, tb);
        }
        // combined like a binary counter, the pending triples in shared memory
        u32 lv = 0;
#pragma unroll 1
        for (; lv + 2 < e && ((sub >> lv) & 1); lv++) {
            const u64 *q = &sm.pend[3 * lv][threadIdx.x];
            gen_pair_acc(b_run, q[0], tp, q[WV_NT], tv, b_run ? q[2 * WV_NT] : 0, tb, sm.r[2 + lv], sm, lv, tp, tv, tb);
        }
        if (lv + 2 < e) {
            u64 *q = &sm.pend[3 * lv][threadIdx.x];
            q[0] = tp;
            q[WV_NT] = tv;
            if (b_run) q[2 * WV_NT] = tb;
        }
    }
#pragma unroll
    for (int j = 0; j < 6; j++) h[j] = acc_red(a[j]);
#pragma unroll
    for (int j = 0; j < 9; j++) h[6 + j] = sm.hs[j][threadIdx.x];
    if (src != GS_NONE) {  // every sum, P and B are linear in it
#pragma unroll
        for (int j = 0; j < 15; j++) h[j] = wmul(hi, h[j]);
        tp = wmul(hi, tp);
        if (b_run) tb = wmul(hi, tb);
    }
    pv = tp;
    vv = tv;
    bv = tb;
}

// Rounds off.. of a general chunk across threads: the threads' triples meet
// in shared memory, round 0's pairs are taken by two warps, the later rounds
// by one, each pair's terms kept in sm.c and summed once at the end (the four
// warps working every round, and summing it, were a third of a chunk's
// instructions).  The folded triple of the chunk goes to sm.lvl.
__device__ __forceinline__ void gen_cross(bool hasB, u64 p, u64 v, u64 b, u32 off, u32 tid, u32 nr, GenSmem &sm)
{
    const u32 ncross = nr - off;
    sm.x[0][tid] = p;
    sm.x[1][tid] = v;
    if (hasB) sm.x[2][tid] = b;
    __syncthreads();
    u32 base = 0;  // round kk's terms start here
#pragma unroll 1
    for (u32 kk = 0; kk < ncross; kk++) {
        const u32 np = 1u << (ncross - 1 - kk);  // pairs
        if (tid < np) {
            u64 c0, c1, c2;
            b = 0;
            gen_pair(hasB, sm.x[0][2 * tid], sm.x[0][2 * tid + 1], sm.x[1][2 * tid], sm.x[1][2 * tid + 1],
                     hasB ? sm.x[2][2 * tid] : 0, hasB ? sm.x[2][2 * tid + 1] : 0, sm.r[off + kk], c0, c1, c2, p, v, b);
            sm.c[0][base + tid] = c0;
            sm.c[1][base + tid] = c1;
            sm.c[2][base + tid] = c2;
        }
        if (np > 32) __syncthreads();  // two warps read what either wrote
        else if (tid < 32) __syncwarp();
        if (tid < np) {
            sm.x[0][tid] = p;
            sm.x[1][tid] = v;
            if (hasB) sm.x[2][tid] = b;
        }
        if (np > 32) __syncthreads();
        else if (tid < 32) __syncwarp();
        base += np;
    }
    if (tid == 0) {
        sm.lvl[0] = p;
        sm.lvl[1] = v;
        sm.lvl[2] = hasB ? b : 0;
    }
}

// One chunk of a GEN wave.
__device__ __noinline__ int gen_chunk(const Globals &G, const GenWave &W, u32 chunk, u32 *ctr)
{
    GenSmem &sm = reinterpret_cast<WaveSmem *>(wv_dyn)->gen;
    const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const u32 nr = W.nr, e = W.e;
    const u32 na = 1u << (nr - e);
    const u64 base = (u64)chunk << nr;
    const bool hasB = (W.flags & WF_HASB) != 0;
    if (e > 0 && tid < na) prefetch_l1(W.inV + base + ((u64)tid << e));  // while the challenges come
    if (tid < nr) sm.r[tid] = G.chal[W.chal_off + tid];
    __syncthreads();
    u64 pv = 0, vv = 0, bv = 0;
    if (e > 0) {
        u64 h[15];
#pragma unroll
        for (int i = 0; i < 15; i++) h[i] = 0;
        if (tid < na) {
            const u64 x0 = base + ((u64)tid << e);
            gen_regs_runs(W, x0, e, hasB, sm, h, pv, vv, bv);
        }
        u64 h16[16];
#pragma unroll
        for (int i = 0; i < 16; i++) h16[i] = (i < 15) ? h[i] : 0;
        const u64 s = warp_sum16(h16);
        if ((lane & 1) == 0) sm.w[warp][lane >> 1] = s;
    } else if (tid < na) {
        const u64 x = base + tid;
        const bool ext = W.r0 == 0;
        vv = ld_in(W.inV + x, ext);
        if (W.src == GS_NONE) {
            pv = ld_in(W.inP + x, ext);
            bv = hasB ? ld_in(W.inB + x, ext) : 0;
        } else {
            const u64 xn = W.src == GS_TREE2 ? x | 1 : W.src == GS_PAIR2 ? x & ~1ull : x;
            const ulonglong2 t = gen_source(W, x, vv, xn != x ? ld_in(W.inV + xn, ext) : vv);
            pv = t.x;
            bv = t.y;
        }
    }
    const int next = claim_task(ctr);
    gen_cross(hasB || source_b(W.src), pv, vv, bv, e, tid, nr, sm);
    __syncthreads();
    // four threads a value: in-register rounds from the warps' sums, cross
    // rounds from their pairs' terms
    for (u32 o = tid >> 2; o < 3 * nr; o += WV_NT / 4) {
        const u32 k = o / 3, t = o - 3 * k, q = tid & 3;
        u64 s = 0;
        if (k < e) {
            s = sm.w[q][o];
        } else {
            const u32 np = 1u << (nr - 1 - k), first = (1u << (nr - e)) - 2 * np;
            for (u32 i = q; i < np; i += 4) s = wred(s + sm.c[t][first + i]);
        }
        const u32 m = 0xFu << (threadIdx.x & 28);
        s = wred(s + __shfl_xor_sync(m, s, 1));
        s = wred(s + __shfl_xor_sync(m, s, 2));
        if (q == 0) W.part[((u64)k * W.nchunks + chunk) * 3 + t] = s;
    }
    if (!(W.flags & WF_LAST) && tid == 0) {
        W.outP[chunk] = sm.lvl[0];
        W.outV[chunk] = sm.lvl[1];
        if (W.outB) W.outB[chunk] = sm.lvl[2];
    }
    return next;
}

// ---- line reduction -----------------------------------------------------------------
// q(t) = V~_{i+1}(l(t)), folding V_{i+1} with coordinates a_k + b_k t in
// coefficient form (degree grows by one per folded coordinate):
//   out_c = A_c + a (B_c - A_c) + b (B_{c-1} - A_{c-1}),  c = 0 .. deg + 1.
// A first-wave chunk folds e coordinates per thread in registers; the next kk
// are folded in one step, since the result is the sum over the threads of
// their polynomials times weight polynomials that the coins alone fix
// (k_coins): 8 (e + 1) multiply-adds a thread and one sum over the CTA.
// Folding those coordinates level by level through shared memory was half of
// a chunk's time (10 us of 20) and most of a small circuit's.

// One level of coefficient folding in registers: D+1 -> D+2 coefficients.
template <int D>
__device__ __forceinline__ void line_fold(const u64 (&A)[D + 1], const u64 (&B)[D + 1], u64 a, u64 b,
                                          u64 (&out)[D + 2])
{
    u64 d[D + 1];
#pragma unroll
    for (int c = 0; c <= D; c++) d[c] = B[c] + (2 * FP_P) - A[c];
    out[0] = wlin1(A[0], d[0], a);
#pragma unroll
    for (int c = 1; c <= D; c++) out[c] = wlin2(A[c], d[c], d[c - 1], a, b);
    out[D + 1] = wlin1(0, d[D], b);
}

// 8 consecutive entries -> one cubic (coordinates 0, 1, 2 of the run).
__device__ __forceinline__ void line_run8(const u64 *v, const u64 *la, const u64 *lb, u64 (&out)[4])
{
    u64 l1[4][2];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const u64 dd = v[2 * q + 1] + (2 * FP_P) - v[2 * q];
        l1[q][0] = wlin1(v[2 * q], dd, la[0]);
        l1[q][1] = wlin1(0, dd, lb[0]);
    }
    u64 l2[2][3];
    line_fold<1>(l1[0], l1[1], la[1], lb[1], l2[0]);
    line_fold<1>(l1[2], l1[3], la[1], lb[1], l2[1]);
    line_fold<2>(l2[0], l2[1], la[2], lb[2], out);
}

// e coordinates (3..8) of a thread's 2^e consecutive entries: runs of 8
// (cubics over coordinates 0..2), combined like a binary counter over
// coordinates 3, 4, .. (a rolled loop keeps one copy of the run code; from
// coordinate 6 on the pending polynomials wait in sm.part); the polynomial to
// sm.part[0..e][tid].
__device__ __forceinline__ void line_regs(const u64 *entries, u32 e, LineSmem &sm)
{
    const u32 tid = threadIdx.x, nruns = 1u << (e - 3);
    u64 la[3], lb[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        la[k] = sm.a[k];
        lb[k] = sm.b[k];
    }
    u64 c0[4] = {0, 0, 0, 0}, q0[5] = {0, 0, 0, 0, 0}, s0[6] = {0, 0, 0, 0, 0, 0};
    u64 *const dst = &sm.part[0][tid];
    auto store = [](u64 *to, const auto &v) {
#pragma unroll
        for (u32 i = 0; i < sizeof(v) / sizeof(u64); i++) to[i * (WV_NT + 4)] = v[i];
    };
#pragma unroll 1
    for (u32 run = 0; run < nruns; run++) {
        if (!(run & 1) && run + 2 < nruns) prefetch_l1(entries + 8 * (run + 2));  // the next line
        u64 v[8];
        ldg4(entries + 8 * run, v[0], v[1], v[2], v[3]);
        ldg4(entries + 8 * run + 4, v[4], v[5], v[6], v[7]);
        u64 c[4];
        line_run8(v, la, lb, c);
        if (nruns == 1) store(dst, c);
        if (!(run & 1)) {
#pragma unroll
            for (int i = 0; i < 4; i++) c0[i] = c[i];
            continue;
        }
        u64 q[5];
        line_fold<3>(c0, c, sm.a[3], sm.b[3], q);
        if (nruns == 2) store(dst, q);
        if (!(run & 2)) {
#pragma unroll
            for (int i = 0; i < 5; i++) q0[i] = q[i];
            continue;
        }
        u64 t5[6];
        line_fold<4>(q0, q, sm.a[4], sm.b[4], t5);
        if (nruns == 4) store(dst, t5);
        if (!(run & 4)) {
#pragma unroll
            for (int i = 0; i < 6; i++) s0[i] = t5[i];
            continue;
        }
        u64 p[7];
        line_fold<5>(s0, t5, sm.a[5], sm.b[5], p);
        if (nruns == 8) store(dst, p);
        if (!(run & 8)) {
            store(dst, p);
            continue;
        }
        u64 p0[7], p6[8];
#pragma unroll
        for (int i = 0; i < 7; i++) p0[i] = sm.part[i][tid];
        line_fold<6>(p0, p, sm.a[6], sm.b[6], p6);
        if (nruns == 16) store(dst, p6);
        if (!(run & 16)) {
            store(&sm.part[8][tid], p6);
            continue;
        }
        u64 r0[8], p7[9];
#pragma unroll
        for (int i = 0; i < 8; i++) r0[i] = sm.part[8 + i][tid];
        line_fold<7>(r0, p6, sm.a[7], sm.b[7], p7);
        store(dst, p7);
    }
}

// One chunk of one line wave, by the whole CTA.
__device__ __noinline__ int line_chunk(const Globals &G, const LineWaveDev &W, u32 chunk, u32 *ctr)
{
    LineSmem &sm = reinterpret_cast<WaveSmem *>(wv_dyn)->line;
    const u32 tid = threadIdx.x, e = W.e, kk = W.kk, l0 = W.l0;
    const u32 deg0 = l0 + e, C = deg0 + kk + 1;  // a thread's degree; the result's coefficients
    if (tid < e) {
        const u64 a = G.chal[W.a_off + l0 + tid];
        sm.a[tid] = a;
        sm.b[tid] = f_sub(G.chal[W.b_off + l0 + tid], a);
    }
    const bool on = tid < (1u << kk);
    const u64 npoly = (u64)W.nchunks << W.nl;
    const u64 y = ((u64)chunk << kk) + tid;  // the thread's polynomial in the wave's input
    __syncthreads();
    if (e && on) line_regs(W.in + (y << e), e, sm);
    u64 w[8];
#pragma unroll
    for (u32 b = 0; b < 8; b++) w[b] = (on && b <= kk) ? __ldg(W.wt + (b << kk) + tid) : 0;
    // coefficient c of the product is complete once p_c is in: eight
    // accumulators in turn
    acc128 a[8];
#pragma unroll
    for (int i = 0; i < 8; i++) acc_zero(a[i]);
#pragma unroll 1
    for (u32 c0 = 0; c0 < C; c0 += 8) {
#pragma unroll
        for (u32 i = 0; i < 8; i++) {
            const u32 c = c0 + i;
            if (c < C) {
                if (c <= deg0 && on) {
                    const u64 p = e ? sm.part[c][tid] : l0 ? __ldcg(W.in + c * npoly + y) : __ldg(W.in + y);
#pragma unroll
                    for (u32 b = 0; b < 8; b++) mac(a[(i + b) & 7], p, w[b]);
                }
                sm.part[c][tid] = acc_red(a[i]);
                acc_zero(a[i]);
            }
        }
    }
    const int next = claim_task(ctr);
    __syncthreads();
    {
        const u32 c = tid >> 2, q = tid & 3;
        u64 s = 0;
        if (c < C) {
#pragma unroll 1
            for (u32 i = q; i < (1u << kk); i += 8)
                s = wred(s + sm.part[c][i] + (i + 4 < (1u << kk) ? sm.part[c][i + 4] : 0));
        }
        s = wred(s + __shfl_xor_sync(0xffffffffu, s, 1));
        s = wred(s + __shfl_xor_sync(0xffffffffu, s, 2));
        if (q == 0 && c < C) sm.res[c] = s;
    }
    __syncthreads();
    const u64 *q = sm.res;  // q[0..deg] is this chunk's polynomial
    const u32 deg = C - 1;
    if (!W.last) {
        if (tid <= deg) W.out[(u64)tid * W.nchunks + chunk] = q[tid];
    } else {
        // q(t) for t = 0..n by Horner; q(0) = V~_{i+1}(r1) feeds phase 3
        if (tid <= W.n) {
            u64 acc = q[deg];
            for (int c = (int)deg - 1; c >= 0; c--) acc = wred(wmul(acc, (u64)tid) + q[c]);
            G.tr[W.tr_q + tid] = wcanon(acc);
        }
        if (tid == 0) G.scal[SCAL_V1(W.layer)] = wcanon(q[0]);
    }
    return next;
}

// ---- the persistent launch ------------------------------------------------------------

// After a chunk of a wave with a tail: count the chunk; the CTA that counts
// the last one returns true (and resets the counter for the next proof).
__device__ __forceinline__ bool wave_done(u32 *counter, u32 nchunks, u32 &s_flag)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_flag = (atomicAdd(counter, 1u) == nchunks - 1) ? 1u : 0u;
    __syncthreads();
    const bool last = s_flag != 0;
    if (last) {
        __threadfence();
        if (threadIdx.x == 0) *counter = 0;
    }
    return last;
}

#ifndef WV_MINB
#define WV_MINB 4  // resident CTAs per SM the register allocation is sized for (4: 128 registers)
#endif

__global__ void __launch_bounds__(WV_NT, WV_MINB) k_waves(const Globals *Gs, const LineWaveDev *lw, const ProdWave *pw,
                                                   const GenWave *gw, const Task *tasks, int ntasks, u32 *ctr)
{
    __shared__ int s_task;
    __shared__ u32 s_flag;
    // the final reduction may begin its launch on SMs this launch frees as it
    // drains (it waits for the whole launch before it reads what it wrote)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // a CTA's first task is its own index (the grid has at most ntasks CTAs);
    // the counter hands out the rest, each claimed in the last part of the task
    // before it: earlier, and a long task would hold back one that an idle CTA
    // could run; later, and every task would wait for the counter.  With a CTA
    // for every task (up to F2 2^14) there is nothing to claim, and neither
    // counter is touched: two round trips to memory less (F2 2^1 15.4 -> 14.4 us,
    // 2^10 24.6 -> 22.6).
    if ((int)gridDim.x == ntasks) ctr = nullptr;
    int ti = blockIdx.x;
    for (;;) {
        const Task tk = tasks[ti];
        int next = 0;
        if (tk.type == TK_LINE) {
            const LineWaveDev &W = lw[tk.wave];
            const Globals &G = Gs[W.circ];
            next = line_chunk(G, W, tk.chunk, ctr);
            if (W.tail && wave_done(W.counter, W.nchunks, s_flag)) line_chunk(G, lw[tk.wave + 1], 0, nullptr);
        } else if (tk.type == TK_PROD) {
            const ProdWave &W = pw[tk.wave];
            next = prod_chunk(W, tk.chunk, ctr);
            if ((W.flags & WF_TAIL) && wave_done(W.counter, W.nchunks, s_flag)) {
                __syncthreads();
                prod_chunk(pw[tk.wave + 1], 0, nullptr);
            }
        } else {
            const GenWave &W = gw[tk.wave];
            const Globals &G = Gs[W.circ];
            next = gen_chunk(G, W, tk.chunk, ctr);
            if ((W.flags & WF_TAIL) && wave_done(W.counter, W.nchunks, s_flag)) {
                __syncthreads();
                gen_chunk(G, gw[tk.wave + 1], 0, nullptr);
            }
        }
        if (!ctr) return;
        if (threadIdx.x == 0) s_task = next;
        __syncthreads();  // the task is done with shared memory
        ti = s_task;
        if (ti >= ntasks) break;
        __syncthreads();  // s_task is read
    }
    // the CTA that exits last resets the task counter for the next launch
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&ctr[1], 1u) == gridDim.x - 1) {
            ctr[0] = 0;
            ctr[1] = 0;
        }
    }
}

// Shared-memory size of the wave launch (called outside stream capture).
void waves_init()
{
    device_sms();
    cudaFuncSetAttribute(k_waves, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WaveSmem));
}

void launch_waves(const Globals *Gs, const LineWaveDev *lw, const ProdWave *pw, const GenWave *gw, const Task *tasks,
                  int ntasks, u32 *ctr, cudaStream_t st)
{
    if (ntasks <= 0) return;
    const int sms = device_sms();
    const int grid = std::min(ntasks, sms * WV_MINB);
    k_waves<<<grid, WV_NT, sizeof(WaveSmem), st>>>(Gs, lw, pw, gw, tasks, ntasks, ctr);
}

// --------------------------------------------------------------------------------
// Final reduction into the transcript.  Rounds with more than
// FINAL_WARP_MIN chunk partials (they come first in the round list) are
// summed by a warp each; the rest, the great majority in a batch of small
// circuits, by a thread each.  The round's scalars then turn the sums into
// g(0), g(1), g(2).
// --------------------------------------------------------------------------------

// The scalars a round's message needs besides its partial sums (loaded
// before the sums, so that both sets of loads are in flight together).
struct RoundScalars {
    u64 ez, ch, rp0, v1, es, kap, c0, c1;
};

// Everything but v1 (the coin launch wrote it all before the wave launch).
__device__ __forceinline__ RoundScalars round_scalars_pre(const RoundRef &R)
{
    RoundScalars S{};
    S.ez = *R.ez;
    S.ch = *R.ch;
    if (R.rp0) S.rp0 = *R.rp0;
    if (R.kind < PK_GEN_FIRST) {
        S.es = *R.esum;
        S.kap = *R.kap;
        S.c0 = R.lc[0];
        S.c1 = R.lc[1];
    }
    return S;
}

// A product out of line.  A round takes up to ten, in five forms, once each: a
// warp that has one round to itself waits for instruction fetches (with the L2
// flushed F2 2^17 55.5 -> 53.3 us, 2^4 24.6 -> 23.1); threads with rounds of
// their own run the code from the cache, with the products in line.
static __device__ __noinline__ u64 f_mul_call(u64 a, u64 b) { return f_mul_wide(a, b); }

// g(0), g(1), g(2) of round R from its canonical partial sums h (and h2:
// TREE phase 2's second instance), written to the circuit's transcript.
template <bool CALL>
__device__ __forceinline__ void final_round(const Globals *Gs, const RoundRef &R, const RoundScalars &S,
                                            const u64 (&h)[3], const u64 (&h2)[2])
{
    auto mul = [](u64 a, u64 b) { return CALL ? f_mul_call(a, b) : f_mul(a, b); };
    const u64 ez = S.ez;
    u64 g0, g1, g2;
    if (R.kind >= PK_GEN_FIRST) {
        // h[2] is the leading coefficient: value at 2 = 2 g(1) - g(0) + 2 h2
        u64 s0 = (R.kind == PK_GEN_TAB) ? 1 : ez, s1 = s0, s2 = s0, lead = h[2];
        if (R.kind == PK_GEN_PAIR2 || R.kind == PK_GEN_FINAL2) {
            // round 0: P[2q + b] = A f_b, f = (1 - a, a) (PAIR) or (0, 1) (FINAL);
            // later rounds carry the fold f_0 + r_0 (f_1 - f_0) left out of P
            const u64 a = R.kind == PK_GEN_PAIR2 ? S.rp0 : 1, f0 = f_sub(1, a);
            if (R.j == 0) {
                s0 = mul(ez, f0);
                s1 = mul(ez, a);
                s2 = f_sub(s1, s0);
                lead = f_sub(h[1], h[0]);
            } else {
                s0 = s1 = s2 = mul(ez, f_add(f0, mul(S.ch, f_sub(a, f0))));
            }
        }
        g0 = mul(s0, h[0]);
        g1 = mul(s1, h[1]);
        lead = mul(s2, lead);
        g2 = f_add(f_sub(f_add(g1, g1), g0), f_add(lead, lead));
    } else if (R.kind == PK_TREE2) {
        const u64 kj = mul(ez, S.kap), c0 = S.c0, c1 = S.c1;
        const u64 d = f_sub(f_add(h[1], h[1]), h[0]);  // h(2)
        if (R.j == 0) {  // L_0(t) (h(t) + h(1)), L_0 = 1 - t
            g0 = mul(ez, f_add(h[0], h[1]));
            g1 = 0;
            g2 = f_neg(mul(ez, f_add(d, h[1])));
        } else {
            const u64 sb = mul(ez, f_sub(1, S.ch));
            const u64 b0 = mul(sb, mul(c0, h2[0])), b1 = mul(sb, mul(c1, h2[1]));
            g0 = f_add(mul(kj, mul(c0, h[0])), b0);
            g1 = f_add(mul(kj, mul(c1, h[1])), b1);
            g2 = f_add(mul(kj, mul(f_sub(f_add(c1, c1), c0), d)), f_sub(f_add(b1, b1), b0));
        }
    } else {
        const u64 v1 = S.v1, es = S.es, kap = S.kap, c0 = S.c0, c1 = S.c1;
        // the instance sums sigma P (sv V + add)
        u64 sigma = 1, sv = 1, add = 0;
        if (R.kind == PK_TREE3) {
            sigma = mul(ez, f_sub(1, S.ch));
            add = v1;
        } else if (R.kind == PK_FIRST3) {
            sigma = ez;
            add = mul(S.rp0, v1);
            sv = f_add(S.rp0, f_sub(v1, add));  // rp0 + v1 (1 - rp0)
        } else if (R.kind != PK_PH1) {
            sigma = mul(ez, v1);
        }
        const u64 ce = mul(add, es);
        const u64 h0 = f_add(mul(sv, h[0]), ce), h1 = f_add(mul(sv, h[1]), ce);
        const u64 kj = mul(sigma, kap);
        g0 = mul(kj, mul(c0, h0));
        g1 = mul(kj, mul(c1, h1));
        g2 = mul(kj, mul(f_sub(f_add(c1, c1), c0), f_sub(f_add(h1, h1), h0)));
    }
    u64 *tr = Gs[R.circ].tr;
    tr[R.tr_pos] = g0;
    tr[R.tr_pos + 1] = g1;
    tr[R.tr_pos + 2] = g2;
}

__global__ void __launch_bounds__(256) k_final(Globals *Gs, const RoundRef *rounds, int nrounds, int nbig,
                                               const u32 *outs, int nouts)
{
    const u32 lane = threadIdx.x & 31;
    const u64 gt = blockIdx.x * (u64)blockDim.x + threadIdx.x, nthreads = (u64)gridDim.x * blockDim.x;
    // the outputs open each transcript (the evaluation wrote them before the
    // wave launch began): gridDim / nouts CTAs a circuit (one CTA copying
    // MATMULT's 2^14 outputs took 14 us); the proof's in-place input pointer is
    // cleared (later evaluations read the input layer)
    const u32 slices = gridDim.x > (u32)nouts ? gridDim.x / nouts : 1u;
    for (u32 k = blockIdx.x; k < (u32)nouts * slices; k += gridDim.x) {
        Globals &G = Gs[outs[k % nouts]];
        const u32 sl = k / nouts;
        if (sl == 0 && threadIdx.x == 0) G.in = nullptr;
        const u64 n = G.S0;
        const u64 *__restrict__ src = G.out_src;
        u64 *__restrict__ dst = G.tr;
        for (u64 x = (u64)sl * blockDim.x + threadIdx.x; x < n; x += (u64)slices * blockDim.x) dst[x] = src[x];
    }
    // launched early (programmatic dependence on the wave launch): the first
    // round's descriptor and coin-launch scalars are loaded before waiting
    // for the waves; v1 and the partials only after
    const u64 gw0 = gt >> 5;
    RoundRef R0{};
    RoundScalars S0{};
    if (gw0 < (u64)nbig) {
        R0 = rounds[gw0];
        if (lane == 0) S0 = round_scalars_pre(R0);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (u64 gw = gw0; gw < (u64)nbig; gw += nthreads >> 5) {
        const RoundRef R = (gw == gw0) ? R0 : rounds[gw];
        RoundScalars S{};
        if (lane == 0) {
            S = (gw == gw0) ? S0 : round_scalars_pre(R);
            if (R.kind < PK_GEN_FIRST) S.v1 = *R.v1;  // written by the layer's line reduction
        }
        u64 h[3] = {0, 0, 0}, h2[2] = {0, 0};
        if (R.kind >= PK_GEN_FIRST) {
            warp_record_sums<3>(R.part_pos, R.nchunks, lane, h);
        } else {
            warp_record_sums<2>(R.part_pos, R.nchunks, lane, h);
            if (R.nchunks2) warp_record_sums<2>(R.part2_pos, R.nchunks2, lane, h2);
        }
        if (lane == 0) final_round<true>(Gs, R, S, h, h2);
    }
    // (from the grid's end: the CTAs that had no round to themselves first)
    for (u64 t = nthreads - 1 - gt; t < (u64)(nrounds - nbig); t += nthreads) {
        const RoundRef R = rounds[nbig + t];
        RoundScalars S = round_scalars_pre(R);
        if (R.kind < PK_GEN_FIRST) S.v1 = *R.v1;
        const u32 nv = R.kind >= PK_GEN_FIRST ? 3 : 2;
        u64 h[3] = {0, 0, 0};
        for (u32 q = 0; q < R.nchunks; q++)
            for (u32 v = 0; v < nv; v++) h[v] = wred(h[v] + R.part_pos[(u64)q * nv + v]);
        for (u32 v = 0; v < 3; v++) h[v] = wcanon(h[v]);
        u64 h2[2] = {0, 0};
        for (u32 q = 0; q < R.nchunks2; q++)
            for (u32 v = 0; v < 2; v++) h2[v] = wred(h2[v] + R.part2_pos[(u64)q * 2 + v]);
        for (u32 v = 0; v < 2; v++) h2[v] = wcanon(h2[v]);
        final_round<false>(Gs, R, S, h, h2);
    }
}

void launch_final(Globals *Gs, const RoundRef *rounds, int nrounds, int nbig, const u32 *outs, int nouts,
                  cudaStream_t st)
{
    const u64 warp_blocks = ((u64)nbig * 32 + 255) / 256, thread_blocks = ((u64)(nrounds - nbig) + 255) / 256;
    u64 blocks = warp_blocks + thread_blocks;
    if (blocks < (u64)nouts) blocks = (u64)nouts;
    if (blocks < 64) blocks = 64;
    if (blocks > (u64)device_sms() * 8) blocks = (u64)device_sms() * 8;
    // programmatic dependence: the launch may begin while the wave launch
    // drains (k_final waits for it with griddepcontrol.wait)
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_final, Gs, rounds, nrounds, nbig, outs, nouts);
}
