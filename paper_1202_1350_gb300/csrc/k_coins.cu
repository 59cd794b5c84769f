// k_coins.cu -- the verifier's coins and everything derived from them alone,
// in one launch: the challenges and layer points (Sec. 3.1: z_{i+1} is the
// point the line reduction moves to), the split eq tables of those points,
// and the factor tables of the product-weighted sum-checks.
//
// Every challenge is a function of the seed (challenge c = draw c + 1 of the
// splitmix64 stream, Sec. 3.1's "verifier picks at random", made
// reproducible), so each CTA derives the challenges its job needs itself and
// no CTA waits for another.  A draw equal to p is rejected and the stream
// shifts (probability 2^-61 per draw): each CTA finds out whether any of its
// circuit's draws is (eight products, draws_rejected) and then walks the
// stream to each of its challenges.
#include <cuda_runtime.h>
#include "coins.cuh"

#define CN_NT 256

// Every loop here is kept rolled: a CTA runs each piece of code a few times at
// most, so the launch waits for instruction fetches, not for issue slots.

// Setup role: all challenges, all points, eq(z_i, r_P) per layer, shared by
// `n` CTAs (a warp takes one layer: one CTA for all of F0's 78 layers was the
// end of the launch, 16 us).
__device__ void coins_setup(const Globals &G, bool rej, u32 slice, u32 n)
{
    const u32 t0 = slice * blockDim.x + threadIdx.x, nt = n * blockDim.x;
    if (!rej) {
#pragma unroll 1
        for (u32 c = t0; c < G.nchal; c += nt) G.chal[c] = splitmix64_at(G.seed, (u64)c + 1) >> 3;
    } else if (t0 == 0) {
        u64 k = 1;
#pragma unroll 1
        for (u32 c = 0; c < G.nchal; c++) {
            u64 x;
            do { x = splitmix64_at(G.seed, k++) >> 3; } while (x == FP_P);
            G.chal[c] = x;
        }
    }
    const LayerDev *L = G.layers;
#pragma unroll 1
    for (u32 k = t0; k < L[0].s; k += nt) G.pts[L[0].z_off + k] = chal_of(G, rej, k);
#pragma unroll 1
    for (u32 qi = t0; qi < G.nz; qi += nt) {
        const u32 i = G.zmap[qi] >> 8, k = G.zmap[qi] & 0xFF;
        G.pts[((i + 1 < G.d) ? L[i + 1].z_off : G.zd_off) + k] = zcoord(G, rej, i + 1, k);
    }
    // eq(z_i, r_P): a warp per layer, a lane per coordinate (s_i <= 30)
    const u32 lane = threadIdx.x & 31;
#pragma unroll 1
    for (u32 i = t0 >> 5; i < G.d; i += nt >> 5) {
        u64 f = 1;
        if (lane < L[i].s) {
            const u64 z = zcoord(G, rej, i, lane), rp = chal_of(G, rej, L[i].chal_off + lane);
            f = f_add(f_mul(z, rp), f_mul(f_sub(1, z), f_sub(1, rp)));
        }
        f = warp_prod(f);
        if (lane == 0) G.scal[SCAL_EQZRP(i)] = f;
    }
}

// Eq-table role: lo[j] = prod_{k<h} eq(x_k, bit_k j), hi[j] = prod_{k<n-h}
// eq(x_{h+k}, bit_k j).  Each half is a product of two sub-tables over its
// low and high coordinates, built by direct products, so every entry costs
// one product.
__device__ void coins_eq(const Globals &G, bool rej, const EqJob &J)
{
    const EqTab &t = J.t;
    __shared__ u64 x[64], xm[64];
    __shared__ u64 sub[4][256];
#pragma unroll 1
    for (u32 k = threadIdx.x; k < t.n; k += blockDim.x) {
        x[k] = chal_of(G, rej, J.off + k);
        xm[k] = f_sub(1, x[k]);
    }
    __syncthreads();
    const u32 m[2] = {t.h, t.n - t.h};
    const u32 c0[2] = {0, t.h};
#pragma unroll 1
    for (u32 j = 0; j < 2; j++) {
        const u32 m1 = m[j] / 2, m2 = m[j] - m1;
#pragma unroll 1
        for (u32 e = threadIdx.x; e < (1u << m1) + (1u << m2); e += blockDim.x) {
            const bool lowp = e < (1u << m1);
            const u32 idx = lowp ? e : e - (1u << m1);
            const u32 cnt = lowp ? m1 : m2, off = c0[j] + (lowp ? 0 : m1);
            u64 v = 1;
#pragma unroll 1
            for (u32 k = 0; k < cnt; k++) v = f_mul(v, ((idx >> k) & 1) ? x[off + k] : xm[off + k]);
            sub[2 * j + (lowp ? 0 : 1)][idx] = v;
        }
    }
    __syncthreads();
    u64 *dst[2] = {t.lo, t.hi};
#pragma unroll 1
    for (u32 j = 0; j < 2; j++) {
        const u32 m1 = m[j] / 2;
#pragma unroll 1
        for (u32 e = threadIdx.x; e < (1u << m[j]); e += blockDim.x)
            dst[j][e] = f_mul(sub[2 * j][e & ((1u << m1) - 1)], sub[2 * j + 1][e >> m1]);
    }
}

// Linear factor L_m of a product-weighted instance, from the coins (the kinds'
// factors: the PK_* list).  Most are w e, the two points' coordinates iw and
// ie multiplied entry by entry, or one of them alone.
__device__ void prod_factor(const Globals &G, bool rej, const SciDev &S, u32 m, u64 &c0, u64 &c1)
{
    const LayerDev &L = G.layers[S.layer];
    const u32 rP = L.chal_off, r1 = L.chal_off + L.s;
    const u32 none = 0xFFFFFFFFu;
    u32 iw = none, ie = none;  // challenges of w's and e's coordinate
    c0 = c1 = 1;
    const u32 Lb = L.s / 3;
    switch (S.kind) {
    case PK_PH1: {
        const u64 z = zcoord(G, rej, S.layer, m);
        c0 = f_sub(1, z);
        c1 = z;
        return;
    }
    case PK_TREE2:
        if (m == 0) {
            c1 = 0;
            return;
        }
        iw = rP + m - 1;
        break;
    case PK_TREE2B: iw = rP + m; break;
    case PK_TREE3:
        if (m == 0) {
            c0 = 0;
            return;
        }
        iw = rP + m - 1;
        ie = r1 + m;
        break;
    case PK_FINAL3:
        if (m == 0) c0 = 0;
        else iw = rP + m - 1;
        ie = r1 + m;
        break;
    case PK_FIRST3:
        iw = rP + m + 1;
        ie = r1 + m;
        break;
    case PK_MM3:
        if (m < Lb) {
            iw = rP + Lb + m;
        } else {
            iw = rP + m - Lb;
            ie = r1 + m - Lb;
            if (m == 2 * Lb) {  // the top bit
                c0 = 0;
                c1 = f_sub(1, chal_of(G, rej, r1 + 2 * Lb));
#pragma unroll 1
                for (u32 b = 0; b < Lb; b++) {
                    const u64 x = chal_of(G, rej, rP + 2 * Lb + b), y = chal_of(G, rej, r1 + Lb + b);
                    c1 = f_mul(c1, f_add(f_mul(x, y), f_mul(f_sub(1, x), f_sub(1, y))));
                }
                return;
            }
        }
        break;
    default:  // PK_SQ3, PK_PAIR3
        iw = rP + m;
        ie = r1 + m;
        break;
    }
    const u64 w = iw == none ? 0 : chal_of(G, rej, iw), e = ie == none ? 0 : chal_of(G, rej, ie);
    if (iw != none) {
        c0 = f_mul(c0, f_sub(1, w));
        c1 = f_mul(c1, w);
    }
    if (ie != none) {
        c0 = f_mul(c0, f_sub(1, e));
        c1 = f_mul(c1, e);
    }
    if (S.kind == PK_PAIR3 && m == 0) {
        c0 = f_add(c0, c1);
        c1 = 0;
    }
}

// prod over the coordinates a .. a + n - 1 but a + skip (skip < 0 or >= n:
// none is left out) of e_m (m below a + skip) or c_m (above it) at y's bits.
__device__ __forceinline__ u64 part_prod(const u64 (*c)[2], const u64 (*e)[2], u32 a, u32 n, int skip, u32 y)
{
    u64 v = 1;
#pragma unroll 1
    for (int m = 0; m < (int)n; m++) {
        if (m == skip) continue;
        v = f_mul(v, m < skip ? e[a + m][y & 1] : c[a + m][y & 1]);
        y >>= 1;
    }
    return v;
}

// Weights over kk <= 7 coordinates are products of a part over the lower h =
// ceil(kk / 2) of them and one over the rest, each a product of at most four
// factors from these tables.
struct VecParts {
    u64 ea[16], eb[8];      // all e
    u64 ca[16], cb[8];      // all c
    u64 ma[4][8], mb[3][4]; // coordinate j left out: e below it, c above
};

// Word t < 92 of the tables: the arguments of its part_prod and where it goes
// (NULL: kk needs no such word).
__device__ __forceinline__ u64 *vec_part_job(VecParts &V, u32 t, u32 kk, u32 &a, u32 &n, int &skip, u32 &y)
{
    const u32 h = (kk + 1) / 2, g = kk - h;
    const bool lower = t < 32 || (t >= 48 && t < 80);
    a = lower ? 0 : h;
    n = lower ? h : g;
    if (t < 48) {  // ea, ca (16 each), eb, cb (8 each)
        const u32 w = lower ? 16 : 8, k = lower ? t : t - 32;
        const bool all_c = k >= w;
        y = k & (w - 1);
        skip = all_c ? -1 : 99;
        if (y >= (1u << n)) return nullptr;
        return lower ? (all_c ? V.ca : V.ea) + y : (all_c ? V.cb : V.eb) + y;
    }
    const u32 j = lower ? (t - 48) >> 3 : (t - 80) >> 2;
    y = lower ? t & 7 : t & 3;
    skip = (int)j;
    if (j >= n || y >= (1u << (n - 1))) return nullptr;
    return lower ? &V.ma[j][y] : &V.mb[j][y];
}

// Message weights of kk coordinates (layout: ProdWave::wblk).
__device__ __forceinline__ void coins_vec(u64 *T, u32 kk, const VecParts &V)
{
    const u32 half = 1u << (kk - 1), words = vec_words(kk), h = (kk + 1) / 2;
#pragma unroll 1
    for (u32 idx = threadIdx.x; idx < words; idx += blockDim.x) {
        const u32 i = idx / (16 * kk), rem = idx - i * 16 * kk, j = rem >> 4, y = 16 * i + (rem & 15);
        u64 v = 0;
        if (y < half) {
            if (j < h)
                v = f_mul(V.ma[j][y & ((1u << (h - 1)) - 1)], V.cb[y >> (h - 1)]);
            else
                v = f_mul(V.ea[y & ((1u << h) - 1)], V.mb[j - h][y >> h]);
        }
        T[idx] = v;
    }
}

// Product-weight role, one PROD wave: the wave's weight block and, for the
// first wave of an SCI, its factors, kappa_j (without sigma) and esum_j =
// prod_{m>j} (c0_m + c1_m).
__device__ void coins_prep(const Globals &G, bool rej, const SciDev &S, const ProdWave &W)
{
    __shared__ u64 c[32][2], e[PR_C + PR_R][2];
    __shared__ VecParts col, row;
    const u32 tid = threadIdx.x;
    if (tid < S.n) prod_factor(G, rej, S, tid, c[tid][0], c[tid][1]);
    if (tid >= 32 && tid < 32 + W.nr) {
        const u64 r = chal_of(G, rej, S.chal_off + W.r0 + tid - 32);
        e[tid - 32][0] = f_sub(1, r);
        e[tid - 32][1] = r;
    }
    __syncthreads();
    if (S.kind == PK_TREE2B) {  // a folded coordinate keeps its factor
        if (tid < 2 * W.nr) e[tid >> 1][tid & 1] = f_mul(e[tid >> 1][tid & 1], c[W.r0 + (tid >> 1)][tid & 1]);
        __syncthreads();
    }
    const u32 kc = W.kc, kr = W.kr, r0 = W.r0;
    u64 *blk = W.wblk;
    u64 *olo = blk + pw_outer(kc, kr);
    // the parts of the columns' weights (92 words), of the rows' and the outer
    // tables, one loop around one copy of the product's code
    const u32 nlo = 1u << W.ho, nhi = 1u << (W.no - W.ho), njob = 192 + nlo + nhi;
#pragma unroll 1
    for (u32 t = tid; t < njob; t += CN_NT) {
        u32 a = 0, n = 0, y = 0;
        int skip = -1;
        u64 *dst = nullptr;
        if (t < 192) {
            const bool rows = t >= 96;
            const u32 k = rows ? t - 96 : t;
            if (k < 92 && !(rows && kr == 0)) {
                dst = vec_part_job(rows ? row : col, k, rows ? kr : kc, a, n, skip, y);
                if (rows) a += kc;
            }
        } else {
            const u32 x = t - 192;
            const bool hi = x >= nlo;
            dst = olo + x;
            a = W.nr + (hi ? W.ho : 0);
            n = hi ? W.no - W.ho : W.ho;
            y = hi ? x - nlo : x;
        }
        if (dst) *dst = part_prod(c + r0, e, a, n, skip, y);
    }
    if (tid >= 224) {
        const u32 j = tid - 224;
        if (j < 4) blk[pw_last(kc, kr) + j] = j < 2 ? e[kc - 1][j] : (kr ? e[kc + kr - 1][j - 2] : 0);
        if (r0 == 0 && S.Lc) {
            // kappa_j = prod_{m<j} L_m(r_m), esum_j = prod_{m>j} (c0_m + c1_m): warp scans
            const bool in = j < S.n;
            const u64 r = in ? chal_of(G, rej, S.chal_off + j) : 0;
            const u64 a = in ? f_add(c[j][0], f_mul(r, f_sub(c[j][1], c[j][0]))) : 1;
            const u64 b = in ? f_add(c[j][0], c[j][1]) : 1;
            u64 pre = __shfl_up_sync(0xffffffffu, warp_scan_mul(a), 1);
            u64 suf = __shfl_down_sync(0xffffffffu, warp_rscan_mul(b), 1);
            if (j == 0) pre = 1;
            if (j == 31) suf = 1;
            if (in) {
                S.Lc[2 * j] = c[j][0];
                S.Lc[2 * j + 1] = c[j][1];
                S.kap[j] = pre;
                S.esum[j] = suf;
            }
        }
    }
    __syncthreads();
#pragma unroll 1
    for (u32 k = 0; k < (kr ? 2u : 1u); k++)
        coins_vec(blk + (k ? pw_trow(kc, kr) : pw_tcol(kr)), k ? kr : kc, k ? row : col);
    if (kr) {
        if (tid < (1u << PR_C)) {
            blk[tid] = f_mul(col.ea[tid & 15], col.eb[tid >> 4]);
        } else if (tid - (1u << PR_C) < (1u << kr)) {
            const u32 y = tid - (1u << PR_C), h = (kr + 1) / 2;
            blk[pw_roww(kr) + y] = f_mul(row.ca[y & ((1u << h) - 1)], row.cb[y >> h]);
        }
    }
}

// Line-weight role, one line wave: the weight polynomials over its kk
// coordinates (LineWaveDev::wt), each a product of a polynomial over the lower
// half of the coordinates and one over the upper half.
__device__ void coins_line(const Globals &G, bool rej, const LineWaveDev &W)
{
    __shared__ u64 a[8], b[8];
    __shared__ u64 part[24][5];  // 16 lower, 8 upper polynomials of degree <= 4
    const u32 tid = threadIdx.x, kk = W.kk, h = (kk + 1) / 2, g = kk - h;
    if (tid < kk) {
        const u32 k = W.l0 + W.e + tid;
        const u64 x = chal_of(G, rej, W.a_off + k);
        a[tid] = x;
        b[tid] = f_sub(chal_of(G, rej, W.b_off + k), x);
    }
    __syncthreads();
    const bool up = tid >= 16;
    const u32 m0 = up ? h : 0, nm = up ? g : h, y = up ? tid - 16 : tid;
    if (tid < 24 && y < (1u << nm)) {
        u64 *q = part[tid];
        q[0] = 1;
#pragma unroll 1
        for (u32 m = 0; m < nm; m++) {
            const bool one = (y >> m) & 1;  // l_m = a + b t, 1 - l_m
            const u64 c0 = one ? a[m0 + m] : f_sub(1, a[m0 + m]), c1 = one ? b[m0 + m] : f_neg(b[m0 + m]);
            q[m + 1] = f_mul(c1, q[m]);
#pragma unroll 1
            for (u32 j = m; j > 0; j--) q[j] = f_add(f_mul(c0, q[j]), f_mul(c1, q[j - 1]));
            q[0] = f_mul(c0, q[0]);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (u32 idx = tid; idx < ((kk + 1) << kk); idx += CN_NT) {
        const u32 y2 = idx & ((1u << kk) - 1), c = idx >> kk;
        const u64 *lo = part[y2 & ((1u << h) - 1)], *hi = part[16 + (y2 >> h)];
        u64 v = 0;
#pragma unroll 1
        for (u32 j = c > h ? c - h : 0; j <= c && j <= g; j++) v = f_add(v, f_mul(lo[c - j], hi[j]));
        W.wt[idx] = v;
    }
}

// CTAs [0, nsetup): setup, slice `chunk` of circuit `wave` of each item (8
// layers a slice); then one per eq job; one per PROD wave; one per line wave.
__global__ void __launch_bounds__(CN_NT) k_coins(const Globals *Gs, const Item *setups, int nsetup,
                                                 const EqJob *eqjobs, int neq, const SciDev *scis,
                                                 const ProdWave *pw, int npw, const LineWaveDev *lw)
{
    int b = blockIdx.x;
    if (b < nsetup) {
        const Item it = setups[b];
        const Globals &G = Gs[it.wave];
        coins_setup(G, draws_rejected(G), it.chunk, coin_setups(G.d));
        return;
    }
    b -= nsetup;
    if (b < neq) {
        const EqJob J = eqjobs[b];
        const Globals &G = Gs[J.circ];
        coins_eq(G, draws_rejected(G), J);
        return;
    }
    b -= neq;
    if (b < npw) {
        const ProdWave &W = pw[b];
        const Globals &G = Gs[W.circ];
        coins_prep(G, draws_rejected(G), scis[W.sci], W);
        return;
    }
    const LineWaveDev &W = lw[b - npw];
    const Globals &G = Gs[W.circ];
    coins_line(G, draws_rejected(G), W);
}

void launch_coins(const Globals *Gs, const Item *setups, int nsetup, const EqJob *eqjobs, int neq,
                  const SciDev *scis, const ProdWave *pw, int npw, const LineWaveDev *lw, int nlw, cudaStream_t st)
{
    const int grid = nsetup + neq + npw + nlw;
    if (grid > 0) k_coins<<<grid, CN_NT, 0, st>>>(Gs, setups, nsetup, eqjobs, neq, scis, pw, npw, lw);
}
