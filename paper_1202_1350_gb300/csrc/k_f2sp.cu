// k_f2sp.cu -- the special-purpose non-interactive F2 protocol (outlined in
// Sec. 3.2; prover and verifier parallelisation in Sec. 4.2; memory access in
// Sec. 5.2; GPU results in Sec. 6.3).
//
// The frequency vector a (n = v h entries) is a v x h grid, a(x, y) at
// x h + y.  Row x is the polynomial f_x of degree < h with f_x(w^y) = a(x, y),
// w a generator of the subgroup of order h of F_p^*; the proof is
// s(Y) = sum_x f_x(Y)^2 at the 2h points u^k (u of order 2h, u^2 = w).  The
// verifier keeps f_x(r) for a secret random r, accepts iff
// s(r) = sum_x f_x(r)^2 and answers F2 = sum_{k even} s(u^k).
//
// Prover (the paper's per-row transform by the Prime Factor FFT, Sec. 4.2).
// The even points u^{2y} = w^y are the nodes: s there is the column's sum of
// squares.  For the odd points u w^y: the row's coefficients are the inverse
// DFT of its values over the subgroup of order h, c_j = (1/h) sum_y a_y w^{-jy},
// and f(u w^y) = sum_j (c_j u^j) w^{jy} is a forward DFT of the twisted
// coefficients.  h = q_1 ... q_m with pairwise coprime odd prime powers
// q_i <= 61, so each DFT is an m-dimensional DFT with no twiddles between
// dimensions (Good-Thomas), the root of dimension i being w^{N_i}, N_i = h/q_i.
// The inverse transform takes index y at digits (y N_i^{-1} mod q_i) and leaves
// coefficient j at digits (j mod q_i); the forward one takes j at digits
// (j mod q_i), so nothing moves between the two, and leaves output k at the
// digits with k = sum_i k_i N_i.
//
// A small DFT of odd size q pairs inputs and outputs of opposite sign:
//   X_{+-k} = x_0 + sum_{j<=(q-1)/2} (x_j + x_{q-j}) c_jk +- (x_j - x_{q-j}) s_jk,
// c, s = (w^{jk} +- w^{-jk})/2, i.e. (q-1)/2 products per output instead of q,
// and a thread holds a whole line of q values in registers (the sums, then the
// differences, for q > 13), so a value is read from and written to shared
// memory once per pass, in place, instead of q times.
//
// Verifier.  f_x(r) = sum_y a(x, y) L_y(r) with the subgroup's Lagrange basis
// L_y(r) = w^y (r^h - 1) / (h (r - w^y)), streamed over whole rows; at the end
// s(r) = sum_k s_k u^k (r^{2h} - 1) / (2h (r - u^k)) over the 2h proof points
// (an indicator basis when r lies in the subgroup).
#include <cuda_runtime.h>

#include "plan.h"

#define SP_NT 256
// Prover CTA: 1024 threads (64 registers each) when every dimension is at most
// 13, whose lines fit that; 512 (128 registers) otherwise.  A line's products
// are dependent chains, so warps in flight matter: at 4995 x 5005 16 warps an
// SM issued in 42 % of the cycles.  (Both spill a few words around the calls of
// the passes, once a pass; the lines' loops do not.)
#define SP_PNT 1024
#define SP_PNT_BIG 512

// Geometry and tables of the prover's transform (device pointers; built on
// the host by vc_f2sp_create).
struct SpFft {
    u32 h, m;             // h = q_0 ... q_{m-1}
    u32 q[8], st[8];      // dimension sizes, largest first, and the strides of their digits
    u32 magic[8];         // ceil(2^32 / st): floor(i / st) = (i magic) >> 32 for i < 2^16
    u32 cso[8], ncs;      // offset of dimension i's (c, s) pairs in cs, and their number
    u32 rb, groups;       // rows a CTA transforms together; accumulators per column
    const u64 *cs;        // per dimension, k = 1..(q-1)/2, j = 1..(q-1)/2: c_jk, s_jk
    const u32 *pin;       // input slot of index y (digits y N_i^{-1} mod q_i)
    const u64 *twist;     // slot P -> u^j / h (j the coefficient at P)
    const u32 *idx;       // slot P -> the index k of the forward transform's output there
};

// One line of Q values at p, p + st, ...: its DFT (the inverse one, without
// the factor 1/Q, swaps outputs k and Q - k), in place; with TW times
// tw[slot].  Up to 13 values the sums and differences stay in registers
// together; beyond, the differences wait in shared memory for the sums' half.
// Values between passes are below 3 2^61 (lazy sums of two W values, or a
// difference plus 2 p): the next pass's sums and differences, below 2^64, are
// brought back to W.
// Lines of more than 13 values may be shared by T lanes of a warp (adjacent
// ones, `mask`; this one is lane t of them): each holds all the sums, then all
// the differences, and takes every T-th output pair.  Few rows leave few lines,
// and one of 61 values is 3,600 products one after another.
template <int Q, bool INV, bool TW>
__device__ __forceinline__ void sp_line(u64 *p, u32 st, const ulonglong2 *cs, const u64 *__restrict__ tw, u32 T,
                                        u32 t, u32 mask)
{
    constexpr int N = (Q - 1) / 2;
    const u64 x0 = p[0];
    auto put = [&](u32 k, u64 v) { p[k * st] = TW ? wmul(v, __ldg(tw + k * st)) : v; };
    u64 s[N];
    if constexpr (Q <= 13) {
        u64 d[N];
        u64 t = wred(x0);
#pragma unroll
        for (int j = 0; j < N; j++) {
            const u64 a = p[(j + 1) * st], b = p[(Q - 1 - j) * st];
            s[j] = wred(a + b);
            d[j] = wred(a + (4 * FP_P) - b);
            t += s[j];  // at most seven W values: below 2^64
        }
        put(0, wred(t));
#pragma unroll 1
        for (int k = 1; k <= N; k++) {
            acc128 c, e;  // at most six products and x0
            c.lo = x0;
            c.hi = 0;
            acc_zero(e);
#pragma unroll
            for (int j = 0; j < N; j++) {
                const ulonglong2 w = cs[(k - 1) * N + j];
                mac(c, s[j], w.x);
                mac(e, d[j], w.y);
            }
            const u64 C = acc_red7(c), S = acc_red7(e);
            put(INV ? Q - k : k, C + S);
            put(INV ? k : Q - k, C + (2 * FP_P) - S);
        }
    } else {
        u64 sum = wred(x0);
#pragma unroll
        for (int j = 0; j < N; j++) {
            const u64 a = p[(j + 1) * st], b = p[(Q - 1 - j) * st];
            s[j] = wred(a + b);
            if (T == 1) p[(Q - 1 - j) * st] = wred(a + (4 * FP_P) - b);
            sum += s[j];
            if ((j & 3) == 3) sum = wred(sum);
        }
        if (T > 1) {
            __syncwarp(mask);  // every lane has its sums
#pragma unroll 1
            for (u32 k = t + 1; k <= N; k += T) p[(Q - k) * st] = wred(p[k * st] + (4 * FP_P) - p[(Q - k) * st]);
        }
        if (t == 0) put(0, wred(sum));
#pragma unroll 1
        for (u32 k = t + 1; k <= N; k += T) {
            acc128 c0, c1;  // N <= 30 products of W and canonical values: below 2^128
            c0.lo = x0;
            c0.hi = 0;
            acc_zero(c1);
#pragma unroll
            for (int j = 0; j < N; j++) mac((j & 1) ? c1 : c0, s[j], cs[(k - 1) * N + j].x);
            p[k * st] = wred(acc_red(c0) + acc_red(c1));
        }
        if (T > 1) __syncwarp(mask);  // the differences are there
#pragma unroll
        for (int j = 0; j < N; j++) s[j] = p[(Q - 1 - j) * st];
        if (T > 1) __syncwarp(mask);  // and read: their slots take outputs
#pragma unroll 1
        for (u32 k = t + 1; k <= N; k += T) {
            acc128 e0, e1;
            acc_zero(e0);
            acc_zero(e1);
#pragma unroll
            for (int j = 0; j < N; j++) mac((j & 1) ? e1 : e0, s[j], cs[(k - 1) * N + j].y);
            const u64 C = p[k * st], S = wred(acc_red(e0) + acc_red(e1));
            put(INV ? Q - k : k, C + S);
            put(INV ? k : Q - k, C + (2 * FP_P) - S);
        }
    }
}

// Kinds of pass: inverse, forward, and the middle one along the outermost
// digit (inverse, twist, forward on the same line, so the row does not go
// through shared memory and a barrier in between).
enum { SP_INV = 0, SP_FWD = 1, SP_MID = 2 };

// One pass over `nrows` rows in buf: a thread per line, or T where the lines of
// more than 13 values are at most 1/T of the CTA's threads (100 rows of 61, one
// line a CTA: 31 us, 103 with a thread a line, 39 with a thread a value; 152 of
// 2501 = 41 61: 79, 141 and 122).  Lines of all the rows are numbered together (line J starts at
// (J / st) q st + J mod st).
template <int Q, int KIND, int NT>
__device__ __forceinline__ void sp_pass_q(u64 *buf, u32 nrows, const SpFft &F, u32 d, const ulonglong2 *cs)
{
    const u32 st = F.st[d], n = nrows * (F.h / Q);
    const ulonglong2 *w = cs + F.cso[d];
    u32 T = 1;
    if (Q > 13)
        while (T < 32 && 2 * T * n <= NT) T *= 2;
    const u32 t = threadIdx.x & (T - 1), mask = (T == 32 ? ~0u : (1u << T) - 1) << (threadIdx.x & 31 & ~(T - 1));
    for (u32 J = threadIdx.x / T; J < n; J += NT / T) {
        const u32 o = st == 1 ? J : __umulhi(J, F.magic[d]), in = J - o * st;
        u64 *p = buf + o * Q * st + in;
        if (KIND == SP_MID) {  // outermost digit: o is the row, `in` the line's first slot
            sp_line<Q, true, true>(p, st, w, F.twist + in, T, t, mask);
            if (T > 1) __syncwarp(mask);
            sp_line<Q, false, false>(p, st, w, nullptr, T, t, mask);
        } else if (KIND == SP_INV) {
            sp_line<Q, true, false>(p, st, w, nullptr, T, t, mask);
        } else {
            sp_line<Q, false, false>(p, st, w, nullptr, T, t, mask);
        }
    }
}

template <int KIND, int NT>
__device__ __noinline__ void sp_pass(u64 *buf, u32 nrows, const SpFft &F, u32 d, const ulonglong2 *cs)
{
    switch (F.q[d]) {
    case 3: sp_pass_q<3, KIND, NT>(buf, nrows, F, d, cs); break;
    case 5: sp_pass_q<5, KIND, NT>(buf, nrows, F, d, cs); break;
    case 7: sp_pass_q<7, KIND, NT>(buf, nrows, F, d, cs); break;
    case 9: sp_pass_q<9, KIND, NT>(buf, nrows, F, d, cs); break;
    case 11: sp_pass_q<11, KIND, NT>(buf, nrows, F, d, cs); break;
    case 13: sp_pass_q<13, KIND, NT>(buf, nrows, F, d, cs); break;
    default:
        if constexpr (NT == SP_PNT_BIG) switch (F.q[d]) {
            case 25: sp_pass_q<25, KIND, NT>(buf, nrows, F, d, cs); break;
            case 31: sp_pass_q<31, KIND, NT>(buf, nrows, F, d, cs); break;
            case 41: sp_pass_q<41, KIND, NT>(buf, nrows, F, d, cs); break;
            case 61: sp_pass_q<61, KIND, NT>(buf, nrows, F, d, cs); break;
            default: break;  // vc_f2sp_create admits no other size
            }
    }
}

// Column partials of the proof for the CTA's rows (consecutive, F.rb at a
// time): part[cta][2y] = sum a(x, y)^2, part[cta][2k + 1] = sum f_x(u w^k)^2.
template <int NT>
__global__ void __launch_bounds__(NT, 1) k_sp_prove(const u64 *__restrict__ a, u64 v, SpFft F, u64 *part,
                                                        u32 *status)
{
    extern __shared__ __align__(16) u64 sp_dyn[];
    const u32 h = F.h, gh = F.groups * h;
    ulonglong2 *cs = reinterpret_cast<ulonglong2 *>(sp_dyn);
    u64 *buf = sp_dyn + 2 * F.ncs, *acc_e = buf + F.rb * h, *acc_o = acc_e + gh;
    for (u32 i = threadIdx.x; i < gh; i += NT) acc_e[i] = acc_o[i] = 0;
    for (u32 i = threadIdx.x; i < F.ncs; i += NT) cs[i] = make_ulonglong2(F.cs[2 * i], F.cs[2 * i + 1]);
    bool bad = false;
    const u64 x0 = v * blockIdx.x / gridDim.x, x1 = v * (blockIdx.x + 1) / gridDim.x;
    for (u64 x = x0; x < x1; x += F.rb) {
        const u32 nr = (u32)(x1 - x < F.rb ? x1 - x : F.rb);
        const u64 *rows = a + x * h;
        __syncthreads();  // the previous rows are done with the buffer
        for (u32 e = threadIdx.x; e < gh; e += NT) {
            const u32 g = F.groups == 1 ? 0 : e / h, y = e - g * h;
            const u32 slot = __ldg(F.pin + y);
            u64 sum = acc_e[e];
            for (u32 r = g; r < nr; r += F.groups) {
                u64 val = __ldg(rows + (u64)r * h + y);
                bad |= val >= FP_P;
                val = val >= FP_P ? 0 : val;
                buf[r * h + slot] = val;
                sum = wred(sum + wmul(val, val));
            }
            acc_e[e] = sum;
        }
        // the next rows on their way into L2 while these are transformed
        if (x + F.rb < x1) {
            const u64 *nx = rows + (u64)F.rb * h;
            const u64 left = (x1 - x - F.rb) * h, want = (u64)F.rb * h;
            for (u64 o = threadIdx.x * 16; o < (left < want ? left : want); o += NT * 16)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + o));
        }
        __syncthreads();
        if (F.m == 0) {  // h = 1: only the twist (u^0 / 1)
            for (u32 i = threadIdx.x; i < nr; i += NT) buf[i] = wmul(buf[i], F.twist[0]);
            __syncthreads();
        } else {
            for (u32 d = F.m - 1; d > 0; d--) {
                sp_pass<SP_INV, NT>(buf, nr, F, d, cs);
                __syncthreads();
            }
            sp_pass<SP_MID, NT>(buf, nr, F, 0, cs);
            __syncthreads();
            for (u32 d = 1; d < F.m; d++) {
                sp_pass<SP_FWD, NT>(buf, nr, F, d, cs);
                __syncthreads();
            }
        }
        for (u32 e = threadIdx.x; e < gh; e += NT) {
            const u32 g = F.groups == 1 ? 0 : e / h, i = e - g * h;
            u64 sum = acc_o[e];
            for (u32 r = g; r < nr; r += F.groups) {
                const u64 f = wred(buf[r * h + i]);
                sum = wred(sum + wmul(f, f));
            }
            acc_o[e] = sum;
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, ST_BAD_INPUT);
    u64 *out = part + (u64)blockIdx.x * 2 * h;
    for (u32 i = threadIdx.x; i < h; i += NT) {
        u64 se = 0, so = 0;
        for (u32 g = 0; g < F.groups; g++) {
            se = wred(se + acc_e[g * h + i]);
            so = wred(so + acc_o[g * h + i]);
        }
        out[2 * i] = wcanon(se);
        out[2 * __ldg(F.idx + i) + 1] = wcanon(so);
    }
}

// proof[k] = sum over CTAs of part[cta][k]: a CTA takes 32 entries, its warps
// the partials in turn (a thread an entry left one chain of 152 loads: 23 us).
__global__ void __launch_bounds__(SP_NT) k_sp_reduce(const u64 *__restrict__ part, u32 nparts, u64 n2, u64 *proof)
{
    __shared__ u64 sh[SP_NT / 32][32];
    const u32 lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
    const u64 m = blockIdx.x * (u64)32 + lane;
    u64 s = 0;
    if (m < n2) {
#pragma unroll 4
        for (u32 k = wv; k < nparts; k += SP_NT / 32) s = wred(s + part[(u64)k * n2 + m]);
    }
    sh[wv][lane] = s;
    __syncthreads();
    if (wv == 0 && m < n2) {
        for (u32 k = 1; k < SP_NT / 32; k++) s = wred(s + sh[k][lane]);
        proof[m] = wcanon(s);
    }
}

__device__ u64 f_pow(u64 b, u64 e)
{
    u64 r = 1;
    while (e) {
        if (e & 1) r = f_mul(r, b);
        b = f_mul(b, b);
        e >>= 1;
    }
    return r;
}

// The verifier's secret point: the seed's first accepted draw.
__device__ u64 sp_secret(u64 seed)
{
    for (u64 k = 1;; k++) {
        const u64 r = splitmix64_at(seed, k) >> 3;
        if (r != FP_P) return r;
    }
}

// Verifier setup, every CTA: r from the seed (res[0] = r, written by CTA 0);
// L[y] = L_y(r) over the nodes pw[2y] (y < h) and M[k] = the basis at r over
// the proof points pw[k] (k < 2h), grid-stride; row values zeroed.
__global__ void __launch_bounds__(SP_NT) k_sp_vbegin(u64 seed, u64 v, u64 h, u64 inv_h, const u64 *pw, u64 *L,
                                                     u64 *M, u64 *acc, u64 *res)
{
    const u64 r = sp_secret(seed);
    const u64 gt = blockIdx.x * (u64)SP_NT + threadIdx.x, nth = (u64)gridDim.x * SP_NT;
    if (gt == 0) res[0] = r;
    for (u64 x = gt; x < v; x += nth) acc[x] = 0;
    const u64 rh = f_pow(r, h), r2h = f_mul(rh, rh);
    const u64 ch = f_mul(f_sub(rh, 1), inv_h);                        // (r^h - 1) / h
    const u64 c2h = f_mul(f_mul(f_sub(r2h, 1), inv_h), FP_INV2);      // (r^2h - 1) / (2h)
    for (u64 e = gt; e < 3 * h; e += nth) {
        // e < h: node y = e (point pw[2y]); else proof point k = e - h
        const bool node = e < h;
        const u64 k = node ? 2 * e : e - h;
        const u64 pt = pw[k];
        const bool in_group = node ? (rh == 1) : (r2h == 1);
        u64 val;
        if (in_group) {
            val = (r == pt) ? 1 : 0;  // r is a point of the set: indicator basis
        } else {
            val = f_mul(f_mul(pt, node ? ch : c2h), f_inv(f_sub(r, pt)));
        }
        if (node) L[e] = val;
        else M[k] = val;
    }
}

// Streaming pass over whole rows [x0, x0 + nrows): acc[x] += sum_y a(x, y) L[y]
// (one warp per row; rows given contiguously, row x at rows[(x - x0) h]).
// Bound by HBM when enough loads are in flight: a lane issues SP_VU entries'
// loads before their products (rows start at any multiple of 8 bytes, so
// loads are 8 bytes wide), and CTAs of two warps spread the rows evenly over
// the SMs.
#define SP_VU 8
#define SP_VNT 64
__global__ void __launch_bounds__(SP_VNT) k_sp_vabsorb(const u64 *__restrict__ rows, u64 x0, u64 nrows, u64 h,
                                                       const u64 *__restrict__ L, u64 *acc, u32 *status)
{
    const u32 lane = threadIdx.x & 31, n = (u32)h;
    const u64 wid = (blockIdx.x * (u64)SP_VNT + threadIdx.x) >> 5, nw = ((u64)gridDim.x * SP_VNT) >> 5;
    for (u64 x = wid; x < nrows; x += nw) {
        const u64 *row = rows + x * h;
        u64 red = 0;
        bool bad = false;
        u64 val[SP_VU];
        auto load = [&](u32 y0) {
#pragma unroll
            for (u32 u = 0; u < SP_VU; u++) val[u] = y0 + 32 * u < n ? __ldcs(row + y0 + 32 * u) : 0;
        };
        load(lane);
        for (u32 y0 = lane; y0 < n; y0 += 32 * SP_VU) {
            u64 cur[SP_VU];
#pragma unroll
            for (u32 u = 0; u < SP_VU; u++) cur[u] = val[u];
            load(y0 + 32 * SP_VU);  // the next entries arrive during this batch's products
            acc128 s;
            acc_zero(s);
#pragma unroll
            for (u32 u = 0; u < SP_VU; u++) {
                const u32 y = y0 + 32 * u;
                bad |= cur[u] >= FP_P;
                mac(s, cur[u] >= FP_P ? 0 : cur[u], y < n ? __ldg(L + y) : 0);
            }
            red = wred(red + acc_red(s));
        }
        const u64 t = warp_wsum(red);
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, ST_BAD_INPUT);
        if (lane == 0) acc[x0 + x] = f_add(acc[x0 + x], wcanon(t));
    }
}

// Verifier end (one CTA): res[0] = accept, res[1] = F2 answer (the even
// points), res[2] = s(r), res[3] = sum_x f_x(r)^2.
#define SP_ENT 1024
#define SP_EU 8
__global__ void __launch_bounds__(SP_ENT) k_sp_vend(const u64 *__restrict__ proof, u64 v, u64 h,
                                                    const u64 *__restrict__ M, const u64 *__restrict__ acc, u64 *res)
{
    const u64 n2 = 2 * h;
    u64 lhs = 0, rhs = 0, ans = 0;
    bool bad = false;
    for (u64 x0 = threadIdx.x; x0 < v; x0 += SP_ENT * SP_EU) {  // SP_EU loads in flight per thread
        u64 f[SP_EU];
#pragma unroll
        for (u32 u = 0; u < SP_EU; u++) f[u] = x0 + u * SP_ENT < v ? acc[x0 + u * SP_ENT] : 0;
#pragma unroll
        for (u32 u = 0; u < SP_EU; u++) lhs = wred(lhs + wmul(f[u], f[u]));
    }
    for (u64 k0 = threadIdx.x; k0 < n2; k0 += SP_ENT * SP_EU) {
        u64 s[SP_EU], m[SP_EU];
#pragma unroll
        for (u32 u = 0; u < SP_EU; u++) {
            const u64 k = k0 + u * SP_ENT;
            s[u] = k < n2 ? proof[k] : 0;
            m[u] = k < n2 ? M[k] : 0;
        }
#pragma unroll
        for (u32 u = 0; u < SP_EU; u++) {
            bad |= s[u] >= FP_P;
            const u64 t = s[u] >= FP_P ? 0 : s[u];
            rhs = wred(rhs + wmul(t, m[u]));
            if ((k0 & 1) == 0) ans = wred(ans + t);  // the stride is even: the point's parity is k0's
        }
    }
    __shared__ u64 sh[3][SP_ENT / 32];
    lhs = warp_wsum(lhs);
    rhs = warp_wsum(rhs);
    ans = warp_wsum(ans);
    const u32 lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][wv] = lhs;
        sh[1][wv] = rhs;
        sh[2][wv] = ans;
    }
    const int anybad = __syncthreads_or(bad);
    if (threadIdx.x < 32) {
        lhs = warp_wsum(lane < SP_ENT / 32 ? sh[0][lane] : 0);
        rhs = warp_wsum(lane < SP_ENT / 32 ? sh[1][lane] : 0);
        ans = warp_wsum(lane < SP_ENT / 32 ? sh[2][lane] : 0);
        if (lane == 0) {
            lhs = wcanon(lhs);
            rhs = wcanon(rhs);
            res[0] = (!anybad && lhs == rhs) ? 1 : 0;
            res[1] = wcanon(ans);
            res[2] = rhs;
            res[3] = lhs;
        }
    }
}

// Rows a CTA transforms together, its accumulators per column and its shared
// memory.  About 14,000 values at once: at h = 5005 two rows, whose lines
// (2 x 385 of size 13 up to 2 x 1001 of size 5) fill the threads better than
// one row's and halve the barriers; short rows many at a time.  At most the
// CTA's share of the rows, and what 227 KB hold.
static void sp_prove_shape(u64 v, u64 h, u32 nt, u32 ncs, u32 *rb, u32 *groups, size_t *smem)
{
    const u64 ctas = sp_prove_ctas(v), share = (v + ctas - 1) / ctas;
    const u64 room = 227 * 1024 / 8 - 2 * ncs;
    u64 r = 14000 / h, g;
    if (r > share) r = share;
    if (r < 1) r = 1;
    while (true) {
        g = nt / h;
        if (g > r) g = r;
        if (g < 1) g = 1;
        if (r == 1 || (r + 2 * g) * h <= room) break;
        r--;
    }
    *rb = (u32)r;
    *groups = (u32)g;
    *smem = (size_t)((r + 2 * g) * h + 2 * ncs) * sizeof(u64);
}

u32 sp_prove_ctas(u64 v) { return (u32)(v < (u64)device_sms() ? v : (u64)device_sms()); }

void sp_init()
{
    cudaFuncSetAttribute(k_sp_prove<SP_PNT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaFuncSetAttribute(k_sp_prove<SP_PNT_BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

void launch_sp_prove(const u64 *a, u64 v, const SpFftHost &H, u64 *part, u32 nparts, u64 *proof, u32 *status,
                     cudaStream_t st)
{
    SpFft F{};
    F.h = H.h;
    F.m = H.m;
    F.ncs = H.ncs;
    for (u32 i = 0; i < 8; i++) {
        F.q[i] = H.q[i];
        F.st[i] = H.st[i];
        F.magic[i] = H.magic[i];
        F.cso[i] = H.cso[i];
    }
    F.cs = H.cs;
    F.pin = H.pin;
    F.twist = H.twist;
    F.idx = H.idx;
    size_t smem = 0;
    const bool big = H.m && H.q[0] > 13;  // the largest dimension is first
    sp_prove_shape(v, H.h, big ? SP_PNT_BIG : SP_PNT, H.ncs, &F.rb, &F.groups, &smem);
    if (big)
        k_sp_prove<SP_PNT_BIG><<<nparts, SP_PNT_BIG, smem, st>>>(a, v, F, part, status);
    else
        k_sp_prove<SP_PNT><<<nparts, SP_PNT, smem, st>>>(a, v, F, part, status);
    k_sp_reduce<<<(unsigned)((2 * H.h + 31) / 32), SP_NT, 0, st>>>(part, nparts, 2 * H.h, proof);
}

void launch_sp_vbegin(u64 seed, u64 v, u64 h, u64 inv_h, const u64 *pw, u64 *L, u64 *M, u64 *acc, u64 *res,
                      cudaStream_t st)
{
    k_sp_vbegin<<<grid_for_items(3 * h > v ? 3 * h : v, SP_NT, 4), SP_NT, 0, st>>>(seed, v, h, inv_h, pw, L, M, acc,
                                                                                  res);
}

void launch_sp_vabsorb(const u64 *rows, u64 x0, u64 nrows, u64 h, const u64 *L, u64 *acc, u32 *status,
                       cudaStream_t st)
{
    k_sp_vabsorb<<<grid_for_items(nrows * 32, SP_VNT, 32), SP_VNT, 0, st>>>(rows, x0, nrows, h, L, acc, status);
}

void launch_sp_vend(const u64 *proof, u64 v, u64 h, const u64 *M, const u64 *acc, u64 *res, cudaStream_t st)
{
    k_sp_vend<<<1, SP_ENT, 0, st>>>(proof, v, h, M, acc, res);
}
