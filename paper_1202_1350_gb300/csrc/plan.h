// plan.h -- launch-plan descriptors shared by the host planner and the kernels.
//
// A proof is a fixed sequence of launches whose shapes depend only on the
// circuit's shape, so vc_circuit_create computes every descriptor once and
// uploads it; a proof only replays the plan with a new seed and new inputs.
//
// Because the verifier's coins are a function of the seed alone, every
// challenge is known before the first message is computed.  The prover uses
// this to run all d layer iterations, and within a layer its three sum-check
// phases and its line reduction, concurrently: each is an independent
// "sum-check instance" (SCI) or line job over its own tables.  The rounds of
// one SCI stay in order (each round folds the tables with its challenge).
#pragma once
#include "field.cuh"

enum : u32 {
    W_SQUARE = 0, W_TREE = 1, W_MATMULT = 2, W_F0_FIRST = 3, W_F0_PAIR = 4, W_F0_FINAL = 5,
    W_EXPLICIT = 6
};

// Split table of eq(x, .) over n coordinates: eq(x, b) = lo[b mod 2^h] * hi[b >> h]
// with h = ceil(n/2) (Sec. 4.1.1's per-gate eq factor at one product per gate).
struct EqTab {
    u64 *lo;        // 2^h entries
    u64 *hi;        // 2^(n-h) entries
    const u64 *pt;  // the point, n coordinates (device)
    u32 n, h;
};

__device__ __forceinline__ u64 eq_at(const EqTab &t, u64 b)
{
    return f_mul(t.lo[b & ((1ull << t.h) - 1)], t.hi[b >> t.h]);
}

// One layer iteration (layer i relates V_i to V_{i+1}).
struct LayerDev {
    u32 s, sn;        // s_i, s_{i+1}
    u32 kind;         // W_*
    u32 has_add;      // layer has ADD gates (else the B tables are zero)
    u32 chal_off;     // first round challenge of this layer in chal[]
    u32 z_off;        // z_i in pts[] (s_i coordinates)
    u64 *V;           // layer i values
    u64 *Vn;          // layer i+1 values
    u64 tr_msg;       // transcript offset of the layer's round values
    u64 tr_q;         // transcript offset of q(0..s_{i+1})
    EqTab trp, tr1, tr2;  // eq tables of r_P, r1, r2 (r1, r2: table-built layers, verifier)
    u64 *P2, *B2, *P3, *B3;   // EXPLICIT: phase-2/3 tables over layer i+1 (B* NULL if !has_add)
    u64 *mu, *mei;            // MATMULT: tables of k_mm_tables (n entries each; mei then n zeros)
    const unsigned char *type;  // EXPLICIT only
    const u32 *in1, *in2;
    const u32 *by1_off, *by1_g;  // gates grouped by in1: offsets [S_{i+1}+1], gate ids [S_i]
    const u32 *by2_off, *by2_g;  // gates grouped by in2
};

// In-neighbours and operation of gate g of layer i (Sec. 6.2.1 circuits):
// computed from the index for the structured kinds (a tree gate reads 2g and
// 2g+1, as in Sec. 5.1.4), read for EXPLICIT layers.
__device__ __forceinline__ void gate_wiring(const LayerDev &L, u64 g, u64 &a, u64 &b, u32 &mul)
{
    switch (L.kind) {
    case W_SQUARE: a = g; b = g; mul = 1; break;
    case W_TREE: a = 2 * g; b = 2 * g + 1; mul = 0; break;
    case W_MATMULT: {
        const u32 Lb = L.s / 3;
        const u64 n = 1ull << Lb, m = n - 1;
        const u64 k = g & m, j = (g >> Lb) & m, ii = g >> (2 * Lb);
        a = (ii << Lb) | k;
        b = (1ull << (2 * Lb)) | (k << Lb) | j;
        mul = 1;
        break;
    }
    case W_F0_FIRST: a = g >> 1; b = g >> 1; mul = (g & 1) ? 0 : 1; break;
    case W_F0_PAIR: a = g; b = g & ~1ull; mul = 1; break;
    case W_F0_FINAL: a = 2 * g + 1; b = 2 * g + 1; mul = 1; break;
    default: a = L.in1[g]; b = L.in2[g]; mul = L.type[g]; break;
    }
}

// Per-layer scalars written during a proof: scal[2 i] = eq(z_i, r_P),
// scal[2 i + 1] = V~_{i+1}(r1) (= q_i(0)).
#define SCAL_EQZRP(i) (2 * (i))
#define SCAL_V1(i) (2 * (i) + 1)

// Flags of a sum-check wave.  WF_TAIL: the next descriptor (a single chunk)
// is run by the CTA that finishes this wave's last chunk.
// WF_ODD: a PROD wave over the odd entries of its input table; WF_HOST: over
// values in host memory.
enum : u32 { WF_HASB = 2, WF_LAST = 4, WF_TAIL = 8, WF_ODD = 16, WF_HOST = 32 };

// Kinds of sum-check instance (SCI).  Product-weighted ones (< PK_GEN_FIRST)
// keep P = sigma prod_m L_m(x_m) implicit; general ones fold P, V, B tables.
// Phase 3's gates with in2 = x have a product-form weight over x in every
// structured kind, so it needs no table: with w, e the factors eq(r_P, .),
// eq(r1, .) of the gates and their first in-neighbours,
//   SQUARE    L_m = w_m e_m;
//   TREE      L_0 = (0, 1), L_m = w_{m-1} e_m, summed with V + v1;
//   F0_PAIR   in2 = 2q of gates 2q, 2q+1: L_0 = (w_0(0) e_0(0) + w_0(1) e_0(1), 0), L_m = w_m e_m;
//   F0_FINAL  in2 = 2q+1: L_0 = (0, e_0(1)), L_m = w_{m-1} e_m;
//   F0_FIRST  gates 2x (MUL), 2x+1 (ADD): L_m = w_{m+1} e_m, and per entry
//             (w_0(0) v1 + w_0(1)) V + w_0(1) v1;
//   MATMULT   x = (j, k, 1): L = w over j, w e over k, and on the top bit (0,
//             the sum over i of w e, times e's own top factor).
enum : u32 {
    PK_PH1 = 0,        // phase 1 of any layer: P = eq(z_i, .), V = V_i
    PK_TREE3 = 1,
    PK_SQ3 = 2,        // sigma = eq(z,rP) v1, as for the next three
    PK_PAIR3 = 3,
    PK_FINAL3 = 4,
    PK_MM3 = 5,
    PK_FIRST3 = 6,
    // TREE phase 2: P[2g] = eq(rP, g), B[2g] = P[2g] V[2g+1] (times eq(z, rP)).
    // P is a product over the coordinates, L_0 = (1, 0).  Folding B by r_0
    // leaves (1 - r_0) eq(rP, g) V[2g+1], whose sums and folds are again linear
    // in V with product weights, those of a folded coordinate e_m L_m instead
    // of e_m: an instance of its own over the odd entries (PK_TREE2B), whose
    // sums join round j >= 1 of PK_TREE2 in the final reduction.
    PK_TREE2 = 7,
    PK_TREE2B = 8,
    PK_GEN_FIRST = 16,
    PK_GEN_EZ = 16,    // phase 2 of SQUARE, F0 and (values in host memory) TREE layers, P and B formed from
                       // the wiring (times eq(z, rP))
    PK_GEN_PAIR2 = 17,   // phase 2 of F0_PAIR and
    PK_GEN_FINAL2 = 18,  // F0_FINAL layers with a first wave in registers (bil_run)
    PK_GEN_TAB = 19    // tables built by k_build23 (EXPLICIT) or k_mm_tables (MATMULT)
};

// Source of the first GEN wave's P and B.
//   SQ2     P[x] = eq(rP, x) V[x]
//   PAIR2   P[2q] = eq(rP, 2q) V[2q], P[2q+1] = eq(rP, 2q+1) V[2q]
//   FINAL2  P[2q+1] = eq(rP, q) V[2q+1], P[2q] = 0
//   FIRST2  P[x] = eq(rP, 2x) V[x] + eq(rP, 2x+1), B[x] = eq(rP, 2x+1) V[x]
//   MM2     P[(k, i, 0)] = u[k] ei[i] (inP, inB: the tables of k_mm_tables), P[(., ., 1)] = 0
//   TREE2   P[2g] = eq(rP, g), B[2g] = P[2g] V[2g+1], P and B 0 at odd entries
//           (values in host memory only: one pass over V, where PK_TREE2 and
//           PK_TREE2B are two and the odd entries' sectors cross the link twice)
enum : u32 { GS_NONE = 0, GS_SQ2 = 1, GS_PAIR2 = 2, GS_FINAL2 = 3, GS_FIRST2 = 4, GS_MM2 = 5, GS_TREE2 = 6 };

// PROD: a chunk of more than 2^PR_C entries is a matrix of 2^kr rows of 2^PR_C
// columns, kr <= PR_R (128 threads per CTA)
#define PR_C 7
#define PR_R 7
// Words of the message-weight table of kk coordinates (see ProdWave::wblk).
__host__ __device__ __forceinline__ u32 vec_slots(u32 kk) { return kk > 5 ? 1u << (kk - 5) : 1u; }
__host__ __device__ __forceinline__ u32 vec_words(u32 kk) { return vec_slots(kk) * kk * 16; }
#define GN_M 5  // GEN: at most 2^5 entries per thread (128 threads per CTA)
// Evaluation runs holding F0_PAIR layers take chunks of at most 2^8 input
// entries: one pair per thread of a 256-thread evaluation CTA.
#define EV_PAIR_CHUNK 8

struct SciDev {
    u32 circ;
    u32 n;         // rounds
    u32 kind;      // PK_*
    u32 layer;
    u32 chal_off;  // challenge of round k: chal[chal_off + k]
    u64 tr_off;    // transcript offset of round 0's three values
    u64 *Lc;       // PROD: factors c0_m, c1_m (2n), written by the coin launch
    u64 *kap;      // PROD: prod_{m<j} L_m(r_m)
    u64 *esum;     // PROD: prod_{m>j} (c0_m + c1_m)
};

// One wave of a PROD SCI: each CTA takes a chunk of 2^nr entries, nr = kc + kr
// (kc low coordinates: columns, kr high ones: rows; kr > 0 only with kc = PR_C).
// wblk, the wave's weights (k_coins; e_m(b) the fold's factor of local
// coordinate m, L_m the instance's):
//   kr > 0: colw[x] = prod_{m<kc} e_m(x_m) (2^kc words, the fold of the columns),
//           roww[y] = prod_{m>=kc} L_m(y_m) (2^kr words, the rows' weight)
//   message weights of the columns, and of the rows if kr > 0: over the kk
//           coordinates from a, entry y of round j (y: the other kk - 1 bits)
//           prod_{m<j} e_{a+m}(y_m) prod_{m>j} L_{a+m}(y_{m-1}), at
//           word (y / 16) 16 kk + 16 j + y mod 16
//   e(0), e(1) of the last column coordinate, then of the last row coordinate
//   outer lo / hi: split table of prod_{m >= r0+nr} L_m over the chunk index
struct ProdWave {
    u32 circ;
    u32 sci;
    u32 r0, nr, kc, kr;
    u32 nchunks;
    u32 flags;
    u32 no, ho;        // coordinates beyond the chunk (r0+nr..n-1) and their split
    const u64 *in;     // entries of this wave's table
    u64 *out;          // one folded value per chunk (unused on the last wave)
    u64 *wblk;
    u64 *part;         // partials: part[(k * nchunks + chunk) * 2 + t]
    u32 *counter;      // chunks finished (WF_TAIL only; reset by the last)
};
// Offsets in wblk.
__host__ __device__ __forceinline__ u32 pw_roww(u32 kr) { return kr ? 1u << PR_C : 0u; }
__host__ __device__ __forceinline__ u32 pw_tcol(u32 kr) { return kr ? (1u << PR_C) + (1u << kr) : 0u; }
__host__ __device__ __forceinline__ u32 pw_trow(u32 kc, u32 kr) { return pw_tcol(kr) + vec_words(kc); }
__host__ __device__ __forceinline__ u32 pw_last(u32 kc, u32 kr) { return pw_trow(kc, kr) + (kr ? vec_words(kr) : 0u); }
__host__ __device__ __forceinline__ u32 pw_outer(u32 kc, u32 kr) { return pw_last(kc, kr) + 4; }

// One wave of a GEN SCI.
struct GenWave {
    u32 circ;
    u32 sci;
    u32 r0, nr, e;
    u32 nchunks;
    u32 flags;
    u32 src;           // GS_* (first wave only)
    u32 layer;
    u32 chal_off;
    u32 pad;
    u32 th;            // first wave with a source: its factor of entry x (SQ2, PAIR2, MM2), x / 2 (FINAL2, TREE2)
                       // or 2 x (FIRST2) is lo[index mod 2^th] hi[index >> th]; lo is inP, hi is inB
    u32 pad2;
    const u64 *inP, *inV, *inB;
    u64 *outP, *outV, *outB;
    u64 *part;         // partials: part[(k * nchunks + chunk) * 3 + t]
    u32 *counter;      // chunks finished (WF_TAIL only; reset by the last)
};

// Line reduction of layer i (q(t) = V~_{i+1}(l(t)), l(t) = r1 + t (r2 - r1)),
// computed by folding V_{i+1} with the coordinates a_k + b_k t in coefficient
// form: after folding j coordinates each entry is a polynomial of degree j.
// A wave folds nl = e + kk coordinates of each chunk: e in registers (2^e
// consecutive entries a thread; 0 or 3..8), kk in one step, as the sum over
// the 2^kk threads of their polynomials times the weight polynomials
// prod_m (l_m or 1 - l_m) (wt: coefficient b of thread y at b 2^kk + y).
struct LineWaveDev {
    u32 circ;
    u32 layer;
    u32 n;        // s_{i+1}
    u32 l0, nl;   // coordinates [l0, l0 + nl) folded by this wave
    u32 e, kk;
    u32 nchunks;
    u32 last;
    const u64 *in;  // l0 == 0: V_{i+1}; else coefficient c of poly q at c (nchunks << nl) + q
    u64 *out;       // coefficient c of chunk's poly at c nchunks + chunk (unused on the last wave)
    u64 *wt;        // (kk + 1) 2^kk words
    u32 a_off;      // a_k = chal[a_off + k] (= r1), b_k = chal[b_off + k] - a_k
    u32 b_off;
    u64 tr_q;
    u32 tail;       // the next descriptor (one chunk) is run by this wave's last CTA
    u32 pad;
    u32 *counter;   // CTAs of this wave that finished (tail only; reset by the last)
};

// Work item of a merged launch: which wave descriptor and which chunk.
struct Item {
    u32 wave;
    u32 chunk;
};

// Task of the persistent wave launch: one chunk of a line, PROD or GEN wave.
enum : u32 { TK_LINE = 0, TK_PROD = 1, TK_GEN = 2 };
struct Task {
    u32 type;
    u32 wave;   // index into the plan's line, PROD or GEN wave descriptors
    u32 chunk;
    u32 pad;
};

// Final reduction of one round: sum the chunks' partials (2 per chunk for
// PROD, 3 for GEN) and write g(0), g(1), g(2) at tr[tr_pos].  Every scalar
// the round needs is reached through its own pointer, so the loads are
// independent of one another.
struct RoundRef {
    u64 tr_pos;
    const u64 *part_pos;
    u32 nchunks;
    u32 kind;         // PK_* of the instance
    u32 circ;
    u32 sci;
    u32 j;            // round index within the SCI
    u32 nchunks2;     // TREE phase 2, j >= 1: the PK_TREE2B instance's partials of the round
    const u64 *part2_pos;
    const u64 *ez;    // eq(z_i, r_P) of the layer
    const u64 *v1;    // V~_{i+1}(r1) of the layer
    const u64 *ch;    // the first challenge of phase 2
    const u64 *rp0;   // the first challenge of phase 1 (NULL without one)
    const u64 *lc;    // PROD: c0, c1 of round j
    const u64 *kap;   // PROD: kappa_j
    const u64 *esum;  // PROD: esum_j
};

// Per-circuit globals.  Each circuit keeps one copy in device memory (and a
// batch keeps one per member); kernels find theirs through the `circ` index of
// their work descriptor.  seed and tr change per proof and are written on the
// stream by k_params (or from a parameter table for a batch) before the
// proof's launches, so a captured launch sequence can be replayed.
struct Globals {
    u64 seed;
    u32 d;
    u32 nchal;
    u64 *chal;        // nchal challenges
    u64 *pts;         // z_0 .. z_d
    u64 *scal;        // per-layer scalars (SCAL_*)
    u64 *tr;          // transcript (device)
    u32 *status;      // error flags (bit 0: non-canonical input)
    LayerDev *layers;
    u64 *invfact;     // 1/k! for k < 64 (verifier)
    const u32 *zmap;  // flattened coordinates of z_1..z_d: layer << 8 | k
    u32 nz;
    u32 zd_off;       // z_d in pts[]
    u64 S0;           // outputs
    const u64 *out_src;  // where the final reduction reads the outputs (layer 0, or a
                         // copy of it when the layer values rotate through device slots)
    const u64 *in;    // this proof's inputs when the first evaluation launch reads them
                      // in place (it also writes the input layer's values); set by
                      // k_params, cleared by k_final; NULL: the inputs are in layer d
};

// A run of block-local layers evaluated by one launch (k_eval_seg): layers
// i_hi down to i_lo, chunks of 2^c entries of layer i_hi + 1 per CTA.  The
// CTA that finishes last then evaluates layers i_lo - 1 down to tail_lo
// alone (tail_lo == i_lo: no tail); `counter` counts finished CTAs and is
// reset by the last one.
struct EvalSeg {
    u32 circ;
    u32 i_hi, i_lo;
    u32 c;
    u32 nchunks;
    u32 check_input;  // the run's input layer is the circuit's input layer
    u32 tail_lo;
    u32 warp_from;       // first run layer whose blocks all fit one warp (i_lo - 1: none)
    u32 *counter;
    u32 tail_warp_from;  // first tail layer from which all fit one warp (tail_lo - 1: none)
    u32 pad2;
};

// A layer evaluated on its own (MATMULT or EXPLICIT wiring), by items of 256
// `reps` gates: about 1024 CTAs for wide layers, a gate a thread below 2^19.
#define EVL_REPS 8u
__host__ __device__ __forceinline__ u32 eval_reps(u32 s) { return s <= 18 ? 1u : s >= 21 ? EVL_REPS : 1u << (s - 18); }
struct LayerEval {
    u32 circ;
    u32 layer;
    u32 reps;
    u32 pad;
};

// Work item of k_build23: BUILD_ENTRIES entries of layer i+1's phase-2/3 tables.
struct BuildItem {
    u32 circ;
    u32 layer;
    u32 block;
    u32 pad;
};

// Parameters of one proof in a batch (written from the host each call).
struct CallParams {
    u64 seed;
    u64 *tr;
    const u64 *in;       // the member's inputs (device memory) for the gather launch
    const u64 *in_eval;  // the same when the member's first evaluation launch reads them in
                         // place (written to Globals::in), else NULL
};

// A piece of one batch member's input copy: count entries from the member's
// inputs (CallParams::in) at `start` to dst (its input layer, at `start`).
struct GatherChunk {
    u64 *dst;
    u64 start;
    u32 member;
    u32 count;
};
#define GATHER_CHUNK 2048

#define ST_BAD_INPUT 1u
#define ST_TIMEOUT 2u
#define VC_RESULT_WORDS 8  // verifier result words (device)

// ---- launch entry points (implemented in the .cu files) -------------------------
// An eq table to build, its point the challenges chal[off ..].
struct EqJob {
    EqTab t;
    u32 circ;
    u32 off;
};

void launch_params(Globals *G, u64 seed, u64 *tr, const u64 *in, cudaStream_t st);
const void *params_kernel();   // k_params, to find its node in a captured graph
const void *vparams_kernel();  // k_vparams, likewise
void launch_params_batch(Globals *Gs, const CallParams *cp, int n, cudaStream_t st);
// Every member's inputs into its input layer, one launch (all inputs device memory).
void launch_gather_inputs(const CallParams *cp, const GatherChunk *chunks, int nchunks, cudaStream_t st);
// One launch: setup of every circuit (challenges, points, eq(z_i, r_P), by
// coin_setups(d) CTAs listed as {circuit, slice}), the eq tables and the
// weights of the PROD waves and of the line waves.
__host__ __device__ __forceinline__ u32 coin_setups(u32 d) { return (d + 7) / 8; }
void launch_coins(const Globals *Gs, const Item *setups, int nsetup, const EqJob *eqjobs, int neq,
                  const SciDev *scis, const ProdWave *pw, int npw, const LineWaveDev *lw, int nlw, cudaStream_t st);
void launch_eval_layers(const Globals *Gs, const LayerEval *le, const Item *items, int nitems, cudaStream_t st);
// maxblock: the largest block (entries) of any run layer or tail output in
// the launch (<= 2048); it sizes the two shared-memory buffers.
void launch_eval_segs(const Globals *Gs, const EvalSeg *segs, const Item *items, int nitems, u32 maxblock,
                      cudaStream_t st,
                      bool after_params = false);
void launch_check_canonical(const u64 *x, u64 n, u32 *status, cudaStream_t st);
void launch_check_inputs(const Globals *Gs, const Item *items, int nitems, cudaStream_t st);
void launch_build23(const Globals *Gs, const BuildItem *items, int nitems, cudaStream_t st);
// MATMULT layers' phase-2 factors (BuildItem: MM_ROWS rows of the second matrix).
#define MM_ROWS 8u
void launch_mm_tables(const Globals *Gs, const BuildItem *items, int nitems, cudaStream_t st);
// Explicit layers: an entry w of layer i+1 read by more than BUILD_HEAVY
// gates is summed after launch_build23 by npieces CTAs of up to
// BUILD_PIECE gates each (kind 1: its in1 list, 2: its in2 list); each writes
// its sums to part[2 piece ..], and the last to finish (ctr) adds them all to
// the entry's tables.
#define BUILD_HEAVY 32u
#define BUILD_PIECE 512u
#define BUILD_LANES 8u    // k_build23: threads per entry
#define BUILD_ENTRIES (256u / BUILD_LANES)
struct HeavyItem {
    u32 circ, layer, w, kind;
    u32 piece, npieces, pad0, pad1;
    u64 *part;  // 2 npieces u64
    u32 *ctr;   // zero between proofs (reset by the last piece)
};
void launch_build_heavy(const Globals *Gs, const HeavyItem *items, int nitems, cudaStream_t st);
// One persistent launch over `tasks` (ctr: two zeroed counters, left zeroed).
void launch_waves(const Globals *Gs, const LineWaveDev *lw, const ProdWave *pw, const GenWave *gw, const Task *tasks,
                  int ntasks, u32 *ctr, cudaStream_t st);
// Rounds [0, nbig) are reduced a warp each: all rounds when there are at most
// FINAL_ALL_WARPS (the warps of one full launch), else those with more than
// FINAL_WARP_MIN chunk partials; the rest a thread each (those with up to 8 a
// thread: 196.6 us for the 56-circuit batch, so 194.3).
#define FINAL_WARP_MIN 2u
#define FINAL_ALL_WARPS ((u32)device_sms() * 8u * 8u)
void launch_final(Globals *Gs, const RoundRef *rounds, int nrounds, int nbig, const u32 *outs, int nouts,
                  cudaStream_t st);
void prove_kernels_init();
void waves_init();

// verifier
// Per-call pointers of a verification, written on the stream before the
// verifier's captured launches (so that the launches can be replayed).
struct VerifyPtrs {
    const u64 *tr;      // transcript (device)
    const u64 *inputs;  // S_d inputs (device)
    int *accept_out;    // optional device int receiving the accept bit
    u64 pad;
};

struct VerifyDev {
    u32 d;
    u64 tr_len;
    const VerifyPtrs *vp;  // device
    u64 *mle_part;      // partial sums of the input MLE
    u32 mle_blocks;
    u64 *result;        // [2] accept bit, [3] a check failed (k_vcheck writes both); others unused
    u64 *wire;          // generic add~/mult~ per layer (EXPLICIT layers)
    u64 *wire_part;     // their per-CTA partial sums (two per CTA, VwireItem::part_off)
    u32 *wire_ctr;      // per layer: CTAs done (reset by the last)
    u32 mle_out_blocks; // blocks of the output-MLE partials (after the input's; 0: formed by k_vcheck)
    const u32 *round_layer;  // per global round: layer << 8 | round within layer
    u32 nrounds;
};
// One CTA's share of an explicit layer's generic wiring sum: gates
// [block, block + 1) * ceil(S_i / nblocks); partial sums at part_off + block.
struct VwireItem {
    u32 layer, block, nblocks, part_off;
};
void launch_init_invfact(u64 *invfact, cudaStream_t st);
// result: VC_RESULT_WORDS words, cleared by the launch
void launch_vparams(Globals *G, VerifyPtrs *vp, u64 seed, const u64 *tr, const u64 *inputs, int *accept,
                    u64 *result, cudaStream_t st);
// The verifier's launches after its coin launch was issued on st: the MLE
// partial sums on st_mle (forked from st before the coins, so both run
// together), joined back into st through ev_join, then the checks.
u32 vmle_log(u32 n);
void launch_verify(const Globals *Gd, const Globals &G, const VerifyDev &V, u32 nd, u32 n0, const VwireItem *wire_items,
                   int n_wire, cudaStream_t st_mle, cudaEvent_t ev_join, cudaStream_t st);
// The verifier in two passes.  Input pass: the input's MLE partial sums (the
// coins are launched beside it by the caller).  Transcript pass, with the
// transcript and accept pointer as arguments: the claimed outputs' MLE
// partial sums (many outputs only), add~/mult~ of explicit layers, the checks
// (the eq tables of explicit layers are launched before it by the caller).
void launch_verify_input(const Globals *Gd, const Globals &G, const VerifyDev &V, u32 nd, u32 n0, cudaStream_t st);
void launch_verify_transcript(const Globals *Gd, const Globals &G, const VerifyDev &V, u32 nd, u32 n0,
                              const VwireItem *wire_items, int n_wire, const u64 *tr, int *accept,
                              cudaStream_t st);
void launch_vparams_in(Globals *G, VerifyPtrs *vp, u64 seed, const u64 *inputs, cudaStream_t st);
const void *vparams_in_kernel();
// Circuits with at most this many outputs have their claimed outputs' MLE
// formed inside the check launch, by one warp (more: k_vmle partial sums).
#define VC_OUT_INLINE 256u

// Per-gate prover (k_pergate.cu): one descriptor per layer.
struct PgLayer {
    u32 layer;         // i
    u32 s, sn, n;      // s_i, s_{i+1}, rounds s_i + 2 s_{i+1}
    u32 blk0, nblk;    // CTAs of the gate launches covering this layer's gates
    u32 lblk0, lnblk;  // CTAs of the line launch covering V_{i+1}
    u64 *preP;         // eq over the bound p coordinates (S_i entries; eq(r_P, .) after phase 1)
    u64 *preA, *preB;  // the same over the bound w1 / w2 coordinates (S_{i+1} each)
    u64 *suf;          // phase-1 suffix tables of z_i (S_i - 1 entries)
    u64 *fa, *fb;      // V_{i+1} folded with the bound coordinates (S_{i+1}/2, S_{i+1}/4)
    u64 *v1;           // V~_{i+1}(r1)
    u64 *part;         // per-CTA partial sums of the current round, 3 per CTA
    u64 *ltab;         // line: split eq tables of l(t), t = 0..s_{i+1}
    u64 *lpart;        // line: per-CTA partial sums, s_{i+1} + 1 per CTA
};
// Every launch of a per-gate proof after the evaluation and the coins.
void launch_pergate(const Globals *G, const PgLayer *pl, int nl, const u32 *blk_layer, u32 nblk,
                    const u32 *lblk_layer, u32 nlblk, u32 nrounds, cudaStream_t st);
u32 pergate_gpt();  // gates (and line entries) per CTA

// Special-purpose non-interactive F2 protocol (k_f2sp.cu).  The prover's
// transform (built by vc_f2sp_create): h = q_0 ... q_{m-1}, pairwise coprime
// prime powers <= 61; device tables.
struct SpFftHost {
    u32 h, m, ncs;
    u32 q[8], st[8], magic[8], cso[8];
    const u64 *cs;  // per dimension: its root's (c, s) pairs
    const u32 *pin, *idx;
    const u64 *twist;
};
void sp_init();
u32 sp_prove_ctas(u64 v);
void launch_sp_prove(const u64 *a, u64 v, const SpFftHost &H, u64 *part, u32 nparts, u64 *proof, u32 *status,
                     cudaStream_t st);
void launch_sp_vbegin(u64 seed, u64 v, u64 h, u64 inv_h, const u64 *pw, u64 *L, u64 *M, u64 *acc, u64 *res,
                      cudaStream_t st);
void launch_sp_vabsorb(const u64 *rows, u64 x0, u64 nrows, u64 h, const u64 *L, u64 *acc, u32 *status,
                       cudaStream_t st);
void launch_sp_vend(const u64 *proof, u64 v, u64 h, const u64 *M, const u64 *acc, u64 *res, cudaStream_t st);

// SM count of the current device (queried once per device; 1 if the query
// fails), and the grid of a grid-stride loop over n items capped at per_sm
// CTAs per SM.
int device_sms();
unsigned grid_for_items(u64 n, unsigned threads, unsigned per_sm);
void launch_field_mul(const u64 *a, const u64 *b, u64 *out, u64 n, cudaStream_t st);
double run_field_mul_rate(int variant, u64 iters, int sms, u64 *sink);
