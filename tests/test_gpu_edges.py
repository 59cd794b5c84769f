"""The kernels at the sizes where their splits change: chunk shapes of the sum-
check waves, chains of power layers around a warp's 32 lanes, gate lists around
the build's pieces, wide evaluation layers, seeds with a rejected coin, and the
row groups of the special-purpose F2 prover.  Every result equals the CPU
oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from gpu_util import ensure_built, first_mismatch, gpu_prove, oracle_prove, to_np
from paper_1202_1350_gb300 import EXPLICIT, F0_FINAL, F0_FIRST, F0_PAIR, MATMULT, SQUARE, TREE, circuits, vc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P = (1 << 61) - 1
M64 = (1 << 64) - 1
GAMMA = 0x9E3779B97F4A7C15


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, np.uint64)).view(np.int64).copy()).cuda()


def elements(seed, n):
    """n field elements over the whole range, both ends among them."""
    x = oracle.splitmix64(seed, n) >> np.uint64(3)
    x[x == P] = 0
    x[::7] = P - 1
    x[3::11] = 0
    return x


def check(widths, kinds, x, seed, explicit=None):
    g, o = gpu_prove(widths, kinds, x, seed, explicit), oracle_prove(widths, kinds, x, seed, explicit)
    assert len(g) == len(o)
    assert first_mismatch(g, o) is None, f"first mismatch at {first_mismatch(g, o)}"


# product-weighted chunks of 2^13 end at 13 and 18 coordinates, those of 2^14
# begin at 19; line chunks of 2^12 and 2^13 part at widths of 2^16; rows of a
# chunk are 2^0 .. 2^7 over 2^7 columns
@pytest.mark.parametrize("logn", [14, 15, 17, 18, 19])
def test_f2_chunk_shapes(logn):
    check(*circuits.f2(logn), elements(logn, 1 << logn), 5 + logn)


# general chunks of 2^10, 2^11 and 2^12 (layers of 12, 13, 15 and 16 coordinates)
@pytest.mark.parametrize("logn", [5, 7, 11, 13, 14])
def test_f0_chunk_shapes(logn):
    check(*circuits.f0(logn), elements(100 + logn, 1 << logn), 9)


def test_matmult_64():
    check(*circuits.matmult(6), elements(60, 1 << 13), 13)


# power layers whose chains of points are found 32 layers at a time, alone and
# under a tree, over widths of a part of a warp, a warp and a chunk
@pytest.mark.parametrize("pairs", [0, 1, 2, 30, 31, 32, 33, 64])
@pytest.mark.parametrize("s", [1, 5, 9])
def test_power_chains(pairs, s):
    widths = [s - 1, s] + [s + 1] * (pairs + 1) + [s]
    kinds = [TREE, F0_FINAL] + [F0_PAIR] * pairs + [F0_FIRST]
    check(widths, kinds, elements(s, 1 << s), 21)
    # a chain that ends on the inputs, beside squaring layers
    if pairs:
        check([s, s, s + 1] + [s + 1] * pairs, [SQUARE, F0_FINAL] + [F0_PAIR] * pairs, elements(s, 2 << s), 22)


# matrix products over the circuit's inputs and over computed values
@pytest.mark.parametrize("L", [1, 3, 4])
def test_matmult_over_computed_values(L):
    w, k = circuits.matmult(L)
    shapes = [(w, k), (w + [2 * L + 1], k + [SQUARE]), (w + [2 * L + 2], k + [TREE])]
    specs = [(w, k, elements(L, 1 << w[-1])) for w, k in shapes]
    for w, k, x in specs:
        check(w, k, x, 17)
    hs = [vc.vc_circuit_create(w, k, None) for w, k, _ in specs]  # and merged
    b = vc.vc_batch_create(hs)
    try:
        for call in range(2):
            trs = [torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda") for h in hs]
            vc.vc_batch_prove(b, [dev(x) for *_, x in specs], [31 + call] * len(hs), trs)
            vc.vc_batch_sync(b)
            for (w, k, x), tr in zip(specs, trs):
                assert (to_np(tr) == oracle_prove(w, k, x, 31 + call)).all()
    finally:
        vc.vc_batch_destroy(b)
        for h in hs:
            vc.vc_circuit_destroy(h)


# one entry read by `reads` gates: eight threads, and pieces of 512 gates past 32
@pytest.mark.parametrize("reads", [7, 8, 9, 31, 32, 33, 511, 512, 513, 1025])
def test_explicit_list_lengths(reads):
    S, Sn = 1 << 11, 1 << 6
    rng = np.random.default_rng(reads)
    in1 = rng.integers(1, Sn, S).astype(np.uint32)
    in2 = rng.integers(1, Sn, S).astype(np.uint32)
    in1[rng.permutation(S)[:reads]] = 0
    in2[rng.permutation(S)[:reads]] = 0
    ex = [(rng.integers(0, 2, S).astype(np.uint8), in1, in2)]
    check([11, 6], [EXPLICIT], elements(reads, Sn), 41, ex)


# one, two, four and eight gates a thread of an evaluation CTA
@pytest.mark.parametrize("s", [18, 19, 20, 21])
def test_wide_evaluation_layers(s):
    S, Sn = 1 << s, 1 << 10
    rng = np.random.default_rng(s)
    ex = [(rng.integers(0, 2, S).astype(np.uint8), rng.integers(0, Sn, S).astype(np.uint32),
           rng.integers(0, Sn, S).astype(np.uint32))]
    check([s, 10], [EXPLICIT], elements(s, Sn), 43, ex)


def unmix(z):
    """The state that splitmix64's output function takes to z."""
    z ^= (z >> 31) ^ (z >> 62)
    z = z * pow(0x94D049BB133111EB, -1, 1 << 64) & M64
    z ^= (z >> 27) ^ (z >> 54)
    z = z * pow(0xBF58476D1CE4E5B9, -1, 1 << 64) & M64
    return z ^ (z >> 30) ^ (z >> 60)


# each of the eight outputs that draw p, as the first, a middle, the last and
# the first unused draw
@pytest.mark.parametrize("low", range(8))
def test_rejected_coins(low):
    w, k = circuits.f2(6)
    nchal = w[0] + sum(w[i] + 2 * w[i + 1] + 1 for i in range(len(k)))
    x = elements(low, 1 << 6)
    h = vc.vc_circuit_create(w, k, None)
    tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
    try:
        for draw in (1, nchal // 2, nchal, nchal + 1):
            seed = (unmix(8 * P + low) - draw * GAMMA) & M64
            assert int(oracle.splitmix64(seed, draw)[-1]) >> 3 == P
            assert vc.vc_prove_verify(h, dev(x), seed, tr)
            assert (to_np(tr) == oracle_prove(w, k, x, seed)).all(), draw
    finally:
        vc.vc_circuit_destroy(h)


# rows of a CTA's batch: one, a part, several groups, more rows than a wave of
# CTAs takes, with every dimension small (1024 threads) and with a large one
@pytest.mark.parametrize("v,h", [(2, 9), (19, 13), (19, 61), (305, 7), (700, 3), (37, 143), (157, 65), (9, 123),
                                 (40, 315)])
def test_f2sp_row_groups(v, h):
    a = elements(v + h, v * h)
    s = vc.vc_f2sp_create(v, h)
    try:
        out = torch.empty(2 * h, dtype=torch.int64, device="cuda")
        vc.vc_f2sp_prove(s, dev(a), out)
        proof = oracle.f2sp_prove(a, v, h)
        assert (to_np(out) == proof).all()
        vc.vc_f2sp_verify_begin(s, 77)
        vc.vc_f2sp_verify_absorb(s, dev(a), 0, v)
        ok, f2 = vc.vc_f2sp_verify_end(s, dev(proof))
        assert ok and f2 == sum(int(t) * int(t) for t in a) % P
    finally:
        vc.vc_f2sp_destroy(s)


# values in host memory: addition layers of a part of a warp, one and several
# registers' runs, one and several chunks; against every other kind's layers
@pytest.mark.parametrize("family,logn", [("f2", n) for n in (1, 2, 3, 7, 8, 9, 10, 12, 13, 14, 16)] +
                         [("f0", 9), ("matmult", 4)])
def test_host_values_addition_layers(family, logn):
    w, k = circuits.by_name(family, logn)
    x = elements(logn, 1 << w[-1])
    h = vc.vc_circuit_create(w, k, host_values=True)
    try:
        tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
        vc.vc_prove(h, dev(x), 51, tr)
        vc.vc_circuit_sync(h)
        assert (to_np(tr) == oracle_prove(w, k, x, 51)).all()
        assert vc.vc_verify(h, dev(x), 51, tr)
    finally:
        vc.vc_circuit_destroy(h)
