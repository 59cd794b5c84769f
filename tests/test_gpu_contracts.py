"""What the entry points promise beside their results: pointers they take,
stages they mark, tile shapes they keep to, and paths that only wide or
unevenly split tables reach.  Every result equals the CPU oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import ensure_built, oracle_prove, to_np
from paper_1202_1350_gb300 import EXPLICIT, SQUARE, TREE, circuits, vc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P = (1 << 61) - 1


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


# a proof buffer at any byte of device memory, as a copy takes it
@pytest.mark.parametrize("offset", [0, 1, 4, 8, 12])
def test_f2sp_proof_at_any_byte(offset):
    v, h = 19, 13
    a = elements(offset, v * h)
    want = oracle.f2sp_prove(a, v, h)
    buf = torch.full((16 * h + 32,), 0x5A, dtype=torch.uint8, device="cuda")
    s = vc.vc_f2sp_create(v, h)
    try:
        da = dev(a)
        assert vc.lib().vc_f2sp_prove(s, da.data_ptr(), buf.data_ptr() + offset, None) == vc.VC_OK
        torch.cuda.synchronize()
    finally:
        vc.vc_f2sp_destroy(s)
    got = buf.cpu().numpy()
    assert (got[offset:offset + 16 * h].view(np.uint64) == want).all()
    assert (got[:offset] == 0x5A).all() and (got[offset + 16 * h:] == 0x5A).all()


# lines of 25, 31, 41 and 61 values on 32 lanes, then on 16, 8, 4, 2 and one
@pytest.mark.parametrize("v,h", [(3, 25), (3, 31), (3, 41), (100, 61), (3040, 61), (6080, 61), (2000, 155), (30400, 61),
                                 (17176, 123)])
def test_f2sp_shared_lines(v, h):
    a = elements(v + h, v * h)
    s = vc.vc_f2sp_create(v, h)
    try:
        out = torch.empty(2 * h, dtype=torch.int64, device="cuda")
        vc.vc_f2sp_prove(s, dev(a), out)
    finally:
        vc.vc_f2sp_destroy(s)
    assert (out.cpu().numpy().view(np.uint64) == oracle.f2sp_prove(a, v, h)).all()


# two and three large factors in one row length: the even points in closed form,
# and the polynomial through all of them at the verifier's secret points
@pytest.mark.parametrize("v,h", [(2, 775), (304, 775), (152, 2501), (2, 4575), (3, 6355)])
def test_f2sp_two_large_factors(v, h):
    a = elements(v + h, v * h)
    s = vc.vc_f2sp_create(v, h)
    try:
        da, out = dev(a), torch.empty(2 * h, dtype=torch.int64, device="cuda")
        vc.vc_f2sp_prove(s, da, out)
        even = out.cpu().numpy().view(np.uint64)[::2]
        want = (a.astype(object).reshape(v, h) ** 2).sum(axis=0) % P
        assert [int(t) for t in even] == [int(t) for t in want]
        for seed in (1, 2):
            vc.vc_f2sp_verify_begin(s, seed)
            vc.vc_f2sp_verify_absorb(s, da, 0, v)
            assert vc.vc_f2sp_verify_end(s, out) == (True, int(want.sum()) % P)
    finally:
        vc.vc_f2sp_destroy(s)


def prove_us(v, h):
    """Device time of a special-purpose proof, the least of twenty."""
    a = dev(elements(1, v * h))
    out = torch.empty(2 * h, dtype=torch.int64, device="cuda")
    s = vc.vc_f2sp_create(v, h)
    try:
        best = float("inf")
        for _ in range(20):
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            vc.vc_f2sp_prove(s, a, out)
            e.record()
            e.synchronize()
            best = min(best, b.elapsed_time(e) * 1e3)
        return best
    finally:
        vc.vc_f2sp_destroy(s)


def test_f2sp_few_rows_of_a_large_factor():
    """One row of 61 a CTA takes about as long as one of 91 = 7 13 (a line of 61
    in one thread took 3.5 times as long, and twice a thread per value's)."""
    assert prove_us(100, 61) < 2 * prove_us(100, 91)


W, BY_SIZE = vc.VC_SPLIT_WIDEST, vc.VC_TILE_BY_SIZE


def tiles_of(pr, gn, ln, ev, split):
    return {"pr_chunk_log": pr, "gn_chunk_log": gn, "line_chunk_log": ln, "eval_chunk_log": ev, "pr_split_log": split}


def first_chunks(widths, kinds, pr, gn, ln, split):
    """Chunks of every instance's and line's first wave (SQUARE and TREE
    layers), by the documented meaning of the tile shapes."""
    widest = max(widths)
    split = widest if split == W else split

    def chunks(n, c):
        return 1 << (n - min(n, c)) if n > 0 else 0

    total = 0
    for i, kind in enumerate(kinds):
        si, sn = widths[i], widths[i + 1]
        prod = [si, sn] if kind == SQUARE else [si, sn, sn - 1, sn]
        total += sum(chunks(n, pr - 1 if n < split and pr > 1 else pr) for n in prod)
        total += chunks(sn, gn) if kind == SQUARE else 0
        total += 1 << (sn - min(sn, ln))
    return total


# numbers at the top of their range, below it, and with each kind of split
@pytest.mark.parametrize("shape", [(13, 12, 13, 11, W), (13, 12, 13, 11, 0), (13, 12, 13, 11, 15), (12, 11, 12, 11, W),
                                   (13, 10, 9, 10, 14), (1, 7, 7, 11, W)])
@pytest.mark.parametrize("logn", [12, 15, 17, 21])
def test_explicit_tiles_are_used_as_they_are(shape, logn):
    w, k = circuits.f2(logn)
    pr, gn, ln, ev, split = shape
    h = vc.vc_circuit_create_tiles(w, k, tiles_of(*shape))
    try:
        assert vc.vc_circuit_get_tiles(h) == tiles_of(*shape)
        assert vc.vc_circuit_get_info(h)["wave_tasks"] == first_chunks(w, k, pr, gn, ln, split)
    finally:
        vc.vc_circuit_destroy(h)


@pytest.mark.parametrize("logn", [13, 20])
def test_default_tiles_are_named_by_size(logn):
    """What a circuit without tiles reports is what it was planned with: the
    same shapes again give the same plan, and a numeric split leaves the sizes
    of wider instances' chunks alone.  (Sizes that no test has tuned: a recorded
    choice would be what such a circuit reports.)"""
    w, k = circuits.f2(logn)
    hs = [vc.vc_circuit_create(w, k)]
    try:
        t = vc.vc_circuit_get_tiles(hs[0])
        assert t == tiles_of(BY_SIZE, BY_SIZE, BY_SIZE, 11, W)
        hs.append(vc.vc_circuit_create_tiles(w, k, t))
        hs.append(vc.vc_circuit_create_tiles(w, k, dict(t, pr_split_log=0)))
        tasks = [vc.vc_circuit_get_info(h)["wave_tasks"] for h in hs]
        assert tasks[0] == tasks[1] and tasks[2] <= tasks[0]
    finally:
        for h in hs:
            vc.vc_circuit_destroy(h)


# explicit shapes whose general first waves form their tables with one entry, 4
# and 32 entries a thread, from split tables with several upper factors
@pytest.mark.parametrize("family,logn", [("f0", 11), ("f2", 12), ("matmult", 6)])
@pytest.mark.parametrize("gn", [7, 9, 12])
def test_explicit_general_chunks(family, logn, gn):
    w, k = circuits.by_name(family, logn)
    x = elements(gn, 1 << w[-1])
    h = vc.vc_circuit_create_tiles(w, k, tiles_of(13, gn, 13, 11, W))
    try:
        tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
        vc.vc_prove(h, dev(x), 61, tr)
        vc.vc_circuit_sync(h)
        assert (to_np(tr) == oracle_prove(w, k, x, 61)).all()
    finally:
        vc.vc_circuit_destroy(h)


# a single general instance of 10 .. 13 coordinates, in a circuit and beside others
@pytest.mark.parametrize("logn", [10, 11, 12, 13])
def test_lone_general_instances(logn):
    for w, k in (circuits.f2(logn), ([logn - 1, logn], [TREE]), ([logn, logn], [SQUARE]),
                 ([logn] * 4, [SQUARE] * 3)):
        x = elements(logn, 1 << w[-1])
        h = vc.vc_circuit_create(w, k)
        try:
            tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
            assert vc.vc_prove_verify(h, dev(x), 71, tr)
            assert (to_np(tr) == oracle_prove(w, k, x, 71)).all()
        finally:
            vc.vc_circuit_destroy(h)


def stage_times(widths, kinds, x, explicit=None):
    """(start, end) of every stage in ms after the proof's start, negative for
    a stage that the proof did not mark."""
    h = vc.vc_circuit_create(widths, kinds, explicit)
    try:
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(2 * vc.NUM_STAGES)]
        for e in evs:
            e.record()
        torch.cuda.synchronize()
        vc.vc_circuit_set_stage_events(h, evs)
        tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
        xd = dev(x)
        for _ in range(2):
            vc.vc_prove(h, xd, 81, tr)
        vc.vc_circuit_sync(h)
        torch.cuda.synchronize()
        assert (to_np(tr) == oracle_prove(widths, kinds, x, 81, explicit)).all()
        t = [evs[0].elapsed_time(e) for e in evs]
        return list(zip(t[::2], t[1::2]))
    finally:
        vc.vc_circuit_destroy(h)


PROOF, TABLES, EVAL, WAVES, WAVESN, BUILD, TABWAVES, FINAL = range(8)


def test_stages_of_matrix_products():
    """The launch that forms MATMULT layers' factors is inside a marked stage,
    wherever it runs (the marks of one stream are ordered among themselves)."""
    L = 4
    w, k = circuits.matmult(L)
    t = stage_times(w, k, elements(1, 1 << w[-1]))  # over the inputs: beside the evaluation
    assert t[BUILD][0] < 0 and 0 <= t[TABLES][0] <= t[TABLES][1] and 0 <= t[EVAL][1] <= t[WAVES][0]
    w, k = w + [2 * L + 1], k + [SQUARE]  # over computed values: a stage before the waves
    t = stage_times(w, k, elements(2, 1 << w[-1]))
    assert t[EVAL][1] <= t[BUILD][0] <= t[BUILD][1] <= t[WAVES][0] <= t[WAVES][1] <= t[FINAL][0]
    S = 1 << w[-1]  # with explicit layers, whose tables come after the waves
    ex = [None] * len(k) + [(np.arange(S, dtype=np.uint8) % 2, np.arange(S, dtype=np.uint32),
                             np.arange(S, dtype=np.uint32)[::-1].copy())]
    w, k = w + [2 * L + 1], k + [EXPLICIT]
    t = stage_times(w, k, elements(3, 1 << w[-1]), ex)
    assert t[WAVES][1] <= t[BUILD][0] <= t[BUILD][1] <= t[TABWAVES][0] <= t[FINAL][0]


# layers of 22 and 23 coordinates: line chunks of 8 coordinates a thread and a
# third line wave, product-weighted chunks of 2^14 whose next wave has one or two
# row coordinates over values that the same launch wrote; with explicit shapes two
# to four
@pytest.mark.parametrize("widths,kinds,shapes", [
    ([21, 22], [TREE], [None, (11, 12, 13, 11, 0), (12, 11, 12, 11, W)]),
    ([22, 22], [SQUARE], [None, (9, 12, 13, 11, 0)]),
    ([22, 23], [TREE], [None])])
def test_wide_layers(widths, kinds, shapes):
    x = elements(sum(widths), 1 << widths[-1])
    want = oracle_prove(widths, kinds, x, 91)
    xd = dev(x)
    for shape in shapes:
        h = vc.vc_circuit_create(widths, kinds) if shape is None else \
            vc.vc_circuit_create_tiles(widths, kinds, tiles_of(*shape))
        try:
            tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
            for _ in range(2):
                assert vc.vc_prove_verify(h, xd, 91, tr), shape
                assert (to_np(tr) == want).all(), shape
                tr.zero_()
        finally:
            vc.vc_circuit_destroy(h)


# later product-weighted waves of 2^8 chunks (one row coordinate) and of a part
@pytest.mark.parametrize("pr,logn", [(8, 17), (8, 16), (9, 18), (10, 15)])
def test_later_waves_with_rows(pr, logn):
    w, k = circuits.f2(logn)
    x = elements(pr, 1 << logn)
    h = vc.vc_circuit_create_tiles(w, k, tiles_of(pr, 12, 13, 11, 0))
    try:
        tr = torch.empty(vc.vc_transcript_len(h), dtype=torch.int64, device="cuda")
        vc.vc_prove(h, dev(x), 101, tr)
        vc.vc_circuit_sync(h)
        assert (to_np(tr) == oracle_prove(w, k, x, 101)).all()
    finally:
        vc.vc_circuit_destroy(h)


def test_multiply_accumulate_rate_is_of_whole_products():
    """Variant 4's exact multiply-accumulates against variant 2's pair steps
    (three products each).  The multiply pipe bounds both: a product is four
    wide ones, eight of the 10.5 pipe cycles a product of the pair step takes
    by the counters, so a multiply-accumulate is at most 10.5 / 8 = 1.31 times as
    fast (1.5 times when parts of the products left the loop)."""
    pair, mac = (max(vc.vc_field_mul_rate(0, v, 1 << 12) for _ in range(3)) for v in (2, 4))
    assert mac < 1.35 * pair
