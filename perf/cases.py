"""What is timed when this framework's speed is judged: the work its users have it do.

A case is one call (or the two or three calls that belong together) through
the package's public entry points: proofs of the paper's circuits, their
verification, merged batches, and the special-purpose F2 protocol.  Sizes are
those of the benchmark's workloads and size sweep and of the serving mix.
Inputs, circuit handles and transcripts are device-resident, as in the
benchmark; every proof starts from the inputs and a seed, nothing is reused
from one pass to the next.
"""
from __future__ import annotations

import math

import torch

from paper_1202_1350_gb300 import api, circuits, vc

P = (1 << 61) - 1
DEVICE = "cuda:0"

# rows of the special-purpose protocol's grid: products of distinct members of
# {9, 3, 25, 5, 7, 11, 13, 31, 41, 61}, from about a hundred to the largest allowed
F2SP_H = [h for h in range(91, 7001) if vc.f2sp_valid_h(h)]


def listed():
    return [
        # the smallest call: one short proof, verified as it is made (a served
        # request of the smallest size); launches and latency are all there is
        {"name": "f2_2e10_prove_verify", "op": "prove_verify", "circuit": "f2", "log": 10, "log2": 0},
        # the headline workload: proof and verification of F2 over 2^20 counts
        {"name": "f2_2e20_prove_verify", "op": "prove_verify", "circuit": "f2", "log": 20, "log2": 0},
        # the largest served request
        {"name": "f2_2e22_prove", "op": "prove", "circuit": "f2", "log": 22, "log2": 0},
        # distinct elements: 62 power layers over few and over many inputs (a deep circuit)
        {"name": "f0_2e11_prove", "op": "prove", "circuit": "f0", "log": 11, "log2": 0},
        {"name": "f0_2e16_prove", "op": "prove", "circuit": "f0", "log": 16, "log2": 0},
        # matrix product of 128 x 128 matrices, 2^14 outputs
        {"name": "matmult_128_prove", "op": "prove", "circuit": "matmult", "log": 7, "log2": 0},
        # explicit wiring with gates that share constants: text of 2^14, pattern of 2^4
        {"name": "pattern_2e14_prove", "op": "prove", "circuit": "pattern", "log": 14, "log2": 4},
        # the verifier alone, from a transcript that arrived: explicit wiring and 68 layers
        {"name": "matmult_check_32_verify", "op": "verify", "circuit": "matmult_check", "log": 5, "log2": 0},
        # many uneven proofs in merged launches: 48 F2 (2^8..2^18), 8 MatMult (16, 32, 64)
        {"name": "batch_56_prove", "op": "batch", "n_f2": 48, "n_mm": 8, "mix": 3},
        # special-purpose F2: about 2^20 and 25 million counts, prover
        {"name": "f2sp_1048x1001_prove", "op": "f2sp_prove", "v": 1048, "h": 1001},
        {"name": "f2sp_4995x5005_prove", "op": "f2sp_prove", "v": 4995, "h": 5005},
        # and its verifier over rows that are on the device
        {"name": "f2sp_4995x5005_verify", "op": "f2sp_verify", "v": 4995, "h": 5005},
    ]


def draw(rng):
    plain = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in plain:
            return case


def _draw(rng):
    op = rng.choice(["prove", "prove", "prove", "prove_verify", "prove_verify", "verify", "batch", "f2sp_prove",
                     "f2sp_verify"])
    if op == "batch":
        n = int(round(math.exp(rng.uniform(math.log(8), math.log(64)))))
        return {"op": op, "n_f2": n - n // 8, "n_mm": n // 8, "mix": rng.randrange(1 << 20)}
    if op in ("f2sp_prove", "f2sp_verify"):
        h = rng.choice(F2SP_H)
        n = math.exp(rng.uniform(math.log(1 << 14), math.log(8 << 20)))
        return {"op": op, "v": max(1, int(n / h)), "h": h}
    name = rng.choice(["f2", "f2", "f2", "f0", "f0", "matmult", "pattern", "pattern", "matmult_check"])
    log2 = 0
    if name == "f2":
        log, log2 = rng.randint(8, 22), rng.randint(0, 6)
    elif name == "f0":
        log, log2 = rng.randint(6, 16), rng.randint(0, 4)
    elif name == "matmult":
        log = rng.randint(3, 7)
    elif name == "pattern":
        log, log2 = rng.randint(7, 15), rng.randint(2, 5)
    else:
        log = rng.randint(2, 5)
    return {"op": op, "circuit": name, "log": log, "log2": log2}


def _shape(case):
    """(log widths, wiring kinds, explicit layers or None)."""
    c, n = case["circuit"], case["log"]
    if c == "pattern":
        return circuits.pattern_match(n, case["log2"])
    if c == "matmult_check":
        return circuits.matmult_check(n)
    return (*_grouped(c, n, case["log2"]), None)


def _grouped(name, log, log2):
    """(log widths, wiring kinds) of a benchmark circuit; F2 and F0 of
    2^log2 groups of counts at once: the tree stops 2^log2 outputs wide."""
    w, kinds = circuits.by_name(name, log)
    return w[log2:], kinds[log2:]


def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _ints(g, n, hi):
    return torch.randint(0, hi + 1, (n,), generator=g, device=DEVICE, dtype=torch.int64)


def _inputs(name, log, log2, g):
    """The circuit's inputs in earnest: counts in [0, 2^16], frequencies from
    Poisson(1), matrix entries in [0, 2^10], text over four symbols with the
    pattern planted, a claimed product with up to n wrong entries."""
    n = 1 << log
    if name == "f2":
        return _ints(g, n, 1 << 16)
    if name == "f0":
        return torch.poisson(torch.ones(n, device=DEVICE), generator=g).long().clamp_(max=1 << 10)
    if name == "matmult":
        return _ints(g, 2 * n * n, 1 << 10)
    if name == "pattern":
        q = 1 << log2
        x = torch.zeros(2 * n, dtype=torch.int64, device=DEVICE)
        x[:n + q] = _ints(g, n + q, 3)
        for k in range(3):
            at = (k * n) // 3
            if at + q <= n:
                x[at:at + q] = x[n:n + q]
        x[n + q] = P - 1
        x[n + q + 1] = 1
        return x
    ab = _ints(g, 2 * n * n, 1 << 10)
    a, b = ab[:n * n].reshape(n, n).double(), ab[n * n:].reshape(n, n).double()
    c = (a @ b).long().reshape(-1)  # below 2^53: exact
    c[_ints(g, int(_ints(g, 1, n).item()), n * n - 1)] += 1
    x = torch.zeros(4 * n * n, dtype=torch.int64, device=DEVICE)
    x[:2 * n * n] = ab
    x[2 * n * n:3 * n * n] = c
    x[3 * n * n] = P - 1
    return x


class _F2sp:
    """Owner of a special-purpose F2 handle."""

    def __init__(self, v, h):
        self.handle = vc.vc_f2sp_create(v, h)

    def __del__(self):
        vc.vc_f2sp_destroy(self.handle)


def _batch_jobs(case):
    g = torch.Generator().manual_seed(case["mix"])
    f2 = torch.randint(8, 19, (case["n_f2"],), generator=g).tolist()
    mm = torch.randint(4, 7, (case["n_mm"],), generator=g).tolist()
    return [("f2", n) for n in f2] + [("matmult", n) for n in mm]


def _f2sp_counts(case, seed):
    return _ints(_gen(seed), case["v"] * case["h"], 1 << 16)


def prepare(case, seed):
    op, g = case["op"], _gen(seed)
    proof_seed = seed * 2654435761 + 1
    if op == "batch":
        jobs = _batch_jobs(case)
        cs = [api.Circuit(*circuits.by_name(name, n)) for name, n in jobs]
        return {"op": op, "batch": api.Batch(cs), "circuits": cs,
                "inputs": [_inputs(name, n, 0, g) for name, n in jobs],
                "seeds": [proof_seed + j for j in range(len(jobs))],
                "transcripts": [c.new_transcript() for c in cs]}
    if op in ("f2sp_prove", "f2sp_verify"):
        own = _F2sp(case["v"], case["h"])
        st = {"op": op, "f2sp": own, "v": case["v"], "counts": _f2sp_counts(case, seed), "seed": proof_seed,
              "proof": torch.empty(2 * case["h"], dtype=torch.int64, device=DEVICE)}
        if op == "f2sp_verify":  # the proof that the verifier was sent
            vc.vc_f2sp_prove(own.handle, st["counts"], st["proof"])
        return st
    c = api.Circuit(*_shape(case))
    st = {"op": op, "circuit": c, "inputs": _inputs(case["circuit"], case["log"], case["log2"], g),
          "seed": proof_seed, "transcript": c.new_transcript(),
          "accept": torch.zeros(1, dtype=torch.int32, device=DEVICE)}
    if op == "verify":  # the transcript that the verifier was sent
        c.prove(st["inputs"], st["seed"], st["transcript"])
    return st


def run(state):
    op = state["op"]
    if op == "prove":
        return vc.vc_prove(state["circuit"].handle, state["inputs"], state["seed"], state["transcript"])
    if op == "prove_verify":
        vc.vc_prove_verify(state["circuit"].handle, state["inputs"], state["seed"], state["transcript"],
                           accept=state["accept"])
        return [state["transcript"], state["accept"]]
    if op == "verify":
        vc.vc_verify(state["circuit"].handle, state["inputs"], state["seed"], state["transcript"],
                     accept=state["accept"])
        # what the verifier learns: the claimed answer (it opens the transcript) and whether to believe it
        return [state["transcript"][:state["circuit"].n_outputs], state["accept"]]
    if op == "batch":
        return state["batch"].prove(state["inputs"], state["seeds"], state["transcripts"], sync=False)
    h = state["f2sp"].handle
    if op == "f2sp_prove":
        return vc.vc_f2sp_prove(h, state["counts"], state["proof"])
    vc.vc_f2sp_verify_begin(h, state["seed"])
    vc.vc_f2sp_verify_absorb(h, state["counts"], 0, state["v"])
    accept, f2 = vc.vc_f2sp_verify_end(h, state["proof"])
    return [int(accept), f2]


def _widths(case):
    if case["op"] == "batch":
        return [circuits.by_name(name, n)[0] for name, n in _batch_jobs(case)]
    if case["circuit"] == "pattern":  # the widths alone: no gate arrays
        a, b = case["log"], case["log2"]
        return [[*range(a + 1)] + [a + 1] * 60 + [*range(a, a + b)] + [a + b, a + b, a + 1, a + 1]]
    if case["circuit"] == "matmult_check":
        m = case["log"]
        return [[*range(2 * m + 1)] + [2 * m + 1] * 60 + [*range(2 * m, 3 * m + 1)] + [3 * m + 1, 2 * m + 2]]
    return [_grouped(case["circuit"], case["log"], case["log2"])[0]]


def work(case):
    """Bytes: inputs (and, for the verifier, the transcript) read once, results
    written once.  Operations: field multiply-adds, two each.  A proof needs
    at least one per gate, and one per entry of the table in each of a layer's
    three sum-check phases and in its line reduction; the verifier one per
    input; the special-purpose prover a square per count and per extended
    value and the two transforms between them, at least log2 h each per
    entry; its verifier one per count."""
    op = case["op"]
    if op in ("f2sp_prove", "f2sp_verify"):
        n, h = case["v"] * case["h"], case["h"]
        if op == "f2sp_prove":
            return {"bytes": 8 * (n + 2 * h), "flops": 2 * n * (2 + math.log2(h))}
        return {"bytes": 8 * (n + 2 * h), "flops": 2 * n}
    total_bytes = flops = 0
    for w in _widths(case):
        tr = 8 * circuits.transcript_len(w)
        total_bytes += 8 * (1 << w[-1]) + tr
        if op == "verify":
            flops += 2 * (1 << w[-1])
            continue
        flops += 2 * sum((1 << a) * 2 + 3 * (1 << b) for a, b in zip(w[:-1], w[1:]))
        if op == "prove_verify":
            flops += 2 * (1 << w[-1])
    return {"bytes": total_bytes, "flops": flops}


def exact(case, seed):
    """Transcripts and proofs are whole numbers modulo p with no value in
    floating point to be near to; the verifier's answers are known."""
    op = case["op"]
    if op in ("prove_verify", "verify"):
        return [None, torch.ones(1, dtype=torch.int32)]
    if op == "f2sp_verify":
        a = _f2sp_counts(case, seed)
        return [1, int((a * a).sum().item()) % P]  # counts up to 2^16: the sum is far below 2^63
    return None
