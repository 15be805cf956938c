"""Performance cases of the sliced tensor-network contractor.

Each case is one call a program makes through the package's public entry
points (`paper_2111_01066_gb300.tn`), with the plan or the buffers it keeps
between calls:

* ``plan``     amplitudes of correlated batches of a random circuit:
               ``Plan.contract_slices`` over all slices or a range of them;
* ``pair``     one pairwise contraction of two device tensors
               (``contract_pair``), operands stored ready for streaming
               ("kfast": contracted wires first) or in any order ("random");
* ``permute``  one index permutation (``permute``);
* ``score``    linear XEB of a set of amplitudes and, where asked, frugal
               sampling from it (``xeb``, ``frugal_sample``).

Circuits come from the repository's seeded generator; every tensor dimension
is a power of two because every wire has dimension two, so the ragged sizes
are odd ranks, odd batch counts, slice ranges that start and end inside a
chunk, and amplitude counts.
"""
import functools
import math

import numpy as np
import torch

import rqcgen
from paper_2111_01066_gb300 import tn

PRECISIONS = ("fp32", "tf32", "bf16x3", "fp16x3")


def _plan(name, rows, cols, cycles, circuit_seed, k_open, precision, **more):
    case = dict(name=name, kind="plan", rows=rows, cols=cols, cycles=cycles, circuit_seed=circuit_seed, missing=0,
                k_open=k_open, log2_bound=30, log2_slices=0, log2_chunk=0, trials=64, plan_seed=1, mem_weight=32.0,
                precision=precision, complex_mult=4, first=0, count=0, parts=1, batches=2)
    case.update(more)
    return case


def listed():
    return [
        # a small circuit checked against a state vector: its 32 slices are
        # contracted in three ragged ranges for three batches; launches and
        # latency are all there is
        _plan("plan_12q_fp32", 3, 4, 8, 1, 8, "fp32", log2_slices=5, log2_chunk=3, trials=8, parts=3, batches=3),
        # the 30-qubit circuit in the default precision, unsliced: 148 small steps
        _plan("plan_30q_fp32", 5, 6, 14, 2, 10, "fp32", log2_bound=26),
        # the same circuit sliced over five wires, FP16 split products
        _plan("plan_30q_fp16x3", 5, 6, 14, 2, 10, "fp16x3", log2_bound=26, log2_slices=5),
        # the 42-qubit batch, all 2^12 slices: the library's main workload
        _plan("plan_42q_bf16x3", 6, 7, 16, 3, 12, "bf16x3", log2_bound=28, log2_slices=12, trials=128,
              mem_weight=128.0),
        # one worker's share of that batch in plain FP32: a slice range with
        # ragged ends over chunks of 2^8
        _plan("plan_42q_fp32_range", 6, 7, 16, 3, 12, "fp32", log2_bound=28, log2_slices=12, log2_chunk=8, trials=128,
              mem_weight=128.0, first=1100, count=900, batches=1),
        # the 53-qubit circuit: one 1024-slice chunk of its 2^20 slices
        _plan("plan_53q_bf16x3_chunk", 6, 9, 20, 5, 6, "bf16x3", missing=1, log2_slices=20, log2_chunk=10, trials=128,
              plan_seed=5, first=5 * 1024, count=1024),
        # a compute-bound step: 4096 x 2048 x 4096, split BF16
        dict(name="pair_square_bf16x3", kind="pair", nm=12, nk=11, nn=12, batch=1, precision="bf16x3", complex_mult=4,
             layout="kfast", wire_seed=1),
        # a skewed, memory-bound step whose operands are stored in any order
        dict(name="pair_skewed_tf32", kind="pair", nm=18, nk=6, nn=7, batch=1, precision="tf32", complex_mult=4,
             layout="random", wire_seed=2),
        # many middling instances at once, three products per complex product
        dict(name="pair_batched_bf16x3_3m", kind="pair", nm=9, nk=8, nn=7, batch=45, precision="bf16x3",
             complex_mult=3, layout="kfast", wire_seed=3),
        # the smallest kind of step: launch latency
        dict(name="pair_small_fp32", kind="pair", nm=7, nk=5, nn=4, batch=1, precision="fp32", complex_mult=4,
             layout="random", wire_seed=4),
        # an index permutation of a 2^27-element tensor
        dict(name="permute_27", kind="permute", rank=27, batch=1, perm_seed=5),
        # verification of a million amplitudes, and 2000 samples from them
        dict(name="score_1m", kind="score", count=1000000, n_qubits=53, samples=2000, draws=64),
    ]


def draw(rng):
    kind = rng.choice(("plan", "plan", "plan", "pair", "pair", "pair", "pair", "permute", "permute", "score"))
    precision = rng.choice(PRECISIONS)
    complex_mult = 4 if precision == "fp32" else rng.choice((4, 4, 3))
    if kind == "plan":
        c = _plan(None, rng.randint(3, 5), rng.randint(4, 6), rng.randint(8, 14), rng.randint(10, 10000),
                  rng.randint(3, 10), precision, complex_mult=complex_mult, log2_bound=26,
                  log2_slices=rng.randint(0, 6), trials=rng.choice((8, 16, 32)), parts=rng.randint(1, 3),
                  batches=rng.randint(2, 5))
        del c["name"]
        return c
    if kind == "pair":
        while True:
            nm, nk, nn = rng.randint(2, 20), rng.randint(1, 13), rng.randint(0, 12)
            batch = int(round(2 ** rng.uniform(0, 6)))
            lb = math.log2(batch)
            if max(nm + nk, nk + nn, nm + nn) + lb <= 27 and nm + nk + nn + lb <= 36 and nn <= nm:
                return dict(kind="pair", nm=nm, nk=nk, nn=nn, batch=batch, precision=precision,
                            complex_mult=complex_mult, layout=rng.choice(("kfast", "random")),
                            wire_seed=rng.randint(10, 10000))
    if kind == "permute":
        rank = rng.randint(8, 27)
        return dict(kind="permute", rank=rank, batch=rng.randint(1, 5) if rank <= 24 else 1,
                    perm_seed=rng.randint(10, 10000))
    return dict(kind="score", count=int(2 ** rng.uniform(4, 20)), n_qubits=rng.randint(20, 53),
                samples=int(2 ** rng.uniform(0, 11)), draws=64)


# ------------------------------------------------------------------ the parts of a case


def _circuit(case):
    circ = rqcgen.sycamore_style(case["rows"], case["cols"], case["cycles"], case["circuit_seed"], case["missing"])
    n = circ.n_qubits
    open_mask = ((1 << case["k_open"]) - 1) << (n - case["k_open"])
    return circ, open_mask


def _make_plan(case, circ, open_mask):
    return tn.Plan(tn.Network(circ), open_mask=open_mask, max_log2_intermediate=case["log2_bound"],
                   min_log2_slices=case["log2_slices"], log2_batch_slices=case["log2_chunk"], trials=case["trials"],
                   seed=case["plan_seed"], mem_weight=case["mem_weight"], precision=case["precision"],
                   complex_mult=case["complex_mult"])


def _ranges(case, total):
    """The slice range of the case, cut into its parts at ragged places."""
    first, count = case["first"], case["count"] or total - case["first"]
    parts = min(case["parts"], count)
    cuts = [first + (count * i * i) // (parts * parts) for i in range(parts)] + [first + count]
    cuts = sorted(set(cuts))
    return [(a, b - a) for a, b in zip(cuts, cuts[1:])]


def _bitstrings(case, seed, n_qubits, open_mask):
    """Distinct closed bits of every batch, so that each is a new batch for the plan."""
    rng = np.random.default_rng([seed, 11])
    out = []
    while len(out) < case["batches"]:
        bits = int(sum(int(b) << q for q, b in enumerate(rng.integers(0, 2, size=n_qubits)))) & ~open_mask
        if bits not in out:
            out.append(bits)
    return out


def _pair_wires(case):
    rng = np.random.default_rng([case["wire_seed"], 7])
    nm, nk, nn = case["nm"], case["nk"], case["nn"]
    wires = list(range(nm + nk + nn))
    m, k, n = wires[:nm], wires[nm:nm + nk], wires[nm + nk:]
    mix = lambda v: [int(w) for w in rng.permutation(v)]  # noqa: E731
    if case["layout"] == "kfast":
        return k + m, k + n, m + n
    return mix(m + k), mix(k + n), mix(m + n)


def _normal(shape, seed, dtype, scale):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=dtype, device="cuda") * scale


def _perm(case):
    return [int(p) for p in np.random.default_rng([case["perm_seed"], 9]).permutation(case["rank"])]


def _amplitudes(case, seed):
    """Amplitudes of a random state (Porter-Thomas: complex Gaussian of variance 2^-n)."""
    return _normal((case["count"],), seed, torch.complex128, 2.0 ** (-case["n_qubits"] / 2))


# ------------------------------------------------------------------ one pass


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "plan":
        circ, open_mask = _circuit(case)
        s["plan"] = _make_plan(case, circ, open_mask)
        total = 1 << len(s["plan"].sliced_wires())
        s["ranges"] = _ranges(case, total)
        s["bits"] = _bitstrings(case, seed, circ.n_qubits, open_mask)
        s["out"] = torch.zeros(case["batches"] << case["k_open"], dtype=torch.complex128, device="cuda")
    elif case["kind"] == "pair":
        s["wires"] = _pair_wires(case)
        a_w, b_w, c_w = s["wires"]
        # tensors of about unit norm, as intermediates of a unit-norm state are
        s["a"] = _normal((case["batch"], 1 << len(a_w)), 2 * seed, torch.complex64, 2.0 ** (-len(a_w) / 2))
        s["b"] = _normal((case["batch"], 1 << len(b_w)), 2 * seed + 1, torch.complex64, 2.0 ** (-len(b_w) / 2))
        s["c"] = torch.zeros((case["batch"], 1 << len(c_w)), dtype=torch.complex64, device="cuda")
    elif case["kind"] == "permute":
        s["perm"] = _perm(case)
        s["x"] = _normal((case["batch"], 1 << case["rank"]), seed, torch.complex64, 2.0 ** (-case["rank"] / 2))
        s["y"] = torch.zeros_like(s["x"])
    else:
        s["amps"] = _amplitudes(case, seed)
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        shape = (case["samples"], case["draws"])
        s["candidates"] = torch.randint(0, case["count"], shape, generator=g, device="cuda")
        s["uniforms"] = torch.rand(shape, generator=g, dtype=torch.float64, device="cuda")
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "plan":
        out = state["out"]
        out.zero_()
        for first, count in state["ranges"]:
            state["plan"].contract_slices(first, count, state["bits"], out)
        return out
    if case["kind"] == "pair":
        a_w, b_w, c_w = state["wires"]
        tn.contract_pair(state["a"], a_w, state["b"], b_w, state["c"], c_w, batch=case["batch"],
                         precision=case["precision"], complex_mult=case["complex_mult"])
        return state["c"]
    if case["kind"] == "permute":
        tn.permute(state["x"], state["y"], case["rank"], state["perm"], case["batch"])
        return state["y"]
    f = tn.xeb(state["amps"], case["n_qubits"])
    first = tn.frugal_sample(state["amps"], case["n_qubits"], 10.0, state["candidates"], state["uniforms"])
    return {"xeb": f, "first": np.array(first, dtype=np.int64)}


# ------------------------------------------------------------------ what a pass cannot do without


@functools.lru_cache(maxsize=64)
def _plan_work(key):
    """Complex multiply-adds of the case's contraction tree (8 flops each): the
    steps that depend on the slices for every chunk, those that depend on the
    closed bits alone once per batch; bytes: the gates in, the amplitudes out."""
    case = dict(key)
    circ, open_mask = _circuit(case)
    plan = _make_plan(case, circ, open_mask)
    info = plan.info()
    per_chunk = per_batch = 0.0
    for i, (m, k, n, b) in enumerate(plan.step_shapes()):
        flags = plan.step_layout(i)["dep_flags"]
        if flags & 1:
            per_chunk += 8.0 * 2.0 ** (m + k + n + b)
        elif flags:
            per_batch += 8.0 * 2.0 ** (m + k + n + b)
    total = 1 << info["log2_slices"]
    count = case["count"] or total - case["first"]
    chunks = max(1.0, count / 2.0 ** info["log2_batch_slices"])
    data = 16.0 * sum(m.size for m in circ.gate_matrices) + 16.0 * 2 ** case["k_open"]
    return {"bytes": case["batches"] * data, "flops": case["batches"] * (per_chunk * chunks + per_batch)}


def work(case):
    if case["kind"] == "plan":
        return _plan_work(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    if case["kind"] == "pair":
        m, k, n = 2.0 ** case["nm"], 2.0 ** case["nk"], 2.0 ** case["nn"]
        return {"bytes": 8.0 * case["batch"] * (m * k + k * n + m * n), "flops": 8.0 * case["batch"] * m * k * n}
    if case["kind"] == "permute":
        return {"bytes": 16.0 * case["batch"] * 2.0 ** case["rank"], "flops": 0.0}
    draws = case["samples"] * case["draws"]
    return {"bytes": 16.0 * case["count"] + 32.0 * draws + 8.0 * case["samples"],
            "flops": 4.0 * case["count"] + 6.0 * draws}


# four times the error against 64 bits seen over these ranges (TF32: an operand's
# rounding may also be a truncation; the split modes: the tensor cores' own
# 32-bit accumulation over the longest contractions counts too)
PLAN_TOLERANCE = {"fp32": 6e-6, "tf32": 2e-2, "bf16x3": 2e-4, "fp16x3": 1e-4}
PAIR_TOLERANCE = {"fp32": 6e-6, "tf32": 3e-3, "bf16x3": 8e-5, "fp16x3": 6e-5}


def tolerance(case):
    if case["kind"] == "plan":
        return {"rel": PLAN_TOLERANCE[case["precision"]]}
    if case["kind"] == "pair":
        return {"rel": PAIR_TOLERANCE[case["precision"]]}
    if case["kind"] == "permute":
        return "exact"
    # the XEB of a random state is a mean near 1 less 1; the samples are whole numbers
    return {"rel": 1e-10}


# ------------------------------------------------------------------ the same in 64 bits


def _state_vector(circ):
    """The circuit's state in complex128 on the GPU: every single-qubit gate is
    merged into the next two-qubit gate of its qubit, so the state is passed
    over once per two-qubit gate."""
    n = circ.n_qubits
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    waiting = {q: np.eye(2, dtype=np.complex128) for q in range(n)}

    def two(q0, q1, u):
        # u[(o0, o1), (i0, i1)], row/column index 2 b(q0) + b(q1)
        lo, hi = min(q0, q1), max(q0, q1)
        v = psi.view(1 << (n - 1 - hi), 2, 1 << (hi - lo - 1), 2, 1 << lo)
        at = (lambda b0, b1: v[:, b0, :, b1]) if q0 == hi else (lambda b0, b1: v[:, b1, :, b0])
        old = [at(b >> 1, b & 1).clone() for b in range(4)]
        for r in range(4):
            new = torch.zeros_like(old[0])
            for c in range(4):
                if u[r, c] != 0:
                    new.add_(old[c], alpha=complex(u[r, c]))
            at(r >> 1, r & 1).copy_(new)
            del new

    for (q0, q1), u in zip(circ.gate_qubits.tolist(), circ.gate_matrices):
        if q1 < 0:
            waiting[q0] = u @ waiting[q0]
        else:
            two(q0, q1, u @ np.kron(waiting[q0], waiting[q1]))
            waiting[q0] = waiting[q1] = np.eye(2, dtype=np.complex128)
    for q in range(0, n - 1, 2):
        two(q, q + 1, np.kron(waiting[q], waiting[q + 1]))
    if n % 2:
        two(n - 1, 0, np.kron(waiting[n - 1], np.eye(2)))
    return psi


def _source(positions):
    """Index of every element's source where bit p of an element's index is bit positions[p] of its source's."""
    at = torch.zeros(1, dtype=torch.int64, device="cuda")
    for p in positions:
        at = torch.cat([at, at + (1 << p)])
    return at


def exact(case, seed):
    if case["kind"] == "plan":
        circ, open_mask = _circuit(case)
        if circ.n_qubits > 30 or case["first"] or case["count"]:
            return None
        psi = _state_vector(circ)
        # the open qubits are the top ones: a batch is a strided run of the state
        return torch.cat([psi[b::1 << (circ.n_qubits - case["k_open"])]
                          for b in _bitstrings(case, seed, circ.n_qubits, open_mask)]).clone()
    if case["kind"] == "pair":
        if case["nm"] + case["nk"] + case["nn"] + math.log2(case["batch"]) > 40:
            return None
        s = prepare(case, seed)
        (a_w, b_w, c_w), nm, nk, nn = s["wires"], case["nm"], case["nk"], case["nn"]
        m = [w for w in a_w if w not in b_w]
        n = [w for w in b_w if w not in a_w]
        k = [w for w in a_w if w in b_w]

        def ordered(x, have, want):
            return x[_source([have.index(w) for w in want])]

        out = torch.empty(s["c"].shape, dtype=torch.complex128, device="cuda")
        for i in range(case["batch"]):
            a = ordered(s["a"][i], a_w, k + m).reshape(1 << nm, 1 << nk).to(torch.complex128)
            b = ordered(s["b"][i], b_w, k + n).reshape(1 << nn, 1 << nk).to(torch.complex128)
            c = (b @ a.t()).reshape(-1)                  # stored [m fastest, n]
            out[i] = ordered(c, m + n, c_w)
        return out
    if case["kind"] == "permute":
        s = prepare(case, seed)
        return s["x"][:, _source(s["perm"])].to(torch.complex128)
    s = prepare(case, seed)
    p = s["amps"].real ** 2 + s["amps"].imag ** 2
    f = float(p.mean()) * 2.0 ** case["n_qubits"] - 1.0
    ok = s["uniforms"] * 10.0 < p[s["candidates"]] * 2.0 ** case["n_qubits"]
    first = torch.where(ok.any(1), ok.to(torch.int8).argmax(1), torch.full((), -1, device="cuda"))
    return {"xeb": f, "first": first.cpu().numpy()}
