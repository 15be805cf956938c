"""Kernel variants at the sizes where their tiles, splits and dispatch rules change."""
import numpy as np
import pytest

from oracle import pairwise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2111_01066_gb300 import tn
    torch.cuda.set_device(0)
    return tn, torch


def _pair_case(torch, shape, batch, layout, seed, misaligned=False):
    nm, nk, nn = shape
    rng = np.random.default_rng(seed)
    w = list(range(nm + nk + nn))
    m, k, n = w[:nm], w[nm:nm + nk], w[nm + nk:]
    if layout == "kfast":
        a_w, b_w, c_w = k + m, k + n, m + n
    else:
        a_w, b_w, c_w = (list(rng.permutation(v)) for v in (m + k, k + n, m + n))
    draw = lambda r: ((rng.normal(size=(batch, 2 ** r)) + 1j * rng.normal(size=(batch, 2 ** r))) / 2).astype(np.complex64)
    a, b = draw(nm + nk), draw(nk + nn)

    def dev(x):   # misaligned: one element past a 16-byte boundary
        pad = 1 if misaligned else 0
        t = torch.empty(x.size + pad, dtype=torch.complex64, device="cuda")[pad:].view(x.shape)
        return t.copy_(torch.from_numpy(x))

    c = dev(np.full((batch, 2 ** (nm + nn)), np.nan, dtype=np.complex64))
    return (a, a_w, b, b_w, c_w), (dev(a), a_w, dev(b), b_w, c, c_w)


@pytest.mark.parametrize("misaligned", [False, True])
@pytest.mark.parametrize("layout", ["kfast", "random"])
@pytest.mark.parametrize("shape,batch", [
    ((5, 5, 5), 1), ((4, 6, 5), 3), ((6, 7, 4), 2), ((0, 1, 0), 1), ((5, 0, 5), 1),        # 32x32: one tile, one chunk
    ((6, 6, 6), 1), ((5, 8, 5), 1), ((7, 10, 6), 1), ((3, 13, 2), 5), ((6, 8, 1), 7),      # split-K clusters of 2, 4, 8
    ((3, 2, 17), 1), ((10, 5, 5), 20),                                                      # many 32x32 tiles
    ((7, 3, 6), 130), ((12, 4, 9), 1), ((8, 2, 13), 3),                                     # 128x64: short and whole k
    ((14, 3, 2), 2), ((15, 5, 1), 1), ((9, 4, 0), 200), ((12, 6, 4), 5), ((13, 1, 3), 9),  # 256x4 and 128x16
    ((6, 4, 8), 33), ((5, 6, 9), 70)])                                                      # 64x64
def test_fp32_tilings_at_their_edges(env, shape, batch, layout, misaligned):
    """Every CUDA-core tiling the dispatch rule picks, at tile edges, with part
    tiles, k split over thread groups and clusters, and operands that rule
    16-byte loads out: within the rounding bound of FP32 sums in any order,
    |error| <= (2 k + 2) u sum |a| |b|, u = 2^-24 (each component is a sum of 2k
    products)."""
    tn, torch = env
    (a, a_w, b, b_w, c_w), dev = _pair_case(torch, shape, batch, layout, sum(shape) * 100 + batch, misaligned)
    tn.contract_pair(*dev, batch=batch)
    tn.device_sync()
    got = dev[4].cpu().numpy()
    for i in range(batch):
        want = pairwise.contract_pair(a[i].astype(np.complex128), a_w, b[i].astype(np.complex128), b_w, c_w)
        mag = pairwise.contract_pair(np.abs(a[i]).astype(np.complex128), a_w, np.abs(b[i]).astype(np.complex128), b_w,
                                     c_w).real
        bound = (2 * 2 ** shape[1] + 2) * 2.0 ** -24 * mag
        assert np.all(np.abs(got[i].real - want.real) <= bound)
        assert np.all(np.abs(got[i].imag - want.imag) <= bound)


@pytest.mark.parametrize("prec", ["fp32", "fp16x3"])
def test_chunk_graphs_across_calls(env, prec):
    """The chunk's two launch sequences (with and without a batch's prologue) run
    eagerly, then captured, in calls of few and of many chunks: the parameter
    buffer (1024 chunks at first) grows after the capture, batches open with a
    new bitstring or the previous one, and every call gives the state vector's
    amplitudes."""
    import rqcgen
    from oracle import statevector as sv
    tn, torch = env
    circ, _, _ = rqcgen.config_circuit("c1")
    om = 0b111100001111
    psi = sv.simulate(circ)
    plan = tn.Plan(tn.Network(circ), open_mask=om, max_log2_intermediate=30, min_log2_slices=5, log2_batch_slices=1,
                   trials=8, precision=prec)
    n = 1 << plan.info()["log2_slices"]
    per = n >> plan.info()["log2_batch_slices"]
    many = 1024 // per + 3
    rng = np.random.default_rng(5)
    draw = lambda count: [int(b) << 4 for b in rng.integers(0, 16, size=count)]
    for bits in ([0x30], [0x30, 0x30, 0x50], draw(3), draw(many), draw(2)):
        out = torch.zeros(len(bits) << 8, dtype=torch.complex128, device="cuda")
        plan.contract_slices(0, n, bits, out)
        plan.sync()
        want = np.concatenate([sv.batch_amplitudes(psi, circ.n_qubits, b, om) for b in bits])
        got = out.cpu().numpy()
        assert np.linalg.norm(got - want) < (1e-5 if prec == "fp32" else 1e-4) * np.linalg.norm(want)


@pytest.mark.parametrize("count", [1, 7, 255, 1024, 1025, 4096, 100003, 4 * 152 * 1024 - 1, 4 * 152 * 1024 + 1, 2000003])
def test_xeb_block_counts(env, count):
    """One block, a few, the most, and more rounds than one per block; twice in a
    row (the ticket is left at zero), the same bits both times.  |error| <= 2^n
    mean * (terms a thread adds + the trees) * 2^-53, below 1e-12 here."""
    tn, torch = env
    rng = np.random.default_rng(count)
    a = (rng.normal(size=count) + 1j * rng.normal(size=count)) * 2.0 ** -10
    t = torch.from_numpy(a).cuda()
    f = tn.xeb(t, 20)
    want = 2.0 ** 20 * np.mean(a.real ** 2 + a.imag ** 2) - 1.0
    assert abs(f - want) <= 1e-12 * (1.0 + abs(want))
    assert tn.xeb(t, 20) == f


def test_scoring_calls_from_several_threads(env):
    """tn_xeb and tn_frugal_sample share one scratch area per device: calls from
    several threads, each on a stream of its own, give what they give alone,
    and leave the area fit for the next call."""
    import threading
    tn, torch = env
    rng = np.random.default_rng(11)
    jobs = []
    for t, count in enumerate((3001, 100003, 500000, 1 << 20)):
        a = torch.from_numpy((rng.normal(size=count) + 1j * rng.normal(size=count)) * 2.0 ** -10).cuda()
        cand = torch.from_numpy(rng.integers(0, count, size=(50 + t, 16))).cuda()
        u = torch.from_numpy(rng.random((50 + t, 16))).cuda()
        jobs.append((a, cand, u, tn.xeb(a, 20), tn.frugal_sample(a, 20, 10.0, cand, u)))
    wrong = []

    def work(job, stream):
        a, cand, u, f, first = job
        for _ in range(100):
            if tn.xeb(a, 20, stream=stream) != f or tn.frugal_sample(a, 20, 10.0, cand, u, stream=stream) != first:
                wrong.append(a.numel())

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(j, torch.cuda.Stream())) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    for a, cand, u, f, first in jobs:
        assert tn.xeb(a, 20) == f and tn.frugal_sample(a, 20, 10.0, cand, u) == first


@pytest.mark.parametrize("misaligned", [False, True])
@pytest.mark.parametrize("kind", ["random", "identity", "reverse", "rotate", "swap ends"])
@pytest.mark.parametrize("rank,batch", [(9, 3), (10, 1), (11, 3), (12, 1), (13, 5), (12, 700), (14, 153), (22, 1)])
def test_permute_tiles_bit_exact(env, rank, batch, kind, misaligned):
    """Both tile sizes (4096 elements from four tiles per SM on), one tile to many
    per block, orders whose tile bits are the same or disjoint on both sides,
    arrays that rule 16-byte accesses out; nothing outside the output is written."""
    tn, torch = env
    perm = {"random": lambda: [int(p) for p in np.random.default_rng(rank).permutation(rank)],
            "identity": lambda: list(range(rank)), "reverse": lambda: list(range(rank))[::-1],
            "rotate": lambda: [(p + 4) % rank for p in range(rank)],
            "swap ends": lambda: [rank - 1] + list(range(1, rank - 1)) + [0]}[kind]()
    n = batch << rank
    pad = 1 if misaligned else 0
    x = torch.arange(n + 2, device="cuda", dtype=torch.float32)[pad:pad + n]
    x = torch.complex(x, -x)
    xin = torch.zeros(n + 2, dtype=torch.complex64, device="cuda")
    xin[pad:pad + n] = x
    y = torch.full((n + 2,), 7.0, dtype=torch.complex64, device="cuda")
    tn.permute(xin[pad:pad + n], y[pad:pad + n], rank, perm, batch)
    at = torch.zeros(1, dtype=torch.int64, device="cuda")
    for p in perm:
        at = torch.cat([at, at + (1 << p)])
    want = x.view(batch, 1 << rank)[:, at].reshape(-1)
    assert torch.equal(y[pad:pad + n], want)
    rest = torch.cat([y[:pad], y[pad + n:]])
    assert torch.all(rest == 7.0)


PAIR_REL = {("tf32", 4): 3e-3, ("tf32", 3): 3e-3, ("bf16x3", 4): 4e-5, ("bf16x3", 3): 4e-5, ("fp16x3", 4): 2e-5,
            ("fp16x3", 3): 2e-5}


@pytest.mark.parametrize("prec,cm", sorted(PAIR_REL))
@pytest.mark.parametrize("shape,batch,layout,misaligned", [
    ((14, 2, 9), 1, "random", False), ((13, 3, 9), 1, "kfast", False), ((13, 5, 7), 1, "kfast", True),   # around a k chunk
    ((14, 6, 3), 5, "kfast", False), ((9, 13, 3), 3, "random", False),                                  # narrow, split k
    ((4, 10, 6), 40, "random", False), ((6, 6, 9), 17, "kfast", False),                                 # part row tiles
    ((8, 9, 8), 2, "kfast", False), ((10, 7, 9), 1, "random", False), ((9, 11, 6), 1, "kfast", False)])  # SM pairs
def test_tensor_core_tiles_at_their_edges(env, shape, batch, layout, misaligned, prec, cm):
    """Tensor-core contractions around a k chunk (16), with narrow and part
    tiles, several instances and split k, operands in streaming or any order, or
    off a 16-byte boundary (no tensor-map or 16-byte loads).  Norm-wise: TF32
    operands carry 2^-11, the split modes 2^-16 (BF16) or 2^-21 (FP16) plus the
    tensor cores' 32-bit accumulation over 2^13 products at most."""
    tn, torch = env
    (a, a_w, b, b_w, c_w), dev = _pair_case(torch, shape, batch, layout, sum(shape) * 10 + batch, misaligned)
    tn.contract_pair(*dev, batch=batch, precision=prec, complex_mult=cm)
    tn.device_sync()
    fp32 = torch.empty_like(dev[4])
    tn.contract_pair(*dev[:4], fp32, dev[5], batch=batch)   # on the tensor cores: not the bits of the FP32 call
    assert not torch.equal(torch.view_as_real(dev[4]), torch.view_as_real(fp32))
    got = dev[4].cpu().numpy()
    for i in {0, batch - 1}:
        want = pairwise.contract_pair(a[i].astype(np.complex128), a_w, b[i].astype(np.complex128), b_w, c_w)
        assert np.linalg.norm(got[i] - want) <= PAIR_REL[prec, cm] * np.linalg.norm(want)


@pytest.mark.parametrize("misaligned", [False, True])
@pytest.mark.parametrize("layout", ["kfast", "random"])
@pytest.mark.parametrize("shape,batch", [((18, 7, 0), 1), ((17, 7, 1), 1), ((16, 7, 2), 1), ((14, 3, 2), 70), ((15, 10, 1), 3),
                                         ((4, 9, 0), 4100)])
@pytest.mark.parametrize("prec,cm", sorted(PAIR_REL))
def test_tensor_core_padded_columns(env, prec, cm, shape, batch, layout, misaligned):
    """Fewer columns than the narrowest tile has (8, or 16 with 3M): the images'
    other columns are zero and no result of theirs is stored.  Against 64 bits,
    and on the tensor cores: not the bits of the FP32 call."""
    tn, torch = env
    nm, nk, nn = shape
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    rng = np.random.default_rng(sum(shape))
    w = list(range(nm + nk + nn))
    m, k, n = w[:nm], w[nm:nm + nk], w[nm + nk:]
    a_w, b_w, c_w = (k + m, k + n, m + n) if layout == "kfast" else \
        tuple([int(x) for x in rng.permutation(v)] for v in (m + k, k + n, m + n))
    pad = 1 if misaligned else 0

    def draw(r):
        t = torch.randn((batch << r) + pad, generator=g, dtype=torch.complex64, device="cuda")
        return t[pad:].view(batch, 1 << r)

    def ordered(x, have, want):
        at = torch.zeros(1, dtype=torch.int64, device="cuda")
        for q in want:
            at = torch.cat([at, at + (1 << have.index(q))])
        return x[:, at]

    a, b = draw(nm + nk), draw(nk + nn)
    buf = torch.full(((batch << (nm + nn)) + 2,), 7.0, dtype=torch.complex64, device="cuda")
    c = buf[pad:pad + (batch << (nm + nn))].view(batch, -1)
    tn.contract_pair(a, a_w, b, b_w, c, c_w, batch=batch, precision=prec, complex_mult=cm)
    tn.device_sync()
    x = ordered(a, a_w, k + m).view(batch, 1 << nm, 1 << nk).to(torch.complex128)
    y = ordered(b, b_w, k + n).view(batch, 1 << nn, 1 << nk).to(torch.complex128)
    want = ordered(torch.bmm(y, x.transpose(1, 2)).reshape(batch, -1), m + n, c_w)
    assert float((c.to(torch.complex128) - want).norm() / want.norm()) <= PAIR_REL[prec, cm]
    assert torch.all(buf[:pad] == 7.0) and torch.all(buf[pad + (batch << (nm + nn)):] == 7.0)
    fp32 = torch.empty_like(c)
    tn.contract_pair(a, a_w, b, b_w, fp32, c_w, batch=batch)
    assert not torch.equal(torch.view_as_real(c), torch.view_as_real(fp32))


@pytest.mark.parametrize("prec,slices,chunk", [("fp32", 0, 0), ("fp32", 5, 2), ("tf32", 4, 2), ("bf16x3", 4, 0),
                                               ("fp16x3", 4, 1)])
def test_chunks_side_by_side(env, prec, slices, chunk):
    """Chunks of one call run side by side, 16 at most, filled up to a power of
    two: any number of batches, whole or in ragged slice ranges, gives the bits of
    a plan with room for one lane that gets one chunk a call, and the state
    vector's amplitudes; with the CUDA-core steps that these sizes have, then
    with tensor-core kernels wherever they can run."""
    import rqcgen
    from oracle import statevector as sv
    tn, torch = env
    circ = rqcgen.sycamore_style(4, 4, 9, 7, 0)
    om = 0b1111110000000000
    psi = sv.simulate(circ)
    net = tn.Network(circ)
    make = lambda arena=0: tn.Plan(net, open_mask=om, max_log2_intermediate=30, min_log2_slices=slices, trials=8,
                                   log2_batch_slices=chunk, precision=prec, max_arena_bytes=arena)
    plan = make()
    single = make(plan.info()["arena_bytes"])
    assert single.step_shapes() == plan.step_shapes()
    n, per = 1 << plan.info()["log2_slices"], 1 << plan.info()["log2_batch_slices"]
    rng = np.random.default_rng(3)
    for tensor_cores in ([False, True] if prec != "fp32" else [False]):
        if tensor_cores:
            kid = {v: k for k, v in tn.Plan.KERNELS.items()}["tc_" + prec]
            forced = [(kid, -1, 0, 0, 1) if shape[0] >= 4 else t
                      for t, shape in zip(plan.get_tuning(), plan.step_shapes())]
            for p in (plan, single):
                p.set_tuning(forced)
            assert sum(t[0] == kid for t in plan.get_tuning()) >= 3
        for count in (1, 3, 2, 17, 16, 5):
            bits = [int(b) for b in rng.integers(0, 1 << 10, size=count)]
            out = torch.zeros(count << 6, dtype=torch.complex128, device="cuda")
            alone = torch.zeros_like(out)
            cuts = sorted({0, n // 3, n})
            for lo, hi in zip(cuts, cuts[1:]):
                plan.contract_slices(lo, hi - lo, bits, out)
                for i, b in enumerate(bits):
                    at = lo
                    while at < hi:
                        end = min(hi, (at // per + 1) * per)
                        single.contract_slices(at, end - at, [b], alone[i << 6:(i + 1) << 6])
                        at = end
            plan.sync()
            single.sync()
            want = np.concatenate([sv.batch_amplitudes(psi, circ.n_qubits, b, om) for b in bits])
            got = out.cpu().numpy()
            tol = {"fp32": 1e-5, "tf32": 2e-2 if tensor_cores else 1e-5}.get(prec, 1e-4)
            assert np.linalg.norm(got - want) < tol * np.linalg.norm(want)
            assert torch.equal(torch.view_as_real(out), torch.view_as_real(alone)), (count, tensor_cores)


@pytest.fixture(scope="module")
def wide_plans(env):
    """35 qubits, 14 cycles, 8 chunks of one slice: a plan of several lanes whose
    chunks hold tensor-core steps (from 2^25 multiply-adds), some of them with a
    B that depends on no slice; and the same circuit's FP32 amplitudes."""
    import rqcgen
    tn, torch = env
    circ = rqcgen.sycamore_style(5, 7, 14, 44, 0)
    net = tn.Network(circ)
    make = lambda prec, cm=4, arena=0: tn.Plan(net, open_mask=255 << 27, max_log2_intermediate=26, trials=8,
                                               precision=prec, complex_mult=cm, max_arena_bytes=arena,
                                               forced_slices=[(34, 22), (34, 21), (34, 20)])
    bits = [int(b) for b in np.random.default_rng(9).integers(0, 1 << 27, size=3)]
    ref = torch.zeros(3 << 8, dtype=torch.complex128, device="cuda")
    make("fp32").contract_slices(0, 8, bits, ref)
    torch.cuda.synchronize()
    return make, bits, ref


@pytest.mark.parametrize("prec,cm", [("tf32", 4), ("bf16x3", 4), ("fp16x3", 4), ("bf16x3", 3), ("fp16x3", 3)])
def test_lanes_with_tensor_core_steps(env, wide_plans, prec, cm):
    """Tensor-core steps run once per lane, each lane with its own operands, FP16
    maxima and B' images: calls of several chunks, of one batch or of several, give
    the bits of a plan that gets them one chunk a call, and the FP32
    amplitudes; images of a B that no slice changes are built with its prologue,
    not with every chunk, in either."""
    tn, torch = env
    make, bits, ref = wide_plans
    many = make(prec, cm)
    one = make(prec, cm, arena=many.info()["arena_bytes"])   # room for one lane
    assert one.step_shapes() == many.step_shapes()
    want = torch.zeros_like(ref)
    for i, b in enumerate(bits):
        for c in range(8):
            one.contract_slices(c, 1, [b], want[i << 8:(i + 1) << 8])
    kernels = [k for _, k in one.step_times(1)]
    flags = [one.step_layout(i)["dep_flags"] for i in range(len(kernels))]
    tc = sum(k.startswith("tc") and bool(f & 1) for k, f in zip(kernels, flags))
    assert tc >= 2
    rel = {"tf32": 2e-2, "bf16x3": 1e-4, "fp16x3": 1e-4}[prec]
    assert float((want - ref).norm() / ref.norm()) < rel
    for cuts, batches in (([0, 8], [[0, 1, 2]]), ([0, 1, 8], [[0], [1, 2]]), ([0, 3, 4, 8], [[2], [1], [0]]),
                          ([0, 2, 4, 6, 8], [[0, 1], [2]])):
        out = torch.zeros_like(ref)
        for group in batches:
            part = torch.zeros(len(group) << 8, dtype=torch.complex128, device="cuda")
            for lo, hi in zip(cuts, cuts[1:]):
                many.contract_slices(lo, hi - lo, [bits[i] for i in group], part)
            for j, i in enumerate(group):
                out[i << 8:(i + 1) << 8] = part[j << 8:(j + 1) << 8]
        many.sync()
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(want)), (cuts, batches)
    assert many.chunk_launches() == one.chunk_launches()


def test_lanes_weigh_a_heavy_prologue(env):
    """30 closed qubits beside 6 open ones of which alone wires are sliced: the
    prologue of a batch (2^24.8 multiply-adds) outweighs its 16 chunks (2^11).
    More lanes save launches but repeat the prologue, so a call of all chunks takes
    no longer than the same chunks in two calls of half the lanes (329 us
    against 231 with as many lanes as there is room for), and gives the same bits."""
    import rqcgen
    tn, torch = env
    big, small = rqcgen.sycamore_style(5, 6, 14, 17, 0), rqcgen.sycamore_style(2, 3, 8, 18, 0)
    n = big.n_qubits
    circ = rqcgen.Circuit(n + 6, np.concatenate([big.gate_qubits, np.where(small.gate_qubits >= 0,
                                                                           small.gate_qubits + n, -1)]),
                          list(big.gate_matrices) + list(small.gate_matrices),
                          np.concatenate([big.gate_layer, small.gate_layer]))
    net = tn.Network(circ)
    per = net.gates_per_qubit()
    make = lambda **kw: tn.Plan(net, open_mask=63 << n, max_log2_intermediate=26, trials=8,
                                forced_slices=[(n + j, per[n + j] - 2) for j in range(4)], **kw)
    plan = make()
    work = {0: 0.0, 1: 0.0, 2: 0.0}
    for i, shape in enumerate(plan.step_shapes()):
        f = plan.step_layout(i)["dep_flags"]
        work[1 if f & 1 else f] += 2.0 ** sum(shape)
    assert work[2] > 100 * work[1]
    single = make(max_arena_bytes=plan.info()["arena_bytes"])   # room for one lane
    rng = np.random.default_rng(4)
    draw = lambda: [int(b) for b in rng.integers(0, 1 << n, size=1)]

    def amplitudes(p, bits, parts):
        out = torch.zeros(64, dtype=torch.complex128, device="cuda")
        for lo in range(0, 16, 16 // parts):
            p.contract_slices(lo, 16 // parts, bits, out)
        return torch.view_as_real(out)

    for _ in range(3):
        bits = draw()
        want = amplitudes(single, bits, 16)
        assert float(want.abs().max()) > 0.0
        for parts in (1, 2, 4):
            assert torch.equal(amplitudes(plan, bits, parts), want)

    def us(parts):
        best = float("inf")
        for _ in range(5):
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(20):
                amplitudes(plan, draw(), parts)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1) * 50)
        return best

    whole, halves = us(1), us(2)
    assert whole < 1.15 * halves, (whole, halves)


def test_later_calls_do_not_wait(env):
    """Only the first call of a plan synchronises: calls with other numbers of
    chunks return while earlier work of another stream still runs (half a second of
    sleep on the legacy stream, which a blocking copy would wait for)."""
    import time
    import rqcgen
    tn, torch = env
    circ = rqcgen.sycamore_style(4, 4, 9, 7, 0)
    plan = tn.Plan(tn.Network(circ), open_mask=0b1111110000000000, max_log2_intermediate=30, trials=8)
    out = torch.zeros(16 << 6, dtype=torch.complex128, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    plan.contract_slices(0, 1, [1], out, stream=side)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda._sleep(1000)   # its kernel is loaded
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.default_stream()):
        e0.record()
        torch.cuda._sleep(1_000_000_000)
        e1.record()
    t0 = time.perf_counter()
    for count in (2, 5, 3, 16, 9, 16, 1):
        plan.contract_slices(0, 1, [4 * i + count for i in range(count)], out, stream=side)
    host = time.perf_counter() - t0
    side.synchronize()
    torch.cuda.synchronize()
    assert e0.elapsed_time(e1) > 400.0 and host < 0.2


def test_selection_estimates_calls_of_many_chunks(env):
    """A candidate's estimate for all slices is what the chosen plan then takes: a
    plan of small chunks runs several side by side, and is timed so."""
    import rqcgen
    tn, torch = env
    circ = rqcgen.sycamore_style(4, 4, 9, 7, 0)
    om = 0b1111110000000000
    plan, est = tn.select_plan(tn.Network(circ), 3, 5, open_mask=om, max_log2_intermediate=30, min_log2_slices=5,
                               trials=8, log2_batch_slices=1)
    info = plan.info()
    assert info["log2_slices"] - info["log2_batch_slices"] >= 4
    out = torch.zeros(1 << 6, dtype=torch.complex128, device="cuda")
    best = float("inf")
    for _ in range(20):
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        plan.contract_slices(0, 1 << info["log2_slices"], [5], out)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e-3)
    assert best / 2.5 < min(est) < 2.5 * best, (est, best)
