"""The allocation-free pairwise contraction (tn_contract_pair_noalloc).

Callers that cannot allocate device memory (their memory belongs to another
allocator, or their host forbids allocation once it runs) use this entry
point; it must give what tn_contract_pair gives.  Each case runs it twice in a
row on different inputs, because every call reuses the same static scratch
array and must not be affected by what the previous call left there.  Each
result is compared with the FP64 oracle contraction of the same host operands
and with tn_contract_pair.  Collected last so that a run stopping at the first
failure has run every other test.
"""
import ctypes
import math

import numpy as np
import pytest

from oracle import pairwise

pytestmark = pytest.mark.gpu

# element-wise bound on |C - C_ref| as a multiple of sqrt(K) rms(A) rms(B)
PAIR_TOL = {("fp32", 4): 1e-5, ("tf32", 4): 3e-3, ("bf16x3", 4): 5e-5, ("fp16x3", 4): 2e-5,
            ("tf32", 3): 6e-3, ("bf16x3", 3): 1e-4, ("fp16x3", 3): 4e-5}


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2111_01066_gb300 import tn
    torch.cuda.set_device(0)
    return tn, torch


def _operands(torch, rng, batch, a_w, b_w):
    a = ((rng.normal(size=(batch, 2 ** len(a_w))) + 1j * rng.normal(size=(batch, 2 ** len(a_w)))) / 2)
    b = ((rng.normal(size=(batch, 2 ** len(b_w))) + 1j * rng.normal(size=(batch, 2 ** len(b_w)))) / 2)
    a = a.astype(np.complex64)
    b = b.astype(np.complex64)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    return a, b, dev(a), dev(b)


def _noalloc(tn, ta, a_w, tb, b_w, tc, c_w, batch, prec, cm, torch):
    """The entry point called through the C ABI (ctypes), as a C caller would."""
    lib = tn.load()
    return lib.tn_contract_pair_noalloc(
        ctypes.c_void_p(ta.data_ptr()), tn._i32(a_w), len(a_w), ctypes.c_void_p(tb.data_ptr()), tn._i32(b_w),
        len(b_w), ctypes.c_void_p(tc.data_ptr()), tn._i32(c_w), len(c_w), batch, tn.PREC[prec], cm,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("prec,cm", [("fp32", 4), ("tf32", 4), ("bf16x3", 4), ("fp16x3", 4),
                                     ("bf16x3", 3), ("fp16x3", 3)])
@pytest.mark.parametrize("shape", [(9, 9, 7), (12, 6, 7), (3, 2, 5), (8, 12, 4)])
def test_noalloc_matches_oracle_and_contract_pair_on_two_calls(env, prec, cm, shape):
    tn, torch = env
    nm, nk, nn = shape
    batch = 2
    rng = np.random.default_rng(sum(shape) + len(prec) + cm)
    wires = list(range(10, 10 + nm + nk + nn))
    m_w, k_w, n_w = wires[:nm], wires[nm:nm + nk], wires[nm + nk:]
    a_w = list(rng.permutation(m_w + k_w))
    b_w = list(rng.permutation(k_w + n_w))
    c_w = list(rng.permutation(m_w + n_w))
    tol = PAIR_TOL[(prec, cm)]
    for call in range(2):
        a, b, ta, tb = _operands(torch, rng, batch, a_w, b_w)
        ref = torch.empty((batch, 2 ** len(c_w)), dtype=torch.complex64, device="cuda")
        tn.contract_pair(ta, a_w, tb, b_w, ref, c_w, batch=batch, precision=prec, complex_mult=cm)
        got = torch.full_like(ref, float("nan"))
        st = _noalloc(tn, ta, a_w, tb, b_w, got, c_w, batch, prec, cm, torch)
        assert st == tn.TN_OK, tn.load().tn_last_error()
        tn.device_sync()     # no bounded wait ran out in either call
        if prec != "fp32" and nm + nk + nn >= 24:   # on the tensor cores: other bits than the FP32 call's
            plain = torch.empty_like(ref)
            tn.contract_pair(ta, a_w, tb, b_w, plain, c_w, batch=batch)
            assert not torch.equal(torch.view_as_real(got), torch.view_as_real(plain))
        g, r = got.cpu().numpy(), ref.cpu().numpy()
        for i in range(batch):
            want = pairwise.contract_pair(a[i].astype(np.complex128), a_w, b[i].astype(np.complex128), b_w, c_w)
            scale = math.sqrt(2 ** nk) * np.sqrt(np.mean(np.abs(a[i]) ** 2) * np.mean(np.abs(b[i]) ** 2))
            assert np.all(np.isfinite(g[i]))
            assert np.max(np.abs(g[i] - want)) <= tol * scale * 8, f"call {call}: vs oracle"
            assert np.max(np.abs(g[i] - r[i])) <= tol * scale * 8, f"call {call}: vs tn_contract_pair"


def test_noalloc_rejects_scratch_beyond_the_static_array(env):
    tn, torch = env
    # B with k = 2^10, n = 2^12 complex entries: about 64 MiB of B' images > 32 MiB
    a_w = list(range(0, 4)) + list(range(100, 110))
    b_w = list(range(100, 110)) + list(range(200, 212))
    c_w = list(range(0, 4)) + list(range(200, 212))
    ta = torch.zeros(2 ** len(a_w), dtype=torch.complex64, device="cuda")
    tb = torch.zeros(2 ** len(b_w), dtype=torch.complex64, device="cuda")
    tc = torch.zeros(2 ** len(c_w), dtype=torch.complex64, device="cuda")
    st = _noalloc(tn, ta, a_w, tb, b_w, tc, c_w, 1, "bf16x3", 4, torch)
    assert st == tn.TN_ERR_ARG
    assert b"static array" in tn.load().tn_last_error()


@pytest.mark.parametrize("prec,cm", [("tf32", 4), ("bf16x3", 4), ("fp16x3", 4), ("tf32", 3), ("bf16x3", 3)])
@pytest.mark.parametrize("shape,batch", [((7, 5, 5), 4096), ((4, 4, 4), 16384), ((6, 7, 6), 512), ((5, 9, 5), 200)])
def test_noalloc_takes_many_small_instances(env, prec, cm, shape, batch):
    """Instances under 2^20 multiply-adds are accepted whatever their number:
    where the B' images of all of them exceed the static array they run on the
    CUDA cores, within the rounding bound of FP32 sums in any order,
    |error| <= (2 k + 2) u sum |a| |b|, u = 2^-24 (each component is a sum of 2k
    products)."""
    tn, torch = env
    nm, nk, nn = shape
    rng = np.random.default_rng(sum(shape) + batch)
    wires = list(range(nm + nk + nn))
    m_w, k_w, n_w = wires[:nm], wires[nm:nm + nk], wires[nm + nk:]
    a_w, b_w, c_w = k_w + m_w, list(rng.permutation(k_w + n_w)), list(rng.permutation(m_w + n_w))
    a, b, ta, tb = _operands(torch, rng, batch, a_w, b_w)
    tc = torch.full((batch, 2 ** len(c_w)), float("nan"), dtype=torch.complex64, device="cuda")
    st = _noalloc(tn, ta, a_w, tb, b_w, tc, c_w, batch, prec, cm, torch)
    assert st == tn.TN_OK, tn.load().tn_last_error()
    tn.device_sync()
    got = tc.cpu().numpy()
    assert np.all(np.isfinite(got.view(np.float32)))
    for i in {0, 1, batch // 2, batch - 1}:
        want = pairwise.contract_pair(a[i].astype(np.complex128), a_w, b[i].astype(np.complex128), b_w, c_w)
        mag = pairwise.contract_pair(np.abs(a[i]).astype(np.complex128), a_w, np.abs(b[i]).astype(np.complex128), b_w,
                                     c_w).real
        bound = (2 * 2 ** nk + 2) * 2.0 ** -24 * mag
        assert np.all(np.abs(got[i].real - want.real) <= bound)
        assert np.all(np.abs(got[i].imag - want.imag) <= bound)


@pytest.mark.parametrize("shape,batch", [((10, 14, 3), 12), ((12, 14, 4), 3), ((12, 15, 3), 3), ((11, 14, 4), 5),
                                         ((11, 16, 3), 3)])
def test_noalloc_divides_k_beside_the_images(env, shape, batch):
    """Partial sums and B' images that fill the static array between them: k is
    still divided as far as both fit, so the tensor cores' 32-bit accumulation
    runs over at most 2^13 of the k (norm-wise 4e-5 at BF16x3; it grows with the
    length of the chain, and one pass over these k is 1.1e-4 to 4.6e-4 off)."""
    tn, torch = env
    nm, nk, nn = shape
    wires = list(range(nm + nk + nn))
    m_w, k_w, n_w = wires[:nm], wires[nm:nm + nk], wires[nm + nk:]
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    draw = lambda r: torch.randn((batch, 1 << r), generator=g, dtype=torch.complex64, device="cuda")
    ta, tb = draw(nm + nk), draw(nk + nn)
    tc = torch.full((batch, 1 << (nm + nn)), float("nan"), dtype=torch.complex64, device="cuda")
    st = _noalloc(tn, ta, k_w + m_w, tb, k_w + n_w, tc, m_w + n_w, batch, "bf16x3", 4, torch)
    assert st == tn.TN_OK, tn.load().tn_last_error()
    tn.device_sync()
    want = torch.bmm(tb.view(batch, 1 << nn, 1 << nk).to(torch.complex128),
                     ta.view(batch, 1 << nm, 1 << nk).to(torch.complex128).transpose(1, 2)).reshape(batch, -1)
    assert float((tc.to(torch.complex128) - want).norm() / want.norm()) <= 4e-5
