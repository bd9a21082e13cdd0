"""Failure detection on the GPU without faulting it.  A fault-injection hook
makes the first CTA of a split plan's forward GEMM never arm its first
pipeline stage: every bounded wait downstream runs out (about 2 s), the CTA
drains its copies, frees its tensor memory and records SHT_ERR_TIMEOUT, which
sht_plan_status reports; the context stays usable.  A second hook fails a
plan's device allocation as if the GPU were out of memory."""
import os

import numpy as np
import pytest
import torch

import oracle as O
from paper_1711_11296_gb300 import workloads as W
from sht_testutil import built_lib, rel_l2, to_cuda

pytestmark = pytest.mark.gpu

SHT_ERR_ALLOC, SHT_ERR_TIMEOUT = -2, -5


@pytest.fixture(scope="module")
def sht():
    built_lib()
    from paper_1711_11296_gb300 import sht as S
    return S


def _with_env(name, value, fn):
    os.environ[name] = value
    try:
        return fn()
    finally:
        del os.environ[name]


def test_bounded_wait_timeout_is_reported_and_context_survives(sht):
    N, J, I, F = 7, 15, 16, 1
    p = _with_env("SHT_INJECT_STALL", "1", lambda: sht.Plan(N, J, I, F, "bf16x3"))
    x = W.random_grid(F, J, I, seed=1701).astype(np.float32).astype(np.float64)
    p.forward(to_cuda(x, torch.float32))
    with pytest.raises(sht.SHTError) as ei:
        p.status()
    assert ei.value.code == SHT_ERR_TIMEOUT
    p.status()                      # reading the status cleared it
    p.close()
    # the device is healthy: a fresh plan computes the right answer
    q = sht.Plan(N, J, I, F, "bf16x3")
    got = q.forward(to_cuda(x, torch.float32)).cpu().numpy()
    assert rel_l2(got, O.analysis(x, N)) <= 1e-6
    q.status()


def test_injected_allocation_failure(sht):
    for k in (1, 3):
        with pytest.raises(sht.SHTError) as ei:
            _with_env("SHT_INJECT_ALLOC_FAIL", str(k), lambda: sht.Plan(31, 65, 128, 2, "fp64"))
        assert ei.value.code == SHT_ERR_ALLOC
    p = sht.Plan(31, 65, 128, 2, "fp64")    # nothing leaked into the next plan
    x = W.random_grid(2, 65, 128, seed=1702)
    assert rel_l2(p.forward(to_cuda(x, torch.float64)).cpu().numpy(), O.analysis(x, 31)) < 1e-12


# ---- the FP64 plans' tensor-core tables ----
from sht_testutil import assert_fp64_close  # noqa: E402

# Plans whose contractions are sliced; the last one's columns and nodes fill no tile.
SLICED = [(63, 129, 256, 64), (40, 71, 96, 321), (62, 131, 128, 65)]


def _check_all(sht, p, N, J, I, F):
    x = W.random_grid(F, J, I, seed=1703)
    a = W.random_spectrum(N, F, "flat", seed=1704)
    assert_fp64_close(p.forward(to_cuda(x, torch.float64)).cpu().numpy(), O.analysis(x, N))
    assert_fp64_close(p.inverse(to_cuda(a, torch.complex128)).cpu().numpy(),
                      O.synthesis(a, N, J, I))
    # adjoints by their definition: <A x, a> = <x, A^T a>, over the fields together
    gx, ga = to_cuda(x, torch.float64), to_cuda(a, torch.complex128)
    for lhs, rhs in (((p.forward(gx).conj() * ga).real.sum(), (gx * p.adjoint(0, ga)).sum()),
                     ((gx * p.inverse(ga)).sum(), (p.adjoint(1, gx).conj() * ga).real.sum())):
        assert abs(lhs.item() - rhs.item()) <= 1e-11 * max(abs(lhs.item()), 1.0)
    p.status()


@pytest.mark.parametrize("k", range(16, 28))
def test_plan_without_the_memory_for_tensor_tables(sht, k):
    # the tables' allocations follow the plan's own fifteen; each of them failing
    # leaves a plan on the FP64 pipe that says so
    N, J, I, F = SLICED[0]
    p = _with_env("SHT_INJECT_ALLOC_FAIL", str(k), lambda: sht.Plan(N, J, I, F, "fp64"))
    assert p.tensor_tables == {"on": False, "bytes": 0}
    if k in (16, 27):
        _check_all(sht, p, N, J, I, F)


@pytest.mark.parametrize("N,J,I,F", SLICED)
def test_tensor_tables_given_back_and_rebuilt(sht, N, J, I, F):
    p = sht.Plan(N, J, I, F, "fp64")
    had = p.tensor_tables
    assert had["on"] and had["bytes"] > 0
    x = to_cuda(W.random_grid(F, J, I, seed=1705), torch.float64)
    sliced = p.forward(x)
    p.set_tensor_tables(False)
    assert p.tensor_tables == {"on": False, "bytes": 0}
    _check_all(sht, p, N, J, I, F)
    p.set_reduced(True)
    _check_all(sht, p, N, J, I, F)
    p.set_reduced(False)
    p.set_tensor_tables(True)
    assert p.tensor_tables == had
    assert torch.equal(p.forward(x), sliced)
    _check_all(sht, p, N, J, I, F)


def test_tensor_tables_where_there_are_none(sht):
    for p in (sht.Plan(31, 65, 128, 2, "fp64"), sht.Plan(63, 129, 256, 64, "bf16x3")):
        assert p.tensor_tables == {"on": False, "bytes": 0}
        with pytest.raises(sht.SHTError):
            p.set_tensor_tables(True)


def test_tensor_tables_leave_most_of_the_memory(sht):
    # with less than eight times their size free, a plan does without, unless told
    N, J, I, F = SLICED[0]
    need = sht.Plan(N, J, I, F, "fp64").tensor_tables["bytes"]
    make = lambda: sht.Plan(N, J, I, F, "fp64")
    assert _with_env("SHT_INJECT_FREE_BYTES", str(8 * need), make).tensor_tables["on"]
    p = _with_env("SHT_INJECT_FREE_BYTES", str(8 * need - 1), make)
    assert not p.tensor_tables["on"]
    p.set_tensor_tables(True)
    assert p.tensor_tables == {"on": True, "bytes": need}
