"""FP32 FFT shapes read at run time, against the oracle: regular rows of
lengths without a compile-time kernel (one to three passes of register DFT
sizes, odd ones among them), reduced-grid rows of compile-time lengths that a
half-spacing shift sends to the run-time kernel, and rows transformed by
Bluestein's method with convolution lengths on either side of and equal to
the compile-time ones.

Tolerance: the split transform's (1e-6, relative L2); the FFT's rounding is
an order below it."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1711_11296_gb300 import workloads as W
from sht_testutil import built_lib, rel_l2, to_cuda

pytestmark = pytest.mark.gpu

TOL = 1e-6
N, J = 12, 27


@pytest.fixture(scope="module")
def sht():
    built_lib()
    from paper_1711_11296_gb300 import sht as S
    return S


@pytest.mark.parametrize("L", [15, 25, 27, 32, 45, 81, 96, 125, 160, 192, 225, 243, 250, 288,
                               375, 384, 405, 480, 500, 625, 720, 768, 810, 900, 960, 1000,
                               1125, 1350, 1536, 1600, 2000, 2048, 4096])
@pytest.mark.parametrize("F", [1, 5])
def test_regular_rows(sht, L, F):
    I = 2 * L
    p = sht.Plan(N, J, I, F, "bf16x3")
    x = W.random_grid(F, J, I, seed=2500 + L).astype(np.float32).astype(np.float64)
    a = W.random_spectrum(N, F, "flat", seed=2600 + L).astype(np.complex64)
    assert rel_l2(p.forward(to_cuda(x, torch.float32)).cpu().numpy(), O.analysis(x, N)) <= TOL
    got = p.inverse(torch.from_numpy(a).cuda()).cpu().numpy()
    assert rel_l2(got, O.synthesis(a.astype(np.complex128), N, J, I)) <= TOL
    p.status()


def _reduced(sht, pts, shift, F):
    p = sht.Plan(N, J, max(pts), F, "bf16x3", grid="reduced", lat_points=pts, half_shift=shift)
    x = np.random.default_rng(sum(pts)).standard_normal((F, sum(pts)))
    x = x.astype(np.float32).astype(np.float64)
    a = W.random_spectrum(N, F, "flat", seed=2700 + pts[0]).astype(np.complex64)
    got = p.forward(to_cuda(x, torch.float32)).cpu().numpy()
    spacings = None if shift is None else [0.5 * v for v in shift]
    ref = O.analysis_reduced(x, N, J, pts, shifts=spacings)
    assert rel_l2(got, ref) <= TOL
    got = p.inverse(torch.from_numpy(a).cuda()).cpu().numpy()
    ref = O.synthesis_reduced(a.astype(np.complex128), N, J, pts, shifts=spacings)
    assert rel_l2(got, ref) <= TOL
    p.status()


@pytest.mark.parametrize("L", [64, 128, 256, 320, 512, 640, 1024, 1280])
def test_shifted_rows_of_compile_time_lengths(sht, L):
    _reduced(sht, [2 * L] * J, [1] * J, 3)


@pytest.mark.parametrize("L2", [64, 256, 320, 512, 640, 1024, 1280, 1350])
@pytest.mark.parametrize("F", [1, 6])
def test_bluestein_convolution_lengths(sht, L2, F):
    # the longest row whose convolution takes L2 points and has a prime factor
    # above 5, and shorter rows beside it
    L = max(k for k in range(14, L2 // 2 + 1) if 2 * k - 1 <= L2 and _big_prime(k))
    pts = [2 * L - 2 * (j % 3) if j != J // 2 else 2 * L for j in range((J + 1) // 2)]
    pts = pts + pts[-2::-1]
    _reduced(sht, pts, None, F)


def _big_prime(n):
    for q in (2, 3, 5):
        while n % q == 0:
            n //= q
    return n > 1


def test_reduced_grid_captured_in_a_graph(sht):
    # the side-by-side launches of a reduced grid's FFTs (classes, run-time
    # shapes, Bluestein rows) keep their order when captured and replayed
    F = 3
    pts = [2 * L for L in (15, 31, 64, 64, 90, 96, 101, 128, 128, 128, 133, 256, 256, 320)]
    pts = pts + pts[-2::-1]
    p = sht.Plan(N, J, max(pts), F, "bf16x3", grid="reduced", lat_points=pts)
    a = torch.from_numpy(W.random_spectrum(N, F, "flat", seed=2800).astype(np.complex64)).cuda()
    grid, spec = p.empty_grid(), p.empty_spec()
    p.inverse(a, out=grid)
    p.forward(grid, out=spec)
    ref_grid, ref_spec = grid.clone(), spec.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.inverse(a, out=grid)
        p.forward(grid, out=spec)
    for _ in range(20):
        grid.zero_()
        spec.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(grid, ref_grid) and torch.equal(spec, ref_spec)
    p.status()


@pytest.mark.parametrize("I", [40, 128, 1280])
@pytest.mark.parametrize("k,offset", [(1, 0), (1, 2), (1, 4), (2, 0)])
def test_restriction_reads_any_alignment(sht, I, k, offset):
    # the nested rows' 16-byte loads (k = 1, aligned) and the copies of other
    # strides and alignments give the transform of the injected grid
    F, Nc, Jc = 3, 7, 15
    p = sht.Plan(Nc, Jc, I, F, "bf16x3")
    shape = (F, 2 ** k * (Jc + 1) - 1, 2 ** k * I)
    n = int(np.prod(shape))
    buf = torch.randn(n + offset, device="cuda", generator=torch.Generator("cuda").manual_seed(I))
    fine = buf[offset:].view(shape)
    ref = p.forward(p.inject_nested(fine, k))
    assert torch.equal(p.restrict_nested(fine, k), ref)


# Grids of few values of L > 320 (the cases above) take the kernel of the radices
# up to 10; these have enough of them for the kernel of all register sizes.
@pytest.mark.parametrize("L,F", [(96, 200), (100, 201), (150, 200), (240, 100), (288, 100),
                                 (300, 101), (375, 64), (625, 64), (720, 40), (800, 40),
                                 (900, 40), (1125, 41), (1536, 40), (1600, 40), (2000, 24),
                                 (2048, 25)])
def test_regular_rows_of_many_fields(sht, L, F):
    J, I = 201, 2 * L
    p = sht.Plan(N, J, I, F, "bf16x3")
    x = W.random_grid(F, J, I, seed=2500 + L).astype(np.float32).astype(np.float64)
    a = W.random_spectrum(N, F, "flat", seed=2600 + L).astype(np.complex64)
    assert rel_l2(p.forward(to_cuda(x, torch.float32)).cpu().numpy(), O.analysis(x, N)) <= TOL
    got = p.inverse(torch.from_numpy(a).cuda()).cpu().numpy()
    assert rel_l2(got, O.synthesis(a.astype(np.complex128), N, J, I)) <= TOL
    p.status()


def test_both_runtime_kernels_agree(sht):
    # the same fields in a plan of 3 fields (radices up to 10) and of 64 (30 24), forward,
    # inverse, onto a grid, strided; both within the FFT's rounding
    J, I, F = 101, 1440, 64
    gen = torch.Generator("cuda").manual_seed(2800)
    x = torch.randn(F, J, I, device="cuda", generator=gen)
    fine = torch.randn(F, 2 * J + 1, 2 * I, device="cuda", generator=gen)
    a = torch.from_numpy(W.random_spectrum(N, F, "flat", seed=2801).astype(np.complex64)).cuda()
    p, q = sht.Plan(N, J, I, F, "bf16x3"), sht.Plan(N, J, I, 3, "bf16x3")
    pick = slice(5, 8)
    b = a[:, pick].contiguous()

    def close(got, ref):
        assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) <= 5e-7

    close(q.forward(x[pick].contiguous()), p.forward(x)[:, pick])
    close(q.inverse(b), p.inverse(a)[pick])
    close(q.prolong_spectral(b, N, out=x[pick].clone(), add=True),
          p.prolong_spectral(a, N, out=x.clone(), add=True)[pick])
    close(q.restrict_nested(fine[pick].contiguous(), 1), p.restrict_nested(fine, 1)[:, pick])


@pytest.mark.parametrize("L", [384, 480, 768, 960])
@pytest.mark.parametrize("prec,tol", [("bf16x3", TOL), ("fp64", 1e-12)])
def test_shifted_and_plain_rows_of_later_compile_time_lengths(sht, L, prec, tol):
    # shifted rows go to the run-time kernel, plain ones beside them to the
    # compile-time one (FP64: the run-time one)
    pts, shift = [2 * L] * J, [j % 2 for j in range((J + 1) // 2)]
    shift = shift + shift[-2::-1]
    p = sht.Plan(N, J, 2 * L, 3, prec, grid="reduced", lat_points=pts, half_shift=shift)
    x = np.random.default_rng(L).standard_normal((3, sum(pts))).astype(np.float32)
    x = x.astype(np.float64)
    a = W.random_spectrum(N, 3, "flat", seed=2900 + L).astype(np.complex64).astype(np.complex128)
    spacings = [0.5 * v for v in shift]
    got = p.forward(to_cuda(x, p.real_dtype)).cpu().numpy()
    assert rel_l2(got, O.analysis_reduced(x, N, J, pts, shifts=spacings)) <= tol
    got = p.inverse(to_cuda(a, p.complex_dtype)).cpu().numpy()
    assert rel_l2(got, O.synthesis_reduced(a, N, J, pts, shifts=spacings)) <= tol
    p.status()
