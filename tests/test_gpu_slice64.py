"""FP64 contractions on the tensor cores (sliced operands) against the CPU
oracle, at the edges of their tiles: one more and one fewer row, node or
column than a multiple of 16, 64 or 128, both orientations of the product,
column ranges of 1e-300 .. 1e300, and non-finite columns; and the small
contractions with a thread per output.

Tolerance: a slice carries its operand to 2^-55 of the row or column
maximum, so a sum of K products is within 2 K 2^-55 of (row maximum x column
maximum) besides the final rounding; with K <= 322 and |P~| <= 26 that is
below 5e-13 of the largest column, and the FP64 tolerance of the other tests
(1e-12) covers it."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1711_11296_gb300 import workloads as W
from sht_testutil import assert_fp64_close, built_lib, to_cuda

pytestmark = pytest.mark.gpu

# (N, J, I, F): columns are 2 F, parity rows at most N / 2 + 1, nodes J / 2.
# All above the size up to which the FP64 pipe keeps a transform.
CASES = [
    (63, 129, 256, 60),     # 120 columns, 64 nodes + the Equator
    (63, 127, 256, 64),     # 128 columns, 63 nodes
    (62, 131, 128, 65),     # 130 columns, 65 nodes
    (127, 257, 512, 8),     # 16 columns, 128 nodes, rows up to 64
    (127, 259, 512, 9),     # 18 columns, 129 nodes
    (129, 263, 288, 33),    # 66 columns
    (31, 65, 128, 450),     # 900 columns, 16 rows
    (33, 69, 72, 400),      # 17 rows
    (40, 71, 96, 321),      # inexact grid (J < 2 N + 1)
]

# Either side of the tile widths 32, 64 and 80: by columns, then by rows.
WIDTHS = [(159, 321, 640, 16), (159, 321, 640, 17), (159, 321, 640, 32), (159, 321, 640, 33),
          (159, 321, 640, 40), (159, 321, 640, 41),
          (95, 193, 192, 64), (127, 257, 288, 64), (159, 321, 640, 64), (161, 325, 648, 64)]

# Transforms with a thread per output, on either side of its row chunks.
SMALL = [(31, 65, 128, 1), (42, 87, 180, 4), (63, 129, 256, 5), (159, 321, 640, 1),
         (12, 27, 30, 300), (0, 1, 2, 3)]


@pytest.fixture(scope="module")
def sht():
    built_lib()
    from paper_1711_11296_gb300 import sht as S
    return S


@pytest.mark.parametrize("N,J,I,F", CASES + WIDTHS + SMALL)
def test_matches_oracle(sht, N, J, I, F):
    p = sht.Plan(N, J, I, F, "fp64")
    x = W.random_grid(F, J, I, seed=2100 + N)
    a = W.random_spectrum(N, F, "flat", seed=2200 + N)
    assert_fp64_close(p.forward(to_cuda(x, torch.float64)).cpu().numpy(), O.analysis(x, N))
    assert_fp64_close(p.inverse(to_cuda(a, torch.complex128)).cpu().numpy(),
                      O.synthesis(a, N, J, I))
    p.status()


def test_columns_are_scaled_alone(sht):
    # columns at the ends of the FP64 range, and an all-zero one: each
    # field's result is that of the field alone, scaled (powers of two)
    N, J, I, F = 63, 129, 256, 60
    p = sht.Plan(N, J, I, F, "fp64")
    a = W.random_spectrum(N, 1, "flat", seed=2300)
    scale = np.tile([1.0, 2.0 ** -990, 2.0 ** 990, 0.0, 2.0 ** 40, 2.0 ** -40], F // 6)
    t = p.inverse(to_cuda(a * scale, torch.complex128)).cpu().numpy()
    for f, s in enumerate(scale):
        ref = t[0] * s
        assert np.abs(t[f] - ref).max() <= 1e-14 * np.abs(ref).max()
    s0 = p.forward(to_cuda(t, torch.float64)).cpu().numpy()
    for f, s in enumerate(scale):
        ref = s0[:, 0] * s
        assert np.abs(s0[:, f] - ref).max() <= 1e-14 * np.abs(ref).max()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_fields_stay_apart(sht, bad):
    N, J, I, F = 63, 129, 256, 60
    p = sht.Plan(N, J, I, F, "fp64")
    x = W.random_grid(F, J, I, seed=2400)
    y = x.copy()
    y[3, 17, 40] = bad
    good = p.forward(to_cuda(x, torch.float64)).cpu().numpy()
    got = p.forward(to_cuda(y, torch.float64)).cpu().numpy()
    keep = [f for f in range(F) if f != 3]
    np.testing.assert_array_equal(got[:, keep], good[:, keep])
    assert not np.isfinite(got[:, 3]).any()
    a = W.random_spectrum(N, F, "flat", seed=2401)
    b = a.copy()
    b[100, 2] = bad
    good = p.inverse(to_cuda(a, torch.complex128)).cpu().numpy()
    got = p.inverse(to_cuda(b, torch.complex128)).cpu().numpy()
    keep = [f for f in range(F) if f != 2]
    np.testing.assert_array_equal(got[keep], good[keep])
    assert not np.isfinite(got[2]).any()


# Constant fields: the column's digits are then the same at every node, as are
# those of P~_0^0, and the products' sums do not average out (N = 774 with J =
# 2 N + 3 is the worst of the truncations 303 .. 1023 for the cotangent of a
# mean; J = 2301 has more than 1024 nodes).  Tolerance: an exact sum has the
# operands' rounding, 2^-56 of the maxima for each of K <= 1151 terms of one
# sign, and the FFT's (2e-16); 1e-13 is far above both.
@pytest.mark.parametrize("N,J,I,F,c", [
    (774, 1551, 1600, 2, None), (928, 1859, 1920, 2, None), (639, 1281, 1280, 2, 0.949412),
    (639, 1281, 1280, 2, 0.98831), (100, 2301, 216, 4, None), (100, 2301, 216, 4, 0.949412),
])
def test_constant_fields(sht, N, J, I, F, c):
    p = sht.Plan(N, J, I, F, "fp64")
    c = 1.0 / (J * I) if c is None else c
    noise = np.random.default_rng(2500 + N).standard_normal((J, I)) * (1e-6 * c)
    x = np.stack([np.full((J, I), c), c + noise] + [np.full((J, I), -3.0 * c)] * (F - 2))
    got = p.adjoint(1, to_cuda(x, torch.float64)).cpu().numpy()
    p.status()
    # X_0^0 = sum over the points x P~_0^0, in extended precision
    ref = x.astype(np.longdouble).sum(axis=(1, 2)) * np.sqrt(np.longdouble(0.5))
    assert np.abs(got[0] / ref.astype(np.float64) - 1.0).max() <= 1e-13


# The segments of a long sum: fields whose digits are random, so that the whole
# range of rows and columns is summed, against the oracle.
@pytest.mark.parametrize("N,J,I,F", [
    (20, 2051, 48, 40),     # 1026 nodes: three segments of a forward sum
    (20, 8191, 48, 12),     # 4096 nodes, the most that are sliced
    (340, 700 + 1, 720, 3), # two segments forward, one inverse
])
def test_long_sums(sht, N, J, I, F):
    p = sht.Plan(N, J, I, F, "fp64")
    x = W.random_grid(F, J, I, seed=2600 + J)
    a = W.random_spectrum(N, F, "flat", seed=2700 + J)
    assert_fp64_close(p.forward(to_cuda(x, torch.float64)).cpu().numpy(), O.analysis(x, N))
    assert_fp64_close(p.inverse(to_cuda(a, torch.complex128)).cpu().numpy(),
                      O.synthesis(a, N, J, I))
    p.status()


def test_more_than_a_million_fields(sht):
    # 2 F columns in blocks of 32: more blocks than a grid's second dimension holds
    N, J, I, F = 1, 5, 8, (1 << 20) + 1
    p = sht.Plan(N, J, I, F, "fp64")
    x = torch.randn(F, J, I, dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(2800))
    got = p.forward(x)
    pick = [0, 1, 12345, F - 2, F - 1]
    assert_fp64_close(got[:, pick].cpu().numpy(), O.analysis(x[pick].cpu().numpy(), N))
    back = p.inverse(got)
    assert_fp64_close(back[pick].cpu().numpy(), O.synthesis(got[:, pick].cpu().numpy(), N, J, I))
    p.status()
