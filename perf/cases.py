"""Performance cases: the transforms a user of this library runs, over the
sizes, precisions, grids and directions it is used with.

Every case goes through ``paper_1711_11296_gb300.sht``.  ``prepare`` makes
the plan (or the group of plans) that a program keeps for its whole run and
the seeded fields of one step; ``run`` is one step on them.

Kinds of step:

* ``pair``: synthesis then analysis of F field-levels, the spectral part of
  a model's time step (optionally on a reduced or polyhedral grid).
* ``forward`` / ``inverse``: one transform alone (initialisation and
  diagnostics read a grid; output writes one).
* ``grad``: analysis of a grid and the gradient of a loss on the spectrum
  back to the grid, through autograd (training, data assimilation).
* ``grad_inverse``: the same for the synthesis.
* ``group``: synthesis then analysis of an uneven ensemble, four truncations
  in one grouped launch per stage.
* ``alias``: the quadratic and cubic products of three synthesised fields,
  analysed (nonlinear terms).
* ``restrict``: the coarse spectrum of a nested fine grid (multigrid).
"""
import math

import numpy as np
import torch

from paper_1711_11296_gb300 import sht

ENVELOPES = ("energy^-2", "uniform^-1/3")


def _case(name, kind, N, J, I, F, precision, grid="cc"):
    return {"name": name, "kind": kind, "N": N, "J": J, "I": I, "F": F,
            "precision": precision, "grid": grid}


def listed():
    return [
        # the smallest call: one scalar field at T31 (the paper's smallest
        # shallow-water truncation), bound by launches and their gaps
        _case("t31_fp64_pair_1", "pair", 31, 65, 128, 1, "fp64"),
        # a few levels of a small ensemble member: an odd field count
        _case("t63_bf16x3_pair_7", "pair", 63, 129, 256, 7, "bf16x3"),
        # a dynamical-core step at Tc159, 4 fields x 64 levels, in the
        # paper's precision and in the split one
        _case("t159_fp64_pair_256", "pair", 159, 321, 640, 256, "fp64"),
        _case("t159_bf16x3_pair_256", "pair", 159, 321, 640, 256, "bf16x3"),
        # an FP64 gradient at T319, 100 levels (adjoint-based assimilation)
        _case("t319_fp64_grad_100", "grad", 319, 641, 1280, 100, "fp64"),
        # reading 3 fields x 100 levels of grid data at T319, two FP16 terms
        _case("t319_fp16x2_forward_300", "forward", 319, 641, 1280, 300, "fp16x2"),
        # the library's headline step: T639, 4 fields x 64 levels, split
        _case("t639_bf16x3_pair_256", "pair", 639, 1281, 2560, 256, "bf16x3"),
        # the same in FP64, the largest case
        _case("t639_fp64_pair_256", "pair", 639, 1281, 2560, 256, "fp64"),
        # two members of the uneven ensemble T63 / T127 / T255 / T511,
        # 32 levels x 2 fields each, grouped
        _case("ensemble_bf16x3_128", "group", 511, 1025, 2048, 128, "bf16x3"),
        # nonlinear terms at the paper's aliasing resolution Tc479
        _case("tc479_bf16x3_alias_64", "alias", 479, 959, 1920, 64, "bf16x3"),
        # a step on the octahedral grid, whose rows have any even length
        _case("octahedral_t319_bf16x3_pair_64", "pair", 319, 641, 0, 64, "bf16x3",
              "octahedral"),
        # multigrid restriction T511 grid -> T255 spectrum
        _case("t255_bf16x3_restrict_64", "restrict", 255, 511, 1024, 64, "bf16x3"),
    ]


def _smooth_even(n):
    """The smallest even 2-3-5-smooth number >= n."""
    n += n % 2
    while True:
        r = n // 2
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if r == 1:
            return n
        n += 2


def draw(rng):
    """One more case: truncations 21..639 and 1..300 fields over their
    logarithms (powers of two, multiples and odd counts), every precision and
    step, longitudes for cubic, quadratic or linear truncation."""
    top = _work_units(listed()[7])
    while True:
        kind = rng.choice(["pair", "pair", "pair", "pair", "forward", "inverse", "grad",
                           "grad_inverse", "group", "alias", "restrict"])
        precision = rng.choice(["fp64", "fp64", "bf16x3", "bf16x3", "bf16x3", "fp16x2",
                                "fp16x3", "bf16x2"])
        grid = "cc"
        if kind == "pair":
            grid = rng.choice(["cc"] * 6 + ["fejer1", "octahedral", "icositetrahedral",
                                            "smooth", "fast"])
        N = int(round(math.exp(rng.uniform(math.log(21), math.log(639)))))
        if rng.random() < 0.6:   # truncations as models use them: N + 1 a multiple of 8
            N = max(23, (N + 1) // 8 * 8 - 1)
        F = int(round(math.exp(rng.uniform(0.0, math.log(300)))))
        if rng.random() < 0.5 and F > 4:
            F = F // 4 * 4
        if kind == "group":
            N = max(63, (N + 1) // 8 * 8 - 1)
        if kind in ("group", "alias"):
            F = min(F, 128)
        if kind == "restrict":
            N = min(N, 319)
            F = min(F, 128)
            J = 2 * N + 1
        else:
            J = 2 * N + 3
        if grid == "octahedral":
            I = 0
            J = 2 * N + 3
        elif grid == "icositetrahedral":
            # 6 j points up to 30 degrees: the tropical rows have 2 (J + 1)
            # of them, more than 2 N
            I = 0
            J = 2 * N + 3
        else:
            if kind == "alias" or grid in ("smooth", "fast"):
                per = 4
            else:
                per = rng.choice([4, 4, 4, 3, 2])
            I = _smooth_even(per * (N + 1))
        case = {"kind": kind, "N": N, "J": J, "I": I, "F": F, "precision": precision,
                "grid": grid}
        if _work_units(case) <= top:
            return case


def _sizes(case):
    """[(N, J, I)] of the case's plans (one, or the four of a group)."""
    N, J, I = case["N"], case["J"], case["I"]
    if case["kind"] != "group":
        return [(N, J, I)]
    out = []
    for d in (8, 4, 2):
        n = (N + 1) // d - 1
        out.append((n, 2 * n + 3, _smooth_even(4 * (n + 1))))
    return out + [(N, J, I)]


def _ncoef(N):
    return (N + 1) * (N + 2) // 2


def _points(case):
    """Grid points per field (the reduced grids by their leading fraction)."""
    J, I = case["J"], case["I"]
    if case["grid"] == "octahedral":
        return sum(_octahedral(J))
    if case["grid"] == "icositetrahedral":
        return sum(_icositetrahedral(J)[0])
    return J * I * (0.75 if case["grid"] in ("smooth", "fast") else 1.0)


def _transform_work(N, J, points, I, F, fp64):
    """Bytes and flops of one transform: grid and spectrum once, the
    Legendre functions once; folded Legendre sums and real row FFTs."""
    b = 8 if fp64 else 4
    jh = (J + 1) // 2
    nbytes = points * F * b + 2 * b * _ncoef(N) * F + b * _ncoef(N) * jh
    flops = 4.0 * _ncoef(N) * jh * F + 2.5 * points * F * math.log2(max(I, 2))
    return nbytes, flops


def work(case):
    fp64 = case["precision"] == "fp64"
    F = case["F"]
    nb = fl = 0.0
    for N, J, I in _sizes(case):
        row = I or 4 * (N + 1)
        pts = _points(case) if case["kind"] != "group" else J * I
        b1, f1 = _transform_work(N, J, pts, row, F, fp64)
        times = {"pair": 2, "group": 2, "grad": 2, "grad_inverse": 2, "alias": 5}.get(
            case["kind"], 1)
        if case["kind"] == "alias":
            # U, V, W in, two product grids and two spectra out
            b = 8 if fp64 else 4
            nb += 5 * 2 * b * _ncoef(N) * F + 2 * pts * F * b + b * _ncoef(N) * (J + 1) / 2
        else:
            nb += times * b1
        fl += times * f1
    return {"bytes": float(nb), "flops": float(fl)}


def _work_units(case):
    w = work(case)
    # FP64 arithmetic is the slower of the two on this hardware
    return max(w["bytes"], w["flops"] / (0.2 if case["precision"] == "fp64" else 50))


# -- inputs ------------------------------------------------------------------

def _dtypes(case):
    if case["precision"] == "fp64":
        return torch.float64, torch.complex128
    return torch.float32, torch.complex64


def _degrees(N, device):
    """(n, m) of every packed row, m-major."""
    m = torch.repeat_interleave(torch.arange(N + 1, device=device),
                                torch.arange(N + 1, 0, -1, device=device))
    first = torch.cumsum(torch.arange(N + 1, 0, -1, device=device), 0) - torch.arange(
        N + 1, 0, -1, device=device)
    n = torch.arange(_ncoef(N), device=device) - first[m] + m
    return n, m


def _spectrum(N, F, gen, dtype, envelope="energy^-2"):
    """Random spectrum of real fields: energy falling as (n + 1)^-2, or the
    amplitude law of the aliasing experiment."""
    dev = gen.device
    n, m = _degrees(N, dev)
    nf = n.to(torch.float64)
    rd = torch.float64 if dtype == torch.complex128 else torch.float32
    shape = (_ncoef(N), F)
    if envelope == "energy^-2":
        amp = (nf + 1) ** -1.0 / torch.sqrt(2.0 * (2.0 * nf + 1.0))
        re = torch.randn(shape, generator=gen, device=dev, dtype=rd)
        im = torch.randn(shape, generator=gen, device=dev, dtype=rd)
    else:
        amp = (nf + 1) ** (-1.0 / 3.0)
        re = 1 + torch.rand(shape, generator=gen, device=dev, dtype=rd)
        im = 1 + torch.rand(shape, generator=gen, device=dev, dtype=rd)
    amp = amp.to(rd)[:, None]
    im[m == 0] = 0
    return torch.complex(re * amp, im * amp)


def _grid_field(F, J, I, gen, dtype):
    """Grid data as a model holds it: a zonal flow and a planetary wave per
    field, with weather (white noise) on top."""
    dev = gen.device
    th = math.pi * torch.arange(1, J + 1, device=dev, dtype=torch.float64) / (J + 1)
    lam = 2 * math.pi * torch.arange(I, device=dev, dtype=torch.float64) / I
    a = torch.rand((F, 3), generator=gen, device=dev, dtype=dtype)
    s, c = torch.sin(th).to(dtype), torch.cos(th).to(dtype)
    wave = ((s ** 4 * c)[:, None] * torch.cos(4 * lam).to(dtype)[None, :])
    x = torch.randn((F, J, I), generator=gen, device=dev, dtype=dtype)
    x.mul_(0.3)
    x.add_((10 * a[:, 0, None] + 20 * a[:, 1, None] * s ** 2)[:, :, None])
    for f in range(F):
        x[f].add_(wave, alpha=float(5 + f % 3))
    return x


def _octahedral(J):
    jh = (J + 1) // 2
    north = [20 + 4 * j for j in range(jh)]
    return north + north[-2::-1]


def _icositetrahedral(J):
    jh = (J + 1) // 2
    j30 = max(1, int((J + 1) / 3.0 + 0.5))
    pts = [6 * min(j, j30) for j in range(1, jh + 1)]
    sh = [(j - j30) % 2 if j > j30 else 0 for j in range(1, jh + 1)]
    return pts + pts[-2::-1], sh + sh[-2::-1]


def _plan(case, N, J, I):
    F, prec, grid = case["F"], case["precision"], case["grid"]
    if grid in ("cc", "fejer1"):
        return sht.Plan(N, J, I, F, prec, grid=grid)
    if grid == "octahedral":
        return sht.Plan(N, J, 0, F, prec, grid="reduced",
                        lat_points=sht.octahedral_grid_sizes(J))
    if grid == "icositetrahedral":
        pts, sh = sht.icositetrahedral_grid_sizes(J)
        return sht.Plan(N, J, 0, F, prec, grid="reduced", lat_points=pts, half_shift=sh)
    one = sht.Plan(N, J, I, 1, "fp64")
    sizes = one.reduced_grid_sizes(grid)
    one.close()
    return sht.Plan(N, J, I, F, prec, grid="reduced", lat_points=sizes)


def _inputs(case, seed):
    """The step's seeded tensors (no plan needed)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    rd, cd = _dtypes(case)
    N, J, I, F = case["N"], case["J"], case["I"], case["F"]
    kind = case["kind"]
    if kind == "group":
        return {"specs": [_spectrum(n, F, gen, cd) for n, _, _ in _sizes(case)]}
    if kind == "alias":
        return {"specs": [_spectrum(N, F, gen, cd, "uniform^-1/3") for _ in range(3)]}
    if kind == "restrict":
        return {"grid": _grid_field(F, 2 * J + 1, 2 * I, gen, rd)}
    if kind == "forward":
        return {"grid": _grid_field(F, J, I, gen, rd)}
    if kind == "grad":
        return {"grid": _grid_field(F, J, I, gen, rd), "cot": _spectrum(N, F, gen, cd)}
    if kind == "grad_inverse":
        return {"spec": _spectrum(N, F, gen, cd), "cot": _grid_field(F, J, I, gen, rd)}
    return {"spec": _spectrum(N, F, gen, cd)}


def prepare(case, seed):
    state = {"kind": case["kind"], **_inputs(case, seed)}
    if case["kind"] == "group":
        state["plans"] = [_plan(case, n, j, i) for n, j, i in _sizes(case)]
        state["group"] = sht.Group(state["plans"])
        state["grids"] = [p.empty_grid() for p in state["plans"]]
        state["outs"] = [p.empty_spec() for p in state["plans"]]
        return state
    p = state["plan"] = _plan(case, case["N"], case["J"], case["I"])
    kind = case["kind"]
    # result buffers that a time loop keeps
    if kind in ("pair", "inverse"):
        state["out_grid"] = p.empty_grid()
    if kind in ("pair", "forward", "restrict"):
        state["out_spec"] = p.empty_spec()
    if kind == "alias":
        state["grids"] = [p.empty_grid(), p.empty_grid()]
        state["outs"] = [p.empty_spec(), p.empty_spec()]
    if kind == "grad":
        state["grid"].requires_grad_()
    if kind == "grad_inverse":
        state["spec"].requires_grad_()
    return state


def run(state):
    kind = state["kind"]
    if kind == "group":
        grids = state["group"].inverse(state["specs"], out=state["grids"])
        specs = state["group"].forward(grids, out=state["outs"])
        return {"grids": grids, "specs": specs}
    p = state["plan"]
    if kind == "pair":
        grid = p.inverse(state["spec"], out=state["out_grid"])
        return {"grid": grid, "spec": p.forward(grid, out=state["out_spec"])}
    if kind == "forward":
        return {"spec": p.forward(state["grid"], out=state["out_spec"])}
    if kind == "inverse":
        return {"grid": p.inverse(state["spec"], out=state["out_grid"])}
    if kind == "restrict":
        return {"spec": p.restrict_nested(state["grid"], 1, out=state["out_spec"])}
    if kind == "alias":
        q, c = p.alias_products(*state["specs"], grids=state["grids"], out=state["outs"])
        return {"spec_q": q, "spec_c": c, "grid_q": state["grids"][0],
                "grid_c": state["grids"][1]}
    if kind == "grad":
        spec = sht.analysis(state["grid"], p)
        (g,) = torch.autograd.grad(spec, state["grid"], state["cot"])
        return {"spec": spec.detach(), "grad": g}
    if kind == "grad_inverse":
        grid = sht.synthesis(state["spec"], p)
        (g,) = torch.autograd.grad(grid, state["spec"], state["cot"])
        return {"grid": grid.detach(), "grad": g}
    raise ValueError(kind)


# -- the same in 64 bits, from the equations -----------------------------------

def _theta_weights(J, grid, dev):
    """Colatitudes and quadrature weights (Fejer's second rule, the paper's
    Clenshaw-Curtis form without the poles, or his first)."""
    j = torch.arange(1, J + 1, device=dev, dtype=torch.float64)
    if grid == "fejer1":
        th = math.pi * (j - 0.5) / J
        p = torch.arange(1, J // 2 + 1, device=dev, dtype=torch.float64)
        w = 2.0 / J * (1 - 2 * (torch.cos(2 * th[:, None] * p) / (4 * p * p - 1)).sum(1))
        return th, w
    th = math.pi * j / (J + 1)
    p = torch.arange(1, (J + 1) // 2 + 1, device=dev, dtype=torch.float64)
    w = 4 * torch.sin(th) / (J + 1) * (torch.sin(th[:, None] * (2 * p - 1)) / (2 * p - 1)).sum(1)
    return th, w


def _legendre(N, th):
    """P[m, n - m, j], normalised so that the integral of P^2 over mu is 1.
    Rows beyond the last are zero.  (Sectoral values below 1e-300 vanish;
    what they would grow to by n = N is far below the rounding.)"""
    dev = th.device
    mu, s = torch.cos(th), torch.sin(th)
    m = torch.arange(N + 1, device=dev, dtype=torch.float64)
    logc = 0.5 * torch.cumsum(torch.cat([m[:1], torch.log((2 * m[1:] + 1) / (2 * m[1:]))]), 0)
    P = torch.zeros((N + 1, N + 1, len(th)), device=dev, dtype=torch.float64)
    P[:, 0] = math.sqrt(0.5) * torch.exp(logc[:, None] + m[:, None] * torch.log(s)[None])

    def eps(n, mm):
        return torch.sqrt((n * n - mm * mm) / (4 * n * n - 1))[:, None]

    for k in range(1, N + 1):
        mm = m[:N + 1 - k]
        n = mm + k
        nxt = mu * P[:N + 1 - k, k - 1]
        if k > 1:
            nxt = nxt - eps(n - 1, mm) * P[:N + 1 - k, k - 2]
        P[:N + 1 - k, k] = nxt / eps(n, mm)
    return P


class _Exact:
    """Analysis, synthesis and their adjoints on rows of any length."""

    def __init__(self, N, J, F, sizes, shift, grid, dev):
        self.N, self.J, self.F, self.sizes, self.shift = N, J, F, sizes, shift
        self.th, self.w = _theta_weights(J, grid, dev)
        jh = (J + 1) // 2
        # one hemisphere: P(pi - th) = (-1)^(n - m) P(th)
        self.P = _legendre(N, self.th[:jh])
        self.dev, self.jh = dev, jh
        self.off = [0] + list(np.cumsum(sizes))
        self.regular = len(set(sizes)) == 1 and not any(shift)

    def _rows(self, m):
        a = m * (self.N + 1) - m * (m - 1) // 2
        return a, a + self.N - m + 1

    def to_fourier(self, spec):
        """[M, J, F] zonal coefficients of a spectrum."""
        out = torch.zeros((self.N + 1, self.J, self.F), device=self.dev, dtype=torch.complex128)
        for m in range(self.N + 1):
            a, b = self._rows(m)
            x = torch.view_as_real(spec[a:b]).reshape(b - a, -1)
            S = self.P[m, 0:b - a:2].T @ x[0::2]
            A = self.P[m, 1:b - a:2].T @ x[1::2] if b - a > 1 else torch.zeros_like(S)
            o = torch.view_as_real(out[m]).view(self.J, -1)
            o[:self.jh] = S + A
            o[self.jh:] = torch.flip((S - A)[:self.jh - 1], (0,))
        return out

    def from_fourier(self, four):
        """Spectrum of [M, J, F] zonal coefficients (already weighted)."""
        n = _ncoef(self.N)
        out = torch.zeros((n, self.F), device=self.dev, dtype=torch.complex128)
        for m in range(self.N + 1):
            a, b = self._rows(m)
            x = torch.view_as_real(four[m]).reshape(self.J, -1)
            south = torch.flip(x[self.jh:], (0,))
            S, A = x[:self.jh].clone(), x[:self.jh].clone()
            S[:self.jh - 1] += south
            A[:self.jh - 1] -= south
            A[self.jh - 1] = 0
            o = torch.view_as_real(out[a:b]).view(b - a, -1)
            o[0::2] = self.P[m, 0:b - a:2] @ S
            o[1::2] = self.P[m, 1:b - a:2] @ A
        return out

    def _classes(self):
        """(row length, shifted, rows) of the distinct kinds of row."""
        kinds = {}
        for j in range(self.J):
            kinds.setdefault((self.sizes[j], self.shift[j]), []).append(j)
        return [(I, sh, js) for (I, sh), js in kinds.items()]

    def _index(self, I, js):
        return (torch.tensor([self.off[j] for j in js], device=self.dev)[:, None]
                + torch.arange(I, device=self.dev))

    def rows_to_grid(self, four, half=False, scale=None):
        """Sum over m of c_m Re(Y_m e^{i m lambda}), c_0 = 1 and c_m = 2 (or
        1, half): the grid [F, J, I] (regular) or [F, points]."""
        out = torch.empty((self.F, self.off[-1]), device=self.dev, dtype=torch.float64)
        step = max(1, int(2e9 // (16 * self.F * max(self.sizes))))
        for I, sh, js_all in self._classes():
            for at in range(0, len(js_all), step):
                js = js_all[at:at + step]
                k = min(self.N, I // 2 - 1) + 1
                y = torch.zeros((len(js), self.F, I // 2 + 1), device=self.dev,
                                dtype=torch.complex128)
                y[:, :, :k] = four[:k, js].permute(1, 2, 0)
                if sh:
                    y[:, :, :k] *= torch.exp(1j * math.pi / I * torch.arange(
                        k, device=self.dev, dtype=torch.float64))
                if half:
                    y[:, :, 1:] *= 0.5
                y[:, :, 0] = y[:, :, 0].real.to(torch.complex128)
                x = torch.fft.irfft(y, n=I, norm="forward")
                if scale is not None:
                    x *= scale[js][:, None, None]
                out[:, self._index(I, js).reshape(-1)] = x.permute(1, 0, 2).reshape(self.F, -1)
        return out.view(self.F, self.J, -1) if self.regular else out

    def grid_to_rows(self, grid, scale, c1=1.0):
        """[M, J, F]: c_m scale_j sum_i x e^{-i m lambda}."""
        x = grid.reshape(self.F, -1)
        out = torch.zeros((self.N + 1, self.J, self.F), device=self.dev, dtype=torch.complex128)
        step = max(1, int(2e9 // (16 * self.F * max(self.sizes))))
        for I, sh, js_all in self._classes():
            for at in range(0, len(js_all), step):
                js = js_all[at:at + step]
                k = min(self.N, I // 2 - 1) + 1
                r = x[:, self._index(I, js).reshape(-1)].view(self.F, len(js), I)
                y = torch.fft.rfft(r.to(torch.float64))[:, :, :k]
                if sh:
                    y = y * torch.exp(-1j * math.pi / I * torch.arange(
                        k, device=self.dev, dtype=torch.float64))
                y = y * scale[js][None, :, None]
                if c1 != 1.0:
                    y[:, :, 1:] *= c1
                out[:k, js] = y.permute(2, 1, 0)
        return out

    def _wI(self):
        return self.w / torch.tensor(self.sizes, device=self.dev, dtype=torch.float64)

    def inverse(self, spec):
        return self.rows_to_grid(self.to_fourier(spec))

    def forward(self, grid):
        out = self.from_fourier(self.grid_to_rows(grid, self._wI()))
        out[:self.N + 1] = out[:self.N + 1].real.to(torch.complex128)
        return out

    def adjoint_forward(self, spec):
        return self.rows_to_grid(self.to_fourier(spec), half=True, scale=self._wI())

    def adjoint_inverse(self, grid):
        one = torch.ones(self.J, device=self.dev, dtype=torch.float64)
        out = self.from_fourier(self.grid_to_rows(grid, one, 2.0))
        out[:self.N + 1] = out[:self.N + 1].real.to(torch.complex128)
        return out


def _reduced_sizes(N, J, I, rule, dev):
    """The 1e-16 reduction rule: I_j >= 4 M_j + 1 longitudes, an even
    2-3-5-smooth count or one of the compile-time FFT lengths."""
    th, _ = _theta_weights(J, "cc", dev)
    jh = (J + 1) // 2
    P = _legendre(N, th[:jh])
    seen = (P.abs() >= 1e-16).any(1)   # [M, jh]
    mmax = (seen * torch.arange(N + 1, device=dev)[:, None]).amax(0).tolist()
    north = []
    for mj in mmax:
        need = 4 * mj + 1
        n = _smooth_even(need)
        if rule == "fast":
            n = next((2 * L for L in (64, 128, 256, 320, 512, 640, 1024, 1280)
                      if 2 * L >= need), I)
        north.append(min(I, n))
    return north + north[-2::-1]


def _exact_of(case, N, J, I):
    dev = torch.device("cuda")
    shift = [0] * J
    grid = case["grid"]
    if grid == "octahedral":
        sizes = _octahedral(J)
    elif grid == "icositetrahedral":
        sizes, shift = _icositetrahedral(J)
    elif grid in ("smooth", "fast"):
        sizes = _reduced_sizes(N, J, I, grid, dev)
    else:
        sizes = [I] * J
    return _Exact(N, J, case["F"], sizes, shift, "fejer1" if grid == "fejer1" else "cc", dev)


def exact(case, seed):
    kind, x = case["kind"], _inputs(case, seed)
    c128, f64 = torch.complex128, torch.float64
    if kind == "group":
        grids, specs = [], []
        for (n, j, i), s in zip(_sizes(case), x["specs"]):
            e = _exact_of(case, n, j, i)
            grids.append(e.inverse(s.to(c128)))
            specs.append(e.forward(grids[-1]))
        return {"grids": grids, "specs": specs}
    e = _exact_of(case, case["N"], case["J"], case["I"])
    if kind == "pair":
        g = e.inverse(x["spec"].to(c128))
        packed = case["grid"] not in ("cc", "fejer1")
        return {"grid": g.reshape(case["F"], -1) if packed else g, "spec": e.forward(g)}
    if kind == "forward":
        return {"spec": e.forward(x["grid"].to(f64))}
    if kind == "inverse":
        return {"grid": e.inverse(x["spec"].to(c128))}
    if kind == "restrict":
        return {"spec": e.forward(x["grid"][:, 1::2, ::2].to(f64))}
    if kind == "alias":
        u, v, w = (e.inverse(s.to(c128)) for s in x["specs"])
        u *= v
        q = e.forward(u)
        w *= u
        return {"spec_q": q, "spec_c": e.forward(w), "grid_q": u, "grid_c": w}
    if kind == "grad":
        return {"spec": e.forward(x["grid"].to(f64)), "grad": e.adjoint_forward(x["cot"].to(c128))}
    return {"grid": e.inverse(x["spec"].to(c128)), "grad": e.adjoint_inverse(x["cot"].to(f64))}
