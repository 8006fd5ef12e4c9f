"""The two-float forms over steps and data scales: u(x) = L^2 u0(x / L) has the
Hessian of u0 on a cube of edge L, s u0 has s times the Hessian and s^3 times the
right-hand side.  FP64 arithmetic gives the same relative errors at every scale,
and so must every FP64 cycle and single step, whose two-float arithmetic has
FP32's range.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1411_7018_gb300 import libma as M
from paper_1411_7018_gb300 import problems as P

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps
INNER = (slice(1, -1),) * 3

# cube edge L and data scale s; 257^3 with L = 4e-5 has 1 / (64 h^6) beyond FP32, s = 1e7 has |u| beyond 2^20
SCALES = [(1e-6, 1.0), (4e-5, 1.0), (1e-4, 1.0), (1e-3, 1.0), (1e3, 1.0), (1.0, 1e-3), (1.0, 1e-7), (1.0, 1e-8),
          (1.0, 1e7), (1e-4, 1e-7)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    M.load()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def scaled(n, length, s, amp):
    """(u, f, h) of Example 4 with a seeded roughness, scaled."""
    pr = P.make("exp", n)
    u = pr.u.copy()
    u[INNER] += amp * np.random.default_rng(n).standard_normal((n - 2,) * 3)
    return s * length ** 2 * u, s ** 3 * pr.f, length / (n - 1)


@pytest.mark.parametrize("length,s", SCALES)
@pytest.mark.parametrize("n", [9, 33, 35, 65, 129, 257])
def test_residual_and_coarse_rhs_over_scales(n, length, s):
    """Against the oracle's FP64 forms, within the bound those are held to: 64 roundings of |u| / h^2
    in a second difference, times the largest cofactor (all relative to the scale)."""
    u, f, h = scaled(n, length, s, 1e-2 / (n - 1) ** 2)
    bound = 64.0 * EPS * np.max(np.abs(u)) / h ** 2 * (s * np.exp(1.5) * 4.0) ** 2
    out = torch.full_like(dev(u), 7.0)
    M.ma_residual_f2(dev(u), dev(f), out, n, h)
    assert np.max(np.abs(host(out) - O.residual(u, f, h))) <= bound
    r = 1e-3 * f
    M.ma_coarse_rhs(dev(u), dev(r), out, n, h)
    assert np.max(np.abs(host(out) - O.coarse_rhs(u, r, h))) <= bound


@pytest.mark.parametrize("n", [33, 65])
@pytest.mark.parametrize("rhs", [0.0, 1e-30, 1e-25, 1e-21, 1e30, 1e39, 1e300, np.inf, np.nan])
def test_operators_keep_the_range_of_the_other_term(n, rhs):
    """A right-hand side far from det(D^2 u), as large, small or odd as FP64 has them."""
    u, f, h = scaled(n, 1.0, 1.0, 0.0)
    b = np.full_like(f, rhs)
    bound = 64.0 * EPS * (np.max(np.abs(u)) / h ** 2 * (np.exp(1.5) * 4.0) ** 2 + (rhs if np.isfinite(rhs) else 0.0))
    out = torch.zeros_like(dev(u))
    for call, ref in ((M.ma_residual_f2, O.residual(u, b, h)), (None, O.coarse_rhs(u, b, h))):
        if call:
            call(dev(u), dev(b), out, n, h)
        else:
            M.ma_coarse_rhs(dev(u), dev(b), out, n, h)
        got, ref = host(out)[INNER], ref[INNER]
        if np.isfinite(rhs):
            assert np.max(np.abs(got - ref)) <= bound
        else:
            assert np.array_equal(got, ref, equal_nan=True)


def _cycled(n, length, s, precision, cycles, **kw):
    u, f, h = scaled(n, length, s, 1e-3 / (n - 1))
    H = M.Hierarchy(M.make_desc(n, length=length, precision=precision, **kw))
    H.set_rhs_bc(dev(f), dev(u))
    H.vcycle(cycles)
    out = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    H.get_solution(out)
    H.close()
    return host(out) / (s * length ** 2)


@pytest.mark.parametrize("length,s", SCALES)
@pytest.mark.parametrize("n,kw", [(17, dict(coarsest_n=5)), (33, {}), (65, {}), (257, {})])
def test_fp64_cycles_over_scales(n, kw, length, s):
    """Two V-cycles at a scale against the unscaled ones: the same method on data that differ by a
    rounding; whole cycles are held to 1e-12."""
    ref = _cycled(n, 1.0, 1.0, M.MA_FP64, 2, **kw)
    assert np.max(np.abs(_cycled(n, length, s, M.MA_FP64, 2, **kw) - ref)) <= 1e-12 * np.max(np.abs(ref))


def _solved(n, length, s, precision, tol):
    _, f, h = scaled(n, length, s, 0.0)
    pr = P.make("exp", n)
    H = M.Hierarchy(M.make_desc(n, length=length, precision=precision))
    H.set_rhs_bc(dev(f), dev(s * length ** 2 * pr.initial()))
    res = H.solve(tol=tol, max_cycles=25)
    out = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    H.get_solution(out)
    H.close()
    return host(out) / (s * length ** 2), res


# the norms are taken in FP32: sums of squares of f beyond 1e19 overflow there, so no s = 1e7
@pytest.mark.parametrize("length,s", [v for v in SCALES if v[1] <= 1.0])
@pytest.mark.parametrize("n,precision,tol", [(33, M.MA_FP64, 1e-11), (65, M.MA_FP64, 1e-11), (257, M.MA_FP64, 1e-10),
                                             (33, M.MA_MIXED, 1e-10)])
def test_solves_over_scales(n, precision, tol, length, s):
    """Whole solves converge, and to the unscaled solution: with residuals of tol max f both are within
    tol |u| of the discrete one (det is of degree 3 in u: a third of it, on average)."""
    ref, _ = _solved(n, 1.0, 1.0, precision, tol)
    got, res = _solved(n, length, s, precision, tol)
    assert res.res <= tol
    assert np.max(np.abs(got - ref)) <= 10 * tol * np.max(np.abs(ref))
