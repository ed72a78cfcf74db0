"""Step lengths of the conjugate gradients near the top of FP32 and beyond: residuals
so large that p.Ap lies between 2^126 and 2^128, where an approximate division
returns zero and a component never leaves its start, and squares beyond FP32.  Every
size class, against the FP64 oracle, gates as in test_gpu_components."""
import numpy as np
import pytest

from oracle import spider_oracle as O
from paper_2508_12117_gb300 import binding
from test_gpu_components import _check

pytestmark = pytest.mark.gpu

KW = dict(sigma=0.005, kappa=0.03, p=0.25, ell=40.0, eps_w=1e-5)


def _first_pap(P):
    """p.Ap and |u|^2 of the first iteration in FP64 (Jacobi preconditioner)."""
    r = P.dt - (P.init[P.i, 3] - P.init[P.j, 3])
    sw = np.sqrt(P.w)
    lam = KW["sigma"] ** 2 / KW["kappa"] ** 2
    u, d = np.zeros(P.M), np.full(P.M, lam)
    for e, s in ((P.i, 1.0), (P.j, -1.0)):
        np.add.at(u, e, s * sw * r)
        np.add.at(d, e, P.w)
    y = u / d
    return float(lam * (y @ y) + P.w @ (y[P.i] - y[P.j]) ** 2), float(u @ u)


def _solve(m, log2_pap):
    """A path of m events whose first p.Ap is 2^log2_pap, against the oracle; |u|^2."""
    rng = np.random.default_rng(m)
    xyz = np.c_[np.sort(rng.uniform(0.0, 30.0, (m, 2)), axis=0), rng.uniform(5.0, 12.0, m)]
    th0 = np.c_[xyz, rng.uniform(0.0, 100.0, m)]
    i, j = np.arange(m - 1), np.arange(1, m)
    k, sta = np.zeros(m - 1, np.int32), np.array([[40.0, 5.0, 0.0]])
    noise = rng.normal(0.0, 1.0, m - 1)

    def problem(scale):
        dt = th0[i, 3] - th0[j, 3] + scale * noise
        return dt, O.Problem(th0, sta, i, j, k, dt, O.Model("homogeneous", v0=6.0),
                             sig_e=np.array([0.5, 0.5, 0.5, 0.1]), sig_c=np.full(4, 0.01), **KW)

    scale = np.sqrt(2.0 ** log2_pap / _first_pap(problem(1e9)[1])[0]) * 1e9
    dt, P = problem(scale)
    pap, uu = _first_pap(P)
    assert abs(np.log2(pap) - log2_pap) < 0.1
    ctx = binding.Context(th0, i, j, k, dt, sta, binding.Net(binding.TT_HOMOGENEOUS, v0=6.0),
                          binding.make_config(block_obs=4096, batch_n=0, **KW))
    _check(ctx, P)
    ctx.close()
    return uu


@pytest.mark.parametrize("m", [50, 200, 400, 900, 1500])
def test_large_residuals_converge(m):
    assert _solve(m, 126.6) < 2.0 ** 127.9


@pytest.mark.parametrize("m", [50, 200, 400, 900, 1500])
def test_squares_beyond_fp32_converge(m):
    assert _solve(m, 150.0) > 2.0 ** 129
