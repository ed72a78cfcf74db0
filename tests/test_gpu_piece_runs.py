"""Components of several CTAs that are made of very many pieces: their pieces are
ordered in runs of 4096 (bisection between runs), at the edges of a run and far
beyond it, against the FP64 oracle, and the time of a component must not grow with
the square of its pieces.  Gates as in test_gpu_components."""
import numpy as np
import pytest

from oracle import spider_oracle as O
from paper_2508_12117_gb300 import binding
from test_gpu_components import _check

pytestmark = pytest.mark.gpu


def _problem(m, n, block_obs, batch_n=0):
    """m events at one station: a path and random chords, n observations."""
    rng = np.random.default_rng(m + n)
    xyz = np.c_[np.sort(rng.uniform(0.0, 30.0, (m, 2)), axis=0), rng.uniform(5.0, 12.0, m)]
    th0 = np.c_[xyz, rng.uniform(0.0, 100.0, m)]
    i = rng.integers(0, m, n)
    j = (i + rng.integers(1, m, n)) % m
    i[:m - 1], j[:m - 1] = np.arange(m - 1), np.arange(1, m)
    dt = th0[i, 3] - th0[j, 3] + rng.normal(0.0, 0.05, n)
    k, sta = np.zeros(n, np.int32), np.array([[40.0, 5.0, 0.0]])
    kw = dict(sigma=0.005, kappa=0.03, p=0.25, ell=40.0, eps_w=1e-5)
    ctx = binding.Context(th0, i, j, k, dt, sta, binding.Net(binding.TT_HOMOGENEOUS, v0=6.0),
                          binding.make_config(block_obs=block_obs, batch_n=batch_n, **kw))
    P = O.Problem(th0, sta, i, j, k, dt, O.Model("homogeneous", v0=6.0), sig_e=np.array([0.5, 0.5, 0.5, 0.1]),
                  sig_c=np.full(4, 0.01), batch_n=batch_n, block_obs=block_obs, **kw)
    return ctx, P


@pytest.mark.parametrize("n", [1025, 4096, 4097, 8193, 50000])
def test_components_of_many_pieces(n):
    ctx, P = _problem(600, n, 1)
    _check(ctx, P)
    assert ctx.spider_info()["units_global"] == 1
    a, _ = ctx.spider_grad_logpost(0)
    b, _ = ctx.spider_grad_logpost(0)
    assert np.array_equal(a, b)
    ctx.close()


def test_minibatch_of_many_pieces():
    """Half of the one-observation blocks, selected in the order of the draw."""
    ctx, P = _problem(600, 40000, 1, batch_n=20000)
    for seed in (3, 4):
        _check(ctx, P, seed, P.batch(seed))
    assert ctx.spider_info()["units_global"] >= 1
    ctx.close()


def test_time_does_not_grow_with_the_square_of_the_pieces():
    """The same rows and entries cut into 96,000 pieces and into at most 3,000:
    pieces compared with each other took about ten times the iteration."""
    ms = []
    for block_obs in (1, 64):
        ctx, _ = _problem(1200, 96000, block_obs)
        ctx.spider_set_timing(True)
        t = []
        for _ in range(6):
            ctx.spider_grad_logpost(0)
            t.append(ctx.spider_last_whiten_timing()["cta_passes"])
        ms.append(float(np.median(t[1:])))
        ctx.close()
    print(f"several-CTA phase: 96,000 pieces {ms[0]:.2f} ms, {ms[1]:.2f} ms in blocks of 64")
    assert ms[0] <= 3.0 * ms[1] + 1.0
