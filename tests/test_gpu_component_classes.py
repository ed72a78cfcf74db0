"""Many components of one size, so that the largest size class a catalog can
reach is each one in turn (larger classes are not launched), with more
components than CTAs are resident.  Against the FP64 oracle, gates as in
test_gpu_components."""
import numpy as np
import pytest

from oracle import spider_oracle as O
from paper_2508_12117_gb300 import binding
from test_gpu_components import _rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,stations,block_obs", [(60, 700, 4096), (200, 350, 4096), (400, 180, 4096), (900, 170, 4096),
                                                  (1100, 90, 4096), (1200, 3, 4)])
def test_components_of_the_largest_class_reached(m, stations, block_obs):
    """Every station a component of m rows; the last with blocks so small that a
    component's pieces, not its rows, put it in the class of several CTAs."""
    rng = np.random.default_rng(m)
    xyz = np.c_[np.sort(rng.uniform(0.0, 30.0, (m, 2)), axis=0), rng.uniform(5.0, 12.0, m)]
    th0 = np.c_[xyz, rng.uniform(0.0, 100.0, m)]
    a = np.arange(m - 1)
    per = [np.concatenate([np.c_[a, a + 1], (c := rng.integers(0, m, (2 * m, 2)))[c[:, 0] != c[:, 1]]])
           for _ in range(stations)]
    i, j = (np.concatenate([p[:, e] for p in per]) for e in (0, 1))
    k = np.concatenate([np.full(len(p), s, np.int32) for s, p in enumerate(per)])
    sta = np.c_[rng.uniform(-10.0, 40.0, (stations, 2)), np.zeros(stations)]
    dt = th0[i, 3] - th0[j, 3] + rng.normal(0.0, 0.05, len(i))
    kw = dict(sigma=0.005, kappa=0.03, p=0.25, ell=40.0, eps_w=1e-5)
    ctx = binding.Context(th0, i, j, k, dt, sta, binding.Net(binding.TT_HOMOGENEOUS, v0=6.0),
                          binding.make_config(block_obs=block_obs, batch_n=0, **kw))
    P = O.Problem(th0, sta, i, j, k, dt, O.Model("homogeneous", v0=6.0), sig_e=np.array([0.5, 0.5, 0.5, 0.1]),
                  sig_c=np.full(4, 0.01), batch_n=0, block_obs=block_obs, **kw)
    g, _ = ctx.spider_grad_logpost(0)
    _, go, info = O.log_posterior(P, P.init)
    assert _rel(g, go) <= 1e-5
    assert ctx.spider_info()["components"] == stations
    g2, _ = ctx.spider_grad_logpost(0)
    assert np.array_equal(g, g2)
    ctx.close()
