"""Conjugate gradients on the whitening components at the edges of their size
classes (one warp, CTAs of 8, 16 and 32 warps, several CTAs) against the FP64
oracle: one station, so a component has as many rows as its event graph has
events.  Gates are the FP32 ones of the other parity tests: gradient and
q = Sigma^-1 r rel-L2 <= 1e-5."""
import numpy as np
import pytest

from oracle import spider_oracle as O
from paper_2508_12117_gb300 import binding

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _problem(graph, m, block_obs, batch_n=0, seed=0):
    """m events observed at one station, linked as a path with random chords
    ("mesh": even rows) or to event 0 and to their neighbour ("star": one row
    with an entry per event)."""
    rng = np.random.default_rng(seed + m)
    xyz = np.sort(rng.uniform(0.0, 30.0, (m, 3)), axis=0)
    xyz[:, 2] = rng.uniform(5.0, 12.0, m)
    th0 = np.c_[xyz, rng.uniform(0.0, 100.0, m)]
    a = np.arange(m - 1)
    if graph == "mesh":
        c = rng.integers(0, m, (3 * m, 2))
        c = c[c[:, 0] != c[:, 1]]
        pairs = np.concatenate([np.c_[a, a + 1], c]) if m > 2 else np.c_[a, a + 1]
    else:
        pairs = np.concatenate([np.c_[np.zeros(m - 1, int), a + 1], np.c_[a[1:], a[1:] + 1]])
    i, j = pairs[:, 0], pairs[:, 1]
    k = np.zeros(len(i), np.int32)
    sta = np.array([[40.0, 5.0, 0.0]])
    dt = th0[i, 3] - th0[j, 3] + rng.normal(0.0, 0.05, len(i))
    kw = dict(sigma=0.005, kappa=0.03, p=0.25, ell=40.0, eps_w=1e-5)
    cfg = binding.make_config(block_obs=block_obs, batch_n=batch_n, **kw)
    ctx = binding.Context(th0, i, j, k, dt, sta, binding.Net(binding.TT_HOMOGENEOUS, v0=6.0), cfg)
    P = O.Problem(th0, sta, i, j, k, dt, O.Model("homogeneous", v0=6.0), sig_e=np.array([0.5, 0.5, 0.5, 0.1]),
                  sig_c=np.full(4, 0.01), batch_n=batch_n, block_obs=block_obs, **kw)
    return ctx, P


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def _check(ctx, P, seed=0, sel=None):
    g, _ = ctx.spider_grad_logpost(seed)
    _, go, info = O.log_posterior(P, P.init, sel)
    idx, _, q = ctx.spider_debug_obs(P.N)
    qo = info["q"] if sel is None else info["q"][np.searchsorted(sel, idx)]
    rg, rq = _rel(g, go), _rel(q, qo if sel is not None else qo[idx])
    print(f"gradient rel-L2 {rg:.2e}, q rel-L2 {rq:.2e}, iterations {ctx.spider_last_timing()['pcg_iters']}")
    assert rg <= TOL and rq <= TOL


@pytest.mark.parametrize("graph", ["mesh", "star"])
@pytest.mark.parametrize("m", [2, 3, 33, 64, 65, 255, 256, 257, 511, 513, 1024, 1025, 2500, 5000])
def test_component_sizes(graph, m):
    ctx, P = _problem(graph, m, 4096)
    _check(ctx, P)
    assert ctx.spider_info()["components"] == 1
    ctx.close()


@pytest.mark.parametrize("m,block_obs", [(40, 2), (60, 8), (300, 4), (700, 2), (1500, 16)])
def test_components_of_many_pieces(m, block_obs):
    """Tiny blocks: a component's rows are shared by many pieces (more than its
    row count would take, so the piece limits of the classes are crossed)."""
    ctx, P = _problem("mesh", m, block_obs)
    _check(ctx, P)
    ctx.close()


@pytest.mark.parametrize("m", [300, 3000])
def test_minibatch_components(m):
    """Half of the blocks per step: pieces solved with their inverses beside
    components of every class, gradients of two seeds and a reproducible chain."""
    ctx, P = _problem("mesh", m, 32, batch_n=2 * m)
    for seed in (3, 4):
        _check(ctx, P, seed, P.batch(seed))
    b, _ = _problem("mesh", m, 32, batch_n=2 * m)
    for s in range(4):
        ctx.spider_sgld_step(1e-6, 50 + s)
        b.spider_sgld_step(1e-6, 50 + s)
    assert np.array_equal(ctx.spider_get_state()[0], b.spider_get_state()[0])
    ctx.close()
    b.close()
