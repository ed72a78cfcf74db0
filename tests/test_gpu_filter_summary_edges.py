"""Edges of the observation filters and the posterior summaries: medians of several
sub-problems (histograms in shared memory up to eight, in global memory beyond), odd
and even counts, ties; series whose lengths are no multiple of the lags taken
together, a wrapped sample ring, and lengths that leave fewer warps a CTA."""
import numpy as np
import pytest

from oracle import spider_oracle as O
from paper_2508_12117_gb300 import binding

pytestmark = pytest.mark.gpu

NET = (binding.TT_HOMOGENEOUS, 6.0)


class _Cat:
    def __init__(self, M, N, seed, distinct=None):
        rng = np.random.default_rng(seed)
        self.M, self.N, self.S = M, N, 4
        self.init_xyzt = np.c_[rng.uniform(0, 20, (M, 2)), rng.uniform(5, 12, M), rng.uniform(0, 100, M)]
        i, s, k = rng.integers(0, M, N), rng.integers(1, M, N), rng.integers(0, 4, N)
        noise = rng.standard_t(2, N) * 0.05
        if distinct:                                   # repeated observations: equal residuals
            i, s, k, noise = (a[np.arange(N) % distinct] for a in (i, s, k, noise))
        self.i, self.j, self.k = i.astype(np.int32), ((i + s) % M).astype(np.int32), k.astype(np.int32)
        self.dt = self.init_xyzt[self.i, 3] - self.init_xyzt[self.j, 3] + noise
        self.stations = np.c_[rng.uniform(-10, 30, (4, 2)), np.zeros(4)]


@pytest.mark.parametrize("chains", [1, 2, 3, 40])
def test_masks_of_several_sub_problems(chains):
    """Bit for bit: median, MAD and mask of the FP32 residuals of every sub-problem
    (4, 8, 12 and 160 of them)."""
    cats = [_Cat(20, 301, 1), _Cat(30, 400, 2), _Cat(5, 1, 3), _Cat(12, 260, 4, distinct=7)]
    ctx = binding.Context.batch(cats, chains, binding.Net(*NET),
                                binding.make_config(sigma=0.01, kappa=0.0, block_obs=1))
    keep, med, mad = ctx.spider_outlier_mask(4.0)
    idx, r, _ = ctx.spider_debug_obs(ctx.N)
    res = np.empty(ctx.N, np.float32)
    res[idx] = r
    off = 0
    for s, cat in enumerate(c for c in cats for _ in range(chains)):
        x = res[off:off + cat.N]
        mid = [(cat.N - 1) // 2, cat.N // 2]
        m = np.float32(0.5) * np.float32(np.sort(x)[mid].sum(dtype=np.float32))
        a = np.abs(x - m)
        d = np.float32(0.5) * np.float32(np.sort(a)[mid].sum(dtype=np.float32))
        assert med[s] == m and mad[s] == d, s
        assert np.array_equal(keep[off:off + cat.N], a <= np.float32(4.0) * d), s
        off += cat.N
    again = ctx.spider_outlier_mask(4.0)               # counters and histograms were left clean
    assert all(np.array_equal(p, q) for p, q in zip((keep, med, mad), again))
    ctx.close()


@pytest.mark.parametrize("cap,steps", [(5, 1), (5, 2), (7, 3), (8, 6), (33, 50), (301, 450), (1030, 1200),
                                       (2049, 2100), (4096, 4100)])
def test_summaries_of_any_length(cap, steps):
    cat = _Cat(6, 60, 9)
    ctx = binding.Context(cat.init_xyzt, cat.i, cat.j, cat.k, cat.dt, cat.stations, binding.Net(*NET),
                          binding.make_config(sigma=0.01, kappa=0.0, thin=1, sample_cap=cap))
    for t in range(steps):
        ctx.spider_sgld_step(2e-6, 70 + t)
    samples = ctx.spider_samples(cap)
    assert samples.shape[0] == min(cap, steps)
    truth = samples.mean(axis=0) + 1e-4
    if steps == 1:                                     # a summary needs two samples
        with pytest.raises(binding.SpiderError):
            ctx.spider_uq(truth, 2.5, 97.5)
        ctx.close()
        return
    uq = ctx.spider_uq(truth, 2.5, 97.5)
    med, half, calib, ess = O.uq_stats(samples, truth, 2.5, 97.5)
    assert np.abs(uq["median"] - med).max() <= 1e-9
    assert np.abs(uq["halfwidth"] - half).max() <= 1e-9
    assert np.array_equal(uq["calib"], calib)
    print(f"n {samples.shape[0]}: ESS rel {np.abs(uq['ess'] / ess - 1).max():.1e}")
    assert np.abs(uq["ess"] / ess - 1).max() <= 1e-9
    ctx.close()
