"""Contexts of different block sizes live side by side."""
import numpy as np
import pytest

from paper_2508_12117_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def test_older_context_with_larger_blocks_still_steps():
    """The per-block kernels' shared memory follows the context's largest block;
    a context created later with smaller blocks leaves the older one's launches
    valid."""
    cat = synth.make_catalog(1)
    a = binding.Context.from_catalog(cat, block_obs=4096)
    want, _ = a.spider_grad_logpost(0)
    b = binding.Context.from_catalog(cat, block_obs=16)
    got, _ = a.spider_grad_logpost(0)
    assert np.array_equal(got, want)
    b.spider_grad_logpost(0)
    a.close()
    b.close()
