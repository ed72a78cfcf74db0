"""Ranges of the pool of the whitening components' matrix entries: the largest
accepted catalog (N < 2^30 observations, so up to 4 N entries with padding) must
stay inside the 32-bit cursor, every slice inside its range and all slices inside
the pool.  Checked on the CPU through the header the kernels use."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2508_12117_gb300", "csrc")
I31 = (1 << 31) - 1


@pytest.fixture(scope="module")
def pool(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("pool") / "pool_harness.so")
    subprocess.run(["g++", "-O2", "-fPIC", "-shared", "-std=c++17", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "pool_harness.cpp"), "-o", so], check=True, capture_output=True)
    L = C.CDLL(so)
    L.pool_begin.restype = L.pool_size.restype = C.c_int64
    L.pool_begin.argtypes = [C.c_int32]
    L.pool_size.argtypes = [C.c_int64, C.c_int64]
    return L


def _lengths(rng, kind, rows):
    if kind == "even":
        return rng.integers(4, 9, rows)
    if kind == "uneven":
        return np.where(rng.random(rows) < 0.05, rng.integers(50, 400, rows), 1)
    return np.ones(rows, int)


@pytest.mark.parametrize("kind", ["even", "uneven", "ones"])
@pytest.mark.parametrize("rows", [33, 65, 1000, 4001])
def test_slices_stay_inside_the_pool(pool, kind, rows):
    """Components of the worst row counts, nothing kept in shared memory: the
    grains taken fit the pool, and a slice's entries fit its grains."""
    rng = np.random.default_rng(rows)
    taken = entries = pairs = 0
    for _ in range(50):
        length = _lengths(rng, kind, rows)
        for a in range(0, rows, 32):
            x = length[a:a + 32]
            rest, steps = int(x.sum()), (int(x.max()) + 3) // 4 * 4
            used = 32 * steps if pool.pool_is_padded(steps, rest) else rest
            grains = pool.pool_takes(steps, rest)
            assert used <= 4 * grains
            taken += grains
        entries += int(length.sum())
        pairs += rows
    assert 4 * taken <= pool.pool_size((entries + 1) // 2, pairs)


@pytest.mark.parametrize("rows", [32, 31])
def test_largest_catalog_fits_the_cursor(pool, rows):
    """N = 2^30 - 1 observations in slices of `rows` even rows of eight entries
    (padded to twice as many at most): the cursor and the end of the last slice."""
    N, P = (1 << 30) - 1, (1 << 31) - 1
    per = rows * 8
    count = 2 * N // per
    cursor = count * pool.pool_takes(8, per)
    assert cursor <= I31 and pool.pool_size(N, P) // 4 <= I31
    last = cursor - pool.pool_takes(8, per)
    assert pool.pool_begin(last) == pool.pool_begin(~last) == 4 * last
    assert pool.pool_begin(last) + 32 * 8 <= pool.pool_size(N, P)


@pytest.mark.parametrize("steps,rest", [(1 << 27, 1 << 30), (1 << 30, (1 << 31) - 2), (1 << 26, 1 << 30)])
def test_positions_inside_a_slice_fit_32_bits(pool, steps, rest):
    """A handful of pairs that hold every observation: 32 steps of the padded
    layout would pass 2^31, so the slice is not padded."""
    assert not pool.pool_is_padded(steps, rest)
    assert 0 < pool.pool_takes(steps, rest) <= (rest + 3) // 4
