"""The form of the FP32 travel-time kernel inside a step follows the pairs that the
step can have, not the catalog's."""
import ctypes as C

import pytest

from test_mlp32_shape import lib  # noqa: F401


@pytest.mark.parametrize("H,P,n_b,nodes,narrow", [
    (128, 3_000_000, 2, 300, 1),      # a small minibatch of a large catalog
    (128, 3_000_000, 100, 3000, 0),   # a large one
    (128, 600, 100, 3000, 1),         # a small catalog, every block
    (128, 4864, 1 << 20, 8192, 1), (128, 4865, 1 << 20, 8192, 0),
    (64, 1 << 30, 1, 2 * 4864, 1), (64, 1 << 30, 1, 2 * 4864 + 1, 0),
])
def test_form_follows_the_step(lib, H, P, n_b, nodes, narrow):  # noqa: F811
    f = lib.mlp32_step_is_narrow
    f.argtypes = [C.c_int, C.c_longlong, C.c_longlong, C.c_longlong, C.c_int]
    assert f(H, P, n_b, nodes, 152) == narrow
