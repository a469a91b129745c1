"""The shapes that the pass over a group's carriers may take, without a GPU:
whatever the grid, the tables, the period and the number of slots, a block has
the 256 threads that its barriers count, and its sizes are ones that exist."""
import ctypes as C
import itertools

import pytest

from paper_1807_04733_gb300 import build as B
from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

SMEM = 227 * 1024 - 2048


@pytest.fixture(scope="module")
def shapes():
    B.build()
    f = pic.lib().pic_group_shapes
    f.argtypes = [C.c_int] * 5 + [C.c_uint, C.c_longlong, C.c_int, C.c_longlong, C.c_void_p, C.c_int]

    def get(n_stacks, n_e, layers, cells, me, flags, slots):
        out = (C.c_int * 300)()
        n = f(n_stacks, n_e, layers, cells, me, flags, slots, 152, SMEM, out, 100)
        assert n <= 100
        return [tuple(out[3 * i: 3 * i + 3]) for i in range(n)]
    return get


@pytest.mark.parametrize("flags", [0, W.FLAG_VELOCITY, W.FLAG_WEIGHTS])
@pytest.mark.parametrize("n_stacks,layers", [(1, 1), (1, 2), (1, 6), (1, 16), (64, 3)])
def test_every_shape_has_the_threads_of_its_barriers(shapes, n_stacks, layers, flags):
    seen = 0
    for n_e, cells, me, slots in itertools.product(
            [1, 4, 30, 60, 100, 200, 255], [1, 20, 115, 278, 315, 360, 500, 700, 1500, 5000, 20000],
            [1, 2, 3, 4, 50], [0, 10 ** 4, 900_000, 940_000, 1_870_000, 8 << 20, (8 << 20) + 1, 1 << 30]):
        for m, quads, warps in shapes(n_stacks, n_e, layers, cells, me, flags, slots):
            seen += 1
            assert 8 <= warps <= 16 and quads in (2, 4, 8) and 1 <= m <= 8, (n_e, cells, me, slots)
            assert m <= 4 or slots <= 8 << 20
            # no kernel of 1024-slot sub-tiles with densities
            assert quads <= 4 or me >= 4 or flags & W.FLAG_WEIGHTS
            # groups of one step: densities every step and few slots
            assert m > 1 or (me == 1 and slots <= 2 << 20)
    assert seen > 1000


def test_known_shapes(shapes):
    """The usual grids have shapes of several steps; the 315-cell, 60-bin grid
    with densities in most steps and many slots had one of six warps."""
    assert shapes(1, 30, 2, 115, 1, 0, 400_000)[0][0] >= 4
    assert shapes(1, 60, 2, 315, 50, 0, 400_000_000)[0][:2] == (4, 8)
    for me in (1, 2, 3):
        assert shapes(1, 60, 2, 315, me, 0, 1_200_000) == []
        assert all(w >= 8 for _, _, w in shapes(1, 60, 2, 315, me, 0, 40_000))
