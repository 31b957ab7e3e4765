"""Dispatch order of the FP64 step launches on the tiles that they run on (host logic, no
GPU): every tile column of every problem is covered by items whose planes join up from 0
to n - 1, at the sizes where the tile changes (8 x 8, 14 x 9, 32 x 8 nodes) and for the
depths from one plane up.  tests/test_step_items.py covers FP32 and the 32 x 8 tile."""
import numpy as np
import pytest

from paper_2508_07780_gb300.binding import DDFDError, step_items64


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_07780_gb300 import build
    build.build()


def cube_box(n, fem):
    a = (n - fem) // 2
    return (a, a + fem - 1, a + 2, fem - 4)


# n, FEM cubes, the tile of the launch
CASES = [(7, [5], (8, 8)), (13, [9], (8, 8)), (41, [21], (8, 8)), (48, [46], (8, 8)), (49, [25], (14, 9)),
         (33, [31, 9], (8, 8)), (33, [31, 20, 9] * 4, (14, 9)), (65, [33] * 16, (14, 9)), (161, [121], (14, 9)),
         (447, [101], (14, 9)), (448, [446], (14, 9)), (449, [225], (32, 8)), (1024, [9], (32, 8))]


@pytest.mark.parametrize("n,fems,tile", CASES, ids=lambda v: str(v) if isinstance(v, int) else f"{len(v)}-{v[0]}")
@pytest.mark.parametrize("kz", [1, 5, 12, 64])
def test_every_column_is_covered_once(n, fems, tile, kz):
    items, got = step_items64(n, [cube_box(n, f) for f in fems], kz)
    assert got == tile
    it = items.astype(np.int64)
    tx, ty, z0, nz, pr = it & 31, (it >> 5) & 127, (it >> 12) & 1023, ((it >> 22) & 63) + 1, it >> 28
    gx, gy = -(-n // tile[0]), -(-n // tile[1])
    assert gx <= 32 and gy <= 128 and tx.max() == gx - 1 and ty.max() == gy - 1
    assert pr.max() == len(fems) - 1 and nz.max() <= kz
    col = tx + gx * (ty + gy * pr)
    o = np.lexsort((z0, col))
    col, z0, end = col[o], z0[o], np.minimum(z0[o] + nz[o], n)
    first = np.r_[True, col[1:] != col[:-1]]
    assert np.array_equal(col[first], np.arange(gx * gy * len(fems)))      # every column
    assert (z0[first] == 0).all() and (end[np.r_[first[1:], True]] == n).all()
    assert (z0[1:][~first[1:]] == end[:-1][~first[1:]]).all()              # its planes join up


def test_argument_checks():
    for args in ((5, [(1, 3, 2, 0)], 8), (41, [(10, 50, 12, 4)], 8), (41, [cube_box(41, 11)], 65), (41, [], 8)):
        with pytest.raises(DDFDError):
            step_items64(*args)
