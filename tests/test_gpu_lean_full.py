"""FP32: a tile's nodes come out the same from the lean loop (items without FEM-cube or free
nodes) and from the full one.  Which loop runs a tile is decided by the FEM cube alone; in
vacuum the FEM rows equal the finite-difference ones to the bit (s = 0, damping 0: products
with 0 and 1), so that runs with a cube that fills the grid, where every tile below the
last ragged row runs the full loop, and with a cube of five nodes, where all but the middle
ones run the lean loop, must agree on every node: at the side faces, mirrored or absorbing,
the top face with its source and its detectors' residuals, edges and corners, and the x
tail of n = 32 m + 1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STEPS, KEEP = 70, [1, 20, 45, 70]


def solve(n, fems, faces, direction, **kw):
    from paper_2508_07780_gb300 import Batch, Problem
    det = [[0, 0], [n - 1, n - 1], [n - 1, 3], [5, n - 1], [n // 2, n // 2], [n // 2, n // 2], [31, 16], [0, 40]]
    cfg = [dict(n=n, fem_n=f, n_steps=STEPS, precision="fp32", det_ij=det, src_dir=[direction], absorbing_faces=faces,
                t0=0.1, width=0.05, freq=5.0, t1=0.3, **kw) for f in fems]
    h = Problem(**cfg[0]) if len(cfg) == 1 else Batch(cfg)
    members = [h] if len(cfg) == 1 else h.members
    for m in members:
        m.set_coeffs(np.ones(m.n_free), np.zeros(m.n_free))
        if len(cfg) == 1:
            m.set_capture(KEEP)
    tr = h.forward()
    tr = [tr] if len(cfg) == 1 else tr
    eobs = np.random.default_rng(7).standard_normal((1, STEPS + 1, len(det), 3))
    h.adjoint(eobs if len(cfg) == 1 else [eobs] * len(cfg))
    out = [np.stack(tr)]
    if len(cfg) == 1:
        out += [h.get_capture(0, i) for i in range(len(KEEP))] + [h.get_capture(1, i) for i in range(len(KEEP) - 1)]
    h.close()
    return out


@pytest.mark.parametrize("n", [47, 63, 65])
@pytest.mark.parametrize("faces", [0, 3, 63])
@pytest.mark.parametrize("direction", [[0.0, 0.0, -1.0], [0.3, -0.2, -0.9]])
def test_lean_and_full_loops_agree(n, faces, direction):
    from paper_2508_07780_gb300 import build
    build.build()
    lean = solve(n, [5], faces, direction)
    for kw in (dict(), dict(tile_kz=n), dict(mem_budget=1 << 36)):
        full = solve(n, [n - 2], faces, direction, **kw)
        for i, (x, y) in enumerate(zip(lean, full)):
            assert np.abs(x).max() > 0 and np.isfinite(x).all()
            assert np.array_equal(x, y), (kw, i)


def test_lean_and_full_loops_agree_in_a_batch():
    from paper_2508_07780_gb300 import build
    build.build()
    (tr,) = solve(65, [5, 63, 33], 63, [0.3, -0.2, -0.9])
    assert np.abs(tr[0]).max() > 0
    assert np.array_equal(tr[0], tr[1]) and np.array_equal(tr[0], tr[2])
