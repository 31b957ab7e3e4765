"""The FP32 step kernel (csrc/ddfd_step.cu) where its quads, tiles and rings can
go wrong: grids of n mod 4 = 0..3 and n = 32 m + 1 (the x tail), FEM cubes at any
offset from the quads, across tiles and z ranges, absorbing faces on every side,
oblique incidence, item depths from two planes to more than the rings hold.

Against the oracle with the FP32 bars (relative L2 1e-4 on traces, fields, mu and J,
1e-3 on the gradient).  A handle with a memory budget keeps the history's rows
unpadded and evaluates the oblique pulse in the kernel: every bit must agree, as it
must between item depths."""
import numpy as np
import pytest

from helpers import capture_steps, rel_l2, run_gpu, run_oracle
from synth import workload

pytestmark = pytest.mark.gpu

# n, fem_n; the cube's first free node is at offset 3, 4, 3, 5, 4, 3, 3, 8, 10, 3, 13 + ... from x = 0
GRIDS = [(7, 5), (9, 5), (10, 8), (15, 9), (16, 12), (28, 26), (31, 29), (33, 21), (34, 18), (35, 33), (65, 9)]


@pytest.fixture(scope="module")
def reference():
    from paper_2508_07780_gb300 import build
    build.build()
    seen = {}

    def get(n, fem):
        if (n, fem) not in seen:
            w = workload("tiny", n=n, fem_n=fem, n_steps=2 * n + 20, seed=n, dir_seed=n, det_per_side=3,
                         extra={"det": [[0, 0], [n - 1, n - 1], [n - 1, 2], [n // 2, n // 2], [n // 2, n // 2], [3, n - 1]]})
            e, m = capture_steps(w.n_steps)
            seen[n, fem] = (w, e, m, run_oracle(w, keep_e=e, keep_mu=m, absorbing=63))
        return seen[n, fem]
    return get


@pytest.mark.parametrize("n,fem", GRIDS)
def test_fp32_step_at_tile_edges(reference, n, fem):
    w, e, m, ref = reference(n, fem)
    first = None
    for kw in (dict(), dict(mem_budget=1 << 36), dict(tile_kz=2, tile_kz_lean=2), dict(tile_kz=min(n, 5), tile_kz_lean=19)):
        out = run_gpu(w, ref["eobs"], precision="fp32", keep_e=e, keep_mu=m, absorbing_faces=63, **kw)
        if first is None:
            first = out
            assert rel_l2(out["trace"], ref["trace"]) <= 1e-4
            for k in e:
                assert rel_l2(out["E"][k], ref["E"][k]) <= 1e-4, k
            for k in m:
                assert rel_l2(out["mu"][k], ref["mu"][k]) <= 1e-4, k
            assert abs(out["J"] - ref["J"]) <= 1e-4 * abs(ref["J"])
            assert rel_l2(out["g_eps"], ref["g_eps"]) <= 1e-3 and rel_l2(out["g_sig"], ref["g_sig"]) <= 1e-3
        else:
            assert np.array_equal(out["trace"], first["trace"]) and out["J"] == first["J"], kw
            assert np.array_equal(out["g_eps"], first["g_eps"]) and np.array_equal(out["g_sig"], first["g_sig"]), kw
            assert all(np.array_equal(out["mu"][k], first["mu"][k]) for k in m), kw
