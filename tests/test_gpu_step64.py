"""The FP64 step kernels (csrc/ddfd_step64.cu) where their tiling can go wrong,
against the oracle: one to three tiles and a ragged rest per axis, FEM cubes
that fill the grid or lie across the edges of tiles and of z ranges, every z
depth from one plane up, and depths of several planes that start or end
inside the cube.

Bar: relative L2 1e-12 on traces, fields, mu, J and the gradient, the bar of the FP64
path (a few hundred steps of a scheme whose rounding is 1e-16 a step)."""
import numpy as np
import pytest

from helpers import capture_steps, rel_l2, run_gpu, run_oracle
from synth import workload

pytestmark = pytest.mark.gpu

# n, fem_n (n - 2: the cube's rows start two nodes from the boundary)
GRIDS = [(7, 5), (9, 7), (10, 7), (15, 13), (16, 14), (17, 15), (19, 8), (28, 26), (29, 17), (33, 31), (34, 13)]


@pytest.fixture(scope="module")
def reference():
    from paper_2508_07780_gb300 import build
    build.build()
    seen = {}

    def get(n, fem):
        if (n, fem) not in seen:
            w = workload("tiny", n=n, fem_n=fem, n_steps=3 * n // 2 + 20, seed=n, dir_seed=n, det_per_side=3)
            e, m = capture_steps(w.n_steps)
            seen[n, fem] = (w, e, m, run_oracle(w, keep_e=e, keep_mu=m, absorbing=1 | 2 | 8 | 16))
        return seen[n, fem]
    return get


@pytest.mark.parametrize("n,fem", GRIDS)
def test_fp64_step_at_tile_edges(reference, n, fem):
    w, e, m, ref = reference(n, fem)
    first = None
    for kz in (0, 2, 3, n - 1):
        out = run_gpu(w, ref["eobs"], precision="fp64", keep_e=e, keep_mu=m, absorbing_faces=1 | 2 | 8 | 16, tile_kz=kz)
        assert rel_l2(out["trace"], ref["trace"]) <= 1e-12
        for k in e:
            assert rel_l2(out["E"][k], ref["E"][k]) <= 1e-12, (kz, k)
        for k in m:
            assert rel_l2(out["mu"][k], ref["mu"][k]) <= 1e-12, (kz, k)
        assert abs(out["J"] - ref["J"]) <= 1e-12 * abs(ref["J"])
        assert rel_l2(out["g_eps"], ref["g_eps"]) <= 1e-12 and rel_l2(out["g_sig"], ref["g_sig"]) <= 1e-12
        if first is not None:  # the depth changes no bit
            assert np.array_equal(out["trace"], first["trace"]) and np.array_equal(out["g_eps"], first["g_eps"])
        first = first or out


def test_fp64_tiles_of_small_and_large_launches_agree(reference):
    """The tile shape goes by the nodes of a launch: one problem of 33^3 nodes runs on
    8 x 8 tiles (checked against the oracle above), twelve together on 14 x 9; the
    arithmetic per node is the same, so every bit is."""
    from paper_2508_07780_gb300 import Batch
    rng = np.random.default_rng(3)
    ws = [workload("tiny", n=33, fem_n=f, n_steps=60, seed=f, dir_seed=f, det_per_side=3) for f in (31, 20, 9)] * 4
    kw = [dict(n=33, fem_n=w.fem_n, n_steps=60, precision="fp64", src_dir=w.directions(), det_ij=w.detectors(),
               absorbing_faces=1 | 2 | 4) for w in ws]
    b = Batch(kw)
    for m, w in zip(b.members, ws):
        m.set_coeffs(*w.model())
    traces = b.forward()
    eobs = [t + 1e-3 * rng.standard_normal(t.shape) for t in traces]
    b.adjoint(eobs)
    for i in (0, 1, 2, 11):
        w = ws[i]
        alone = run_gpu(w, eobs[i], precision="fp64", absorbing_faces=1 | 2 | 4)
        ge, gs = b.members[i].gradient()
        assert np.abs(ge).max() > 0
        assert np.array_equal(alone["trace"], traces[i])
        assert np.array_equal(alone["g_eps"], ge) and np.array_equal(alone["g_sig"], gs)
    b.close()


def test_fp64_tiles_of_large_grids_against_fp32():
    """Grids beyond 448 nodes run on 32 x 8 tiles.  Ten steps of a 450^3 grid whose FEM
    rows reach to two nodes below the top face, against the FP32 kernel, whose rows are
    written as block stencils: 1e-5 covers its rounding (1e-7 a step) several times over."""
    from paper_2508_07780_gb300 import Problem, build
    build.build()
    n, fem, nt = 450, 448, 10
    nf = fem - 4
    z = np.arange(nf)
    eps = np.broadcast_to((4.0 + 3.0 * ((z // 5) % 3))[:, None, None] + ((z // 7) % 2)[None, None, :], (nf, nf, nf)).ravel()
    sig = np.broadcast_to((0.1 * ((z // 3) % 4))[None, :, None], (nf, nf, nf)).ravel()
    det = [[0, 0], [449, 449], [31, 8], [32, 7], [447, 225], [448, 16]]
    out = {}
    for prec in ("fp64", "fp32"):
        p = Problem(n=n, fem_n=fem, n_steps=nt, precision=prec, det_ij=det, freq=2.0, t0=0.05, width=0.5,
                    src_dir=[[0.3, -0.2, -0.9]])
        p.set_coeffs(eps, sig)
        tr = p.forward()
        p.adjoint(0.5 * tr + 1e-3)
        out[prec] = (tr, *p.gradient())
        p.close()
    for a, b in zip(out["fp64"], out["fp32"]):
        assert np.abs(a).max() > 0 and rel_l2(b, a) <= 1e-5
