"""The rows of a refined mesh that run as Kuhn block stencils against gathering them
element by element, which the same cube as an element handle does for all of its rows.
Four fifths of the rows are stencil rows here.  In FP64 they are bound by the SMs' FP64
units: spread over all thread blocks the mesh's gather takes 0.60 of the element
handle's, on the first 46 of 302 thread blocks 0.78 (forward; adjoint 0.58, 0.74); the
bar lies between.  FP32 is bound by latency (0.80, 0.67)."""
import numpy as np
import pytest

from synth.mesh import refined_fem_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("fp64", 0.68), ("fp32", 0.9)])
def test_stencil_rows_cost_less_than_gathered_ones(prec, bar):
    from paper_2508_07780_gb300 import Problem, build
    build.build()
    n, fem = 61, 31
    nf, f0 = fem - 4, (n - fem) // 2 + 2
    e = 1 + 5 * np.random.default_rng(1).random(nf ** 3)
    mesh = refined_fem_mesh(n, fem, e, 0 * e, beta_eps=0.9, beta_sig=0.0, region=(f0 + nf // 3, f0 + nf // 3 + 8))
    ms = {}
    for kind, kw in (("mesh", dict(mesh=mesh)), ("ebe", dict(fem_kind=1))):
        p = Problem(n=n, fem_n=fem, n_steps=4, precision=prec, det_ij=[[0, 0]], **kw)
        p.set_coeffs(np.full(p.n_free, 3.0), np.full(p.n_free, 0.1))
        p.forward()
        p.time_gather(reps=20)
        ms[kind] = np.min([p.time_gather(reps=50)[:2] for _ in range(5)], axis=0)
        p.close()
    print(prec, ms)
    assert (ms["mesh"] <= bar * ms["ebe"]).all()
