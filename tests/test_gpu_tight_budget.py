"""Handles whose memory budget has no room for the layouts that are chosen for speed
(gather blocks of 64 rows, items of one or two planes): they are created in the form
that takes the least memory, and give the same bits.

BYTES: device bytes of handles with gather blocks of 128 rows and one table entry per
tile of 32 x 16 (FP64 32 x 8) nodes and 8 planes, the least that these sizes were ever
created in."""
import numpy as np
import pytest

from synth.mesh import refined_fem_mesh

pytestmark = pytest.mark.gpu

BYTES = {
    ("fp32", 13, 9, 40, "stencil"): 249504, ("fp32", 13, 9, 40, "ebe"): 498964, ("fp32", 13, 9, 40, "mesh"): 354860,
    ("fp32", 24, 12, 40, "ebe"): 1939000, ("fp32", 24, 12, 40, "mesh"): 1698620,
    ("fp32", 41, 21, 60, "stencil"): 8977076, ("fp32", 41, 21, 60, "ebe"): 14085376,
    ("fp64", 13, 9, 40, "stencil"): 470560, ("fp64", 13, 9, 40, "ebe"): 975260, ("fp64", 24, 12, 40, "mesh"): 3271608,
    ("fp64", 41, 21, 60, "stencil"): 17367280, ("fp64", 41, 21, 60, "ebe"): 27550508,
}


def config(prec, n, fem, steps, kind):
    c = dict(n=n, fem_n=fem, n_steps=steps, precision=prec, det_ij=[[1, 1], [2, 5]], t0=0.1, width=0.035, freq=10.0)
    if kind == "ebe":
        c["fem_kind"] = 1
    elif kind == "mesh":
        nf, f0 = fem - 4, (n - fem) // 2 + 2
        e = 1 + 5 * np.random.default_rng(1).random(nf ** 3)
        c["mesh"] = refined_fem_mesh(n, fem, e, 0 * e, beta_eps=0.9, beta_sig=0.0,
                                     region=(f0 + nf // 3, f0 + min(nf // 3 + 8, 2 * nf // 3)))
    return c


def solve(handle, members):
    g = np.random.default_rng(3)
    for m in members:
        m.set_coeffs(1 + 5 * g.random(m.n_free), g.random(m.n_free))
    tr = handle.forward()
    rows = list(tr) if isinstance(tr, list) else [tr]
    eobs = [0.5 * t + 1e-2 * g.standard_normal(t.shape) for t in rows]
    handle.adjoint(eobs if isinstance(tr, list) else eobs[0])
    return rows + [x for m in members for x in m.gradient()]


@pytest.mark.parametrize("key", list(BYTES), ids=lambda k: "-".join(map(str, k)))
def test_least_bytes_are_enough(key):
    from paper_2508_07780_gb300 import Problem, build
    build.build()
    c = config(*key)
    out = []
    for budget in (1 << 40, BYTES[key]):
        p = Problem(**c, mem_budget=budget)
        assert p.get_info().device_bytes <= budget
        out.append(solve(p, [p]))
        p.close()
    assert np.abs(out[0][0]).max() > 0
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_batch_members_under_a_tight_budget(prec):
    from paper_2508_07780_gb300 import Batch, build
    build.build()
    out, budget = [], 1 << 40
    for _ in range(2):
        b = Batch([dict(config(prec, 24, 12, 40, k), mem_budget=budget) for k in ("ebe", "ebe")])
        budget = b.members[0].get_info().device_bytes - 1
        out.append(solve(b, b.members))
        b.close()
    assert np.abs(out[0][0]).max() > 0
    for x, y in zip(*out):
        assert np.array_equal(x, y)
