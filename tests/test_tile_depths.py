"""The tile depths that a batch reports are depths that a configuration takes: FP64
launches of small grids run one plane an item by default."""
import numpy as np
import pytest

CFG = dict(n=33, fem_n=17, n_steps=90, det_ij=[[3, 4], [32, 32], [16, 0]])


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_07780_gb300 import build
    build.build()


@pytest.mark.parametrize("prec,kw,ok", [("fp64", dict(tile_kz=1), True), ("fp64", dict(tile_kz_lean=1), True),
                                        ("fp64", dict(tile_kz=33), True), ("fp32", dict(tile_kz=2, tile_kz_lean=2), True),
                                        ("fp32", dict(tile_kz=1), False), ("fp32", dict(tile_kz_lean=1), False),
                                        ("fp64", dict(tile_kz=-1), False), ("fp64", dict(tile_kz=34), False),
                                        ("fp64", dict(tile_kz_lean=65), False)])
def test_accepted_depths(prec, kw, ok):
    from paper_2508_07780_gb300 import DDFDError, Problem
    try:
        Problem(**CFG, precision=prec, **kw).close()
        code = 0
    except DDFDError as e:
        code = e.code
    assert code in ((0, -4) if ok else (-1,))  # -4: accepted, but this machine has no GPU


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_reported_depths_are_accepted_and_change_no_bit(prec):
    from paper_2508_07780_gb300 import Batch
    out = []
    kw = {}
    for _ in range(2):
        b = Batch([dict(CFG, precision=prec, **kw)] * 2)
        i = b.get_info()
        kw = dict(tile_kz=i.tile_kz, tile_kz_lean=i.tile_kz_lean)
        for m in b.members:
            g = np.random.default_rng(1)
            m.set_coeffs(1 + g.random(m.n_free), g.random(m.n_free))
        tr = b.forward()
        b.adjoint([0.5 * t + 1e-3 for t in tr])
        out.append((tr[1], *b.members[1].gradient(), kw))
        b.close()
    assert out[0][3] == out[1][3]
    for x, y in zip(out[0][:3], out[1][:3]):
        assert np.abs(x).max() > 0 and np.array_equal(x, y)
