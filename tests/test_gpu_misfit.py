"""ddfd_misfit_noalloc at the edges of its row split (a warp a row up to 341
detectors, else a thread block; 256 or 1024 threads for the total): against the
plain sum in numpy FP64.  Bar: 1e-13 relative -- every term is positive, so the
summation order moves the result by a few ulps times log2 of the row length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_src,n_steps,n_det,frac", [(1, 1, 1, 0.0), (1, 7, 10, 0.3), (2, 33, 11, 0.1), (1, 300, 64, 0.1),
                                                      (1, 40, 341, 0.2), (3, 20, 342, 0.2), (1, 2047, 3, 0.1),
                                                      (2, 1023, 5, 0.1), (1, 2048, 3, 0.9), (5, 9, 1024, 0.0),
                                                      (8, 8191, 1, 0.1), (1, 5, 0, 0.1)])
def test_misfit_noalloc_row_split(n_src, n_steps, n_det, frac):
    torch = pytest.importorskip("torch")
    from paper_2508_07780_gb300 import build, misfit_noalloc
    build.build()
    rng = np.random.default_rng(n_det + n_steps)
    tr = rng.standard_normal((n_src, n_steps + 1, n_det, 3))
    eo = tr + 0.1 * rng.standard_normal(tr.shape)
    tau = 1e-3
    t, T, dl = np.arange(n_steps + 1) * tau, n_steps * tau, frac * n_steps * tau
    z = np.ones(n_steps + 1) if dl <= 0 else np.where(t <= T - dl, 1.0, 0.5 * (1 + np.cos(np.pi * (t - T + dl) / dl)))
    z[0] = 0.0
    want = 0.5 * tau * float((((tr - eo) ** 2).sum((2, 3)) * z).sum())
    J = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    a, b = (torch.tensor(v, device="cuda") for v in (tr, eo))
    for _ in range(2):
        misfit_noalloc(a, b, n_src, n_steps, n_det, tau, frac, J)
    assert abs(J.item() - want) <= 1e-13 * want
