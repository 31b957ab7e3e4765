"""ddfd_misfit_noalloc with short tapers: z(t) = (1 + cos(pi (t - T + dl) / dl)) / 2 for
t > T - dl, dl = z_delta_frac T, is exactly 0 at t = T however short dl is.  Against
numpy FP64; the residual of the tapered rows is 1e3 times that of the others, so that
an error of z is seen in the sum.  Bar 1e-13 relative: every term is positive, and z
is 0 at the end or, over several tapered rows, rounded to 1e-16 of one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_det", [3, 400])       # a warp a row, a thread block a row
@pytest.mark.parametrize("tau", [1e-3, 0.3 / 160, 0.25 / 64])
@pytest.mark.parametrize("n_steps,frac", [(300, 1e-12), (300, 1e-15), (77, 1e-9), (1000, 1e-6), (400, 2.5e-3), (400, 0.0101)])
def test_short_tapers(n_steps, frac, tau, n_det):
    torch = pytest.importorskip("torch")
    from paper_2508_07780_gb300 import build, misfit_noalloc
    build.build()
    rng = np.random.default_rng(n_steps)
    tr = rng.standard_normal((1, n_steps + 1, n_det, 3))
    t, T, dl = np.arange(n_steps + 1) * tau, n_steps * tau, frac * (n_steps * tau)
    tr[:, t > T - dl] *= 1e3
    z = np.where(t <= T - dl, 1.0, 0.5 * (1 + np.cos(np.pi * (t - T + dl) / dl)))
    z[0] = 0.0
    assert z[-1] == (1.0 if T - dl == T else 0.0)
    want = 0.5 * tau * float(((tr ** 2).sum((0, 2, 3)) * z).sum())
    J = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    misfit_noalloc(torch.tensor(tr, device="cuda"), torch.zeros(tr.shape, dtype=torch.float64, device="cuda"), 1,
                   n_steps, n_det, tau, frac, J)
    assert abs(J.item() - want) <= 1e-13 * want
