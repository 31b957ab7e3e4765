"""Handles on a device that is nearly full: FP32 history rows are padded to 16 bytes
where they fit, and a handle that fits only without the padding still has to be
created.  The device is filled with one buffer up to halfway between the bytes that
the handle needs unpadded (those of the same handle with a memory budget, which never
pads) and padded."""
import gc

import pytest

pytestmark = pytest.mark.gpu


def padded_row(n, fem):
    f0, nf = (n - fem) // 2 + 2, fem - 4
    return (f0 + nf - f0 // 4 * 4 + 3) // 4 * 4, nf


@pytest.mark.parametrize("batched", [False, True])
def test_a_handle_that_fits_only_unpadded_is_created(batched):
    torch = pytest.importorskip("torch")
    from paper_2508_07780_gb300 import Batch, Problem, build
    build.build()
    det = [[0, 0], [5, 7], [100, 60]]
    if batched:  # two members, whose snapshots (23 GB) come after the choice of the layout
        cfg = dict(n=200, fem_n=105, n_steps=60000, n_snapshots=60, precision="fp32", det_ij=det)
        levels, make = 1001, lambda **kw: Batch([dict(cfg, **kw)] * 2)
    else:        # fields of 22 GB
        cfg = dict(n=720, fem_n=25, n_steps=40000, precision="fp32", det_ij=det)
        levels, make = 40001, lambda **kw: Problem(**cfg, **kw)
    hp, nf = padded_row(cfg["n"], cfg["fem_n"])
    more = levels * 3 * (hp - nf) * nf * nf * 4 * (2 if batched else 1)
    assert more > 5e8
    h = make(mem_budget=1 << 40)
    need = h.get_info().device_bytes
    h.close()
    gc.collect()  # (what earlier tests left would be freed between the two calls)
    torch.cuda.empty_cache()
    fill = torch.cuda.mem_get_info()[0] - need - more // 2
    assert fill > 0
    hold = torch.empty(fill, dtype=torch.uint8, device="cuda")
    try:
        h = make()
        got = h.get_info().device_bytes
        h.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert got < need + more // 4
    # with the device free again the rows are padded
    h = make()
    assert h.get_info().device_bytes >= need + more
    h.close()
