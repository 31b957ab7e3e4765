"""Reads of a kernel that is launched as the programmatic dependent of the kernel
before it: it may start while that one still writes, so that the non-coherent load
path (__ldg, ld.global.nc, const __restrict__ parameters), specified for data that
nothing writes during the kernel's life, is not for the fields, the history or the
gather's rows.  The first adjoint step after a replayed checkpoint segment reads the
history level that the kernel before it writes."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_07780_gb300", "csrc")


@pytest.mark.parametrize("name", ["ddfd_step.cu", "ddfd_step64.cu", "ddfd_step_common.h", "ddfd_ebe.cu"])
def test_chained_kernels_have_no_non_coherent_loads(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    assert not re.findall(r"__ldg|\.nc\b|__restrict__", src)


@pytest.mark.gpu
@pytest.mark.parametrize("prec,kw", [("fp64", {}), ("fp32", {}), ("fp32", dict(mem_budget=1 << 36))])
@pytest.mark.parametrize("nsnap", [25, 50])
def test_short_segments_are_bitwise_the_full_history(prec, kw, nsnap):
    """50 steps in segments of two steps and of one: every adjoint step, or every
    second one, follows a replay.  A memory budget keeps the FP32 history unpadded,
    which is read by other loads."""
    from paper_2508_07780_gb300 import build
    from helpers import run_gpu
    from synth import workload
    build.build()
    w = workload("tiny", n=34, fem_n=31, n_steps=50, seed=5, dir_seed=5)
    eobs = 1e-3 * np.random.default_rng(2).standard_normal((1, 51, w.detectors().shape[0], 3))
    full = run_gpu(w, eobs, precision=prec, **kw)
    for _ in range(3):
        ck = run_gpu(w, eobs, precision=prec, n_snapshots=nsnap, **kw)
        assert np.abs(ck["g_eps"]).max() > 0
        for key in ("trace", "g_eps", "g_sig"):
            assert np.array_equal(full[key], ck[key]), key
