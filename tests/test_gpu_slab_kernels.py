"""y-bands whose size takes another FP64 step kernel than the whole domain's: the two order their sums differently, so
a band's own rows equal the single-domain step to round-off.  1e-12 of the largest stored value after three steps
of a rough state of order one, as between the kernels themselves (test_gpu_strip_edges); a stale halo row moves such
a state by about 1e-2."""
import ctypes

import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_bands_of_rectangles_equal_a_domain_of_strips():
    from paper_1810_07802_gb300 import build, slab, solver

    build.build()
    which = solver.lib().dugks_step_kernel
    cfg, f = W.random_state(1024, 1024, seed=31, rho_ratio=100.0)
    with solver.Solver(cfg, **f) as whole:
        assert which(whole.h, ctypes.POINTER(ctypes.c_int32)()) == 1
        whole.step(3)
        ref = whole.distributions()
    bands = []
    for r0, r1 in slab.bands(cfg["ny"], 8):
        bcfg, bfields = slab.band_problem(cfg, f, r0, r1)
        bands.append(slab.Band(solver.Solver(bcfg, **bfields), r0, r1, cfg))
        assert which(bands[-1].stepper.h, ctypes.POINTER(ctypes.c_int32)()) == 2
    slab.step_bands(slab.LocalExchange(bands), bands, 3)
    for b in bands:
        for got, r in zip(b.stepper.distributions(), ref):
            assert np.abs(got[:, b.own] - r[:, b.r0:b.r1]).max() <= 1e-12 * np.abs(r).max()
        b.stepper.close()
