"""The read-out of FP32 states: stored values are widened to FP64 by integer operations, which zeros of both signs
and denormals take another way through than normal values.  Sums of nine values of 24 bits within 20 binary orders
of one another (and of denormals among themselves) are exact in FP64, so phi has to be equal bit for bit."""
import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["normal", "denormal", "zero"])
def test_widened_values_are_exact(kind):
    import torch
    from paper_1810_07802_gb300 import build, solver

    build.build()
    nx, ny = 37, 11
    cfg, f = W.random_state(nx, ny, seed=5, rho_ratio=10.0, model="coupled", bc_y="periodic")
    rng = np.random.default_rng(3)
    bits = {"normal": rng.integers(107 << 23, 127 << 23, (9, ny, nx)),
            "denormal": rng.integers(1, 1 << 23, (9, ny, nx)),
            "zero": np.zeros((9, ny, nx), np.int64)}[kind]
    v = (bits | rng.integers(0, 2, (9, ny, nx)) << 31).astype(np.uint32).view(np.float32)
    with solver.Solver(dict(cfg, precision="fp32", phi_ref=0.0), **f) as s:
        buf = s.row_buffer(ny)
        s.get_rows(0, ny, buf)
        s.sync()
        buf[:9] = torch.from_numpy(v).to(buf.device)
        torch.cuda.synchronize()
        s.set_rows(0, ny, buf)
        s.sync()
        phi = s.macros()["phi"].reshape(ny, nx)
    assert np.array_equal(phi, v.astype(np.float64).sum(axis=0))
