"""The FP32 strips repeat the tile kernels' operations in their order: every bit of the state is equal, step after
step, in every model, boundary, reconstruction and closure."""
import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_1810_07802_gb300 import build, solver

    build.build()
    solver.lib()
    return solver


@pytest.mark.parametrize("recon", ["central", "upwind"])
@pytest.mark.parametrize("bc_y", ["periodic", "wall"])
@pytest.mark.parametrize("kind", ["reciprocal", "linear", "rotation", "sampled"])
@pytest.mark.parametrize("nx,ny", [(3, 3), (29, 8), (113, 70), (509, 387)])
def test_strips_give_the_bits_of_the_tiles(S, nx, ny, kind, bc_y, recon):
    model = "coupled" if kind in ("reciprocal", "linear") else "ac"
    cfg, f = W.random_state(nx, ny, seed=7 * nx + ny, rho_ratio=100.0, model=model, bc_y=bc_y)
    cfg = dict(cfg, precision="fp32", phi_ref=0.5, recon=recon)
    r = np.random.default_rng(nx + ny)
    if kind == "linear":
        cfg = dict(cfg, visc="linear", gravity_mode=1, gx=1e-5, gy=-2e-5, rho_ref=30.0)
    elif kind == "rotation":
        cfg = dict(cfg, velocity_field="rotation", vel_u0=0.02, vel_length=float(max(nx, ny)))
    elif kind == "sampled":
        cfg = dict(cfg, velocity_field="sampled")
        f = dict(f, ux0=None, uy0=None)
    with S.Solver(dict(cfg, tile_shape=0), **f) as strip, S.Solver(dict(cfg, tile_shape=1), **f) as tile:
        if kind == "sampled":   # cells and faces
            v = 0.02 * r.standard_normal((4, ny, nx))
            for s in (strip, tile):
                s.set_velocity_field(*v)
        for n in range(1, 5):
            strip.step(1)
            tile.step(1)
            a, b = strip.get_state(), tile.get_state()
            assert np.array_equal(a, b), "step %d: %d values differ" % (n, (a != b).sum())
