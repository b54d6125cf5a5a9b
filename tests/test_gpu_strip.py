"""The strip and rectangle step kernels (the default path of the central reconstruction) at the sizes where they
can go wrong: one column or row more or less than a strip (28 columns) or a chunk, grids narrower than a warp,
rows that are no multiple of 16 bytes, one-row chunks, walls in the first and last chunk.

FP64 against the oracle at the parity bar (1e-10).  FP32 against the tile kernels, which do the same operations in
the same order on the same state: after three steps of a rough state of order one, a few units in the last place of
the largest stored value (4e-7 of it, as for bands of one problem; FP64 1e-12, as between the batched and the
single-problem kernels)."""
import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(3, 3), (4, 200), (27, 5), (28, 9), (29, 8), (32, 33), (57, 12), (60, 4), (113, 70), (255, 31)]


@pytest.fixture(scope="module")
def S():
    from paper_1810_07802_gb300 import build, solver

    build.build()
    solver.lib()
    return solver


def problem(nx, ny, model, bc_y):
    cfg, f = W.random_state(nx, ny, seed=7 * nx + ny, rho_ratio=100.0, model=model, bc_y=bc_y)
    if model == "ac":
        cfg = dict(cfg, velocity_field="rotation", vel_u0=0.02, vel_length=float(nx))
    return cfg, f


def stepped(S, cfg, f, steps):
    with S.Solver(cfg, **f) as s:
        s.step(steps)
        s.sync()
        return np.concatenate([a.reshape(-1, s.ny, s.nx) for a in s.distributions()])


@pytest.mark.parametrize("bc_y", ["periodic", "wall"])
@pytest.mark.parametrize("model", ["coupled", "ac"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_small_grids(S, nx, ny, model, bc_y):
    from oracle.oracle import Oracle

    cfg, f = problem(nx, ny, model, bc_y)
    o = Oracle(cfg, **f)
    o.step(4)
    ref = np.concatenate([a.reshape(-1, ny, nx) for a in o.state()])
    assert np.abs(stepped(S, cfg, f, 4) - ref).max() <= 1e-10
    cfg32 = dict(cfg, precision="fp32", phi_ref=0.5)
    strip, tile = (stepped(S, dict(cfg32, tile_shape=k), f, 3) for k in (0, 1))
    assert np.abs(strip - tile).max() <= 4e-7 * np.abs(tile).max()


@pytest.mark.parametrize("bc_y", ["periodic", "wall"])
@pytest.mark.parametrize("model", ["coupled", "ac"])
@pytest.mark.parametrize("precision,nx,ny", [("fp64", 1003, 777), ("fp32", 1003, 777), ("fp32", 2049, 530)])
def test_large_grids_against_the_tile_kernels(S, precision, nx, ny, model, bc_y):
    cfg, f = problem(nx, ny, model, bc_y)
    cfg = dict(cfg, precision=precision, phi_ref=0.5)
    strip, tile = (stepped(S, dict(cfg, tile_shape=k), f, 3) for k in (0, 1))
    assert np.abs(strip - tile).max() <= (1e-12 if precision == "fp64" else 4e-7) * np.abs(tile).max()


@pytest.mark.parametrize("bc_y", ["periodic", "wall"])
@pytest.mark.parametrize("model", ["coupled", "ac"])
@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 200), (25, 6), (26, 9), (27, 8), (53, 12), (130, 70), (1003, 777)])
def test_upwind_strips_against_the_tile_kernels(S, nx, ny, model, bc_y):
    """The FP32 upwind strips (26 columns of their own, three-row halo) against the tile kernel's slopes."""
    cfg, f = problem(nx, ny, model, bc_y)
    cfg = dict(cfg, precision="fp32", phi_ref=0.5, recon="upwind")
    strip, tile = (stepped(S, dict(cfg, tile_shape=k), f, 3) for k in (0, 1))
    assert np.abs(strip - tile).max() <= 4e-7 * np.abs(tile).max()


@pytest.mark.parametrize("bc_y", ["periodic", "wall"])
@pytest.mark.parametrize("model", ["coupled", "ac"])
@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 200), (7, 5), (33, 17), (130, 70), (403, 277)])
def test_upwind_rectangles_against_the_tile_kernels(S, nx, ny, model, bc_y):
    """FP64 upwind: rectangles with two-cell record halos, cut by the domain's edge, beside walls, wrapped twice."""
    cfg, f = problem(nx, ny, model, bc_y)
    cfg = dict(cfg, recon="upwind")
    rect, tile = (stepped(S, dict(cfg, tile_shape=k), f, 3) for k in (0, 1))
    assert np.abs(rect - tile).max() <= 1e-12 * np.abs(tile).max()
