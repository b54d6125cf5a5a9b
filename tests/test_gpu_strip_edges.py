"""FP64 strips at the sizes where they can go wrong, alone and in batches: a last chunk of one or two rows (beside the
top wall too), a strip with a single column of its own, grids narrower than a warp, members of one group with
chunks of different heights, more members than a launch carries.

The kernel that steps a problem is asked for, so that a size that no longer reaches the strips fails.  FP64 against the
tile kernels at 1e-12 of the largest stored value after three steps of a rough state of order one (as between
the batched and the single-problem kernels), FP32 at 4e-7 of it."""
import ctypes

import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KINDS = [("coupled", "periodic"), ("ac", "periodic"), ("ac", "wall")]   # (coupled FP64 between walls has no strips)


@pytest.fixture(scope="module")
def S():
    from paper_1810_07802_gb300 import build, solver

    build.build()
    solver.lib()
    return solver


def problem(nx, ny, model, bc_y, precision="fp64"):
    cfg, f = W.random_state(nx, ny, seed=7 * nx + ny, rho_ratio=100.0, model=model, bc_y=bc_y)
    if model == "ac":
        cfg = dict(cfg, velocity_field="rotation", vel_u0=0.02, vel_length=float(max(nx, ny)))
    return dict(cfg, precision=precision, phi_ref=0.5), f


def kernel(S, s):
    """(0 tiles, 1 strips, 2 rectangles; rows of a strip's chunk or 0)."""
    rows = ctypes.c_int32(-1)
    return S.lib().dugks_step_kernel(s.h, ctypes.byref(rows)), rows.value


def state(s):
    s.sync()
    return np.concatenate([a.reshape(-1, s.ny, s.nx) for a in s.distributions()])


def tiles(S, cfg, f, steps):
    with S.Solver(dict(cfg, tile_shape=1), **f) as s:
        assert kernel(S, s) == (0, 0)
        s.step(steps)
        return state(s)


@pytest.mark.parametrize("model,bc_y", KINDS)
@pytest.mark.parametrize("nx,ny,last", [(27, 9137, 1), (27, 9274, 2), (28, 9137, 1), (28, 9274, 2), (56, 9137, 1),
                                        (84, 9411, 3), (1401, 507, 1), (1401, 508, 2)])
def test_fp64_strips(S, nx, ny, last, model, bc_y):
    cfg, f = problem(nx, ny, model, bc_y)
    with S.Solver(cfg, **f) as s:
        which, rows = kernel(S, s)
        assert which == 1 and ny % rows == last
        s.step(3)
        got = state(s)
    ref = tiles(S, cfg, f, 3)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


def stepped_together(S, problems, steps, strips):
    import torch

    st = torch.cuda.Stream()
    solvers = [S.Solver(c, stream=st, **f) for c, f in problems]
    assert all((kernel(S, s)[1] > 0) == strips for s in solvers)
    with S.Batch(stream=st) as b:
        for s in solvers:
            b.add(s)
        b.step(steps)
        b.sync()
    out = [state(s) for s in solvers]
    for s in solvers:
        s.close()
    return out


@pytest.mark.parametrize("model,bc_y", KINDS)
def test_fp64_strips_in_a_batch(S, model, bc_y):
    """Below 2,048 tiles, so that the batch's own kernel steps them; grids of one and of 18 strips, odd rows."""
    problems = [problem(nx, ny, model, bc_y) for nx, ny in ((496, 512), (32, 8171), (16, 16000), (3, 9737), (31, 7999))]
    for (cfg, f), got in zip(problems, stepped_together(S, problems, 3, True)):
        ref = tiles(S, cfg, f, 3)
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max(), (cfg["nx"], cfg["ny"])


def test_walled_coupled_fp64_members_take_the_tiles(S):
    problems = [problem(nx, ny, "coupled", "wall") for nx, ny in ((496, 512), (32, 8171), (33, 17))]
    for (cfg, f), got in zip(problems, stepped_together(S, problems, 3, False)):
        ref = tiles(S, cfg, f, 3)
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max(), (cfg["nx"], cfg["ny"])


@pytest.mark.parametrize("model,bc_y", [("coupled", "wall"), ("coupled", "periodic"), ("ac", "periodic")])
def test_more_members_than_one_launch_carries(S, model, bc_y):
    """70 and 130 FP32 members of one group: two and three launches a step, the last of them of few members."""
    for n in (70, 130):
        problems = [problem(29 + 3 * (i % 37), 11 + i, model, bc_y, "fp32") for i in range(n)]
        for (cfg, f), got in zip(problems, stepped_together(S, problems, 3, True)):
            ref = tiles(S, cfg, f, 3)
            assert np.abs(got - ref).max() <= 4e-7 * np.abs(ref).max(), (cfg["nx"], cfg["ny"])


@pytest.mark.parametrize("precision,model,bc_y", [("fp64",) + k for k in KINDS] + [("fp32", "coupled", "periodic"),
                                                                                   ("fp32", "coupled", "wall")])
def test_chunk_heights_of_a_group_change_no_bits(S, precision, model, bc_y):
    """The rows of a chunk are chosen for a whole group: a member alone has others, and the same bits."""
    problems = [problem(nx, ny, model, bc_y, precision) for nx, ny in ((496, 512), (32, 8171), (31, 7999))]
    together = stepped_together(S, problems, 5, True)
    for p, got in zip(problems, together):
        assert np.array_equal(got, stepped_together(S, [p], 5, True)[0]), (p[0]["nx"], p[0]["ny"])
