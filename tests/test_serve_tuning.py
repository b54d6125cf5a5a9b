"""What the serving loop's tuner pins a problem to: never to a kernel slower than the library's own choice, and a
shape per reconstruction."""
import pytest

from paper_1810_07802_gb300 import workloads as W


def test_reconstructions_of_one_size_are_tuned_apart():
    """An upwind problem takes tile shape 1 only: the shape of a central problem of its size is refused."""
    from paper_1810_07802_gb300.serve import AutotuneCache

    cache = AutotuneCache(tuner=lambda cfg, trial_steps: (1 if cfg.get("recon") == "upwind" else 3, [1.0]))
    central = dict(nx=64, ny=64, precision="fp32")
    assert [cache(dict(central, recon=r), {}) for r in ("central", "upwind", "central")] == [3, 1, 3]
    assert cache(central, {}) == 3 and len(cache.shapes) == 2


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,recon,bc_y", [(256, 256, "central", "periodic"), (4, 256, "central", "wall")])
def test_fp32_problems_keep_the_library_choice(nx, ny, recon, bc_y):
    """The FP32 strips step both faster than any tile: 11.3 us against 12.9 in a batch of one, 4 x 256 6 against 15."""
    from paper_1810_07802_gb300 import build
    from paper_1810_07802_gb300.serve import AutotuneCache

    build.build()
    cfg, f = W.random_state(nx, ny, seed=2, rho_ratio=10.0, bc_y=bc_y)
    assert AutotuneCache(trial_steps=20)(dict(cfg, precision="fp32", phi_ref=0.5, recon=recon), f) == 0


@pytest.mark.gpu
def test_a_server_tunes_upwind_and_central_requests_of_one_size():
    from paper_1810_07802_gb300 import build
    from paper_1810_07802_gb300.serve import AutotuneCache, BatchingServer, Request

    build.build()
    reqs = []
    for i, recon in enumerate(("central", "upwind", "central", "upwind")):
        cfg, f = W.random_state(40, 64, seed=i)
        reqs.append(Request(i, recon, dict(cfg, recon=recon), f, 4, 0.0))
    recs = BatchingServer(1 << 30, max_members=4, chunk=4, tile_policy=AutotuneCache(trial_steps=4)).run(reqs)
    assert len(recs) == 4 and all(r.error is None for r in recs)
