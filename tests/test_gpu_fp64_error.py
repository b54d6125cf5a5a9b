"""Round-off of the FP64 step kernels, against the oracle's own source compiled in extended precision (80 or 128 bits):
the rectangles are no further from it than the tile kernels.  (A 64-bit run cannot tell: its own round-off is of the
same size, and nearer to that of a kernel that sums in its order.)"""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu

REAL = ctypes.c_longdouble


@pytest.fixture(scope="module")
def extended(tmp_path_factory):
    """The oracle with every double, literals included, a long double."""
    from oracle import oracle

    d = tmp_path_factory.mktemp("extended")
    for name in ("dugks_oracle.c", "dugks_oracle.h"):
        with open(os.path.join(os.path.dirname(oracle.__file__), name)) as f:
            text = re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S)
        text = re.sub(r"(?<![\w.])(\d+\.\d*(?:[eE][-+]?\d+)?|\d+[eE][-+]?\d+)(?![\w.])", r"\1L", text)
        text = re.sub(r"\bdouble\b", "long double", text).replace("<math.h>", "<tgmath.h>")
        (d / name).write_text(text)
    so = str(d / "extended.so")
    subprocess.run(["gcc", "-std=gnu99", "-O2", "-fPIC", "-shared", "-o", so, str(d / "dugks_oracle.c"), "-lm"], check=True)
    lib = ctypes.CDLL(so)

    class Params(ctypes.Structure):
        _fields_ = [(n, REAL if t is ctypes.c_double else t) for n, t in oracle.OracleParams._fields_]

    ptr = ctypes.POINTER(REAL)
    lib.oracle_create.restype = ctypes.c_void_p
    lib.oracle_create.argtypes = [ctypes.POINTER(Params)] + [ptr] * 4
    lib.oracle_step.argtypes = [ctypes.c_void_p, ctypes.c_long]
    lib.oracle_get_state.argtypes = [ctypes.c_void_p] + [ptr] * 3
    lib.oracle_destroy.argtypes = [ctypes.c_void_p]

    def run(cfg, fields, steps):
        p, q = Params(), oracle.make_params(cfg)
        for n, _ in Params._fields_:
            setattr(p, n, getattr(q, n))
        keep = [np.ascontiguousarray(fields.get(k), dtype=np.longdouble) if fields.get(k) is not None else None
                for k in ("phi0", "ux0", "uy0", "p0")]
        h = lib.oracle_create(ctypes.byref(p), *[None if a is None else a.ctypes.data_as(ptr) for a in keep])
        assert h
        lib.oracle_step(h, steps)
        out = [np.zeros((n, cfg["ny"], cfg["nx"]), np.longdouble) for n in (9, 9, 2)]
        lib.oracle_get_state(h, *[a.ctypes.data_as(ptr) for a in out])
        lib.oracle_destroy(h)
        return np.concatenate(out)

    return run


@pytest.mark.parametrize("recon", ["central", "upwind"])
@pytest.mark.parametrize("bc_y", ["periodic", "wall"])
@pytest.mark.parametrize("model", ["coupled", "ac"])
def test_rectangles_round_no_worse_than_the_tiles(extended, model, bc_y, recon):
    from paper_1810_07802_gb300 import build, solver

    build.build()
    nx, ny, steps = 45, 38, 8
    cfg, f = W.random_state(nx, ny, seed=4, rho_ratio=100.0, model=model, bc_y=bc_y)
    cfg = dict(cfg, recon=recon)
    if model == "ac":
        cfg.update(velocity_field="rotation", vel_u0=0.02, vel_length=float(nx))
    exact = extended(cfg, f, steps)
    err = []
    for k in (0, 1):
        with solver.Solver(dict(cfg, tile_shape=k), **f) as s:
            s.step(steps)
            s.sync()
            got = np.concatenate([a.reshape(-1, ny, nx) for a in s.distributions()])
        err.append(float(np.sqrt(np.sum((got - exact) ** 2) / np.sum(exact ** 2))))
    print("\n%s %s %s: rectangles %.2e, tiles %.2e" % (model, bc_y, recon, *err), end="")
    assert err[0] <= err[1], err
