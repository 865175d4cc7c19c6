"""The resident stage loop (many steps of a small solver in one launch,
params.kernel = 0) against the stage kernels, which advance one stage per
launch: the arithmetic is the same value by value, so FP32 and 16-bit states
are bitwise equal and FP64 agrees to rounding and with the oracle to 1e-12."""
import numpy as np
import pytest

from paper_1812_00390_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


# one tile of two cells; a few tiles; every boundary kind; polygons; one tile on
# (nearly) every SM; three and four tiles per SM (FP64 beyond the loop's sizes)
MESHES = {
    "two_cells": lambda: mg.two_triangles(),
    "two_cells_periodic": lambda: mg.two_triangles(periodic=True),
    "channel_1_wide": lambda: mg.couette(40, 1),
    "couette": lambda: mg.couette(),
    "symmetry": lambda: mg.channel(nx=30, ny=17, top_bottom="symmetry"),
    "pressure_outlet": lambda: mg.channel(nx=33, ny=15, top_bottom="symmetry", external=0),
    "bricks": lambda: mg.bricks(62, 41),
    "periodic": lambda: mg.periodic_tri(71, 53, lx=71.0, ly=53.0),
    "cavity": lambda: mg.cavity(127, 20.0),
    "cylinder": lambda: mg.cylinder_hybrid(n_rad=70, n_circ=171, n_tri_rings=90, seed=5),
    "periodic_73k": lambda: mg.periodic_tri(192, 190, lx=192.0, ly=190.0),
    "cavity_103k": lambda: mg.cavity(321, 20.0),
    "bricks_50k": lambda: mg.bricks(400, 240),
}


def start(n, seed):
    rho, u, dev = mg.random_state(n, seed=seed)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    e = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]], float)
    eu = u @ e.T
    return rho[:, None] * w * (1 + 3 * eu + 4.5 * eu ** 2 - 1.5 * (u ** 2).sum(1)[:, None]) + 0.01 * dev


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16", "fp64"])
@pytest.mark.parametrize("scheme", ["rk2", "euler", "ab2", "rk4"])
@pytest.mark.parametrize("name", list(MESHES))
def test_resident_loop_equals_stage_kernels(fv, name, scheme, prec):
    m = MESHES[name]()
    f0 = start(m.n_cell, 41)
    h = fv.Mesh(m)
    out = []
    for kernel in (0, 128):
        s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme=scheme, precision=prec, u_max=0.1, kernel=kernel))
        s.set_f(f0)
        for n in (1, 2, 7, 40):      # odd and even numbers of stages, one launch after another
            s.step(n)
        a = s.get_f()
        s.set_f(a)                   # a new start: AB2 begins again
        s.step(3)
        out.append((a, s.get_f()))
        s.close()
    for x, y in zip(*out):
        assert np.isfinite(x).all()
        if prec == "fp64":
            assert np.abs(x - y).max() <= 1e-14 * np.abs(y).max()
        else:
            assert np.array_equal(x, y)


@pytest.mark.parametrize("name,scheme", [("couette", "euler"), ("bricks", "rk4"), ("cavity", "rk2"), ("symmetry", "ab2")])
def test_resident_loop_matches_oracle(fv, orc, name, scheme):
    m = MESHES[name]()
    o = orc.Oracle(m)
    dt = o.cfl_dt(0.3, 0.1, 0.1, scheme)
    f0 = start(m.n_cell, 43)
    s = fv.Solver(fv.Mesh(m), fv.make_params(0.1, dt=dt, scheme=scheme, precision="fp64"))
    s.set_f(f0)
    s.step(25)
    o.set_f(f0)
    o.run(scheme, 0.1, dt, 25)
    ref = o.get_f()
    assert np.abs(s.get_f() - ref).max() <= 1e-12 * np.abs(ref).max()
    s.close()


@pytest.mark.parametrize("prec", ["fp32", "fp16", "fp64"])
def test_resident_loop_many_stages_and_instances(fv, prec):
    """More stages than one launch advances, on instances of their own tau
    whose tiles straddle instance boundaries."""
    hs = [fv.Mesh(mg.couette(8, 3)), fv.Mesh(mg.two_triangles()), fv.Mesh(mg.cavity(21, 3.0)), fv.Mesh(mg.bricks(6, 4))]
    mesh, out = fv.Mesh.concat(hs), []
    for kernel in (0, 128):
        s = fv.Solver(mesh, [fv.make_params(t, scheme="rk2", precision=prec, kernel=kernel) for t in (0.24, 0.2, 0.05, 0.1)])
        s.step(1500)
        out.append(s.get_f())
        s.close()
    assert np.abs(out[0] - out[1]).max() <= (1e-13 if prec == "fp64" else 0.0)
