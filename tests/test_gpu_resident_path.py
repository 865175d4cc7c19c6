"""Which path fvlbm_step takes on a small mesh: the resident loop is the one that
runs where it is meant to (its comparison with the stage kernels would say nothing
otherwise), and in FP64, too, the path cannot be seen in the state."""
import numpy as np
import pytest
import torch

from paper_1812_00390_gb300 import meshgen as mg
from test_gpu_resident import MESHES, start

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


# tiles per SM of each mesh on 152 SMs: FP32 and 16-bit, FP64 (0: beyond the loop's size;
# 103,000 quads are in more tiles than fit, the stage kernels run them)
PER_SM = {"two_cells": (1, 1), "two_cells_periodic": (1, 1), "channel_1_wide": (1, 1), "couette": (1, 1),
          "symmetry": (1, 1), "pressure_outlet": (1, 1), "bricks": (1, 1), "periodic": (1, 0), "cavity": (1, 0),
          "cylinder": (2, 0), "periodic_73k": (3, 0), "cavity_103k": (0, 0), "bricks_50k": (2, 0)}


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16", "fp64"])
@pytest.mark.parametrize("name", list(MESHES))
def test_small_meshes_run_the_resident_loop(fv, name, prec):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("the table is for 152 SMs")
    h, per_sm = fv.Mesh(MESHES[name]()), PER_SM[name][prec == "fp64"]
    s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme="euler", precision=prec, u_max=0.1))
    got = s.resident_info()
    assert (got["tile"] > 0) == (per_sm > 0) and -(-got["tiles"] // sms) == per_sm
    s.step(1)                        # a single stage runs by itself
    assert s.resident_info()["launches"] == 0
    s.step(2100)                     # 2048 stages and the rest
    assert s.resident_info()["launches"] == (2 if per_sm else 0)
    torch.cuda.synchronize()         # (in 16 bits the stretched cavity diverges at this tau, on every path)
    s.close()
    s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme="euler", precision=prec, u_max=0.1, kernel=128))
    s.step(3)
    assert s.resident_info() == {"tile": 0, "tiles": 0, "launches": 0}
    s.close()


# the largest of the loop's range: four tiles per SM (two of polygons)
LARGEST = {"quads_96k": lambda: mg.cavity(310, 20.0), "triangles_110k": lambda: mg.periodic_tri(235, 235, lx=235.0, ly=235.0),
           "polygons_53k": lambda: mg.bricks(460, 230)}


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name,scheme", [("quads_96k", "rk2"), ("quads_96k", "ab2"), ("triangles_110k", "rk4"),
                                         ("polygons_53k", "rk2")])
def test_largest_resident_meshes_equal_stage_kernels(fv, name, scheme, prec):
    m = LARGEST[name]()
    h, f0, out = fv.Mesh(m), start(m.n_cell, 49), []
    for kernel in (0, 128):
        s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme=scheme, precision=prec, u_max=0.1, kernel=kernel))
        s.set_f(f0)
        for n in (2, 21):
            s.step(n)
        assert s.resident_info()["launches"] == (0 if kernel else 2)
        out.append(s.get_f())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(*out)


FP64_MESHES = dict({k: MESHES[k] for k in ("two_cells", "two_cells_periodic", "channel_1_wide", "couette", "symmetry",
                                           "pressure_outlet", "bricks", "periodic")},
                   cavity_5k=lambda: mg.cavity(75, 20.0),
                   hybrid=lambda: mg.cylinder_hybrid(n_rad=12, n_circ=48, first=0.02, growth=1.12, r_far=8.0,
                                                     n_tri_rings=12, seed=4))


@pytest.mark.parametrize("scheme", ["euler", "ab2", "rk2", "rk4"])
@pytest.mark.parametrize("name", list(FP64_MESHES))
def test_fp64_state_is_the_same_bits_on_every_path(fv, name, scheme):
    m = FP64_MESHES[name]()
    h, f0, out = fv.Mesh(m), start(m.n_cell, 47), {}
    # whole calls and single steps with the automatic choice, the two-kernel stage, fused tiles
    for kernel, calls in ((0, [50]), (0, [1] * 50), (1, [50]), (128, [49, 1]), (256, [50])):
        s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme=scheme, precision="fp64", u_max=0.1, kernel=kernel))
        s.set_f(f0)
        for n in calls:
            s.step(n)
        out[kernel, len(calls)] = s.get_f()
        s.close()
    first = out[0, 1]
    assert np.isfinite(first).all()
    for x in out.values():
        assert np.array_equal(x, first)


def test_fp64_two_kernel_stage_is_the_same_bits_as_fused_tiles_on_a_large_mesh(fv):
    """A thread per cell in both (beyond the sizes that take four lanes per cell)."""
    m = mg.cavity(600, 20.0)
    h, f0, out = fv.Mesh(m), start(m.n_cell, 48), []
    for kernel in (1, 256):
        s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme="rk2", precision="fp64", u_max=0.1, kernel=kernel))
        s.set_f(f0)
        s.step(3)
        out.append(s.get_f())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(*out)


@pytest.mark.parametrize("name,make", [("quads", lambda m: mg.cavity(m, 20.0)), ("polygons", lambda m: mg.bricks(2 * m, m))])
def test_fp64_state_is_the_same_bits_on_both_sides_of_the_lanes_limit(fv, name, make):
    """Four lanes per cell below 1300 cells per SM (750 of polygons), a boundary face counting
    as eight cells less, a thread per cell from there."""
    for side in ((460, 462) if name == "quads" else (362, 366)):
        m = make(side)
        h, f0, out = fv.Mesh(m), start(m.n_cell, 59), []
        for kernel in (1, 256):
            s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme="rk2", precision="fp64", u_max=0.1, kernel=kernel))
            s.set_f(f0)
            s.step(3)
            out.append(s.get_f())
            s.close()
        assert np.isfinite(out[0]).all() and np.array_equal(*out)
