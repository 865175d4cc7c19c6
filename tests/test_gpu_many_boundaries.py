"""Meshes whose cells have more boundary faces than neighbours (instances of a few
cells, a channel one cell wide): tiles with up to two ghost rows per thread of the
fused stage give the bits of the two-kernel stage."""
import numpy as np
import pytest

from paper_1812_00390_gb300 import meshgen as mg
from test_gpu_resident import start

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


MESHES = {"two_triangles": ([mg.two_triangles], 3001), "three_squared": ([lambda: mg.cavity(3, 1.0)], 500),
          "one_wide": ([lambda: mg.couette(2500, 1)], 1), "bricks": ([lambda: mg.bricks(4, 3)], 300),
          "uneven": ([mg.two_triangles, lambda: mg.cavity(40, 8.0), lambda: mg.couette(30, 1)], 3)}


@pytest.mark.parametrize("kernel", [128, 256, 512, 1024])
@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16", "fp64"])
@pytest.mark.parametrize("name", list(MESHES))
def test_fused_stage_equals_two_kernels(fv, name, prec, kernel):
    makes, times = MESHES[name]
    if prec == "fp64" and kernel == 1024:
        pytest.skip("does not fit in FP64")
    ms = [m() for m in makes]
    h = fv.Mesh.concat([fv.Mesh(m) for m in ms] * times)
    f0 = np.concatenate([start(m.n_cell, 70 + k) for k, m in enumerate(ms)] * times)
    out = []
    for k in (kernel, 1):
        s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme="rk2", precision=prec, u_max=0.1, kernel=k))
        s.set_f(f0)
        s.step(7)
        out.append(s.get_f())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(*out)


def test_tiles_are_not_cut_by_their_boundary_faces(fv):
    h = fv.Mesh.concat([fv.Mesh(mg.two_triangles())] * 3000)
    i = fv.plan_info(h, fv.make_params(0.1, precision="fp32", kernel=512))
    assert i["violations"] == 0 and i["mean_tile_cells"] > 480
