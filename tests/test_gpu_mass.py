"""fvlbm_mass_noalloc is the reduction of fvlbm_mass on another scratch: the same bits."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
def test_noalloc_mass_is_the_same_bits(fv, prec):
    # one chunk of 4096 cells; several and a remainder; a chunk of two cells
    ms = [mg.cavity(64, 5.0), mg.cavity(233, 20.0), mg.two_triangles(), mg.couette(64, 16)]
    h = fv.Mesh.concat([fv.Mesh(m) for m in ms])
    s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme="euler", precision=prec, u_max=0.1))
    s.set_f(np.concatenate([start(m.n_cell, 60 + k) for k, m in enumerate(ms)]))
    for n in (0, 3):
        s.step(n)
        assert np.array_equal(s.mass_noalloc(), s.mass())
    s.close()
