"""A partitioned solve that is given a new state after it has run: the schemes
with a history start again, whatever was recorded of the steps before."""
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


def start(m, seed):
    rho, u, dev = mg.random_state(m.n_cell, seed=seed)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    e = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]], float)
    eu = u @ e.T
    return rho[:, None] * w * (1 + 3 * eu + 4.5 * eu ** 2 - 1.5 * (u ** 2).sum(1)[:, None]) + 0.01 * dev


@pytest.mark.parametrize("scheme", ["ab2", "euler"])
@pytest.mark.parametrize("prec,kernel", [("fp64", 1), ("fp64", 128), ("fp32", 1), ("fp32", 128)])
@pytest.mark.parametrize("n_parts,first", [(2, 120), (3, 121)])   # an even and an odd number of steps before the new state
def test_new_state_after_recorded_steps(fv, scheme, prec, kernel, n_parts, first):
    m = mg.cylinder_hybrid(n_rad=12, n_circ=48, first=0.02, growth=1.12, r_far=8.0, n_tri_rings=12, seed=4)
    h, p = fv.Mesh(m), fv.make_params(0.1, cfl=0.3, scheme=scheme, precision=prec, kernel=kernel, u0=(0.02, 0.0))
    one, dd = fv.Solver(h, p), fv.DDSolver(fv.Partition(h, n_parts), p)
    for seed, n in ((1, first), (2, 40), (3, 16), (4, 35)):
        f = start(m, seed)
        for s in (one, dd):
            s.set_f(f)
            s.step(n)
            s.step(17)
        assert np.array_equal(dd.get_f(), one.get_f())
    one.close()
    dd.close()
