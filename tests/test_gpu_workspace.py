"""The binding's workspace is torch memory used on the solver's own stream."""
import pytest
import torch

from paper_1812_00390_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


@pytest.mark.parametrize("handle", [False, True])
def test_workspace_is_not_given_away_while_launches_use_it(fv, handle):
    side = torch.cuda.Stream()
    s = fv.Solver(fv.Mesh(mg.cavity(128, 20.0)), fv.make_params(5e-4, scheme="rk2", precision="fp64"),
                  stream=side.cuda_stream if handle else side)
    n, at = s.workspace_bytes, s._ws.data_ptr()
    s.step(2000)                     # tens of milliseconds
    s.close()
    del s
    other = torch.empty(n, dtype=torch.uint8, device="cuda")   # its memory is not touched
    assert not side.query()
    assert not at <= other.data_ptr() < at + n
    side.synchronize()
