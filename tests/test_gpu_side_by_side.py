"""Small solvers stepped side by side on streams of their own: where their resident
launches would have to take turns they run overlapping stage kernels instead, and
return to the resident loop when they are alone again."""
import numpy as np
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


def launches(solvers):
    return [s.resident_info()["launches"] for s in solvers]


@pytest.mark.parametrize("n_solvers,make,prec,shared", [
    (4, lambda: mg.cavity(128, 20.0), "fp32", False),      # each fills the GPU
    (6, lambda: mg.cavity(64, 20.0), "fp64", False),
    (8, lambda: mg.couette(64, 16), "fp32", True),         # all fit on it at once
])
def test_rounds_of_solvers(fv, n_solvers, make, prec, shared):
    """From rest, the plate or lid moving."""
    n, h = 1500, fv.Mesh(make())
    p = fv.make_params(5e-4 if not shared else 0.24, scheme="rk2", precision=prec)
    ss = [fv.Solver(h, p) for _ in range(n_solvers)]
    seen, rounds = [], 10                                  # (the graphs of stage kernels have to pay first)
    for _ in range(rounds):
        for s in ss:
            s.step(n)
        for s in ss:
            s.sync()
        seen.append(launches(ss))
    assert all(x > 0 for x in seen[0])                     # in turns to begin with
    if shared:
        assert all(b > a for a, b in zip(seen[-2], seen[-1]))
    else:
        assert seen[-1] == seen[-2]                        # stage kernels in the end
    ss[0].step(n)                                          # was joined in its last call
    ss[0].sync()
    before = launches(ss[:1])
    ss[0].step(n)                                          # nobody else since
    assert launches(ss[:1]) > before
    ref = fv.Solver(h, p)
    for _ in range(rounds):
        ref.step(n)
        ref.sync()                                         # alone: in the resident loop throughout
    out = ref.get_f()
    assert np.isfinite(out).all()
    for s in ss[1:]:
        assert np.array_equal(s.get_f(), out)
    for s in ss:
        s.close()


def test_short_calls_and_one_stream_stay_in_the_loop(fv):
    h = fv.Mesh(mg.cavity(128, 20.0))
    p = fv.make_params(5e-4, scheme="rk2", precision="fp32")
    one = torch.cuda.Stream()
    for streams, n in ((None, 31), (one, 500)):
        ss = [fv.Solver(h, p, stream=streams) for _ in range(4)]
        for _ in range(3):
            for s in ss:
                s.step(n)
        assert launches(ss) == [3] * 4
        for s in ss:
            s.sync()
            s.close()
