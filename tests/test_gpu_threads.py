"""Small solvers stepped by a thread each on streams of their own, made and closed
while others step: what they know of one another does not show in their states."""
import threading

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


def test_threads_of_solvers(fv):
    h = fv.Mesh(mg.cavity(128, 20.0))
    p = fv.make_params(5e-4, scheme="rk2", precision="fp32")
    ref = fv.Solver(h, p)
    ref.step(960)
    want = ref.get_f()
    ref.close()
    got, errors = {}, []

    def work(k):
        try:
            for turn in range(3):
                s = fv.Solver(h, p)
                for n in (320, 1, 63, 576):
                    s.step(n)
                    if (k + turn) % 2:
                        s.sync()
                got[k, turn] = s.get_f()
                s.close()
        except Exception as e:   # noqa: BLE001 - handed to the main thread
            errors.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors and len(got) == 18
    assert all(np.array_equal(f, want) for f in got.values())
