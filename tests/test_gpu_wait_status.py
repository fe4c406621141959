"""GPU: a bounded wait that gives up shows in the plan's next status-reading call, once, and only in that plan's.
The wait is the fused kernels' own, with the plan's flag, on a barrier that nothing completes (1 ms budget).
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2406_06640_gb300 as pg  # noqa: E402

pytestmark = pytest.mark.gpu

OK, EINVAL, ETIMEOUT = 0, 1, 6
M = 32
POS = np.array([(0, 0), (4, 6), (9, 2)], np.int32)
PRM = dict(M=M, K=2, N=3, obj_h=M + 9, obj_w=M + 9, sigma1=1.0, sigma2=1.0, kernel_size=11)


def _inputs():
    dev = torch.device("cuda:0")
    I = torch.rand(3, M, M, device=dev) * 20 + 1
    return I, torch.ones(M + 9, M + 9, device=dev, dtype=torch.complex64), \
        torch.ones(2, M, M, device=dev, dtype=torch.complex64)


def _errors(plan):
    lib, e, n = pg.load(), ctypes.c_double(), ctypes.c_int32()
    buf = (ctypes.c_double * 4)()
    return {"error": lambda: lib.ptycho_error(plan._h, ctypes.byref(e)),
            "history": lambda: lib.ptycho_error_history(plan._h, buf, 4, ctypes.byref(n)),
            "batch": lambda: lib.ptycho_error_batch(plan._h, buf)}


@pytest.mark.parametrize("call", ["error", "history"])
@pytest.mark.parametrize("minibatch", [0, 2])
def test_single_plan(call, minibatch):
    from paper_2406_06640_gb300.engine import Reconstruction

    lib = pg.load()
    I, O, P = _inputs()
    rec = Reconstruction(dict(PRM, minibatch=minibatch), I, POS)
    other = Reconstruction(PRM, I, POS)
    rec.iterate(O, P, 1)
    other.iterate(O, P, 1)
    read, other_read = _errors(rec._plan)[call], _errors(other._plan)[call]
    assert read() == OK
    assert lib.ptycho_plan_wait_selftest(rec._plan._h, 0, 1_000_000, 1) == OK  # completed: no timeout
    assert read() == OK
    assert lib.ptycho_plan_wait_selftest(rec._plan._h, 0, 1_000_000, 0) == OK
    assert other_read() == OK
    assert read() == ETIMEOUT and "gave up" in lib.ptycho_last_error().decode()
    assert read() == OK
    rec.iterate(O, P, 1)
    assert read() == OK
    assert lib.ptycho_plan_wait_selftest(rec._plan._h, 1, 1_000_000, 0) == EINVAL
    rec.close()
    other.close()


def test_batch_plan():
    from paper_2406_06640_gb300.engine import ReconstructionBatch

    lib = pg.load()
    I, O, P = _inputs()
    batch = ReconstructionBatch([(PRM, I, POS), (dict(PRM, engine="dm"), I, POS)])
    batch.iterate([O, O.clone()], [P, P.clone()], 1)
    read = _errors(batch._plan)["batch"]
    for member in (0, 1):
        assert read() == OK
        assert lib.ptycho_plan_wait_selftest(batch._plan._h, member, 1_000_000, 0) == OK
        assert read() == ETIMEOUT
    assert read() == OK
    assert lib.ptycho_plan_wait_selftest(batch._plan._h, 2, 1_000_000, 0) == EINVAL
    batch.close()
