"""GPU: many plans alive at a time, made and closed in any order and from several threads. Each reads its own error
(the plans' host words share blocks of 64) and reports its own timeout.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2406_06640_gb300 as pg  # noqa: E402

pytestmark = pytest.mark.gpu

M = 16
POS = np.array([(0, 0), (4, 6), (9, 2)], np.int32)


def _plan(i, stream=None):
    from paper_2406_06640_gb300.engine import Reconstruction

    gen = torch.Generator(device="cuda").manual_seed(i)
    I = torch.rand(3, M, M, device="cuda", generator=gen) * 20 + 1
    torch.cuda.synchronize()
    prm = dict(M=M, K=1, N=3, obj_h=M + 9, obj_w=M + 9, sigma1=1.0, sigma2=1.0, kernel_size=11)
    return Reconstruction(prm, I, POS, stream)


def _run(rec, n):
    O = torch.ones(M + 9, M + 9, device="cuda", dtype=torch.complex64)
    P = torch.ones(1, M, M, device="cuda", dtype=torch.complex64)
    torch.cuda.synchronize()
    rec.iterate(O, P, n)
    return rec.error()


def test_plans_keep_their_own_words():
    expected = []
    for i in range(150):
        rec = _plan(i)
        expected.append(_run(rec, 2))
        rec.close()
    assert len(set(expected)) == 150
    recs = {i: _plan(i) for i in range(150)}
    for i in list(range(0, 150, 3)) + list(range(149, 90, -2)):  # leave blocks partly and wholly empty
        if i in recs:
            recs.pop(i).close()
    lib = pg.load()
    some = sorted(recs)[5]
    assert lib.ptycho_plan_wait_selftest(recs[some]._plan._h, 0, 1_000_000, 0) == 0
    for i, rec in recs.items():
        if i != some:
            assert _run(rec, 2) == expected[i], i
    with pytest.raises(pg.PtychoError):
        _run(recs[some], 2)
    recs.update({i: _plan(i) for i in range(0, 150, 3)})  # words given back are taken again, cleared
    for i in range(0, 150, 3):
        assert _run(recs[i], 2) == expected[i], i
    for rec in recs.values():
        rec.close()


def test_plans_of_several_threads():
    expected = {}
    for i in range(40):
        rec = _plan(i)
        expected[i] = _run(rec, 1)
        rec.close()
    wrong = []

    def work(first):
        stream = torch.cuda.Stream()
        for _ in range(3):
            recs = [(i, _plan(i, stream)) for i in range(first, 40, 4)]
            wrong.extend(i for i, rec in recs if _run(rec, 1) != expected[i])
            for _, rec in reversed(recs):
                rec.close()

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
