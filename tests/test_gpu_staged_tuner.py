"""GPU: timing the staged passes for a plan leaves nothing behind. A plan whose chunk was tuned gives, bit by bit, what
a plan with that chunk fixed gives; the simultaneous engine and the difference map, whose passes differ, are tuned
each by its own.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", ["dm", "pie"])
def test_tuned_plan_equals_fixed_plan(engine):
    import paper_2406_06640_gb300 as pg
    from paper_2406_06640_gb300.engine import Reconstruction

    dev = torch.device("cuda:0")
    p = make_problem(0, scan_side=4, obj_side=256 + 3 * 48 + 9, M=256, K=3, sigma=1.0)
    prm = dict(p.params, sigma1=1.0, sigma2=1.0, kernel_size=9, engine=engine)  # a class no other test plans
    out = []
    chunk = 0
    try:
        for _ in range(2):
            pg.set_staged_chunk(chunk)
            O = torch.from_numpy(p.O0.astype(np.complex64)).to(dev)
            P = torch.from_numpy(p.P0.astype(np.complex64)).to(dev)
            rec = Reconstruction(prm, torch.from_numpy(p.I).to(dev), p.positions)
            chunk = rec.staged_chunk()
            rec.iterate(O, P, 3)
            out.append((O, P, rec.errors(3)))
            rec.close()
    finally:
        pg.set_staged_chunk(0)
    assert chunk in (4, 8, 16) and torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
