"""GPU: iterations captured into a caller's CUDA graph and replayed. ptycho_error returns E of the last iteration the
host asked for (the plan's ring of errors is indexed by calls), also where replays have run past it, and objects
and probes are those of as many plain iterations.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,engine", [(32, 2, "pie"), (128, 2, "pie"), (32, 2, "dm"), (256, 1, "pie")])
def test_error_of_replayed_iterations(M, K, engine):
    from paper_2406_06640_gb300.engine import Reconstruction

    dev = torch.device("cuda:0")
    p = make_problem(0, scan_side=3, obj_side=M + 24 * M // 64 + 9, M=M, K=K, sigma=1.0)
    prm = dict(p.params, sigma1=1.0, sigma2=1.0, engine=engine, windows=[])
    I = torch.from_numpy(p.I).to(dev)

    def start(stream=None):
        return (Reconstruction(prm, I, p.positions, stream), torch.from_numpy(p.O0.astype(np.complex64)).to(dev),
                torch.from_numpy(p.P0.astype(np.complex64)).to(dev))

    plain, O, P = start()
    E, states = [], []
    for _ in range(6):
        plain.iterate(O, P, 1)
        E.append(plain.error())
        states.append((O.clone(), P.clone()))
    plain.close()
    assert len(set(E)) == 6

    s = torch.cuda.Stream()
    rec, O, P = start(s)
    torch.cuda.synchronize()
    rec.iterate(O, P, 1)
    assert rec.error() == E[0]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        rec.iterate(O, P, 1)
    with torch.cuda.stream(s):
        for _ in range(4):
            g.replay()
    assert rec.error() == E[1]  # two iterations asked for, five run
    assert torch.equal(O, states[4][0]) and torch.equal(P, states[4][1])
    rec.iterate(O, P, 1)
    assert rec.error() == E[2] and rec.errors(3) == E[:3]
    assert torch.equal(O, states[5][0])
    rec.close()
