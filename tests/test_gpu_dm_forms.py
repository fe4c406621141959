"""GPU: the two forms of the difference map's launch (a cluster of K CTAs per position for few positions and many
modes, one CTA per position otherwise) on both sides of the line between them, against the FP64 oracle: object,
probe and E within 1e-4 (as test_gpu_parity.py), and two runs equal bit by bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 1e-4


def _run(prob, prm, n_iter):
    from paper_2406_06640_gb300.engine import Reconstruction

    dev = torch.device("cuda:0")
    O = torch.from_numpy(prob.O0.astype(np.complex64)).to(dev)
    P = torch.from_numpy(prob.P0.astype(np.complex64)).to(dev)
    rec = Reconstruction(prm, torch.from_numpy(prob.I).to(dev), prob.positions)
    rec.iterate(O, P, n_iter)
    E = np.array(rec.errors(n_iter))
    rec.close()
    return O.cpu().numpy(), P.cpu().numpy(), E


@pytest.mark.parametrize("geometry", ["far", "near"])
@pytest.mark.parametrize("M,K,side", [(8, 8, 3), (8, 3, 8), (16, 5, 3), (16, 2, 5), (32, 7, 3), (32, 8, 13),
                                      (64, 4, 3), (64, 2, 3), (128, 2, 2), (128, 8, 2), (128, 1, 2), (128, 3, 8)])
def test_difference_map(M, K, side, geometry):
    s = max(M / 64, 0.25)
    p = make_problem(0, scan_side=side, obj_side=int(M + (side - 1) * 10 * s + 9), M=M, K=K, geometry=geometry,
                     sigma=1.0)
    prm = dict(p.params, engine="dm", sigma1=1.0, sigma2=1.0, windows=[(2, 2)], alpha1=1.0, alpha2=0.2)
    O, P, E = _run(p, prm, 3)
    Oo, Po, Eo = oracle.iterate(p.I, p.positions, p.O0, p.P0, oracle.Params.from_dict(prm), 3)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    assert rel(O, Oo) < TOL and rel(P, Po) < TOL and np.max(np.abs(E - Eo) / np.array(Eo)) < TOL
    O2, P2, E2 = _run(p, prm, 3)
    assert np.array_equal(O, O2) and np.array_equal(P, P2) and np.array_equal(E, E2)
