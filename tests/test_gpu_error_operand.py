"""GPU: the measured counts under the error E. With an object of zeros the model intensity is exactly 0 and every
term of E is I^2, so E = 1; with I = 2 the terms (4) and their sums are exact, and squaring the rounded root
instead of taking I gives E = 1 - 1.2e-7. Bar 1e-12: nothing but the final FP64 square root rounds.

Launches that read the counts for E: the staged passes, the difference map, batch members and small mini-batches
(a single plan up to 128^2 reads sqrt(I) alone and squares it).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _problem(M, K, **kw):
    dev = torch.device("cuda:0")
    pos = np.array([(0, 0), (3, 5), (9, 2)], np.int32)
    I = torch.full((3, M, M), 2.0, device=dev)
    prm = dict(M=M, K=K, N=3, obj_h=M + 9, obj_w=M + 5, sigma1=1.0, sigma2=1.0, kernel_size=11, **kw)
    O = torch.zeros(M + 9, M + 5, device=dev, dtype=torch.complex64)
    P = torch.ones(K, M, M, device=dev, dtype=torch.complex64)
    return prm, I, pos, O, P


@pytest.mark.parametrize("kw", [dict(M=256, K=2), dict(M=256, K=1, geometry="near", fresnel_F=10.0),
                                dict(M=512, K=1), dict(M=256, K=2, engine="dm"), dict(M=32, K=2, engine="dm"),
                                dict(M=64, K=1, engine="dm"), dict(M=128, K=2, engine="dm"),
                                dict(M=128, K=4, minibatch=2, order_seed=3)])
@pytest.mark.parametrize("blur", ["amplitude", "intensity"])
def test_single_plan(kw, blur):
    from paper_2406_06640_gb300.engine import Reconstruction

    prm, I, pos, O, P = _problem(blur_domain=blur, **kw)
    rec = Reconstruction(prm, I, pos)
    rec.iterate(O, P, 1)
    assert abs(rec.error() - 1.0) < 1e-12
    rec.close()


@pytest.mark.parametrize("M", [8, 32, 64, 128, 256])
@pytest.mark.parametrize("blur", ["amplitude", "intensity"])
def test_batch_member(M, blur):
    from paper_2406_06640_gb300.engine import ReconstructionBatch

    prm, I, pos, O, P = _problem(M, 2, blur_domain=blur)
    batch = ReconstructionBatch([(prm, I, pos)])
    batch.iterate([O], [P], 1)
    assert abs(batch.errors()[0] - 1.0) < 1e-12
    batch.close()
