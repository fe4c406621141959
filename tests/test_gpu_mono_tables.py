"""GPU: the strip monochromatisation kernels at the ends of their shared-memory tables: the last spectrum whose
fraction tables fit, the first without them, and the largest accepted. Criterion of test_gpu_mono.py: x within 1e-4
of the FP64 oracle per pattern, residual norms within 1e-4 of the pattern's norm (FP32 stays below 6e-6).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mono  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.mark.parametrize("M,J", [(64, 16), (64, 17), (64, 63), (64, 64), (128, 47), (128, 48)])
def test_table_ends(M, J):
    from paper_2406_06640_gb300.engine import monochromatise

    rng = np.random.default_rng(10 * M + J)
    B = rng.uniform(0.0, 1e3, size=(3, M, M)).astype(np.float32)
    scales = [1.0, 0.7, 2.5] + list(rng.uniform(0.5, 2.5, J - 3))
    weights = rng.uniform(0.1, 1.0, J)
    x, r = monochromatise(torch.from_numpy(B).cuda(), scales, weights, 3, with_residuals=True)
    X, R = x.cpu().numpy().astype(np.float64), r.cpu().numpy()
    Xo, Ro = mono.monochromatise(B.astype(np.float64), scales, weights, 3)
    for n in range(3):
        assert np.linalg.norm(X[n] - Xo[n]) <= TOL * np.linalg.norm(Xo[n]), n
        assert np.max(np.abs(R[n] - Ro[n])) <= TOL * Ro[n][0], n
