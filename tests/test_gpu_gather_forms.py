"""GPU: the sums of the object and probe updates. The two forms of the gather (a cluster of eight blocks per tile for
long position lists, one block per band for short ones) add the same terms in the same order, so what they have
in common is equal bit by bit; chunks of the staged passes against the FP64 oracle (1e-4, as test_gpu_parity.py).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def _average_list(pos, M, tile=32):
    used = {}
    for y, x in pos:
        for a in range(y // tile, (y + M - 1) // tile + 1):
            for b in range(x // tile, (x + M - 1) // tile + 1):
                used[a, b] = used.get((a, b), 0) + 1
    return sum(used.values()) / len(used)


def _run(prm, I, pos, O, P, n_iter=1):
    from paper_2406_06640_gb300.engine import Reconstruction

    dev = torch.device("cuda:0")
    O, P = torch.from_numpy(O).to(dev), torch.from_numpy(P).to(dev)
    rec = Reconstruction(dict(prm, N=len(pos), obj_h=O.shape[0], obj_w=O.shape[1]), torch.from_numpy(I).to(dev),
                         pos.astype(np.int32))
    rec.iterate(O, P, n_iter)
    rec.close()
    return O.cpu().numpy(), P.cpu().numpy()


@pytest.mark.parametrize("M,K", [(8, 1), (32, 2), (64, 1), (128, 2)])
def test_probe_sums_do_not_depend_on_the_form(M, K):
    """On a constant object the boxes, and so the partials, are the same wherever they lie."""
    N, rng = 600, np.random.default_rng(M)
    I = rng.uniform(0.5, 20.0, (N, M, M)).astype(np.float32)
    P = (rng.standard_normal((K, M, M, 2)) @ [1, 1j]).astype(np.complex64)
    side = 25 * M + 8
    dense = np.stack(np.divmod(np.arange(N), 25), 1) % 8
    sparse = np.stack(np.divmod(np.arange(N), 25), 1) * M
    assert _average_list(dense, M) >= 24 > _average_list(sparse, M)
    O = np.full((side, side), 0.7 + 0.2j, np.complex64)
    prm = dict(M=M, K=K, sigma1=1.0, sigma2=1.0, kernel_size=11, eps_mod=1e-3)
    assert np.array_equal(_run(prm, I, dense, O, P)[1], _run(prm, I, sparse, O, P)[1])


@pytest.mark.parametrize("M", [16, 64, 128])
def test_object_sums_do_not_depend_on_the_form(M):
    """A dense patch, alone and with enough lone positions beside it to bring the average list below the line."""
    rng = np.random.default_rng(M)
    patch = rng.integers(0, 30, (150, 2))
    n = int(np.ceil(np.sqrt(20 * 150 / 4)))  # lone boxes cover four tiles or more each
    lone = np.stack(np.divmod(np.arange(n * n), n), 1) * M + M + 64
    side = int(lone.max()) + M + 3
    both = np.concatenate([patch, lone])
    assert _average_list(patch, M) >= 24 > _average_list(both, M)
    I = rng.uniform(0.5, 20.0, (len(both), M, M)).astype(np.float32)
    P = (rng.standard_normal((1, M, M, 2)) @ [1, 1j]).astype(np.complex64)
    O = np.full((side, side), 0.7 + 0.2j, np.complex64)
    prm = dict(M=M, K=1, sigma1=1.0, sigma2=1.0, kernel_size=11, eps_mod=1e-3)
    a, b = _run(prm, I[:150], patch, O, P)[0], _run(prm, I, both, O, P)[0]
    assert np.array_equal(a[:30 + M, :30 + M], b[:30 + M, :30 + M])


@pytest.mark.parametrize("chunk", [4, 32])
@pytest.mark.parametrize("engine", ["pie", "dm"])
def test_staged_chunks(chunk, engine):
    """70 positions: a last chunk shorter than the groups of the final pass."""
    import paper_2406_06640_gb300 as pg

    p = make_problem(0, scan_side=9, obj_side=256 + 8 * 48 + 9, M=256, K=2, sigma=1.5)
    prm = dict(p.params, N=70, sigma1=1.5, sigma2=1.5, engine=engine)
    I, pos = np.ascontiguousarray(p.I[:70]), p.positions[:70]
    pg.set_staged_chunk(chunk)
    try:
        O, P = _run(prm, I, pos, p.O0.astype(np.complex64), p.P0.astype(np.complex64))
    finally:
        pg.set_staged_chunk(0)
    Oo, Po, _ = oracle.iterate(I, pos, p.O0, p.P0, oracle.Params.from_dict(prm), 1)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    assert rel(O, Oo) < 1e-4 and rel(P, Po) < 1e-4
