"""GPU: the work items of batch plans. They depend on the class and the device, not on what the process planned
before; a class never leaves CTA slots idle while its items can be cut; few positions with several modes run a
cluster of K CTAs per position. Every form against the FP64 oracle (1e-4, as test_gpu_batch.py), and two runs
equal bit by bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(M, K, side, geometry="far", **kw):
    s = max(M / 64, 0.25)
    p = make_problem(0, scan_side=side, obj_side=int(M + (side - 1) * 12 * s + 9), M=M, K=K, geometry=geometry, sigma=1.0)
    return p, dict(p.params, sigma1=1.0, sigma2=1.0, **kw)


def _plan(probs):
    from paper_2406_06640_gb300.engine import ReconstructionBatch

    dev = torch.device("cuda:0")
    return ReconstructionBatch([(prm, torch.from_numpy(p.I).to(dev), p.positions) for p, prm in probs])


def _items(probs):
    batch = _plan(probs)
    out = (batch.items(), batch.classes())
    batch.close()
    return out


def _run(probs, n_iter):
    dev = torch.device("cuda:0")
    batch = _plan(probs)
    O = [torch.from_numpy(p.O0.astype(np.complex64)).to(dev) for p, _ in probs]
    P = [torch.from_numpy(p.P0.astype(np.complex64)).to(dev) for p, _ in probs]
    batch.iterate(O, P, n_iter)
    E = batch.errors()
    batch.close()
    return [o.cpu().numpy() for o in O], [p.cpu().numpy() for p in P], E


@pytest.mark.parametrize("M,K", [(32, 2), (128, 1)])
def test_items_do_not_depend_on_earlier_plans(M, K):
    small = [_problem(M, K, 3, kernel_size=9)]
    before = _items(small)
    assert before[0][0]["items"] == small[0][0].N and before[0][0]["item_len"] == 1
    large = 4 * [_problem(M, K, 24, kernel_size=9)]
    big = _items(large)
    assert big[0][0]["ctas"] < big[0][0]["items"]
    assert _items(small) == before
    assert _items(large)[0] == big[0]


def _check(probs, n_iter):
    O, P, E = _run(probs, n_iter)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    for b, (p, prm) in enumerate(probs):
        Oo, Po, Eo = oracle.iterate(p.I, p.positions, p.O0, p.P0, oracle.Params.from_dict(prm), n_iter)
        assert rel(O[b], Oo) < 1e-4 and rel(P[b], Po) < 1e-4 and abs(E[b] - Eo[-1]) < 1e-4 * Eo[-1], b
    O2, P2, E2 = _run(probs, n_iter)
    assert all(np.array_equal(x, y) for x, y in zip(O + P, O2 + P2)) and E == E2


@pytest.mark.parametrize("geometry", ["far", "near"])
@pytest.mark.parametrize("M,K", [(8, 8), (16, 6), (32, 5), (64, 4), (128, 3), (128, 8)])
def test_clusters_for_few_positions(M, K, geometry):
    probs = [_problem(M, K, side, geometry, kernel_size=size) for side, size in ((1, 11), (3, 11), (2, 21))]
    for it, members in zip(_items(probs)[0], ((0, 1), (2,))):
        T = sum(probs[b][0].N for b in members)
        assert it == dict(item_len=1, items=T, ctas_per_item=K, ctas=T * K)
    _check(probs, 2)


def test_items_of_two_positions():
    probs = [_problem(128, 1, 10), _problem(128, 1, 15)]
    it = _items(probs)[0][0]
    slots = torch.cuda.get_device_properties(0).multi_processor_count
    assert it["item_len"] == 2 and it["items"] == 50 + 113 >= slots and it["ctas_per_item"] == 1
    _check(probs, 1)
