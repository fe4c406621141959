"""GPU: an object of more than 2^31 pixels. Boxes in its last rows, whose pixel indices exceed 31 bits, are updated
like the same boxes in a small object, bit by bit (same patterns, same order of every sum), and the rest of it
stays as it was.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

W = 16384
H = (1 << 31) // W + 64  # object, 17 GB; the plan's per-pixel maps take another 60 GB
M, SIDE = 16, 48


@pytest.mark.parametrize("engine", ["pie", "dm"])
def test_boxes_beyond_2_to_the_31(engine):
    from paper_2406_06640_gb300.engine import Reconstruction

    dev = torch.device("cuda:0")
    if torch.cuda.mem_get_info(dev)[0] < 110e9:
        pytest.skip("needs 110 GB of device memory")
    rng = np.random.default_rng(7)
    pos = np.array([(0, 0), (5, 20), (20, 7), (32, 32), (17, 30)], np.int32)
    I = torch.from_numpy(rng.uniform(1, 50, (len(pos), M, M)).astype(np.float32)).to(dev)
    P0 = torch.from_numpy((rng.standard_normal((1, M, M, 2)) @ [1, 1j]).astype(np.complex64)).to(dev)

    def run(h, w, corner):
        O, P = torch.ones(h, w, device=dev, dtype=torch.complex64), P0.clone()
        rec = Reconstruction(dict(M=M, K=1, N=len(pos), obj_h=h, obj_w=w, sigma1=1.0, sigma2=1.0, kernel_size=11,
                                  engine=engine), I, pos + np.array(corner, np.int32))
        rec.iterate(O, P, 2)
        E = rec.errors(2)
        rec.close()
        return O, P, E

    Os, Ps, Es = run(SIDE, SIDE, (0, 0))
    r0, c0 = H - SIDE, W - SIDE
    assert r0 * W >= 1 << 31
    Ob, Pb, Eb = run(H, W, (r0, c0))
    assert torch.equal(Ob[r0:, c0:], Os) and torch.equal(Pb, Ps) and Eb == Es
    Ob[r0:, c0:] = 1
    one = torch.ones(8192, W, device=dev, dtype=torch.complex64)
    for r in range(0, H, 8192):
        assert torch.equal(Ob[r:r + 8192], one[:min(8192, H - r)])
    del Ob, one
    torch.cuda.empty_cache()
