"""Learned data term and adjoint kernels where their paths differ: depth ranges
that are a multiple of four or not, arrays longer than one block's chunk, a
row too long to be staged, outputs that do not start on 16 bytes."""
import numpy as np
import pytest

from oracle import learned

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import build
    build.build()
    from paper_1803_01516_gb300 import gazecut
    return gazecut


@pytest.mark.parametrize("h,ng,D", [(1, 1, 2), (3, 41, 5), (7, 65, 16), (17, 130, 23), (2, 9, 64),
                                    (33, 64, 4), (1, 3, 4097), (1, 2, 6400)])
@pytest.mark.parametrize("off", [0, 1])
def test_edges(gc, h, ng, D, off):
    rng = np.random.default_rng(h * 1000 + D)
    w = ng + 2 * (D - 1)
    L, R = (rng.integers(0, 256, size=(h, w)).astype(np.uint8) for _ in range(2))
    X = rng.integers(0, D, size=(h, ng)).astype(np.int32)
    w1, w2, tau = 0.75, 0.6, 33.0
    p = gc.Params(w=w, h=h, D=D, tau=0, lam=3, inhibit=5)
    Ld, Rd, Xd = (torch.from_numpy(a).cuda() for a in (L, R, X))
    n = h * ng * D
    cost = torch.full((n + off,), -7, dtype=torch.int32, device="cuda")[off:]
    gc.gs_stereo_cost_volume_f32(Ld, Rd, p, w1, w2, tau, 256.0, cost)
    ref = learned.cost_volume_f32(L, R, D, 2 * (D - 1), w1, w2, tau, 256.0)
    assert np.array_equal(cost.cpu().numpy().reshape(ref.shape), ref)
    guard = torch.full((n + off + 8,), -1.0, dtype=torch.float32, device="cuda")
    dcost = guard[off:off + n]
    counts = torch.zeros(2, dtype=torch.int64, device="cuda")
    gc.gs_energy_backward(Xd, p, 0.75, dcost, counts)
    onehot, J, V = learned.energy_adjoint(X, D, 1)
    assert np.array_equal(dcost.cpu().numpy().reshape(onehot.shape), 0.75 * onehot)
    assert (guard[off + n:] == -1).all()
    assert counts.cpu().tolist() == [J, V]
    sums = torch.zeros(3, dtype=torch.int64, device="cuda")
    gc.gs_cost_volume_f32_backward(Ld, Rd, p, w1, w2, tau, Xd, sums)
    assert tuple(sums.cpu().tolist()) == learned.cost_grad_sums(L, R, D, 2 * (D - 1), w1, w2, tau, X)
