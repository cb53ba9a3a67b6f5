"""Block cuts at the edges of the digit-line transform: blocks of one column
with as many labels as a block may hold (32 lines of one, one line of 32), one
row, weights of zero, and grids whose last blocks are cut off."""
import numpy as np
import pytest

from oracle import level2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,ng,D,b,lam,inh,vi", [
    (9, 1, 32, 3, 3, 7, 1), (10, 1, 9, 3, 3, 7, 1), (1, 13, 9, 3, 2, 40, 1), (1, 1, 5, 2, 1, 1, 1),
    (7, 11, 9, 3, 0, 0, 1), (8, 7, 9, 3, 5, 0, 1), (8, 7, 9, 3, 0, 6, 0), (13, 16, 6, 2, 4, 9, 1),
    (5, 8, 3, 1, 4, 9, 1),
])
def test_block_lines(h, ng, D, b, lam, inh, vi):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    rng = np.random.default_rng(h * 100 + ng * 10 + D)
    C = rng.integers(0, 25, size=(h, ng, D)).astype(np.int32)
    X = rng.integers(0, D, size=(h, ng)).astype(np.int32)
    lo, hi = np.zeros_like(X), np.full_like(X, D - 1)
    p = gc.Params(w=ng + 2 * (D - 1), h=h, D=D, tau=0, lam=lam, inhibit=inh, vertical_inhibit=vi)
    Xd = torch.from_numpy(X).cuda()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    gc.gs_block_descent(torch.from_numpy(C).cuda().reshape(-1), p, b, torch.from_numpy(lo).cuda(),
                        torch.from_numpy(hi).cuda(), Xd, 2, st)
    ref = level2.block_descent(C, X, lam, inh, vi, b, lo, hi, 2)
    assert int(st.item()) == gc.GS_OK
    assert np.array_equal(Xd.cpu().numpy(), ref)
