"""Relabel passes end at their fixed point however the warps of a tile interleave:
repeated solves of chains that many warps share, with costs that let distances
run far along and across the chains, always give the canonical cut."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("D,tile,bt", [(64, (8, 4), 512), (64, (8, 2), 256), (40, (8, 5), 512),
                                       (17, (16, 8), 512), (48, (8, 8), 512)])
@pytest.mark.parametrize("direction", [1, 2])
def test_repeated_relaxations(D, tile, bt, direction):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    h, ng = 21, 37                                   # no tile divides either
    rng = np.random.default_rng(D + tile[1])
    C = rng.integers(0, 2, size=(h, ng, D)).astype(np.int32) * rng.integers(0, 40, size=(h, ng, 1),
                                                                            dtype=np.int32)
    p = gc.Params(w=ng + 2 * (D - 1), h=h, D=D, tau=0, lam=2, inhibit=11, direction=direction)
    o = gc.SolveOpts(tile_w=tile[0], tile_h=tile[1], cta_threads=bt)
    ref = oracle.solve(C, 2, 11, 1)
    c, b = torch.from_numpy(C).cuda(), gc.Buffers(p, o)
    for _ in range(6):
        X, flow, status = gc.solve_costs(c, p, o, b)
        assert int(status.item()) == gc.GS_OK and int(flow.item()) == ref["flow"]
        assert np.array_equal(X.cpu().numpy(), ref["labels"])
