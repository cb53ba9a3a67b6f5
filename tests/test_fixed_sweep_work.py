"""A round of fixed-sweep mode, its work per visit left to the library: once few
nodes are active a visit takes a unit of flow 4 x 8 arcs far within its tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("hops", [1, 15, 17, 24, 31])
def test_a_tail_round_crosses_a_tile(hops):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    # one row of 70 sites in tiles of 32 x 1, one layer: the only excess at site 0,
    # the only sink capacity `hops` sites to its right, arcs of capacity 1
    # between neighbours; one active node of 96 makes it a tail
    C = np.zeros((1, 70, 2), dtype=np.int32)
    C[0, 0, 0] = 1
    C[0, hops, 1] = 1
    p = gc.Params(w=72, h=1, D=2, tau=0, lam=1, inhibit=0, direction=1)
    o = gc.SolveOpts(mode=gc.GS_MODE_FIXED_SWEEPS, fixed_sweeps=1, tile_w=32, tile_h=1,
                     relabel_passes=64)
    X, flow, status = gc.solve_costs(torch.from_numpy(C).cuda(), p, o)
    assert int(status.item()) == gc.GS_OK
    assert int(flow.item()) == 1          # E = 1: either the site's own cost or one jump
