"""Graph build at its edges: fewer layers than the block has warps, layers that
the warps share unevenly, a depth range too long for the staged costs, one
site more than a group of 32 -- the cut of the built graph (node-parallel
engine) against the oracle, with and without the chain preflow."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,ng,D", [(3, 33, 2), (2, 32, 3), (3, 31, 9), (2, 65, 10), (2, 5, 18),
                                    (2, 3, 385)])
@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("direction", [1, 2])
def test_build_edges(h, ng, D, flags, direction):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    C = np.random.default_rng(h * ng + D).integers(0, 20, size=(h, ng, D)).astype(np.int32)
    p = gc.Params(w=ng + 2 * (D - 1), h=h, D=D, tau=0, lam=3, inhibit=9, direction=direction)
    o = gc.SolveOpts(engine=gc.GS_ENGINE_SIMPLE)
    b = gc.Buffers(p, o)
    gc.gs_build_graph_flags(torch.from_numpy(C).cuda().reshape(-1), p, flags, b.graph, b.status)
    gc.gs_maxflow_solve(b.graph, p, o, b.work, b.status)
    gc.gs_extract_labels(b.graph, p, o, b.work, b.labels, b.flow, b.status)
    ref = oracle.solve(C, 3, 9, 1)
    assert int(b.status.item()) == gc.GS_OK and int(b.flow.item()) == ref["flow"]
    assert np.array_equal(b.labels.cpu().numpy(), ref["labels"])
