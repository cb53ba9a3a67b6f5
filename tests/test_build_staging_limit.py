"""Graph build around the longest chains whose costs are staged in shared memory
beside the kernel's own sums: the cut of the built graph (node-parallel
engine) against the oracle on both sides of the limit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("D", [379, 380, 381, 382, 383, 384])
def test_build_around_the_staging_limit(D):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    C = np.random.default_rng(D).integers(0, 20, size=(2, 3, D)).astype(np.int32)
    p = gc.Params(w=3 + 2 * (D - 1), h=2, D=D, tau=0, lam=3, inhibit=9)
    o = gc.SolveOpts(engine=gc.GS_ENGINE_SIMPLE)
    b = gc.Buffers(p, o)
    X, flow, status = gc.solve_costs(torch.from_numpy(C).cuda().reshape(-1), p, o, b)
    ref = oracle.solve(C, 3, 9, 1)
    assert int(status.item()) == gc.GS_OK and int(flow.item()) == ref["flow"]
    assert np.array_equal(X.cpu().numpy(), ref["labels"])
