"""Tile shapes of the persistent solver at their edges: blocks of four chain
layers with 1 to 4 layers left in the last one, one or two blocks per thread,
tile widths with code of their own (8, 16) and without (4, 32), rows that do
not fill a warp, tiles that the grid cuts off."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bt,tile,D,fits", [
    (256, (32, 3), 22, True),     # two blocks per thread of 512, not of 256
    (256, (8, 3), 86, True),
    (512, (32, 8), 16, True),     # 256 sites x 15 layers: nine fields of exactly 180 KB
    (512, (32, 8), 17, False),
    (512, (4, 1), 280, True),     # long chains, the narrowest tile
    (256, (8, 9), 4, False),
])
def test_shapes_accepted(bt, tile, D, fits):
    from paper_1803_01516_gb300 import build
    build.build()
    from paper_1803_01516_gb300 import gazecut as gc
    p = gc.Params(w=2 * (D - 1) + 64, h=40, D=D, tau=30, lam=3)
    o = gc.SolveOpts(cta_threads=bt, tile_w=tile[0], tile_h=tile[1])
    if fits:
        info = gc.gs_tile_info(p, o)
        assert (info["tile_w"], info["tile_h"]) == tile
        assert info["smem_bytes"] <= 180 * 1024
    else:
        with pytest.raises(RuntimeError):
            gc.gs_tile_info(p, o)


@pytest.mark.gpu
@pytest.mark.parametrize("D", [2, 4, 5, 6, 7, 8, 18])
@pytest.mark.parametrize("tile,bt", [((8, 8), 256), ((8, 8), 512), ((16, 8), 512), ((16, 8), 256),
                                     ((32, 8), 512), ((32, 3), 256), ((4, 8), 256), ((4, 1), 512),
                                     ((8, 3), 256), ((16, 5), 512)])
def test_tile_edges_exact(D, tile, bt):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    h, ng = 19, 43                                   # no tile divides either
    rng = np.random.default_rng(100 * D + tile[0] + tile[1])
    C = rng.integers(0, 31, size=(h, ng, D)).astype(np.int32)
    p = gc.Params(w=ng + 2 * (D - 1), h=h, D=D, tau=0, lam=4, inhibit=37)
    o = gc.SolveOpts(cta_threads=bt, tile_w=tile[0], tile_h=tile[1])
    try:
        gc.gs_tile_info(p, o)
    except RuntimeError:
        pytest.skip("the shape does not fit this depth range")
    ref = oracle.solve(C, 4, 37, 1)
    for direction in (1, 2):
        p.direction = direction
        X, flow, status = gc.solve_costs(torch.from_numpy(C).cuda(), p, o)
        assert int(status.item()) == gc.GS_OK and int(flow.item()) == ref["flow"]
        assert np.array_equal(X.cpu().numpy(), ref["labels"])


@pytest.mark.parametrize("bt,D,shape", [
    (512, 17, (16, 8)), (512, 18, (16, 6)), (512, 21, (16, 6)), (512, 22, (8, 8)),
    (512, 33, (8, 8)), (512, 34, (8, 7)),
    (512, 37, (8, 7)), (512, 38, (8, 6)), (512, 41, (8, 6)), (512, 42, (8, 5)),
    (512, 49, (8, 5)), (512, 50, (8, 4)), (512, 65, (8, 4)), (512, 66, (8, 3)),
    (256, 9, (16, 8)), (256, 10, (8, 8)), (256, 17, (8, 8)),
    (256, 18, (8, 6)), (256, 22, (8, 5)),
])
def test_own_shape_fills_the_threads(bt, D, shape):
    """The library's own tile at both ends of each range of blocks of four
    layers: at most one block per thread."""
    from paper_1803_01516_gb300 import build
    build.build()
    from paper_1803_01516_gb300 import gazecut as gc
    p = gc.Params(w=2 * (D - 1) + 64, h=40, D=D, tau=30, lam=3)
    info = gc.gs_tile_info(p, gc.SolveOpts(cta_threads=bt))
    assert (info["tile_w"], info["tile_h"]) == shape
    assert info["tile_w"] * info["tile_h"] * ((D + 2) // 4) <= bt


@pytest.mark.gpu
@pytest.mark.parametrize("D,bt", [(10, 256), (18, 512), (22, 512), (25, 256), (34, 512), (38, 512),
                                  (45, 512), (66, 512)])
def test_own_shape_exact(D, bt):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_01516_gb300 import gazecut as gc
    h, ng = 23, 35                                   # no tile divides either
    C = np.random.default_rng(D).integers(0, 31, size=(h, ng, D)).astype(np.int32)
    p = gc.Params(w=ng + 2 * (D - 1), h=h, D=D, tau=0, lam=4, inhibit=37)
    ref = oracle.solve(C, 4, 37, 1)
    X, flow, status = gc.solve_costs(torch.from_numpy(C).cuda(), p, gc.SolveOpts(cta_threads=bt))
    assert int(status.item()) == gc.GS_OK and int(flow.item()) == ref["flow"]
    assert np.array_equal(X.cpu().numpy(), ref["labels"])


@pytest.mark.parametrize("w,h,D,shape", [(384, 288, 16, (8, 8)), (400, 300, 17, (8, 8)),
                                         (400, 300, 18, (8, 6)), (400, 300, 20, (8, 6)),
                                         (500, 400, 8, (16, 8)), (500, 400, 9, (16, 8))])
def test_shipped_shape_fills_the_threads(w, h, D, shape, monkeypatch, tmp_path):
    """Shipped entries at both ends of their bucket's chain lengths: at most one
    block of layers per thread; a shape from the caller's own cache stays."""
    import json
    from paper_1803_01516_gb300 import build
    build.build()
    from paper_1803_01516_gb300 import autotune
    from paper_1803_01516_gb300 import gazecut as gc
    monkeypatch.setenv("GAZECUT_TUNE_CACHE", str(tmp_path / "cache.json"))
    p = gc.Params(w=w, h=h, D=D, tau=30, lam=10)
    o = autotune.tuned_opts(p)
    info = gc.gs_tile_info(p, o)
    assert o.cta_threads == 256 and (info["tile_w"], info["tile_h"]) == shape
    with open(autotune.cache_path(), "w") as f:
        json.dump({autotune.bucket(p): {"best": [16, 8, 0, 8, 8, 16, 256]}}, f)
    o = autotune.tuned_opts(p)
    assert (o.tile_w, o.tile_h) == (8, 8)
