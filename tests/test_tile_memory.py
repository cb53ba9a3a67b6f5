"""Shared memory that a launch of the persistent solver really takes, over every
tile shape and chain length, and the shapes that are refused."""
import pytest


@pytest.fixture(scope="module")
def gc():
    from paper_1803_01516_gb300 import build
    build.build()
    from paper_1803_01516_gb300 import gazecut
    return gazecut


KB = 1024
STATIC = 1 * KB          # static shared memory of the kernel, at most
RESERVED = 1 * KB        # the system's share of every resident block


def _tile(gc, D, bt, tile=(0, 0)):
    p = gc.Params(w=2 * (D - 1) + 64, h=40, D=D, tau=30, lam=3)
    o = gc.SolveOpts(cta_threads=bt, tile_w=tile[0], tile_h=tile[1])
    n = gc.gs_tile_smem_bytes(p, o)
    return (gc.gs_tile_info(p, o) if n else None), n


@pytest.mark.parametrize("bt", [512, 256])
@pytest.mark.parametrize("tw", [0, 4, 8, 16, 32])
def test_every_accepted_tile_fits_a_block(gc, bt, tw):
    for th in range(1, 9) if tw else [0]:
        for D in range(2, 300):
            info, n = _tile(gc, D, bt, (tw, th))
            if not n:
                continue
            assert n == info["launch_smem_bytes"]
            w, h = info["tile_w"], info["tile_h"]
            # nine fields of rows, layers (one of padding) and sites with their halo,
            # two lists of 16-bit entries
            assert n >= 4 * (9 * (h + 2) * D * (w + 2) + w * h * (D - 1))
            assert n + STATIC <= 227 * KB, (bt, w, h, D)


def test_own_shapes_leave_room_for_two_blocks(gc):
    for D in range(2, 66):
        _, n = _tile(gc, D, 256)
        assert 2 * (n + STATIC + RESERVED) <= 228 * KB, D


def test_no_tile_no_bytes(gc):
    assert gc.gs_tile_smem_bytes(gc.Params(w=10, h=4, D=16, tau=1, lam=1), gc.SolveOpts()) == 0
    p = gc.Params(w=2 * 499 + 64, h=4, D=500, tau=1, lam=1)
    assert gc.gs_tile_smem_bytes(p, gc.SolveOpts()) == 0
    with pytest.raises(RuntimeError):
        gc.gs_tile_info(p, gc.SolveOpts())


@pytest.mark.parametrize("D", [2, 4, 5, 6, 7, 8, 18])
@pytest.mark.parametrize("tile,bt,longest", [
    ((8, 8), 256, 33), ((8, 8), 512, 49), ((16, 8), 512, 28), ((16, 8), 256, 17),
    ((32, 8), 512, 16), ((32, 3), 256, 22), ((4, 8), 256, 65), ((4, 1), 512, 285),
    ((8, 3), 256, 86), ((16, 5), 512, 41),
])
def test_accepted_and_refused(gc, D, tile, bt, longest):
    """A shape is refused above its longest chain (4096 nodes, 8 for each of the
    threads asked for, nine fields of 180 KB) and nowhere below."""
    info, n = _tile(gc, D, bt, tile)
    assert bool(n) == (D <= longest)
    if n:
        assert (info["tile_w"], info["tile_h"]) == tile
