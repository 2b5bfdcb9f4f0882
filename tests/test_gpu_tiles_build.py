"""Tile records of volumes whose tiles hold any number of segments: below, at and
past what a thread counts by itself (16 segments of an ID tile, 24 of a merged
one), pools that run full in any stage, and rows longer than a warp's part.
Counts are whole numbers, equal to the oracle's."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2009_02702_gb300 import mg as _mg
    _mg.lib()
    return _mg


def tile_boxes(dims, rng, n=80):
    d = np.array(dims)
    lo = np.minimum(rng.integers(0, 1 + d // 8, (n, 3)) * 8 + rng.integers(-1, 2, (n, 3)), d - 1).clip(0)
    side = np.minimum(rng.choice([1, 2, 3, 8, 16, 32, 64, 2000], (n, 3)), d - lo)
    return np.concatenate([np.concatenate([lo, side], 1), [[0, 0, 0, *dims]]]).astype(np.int32)


def check(mg, vol, S, rng):
    dims = vol.shape[::-1]
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = tile_boxes(dims, rng)
    t = torch.from_numpy(bx).cuda()
    ref = oracle.box_hist(vol, S, bx)
    assert np.array_equal(mg.mg_query_boxes(g, t).cpu().numpy(), ref)
    back = mg.mg_graph_import(mg.mg_graph_export(g))
    assert np.array_equal(mg.mg_query_boxes(back, t).cpu().numpy(), ref)
    mg.mg_sync_status(g)
    back.close()
    g.close()


@pytest.mark.parametrize("kinds", [1, 2, 3, 4, 5, 15, 16, 17, 24, 25, 40])
@pytest.mark.parametrize("dims", [(96, 64, 48), (71, 50, 37)])
def test_tiles_of_any_number_of_segments(mg, kinds, dims):
    # every region of 16^3 draws from `kinds` segments of its own, in any order and any counts
    S = 32768
    rng = np.random.default_rng([kinds, *dims])
    shape = dims[::-1]
    z, y, x = np.meshgrid(*(np.arange(n) // 16 for n in shape), indexing="ij")
    first = rng.integers(0, S - kinds, 4096)[(z * 16 + y) * 16 + x]
    vol = (first + np.minimum(rng.geometric(0.2, shape) - 1, kinds - 1)).astype(np.uint16)
    check(mg, vol, S, rng)


@pytest.mark.parametrize("share", [0.02, 0.1, 0.3, 1.0])
def test_pools_that_run_full(mg, share):
    # a part of the volume is noise: the lists fit, or run out in one stage or another
    dims, S = (160, 128, 96), 3000
    rng = np.random.default_rng(int(100 * share))
    vol = np.full(dims[::-1], 7, np.uint16)
    n = int(share * dims[2])
    vol[:n] = rng.integers(0, S, vol[:n].shape)
    check(mg, vol, S, rng)


@pytest.mark.parametrize("dims", [(60000, 1, 1), (1, 9000, 3), (2049, 5, 2), (3, 2, 4097), (1023, 1, 17)])
def test_long_rows(mg, dims):
    S = 900
    rng = np.random.default_rng(dims)
    vol = (np.arange(np.prod(dims)) // 37 % S).astype(np.uint16).reshape(dims[::-1])
    check(mg, vol, S, rng)
