"""Box histograms read through tile and node records: volumes and boxes at the
edges of the tiles (8 and 16 cubes), segments past the four of an inline
record, volumes whose records do not fit, and 16-bit weights.  Counts are whole
numbers, equal to the oracle's; the plain schedule reads cubes only."""
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


def volume(kind, dims, S, rng):
    nx, ny, nz = dims
    if kind == "noise":      # every tile holds many segments: no room for their lists
        return rng.integers(0, S, (nz, ny, nx)).astype(np.uint16)
    if kind == "bricks":     # five to eight segments a tile: records that are lists
        z, y, x = np.meshgrid(np.arange(nz) // 5, np.arange(ny) // 3, np.arange(nx) // 4, indexing="ij")
        return ((x * 7919 + y * 104729 + z * 1299709) % S).astype(np.uint16)
    p = rng.random((S, 3)) * np.array([nz, ny, nx])
    g = np.stack(np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"), -1).reshape(-1, 3)
    best = np.zeros(len(g), np.uint16)
    d = np.full(len(g), np.inf)
    for s in range(S):
        e = ((g - p[s]) ** 2).sum(1)
        best[e < d] = s
        d = np.minimum(d, e)
    return best.reshape(nz, ny, nx)


def boxes_at_edges(dims, rng, n=150):
    """Corners at multiples of 8 and 16 and one voxel beside them, thin slabs
    and lines along each axis, and the whole volume."""
    d = np.array(dims)
    lo = np.minimum(rng.integers(0, 1 + d // 8, (n, 3)) * 8 + rng.integers(-1, 2, (n, 3)), d - 1).clip(0)
    hi = np.minimum(rng.integers(0, 1 + d // 8, (n, 3)) * 8 + rng.integers(-1, 2, (n, 3)), d).clip(1)
    lo, hi = np.minimum(lo, hi), np.maximum(lo, hi)
    side = np.maximum(hi - lo, 1)
    thin = rng.integers(0, 3, n)
    side[np.arange(n), thin] = np.minimum(side[np.arange(n), thin], rng.integers(1, 4, n))
    line = rng.random(n) < 0.3
    side[line, (thin[line] + 1) % 3] = rng.integers(1, 6, line.sum())
    whole = np.array([[0, 0, 0, *dims], [0, 0, dims[2] - 1, dims[0], dims[1], 1], [1, 1, 1, *(d - 1).clip(1)]])
    lo = np.minimum(lo, d - 1)
    return np.concatenate([np.concatenate([lo, side], 1), whole]).astype(np.int32)


CASES = [("cells", (16, 16, 16), 1), ("cells", (131, 67, 70), 23), ("cells", (7, 130, 33), 9),
         ("bricks", (128, 96, 64), 300), ("bricks", (97, 50, 66), 2500), ("noise", (72, 64, 48), 700),
         ("noise", (64, 40, 64), 32768)]


@pytest.mark.parametrize("kind,dims,S", CASES)
def test_counts_through_records(mg, kind, dims, S):
    rng = np.random.default_rng([len(kind), S, *dims])
    vol = volume(kind, dims, S, rng)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = boxes_at_edges(dims, rng)
    ref = oracle.box_hist(vol, S, bx)
    t = torch.from_numpy(bx).cuda()
    hists = [mg.mg_query_boxes(g, t), mg.mg_query_boxes(g, t, chunk_cubes=37)]
    if S <= 18000:   # two fp32 bins a segment fill an SM's shared memory beyond that
        hists.append(mg.mg_query_boxes(g, t, hist="f32"))
    plan = mg.QueryPlan(g, max_Q=len(bx), max_blocks=len(bx) * 4096, max_chunks=len(bx) * 4096)
    hists += [plan.run(t), mg.mg_query_boxes(g, t, schedule="plain")]
    back = mg.mg_graph_import(mg.mg_graph_export(g))
    hists.append(mg.mg_query_boxes(back, t))
    for h in hists:
        assert np.array_equal(h.cpu().numpy().astype(np.int64), ref.astype(np.int64))
    mg.mg_sync_status(g)
    plan.close()
    back.close()
    g.close()


@pytest.mark.parametrize("alpha,u", [("f16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("kind,dims,S", [("cells", (131, 67, 70), 23), ("bricks", (97, 50, 66), 2500)])
def test_sixteen_bit_weights_through_records(mg, kind, dims, S, alpha, u):
    # each unit of a box's weight crosses at most D rounded weights
    rng = np.random.default_rng([S, *dims])
    vol = volume(kind, dims, S, rng)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = boxes_at_edges(dims, rng)
    ref = oracle.box_hist(vol, S, bx).astype(np.float64)
    h = mg.mg_query_boxes(g, torch.from_numpy(bx).cuda(), hist="f32", alpha=alpha).cpu().numpy().astype(np.float64)
    mg.mg_sync_status(g)
    assert (np.abs(h - ref).sum(1) <= 1.5 * g.info["depth"] * u * ref.sum(1)).all()
    assert ((h != 0) <= (ref != 0)).all()
    g.close()


@pytest.mark.parametrize("threads", [128, 256, 512])
def test_most_segments_of_a_float_histogram(mg, threads):
    # the largest histograms leave room for a few warps' block descriptors only
    dims, S = (40, 32, 24), 18600
    rng = np.random.default_rng(threads)
    vol = volume("noise", dims, S, rng)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = boxes_at_edges(dims, rng, 40)
    h = mg.mg_query_boxes(g, torch.from_numpy(bx).cuda(), hist="f32", block_threads=threads).cpu().numpy()
    mg.mg_sync_status(g)
    assert np.array_equal(h.astype(np.int64), oracle.box_hist(vol, S, bx).astype(np.int64))
    g.close()


@pytest.mark.parametrize("dims,S,third", [((64, 48, 40), 16384, 0.0), ((64, 48, 40), 5, 0.01), ((61, 47, 39), 997, 0.004)])
def test_tiles_of_two_segments(mg, dims, S, third):
    # pairs that share and differ in any bits, one segment a single voxel or all but one, and strays among them
    rng = np.random.default_rng([S, *dims])
    nx, ny, nz = dims
    cell = tuple((n + 7) // 8 for n in (nz, ny, nx))

    def spread(v):
        return v.repeat(8, 0).repeat(8, 1).repeat(8, 2)[:nz, :ny, :nx]

    a, b, share = (spread(v) for v in (rng.integers(0, S, cell), rng.integers(0, S, cell), rng.random(cell) ** 3))
    vol = np.where(rng.random((nz, ny, nx)) < share, a, b)
    vol = np.where(rng.random(vol.shape) < third, rng.integers(0, S, vol.shape), vol).astype(np.uint16)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = boxes_at_edges(dims, rng)
    h = mg.mg_query_boxes(g, torch.from_numpy(bx).cuda()).cpu().numpy()
    mg.mg_sync_status(g)
    assert np.array_equal(h.astype(np.int64), oracle.box_hist(vol, S, bx).astype(np.int64))
    g.close()


@pytest.mark.parametrize("S", [352, 1040, 1100, 1200, 1480, 2048])
def test_default_shapes_of_float_histograms(mg, S):
    # both CTA sizes that an untuned batch can take, and its chunk lengths; the bound of the 16-bit weights as above
    dims = (96, 64, 48)
    rng = np.random.default_rng(S)
    vol = volume("bricks", dims, S, rng)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    for n in (1, 40, 900):
        bx = boxes_at_edges(dims, rng, n)
        ref = oracle.box_hist(vol, S, bx).astype(np.float64)
        t = torch.from_numpy(bx).cuda()
        assert np.array_equal(mg.mg_query_boxes(g, t, hist="f32").cpu().numpy().astype(np.float64), ref)
        plan = mg.QueryPlan(g, max_Q=len(bx), hist="f32", alpha="f16", max_blocks=len(bx) * 4096, max_chunks=len(bx) * 4096)
        for h in (mg.mg_query_boxes(g, t, hist="f32", alpha="f16"), plan.run(t)):
            h = h.cpu().numpy().astype(np.float64)
            assert (np.abs(h - ref).sum(1) <= 1.5 * g.info["depth"] * 2.0 ** -11 * ref.sum(1)).all()
        mg.mg_sync_status(g)
        plan.close()
    g.close()
