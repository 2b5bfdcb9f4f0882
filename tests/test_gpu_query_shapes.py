"""Launch shapes of the batched box query at the limits of shared memory, and
plans whose launches were refused.  Counts are whole numbers, equal to the
oracle's."""
import ctypes

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


def noise(dims, S, seed):
    rng = np.random.default_rng(seed)
    return rng.integers(0, S, dims[::-1]).astype(np.uint16)


def some_boxes(dims, n, seed):
    rng = np.random.default_rng(seed)
    d = np.array(dims)
    lo = rng.integers(0, d, (n, 3))
    return np.concatenate([lo, rng.integers(1, d - lo + 1)], 1).astype(np.int32)


def test_a_plan_goes_on_after_a_refused_launch(mg):
    """Two graphs whose fp32 histograms take the same kernel, one of them nearly
    all shared memory of an SM: should a run of its plan be refused after the
    other graph's calls, the next run starts from clean counters."""
    dims, S = (40, 32, 24), 18620
    vol = noise(dims, S, 1)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    other = mg.mg_build(torch.from_numpy(noise(dims, 2500, 2)).cuda(), 2500)
    batches = [some_boxes(dims, 60, k) for k in range(3)]
    t = [torch.from_numpy(b).cuda() for b in batches]
    plan = mg.QueryPlan(g, max_Q=60, hist="f32")
    mg.mg_query_boxes(other, t[0], hist="f32")
    try:
        plan.run(t[0])
    except mg.MGError as e:
        assert e.status == mg.MG_ERR_CUDA
    mg.mg_query_boxes(g, t[1], hist="f32")
    for k in (2, 0):
        h = plan.run(t[k]).cpu().numpy()
        assert np.array_equal(h.astype(np.int64), oracle.box_hist(vol, S, batches[k]).astype(np.int64)), k
    mg.mg_sync_status(g)
    plan.close()
    g.close()
    other.close()


# 18002-18004 at 512 threads and 18685-18686 at 256: dynamic shared memory fits
# an SM by itself, but not with the kernel's static variables
@pytest.mark.parametrize("S", [17299, 18003, 18333, 18602, 18686])
def test_every_shape_of_the_largest_float_histograms(mg, S):
    dims = (40, 32, 24)
    vol = noise(dims, S, S)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = some_boxes(dims, 40, S)
    t = torch.from_numpy(bx).cuda()
    ref = oracle.box_hist(vol, S, bx).astype(np.int64)
    most = 512 if S < 18660 else 256   # 16 warps' queues fit beside the histogram up to there
    for threads in (0, 128, 256, 512)[:3 + (most == 512)]:
        h = mg.mg_query_boxes(g, t, hist="f32", block_threads=threads)
        assert np.array_equal(h.cpu().numpy().astype(np.int64), ref), threads
    if most == 512:
        assert mg.mg_query_autotune(g, t, hist="f32")["block_threads"] in (128, 256, 512)
    assert np.array_equal(mg.mg_query_boxes(g, t, hist="f32").cpu().numpy().astype(np.int64), ref)
    mg.mg_sync_status(g)
    g.close()


def test_plans_of_two_graphs_keep_their_shared_memory(mg):
    """The limit of a kernel's shared memory is the same for every caller."""
    dims, S = (40, 32, 24), 18620
    vol = noise(dims, S, 1)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    other = mg.mg_build(torch.from_numpy(noise(dims, 2500, 2)).cuda(), 2500)
    bx = some_boxes(dims, 60, 5)
    t = torch.from_numpy(bx).cuda()
    plan = mg.QueryPlan(g, max_Q=60, hist="f32")
    mg.mg_query_boxes(other, t, hist="f32")
    h = plan.run(t).cpu().numpy()
    assert np.array_equal(h.astype(np.int64), oracle.box_hist(vol, S, bx).astype(np.int64))
    plan.close()
    g.close()
    other.close()


@pytest.mark.parametrize("layout", ["dense", "csr"])
def test_direct_batch_within_a_small_allocator(mg, layout):
    """1,000 boxes of 64^3 could have 2.7 M blocks (33 MB) and have under
    200,000: without memory for the worst case the batch is planned exactly."""
    dims, S = (64, 64, 64), 64
    vol = (np.arange(64 ** 3).reshape(64, 64, 64) // 97 % S).astype(np.uint16)
    ids = torch.from_numpy(vol).cuda()
    state = {"most": 1 << 40, "refused": 0}

    def alloc(ctx, nbytes, stream):
        if nbytes > state["most"]:
            state["refused"] += 1
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))

    def free(ctx, ptr, nbytes, stream):
        torch.cuda.caching_allocator_delete(int(ptr))

    a = mg.mg_allocator(None, mg.ALLOC_FN(alloc), mg.FREE_FN(free))
    h = ctypes.c_void_p()
    st = mg.lib().mg_build(ids.data_ptr(), *dims, S, ctypes.byref(mg.mg_build_opts(2)), ctypes.byref(a),
                           torch.cuda.current_stream().cuda_stream, ctypes.byref(h))
    assert st == mg.MG_OK
    g = mg.Graph(h.value, 0, a)
    bx = some_boxes(dims, 1000, 7)
    t = torch.from_numpy(bx).cuda()
    ref = oracle.box_hist(vol, S, bx)
    state["most"] = 8 << 20
    for k in range(3):   # (the scratch of a stream grows to what its calls took)
        if layout == "dense":
            got = mg.mg_query_boxes(g, t).cpu().numpy()
        else:
            off, seg, cnt = (x.cpu().numpy() for x in mg.mg_query_boxes(g, t, layout="csr"))
            got = np.zeros_like(ref)
            for q in range(len(bx)):
                got[q, seg[off[q]:off[q + 1]]] = cnt[off[q]:off[q + 1]]
        assert np.array_equal(got, ref), k
    assert state["refused"] > 0
    mg.mg_sync_status(g)
    g.close()


@pytest.mark.parametrize("hist,alpha", [("u32", "f32"), ("f32", "f32"), ("f32", "f16")])
def test_direct_batches_on_both_sides_of_the_worst_case_bound(mg, hist, alpha):
    """1,528 boxes of 64^3 have fewer than 2^22 blocks whatever they are and are
    planned in one launch; 1,529 boxes are not."""
    dims, S = (64, 64, 64), 64
    assert 1528 * 14 ** 3 < 1 << 22 <= 1529 * 14 ** 3
    vol = (np.arange(64 ** 3).reshape(64, 64, 64) // 97 % S).astype(np.uint16)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = some_boxes(dims, 1529, 8)
    t = torch.from_numpy(bx).cuda()
    one = mg.mg_query_boxes(g, t[:1528].contiguous(), hist=hist, alpha=alpha).cpu().numpy().astype(np.float64)
    many = mg.mg_query_boxes(g, t, hist=hist, alpha=alpha).cpu().numpy().astype(np.float64)
    mg.mg_sync_status(g)
    ref = oracle.box_hist(vol, S, bx).astype(np.float64)
    if alpha == "f32":
        assert np.array_equal(one, ref[:1528]) and np.array_equal(many, ref)
    else:   # the same shares, at most one a cube (8/3 of the three areas), summed in another order
        assert (np.abs(one - many[:1528]) <= 8 * 64 ** 2 * 2.0 ** -24 * np.maximum(one, many[:1528])).all()
    g.close()


@pytest.mark.parametrize("S", [64, 1182, 2500])
def test_chunks_of_every_length_the_default_takes(mg, S):
    """Batches whose default chunks run from 128 items to 2,048, direct and by a
    plan made for just as many boxes: few and many, histograms per warp and per CTA."""
    dims = (160, 96, 80)
    z, y, x = np.meshgrid(*(np.arange(n) // k for n, k in zip(dims[::-1], (9, 7, 11))), indexing="ij")
    vol = ((x * 7919 + y * 104729 + z * 1299709) % S).astype(np.uint16)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    for Q in (1, 60, 700, 9000):
        bx = some_boxes(dims, Q, Q)
        t = torch.from_numpy(bx).cuda()
        ref = oracle.box_hist(vol, S, bx).astype(np.int64)
        for hist in ("u32", "f32"):
            plan = mg.QueryPlan(g, max_Q=Q, hist=hist, max_blocks=4096 * Q)
            for h in (mg.mg_query_boxes(g, t, hist=hist), plan.run(t)):
                assert np.array_equal(h.cpu().numpy().astype(np.int64), ref), (Q, hist)
            plan.close()
    mg.mg_sync_status(g)
    g.close()


@pytest.mark.parametrize("S", [2049, 3000, 18000])
def test_rows_of_many_segments(mg, S):
    """Noise: a cube of level 2 holds some 64 segments, one of level 3 some 500, at
    every place of a warp's step, added by all its lanes."""
    dims = (64, 48, 40)
    vol = noise(dims, S, S)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = np.concatenate([some_boxes(dims, 200, S), [[0, 0, 0, *dims], [8, 8, 8, 16, 16, 16], [3, 0, 0, 5, 48, 40]]])
    bx = bx.astype(np.int32)
    t = torch.from_numpy(bx).cuda()
    ref = oracle.box_hist(vol, S, bx).astype(np.float64)
    for hist in ("u32", "f32"):
        for kw in (dict(), dict(chunk_cubes=37), dict(schedule="plain")):
            assert np.array_equal(mg.mg_query_boxes(g, t, hist=hist, **kw).cpu().numpy().astype(np.float64), ref)
    for alpha, u in (("f16", 2.0 ** -11), ("bf16", 2.0 ** -8)):   # each unit crosses at most D rounded weights
        h = mg.mg_query_boxes(g, t, hist="f32", alpha=alpha).cpu().numpy().astype(np.float64)
        assert (np.abs(h - ref).sum(1) <= 1.5 * g.info["depth"] * u * ref.sum(1)).all()
        assert ((h != 0) <= (ref != 0)).all()
    mg.mg_sync_status(g)
    g.close()


def test_fixed_scratch_filled_to_its_limit(mg):
    """The scratch-free call takes short chunks for small batches; a batch whose
    blocks leave no room for them is planned with long ones before it is refused."""
    dims, S = (255, 255, 255), 50
    z, y, x = np.meshgrid(*(np.arange(n) // 32 for n in dims), indexing="ij")
    vol = ((x + 8 * y + 64 * z) % S).astype(np.uint16)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    one = np.array([[1, 1, 1, 253, 253, 253]], np.int32)
    ref = oracle.box_hist(vol, S, one)[0]
    out = torch.empty((4000, S), dtype=torch.uint32, device="cuda")

    def fits(Q):
        t = torch.from_numpy(one.repeat(Q, 0)).cuda()
        try:
            mg.mg_query_boxes_noalloc(g, t, out=out[:Q])
        except mg.MGError as e:
            assert e.status == mg.MG_ERR_CAPACITY
            return False
        return True

    lo, hi = 1, 4000
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if fits(mid) else (lo, mid)
    for Q in (1, lo - 20, lo):
        assert fits(Q)
        got = out[:Q].cpu().numpy()
        assert (got == ref).all(), Q
    # 12 bytes a block and 8 a chunk, at most one chunk a box more than its cubes fill
    blocks = 13 ** 3
    cubes = int(mg.mg_count_cubes(g, torch.from_numpy(one).cuda()).cpu().numpy()[0])
    assert (lo + 1) * (12 * blocks + 8 * (cubes // 2048 + 1)) > (60 << 20)
    mg.mg_sync_status(g)
    g.close()


@pytest.mark.parametrize("chunk,threads", [(16384, 256), (3000, 128), (100, 256), (1024, 512), (0, 0)])
def test_recorded_shapes_and_small_batches(mg, chunk, threads):
    """A recorded length is for batches that fill it; what fits a plan's capacity in
    recorded chunks fits it in shorter ones (noise: items are cubes)."""
    dims, S = (64, 64, 64), 700
    vol = noise(dims, S, 3)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    one = np.array([[1, 1, 1, 62, 62, 62]], np.int32)
    cubes = int(mg.mg_count_cubes(g, torch.from_numpy(one).cuda()).cpu().numpy()[0])
    for hist in (0, 1):
        assert mg.lib().mg_query_set_tuning(g.handle, hist, chunk, threads) == mg.MG_OK
    fits = -(-cubes // (chunk or 2048))
    for hist, alpha in (("u32", "f32"), ("f32", "f32"), ("f32", "bf16")):
        for bx in (one, some_boxes(dims, 50, 1), some_boxes(dims, 3000, 2)):
            t = torch.from_numpy(bx).cuda()
            ref = oracle.box_hist(vol, S, bx).astype(np.float64)
            plan = mg.QueryPlan(g, max_Q=len(bx), hist=hist, alpha=alpha, max_blocks=4096 * len(bx),
                                max_chunks=fits * len(bx))
            for h in (mg.mg_query_boxes(g, t, hist=hist, alpha=alpha), plan.run(t)):
                h = h.cpu().numpy().astype(np.float64)
                if alpha == "f32":
                    assert np.array_equal(h, ref)
                else:
                    assert (np.abs(h - ref).sum(1) <= 1.5 * g.info["depth"] * 2.0 ** -8 * ref.sum(1)).all()
            plan.close()
    mg.mg_sync_status(g)
    g.close()


def test_a_shape_tuned_for_some_weights(mg):
    dims, S = (64, 64, 64), 700
    vol = noise(dims, S, 4)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = some_boxes(dims, 4000, 4)
    t = torch.from_numpy(bx).cuda()
    ref = oracle.box_hist(vol, S, bx).astype(np.float64)
    for alpha in ("f16", "f32"):
        r = mg.mg_query_autotune(g, t, hist="f32", alpha=alpha)
        assert r["chunk_cubes"] in (1024, 2048, 4096, 8192, 16384) and r["block_threads"] in (128, 256, 512)
        for other, u in (("f32", 0.0), ("f16", 2.0 ** -11), ("bf16", 2.0 ** -8)):
            h = mg.mg_query_boxes(g, t, hist="f32", alpha=other).cpu().numpy().astype(np.float64)
            assert (np.abs(h - ref).sum(1) <= 1.5 * g.info["depth"] * u * ref.sum(1)).all()
    mg.mg_sync_status(g)
    g.close()


@pytest.mark.parametrize("S,hist,alpha", [(64, "u32", "f32"), (64, "f32", "f16"), (2500, "f32", "f32"), (15000, "u32", "f32")])
@pytest.mark.parametrize("max_chunks", [0, 40000])
def test_plan_made_for_many_boxes_runs_few(mg, S, hist, alpha, max_chunks):
    """Runs take chunks by their own size, where the plan's chunk map holds them."""
    dims = (96, 80, 64)
    vol = noise(dims, S, 9)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = some_boxes(dims, 5000, 9)
    t = torch.from_numpy(bx).cuda()
    plan = mg.QueryPlan(g, max_Q=5000, hist=hist, alpha=alpha, max_blocks=5000 * 2048, max_chunks=max_chunks)
    for Q in (1, 5000, 7, 64, 65, 900, 5000, 2):
        b = bx[:Q]
        h = plan.run(t[:Q].contiguous()).cpu().numpy().astype(np.float64)
        ref = oracle.box_hist(vol, S, b).astype(np.float64)
        u = 2.0 ** -11 if alpha == "f16" else 0.0
        assert (np.abs(h - ref).sum(1) <= 1.5 * g.info["depth"] * u * ref.sum(1)).all(), Q
        mg.mg_sync_status(g)
    plan.close()
    g.close()


def test_server_batches_of_few_and_of_many(mg):
    dims, S = (96, 80, 64), 2500
    vol = noise(dims, S, 10)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    bx = some_boxes(dims, 1200, 10)
    ref = oracle.box_hist(vol, S, bx)
    for hist in ("u32", "f32"):
        srv = mg.Server(slots=2, max_batch=512, hist=hist)
        v = srv.add_volume(g, 4)
        late = [srv.submit_box(v, b) for b in bx[:1100]]   # queued before the start: full batches
        srv.start()
        for k, (ticket, out) in enumerate(late):
            srv.wait(ticket, timeout=60.0)
            assert np.array_equal(out.astype(np.int64), ref[k].astype(np.int64)), k
        for k in range(1100, 1200):                        # one by one
            ticket, out = srv.submit_box(v, bx[k])
            srv.wait(ticket, timeout=60.0)
            assert np.array_equal(out.astype(np.int64), ref[k].astype(np.int64)), k
        st = srv.stats()
        assert st["max_batch_seen"] > 64 and st["failed"] == 0
        srv.close()
    g.close()
