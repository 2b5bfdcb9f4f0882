"""Calls captured into CUDA graphs: what a captured call leaves behind (the
propagation's counters, the scratch of a stream) serves later eager calls and
every replay, in any order."""
import threading

import pytest

from paper_2009_02702_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS, S = (61, 47, 38), 40


@pytest.fixture(scope="module")
def mg():
    from paper_2009_02702_gb300 import mg as _mg
    _mg.lib()
    return _mg


def build(mg, own_allocator):
    """Memory from torch's allocator, or stream-ordered from the library itself."""
    vol = synth.make_volume(2, dims=DIMS, S=S)
    return mg.mg_build(torch.from_numpy(vol).cuda(), S, use_torch_allocator=not own_allocator)


def capture(f, stream):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        f()
    return graph


@pytest.mark.parametrize("own_allocator", [True, False])
@pytest.mark.parametrize("warm", ["cold", "propagated", "queried"])
def test_propagation_captured_on_a_stream(mg, own_allocator, warm):
    g = build(mg, own_allocator)
    tfs = [torch.from_numpy(synth.make_tf(3, S, 4, frame=k)).cuda() for k in range(3)]
    ref = [mg.mg_propagate_tf(g, t) for t in tfs]
    s = torch.cuda.Stream()
    tf = tfs[0].clone()
    out = torch.empty_like(ref[0])
    torch.cuda.synchronize()
    if warm == "propagated":
        mg.mg_propagate_tf(g, tfs[1], stream=s)
    elif warm == "queried":
        mg.mg_query_boxes(g, torch.tensor([[0, 0, 0, *DIMS]], dtype=torch.int32, device="cuda"), stream=s)
    graph = capture(lambda: mg.mg_propagate_tf(g, tf, out=out, stream=s), s)
    # eager calls on the captured stream before, between and beside the replays
    other = torch.cuda.Stream()
    for k in range(3):
        eager = mg.mg_propagate_tf(g, tfs[k], stream=s)
        torch.cuda.synchronize()
        assert torch.equal(eager, ref[k])
        tf.copy_(tfs[k])
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            graph.replay()
        eager = mg.mg_propagate_tf(g, tfs[2 - k], stream=s)
        torch.cuda.synchronize()
        assert torch.equal(out, ref[k]) and torch.equal(eager, ref[2 - k])
    mg.mg_sync_status(g)
    del graph
    g.close()


@pytest.mark.parametrize("own_allocator", [True, False])
def test_scratch_outlives_its_growth(mg, own_allocator):
    """A frame marched with empty space skipped takes scratch; a query with more
    scratch on the same stream makes it grow between the replays."""
    g = build(mg, own_allocator)
    tf = synth.make_tf(3, S, 4)
    tf[5:, 3] = 0.0
    vals = mg.mg_propagate_tf(g, torch.from_numpy(tf).cuda())
    opac = vals[:, 3].contiguous()
    cam = synth.orbit_camera(3, dims=DIMS, width=64, height=48, frame=1, base_step=0.5)
    boxes = torch.from_numpy(synth.make_boxes(1, Q=300, dims=DIMS, box_max=61)).cuda()
    ref = mg.mg_raymarch(g, vals, cam, opacity=opac)
    hist = mg.mg_query_boxes(g, boxes)
    image = torch.empty_like(ref)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(2):   # the second call makes the stream's scratch fit
        mg.mg_raymarch(g, vals, cam, opacity=opac, image=image, stream=s)
    graph = capture(lambda: mg.mg_raymarch(g, vals, cam, opacity=opac, image=image, stream=s), s)
    for _ in range(3):
        image.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(image, ref)
        again = mg.mg_query_boxes(g, boxes, stream=s)
        torch.cuda.synchronize()
        assert torch.equal(again.cpu(), hist.cpu())
        filler = torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda")   # over whatever was given back
        torch.cuda.synchronize()
        del filler
    mg.mg_sync_status(g)
    del graph
    g.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_first_16_bit_call_captured(mg, storage):
    """The weights it would make cannot come from a capture: it is refused, and
    nothing of it is kept."""
    ref = mg.mg_propagate_tf(build(mg, True), torch.from_numpy(synth.make_tf(3, S, 4)).cuda(), storage=storage)
    g = build(mg, True)
    tf = torch.from_numpy(synth.make_tf(3, S, 4)).cuda()
    out = torch.empty_like(ref)
    s = torch.cuda.Stream()
    with pytest.raises(mg.MGError) as e:
        capture(lambda: mg.mg_propagate_tf(g, tf, storage=storage, out=out, stream=s), s)
    assert e.value.status == mg.MG_ERR_CUDA
    got = mg.mg_propagate_tf(g, tf, storage=storage, stream=s)
    torch.cuda.synchronize()
    assert torch.equal(got, ref)
    graph = capture(lambda: mg.mg_propagate_tf(g, tf, storage=storage, out=out, stream=s), s)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    mg.mg_sync_status(g)
    del graph
    g.close()


def test_first_16_bit_calls_of_several_threads(mg):
    """Weights and records are made once and read only when they are there."""
    tf = torch.from_numpy(synth.make_tf(3, S, 4)).cuda()
    boxes = torch.from_numpy(synth.make_boxes(1, Q=50, dims=DIMS, box_max=61)).cuda()
    work = [lambda g, s: mg.mg_propagate_tf(g, tf, storage="f16", stream=s),
            lambda g, s: mg.mg_query_boxes(g, boxes, hist="f32", alpha="f16", stream=s)]
    g = build(mg, True)
    ref = [f(g, None) for f in work]
    torch.cuda.synchronize()
    g.close()
    for _ in range(5):
        g = build(mg, True)
        streams = [torch.cuda.Stream() for _ in range(8)]
        out = [None] * 8
        gate = threading.Barrier(8)

        def go(k):
            gate.wait()
            out[k] = work[k % 2](g, streams[k])

        threads = [threading.Thread(target=go, args=(k,)) for k in range(8)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        for k in range(8):
            # (the order of the fp32 sums of a histogram differs from run to run)
            assert torch.equal(out[k], ref[0]) if k % 2 == 0 else torch.allclose(out[k], ref[1], rtol=1e-4, atol=1e-3), k
        mg.mg_sync_status(g)
        g.close()
