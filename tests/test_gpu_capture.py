"""Calls captured into CUDA graphs: what a captured call leaves behind (the
propagation's counters, the scratch of a stream) serves later eager calls and
every replay, in any order."""
import numpy as np
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
