"""Propagation over row shapes and TF layouts at the edges of its tiles: rows of
one, two, three and more vectors, RGBA tables on and off a 16-byte boundary,
graphs of one level, of a few nodes and of more than one tile per level, and
repeated launches on several streams.  Against fp64 level by level, within the
rounding of the storage type: each level rounds the weight and the value once,
(2 D + 1) u of the largest input."""
import numpy as np
import pytest

from paper_2009_02702_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = {"f32": 2.0 ** -24, "f16": 2.0 ** -11, "bf16": 2.0 ** -8}


@pytest.fixture(scope="module")
def graphs():
    from paper_2009_02702_gb300 import mg
    vols = [np.zeros((1, 1, 1), np.uint16), np.arange(8, dtype=np.uint16).reshape(2, 2, 2),
            synth.make_volume(1, dims=(40, 33, 21), S=30), synth.make_volume(1, dims=(96, 96, 96), S=700)]
    out = []
    for v in vols:
        S = int(v.max()) + 1
        out.append((mg.mg_build(torch.from_numpy(v).cuda(), S), S))
    return mg, out


def exact(mg, g, tf):
    p, q, a, b = (x.astype(np.int64) for x in mg.mg_graph_copy_nodes(g))
    v = np.zeros((g.N, tf.shape[1]))
    v[:g.S] = tf
    bk = g.info["bucket"]
    for lo, hi in zip(bk[1:-1], bk[2:]):
        w = (b[lo:hi] / (a[lo:hi] + b[lo:hi]))[:, None]
        v[lo:hi] = (1 - w) * v[p[lo:hi]] + w * v[q[lo:hi]]
    return v


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("k,C,shift", [(1, 1, 0), (1, 2, 0), (1, 3, 0), (1, 4, 0), (1, 4, 1), (1, 5, 0), (1, 6, 0),
                                       (1, 7, 1), (1, 8, 0), (1, 12, 0), (1, 16, 0), (2, 4, 0), (3, 4, 2), (5, 4, 0),
                                       (7, 4, 0), (8, 4, 0), (4, 2, 0), (2, 6, 0)])
def test_rows(graphs, storage, k, C, shift):
    mg, gs = graphs
    rng = np.random.default_rng([k, C])
    for g, S in gs:
        tf = rng.random((k, S, C), dtype=np.float32)
        flat = torch.zeros(k * S * C + shift, device="cuda")
        dev = flat[shift:].view(k, S, C)
        dev.copy_(torch.from_numpy(tf))
        streams = [torch.cuda.Stream() for _ in range(2)]
        torch.cuda.synchronize()
        outs = []
        for s in streams * 2:   # each stream's second launch finds its words as the first left them
            with torch.cuda.stream(s):
                outs.append(mg.mg_propagate_tf(g, dev[0], storage=storage) if k == 1
                            else mg.mg_propagate_tf_multi(g, dev, storage=storage))
        torch.cuda.synchronize()
        mg.mg_sync_status(g)
        ref = np.concatenate([exact(mg, g, t.astype(np.float64)) for t in tf], 1)
        bound = (2 * g.info["depth"] + 1) * U[storage]
        for o in outs:
            assert torch.equal(o, outs[0])
            assert np.abs(o.double().cpu().numpy() - ref).max() <= bound
