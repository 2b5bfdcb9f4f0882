"""Ray-sample lookups whose rows are copied by one or two samples a thread, at
the edges of a CTA's samples.  Values are copied: equal bits."""
import numpy as np
import pytest

from paper_2009_02702_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("C", [1, 3, 7, 8, 9, 12, 15, 16])
def test_rows_of_every_width(storage, C):
    from paper_2009_02702_gb300 import mg
    dims, S = (41, 30, 23), 25
    g = mg.mg_build(torch.from_numpy(synth.make_volume(1, dims=dims, S=S)).cuda(), S)
    rng = np.random.default_rng(C)
    vals = torch.from_numpy(rng.random((g.N, C)).astype(np.float32)).cuda().to(
        torch.float16 if storage == "f16" else torch.float32)
    ids = [mg.mg_graph_copy_mip(g, l).ravel() for l in range(g.info["levels"])]
    smp = synth.make_samples(1, dims=dims, width=40, height=20)[:600]
    lev = np.clip(np.floor(smp[:, 3] + np.float32(0.5)), 0, g.info["levels"] - 1).astype(int)
    node = np.empty(len(smp), np.int64)
    for i, l in enumerate(lev):
        d = g.info["dims"][l]
        v = [min(int(min(max(smp[i, k], 0.0), g.info["dims"][0][k])) >> l, d[k] - 1) for k in range(3)]
        node[i] = ids[l][(v[2] * d[1] + v[1]) * d[0] + v[0]]
    ref = vals.cpu()[torch.from_numpy(node)]
    t = torch.from_numpy(smp).cuda()
    for P in (1, 127, 128, 129, 255, 256, 257, 600):
        assert torch.equal(mg.mg_render_lookup(g, vals, t[:P].contiguous()).cpu(), ref[:P]), P
    g.close()
