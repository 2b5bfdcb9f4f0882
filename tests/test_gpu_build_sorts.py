"""Builds whose levels are sorted in each of the sort's tile sizes: noise volumes
with topological levels of 5 thousand to 1.2 million nodes, on both sides of
65,536, 131,072 and 262,144.  Node table and mips equal the oracle's."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,S", [((18, 20, 26), 30000), ((64, 64, 32), 60000), ((66, 64, 32), 60000),
                                    ((64, 64, 66), 60000), ((130, 64, 64), 60000), ((40, 40, 40), 3)])
def test_levels_on_both_sides_of_the_sort_sizes(dims, S):
    from paper_2009_02702_gb300 import mg
    nx, ny, nz = dims
    vol = np.random.default_rng([S, *dims]).integers(0, S, (nz, ny, nx)).astype(np.uint16)
    g, og = mg.mg_build(torch.from_numpy(vol).cuda(), S), oracle.Graph(vol, S)
    assert g.N == og.N and g.info["bucket"] == og.bucket.tolist()
    for got, want in zip(mg.mg_graph_copy_nodes(g), (og.p, og.q, og.a, og.b)):
        assert (got == want[: og.N]).all()
    for level in range(og.L):
        assert (mg.mg_graph_copy_mip(g, level) == og.mip(level)).all(), level
    g.close()
