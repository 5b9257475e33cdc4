"""Edges of the GPU kernels' work splits: sizes at which a warp, tile or chunk is partly filled,
exactly filled or exceeded, each against the CPU oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return pytest.importorskip("torch")


@pytest.fixture(scope="module")
def css():
    import paper_2605_20918_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(css):
    c = css.Context(0)
    yield c
    c.close()


def _complete(n):
    adj = np.array([j for i in range(n) for j in range(n) if j != i], np.int32)
    return np.arange(n + 1, dtype=np.int32) * (n - 1), adj


def _ring(n):
    i = np.arange(n)
    adj = np.stack([(i - 1) % n, (i + 1) % n], axis=1).reshape(-1).astype(np.int32)
    return np.arange(n + 1, dtype=np.int32) * 2, adj


# complete graphs: as many colours as vertices, around the 256 colours of one search and the 32
# parents of one look; rings: one vertex per warp, several, and more than the 32 a warp watches at once
@pytest.mark.parametrize("graph,n", [(_complete, 33), (_complete, 256), (_complete, 300), (_ring, 20_001),
                                     (_ring, 400_000)])
def test_colour_graph_splits(torch, ctx, graph, n):
    ptr, adj = graph(n)
    col = torch.empty(n, dtype=torch.int32, device="cuda")
    nc = ctx.color_graph(torch.as_tensor(ptr, device="cuda"), torch.as_tensor(adj, device="cuda"), 1004, col)
    ref, nref = oracle.color_graph(ptr, adj, 1004)
    assert nc == nref and np.array_equal(col.cpu().numpy(), ref)
