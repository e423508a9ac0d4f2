"""Aggregates of graphs with many dense parts, where no vertex is a hub and the
call has no adjacency bitmap: out-degrees around the limits of the warp, CTA
and bit-matrix forms. Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from helpers import closed_complete
from test_gpu_parity import assert_same, ni  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _count_batch(ni, graphs):  # noqa: F811
    rowptr, colidx, vo, eo = gg.pack(graphs)
    # no bitmap: its rows (6 bytes a word, 4 bytes an entry) hold under half of the entries
    deg = np.sort(np.diff(rowptr))[::-1].astype(np.int64)
    words = np.cumsum(np.arange(len(deg)) // 32 + 1)
    rows = int(np.searchsorted(6 * words, 4 * len(colidx), side="right"))
    assert 2 * deg[:rows].sum() < len(colidx)
    dev = torch.device("cuda:0")
    out = ni.count_batch(torch.from_numpy(rowptr.astype(np.int32)).to(dev), torch.from_numpy(colidx).to(dev),
                         torch.from_numpy(vo).to(dev), torch.from_numpy(eo).to(dev))
    ni.check()
    return out.cpu().numpy(), vo


@pytest.mark.parametrize("n,p,copies", [(90, 0.8, 220), (160, 0.6, 200)])
def test_random_dense_graphs(ni, n, p, copies):  # noqa: F811
    graphs = [gg.er(n, p, 70 + i) for i in range(copies)]
    got, vo = _count_batch(ni, graphs)
    for i, (rp, ci) in enumerate(graphs):
        assert_same(got[vo[i]:vo[i + 1]], oracle.count(rp, ci), f"graph {i}")


@pytest.mark.parametrize("k", [66, 257, 258, 1153, 1154])   # out-degrees up to k - 1
def test_a_clique_among_cliques(ni, k):  # noqa: F811
    got, vo = _count_batch(ni, [gg.complete(k)] + [gg.complete(100)] * 1000)
    exp = [np.tile(np.array(closed_complete(s), dtype=np.int64), (s, 1)) for s in [k] + [100] * 1000]
    assert_same(got, np.concatenate(exp), f"K{k}")
