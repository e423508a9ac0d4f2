"""Triangle and aggregate stages over the adjacency bitmap of the hubs and over
streamed rows: out-degrees around the 8, 32 and 64 entries of the warp tier's
layouts, and skewed graphs whose roots have out-neighbours on both sides of
the bitmap's first row. Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_parity import assert_same, gpu_count, ni, tuning  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _cliques(sizes, copies):
    """Disjoint complete graphs: out-degrees size - 1 down to 0."""
    edges, n = [], 0
    for k in sizes * copies:
        edges += [(n + i, n + j) for i in range(k) for j in range(i + 1, k)]
        n += k
    return gg.from_edges(n, edges)


@pytest.mark.parametrize("name,make", [
    # few entries: streamed rows
    ("cliques 2..12, one warp each", lambda: _cliques(list(range(2, 13)), 3)),
    ("cliques 31..36", lambda: _cliques([31, 32, 33, 34, 35, 36], 2)),
    ("cliques 63..67", lambda: _cliques([63, 64, 65, 66, 67], 1)),
    # enough entries for a bitmap that covers every vertex
    ("cliques 2..70", lambda: _cliques(list(range(2, 71)), 1)),
    # a bitmap of some vertices only, not used (no hubs)
    ("sparse, four small roots a warp", lambda: gg.er_mean_degree(200000, 6, 21)),
    ("sparse with triangles", lambda: gg.chunglu_batch(1, 2.8, 6.0, 90000, 90001, 4)[0]),
    # used
    ("hubs, part of the rows", lambda: gg.rmat(13, 16, seed=31)),
])
def test_against_the_oracle(ni, name, make):  # noqa: F811
    rp, ci = make()
    assert_same(gpu_count(ni, rp, ci), oracle.count(rp, ci), name)


def test_probed_rows_equal_searched_rows(tuning):  # noqa: F811
    # R-MAT 17 has roots of every tier with out-neighbours outside the bitmap;
    # with these limits the CTA tiers search N+(u) instead of probing
    rp, ci = gg.rmat(17, 16, seed=32)
    got = gpu_count(tuning, rp, ci)
    tuning.set_tuning(tri_bits_maxd=2, tri_hash_maxd=2)
    assert_same(got, gpu_count(tuning, rp, ci), "probed against searched")
    assert np.all(got >= 0)
