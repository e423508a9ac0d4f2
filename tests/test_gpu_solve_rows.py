"""The orbit solve of large graphs: degrees around the one from which a vertex
has a warp to itself, next to each other in the caller's order and spread over
it. Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_parity import assert_same, gpu_count, ni  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.mark.parametrize("spread", [False, True])
def test_degrees_around_a_warp_each(ni, spread):  # noqa: F811
    n, edges, top = 15000, [], 40
    for h, d in enumerate([0, 1, 7, 8, 9, 62, 63, 64, 65, 127, 128, 129, 511, 512, 600] * 2):
        edges += [(h, top + i) for i in range(d)]            # a star
        edges += [(top + i, top + i + 1) for i in range(0, d - 1, 3)]   # with triangles
        top += d
    assert top <= n
    if spread:
        perm = np.random.default_rng(3).permutation(n)
        edges = [(int(perm[a]), int(perm[b])) for a, b in edges]
    rp, ci = gg.from_edges(n, edges)
    assert_same(gpu_count(ni, rp, ci), oracle.count(rp, ci), f"spread {spread}")
