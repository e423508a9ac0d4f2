"""The key-tiled 4-cycle tier at the edges of its layout: roots whose counts
pass 16 bits, several counter groups, runs found by search instead of by
index, and a single group whose last id range is short. Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from helpers import closed_complete_bipartite
from test_gpu_parity import assert_same, gpu_count, ni, tuning  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("a,b", [(5, 65534), (5, 65535), (3, 70000)])
def test_counts_around_sixteen_bits(ni, a, b):  # noqa: F811
    # the roots of side A have b in-neighbours and c = b for the other A's
    assert_same(gpu_count(ni, *gg.complete_bipartite(a, b)), closed_complete_bipartite(a, b), f"K{a},{b}")


def test_wide_root_with_keys_of_every_width(ni):  # noqa: F811
    # a hub joined to every vertex of a power-law graph G0: psi_8 by
    # c_xw = c0_xw + 1 inside G0 and c_xh = d0(x)
    import scipy.sparse as sp
    n = 70000
    rp, ci = gg.chunglu(n, 2.2, 6.0, 11)
    d0 = np.diff(rp).astype(np.int64)
    a0 = sp.csr_matrix((np.ones(len(ci), np.int64), ci, rp), shape=(n, n))
    c0 = (a0 @ a0).tocoo()
    off = c0.row != c0.col
    exp = np.bincount(c0.row[off], weights=(c0.data[off] + 1) * c0.data[off] // 2, minlength=n).astype(np.int64)
    exp += d0 * (d0 - 1) // 2
    rp2 = np.concatenate([rp.astype(np.int64) + np.arange(n + 1), [rp[-1] + 2 * n]])
    ci2 = np.concatenate([np.insert(ci, rp[1:], n), np.arange(n)]).astype(np.int32)
    got = gpu_count(ni, rp2.astype(np.int32), ci2)
    assert np.array_equal(got[:n, 8], exp)
    assert got[n, 8] == int((d0 * (d0 - 1) // 2).sum())


@pytest.mark.parametrize("name,make", [
    ("several groups, indexed", lambda: gg.er_mean_degree(600000, 14, 3)),
    ("several groups, searched", lambda: gg.er_mean_degree(1200000, 3, 4)),
    ("one group, 1024 threads", lambda: gg.chunglu(12289, 2.3, 10.0, 5)),
    ("one group, 256 threads", lambda: gg.chunglu(12288, 2.3, 10.0, 6)),
])
def test_groups_with_every_root_in_the_tier(tuning, name, make):  # noqa: F811
    rp, ci = make()
    tuning.set_tuning(c4_warp_maxw=2, c4_team_minw=2)
    assert_same(gpu_count(tuning, rp, ci), oracle.count(rp, ci), name)
