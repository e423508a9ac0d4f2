"""The orbit solve's lines: vertices of degree 2048 and more take a CTA; in
graphs of many vertices and a high mean degree the vertices up to 2.5 times the
mean are solved 32 at a time. Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_parity import assert_same, gpu_count, ni  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [9000, 12000])   # fewer vertices than the grid has warps, and more
def test_degrees_around_a_cta_each(ni, n):  # noqa: F811
    rng = np.random.default_rng(n)
    degrees = [2047, 2048, 2049, 2303, 2304, 4097, 8191, n - 40]
    pool = n - len(degrees)
    edges = {(int(a), int(a) + 1 + int(rng.integers(0, 9))) for a in rng.integers(0, pool - 10, n)}
    for i, d in enumerate(degrees):
        edges |= {(int(v), pool + i) for v in rng.choice(pool, size=d, replace=False)}
    rp, ci = gg.from_edges(n, sorted(edges))
    assert set(degrees) <= set(np.diff(rp).tolist())
    exp = oracle.count(rp, ci)
    assert_same(gpu_count(ni, rp, ci), exp, f"n = {n}")
    h = [torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in (rp, ci)]
    got = ni.count_host(*h)
    torch.cuda.synchronize()
    ni.check()
    assert_same(got.numpy(), exp, f"n = {n}, host buffers")


@pytest.mark.parametrize("n", [97280 - 1, 97280])   # 640 vertices a multiprocessor of 152
def test_mean_degree_above_a_warp_each(ni, n):  # noqa: F811
    rp, ci = gg.er_mean_degree(n, 72, 9)
    got = gpu_count(ni, rp, ci)
    d = np.diff(rp).astype(np.int64)
    v = np.unique(np.concatenate([np.argsort(d)[[0, -1]], np.arange(0, n, n // 60), [n - 1]])).astype(np.int32)
    assert_same(got[v], oracle.count_vertices(rp, ci, v), f"n = {n}")
    # psi_1 of every vertex from its neighbours' degrees
    psi1 = np.add.reduceat(d[ci], rp[:-1]) - d
    assert (got[:, 0] == d).all() and (got[:, 1] == psi1).all()
    # psi_9 from the neighbours' triangles: paws whose vertex of degree 1 this is
    t = got[:, 3]
    assert (got[:, 9] == np.add.reduceat(t[ci], rp[:-1]) - 2 * t).all()
