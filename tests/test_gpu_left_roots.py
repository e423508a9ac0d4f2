"""4-cycle roots with many repeated keys in graphs that start with the filter:
who takes the roots it leaves (four warps each while they are few, a warp each
in graphs of up to 2048 vertices a multiprocessor when they are many, always a
warp each beyond), and graphs of many triangles, which go without it.
Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from helpers import closed_complete_bipartite
from test_gpu_parity import assert_same, gpu_count, ni, tuning  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FEW, TABLE_MAXW = 8192, 1152


def _union(graphs, isolated=0):
    rp, ci, n = [np.zeros(1, np.int64)], [], 0
    for a, b in graphs:
        rp.append(rp[-1][-1] + a[1:].astype(np.int64))
        ci.append(b.astype(np.int64) + n)
        n += len(a) - 1
    rp.append(np.full(isolated, rp[-1][-1]))
    return np.concatenate(rp).astype(np.int32), np.concatenate(ci).astype(np.int32)


@pytest.mark.parametrize("copies,isolated", [(60, 0), (800, 0), (800, 300000), (60, 600000)])
def test_bipartite_parts(ni, copies, isolated):  # noqa: F811
    # no triangles; nearly every wedge of a root ends where another one does
    import bench

    sides = [(14, 14), (12, 30), (36, 36), (20, 64)]
    rp, ci = _union([gg.complete_bipartite(a, b) for a, b in sides] * copies, isolated)
    sh = bench.Shape(rp, ci)
    w = sh.w_root
    left = (w <= TABLE_MAXW) & (sh.din >= 2) & (sh.din <= 64)
    sure = int((left & (w > 64 + 32)).sum())   # at most 64 different keys: over 32 repeats
    assert sh.n > 32 * 152 and sure > 0
    if isolated:
        assert 2048 * 152 < sh.n < 1 << 21     # packed tables, a warp each
    else:
        assert sh.n <= 2048 * 152 and (sure > FEW if copies > 100 else int(left.sum()) <= FEW)
    assert (w > TABLE_MAXW).any()              # and some for the wider tiers
    exp = [closed_complete_bipartite(a, b) for a, b in sides] * copies + [np.zeros((isolated, 15), np.int64)]
    assert_same(gpu_count(ni, rp, ci), np.concatenate(exp), f"{copies} copies, {isolated} isolated vertices")


def _ring(n, k, seed):
    """A ring of n vertices joined to their k nearest, one edge in ten moved."""
    rng = np.random.default_rng(seed)
    u = np.repeat(np.arange(n), k // 2)
    v = (u + np.tile(np.arange(1, k // 2 + 1), n)) % n
    v = np.where(rng.random(len(v)) < 0.1, rng.integers(0, n, len(v)), v)
    return gg.from_edges(n, sorted({(min(a, b), max(a, b)) for a, b in zip(u.tolist(), v.tolist()) if a != b}))


@pytest.mark.parametrize("n,k,isolated", [(4900, 16, 0), (6000, 60, 0), (20000, 24, 0), (60000, 16, 260000),
                                          (200000, 24, 0)])
def test_overlapping_neighbourhoods(ni, n, k, isolated):  # noqa: F811
    rp, ci = _ring(n, k, 5)
    exp = np.concatenate([oracle.count(rp, ci), np.zeros((isolated, 15), np.int64)])
    # over a third of the pairs of neighbours are edges
    assert 3 * 2 * exp[:, 3].sum() > (exp[:, 0] * (exp[:, 0] - 1)).sum()
    rp = np.concatenate([rp, np.full(isolated, rp[-1], rp.dtype)])
    assert_same(gpu_count(ni, rp, ci), exp, f"ring {n}, {k}")


def test_tables_at_once_past_twenty_one_bits(ni):  # noqa: F811
    # split tables; mean degree 12 and over a third of the pairs closed
    k, copies = 15, (1 << 21) // 15 + 1000
    one = gg.complete(k)
    rp, ci = _union([one])
    n, m = k * copies, len(ci)
    rp = np.concatenate([[0], (rp[1:].astype(np.int64)[None] + m * np.arange(copies)[:, None]).ravel()]).astype(np.int32)
    ci = (ci.astype(np.int64)[None] + k * np.arange(copies)[:, None]).ravel().astype(np.int32)
    got = gpu_count(ni, rp, ci)
    assert n > 1 << 21 and (got == oracle.count(*one)[0]).all()


def test_lowered_limit_of_the_warp_tables(tuning):  # noqa: F811
    rp, ci = _ring(20000, 24, 6)
    exp = oracle.count(rp, ci)
    for maxw in (2, 33, 200):
        tuning.set_tuning(c4_warp_maxw=maxw)
        assert_same(gpu_count(tuning, rp, ci), exp, f"c4_warp_maxw {maxw}")


@pytest.mark.parametrize("graphs,n,p", [(40, 300, 0.1), (30, 700, 0.02), (20, 700, 0.04)])
def test_batches_of_random_graphs(ni, graphs, n, p):  # noqa: F811
    # eight and more repeated keys per root of (n p)^2 / 3 wedges, and fewer
    gs = [gg.er(n, p, 30 + i) for i in range(graphs)]
    assert (((n * p) ** 2 / 3) ** 2 / (2 * n) >= 8) == (p > 0.03) and graphs * n > 32 * 152
    rowptr, colidx, vo, eo = gg.pack(gs)
    dev = torch.device("cuda:0")
    out = ni.count_batch(torch.from_numpy(rowptr.astype(np.int32)).to(dev), torch.from_numpy(colidx).to(dev),
                         torch.from_numpy(vo).to(dev), torch.from_numpy(eo).to(dev))
    ni.check()
    got = out.cpu().numpy()
    for i, (rp, ci) in enumerate(gs):
        assert_same(got[vo[i]:vo[i + 1]], oracle.count(rp, ci), f"graph {i}")


@pytest.mark.parametrize("n", [16 * 152, 16 * 152 + 1, 32 * 152, 32 * 152 + 1])   # small graphs' lines (152 multiprocessors)
@pytest.mark.parametrize("k", [12, 24])
def test_small_graphs(ni, n, k):  # noqa: F811
    rp, ci = _ring(n, k, n)
    assert_same(gpu_count(ni, rp, ci), oracle.count(rp, ci), f"ring {n}, {k}")
