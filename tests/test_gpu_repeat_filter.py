"""4-cycle roots that a Bloom filter of their keys settles without a count
table: in-neighbour counts around 8, 32 and 64, numbers of repeated keys
around what the filter's lists hold, rows past one step of the walk, and
wedge counts around its limits, with packed and with split tables behind it.
Integers: exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_parity import assert_same, gpu_count, ni, tuning  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HUBS, HUB_LEAVES = 60, 200


def _roots(specs, n, seed):
    """For every (D, r, L) a vertex u, above its D neighbours v in the degree
    order (it is joined to all hubs), whose r repeated keys are joined to two
    or three of the v each, and whose v have L further neighbours each."""
    rng = np.random.default_rng(seed)
    edges, top = [], HUBS
    for h in range(HUBS):
        edges += [(h, top + i) for i in range(HUB_LEAVES)]
        top += HUB_LEAVES
    for d, r, extra in specs:
        u, v, top = top, np.arange(top + 1, top + 1 + d), top + 1 + d
        edges += [(h, u) for h in range(HUBS)] + [(u, x) for x in v]
        for _ in range(r):
            edges += [(x, top) for x in rng.choice(v, size=int(rng.integers(2, min(3, d) + 1)), replace=False)]
            top += 1
        for x in v:
            edges += [(x, top + i) for i in range(extra)]
            top += extra
    for a, b in [(2, 2), (3, 8), (4, 7), (8, 8), (5, 15)]:   # low degrees: few and many repeated keys
        edges += [(top + i, top + a + j) for i in range(a) for j in range(b)]
        top += a + b
    assert top <= n
    return gg.from_edges(n, edges)


@pytest.mark.parametrize("n", [20000, 40000, (1 << 21) + 7])
def test_against_the_oracle(ni, n):  # noqa: F811
    around = [(d, r, 2) for d in (2, 7, 8, 9, 31, 32, 33, 63, 64, 65) for r in (0, 1, 5) if d > 2]
    lists = [(d, r, 1) for d in (8, 40) for r in (15, 16, 17, 31, 32, 33)]
    long_rows = [(4, 1, 31), (4, 2, 32), (9, 1, 33), (33, 2, 17), (12, 0, 49)]
    # W around sqrt(48 n) (979, 1385) and around 1536
    limits = [(40, 2, 24), (40, 3, 25), (40, 5, 34), (40, 2, 35), (48, 0, 32), (51, 3, 30), (64, 1, 24)]
    rp, ci = _roots(around + lists if n == 20000 else lists + long_rows + limits, n, n)
    assert_same(gpu_count(ni, rp, ci), oracle.count(rp, ci), f"n = {n}")


def test_random_graph_equals_the_counting_tiers(tuning):  # noqa: F811
    rp, ci = gg.er_mean_degree(60000, 30, 8)
    got = gpu_count(tuning, rp, ci)
    tuning.set_tuning(c4_warp_maxw=2)
    assert_same(got, gpu_count(tuning, rp, ci), "filter against tables")


@pytest.mark.parametrize("graphs,hi", [(150, 60), (90, 149), (40, 400)])
def test_batch_equals_the_union(ni, graphs, hi):  # noqa: F811
    # more vertices in all than the filter's least; graphs of under and over
    # 150 vertices on average take different kernels
    gs = [gg.er_mean_degree(hi - 5 * (i % 4), 12, i) for i in range(graphs)]
    rp = np.concatenate([[0]] + [np.diff(r) for r, _ in gs]).cumsum()
    v = np.concatenate([[0], np.cumsum([len(r) - 1 for r, _ in gs])])
    e = np.concatenate([[0], np.cumsum([len(c) for _, c in gs])])
    assert v[-1] > 4864
    dev = torch.device("cuda", 0)
    on = lambda a, t: torch.from_numpy(np.ascontiguousarray(a, dtype=t)).to(dev)  # noqa: E731
    out = ni.count_batch(on(rp, np.int32), on(np.concatenate([c for _, c in gs]), np.int32), on(v, np.int64), on(e, np.int64))
    union = np.concatenate([c.astype(np.int64) + v[i] for i, (_, c) in enumerate(gs)]).astype(np.int32)
    assert_same(out.cpu().numpy(), oracle.count(rp.astype(np.int32), union), f"{graphs} graphs of up to {hi}")
