"""Malformed CSR input through the device entry points: the error is reported,
nothing is touched out of range, and the next call on the stream is right."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_parity import assert_same, gpu_count, ni, tuning  # noqa: F401 (fixtures)
from test_zz_no_alloc import _run, lib  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _rows_that_overlap(n, m):
    """Offsets 0, m, 0, m, ...: every other row is in range and holds all m
    entries, so that the degrees sum to about n m / 2."""
    rp = np.zeros(n + 1, np.int32)
    rp[1::2] = m
    rp[n] = m
    return rp, (np.arange(m) % n).astype(np.int32)


@pytest.mark.parametrize("n,m", [(3, 2), (1501, 6000), (2048, 40000),   # one tile of vertices
                                 (2049, 9000), (30000, 120000),        # several
                                 (6000, 1 << 20)])                      # the sum passes 2^31
def test_overlapping_rows_stop_the_call(ni, lib, n, m):  # noqa: F811
    from paper_2606_29651_gb300 import Status
    rp, ci = _rows_that_overlap(n, m)
    dev = torch.device("cuda:0")
    a, b = torch.from_numpy(rp).to(dev), torch.from_numpy(ci).to(dev)
    ni.last_status()
    for call in (ni.count, ni.count_induced):
        call(a, b)
        assert ni.last_status() == Status.EINVAL
    ni.count_batch(a, b, torch.tensor([0, n], device=dev), torch.tensor([0, m], device=dev))
    assert ni.last_status() == Status.EINVAL
    ha, hb = a.cpu().pin_memory(), b.cpu().pin_memory()
    hout = ni.count_host(ha, hb)
    assert hout.shape == (n, 15)
    assert ni.last_status() == Status.EINVAL
    # the rows are not looked at: their loops and repeats are not reported
    status = torch.full((1,), 7, dtype=torch.int32, device=dev)
    _run(lib, "noalloc", rp, ci, status)
    assert int(status.item()) == 1 << Status.EINVAL
    good = gg.rmat(10, 8, seed=2)
    assert_same(gpu_count(ni, *good), oracle.count(*good), "the next call")


def test_too_many_in_neighbours_are_reported(ni):  # noqa: F811
    # 60 rows of 2000 entries whose vertices do not list them back: roots of
    # the key-tiled 4-cycle tier with more in-entries than half of the CSR
    from paper_2606_29651_gb300 import Status
    n, hubs = 6000, 60
    rp = np.concatenate([np.zeros(n - hubs + 1, np.int32), 2000 * np.arange(1, hubs + 1, dtype=np.int32)])
    ci = np.tile(np.arange(0, 4000, 2, dtype=np.int32), hubs)
    dev = torch.device("cuda:0")
    ni.last_status()
    ni.count(torch.from_numpy(rp).to(dev), torch.from_numpy(ci).to(dev))
    assert ni.last_status() == Status.ENOTSIMPLE


def _graph(kind):
    if kind == "hubs":      # bitmap, filter, key-tiled tier with one group
        return gg.rmat(14, 16, seed=5)
    if kind == "random":    # streamed rows, filter
        return gg.er_mean_degree(20000, 30, 6)
    if kind == "groups":    # key-tiled tier with several groups (all roots sent there)
        return gg.er_mean_degree(600000, 14, 7)
    return gg.er(1501, 0.3, 8)   # dense: bitmap of every row


def _spoil(how, rp, ci, seed):
    """A copy of the columns with rows spoilt, and the status that reports it."""
    from paper_2606_29651_gb300 import Status
    rng = np.random.default_rng(seed)
    ci, d = ci.copy(), np.diff(rp)
    rows = np.argsort(d)[::-1][:200].tolist() + rng.choice(np.flatnonzero(d > 1), 2000).tolist()
    if how == "anything":
        ci[:] = rng.integers(0, len(rp) - 1, len(ci))
        return ci, Status.ENOTSIMPLE
    for x in dict.fromkeys(rows):
        a, b = int(rp[x]), int(rp[x + 1])
        if how == "reversed":
            ci[a:b] = ci[a:b][::-1]
        elif how == "shuffled":
            ci[a:b] = rng.permutation(ci[a:b])
        elif how == "repeated":
            ci[a:b] = ci[a]
        elif how == "loops":   # (a row of n loops is n^3 triangles and K4s: short ones only)
            ci[a:min(b, a + 60)] = x
        else:
            ci[a + int(rng.integers(0, b - a))] = rng.choice([-1, len(rp) - 1, len(rp) + 5, 2**31 - 1, -2**31])
    return ci, Status.EINVAL if how == "out of range" else Status.ENOTSIMPLE


@pytest.mark.parametrize("kind", ["hubs", "random", "groups", "dense"])
@pytest.mark.parametrize("how", ["reversed", "shuffled", "repeated", "loops", "out of range", "anything"])
def test_malformed_rows_in_large_graphs(tuning, kind, how):  # noqa: F811
    rp, ci = _graph(kind)
    bad, status = _spoil(how, rp, ci, 9)
    dev = torch.device("cuda:0")
    a, b = torch.from_numpy(rp).to(dev), torch.from_numpy(bad).to(dev)
    if kind == "groups":
        tuning.set_tuning(c4_warp_maxw=2, c4_team_minw=2)
    tuning.last_status()
    tuning.count(a, b)
    assert tuning.last_status() == status
    tuning.count_host(*(keep := [a.cpu().pin_memory(), b.cpu().pin_memory()]))
    assert tuning.last_status() == status and len(keep) == 2
    good = gg.rmat(10, 8, seed=2)
    assert_same(gpu_count(tuning, *good), oracle.count(*good), "the next call")
