"""Row relabelling at the edges of its forms: rows of up to 64 entries, of up
to 511 (a warp, the first 64 entries kept in registers) and longer ones (a CTA,
a part of the row per warp), with neighbours of many degree classes. Integers:
exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_parity import assert_same, gpu_count, ni, tuning  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _rows(degrees, pool, seed):
    """A vertex of every given degree, joined to random vertices of a pool that
    has edges of its own (degrees 0 to about 40)."""
    rng = np.random.default_rng(seed)
    edges = {(int(a), int(a + 1 + rng.integers(0, 40))) for a in rng.integers(0, pool - 41, 6 * pool // 10) for _ in range(2)}
    for i, d in enumerate(degrees):
        edges |= {(int(v), pool + i) for v in rng.choice(pool, size=d, replace=False)}
    return gg.from_edges(pool + len(degrees), sorted(edges))


@pytest.mark.parametrize("degrees", [
    [63, 64, 65, 66, 95, 96, 97, 127, 128, 129],
    [511, 512, 513, 639, 640, 641, 767, 768, 769],           # parts of 64 and 96 entries, the last ones short
    [1023, 1024, 1025, 1151, 1152, 1153, 8191, 8192, 8193],  # several steps of a part
])
@pytest.mark.parametrize("long_row_class", [32, 20])   # rows from degree 512, 64 on get a CTA
def test_rows_around_the_limits(tuning, degrees, long_row_class):  # noqa: F811
    rp, ci = _rows(degrees, 9000, len(degrees) + degrees[0])
    assert set(degrees) <= set(np.diff(rp).tolist())
    tuning.set_tuning(long_row_class=long_row_class)
    assert_same(gpu_count(tuning, rp, ci), oracle.count(rp, ci), f"{degrees}, {long_row_class}")


@pytest.mark.parametrize("degree,at", [(100, 64), (100, 99), (1000, 1), (1000, 128), (1000, 999), (8192, 1056), (8192, 8191)])
def test_unsorted_entries_are_reported(ni, degree, at):  # noqa: F811
    from paper_2606_29651_gb300 import Status
    rp, ci = _rows([degree], 9000, 1)
    ci = ci.copy()
    p = int(rp[9000]) + at
    ci[[p - 1, p]] = ci[[p, p - 1]]
    dev = torch.device("cuda:0")
    ni.last_status()
    ni.count(torch.from_numpy(rp).to(dev), torch.from_numpy(ci).to(dev))
    assert ni.last_status() == Status.ENOTSIMPLE
