"""Every kernel is traced under its own name."""
import pytest

import graphgen as gg
from test_gpu_parity import ni  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,first", [(4000, "k_c4_warp"), (8000, "k_c4_filter")])
def test_first_four_cycle_kernel(ni, n, first):  # noqa: F811
    # up to 32 vertices a multiprocessor (152: 4864) the tables come first
    rp, ci = gg.er_mean_degree(n, 10, 3)
    dev = torch.device("cuda:0")
    a, b = torch.from_numpy(rp).to(dev), torch.from_numpy(ci).to(dev)
    torch.cuda.synchronize()
    ni.profile_reset()
    ni.profile_enable(True)
    try:
        ni.count(a, b)
        torch.cuda.synchronize()
    finally:
        ni.profile_enable(False)
    launched = {k for k, v in ni.profile_read().items() if v[1] > 0}
    ni.check()
    assert launched & {"k_c4_warp", "k_c4_filter"} == {first}
    assert ("k_c4_warp_left" in launched) == (first == "k_c4_filter")
