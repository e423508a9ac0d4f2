"""The bench's account of which kernel takes a 4-cycle root first follows the
library's limits: table sizes, the filter's predicate, small graphs, hubs."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402
import graphgen as gg  # noqa: E402


def _padded(rp, ci, n):
    return np.concatenate([rp, np.full(n - len(rp) + 1, rp[-1], rp.dtype)]), ci


@pytest.mark.parametrize("name,make", [
    ("small", lambda: gg.er_mean_degree(2400, 48, 5)),
    ("few", lambda: gg.er_mean_degree(3000, 48, 5)),
    ("packed tables", lambda: gg.er_mean_degree(9000, 50, 6)),
    ("split tables", lambda: _padded(*gg.er_mean_degree(9000, 50, 6), (1 << 21) + 9)),
    ("hubs", lambda: gg.rmat(14, 16, seed=3)),
])
def test_every_root_goes_to_one_kernel(name, make):
    sh = bench.Shape(*make())
    w, routes = sh.w_root, sh.c4_routes()
    live = (sh.din >= 2) & (w >= 2)
    assert (sum(m.astype(int) for m in routes.values()) == live).all(), name
    if name in ("small", "few"):
        limit = 32 if name == "small" else 128
        assert set(routes) == {"k_c4_warp", "k_c4_mid", "k_c4_cta", "k_c4_tiled"}
        assert w[routes["k_c4_warp"]].max() <= limit < w[routes["k_c4_mid"]].min()
        return
    f, left = routes["k_c4_filter"], routes["k_c4_warp_left"]
    assert (w[f] ** 2 <= 48 * sh.n).all() and w[f].max() <= 2048 and sh.din[f].max() <= 64
    table = 768 if name == "split tables" else 1152
    # what the filter may not take goes by the table's limit
    other = live & ~f
    assert (left == (other & (w <= table) & (sh.din <= 1024))).all()
    assert routes["k_c4_tiled"][sh.din > 1024].all() and ((sh.din > 1024).any() or name != "hubs")
    assert w[routes["k_c4_mid"]].max() <= 6144


def test_filter_limit_follows_the_tuning_value():
    sh = bench.Shape(*gg.er_mean_degree(100000, 44, 7))
    w = sh.w_root
    for maxw in (300, 1200, 1536):
        f = sh.c4_routes(maxw)["k_c4_filter"]
        assert w[f].max() <= min(maxw * 4 // 3, int((48 * sh.n) ** 0.5))
        assert w[f].max() > maxw


def test_launched_bytes_sum_to_the_wedges():
    rp, ci = gg.er_mean_degree(20000, 30, 8)
    sh = bench.Shape(rp, ci)
    ab = bench.algorithmic_bytes(rp, ci, shape=sh)
    per = bench.launched_bytes(ab, sh)
    c4 = sum(v for k, v in per.items() if k.startswith("k_c4"))
    assert 0.999 * ab["B_c4"] < c4 <= ab["B_c4"]
    assert per["k_tri_warp"] == ab["per_kernel"]["k_tri_warp"]
