"""The built-in rules that choose a size class's team, on the CPU (fakes of the CUDA calls).

Sizes of the rules' own making must run on whatever the GPU reports it can hold; sizes that a
caller asks for are reported when they cannot.
"""
import ctypes

import numpy as np
import pytest

from host_probe import load
from paper_2605_00830_gb300 import fastged as F
from paper_2605_00830_gb300 import workloads as W
from test_host_tuning import _probe_classes


@pytest.fixture
def lib():
    L = load()
    L.fastged_autotune_clear()
    L.fake_set_shape_ms(0, 0, 0.0)
    yield L
    L.fake_set_max_cluster(16, 0)
    L.fastged_autotune_clear()


@pytest.mark.parametrize("error", [0, 1])
@pytest.mark.parametrize("fits", [16, 8, 4, 2, 1])
def test_a_cluster_of_the_rule_that_does_not_fit_is_halved(lib, fits, error):
    w = W.config4(3, n_range=(600, 700))       # the rule takes 16 CTAs for K = 5000
    lib.fake_set_max_cluster(fits, error)
    cls = _probe_classes(lib, w, 5000, full=True)
    assert [c["cluster"] for c in cls] == [fits] * len(cls)
    for c in cls:
        assert c["grid"] == min((152 if fits > 1 else 304) // fits, c["n_order"]) * fits


def test_a_cluster_asked_for_is_refused_when_it_does_not_fit(lib):
    w = W.config4(3, n_range=(600, 700))
    lib.fake_set_max_cluster(8, 0)
    c = (ctypes.c_int32 * 6)(*w.cost)
    mm = F.Marshalled(w.graphs, w.pairs)
    o = F.make_options(team=F.FASTGED_TEAM_CTA, cluster=16)
    assert lib.probe_flatten(ctypes.addressof(mm.pl), 5000, ctypes.addressof(o), c) == F.FASTGED_ERR_CUDA


@pytest.mark.parametrize("max_sms,cluster,grid", [(0, 16, 48), (152, 16, 48), (48, 16, 48),
                                                  (47, 8, 24), (16, 8, 16), (8, 8, 8), (4, 8, 8)])
def test_sixteen_ctas_per_pair_stay_within_the_cap(lib, max_sms, cluster, grid):
    """Three pairs of one class; the sizes of eight CTAs and less are the rule's for any cap."""
    w = W.config4(3, n_range=(600, 700))
    (c,) = _probe_classes(lib, w, 1024, full=True, max_sms=max_sms)
    assert (c["cluster"], c["grid"]) == (cluster, grid)


def _paths(sizes, n_pad=0):
    """Pairs of equal path graphs of the given sizes, and n_pad pairs of 70-vertex ones."""
    g = [W.Graph(n, np.zeros(n, np.int32), np.stack([np.arange(n - 1), np.arange(1, n)], 1).astype(np.int32))
         for n in list(sizes) + [70] * n_pad]
    return W.Workload("paths", g, np.repeat(np.arange(len(g), dtype=np.int32), 2).reshape(-1, 2),
                      W.UNIT_COSTS, 128)


def _warps(lib, w, K, **opts):
    """Whether the batch's single-word class of at most 31 target vertices takes one-warp teams."""
    cls = _probe_classes(lib, w, K, team=F.FASTGED_TEAM_AUTO, full=True, **opts)
    (c,) = [c for c in cls if c["n2max"] <= 31]
    return bool(c["warp"])


# one CTA per pair while the largest gain of a pair, (K - 32) n1 (n2 + 1), is at least
# 12,000 + 380 levels per SM; by hand for the 152 SMs of the fakes
@pytest.mark.parametrize("n,K,opts,most", [
    (20, 100, {}, 331),                  # 68 * 420 = 28,560: 16,560 * 152 / (380 * 20) = 331.2
    (20, 64, {}, 28),                    # 32 * 420 = 13,440:  1,440 * 152 / 7,600 = 28.8
    (20, 63, {}, 0), (15, 128, {}, 0),   # below 64 nodes or 16 source vertices: never
    (31, 128, {}, 1073),                 # 96 * 992 = 95,232: 83,232 * 152 / 11,780 = 1,073.9
    (20, 100, {"max_sms": 10}, 54),      # 25 SMs: 16,560 * 25 / 7,600 = 54.5
    (20, 100, {"max_sms": 1}, 5),        # 2.5 SMs: 5.4
    (20, 100, {"max_sms": 100}, 331)])   # 250 SMs: no more than there are
def test_few_pairs_take_a_cta_each(lib, n, K, opts, most):
    if most:
        assert not _warps(lib, _paths([n] * most), K, **opts)
    assert _warps(lib, _paths([n] * (most + 1)), K, **opts)


def test_the_largest_gain_decides_and_the_batch_bounds_it(lib):
    # 100 pairs, 2,000 levels: 12,000 + 5,000. One K = 64 among K = 32 gains 13,440, one K = 100
    # 28,560
    w = _paths([20] * 100)
    for top, warps in ((32, True), (64, True), (100, False)):
        kpp = np.full(100, 32, np.int32)
        kpp[57] = top
        assert _warps(lib, w, 128, k_per_pair=kpp) == warps
    # batches of more than 8 * 152 pairs keep their one-warp classes
    for pad, warps in ((1116, False), (1117, True)):
        assert _warps(lib, _paths([20] * 100, pad), 100) == warps
