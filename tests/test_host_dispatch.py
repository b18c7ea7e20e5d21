"""The built-in rules that choose a size class's team, on the CPU (fakes of the CUDA calls).

Sizes of the rules' own making must run on whatever the GPU reports it can hold; sizes that a
caller asks for are reported when they cannot.
"""
import ctypes

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
