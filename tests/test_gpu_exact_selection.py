"""The exact selection (GPU, against the oracle): kept sets past the histogram window, where the
level is scored again, and over too many of its buckets, where its bytes decide.

Costs of 700-3,001 put nearly every level's kept PEDs thousands apart; a window of 2 sends every
level whose kept set has two PEDs there. One-warp, one-CTA and cluster teams; each word class;
rows of neighbour counts with more prior neighbours than a warp has lanes; beams of one node, of
odd sizes, and past the 2,048 that are ranked instead of sorted. Costs, maps and evaluation counts
are whole numbers: equality.
"""
import numpy as np
import pytest

from paper_2605_00830_gb300 import build as B
from paper_2605_00830_gb300 import fastged as F
from paper_2605_00830_gb300 import workloads as W
from parity_util import assert_parity, gpu_run, single

pytestmark = pytest.mark.gpu

FAR = (1000, 3001, 2999, 700, 1500, 901)
FAR_FOLDED = (1000, 3001, 2999, 700, 1500, 1500)
SMALL_FAR = (100, 301, 299, 70, 150, 91)   # PEDs of molecules below 2^16: single-word teams


@pytest.fixture(scope="module", params=["normal", "checked"], autouse=True)
def library(request):
    saved = F._LIB
    F._LIB = F.load(B.build(checked=request.param == "checked"))
    yield
    F._LIB = saved


def _pairs(n1, n2, p2, labelled, count=2):
    out = []
    for k in range(count):
        st = W.Stream(100 * n2 + k, 12)
        g1, g2 = W.erdos_renyi(st, n1, 0.3, 4), W.erdos_renyi(st, n2, p2, 4)
        if labelled:
            for g in (g1, g2):
                g.elabel = st.randint(0, 2, g.m).astype(np.int32)
        out.append((g1, g2))
    return out


@pytest.mark.parametrize("window", [0, 2])
@pytest.mark.parametrize("cost", [FAR, FAR_FOLDED, SMALL_FAR], ids=["far", "folded", "small"])
@pytest.mark.parametrize("labelled", [False, True])
@pytest.mark.parametrize("n2", [20, 33, 64, 100, 200, 300, 600])
def test_word_classes(n2, labelled, cost, window):
    # 300 and 600 vertices: sparse, so that unlabelled pairs keep rows of counts
    w = single(_pairs(14, n2, 4.0 / n2 if n2 > 256 else 0.2, labelled), cost, 70)
    for opts in ({}, {"team": F.FASTGED_TEAM_CTA, "cluster": 1}, {"team": F.FASTGED_TEAM_CTA, "cluster": 4}):
        assert_parity(w, gpu_run(w, hist_window=window, **opts))


@pytest.mark.parametrize("K", [1, 2, 31, 127, 128, 2047, 2049, 3000])
@pytest.mark.parametrize("n2,window,cost", [(18, 0, SMALL_FAR), (18, 2, W.SETTING1_COSTS),
                                            (70, 0, FAR), (300, 2, W.UNIT_COSTS), (300, 0, FAR)])
def test_beams(n2, window, cost, K):
    w = single(_pairs(9, n2, 4.0 / n2 if n2 > 256 else 0.3, False), cost, K)
    assert_parity(w, gpu_run(w, hist_window=window))


@pytest.mark.parametrize("cost", [FAR, FAR_FOLDED], ids=["unfolded", "folded"])
@pytest.mark.parametrize("leaves", [31, 32, 33, 100, 127])
def test_counts_with_many_prior_neighbours(leaves, cost):
    """The source's last vertex neighbours the first `leaves` ones."""
    n = leaves + 1
    src = W.Graph(n, np.arange(n, dtype=np.int32) % 3,
                  np.stack([np.arange(leaves), np.full(leaves, leaves)], 1).astype(np.int32))
    st = W.Stream(leaves, 13)
    w = single([(src, W.erdos_renyi(st, 290, 0.02, 3))], cost, 20)
    for cluster in (1, 2):
        assert_parity(w, gpu_run(w, cluster=cluster))
