"""Cluster teams at levels with fewer nodes than CTAs, in the exact selection (GPU, oracle).

A CTA without nodes has no column list at such a level. Targets that fill their bitset words
(128, 256, 512, 1024 vertices) and one vertex less; beams of one node (every level has idle
CTAs) and beams wider than the target (level 0 keeps more than 31 PEDs when a deletion costs 40
more than a substitution, or lies past the 127 offsets of a score byte when every vertex label
differs). Both the normal and the bounds-checked library. Costs, maps and evaluation counts are
whole numbers: equality.
"""
import pytest

from paper_2605_00830_gb300 import build as B
from paper_2605_00830_gb300 import fastged as F
from paper_2605_00830_gb300 import workloads as W
from parity_util import assert_parity, gpu_run, single

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["normal", "checked"], autouse=True)
def library(request):
    saved = F._LIB
    F._LIB = F.load(B.build(checked=request.param == "checked"))
    yield
    F._LIB = saved


# vertex costs: a wide first level, and one past the score bytes' window (labels of the two
# graphs are disjoint there)
WIDE = (2, 42, 4, 1, 2, 2)
FAR = (200, 300, 4, 150, 160, 170)


@pytest.mark.parametrize("cost", [WIDE, FAR], ids=["wide", "far"])
@pytest.mark.parametrize("n2", [127, 128, 255, 256, 511, 512, 1024])
@pytest.mark.parametrize("labelled", [False, True])
def test_idle_ctas_in_the_exact_selection(n2, labelled, cost):
    st = W.Stream(n2, 11)
    g1, g2 = W.erdos_renyi(st, 6, 0.5, 3), W.erdos_renyi(st, n2, 3.0 / n2, 3)
    if cost is FAR:
        g2.vlabel = g2.vlabel + 10
    if labelled:
        for g in (g1, g2):
            g.elabel = st.randint(0, 2, g.m).astype("int32")
    # two-word pairs take clusters from 2^14 successors of a level on
    for K in ((n2 + 40,) if n2 <= 128 else (1, n2 + 40)):
        w = single([(g1, g2)], cost, K)
        for cluster in (2, 16):
            assert_parity(w, gpu_run(w, cluster=cluster))
