"""Large sparse pairs scored from rows of neighbour counts (GPU, against the oracle).

Targets of eight and more words, no edge labels, at most eight prior neighbours per source vertex
in the mean, no degree above 127: both sides of each bound, the two-term costs (insertion and
deletion of an edge differ) beside the folded ones, the exact selection after such a pass (a
window of 2 sends every level there), target sizes around the words and around the eight
columns of a lane, and labelled and unlabelled pairs in one batch. One-CTA and cluster teams.
Costs, maps and evaluation counts are whole numbers: equality.
"""
import numpy as np
import pytest

from paper_2605_00830_gb300 import build as B
from paper_2605_00830_gb300 import fastged as F
from paper_2605_00830_gb300 import workloads as W
from parity_util import assert_parity, gpu_run, single

pytestmark = pytest.mark.gpu

UNFOLDED = (2, 4, 3, 1, 5, 2)   # an inserted edge costs 2, a deleted one 5


@pytest.fixture(scope="module", params=["normal", "checked"], autouse=True)
def library(request):
    saved = F._LIB
    F._LIB = F.load(B.build(checked=request.param == "checked"))
    yield
    F._LIB = saved


def _sparse(seed, n, m, labels=4):
    """n vertices, m distinct random edges."""
    st = W.Stream(n, seed)
    key = np.unique(st.randint(0, n * n - 1, 3 * m + 64))
    u, v = key // n, key % n
    e = np.stack([u, v], 1)[u < v]
    e = e[np.argsort(st.uniform(len(e)), kind="stable")][:m]
    assert len(e) == m
    return W.Graph(n, st.randint(0, labels - 1, n).astype(np.int32), e.astype(np.int32))


def _star(n, degree, hub):
    """A hub with `degree` leaves (the lowest other ids), the other vertices isolated."""
    leaves = [v for v in range(n) if v != hub][:degree]
    return W.Graph(n, np.arange(n, dtype=np.int32) % 3,
                   np.array([(min(hub, v), max(hub, v)) for v in leaves], np.int32))


def _check(w, **opts):
    for cluster in (1, 4):
        assert_parity(w, gpu_run(w, cluster=cluster, **opts))


@pytest.mark.parametrize("window", [0, 2])
@pytest.mark.parametrize("cost", [W.SETTING1_COSTS, UNFOLDED], ids=["folded", "unfolded"])
@pytest.mark.parametrize("n2", [257, 511, 512, 513, 520, 1023, 1024])
def test_target_sizes(n2, cost, window):
    w = single([(_sparse(1, 40, 70), _sparse(2, n2, 2 * n2))], cost, 60)
    _check(w, hist_window=window)


@pytest.mark.parametrize("scale", [1, 40])
def test_whole_searches_with_two_term_costs(scale):
    pairs = [(_sparse(k, 150, 300), _sparse(k + 9, 280 + 3 * k, 600)) for k in range(3)]
    _check(single(pairs, tuple(scale * c for c in UNFOLDED), 50))


@pytest.mark.parametrize("cost", [W.UNIT_COSTS, UNFOLDED], ids=["folded", "unfolded"])
@pytest.mark.parametrize("degree", [127, 128])
@pytest.mark.parametrize("hub_last", [False, True])
def test_degree_bounds(degree, hub_last, cost):
    """Hubs of 127 neighbours are the highest counts a byte has to hold (127 in the image and
    127 among the prior neighbours' images); 128 goes back to the popcounts."""
    n = 150
    s, t = _star(n, degree, n - 1 if hub_last else 0), _star(300, degree, 299 if hub_last else 0)
    other = _star(300, 127, 140)
    _check(single([(s, t), (s, other), (_star(n, 127, n - 1), t)], cost, 30))


@pytest.mark.parametrize("extra", [0, 1])
def test_mean_degree_bound(extra):
    w = single([(_sparse(3, 40, 320 + extra), _sparse(4, 270, 500))], W.UNIT_COSTS, 50)
    _check(w)


@pytest.mark.parametrize("window", [0, 2])
def test_labelled_and_unlabelled_pairs_in_one_batch(window):
    plain, lab = ([(_sparse(10 + k, 60, 110), _sparse(20 + k, 300 + 250 * (k % 2), 700)) for k in range(3)]
                  for _ in range(2))
    st = W.Stream(3, 3)
    for a, b in lab:
        for g in (a, b):
            g.elabel = st.randint(0, 2, g.m).astype(np.int32)
    zero = [(_sparse(30, 60, 110), _sparse(31, 300, 700))]   # labels that are all 0 count as none
    for g in zero[0]:
        g.elabel = np.zeros(g.m, np.int32)
    _check(single(plain + lab + zero, W.SETTING1_COSTS, 40), hist_window=window)
