"""Sizes where the score bytes and their histogram window can go wrong (GPU, against the oracle).

Columns: target graphs around the chunks of 32 columns and quads of four, and around the words
of a bitset. Nodes: beams around the groups of 32 nodes and the lanes a short group is spread
over. Window: source graphs whose levels start far above the best parent's PED (a clique after
an edgeless part and the reverse), so that the predicted anchor is too low or too high and the
exact selection takes over. Costs, maps and evaluation counts are whole numbers: equality.
"""
import numpy as np
import pytest

from paper_2605_00830_gb300 import fastged as F
from paper_2605_00830_gb300 import workloads as W
from parity_util import assert_parity, gpu_run, single

pytestmark = pytest.mark.gpu


def _labelled(st, n, p):
    g = W.erdos_renyi(st, n, p, 3)
    g.elabel = st.randint(0, 2, g.m).astype(np.int32)
    return g


@pytest.mark.parametrize("n2", [1, 2, 3, 4, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("labelled", [False, True])
def test_column_edges(n2, labelled):
    st = W.Stream(n2, 5)
    make = _labelled if labelled else (lambda s, n, p: W.erdos_renyi(s, n, p, 3))
    w = single([(make(st, 9, 0.4), make(st, n2, 0.3)) for _ in range(3)], W.SETTING1_COSTS, 40)
    assert_parity(w, gpu_run(w, team=F.FASTGED_TEAM_CTA))


@pytest.mark.parametrize("K", [1, 2, 3, 5, 9, 17, 31, 33, 255, 257, 600])
def test_beam_edges(K):
    st = W.Stream(K, 6)
    w = single([(_labelled(st, 10, 0.3), _labelled(st, n, 0.3)) for n in (8, 20, 40, 70)],
               W.SETTING2_COSTS, K)
    assert_parity(w, gpu_run(w, team=F.FASTGED_TEAM_CTA))


def _clique_and_isolated(n, clique_first):
    ids = np.arange(n) if clique_first else np.arange(n)[::-1]
    half = ids[:n // 2]
    e = [(min(a, b), max(a, b)) for x, a in enumerate(half) for b in half[x + 1:]]
    return W.Graph(n, np.arange(n, dtype=np.int32) % 3, np.array(sorted(e), np.int32).reshape(-1, 2))


@pytest.mark.parametrize("cluster", [1, 4])
@pytest.mark.parametrize("clique_first", [False, True])
@pytest.mark.parametrize("scale", [1, 9, 700])
def test_anchor_jumps(cluster, clique_first, scale):
    costs = tuple(scale * c for c in W.SETTING1_COSTS)
    st = W.Stream(scale, 7)
    g1 = _clique_and_isolated(36, clique_first)
    w = single([(g1, W.erdos_renyi(st, 140, 0.3, 3)), (g1, W.erdos_renyi(st, 30, 0.6, 3))], costs, 30)
    assert_parity(w, gpu_run(w, team=F.FASTGED_TEAM_CTA, cluster=cluster))


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n2", [1, 2, 3, 4, 7, 8, 15, 16, 30, 31, 32, 33, 62, 63])
def test_one_warp_column_edges(n2, variant):
    st = W.Stream(n2, 8)
    w = single([(_labelled(st, n1, 0.4), _labelled(st, n2, 0.3)) for n1 in (1, 9, 31)],
               W.SETTING1_COSTS, 40)
    assert_parity(w, gpu_run(w, variant=variant), variant=variant)


@pytest.mark.parametrize("K", [1, 2, 3, 5, 9, 17, 31, 33, 97, 127, 128])
def test_one_warp_beam_edges(K):
    st = W.Stream(K, 9)
    w = single([(_labelled(st, 12, 0.3), _labelled(st, n, 0.3)) for n in (8, 20, 40)],
               W.SETTING2_COSTS, K)
    for window in (0, 2, 17):
        assert_parity(w, gpu_run(w, hist_window=window))


@pytest.mark.parametrize("scale", [1, 9, 120])
def test_one_warp_wide_offsets(scale):
    """PED offsets past the 127 of a score byte, up to the 16 bits a one-warp pair allows."""
    costs = tuple(scale * c for c in W.SETTING1_COSTS)
    st = W.Stream(scale, 10)
    w = single([(_clique_and_isolated(16, f), W.erdos_renyi(st, 25, 0.5, 3)) for f in (False, True)],
               costs, 60)
    for variant in (0, 1):
        assert_parity(w, gpu_run(w, variant=variant), variant=variant)
