"""The one-warp kernel on molecule sizes and beams (GPU, against the oracle).

Small batches of K >= 64 take CTA teams unless few SMs are theirs, so these run under
max_sms = 1, where batches of this size keep one warp each (asserted on the plan: CTAs of 128
threads, which CTA teams of K > 32 never have by themselves). Both the normal and the
bounds-checked library; in the latter a selection list declared too short must be reported.
Costs, maps and evaluation counts are whole numbers: equality.
"""
import numpy as np
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
    yield request.param
    F._LIB = saved


def _with(w, **fields):
    for k, v in fields.items():
        setattr(w, k, v)
    return w


def _labelled(n_pairs, max_label):
    w = W.config2(n_pairs, seed=17)
    st = W.Stream(17, 99)
    for g in w.graphs:
        g.elabel = st.randint(0, max_label, g.m).astype(np.int32)
    return w


def _unlabelled(n_pairs):
    w = W.config2(n_pairs, seed=18)
    for g in w.graphs:
        g.elabel = None
    return w


def _limits():
    """PEDs above 2^15, the highest a single-word pair may have is below 2^16."""
    pairs = []
    for k in range(24):
        st = W.Stream(31, k)
        big, small = W.molecule_like(st, 39), W.molecule_like(st, 5 + k % 4)
        pairs += [(big, small), (small, big)]
    return single(pairs, (1000, 1200, 0, 250, 300, 0), 100)


CASES = {
    "setting1": lambda: (W.config2(300), {}),
    "full_beam": lambda: (_with(W.config2(200), K=128), {}),
    "window_2": lambda: (W.config2(120), {"hist_window": 2}),
    "window_17": lambda: (W.config2(120), {"hist_window": 17}),
    "setting2": lambda: (_with(W.config2(120), cost=W.SETTING2_COSTS), {}),
    "large_costs": lambda: (_with(W.config2(120), cost=(100, 301, 299, 70, 150, 91)), {}),
    "ped_limits": lambda: (_limits(), {}),
    "per_pair_k": lambda: (_with(W.config2(150), k_per_pair=W.Stream(31, 2).randint(1, 100, 150).astype(np.int32)), {}),
    "variant_b": lambda: (W.config2(120), {"variant": 1}),
    "degree_order": lambda: (W.config2(120), {"vertex_order": F.FASTGED_ORDER_DEGREE}),
    "unlabelled": lambda: (_unlabelled(100), {}),
    "eight_planes": lambda: (_labelled(120, 6), {}),
}


def _on_warps(w, **opts):
    mm = F.marshal(w)
    with F.FastGED(w.cost) as g:
        plan = F.fastged_plan_create(g.h, mm, w.K, F.make_options(max_sms=1, k_per_pair=w.k_per_pair, **opts))
        threads = F.fastged_plan_info(plan)["block_threads"]
        F.fastged_plan_destroy(plan)
    return set(threads) == {128}


@pytest.mark.parametrize("name", sorted(CASES))
def test_one_warp_teams_match_oracle(name):
    w, opts = CASES[name]()
    assert _on_warps(w, **opts)
    assert_parity(w, gpu_run(w, max_sms=1, **opts), variant=opts.get("variant", 0),
                  order=1 if opts.get("vertex_order") else 0)


def test_one_warp_teams_report_an_index_past_its_array(library, monkeypatch):
    if library != "checked":
        pytest.skip("the bounds checks are in the checked library")
    w = W.config2(120)
    assert _on_warps(w)
    monkeypatch.setenv("FASTGED_CHECK_SHRINK_SEL", "1")
    with pytest.raises(F.FastGEDError) as ei:
        gpu_run(w, max_sms=1)
    assert ei.value.code == F.FASTGED_ERR_CUDA and "bounds check" in str(ei.value)
    monkeypatch.delenv("FASTGED_CHECK_SHRINK_SEL")
    assert_parity(w, gpu_run(w, max_sms=1))
