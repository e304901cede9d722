"""The two forms of a walk on the GPU, against the oracle: small batches walk
one probe per thread in a single launch, larger ones (or any batch when
PV_OPT_WALK_TAIL_HOP names a hop) are regrouped by switch.  The other walk
tests use small batches, so here the regrouped form runs their inputs, and
the thread form runs at the edges of its grid and at the batch size where
the library changes over."""
import numpy as np
import pytest

import oracle
import test_gpu_policies as TP
import test_gpu_walk as TW
from paper_2602_16100_gb300 import binding as B
from paper_2602_16100_gb300 import workloads as W

pytestmark = pytest.mark.gpu

THREAD_WALK_MAX = 1 << 20   # kThreadWalkMax of the library


@pytest.fixture(params=[0, 1, 6])
def regrouped(validator, request):
    """The validator with regrouped walks: every hop, or a tail launch from hop 1 or 6."""
    validator.set_option(B.PV_OPT_WALK_TAIL_HOP, request.param)
    yield validator
    validator.set_option(B.PV_OPT_WALK_TAIL_HOP, -1)


@pytest.mark.parametrize("k,rules,cap,mask_all", [(4, 100, 8, True), (8, 600, 32, False), (6, 2000, 255, True)])
def test_regrouped_fat_trees(regrouped, k, rules, cap, mask_all):
    TW.test_fat_trees(regrouped, k, rules, cap, mask_all, 2)


def test_regrouped_random_graph(regrouped):
    TW.test_random_graph_network(regrouped, 2)


@pytest.mark.parametrize("seed,cap", [(1, 32), (2, 3), (3, 255)])
def test_regrouped_policies(regrouped, seed, cap):
    TP.test_random_policies(regrouped, seed, cap, 2)


@pytest.mark.parametrize("form", ["records", "columns"])
@pytest.mark.parametrize("policy_form", ["per_group", "per_probe", "per_pair_of_groups", "none"])
def test_regrouped_flows(regrouped, policy_form, form):
    TP.test_flow_verification_direct_and_regrouped_first_hop_agree(regrouped, policy_form, form)


def _random_sources(net, pr, seed):
    st = W.Stream(seed, "sources")
    pr["src_host"] = st.ints(0, net.num_hosts + 2, len(pr))       # a few out of range
    ok = pr["src_host"] < net.num_hosts
    pr["src_ip"][ok] = net.host_ip[pr["src_host"][ok]]
    return pr


@pytest.mark.parametrize("m", [1, 31, 33, 65, 152 * 256 - 1, 152 * 256, 152 * 256 + 1])
@pytest.mark.parametrize("cycles", [0, 1])
def test_thread_walk_grid_edges(validator, m, cycles):
    """One probe, ragged warps and blocks, and both block sizes; visit counts add up."""
    d = W.fat_tree(seed=11, k=4, rules_per_switch=120, num_probes=m, hop_cap=24)
    net, pr = d["network"], _random_sources(d["network"], d["probes"].probes, m)
    pr["allowed_mask"][::2] = 0xFFFFFFFF
    o = oracle.verify_probes(net, pr, 24)
    validator.set_option(B.PV_OPT_WALK_CYCLES, cycles)
    try:
        g = TW._gpu_walk(validator, net, pr, 24)
    finally:
        validator.set_option(B.PV_OPT_WALK_CYCLES, 0)
    assert (g == o).all()
    ran = o["status"] != W.ST_NOSRC
    want = int(o["hops"][ran].astype(np.int64).sum()) - int((o["status"] == W.ST_VIOLATION).sum())
    total = B.pv_get_stat(validator.ctx, B.PV_STAT_WALK_LIVE_TOTAL)
    assert total == want if cycles else total <= want


@pytest.mark.parametrize("m", [THREAD_WALK_MAX, THREAD_WALK_MAX + 1])
def test_forms_agree_at_the_changeover(validator, m):
    """Each form on both sides of the changeover (lanes of the thread form
    draw several probes each here), the oracle on a sample."""
    e = W.end_to_end(seed=44, num_switches=60, num_intents=1, probes_per_intent=m, rules_per_switch=200)
    net, pr = e.network, _random_sources(e.network, e.probes.probes, 5)
    pr["allowed_mask"] = W.Stream(6, "masks").ints(0, 0xFFFFFFFF, m).astype(np.uint32)
    auto = TW._gpu_walk(validator, net, pr, 32)
    validator.set_option(B.PV_OPT_WALK_TAIL_HOP, 5)
    try:
        regrouped = TW._gpu_walk(validator, net, pr, 32)
    finally:
        validator.set_option(B.PV_OPT_WALK_TAIL_HOP, -1)
    assert (auto == regrouped).all()
    idx = np.arange(0, m, 97)
    assert (auto[idx] == oracle.verify_probes(net, pr[idx], 32)).all()
