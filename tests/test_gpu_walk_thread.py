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
from netbuild import make_net

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


def _scattered_net(seed, n, hosts, wide):
    """Four switches in a ring, n random rules each: prefixes of every length
    0-32 of host and of arbitrary addresses, ports all `wide` or of mixed
    widths; `hosts` hosts at addresses scattered over the whole range."""
    r = np.random.default_rng(seed)
    ips = np.unique(np.concatenate([[0, 0xFFFFFFFF], r.integers(0, 1 << 32, hosts)]))[:hosts] if hosts > 2 else \
        r.integers(0, 1 << 32, hosts)
    t = np.zeros((4, n), W.RULE_DTYPE)
    t["priority"] = r.integers(0, 50, t.shape)            # many ties
    t["in_port"] = np.where(r.random(t.shape) < 0.5, W.ANY_PORT, r.integers(0, 4, t.shape))
    for a, ln in (("src_ip", "src_len"), ("dst_ip", "dst_len")):
        t[a] = np.where(r.random(t.shape) < 0.8, r.choice(ips, t.shape), r.integers(0, 1 << 32, t.shape))
        t[ln] = r.integers(0, 33, t.shape)
    t["src_len"] = np.where(r.random(t.shape) < 0.5, 0, t["src_len"])
    t["dport_lo"] = 0 if wide else r.integers(0, 65536, t.shape)
    t["dport_hi"] = 65535 if wide else np.minimum(65535, t["dport_lo"].astype(np.int64)
                                                  + (1 << r.integers(0, 17, t.shape)) - 1)
    if wide:
        t["in_port"] = np.where(t["src_len"] == 0, r.integers(0, 4, t.shape), t["in_port"])   # no segments
    t["action"] = np.where(r.random(t.shape) < 0.1, W.DROP, r.integers(0, 4, t.shape))
    nets = make_net([4] * 4, [(i, 2, (i + 1) % 4, 3) for i in range(4)], [(i % 4, i // 4 % 2, int(x)) for i, x in enumerate(ips)],
                    [0, 1, 2, 3], [[x.reshape(1) for x in t[s]] for s in range(4)])
    return nets


@pytest.mark.parametrize("n,hosts,wide,lane_max", [(40, 2, False, 96), (40, 8, False, 0), (200, 8, False, 96),
                                                   (600, 8, False, 65535), (31, 8, True, 96), (32, 8, True, 96),
                                                   (33, 8, True, 96), (65, 8, True, 96), (400, 8, True, 65535),
                                                   (400, 8, True, 96)])
@pytest.mark.parametrize("tail", [-1, 0])
def test_candidate_filter(validator, n, hosts, wide, lane_max, tail):
    """The filter of the first-match index: addresses at class boundaries and
    at both ends of the range, prefixes of every length, lists of 31 to 400
    candidates (one and several per filter bit), fewer hosts than classes,
    and tables whose filter does not fit the hop kernel's stage (400 rules of
    every port: 205 KB of items)."""
    net = _scattered_net(n + hosts, n, hosts, wide)
    r = np.random.default_rng(n)
    m = 3000
    pr = np.zeros(m, W.PROBE_DTYPE)
    ends = np.concatenate([net.host_ip, net.host_ip - np.uint32(1), net.host_ip + np.uint32(1)])
    for f in ("src_ip", "dst_ip"):
        pr[f] = np.where(r.random(m) < 0.8, r.choice(ends, m), r.integers(0, 1 << 32, m))
    pr["src_host"] = r.integers(0, hosts, m)
    pr["dport"] = r.integers(0, 65536, m)
    pr["allowed_mask"] = r.integers(1, 16, m)
    validator.set_option(B.PV_OPT_WALK_TAIL_HOP, tail)
    validator.set_option(B.PV_OPT_WALK_LANE_MAX, lane_max)
    validator.set_option(B.PV_OPT_WALK_STATS, 1)
    try:
        g = TW._gpu_walk(validator, net, pr, 20, 2)
        assert B.pv_get_stat(validator.ctx, B.PV_STAT_WALK_INDEX_MISMATCHES) == 0
        validator.set_option(B.PV_OPT_WALK_STATS, 0)
        g2 = TW._gpu_walk(validator, net, pr, 20, 2)
    finally:
        for o, x in ((B.PV_OPT_WALK_TAIL_HOP, -1), (B.PV_OPT_WALK_LANE_MAX, 96), (B.PV_OPT_WALK_STATS, 0)):
            validator.set_option(o, x)
    o = oracle.verify_probes(net, pr, 20)
    assert (g == o).all() and (g2 == o).all()
