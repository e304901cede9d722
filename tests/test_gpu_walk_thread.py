"""The two forms of a walk on the GPU, against the oracle: small batches walk
one probe per thread in a single launch, larger ones (or any batch when
PV_OPT_WALK_TAIL_HOP names a hop) are regrouped by switch.  The other walk
tests use small batches, so here the regrouped form runs their inputs, and
the thread form runs at the edges of its grid and at the batch size where
the library changes over."""
import numpy as np
import pytest
import torch

import oracle
import test_gpu_policies as TP
import test_gpu_walk as TW
from paper_2602_16100_gb300 import binding as B
from paper_2602_16100_gb300 import workloads as W
from paper_2602_16100_gb300.validator import empty_device, to_device, to_numpy
from netbuild import ip, make_net, rule

pytestmark = pytest.mark.gpu

THREAD_WALK_MAX = 1 << 20   # kThreadWalkMax of the library
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1


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


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_regrouped_index_stress_tables(regrouped, seed):
    TW.test_index_stress_tables(regrouped, seed)


def test_regrouped_long_destination_runs(regrouped):
    TW.test_long_destination_runs_split_into_segments(regrouped)


def test_regrouped_forwarding_cycles(regrouped):
    TW.test_forwarding_cycles_finish_with_the_full_walk_result(regrouped)


def test_regrouped_bounces_on_asymmetric_cabling(regrouped):
    TW.test_bounces_on_asymmetric_cabling_are_walked_out(regrouped)


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


@pytest.mark.parametrize("m", [1, 31, 33, 65, SMS * 256 - 1, SMS * 256, SMS * 256 + 1])
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


def _deep_net(n):
    """Three switches in a line, two hosts each.  n rules of one port bucket at
    every switch, each for one source address above every host's or for one
    port of the hosts (so that the candidate filter keeps most of them), a run
    of destination rules in their midst and the routes below them."""
    hosts = [(s, h, ip(10, s, h, 1)) for s in range(3) for h in range(2)]
    tables = []
    for s in range(3):
        t = [rule(1000, hosts[0][2], 32, W.DROP, src_ip=0xF0000000 + i, src_len=32, lo=0, hi=255) for i in range(n)]
        for i, r in enumerate(t):
            r["priority"] = 40000 - 2 * i
            r["action"] = i % 4 if i % 5 else W.DROP
            r["dst_len"] = 0 if i % 2 else 32
            if i % 3 == 0:      # and one port of any host
                r["src_ip"], r["src_len"], r["dst_len"], r["dport_lo"], r["dport_hi"] = ip(10, 0, 0, 0), 8, 0, i % 251, i % 251
        mid = [rule(40001 - n, ip(99, k, 0, 0), 16, 2 if k % 2 else 3) for k in range(7)]
        low = [rule(100, a, 32, h if s2 == s else 3 if s2 > s else 2) for s2, h, a in hosts] + [rule(1, 0, 0, 3)]
        tables.append(t + mid + low)
    return make_net([4] * 3, [(0, 3, 1, 2), (1, 3, 2, 2)], hosts, [0, 1, 2], tables)


def _deep_probes(net, n, m, seed):
    """Sources of rules at both sides of a lane's and a warp's steps, at the end, of none; a third past the bucket."""
    r = np.random.default_rng(seed)
    depth = np.unique(np.clip([0, 1, 15, 16, 17, 31, 32, 33, 63, 64, n // 2 - 1, n // 2, n - 2, n - 1, n], 0, n))
    pr = np.zeros(m, W.PROBE_DTYPE)
    pr["src_ip"] = np.where(r.random(m) < 0.7, 0xF0000000 + r.choice(depth, m), 0xF0000000 + r.integers(0, n + 9, m))
    dst = np.concatenate([net.host_ip, [ip(99, k, 3, 3) for k in range(8)], [5]]).astype(np.uint32)
    pr["dst_ip"] = r.choice(dst, m)
    pr["src_host"] = r.integers(0, net.num_hosts + 1, m)
    pr["dport"] = np.where(r.random(m) < 0.7, r.integers(0, 256, m), r.integers(0, 65536, m))
    pr["allowed_mask"] = np.where(r.random(m) < 0.8, 7, r.integers(0, 8, m))
    return pr


@pytest.mark.parametrize("n,m", [(95, 3000), (96, 1), (96, 3001), (97, 1 << 17), (97, (1 << 17) + 1), (255, 140_000),
                                 (256, 140_000), (300, 1500), (2999, 700), (3000, 701), (6000, 900)])
def test_long_candidate_lists(validator, n, m):
    """Lists past what a lane tests alone: every depth of the match, interval
    searches behind it, both sides of the rules on list length and batch size;
    visit counts add up and no first match differs from a plain scan's."""
    net = _deep_net(n)
    pr = _deep_probes(net, n, m, n + m)
    idx = np.arange(0, m, 1 + m // 20000)
    o = oracle.verify_probes(net, pr[idx], 20)
    validator.set_option(B.PV_OPT_WALK_CYCLES, 1)
    try:
        g = TW._gpu_walk(validator, net, pr, 20, 2)
        assert (g[idx] == o).all()
        ran = g["status"] != W.ST_NOSRC
        want = int(g["hops"][ran].astype(np.int64).sum()) - int((g["status"] == W.ST_VIOLATION).sum())
        assert B.pv_get_stat(validator.ctx, B.PV_STAT_WALK_LIVE_TOTAL) == want
        validator.set_option(B.PV_OPT_WALK_STATS, 1)
        assert (TW._gpu_walk(validator, net, pr, 20, 2) == g).all()
        assert B.pv_get_stat(validator.ctx, B.PV_STAT_WALK_INDEX_MISMATCHES) == 0
    finally:
        validator.set_option(B.PV_OPT_WALK_CYCLES, 0)
        validator.set_option(B.PV_OPT_WALK_STATS, 0)


@pytest.mark.parametrize("n", [95, 96, 700])
@pytest.mark.parametrize("policies", [False, True])
def test_long_candidate_lists_regrouped_and_flows(validator, n, policies):
    """The same lists in a regrouped walk's last hops (most blocks with no
    probe left) and for compact flows, with and without path policies."""
    v, net, ppg, groups = validator, _deep_net(n), 40, 30
    m = ppg * groups
    pr = _deep_probes(net, n, m, n)
    v.load_network(net)
    pol = W.PathPolicies(1, np.array([0, 1], np.uint32), np.array([1], np.uint16), np.array([0, 2], np.uint32),
                         np.array([0, 2], np.uint16), np.ones(1, np.uint8)) if policies else None
    if policies:
        v.load_policies(pol)
    r = np.random.default_rng(n)
    assign = r.integers(0, net.num_hosts + 1, groups).astype(np.uint32)
    masks = r.choice([7, 7, 5, 3], groups).astype(np.uint32)
    flows = pr.copy()
    flows["allowed_mask"] = np.repeat(masks, ppg)
    bound = oracle.bind_probes(flows, ppg, 1, assign, net.host_ip)
    d = v.device
    for tail in (-1, 1, 2):
        v.set_option(B.PV_OPT_WALK_TAIL_HOP, tail)
        try:
            for form, x in (("probes", pr), ("flows", bound)):
                out, hits = empty_device(4 * m, d), empty_device(4 * m, d)
                if form == "probes" and policies:
                    B.pv_verify_probes_constrained(v.ctx, m, to_device(x, d), 20, None, m, out, hits)
                elif form == "probes":
                    B.pv_verify_probes(v.ctx, m, to_device(x, d), 20, out)
                else:
                    cols = [to_device(np.ascontiguousarray(pr[f]), d) for f in ("dst_ip", "dport")]
                    a = (v.ctx, m, *cols, ppg, 1, to_device(assign, d), to_device(masks, d), 20)
                    if policies:
                        B.pv_verify_flow_columns_constrained(*a, None, m, 0, None, out, hits)
                    else:
                        B.pv_verify_flow_columns(*a, None, out)
                v.sync()
                if policies:
                    want, oh = oracle.verify_constrained(net, x, 20, pol, probes_per_policy=m)
                    assert (to_numpy(hits, np.uint32) == oh).all(), (tail, form)
                else:
                    want = oracle.verify_probes(net, x, 20)
                assert (to_numpy(out, W.RESULT_DTYPE) == want).all(), (tail, form)
        finally:
            v.set_option(B.PV_OPT_WALK_TAIL_HOP, -1)
