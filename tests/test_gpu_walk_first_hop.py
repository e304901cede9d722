"""Regrouped walks of compact flows: the kernels that write the first hop's
records (one block per group from kGroupInitMin flows, whole ranges of probes
otherwise) at the edges of their ranges, against the oracle, and the hop grid
of large batches against the same flows in smaller calls."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_16100_gb300 import binding as B
from paper_2602_16100_gb300 import workloads as W
from paper_2602_16100_gb300.validator import empty_device, to_device, to_numpy

pytestmark = pytest.mark.gpu

GROUP_MIN = 2560        # kGroupInitMin of the library
COLUMNS_MAX = 10912     # largest groups whose slices fit a block: two columns,
RECORDS_MAX = 8190      # and 8-byte records


@pytest.mark.parametrize("form", ["records", "columns"])
@pytest.mark.parametrize("policy", [False, True])
@pytest.mark.parametrize("ppg,pods", [(1, 1), (3, 5), (255, 2), (257, 7), (GROUP_MIN - 1, 3), (GROUP_MIN, 3),
                                      (GROUP_MIN + 1, 16), (GROUP_MIN + 1, 17), (RECORDS_MAX, 1), (RECORDS_MAX + 1, 5),
                                      (COLUMNS_MAX, 13), (COLUMNS_MAX + 1, 3)])
def test_group_sizes(validator, ppg, pods, policy, form):
    v, groups = validator, 4 if ppg > 300 else 61
    e = W.end_to_end(seed=7 + ppg, num_switches=24, num_intents=groups, probes_per_intent=ppg, rules_per_switch=90)
    v.load_cluster(e.cluster)
    v.load_network(e.network)
    M, H = groups * ppg - (ppg > 40) * 33, e.network.num_hosts      # ragged last group
    st = W.Stream(pods, "assign")
    assign = st.ints(0, H + 2, groups * pods).astype(np.uint32)
    assign[assign >= H] = W.UNPLACED
    probes = oracle.bind_probes(e.probes.probes[:M], ppg, pods, assign, e.network.host_ip)
    dev, sizes = v.alloc_end_to_end(e)
    dassign, dp, out = to_device(assign, v.device), empty_device(M * 16, v.device), empty_device(M * 4, v.device)
    dst = empty_device(M * 4 + 4, v.device)[4:]          # columns need only their element alignment
    dst.copy_(dev["dst"][: M * 4])
    dport = empty_device(M * 2 + 2, v.device)[2:]
    dport.copy_(dev["dport"][: M * 2])
    flows = [dev["flows"]] if form == "records" else [dst, dport]
    cap = sizes["hop_cap"]
    v.set_option(B.PV_OPT_WALK_TAIL_HOP, 1)
    try:
        if policy:
            pol = W.path_policies(43, e.network, 2 * groups, forbid_max=1, must_max=2, hubs=6, p_noop=0.1)
            v.load_policies(pol)
            hits = empty_device(M * 4, v.device)
            call = B.pv_verify_flows_constrained if form == "records" else B.pv_verify_flow_columns_constrained
            call(v.ctx, M, *flows, ppg, pods, dassign, dev["masks"], cap, None, ppg, 0, dp, out, hits)
            v.sync()
            want, oh = oracle.verify_constrained(e.network, probes, cap, pol, probes_per_policy=ppg)
            assert (to_numpy(hits, np.uint32) == oh).all()
        else:
            call = B.pv_verify_flows if form == "records" else B.pv_verify_flow_columns
            call(v.ctx, M, *flows, ppg, pods, dassign, dev["masks"], cap, dp, out)
            v.sync()
            want = oracle.verify_probes(e.network, probes, cap)
    finally:
        v.set_option(B.PV_OPT_WALK_TAIL_HOP, -1)
    assert (to_numpy(out, W.RESULT_DTYPE) == want).all()
    assert (to_numpy(dp, W.PROBE_DTYPE) == probes).all()


def test_large_batches_equal_their_parts(validator):
    """60 million flows (more hop blocks than fit at once) and the same flows
    in calls of at most 3 million."""
    v, ppg, pods, groups = validator, 3000, 3, 1000
    e = W.end_to_end(seed=3, num_switches=48, num_intents=groups, probes_per_intent=ppg, rules_per_switch=120)
    v.load_cluster(e.cluster)
    v.load_network(e.network)
    part, copies, H = groups * ppg, 20, e.network.num_hosts
    dev, sizes = v.alloc_end_to_end(e)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    assign = torch.randint(0, H, (copies, groups * pods), generator=g, device="cuda", dtype=torch.int32)
    dst, dport = dev["dst"][: part * 4].repeat(copies), dev["dport"][: part * 2].repeat(copies)
    masks = dev["masks"][: groups * 4].repeat(copies)
    whole = empty_device(copies * part * 4, v.device)
    B.pv_verify_flow_columns(v.ctx, copies * part, dst, dport, ppg, pods, assign.view(torch.uint8).flatten(), masks,
                             sizes["hop_cap"], None, whole)
    one = empty_device(part * 4, v.device)
    for c in range(copies):
        B.pv_verify_flow_columns(v.ctx, part, dev["dst"], dev["dport"], ppg, pods, assign[c].view(torch.uint8), dev["masks"],
                                 sizes["hop_cap"], None, one)
        v.sync()
        assert torch.equal(whole[c * part * 4:(c + 1) * part * 4], one)
