"""Performance cases of the privacy-intent validator: what programs that use
the library have it do, called through ``Validator`` and the binding.

Kinds of case
  walk      probe walks over loaded flow tables (pv_verify_probes)
  place     node selectors of pods against a loaded cluster (pv_eval_selectors)
  affinity  the multi-term form of them (pv_eval_selector_terms)
  reach     jurisdiction-masked reachability (pv_compliant_reach)
  schedule  constrained paths and their per-hop rules (pv_schedule_paths,
            pv_compile_path_rules)
  intents   the whole check of a batch of intents on device-resident inputs:
            selectors, placement, walks, verdicts; with or without path policies
  reload    the same check from host memory after a change of the cluster and
            the tables: both are loaded again, inputs are uploaded, verdicts
            read back

Networks: "ring" is a small ring with chords; "mesh" a random graph of
average degree 5 with two hosts per switch; "fat" a k-ary fat tree.  All
outputs are whole numbers, so every tolerance is "exact".
"""
import math
import weakref

import numpy as np
import torch

from paper_2602_16100_gb300 import binding as B
from paper_2602_16100_gb300 import workloads as W
from paper_2602_16100_gb300.validator import Validator, empty_device, to_device

HOP_CAP = 32
MAX_PATH = 64        # visits of a scheduled path
RULE_PRIORITY = 60000


def listed():
    return [
        # a handful of probes after a small change: 8 switches, 1,000 probes; launches and latency count
        dict(name="walk_ring_1k", kind="walk", net="ring", switches=8, rules=64, probes=1000),
        # the flows of a few tenants re-checked on a mid-size network, an odd count
        dict(name="walk_mesh_100k", kind="walk", net="mesh", switches=512, rules=1000, probes=100_003),
        # audit of a data centre: a k=16 fat tree (320 switches) with 2,000 rules each, 10 million probes
        dict(name="walk_fat_10m", kind="walk", net="fat", switches=320, rules=2000, probes=10_000_000),
        # the pods of one deployment against a 5,000-node cluster
        dict(name="place_777", kind="place", nodes=5000, keys=64, pods=777, absent=0.1),
        # every pod of a large cluster
        dict(name="place_100k", kind="place", nodes=5000, keys=64, pods=100_000, absent=0.0),
        # the same cluster with node affinity: up to three ORed terms per pod
        dict(name="affinity_50k", kind="affinity", nodes=4999, keys=64, pods=50_001, absent=0.0),
        # all-source compliant reach of a continuum WAN (links both ways)
        dict(name="reach_wan_4096", kind="reach", directed=False, vertices=4096, sources=4096, masks=64),
        # the same question where links are one-way
        dict(name="reach_directed_3k", kind="reach", directed=True, vertices=3001, sources=3001, masks=24),
        # enforcement: weighted paths under policies for 10,000 flows, compiled to rules
        dict(name="schedule_10k", kind="schedule", switches=512, rules=1000, requests=10_000, weighted=True),
        # a small batch of new intents with path policies; latency counts
        dict(name="intents_policies_300", kind="intents", switches=512, rules=1000, intents=301, flows=250, policies=True),
        # the full audit: 10,000 intents, 50 million flows
        dict(name="intents_10k", kind="intents", switches=512, rules=1000, intents=10_000, flows=5000, policies=False),
        # the control loop after a change of labels and rules, from host memory
        dict(name="reload_1k", kind="reload", switches=512, rules=1000, intents=1000, flows=1000, policies=False),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["walk", "walk", "place", "affinity", "reach", "schedule", "intents", "intents", "reload"])
    switches = _log(rng, 40, 512)
    rules = switches + rng.randint(60, 500)   # a mesh switch routes to every other one, then has its ACL
    if kind == "walk":
        net = rng.choice(["ring", "mesh", "fat"])
        if net == "ring":
            return dict(kind=kind, net=net, switches=rng.randint(5, 24), rules=rng.randint(60, 120), probes=_log(rng, 1, 300_000))
        if net == "mesh":
            return dict(kind=kind, net=net, switches=switches, rules=rules, probes=_log(rng, 100, 5_000_000))
        k = rng.choice([4, 6, 8, 12, 16])
        return dict(kind=kind, net=net, switches=k * k // 4 + k * k, rules=rng.randint(300, 2000), probes=_log(rng, 1000, 10_000_000))
    if kind in ("place", "affinity"):
        return dict(kind=kind, nodes=_log(rng, 16, 5000), keys=rng.randint(8, 64), absent=rng.choice([0.0, 0.1]),
                    pods=_log(rng, 32, 100_000 if kind == "place" else 50_000))
    if kind == "reach":
        directed = rng.random() < 0.5
        v = _log(rng, 200, 3000 if directed else 4096)
        return dict(kind=kind, directed=directed, vertices=v, sources=rng.randint(1, v),
                    masks=rng.randint(1, 24 if directed else 64))
    if kind == "schedule":
        return dict(kind=kind, switches=switches, rules=rules, requests=_log(rng, 50, min(10_000, switches * switches)),
                    weighted=rng.random() < 0.5)
    big = kind == "intents"
    intents = _log(rng, 20, 10_000 if big else 2000)
    flows = _log(rng, 20, min(5000, 50_000_000 // intents if big else 2_000_000 // intents))
    return dict(kind=kind, switches=switches, rules=rules, intents=intents, flows=flows,
                policies=big and rng.random() < 0.5)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _ints(g, lo, hi, *shape):
    """Integers uniform in [lo, hi]."""
    return torch.randint(lo, hi + 1, shape, generator=g, device="cuda")


def _zipf_weights(n, s=1.1):
    return 1.0 / torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** s


def _zipf(g, n, *shape):
    c = torch.cumsum(_zipf_weights(n), 0)
    u = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * c[-1]
    return torch.searchsorted(c, u).clamp_(max=n - 1)


def _sets(g, n, k, count):
    """count draws of k values of Zipf(n) without replacement, in draw order (exponential races)."""
    out = []
    w = _zipf_weights(n).float()
    for lo in range(0, count, 1 << 18):
        m = min(1 << 18, count - lo)
        t = torch.empty((m, n), device="cuda").exponential_(generator=g) / w
        out.append(torch.topk(t, min(k, n), dim=1, largest=False).indices)
    return torch.cat(out) if out else torch.zeros((0, k), dtype=torch.int64, device="cuda")


def _offsets(n):
    o = torch.zeros(len(n) + 1, dtype=torch.int64, device="cuda")
    o[1:] = torch.cumsum(n, 0)
    return o


def _u8(t):
    return t.contiguous().view(torch.uint8).reshape(-1)


def _exprs(key, op, nvals, vals):
    """pv_expr records from columns; value slots past nvals repeat the first value."""
    r = torch.zeros((len(key), 10), dtype=torch.int16, device="cuda")
    r[:, 0] = key.to(torch.int16)
    r[:, 1] = (op | nvals << 8).to(torch.int16)
    slot = torch.arange(8, device="cuda")[None, :]
    r[:, 2:] = torch.where(slot < nvals[:, None], vals, vals[:, :1]).to(torch.int16)
    return _u8(r)


def _cluster(seed, c):
    g = _gen(seed)
    labels = _zipf(g, 256, c["keys"], c["nodes"])
    if c["absent"]:
        labels[torch.rand(labels.shape, generator=g, device="cuda") < c["absent"]] = W.ABSENT
    return W.Cluster(c["nodes"], c["keys"], labels.cpu().numpy().astype(np.uint16).reshape(-1))


def _selector_lists(g, lists, keys, max_exprs):
    """Expression lists: 1 .. max_exprs expressions on distinct keys, 40% equality, 30% In, 20% NotIn, 10% Exists."""
    n = _ints(g, 1, min(max_exprs, keys), lists)
    offs = _offsets(n)
    E = int(offs[-1])
    lst = torch.repeat_interleave(torch.arange(lists, device="cuda"), n)
    slot = torch.arange(E, device="cuda") - offs[lst]
    key = torch.rand((lists, keys), generator=g, device="cuda").argsort(1)[lst, slot]
    u = torch.rand(E, generator=g, device="cuda")
    op = torch.where(u < 0.7, W.OP_IN, torch.where(u < 0.9, W.OP_NOTIN, W.OP_EXISTS))
    nvals = torch.where(u < 0.4, 1, torch.where(u < 0.9, _ints(g, 1, 8, E), 0))
    return offs, E, dict(key=key, op=op, nvals=nvals, vals=_sets(g, 256, 8, E))


def _mesh(seed, S, rules, regions=16):
    """Random connected switch graph (average degree 5), two hosts per switch;
    /24 BFS routes, /32 local delivery and an ACL fill to ``rules`` rules per
    switch (prefixes /8-/32, port ranges up to 1,024 wide, 5% shadowed)."""
    r = np.random.default_rng([seed, 11])
    perm = r.permutation(S)
    edges = {tuple(sorted((int(perm[i]), int(perm[r.integers(0, i)])))) for i in range(1, S)}
    while len(edges) < min(S * 5 // 2, S * (S - 1) // 2):
        a, b = (int(x) for x in r.integers(0, S, 2))
        if a != b:
            edges.add((min(a, b), max(a, b)))
    adj = np.zeros((S, S), bool)
    e = np.array(sorted(edges))
    adj[e[:, 0], e[:, 1]] = adj[e[:, 1], e[:, 0]] = True
    dist = np.where(np.eye(S, dtype=bool), 0, -1)
    a32, level = adj.astype(np.float32), 0
    while (dist < 0).any():
        dist = np.where((dist < 0) & ((dist == level).astype(np.float32) @ a32 > 0), level + 1, dist)
        level += 1
    deg = adj.sum(1)
    port_offs = np.concatenate([[0], np.cumsum(2 + deg)])
    peer = np.zeros(port_offs[-1], np.int64)
    port_to = np.cumsum(adj, 1) + 1          # port of s towards neighbour u
    u, v = np.nonzero(adj)
    peer[port_offs[u] + port_to[u, v]] = v << 8 | port_to[v, u]
    hosts = np.arange(2 * S)
    peer[port_offs[hosts // 2] + hosts % 2] = W.HOST_BIT | hosts
    host_ip = (10 << 24 | (hosts // 2) << 8 | (hosts % 2 + 1)).astype(np.uint32)
    next_port = np.zeros((S, S), np.int64)
    for s in range(S):
        nb = np.nonzero(adj[s])[0]
        next_port[s] = port_to[s, nb[np.argmax(dist[nb] == dist[s] - 1, axis=0)]]
    n = max(rules, S + 1)
    t = np.zeros((S, n), W.RULE_DTYPE)
    t["priority"], t["in_port"], t["dport_hi"] = W.ROUTING_PRIORITY, W.ANY_PORT, 65535
    other = np.arange(S - 1)[None, :] + (np.arange(S - 1)[None, :] >= np.arange(S)[:, None])
    t["dst_ip"][:, :S - 1], t["dst_len"][:, :S - 1] = 10 << 24 | other << 8, 24
    t["action"][:, :S - 1] = np.take_along_axis(next_port, other, 1)
    t["dst_ip"][:, S - 1:S + 1], t["dst_len"][:, S - 1:S + 1] = host_ip.reshape(S, 2), 32
    t["action"][:, S - 1:S + 1] = [0, 1]
    a = t[:, S + 1:]
    shape = a.shape
    if a.size:
        a["priority"] = r.integers(W.ROUTING_PRIORITY + 1, 65536, shape)
        for ip, ln in (("src_ip", "src_len"), ("dst_ip", "dst_len")):
            a[ln] = r.integers(8, 33, shape)
            a[ip] = host_ip[r.integers(0, 2 * S, shape)] & (0xFFFFFFFF << (32 - a[ln].astype(np.int64)) & 0xFFFFFFFF)
        a["dport_lo"] = r.integers(0, 65536, shape)
        a["dport_hi"] = np.minimum(a["dport_lo"].astype(np.int64) + r.integers(0, 1024, shape), 65535)
        ports = (2 + deg)[:, None]
        a["in_port"] = np.where(r.random(shape) < 0.75, W.ANY_PORT, r.integers(0, ports, shape))
        a["action"] = np.where(r.random(shape) < 0.2, W.DROP, r.integers(0, ports, shape))
        s, i = np.nonzero(r.random(shape) < 0.05)      # shadowed: a narrower copy below the rule it copies
        c = a[s, r.integers(0, shape[1], len(s))]
        c["dst_len"] = np.minimum(32, c["dst_len"] + r.integers(0, 9, len(s)))
        c["priority"] = r.integers(W.ROUTING_PRIORITY, np.maximum(c["priority"], W.ROUTING_PRIORITY + 1), len(s))
        c["action"] = a["action"][s, i]
        a[s, i] = c
    t = np.take_along_axis(t, r.random((S, n)).argsort(1), 1)
    return W.Network(S, (np.arange(S + 1) * n).astype(np.uint32), t.reshape(-1), r.integers(0, regions, S).astype(np.uint8),
                     port_offs.astype(np.uint32), peer.astype(np.int32), 2 * S, (hosts // 2).astype(np.uint16),
                     (hosts % 2).astype(np.uint16), host_ip)


def _network(seed, c):
    if c.get("net") == "ring":
        return W.tiny(seed=seed, num_switches=c["switches"], rules_per_switch=c["rules"], num_pods=1, num_probes=1)["network"]
    if c.get("net") == "fat":
        k = int(round(math.sqrt(c["switches"] * 4 / 5)))
        return W.fat_tree(seed=seed, k=k, rules_per_switch=c["rules"], num_probes=1)["network"]
    return _mesh(seed, c["switches"], c["rules"])


def _probes(seed, net, m):
    """Uniform host pairs and ports, a random region mask each: pv_probe records as int32 [m, 4]."""
    g = _gen(seed + 1)
    ip = torch.from_numpy(net.host_ip.astype(np.int64)).cuda()
    src, dst = _ints(g, 0, net.num_hosts - 1, m), _ints(g, 0, net.num_hosts - 1, m)
    bits = int(net.switch_region.max()) + 1
    p = torch.empty((m, 4), dtype=torch.int32, device="cuda")
    p[:, 0], p[:, 1] = ip[src].int(), ip[dst].int()
    p[:, 2] = (_ints(g, 0, 65535, m) | src << 16).int()
    p[:, 3] = _ints(g, 0, (1 << bits) - 1, m).int()
    return p


def _intents(seed, c, net):
    """Cluster (node n = host n, key 0 = its region) and the inputs of a batch
    of intents: 2-8 permitted regions each, a region term and 0-3 more, four
    pods, ``flows`` flows to uniform hosts."""
    g = _gen(seed + 2)
    N, I, F, K = net.num_hosts, c["intents"], c["flows"], 32
    region = torch.from_numpy(net.switch_region[net.host_switch].astype(np.int64)).cuda()
    nreg = int(net.switch_region.max()) + 1
    labels = _zipf(g, 64, K, N)
    labels[0] = region
    cluster = W.Cluster(N, K, labels.cpu().numpy().astype(np.uint16).reshape(-1))
    pick = torch.rand((I, max(nreg, 8)), generator=g, device="cuda")
    pick[:, nreg:] = 2.0
    pick = pick.argsort(1)[:, :8]
    pop = _ints(g, 2, min(8, nreg), I)
    masks = torch.where(torch.arange(8, device="cuda")[None, :] < pop[:, None], torch.ones_like(pick) << pick, 0).sum(1)
    n = 1 + _ints(g, 0, 3, I)
    offs = _offsets(n)
    E = int(offs[-1])
    lst = torch.repeat_interleave(torch.arange(I, device="cuda"), n)
    slot = torch.arange(E, device="cuda") - offs[lst]
    key = torch.rand((I, K - 1), generator=g, device="cuda").argsort(1)[lst, (slot - 1).clamp(min=0)] + 1
    more = torch.where(torch.rand(E, generator=g, device="cuda") < 0.7, 1, _ints(g, 2, 4, E))
    first = slot == 0
    exprs = _exprs(torch.where(first, 0, key), torch.zeros_like(key), torch.where(first, pop[lst], more),
                   torch.where(first[:, None], pick[lst], _sets(g, 64, 8, E)))
    ip = torch.from_numpy(net.host_ip.astype(np.int64)).cuda()
    M = I * F
    inputs = {"offs": _u8(offs.int()), "exprs": exprs,
              "draws": _u8(torch.randint(0, 1 << 62, (I * 4,), generator=g, device="cuda")),
              "masks": _u8(masks.int()), "dst": _u8(ip[_ints(g, 0, N - 1, M)].int()),
              "dport": _u8(_ints(g, 0, 65535, M).to(torch.int16))}
    sizes = {"intents": I, "pods": 4, "probes_per_intent": F, "num_exprs": E, "hop_cap": HOP_CAP}
    return cluster, inputs, sizes


def _intent_outputs(sizes, nodes, policies):
    I, M, words = sizes["intents"], sizes["intents"] * sizes["probes_per_intent"], W.words_per_row(nodes)
    n = {"bits": I * words * 4, "flags": I, "assign": I * 16, "results": M * 4, "pass": I, "counts": I * 32}
    if policies:
        n["hits"] = M * 4
    return {k: empty_device(b, "cuda") for k, b in n.items()}


def _reach_query(seed, c):
    V = c["vertices"]
    if not c["directed"]:
        q = W.continuum_wan(seed=seed, num_vertices=V, num_masks=c["masks"],
                            num_sources=None if c["sources"] == V else c["sources"])
        return q.graph, q.sources, q.masks
    r = np.random.default_rng([seed, 12])
    graph = W.random_digraph(seed, V, 6 * V, num_regions=32)
    masks = np.array([np.bitwise_or.reduce(1 << r.permutation(32)[:r.integers(8, 25)]) for _ in range(c["masks"])], np.int64)
    src = np.arange(V) if c["sources"] == V else r.integers(0, V, c["sources"])
    return graph, src.astype(np.uint32), masks.astype(np.uint32)


class State(dict):
    """A prepared case: its context, plan and buffers; the context is closed with the state."""

    def __init__(self, case):
        super().__init__(case=case, v=Validator(torch.cuda.current_device()))
        weakref.finalize(self, self["v"].close)


def prepare(case, seed):
    s = State(case)
    v, kind = s["v"], case["kind"]
    if kind == "walk":
        net = _network(seed, case)
        v.load_network(net)
        s.update(probes=_u8(_probes(seed, net, case["probes"])), out=empty_device(case["probes"] * 4, "cuda"))
    elif kind in ("place", "affinity"):
        v.load_cluster(_cluster(seed, case))
        s.update(_placement_inputs(seed, case))
        words = W.words_per_row(case["nodes"])
        s.update(words=words, bits=empty_device(case["pods"] * words * 4, "cuda"), flags=empty_device(case["pods"], "cuda"))
    elif kind == "reach":
        graph, src, masks = _reach_query(seed, case)
        s.update(graph=v.upload_graph(graph), src=to_device(src, "cuda"), masks=to_device(masks, "cuda"),
                 out=empty_device(len(masks) * len(src) * W.words_per_row(case["vertices"]) * 4, "cuda"))
    elif kind == "schedule":
        net = _network(seed, case)
        v.load_network(net)
        R = case["requests"]
        v.load_policies(W.path_policies(seed, net, R))
        req = W.path_requests(seed, net, R, num_policies=R, extra_regions=(6, 14))
        weights = _ints(_gen(seed), 1, 16, len(net.port_peer)).to(torch.int16)
        s.update(req=to_device(req, "cuda"), weights=_u8(weights) if case["weighted"] else None,
                 visits=torch.zeros(R * MAX_PATH, dtype=torch.int32, device="cuda"), len=empty_device(R, "cuda"),
                 status=empty_device(R, "cuda"), rules=empty_device(R * MAX_PATH * 20, "cuda"),
                 rule_switch=empty_device(R * MAX_PATH * 2, "cuda"))
    else:
        net = _network(seed, case)
        cluster, inputs, sizes = _intents(seed, case, net)
        dev = {**inputs, **_intent_outputs(sizes, cluster.num_nodes, case["policies"])}
        s.update(dev=dev, sizes=sizes)
        v.load_cluster(cluster)
        v.load_network(net)
        if case["policies"]:
            v.load_policies(W.path_policies(seed, net, case["intents"]))
        if kind == "reload":
            host = {k: t.cpu().pin_memory() for k, t in inputs.items()}
            host["pass"], host["counts"] = (torch.zeros(dev[k].numel(), dtype=torch.uint8).pin_memory()
                                            for k in ("pass", "counts"))
            s.update(host=host, cluster=cluster, net=net, stream=torch.cuda.Stream(), copy_stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    return s


def _placement_inputs(seed, case):
    g = _gen(seed + 1)
    P = case["pods"]
    assign = _u8(_ints(g, 0, case["nodes"] - 1, P).int())
    if case["kind"] == "place":
        offs, E, cols = _selector_lists(g, P, case["keys"], 8)
        return dict(offs=_u8(offs.int()), num_exprs=E, exprs=_exprs(**cols), assign=assign)
    terms = _offsets(_ints(g, 0, 3, P))
    T = int(terms[-1])
    offs, E, cols = _selector_lists(g, T, case["keys"], 4)
    return dict(terms=_u8(terms.int()), num_terms=T, offs=_u8(offs.int()), num_exprs=E, exprs=_exprs(**cols), assign=assign)


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def run(s):
    case, v = s["case"], s["v"]
    kind, stream = case["kind"], torch.cuda.current_stream()
    if kind == "walk":
        return v.verify_probes(s["probes"], case["probes"], HOP_CAP, s["out"], stream)
    if kind == "place":
        return v.eval_selectors(s["offs"], s["num_exprs"], s["exprs"], s["assign"], case["pods"], s["words"], s["bits"],
                                s["flags"], stream)
    if kind == "affinity":
        B.pv_eval_selector_terms(v.ctx, case["pods"], s["terms"], s["num_terms"], s["offs"], s["num_exprs"], s["exprs"],
                                 s["assign"], s["bits"], s["words"], s["flags"], stream)
        return s["bits"], s["flags"]
    if kind == "reach":
        return v.compliant_reach(s["graph"], case["sources"], s["src"], case["masks"], s["masks"], d_reach=s["out"],
                                 stream=stream)
    if kind == "schedule":
        R = case["requests"]
        B.pv_schedule_paths(v.ctx, R, s["req"], s["weights"], MAX_PATH, s["visits"], s["len"], s["status"], stream)
        B.pv_compile_path_rules(v.ctx, R, s["req"], MAX_PATH, s["visits"], s["len"], s["status"], RULE_PRIORITY, s["rules"],
                                s["rule_switch"], stream)
        return s["visits"], s["len"], s["status"], s["rules"], s["rule_switch"]
    if kind == "intents":
        v.run_end_to_end(s["dev"], s["sizes"], stream)
        return {k: s["dev"][k] for k in ("pass", "counts", "results", "bits", "flags", "assign", "hits") if k in s["dev"]}

    def loads():
        v.load_cluster(s["cluster"])
        v.begin_network(s["net"])
        return v.finish_network

    v.run_end_to_end_from_host(s["host"], s["dev"], s["sizes"], s["stream"], s["copy_stream"], loads=loads)
    v.sync(s["stream"])
    return {**{k: s["host"][k] for k in ("pass", "counts")}, **{k: s["dev"][k] for k in ("results", "bits", "flags", "assign")}}


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def work(case):
    """Bytes of the inputs and outputs (averages where they are drawn);
    "flops": integer operations of the definition, one per node and
    expression, per probe, or per (mask, source, edge) word of 32 vertices."""
    kind = case["kind"]
    if kind == "walk":
        return {"bytes": 20 * case["probes"], "flops": 3 * case["probes"]}
    if kind in ("place", "affinity"):
        P, words = case["pods"], W.words_per_row(case["nodes"])
        E = 4.5 * P if kind == "place" else 1.5 * 2.5 * P
        extra = 0 if kind == "place" else 4 * P + 4 * 1.5 * P
        return {"bytes": int(P * (4 * words + 9) + 20 * E + extra + 2 * case["nodes"] * case["keys"]),
                "flops": int(E * case["nodes"])}
    if kind == "reach":
        rows, V = case["masks"] * case["sources"], case["vertices"]
        return {"bytes": rows * W.words_per_row(V) * 4 + 29 * V, "flops": rows * 6 * V // 32}
    if kind == "schedule":
        R = case["requests"]
        # request, path of about 8 visits, length and status; every rule slot and its switch
        return {"bytes": R * (16 + 4 * 8 + 2 + MAX_PATH * 22), "flops": R * 5 * case["switches"]}
    I, M, N = case["intents"], case["intents"] * case["flows"], 2 * case["switches"]
    n = I * (W.words_per_row(N) * 4 + 2.5 * 20 + 4 + 32 + 4 + 1 + 16 + 1 + 32) + M * (6 + 4 + (4 if case["policies"] else 0))
    if kind == "reload":   # the tables and labels come in too
        n += case["switches"] * max(case["rules"], case["switches"] + 1) * 20 + 32 * N * 2
    return {"bytes": int(n), "flops": int(3 * M + 2.5 * I * N)}


def tolerance(case):
    return "exact"


# ----------------------------------------------------------------------------
# the same outputs by definition, in plain torch
# ----------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "walk":
        return _exact_walk(case, seed)
    if kind in ("place", "affinity"):
        return _exact_placement(case, seed)
    if kind == "reach":
        return _exact_reach(case, seed)
    return None   # chains of the above, and of a path search per request


def _pack(rows, words):
    """bool [n, items] -> bytes of LSB-first bitset rows of ``words`` words."""
    n, items = rows.shape
    b = torch.zeros((n, words * 32), dtype=torch.uint8, device=rows.device)
    b[:, :items] = rows
    weight = (1 << torch.arange(8, device=rows.device)).to(torch.uint8)
    return (b.view(n, words * 4, 8) * weight).sum(2).to(torch.uint8).reshape(-1)


def _exact_placement(case, seed):
    s = _placement_inputs(seed, case)
    N, P, words = case["nodes"], case["pods"], W.words_per_row(case["nodes"])
    labels = torch.from_numpy(_cluster(seed, case).labels.astype(np.int64)).cuda().view(case["keys"], N)
    raw = s["exprs"].view(torch.int16).view(-1, 10).long() & 0xFFFF
    key, op, nvals, vals = raw[:, 0], raw[:, 1] & 0xFF, raw[:, 1] >> 8, raw[:, 2:]
    offs = s["offs"].view(torch.int32).long()
    terms = s["terms"].view(torch.int32).long() if "terms" in s else torch.arange(P + 1, device="cuda")
    assign = s["assign"].view(torch.int32).long()
    listed_in = torch.arange(8, device="cuda")[None, :] < nvals[:, None]
    carried = torch.zeros((case["keys"], 65536), dtype=torch.bool, device="cuda")
    carried[torch.arange(case["keys"], device="cuda")[:, None].expand(-1, N), labels] = True
    bad_value = (listed_in & (op == W.OP_IN)[:, None] & ~carried[key[:, None], vals]).any(1)
    bits, flags = [], []
    for lo in range(0, P, 2048):
        hi = min(P, lo + 2048)
        t0, t1 = int(terms[lo]), int(terms[hi])
        e0, e1 = int(offs[t0]), int(offs[t1])
        unknown = torch.zeros(hi - lo, dtype=torch.bool, device="cuda")
        term_ok = torch.ones((t1 - t0, N), dtype=torch.bool, device="cuda")
        pod_of = torch.repeat_interleave(torch.arange(hi - lo, device="cuda"), terms[lo + 1:hi + 1] - terms[lo:hi])
        if e1 > e0:
            val = labels[key[e0:e1]]
            inset = torch.zeros(val.shape, dtype=torch.bool, device="cuda")
            for j in range(8):
                inset |= (val == vals[e0:e1, j:j + 1]) & listed_in[e0:e1, j:j + 1]
            o = op[e0:e1, None]
            m = torch.where(o == W.OP_IN, inset, torch.where(o == W.OP_NOTIN, ~inset, (val != W.ABSENT) ^ (o == W.OP_DOESNOTEXIST)))
            term_of = torch.repeat_interleave(torch.arange(t1 - t0, device="cuda"), offs[t0 + 1:t1 + 1] - offs[t0:t1])
            misses = torch.zeros((t1 - t0, N), dtype=torch.int32, device="cuda").index_add_(0, term_of, (~m).int())
            term_ok = misses == 0
            unknown[pod_of[term_of[bad_value[e0:e1]]]] = True
        hits = torch.zeros((hi - lo, N), dtype=torch.int32, device="cuda").index_add_(0, pod_of, term_ok.int())
        ok = (hits > 0) | (terms[lo + 1:hi + 1] == terms[lo:hi])[:, None]
        a_ok = ok.gather(1, assign[lo:hi, None])[:, 0]
        bits.append(_pack(ok, words))
        flags.append((a_ok * 1 + ~ok.any(1) * 2 + unknown * 4 + (a_ok & ~unknown) * 8).to(torch.uint8))
    return torch.cat(bits), torch.cat(flags)


def _exact_reach(case, seed):
    graph, src, masks = _reach_query(seed, case)
    V, words = case["vertices"], W.words_per_row(case["vertices"])
    adj = torch.zeros((V, V), dtype=torch.float16, device="cuda")
    u = torch.from_numpy(np.repeat(np.arange(V), np.diff(graph.offs.astype(np.int64)))).cuda()
    adj[u, torch.from_numpy(graph.cols.astype(np.int64)).cuda()] = 1
    region, src = (torch.from_numpy(x.astype(np.int64)).cuda() for x in (graph.region, src))
    out = []
    for mask in masks:
        ok = (int(mask) >> region) & 1 == 1
        idx = torch.nonzero(ok)[:, 0]   # closure of the permitted subgraph by squaring
        r = ((adj[idx][:, idx] + torch.eye(len(idx), device="cuda", dtype=torch.float16)) > 0).half()
        while True:
            r2 = ((r @ r) > 0).half()
            if torch.equal(r2, r):
                break
            r = r2
        full = torch.zeros((V, V), dtype=torch.bool, device="cuda")
        full[idx[:, None], idx[None, :]] = r > 0
        out.append(_pack(full[src], words))
    return torch.cat(out)


def _exact_walk(case, seed):
    net = _network(seed, case)
    p = _probes(seed, net, case["probes"]).long() & 0xFFFFFFFF
    M = len(p)

    def dev(a):
        return torch.from_numpy(a.astype(np.int64)).cuda()

    ro, po = net.rule_offs.astype(np.int64), dev(net.port_offs)
    peer, region, host_ip = dev(net.port_peer), dev(net.switch_region), dev(net.host_ip)
    src = p[:, 2] >> 16
    here, in_port = dev(net.host_switch)[src], dev(net.host_port)[src]
    out = torch.zeros(M, dtype=torch.int64, device="cuda")
    live = torch.arange(M, device="cuda")

    def finish(which, status, hops):
        out[live[which]] = status | hops << 8 | here[which] << 16

    for hop in range(HOP_CAP):
        ok = (p[live, 3] >> region[here]) & 1 == 1
        finish(~ok, W.ST_VIOLATION, hop + 1)
        live, here, in_port = live[ok], here[ok], in_port[ok]
        order = here.argsort()
        live, here, in_port = live[order], here[order], in_port[order]
        act = torch.full_like(here, W.DROP)
        count = torch.bincount(here, minlength=net.num_switches).tolist()
        at = 0
        for s, n in enumerate(count):
            rules = net.rules[ro[s]:ro[s + 1]]
            rules = rules[np.argsort(-rules["priority"].astype(np.int64), kind="stable")]
            if n and len(rules):
                r = {f: dev(rules[f])[None, :] for f in rules.dtype.names}
                ms, md = ((0xFFFFFFFF << (32 - r[f])) & 0xFFFFFFFF for f in ("src_len", "dst_len"))
                for lo in range(at, at + n, 16384):
                    k = slice(lo, min(lo + 16384, at + n))
                    h = p[live[k]]
                    port = h[:, 2:3] & 0xFFFF
                    m = ((h[:, :1] ^ r["src_ip"]) & ms == 0) & ((h[:, 1:2] ^ r["dst_ip"]) & md == 0)
                    m &= (port >= r["dport_lo"]) & (port <= r["dport_hi"])
                    m &= (r["in_port"] == W.ANY_PORT) | (r["in_port"] == in_port[k, None])
                    first = m.to(torch.uint8).argmax(1)
                    act[k] = torch.where(m.any(1), r["action"][0][first], W.DROP)
            at += n
        nxt = torch.where(act == W.DROP, torch.full_like(act, W.PEER_NONE), peer[(po[here] + act).clamp(max=len(peer) - 1)])
        finish(nxt < 0, W.ST_DROP, hop + 1)
        at_host = (nxt >= 0) & (nxt & W.HOST_BIT != 0)
        mine = at_host & (host_ip[(nxt & ~W.HOST_BIT).clamp(0, net.num_hosts - 1)] == p[live, 1])
        finish(mine, W.ST_COMPLIANT, hop + 1)
        finish(at_host & ~mine, W.ST_MISDELIVERED, hop + 1)
        go = (nxt >= 0) & ~at_host
        if hop + 1 == HOP_CAP:
            finish(go, W.ST_LOOP, HOP_CAP)
        live, here, in_port = live[go], (nxt >> 8)[go], (nxt & 0xFF)[go]
        if not len(live):
            break
    return torch.from_numpy(out.cpu().numpy().astype(np.uint32).view(np.uint8)).cuda()
