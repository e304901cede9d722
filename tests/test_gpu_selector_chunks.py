"""The selector rows kernel resolves the expressions of a chunk of pods
together: chunk sizes, lists that run past a chunk's slots, malformed lists
among well-formed ones and arrays at the least alignment, against the oracle,
for expression lists and for terms."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_16100_gb300 import binding as B
from paper_2602_16100_gb300 import workloads as W
from paper_2602_16100_gb300.validator import empty_device, to_device, to_numpy

pytestmark = pytest.mark.gpu

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1


def _cluster(n, seed):
    r = np.random.default_rng(seed)
    labels = r.integers(0, 9, (12, n)).astype(np.uint16)
    labels[r.random((12, n)) < 0.15] = W.ABSENT
    return W.Cluster(n, 12, labels.reshape(-1))


def _exprs(r, count, bad=0.0):
    e = np.zeros(count, W.EXPR_DTYPE)
    e["key"] = r.integers(0, 12, count)
    e["op"] = r.choice([0, 0, 1, 1, 1, 2, 3], count)
    e["nvals"] = np.where(e["op"] < 2, r.integers(1, 9, count), 0)
    e["vals"] = r.integers(0, 10, (count, 8))            # 9 is carried by no node
    hit = r.random(count) < bad
    e["key"][hit] = r.integers(12, 60000, hit.sum())
    return e


def _offsets(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.uint32)


def _shift(a, dev, by):
    """The array's bytes on the device, `by` bytes past an aligned address."""
    t = empty_device(a.nbytes + 16, dev)
    t[by:by + a.nbytes].copy_(to_device(a, dev))
    return t[by:]


def _lists(v, c, offs, ex, assign, words):
    P, d = len(offs) - 1, v.device
    bits, flags = empty_device(P * words * 4, d), empty_device(P, d)
    B.pv_eval_selectors(v.ctx, P, to_device(offs, d), len(ex), _shift(ex, d, 4), to_device(assign, d), bits, words, flags)
    v.sync()
    return to_numpy(bits, np.uint32, (P, words)), to_numpy(flags, np.uint8)


@pytest.mark.parametrize("P", [1, 7, 9, 31, 33, SMS * 32 + 1, SMS * 128 + 5])
@pytest.mark.parametrize("n", [33, 5121])
def test_chunk_sizes(validator, P, n):
    if n > 5000 and P > 5000:
        n = 161
    r = np.random.default_rng(P)
    c = _cluster(n, 1)
    validator.load_cluster(c)
    offs = _offsets(r.integers(0, 9, P))
    ex = _exprs(r, int(offs[-1]), bad=0.01)
    assign = r.integers(0, n + 2, P).astype(np.uint32)
    words = W.words_per_row(n) + (4 if P % 2 else 0)
    g, gf = _lists(validator, c, offs, ex, assign, words)
    o, of = oracle.eval_selectors(n, 12, c.labels, offs, ex, assign, words=words)
    assert (g == o).all() and (gf == of).all()


@pytest.mark.parametrize("lens", [[320] + [1] * 40, [100, 100, 100, 20, 5, 0, 0, 6], [319, 1, 1, 0, 3], [321, 2, 0, 900, 1],
                                  [33] * 32, [0] * 50])
def test_lists_past_the_slots(validator, lens):
    r = np.random.default_rng(len(lens))
    c = _cluster(200, 2)
    validator.load_cluster(c)
    offs = _offsets(lens)
    ex = _exprs(r, int(offs[-1]))
    ex["op"] = np.where(r.random(len(ex)) < 0.97, 1, ex["op"])      # mostly NotIn: long lists leave nodes
    ex["nvals"] = np.where(ex["op"] < 2, np.maximum(1, ex["nvals"] // 4), 0)
    ex["vals"] = np.where(np.arange(8) < 1, 9, ex["vals"])
    assign = r.integers(0, 200, len(lens)).astype(np.uint32)
    words = W.words_per_row(200)
    g, gf = _lists(validator, c, offs, ex, assign, words)
    o, of = oracle.eval_selectors(200, 12, c.labels, offs, ex, assign)
    assert (g == o).all() and (gf == of).all()
    # the same lists as one term each, the expressions only 2-byte aligned
    P, d = len(lens), validator.device
    bits, flags = empty_device(P * words * 4, d), empty_device(P, d)
    terms = np.arange(P + 1, dtype=np.uint32)
    B.pv_eval_selector_terms(validator.ctx, P, to_device(terms, d), P, to_device(offs, d), len(ex), _shift(ex, d, 2),
                             to_device(assign, d), bits, words, flags)
    validator.sync()
    o, of = oracle.eval_selector_terms(200, 12, c.labels, terms, offs, ex, assign)
    assert (to_numpy(bits, np.uint32, (P, words)) == o).all() and (to_numpy(flags, np.uint8) == of).all()


def test_malformed_among_well_formed(validator):
    """Offsets that decrease or pass the end, in the middle of a chunk: only
    the pods that they bound are affected (lists and terms)."""
    r = np.random.default_rng(5)
    c = _cluster(300, 3)
    validator.load_cluster(c)
    P, words = 100, W.words_per_row(300)
    offs = _offsets(r.integers(1, 6, P))
    ex = _exprs(r, int(offs[-1]))
    assign = r.integers(0, 300, P).astype(np.uint32)
    for at, to in ((40, 3), (50, len(ex) + 9), (70, 0xFFFFFFFF)):
        bad = offs.copy()
        bad[at] = to
        g, gf = _lists(validator, c, bad, ex, assign, words)
        o, of = oracle.eval_selectors(300, 12, c.labels, bad, ex, assign)
        assert (g == o).all() and (gf == of).all(), (at, to)
        d = validator.device
        pods = np.concatenate([np.arange(0, P, 2), [P]]).astype(np.uint32)     # two terms a pod
        n = len(pods) - 1
        bits, flags = empty_device(n * words * 4, d), empty_device(n, d)
        B.pv_eval_selector_terms(validator.ctx, n, to_device(pods, d), P, to_device(bad, d), len(ex), to_device(ex, d),
                                 to_device(assign[:n], d), bits, words, flags)
        validator.sync()
        o, of = oracle.eval_selector_terms(300, 12, c.labels, pods, bad, ex, assign[:n])
        assert (to_numpy(bits, np.uint32, (n, words)) == o).all() and (to_numpy(flags, np.uint8) == of).all(), (at, to)


@pytest.mark.parametrize("n", [161, 5120, 5121, 11000])
def test_more_expressions_than_lanes(validator, n):
    """Pods of 31 to 130 expressions in one list, in one term and over several,
    most of them with nodes left at the end, in rows of one span and more."""
    r = np.random.default_rng(n)
    c = _cluster(n, 6)
    validator.load_cluster(c)
    lens = np.concatenate([[31, 32, 33, 34, 64, 65, 96, 97, 130, 0, 1], r.integers(0, 70, 60)])
    offs = _offsets(lens)
    ex = _exprs(r, int(offs[-1]))
    ex["op"] = np.where(r.random(len(ex)) < 0.985, 1, ex["op"])
    ex["nvals"] = np.where(ex["op"] < 2, np.maximum(1, ex["nvals"] // 4), 0)
    ex["vals"] = np.where(r.random((len(ex), 8)) < 0.97, 10 + np.arange(8), ex["vals"])    # mostly values of no node
    P, words, d = len(lens), W.words_per_row(n) + 4, validator.device
    assign = r.integers(0, n + 2, P).astype(np.uint32)
    g, gf = _lists(validator, c, offs, ex, assign, words)
    o, of = oracle.eval_selectors(n, 12, c.labels, offs, ex, assign, words=words)
    assert (g == o).all() and (gf == of).all()
    assert 5 < (of[lens > 32] & W.F_EMPTY == 0).sum() < (lens > 32).sum()
    pods = np.unique(np.concatenate([[0, P], r.integers(0, P, 30)])).astype(np.uint32)     # 1 to several terms a pod
    n_pods = len(pods) - 1
    bits, flags = empty_device(n_pods * words * 4, d), empty_device(n_pods, d)
    B.pv_eval_selector_terms(validator.ctx, n_pods, to_device(pods, d), P, to_device(offs, d), len(ex), to_device(ex, d),
                             to_device(assign[:n_pods], d), bits, words, flags)
    validator.sync()
    o, of = oracle.eval_selector_terms(n, 12, c.labels, pods, offs, ex, assign[:n_pods], words=words)
    assert (to_numpy(bits, np.uint32, (n_pods, words)) == o).all() and (to_numpy(flags, np.uint8) == of).all()


@pytest.mark.parametrize("n", [161, 5121])
@pytest.mark.parametrize("warps,more", [(24, 0), (24, 1), (40, 0), (40, 1)])
def test_terms_around_a_pod_a_warp(validator, n, warps, more):
    """As many pods as 24 or 40 warps an SM, and one more (the form with a pod to
    a warp runs between): 0 to 3 terms a pod and now and then 40, empty terms,
    more than 32 expressions, bad expressions, offsets that decrease."""
    P = SMS * warps + more
    r = np.random.default_rng(P + n)
    c = _cluster(n, 7)
    validator.load_cluster(c)
    terms = np.where(r.random(P) < 0.005, 40, r.integers(0, 4, P))
    pods = _offsets(terms)
    offs = _offsets(np.where(r.random(pods[-1]) < 0.004, r.integers(25, 60, pods[-1]), r.integers(0, 5, pods[-1])))
    offs[50:60] = offs[50:60][::-1]
    ex = _exprs(r, int(offs[-1]), bad=0.002)
    assign = r.integers(0, n + 2, P).astype(np.uint32)
    words, d = W.words_per_row(n), validator.device
    bits, flags = empty_device(P * words * 4, d), empty_device(P, d)
    B.pv_eval_selector_terms(validator.ctx, P, to_device(pods, d), len(offs) - 1, to_device(offs, d), len(ex),
                             to_device(ex, d), to_device(assign, d), bits, words, flags)
    validator.sync()
    o, of = oracle.eval_selector_terms(n, 12, c.labels, pods, offs, ex, assign)
    assert (to_numpy(bits, np.uint32, (P, words)) == o).all() and (to_numpy(flags, np.uint8) == of).all()
