"""Compliant reach where the library's choice of kernel changes: the hub search
of directed graphs (taken when there are more (mask, 64 sources) items than
blocks fit the GPU at once) and the component table of symmetric ones, against
the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_16100_gb300 import binding as B
from paper_2602_16100_gb300 import workloads as W
from paper_2602_16100_gb300.validator import Validator, to_device, to_numpy

pytestmark = pytest.mark.gpu

HUB_MIN_V = 1000   # kHubMinV of the library
# more than this many (mask, 64 sources) items on HUB_MIN_V vertices or more: hub search
ITEMS = 4 * (torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1)


def _graph(V, a, b, regions, seed):
    o = np.lexsort((b, a))
    a, b = np.asarray(a)[o], np.asarray(b)[o]
    offs = np.zeros(V + 1, np.int64)
    np.add.at(offs, a + 1, 1)
    return W.Graph(V, np.cumsum(offs).astype(np.uint32), b.astype(np.uint32),
                   np.random.default_rng(seed).integers(0, regions, V).astype(np.uint8))


def _check(v, g, src, masks, components):
    out = v.compliant_reach(v.upload_graph(g), len(src), to_device(src.astype(np.uint32), v.device), len(masks),
                            to_device(masks.astype(np.uint32), v.device))
    v.sync()
    assert B.pv_get_stat(v.ctx, B.PV_STAT_REACH_COMPONENTS) == components
    want = oracle.compliant_reach(g, src.astype(np.uint32), masks.astype(np.uint32))
    assert (to_numpy(out, np.uint32, want.shape) == want).all()


def _edges(kind, V, r):
    if kind == "giant":          # one large strongly connected component and tendrils
        return r.integers(0, V, 6 * V), r.integers(0, V, 6 * V)
    if kind == "dag":            # none: every source is swept
        a, b = r.integers(0, V, 4 * V), r.integers(0, V, 4 * V)
        return np.minimum(a, b), np.maximum(a, b)
    if kind == "tail":           # a component whose sources outside it reach more than a queue holds
        core, n = V // 2, 6 * (V // 2)
        path = np.arange(core, V - 1)
        return np.concatenate([r.integers(0, core, n), path, path[-1:] + 1]), \
            np.concatenate([r.integers(0, core, n), path + 1, [0]])
    if kind == "two":            # two components, the first hub may sit in the smaller
        h = V // 3
        return np.concatenate([r.integers(0, h, 8 * h), r.integers(h, V, 5 * (V - h))]), \
            np.concatenate([r.integers(0, h, 8 * h), r.integers(h, V, 5 * (V - h))])
    if kind == "ring":           # as many levels as vertices, each in the component
        return np.arange(V), (np.arange(V) + 1) % V
    if kind == "spur":           # the same with a dead end, past the levels that are searched
        return np.concatenate([np.arange(V - 1), [0]]), np.concatenate([(np.arange(V - 1) + 1) % (V - 1), [V - 1]])
    a = np.arange(V - 1)         # a long path: searched for some levels only
    return a, a + 1


@pytest.mark.parametrize("kind", ["giant", "dag", "tail", "two", "path", "ring", "spur"])
@pytest.mark.parametrize("V,num_masks", [(700, 64), (HUB_MIN_V - 1, 64), (HUB_MIN_V, 64), (1321, 120)])
def test_hub_search(validator, kind, V, num_masks):
    r = np.random.default_rng(V + len(kind))
    g = _graph(V, *_edges(kind, V, r), 5, 3)
    src = np.concatenate([np.arange(V), [0, V - 1, V, 0xFFFFFFFF]])      # duplicates, out of range
    masks = r.integers(0, 32, num_masks)
    masks[:3] = [31, 0, 1]
    assert (len(src) + 63) // 64 * num_masks > ITEMS
    _check(validator, g, src, masks, 0)


@pytest.mark.parametrize("past", [0, 1])
def test_either_side_of_the_item_limit(validator, past):
    masks = ITEMS // 2 + past
    r = np.random.default_rng(masks)
    g = _graph(1030, *_edges("giant", 1030, r), 4, 1)
    _check(validator, g, np.arange(128), r.integers(1, 16, masks), 0)


@pytest.mark.parametrize("bad", ["offsets", "columns"])
def test_hub_search_malformed(validator, bad):
    """Malformed offsets (no edges) and columns out of range (skipped), reported by the next sync."""
    r = np.random.default_rng(9)
    g = _graph(1200, *_edges("giant", 1200, r), 3, 2)
    if bad == "offsets":
        g.offs[200] = g.offs[-1] + 7
    else:
        g.cols[::9] = 1200 + np.arange(len(g.cols[::9]))
    src, masks = np.arange(1200), r.integers(0, 8, 100)
    v = validator
    out = v.compliant_reach(v.upload_graph(g), 1200, to_device(src.astype(np.uint32), v.device), 100,
                            to_device(masks.astype(np.uint32), v.device))
    with pytest.raises(B.PVError) as e:
        v.sync()
    assert e.value.code == B.PV_EINVAL
    assert B.pv_get_stat(v.ctx, B.PV_STAT_REACH_COMPONENTS) == (1 if bad == "offsets" else 0)
    want = oracle.compliant_reach(g, src.astype(np.uint32), masks.astype(np.uint32))
    assert (to_numpy(out, np.uint32, want.shape) == want).all()


@pytest.mark.parametrize("group,num_masks", [(1, 7), (2, 2000), (5, 2000), (2, 7)])
def test_component_table(validator, group, num_masks):
    """Vertices alone, and components of `group`: fewer and more of them than
    the mask's table holds (2,000 masks leave it 262 rows)."""
    V = 2003
    v = np.arange(V)
    a = v[(v % group != group - 1) & (v + 1 < V)] if group > 1 else v[:0]
    g = _graph(V, np.concatenate([a, a + 1]), np.concatenate([a + 1, a]), 3, 4)
    r = np.random.default_rng(group)
    src = np.concatenate([r.integers(0, V, 5), [V - 1, 0, V]])
    _check(validator, g, src, r.integers(0, 8, num_masks), 1)


def _pairs_graph(V):
    """Components of two vertices, one region."""
    a = np.arange(0, V - 1, 2)
    return _graph(V, np.concatenate([a, a + 1]), np.concatenate([a + 1, a]), 1, 4)


def test_scratch_stays_bounded(validator):
    """The component table takes 128 MB at most, whatever the caller's rows
    (1 GB here); components past it are exact."""
    v, V, masks = Validator(0), 8192, np.ones(64, np.uint32)
    masks[::3] = 2
    try:
        g, src = _pairs_graph(V), np.arange(2 * V) % V
        out = v.compliant_reach(v.upload_graph(g), len(src), to_device(src.astype(np.uint32), v.device), 64,
                                to_device(masks, v.device))
        v.sync()
        assert B.pv_get_stat(v.ctx, B.PV_STAT_SCRATCH_BYTES) < 180 << 20
        rows = out.view(torch.int32).view(64, len(src), -1)
        want = oracle.compliant_reach(g, src.astype(np.uint32), masks[:2])
        assert (to_numpy(rows[:2].contiguous().view(torch.uint8).flatten(), np.uint32, want.shape) == want).all()
        for m in range(2, 64):
            assert torch.equal(rows[m], rows[0 if m % 3 == 0 else 1])
    finally:
        v.close()


def _fill_memory():
    """Tensors that leave about 16 to 32 MB of the GPU's memory (what other
    allocators hold unused included)."""
    torch.cuda.empty_cache()
    hold = [torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")]
    for chunk in (64 << 20, 16 << 20):
        try:
            while True:
                hold.append(torch.empty(chunk, dtype=torch.uint8, device="cuda"))
        except torch.cuda.OutOfMemoryError:
            pass
    del hold[-1]
    torch.cuda.empty_cache()
    return hold


@pytest.mark.parametrize("directed", [False, True])
def test_little_memory_left(validator, directed):
    """Beside rows that leave little memory the call still runs (by sweeps)."""
    v, V = Validator(0), 4096
    try:
        if directed:
            g = _graph(V, *_edges("giant", V, np.random.default_rng(2)), 5, 3)
        else:
            g = _pairs_graph(V)
        src, masks = np.arange(V).astype(np.uint32), np.array([31, 1, 6] * 21 + [2], np.uint32)
        graph, d_src, d_masks = v.upload_graph(g), to_device(src, v.device), to_device(masks, v.device)
        out = torch.zeros(len(masks) * V * (V // 8), dtype=torch.uint8, device="cuda")
        v.sync()
        torch.cuda.synchronize()
        hold = _fill_memory()
        try:
            v.compliant_reach(graph, V, d_src, len(masks), d_masks, d_reach=out)
            v.sync()
        finally:
            del hold
            torch.cuda.empty_cache()
        assert B.pv_get_stat(v.ctx, B.PV_STAT_SCRATCH_BYTES) < 40 << 20      # the table would take 64 MB
        want = oracle.compliant_reach(g, src, masks[:3])
        assert (to_numpy(out[: want.size * 4], np.uint32, want.shape) == want).all()
    finally:
        v.close()


@pytest.mark.parametrize("V,num_masks", [(1, 1), (31, 3), (1023, 1), (1024, 2), (3001, 1), (3001, 40), (9001, 5),
                                         (16384, 1), (16384, 17)])
def test_few_masks_and_rows(validator, V, num_masks):
    """Several blocks to a mask's table and few rows to a warp: components of
    one to many vertices, some of them whole regions apart."""
    r = np.random.default_rng(V)
    a, b = r.integers(0, V, V // 2), r.integers(0, V, V // 2)
    g = _graph(V, np.concatenate([a, b]), np.concatenate([b, a]), 4, V)
    src = np.concatenate([r.integers(0, V, min(V, 700)), [0, V - 1, V]])
    _check(validator, g, src, np.concatenate([[15], r.integers(0, 16, num_masks - 1)]), 1)
