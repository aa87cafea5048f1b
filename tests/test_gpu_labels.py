"""Distance labels at the sizes where the labelling kernels can go wrong: lists below, at and
above a sorting tile, searches stopped early (successors looked up every round instead of kept),
capped outputs."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1801_05857_gb300 import gx, inputs

pytestmark = pytest.mark.gpu


def _rows(hist, label, max_dist):
    return sorted(zip(map(tuple, hist), [int(round(float(x) * max_dist)) for x in label]))


def _expected(net, levels, max_dist):
    """Histograms and distances of the states of the first `levels` levels, by their definition:
    distances run through stored states only."""
    seen = {tuple(p.initial for p in net.procs)}
    succ, level = {}, list(seen)
    for _ in range(levels):
        fresh = []
        for s in level:
            succ[s] = [tuple(t) for t in oracle.successors(net, np.array(s, dtype=np.uint32))]
            for t in succ[s]:
                if t not in seen:
                    seen.add(t)
                    fresh.append(t)
        level = fresh
    for s in level:  # found, not expanded by the search
        succ[s] = [tuple(t) for t in oracle.successors(net, np.array(s, dtype=np.uint32))]
    dist = {s: 0 for s in seen if not succ[s]}
    for r in range(1, max_dist + 1):
        near = [s for s in seen if s not in dist and any(dist.get(t) == r - 1 for t in succ[s])]
        if not near:
            break
        dist.update((s, r) for s in near)
    hist = np.array([np.bincount(s, minlength=16) for s in seen])
    return _rows(hist, [min(dist.get(s, max_dist), max_dist) / max_dist for s in seen], max_dist)


def _label(net, max_levels, max_dist, cap=None):
    import torch
    h = gx.load_network(net)
    o = gx.default_opts(table_bytes=1 << 20, hash_rounds=32, max_levels=max_levels, bucket_words=8, group_lanes=1)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    s = gx.stats(h)
    if cap is None:
        hist, label = gx.training_set(h, ws, max_dist)
    else:
        dist = torch.empty(s["table_slots"], dtype=torch.int32, device="cuda")
        hist = torch.zeros((max(cap, 1), 16), dtype=torch.uint8, device="cuda")
        label = torch.zeros(max(cap, 1), dtype=torch.float32, device="cuda")
        n = ctypes.c_uint64()
        gx._check(gx.lib().gx_training_set(h.handle, ws.data_ptr(), ws.numel(), None, dist.data_ptr(), max_dist,
                                           hist.data_ptr(), label.data_ptr(), cap, ctypes.byref(n)))
        assert n.value == s["states"]
        hist, label = hist[:cap], label[:cap]
    return s, hist.cpu().numpy().astype(np.int64), label.cpu().numpy()


@pytest.mark.parametrize("max_levels", [0, 1, 5, 9])
@pytest.mark.parametrize("max_dist", [1, 3, 64])
@pytest.mark.parametrize("net", [inputs.random_network(6, 5, 5, 0, 2, 6, n_sync=2, parties=2),
                                 inputs.planted_network(1, 4, n_traps=2)], ids=lambda n: n.name)
def test_labels_of_complete_and_stopped_searches(cuda, net, max_dist, max_levels):
    s, hist, label = _label(net, max_levels, max_dist)
    assert _rows(hist, label, max_dist) == _expected(net, max_levels or s["n_levels"], max_dist)


@pytest.mark.parametrize("cap", [1, 2, 3, 1023, 1024, 1025, 2047, 2048, 2049, 4097, 9000])
def test_examples_come_sorted_at_every_size(cuda, cap):
    """Outputs capped below, at and above the sort's tile (and its power-of-two padding)."""
    net = inputs.token_ring(7)  # 10,206 states
    s, hist, label = _label(net, 0, 16, cap=cap)
    n = min(cap, s["states"])
    words = np.ascontiguousarray(hist.astype(np.uint8)).view("<u4").reshape(n, 4)
    keys = [tuple(w) + (float(x),) for w, x in zip(words.tolist(), label)]
    assert keys == sorted(keys)
    assert hist.sum(1).tolist() == [7] * n  # every row is a state's histogram


@pytest.mark.parametrize("offset", [1, 4, 8])
@pytest.mark.parametrize("cap", [1, 2, 2049, 10206])
def test_examples_at_odd_addresses(cuda, cap, offset):
    """The histograms' address need not be a multiple of 16: the same examples as at one (with
    cap below the states found, which ones are written is open: they are sorted histograms)."""
    import torch
    net = inputs.token_ring(7)  # 10,206 states
    h = gx.load_network(net)
    o = gx.default_opts(table_bytes=1 << 20, hash_rounds=32)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    s = gx.stats(h)
    dist = torch.empty(s["table_slots"], dtype=torch.int32, device="cuda")
    flat = torch.full((16 * cap + offset + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    assert flat.data_ptr() % 16 == 0
    label = torch.zeros(cap, dtype=torch.float32, device="cuda")
    n = ctypes.c_uint64()
    gx._check(gx.lib().gx_training_set(h.handle, ws.data_ptr(), ws.numel(), None, dist.data_ptr(), 16,
                                       flat.data_ptr() + offset, label.data_ptr(), cap, ctypes.byref(n)))
    assert n.value == s["states"]
    got = flat.cpu().numpy()
    assert (got[:offset] == 0xA5).all() and (got[offset + 16 * cap:] == 0xA5).all()
    hist = got[offset:offset + 16 * cap].reshape(cap, 16)
    keys = [tuple(w) + (float(x),) for w, x in zip(np.ascontiguousarray(hist).view("<u4").tolist(), label.cpu())]
    assert keys == sorted(keys) and (hist.sum(1) == 7).all()
    if cap >= s["states"]:
        want_hist, want_label = gx.training_set(h, ws, 16)
        assert (want_hist.cpu().numpy() == hist).all() and torch.equal(want_label, label)
