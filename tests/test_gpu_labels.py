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


def _examples(h, ws, max_dist, cap):
    """gx_training_set with room for cap examples: (states found, histograms, labels)."""
    import torch
    dist = torch.empty(gx.stats(h)["table_slots"], dtype=torch.int32, device="cuda")
    hist = torch.zeros((max(cap, 1), 16), dtype=torch.uint8, device="cuda")
    label = torch.zeros(max(cap, 1), dtype=torch.float32, device="cuda")
    n = ctypes.c_uint64()
    gx._check(gx.lib().gx_training_set(h.handle, ws.data_ptr(), ws.numel(), None, dist.data_ptr(), max_dist,
                                       hist.data_ptr() if cap else None, label.data_ptr() if cap else None, cap,
                                       ctypes.byref(n)))
    k = min(n.value, cap)
    return n.value, hist[:k].cpu().numpy().astype(np.int64), label[:k].cpu().numpy()


@pytest.mark.parametrize("change", ["fewer", "more"])
@pytest.mark.parametrize("max_levels", [0, 5])
def test_labels_of_the_table_as_it_is_now(cuda, max_levels, change):
    """The examples are those of the states the workspace's table holds at the call: a third of
    them taken out, or states put in that the search had not found, each in its own bucket."""
    import torch
    net = inputs.planted_network(1, 4, n_traps=2)
    h = gx.load_network(net)
    o = gx.default_opts(table_bytes=1 << 22, hash_rounds=32, max_levels=max_levels, bucket_words=8, group_lanes=1,
                        global_cache_log2=0)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    s = gx.stats(h)
    assert s["slot_words"] == 1
    table = ws[ws.numel() - 4 * s["table_slots"]:].view(torch.int32)  # the last part of the workspace
    at = torch.nonzero(table).flatten()
    assert len(at) == s["states"]
    if change == "fewer":
        # (whole buckets' first slots only when nothing is behind them: a lookup ends at an empty slot)
        first = at[(at % 8 == 0) & (table[(at // 8) * 8 + 1] == 0)]
        table[first[::3]] = 0
    else:
        lay = gx.layout(h)
        top = int(lay["field_bits"].sum())
        have = set((table[at].cpu().numpy().astype(np.int64) & 0x7FFFFFFF).tolist())
        new = [v for v in range(1 << top) if v not in have][::7][:50]
        empty = torch.nonzero(table.view(-1, 8)[:, 0] == 0).flatten()[:len(new)]
        table[empty * 8] = torch.tensor([v - (1 << 31) for v in new], dtype=torch.int32, device="cuda")
    now = table[torch.nonzero(table).flatten()].cpu().numpy().astype(np.int64) & 0x7FFFFFFF
    lay = gx.layout(h)
    states = [tuple(int(v >> int(sh)) & ((1 << int(b)) - 1) for sh, b in zip(lay["field_offset"], lay["field_bits"]))
              for v in now]
    n, hist, label = _examples(h, ws, 8, len(states))
    assert n == len(states)
    if change == "more":  # put in at buckets of no meaning: no lookup finds them, and each is an example
        found = {tuple(int(v >> int(sh)) & ((1 << int(b)) - 1) for sh, b in zip(lay["field_offset"], lay["field_bits"]))
                 for v in have}
    else:
        found = set(states)
    succ = {x: [tuple(t) for t in oracle.successors(net, np.array(x, dtype=np.uint32))] for x in states}
    dist = {x: 0 for x in states if not succ[x]}
    for r in range(1, 9):
        near = [x for x in states if x not in dist and any(t in found and dist.get(t) == r - 1 for t in succ[x])]
        dist.update((x, r) for x in near)
    want = _rows(np.array([np.bincount(x, minlength=16) for x in states]),
                 [min(dist.get(x, 8), 8) / 8 for x in states], 8)
    assert _rows(hist, label, 8) == want


class _PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("loc_type", ctypes.c_int),
                ("loc_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@pytest.mark.parametrize("n_procs", [10, 11])
def test_labels_without_room_for_lists(cuda, n_procs):
    """A device memory pool of 32 MiB: it holds the lists of 1,080,000 states without their
    successors, and no lists of 5,400,000 states.  The call goes without them, counts with
    no memory at all, and writes examples of the same states."""
    import torch
    net = inputs.planted_network(1, n_procs, n_traps=2)
    h = gx.load_network(net)
    o = gx.default_opts(table_bytes=1 << 26, hash_rounds=32)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    states = gx.stats(h)["states"]
    too_much = 28 * states + (4 * gx.stats(h)["transitions"] if n_procs == 10 else 0)
    assert too_much > 2 * (32 << 20)
    n, hist, label = _examples(h, ws, 64, states)
    rows = lambda x, y: set(map(tuple, np.concatenate([x, np.rint(y * 64).astype(np.int64)[:, None]], 1).tolist()))
    want = rows(hist, label)
    cu = ctypes.CDLL("libcuda.so.1")
    default, small = ctypes.c_void_p(), ctypes.c_void_p()
    props = _PoolProps(alloc_type=1, loc_type=1, loc_id=torch.cuda.current_device(), max_size=32 << 20)
    assert cu.cuDeviceGetMemPool(ctypes.byref(default), torch.cuda.current_device()) == 0
    assert cu.cuMemPoolCreate(ctypes.byref(small), ctypes.byref(props)) == 0
    try:
        assert cu.cuDeviceSetMemPool(torch.cuda.current_device(), small) == 0
        p = ctypes.c_uint64()
        if cu.cuMemAllocFromPoolAsync(ctypes.byref(p), ctypes.c_size_t(too_much), small, None) == 0:
            cu.cuMemFreeAsync(p, None)
            pytest.skip("the driver does not hold the pool to its limit")
        assert _examples(h, ws, 64, 0)[0] == states
        n, hist, label = _examples(h, ws, 64, 1000)
        assert n == states and len(hist) == 1000
        assert rows(hist, label) <= want
    finally:
        assert cu.cuDeviceSetMemPool(torch.cuda.current_device(), default) == 0
        torch.cuda.synchronize()
        cu.cuMemPoolDestroy(small)


def test_labels_of_more_than_2_32_states(cuda):
    """The 5.37e9-state network in its 128 GiB table: counted and labelled without lists (their
    indexes have 32 bits).  No state of it is a deadlock, so every label is 1."""
    import torch
    free, _ = torch.cuda.mem_get_info()
    if free < (210 << 30):
        pytest.skip("needs 210 GiB of free device memory")
    h = gx.load_network(inputs.workload("scaled"))
    o = gx.default_opts(table_bytes=4 << 35, bucket_words=8, group_lanes=1, hash_rounds=64)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    s = gx.stats(h)
    assert s["states"] >= 1 << 32 and s["deadlock_count"] == 0
    n, hist, label = _examples(h, ws, 1, 4097)
    del ws
    torch.cuda.empty_cache()
    assert n == s["states"]
    assert (hist.sum(1) == 16).all() and (label == 1.0).all()
