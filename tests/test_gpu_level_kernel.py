"""The level kernel's queues, rounds and caches at the sizes where they can go wrong,
against the CPU oracle (bit-exact, including the digest of the visited set)."""
import pytest

import oracle
from paper_1801_05857_gb300 import gx, inputs

pytestmark = pytest.mark.gpu


def _mostly_still(n_procs, moving, n_states=2):
    """n_procs processes of which the first `moving` cycle through their states: n_states ** moving states."""
    cycle = [(s, 0, (s + 1) % n_states) for s in range(n_states)]
    return inputs.Network(1, [inputs.LTS(n_states, 0, cycle if p < moving else []) for p in range(n_procs)], [])


NETS = {
    1: inputs.random_network(7, 6, 8, 1, 3, 8, n_sync=2, parties=2),
    2: inputs.random_network(1, 10, 16, 1, 3, 12, n_sync=4, parties=2, cluster=4),
    4: inputs.random_network(1, 15, 16, 1, 3, 16, n_sync=8, parties=3, cluster=4),
}
_want = {}


def _oracle(key, net):
    if key not in _want:
        _want[key] = oracle.explore(net)
    return _want[key]


def _check(key, net, **opts):
    r = _oracle(key, net)
    h = gx.load_network(net)
    o = gx.default_opts(**opts)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    s = gx.stats(h)
    assert (s["states"], s["transitions"], gx.levels(h)) == (r.states, r.transitions, r.levels)
    assert (s["deadlock_count"], s["deadlock_sum"], s["deadlock_xor"]) == (r.deadlock_count, r.deadlock_sum,
                                                                          r.deadlock_xor)
    assert gx.set_digest(h, ws) == (r.states, r.set_sum, r.set_xor)
    return s


@pytest.mark.parametrize("bucket,group", [(4, 0), (8, 1), (8, 0), (16, 2), (32, 1), (32, 0)])
@pytest.mark.parametrize("W", [1, 2, 4])
def test_crowded_tables_take_further_hash_rounds(cuda, W, bucket, group):
    """The smallest power-of-two table that holds the states at up to 90 % (here 62-84 %):
    vectors that meet a full bucket go back to their warp's queue with the next
    hash-constant set (buckets of up to four slots certainly overflow)."""
    r = _oracle(W, NETS[W])
    slots = 1
    while slots < r.states / 0.9:
        slots *= 2
    s = _check(W, NETS[W], table_bytes=slots * 4 * W, frontier_states=slots, bucket_words=bucket,
               group_lanes=min(group, bucket // W), hash_rounds=64, warp_cache_log2=0, global_cache_log2=0)
    assert s["slot_words"] == W
    assert s["probes"] > r.transitions if bucket // W <= 4 else s["probes"] >= r.transitions


@pytest.mark.parametrize("log2", [1, 9, 16, 24, 25])
@pytest.mark.parametrize("W", [1, 2, 4])
def test_seen_cache_entries_of_every_width(cuda, W, log2):
    """Keys of 18, 40 and 60 bits in caches of 2^1 to 2^25 entries: entries of 16, 32 and 64
    bits, and indexes longer than the key."""
    s = _check(W, NETS[W], table_bytes=1 << 25, frontier_states=1 << 21, bucket_words=8, group_lanes=1,
               global_cache_log2=log2, warp_cache_log2=0)
    assert s["global_cache_entries"] == 1 << log2 and s["slot_words"] == W


@pytest.mark.parametrize("moving", [1, 2, 5, 13, 16])
@pytest.mark.parametrize("ctas", [1, 0])
def test_levels_below_at_and_above_one_state_per_warp(cuda, moving, ctas):
    """Binomial level sizes from 1 to 12,870 states, on a full grid and on 1216 warps."""
    s = _check(("still", moving), _mostly_still(20, moving), table_bytes=1 << 20, ctas_per_sm=ctas)
    assert s["states"] == 2 ** moving


@pytest.mark.parametrize("n_procs", [40, 70])
@pytest.mark.parametrize("ctas", [1, 0])
def test_levels_of_a_few_states_per_warp(cuda, n_procs, ctas):
    """The same levels with 2- and 4-word vectors: up to 11 states a warp, of which 1 to 8 are
    shared out among 32 to 4 lanes each."""
    s = _check(("few", n_procs), _mostly_still(n_procs, 16), table_bytes=1 << 22, ctas_per_sm=ctas)
    assert s["slot_words"] == (2 if n_procs == 40 else 4)


@pytest.mark.parametrize("n_procs", [31, 32, 33, 62])
def test_batched_networks_with_more_processes_than_lanes(cuda, n_procs):
    nets = [_mostly_still(n_procs, 9), _mostly_still(12, 7), NETS[1]]
    b = gx.batch_create(nets)
    o = gx.batch_opts(table_slots=1 << 16, hash_rounds=32)
    gx.batch_explore(b, o, gx.batch_alloc_workspace(b, o))
    for i, net in enumerate(nets):
        r = oracle.explore(net)
        s = gx.batch_stats(b, i)
        assert (s["states"], s["transitions"], gx.batch_levels(b, i)) == (r.states, r.transitions, r.levels)
        assert (s["deadlock_count"], s["deadlock_sum"]) == (r.deadlock_count, r.deadlock_sum)


@pytest.mark.parametrize("wide", [0, gx.BATCH_WIDE_OFF])
@pytest.mark.parametrize("count", [1, 32, 33, 70])
def test_batches_of_any_number_of_networks(cuda, count, wide):
    """Levels end network by network: one network alone, a full window of the search for
    open networks and one more; networks of very different depth and size, large ones last."""
    nets = [inputs.token_ring(3 + i % 6) if i % 2 else inputs.random_network(i, 4 + i % 4, 5, 0, 2, 6, n_sync=2, parties=2)
            for i in range(count)]
    b = gx.batch_create(nets)
    o = gx.batch_opts(table_slots=1 << 16, hash_rounds=32, wide_factor=wide)
    ws = gx.batch_alloc_workspace(b, o)
    for _ in range(2):
        gx.batch_explore(b, o, ws)
        for i, net in enumerate(nets):
            r = oracle.explore(net)
            s = gx.batch_stats(b, i)
            assert s["complete"] == 1
            assert (s["states"], s["transitions"], s["explored"]) == (r.states, r.transitions, r.explored)
            assert (s["deadlock_count"], s["deadlock_sum"]) == (r.deadlock_count, r.deadlock_sum)
            assert (s["first_deadlock_level"], gx.batch_levels(b, i)) == (r.first_deadlock_level, r.levels)


@pytest.mark.parametrize("words,bucket,group", [(1, 8, 8), (1, 8, 2), (1, 32, 32), (2, 16, 4), (4, 16, 4)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 100_003])
def test_find_or_put_of_any_number_of_keys(cuda, n, words, bucket, group):
    """The lanes of a warp take its keys as they become free: remainders of the 64 it holds,
    keys that occur twice, and (one hash-constant set, nearly full buckets) keys with no place."""
    import torch
    g = torch.Generator().manual_seed(n)
    some = torch.randint(0, 1 << 30, ((n + 1) // 2, words), generator=g, dtype=torch.int32)
    keys = torch.cat([some, some])[torch.randperm(2 * len(some), generator=g)][:n].contiguous()
    distinct = torch.unique(keys, dim=0)
    for rounds, slots in ((32, 4 * n), (1, n // 2)):
        table_words = max(2 * bucket, 1 << (slots * words - 1).bit_length())
        table = torch.zeros(table_words, dtype=torch.int32, device="cuda")
        counters = torch.zeros(3, dtype=torch.int64, device="cuda")
        result = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
        gx.find_or_put(keys.cuda(), words, table, counters, result, bucket, group, rounds)
        ins, fnd, full = counters.tolist()
        got = torch.bincount(result.cpu().long(), minlength=3).tolist()
        assert got == [fnd, ins, full] and ins + fnd + full == n
        # the table holds the inserted keys, each once, and every key that was placed
        rows = table.cpu().view(-1, words)
        held = rows[(rows != 0).all(1)] & 0x7FFFFFFF
        assert len(held) == ins == len(torch.unique(held, dim=0))
        placed = torch.unique(keys[result.cpu() != 2], dim=0)
        assert torch.equal(torch.unique(held, dim=0), placed)
        if rounds == 32:
            assert (ins, fnd, full) == (len(distinct), n - len(distinct), 0)


# 4-word vectors of 60, 64 (the longest 64-bit cache key, all ones reached) and 65 field bits
WIDE_NETS = {
    60: NETS[4],
    64: _mostly_still(16, 4, 16),
    65: inputs.Network(1, _mostly_still(16, 4, 16).procs + _mostly_still(1, 1).procs, []),
}
WIDE_NETS[64].procs[4:] = [inputs.LTS(16, 15, [])] * 12


@pytest.mark.parametrize("passes", [1, 2])
@pytest.mark.parametrize("log2", [1, 2, 3, 7])
@pytest.mark.parametrize("bits", [60, 64, 65])
def test_small_warp_caches_of_4_word_vectors_lose_no_state(cuda, bits, log2, passes):
    """The per-warp cache of 4-word vectors, entries of 8 bytes up to 64 field bits and of 16
    above: with a few of them every batch has many lanes that miss on the same entry, and
    only one of them may write it.  An entry made of two vectors could equal a third, which
    would then never be stored."""
    net = WIDE_NETS[bits]
    assert gx.layout(gx.load_network(net))["field_bits"].sum() == bits
    s = _check(("wide", bits), net, table_bytes=1 << 24, bucket_words=8, group_lanes=1, hash_rounds=32, host_loop=1,
               region_passes=passes, warp_cache_log2=log2, global_cache_log2=0)
    assert s["slot_words"] == 4 and s["region_passes"] == passes and s["global_cache_entries"] == 0


@pytest.mark.parametrize("passes", [1, 2])
@pytest.mark.parametrize("n", [6, 7])
def test_few_state_levels_hand_over_in_a_stopped_search(cuda, n, passes):
    """A search whose levels grow past the few-state kernel's limit (512 states) stops at its
    first deadlock: what that kernel did before the hand-over, the large levels after it
    (one or two region passes) and the stop give the oracle's results."""
    net = inputs.random_network(8, n, 8, 0, 3, 8, n_sync=n - 1, parties=2)
    r = _want[("stopped", n)] = oracle.explore(net, stop_at_first_deadlock=True)
    assert max(r.levels) > 512 and r.deadlock_count and not r.complete
    s = _check(("stopped", n), net, table_bytes=1 << 24, bucket_words=8, group_lanes=1, hash_rounds=32,
               region_passes=passes, stop_at_first_deadlock=1)
    assert s["complete"] == 0 and s["first_deadlock_level"] == r.first_deadlock_level


def _star(n_states, n_procs, moving):
    """One process that can go from its first state to any of n_states - 1 others (its tables take
    8 n_states bytes), beside n_procs two-state processes of which `moving` cycle."""
    net = _mostly_still(n_procs, moving)
    net.procs.append(inputs.LTS(n_states, 0, [(0, 0, s) for s in range(1, n_states)]))
    return net


@pytest.mark.parametrize("loop", [0, 1])
def test_networks_of_different_table_sizes_take_turns(cuda, loop):
    """Kernels staged with 0.5, 56 and 40 KB of network tables and with an explicit warp cache,
    one after the other and again on their cached graphs: what one search asks of a kernel
    (shared memory, its split with the L1) is not changed by another's."""
    runs = []
    for key, net, kw in [("small", _mostly_still(70, 5), {}), ("star7000", _star(7000, 70, 2), {}),
                         ("star5000", _star(5000, 70, 2), dict(warp_cache_log2=9)),
                         ("small_cached", _mostly_still(70, 6), dict(global_cache_log2=16))]:
        o = gx.default_opts(table_bytes=1 << 24, bucket_words=8, group_lanes=1, hash_rounds=32, host_loop=loop, **kw)
        h = gx.load_network(net)
        runs.append((key, net, h, o, gx.alloc_workspace(h, o)))
    for order in ([0, 1, 2, 3], [1, 0, 2, 1, 3, 2, 0, 1]):
        for i in order:
            key, net, h, o, ws = runs[i]
            r = _oracle(key, net)
            gx.explore(h, o, ws)
            s = gx.stats(h)
            assert (s["states"], s["transitions"], gx.levels(h)) == (r.states, r.transitions, r.levels)
            assert s["slot_words"] == 4 and gx.set_digest(h, ws) == (r.states, r.set_sum, r.set_xor)


def test_searches_of_several_threads(cuda):
    """Four threads, a stream and a network each, of different table sizes and caches: every
    search takes the shared memory it needs, whatever the others ask for in between."""
    import threading
    import torch
    runs = [("small", _mostly_still(70, 5), {}), ("star7000", _star(7000, 70, 2), {}),
            ("star5000", _star(5000, 70, 2), dict(warp_cache_log2=9, host_loop=1)),
            ("small_cached", _mostly_still(70, 6), dict(global_cache_log2=16))]
    want = [_oracle(key, net) for key, net, _ in runs]
    bad = []

    def work(i):
        try:
            torch.cuda.set_device(0)
            key, net, kw = runs[i]
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                o = gx.default_opts(table_bytes=1 << 22, bucket_words=8, group_lanes=1, hash_rounds=32, **kw)
                for _ in range(5):  # (a handle each: its graph is built anew)
                    h = gx.load_network(net)
                    ws = gx.alloc_workspace(h, o)
                    for _ in range(4):
                        gx.explore(h, o, ws, stream)
                        s = gx.stats(h)
                        assert (s["states"], s["transitions"], gx.levels(h)) == (
                            want[i].states, want[i].transitions, want[i].levels), key
                    stream.synchronize()
        except Exception as e:  # noqa: BLE001 -- reported by the main thread
            bad.append((runs[i][0], repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(runs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad


def test_workspace_without_room_for_the_automatic_cache(cuda):
    """4-word vectors in 2^26 slots: a workspace with no room for the GPU-wide cache is searched
    without it; one byte less is refused."""
    import torch
    h = gx.load_network(NETS[4])
    kw = dict(table_bytes=1 << 30, bucket_words=8, group_lanes=1, hash_rounds=32)
    need = gx.workspace_bytes(h, gx.default_opts(global_cache_log2=0, **kw))
    full = gx.workspace_bytes(h, gx.default_opts(**kw))
    assert full > need
    r = _oracle(4, NETS[4])
    for size, entries in ((full, 1 << 23), (need, 0)):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        gx.explore(h, gx.default_opts(**kw), ws)
        s = gx.stats(h)
        assert (s["states"], s["transitions"], gx.levels(h)) == (r.states, r.transitions, r.levels)
        assert gx.set_digest(h, ws) == (r.states, r.set_sum, r.set_xor)
        assert s["slot_words"] == 4 and s["global_cache_entries"] == entries
    with pytest.raises(gx.GxError) as e:
        gx.explore(h, gx.default_opts(**kw), torch.empty(need - 1, dtype=torch.uint8, device="cuda"))
    assert e.value.status == gx.GX_ERR_OOM


@pytest.mark.parametrize("passes", [1, 2])
@pytest.mark.parametrize("net", [inputs.workload("tiny"), inputs.token_ring(8), NETS[4]], ids=lambda n: n.name or "net")
def test_launch_count_counts_a_launch_once(cuda, net, passes):
    """The few-state kernel is launched at the start and whenever a level falls to 256 states, and
    takes levels of up to 512; every other level is an expansion per region pass and an advance
    step.  With levels driven by the host each expansion is a launch."""
    h = gx.load_network(net)
    o = gx.default_opts(table_bytes=1 << 24, hash_rounds=32, region_passes=passes)
    gx.explore(h, o, gx.alloc_workspace(h, o))
    sizes, n, i = gx.levels(h), 2, 0  # initialisation, start
    while i < len(sizes):
        n += 1
        while i < len(sizes) and sizes[i] <= 512:
            i += 1
        while i < len(sizes):
            n += passes + 1
            i += 1
            if i < len(sizes) and sizes[i] <= 256:
                break
    assert gx.launch_count(h) == n
    o = gx.default_opts(table_bytes=1 << 24, hash_rounds=32, region_passes=passes, host_loop=1)
    gx.explore(h, o, gx.alloc_workspace(h, o))
    assert gx.launch_count(h) == 1 + passes * len(sizes)


@pytest.mark.parametrize("W", [1, 2, 4])
def test_partitioned_levels_ask_the_gpu_wide_cache(cuda, W):
    """Levels expanded by the partitioned path leave out the bucket reads of vectors that the
    GPU-wide cache holds, as the level kernel does; without the cache every successor reads."""
    kw = dict(table_bytes=1 << 26, hash_rounds=32, bucket_words=8, group_lanes=1, partition_min_states=1,
              warp_cache_log2=0)
    r = _oracle(W, NETS[W])
    s = _check(W, NETS[W], global_cache_log2=0, **kw)
    assert s["partitioned_levels"] == s["n_levels"] and s["probes"] >= r.transitions
    s = _check(W, NETS[W], global_cache_log2=20, **kw)
    assert s["partitioned_levels"] == s["n_levels"] and s["global_cache_entries"] == 1 << 20
    assert s["probes"] < 0.8 * r.transitions


@pytest.mark.parametrize("opts", [dict(), dict(global_cache_log2=0), dict(region_passes=2), dict(host_loop=1, region_passes=4),
                                  dict(warp_cache_log2=2, global_cache_log2=0, group_lanes=2)], ids=str)
@pytest.mark.parametrize("bits", [60, 64, 65])
def test_4_word_vectors_in_large_tables(cuda, bits, opts):
    """Tables of 2^26 slots and more run level kernels of their own for 4-word vectors (one state
    per lane in every level): the same networks as in the small tables above."""
    kw = dict(table_bytes=1 << 30, hash_rounds=32, bucket_words=8, group_lanes=1)
    kw.update(opts)
    s = _check(("wide", bits), WIDE_NETS[bits], **kw)
    assert s["slot_words"] == 4 and s["table_slots"] == 1 << 26
