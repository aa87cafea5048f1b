"""Performance cases of the framework: the work its users have it do, through its public entry points.

A case is a dict of plain values; `kind` says which part of the framework it exercises:

  explore  full breadth-first exploration of one network (gx.explore): 1-, 2- and 4-word
           vectors, default and tuned table layouts, the safety check, region passes
  search   breadth-first deadlock search that stops at the first deadlock (gx.find_deadlocks)
  guided   deadlock search ordered by a trained scoring network (gx.find_deadlocks)
  batch    many networks in one call (gx.batch_explore)
  score    the scoring network on many states (gx.mlp_forward)
  train    Adam steps on the scoring network (gx.mlp_train)
  label    distance labels of every state of an explored network (gx.training_set)
  table    find-or-put of a key sequence (gx.find_or_put)

The networks come from paper_1801_05857_gb300.inputs with fixed generator arguments, so that a
case's size is known.  Another seed of `prepare` gives another presentation of the network
(processes reordered, local states renumbered): other vectors, hashes and table positions, the
same counts, another digest of the visited set.  Keys, training data and weights are drawn from the seed itself.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1801_05857_gb300 import guide, gx, inputs

# States found by a breadth-first search up to the first deadlock (level 2 n) in
# planted_network(seed, n, n_traps=2), seeds 0..4, for n processes.
PLANTED_SEARCH = {
    6: [10428, 4800, 5760, 7800, 15000],
    7: [34500, 24000, 28800, 30000, 62500],
    8: [247492, 72000, 69120, 150000, 375000],
    9: [1125000, 450000, 345600, 750000, 1875000],
    10: [5625000, 1080000, 1728000, 2250000, 9375000],
    11: [22500000, 5400000, 5529600, 11250000, 46875000],
    12: [140625000, 27000000, 34560000, 45000000, 243750000],
}
# All states of the same networks.
PLANTED_STATES = {
    6: [10440, 4800, 5760, 7800, 15000],
    7: [34500, 24000, 28800, 30000, 62500],
    8: [247500, 72000, 69120, 150000, 375000],
}
# States of the first k networks of the batched workload.
BATCH_STATES = {8: 1740944, 16: 2357840, 32: 4526151, 64: 9348558, 128: 16224222, 256: 30539206}

SCORE_FLOPS = 2 * (16 * 128 + 128 * 128 + 128)  # one state through the scoring network


def listed():
    return [
        # the smallest call: a model of a few hundred states while it is being written
        # (4 processes x 8 states, 32-word buckets, every other option left at its default)
        dict(name="explore_tiny", kind="explore", family="random", gen_seed=0, n_procs=4, n_states=8,
             deg_hi=3, n_labels=6, n_sync=2, parties=2, cluster=0, sync_weight=1.0, table_bytes=4 << 16,
             bucket=32, group=0, rounds=8, passes=0, watch=False, states=640),
        # the token ring of the scaling table with a safety property, default options
        dict(name="explore_ring_safety", kind="explore", family="ring", n_procs=11, table_bytes=1 << 26,
             bucket=8, group=0, rounds=8, passes=0, watch=True, states=22 * 3 ** 10),
        # an ordinary large model: 10 processes x 16 states, 2-word vectors, 6.2e7 states in a
        # 1 GiB table with the layout the bucket sweep recommends (8 words, one lane)
        dict(name="explore_mid", kind="explore", family="random", gen_seed=11, n_procs=10, n_states=16,
             deg_hi=3, n_labels=12, n_sync=4, parties=2, cluster=8, sync_weight=1.0, table_bytes=1 << 30,
             bucket=8, group=1, rounds=32, passes=0, watch=False, states=62208000),
        # wide vectors: 16 processes (3 words, padded to 4), 3-party rules, 1.1e8 states in 4 GiB
        dict(name="explore_wide", kind="explore", family="random", gen_seed=6, n_procs=16, n_states=16,
             deg_hi=2, n_labels=30, n_sync=3, parties=3, cluster=5, sync_weight=6.0, table_bytes=4 << 30,
             bucket=8, group=1, rounds=32, passes=0, watch=False, states=107520000),
        # memory-filling runs: the product network of the memory-scaled workload with the two
        # region passes its 128 GiB table takes, in 8 GiB (3.4e8 states, 62.5 % fill)
        dict(name="explore_filling", kind="explore", family="product", gen_seed=7, n_procs=16, n_states=16,
             blocks="4,4,4,4,4,4,4,4,4,4,4,4,4,5,1,1", n_labels=30, deg_hi=2, table_bytes=8 << 30,
             bucket=8, group=1, rounds=64, passes=2, watch=False, states=4 ** 13 * 5),
        # deadlock search on a model with planted deadlocks, breadth-first
        dict(name="search_bfs", kind="search", net_seed=3, n_procs=12, n_traps=2, table_bytes=1 << 30,
             bucket=8, group=1, rounds=32),
        # the same question asked with a trained guide on a larger model
        dict(name="search_guided", kind="guided", net_seed=1, n_procs=14, n_traps=1, table_bytes=1 << 30, rounds=32),
        # a family of small models checked in one call
        dict(name="batch_256", kind="batch", count=256, bucket=8, group=1, rounds=32, chunk=32),
        # scores of every open state of a large search; a ragged last tile
        dict(name="score_4m", kind="score", n=4000037),
        # training the guide: mini-batches of 1024 from 2^20 labelled states
        dict(name="train_guide", kind="train", n=1 << 20, batch=1024, steps=200, lr=1e-3),
        # labelling one training network (8 processes) with distances to the nearest deadlock
        dict(name="label_states", kind="label", net_seed=1, n_procs=8, n_traps=2, table_bytes=1 << 26, max_dist=64),
        # the isolated hash table: 1e8 distinct keys into 2^27 slots (74.5 % fill), half of them
        # first, then the other half mixed with as many that are known
        dict(name="table_100m", kind="table", distinct=100_000_000, first=50_000_000, second=100_000_000, words=1,
             log2_slots=27, bucket=8, group=1, rounds=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2_at_least(x):
    return 1 << max(0, math.ceil(math.log2(max(1, x))))


def _slot_words(n_procs, n_states):
    bits = max(1, (n_states - 1).bit_length())
    words = -(-n_procs // (31 // bits))
    return 4 if words == 3 else words


def _layout(rng, words):
    """Bucket words, lanes per bucket (0: the default, one lane per slot) and hash rounds."""
    bucket = rng.choice([b for b in (4, 8, 8, 8, 16, 32) if b >= words])
    return dict(bucket=bucket, group=rng.choice([0, 1, 1]), rounds=rng.choice([32, 64]))


def _frontier(slots):
    """Small state spaces have few levels, two of which must fit the frontier together: as large
    as the table.  0: the default, a quarter of it."""
    return slots if slots < 1 << 22 else 0


def draw(rng):
    kind = rng.choice(["ring", "ring", "product", "product", "product", "search", "guided", "batch", "score",
                       "train", "label", "table", "table"])
    if kind == "ring":
        n = rng.randint(2, 14)
        w = _slot_words(n, 5)
        states = 2 * n * 3 ** (n - 1)
        slots = _pow2_at_least(max(4096, states * rng.uniform(1.5, 4.0)))
        return dict(kind="explore", family="ring", n_procs=n, table_bytes=max(1 << 16, slots * 4 * w), passes=0, frontier=_frontier(slots),
                    watch=rng.random() < 0.5, states=states, **_layout(rng, w))
    if kind == "product":
        # blocks of 2..5 local states until the drawn number of states is reached
        want = _log_int(rng, 1000, 200_000_000)
        blocks, states = [], 1
        while states < want and len(blocks) < 20:
            blocks.append(rng.randint(2, 5))
            states *= blocks[-1]
        n_states = rng.choice([5, 7, 8, 11, 16])
        w = _slot_words(len(blocks), n_states)
        slots = _pow2_at_least(max(4096, states * rng.uniform(1.45, 3.0)))
        return dict(kind="explore", family="product", gen_seed=rng.randint(0, 99), n_procs=len(blocks), n_states=n_states,
                    blocks=",".join(map(str, blocks)), n_labels=30, deg_hi=rng.choice([2, 3]),
                    table_bytes=slots * 4 * w, frontier=_frontier(slots), passes=rng.choice([0, 0, 0, 2, 4]), watch=False,
                    states=states, **_layout(rng, w))
    if kind == "search":
        n, net_seed = rng.randint(6, 12), rng.randint(0, 4)
        slots = _pow2_at_least(PLANTED_SEARCH[n][net_seed] * rng.uniform(1.5, 3.0))
        return dict(kind="search", net_seed=net_seed, n_procs=n, n_traps=2, frontier=_frontier(slots),
                    table_bytes=slots * 8, **_layout(rng, 2))
    if kind == "guided":
        return dict(kind="guided", net_seed=rng.randint(0, 4), n_procs=rng.randint(10, 16), n_traps=1,
                    table_bytes=2 << 30, rounds=32)
    if kind == "batch":
        return dict(kind="batch", count=rng.choice(sorted(BATCH_STATES)), bucket=rng.choice([8, 8, 16]), group=1,
                    rounds=32, chunk=rng.choice([32, 64, 128]))
    if kind == "score":
        return dict(kind="score", n=_log_int(rng, 1, 4_000_000))
    if kind == "train":
        return dict(kind="train", n=_log_int(rng, 5_000, 1 << 20), batch=_log_int(rng, 32, 8192),
                    steps=rng.randint(20, 200), lr=1e-3)
    if kind == "label":
        return dict(kind="label", net_seed=rng.randint(0, 4), n_procs=rng.randint(6, 8), n_traps=2,
                    table_bytes=1 << 26, max_dist=rng.choice([32, 64]))
    words = rng.choice([1, 1, 2, 4])
    # duplication: lookups per new key in the second call
    dup = rng.choice([1.5, 2, 5, 21, 100])
    total = _log_int(rng, 10_000, 150_000_000 // words)
    new = max(1, int(total / (1 + dup)))
    first = max(1, min(new, total // 2))
    distinct = first + new
    log2_slots = max(12, math.ceil(math.log2(distinct * rng.uniform(1.34, 3.0))))
    return dict(kind="table", distinct=distinct, first=first, second=max(new, total - first), words=words,
                log2_slots=log2_slots, **_layout(rng, words))


# ---- networks

def _relabel(net, seed, states=True):
    """The same network with its processes in another order and, with `states`, their local
    states numbered differently."""
    r = random.Random(seed)
    order = list(range(net.n_procs))
    r.shuffle(order)  # new process i is old process order[i]
    place = {old: new for new, old in enumerate(order)}
    procs = []
    for old in order:
        p = net.procs[old]
        perm = list(range(p.n_states))
        if states:
            r.shuffle(perm)
        procs.append(inputs.LTS(p.n_states, perm[p.initial], [(perm[s], a, perm[t]) for s, a, t in p.edges]))
    rules = [inputs.Rule([(place[p], a) for p, a in rule.parts], rule.result) for rule in net.rules]
    return inputs.Network(net.n_labels, procs, rules, name=net.name)


def _network(case, seed):
    """The network of an explore, search, guided or label case, and the watched (process, state)."""
    if case["kind"] != "explore":
        net = inputs.planted_network(case["net_seed"], case["n_procs"], n_traps=case["n_traps"])
        if case["kind"] != "guided":
            return _relabel(net, seed), None
        # the guide has learned which local states lead to the traps: their numbers stay, but for
        # one process that numbers its trap before the state in front of it
        lts = net.procs[seed % net.n_procs]
        last = lts.n_states - 1
        swap = {last: last - 1, last - 1: last}
        lts.edges = [(swap.get(s, s), a, swap.get(t, t)) for s, a, t in lts.edges]
        return _relabel(net, seed, states=False), None
    if case["family"] == "product":
        blocks = [int(b) for b in case["blocks"].split(",")]
        net = inputs.product_network(case["gen_seed"], case["n_procs"], case["n_states"], blocks,
                                     n_labels=case["n_labels"], parties=min(3, case["n_procs"]), deg_hi=case["deg_hi"])
        return _relabel(net, seed), None
    if case["family"] == "ring":
        base = inputs.token_ring(case["n_procs"])
        # node 1 must never hold the token; found in its new place by the label it sends with
        net = _relabel(base, seed)
        for p, lts in enumerate(net.procs):
            for s, a, _ in lts.edges:
                if a == 2 and any((p, a) == part for part in net.rules[1].parts[:1]):
                    return net, (p, s)
        raise AssertionError("the ring has no node 1")
    net = inputs.random_network(case["gen_seed"], case["n_procs"], case["n_states"], 1, case["deg_hi"], case["n_labels"],
                                n_sync=case["n_sync"], parties=case["parties"], sync_weight=case["sync_weight"],
                                cluster=case["cluster"])
    return _relabel(net, seed), None


def _explore_opts(case, watched=None):
    kw = dict(table_bytes=case["table_bytes"], bucket_words=case["bucket"], group_lanes=case["group"],
              hash_rounds=case["rounds"])
    if case.get("frontier"):
        kw["frontier_states"] = case["frontier"]
    if case.get("passes"):
        kw["region_passes"] = case["passes"]
    if case.get("watch"):
        kw.update(watch=1, watch_proc=watched[0], watch_state=watched[1])
    return gx.default_opts(**kw)


# ---- prepare

def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _prepare_explore(case, seed):
    net, watched = _network(case, seed)
    h = gx.load_network(net)
    opts = _explore_opts(case, watched)
    return dict(case=case, net=h, opts=opts, ws=gx.alloc_workspace(h, opts))


def _prepare_search(case, seed):
    h = gx.load_network(_network(case, seed)[0])
    opts = _explore_opts(case)
    return dict(case=case, net=h, opts=opts, ws=gx.alloc_workspace(h, opts))


def _prepare_guided(case, seed):
    train = [inputs.planted_network(s, n, n_traps=1 + s % 4) for s in range(6) for n in (6, 7, 8)]
    hist, label = guide.collect_examples(train, 64)
    params, _ = guide.train(hist, label, steps=4000, lr=1e-3)
    h = gx.load_network(_network(case, seed)[0])
    gx.guided_set_weights(h, params)
    opts = gx.default_opts(table_bytes=case["table_bytes"], hash_rounds=case["rounds"])
    return dict(case=case, net=h, opts=opts, ws=gx.guided_alloc_workspace(h, opts))


def _prepare_batch(case, seed):
    nets = [_relabel(net, seed * 1000 + i) for i, net in enumerate(inputs.batch_workload(case["count"]))]
    b = gx.batch_create(nets)
    sizing = gx.batch_opts(hash_rounds=case["rounds"], table_slots=1 << 21)
    ws = gx.batch_alloc_workspace(b, sizing)
    gx.batch_explore(b, sizing, ws)
    counts = [gx.batch_stats(b, i)["states"] for i in range(case["count"])]
    del ws
    opts = gx.batch_opts(hash_rounds=case["rounds"], bucket_words=case["bucket"], group_lanes=case["group"],
                         chunk_states=case["chunk"], expected_states=counts)
    return dict(case=case, batch=b, opts=opts, ws=gx.batch_alloc_workspace(b, opts))


def _examples(n, seed):
    """n histograms of 6..16 processes over 16 local states and labels in [0, 1] that depend on
    them, as distances to a deadlock do."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    procs = torch.randint(6, 17, (n, 1), generator=g, device="cuda")
    picks = torch.randint(0, 16, (n, 16), generator=g, device="cuda")
    inside = (torch.arange(16, device="cuda")[None, :] < procs).to(torch.uint8)
    hist = torch.zeros((n, 16), dtype=torch.uint8, device="cuda").scatter_add_(1, picks, inside)
    share = hist.float() / procs.float()
    weight = torch.rand(16, generator=g, device="cuda")
    label = torch.clamp((share * weight).sum(1) + 0.05 * torch.rand(n, generator=g, device="cuda"), 0, 1)
    return hist.contiguous(), label.contiguous()


def _weights(seed):
    params = torch.empty(gx.MLP_PARAMS, dtype=torch.float32, device="cuda")
    gx.mlp_init(params, seed)
    return params


def _prepare_score(case, seed):
    params = _weights(seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    for lo, n in ((128 * 16, 128), (128 * 16 + 128 + 128 * 128, 128), (gx.MLP_PARAMS - 1, 1)):
        params[lo:lo + n] = 0.1 * torch.randn(n, generator=g, device="cuda")  # biases, as training leaves them
    return dict(case=case, params=params, hist=_examples(case["n"], seed + 1)[0])


def _prepare_train(case, seed):
    hist, label = _examples(case["n"], seed)
    return dict(case=case, params=_weights(seed), hist=hist, label=label, seed=seed)


def _prepare_label(case, seed):
    h = gx.load_network(_network(case, seed)[0])
    opts = gx.default_opts(table_bytes=case["table_bytes"], bucket_words=8, group_lanes=1, hash_rounds=32)
    ws = gx.alloc_workspace(h, opts)
    gx.explore(h, opts, ws)
    return dict(case=case, net=h, ws=ws)


def _prepare_table(case, seed):
    w0 = inputs.key_sequence_device(case["distinct"], 1, seed=seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    first, new = w0[:case["first"]], w0[case["first"]:]
    again = torch.randint(0, case["first"], (case["second"] - len(new),), generator=g, device="cuda")
    second = torch.cat([new, first[again]])[torch.randperm(case["second"], generator=g, device="cuda")]

    def wide(x):  # further words are functions of the first: distinct keys stay distinct
        cols = [x] + [((x.to(torch.int64) * (2654435761 + 2 * k)) & 0x7FFFFFFF).to(torch.int32)
                      for k in range(1, case["words"])]
        return torch.stack(cols, dim=1).reshape(-1).contiguous() if len(cols) > 1 else x.contiguous()

    calls = []
    for keys in (first, second):
        calls.append((wide(keys), torch.empty(len(keys), dtype=torch.uint8, device="cuda")))
    table = torch.zeros((1 << case["log2_slots"]) * case["words"], dtype=torch.int32, device="cuda")
    return dict(case=case, calls=calls, table=table)


# ---- run

def run(state):
    return globals()["_run_" + state["case"]["kind"]](state)


def _signed(x):
    """A 64-bit digest as a signed integer."""
    return x - (1 << 64) if x >= 1 << 63 else x


def _stats(s):
    out = {k: int(s[k]) for k in ("states", "explored", "transitions", "n_levels", "deadlock_count",
                                  "first_deadlock_level", "violation_count", "first_violation_level", "complete")}
    for k in ("deadlock_sum", "deadlock_xor", "violation_sum", "violation_xor"):
        out[k] = _signed(int(s[k]))
    return out


def _sorted_states(a):
    """Reported states in a fixed order (the library gives them in none)."""
    return a[np.lexsort(a.T[::-1])].astype(np.int64) if len(a) else a.astype(np.int64)


def _run_explore(st):
    gx.explore(st["net"], st["opts"], st["ws"])
    out = _stats(gx.stats(st["net"]))
    out["levels"] = np.array(gx.levels(st["net"]), dtype=np.int64)
    # the order of the vectors in the table differs from run to run; its digest names the set
    out["visited"] = [_signed(x) for x in gx.set_digest(st["net"], st["ws"])]
    return out


def _run_search(st):
    found, states = gx.find_deadlocks(st["net"], gx.GX_DL_BFS_FIRST, st["opts"], st["ws"])
    out = _stats(gx.stats(st["net"]))
    out["found"] = found
    out["deadlocks"] = _sorted_states(states)
    out["levels"] = np.array(gx.levels(st["net"]), dtype=np.int64)
    return out


def _run_guided(st):
    # the order in which concurrent pushes fill the bins differs from run to run, so which and how
    # many states were expanded does too; the deadlock (there is one) and its path's length do not
    found, states = gx.find_deadlocks(st["net"], gx.GX_DL_GUIDED, st["opts"], st["ws"])
    return dict(found=found, deadlocks=_sorted_states(states), path_states=len(gx.guided_trace(st["net"])))


def _run_batch(st):
    b = st["batch"]
    gx.batch_explore(b, st["opts"], st["ws"])
    rows, levels = [], []
    for i in range(b.n):
        s = gx.batch_stats(b, i)
        rows.append([_signed(int(s[k])) for k in ("states", "explored", "transitions", "n_levels", "deadlock_count",
                                                  "deadlock_sum", "deadlock_xor", "first_deadlock_level", "complete")])
        levels.extend(gx.batch_levels(b, i))
    return dict(stats=np.array(rows, dtype=np.int64), levels=np.array(levels, dtype=np.int64))


def _run_score(st):
    return gx.mlp_forward(st["params"], st["hist"])


def _run_train(st):
    c = st["case"]
    params = st["params"].clone()  # the optimiser updates them in place
    losses = gx.mlp_train(params, st["hist"], st["label"], c["batch"], c["steps"], c["lr"], st["seed"])
    return dict(params=params, losses=losses)


def _run_label(st):
    hist, label = gx.training_set(st["net"], st["ws"], st["case"]["max_dist"])
    return dict(hist=hist, label=label)


def _run_table(st):
    c = st["case"]
    st["table"].zero_()
    counters = torch.zeros(3, dtype=torch.int64, device="cuda")
    for keys, result in st["calls"]:
        gx.find_or_put(keys, c["words"], st["table"], counters, result, c["bucket"], c["group"], c["rounds"])
    return dict(counters=counters, results=[result for _, result in st["calls"]])


# ---- work

def work(case):
    kind = case["kind"]
    if kind in ("explore", "search"):
        if kind == "search":
            states, w = PLANTED_SEARCH[case["n_procs"]][case["net_seed"]], 2 if case["n_procs"] > 7 else 1
        else:
            states = case["states"]
            w = _slot_words(case["n_procs"], 5 if case["family"] == "ring" else case["n_states"])
        # the cleared table; each state stored, queued as open and read again
        return {"bytes": case["table_bytes"] + 12 * w * states, "flops": 0}
    if kind == "guided":
        # at least: one full batch of open states per step of the path, each state's successors
        # (about 17 new ones) stored, scored and queued
        states = 17 * 8192 * (2 * case["n_procs"] + 1)
        return {"bytes": case["table_bytes"] + 28 * states, "flops": SCORE_FLOPS * states}
    if kind == "batch":
        states = BATCH_STATES[case["count"]]
        return {"bytes": 16 * states + 24 * states, "flops": 0}
    if kind == "score":
        return {"bytes": 20 * case["n"] + 4 * gx.MLP_PARAMS, "flops": SCORE_FLOPS * case["n"]}
    if kind == "train":
        rows = case["batch"] * case["steps"]
        return {"bytes": 20 * rows + 28 * gx.MLP_PARAMS * case["steps"], "flops": 3 * SCORE_FLOPS * rows}
    if kind == "label":
        states = PLANTED_STATES[case["n_procs"]][case["net_seed"]]
        return {"bytes": case["table_bytes"] + 20 * states, "flops": 0}
    n, w = case["first"] + case["second"], case["words"]
    return {"bytes": 4 * w * (n + (1 << case["log2_slots"]) + case["distinct"]) + n, "flops": 0}


# ---- exact values in 64 bits

def exact(case, seed):
    if case["kind"] == "score":
        params, hist = _prepare_score(case, seed)["params"], _examples(case["n"], seed + 1)[0]
        return torch.cat([_net64(_split64(params), h)[0] for h in hist.split(1 << 18)])
    if case["kind"] == "train":
        return _train64(case, seed)
    if case["kind"] == "label":
        return _label64(case, seed)
    return None  # whole numbers throughout, compared as they are


def _split64(params):
    """W1, b1, W2, b2, w3, b3 in float64; the weights are BF16 by definition of the network."""
    p = params.double()
    sizes = (128 * 16, 128, 128 * 128, 128, 128, 1)
    parts = list(torch.split(p, sizes))
    for k in (0, 2, 4):
        parts[k] = parts[k].to(torch.float32).to(torch.bfloat16).double()
    parts[0], parts[2] = parts[0].view(128, 16), parts[2].view(128, 128)
    return parts


def _net64(p, hist):
    x = hist.double()
    n = x.sum(1, keepdim=True)
    x = torch.where(n > 0, x / n.clamp(min=1), torch.zeros_like(x))
    h1 = torch.relu(x @ p[0].T + p[1])
    h2 = torch.relu(h1 @ p[2].T + p[3])
    return h2 @ p[4] + p[5], x, h1, h2


def _train64(case, seed):
    st = _prepare_train(case, seed)
    p = st["params"].double()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    batch, losses = case["batch"], []
    for t in range(case["steps"]):
        # the documented counter-based stream: element j of step t is mix64(seed + t * batch + j) mod n
        with np.errstate(over="ignore"):
            z = np.arange(batch, dtype=np.uint64) + np.uint64((seed + t * batch + 0x9E3779B97F4A7C15) & inputs.M64)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = (z ^ (z >> np.uint64(31))) % np.uint64(case["n"])
        idx = torch.from_numpy(z.astype(np.int64)).cuda()
        w = _split64(p.float())
        y, x, h1, h2 = _net64(w, st["hist"][idx])
        lab = st["label"][idx].double()
        losses.append(((y - lab) ** 2).mean())
        dy = 2 * (y - lab) / batch
        d2 = dy[:, None] * w[4][None, :] * (h2 > 0)
        d1 = (d2 @ w[2]) * (h1 > 0)
        g = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy, dy.sum()[None]])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - case["lr"] * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
    return dict(params=p, losses=torch.stack(losses))


def _label64(case, seed):
    """Distances by breadth-first search forwards and relaxation backwards over integer codes."""
    net, _ = _network(case, seed)
    n, base = net.n_procs, 16
    rule_pairs = {part for r in net.rules for part in r.parts}
    edges = {}  # (process, label) -> list of (from, difference of codes)
    for p, lts in enumerate(net.procs):
        for s, a, t in lts.edges:
            edges.setdefault((p, a), []).append((s, (t - s) * base ** p))

    def successors(codes):
        at = [(codes // base ** p) % base for p in range(n)]
        src, dst = [], []

        def moves(parts, rows, delta):
            if not parts:
                src.append(rows)
                dst.append(codes[rows] + delta)
                return
            p, a = parts[0]
            for s, d in edges.get((p, a), ()):
                keep = at[p][rows] == s
                if keep.any():
                    moves(parts[1:], rows[keep], delta + d)

        everything = np.arange(len(codes))
        for pair in edges:
            if pair not in rule_pairs:
                moves([pair], everything, 0)
        for r in net.rules:
            moves(list(r.parts), everything, 0)
        none = [np.empty(0, dtype=np.int64)]
        return np.concatenate(src + none), np.concatenate(dst + none)

    known = np.array([sum(lts.initial * base ** p for p, lts in enumerate(net.procs))], dtype=np.int64)
    fresh = known
    while len(fresh):
        fresh = np.setdiff1d(np.unique(successors(fresh)[1]), known, assume_unique=True)
        known = np.union1d(known, fresh)
        if len(known) > 1_000_000:
            return None
    src, dst = successors(known)
    dst = np.searchsorted(known, dst)
    dist = np.full(len(known), case["max_dist"], dtype=np.int64)
    dead = np.ones(len(known), dtype=bool)
    dead[src] = False
    dist[dead] = 0
    for d in range(1, case["max_dist"]):
        reach = np.zeros(len(known), dtype=bool)
        reach[src[dist[dst] == d - 1]] = True
        dist[reach & (dist == case["max_dist"])] = d
    hist = np.zeros((len(known), 16), dtype=np.uint8)
    for p in range(n):
        np.add.at(hist, (np.arange(len(known)), (known // base ** p) % base), 1)
    words = hist.view("<u4")
    order = np.lexsort((dist, words[:, 3], words[:, 2], words[:, 1], words[:, 0]))
    return dict(hist=torch.from_numpy(hist[order]), label=torch.from_numpy(dist[order] / case["max_dist"]))
