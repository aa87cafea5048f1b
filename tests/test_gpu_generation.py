"""Successors of rules with many combinations, which lanes of a warp share, against the CPU
oracle: combinations at the edges of the rule that picks the sharing kernels (16) and of the
parts lanes are given, several such rules in a state, and local edges beside them."""
import pytest

import oracle
from paper_1801_05857_gb300 import gx, inputs

pytestmark = pytest.mark.gpu


def _rules(n_procs, rules, local=0, n_states=4):
    """n_procs processes of n_states states; a rule (degrees...) takes as many processes,
    starting with a different one each, of which the j-th has degrees[j] edges from every
    state; the first `local` processes have an edge of their own besides."""
    procs = [inputs.LTS(n_states, 0, []) for _ in range(n_procs)]
    out = []
    for r, degrees in enumerate(rules):
        parts = []
        for j, deg in enumerate(degrees):
            p = (r + j) % n_procs
            parts.append((p, r))
            procs[p].edges += [(s, r, (s + 1 + d % (n_states - 1)) % n_states) for s in range(n_states) for d in range(deg)]
        out.append(inputs.Rule(parts, len(rules)))
    for p in range(local):
        procs[p].edges += [(s, len(rules), (s + 1) % n_states) for s in range(n_states)]
    return inputs.Network(len(rules) + 1, procs, out)


NETS = {
    "combinations_15": _rules(4, [(5, 3)], local=2),
    "combinations_16": _rules(4, [(4, 4)], local=2),
    "combinations_17": _rules(4, [(17, 1)], local=4),
    "combinations_243": _rules(5, [(3,) * 5]),
    "three_rules": _rules(5, [(3, 3, 3), (2, 2), (7, 5, 2)], local=1),
    "many_rules": _rules(6, [(3, 3, 2)] * 6),
    "edges_40": _rules(4, [(40,), (1, 1)], local=3),
    "two_words": _rules(10, [(3, 3, 3), (6, 6)], n_states=16),            # 40 bits
    "four_words": _rules(18, [(3, 3, 3), (5, 4)], local=1, n_states=16),  # 72 bits
}


@pytest.mark.parametrize("count", [1, 3, 40])
@pytest.mark.parametrize("name", NETS)
def test_batches_of_networks_with_many_combinations(cuda, name, count):
    net = NETS[name]
    r = oracle.explore(net)
    h = gx.load_network(net)
    b = gx.batch_create([h] * count)
    o = gx.batch_opts(hash_rounds=64, expected_states=[2 * r.states] * count)
    ws = gx.batch_alloc_workspace(b, o)
    gx.batch_explore(b, o, ws)
    for i in range(count):
        s = gx.batch_stats(b, i)
        assert (s["states"], s["transitions"], s["complete"]) == (r.states, r.transitions, 1)
        assert gx.batch_levels(b, i) == r.levels


@pytest.mark.parametrize("opts", [dict(), dict(bucket_words=16, group_lanes=1), dict(host_loop=1, group_lanes=1),
                                  dict(region_passes=2), dict(watch=1, watch_proc=0, watch_state=1)], ids=str)
@pytest.mark.parametrize("name", NETS)
def test_exploration_of_networks_with_many_combinations(cuda, name, opts):
    net = NETS[name]
    r = oracle.explore(net, watch=(0, 1))
    h = gx.load_network(net)
    o = gx.default_opts(table_bytes=1 << 24, hash_rounds=64, **opts)
    ws = gx.alloc_workspace(h, o)
    gx.explore(h, o, ws)
    s = gx.stats(h)
    assert (s["states"], s["transitions"], gx.levels(h)) == (r.states, r.transitions, r.levels)
    assert gx.set_digest(h, ws) == (r.states, r.set_sum, r.set_xor)
    if opts.get("watch"):
        assert (s["violation_count"], s["violation_xor"]) == (r.violation_count, r.violation_xor)
    if not opts:
        n, levels = gx.explore_noalloc(h, o)
        assert (n["states"], n["transitions"], levels) == (r.states, r.transitions, r.levels)


@pytest.mark.parametrize("name", NETS)
def test_guided_search_of_networks_with_many_combinations(cuda, name):
    import torch
    net = NETS[name]
    r = oracle.explore(net)
    assert r.deadlock_count == 0
    h = gx.load_network(net)
    p = torch.empty(gx.MLP_PARAMS, dtype=torch.float32, device="cuda")
    gx.mlp_init(p, 3)
    gx.guided_set_weights(h, p)
    o = gx.default_opts(table_bytes=1 << 24, hash_rounds=64)
    ws = gx.guided_alloc_workspace(h, o)
    found, _ = gx.find_deadlocks(h, gx.GX_DL_GUIDED, o, ws)
    s = gx.stats(h)
    assert found == 0
    assert (s["states"], s["explored"], s["transitions"]) == (r.states, r.states, r.transitions)
