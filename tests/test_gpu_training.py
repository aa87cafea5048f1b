"""The training kernels at the sizes where they can go wrong: which examples a step draws, batches
below, at and above a tile and above one tile per CTA, and histograms at odd addresses."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_1801_05857_gb300 import gx

pytestmark = pytest.mark.gpu


def _data(n, seed):
    import torch
    rng = np.random.default_rng(seed)
    hist = rng.multinomial(9, np.ones(16) / 16, size=n).astype(np.uint8)
    label = rng.random(n).astype(np.float32)
    p = torch.empty(gx.MLP_PARAMS, dtype=torch.float32, device="cuda")
    gx.mlp_init(p, seed)
    return hist, label, p


def _drawn(seed, step, batch, n):
    """Example numbers of a step: mix64(seed + step * batch + j) mod n (splitmix64)."""
    with np.errstate(over="ignore"):
        z = np.arange(batch, dtype=np.uint64) + np.uint64(seed + step * batch) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return ((z ^ (z >> np.uint64(31))) % np.uint64(n)).astype(np.int64)


@pytest.mark.parametrize("batch", [1, 127, 128, 129, 1000, 256 * 128 + 5])
def test_first_steps_losses_are_those_of_the_drawn_examples(cuda, batch):
    """Step 0's loss at the initial weights, and step 1's at weights one Adam step on (its update
    is lr a parameter at most, so the loss moves little for a small lr)."""
    import torch
    hist, label, p = _data(5000, batch)
    p0 = p.cpu().numpy()
    losses = gx.mlp_train(p, torch.from_numpy(hist).cuda(), torch.from_numpy(label).cuda(), batch, 2, 1e-7, 77)
    for step in range(2):
        idx = _drawn(77, step, batch, len(hist))
        want, _ = omlp.loss_and_grad(p0, hist[idx], label[idx])
        assert abs(float(losses[step]) - want) <= 1e-3 * want + 1e-6
    moved = np.abs(p.cpu().numpy() - p0)
    assert 0 < moved.max() <= 2.1e-7 + 2 ** -24  # at most lr a step, and FP32's rounding of parameters below 1


def test_histograms_at_odd_addresses(cuda):
    import torch
    hist, label, p = _data(300, 4)
    flat = torch.zeros(300 * 16 + 1, dtype=torch.uint8, device="cuda")
    flat[1:] = torch.from_numpy(hist.reshape(-1)).cuda()
    lab = torch.from_numpy(label).cuda()
    odd = flat[1:].view(300, 16)
    assert odd.data_ptr() % 16 == 1
    g0, l0 = gx.mlp_grad(p, torch.from_numpy(hist).cuda(), lab)
    g1, l1 = gx.mlp_grad(p, odd, lab)
    assert torch.equal(g0, g1) and torch.equal(l0, l1)
    assert torch.equal(gx.mlp_forward(p, odd), gx.mlp_forward(p, torch.from_numpy(hist).cuda()))


def test_training_is_reproducible(cuda):
    import torch
    hist, label, p = _data(3000, 9)
    h, lab = torch.from_numpy(hist).cuda(), torch.from_numpy(label).cuda()
    a, b = p.clone(), p.clone()
    la, lb = gx.mlp_train(a, h, lab, 700, 60, 1e-3, 5), gx.mlp_train(b, h, lab, 700, 60, 1e-3, 5)
    assert torch.equal(a, b) and torch.equal(la, lb)
    assert float(la[-10:].mean()) < float(la[:10].mean())


@pytest.mark.parametrize("batch", [1, 300, 256 * 128 + 5])
def test_every_step_is_an_adam_step_at_the_weights_before_it(cuda, batch):
    """Steps 0..4 one by one: the parameters after step k are those before it moved by an Adam
    step whose gradient mlp_grad takes at them, over the examples that step draws, and the
    step's loss is mlp_grad's.  mlp_grad packs the FP32 parameters by a kernel of its own, so
    a weight, bias or transposed copy that the update left stale shows in the next step.

    Tolerance: the gradients are the same sums in the same order, so what differs is FP32
    rounding in the update (under 20 roundings of 2^-24 relative, on an update of a few lr)
    and the rounding of the parameter itself."""
    import torch
    hist, label, p0 = _data(5000, batch)
    dh, dl = torch.from_numpy(hist).cuda(), torch.from_numpy(label).cuda()
    lr, seed, steps = 1e-3, 31, 5
    f = lambda x: float(np.float32(x))
    m = np.zeros(gx.MLP_PARAMS)
    v = np.zeros(gx.MLP_PARAMS)
    b1t = b2t = 1.0
    before = p0.clone()
    for k in range(steps):
        idx = torch.from_numpy(_drawn(seed, k, batch, len(hist))).cuda()
        g, loss = gx.mlp_grad(before, dh[idx].contiguous(), dl[idx].contiguous())
        after = p0.clone()
        losses = gx.mlp_train(after, dh, dl, batch, k + 1, lr, seed)
        assert abs(float(losses[k]) - float(loss)) <= 1e-6 * float(loss)
        g = g.cpu().numpy().astype(np.float64)
        m = f(0.9) * m + f(0.1) * g
        v = f(0.999) * v + f(0.001) * g * g
        b1t, b2t = b1t * 0.9, b2t * 0.999
        c1, c2 = f(np.float32(1) - np.float32(b1t)), f(np.float32(1) - np.float32(b2t))
        move = f(lr) * (m / c1) / (np.sqrt(v / c2) + f(1e-8))
        p = before.cpu().numpy().astype(np.float64)
        got = after.cpu().numpy().astype(np.float64)
        assert (np.abs(got - (p - move)) <= 20 * 2.0 ** -24 * np.abs(move) + 2.0 ** -23 * np.abs(p) + 1e-12).all()
        assert np.abs(got - p).max() > 0.1 * lr
        before = after


def test_scores_with_extreme_biases(cuda):
    """Second-layer biases up to the largest floats (their three BF16 parts must stay finite),
    down to 1e-37, infinite and NaN: the scores are those of the network with the bias added
    to a unit's sum.  w3 scales each unit's part to about 1, exactly (a power of two)."""
    import torch
    hist, _, p = _data(300, 2)
    W1, b1, W2, b2, w3, b3 = omlp.unpack(p.cpu().numpy())
    big = float(np.finfo(np.float32).max)
    for bias in (big, np.nextafter(np.float32(big), np.float32(0)), 3.3895e38, 3.39e38, 1e38, -big, 1.0, 1 / 3, 1e-30,
                 -1e-37, np.inf, -np.inf, np.nan):
        q = p.cpu().numpy().copy()
        b2at = 128 * 16 + 128 + 128 * 128
        q[b2at:b2at + 128] = 0
        q[b2at + 5] = bias
        q[b2at + 128:b2at + 256] = 0
        scale = 2.0 ** -int(np.floor(np.log2(abs(bias)))) if np.isfinite(bias) else 1.0
        q[b2at + 128 + 5] = min(max(scale, 2.0 ** -126), 2.0 ** 120)
        y = gx.mlp_forward(torch.from_numpy(q).cuda(), torch.from_numpy(hist).cuda()).cpu().numpy().astype(np.float64)
        with np.errstate(invalid="ignore"):
            want = omlp.forward(q, hist)
        if np.isnan(bias):
            continue  # (max(NaN, 0) is the hardware's choice; it must only not hang or poison others)
        if np.isinf(bias):
            assert (y == want).all()
            continue
        assert np.isfinite(y).all(), bias
        # (a hidden value of up to 1 may round to the other BF16 neighbour, 2^-9 away: times a weight
        # of at most 128 ** -0.5 and w3 of up to 4, 7e-4)
        assert (np.abs(y - want) <= 1e-3 * np.maximum(1, np.abs(want))).all(), bias
    y0 = gx.mlp_forward(p, torch.from_numpy(hist).cuda()).cpu().numpy()
    assert np.isfinite(y0).all()
