"""Accuracy of the tile network's kernels against 64 bits, tight enough to see a lost split part.

The kernels carry each fp32 activation (and gradient) as three exact bf16 parts, so their errors are
those of fp32 sums: logits within 5, each layer's gradient within 16 units of 2^-24 of its norm (medians
over seeds: a ReLU input within rounding of 0 may flip in single batches).  With two parts, 16 bits of an
activation, the errors are 40 times those limits; the host tests check that the limits notice."""

import numpy as np
import pytest

import synth
from oracle import tcnn as ora

LOGITS, GRADIENT = 5 * 2.0**-24, 16 * 2.0**-24
LAYERS = {"W1": (0, 72), "b1": (72, 80), "W2": (80, 1232), "b2": (1232, 1248), "W3": (1248, 3552), "b3": (3552, 3568),
          "wf": (3568, 3584), "bf": (3584, 3585)}
SEEDS = range(9)


def _batch(seed, n=96):
    rng = np.random.default_rng(seed)
    img = synth.scene(512, 512, seed, n_rect=60, n_checker=10)
    at = rng.integers(0, 448, (n, 2))
    tiles = np.stack([img[y:y + 64, x:x + 64] for y, x in at])
    return tiles, (rng.random(n) < 0.4).astype(np.float32)


def _params(seed):
    """He-uniform weights and small biases, as bf16 keeps them."""
    rng = np.random.default_rng(1000 + seed)
    out = []
    for name, shape in ora.SHAPES:
        fan = int(np.prod(shape[1:])) if len(shape) > 1 else 16 if name == "wf" else 0
        out.append(rng.uniform(-1, 1, int(np.prod(shape))) * ((6.0 / fan) ** 0.5 if fan else 0.05))
    p = np.concatenate(out).astype(np.float32)
    return ((p.view(np.uint32) + 0x8000) & 0xFFFF0000).astype(np.uint32).view(np.float32).astype(np.float64)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("mask", [0xFFFF0000, 0xFFFFFF00])  # one bf16 part of an activation, two
def test_the_limits_notice_a_lost_part(monkeypatch, mask):
    conv = ora.conv_s2

    def cut(x, W, b):
        x = np.ascontiguousarray(x, np.float32)
        return conv((x.view(np.uint32) & np.uint32(mask)).view(np.float32).astype(np.float64), W, b)

    logits, grads = [], {k: [] for k in LAYERS}
    for seed in range(3):
        tiles, labels = _batch(seed, 24)
        p = _params(seed)
        z, _ = ora.forward(tiles, p)
        _, g = ora.loss_grad(tiles, labels, p, pos_weight=3.0)
        with monkeypatch.context() as m:
            m.setattr(ora, "conv_s2", cut)
            zc, _ = ora.forward(tiles, p)
            _, gc = ora.loss_grad(tiles, labels, p, pos_weight=3.0)
        logits.append(_rel(zc, z))
        for k, (a, e) in LAYERS.items():
            grads[k].append(_rel(gc[a:e], g[a:e]))
    assert np.median(logits) > 10 * LOGITS
    for k, v in grads.items():
        assert np.median(v) > 4 * GRADIENT, (k, v)


@pytest.mark.gpu
def test_logits_and_every_layers_gradient():
    torch = pytest.importorskip("torch")
    import paper_2506_07164_gb300 as ofg
    from paper_2506_07164_gb300 import learned

    logits, grads = [], {k: [] for k in LAYERS}
    for seed in SEEDS:
        tiles, labels = _batch(seed)
        net = learned.TileNet(0)
        ofg.of_tcnn_set_params(net.net, _params(seed).astype(np.float32))
        p = ofg.of_tcnn_get_params(net.net, 1).astype(np.float64)
        np.testing.assert_array_equal(p, _params(seed))
        dev = torch.from_numpy(tiles).cuda()
        z, _ = ora.forward(tiles, p)
        logits.append(_rel(net.logits(dev).cpu().numpy().astype(np.float64), z))
        ofg.of_tcnn_loss_grad(net.net, dev, torch.from_numpy(labels).cuda(), len(tiles), pos_weight=3.0)
        g = ofg.of_tcnn_get_params(net.net, 2).astype(np.float64)
        _, go = ora.loss_grad(tiles, labels, p, pos_weight=3.0)
        for k, (a, e) in LAYERS.items():
            grads[k].append(_rel(g[a:e], go[a:e]))
        net.close()
    assert np.median(logits) <= LOGITS, logits
    for k, v in grads.items():
        assert np.median(v) <= GRADIENT, (k, v)


@pytest.mark.gpu
def test_last_bias_gradient_over_many_patches():
    """The sum of every patch's loss derivative, of both signs.  Each is off by a few roundings of its own,
    independently: 8 units of 2^-24 of the sum of their sizes over the square root of their number (or of
    the sum, if larger); and by its logit's error, at most the logits' limit, perhaps all of one sign."""
    torch = pytest.importorskip("torch")
    import paper_2506_07164_gb300 as ofg
    from paper_2506_07164_gb300 import learned

    net = learned.TileNet(0)
    for seed in range(4):
        tiles, labels = _batch(50 + seed, 1000)
        ofg.of_tcnn_set_params(net.net, _params(seed).astype(np.float32))
        p = ofg.of_tcnn_get_params(net.net, 1).astype(np.float64)
        ofg.of_tcnn_loss_grad(net.net, torch.from_numpy(tiles).cuda(), torch.from_numpy(labels).cuda(), 1000, pos_weight=3.0)
        got = float(ofg.of_tcnn_get_params(net.net, 2)[3584])
        z, _ = ora.forward(tiles, p)
        w, sg = np.where(labels > 0.5, 3.0, 1.0) / 1000, 1.0 / (1.0 + np.exp(-z))
        dz = w * (sg - labels)
        bound = 8 * 2.0**-24 * max(np.abs(dz).sum() / 1000**0.5, abs(dz.sum()))
        bound += LOGITS * float(np.sqrt(np.mean(z * z))) * (w * sg * (1 - sg)).sum()
        assert abs(got - dz.sum()) <= bound, (got, dz.sum(), bound)
    net.close()
