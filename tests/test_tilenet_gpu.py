"""The tensor-core forward of the tile-proposal network: numbers of patches around
the grid's size, unaligned patch arrays, infinities, and proposal tiles read in
place against the same patches extracted."""

import numpy as np
import pytest

import synth
from oracle import tcnn as ora

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_07164_gb300 as ofg  # noqa: E402
from paper_2506_07164_gb300 import learned  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ofg.build()
    ofg.load()


def _tiles(n, seed):
    rng = np.random.default_rng(seed)
    img = synth.scene(512, 512, seed, n_rect=60, n_checker=10)
    out = np.zeros((n, 64, 64), np.uint8)
    for i in range(n):
        y, x = rng.integers(0, 448, 2)
        out[i] = img[y:y + 64, x:x + 64]
    out[0] = 0
    out[n // 2] = 255
    out[-1] = rng.integers(0, 256, (64, 64))
    return out


def _bound(tiles, p):
    """Each logit's sum with every term positive, times 2^-17: three layers and a head of fewer than 64
    fp32 operations in a row, each off by at most 2^-23 of that sum."""
    P = ora.unpack(np.abs(p))
    a = np.abs(ora.normalise(tiles))[:, None]
    for w, b in (("W1", "b1"), ("W2", "b2"), ("W3", "b3")):
        a = ora.conv_s2(a, P[w], P[b])
    return (a.mean(axis=(2, 3)) @ P["wf"] + P["bf"][0]) * 2.0**-17


@pytest.mark.parametrize("n", [1, 2, 303, 304, 305, 609])
def test_forward_at_grid_edges(n):
    net = learned.TileNet(3)
    rng = np.random.default_rng(n)
    ofg.of_tcnn_set_params(net.net, rng.normal(scale=0.4, size=ofg.of_tcnn_num_params()).astype(np.float32))
    tiles = _tiles(n, 5)
    z = net.logits(torch.from_numpy(tiles).cuda()).cpu().numpy()
    pq = ofg.of_tcnn_get_params(net.net, 1).astype(np.float64)
    zo, _ = ora.forward(tiles, pq)
    assert (np.abs(z - zo) <= _bound(tiles, pq)).all()
    # The same patches one byte into a buffer.
    buf = torch.zeros(tiles.size + 1, dtype=torch.uint8, device="cuda")
    buf[1:] = torch.from_numpy(tiles).cuda().reshape(-1)
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    ofg.of_tcnn_forward(net.net, buf[1:], n, out)
    np.testing.assert_array_equal(out.cpu().numpy(), z)
    net.close()


@pytest.mark.parametrize("n", [1, 2, 151, 152, 153, 305])
def test_gradient_at_grid_edges(n):
    """Loss and every layer's gradient, one patch per block or fewer and more; the same bounds as the
    existing gradient test (fp32 against float64; a ReLU input within rounding of 0 may flip)."""
    net = learned.TileNet(n)
    tiles = _tiles(n, 6)
    rng = np.random.default_rng(n)
    labels = (rng.random(n) < 0.4).astype(np.float32)
    buf = torch.zeros(tiles.size + 1, dtype=torch.uint8, device="cuda")  # unaligned patches
    buf[1:] = torch.from_numpy(tiles).cuda().reshape(-1)
    lab = torch.from_numpy(labels).cuda()
    for dev in (torch.from_numpy(tiles).cuda(), buf[1:]):
        loss = ofg.of_tcnn_loss_grad(net.net, dev, lab, n, pos_weight=3.0)
        g = ofg.of_tcnn_get_params(net.net, 2).astype(np.float64)
        lo, go = ora.loss_grad(tiles, labels, ofg.of_tcnn_get_params(net.net, 1).astype(np.float64), pos_weight=3.0)
        assert loss == pytest.approx(lo, rel=1e-5)
        assert np.linalg.norm(g - go) / np.linalg.norm(go) < 1e-4
        for a, b in ((0, 72), (72, 80), (80, 1232), (1232, 1248), (1248, 3552), (3552, 3568), (3568, 3584), (3584, 3585)):
            assert np.linalg.norm(g[a:b] - go[a:b]) <= 1e-3 * np.linalg.norm(go[a:b]) + 1e-12, (a, b)
    net.close()


def test_infinite_activations():
    """Activations that overflow stay infinities (not NaN) through the split into parts."""
    net = learned.TileNet(0)
    P = {k: np.zeros(s) for k, s in ora.SHAPES}
    P["W1"][0, 0, 1, 1] = P["W2"][0, 0, 1, 1] = P["W3"][0, 0, 1, 1] = 2.0**126
    P["W1"][0, 0, 0, 0] = 1.0
    for k in ("W1", "W2", "W3"):
        P[k] += (P[k] == 0) * 2.0**-120  # no exact zero weight, so that no 0 * inf arises
    P["wf"][:] = 2.0**-60
    ofg.of_tcnn_set_params(net.net, ora.pack(P).astype(np.float32))
    z = net.logits(torch.from_numpy(np.full((3, 64, 64), 255, np.uint8)).cuda()).cpu().numpy()
    assert np.isposinf(z).all(), z
    net.close()


def test_in_place_tiles_equal_extracted_patches():
    net = learned.TileNet(0).load(learned.DEFAULT_WEIGHTS)
    frames = [torch.from_numpy(synth.scene(w, h, 30 + i)).cuda() for i, (w, h) in enumerate([(500, 300), (331, 217)])]
    det = ofg.Detector(500, 300, max_levels=4, max_features=200, max_batch=2, fast_t_lo=7)
    fr = [(t, t.shape[1], t.shape[0], t.stride(0)) for t in frames]
    ofg.of_detect_learned(det.h, fr, 4, 1.2, 20, 0.04, 200, net.net, 0.1, 0.0, 1, det.out, det.counts)
    for f in range(2):
        for lvl in range(4):
            raw, dims = det.inspect(ofg.OF_BUF_LOGIT, f, lvl)
            n, _ = ofg.of_extract_tiles(det.h, f, lvl)
            t = torch.empty((n, 64, 64), dtype=torch.uint8, device="cuda")
            ofg.of_extract_tiles(det.h, f, lvl, t, n)
            np.testing.assert_array_equal(raw.view(np.float32), net.logits(t).cpu().numpy())
    det.close()
    net.close()
