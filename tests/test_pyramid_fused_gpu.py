"""The fused pyramid kernel against the oracle's levels where its tiling changes:
every tile size the batch's pixels choose, runs cut by the seam bound, frames of
several sizes (and with fewer levels) in one batch, an unaligned source."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2506_07164_gb300 as ofg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ofg.build()
    ofg.load()


# Pixels per batch: below 0.8 M (64-pixel tiles), 3 M (96), 24 M (128), above (160, short runs).
@pytest.mark.parametrize("sizes,scale,levels", [
    ([(500, 333)], 1.2, 8),
    ([(997, 801), (333, 197), (41, 640)], 1.2, 8),
    ([(1283, 1717), (1921, 1081), (60, 50)], 1.3, 7),
    ([(1921, 1081)] * 3 + [(640, 479)] * 60, 1.2, 8),
    ([(1283, 717)] * 30, 2.0, 5),
    ([(130, 90), (97, 4), (3, 130)], 1.2, 12),
])
def test_levels_match_the_oracle(sizes, scale, levels):
    uniq = sorted(set(sizes))
    imgs = {s: synth.scene(s[0], s[1], 60 + i, n_rect=40, n_checker=8) for i, s in enumerate(uniq)}
    dev = []
    for k, s in enumerate(sizes):
        h, w = imgs[s].shape
        if k % 3 == 1:  # rows at an odd pitch: the level-0 copy
            buf = torch.zeros((h, w + 3), dtype=torch.uint8, device="cuda")
            t = buf[:, 1:w + 1]
            t.copy_(torch.from_numpy(imgs[s]).cuda())
        else:
            t = torch.from_numpy(imgs[s]).cuda()
        dev.append(t)
    det = ofg.Detector(max(w for w, _ in sizes), max(h for _, h in sizes), max_levels=levels, max_features=50,
                       max_batch=len(sizes))
    det.detect_batch(dev, levels=levels, scale=scale, fast_t=40, n_features=50)
    torch.cuda.synchronize()
    done = set()
    for f in list(range(min(4, len(sizes)))) + [len(sizes) - 1]:
        if (sizes[f], f % 3 == 1) in done:
            continue
        done.add((sizes[f], f % 3 == 1))
        ws, hs, _ = ofg.of_plan_levels(*sizes[f], levels, scale, 50)
        for lv in range(1, levels):
            if ws[lv] < 1 or hs[lv] < 1:
                break
            g, dims = det.inspect(ofg.OF_BUF_LEVEL, f, lv)
            np.testing.assert_array_equal(g.reshape(dims[1], dims[0]), oracle.pyramid_level(imgs[sizes[f]], levels, scale, lv),
                                          err_msg=f"frame {f} {sizes[f]} level {lv}")
    det.close()
