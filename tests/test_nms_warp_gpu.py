"""The per-warp NMS + Harris kernel on whole 128 x 32 tiles (chosen by tuning, as large
batches choose it): cells from the smallest that an 8-row chunk may meet twice to the
largest of the strip form, thresholds within and beyond 128 above the fallback, no
fallback, ragged widths and heights -- against the oracle."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2506_07164_gb300 as ofg  # noqa: E402

FIELDS = ["x_l", "y_l", "level", "fast_score", "A", "B", "C", "m10", "m01", "key"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ofg.build()
    ofg.load()


@pytest.mark.parametrize("form", [4, 3])  # FAST in strips (flags set by it), or per warp and a flag pass
@pytest.mark.parametrize("w,h,levels,cell,border,t,t_lo", [
    (1601, 1101, 4, 30, 19, 20, 7),
    (1601, 1101, 4, 33, 22, 200, 5),
    (1283, 901, 3, 8, 15, 12, 3),
    (1411, 1029, 3, 9, 16, 20, 7),
    (1300, 990, 3, 17, 20, 30, 2),
    (1601, 1101, 4, 30, 19, 20, 0),
])
def test_whole_tiles_match_the_oracle(form, w, h, levels, cell, border, t, t_lo):
    n, frames = 3000, 2
    imgs = [synth.scene(w, h, 90 + i, background="pink") for i in range(frames)]
    dev = [torch.from_numpy(im).cuda() for im in imgs]
    det = ofg.Detector(w, h, max_levels=levels, max_features=n, max_batch=frames, fast_t_lo=t_lo, cell=cell,
                       border=border)
    tun = ofg.OfTuning(resize_tile_h=32, resize_tma=1, fast_blocks_per_sm=1, nms_blocks_per_sm=2, fast_order=0,
                       nms_order=0, stream_groups=1, fast_cell_tiles=form, nms_tile_h=32, fast_tile_h=32)
    det.set_tuning(dev, tun, levels=levels, fast_t=t, n_features=n)
    for _ in range(2):
        det.detect_batch(dev, levels=levels, fast_t=t, n_features=n)
    torch.cuda.synchronize()
    got = det.batch_results(frames, n)
    for i in range(frames):
        ora = oracle.detect(imgs[i], levels=levels, fast_t=t, fast_t_lo=t_lo, n_features=n, cell=cell, border=border)
        assert len(got[i]) == len(ora) > 0
        for f in FIELDS:
            np.testing.assert_array_equal(got[i][f], ora[f], err_msg=f"frame {i} {f}")
    det.close()
