"""Top-N when thousands of candidates share one key (synthetic grids, calibration targets): no
coarse bin splits them, so the boundary is fixed by position -- for grouped lists (few images, shared
scans of 8 and 4 blocks) and sorted ones (4, 2 and 1 blocks); and the lines between the two."""

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


def _grid():
    """About 10,000 identical corners with a textured patch amid them (better and worse keys)."""
    tile = np.full((16, 16), 60, np.uint8)
    tile[4:11, 4:11] = 200
    tile[4, 4] = tile[10, 10] = 250  # two strict score maxima a tile, of one key
    img = np.tile(tile, (60, 100))
    img[320:560, 400:720] = synth.scene(320, 240, 5, n_rect=60, n_checker=12)
    return img


@pytest.mark.parametrize("frames", [1, 17, 33, 130, 305])
def test_boundary_in_a_run_of_equal_keys(frames):
    img = _grid()
    dev = torch.from_numpy(img).cuda()
    ora = oracle.detect(img, levels=1, fast_t=20, n_features=20000)
    values, first, counts = np.unique(ora["key"], return_index=True, return_counts=True)
    run = counts.argmax()
    start, size = int(first[run]), int(counts[run])
    assert size > 2 * 2048 and start > 0  # more than the first block takes of a bin, and better keys before it
    for n in sorted({max(1, start - 1), start, start + 1, start + size // 2, min(8192, start + size - 1)}):
        det = ofg.Detector(img.shape[1], img.shape[0], max_levels=1, max_features=n, max_batch=frames)
        det.detect_batch([dev] * frames, levels=1, fast_t=20, n_features=n)
        torch.cuda.synchronize()
        for i, got in enumerate(det.batch_results(frames, n)):
            assert len(got) == n
            if i in (0, frames - 1):
                for f in FIELDS:
                    np.testing.assert_array_equal(got[f], ora[f][:n], err_msg=f"{frames} frames, n {n}, frame {i}, {f}")
        det.close()


# Grouped up to 32 images whose squared quotas add up to 16 million or four times the largest: the last
# grouped launch and the first sorted one of 5, 16 and 32 images (8 and 4 blocks an image; 4), four images
# of any quota, and 33 images.
@pytest.mark.parametrize("frames,n", [(8, 4096), (8, 4097), (16, 1024), (16, 1025), (32, 128), (32, 129), (33, 100),
                                      (4, 8192), (5, 1788), (5, 1789), (16, 1000), (16, 1001), (32, 707), (32, 708)])
def test_both_sides_of_the_grouping_lines(frames, n):
    img = synth.scene(900, 700, 8, n_rect=60, n_checker=30, noise_sigma=0.6)  # smooth: long runs of one code
    dev = torch.from_numpy(img).cuda()
    ora = oracle.detect(img, levels=1, fast_t=4, n_features=n)
    det = ofg.Detector(900, 700, max_levels=1, max_features=n, max_batch=frames)
    det.detect_batch([dev] * frames, levels=1, fast_t=4, n_features=n)
    torch.cuda.synchronize()
    for i, got in enumerate(det.batch_results(frames, n)):
        assert len(got) == len(ora) > min(n, 1000) - 1
        if i in (0, frames - 1):
            for f in FIELDS:
                np.testing.assert_array_equal(got[f], ora[f], err_msg=f"frame {i} {f}")
    det.close()


# More slots than the frames can fill, from one for 8 pixels of their 80 x 60 up: the orientation
# kernel looks at the count first.  Grouped lists (1 frame), sorted ones (33), several levels, none.
@pytest.mark.parametrize("frames,levels,n", [(1, 1, 600), (1, 1, 601), (33, 1, 600), (33, 1, 601), (33, 1, 4096), (2, 3, 4096),
                                             (40, 3, 4096)])
@pytest.mark.parametrize("size", [(118, 98), (38, 60)])
def test_slots_beyond_the_keypoints(frames, levels, n, size):
    w, h = size
    img = np.ascontiguousarray(synth.scene(640, 480, 8, n_rect=60, n_checker=30)[100 : 100 + h, 200 : 200 + w])
    dev = torch.from_numpy(img).cuda()
    ora = oracle.detect(img, levels=levels, fast_t=4, n_features=n)
    det = ofg.Detector(w, h, max_levels=levels, max_features=n, max_batch=frames)
    det.detect_batch([dev] * frames, levels=levels, fast_t=4, n_features=n)
    torch.cuda.synchronize()
    for i, got in enumerate(det.batch_results(frames, n)):
        assert len(got) == len(ora)
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ora[f], err_msg=f"frame {i} {f}")
    det.close()


def test_allocation_free_entry_in_a_run_of_equal_keys():
    img = _grid()
    h, w = img.shape
    t = torch.from_numpy(img).cuda()
    out = torch.zeros(8192 * 64, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    ora = oracle.detect(img, levels=1, fast_t=20, n_features=8192)
    for n in (300, 4000, 8192):
        ofg.of_detect_level_noalloc(t, w, h, w, 20, 0, 0.04, n, out, cnt)
        torch.cuda.synchronize()
        got = ofg.keypoints_to_numpy(out[: int(cnt.item()) * 64])
        assert len(got) == n
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ora[f][:n], err_msg=f"n {n} {f}")
