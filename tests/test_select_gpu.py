"""Top-N with clusters of blocks sharing an image: every cluster size the launch
picks (by the number of images), with fewer and more candidates than one block
scans alone, against the oracle and against single-frame calls."""

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


# Images per launch: 4 (8 blocks each), 17 (4), 129 (2), 305 (1).  At t = 4 the
# larger frame holds far more than 4096 candidates on level 0, the small one fewer.
@pytest.mark.parametrize("frames,levels", [(1, 4), (17, 1), (43, 3), (61, 5)])
@pytest.mark.parametrize("w,h,t,n", [(641, 479, 4, 700), (301, 203, 20, 33), (523, 391, 4, 4000)])
def test_every_cluster_size_matches_the_oracle(frames, levels, w, h, t, n):
    scenes = [synth.scene(w, h, 40 + i, background="pink") for i in range(2)]
    dev = [torch.from_numpy(scenes[i % 2]).cuda() for i in range(frames)]
    det = ofg.Detector(w, h, max_levels=levels, max_features=n, max_batch=frames)
    det.detect_batch(dev, levels=levels, fast_t=t, n_features=n)
    torch.cuda.synchronize()
    got = [g.copy() for g in det.batch_results(frames, n)]
    for i in range(2, frames):
        assert np.array_equal(got[i].view(np.uint8), got[i % 2].view(np.uint8)), i
    for i in range(min(2, frames)):
        ora = oracle.detect(scenes[i], levels=levels, fast_t=t, n_features=n)
        assert len(got[i]) == len(ora) > 0
        for f in FIELDS:
            np.testing.assert_array_equal(got[i][f], ora[f], err_msg=f)
    det.close()


def test_radix_path_in_a_cluster():
    """A boundary key shared by more candidates than the sort buffer holds, with a shared scan."""
    tile = synth.scene(64, 64, 9, n_rect=6, n_checker=1, noise_sigma=8.0)
    img = np.tile(tile, (12, 16))
    dev = torch.from_numpy(img).cuda()
    for n in (5, 300, 1500):
        det = ofg.Detector(img.shape[1], img.shape[0], max_levels=1, max_features=n)
        got = det.detect(dev, levels=1, fast_t=3, n_features=n)
        ora = oracle.detect(img, levels=1, fast_t=3, n_features=n)
        assert len(got) == len(ora) == n
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ora[f], err_msg=f)
        det.close()


# Grouped lists (up to 32 images; shared scans of 8 and of 4 blocks) and sorted ones, with
# the ties of a tiled image: runs of one key code beyond the 32 entries read around a
# keypoint, and beyond the 128 read next.
@pytest.mark.parametrize("frames", [1, 17, 33])
@pytest.mark.parametrize("n", [1, 31, 1000, 4097, 8192])
def test_grouped_and_sorted_lists(frames, n):
    tile = synth.scene(64, 64, 9, n_rect=6, n_checker=1, noise_sigma=8.0)
    img = np.tile(tile, (12, 16))
    dev = torch.from_numpy(img).cuda()
    det = ofg.Detector(img.shape[1], img.shape[0], max_levels=1, max_features=n, max_batch=frames)
    det.detect_batch([dev] * frames, levels=1, fast_t=3, n_features=n)
    torch.cuda.synchronize()
    ora = oracle.detect(img, levels=1, fast_t=3, n_features=n)
    for got in det.batch_results(frames, n):
        assert len(got) == len(ora) == n
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ora[f], err_msg=f)
    det.close()


# Thousands of keys that differ in their last bits only: the boundary bin holds more
# than the first block takes, so the cluster splits it by further bits of the keys.
@pytest.mark.parametrize("frames,n", [(1, 1), (1, 2000), (1, 8192), (17, 500)])
def test_a_full_boundary_bin_is_split(frames, n):
    rng = np.random.default_rng(7)
    tile = np.full((16, 16), 60, np.uint8)
    tile[4:11, 4:11] = 200
    img = (np.tile(tile, (60, 80)).astype(np.int16) + rng.integers(-1, 2, (960, 1280))).astype(np.uint8)
    dev = torch.from_numpy(img).cuda()
    det = ofg.Detector(img.shape[1], img.shape[0], max_levels=1, max_features=n, max_batch=frames)
    det.detect_batch([dev] * frames, levels=1, fast_t=20, n_features=n)
    torch.cuda.synchronize()
    ora = oracle.detect(img, levels=1, fast_t=20, n_features=n)
    for got in det.batch_results(frames, n):
        assert len(got) == len(ora) == n
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ora[f], err_msg=f)
    det.close()
