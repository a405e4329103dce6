"""Small batches: parts of cell rows as FAST items, 8- and 16-row NMS tiles, the block
NMS kernel that applies the cell flags, kernels started beside their predecessors'
end -- against the oracle, at every bracket of the batch's cell-row strips (below
700, 1200, 6000) and at the ends of the range of cells and borders."""

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


@pytest.mark.parametrize("w,h,frames,levels,cell,border,t,t_lo", [
    (640, 480, 1, 1, 30, 19, 20, 0),
    (641, 479, 1, 8, 30, 19, 20, 7),
    (333, 217, 2, 5, 8, 15, 12, 3),
    (700, 500, 1, 4, 33, 22, 200, 5),
    (700, 500, 1, 4, 13, 19, 20, 7),
    (57, 300, 1, 3, 30, 19, 20, 7),
    (1283, 901, 1, 8, 30, 19, 20, 7),
    (1283, 901, 1, 8, 30, 19, 20, 0),
    (1500, 1100, 1, 8, 20, 19, 30, 7),
    (1601, 1101, 2, 6, 30, 19, 20, 7),
    (500, 400, 2, 4, 40, 19, 20, 7),
])
def test_every_bracket_matches_the_oracle(w, h, frames, levels, cell, border, t, t_lo):
    n = 600
    imgs = [synth.scene(w, h, 70 + i, background="pink") for i in range(frames)]
    dev = [torch.from_numpy(im).cuda() for im in imgs]
    det = ofg.Detector(w, h, max_levels=levels, max_features=n, max_batch=frames, fast_t_lo=t_lo, cell=cell, border=border)
    for _ in range(3):  # back to back: a call must not see the one before it
        det.detect_batch(dev, levels=levels, fast_t=t, n_features=n)
    torch.cuda.synchronize()
    got = det.batch_results(frames, n)
    for i in range(frames):
        ora = oracle.detect(imgs[i], levels=levels, fast_t=t, fast_t_lo=t_lo, n_features=n, cell=cell, border=border)
        assert len(got[i]) == len(ora) > 0
        for f in FIELDS:
            np.testing.assert_array_equal(got[i][f], ora[f], err_msg=f"frame {i} {f}")
    det.close()
