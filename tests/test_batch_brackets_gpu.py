"""Default dispatch on both sides of every line that a batch's cell-row strips decide: 700 and 1200
(parts of strips, 8- and 16-row NMS tiles), 3000 (block or per-warp NMS kernel), 12000 (launches
chained programmatically or not).  Each frame's records equal those of a call of its own, whose
forms are another bracket's, and one frame's the oracle's."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2506_07164_gb300 as ofg  # noqa: E402

FIELDS = ["x_l", "y_l", "level", "fast_score", "A", "B", "C", "m10", "m01", "key"]
LEVELS, N = 8, 500


def _strips(w, h, border=19, cell=30):
    ws, hs, _ = ofg.of_plan_levels(w, h, LEVELS, 1.2, N)
    x0 = border & ~15
    return sum(-(-(a - border - x0) // 128) * -(-(b - 2 * border) // cell) for a, b in zip(ws, hs)
               if a > 2 * border and b > 2 * border)


def _sizes(target):
    """Frames whose strips add up to the target: large ones first, then smaller ones to fill."""
    out, left = [], target
    for w, h in ((1921, 1080), (1283, 717), (640, 479), (333, 217), (160, 130), (97, 70), (60, 50), (45, 45)):
        s = _strips(w, h)
        while s <= left and (left - s == 0 or len(out) < 60):
            out.append((w, h))
            left -= s
    return out, left


@pytest.mark.parametrize("line", [700, 1200, 3000, 12000])
@pytest.mark.parametrize("below", [True, False])
def test_both_sides_of_every_line(line, below):
    sizes, left = _sizes(line - 1 if below else line)
    assert left == 0
    assert sum(_strips(w, h) for w, h in sizes) == (line - 1 if below else line)
    uniq = sorted(set(sizes))
    imgs = {s: synth.scene(s[0], s[1], 110 + i, background="pink", n_rect=120, n_checker=16) for i, s in enumerate(uniq)}
    dev = {s: torch.from_numpy(imgs[s]).cuda() for s in uniq}
    w, h = max(a for a, _ in sizes), max(b for _, b in sizes)
    det = ofg.Detector(w, h, max_levels=LEVELS, max_features=N, max_batch=len(sizes), fast_t_lo=7)
    one = {s: det.detect(dev[s], levels=LEVELS, fast_t=20, n_features=N) for s in uniq}
    for _ in range(2):
        det.detect_batch([dev[s] for s in sizes], levels=LEVELS, fast_t=20, n_features=N)
    torch.cuda.synchronize()
    for i, got in enumerate(det.batch_results(len(sizes), N)):
        assert np.array_equal(got.view(np.uint8), one[sizes[i]].view(np.uint8)), (i, sizes[i])
    ora = oracle.detect(imgs[sizes[0]], levels=LEVELS, fast_t=20, fast_t_lo=7, n_features=N)
    assert len(ora) > 0
    for f in FIELDS:
        np.testing.assert_array_equal(one[sizes[0]][f], ora[f], err_msg=f)
    det.close()
