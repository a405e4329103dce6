"""Frames with more cells in a row than the threshold pass flags in one round (1024): learned and
plain path against the oracle, and the rounds' index arithmetic on the CPU."""

import os
import re

import numpy as np
import pytest

import paper_2506_07164_gb300 as ofg
import synth

CSRC = os.path.join(os.path.dirname(ofg.__file__), "csrc")
FIELDS = ["x_l", "y_l", "level", "fast_score", "A", "B", "C", "m10", "m01", "key"]


@pytest.mark.parametrize("border,cell", [(4, 8), (19, 8), (19, 30), (15, 33), (31, 13)])
def test_rounds_cover_every_cell_once(border, cell):
    """k_cell_apply: rounds of CA_MAX_CELLS cells, each over the chunks that hold their columns; a cell
    outside the round is left to its own."""
    cap = int(re.search(r"CA_MAX_CELLS = (\d+)", open(os.path.join(CSRC, "of_internal.h")).read()).group(1))
    for w in sorted({min(65535, 2 * border + cap * cell + d) for d in (-1, 0, 1, cell, 5 * cell, cap * cell + 3)} | {65535}):
        rx1, xb0 = w - border, border & ~15
        ncx, n_chunks = -(-(w - 2 * border) // cell), (rx1 - xb0 + 15) >> 4
        cols = np.arange(border, rx1)
        cx, ch = (cols - border) // cell, (cols - xb0) >> 4
        seen = np.zeros(ncx, int)
        for g0 in range(0, ncx, cap):
            ng = min(cap, ncx - g0)
            lo, hi = (border + g0 * cell - xb0) >> 4, min(n_chunks, (border + (g0 + ng) * cell - xb0 + 15) >> 4)
            visited = (ch >= lo) & (ch < hi)
            mine = (cx >= g0) & (cx < g0 + ng)
            assert (visited | ~mine).all()          # every column of the round's cells is read
            assert cx[visited & mine].max() - g0 < cap and cx[visited].max() < ncx
            seen[g0:g0 + ng] += 1
        assert (seen == 1).all()


@pytest.mark.gpu
@pytest.mark.parametrize("w,h,cell,border,t,t_lo", [(8300, 90, 8, 19, 20, 7), (8231, 75, 8, 19, 160, 5),
                                                    (33001, 60, 8, 15, 20, 7), (30800, 80, 30, 19, 20, 7)])
def test_learned_and_plain_match_the_oracle(w, h, cell, border, t, t_lo):
    torch = pytest.importorskip("torch")
    import oracle
    from paper_2506_07164_gb300 import learned

    n = 3000
    part = synth.scene(1650, h, w, n_rect=60, n_checker=30)
    img = np.ascontiguousarray(np.tile(part, (1, -(-w // 1650)))[:, :w])
    img[:, ::7] //= 2
    if t > 128:  # some pixels that strong
        img[:, ::3] = np.where(img[:, ::3] > 100, 255, 0)
    ora = oracle.detect(img, levels=2, fast_t=t, fast_t_lo=t_lo, n_features=n, cell=cell, border=border)
    dev = torch.from_numpy(img).cuda()
    det = ofg.Detector(w, h, max_levels=2, max_features=n, fast_t_lo=t_lo, cell=cell, border=border)
    net = learned.TileNet(1)
    plain = det.detect(dev, levels=2, fast_t=t, n_features=n)
    st = ofg.of_detect_learned(det.h, [(dev, w, h, dev.stride(0))], 2, 1.2, t, 0.04, n, net.net, 0.0, 0.0, 0, det.out,
                               det.counts)
    assert st["proposed"] == st["tiles"] > 0
    torch.cuda.synchronize()
    lrn = det.batch_results(1, n)[0]
    assert len(ora) > 0
    for got in (plain, lrn):
        assert len(got) == len(ora)
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ora[f], err_msg=f)
    det.close()
    net.close()
