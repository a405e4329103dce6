"""Wide loads at the end of a caller's frame: no byte past (h - 1) pitch + w is read.

Host: the kernels' own address arithmetic (csrc/of_edge.cuh), compiled for the CPU and run over every
position that can be near the end.  GPU: the calls that reach it, against the oracle, on frames that
end exactly where their buffer does.
"""

import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2506_07164_gb300 as ofg

b = sys.modules[ofg.build.__module__]  # the build module (the package exports its function under the same name)

PATCH = r"""
#include <cstdio>
#include <vector>
#include "of_edge.cuh"
// Every keypoint of the last rows of w x h frames: the bytes that the places of its patch cover.
int main() {
    const int row_words = 9, size = 31 * row_words;
    long beyond = 0, bad = 0, missing = 0, wide = 0;
    for (int H = 4; H <= 15; ++H)
        for (int border = H; border <= H + 4; ++border)
            for (int w = 2 * border + 1; w <= 2 * border + 20; ++w) {
                const int h = 2 * border + 3, pitch = (w + 15) / 16 * 16, end = (h - 1) * pitch + w;
                for (int y = border; y < h - border; ++y)
                    for (int x = border; x < w - border; ++x) {
                        const ofk::PatchWords p = ofk::patch_words(x, y, H, w, h, row_words);
                        std::vector<char> got(pitch * h + 16, 0);
                        for (int i = 0; i < size; ++i) {
                            const int r = i / row_words, c = i % row_words;
                            const long at = (long)(y - H + r) * pitch + x - H - p.sh + 4 * c;
                            if (i < p.whole && c < p.nw) {
                                if (at % 4 || at < 0 || at + 4 > end) ++bad;
                                else for (int k = 0; k < 4; ++k) got[at + k] = 1;
                            }
                            if (r <= 2 * H && c < p.nw && at + 4 > end) ++wide;  // as whole words
                        }
                        if (p.tail) {
                            const int x0 = x - H - p.sh + 4 * (p.nw - 1);
                            if (p.whole >= size || p.whole / row_words != 2 * H || p.whole % row_words != p.nw - 1) ++bad;
                            for (int i = 0; i < 4 && x0 + i < w; ++i) got[(y + H) * pitch + x0 + i] = 1;
                            ++beyond;
                        }
                        for (int r = -H; r <= H; ++r)
                            for (int c = -H; c <= H; ++c) missing += !got[(y + r) * pitch + x + c];
                    }
            }
    std::printf("%ld %ld %ld %ld\n", bad, missing, beyond, wide);
}
"""


def _host(tmp_path, source):
    (tmp_path / "edge.cpp").write_text(source)
    cuda = os.path.dirname(os.path.dirname(b._nvcc()))
    exe = str(tmp_path / "edge")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", b.CSRC,
                        str(tmp_path / "edge.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0
    return [int(v) for v in r.stdout.split()]


def test_orientation_patch_words_stay_inside_the_frame(tmp_path):
    bad, missing, beyond, wide = _host(tmp_path, PATCH)
    assert bad == 0 and missing == 0
    assert beyond == wide > 0  # whole words alone would pass the end at these positions


CHUNK = r"""
#include <cstdio>
#include "of_edge.cuh"
// Every 16-byte chunk of the patches around the tiles of w x h frames.
int main() {
    long bad = 0, missing = 0, wide = 0;
    for (int w = 39; w <= 90; ++w) {
        const int h = 41, pitch = (w + 15) / 16 * 16, end = (h - 1) * pitch + w;
        for (int y = 0; y < h; ++y)
            for (int x = 0; x < w; x += 16) {
                const int n = ofk::chunk_bytes(x, w), at = y * pitch + x;
                const int read = ofk::chunk_whole(n, y, h) ? 16 : n;
                bad += at + read > end;
                missing += n != (w - x < 16 ? w - x : 16) || read < n;
                wide += at + 16 > end;  // as a whole chunk
            }
    }
    std::printf("%ld %ld %ld\n", bad, missing, wide);
}
"""


def test_network_patch_chunks_stay_inside_the_frame(tmp_path):
    bad, missing, wide = _host(tmp_path, CHUNK)
    assert bad == 0 and missing == 0
    assert wide > 0  # whole chunks alone would pass the end of these frames


def _ending_frame(img, torch):
    """The frame at a 16-byte pitch in a buffer that ends with its last pixel."""
    h, w = img.shape
    pitch = (w + 15) // 16 * 16
    buf = torch.zeros((h - 1) * pitch + w, dtype=torch.uint8, device="cuda")
    view = buf.as_strided((h, w), (pitch, 1))
    view.copy_(torch.from_numpy(img).cuda())
    return view


@pytest.mark.gpu
@pytest.mark.parametrize("border,radius", [(15, 15), (16, 15), (17, 15), (4, 4), (5, 2)])
@pytest.mark.parametrize("w", [333, 334, 335])
def test_keypoints_at_the_last_admissible_pixel(border, radius, w):
    """A corner whose patch ends with the frame (smallest border, ragged width): records as the oracle's."""
    torch = pytest.importorskip("torch")
    import oracle
    import synth

    h = 180
    rng = np.random.default_rng(w)
    img = synth.scene(w, h, w, n_rect=40, n_checker=8)
    cy, cx = h - 1 - border, w - 1 - border  # a square's corner there, its corner pixel the brightest
    img[cy - 20:, cx - 20:] = 90
    img[cy - 8:cy + 1, cx - 8:cx + 1] = 220
    img[cy, cx] = 250
    img[cy + 4:, cx + 4:] = rng.integers(60, 121, (border - 3, border - 3))
    det = ofg.Detector(w, h, max_levels=2, max_features=4000, border=border, orient_radius=radius)
    got = det.detect(_ending_frame(img, torch), levels=2, fast_t=8, n_features=4000)
    ora = oracle.detect(img, levels=2, fast_t=8, n_features=4000, border=border, radius=radius)
    assert len(got) == len(ora) > 0
    assert ((got["level"] == 0) & (got["y_l"] == cy) & (got["x_l"] == cx)).any()
    for f in ("x_l", "y_l", "level", "fast_score", "A", "B", "C", "m10", "m01", "key"):
        np.testing.assert_array_equal(got[f], ora[f], err_msg=f)
    det.close()


@pytest.mark.gpu
@pytest.mark.parametrize("w,h", [(331, 217), (97, 70), (145, 89), (335, 102), (336, 103)])
def test_proposal_patches_at_the_frame_end(w, h):
    """Logits of the tiles read in place, on frames that end with their buffer, equal those of the same
    patches extracted."""
    torch = pytest.importorskip("torch")
    import synth
    from paper_2506_07164_gb300 import learned

    net = learned.TileNet(0).load(learned.DEFAULT_WEIGHTS)
    det = ofg.Detector(w, h, max_levels=2, max_features=200, max_batch=1, fast_t_lo=7)
    t = _ending_frame(synth.scene(w, h, w), torch)
    ofg.of_detect_learned(det.h, [(t, w, h, t.stride(0))], 2, 1.2, 20, 0.04, 200, net.net, 0.1, 0.0, 1, det.out,
                          det.counts)
    for lvl in range(2):
        raw, dims = det.inspect(ofg.OF_BUF_LOGIT, 0, lvl)
        n, _ = ofg.of_extract_tiles(det.h, 0, lvl)
        if n == 0:
            continue
        p = torch.empty((n, 64, 64), dtype=torch.uint8, device="cuda")
        ofg.of_extract_tiles(det.h, 0, lvl, p, n)
        np.testing.assert_array_equal(raw.view(np.float32), net.logits(p).cpu().numpy())
    det.close()
    net.close()
