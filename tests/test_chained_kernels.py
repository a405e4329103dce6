"""Rules that the programmatically chained kernels keep (csrc/of_launch.cuh), read from their sources."""

import os
import re

import pytest

import paper_2506_07164_gb300 as ofg

CSRC = os.path.join(os.path.dirname(ofg.__file__), "csrc")
CHAINED = ["k_pyramid.cu", "k_fast.cu", "k_nms_harris.cu", "k_select.cu", "k_orient.cu"]
# Tables and descriptors that the host writes before a chain starts.
CONSTANT = {"items", "list", "prefix", "slot_img", "xg", "yg"}


def _source(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    # k_resize, before it in the file, is launched plainly, level by level.
    return text[text.index("k_pyramid(const PyrJob"):] if name == "k_pyramid.cu" else text


@pytest.mark.parametrize("name", CHAINED)
def test_non_coherent_loads_read_plan_constants_only(name):
    text = _source(name)
    for m in re.finditer(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?([\w.]+)", text):
        assert m.group(1) in CONSTANT, (name, m.group(0))
