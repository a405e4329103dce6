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


def _body(text, kernel):
    """The kernel's statements: from its opening brace to the matching one."""
    i = text.index("{", text.index(kernel + "("))
    depth, k = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[i + 1:k]
        k += 1


@pytest.mark.parametrize("name,kernel", [("k_pyramid.cu", "k_pyramid"), ("k_fast.cu", "k_fast_cstrip"),
                                         ("k_fast.cu", "k_fast_cells"), ("k_nms_harris.cu", "k_nms_harris"),
                                         ("k_nms_harris.cu", "k_nms_warp"), ("k_select.cu", "k_select"),
                                         ("k_orient.cu", "k_orient")])
def test_every_exit_of_a_chained_kernel_is_behind_its_wait(name, kernel):
    """A wait in every thread (a statement of the kernel's outermost block) comes before each return, or
    directly before it in the same block; a kernel whose last statement is the wait returns nowhere else."""
    body = _body(_source(name), kernel)
    depth, waited, k = 0, False, 0
    for m in re.finditer(r"[{}]|pdl_wait\(\);|\breturn;", body):
        tok = m.group(0)
        if tok == "{":
            depth += 1
        elif tok == "}":
            depth -= 1
        elif tok == "pdl_wait();":
            waited = waited or depth == 0
            k = m.end()
        else:
            assert waited or not body[k:m.start()].strip(), (kernel, body[max(0, m.start() - 200):m.end()])
    assert waited, kernel
