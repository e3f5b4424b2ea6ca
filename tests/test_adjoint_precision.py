"""The precision of the reverse sweep's weight adjoints dL, by the kernel's
source: FP32 sums cover the 32 particles of one warp and one slot each, and
everything beyond that is added in FP64.  (The difference to an FP32 sum over
all of a warp's particles is at most a unit in the last place of dL, below
what the gradient shows, so it cannot be read off a result.)"""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_4624_gb300", "csrc",
                   "pf_adjoint.cu")


def _adjoint():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    start = text.index("k_adjoint(const __grid_constant__ AdjointArgs a)")
    return text[start:text.index("__global__", start)]


def test_weight_adjoints_of_a_threads_particles_are_not_added_in_fp32():
    body = _adjoint()
    stores = re.findall(r"(v\[[^;=]*\])\s*(\+?=)\s*dlw\[q\];", body)
    assert len(stores) == 2, stores  # from the tile's own group and from its second origin
    for target, op in stores:
        assert op == "=" and "[q]" in target, (target, op)
    # across the warps in FP64
    assert len(re.findall(r"\(double\)s_red\[", body)) >= 4
    assert "double r = 0.0" in body
