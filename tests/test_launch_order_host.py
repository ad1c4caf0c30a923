"""Conversions of more than small tensors let the next launch of the stream start behind their own wait, so that no more than one launch waits on the device at a time: the blocks of
a second one would take the places that the first one's blocks need.  That shows in times alone, so the order is checked in the source, on the CPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_16626_b200", "csrc")
KERNELS = ["convert_kernel", "fq_ta_kernel", "amax_slots_kernel", "amax_kernel"]


@pytest.mark.parametrize("kernel", KERNELS)
def test_the_next_launch_starts_behind_the_wait(kernel):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "hif8_convert.cu")).read())
    body = next(p for p in re.split(r"(?=__global__ void)", text)[1:] if re.search(r"\b" + kernel + r"\(const", p))
    body = body[:body.find("\n}\n")]
    # (measuring and stand-alone instantiations, launches of few blocks and element-by-element ones let it start in front: named by the condition)
    in_front = r"if \((early|ALONE \|\| n_vec == 0|n_vec == 0)\) $"
    general = [m.start() for m in re.finditer(r"pdl_launch_dependents\(\)", body) if not re.search(in_front, body[:m.start()])]
    assert general and min(general) > body.index("pdl_wait_prior_grid()")
