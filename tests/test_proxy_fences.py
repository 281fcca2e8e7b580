"""Shared memory that a kernel has read or written itself and then hands to TMA
copies: every thread fences the async proxy, then the CTA meets at a barrier.
A missing fence is a race that no run is sure to show, so this reads the
sources: between the last access of the CTA's own and the first copy that
refills the same bytes there is a fence directly before a barrier."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_17475_gb300", "csrc")
HANDOVER = re.compile(r"fence_proxy_async_smem\(\);\s*(?:return |if \()?__syncthreads(?:_or)?\(")


@pytest.mark.parametrize("file,kernel,last_access,first_copy", [
    # the rotated queries lie in the rings until their fragments are built
    ("tq4.cu", "tq4_split_kernel(", "(qbuf + r * D", "issue(it);"),
    ("tq4_verify.cu", "tq4_verify_pair_kernel(", "qsm[i] = make_uint4(", "issue(it);"),
    # span plan: the combined output of a request, before the next one's copies
    ("tq4.cu", "tq4_split_kernel(", "x[e] = qbuf[", "template <int D, bool VER"),
    ("decode.cu", "decode_span_kernel(", "+ w * WCODES) + h * SROW + d", "run_split(h.b, ctx"),
])
def test_rings_are_fenced_before_copies_refill_them(file, kernel, last_access, first_copy):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    body = text[text.index(kernel):]
    after = body[body.index(last_access):]
    between = after[:after.index(first_copy)]
    assert HANDOVER.search(between), between
