"""Launches overlap the kernels before them on the stream, and every pipeline
wait of a kernel gives up after a time limit.  The limit must measure this
kernel only: a warp that starts waiting while an earlier kernel still runs
(its own operands come behind that kernel) would report a timeout for the other
kernel's time.  Read from the sources: in every role of an overlapping kernel
the wait for the earlier kernel comes before the first bounded wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_27460_gb300", "csrc")


def roles(text, kernel):
    """{role: its source} of a kernel, from its `// ---- role ----` marks."""
    body = text[text.index(kernel + "("):]
    body = body[:body.index("\n}\n")]
    parts = re.split(r"// -{16} (.*?) -{16}", body)
    return dict(zip(parts[1::2], parts[2::2]))


@pytest.mark.parametrize("path,kernel,least", [("vie_tc_topk.cuh", "tc_topk_kernel", 4), ("vie_tc_many.cu", "tc_many_kernel", 3)])
def test_no_bounded_wait_before_the_earlier_kernel_has_finished(path, kernel, least):
    waiting = {r: s for r, s in roles(open(os.path.join(CSRC, path)).read(), kernel).items() if "mbar_wait(" in s}
    assert len(waiting) >= least, list(waiting)
    for role, src in waiting.items():
        code = re.sub(r"//.*", "", src)
        first = code.find("griddep_wait(")
        assert 0 <= first < code.index("mbar_wait("), role
