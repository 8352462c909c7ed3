"""The pipelined kernels are launched while the kernel before them in the stream may still run, for as long as it
likes.  Their waits are bounded, so no role may begin one before it has waited for that kernel.  Read from the source:
provoking it would take a kernel that stalls another one past its limit."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_10639_b200", "csrc")


def _roles(path):
    """The common head of the file's pipelined kernel, and the body of each of its roles (warp 0, warp 1, the rest)."""
    text = re.sub(r"//[^\n]*", "", open(path).read())
    heads = [m.start() for m in re.finditer(r"__global__ void", text)]
    kernel = next(text[a:b] for a, b in zip(heads, heads[1:] + [len(text)]) if "mbar_wait_bounded" in text[a:b])
    marks = [kernel.index(m) for m in ("\n  if (warp == 0) {", "\n  } else if (warp == 1) {")]
    marks.append(kernel.index("\n  } else {", marks[1]))
    marks.append(kernel.index("\n  }\n", marks[2]))
    return kernel[:marks[0]], [kernel[a:b] for a, b in zip(marks, marks[1:])]


@pytest.mark.parametrize("name", ["gemm_sm100.cu", "split_gemm.cu", "stream_gemm.cu"])
def test_every_role_waits_for_the_kernel_before_its_first_bounded_wait(name):
    head, roles = _roles(os.path.join(CSRC, name))
    assert "mbar_wait_bounded" not in head and len(roles) == 3
    for i, body in enumerate(roles):
        assert "mbar_wait_bounded" in body, i
        before = head + body[:body.index("mbar_wait_bounded")]
        assert "grid_dependency_wait" in before, f"role {i}"
