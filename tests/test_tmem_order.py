"""Tensor memory and dependent launches (csrc/conv_tc.cu): a kernel that takes tensor
memory lets the next grid's CTAs in only after a barrier behind its allocation.  An
allocation waits without a limit, so CTAs let in earlier could hold an SM's last columns
and wait for the end of a grid one of whose CTAs waits for columns.  Read from the
source: the order is what can be shown without such a wait."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1610_03918_gb300" / "csrc"


def _kernels():
    out = []
    for path in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        for body in text.split("__global__")[1:]:
            if "tmem_alloc(" in body:
                out.append(pytest.param(body, id=re.search(r"\b(k_\w+)\s*\(", body).group(1)))
    return out


def test_all_kernels_found():
    assert len(_kernels()) == 6


@pytest.mark.parametrize("body", _kernels())
def test_dependents_wait_for_the_allocation(body):
    assert "pdl_enter" not in body and "launch_dependents" not in body
    alloc, release = body.index("tmem_alloc("), body.index("pdl_release()")
    assert body.count("pdl_release()") == 1
    assert alloc < body.index("pdl_wait()") < release
    assert "__syncthreads()" in body[alloc:release]
