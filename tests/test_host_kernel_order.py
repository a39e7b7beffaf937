"""Kernels that take tensor memory let the launches behind them begin only once they have it: a CTA of a later launch keeps the columns it takes until every
launch before it has ended, so one that began beside a CTA still waiting for columns could make the two wait for each other.  Nothing bounds the wait of an
allocation, so the order is checked in the source and not by running into it."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2207_08820_b200" / "csrc"
RELEASE = re.compile(r"\bmm_pdl_release\(\)|\bdependent_begin\(|griddepcontrol\.launch_dependents")


def kernels():
    """(file, text of a kernel up to the next one) of every kernel that takes tensor memory."""
    for path in sorted([*CSRC.glob("*.cu"), *CSRC.glob("*.cuh")]):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        for body in text.split("__global__")[1:]:
            if "tcgen05.alloc" in body:
                yield path.name, body


def test_kernels_are_found():
    assert {name for name, _ in kernels()} >= {"mma_kernel.cuh", "oper_kernel.cuh", "stem.cu"}


@pytest.mark.parametrize("name,body", list(kernels()), ids=[name for name, _ in kernels()])
def test_dependents_are_released_behind_the_allocation(name, body):
    """By the warp that allocates, next, or by any thread behind a barrier."""
    allocated = body.index("tcgen05.alloc")
    barrier = body.index("__syncthreads()", allocated)
    releases = [m.start() for m in RELEASE.finditer(body)]
    assert releases and all(r > barrier or (r > allocated and "}" not in body[allocated:r]) for r in releases)
