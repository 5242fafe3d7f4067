"""Kernels that may be resident while the kernel before them still runs (they call pdl_enter())
read what other kernels of a solve write through ordinary loads: a const __restrict__ pointer
or __ldg lets the compiler use non-coherent loads, whose data has to be constant over the
kernel's whole life and which nothing keeps behind the wait.  Only the stencils' coefficients
and the dense coarse inverse are that old.  Read from the source: no GPU shows a missed order
reliably.  The same goes for asynchronous copies into the shared memory of a CTA that ends
without having waited for them."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_03948_gb300", "csrc")
SETUP = {"diag", "invdiag", "c", "inv"}     # written when a problem or its point is set


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//.*", "", f.read())


def kernels():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            for k in re.finditer(r"__global__.*?\n}\n", source(name), re.S):
                if "pdl_enter()" in k.group(0):
                    yield pytest.param(k.group(0), id=re.search(r"\b(k_\w+)\(", k.group(0)).group(1))


def test_kernels_found():
    assert len(list(kernels())) >= 26


@pytest.mark.parametrize("text", list(kernels()))
def test_noncoherent_pointers_are_setup_data(text):
    names = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", text))
    assert names <= SETUP, names - SETUP


@pytest.mark.parametrize("name", ["legs.cu", "march.cu"])
def test_noncoherent_loads_are_setup_data(name):
    args = re.findall(r"__ldg\(\s*([\w.]+)", source(name))
    assert args and all(a.split(".")[-1] in SETUP for a in args), args


def test_column_kernel_waits_for_its_copies_on_every_path():
    """k_colpcg starts the copy of the coarse inverse's triangle before it knows whether its column
    iterates at all (a zero right-hand side, or one that converged a refinement step ago, does
    not), and the V-cycle, which waits for the copy, only runs in the loop."""
    text = source("column.cu")
    body = text[text.index("void col_pcg("):text.index("k_colpcg(")]
    loop = body.index("for (; sc.active && it < maxit; ++it)")
    assert "col_begin(a)" in text[text.index("k_colpcg("):]
    assert "cp.async.wait_all" in body[loop:]
