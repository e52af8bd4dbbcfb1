"""The rule for kernels launched programmatically, checked in their source: a
grid's writes are visible only to a kernel that has waited for it, so no kernel
reads a vector before its own griddepcontrol.wait (pdl_wait)."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2507_11512_gb300", "csrc")
# loads and copies of data that earlier kernels write, and the local functions that
# the reduction passes wrap them in
DEPENDENT = re.compile(r"\b(ld_dep|ld_group|ld_n|load_line|load_elems|load_w|load_q|ld_cs|"
                       r"stencil_rows|copy_async)\s*(<[^;()]*>)?\s*\(")


def block_end(text, start):
    """Index past the brace that closes the one at `start`."""
    depth, i = 1, start + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return i


def without_lambdas(body):
    """The body without local function bodies (their calls count, not their text)."""
    while True:
        m = re.search(r"auto \w+ = \[&\]\([^)]*\)[^{;]*\{", body)
        if not m:
            return body
        body = body[:m.start()] + body[block_end(body, m.end() - 1):]


def kernels():
    """(name, body) of every __global__ function that waits."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+)\s*\((?=const|T|long|double|float|int|Ws)",
                             text):
            start = text.index("{", m.end())
            body = without_lambdas(text[start:block_end(text, start)])
            if "pdl_wait()" in body:
                out.append((m.group(1), body))
    return out


KERNELS = kernels()


def test_kernels_are_found():
    names = {n for n, _ in KERNELS}
    assert {"cgs2_pass_kernel", "gs_plane_kernel", "gs_colour_kernel", "stencil_spmv_kernel",
            "vcycle_tail_kernel", "residual_norm_kernel"} <= names
    assert len(KERNELS) >= 20


@pytest.mark.parametrize("name,body", KERNELS, ids=[n for n, _ in KERNELS])
def test_no_vector_is_read_before_the_wait(name, body):
    early = DEPENDENT.search(body[:body.index("pdl_wait()")])
    assert early is None, "%s: %s before pdl_wait()" % (name, early.group(1))
