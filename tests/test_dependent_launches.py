"""Dependent launches, read from the sources.  Kernels that call chain_wait start under their predecessor's tail and are
alive while that one still writes.  Only what no kernel of a product writes may be promised to be read-only there:
every __restrict__ parameter and every __ldg of these kernels names matrix data or an index list."""
import glob
import os
import re

import pytest

from _helpers import ROOT

CSRC = os.path.join(ROOT, "paper_2509_17257_gb300", "csrc")
# written when the matrix is built (or replaced, behind a synchronisation), never by a product
STATIC = {"perm", "order", "rowptr", "other", "blk", "S", "leaves", "cl_off", "cl_size", "V", "nptr", "nother", "nblk",
          "near_off", "G", "parent", "son0", "son1", "E", "kron"}


def strip_comments(src):
    return re.sub(r"//[^\n]*", "", src)


def block_end(src, at):
    """Index after the brace block that opens at or after `at`."""
    i = src.index("{", at)
    depth = 0
    while True:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
        if depth == 0:
            return i


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = strip_comments(open(path).read())
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^;{]*?\)\s+)?(k_\w+)\(", src):
            text = src[m.start():block_end(src, m.end())]
            if "chain_wait()" in text:
                yield m.group(1), text[:text.index("{")], text[text.index("{"):]


KERNELS = {name: (sig, body) for name, sig, body in kernels()}


def test_the_chained_kernels_are_found():
    assert {"k_gather", "k_scatter_y", "k_scatter_yc", "k_coupling64", "k_leaf64", "k_leaf_fwd64", "k_up64", "k_down64",
            "k_leaf_up", "k_pairs", "k_tc_gemm"} == set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_restrict_only_on_data_no_product_writes(name):
    sig, _ = KERNELS[name]
    assert set(re.findall(r"__restrict__\s+(\w+)", sig)) <= STATIC


def test_contractions_promise_their_matrix_operand_only():
    src = strip_comments(open(os.path.join(CSRC, "h2_mm64.cu")).read())
    at = src.index("void dot2(")
    text = src[at:block_end(src, at)]
    assert set(re.findall(r"__restrict__\s+(\w+)", text)) == {"a0", "a1"}
    assert set(re.findall(r"__ldg\((\w+)", text)) == {"a0", "a1"}


def test_tensor_memory_is_taken_before_the_successor_may_start():
    """A successor's CTA that took TMEM of an SM first, and then waited for this grid, would leave both waiting: every
    CTA has its TMEM (allocated, and seen by the whole CTA past a barrier) when it lets the next launch start."""
    _, body = KERNELS["k_tc_gemm"]
    alloc = body.index("tcgen05.alloc")
    assert alloc < body.index("__syncthreads()", alloc) < body.index("chain_release()") < body.index("chain_wait()")
