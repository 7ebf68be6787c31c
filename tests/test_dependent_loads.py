"""Kernels that start beside the ones before them in the stream (they call
grid_dependency_wait) read by plain loads: __ldg and const __restrict__
pointers are only for memory that nothing writes during the kernel."""
import glob
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1612_01855_gb300", "csrc")


def _code(path):
    text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _block(text, at):
    """From the bracket at `at` to its match."""
    pairs = {"(": ")", "{": "}"}
    depth, end = 0, at
    while True:
        depth += (text[end] == text[at]) - (text[end] == pairs[text[at]])
        if depth == 0:
            return text[at:end + 1], end + 1
        end += 1


def _kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__", text):
        at = m.end()
        while True:
            name = re.compile(r"\s*(?:void\s+)?(\w+)\s*(?=\()").match(text, at)
            params, end = _block(text, text.index("(", name.end()))
            if name.group(1) in ("__launch_bounds__", "__maxnreg__"):
                at = end
                continue
            if text[end:].lstrip().startswith("{"):
                body, _ = _block(text, text.index("{", end))
                yield name.group(1), params, body
            break


def test_dependent_kernels_read_by_plain_loads():
    found, sources = {}, set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        text = _code(path)
        for name, params, body in _kernels(text):
            if "grid_dependency_wait()" in body:
                found[name] = params
                sources.add(os.path.basename(path))
    assert {"residue_rows_kernel", "rns_product_kernel", "tc_tile_kernel_persistent", "to_float_kernel",
            "pack_w_tf32_kernel", "pack_w_tf32_vec_kernel", "pack_dt_kernel", "pack_dt_f16_kernel",
            "correct_kernel"} <= set(found)
    for name, params in found.items():
        for p in params.strip("()").split(","):
            assert not ("const" in p.split("*")[0] and "__restrict__" in p), (name, p)
    # the device functions and epilogues they call are in the same files, and
    # in those that launch the tile kernel with their own
    for base in sources | {"tc_gemm.cu"}:
        assert "__ldg(" not in _code(os.path.join(CSRC, base)), base
