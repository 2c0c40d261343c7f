"""Kernels launched while the one before them still runs (those that call
wait_for_previous_kernel): what their sources promise the compiler.

A `const __restrict__` parameter says that nobody writes the data while the kernel
lives, which lets loads move above the wait and take the non-coherent path.  Only
tables that are older than the solve (matrix structure, inverses, digits, maps) may
say so; vectors and words of the iteration may not.
"""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_06224_gb300", "csrc")

TABLES = {"kk", "remap0", "item1", "dig_tab", "exp_tab", "job_level", "job_dom", "invp", "inv"}


def source(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def chained_kernels():
    """{name: (parameter text, body)} of every __global__ function that waits."""
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = source(path)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s+)?(\w+)\s*\(", text):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params = text[m.end() : i - 1]
            j = text.index("{", i)
            k, depth = j + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            if "wait_for_previous_kernel()" in text[j:k]:
                out[m.group(1)] = (params, text[j:k])
    return out


def test_only_tables_are_promised_constant():
    kernels = chained_kernels()
    assert {"k_pcg_spmv", "k_pcg_xr", "k_pcg_p", "k_level0_f64tc", "k_level0_f32", "k_coarse_f32", "k_bdot",
            "k_bupdate_xr", "k_bupdate_p"} <= set(kernels)
    for name, (params, _) in kernels.items():
        for p in params.split(","):
            if p.strip().startswith("const") and "__restrict__" in p:
                assert p.split()[-1] in TABLES, (name, p.strip())
    # the helpers through which they read the iteration's vectors
    for path, helper in (("ff_product.cuh", "ff_block_product"), ("primitives.cuh", "sum_children"),
                         ("pcg_state.cuh", "warp_sum_partials")):
        text = source(os.path.join(CSRC, path))
        at = text.index(helper + "(")
        assert "__restrict__" not in text[at : text.index("{", at)], helper


def test_kernels_that_set_all_conv_decide_once_per_block():
    """A grid whose recording block may set all_conv must not let each thread test it:
    the warps of a later block could part, and go on with shared words that nobody set."""
    writers = {n: b for n, (_, b) in chained_kernels().items() if "test_convergence(" in b or "all_conv = 1" in b}
    assert set(writers) == {"k_pcg_p", "k_bupdate_p"}
    for name, body in writers.items():
        assert not re.search(r"if\s*\([^)]*all_conv[^)]*\)\s*return", body), name
        assert body.index("all_conv") < body.index("__syncthreads()") < body.index("if (s_stop)"), name
