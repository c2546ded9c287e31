"""Kernels launched programmatically start while the launch before them may still be writing what they read after their
wait.  CUDA defines the non-coherent load only for memory that nothing writes while the kernel runs, so such a kernel
takes no const __restrict__ pointer, which lets the compiler choose that load, and asks for it itself (__ldg) only for
the unembedding weights, which no kernel writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_08670_gb300", "csrc")
WEIGHTS = {"wy + i"}


def kernels():
    """(file, name, parameters, body) of every __global__ function that waits for the launch before it."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            src = re.sub(r"//[^\n]*", "", f.read())
        src = re.sub(r"__(launch_bounds|cluster_dims)__\([^)]*\)", "", src)
        for m in re.finditer(r"__global__\s+void\s+(\w+)\(([^{]*)\)\s*\{", src):
            at, depth = m.end(), 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[at], 0)
                at += 1
            if "pdl_wait()" in src[m.end():at]:
                yield os.path.basename(path), m.group(1), m.group(2), src[m.end():at]


def test_no_non_coherent_reads_of_what_an_earlier_launch_writes():
    found = list(kernels())
    assert {"adacad_beta_kernel", "select_dense_kernel", "lm_lse_finalize_kernel", "att_combine_kernel",
            "select_from_records_kernel", "agg_select_kernel", "lm_head_pair_kernel"} <= {k[1] for k in found}
    for path, name, params, body in found:
        assert "__restrict__" not in params, (path, name)
        assert set(re.findall(r"__ldg\(([^()]*)\)", body)) <= WEIGHTS, (path, name)
