"""Source checks of the kernels that start while the kernel before them still runs."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_24647_gb300", "csrc")

# Inputs of earlier calls: complete before the first kernel of a call starts.
INPUTS = {"col", "key", "sel", "pk", "pay", "fk", "seg", "pseg", "d_seg", "d_n", "d_nrows", "d_nsel",
          # the fragments' plan, copied ahead of the kernel before
          "ph", "emit_start", "fd"}


def overlapped_kernels():
    """(name, parameter list, body) of every kernel that waits for the one before it."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^\n]*\)\s+)?(\w+)\s*\(([^)]*)\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            if "wait_prior()" in text[m.end():end]:
                yield m.group(1), m.group(2), text[m.end():end]


def test_overlapped_kernels_are_found():
    names = {n for n, _, _ in overlapped_kernels()}
    assert {"filter_write_kernel", "part_scan_kernel", "part_scatter_kernel", "part_direct_kernel",
            "build_insert_kernel", "probe_scan_kernel", "probe_emit_kernel", "probe_seg_kernel", "dense_emit_kernel",
            "frag_emit_kernel"} <= names


def test_no_promise_that_memory_of_the_kernel_before_is_constant():
    for name, params, _ in overlapped_kernels():
        for p in params.split(","):
            m = re.search(r"\bconst\b[^*]*\*\s*__restrict__\s+(\w+)", p)
            assert not m or m.group(1) in INPUTS, f"{name}: {p.strip()}"


def test_no_block_returns_before_its_wait():
    for name, _, body in overlapped_kernels():
        for m in re.finditer(r"\breturn\b", body):
            before = body[:m.start()]
            assert "wait_prior()" in before, f"{name}: a return ahead of wait_prior()"
