"""Orders inside the kernels that a run shows only by hanging or racing, checked on their source."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_18719_gb300", "csrc")


def kernels():
    """(file, name, body) of every __global__ function; a body ends at the first line that is a lone brace."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        for m in re.finditer(r"__global__\s[^;{]*?(\w+)\s*\(\s*(?:const|StreamSrc|Src|float)[^{;]*\{\n", text):
            yield os.path.basename(path), m.group(1), text[m.end():text.index("\n}\n", m.end())]


def test_the_kernels_are_found():
    names = {n for _, n, _ in kernels()}
    assert {"gemm_tc_kernel", "gemm_tc2_kernel", "gemv_stream_kernel", "gemv_cluster_kernel", "gemm_wide_kernel",
            "attn_chunk_tc_kernel", "head_kernel", "norm_scale_kernel"} <= names
    found = sum(len(re.findall(r"\b__global__\b", open(p).read())) for p in glob.glob(os.path.join(CSRC, "*.cu")))
    assert found == len(list(kernels()))


def test_dependents_start_after_the_tensor_memory_is_held():
    # a dependent's CTA that shares the SM could otherwise allocate first and then wait for this kernel
    checked = 0
    for path, name, body in kernels():
        if "tcgen05.alloc" not in body:
            continue
        held = body.index("tc_fence_after()", body.index("tcgen05.alloc"))
        assert body.count("pdl_launch_dependents()") == 1, (path, name)
        if name == "gemv_stream_kernel":  # a static_assert has no such CTA fit beside it
            continue
        assert body.index("pdl_launch_dependents()") > held, (path, name)
        checked += 1
    assert checked == 5
