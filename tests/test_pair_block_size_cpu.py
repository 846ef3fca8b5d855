"""The SM-pair kernels' occupancy query asks for the block that is launched (CPU only, by
reading): a query with more threads than a kernel's __launch_bounds__ may fail, and the call
with it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_16188_gb300", "csrc")


def test_every_query_names_its_kernels_block():
    src = open(os.path.join(CSRC, "gemm_tc2.cuh")).read()
    bound = {k: b for b, k in re.findall(r"__launch_bounds__\((\w+), 1\)\s+(\w+)\(", src)}
    assert bound["wgrad_pair_kernel"] != bound["row_pair_kernel"]
    seen = 0
    for fn in re.split(r"\n(?=template <|int |inline int )", src):
        for kern, threads in re.findall(r"pair_clusters\(\(const void \*\)(\w+)(?:<[^>]*>)?, (\w+),", fn):
            if kern == "kern":
                kern = re.search(r"auto kern = (\w+)<", fn).group(1)
            assert threads == bound[kern], (kern, threads)
            block = re.search(r"cfg\.blockDim = dim3\((\w+)\)", fn)
            assert block is None or block.group(1) == threads
            seen += 1
    assert seen == 4
    body = open(os.path.join(CSRC, "gemm_tc_bwd.cu")).read()
    body = body[body.index("int pair_clusters("):]
    assert "cfg.blockDim = dim3((unsigned)threads);" in body[:body.index("\n}\n")]
