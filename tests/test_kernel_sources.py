"""What no run can show without a fault, read from the kernels' sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_15810_b200", "csrc")


def test_kernels_that_abandon_a_wait_let_their_copies_land():
    """Every kernel that loads behind bounded mbarrier waits ends with settle_if_abandoned, which keeps its shared memory until what is in
    flight has landed: beside the freeing of tensor memory behind the last barrier, in a CTA pair in front of that barrier."""
    single = r"\n  if \(warp == [\w:]+\) tmem_dealloc<\w+>\([^)]*\);\n  if \((?:CG == 1 && )?warp == 0\) settle_if_abandoned\(abort_flag\);"
    pair = r"__syncthreads\(\);\n  if \((?:CG == 2 && )?warp == 0\) settle_if_abandoned\(abort_flag\);\n  (?:if \(CG == 2\) )?cluster_sync_all\(\);"
    for name, singles, pairs in (("gemm.cu", 1, 1), ("gemm_swapped.cu", 1, 0), ("gemm_dense.cu", 1, 0), ("gemm_bf16.cu", 1, 1), ("fp8.cu", 1, 0)):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"[ ]*//[^\n]*", "", f.read())
        assert len(re.findall(single, text)) == singles, name
        assert len(re.findall(pair, text)) == pairs, name
        assert len(re.findall(r"tmem_dealloc<", text)) == max(singles, singles + pairs - (1 if name == "gemm.cu" else 0)), name
