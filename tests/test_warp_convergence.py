"""Aligned warp instructions of the tensor-core products: the lanes of a warp
arrive from bounded waits that each of them makes for itself, so every
tensor-memory load must bring them together first.  Read from the source: a
missing reconvergence need not show on a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_05400_gb300", "csrc")


def test_every_tensor_memory_load_reconverges_its_warp():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "restart_tc.cu")).read())
    loads = [m.start() for m in re.finditer(r'asm volatile\("tcgen05\.ld\.sync', src)]
    assert loads
    for at in loads:
        body = src[src.rindex("__device__ __forceinline__", 0, at):at]
        assert "__syncwarp();" in body
