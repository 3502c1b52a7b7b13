"""The kernels over the sketch's row tiles are launched with two CTAs per SM
(kSketchCtas): every SpMV among them must ask the compiler for registers that
let two CTAs of 512 threads reside, or half of the grid waits.  Read from the
source, since the count of registers is the compiler's."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_05400_gb300", "csrc")


def test_every_tile_spmv_asks_for_two_ctas_per_sm():
    src = open(os.path.join(CSRC, "kernels_df.cu")).read()
    assert "kSketchCtas = 152 * 2" in open(os.path.join(CSRC, "rks_impl.h")).read()
    kernels = re.findall(r"__launch_bounds__\(([^)]*)\)\s+(k_df_spmv_\w+)\(", src)
    tiles = [(b, k) for b, k in kernels if b.startswith("512")]
    assert {k for _, k in tiles} >= {"k_df_spmv_sketch", "k_df_spmv_ell", "k_df_spmv_warp", "k_df_spmv_dia"}
    assert all(b.replace(" ", "") == "512,2" for b, _ in tiles), tiles
