"""The benchmark's flop count: two transforms per field and step, on the tensor cores
and on the CUDA cores alike (their sources hold no other dense product of a step)."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1605_04718_gb300", "csrc")


def test_flops_of_a_solve():
    assert bench.transform_flops(128, 8000) == 2 * 2 * 2 * 128**3 * 8000


def test_cuda_core_solve_has_two_products_beside_the_fallback():
    with open(os.path.join(CSRC, "rd_simt_common.cuh")) as f:
        body = f.read()
    body = body[body.index("void implicit_solve_simt("):]
    body = body[:body.index("\n}\n")]
    fallback = body[body.index("} else {"):]
    fallback = fallback[:fallback.index("\n  }\n")]
    assert len(re.findall(r"smem_gemm<", body)) - len(re.findall(r"smem_gemm<", fallback)) == 2
