"""Argument checks that come before any CUDA call (no GPU)."""
import ctypes

from paper_2109_14403_gb300 import dmn

P = ctypes.c_void_p


def test_gemm_refuses_an_output_that_its_stores_cannot_reach():
    """Rows leave as 16-byte stores: a misaligned output would fault the GPU."""
    L = dmn.load()
    for off in (4, 8):
        assert L.dmn_gemm_bf16_tn(None, 128, 128, 64, P(256), P(512), P(1024 + off)) == dmn.DMN_ERR_ARG
        assert b"16-byte aligned" in L.dmn_last_error()
