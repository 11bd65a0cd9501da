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


def test_fp64_stops_at_depth_nine():
    """A K = 10 tree in FP64 fits no SM: refused with the other argument checks."""
    from paper_2109_14403_gb300 import synthetic as syn
    L = dmn.load()
    w, n, ph = syn.tree(10)
    mats, o, h = dmn.materials_from_rows(syn.materials()), dmn.dmn_options(), P()
    for variant in (0, 11):
        L.dmn_default_options(ctypes.byref(o))
        o.solve_variant = variant
        rc = L.dmn_create(ctypes.byref(h), 10, w.ctypes.data_as(P), n.ctypes.data_as(P), ph.ctypes.data_as(P),
                          ctypes.cast(mats, P), 2, ctypes.byref(o))
        assert rc == dmn.DMN_ERR_ARG and b"does not fit one SM" in L.dmn_last_error()
