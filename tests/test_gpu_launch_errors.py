"""A launch that CUDA refuses is reported once, by the call that made it: nothing is
left in the thread's error state, where the next launch check of the caller (or of
this library) would find it.

The refusal: work for the legacy stream while a blocking stream of the thread is
being captured, which the runtime turns down before anything reaches the GPU."""
import ctypes

import pytest

from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
P = ctypes.c_void_p


class _Legacy:
    cuda_stream = 0


def _call(what):
    """A call on the legacy stream, its buffers and handles ready."""
    from paper_2109_14403_gb300 import DMN
    from paper_2109_14403_gb300.linear import DMNLinear
    from paper_2109_14403_gb300.mlp import MLP
    dev = torch.device("cuda:0")
    if what == "linear":
        C1, C2 = (torch.tensor(x, device=dev) for x in syn.stiffness_pairs(8, seed=1))
        d = DMNLinear(3, *syn.linear_params(3, seed=2), device=dev)
        Ct = d.forward(C1, C2) * 1.1
        f = lambda s: d.loss_grad(C1, C2, Ct, stream=s)  # noqa: E731
    elif what == "eval":
        d = DMN(4, *syn.tree(4), syn.materials(), precision="mixed")
        th = torch.full((8,), 300.0, dtype=torch.float64, device=dev)
        s0 = d.init_state(th)
        a = (torch.zeros((8, 6), dtype=torch.float64, device=dev), th, 1.0, s0)
        b = (torch.empty_like(s0), torch.empty((8, 57), dtype=torch.float64, device=dev),
             *(torch.empty(8, dtype=torch.int32, device=dev) for _ in range(2)))
        f = lambda s: d.eval(*a, *b, stream=s)  # noqa: E731
    else:
        d = MLP(K=3, hidden=128, n_hidden=2, max_batch=64, seed=1)
        x = torch.zeros((64, d.n_in_pad), dtype=torch.bfloat16, device=dev)
        y = d.predict(x)
        f = lambda s: d.predict(x, y, stream=s)  # noqa: E731
    f(None)
    torch.cuda.synchronize()
    return f


@pytest.mark.parametrize("what", ["linear", "eval", "network"])
def test_a_refused_launch_leaves_no_error_behind(what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    f = _call(what)
    rt = ctypes.CDLL("libcudart.so.13")
    s, graph = P(), P()
    assert rt.cudaStreamCreate(ctypes.byref(s)) == 0
    assert rt.cudaStreamBeginCapture(s, 0) == 0
    try:
        with pytest.raises(RuntimeError, match="captur"):
            f(_Legacy)
        left = rt.cudaGetLastError()
    finally:
        rt.cudaStreamEndCapture(s, ctypes.byref(graph))  # the refusal has invalidated the capture
        rt.cudaGetLastError()
        rt.cudaStreamDestroy(s)
    assert left == 0
    f(None)  # and the call works again
    torch.cuda.synchronize()
