"""``dmn_linear_loss_grad`` on either side of the rules that choose its kernels:
children of a level pair on one thread or two (128 samples), eight lanes a sample
and overlapped launches or one (2,048), FP32 level pairs of deep trees, exact and
general powers in each of these, repeated squaring or pow() (q = 16).

Tolerances of ``test_gpu_linear.py``: FP64 laminates 1e-8 of the loss and of the
largest gradient entry, FP32 2e-4 and 5e-3.  Deep trees and large batches take the
FP64 laminates as the reference for the FP32 ones (the oracle differentiates one
sample a second at K = 8); those are checked against the oracle on replicated
samples, where J and its gradient scale by r^(1/q - 1)."""
import functools

import numpy as np
import pytest

import oracle.linear as olin
from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-8, 1e-8), "fp32": (2e-4, 5e-3)}


def _t(a):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _problem(K, n, seed=0):
    normals, v = syn.linear_params(K, seed=200 + K + seed)
    C1, C2 = syn.stiffness_pairs(n, seed=300 + n + seed)
    return normals, v * 1.01, C1, C2


def _grad(K, normals, v, C1, C2, Ct, **kw):
    from paper_2109_14403_gb300.linear import DMNLinear
    d = DMNLinear(K, normals, v, device=torch.device("cuda:0"))
    loss = d.loss_grad(C1, C2, Ct, penalty=10.0, **kw).clone()
    return float(loss[1].item()), d.grad.clone(), d


@pytest.mark.parametrize("K,n", [(2, 129), (3, 300), (4, 1), (4, 128), (4, 129), (5, 127), (5, 2048), (5, 2049), (6, 2049),
                                 (7, 128), (7, 129), (7, 300), (8, 127), (8, 129), (8, 2048), (8, 2049)])
def test_fp32_levels_against_fp64(K, n):
    from paper_2109_14403_gb300.linear import DMNLinear
    normals, v, C1, C2 = _problem(K, n)
    C1, C2 = _t(C1), _t(C2)
    Ct = DMNLinear(K, *syn.linear_params(K, seed=400 + K), device=C1.device).forward(C1, C2)
    J, g, _ = _grad(K, normals, v, C1, C2, Ct, precision="fp64")
    J32, g32, _ = _grad(K, normals, v, C1, C2, Ct, precision="fp32")
    assert abs(J32 - J) <= TOL["fp32"][0] * J
    assert float((g32 - g).abs().max()) <= TOL["fp32"][1] * float(g.abs().max())


@functools.lru_cache(maxsize=None)
def _oracle(K, n, p, q):
    normals, v, C1, C2 = _problem(K, n, seed=1)
    Ct = olin.forward(C1, C2, *syn.linear_params(K, seed=401))
    return (normals, v, C1, C2, Ct), olin.loss_grad(C1, C2, Ct, normals, v, p=p, q=q, penalty=0.0)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("r", [1, 65])  # 33 samples, 2,145
@pytest.mark.parametrize("p,q", [(1.0, 10.0), (2.0, 2.0), (1.5, 3.0), (1.0, 16.0), (1.0, 17.0), (1.0, 64.0),
                                 (2.0, 2.5)])
def test_exponents_in_small_and_large_batches(p, q, r, prec):
    from paper_2109_14403_gb300.linear import DMNLinear
    K = 3
    (normals, v, C1, C2, Ct), (J, gn, gv) = _oracle(K, 33, p, q)
    f = float(r) ** (1.0 / q - 1.0)
    d = DMNLinear(K, normals, v, device=_t(C1).device)
    loss = d.loss_grad(*[_t(np.tile(x, (r, 1, 1))) for x in (C1, C2, Ct)], p=p, q=q, penalty=0.0, precision=prec)
    tl, tg = TOL[prec]
    assert abs(float(loss[0]) - f * J) <= tl * f * J
    g = d.grad.cpu().numpy()
    ref = f * np.concatenate([gn.reshape(-1), gv])
    assert np.abs(g - ref).max() <= tg * np.abs(ref).max()


@pytest.mark.parametrize("p", [1.0, 1.5])
@pytest.mark.parametrize("K,n", [(5, 512), (3, 1023), (8, 64)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_overlapped_and_ordinary_launches_agree(K, n, p, prec):
    """n samples fill what overlaps, twice as many do not (FP64, or a general
    power): the batch twice over scales J and its gradient by 2^(1/q - 1)."""
    from paper_2109_14403_gb300.linear import DMNLinear
    q = 3.0
    normals, v, C1, C2 = _problem(K, n, seed=2)
    C1, C2 = _t(C1), _t(C2)
    Ct = DMNLinear(K, *syn.linear_params(K, seed=402), device=C1.device).forward(C1, C2)
    d = DMNLinear(K, normals, v, device=C1.device)
    J = d.loss_grad(C1, C2, Ct, p=p, q=q, penalty=0.0, precision=prec).clone()
    g, f = d.grad.clone(), 2.0 ** (1.0 / q - 1.0)
    J2 = d.loss_grad(*[torch.cat([x, x]).contiguous() for x in (C1, C2, Ct)], p=p, q=q, penalty=0.0, precision=prec)
    tl, tg = TOL[prec]
    assert abs(float(J2[0]) - f * float(J[0])) <= tl * f * float(J[0])
    assert float((d.grad - f * g).abs().max()) <= tg * f * float(g.abs().max())
