"""The batch reduction and the weight chain of ``dmn_linear_loss_grad`` at the
sizes where they change shape: one block of 128 samples and its neighbours,
many blocks (more than one per thread of the joining block), every depth's
level structure, exponents with and without a general power.

Tolerances as in ``test_gpu_linear.py`` for FP64 laminates: 1e-8 of the loss and
of the largest gradient entry (rounding amplified by the 3x3 jump systems)."""
import numpy as np
import pytest

import oracle.linear as olin
from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _t(a):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


@pytest.mark.parametrize("K,n,p,q", [(1, 1, 1.0, 10.0), (2, 127, 1.0, 10.0), (2, 128, 2.0, 2.0),
                                     (2, 129, 1.5, 3.0), (5, 33, 1.0, 10.0),
                                     (7, 2, 3.0, 1.0)])
def test_loss_and_gradient_against_the_oracle(K, n, p, q):
    from paper_2109_14403_gb300.linear import DMNLinear
    normals, v = syn.linear_params(K, seed=60 + K)
    v = v * 1.01
    tn, tv = syn.linear_params(K, seed=80 + K)
    C1, C2 = syn.stiffness_pairs(n, seed=90 + K)
    Ct = olin.forward(C1, C2, tn, tv)
    J, gn, gv = olin.loss_grad(C1, C2, Ct, normals, v, p=p, q=q, penalty=10.0)
    d = DMNLinear(K, normals, v, device=torch.device("cuda:0"))
    for _ in range(2):  # the second call finds the workspace used
        loss = d.loss_grad(_t(C1), _t(C2), _t(Ct), p=p, q=q, penalty=10.0).cpu().numpy()
    g = d.grad.cpu().numpy()
    scale = max(np.abs(gn).max(), np.abs(gv).max())
    assert abs(loss[0] - J) <= 1e-8 * abs(J)
    assert np.abs(g[:3 * d.N].reshape(-1, 3) - gn).max() <= 1e-8 * scale
    assert np.abs(g[3 * d.N:] - gv).max() <= 1e-8 * scale


def test_more_blocks_than_the_joining_block_has_threads():
    """127 samples 131 times over: J and its gradient scale by r^(1/q - 1)."""
    from paper_2109_14403_gb300.linear import DMNLinear
    K, n, r, q = 2, 127, 131, 10.0
    normals, v = syn.linear_params(K, seed=5)
    C1, C2 = syn.stiffness_pairs(n, seed=6)
    Ct = olin.forward(C1, C2, *syn.linear_params(K, seed=7))
    d = DMNLinear(K, normals, v, device=torch.device("cuda:0"))
    base = d.loss_grad(_t(C1), _t(C2), _t(Ct), q=q, penalty=0.0).clone()
    g = d.grad.clone()
    many = d.loss_grad(*[_t(np.tile(x, (r, 1, 1))) for x in (C1, C2, Ct)], q=q, penalty=0.0)
    f = float(r) ** (1.0 / q - 1.0)
    assert float((many - f * base).abs().max()) <= 1e-8 * float(many[0])
    assert float((d.grad - f * g).abs().max()) <= 1e-8 * float(d.grad.abs().max())


def test_errors_of_zero_and_one_block_of_them():
    """Targets met exactly (up to rounding) in whole blocks: the loss is that
    of the other block."""
    from paper_2109_14403_gb300.linear import DMNLinear
    K, n = 2, 384
    normals, v = syn.linear_params(K, seed=3)
    C1, C2 = (_t(x) for x in syn.stiffness_pairs(n, seed=4))
    d = DMNLinear(K, normals, v, device=torch.device("cuda:0"))
    Ct = d.forward(C1, C2)
    whole = d.loss_grad(C1, C2, Ct, penalty=0.0).cpu().numpy()
    assert 0.0 <= whole[0] < 1e-12
    Ct[128:256] *= 1.1
    loss = d.loss_grad(C1, C2, Ct, penalty=0.0).cpu().numpy()
    e = 0.1 / 1.1  # |1.1 C - C| / |1.1 C| for each of the 128
    assert abs(loss[0] - e * 128 ** 0.1 / n) <= 1e-8 * loss[0]
