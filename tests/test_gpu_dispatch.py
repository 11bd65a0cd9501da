"""Which instance of the solve a launch takes.

FP64 trees of every depth up to 9 take the compact kernel, mixed launches of at
most two CTAs per SM the instance with the larger register budget: results
against the oracle on both sides of the rules (tolerances of
``test_gpu_parity.py``: FP64 stress 1e-10 and tangents 1e-8, mixed 1e-8 and
5e-6, relative 2-norms per point), and the same bits from both mixed instances."""
import numpy as np
import pytest

import oracle
from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(K, n, prec, variant, mats, scale=8.0, dt=0.7):
    from paper_2109_14403_gb300 import DMN
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    w, nrm, ph = syn.tree(K)
    deps, theta = syn.random_walk_k8(n_points=n, n_incr=2)
    deps = deps * scale
    d = DMN(K, w, nrm, ph, mats, tol=1e-12, precision=prec, solve_variant=variant)
    s = d.init_state(torch.full((n,), syn.THETA_START, dtype=torch.float64, device=dev))
    res = []
    for k in range(2):
        s, out, st, it = d.eval(torch.tensor(deps[k], device=dev), torch.tensor(theta[k], device=dev), dt, s)
        res.append((s.cpu().numpy(), out.cpu().numpy(), st.cpu().numpy()))
    d.close()
    return deps, theta, dt, res


@pytest.mark.parametrize("K,mats", [(1, "j2"), (2, "j2"), (3, "j2"), (4, "j2"), (5, "perzyna"), (6, "j2"),
                                    (7, "perzyna"), (8, "j2"), (9, "j2")])
def test_fp64_depths_against_the_oracle(K, mats):
    m = syn.materials() if mats == "j2" else syn.materials_viscoplastic()
    n = 12 if K < 8 else 4
    deps, theta, dt, res = _run(K, n, "fp64", 0, m)
    tree = oracle.Tree(K, *syn.tree(K), m)
    so = tree.init_state(n, syn.THETA_START)
    for k in range(2):
        so, oo, _, _ = oracle.eval_batch(tree, deps[k], theta[k], dt, so)
        _, out, st = res[k]
        assert (st == 0).all()
        for sl, tol, floor in ((slice(0, 6), 1e-10, 1e-3), (slice(6, 42), 1e-8, 1.0), (slice(42, 48), 1e-8, 1e-3),
                               (slice(49, 55), 1e-8, 1e-3)):
            ref = np.maximum(np.linalg.norm(oo[:, sl], axis=1), floor)
            assert (np.linalg.norm(out[:, sl] - oo[:, sl], axis=1) / ref).max() < tol


@pytest.mark.parametrize("K,variant", [(3, 0), (5, 0), (6, 13), (8, 13), (8, 14)])
def test_small_and_large_mixed_launches_agree_in_every_bit(K, variant):
    """The first points of a batch of more than two CTAs per SM against the
    same points alone."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1
    _, _, _, many = _run(K, 2 * sms + 5, "mixed", variant, syn.materials())
    from paper_2109_14403_gb300 import DMN
    dev = torch.device("cuda:0")
    deps, theta = syn.random_walk_k8(n_points=2 * sms + 5, n_incr=2)
    for n in (1, 2 * sms):
        d = DMN(K, *syn.tree(K), syn.materials(), tol=1e-12, precision="mixed", solve_variant=variant)
        s = d.init_state(torch.full((n,), syn.THETA_START, dtype=torch.float64, device=dev))
        for k in range(2):
            s, out, st, it = d.eval(torch.tensor(8.0 * deps[k, :n], device=dev),
                                    torch.tensor(theta[k, :n], device=dev), 0.7, s)
            assert np.array_equal(out.cpu().numpy(), many[k][1][:n])
            assert np.array_equal(s.cpu().numpy(), many[k][0][:n])
        d.close()


@pytest.mark.parametrize("K,maxit,tol,scale", [(7, 1, 1e-12, 8.0), (8, 2, 1e-12, 30.0), (8, 50, 1e-7, 30.0),
                                               (7, 50, 1e-9, 20.0)])
def test_states_of_passes_stored_early_or_late(K, maxit, tol, scale):
    """The compact kernel stores the state beside the last pass's condensation
    or after it, and again if the pass is not accepted: the state is that of
    the owner-mapped kernel, which stores once, also where the iteration ends
    by its limit.  Both stop with the same Newton steps in FP32: their jumps
    differ by the residual the steps leave (tol, or the limit's) and rounding."""
    from paper_2109_14403_gb300 import DMN
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    n = 700
    deps, theta = syn.random_walk_k8(n_points=n, n_incr=2)
    res = {}
    for variant in (3, 13):
        d = DMN(K, *syn.tree(K), syn.materials(), tol=tol, maxit=maxit, precision="mixed", solve_variant=variant)
        s = d.init_state(torch.full((n,), syn.THETA_START, dtype=torch.float64, device=dev))
        s, out, st, it = d.eval(torch.tensor(scale * deps[0], device=dev), torch.tensor(theta[0], device=dev), 1.0, s)
        res[variant] = (s.cpu().numpy(), out.cpu().numpy(), st.cpu().numpy(), it.cpu().numpy())
        d.close()
    a, b = res[3], res[13]
    same = (a[3] == b[3]) & (a[2] == b[2])
    assert same.mean() > 0.99
    N3 = 3 * ((1 << K) - 1)
    assert np.isfinite(b[0]).all()
    assert np.array_equal(a[0][:, :7], b[0][:, :7])
    for lo, hi in ((8, 8 + N3), (8 + N3, a[0].shape[1])):
        x, y = a[0][same, lo:hi], b[0][same, lo:hi]
        assert np.abs(x - y).max() <= 1e-5 * np.abs(x).max()
