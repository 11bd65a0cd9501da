"""``dmn_options.res_floor`` as a caller turns it off: any positive value, however
small, floors the residual's denominator and changes nothing at a loaded point.
A point without load, stress or residual is then 0 / floor = 0: converged after
Algorithm 1's one obligatory step, not a quotient of zeros."""
import numpy as np
import pytest

from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _eval(K, prec, floor, n=12):
    from paper_2109_14403_gb300 import DMN
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    deps = np.zeros((n, 6))
    deps[n // 2:] = syn.random_walk_k8(n_points=n, n_incr=1)[0][0][n // 2:] * 8.0  # the first half without load
    theta = np.full(n, syn.THETA_START)
    d = DMN(K, *syn.tree(K), syn.materials(), tol=1e-10, precision=prec, res_floor=floor)
    s = d.init_state(torch.tensor(theta, device=dev))
    s, out, st, it = d.eval(torch.tensor(deps, device=dev), torch.tensor(theta, device=dev), 1.0, s)
    d.close()
    return [x.cpu().numpy() for x in (s, out, st, it)]


@pytest.mark.parametrize("K", [1, 3, 4, 6, 8, 9])
@pytest.mark.parametrize("floor", [1e-150, 1e-170, 1e-300, 5e-324])
def test_points_without_stress_converge_whatever_the_floor_fp64(K, floor):
    n = 12
    s, out, st, it = _eval(K, "fp64", floor, n)
    s0, out0, st0, it0 = _eval(K, "fp64", 0.0, n)  # the default floor
    assert (st0 == 0).all()
    assert (st == 0).all(), st
    assert (it[:n // 2] == 1).all() and (out[:n // 2, :6] == 0.0).all()
    for a, b in ((s, s0), (out, out0), (it, it0)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("K", [1, 3, 4, 6, 8, 9])
@pytest.mark.parametrize("floor", [1e-30, 1e-50, 1e-300])
def test_points_without_stress_converge_whatever_the_floor_mixed(K, floor):
    """The mixed forms hold the floor in FP32: below its range it was zero."""
    n = 12
    s, out, st, it = _eval(K, "mixed", floor, n)
    s0, out0, st0, it0 = _eval(K, "mixed", 0.0, n)
    assert (st0 == 0).all()
    assert (st == 0).all(), st
    assert (it[:n // 2] == 1).all() and (out[:n // 2, :6] == 0.0).all()
    for a, b in ((s, s0), (out, out0), (it, it0)):
        assert np.array_equal(a, b)
