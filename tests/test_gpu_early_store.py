"""States that the compact mixed kernel stores beside a pass it expects to accept
(``solve_compact.cuh``: the residual before it is below 1e4 tol, with a given start
1e7 tol), where it then is not accepted and the iteration goes on.

The reference is the FP64 kernel, which stores once, at the end, stopped after the
same number of Newton steps.  A stale state is the iterate before the last; each
point's last step, measured by stopping the FP64 iteration one step earlier, is the
scale: the mixed state has to lie within a tenth of it.  The mixed steps differ from
the FP64 ones by 5e-6 of their size (the stated bound of the FP32 tangents), so
points whose last step is below 1e-4 of their jumps are left out.  That a pass was
stored early and went on shows in the iteration counts: from the first residual
below 1e4 tol to the first below tol the point took at least two steps."""
import numpy as np
import pytest

from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _load(K, law, n, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    deps = np.random.default_rng(70 + K).normal(0, scale, size=(n, 6))
    return (torch.tensor(deps, device=dev), torch.full((n,), 300.0, dtype=torch.float64, device=dev),
            1.0)


def _eval(K, law, prec, load, tol, maxit=50, da=None):
    from paper_2109_14403_gb300 import DMN
    mats = syn.materials() if law == "j2" else syn.materials_viscoplastic()
    deps, theta, dt = load
    d = DMN(K, *syn.tree(K), mats, tol=tol, maxit=maxit, precision=prec)
    s = d.init_state(torch.full_like(theta, syn.THETA_START))
    r = d.eval(deps, theta, dt, s) if da is None else d.eval_warm(deps, theta, dt, s, da)
    state, _, st, it = [x.cpu().numpy() for x in r]
    d.close()
    return state, st, it


@pytest.mark.parametrize("K,law,scale,tol", [(7, "j2", 6e-3, 1e-6), (8, "j2", 6e-3, 1e-6), (8, "j2", 1e-2, 1e-7),
                                             (9, "perzyna", 3e-2, 1e-7)])
def test_state_of_the_last_pass_where_an_earlier_one_was_stored(K, law, scale, tol):
    n = 400
    load = _load(K, law, n, scale)
    N3 = 3 * ((1 << K) - 1)
    s, st, it = _eval(K, law, "mixed", load, tol)
    _, _, it_early = _eval(K, law, "mixed", load, 1e4 * tol)
    r, st_r, it_r = _eval(K, law, "fp64", load, tol)
    assert (st == 0).all() and (st_r == 0).all()
    gone_on = (it - it_early >= 2) & (it == it_r)
    before = np.full_like(r, np.nan)  # the iterate before the last
    for m in np.unique(it[gone_on]):
        p, _, _ = _eval(K, law, "fp64", load, tol, maxit=int(m) - 1)
        before[it == m] = p[it == m]
    checked = 0
    for lo, hi in ((8, 8 + N3), (8 + N3, s.shape[1])):  # jumps, internal variables
        last = np.abs(r[:, lo:hi] - before[:, lo:hi]).max(axis=1)
        use = gone_on & (last > 1e-4 * np.abs(r[:, lo:hi]).max(axis=1))
        assert (np.abs(s[use, lo:hi] - r[use, lo:hi]).max(axis=1) <= 0.1 * last[use]).all()
        checked += int(use.sum())
    assert checked >= 40, checked


@pytest.mark.parametrize("K,law,scale", [(7, "j2", 6e-3), (8, "j2", 6e-3), (9, "perzyna", 3e-2)])
def test_state_after_a_failed_start(K, law, scale):
    """A start far off, too few steps to get back: every full pass of the first
    iteration stores the state, and the one from a^n has to replace it."""
    n, tol = 300, 1e-6
    load = _load(K, law, n, scale)
    cold, st, it = _eval(K, law, "mixed", load, tol)
    maxit = int(it.max())
    g = torch.Generator(device="cuda").manual_seed(3)
    da = 10.0 * torch.randn((n, 3 * ((1 << K) - 1)), device="cuda", generator=g)
    s, st_w, it_w = _eval(K, law, "mixed", load, tol, maxit=maxit, da=da)
    retried = (st_w & 4) != 0
    assert retried.sum() >= 100 and (it_w[retried] > it[retried]).all()
    assert ((st_w & 3) == 0).all()
    x, y = s[retried, 8:], cold[retried, 8:]
    assert (np.abs(x - y).max(axis=1) <= 1e-6 * np.abs(y).max(axis=1)).all()
