"""The network's kernels at the sizes where their paths change: batches below
and around the 128-row tile, products on either side of the wide form's rule,
buffers that TMA cannot read in place, states that the 16-byte loads cannot.

Gradients: every entry within six standard deviations of the bf16 rounding
model (``oracle.mlp.grad_error_sigma``, as ``test_gpu_mlp.py``).  Where only the
route changes the values are the same bits."""
import numpy as np
import pytest

from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _net(K, hidden, n_hidden, n):
    from paper_2109_14403_gb300.mlp import MLP
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return MLP(K=K, hidden=hidden, n_hidden=n_hidden, max_batch=n, seed=3)


def _batch(net, n, seed=0):
    rng = np.random.default_rng(seed)
    x = np.zeros((n, net.n_in_pad), np.float32)
    x[:, :net.n_in] = rng.normal(size=(n, net.n_in))
    t = np.zeros((n, net.n_out_pad), np.float32)
    t[:, :net.n_out] = rng.normal(size=(n, net.n_out))
    return torch.tensor(x).to(torch.bfloat16).to("cuda:0"), torch.tensor(t, device="cuda:0")


def _misaligned(a, elems):
    """The same values in a buffer that starts `elems` elements off a 16-byte boundary."""
    buf = torch.empty(a.numel() + 16, dtype=a.dtype, device=a.device)
    v = buf[elems:elems + a.numel()].view(a.shape)
    v.copy_(a)
    assert v.data_ptr() % 16
    return v


@pytest.mark.parametrize("K,hidden,n_hidden,n", [(3, 128, 1, 1), (4, 128, 2, 127), (4, 256, 3, 129), (6, 384, 2, 200),
                                                 (2, 128, 8, 64)])
def test_gradients_of_ragged_batches(K, hidden, n_hidden, n):
    net = _net(K, hidden, n_hidden, n)
    x, t = _batch(net, n)
    p = net.params().astype(np.float64)
    q, o = p.copy(), 0
    for a, b in net.layer_dims():
        q[o:o + a * b] = torch.tensor(p[o:o + a * b], dtype=torch.float32).to(torch.bfloat16).double().numpy()
        o += a * b + b
    loss = torch.full((1,), 7.0, dtype=torch.float32, device="cuda:0")
    net.train_step(x, t, 0.0, loss)
    g = net.grads().astype(np.float64)
    x64, t64 = x.double().cpu().numpy(), t.double().cpu().numpy()
    ref, gref = omlp.loss_and_grads(q, net.layer_dims(), x64, t64, net.n_out)
    sig = omlp.grad_error_sigma(q, net.layer_dims(), x64, t64, net.n_out)
    assert (np.abs(g - gref) <= 6.0 * sig + 1e-6 * np.abs(gref).max()).all()
    assert abs(loss.item() - ref) <= 2e-2 * ref
    net.close()


def test_misaligned_buffers_take_the_same_values():
    n = 300
    res = []
    for off in (None, (1, 1)):
        net = _net(4, 256, 2, n)
        x, t = _batch(net, n, seed=5)
        if off:
            x, t = _misaligned(x, off[0]), _misaligned(t, off[1])
        y = net.predict(x).cpu().numpy()
        loss = torch.zeros(1, dtype=torch.float32, device="cuda:0")
        net.train_step(x, t, 1e-3, loss)
        net.train_step(x, t, 1e-3, loss)
        res.append((y, net.grads(), net.params(), loss.item()))
        net.close()
    for a, b in zip(*res):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 128, 1000])
def test_a_step_without_a_loss_buffer_takes_the_same_gradients(n):
    res = []
    for with_loss in (True, False):
        net = _net(4, 128, 2, n)
        x, t = _batch(net, n, seed=2)
        net.train_step(x, t, 1e-3, torch.zeros(1, dtype=torch.float32, device="cuda:0") if with_loss else None)
        res.append((net.grads(), net.params()))
        net.close()
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_narrow_and_square_tiles_agree():
    """Hidden layers of two 128-column tiles: a row panel for every two SMs runs
    64 columns a tile, one panel more 128."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 2
    n = 128 * (sms // 2) + 1
    net = _net(3, 256, 2, n)
    x, _ = _batch(net, n, seed=4)
    assert torch.equal(net.predict(x)[:n - 1], net.predict(x[:n - 1].contiguous()))
    net.close()


def test_wide_and_tile_forms_agree():
    """Rows of a batch that fills the chip with 128 x 256 tiles against the
    same rows alone."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1
    n = 128 * sms + 77
    net = _net(8, 512, 2, n)
    x, _ = _batch(net, n, seed=6)
    many = net.predict(x)
    few = net.predict(x[:400].contiguous())
    assert torch.equal(many[:400], few)
    assert torch.equal(net.predict(x[n - 130:].contiguous()), many[n - 130:])
    net.close()


@pytest.mark.parametrize("K,words", [(1, 11), (1, 12), (3, 30), (5, 101), (5, 102), (8, 1670)])
def test_input_rows_by_both_loads(K, words):
    """dmn_mlp_input with and without the 16-byte loads against normalised
    dmn_mlp_features, bit for bit; words = state words (odd: word by word)."""
    n = 37
    net = _net(K, 128, 1, n)
    g = torch.Generator(device="cuda:0").manual_seed(words)

    def rand(*s):
        return torch.randn(s, dtype=torch.float64, device="cuda:0", generator=g)

    cur, prev = rand(n, words), rand(n, words)
    cur[0, 8], prev[0, 9], cur[1, 10] = 0.0, 1e-300, 5e-42  # zero, and below the float range
    deps, theta = 1e-3 * rand(n, 6), 300.0 + rand(n)
    f = net.features(deps, theta, cur, prev)
    assert torch.equal(f[:, 8:], cur[:, 8:8 + net.n_out].float() - prev[:, 8:8 + net.n_out].float())
    want = net.normalize_features(f)
    assert torch.equal(net.input(deps, theta, cur, prev), want)
    if words % 2 == 0:
        assert torch.equal(net.input(deps, theta, _misaligned(cur, 1), _misaligned(prev, 1)), want)
    f0 = net.normalize_features(net.features(deps, theta, cur, None))
    assert torch.equal(net.input(deps, theta, cur, None), f0)
    net.close()
