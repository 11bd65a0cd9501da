"""``dmn_gemm_bf16_tn`` and the network's inference on either side of the rules that
choose a GEMM form: tiles for half of the SMs, short and long reductions, output
rows that begin on 32 bytes or only on 16.

Each output is one chain of FP32 additions of exact bf16 products: against an FP64
product the error is at most K 2^-24 of the sum of the products' magnitudes for
IEEE additions, and the bound is four times that, as in ``test_gpu_mlp.py`` (the
tensor core's need not round to nearest).  The same rows through another form
have the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.cuda.get_device_properties(0).multi_processor_count


def _operands(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    return [torch.randn((r, K), device="cuda", generator=g).to(torch.bfloat16) for r in (M, N)]


@pytest.mark.parametrize("tiles_of_half_the_sms", [0, 1])
@pytest.mark.parametrize("N,K", [(256, 64), (256, 512), (512, 2048)])
def test_products_on_both_sides_of_the_form_rule(tiles_of_half_the_sms, N, K):
    from paper_2109_14403_gb300.mlp import gemm_bf16_tn
    M = 128 * -(-(_sms() // 2 + tiles_of_half_the_sms) // (N // 256))
    a, b = _operands(M, N, K)
    ref, mag = a.double() @ b.double().T, a.double().abs() @ b.double().abs().T
    assert ((gemm_bf16_tn(a, b).double() - ref).abs() <= K * 2.0 ** -22 * mag).all()


@pytest.mark.parametrize("offset", [0, 4, 8])  # floats from a 32-byte boundary: 4 is a 16-byte one only
def test_output_alignment_and_more_tiles_than_sms(offset):
    from paper_2109_14403_gb300.mlp import gemm_bf16_tn
    M, N, K = 128 * (_sms() + 3), 512, 128
    a, b = _operands(M, N, K)
    buf = torch.full((M * N + 16,), -7.0, device="cuda")
    c = buf[offset:offset + M * N].view(M, N)
    gemm_bf16_tn(a, b, c)
    assert (buf[:offset] == -7.0).all() and (buf[offset + M * N:] == -7.0).all()
    part = gemm_bf16_tn(a[:256].contiguous(), b)  # four tiles: the other form
    assert torch.equal(c[:256], part)
    ref, mag = a.double() @ b.double().T, a.double().abs() @ b.double().abs().T
    assert ((c.double() - ref).abs() <= K * 2.0 ** -22 * mag).all()


@pytest.mark.parametrize("hidden", [1024, 2048])
def test_inference_with_short_and_long_reductions(hidden):
    """A batch that fills the chip with 128 x 256 tiles against its first and
    last rows alone, which run the tile form."""
    from paper_2109_14403_gb300.mlp import MLP
    n = 128 * (_sms() // 3 + 1) + 45
    net = MLP(K=8, hidden=hidden, n_hidden=2, max_batch=n, seed=5)
    x = torch.zeros((n, net.n_in_pad), device="cuda")
    x[:, :net.n_in] = torch.randn((n, net.n_in), device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    x = x.to(torch.bfloat16)
    many = net.predict(x)
    assert torch.equal(net.predict(x[:130].contiguous()), many[:130])
    assert torch.equal(net.predict(x[n - 61:].contiguous()), many[n - 61:])
    net.close()
