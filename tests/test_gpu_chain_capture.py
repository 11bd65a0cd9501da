"""Chains of overlapped launches (``pdl.cuh``) inside captured graphs: as the first
node, after a copy, after the join of two branches of other kernels, and on
branches beside each other.  A replay gives the bits of the same calls one by one."""
import pytest

from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class _Work:
    """Small calls that run as overlapped chains, each with its own buffers."""

    def __init__(self):
        from paper_2109_14403_gb300 import DMN
        from paper_2109_14403_gb300.linear import DMNLinear
        from paper_2109_14403_gb300.mlp import MLP
        dev = torch.device("cuda:0")
        g = torch.Generator(device="cuda").manual_seed(1)
        self.net = MLP(K=4, hidden=256, n_hidden=3, max_batch=100, seed=2)
        self.rows = torch.zeros((100, self.net.n_in_pad), device=dev)
        self.rows[:, :self.net.n_in] = torch.randn((100, self.net.n_in), device=dev, generator=g)
        self.rows = self.rows.to(torch.bfloat16)
        self.x = torch.zeros_like(self.rows)
        self.y = torch.zeros((100, self.net.n_out), device=dev)
        self.C1, self.C2 = (torch.tensor(c, device=dev) for c in syn.stiffness_pairs(40, seed=3))
        self.lin = DMNLinear(5, *syn.linear_params(5, seed=4), device=dev)
        self.Ct = DMNLinear(5, *syn.linear_params(5, seed=5), device=dev).forward(self.C1, self.C2)
        self.lin.loss_grad(self.C1, self.C2, self.Ct, precision="fp32")  # its workspace
        self.dmn = DMN(4, *syn.tree(4), syn.materials(), tol=1e-12, precision="mixed")
        self.th = torch.full((32,), 300.0, dtype=torch.float64, device=dev)
        self.deps = torch.randn((32, 6), dtype=torch.float64, device=dev, generator=g) * 1e-3
        self.s0 = self.dmn.init_state(torch.full_like(self.th, syn.THETA_START))
        self.s1, self.out, self.st, self.it = self.dmn.eval(self.deps, self.th, 1.0, self.s0)
        torch.cuda.synchronize()

    def predict(self):
        self.x.copy_(self.rows)
        self.net.predict(self.x, self.y)

    def chain(self):  # no copy before it
        self.net.predict(self.x, self.y)

    def grad(self):
        self.lin.loss_grad(self.C1, self.C2, self.Ct, precision="fp32")

    def solve(self):
        self.dmn.eval(self.deps, self.th, 1.0, self.s0, self.s1, self.out, self.st, self.it)

    def results(self):
        torch.cuda.synchronize()
        return [t.clone() for t in (self.y, self.lin.loss, self.s1, self.out)]

    def clear(self):
        for t in (self.y, self.lin.loss, self.s1, self.out):
            t.zero_()
        torch.cuda.synchronize()


def _sequence(w, main, side, order):
    if order == "first":
        w.chain()
        w.grad()
        w.solve()
    elif order == "copy":
        w.predict()
        w.grad()
        w.solve()
        w.grad()
    elif order == "joined":  # two branches end in kernels, the chain follows both
        side.wait_stream(main)
        with torch.cuda.stream(side):
            w.solve()
        w.predict()
        main.wait_stream(side)
        w.grad()
        w.chain()
    else:  # chains on both branches, joined before a solve
        side.wait_stream(main)
        with torch.cuda.stream(side):
            w.grad()
        w.predict()
        main.wait_stream(side)
        w.solve()


@pytest.mark.parametrize("order", ["first", "copy", "joined", "beside"])
def test_captured_chains(order):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w, main, side = _Work(), torch.cuda.Stream(), torch.cuda.Stream()
    w.predict()
    torch.cuda.synchronize()
    w.clear()
    with torch.cuda.stream(main):
        _sequence(w, main, side, order)
    ref = w.results()
    w.clear()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        _sequence(w, main, side, order)
    for _ in range(3):
        w.clear()
        graph.replay()
        for a, b in zip(w.results(), ref):
            assert torch.equal(a, b)
