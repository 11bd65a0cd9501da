"""Evaluations on several streams run side by side: the CTAs of one launch must
not keep those of another off the SMs that have room for them."""
import pytest

from paper_2109_14403_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _graph_us(S, K, n, prec):
    """Shortest of some replays of a graph of S evaluations on as many branches."""
    from paper_2109_14403_gb300 import DMN
    dev = torch.device("cuda:0")
    runs = []
    for i in range(S):
        d = DMN(K, *syn.tree(K), syn.materials(), tol=1e-12, precision=prec)
        g = torch.Generator(device="cuda").manual_seed(1)  # the same points on every branch
        deps = torch.randn((n, 6), dtype=torch.float64, device=dev, generator=g) * 1.6e-3
        theta = torch.full((n,), 300.0, dtype=torch.float64, device=dev)
        s = d.init_state(torch.full((n,), syn.THETA_START, dtype=torch.float64, device=dev))
        s1, out, st, it = d.eval(deps, theta, 1.0, s)
        runs.append((d, (deps, theta, 1.0, s, s1, out, st, it), torch.cuda.Stream()))
    torch.cuda.synchronize()
    graph, main = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=main):
        for d, a, sm in runs:
            sm.wait_stream(main)
            with torch.cuda.stream(sm):
                d.eval(*a)
        for _, _, sm in runs:
            main.wait_stream(sm)
    best = 1e9
    for _ in range(12):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        graph.replay()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * e0.elapsed_time(e1))
    del graph
    for d, _, _ in runs:
        d.close()
    return best


def test_eight_fp64_evaluations_of_a_point_an_sm_overlap():
    """K = 6: eight CTAs fit an SM, so eight launches of a CTA per SM are resident
    together and share its FP64 pipe (about 1.8 times one launch's time); one
    after another they take eight times as long."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = torch.cuda.get_device_properties(0).multi_processor_count - 2
    assert _graph_us(8, 6, n, "fp64") < 3.0 * _graph_us(1, 6, n, "fp64")


@pytest.mark.parametrize("K,variant", [(5, 0), (7, 13), (8, 13)])
def test_instances_on_either_side_of_the_small_launch_rule_agree(K, variant):
    """The instance with the larger register budget serves launches that fill at
    most half of what the SMs hold of it (K = 8: one CTA an SM): the same points
    with the same bits in launches on either side of one and of two an SM."""
    from paper_2109_14403_gb300 import DMN
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev, sms = torch.device("cuda:0"), torch.cuda.get_device_properties(0).multi_processor_count
    d = DMN(K, *syn.tree(K), syn.materials(), tol=1e-12, precision="mixed", solve_variant=variant)
    deps, theta = syn.random_walk_k8(n_points=2 * sms + 1, n_incr=1)
    ref = None
    for n in (2 * sms + 1, 2 * sms, sms + 1, sms):
        s = d.init_state(torch.full((n,), syn.THETA_START, dtype=torch.float64, device=dev))
        s, out, st, it = d.eval(torch.tensor(8.0 * deps[0, :n], device=dev), torch.tensor(theta[0, :n], device=dev),
                                0.7, s)
        ref = ref or (s, out, it)
        assert torch.equal(s, ref[0][:n]) and torch.equal(out, ref[1][:n]) and torch.equal(it, ref[2][:n])
    d.close()
