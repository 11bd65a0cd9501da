"""The work this library is used for, as cases that can be timed and checked.

Kinds of case:
  eval     one load increment at a batch of Gauss points (``DMN.eval``), the
           state a few increments into a load path
  warm     the same started from a predicted jump increment (``DMN.eval_warm``)
  control  one stress-controlled adiabatic increment (``DMN.eval_mixed``)
  linear   loss and gradient of the offline training (``DMNLinear.loss_grad``)
  predict  the warm start's network: input rows and inference (``MLP.input``,
           ``MLP.predict``)
  train    one training step of that network (``MLP.train_step``)

Trees, materials and load paths follow ``synthetic.py`` (sizes as in the
benchmark's workloads and the tests); the loads are drawn on the GPU from the
case's seed.  ``exact`` is Algorithm 1, the laminate algebra, the training
loss and the network again, written directly in FP64 PyTorch.
"""
import math

import numpy as np
import torch

from paper_2109_14403_gb300 import DMN, synthetic as syn
from paper_2109_14403_gb300.linear import DMNLinear
from paper_2109_14403_gb300.mlp import MLP

F64 = torch.float64


def listed():
    return [
        # a small model's whole batch: the K = 4 configuration in plain FP64
        dict(name="ramp_k4_fp64_64", kind="eval", K=4, points=64, precision="fp64", matrix="j2",
             load="ramp", past=5, tol=1e-10),
        # the Gauss points of one 27-point hexahedral element: a macro solver's single call
        dict(name="element_k8_mixed_27", kind="eval", K=8, points=27, precision="mixed", matrix="j2",
             load="walk", past=3, tol=1e-12),
        # the plain FP64 path at K = 8: reference runs and the network's training pairs
        dict(name="walk_k8_fp64_8192", kind="eval", K=8, points=8192, precision="fp64", matrix="j2",
             load="walk", past=3, tol=1e-12),
        # uneven increments (a third of a 65,536-point batch), a few points far into yield
        dict(name="uneven_k7_mixed_21845", kind="eval", K=7, points=21845, precision="mixed", matrix="j2",
             load="uneven", past=3, tol=1e-12),
        # the plastic ramp from a^n, an odd batch
        dict(name="ramp_k8_mixed_30011", kind="eval", K=8, points=30011, precision="mixed", matrix="j2",
             load="ramp", past=4, tol=5e-13),
        # the benchmark's batch, warm-started from a prediction good to about 1e-3
        dict(name="warm_k8_mixed_65536", kind="warm", K=8, points=65536, precision="mixed", matrix="j2",
             load="walk", past=3, tol=5e-13),
        # the large configuration's tree and Perzyna matrix
        dict(name="rate_k9_mixed_16384", kind="eval", K=9, points=16384, precision="mixed", matrix="perzyna",
             load="rate", past=2, tol=1e-12),
        # cyclic stress control with adiabatic heating
        dict(name="cyclic_k8_mixed_4096", kind="control", K=8, points=4096, precision="mixed",
             matrix="cyclic", past=3, tol=1e-12),
        # offline training: the paper's mini-batch, and the benchmark's batch
        dict(name="linear_k8_fp32_32", kind="linear", K=8, samples=32, precision="fp32"),
        dict(name="linear_k8_fp32_65536", kind="linear", K=8, samples=65536, precision="fp32"),
        # the warm start's network: inference on the benchmark's batch, one training step
        dict(name="predict_k8_65536", kind="predict", K=8, points=65536, hidden=512, n_hidden=3),
        dict(name="train_k8_4096", kind="train", K=8, points=4096, hidden=512, n_hidden=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "warm", "control", "linear", "linear", "predict", "train"])
    if kind == "eval":
        K = rng.choice([3, 4, 5, 6, 7, 8, 9])
        precision = rng.choice(["fp64", "mixed", "mixed"])
        matrix = "perzyna" if K == 9 else rng.choice(["j2", "j2", "perzyna"])
        load = "rate" if matrix == "perzyna" else rng.choice(["walk", "ramp", "uneven"])
        # about the work of the largest listed evaluation
        most = min(65536, (1 << 22 if precision == "mixed" else 1 << 20) >> K)
        return dict(kind=kind, K=K, points=_log_int(rng, 8, most), precision=precision, matrix=matrix,
                    load=load, past=rng.randint(1, 4), tol=rng.choice([1e-10, 1e-12]))
    if kind == "warm":
        K = rng.choice([6, 7, 8])
        return dict(kind=kind, K=K, points=_log_int(rng, 64, 65536), precision="mixed", matrix="j2",
                    load=rng.choice(["walk", "ramp"]), past=rng.randint(1, 4), tol=5e-13)
    if kind == "control":
        return dict(kind=kind, K=rng.choice([5, 6, 7, 8]), points=_log_int(rng, 64, 4096), precision="mixed",
                    matrix="cyclic", past=rng.randint(1, 3), tol=1e-12)
    if kind == "linear":
        K = rng.choice([3, 4, 5, 6, 7, 8])
        precision = rng.choice(["fp32", "fp32", "fp64"])
        most = 65536 if precision == "fp32" else 8192
        return dict(kind=kind, K=K, samples=_log_int(rng, 16, most), precision=precision)
    K, hidden = rng.choice([6, 7, 8]), rng.choice([256, 512])
    if kind == "predict":
        return dict(kind=kind, K=K, points=_log_int(rng, 32, 65536), hidden=hidden, n_hidden=3)
    return dict(kind=kind, K=K, points=_log_int(rng, 64, 4096), hidden=hidden, n_hidden=3)


def work(case):
    kind = case["kind"]
    N, L = (1 << case["K"]) - 1, 1 << case["K"]
    if kind in ("eval", "warm", "control"):
        z = {"j2": 7, "perzyna": 13, "cyclic": 13}[case["matrix"]] * (L // 2)
        words = 8 + 3 * N + z
        nbytes = 2 * 8 * words + 56 + 456 + 8 + (12 * N if kind == "warm" else 0)
        if kind == "control":
            nbytes += 1 + 48 + 56 + 456 + 4
        # two passes at least: one Newton step and the pass that accepts it
        return {"bytes": case["points"] * nbytes, "flops": case["points"] * 2 * (N * 1005 + L * 155)}
    if kind == "linear":
        n = case["samples"]
        return {"bytes": n * 3 * 288 + 2 * 8 * (3 * N + L) + 24, "flops": n * N * (975 + 2350)}
    n, h, nh = case["points"], case["hidden"], case["n_hidden"]
    nin, nout = 8 + 3 * N, 3 * N
    macs = nin * h + (nh - 1) * h * h + h * nout
    if kind == "predict":
        # load and two states' jumps in; input rows (bf16) and predictions out
        return {"bytes": n * (56 + 2 * 24 * N + 2 * nin + 4 * nout) + 2 * macs, "flops": 2 * n * macs}
    # x, targets, weights with three moments read and written, gradients out
    return {"bytes": n * (2 * nin + 4 * nout) + macs * 4 * 9, "flops": 6 * n * macs - 2 * n * nin * h}


# --------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) + 1000003)


def _rows(matrix):
    return {"j2": syn.materials, "perzyna": syn.materials_viscoplastic, "cyclic": syn.materials_cyclic}[matrix]()


def _dt(case):
    return {"rate": syn.LARGE_DT}.get(case["load"], 1.0)


def _loads(case, seed):
    """deps [past + 1, n, 6], theta [past + 1, n] of the case's load path."""
    g, n, m = _gen(seed), case["points"], case["past"] + 1
    x = torch.randn((m, n, 6), dtype=F64, device="cuda", generator=g)
    dth = torch.rand((m, n), dtype=F64, device="cuda", generator=g)
    if case["load"] == "walk":
        deps = 2e-4 * x
    elif case["load"] == "ramp":
        deps, dth = 1e-4 * x, torch.full_like(dth, 3.0)
        deps[:, :, 0] += 1e-3
    elif case["load"] == "uneven":
        mag = torch.exp(torch.randn((m, n, 1), dtype=F64, device="cuda", generator=g))
        deps = 1e-3 * mag * x / x.norm(dim=-1, keepdim=True)
    else:  # strain rates N(0, 1e-2)/s, 1 K per increment
        deps, dth = 1e-2 * syn.LARGE_DT * x, torch.ones_like(dth)
    return deps, syn.THETA_START + torch.cumsum(dth, 0)


def _cycle(case, seed):
    """mask, target [past + 1, n, 6], dt and heat capacity of the stress cycles."""
    g, n, m = _gen(seed), case["points"], case["past"] + 1
    amp = torch.tensor(syn.CYCLE_AMPLITUDES, dtype=F64, device="cuda")[
        torch.randint(0, len(syn.CYCLE_AMPLITUDES), (n,), device="cuda", generator=g)]
    # a random direction of the 11-22 plane's normal stresses
    d = torch.randint(0, 2, (n,), device="cuda", generator=g)
    dt = syn.CYCLE_PERIOD / syn.CYCLE_STEPS
    t = dt * torch.arange(1, m + 1, dtype=F64, device="cuda")
    target = torch.zeros((m, n, 6), dtype=F64, device="cuda")
    target[:, torch.arange(n, device="cuda"), d] = torch.sin(2 * math.pi * t / syn.CYCLE_PERIOD)[:, None] * amp
    mask = torch.full((n,), syn.MASK_STRESS_ADIABATIC, dtype=torch.uint8, device="cuda")
    w, _, phase = syn.tree(case["K"])
    return mask, target, dt, syn.effective_heat_capacity(w, phase)


def _iso(E, nu):
    K, G = E / (3 * (1 - 2 * nu)), E / (2 * (1 + nu))
    P1 = torch.zeros((6, 6), dtype=F64, device="cuda")
    P1[:3, :3] = 1.0 / 3.0
    P2 = torch.eye(6, dtype=F64, device="cuda") - P1
    return 3 * K[:, None, None] * P1 + 2 * G[:, None, None] * P2


def _stiffness(case, seed):
    """Phase stiffness pairs (contrast up to 100, a rank-one anisotropy) and
    targets between the phases' Reuss and Voigt means."""
    g, n = _gen(seed), case["samples"]

    def rand(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape or (n,), dtype=F64, device="cuda", generator=g)

    C1 = _iso(torch.ones(n, dtype=F64, device="cuda"), rand(0.1, 0.45))
    C2 = _iso(10.0 ** rand(-2.0, 2.0), rand(0.1, 0.45))
    m = torch.randn((n, 6), dtype=F64, device="cuda", generator=g)
    m = m / m.norm(dim=1, keepdim=True)
    q = (m * torch.linalg.solve(C2, m)).sum(1)
    C2 = C2 - (rand(0.0, 0.5) / q)[:, None, None] * m[:, :, None] * m[:, None, :]
    f, b = rand(0.2, 0.8)[:, None, None], rand(0.2, 0.8)[:, None, None]
    reuss = torch.linalg.inv(f * torch.linalg.inv(C1) + (1 - f) * torch.linalg.inv(C2))
    Ct = b * (f * C1 + (1 - f) * C2) + (1 - b) * reuss
    return [((C + C.transpose(1, 2)) / 2).contiguous() for C in (C1, C2, Ct)]


def _net_shape(case):
    N = (1 << case["K"]) - 1
    nin, nout = 8 + 3 * N, 3 * N
    return nin, nout, -(-nin // 128) * 128, -(-nout // 128) * 128


def _net_params(case, seed):
    """[(W [out, in], b [out])] of every layer, FP32, uniform in +-1/sqrt(fan in)."""
    g, (nin, nout, _, _) = _gen(seed + 17), _net_shape(case)
    dims = [(nin, case["hidden"])] + [(case["hidden"],) * 2] * (case["n_hidden"] - 1) + [(case["hidden"], nout)]
    return [(((2 * torch.rand((o, i), device="cuda", generator=g) - 1) / math.sqrt(i)),
             ((2 * torch.rand((o,), device="cuda", generator=g) - 1) / math.sqrt(i))) for i, o in dims]


def _pad_params(case, layers):
    """The layers in the network's flat order, rows and columns padded with 0."""
    nin, nout, kin, nout_pad = _net_shape(case)
    flat = []
    for k, (W, b) in enumerate(layers):
        out = nout_pad if k == len(layers) - 1 else W.shape[0]
        P = torch.zeros((out, kin if k == 0 else W.shape[1]), dtype=W.dtype, device="cuda")
        P[:W.shape[0], :W.shape[1]] = W
        c = torch.zeros(out, dtype=W.dtype, device="cuda")
        c[:b.shape[0]] = b
        flat += [P.reshape(-1), c]
    return torch.cat(flat)


def _net_rows(case, n, seed):
    """n points' loads, states at t^{n-1} and t^n (jumps only; the rest of a
    block is not read) and targets a^{n+1} - a^n."""
    g, N = _gen(seed), (1 << case["K"]) - 1
    words = 8 + 3 * N + 7 * (1 << (case["K"] - 1))
    words += words & 1
    prev, cur = (torch.zeros((n, words), dtype=F64, device="cuda") for _ in range(2))
    prev[:, 8:8 + 3 * N] = 2e-3 * torch.randn((n, 3 * N), dtype=F64, device="cuda", generator=g)
    cur[:, 8:8 + 3 * N] = prev[:, 8:8 + 3 * N] + 3e-4 * torch.randn((n, 3 * N), dtype=F64, device="cuda", generator=g)
    prev[:, 6] = 293.0 + 10.0 * torch.rand(n, dtype=F64, device="cuda", generator=g)
    cur[:, 6] = prev[:, 6] + torch.rand(n, dtype=F64, device="cuda", generator=g)
    theta = cur[:, 6] + torch.rand(n, dtype=F64, device="cuda", generator=g)
    deps = 2e-4 * torch.randn((n, 6), dtype=F64, device="cuda", generator=g)
    mix = torch.randn((6, 3 * N), device="cuda", generator=_gen(5))  # targets follow the load
    tgt = deps.float() @ mix + 1e-4 * torch.randn((n, 3 * N), device="cuda", generator=g)
    return deps, theta.contiguous(), prev, cur, tgt.contiguous()


def _features(case, deps, theta, prev, cur):
    """The network's features in FP64."""
    N = (1 << case["K"]) - 1
    da = cur[:, 8:8 + 3 * N] - prev[:, 8:8 + 3 * N]
    return torch.cat([deps, theta[:, None], (theta - cur[:, 6])[:, None], da], 1)


def _norms(x):
    """Column means and standard deviations (population)."""
    x = x.double()
    return x.mean(0), x.std(0, unbiased=False)


FIT = 4096  # rows that the normalisation is fitted on


# --------------------------------------------------------------------------- prepare, run
def prepare(case, seed):
    s = {"case": case}
    kind = case["kind"]
    if kind in ("eval", "warm", "control"):
        d = DMN(case["K"], *syn.tree(case["K"]), _rows(case["matrix"]), tol=case["tol"],
                precision=case["precision"])
        theta0 = torch.full((case["points"],), syn.THETA_START, dtype=F64, device="cuda")
        state = d.init_state(theta0)
        s["dmn"] = d
    if kind in ("eval", "warm"):
        deps, theta = _loads(case, seed)
        for k in range(case["past"]):
            state = d.eval(deps[k].contiguous(), theta[k].contiguous(), _dt(case), state)[0]
        s.update(deps=deps[-1].contiguous(), theta=theta[-1].contiguous(), state=state)
        if kind == "warm":
            n3 = 3 * ((1 << case["K"]) - 1)
            da = d.eval(s["deps"], s["theta"], _dt(case), state)[0][:, 8:8 + n3] - state[:, 8:8 + n3]
            noise = torch.randn(da.shape, device="cuda", generator=_gen(seed + 29))
            s["da"] = (da.float() * (1.0 + 1e-3 * noise)).contiguous()
    elif kind == "control":
        mask, target, dt, heat = _cycle(case, seed)
        deps, theta, out = torch.zeros((case["points"], 6), dtype=F64, device="cuda"), theta0.clone(), None
        for k in range(case["past"]):
            state, out = d.eval_mixed(mask, target[k].contiguous(), deps, theta, dt, heat, state, out=out,
                                      predict=k > 0)[:2]
        s.update(mask=mask, target=target[-1].contiguous(), deps=deps, theta=theta, dt=dt, heat=heat,
                 state=state, out=out)
    elif kind == "linear":
        s["net"] = DMNLinear(case["K"], *syn.linear_params(case["K"]))
        s["C1"], s["C2"], s["Ct"] = _stiffness(case, seed)
    else:
        n = case["points"]
        net = MLP(K=case["K"], hidden=case["hidden"], n_hidden=case["n_hidden"], max_batch=max(n, 1), seed=0)
        net.set_params(_pad_params(case, _net_params(case, seed)).cpu().numpy())
        deps, theta, prev, cur, tgt = _net_rows(case, FIT, seed + 1)
        net.fit_normalization(net.features(deps, theta, cur, prev), tgt)
        deps, theta, prev, cur, tgt = _net_rows(case, n, seed)
        s["net"] = net
        if kind == "predict":
            s.update(deps=deps, theta=theta, prev=prev, cur=cur)
        else:
            s["x"] = net.normalize_features(net.features(deps, theta, cur, prev))
            s["t"] = net.normalize_targets(tgt)
            s["loss"] = torch.zeros(1, dtype=torch.float32, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "eval":
        state, out, status, iters = s["dmn"].eval(s["deps"], s["theta"], _dt(case), s["state"])
        return {"state": state, "out": out, "status": status, "iters": iters}
    if kind == "warm":
        state, out, status, iters = s["dmn"].eval_warm(s["deps"], s["theta"], _dt(case), s["state"], s["da"])
        return {"state": state, "out": out, "status": status, "iters": iters}
    if kind == "control":
        # the starts are overwritten by the call: each pass has its own
        deps, theta = s["deps"].clone(), s["theta"].clone()
        state, out, status, iters, outer = s["dmn"].eval_mixed(
            s["mask"], s["target"], deps, theta, s["dt"], s["heat"], s["state"], out=s["out"].clone(), predict=True)
        return {"state": state, "out": out, "deps": deps, "theta": theta, "status": status, "iters": iters,
                "outer": outer}
    if kind == "linear":
        loss = s["net"].loss_grad(s["C1"], s["C2"], s["Ct"], precision=case["precision"])
        return {"loss": loss, "grad": s["net"].grad}
    if kind == "predict":
        x = s["net"].input(s["deps"], s["theta"], s["cur"], s["prev"])
        return {"x": x, "da": s["net"].predict(x)}
    s["net"].train_step(s["x"], s["t"], 1e-3, s["loss"])
    return {"loss": s["loss"], "grads": s["net"].grads()}


# --------------------------------------------------------------------------- exact
def _bmat(n):
    """B [m, 6, 3] of the normals n [m, 3]: B a = sym(a (x) n) as a Mandel vector."""
    r, z = math.sqrt(0.5), torch.zeros_like(n[:, 0])
    x, y, w = n[:, 0], n[:, 1], n[:, 2]
    return torch.stack([torch.stack(c, -1) for c in (
        (x, z, z), (z, y, z), (z, z, w), (z, r * w, r * y), (r * w, z, r * x), (r * y, r * x, z))], -2)


def _inv3(A):
    a, b, c = A.unbind(-1)
    bc, ca, ab = (torch.linalg.cross(u, v) for u, v in ((b, c), (c, a), (a, b)))
    return torch.stack([bc, ca, ab], -2) / (a * bc).sum(-1)[..., None, None]


class _Tree:
    """Levels of a tree, root first: (offset, B, c1, c2, w) of their nodes."""

    def __init__(self, K):
        w, normals, _ = syn.tree(K)
        self.K, self.N, self.nleaf = K, (1 << K) - 1, 1 << K
        wt = torch.tensor(w, dtype=F64, device="cuda")
        n = torch.tensor(normals, dtype=F64, device="cuda")
        n = n / n.norm(dim=1, keepdim=True)
        self.leafw, self.levels = wt, []
        for k in range(K, 0, -1):
            off, cnt = (1 << K) - (1 << k), 1 << (k - 1)
            a, b = wt[0::2], wt[1::2]
            wt = a + b
            self.levels.insert(0, (off, _bmat(n[off:off + cnt]), a / wt, b / wt, wt))

    def strains(self, e, a):
        """Leaf strains [n, 2^K, 6] from the macro strain and the jumps [n, N, 3]."""
        e = e[:, None, :]
        for off, B, c1, c2, _ in self.levels:
            J = (B @ a[:, off:off + len(c1), :, None])[..., 0]
            e = torch.stack([e + c2[:, None] * J, e - c1[:, None] * J], 2).flatten(1, 2)
        return e


def _leaves(row, eps, z, eps_n, theta, dt):
    """A material's leaves at strains eps [n, m, 6]: sig, C, tau = dsig/dtheta,
    D, dd = dD/deps, gg = dD/dtheta, X (dissipation), the new z [n, m, nz]."""
    kind, E, nu, alpha, th0, sy0, dsy0, H = (float(v) for v in row[:8])
    K0, G0 = E / (3 * (1 - 2 * nu)), E / (2 * (1 + nu))
    th = theta[:, None]
    one3 = torch.zeros(6, dtype=F64, device="cuda")
    one3[:3] = 1.0
    P1 = torch.outer(one3, one3) / 3
    P2 = torch.eye(6, dtype=F64, device="cuda") - P1
    vp = kind == 2
    dE = float(row[10]) if vp else 0.0
    r = 1 + dE * (th - th0)
    r, dr = torch.where(r < 1e-3, 1e-3, r), torch.where(r < 1e-3, 0.0, dE)
    K, G, sE = K0 * r, G0 * r, dr / r
    ee = eps - (alpha * (th - th0))[..., None] * one3
    if kind:
        ee = ee - z[..., :6]
    tr = ee[..., :3].sum(-1)
    s = 2 * G[..., None] * (ee - (tr / 3)[..., None] * one3)
    trd = (eps - eps_n)[..., :3].sum(-1)
    D = -3 * K * alpha * th * trd / dt
    gg = -3 * alpha * (K + th * K0 * dr) * trd / dt
    dd = (-3 * K * alpha * th / dt)[..., None] * one3 + torch.zeros_like(eps)
    tau = (K0 * dr * tr - 3 * K * alpha)[..., None] * one3
    X = torch.zeros_like(tr)
    if not kind:
        sig = K[..., None] * tr[..., None] * one3 + s
        C = (3 * K[..., None, None] * P1 + 2 * G[..., None, None] * P2).expand(*tr.shape, 6, 6)
        return sig, C, tau, D, dd, gg, X, z
    sy = sy0 + dsy0 * (th - th0)
    sy, dsy = torch.where(sy < 1e-6, 1e-6, sy), torch.where(sy < 1e-6, 0.0, dsy0)
    sn = s.norm(dim=-1).clamp_min(1e-300)
    q, Nn = math.sqrt(1.5) * sn, s / sn[..., None]
    f, den = q - sy - H * z[..., 6], 3 * G + H
    pl = (f > 0).to(F64)
    if vp:
        m, c = float(row[8]), dt / float(row[9])
        dp = torch.zeros_like(f)
        for _ in range(60):
            phi = ((f - den * dp) / sy).clamp_min(0)
            gp = 1 + c * m * phi ** (m - 1) * den / sy
            dp = torch.minimum((dp - (dp - c * phi ** m) / gp).clamp_min(0), f.clamp_min(0) / den)
        phi = ((f - den * dp) / sy).clamp_min(0)
        cm = c * m * phi ** (m - 1)
        kinv = cm / (sy + cm * den)
    else:
        dp, phi, kinv = f / den, torch.zeros_like(f), 1 / den + torch.zeros_like(f)
    dp, kinv = dp * pl, kinv * pl
    th1 = 1 - 3 * G * dp / q.clamp_min(1e-300)
    dep = math.sqrt(1.5) * dp[..., None] * Nn
    sig = K[..., None] * tr[..., None] * one3 + th1[..., None] * s
    thb = 3 * G * kinv - (1 - th1)
    C = (3 * K[..., None, None] * P1 + (2 * G * th1)[..., None, None] * P2
         - (2 * G * thb)[..., None, None] * Nn[..., :, None] * Nn[..., None, :])
    qn = q - 3 * G * dp
    ddp = (sE * qn - dsy * (1 + phi)) * kinv
    tau = tau + (math.sqrt(2 / 3) * (sE * qn - 3 * G * ddp))[..., None] * Nn
    kk = math.sqrt(1.5) * 2 * G * kinv  # d dp / d eps = kk N
    X = sy * dp / dt
    D = D + X
    gg = gg + (dsy * dp + sy * ddp) / dt
    dd = dd + (sy * kk / dt)[..., None] * Nn
    zn = torch.cat([z[..., :6] + dep, (z[..., 6] + dp)[..., None]], -1)
    if vp:
        v = eps - eps_n - dep
        sv, f1 = (sig * v).sum(-1), th * sE / dt
        D = D + f1 * sv
        dd = dd + f1[..., None] * ((C @ v[..., None])[..., 0] + sig - (qn * kk)[..., None] * Nn)
        gg = gg + sE * (1 - th * sE) * sv / dt + f1 * ((tau * v).sum(-1) - qn * ddp)
        zn = torch.cat([zn, eps], -1)
    return sig, C, tau, D, dd, gg, X, zn


def _pass(T, rows, e, a, st, theta, dt):
    """Leaves, residual and condensation at (e, a): (res, da, out [n, 57], new z)."""
    n = e.shape[0]
    el, en = T.strains(e, a), T.strains(st["eps"], st["a"])
    L = [_leaves(rows[j], el[:, j::2], st["z"] if j else None, en[:, j::2], theta, dt) for j in (0, 1)]

    def leaf(i):
        x, y = (v[i] + torch.zeros((n, T.nleaf // 2) + v[i].shape[2:], dtype=F64, device="cuda") for v in L)
        return torch.stack([x, y], 2).flatten(1, 2)

    S, C, V, gg = leaf(0), leaf(1), torch.stack([leaf(0), leaf(2), leaf(4)], -1), leaf(5)
    D, X = (T.leafw * leaf(3)).sum(1), (T.leafw * leaf(6)).sum(1)
    r2, keep = torch.zeros(n, dtype=F64, device="cuda"), []
    for off, B, c1, c2, w in reversed(T.levels):
        a1, a2 = c1[:, None, None], c2[:, None, None]
        CL, CR, VL, VR, SL, SR = C[:, 0::2], C[:, 1::2], V[:, 0::2], V[:, 1::2], S[:, 0::2], S[:, 1::2]
        Bt = B.transpose(-1, -2)
        r = (w * c1 * c2)[:, None] * (Bt @ (SL - SR)[..., None])[..., 0]
        r2 = r2 + (r * r).sum((1, 2))
        S = c1[:, None] * SL + c2[:, None] * SR
        U = (CL - CR) @ B
        Ki = _inv3(Bt @ ((a2 * CL + a1 * CR) @ B))
        t = Bt @ (VL - VR)
        h, Gm = Ki @ t, Ki @ U.transpose(-1, -2)
        gg = c1 * gg[:, 0::2] + c2 * gg[:, 1::2] - c1 * c2 * (t[..., 2] * h[..., 1]).sum(-1)
        C = a1 * CL + a2 * CR - a1 * a2 * (U @ Gm)
        V = a1 * VL + a2 * VR - a1 * a2 * (U @ h)
        keep.insert(0, (Gm, h[..., 0]))
    res = r2.sqrt() / (T.N * S[:, 0].norm(dim=-1))
    de, da = torch.zeros((n, 1, 6), dtype=F64, device="cuda"), torch.zeros_like(a)
    for (off, B, c1, c2, _), (Gm, h) in zip(T.levels, keep):
        x = -((Gm @ de[..., None])[..., 0] + h)
        da[:, off:off + len(c1)] = x
        J = (B @ x[..., None])[..., 0]
        de = torch.stack([de + c2[:, None] * J, de - c1[:, None] * J], 2).flatten(1, 2)
    out = torch.cat([S[:, 0], C[:, 0].flatten(1), V[:, 0, :, 1], D[:, None], V[:, 0, :, 2], gg, X[:, None]], 1)
    return res, da, out, L[1][7]


def _increment(T, rows, st, deps, theta, dt):
    """Algorithm 1 to rounding: (out [n, 57], state at t^{n+1})."""
    e, a, gamma = st["eps"] + deps, st["a"].clone(), 0.5
    res, da, _, _ = _pass(T, rows, e, a, st, theta, dt)
    done = torch.zeros_like(res, dtype=torch.bool)
    res = torch.full_like(res, math.inf)
    for _ in range(40):
        step = torch.where(done, 0.0, 1.0)[:, None, None]
        trial, scale = a + step * da, 1.0
        r2, d2, out, z = _pass(T, rows, e, trial, st, theta, dt)
        for _ in range(8):
            bad = (r2 >= res) & ~done & (r2 > 1e-15)
            if not bool(bad.any()):
                break
            trial = torch.where(bad[:, None, None], trial - scale * (1 - gamma) * da, trial)
            scale *= gamma
            r2, d2, out, z = _pass(T, rows, e, trial, st, theta, dt)
        a, res, da = trial, r2, d2
        if bool(done.all()):
            break
        done = res < 1e-14
    return out, {"eps": e, "theta": theta, "a": a, "z": z}


def _words(T, st):
    n = st["a"].shape[0]
    x = torch.cat([st["eps"], st["theta"][:, None], torch.zeros((n, 1), dtype=F64, device="cuda"),
                   st["a"].reshape(n, -1), st["z"].reshape(n, -1)], 1)
    return torch.nn.functional.pad(x, (0, x.shape[1] & 1))


def _virgin(T, n, matrix):
    nz = 7 if matrix == "j2" else 13
    z = torch.zeros((n, T.nleaf // 2, nz), dtype=F64, device="cuda")
    return {"eps": torch.zeros((n, 6), dtype=F64, device="cuda"),
            "theta": torch.full((n,), syn.THETA_START, dtype=F64, device="cuda"),
            "a": torch.zeros((n, T.N, 3), dtype=F64, device="cuda"), "z": z}


def _exact_eval(case, seed):
    T, rows = _Tree(case["K"]), _rows(case["matrix"])
    deps, theta = _loads(case, seed)
    n, step, got = case["points"], max(1, (1 << 20) >> case["K"]), []
    for i in range(0, n, step):
        st = _virgin(T, min(step, n - i), case["matrix"])
        for k in range(case["past"] + 1):
            out, st = _increment(T, rows, st, deps[k, i:i + step], theta[k, i:i + step], _dt(case))
        got.append((_words(T, st), out))
    return {"state": torch.cat([x for x, _ in got]), "out": torch.cat([x for _, x in got]), "status": None,
            "iters": None}


def _exact_control(case, seed):
    """All six stresses and the heat balance by Newton on (deps, theta)."""
    T, rows = _Tree(case["K"]), _rows(case["matrix"])
    _, target, dt, heat = _cycle(case, seed)
    n, step, got = case["points"], max(1, (1 << 20) >> case["K"]), []
    for i in range(0, n, step):
        m = min(step, n - i)
        st = _virgin(T, m, case["matrix"])
        x = torch.zeros((m, 7), dtype=F64, device="cuda")  # deps, theta - theta^n
        for k in range(case["past"] + 1):
            for _ in range(8):
                th = st["theta"] + x[:, 6]
                out, new = _increment(T, rows, st, x[:, :6], th, dt)
                r = torch.cat([out[:, :6] - target[k, i:i + m], (heat * x[:, 6] / dt - out[:, 48])[:, None]], 1)
                J = torch.zeros((m, 7, 7), dtype=F64, device="cuda")
                J[:, :6, :6] = out[:, 6:42].reshape(m, 6, 6)
                J[:, :6, 6], J[:, 6, :6], J[:, 6, 6] = out[:, 42:48], -out[:, 49:55], heat / dt - out[:, 55]
                dx = torch.linalg.solve(J, r)
                if float((dx.abs() / torch.tensor([1e-2] * 6 + [1.0], dtype=F64, device="cuda")).max()) < 1e-13:
                    break
                x = x - dx
            st = new
        got.append((_words(T, st), out, x[:, :6], st["theta"]))
    state, out, deps, theta = (torch.cat(v) for v in zip(*got))
    return {"state": state, "out": out, "deps": deps, "theta": theta, "status": None, "iters": None, "outer": None}


def _dmn_l(K, C1, C2, normals, v):
    """DMN^L of the samples: the laminates from the leaves to the root."""
    w = v.clamp_min(0)
    n = normals / normals.norm(dim=1, keepdim=True)
    C = torch.stack([C1, C2], 1).repeat(1, 1 << (K - 1), 1, 1)
    for k in range(K, 0, -1):
        off, cnt = (1 << K) - (1 << k), 1 << (k - 1)
        B, wa, wb = _bmat(n[off:off + cnt]), w[0::2], w[1::2]
        w = wa + wb
        c1 = (wa / w)[:, None, None]
        c2 = 1 - c1
        CL, CR = C[:, 0::2], C[:, 1::2]
        U = (CL - CR) @ B
        Ki = _inv3(B.transpose(1, 2) @ ((c2 * CL + c1 * CR) @ B))
        C = c1 * CL + c2 * CR - c1 * c2 * (U @ Ki @ U.transpose(-1, -2))
    return C[:, 0]


def _exact_linear(case, seed, p=1.0, q=10.0, penalty=1e3):
    K, n = case["K"], case["samples"]
    C1, C2, Ct = _stiffness(case, seed)
    normals, v = (torch.tensor(x, dtype=F64, device="cuda").requires_grad_() for x in syn.linear_params(K))
    step = max(1, (1 << 19) >> K)

    def errors(i):
        d = (Ct[i:i + step] - _dmn_l(K, C1[i:i + step], C2[i:i + step], normals, v)).abs() ** p
        return d.sum((1, 2)) ** (1 / p) / (Ct[i:i + step].abs() ** p).sum((1, 2)) ** (1 / p)

    with torch.no_grad():
        e = torch.cat([errors(i) for i in range(0, n, step)])
        m = e.max()
        S = ((e / m) ** q).sum()
        data, coef = m * S ** (1 / q) / n, S ** (1 / q - 1) / n * (e / m) ** (q - 1)
    for i in range(0, n, step):
        (coef[i:i + step] * errors(i)).sum().backward()
    pen = penalty * (v.clamp_min(0).sum() - 1) ** 2
    pen.backward()
    pen = pen.detach()
    return {"loss": torch.stack([data + pen, data, pen]), "grad": torch.cat([normals.grad.reshape(-1), v.grad])}


def _net_input(case, seed, n):
    f = _features(case, *_net_rows(case, FIT, seed + 1)[:4])
    mean, std = _norms(f)
    deps, theta, prev, cur, tgt = _net_rows(case, n, seed)
    return (_features(case, deps, theta, prev, cur) - mean) / std, tgt.double()


def _net_forward(layers, x):
    for W, b in layers[:-1]:
        z = x @ W.T + b
        x = z * torch.sigmoid(z)
    W, b = layers[-1]
    return x @ W.T + b


def _exact_net(case, seed):
    nin, nout, kin, _ = _net_shape(case)
    x, tgt = _net_input(case, seed, case["points"])
    mean, std = _norms(_net_rows(case, FIT, seed + 1)[4])
    layers = [(W.double().requires_grad_(), b.double().requires_grad_()) for W, b in _net_params(case, seed)]
    if case["kind"] == "predict":
        with torch.no_grad():
            da = _net_forward(layers, x) * std + mean
            return {"x": torch.nn.functional.pad(x, (0, kin - nin)), "da": da}
    loss = ((_net_forward(layers, x) - (tgt - mean) / std) ** 2).mean()
    loss.backward()
    grads = _pad_params(case, [(W.grad, b.grad) for W, b in layers])
    return {"loss": loss.detach().reshape(1), "grads": grads.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("eval", "warm"):
        return _exact_eval(case, seed)
    return {"control": _exact_control, "linear": _exact_linear}.get(kind, _exact_net)(case, seed)
