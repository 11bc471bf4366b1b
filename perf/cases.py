"""The work that users of this library have it do, as cases that can be timed and compared.

Kinds of case (`"kind"`):
  kkt      everything one interior-point iteration asks of the network constraint at an iterate:
           residual y - NN(x), Jacobian, Hessian of lambda^T NN and gradient, one call
           (Net.eval_kkt_dev with device tensors, Net.eval_kkt with host arrays)
  residual the residual alone, as each backtracking step of the line search asks for it
  batch    one iterate of many surrogates of equal hidden widths (Batch.eval_kkt_dev, CUDA graph)
  train    training of the warm-start network on solved instances (WarmStart.train)
  ipm      a whole interior-point solve of the adversarial problem (ipm_adversarial)

Networks are random, with the widths, depths and activations of the workloads in synth/nets.py:
weights N(0, 1/fan_in), small biases; softmax classifiers get the gains of synth.make_classifier.
x ~ U[0,1], lambda ~ N(0,1), as in the problems of synth/problems.py.
"""
import math
import random

import torch

from paper_2509_22462_gb300 import nnc


def _net(name, kind, widths, act, out_act, precision, **more):
    return dict(name=name, kind=kind, widths=" ".join(str(w) for w in widths), act=act,
                out_act=out_act, precision=precision, **more)


def listed():
    return [
        # the plain FP64 method on the tiny classifier: small enough that launches count
        _net("tiny_fp64", "kkt", [784, 128, 128, 10], "tanh", "identity", "fp64"),
        # a small surrogate of odd widths and mixed activations, called with host arrays
        _net("odd_bf16_host", "kkt", [37, 130, 261, 61, 5], "softplus gelu tanh", "identity", "bf16",
             host=True),
        # the classifier of the paper's Table 2 / 3 (5.0M parameters, softmax) in the FP32 form
        _net("classifier5m_fp32", "kkt", [784] + [1024] * 5 + [10], "tanh", "softmax", "fp32"),
        # the 104M classifier: the tensor-core form that is the headline, the compensated form for
        # users who want H itself accurate, and the FP64 form that both are held against
        _net("paper104m_bf16", "kkt", [784] + [4096] * 7 + [10], "tanh", "identity", "bf16"),
        _net("paper104m_bf16x3", "kkt", [784] + [4096] * 7 + [10], "tanh", "identity", "bf16x3"),
        _net("paper104m_fp64", "kkt", [784] + [4096] * 7 + [10], "tanh", "identity", "fp64"),
        # backtracking steps of the line search on that net
        _net("paper104m_residual", "residual", [784] + [4096] * 7 + [10], "tanh", "identity", "bf16"),
        # the largest classifier (sigmoid + softmax, 275M parameters) of Eq. 7
        _net("paper274m_bf16", "kkt", [784] + [8192] * 5 + [10], "sigmoid", "softmax", "bf16"),
        # the stability net of the SCOPF problem: few inputs, 37 margins
        _net("scopf68m_bf16", "kkt", [117] + [4096] * 5 + [37], "tanh", "identity", "bf16"),
        # 64 contingency surrogates n_k -> 1024 x 5 -> 1, n_k ~ U{20..200}, one grouped evaluation
        dict(name="scopf_batch64", kind="batch", count=64, n_min=20, n_max=200, hidden=1024, depth=5,
             act="sigmoid", precision="bf16"),
        # warm-start network, two epochs over 2048 solved loads
        dict(name="warmstart_train", kind="train", n_in=512, h1=256, h2=256, n_out=713, rows=2048,
             epochs=2, batch=64, precision="bf16"),
        # a whole solve of the adversarial problem with the plain FP64 method
        _net("ipm5m_fp64", "ipm", [784] + [1024] * 5 + [10], "tanh", "identity", "fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["kkt", "residual", "batch", "train", "ipm"], [0.62, 0.12, 0.1, 0.1, 0.06])[0]
    if kind == "batch":
        n_min = rng.randint(4, 40)
        return dict(kind=kind, count=_log_int(rng, 4, 64), n_min=n_min, n_max=rng.randint(n_min, 200),
                    hidden=_log_int(rng, 64, 1024), depth=rng.randint(2, 5),
                    act=rng.choice(["sigmoid", "tanh"]), precision=rng.choice(["bf16", "bf16x3"]))
    if kind == "train":
        return dict(kind=kind, n_in=64 * rng.randint(1, 8), h1=64 * rng.randint(1, 4),
                    h2=64 * rng.randint(1, 4), n_out=rng.randint(17, 713), rows=_log_int(rng, 200, 2048),
                    epochs=rng.randint(1, 2), batch=rng.choice([32, 64, 64, 128]),
                    precision=rng.choice(["bf16", "bf16", "fp32"]))
    if kind == "ipm":
        widths = [rng.randint(100, 784)] + [_log_int(rng, 32, 1024)] * rng.randint(1, 4) + [rng.randint(4, 10)]
        return dict(kind=kind, widths=" ".join(map(str, widths)), act="tanh", out_act="identity",
                    precision="fp64")
    precision = rng.choice(["fp64", "fp32", "bf16", "bf16", "bf16x3"])
    top = 2048 if precision in ("fp64", "fp32") else 4096
    hidden, depth = _log_int(rng, 24, top), rng.randint(1, 6)
    same = rng.random() < 0.6   # equal hidden widths, or each its own
    widths = [_log_int(rng, 12, 784)]
    widths += [hidden if same else max(8, int(hidden * rng.uniform(0.4, 1.0))) for _ in range(depth)]
    out_act = rng.choice(["identity", "identity", "softmax"])
    widths += [rng.randint(2, 15) if rng.random() < 0.75 else rng.randint(16, 47)]
    case = dict(kind=kind, widths=" ".join(map(str, widths)),
                act=rng.choice(["tanh", "sigmoid", "softplus", "gelu", "tanh sigmoid softplus"]),
                out_act=out_act, precision=precision)
    if kind == "kkt" and rng.random() < 0.2:
        case["host"] = True
    return case


def _shape(case):
    widths = [int(w) for w in case["widths"].split()]
    names = case["act"].split()
    depth = len(widths) - 2
    return widths, [names[l % len(names)] for l in range(depth)] + [case["out_act"]]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _weights(g, widths, acts):
    """Device FP64 weights and biases of one net."""
    W, b = [], []
    last = len(widths) - 2
    for l in range(last + 1):
        w = _randn(g, widths[l + 1], widths[l]) / math.sqrt(widths[l])
        v = 0.05 * _randn(g, widths[l + 1])
        if acts[-1] == "softmax" and l < last and acts[l] == "sigmoid":
            w *= 4.0
            v = -0.5 * w.sum(1)
        if acts[-1] == "softmax" and l == last:
            w *= 3.0
        W.append(w)
        b.append(v)
    return W, b


def _point(g, widths):
    """An iterate (x, y, lambda) of one net."""
    return _rand(g, widths[0]), _randn(g, widths[-1]), _randn(g, widths[-1])


def _host(tensors):
    return [t.cpu().numpy() for t in tensors]


def _surrogates(case):
    """Widths of the batch's nets, n_k ~ U{n_min..n_max} (part of the case, not of its inputs), and
    their activations."""
    rng = random.Random(case["count"] * 1000 + case["n_max"])
    n = [rng.randint(case["n_min"], case["n_max"]) for _ in range(case["count"])]
    acts = [case["act"]] * case["depth"] + ["identity"]
    return [[k] + [case["hidden"]] * case["depth"] + [1] for k in n], acts


def _train_data(case, g):
    """Loads N(1, 0.1^2) and smooth targets of them, and the initial weights (He et al.)."""
    n_in, h1, h2, n_out = case["n_in"], case["h1"], case["h2"], case["n_out"]
    U = 1.0 + 0.1 * _randn(g, case["rows"], n_in)
    A = _randn(g, n_in, n_out) * (10.0 / math.sqrt(n_in))
    T = torch.tanh((U - 1.0) @ A) + 0.05 * _randn(g, case["rows"], n_out)
    params = []
    for m, k in ((h1, n_in), (h2, h1), (n_out, h2)):
        params += [_randn(g, m, k) * math.sqrt(2.0 / k), torch.zeros(m, dtype=torch.float64)]
    return U, T, params


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "train":
        U, T, params = _train_data(case, g)
        ws = nnc.WarmStart(_host(params), precision=case["precision"])
        return dict(case=case, ws=ws, U=U.cpu().numpy(), T=T.cpu().numpy())
    empty = lambda *s: torch.empty(*s, device="cuda", dtype=torch.float64)  # noqa: E731
    if kind == "batch":
        shapes, acts = _surrogates(case)
        nets = []
        for widths in shapes:
            W, b = _weights(g, widths, acts)
            nets.append(nnc.Net(widths, acts, _host(W), _host(b), case["precision"]))
        batch = nnc.Batch(nets)
        batch.use_graph(True)
        n = batch.n_sum
        return dict(case=case, batch=batch, x=_rand(g, n), y=_randn(g, batch.K), lam=_randn(g, batch.K),
                    out=(empty(batch.K), empty(n), empty(batch.h_sum), empty(n)))
    widths, acts = _shape(case)
    W, b = _weights(g, widths, acts)
    net = nnc.Net(widths, acts, _host(W), _host(b), case["precision"])
    x, y, lam = _point(g, widths)
    state = dict(case=case, net=net)
    if kind == "ipm":
        state["x0"] = x.cpu().numpy()
    elif case.get("host"):
        state["x"], state["y"], state["lam"] = _host((x, y, lam))
    else:
        n, m = widths[0], widths[-1]
        state.update(x=x, y=y, lam=lam, out=(empty(m), empty(m, n), empty(n, n), empty(n)))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        loss = state["ws"].train(state["U"], state["T"], case["epochs"], batch=case["batch"], seed=1)
        return [loss] + state["ws"].params()
    if kind == "batch":
        r, J, H, g = state["out"]
        state["batch"].eval_kkt_dev(state["x"], state["y"], state["lam"], r=r, J=J, H=H, g=g)
        return [r, J, H, g]
    if kind == "ipm":
        result, v, lam = nnc.ipm_adversarial(state["net"], state["x0"], target=3)
        return [result["obj"], v, lam]
    if kind == "residual":
        state["net"].residual_dev(state["x"], state["y"], state["out"][0])
        return [state["out"][0]]
    if case.get("host"):
        return list(state["net"].eval_kkt(state["x"], state["y"], state["lam"]))
    r, J, H, g = state["out"]
    state["net"].eval_kkt_dev(state["x"], y=state["y"], lam=state["lam"], r=r, J=J, H=H, grad=g)
    return [r, J, H, g]


def _kkt_work(widths, acts, value_only=False):
    """(bytes, flops): weights once at the 8 bytes they are given in, inputs and outputs once; value
    pass, reverse sweep with n_out + 1 columns, tangents of the layers that H needs (the first
    layer's are its weights), and the lower triangle of H over the curved layers."""
    n, m = widths[0], widths[-1]
    sizes = [a * b for a, b in zip(widths, widths[1:])]
    nbytes, flops = 8 * (sum(sizes) + sum(widths[1:]) + n + 2 * m), 2 * sum(sizes)
    if not value_only:
        nbytes += 8 * (m + m * n + n * n + n)
        flops += 2 * (m + 1) * sum(sizes)
        curved = [a != "identity" for a in acts]
        need = max([l for l, c in enumerate(curved) if c], default=-1)
        flops += 2 * n * sum(sizes[1:need + 1])
        flops += n * (n + 1) * sum(w for w, c in zip(widths[1:], curved) if c)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "train":
        size = case["h1"] * (case["n_in"] + 1) + case["h2"] * (case["h1"] + 1) + case["n_out"] * (case["h2"] + 1)
        nbytes = 8 * case["rows"] * (case["n_in"] + case["n_out"]) + 8 * size
        return {"bytes": nbytes, "flops": 6 * size * case["rows"] * case["epochs"]}
    if kind == "batch":
        shapes, acts = _surrogates(case)
        each = [_kkt_work(widths, acts) for widths in shapes]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    b, f = _kkt_work(*_shape(case), value_only=kind == "residual")
    # a solve takes about ten iterations, each of which needs everything once
    return {"bytes": 10 * b, "flops": 10 * f} if kind == "ipm" else {"bytes": b, "flops": f}


def _act64(name, z):
    """sigma, sigma', sigma'' of an elementwise activation."""
    if name == "tanh":
        t = torch.tanh(z)
        return t, 1 - t * t, -2 * t * (1 - t * t)
    if name in ("sigmoid", "softplus"):
        s = 1 / (1 + torch.exp(-z))
        if name == "sigmoid":
            return s, s * (1 - s), s * (1 - s) * (1 - 2 * s)
        return z.clamp(min=0) + torch.log1p(torch.exp(-z.abs())), s, s * (1 - s)
    if name == "gelu":
        cdf = 0.5 * (1 + torch.erf(z / math.sqrt(2.0)))
        pdf = torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)
        return z * cdf, cdf + z * pdf, pdf * (2 - z * z)
    return z, torch.ones_like(z), torch.zeros_like(z)


def _exact_kkt(W, b, acts, x, y, lam):
    """Residual, Jacobian, Hessian of lambda^T NN and gradient in 64 bits: forward tangents Zdot_l and
    adjoints abar_l give H = sum_l Zdot_l^T diag(sigma'' abar)_l Zdot_l (plus softmax's own term)."""
    a, slopes, curves = x, [], []
    for l, w in enumerate(W):
        z = w @ a + b[l]
        if acts[l] == "softmax":
            a = torch.softmax(z, 0)
            slopes.append(None)
            curves.append(None)
        else:
            a, d1, d2 = _act64(acts[l], z)
            slopes.append(d1)
            curves.append(d2)
    r = y - a
    adj = torch.cat([torch.eye(len(a), dtype=a.dtype, device=a.device), lam[:, None]], 1)
    soft = None
    if acts[-1] == "softmax":
        pl, lb = a * lam, torch.dot(a, lam)
        soft = torch.diag(pl - lb * a) - torch.outer(a, pl) - torch.outer(pl, a) + 2 * lb * torch.outer(a, a)
    c = [None] * len(W)
    for l in range(len(W) - 1, -1, -1):
        if acts[l] == "softmax":
            adj = a[:, None] * (adj - (a @ adj)[None, :])
        else:
            c[l] = curves[l] * adj[:, -1]
            adj = slopes[l][:, None] * adj
        adj = W[l].T @ adj
    J, g = adj[:, :-1].T.contiguous(), adj[:, -1].contiguous()
    n = len(x)
    H = torch.zeros(n, n, dtype=x.dtype, device=x.device)
    zdot = None
    for l, w in enumerate(W):
        zdot = w if zdot is None else w @ zdot
        if acts[l] == "softmax":
            H += zdot.T @ (soft @ zdot)
        elif acts[l] != "identity":
            H += zdot.T @ (c[l][:, None] * zdot)
        if l + 1 < len(W) and acts[l] != "softmax":
            zdot = slopes[l][:, None] * zdot
    return r, J, H, g


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "ipm"):   # many steps, each of which goes on from the last one's rounding
        return None
    g = _gen(seed)
    if kind == "batch":
        shapes, acts = _surrogates(case)
        nets = [_weights(g, widths, acts) for widths in shapes]
        n, K = sum(w[0] for w in shapes), len(shapes)
        x, y, lam = _rand(g, n), _randn(g, K), _randn(g, K)
        got, at = [], 0
        for k, (W, b) in enumerate(nets):
            m = shapes[k][0]
            got.append(_exact_kkt(W, b, acts, x[at:at + m], y[k:k + 1], lam[k:k + 1]))
            at += m
        return [torch.cat([o[i].reshape(-1) for o in got]) for i in range(4)]
    widths, acts = _shape(case)
    W, b = _weights(g, widths, acts)
    x, y, lam = _point(g, widths)
    if kind == "residual":
        a = x
        for l, w in enumerate(W):
            z = w @ a + b[l]
            a = torch.softmax(z, 0) if acts[l] == "softmax" else _act64(acts[l], z)[0]
        return [y - a]
    out = list(_exact_kkt(W, b, acts, x, y, lam))
    return [o.cpu().numpy() for o in out] if case.get("host") else out
