"""What a user of this framework has it do, as timed cases: single attention layers of the paper's models (8 heads
of 64, 16 layers, Fibonacci or power-of-2 rungs) in evaluation and in training, and one whole stack of layers.

Kinds of a case:
  "fwd"       one forward call with nothing but its inputs, as an evaluation loop makes it: (out, lse)
  "train"     one layer's training step through `fwd` and `bwd` with the buffers that a training program keeps
              (rotated keys, residuals, outputs, workspaces): (out, lse, dq, dk, dv[, dtheta, dd])
  "autograd"  the same step through the `FibAttention` module and torch.autograd: (out, dq, dk, dv, dtheta)
  "stack"     `attention_stack` over `layers` layers without gradients: the last layer's output
"""
import math

import torch

import paper_2606_28560_gb300 as fa

D = 64
DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
RUNGS = {"fib": 15, "pow2": 10}


def _case(kind, dtype, B, T, W, alpha, base="fib", H=8, Hkv=8, rung_grads=True, layers=1, **name):
    return dict(name, kind=kind, dtype=dtype, B=B, H=H, Hkv=Hkv, T=T, W=W, alpha=alpha, base=base,
                rung_grads=rung_grads, layers=layers)


def listed():
    return [
        # one short prompt through the paper's grouped heads (8 query, 2 key/value): latency and launches
        _case("fwd", "bf16", 1, 64, 8, 0.9, Hkv=2, name="fwd_bf16_b1_t64_kv2"),
        # one sequence at the training length in fp32, integer rungs: checking a model against a reference
        _case("fwd", "fp32", 1, 1024, 8, 1.0, name="fwd_fp32_b1_t1024"),
        # an evaluation batch at the training length
        _case("fwd", "bf16", 16, 1024, 8, 0.9, name="fwd_bf16_b16_t1024"),
        # length extrapolation to four times the training length
        _case("fwd", "bf16", 4, 4096, 10, 0.9666667, name="fwd_bf16_b4_t4096"),
        # a layer's training step at the training batch, learned alpha
        _case("train", "bf16", 16, 1024, 8, 0.8801671, name="train_bf16_b16_t1024"),
        # the same with the paper's grouped heads
        _case("train", "bf16", 16, 1024, 8, 1.2371, Hkv=2, name="train_bf16_b16_t1024_kv2"),
        # a fine-tuning step on a few ragged sequences, through the module
        _case("autograd", "bf16", 3, 777, 6, 1.05, name="autograd_bf16_b3_t777"),
        # long-context training, Fibonacci rungs
        _case("train", "bf16", 2, 16384, 12, 1.1, name="train_bf16_b2_t16384_fib"),
        # the reach-matched power-of-2 control under a fixed schedule (no gradient of alpha)
        _case("train", "bf16", 2, 16384, 12, 0.7, base="pow2", rung_grads=False, name="train_bf16_b2_t16384_pow2"),
        # a training step in fp32 at an uneven length
        _case("train", "fp32", 4, 1000, 8, 0.7333333, name="train_fp32_b4_t1000"),
        # a training step with a wider local window than the paper sweeps
        _case("train", "bf16", 4, 1024, 32, 0.9, name="train_bf16_b4_t1024_w32"),
        # evaluation of a whole stack of layers, staggered alpha (four: without projections and residual connections the
        # values of a deeper one shrink towards their mean, and its output is mostly rounding)
        _case("stack", "bf16", 8, 1024, 8, 0.0, layers=4, name="stack4_bf16_b8_t1024"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "train", "train", "train", "autograd", "stack"])
    dtype = "bf16" if kind in ("autograd", "stack") else rng.choice(["bf16", "bf16", "bf16", "fp32"])
    W = rng.choice([6, 8, 10, 12])
    if kind in ("fwd", "train") and dtype == "bf16" and rng.random() < 0.2:
        W = rng.randint(17, 40)
    wide = W > 16 or dtype == "fp32"
    most = 4000 if wide else 8000 if kind == "stack" else 24000    # tokens
    T = _spread(rng, 40, most)
    B = max(1, min(16, _spread(rng, 1, max(1.5, most / T)), most // T))
    base = rng.choice(["fib", "fib", "pow2"])
    Hkv = 8 if kind == "stack" else rng.choice([8, 8, 2])
    return _case(kind, dtype, B, T, W, 0.0 if kind == "stack" else round(rng.uniform(0.5, 1.5), 6), base=base, Hkv=Hkv,
                 rung_grads=kind == "autograd" or rng.random() < 0.75, layers=rng.randint(2, 4) if kind == "stack" else 1)


def _normal(shape, dtype, gen):
    return torch.randn(shape, generator=gen, dtype=torch.float32, device="cuda").to(dtype)


def _tensors(case, seed):
    """q, k, v, dout ~ N(0, 1), in the case's type."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    B, H, Hkv, T, dt = case["B"], case["H"], case["Hkv"], case["T"], DTYPES[case["dtype"]]
    return [_normal((B, h, T, D), dt, gen) for h in (H, Hkv, Hkv, H)]


def _alphas(case):
    if case["kind"] == "stack":
        return [float(a) for a in fa.alpha_schedule("linear", case["layers"])]
    return [case["alpha"]]


def prepare(case, seed):
    q, k, v, g = _tensors(case, seed)
    f = fa.base(case["base"], RUNGS[case["base"]])
    s = dict(case=case, q=q, k=k, v=v, f=f)
    if case["kind"] == "stack":
        s["layers"] = [fa.FibAttention(W=case["W"], offsets=f, theta=fa.theta_of_alpha(a), learned=False)
                       for a in _alphas(case)]
    elif case["kind"] == "autograd":
        s["layer"] = fa.FibAttention(W=case["W"], offsets=f, theta=fa.theta_of_alpha(case["alpha"])).cuda()
        s["g"] = g
        for t in (q, k, v):
            t.requires_grad_(True)
    elif case["kind"] == "train":
        B, H, Hkv, T, W, dt = case["B"], case["H"], case["Hkv"], case["T"], case["W"], DTYPES[case["dtype"]]
        # residuals exist for bf16 and windows up to 16 (see fibattn.h)
        res = fa.residuals_like(q, W, len(f)) if dt == torch.bfloat16 and W <= 16 else None
        s["g"] = g
        s["fwd"] = dict(out=torch.empty_like(q), lse=torch.empty((B, H, T), dtype=torch.float32, device="cuda"),
                        rotated_k=fa.rotated_k_like(k), residuals=res,
                        workspace=torch.empty(max(256, fa.fwd_workspace_bytes(B, H, T, W, len(f), dt, Hkv=Hkv)),
                                              dtype=torch.uint8, device="cuda"))
        s["bwd"] = dict(dq=torch.empty_like(q), dk=torch.empty_like(k), dv=torch.empty_like(v),
                        rotated_k=s["fwd"]["rotated_k"], residuals=res, rung_grads=case["rung_grads"],
                        workspace=torch.empty(fa.bwd_workspace_bytes(B, H, T, W, len(f), dt, Hkv=Hkv),
                                              dtype=torch.uint8, device="cuda"))
    return s


def run(state):
    case, q, k, v = state["case"], state["q"], state["k"], state["v"]
    if case["kind"] == "stack":
        with torch.no_grad():
            return fa.attention_stack(q, state["layers"])
    if case["kind"] == "autograd":
        out = state["layer"](q, k, v)
        grads = torch.autograd.grad(out, (q, k, v, state["layer"].theta), state["g"])
        return (out.detach(),) + grads
    if case["kind"] == "fwd":
        return fa.fwd(q, k, v, case["alpha"], state["f"], case["W"])
    out, lse = fa.fwd(q, k, v, case["alpha"], state["f"], case["W"], **state["fwd"])
    grads = fa.bwd(q, k, v, lse, state["g"], case["alpha"], state["f"], case["W"], out=out, **state["bwd"])
    return (out, lse) + tuple(x for x in grads if x is not None)


def _base64(case):
    n = RUNGS[case["base"]]
    if case["base"] == "pow2":
        return torch.tensor([float(2 ** i) for i in range(n)], dtype=torch.float64)
    f = [1.0, 2.0]
    while len(f) < n:
        f.append(f[-1] + f[-2])
    return torch.tensor(f, dtype=torch.float64)


def work(case):
    """Each input read and each output written once; two FLOPs per multiply-add of the scores and values (forward) and
    of dP, dQ, dK and dV (backward) over the attended rows (a rung reads two), 64 wide."""
    B, H, Hkv, T, W = (case[x] for x in ("B", "H", "Hkv", "T", "W"))
    es = 4 if case["dtype"] == "fp32" else 2
    nq, nk = B * H * T, B * Hkv * T
    total_bytes = total_flops = 0
    for a in _alphas(case):
        rows = sum(T - min(t, T) for t in range(W + 1))
        for f in _base64(case).tolist():
            d = float(torch.tensor(a, dtype=torch.float32) * f)
            if W < d <= T - 1:
                rows += 2 * (T - math.ceil(d))
        fwd = 4 * D * rows * B * H
        if case["kind"] == "stack":
            total_bytes += 2 * nq * D * es
            total_flops += fwd
        elif case["kind"] == "fwd":
            total_bytes += (2 * nq + 2 * nk) * D * es + 4 * nq
            total_flops += fwd
        else:
            total_bytes += (4 * nq + 4 * nk) * D * es + (4 * nq if case["kind"] == "train" else 0)
            total_flops += 3 * fwd
    return {"bytes": total_bytes, "flops": total_flops}


def _rope64(x):
    """Rotate-half RoPE at positions 0..T-1, base 1e4, in 64 bits."""
    T = x.shape[-2]
    ang = torch.arange(T, dtype=torch.float64, device=x.device)[:, None] * \
        1e4 ** (-2.0 * torch.arange(D // 2, dtype=torch.float64, device=x.device) / D)
    a, b = x[..., :D // 2], x[..., D // 2:]
    return torch.cat((a * ang.cos() - b * ang.sin(), b * ang.cos() + a * ang.sin()), dim=-1)


def _attend64(q, k, v, d, W):
    """One batch entry: q [H,T,64], k, v [Hkv,T,64], rung distances d [K], all fp64: (out, lse)."""
    H, T, _ = q.shape
    G = H // k.shape[0]
    q, k = _rope64(q).reshape(-1, G, T, D), _rope64(k)
    i = torch.arange(T, device=q.device)

    def rows(x, dist):                            # row i - dist, a zero row before position 0
        j = i - dist
        return torch.where((j >= 0)[:, None], x[:, j.clamp(min=0)], torch.zeros((), dtype=x.dtype, device=x.device))

    keys, vals, ok = [], [], []
    for t in range(W + 1):
        keys.append(rows(k, t))
        vals.append(rows(v, t))
        ok.append(i >= t)
    for n in range(len(d)):
        dn = float(d[n].detach())
        if dn <= W or dn > T - 1:
            continue
        s0 = math.floor(dn)
        w = d[n] - s0
        keys.append((1 - w) * rows(k, s0) + w * rows(k, s0 + 1))
        vals.append((1 - w) * rows(v, s0) + w * rows(v, s0 + 1))
        ok.append(i >= dn)
    s = torch.stack([(q * x[:, None]).sum(-1) for x in keys], dim=-1) / math.sqrt(D)
    s = s.masked_fill(~torch.stack(ok, dim=-1), -math.inf)
    p = torch.softmax(s, dim=-1)
    out = sum(p[..., n, None] * x[:, None] for n, x in enumerate(vals))
    return out.reshape(H, T, D), torch.logsumexp(s, dim=-1).reshape(H, T)


def exact(case, seed):
    q, k, v, g = (x.double() for x in _tensors(case, seed))
    f = _base64(case).to(q.device)
    W = case["W"]

    def distances(alpha):                         # fl32(alpha f), as a function of alpha
        d = alpha * f
        rounded = (f.float() * torch.tensor(float(alpha), dtype=torch.float32, device=f.device)).double()
        return d + (rounded - d).detach()

    if case["kind"] == "stack":
        x = q
        for a in _alphas(case):
            # the module keeps theta, and alpha comes back from it
            th = torch.tensor(float(torch.tensor(_theta64(a), dtype=torch.float32)), dtype=torch.float64)
            d = distances(torch.tensor(float((0.5 + torch.sigmoid(th)).float()), dtype=torch.float64, device=f.device))
            x = torch.stack([_attend64(x[b], x[b], x[b], d, W)[0] for b in range(case["B"])])
        return x
    if case["kind"] == "autograd":
        th = torch.tensor(_theta64(float(torch.tensor(case["alpha"], dtype=torch.float32))), dtype=torch.float32)
        a32 = float((0.5 + torch.sigmoid(th.double())).float())
    else:
        a32 = float(torch.tensor(case["alpha"], dtype=torch.float32))
    alpha = torch.tensor(a32, dtype=torch.float64, device=f.device)
    if case["kind"] == "fwd":
        got = [_attend64(q[b], k[b], v[b], distances(alpha), W) for b in range(case["B"])]
        return torch.stack([x[0] for x in got]), torch.stack([x[1] for x in got])
    outs, lses, dqs, dks, dvs, dd = [], [], [], [], [], 0
    for b in range(case["B"]):
        leaves = [x[b].clone().requires_grad_(True) for x in (q, k, v)] + [distances(alpha).requires_grad_(True)]
        out, lse = _attend64(*leaves, W)
        grads = torch.autograd.grad(out, leaves, g[b], allow_unused=True)
        outs.append(out.detach())
        lses.append(lse.detach())
        for to, x in zip((dqs, dks, dvs), grads):
            to.append(x)
        dd = dd + (grads[3] if grads[3] is not None else torch.zeros_like(f))
    dtheta = (dd * f).sum() * (a32 - 0.5) * (1.5 - a32)
    out, dq, dk, dv = (torch.stack(x) for x in (outs, dqs, dks, dvs))
    if case["kind"] == "autograd":
        return out, dq, dk, dv, dtheta
    return (out, torch.stack(lses), dq, dk, dv) + ((dtheta.reshape(1), dd) if case["rung_grads"] else ())


def _theta64(alpha):
    """theta with 0.5 + sigmoid(theta) = alpha, the ends of the range at -/+ 30."""
    return -30.0 if alpha <= 0.5 else 30.0 if alpha >= 1.5 else math.log((alpha - 0.5) / (1.5 - alpha))
