"""The work that a program of this library has it do, for measuring its speed and accuracy.

Each case is one pass through the public entry points of the binding: a forward, a training
step (forward and backward), a decode step, or a distillation step.  Shapes are those of
the repository's workloads (`paper_2606_27748_gb300/workloads.py`), of the settings they
stand for (language modelling, long-sequence classification, distillation) and generic ones
around them: head sizes and frequency counts off the tuned d = 64, ragged lengths, fp32.

Inputs follow the workloads' distributions (q, k ~ N(0, 1) d^-1/4, v, dO ~ N(0, 1),
frequencies ~ N(0, 1/d), tau = ln(2 sqrt d) and a quarter to either side), drawn on the GPU.
"""
import math

import torch

from paper_2606_27748_gb300 import flexattn


def _case(name, call, variant, causal, dtype, B, H, N, d, M, tau=False):
    return {"name": name, "call": call, "variant": variant, "causal": causal, "dtype": dtype,
            "B": B, "H": H, "N": N, "d": d, "M": M, "tau": tau}


def listed():
    return [
        # one short fp32 sequence: the smallest call, where latency is all (the first workload)
        _case("fwd_f32_single", "fwd", "s", False, "f32", 1, 1, 256, 32, 32),
        # an encoder batch in bf16 off the tuned head size: image classification with 16
        # frequencies and 1024 pixels
        _case("fwd_bf16_d32", "fwd", "n", False, "bf16", 32, 4, 1024, 32, 16),
        # language-model prefill, stationary kernel
        _case("fwd_s_causal", "fwd", "s", True, "bf16", 8, 12, 4096, 64, 64),
        # the bench's headline: long-context prefill, nonstationary kernel, 128 frequencies
        _case("fwd_n_causal", "fwd", "n", True, "bf16", 4, 16, 16384, 64, 128),
        # the largest forward: long-sequence classification
        _case("fwd_n_noncausal", "fwd", "n", False, "bf16", 8, 8, 65536, 64, 64),
        # language-model training step
        _case("train_s_causal", "train", "s", True, "bf16", 8, 12, 8192, 64, 128),
        # language-model training step with every learnable part, ragged length, small batch
        _case("train_n_causal_tau", "train", "n", True, "bf16", 2, 8, 2000, 64, 64, True),
        # training step on documents of 4000 tokens (non-causal encoder)
        _case("train_n_noncausal", "train", "n", False, "bf16", 32, 8, 4000, 64, 64),
        # the same kind of training step in fp32, a small ragged batch
        _case("train_f32", "train", "n", False, "f32", 4, 4, 1000, 64, 64, True),
        # one token for each of a few streams: interactive decoding
        _case("decode_small", "decode", "n", True, "bf16", 4, 16, 1, 64, 128),
        # one token for each of a full serving batch
        _case("decode_serving", "decode", "n", True, "bf16", 256, 16, 1, 64, 128),
        # one step of distilling softmax attention into the kernel
        _case("distill_train", "distill", "n", False, "bf16", 32, 8, 512, 64, 64),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["fwd", "fwd", "fwd", "train", "train", "decode", "decode", "distill"])
    c = {"call": call, "variant": rng.choice("sn"), "causal": rng.random() < 0.5, "dtype": "bf16",
         "B": 1, "H": 1, "N": 1, "d": 64, "M": rng.choice([64, 128]), "tau": rng.random() < 0.25}
    if call == "distill":
        c.update(B=_log_int(rng, 1, 32), H=rng.choice([4, 8, 12]), N=_log_int(rng, 32, 512),
                 M=64)
        return c
    if call == "decode":
        c.update(causal=True, dtype=rng.choice(["bf16", "bf16", "f32"]), B=_log_int(rng, 1, 200),
                 H=rng.choice([4, 8, 12, 16]))
        return c
    if rng.random() < 0.35:  # fp32 storage, or bf16 off the tuned head size
        c["dtype"] = rng.choice(["f32", "f32", "bf16"])
        c["d"], c["M"] = rng.choice([(16, 16), (32, 16), (32, 32), (48, 40), (64, 16), (64, 64),
                                     (128, 32)])
        if c["dtype"] == "bf16" and c["d"] == 64:
            c["M"] = 16
        c.update(B=_log_int(rng, 1, 16), H=rng.choice([1, 2, 4, 8]),
                 N=_log_int(rng, 33, 4096 if call == "fwd" else 1000))
        return c
    c.update(B=_log_int(rng, 1, 16), H=rng.choice([4, 8, 12, 16]))
    most = 2 ** 22 if call == "fwd" else 2 ** 19
    c["N"] = _log_int(rng, 33, max(64, min(65536 if call == "fwd" else 16384,
                                           most // (c["B"] * c["H"]))))
    return c


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _inputs(c, seed):
    """The tensors of one pass, from the seed alone (also what `exact` starts from)."""
    g = _generator(seed)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    B, H, N, d, M = (c[n] for n in ("B", "H", "N", "d", "M"))
    rows = (B, H, d) if c["call"] == "decode" else (B, H, N, d)

    def normal(shape, scale, dtype):
        return torch.randn(shape, generator=g, device="cuda").mul_(scale).to(dtype)

    t = {"q": normal(rows, d ** -0.25, dt), "k": normal(rows, d ** -0.25, dt)}
    t["W1"] = normal((H, M, d), d ** -0.5, torch.float32)
    t["W2"] = normal((H, M, d), d ** -0.5, torch.float32) if c["variant"] == "n" else None
    t["tau"] = None
    if c["tau"]:
        spread = 0.25 * ((torch.arange(H, device="cuda") % 3).float() - 1)
        t["tau"] = math.log(2 * math.sqrt(d)) + spread
    if c["call"] == "distill":  # the gradient of the batch's mean loss
        t["dloss"] = torch.full((B, H), 1.0 / (B * H), device="cuda")
        return t
    t["v"] = normal(rows, 1.0, dt)
    if c["call"] == "train":
        t["dO"] = normal(rows, 1.0, dt)
    if c["call"] == "decode":  # the running sums of 64 earlier tokens
        S, z = flexattn.decode_state(B, H, M, d)
        for b in range(0, B, 32):
            n = min(32, B - b)
            phi = _phi(normal((n, H, 64, d), d ** -0.25, torch.float32), t["W1"], t["W2"])
            S[b:b + n] = phi.mT @ normal((n, H, 64, d), 1.0, torch.float32)
            z[b:b + n] = phi.sum(-2)
        t["S"], t["z"] = S, z
    return t


def _phi(x, W1, W2):
    """Features [.., N, 2M] of rows x [.., N, d] in x's type, scaled by M^-1/2."""
    W1 = W1.to(x.dtype)
    if W2 is None:
        u = x @ W1.mT
        f = torch.cat([u.cos(), u.sin()], -1)
    else:
        W2 = W2.to(x.dtype)
        u, w = x @ ((W1 + W2) / 2).mT, (x @ ((W1 - W2) / 2).mT).cos()
        f = torch.cat([u.cos() * w, u.sin() * w], -1)
    return f * W1.shape[-2] ** -0.5


def prepare(case, seed):
    """Inputs, and the workspaces a program allocates once for its shapes."""
    s = _inputs(case, seed)
    s["case"] = case
    if case["call"] == "decode":
        s["ws"] = flexattn.decode_workspace(case["B"], case["H"], case["M"], case["d"])
        s["out"] = torch.empty_like(s["q"])
        s["den"] = torch.empty(case["B"], case["H"], device="cuda")
        return s
    shape = flexattn.shape_of(s["q"], s["W1"])
    if case["call"] == "distill":
        s["ws"] = flexattn.awd_bwd_workspace(shape)
        return s
    s["ws"] = flexattn.workspace(shape, case["causal"], False)
    if case["call"] == "train":
        s["ws_bwd"] = flexattn.workspace(shape, case["causal"], True)
    return s


def run(s):
    c = s["case"]
    if c["call"] == "decode":
        flexattn.linattn_decode(s["q"], s["k"], s["v"], s["W1"], s["W2"], s["S"], s["z"],
                                out=s["out"], den=s["den"], ws=s["ws"], tau=s["tau"])
        return {"out": s["out"], "den": s["den"], "S": s["S"], "z": s["z"]}
    if c["call"] == "distill":
        loss, dW1, dW2, dtau = flexattn.awd_loss_bwd(
            s["q"], s["k"], s["W1"], s["W2"], c["causal"], tau=s["tau"], dloss=s["dloss"],
            ws=s["ws"])
        return {"loss": loss, "dW1": dW1, "dW2": dW2, "dtau": dtau}
    out, den = flexattn.linattn_fwd(s["q"], s["k"], s["v"], s["W1"], s["W2"], c["causal"],
                                    ws=s["ws"], tau=s["tau"])
    r = {"out": out, "den": den}
    if c["call"] == "train":
        g = flexattn.linattn_bwd(s["q"], s["k"], s["v"], s["W1"], s["W2"], c["causal"], out, den,
                                 s["dO"], ws=s["ws_bwd"], tau=s["tau"])
        r.update(zip(("dq", "dk", "dv", "dW1", "dW2", "dtau"), g))
    return r


def work(case):
    """Bytes: every input read once, every output written once.  Flops: the projections,
    the running sums and their reads (and their gradients); with N x N pairs only where the
    loss itself is over pairs."""
    c = case
    d, M, e = c["d"], c["M"], 4 if c["dtype"] == "f32" else 2
    Mc = 2 * M if c["variant"] == "n" else M
    rows = c["B"] * c["H"] * c["N"]
    freq = c["H"] * Mc * d * 4
    proj, state = 2 * Mc * d, 2 * 2 * M * d  # flops a row: one projection, one sum over state
    if c["call"] == "decode":
        return {"bytes": rows * (2 * 2 * M * (d + 1) * 4 + 4 * d * e + 4) + freq,
                "flops": rows * (2 * proj + 2 * state)}
    if c["call"] == "distill":
        pairs = c["B"] * c["H"] * c["N"] ** 2 * (0.5 if c["causal"] else 1.0)
        return {"bytes": rows * 2 * d * e + 2 * freq,
                "flops": pairs * (2 * d + 3 * 2 * 2 * M) + rows * 6 * proj}
    w = {"bytes": rows * (4 * d * e + 4) + freq, "flops": rows * (2 * proj + 2 * state)}
    if c["call"] == "train":
        w["bytes"] += rows * (8 * d * e + 4) + 2 * freq
        w["flops"] += rows * (4 * proj + 5 * state)
    return w


def tolerance(case):
    """About four times the largest error against `exact` over a call's outputs (measured:
    fp32 up to 1.1e-6, and more for dtau, a sum that cancels; bf16 forward and decode 1.9e-3,
    gradients up to 6e-3 (dq), the distillation's gradients 6e-4, and more with tau)."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    return {"rel": {"fwd": 8e-3, "decode": 8e-3, "train": 2.5e-2, "distill": 5e-3}[case["call"]]}


def _attend(q, k, v, W1, W2, tau, causal):
    """(out, den) of one batch entry [H, N, d] in 64 bits: the linear form, chunk by chunk."""
    pq, pk = _phi(q, W1, W2), _phi(k, W1, W2)
    if tau is not None:
        pk = pk * torch.exp(k.square().sum(-1, keepdim=True) * torch.exp(-tau)[:, None, None])
    v1 = torch.cat([v, torch.ones_like(v[..., :1])], -1)
    if not causal:
        o = pq @ (pk.mT @ v1)
    else:
        H, N, _ = q.shape
        C = 128
        pad = -N % C
        pq, pk, v1 = (torch.nn.functional.pad(x, (0, 0, 0, pad)).unflatten(1, (-1, C))
                      for x in (pq, pk, v1))
        sums = pk.mT @ v1
        before = torch.cat([torch.zeros_like(sums[:, :1]), sums.cumsum(1)[:, :-1]], 1)
        o = (torch.tril(pq @ pk.mT) @ v1 + pq @ before).flatten(1, 2)[:, :N]
    return o[..., :-1] / o[..., -1:], o[..., -1]


def _distill_loss(q, k, W1, W2, tau, causal):
    """Loss [H] of one batch entry, over the explicit pairs."""
    N, d = q.shape[-2:]
    pk = _phi(k, W1, W2)
    if tau is not None:
        pk = pk * torch.exp(k.square().sum(-1, keepdim=True) * torch.exp(-tau)[:, None, None])
    s, a = q @ k.mT / math.sqrt(d), _phi(q, W1, W2) @ pk.mT
    if causal:
        seen = torch.ones(N, N, dtype=torch.bool, device=q.device).tril()
        s, a = s.masked_fill(~seen, -math.inf), a * seen
    p = torch.softmax(s, -1)
    r = a / a.sum(-1, keepdim=True)
    log_r = torch.where(r > 0, torch.where(r > 0, r, 1.0).log(), math.log(1e-6))
    return -(p * log_r).sum((-1, -2)) / N


def exact(case, seed):
    c = case
    t = {n: x.double() if x is not None else None for n, x in _inputs(c, seed).items()}
    W = {n: t[n] for n in ("W1", "W2", "tau")}
    if c["call"] == "decode":
        pq, pk = (_phi(t[n].unsqueeze(-2), W["W1"], W["W2"]).squeeze(-2) for n in "qk")
        if c["tau"]:
            pk = pk * torch.exp(t["k"].square().sum(-1, keepdim=True) * torch.exp(-W["tau"])[:, None])
        S = t["S"] + pk.unsqueeze(-1) * t["v"].unsqueeze(-2)
        z = t["z"] + pk
        den = (pq * z).sum(-1)
        out = (pq.unsqueeze(-2) @ S).squeeze(-2) / den.unsqueeze(-1)
        return {"out": out, "den": den, "S": S, "z": z}

    learn = c["call"] != "fwd"
    params = [x.requires_grad_(learn) for x in W.values() if x is not None]
    got = {n: [] for n in ("loss", "out", "den", "dq", "dk", "dv")}
    total = None
    for b in range(c["B"]):
        if c["call"] == "distill":
            loss = _distill_loss(t["q"][b], t["k"][b], causal=c["causal"], **W)
            g = torch.autograd.grad((loss * t["dloss"][b]).sum(), params)
            got["loss"].append(loss.detach())
        else:
            x = [t[n][b].requires_grad_(learn) for n in "qkv"]
            out, den = _attend(*x, causal=c["causal"], **W)
            got["out"].append(out.detach())
            got["den"].append(den.detach())
            if not learn:
                continue
            g = torch.autograd.grad((out * t["dO"][b]).sum(), x + params)
            for n, gx in zip(("dq", "dk", "dv"), g):
                got[n].append(gx)
            g = g[3:]
        total = g if total is None else [a + x for a, x in zip(total, g)]
    r = {n: torch.stack(x) for n, x in got.items() if x}
    if learn:
        total = iter(total)
        for n, x in W.items():
            r["d" + n] = next(total) if x is not None else None
    return r
