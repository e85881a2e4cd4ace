"""Non-finite values in the fp32 causal kernels stay where the mask lets them go: rows that do
not see a NaN or infinite value, or a key whose weight overflows, have the bits they have
without it (padding on the right may be anything)."""
import pytest
import torch

from paper_2606_27748_gb300 import build, flexattn

pytestmark = pytest.mark.gpu

# (dtype, B, H, N, d, M): one CTA and several ranges a sequence, one and two frequency groups, the
# plans of short sequences and of many small ones
SHAPES = [("f32", 1, 2, 50, 32, 32), ("f32", 1, 2, 20, 32, 100), ("f32", 39, 8, 70, 16, 16), ("f32", 1, 2, 300, 32, 16), ("f32", 1, 1, 200, 64, 64),
          ("f32", 1, 1, 90, 128, 24), ("bf16", 1, 2, 150, 32, 16)]


def inputs(dtype, B, H, N, d, M, nonstat):
    build.build()
    torch.manual_seed(N + d)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    x = {n: (d ** -0.25 * torch.randn(B, H, N, d, device="cuda")).to(dt) for n in ("q", "k", "v", "g")}
    W1 = torch.randn(H, M, d, device="cuda") * d ** -0.5
    W2 = torch.randn(H, M, d, device="cuda") * d ** -0.5 if nonstat else None
    return x, W1, W2, torch.full((H,), 2.5, device="cuda")


def step(x, W1, W2, tau):
    out, den = flexattn.linattn_fwd(x["q"], x["k"], x["v"], W1, W2, True, tau=tau)
    dq, dk, dv = flexattn.linattn_bwd(x["q"], x["k"], x["v"], W1, W2, True, out, den, x["g"],
                                      tau=tau)[:3]
    return out, den, dq, dk, dv


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("what", ["v nan", "v inf", "k nan", "weight"])
@pytest.mark.parametrize("nonstat", [False, True])
def test_rows_before_a_non_finite_value(shape, what, nonstat):
    x, W1, W2, tau = inputs(*shape, nonstat)
    N, d = shape[3], shape[4]
    tau = tau if what == "weight" else None
    want = step(x, W1, W2, tau)
    for at in sorted({1, 2, 7, N // 2 + 1, N - 1} | {t for t in (63, 64, 66) if t < N}):
        y = {n: t.clone() for n, t in x.items()}
        if what == "weight":  # |k|^2 exp(-tau) > 88: the key's weight is infinite
            y["k"][:, :, at:] = 1.2 * (88 * 12.2 / d) ** 0.5
        else:
            y[what[0]][:, :, at:] = float(what[2:])
        got = step(y, W1, W2, tau)
        for name, a, b in zip(("out", "den", "dq"), got, want):
            assert torch.equal(a[:, :, :at], b[:, :, :at]), f"{name} before {at}"
        assert not torch.isfinite(got[0][:, :, at:]).any(), "the planted value has to show"


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("nonstat", [False, True])
def test_keys_after_a_non_finite_query(shape, nonstat):
    """dk and dv of a key take part only in the rows from its own on."""
    x, W1, W2, _ = inputs(*shape, nonstat)
    N = shape[3]
    want = step(x, W1, W2, None)
    for at in sorted({0, 1, 6, N // 2, N - 2} | {t for t in (62, 63, 65) if t < N - 1}):
        y = {n: t.clone() for n, t in x.items()}
        y["q"][:, :, :at + 1] = float("nan")
        got = step(y, W1, W2, None)
        for name, a, b in zip(("dk", "dv"), got[3:], want[3:]):
            assert torch.equal(a[:, :, at + 1:], b[:, :, at + 1:]), f"{name} after {at}"
        assert not torch.isfinite(got[0][:, :, :at + 1]).any(), "the planted value has to show"
