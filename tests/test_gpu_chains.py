"""Calls of several kernels whose launches overlap (each waits for its predecessor inside the
kernel): calls on alternating inputs, queued without a pause in one workspace and one set of
outputs, give the bits that each call gives alone, and so does the same queue as a CUDA graph,
replayed on new contents of its inputs.  A kernel that read its predecessor's results too
early would see those of the call before."""
import pytest
import torch

from paper_2606_27748_gb300 import build, flexattn

pytestmark = pytest.mark.gpu

# (what, dtype, causal, nonstationary, tau, N, M): partial states and their totals or scan, the
# gradient and dW; the key weights before each of them; the feature maps, statistics and gradient
# of the distillation loss; the fp32 gradient and its dW sum
CASES = [
    ("fwd", "bf16", True, False, True, 300, 64), ("fwd", "bf16", False, True, True, 1300, 128),
    ("fwd", "bf16", False, False, False, 129, 64), ("bwd", "bf16", True, True, True, 1300, 128),
    ("bwd", "bf16", True, False, False, 200, 64), ("bwd", "bf16", False, True, True, 700, 64),
    ("bwd", "bf16", False, False, False, 129, 128), ("awd", "bf16", True, False, True, 300, 128),
    ("awd", "bf16", False, True, False, 257, 64), ("bwd", "f32", True, True, True, 130, 32),
]


@pytest.mark.parametrize("what,dtype,causal,nonstat,tau,N,M", CASES)
def test_queued_and_captured_calls_repeat_single_ones(what, dtype, causal, nonstat, tau, N, M):
    build.build()
    torch.manual_seed(N + M)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    B, H, d = 2, 3, 64

    def draw():
        x = {n: (0.35 * torch.randn(B, H, N, d, device="cuda")).to(dt) for n in ("q", "k", "v", "g")}
        x["tau"] = torch.rand(H, device="cuda") + 2.0 if tau else None
        return x

    W1 = torch.randn(H, M, d, device="cuda")
    W2 = torch.randn(H, M, d, device="cuda") if nonstat else None
    sets = [draw(), draw()]
    if what == "bwd":
        for x in sets:
            x["out"], x["den"] = flexattn.linattn_fwd(x["q"], x["k"], x["v"], W1, W2, causal,
                                                      tau=x["tau"])
    shape = flexattn.shape_of(sets[0]["q"], W1)
    ws = (flexattn.awd_bwd_workspace(shape) if what == "awd" else
          flexattn.workspace(shape, causal, what == "bwd"))

    def call(x):
        if what == "fwd":
            r = flexattn.linattn_fwd(x["q"], x["k"], x["v"], W1, W2, causal, ws=ws, tau=x["tau"])
        elif what == "bwd":
            r = flexattn.linattn_bwd(x["q"], x["k"], x["v"], W1, W2, causal, x["out"], x["den"],
                                     x["g"], ws=ws, tau=x["tau"])
        else:
            r = flexattn.awd_loss_bwd(x["q"], x["k"], W1, W2, causal, tau=x["tau"], ws=ws,
                                      dloss=dloss)
        return [t for t in r if t is not None]

    dloss = torch.rand(B, H, device="cuda")
    want = []
    for x in sets:
        want.append(call(x))
        torch.cuda.synchronize()
    got = [call(sets[i % 2]) for i in range(12)]  # queued: no wait in between
    flexattn.check_status(ws)
    for i, r in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(r, want[i % 2])), f"queued call {i}"

    x = {n: None if t is None else t.clone() for n, t in sets[0].items()}
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        first, second = call(sets[1]), call(x)
    for i in (1, 0, 1):
        for n, t in x.items():
            if t is not None:
                t.copy_(sets[i][n])
        graph.replay()
        flexattn.check_status(ws)
        assert all(torch.equal(a, b) for a, b in zip(first, want[1])), "captured"
        assert all(torch.equal(a, b) for a, b in zip(second, want[i])), "replayed on new inputs"
