"""The distillation loss of one sequence has fewer blocks than the GPU has SMs (128 of 152), that of
two has two an SM.  Launched early, the blocks of one must not pair up on some SMs while others
idle: then one sequence takes as long as two (measured 0.98 of it; 0.65 with one block an SM)."""
import pytest
import torch

from paper_2606_27748_gb300 import build, flexattn

pytestmark = pytest.mark.gpu


def test_one_sequence_is_faster_than_two():
    build.build()
    torch.manual_seed(3)
    N, d, M = 16384, 64, 64
    q, k = ((0.35 * torch.randn(1, 2, N, d, device="cuda")).to(torch.bfloat16) for _ in range(2))
    W1, W2 = (torch.randn(2, M, d, device="cuda") * d ** -0.5 for _ in range(2))

    def measure(H):
        a, b, w1, w2 = q[:, :H].contiguous(), k[:, :H].contiguous(), W1[:H].contiguous(), W2[:H].contiguous()
        ws = flexattn.awd_workspace(flexattn.shape_of(a, w1))
        loss, best = None, float("inf")
        for _ in range(20):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(5):
                loss = flexattn.awd_loss(a, b, w1, w2, ws=ws)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        flexattn.check_status(ws)
        return best, loss

    one, l1 = measure(1)
    two, l2 = measure(2)
    assert torch.equal(l1[:, :1], l2[:, :1])
    assert one < 0.85 * two, (one, two)
