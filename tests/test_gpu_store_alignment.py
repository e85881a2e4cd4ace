"""Result tensors that begin 16 but not 32 bytes into an allocation (the alignment that the entry
points ask for is 16): the same bits as aligned ones, and nothing written around them."""
import pytest
import torch

from paper_2606_27748_gb300 import build, flexattn

pytestmark = pytest.mark.gpu


def _at(shape, offset):
    n = 1
    for x in shape:
        n *= x
    buf = torch.full((n + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    t = buf[offset:offset + n].view(*shape)
    assert t.data_ptr() % 32 == 2 * offset % 32
    return buf, t


@pytest.mark.parametrize("causal,nonstat,M,N", [
    (True, True, 128, 257), (True, False, 64, 130), (False, True, 64, 129), (True, False, 128, 1),
    (False, False, 128, 700)])
def test_results_at_16_byte_offsets(causal, nonstat, M, N):
    build.build()
    torch.manual_seed(N)
    B, H, d = 2, 2, 64
    q, k, v, g = ((0.35 * torch.randn(B, H, N, d, device="cuda")).to(torch.bfloat16) for _ in range(4))
    W1 = torch.randn(H, M, d, device="cuda")
    W2 = torch.randn(H, M, d, device="cuda") if nonstat else None

    def run(offset):
        bufs = [_at((B, H, N, d), offset) for _ in range(4)] + [_at((B, H, N, 2 * M), offset)]
        (out, dq, dk, dv, phi) = (t for _, t in bufs)
        _, den = flexattn.linattn_fwd(q, k, v, W1, W2, causal, out=out)
        flexattn.linattn_bwd(q, k, v, W1, W2, causal, out, den, g, dq=dq, dk=dk, dv=dv)
        flexattn.featmap(k, W1, W2, phi=phi)
        torch.cuda.synchronize()
        for buf, t in bufs:
            assert bool((buf[:offset] == 7).all()) and bool((buf[offset + t.numel():] == 7).all())
        return [t for _, t in bufs]

    for a, b in zip(run(0), run(8)):
        assert torch.equal(a, b)
