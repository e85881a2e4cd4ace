"""The sums of dW over its partial slots: few blocks take 16 loads per thread, many take 8, in the
same order.  Ten heads at once (many blocks) give the bits of each head alone (few blocks), for
slot counts around the loads in flight of a block's four lanes (32 and 64)."""
import pytest
import torch

from paper_2606_27748_gb300 import build, flexattn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 5, 16, 17, 37])
@pytest.mark.parametrize("what,nonstat", [("bwd", False), ("bwd", True), ("awd", True)])
def test_dw_of_many_heads_is_that_of_each(what, nonstat, B):
    build.build()
    torch.manual_seed(B)
    H, N, d, M = 10, 70, 64, 64
    q, k, v, g = ((0.35 * torch.randn(B, H, N, d, device="cuda")).to(torch.bfloat16) for _ in range(4))
    W1 = torch.randn(H, M, d, device="cuda")
    W2 = torch.randn(H, M, d, device="cuda") if nonstat else None

    def run(hs):
        a, b, c, e = (x[:, hs].contiguous() for x in (q, k, v, g))
        w1, w2 = W1[hs].contiguous(), None if W2 is None else W2[hs].contiguous()
        if what == "awd":
            return flexattn.awd_loss_bwd(a, b, w1, w2)[1:3]
        out, den = flexattn.linattn_fwd(a, b, c, w1, w2, False)
        return flexattn.linattn_bwd(a, b, c, w1, w2, False, out, den, e)[3:5]

    every = run(slice(0, H))
    torch.cuda.synchronize()
    for h in (0, 4, 9):
        for x, y in zip(every, run(slice(h, h + 1))):
            assert (x is None) == (y is None)
            assert x is None or torch.equal(x[h], y[0])
