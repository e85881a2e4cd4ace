"""The non-causal tensor-core backward with several chunks per CTA: the batch is large enough
that every sequence (or, with two frequency groups, each group of it) is one CTA's, so buffers,
row sums and sums over chunks are used from one chunk to the next.  Two heads of the batch
against the oracle, and bit-exact repeats of queued calls."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_27748_gb300 import flexattn, workloads
from parity import BF16_REL_L2, assert_close, rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu

H = 8
HEADS = [0, 5]


def check(variant, M, N, tau):
    from paper_2606_27748_gb300 import build
    build.build()
    B = 38 * 64 // M  # 304 (sequence, group) pairs: twice the 152 SMs, no split over CTAs
    w = workloads.Workload("w", variant, False, "bf16", B, H, N, 64, M, 64 ** -0.25, "normal", 41,
                           backward=True)
    ins = workloads.make_inputs(w)
    t64 = workloads.draw_tau(w).astype(np.float64) if tau else None
    q, k, v, dO = (to_dev(ins[n], "bf16") for n in ("q", "k", "v", "dO"))
    W1, W2, tg = (to_dev(x, "f32") for x in (ins["W1"], ins["W2"], t64))
    out, den = flexattn.linattn_fwd(q, k, v, W1, W2, False, tau=tg)
    ws = flexattn.workspace(flexattn.shape_of(q, W1), False, True)
    runs = [flexattn.linattn_bwd(q, k, v, W1, W2, False, out, den, dO, ws=ws, tau=tg)
            for _ in range(4)]
    flexattn.check_status(ws)
    for r in runs[1:]:
        assert all(x is y or torch.equal(x, y) for x, y in zip(r, runs[0])), "not repeatable"
    pick = {n: np.ascontiguousarray(ins[n][:, HEADS]) for n in ("q", "k", "v", "dO")}
    f1, f2, th = (None if x is None else x[HEADS] for x in (ins["W1"], ins["W2"], t64))
    ref = oracle.bwd(pick["q"], pick["k"], pick["v"], f1, f2, False, pick["dO"], tau=th)
    for name, x, r in zip(("dq", "dk", "dv", "dW1", "dW2", "dtau"), runs[0], ref):
        if r is None:
            assert x is None
            continue
        x = to_host(x[:, HEADS] if name in ("dq", "dk", "dv") else x[HEADS])
        if name == "dtau":
            assert rel_l2(x, r) <= BF16_REL_L2, name
        else:
            scale = float(np.sqrt(np.mean(r * r))) if name.startswith("dW") else 1.0
            assert_close(x, r, "bf16", name, max_abs_scale=scale)


@pytest.mark.parametrize("variant,N,tau", [
    ("s", 513, True), ("s", 700, False), ("n", 640, True), ("n", 770, True), ("n", 600, False)])
def test_chunks_of_one_cta(variant, N, tau):
    check(variant, 64, N, tau)


@pytest.mark.parametrize("variant,N,tau", [
    ("s", 513, True), ("s", 700, False), ("n", 640, True), ("n", 770, False)])
def test_chunks_of_one_cluster(variant, N, tau):
    """M = 128: the two CTAs of a sequence exchange rows chunk after chunk."""
    check(variant, 128, N, tau)
