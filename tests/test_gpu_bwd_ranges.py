"""The causal tensor-core backward of small batches, whose sequences are cut into ranges of
128-token chunks (8 chunks and more): against the oracle at edges of the cut (range sizes
that do and do not divide, a ragged last chunk, both group counts), bit-exact repeatability,
and the same call with a workspace that only holds the uncut form."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_27748_gb300 import flexattn, workloads
from parity import BF16_REL_L2, assert_close, rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,M,N,tau", [
    ("s", 64, 897, True), ("s", 128, 1024, False), ("s", 128, 1300, True), ("n", 64, 1023, False),
    ("n", 64, 2500, True), ("n", 128, 1153, False), ("n", 128, 1700, True)])
def test_causal_ranges_match_oracle(variant, M, N, tau):
    from paper_2606_27748_gb300 import build
    build.build()
    w = workloads.Workload("w", variant, True, "bf16", 2, 2, N, 64, M, 64 ** -0.25, "normal", 31,
                           backward=True)
    ins = workloads.make_inputs(w)
    t64 = workloads.draw_tau(w).astype(np.float64) if tau else None
    q, k, v, dO = (to_dev(ins[n], "bf16") for n in ("q", "k", "v", "dO"))
    W1, W2, tg = (to_dev(x, "f32") for x in (ins["W1"], ins["W2"], t64))
    out, den = flexattn.linattn_fwd(q, k, v, W1, W2, True, tau=tg)
    ref = oracle.bwd(ins["q"], ins["k"], ins["v"], ins["W1"], ins["W2"], True, ins["dO"], tau=t64)

    def run(ws):
        n0 = flexattn.kernel_launches()
        g = flexattn.linattn_bwd(q, k, v, W1, W2, True, out, den, dO, ws=ws, tau=tg)
        flexattn.check_status(ws)
        return flexattn.kernel_launches() - n0, [None if x is None else to_host(x) for x in g]

    full = flexattn.workspace(flexattn.shape_of(q, W1), True, True)
    ranges, first = run(full)
    assert ranges == (5 if tau else 4)  # partial states, their scan, the gradient, dW (+ weights)
    _, again = run(full)
    # the least workspace: shrink until refused
    lo, hi = 256, full.numel()
    while hi - lo > 256:
        mid = (lo + hi) // 512 * 256
        try:
            run(full[:mid])
            hi = mid
        except flexattn.FlexError as e:
            assert e.status == flexattn.FLEX_EWORKSPACE
            lo = mid
    uncut, small = run(full[:hi])
    assert uncut == ranges - 2
    for name, x, y, z, r in zip(("dq", "dk", "dv", "dW1", "dW2", "dtau"), first, again, small, ref):
        if r is None:
            assert x is None
            continue
        assert np.array_equal(x, y), f"{name}: not repeatable"
        if name == "dtau":
            assert max(rel_l2(x, r), rel_l2(z, r)) <= BF16_REL_L2, name
            continue
        scale = float(np.sqrt(np.mean(r * r))) if name.startswith("dW") else 1.0
        assert_close(x, r, "bf16", name, max_abs_scale=scale)
        assert_close(z, r, "bf16", f"{name} (least workspace)", max_abs_scale=scale)
