"""The fp32 kernels against the fp64 oracle where their plan changes: chunk and range edges
(chunks of 64 tokens, up to 8 ranges of one sequence), frequency groups of up to 32 with
padding, head sizes up to 128, the reduced chunks of the largest shapes, both storage types,
masks and variants, with and without the norm prefactor."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_27748_gb300 import flexattn, workloads
from parity import BF16_REL_L2, F32_REL_L2, assert_close, rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu

# (variant, causal, dtype, B, H, N, d, M, tau)
CASES = [
    ("s", True, "f32", 1, 1, 1, 32, 32, False), ("n", True, "f32", 1, 2, 64, 64, 64, True),
    ("n", False, "f32", 1, 1, 65, 64, 64, True), ("s", False, "f32", 2, 1, 511, 32, 16, False),
    ("n", True, "f32", 1, 1, 512, 64, 33, True), ("s", True, "f32", 3, 5, 513, 48, 40, True),
    ("n", False, "f32", 1, 3, 300, 4, 3, False), ("s", True, "f32", 1, 2, 200, 12, 7, True),
    ("n", True, "f32", 8, 20, 130, 16, 16, False), ("n", False, "f32", 8, 20, 130, 16, 16, True),
    ("s", True, "f32", 1, 2, 150, 128, 64, True), ("n", False, "f32", 2, 1, 150, 128, 32, False),
    ("n", True, "f32", 1, 2, 100, 64, 100, True), ("s", False, "f32", 1, 1, 90, 88, 169, True),
    ("s", True, "f32", 1, 1, 90, 116, 129, False), ("n", True, "f32", 1, 1, 70, 16, 256, True),
    ("n", True, "bf16", 2, 2, 257, 32, 16, True), ("n", False, "bf16", 4, 3, 1024, 32, 16, False),
    ("s", False, "bf16", 2, 3, 512, 32, 16, True), ("n", False, "f32", 1, 2, 641, 16, 5, True),
    ("s", True, "bf16", 1, 2, 140, 128, 24, True), ("s", False, "bf16", 1, 2, 191, 64, 16, True),
]


def _id(c):
    return "-".join([c[0], "c" if c[1] else "nc", c[2], *map(str, c[3:8]), "tau" if c[8] else "1"])


@pytest.mark.parametrize("c", CASES, ids=_id)
def test_fp32_kernels_match_oracle(c):
    from paper_2606_27748_gb300 import build
    build.build()
    variant, causal, dtype, B, H, N, d, M, tau = c
    w = workloads.Workload("w", variant, causal, dtype, B, H, N, d, M, d ** -0.25 / 2, "normal", 21,
                           backward=True)
    ins = workloads.make_inputs(w)
    t64 = workloads.draw_tau(w).astype(np.float64) if tau else None
    q, k, v, dO = (to_dev(ins[n], dtype) for n in ("q", "k", "v", "dO"))
    W1, W2, tg = (to_dev(x, "f32") for x in (ins["W1"], ins["W2"], t64))
    out, den = flexattn.linattn_fwd(q, k, v, W1, W2, causal, tau=tg)
    ro, rd = oracle.fwd(ins["q"], ins["k"], ins["v"], ins["W1"], ins["W2"], causal, tau=t64)
    assert_close(to_host(out), ro, dtype, "out")
    assert rel_l2(to_host(den), rd) <= F32_REL_L2, "den"  # fp32 for either storage type
    runs = []
    for _ in range(2):
        g = flexattn.linattn_bwd(q, k, v, W1, W2, causal, out, den, dO, tau=tg)
        torch.cuda.synchronize()
        runs.append([None if x is None else to_host(x) for x in g])
    r = oracle.bwd(ins["q"], ins["k"], ins["v"], ins["W1"], ins["W2"], causal, ins["dO"], tau=t64)
    for name, x, y, ref in zip(("dq", "dk", "dv", "dW1", "dW2", "dtau"), *runs, r):
        if ref is None:
            assert x is None
            continue
        assert np.array_equal(x, y), f"{name}: not repeatable"
        scale = 1.0
        if name in ("dW1", "dW2"):
            rms = float(np.sqrt(np.mean(ref * ref)))
            scale = rms if rms > 1e-12 else 1.0
        if name == "dtau":  # a cancelling sum over the keys: held to the storage type's bound
            if N > 1:
                assert rel_l2(x, ref) <= (1e-4 if dtype == "f32" else BF16_REL_L2), name
        else:
            assert_close(x, ref, dtype, name, max_abs_scale=scale)


@pytest.mark.parametrize("variant", ["s", "n"])
@pytest.mark.parametrize("size", [3.0, 9.0e3, 1.1e4, 3.0e6])
def test_fp32_sin_cos_at_exact_arguments(variant, size):
    """One token with one-hot q and k: every projection argument is a frequency or half of one
    exactly, so den = phi(q) . phi(k) shows the sin and cos alone, on both sides of the
    argument size where the kernels change methods.  Each of den's 4 M products has two
    factors within 2^-23 of exact: |error| <= 4 * 2^-23 per frequency's share of the mean."""
    H, M, d = 64, 33, 4
    rng = np.random.default_rng(5)
    W1 = rng.uniform(-size, size, (H, M, d)).astype(np.float32)
    W2 = rng.uniform(-size, size, (H, M, d)).astype(np.float32) if variant == "n" else None
    if W2 is not None:  # halves of sums exact in fp32: few mantissa bits
        step = np.float32(2.0 ** np.floor(np.log2(size / 4096)))
        W1, W2 = (step * np.rint(w / step) for w in (W1, W2))
    x = np.zeros((1, H, 1, d), np.float32)
    x[..., 0] = 1.0
    q, k, v = x, np.float32(0.5) * x, x
    out, den = flexattn.linattn_fwd(*(to_dev(a, "f32") for a in (q, k, v, W1, W2)), False)
    _, rd = oracle.fwd(q, k, v, W1, W2, False)
    assert np.abs(to_host(den) - rd).max() <= 4 * 2.0 ** -23
