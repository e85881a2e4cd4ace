"""The fp32 kernels' plans for short sequences (chunks of 16 and 32 tokens, frequency groups of up
to 128) and for many sequences of small heads (32-token chunks): against the oracle on both
sides of each limit."""
import pytest

import test_gpu_simt

pytestmark = pytest.mark.gpu

# (variant, causal, dtype, B, H, N, d, M, tau)
CASES = [
    ("n", True, "f32", 1, 2, 15, 16, 256, True), ("n", False, "f32", 1, 2, 16, 16, 256, True),
    ("s", True, "f32", 1, 2, 17, 16, 256, False), ("s", False, "f32", 1, 1, 32, 16, 255, True),
    ("n", True, "f32", 1, 1, 33, 16, 130, True), ("n", False, "f32", 2, 1, 1, 64, 64, True),
    ("n", True, "f32", 1, 2, 16, 64, 64, False), ("n", False, "f32", 1, 2, 31, 128, 64, True),
    ("s", True, "f32", 1, 2, 14, 128, 33, True), ("s", True, "bf16", 1, 3, 20, 32, 16, True),
    # more sequences than CTAs that run at once: the fewest threads; 304 and one more
    ("n", False, "f32", 39, 8, 16, 64, 40, True), ("s", True, "f32", 39, 8, 9, 128, 32, True),
    ("n", True, "f32", 39, 8, 30, 16, 100, True), ("n", True, "f32", 39, 8, 3, 4, 3, False),
    ("n", True, "f32", 38, 8, 65, 32, 16, True), ("n", True, "f32", 61, 5, 65, 32, 16, True),
    ("s", False, "f32", 61, 5, 100, 16, 7, True), ("n", False, "bf16", 61, 5, 96, 32, 16, False),
    ("n", False, "f32", 61, 5, 530, 16, 16, True), ("n", True, "f32", 61, 5, 40, 36, 16, True),
]


@pytest.mark.parametrize("c", CASES, ids=test_gpu_simt._id)
def test_short_and_many_sequences_match_oracle(c):
    test_gpu_simt.test_fp32_kernels_match_oracle(c)
