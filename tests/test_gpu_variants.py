"""GPU parity of kernel variants that a rule on sizes chooses between, at the sizes where each can go wrong: one tile
and less, tile edges and remainders, the smallest and largest of a variant's range."""
import numpy as np
import pytest
import torch

from workloads import synthetic as S
from tests.util import rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu


def H():
    import paper_2508_17588_b200 as h
    return h


# One output rounding to bf16 (2^-9 relative at most, 2^-9 / sqrt(3) rms) on top of an fp32 accumulation whose error
# is two orders below it: 2^-9 bounds the relative 2-norm with room to spare.
GEMM_TOL = 2.0 ** -9


@pytest.mark.parametrize("M,N,K", [
    # 148 SMs: CTA pairs on 256 x 256, 224, 192 and 128 tiles; last row tile one row, last column tile 8 columns
    (3841, 2056, 72), (8774, 776, 136), (3073, 3912, 8), (3510, 3080, 520), (2305, 1160, 520), (4097, 3080, 264),
    (681, 3536, 8), (1394, 1024, 1024), (1281, 1160, 1544),
    # one tile per CTA: 128 and 64 columns, K whole or over clusters of two and four CTAs (uneven K runs among them)
    (544, 1968, 8), (640, 3080, 136), (7, 1464, 8), (1, 8, 72), (33, 8, 592), (129, 1096, 520), (257, 520, 1544),
    (136, 2904, 760), (23, 16, 1768), (129, 200, 4104), (300, 776, 3080)])
def test_gemm_tile_variants(M, N, K):
    rng = np.random.default_rng(M + 7 * N + 13 * K)
    a = S.round_bf16(rng.standard_normal((M, K)).astype(np.float32))
    w = S.round_bf16((rng.standard_normal((N, K)) / np.sqrt(K)).astype(np.float32))
    bias = S.round_bf16(rng.standard_normal(N).astype(np.float32))
    guard = torch.full((M + 1, N), 7.0, device="cuda", dtype=torch.bfloat16)
    H().hero_gemm_bf16(to_dev(a, "bf16"), to_dev(w, "bf16"), to_dev(bias, "bf16"), guard[:M], 0)
    H().hero_isolated_status()
    want = a.astype(np.float64) @ w.astype(np.float64).T + bias.astype(np.float64)
    assert rel_l2(to_host(guard[:M]), want) <= GEMM_TOL
    assert bool((guard[M] == 7.0).all())
