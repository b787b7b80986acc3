"""The rules on sizes, on the host: what they choose is what the hardware takes and what was measured to be near the best."""
import pytest

import paper_2508_17588_b200 as H
from paper_2508_17588_b200 import binding as Bd


def test_fp32_gemm_serves_every_row_count_that_its_larger_tile_serves():
    """Row tiles go into a grid dimension of 65535, whichever tile the columns would like better."""
    most = 65535 * 64
    for hidden in (32, 64, 96, 128, 160, 192, 224, 256, 320, 384, 416, 512, 544, 1024):
        for ffn in (4, 36, 96, 128, 4 * hidden):
            for n, k in ((3 * hidden, hidden), (hidden, hidden), (ffn, hidden), (hidden, ffn)):
                for m in (65535 * 32, 65535 * 32 + 1, 8 * 262141, 3000001, most):
                    tile, _ = H.hero_plan_fp32_gemm(m, n, k)
                    assert -(-m // tile) <= 65535, (m, n, k, tile)
    with pytest.raises(H.HeroError) as e:
        H.hero_plan_fp32_gemm(most + 1, 64, 64)
    assert e.value.code == Bd.ERR_ARG
