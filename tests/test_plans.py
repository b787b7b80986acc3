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


# Measured on 148 SMs, launches in a row.
ATTENTION_US = [
    # head_dim, items, heads, queries, keys: us with the keys of a group over 1, 2, 4, 8 thread blocks
    ((32, 1, 8, 310, 1319), (44.27, 36.95, 34.18, 27.1)),
    ((32, 1, 16, 110, 442), (16.33, 12.76, 9.9, 10.33)),
    ((32, 1, 1, 1319, 1319), (44.2, 26.81, 20.94, 19.95)),
    ((32, 1, 2, 442, 442), (16.28, 12.73, 8.59, 7.18)),
    ((32, 1, 18, 250, 500), (18.38, 16.52, 19.44, 20.9)),
    ((64, 1, 2, 600, 1240), (59.59, 35.43, 28.68, 26.02)),
    ((64, 1, 2, 310, 1319), (62.46, 38.24, 22.11, 19.25)),
    ((64, 1, 8, 310, 1319), (62.56, 58.36, 46.04, 48.66)),
    ((64, 1, 16, 64, 2000), (93.82, 52.5, 34.98, 31.77)),
    ((64, 1, 16, 310, 1319), (100.7, 81.31, 78.43, 81.47)),
    ((64, 2, 1, 32, 144), (11.01, 12.2, 7.38)),
    ((128, 1, 2, 110, 442), (37.65, 30.93, 17.07, 11.86)),
    ((128, 1, 4, 110, 442), (37.81, 31.07, 17.14, 22.38)),
    ((128, 1, 8, 310, 1319), (106.7, 128.8, 108.5, 126.2)),
    ((128, 1, 2, 1319, 1319), (107.1, 129, 108.8, 126.6)),
    ((128, 1, 8, 64, 2000), (160.5, 89.9, 46.48, 52.22)),
    ((64, 1, 10, 600, 1240), (96.25, 74.72, 77.81, 96.03)),
    ((64, 1, 16, 1319, 1319), (234, 252.8, 264.2, 302.8)),
    ((32, 1, 16, 1319, 1319), (144.2, 148.9, 153.6, 165.9)),
    ((128, 1, 8, 1319, 1319), (316.8, 323.1, 394.9, 481.7)),
    ((32, 2, 9, 52, 528), (20.2, 14.66, 10.99, 13.41)),
    ((32, 2, 16, 146, 586), (31.42, 30.71, 26.1, 31.24)),
    ((32, 3, 2, 431, 431), (16.33, 16.36, 15.09, 15.2)),
    ((32, 3, 12, 180, 722), (37.4, 36.64, 34.18, 43.32)),
    ((32, 1, 10, 90, 265), (12.22, 10.68, 8.55, 7.45)),
    ((32, 1, 20, 2282, 2282), (459.8, 463.8, 482.4, 548.9)),
    ((32, 1, 16, 707, 2080), (170.8, 121, 130.8, 137.2)),
    ((64, 1, 16, 102, 301), (16.92, 15.57, 18.97, 20.62)),
    ((64, 3, 13, 459, 919), (138.7, 153.6, 167.9, 195.9)),
    ((64, 1, 1, 1304, 2609), (119.5, 66.95, 56.05, 45.59)),
    ((64, 2, 15, 85, 425), (22.67, 26.22, 19.64, 23.89)),
    ((64, 1, 9, 224, 449), (25.55, 18.4, 19.03, 20.61)),
    ((64, 3, 14, 286, 1144), (122.7, 129.6, 135.4, 164.7)),
    ((64, 2, 5, 113, 1130), (53.83, 32.72, 28.61, 25.55)),
    ((128, 1, 4, 333, 1333), (106.6, 65.6, 72.54, 63.86)),
    ((128, 3, 4, 125, 629), (52.55, 36.18, 43.22, 64.49)),
    ((128, 1, 1, 68, 684), (57.28, 40.39, 21.67, 16.57)),
    ((128, 1, 6, 511, 2559), (200.3, 217.4, 167.9, 216)),
    ((128, 1, 1, 535, 1574), (126.1, 75.13, 41.7, 52.01)),
    ((128, 3, 1, 569, 2279), (180.3, 100.3, 102.4, 123.9)),
    ((128, 2, 4, 94, 472), (42.63, 30.94, 17.21, 22.99)),
]


@pytest.mark.parametrize("problem,us", ATTENTION_US, ids=lambda v: "x".join(map(str, v)) if isinstance(v[0], int) else "")
def test_fp32_attention_takes_nearly_the_best_split(problem, us):
    """Within 5 % of the fastest, runs of one problem lying 1 to 2 % apart."""
    head_dim, items, heads, queries, keys = problem
    ctas = H.hero_plan_fp32_attention(items, queries, keys, heads, head_dim)
    assert us[(1, 2, 4, 8).index(ctas)] <= 1.05 * min(us)


def test_fp32_attention_split_is_one_that_the_kernel_runs():
    """A power of two up to eight, less than twice the key tiles, on any number of SMs."""
    for sms in (1, 2, 7, 20, 132, 148, 160):
        for head_dim in (32, 64, 128):
            for items, heads, queries in ((1, 1, 1), (2, 3, 33), (8, 16, 1319), (8, 96, 1 << 20)):
                for keys in (1, 64, 65, 128, 129, 600, 1 << 20):
                    ctas = H.hero_plan_fp32_attention(items, queries, keys, heads, head_dim, sms)
                    assert ctas in (1, 2, 4, 8) and (ctas == 1 or ctas < 2 * -(-keys // 64))
