"""Verify forwards of 17 to 128 rows (the chain of projections that finish their rows) and the first
sizes beyond (pairs of CTAs), through the whole verify step against the float64 oracle: the smallest
and the largest number of rows, both sides of the limits at which token rows are halved between CTAs,
a down projection whose K is split over a cluster (and not a multiple of its eight CTAs' k-steps),
every head size, row groups, prefixes from one cached token to more tiles than key splits.
"""
import pytest

from paper_2505_15380_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,hq,hkv,d,f,gamma,lens,capacity", [
    (64, 2, 1, 128, 256, 1, [5] * 9, None),                        # 18 rows
    (32, 4, 2, 136, 264, 7, [2, 64, 65, 1, 30, 31], None),          # 48 rows, K not a multiple of 16
    (64, 14, 2, 128, 2064, 6, [70, 1, 200, 64, 63, 128, 9], 700),   # 49 rows, K = 129 k-steps over 8 CTAs
    (128, 4, 2, 256, 4864, 7, [600, 33, 129], 900),                 # 24 rows, long K
    (64, 6, 2, 192, 2048, 15, [100, 1, 65, 40, 17, 64, 190, 2], None),   # 128 rows
    (64, 8, 1, 128, 256, 8, [130, 64], 2200),                       # 72 query rows per kv head: two row groups
    (64, 4, 2, 128, 384, 2, [20 + i for i in range(43)], None),     # 129 rows: pairs of CTAs
])
def test_verify_matches_oracle(hd, hq, hkv, d, f, gamma, lens, capacity):
    from tests.gpu_case import run_case
    shape = synth.ModelShape(2, d, hq, hkv, hd, f, 301, 8, 1e4, weight_dtype=synth.BF16)
    wl = synth.Workload("chain", shape, shape, len(lens), gamma, 0.8, 25, tuple(lens), 2, hd + f, hd + f + 1)
    run_case(wl, beta=0.4, sigma=1.0, commit_and_repeat=True, logit_tol=2e-3, capacity=capacity)
    pages = sum(-(-(n + gamma + 1) // 64) for n in lens) + len(lens) + 2
    run_case(wl, beta=0.0, sigma=0.5, logit_tol=2e-3,
             paged=(pages, max(-(-(max(lens) + 2 * gamma + 2) // 64) + 1, 4)))
