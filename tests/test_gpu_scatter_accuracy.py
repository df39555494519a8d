"""The centred scatter against FP64, beside the 4 x 4 and 8 x 8 tiles before it.

The rows of a block are summed in FP32 by subsets, whose sums are joined in FP32
before they go to FP64; with many subsets (17 for K = 33 .. 40) the joining
counts.  BASE holds the rms error of the form before (commit 31d30a4, measured on
a GB300 for the same inputs), relative to sqrt(S_ii S_jj); the bound is 1.05 times
it, for the order of the sums differs.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (K, rows): rms error of the scatter of 31d30a4
BASE = {
    (33, 64): 1.38e-08, (33, 500): 5.14e-09, (33, 5000): 1.87e-09, (40, 2000): 2.70e-09,
    (41, 500): 5.07e-09, (48, 2000): 2.70e-09, (50, 20000): 1.72e-09, (64, 500): 5.96e-09,
    (64, 20000): 2.82e-09, (65, 2000): 2.39e-09, (100, 2000): 2.69e-09, (128, 5000): 4.62e-09,
}


def rms_error(bp, K, R):
    import torch

    rng = np.random.default_rng(K * 7 + R)
    errors = []
    for _ in range(4):
        X = (rng.normal(size=(R, K)) * K ** -0.25 + 0.1 * rng.normal(size=K)).astype(np.float32)
        x = X.astype(np.float64)
        x -= x.mean(0)
        ref = x.T @ x
        xbar = torch.zeros(K, dtype=torch.float64, device="cuda")
        S = torch.zeros(K * K, dtype=torch.float64, device="cuda")
        bp.bpmf_hyper_stats_noalloc(torch.from_numpy(X).cuda(), R, K, xbar, S)
        torch.cuda.synchronize()
        d = np.sqrt(np.diag(ref))
        errors.append(np.mean(((S.cpu().numpy().reshape(K, K) - ref) / np.outer(d, d)) ** 2))
    return float(np.sqrt(np.mean(errors)))


@pytest.mark.parametrize("K,R", sorted(BASE))
def test_no_further_from_fp64_than_before(gpu_lib, K, R):
    assert rms_error(gpu_lib, K, R) <= 1.05 * BASE[K, R]
