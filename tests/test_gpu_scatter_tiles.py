"""Centred scatter at the edges of its tiles, chunks and flushes, against FP64.

Latent dimensions at both edges of every pair of tile columns, row counts at
the edges of a block's chunk of 64 and of the row subsets, each a block of its
own; and one matrix tall enough that the FP32 sums are moved to FP64 on the way
(a block of the allocation-free entry point has more than 6,144 rows).
Bound as the other statistics tests: 1e-5 in units of sqrt(S_ii S_jj).
"""
import numpy as np
import pytest

import synth
from parity_util import random_state

pytestmark = pytest.mark.gpu


def _check(xbar, S, X):
    ref = X.astype(np.float64)
    m = ref.mean(axis=0)
    ref -= m
    R = ref.T @ ref
    scale = np.sqrt(np.outer(np.diag(R), np.diag(R))) + 1e-300
    assert np.max(np.abs(xbar - m)) <= 1e-6 * (np.abs(m).max() + X.std())
    assert np.array_equal(S, S.T)
    assert np.max(np.abs(S - R) / scale) <= 1e-5


@pytest.mark.parametrize("K", [2, 8, 9, 15, 16, 17, 24, 31, 32, 33, 47, 48, 49, 50, 63, 64, 65, 79, 80, 81, 95,
                               96, 97, 111, 112, 113, 127, 128])
@pytest.mark.parametrize("M,N", [(2, 7), (8, 9), (31, 32), (33, 63), (64, 95), (96, 97), (129, 4000)])
def test_edges(gpu_lib, K, M, N):
    bp = gpu_lib
    ds = synth.uniform(M, N, min(M * N, 50), K, seed=K)
    U, V, _, hyper = random_state(ds, K)
    U += np.float32(0.5)
    with bp.Sampler(M, N, ds.train_row, ds.train_col, ds.train_val, K=K, seed=1, path=bp.PATH_BINNED) as s:
        s.set_state(U, V, hyper)
        for side, X in ((0, U), (1, V)):
            s.sample_hyper(side)
            _check(*s.hyper_stats(side), X)


def test_sums_moved_on_the_way(gpu_lib):
    import torch
    bp = gpu_lib
    R, K = 1_600_000, 48
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(R, K, generator=g, device="cuda") * 0.3 + 0.1
    xbar = torch.zeros(K, dtype=torch.float64, device="cuda")
    S = torch.zeros(K, K, dtype=torch.float64, device="cuda")
    bp.bpmf_hyper_stats_noalloc(X, R, K, xbar, S)
    torch.cuda.synchronize()
    _check(xbar.cpu().numpy(), S.cpu().numpy(), X.cpu().numpy())
