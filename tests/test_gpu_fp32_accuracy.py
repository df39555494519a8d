"""The FP32 paths' draws against FP64, beside what FP32 multiply-adds give.

The updates of the one-warp Cholesky run on tensor cores, with every operand split
in two.  That may be no further from FP64 than the plain FP32 form, every
product and sum an FP32 multiply-add.  BASE holds the rms error of that form for
the same inputs (commit 31d30a4, the last with it, measured on a GB300), in
units of the draws' rms; the bound is 1.05 times it, for the order of the sums
differs.  A large K shows the rounding of the accumulators.  The prior is
well-conditioned, so that no row goes to the FP64 redo.
"""
import numpy as np
import pytest

import synth
from parity_util import oracle_sweep

pytestmark = pytest.mark.gpu

# (K, ratings of a row, hub_min or 0): rms error of FP32 multiply-adds
BASE = {
    (56, 8, 0): 5.08e-07, (64, 30, 0): 1.05e-06, (77, 30, 0): 1.10e-06, (88, 30, 0): 1.16e-06,
    (100, 16, 0): 8.32e-07, (112, 30, 0): 1.22e-06, (119, 64, 0): 1.90e-06, (127, 8, 0): 6.14e-07,
    (128, 30, 0): 1.27e-06, (128, 100, 0): 2.20e-06, (112, 24, 16): 9.79e-07, (128, 64, 33): 1.60e-06,
}


def inputs(K, d):
    rng = np.random.default_rng(1000 * K + d)
    M, N = max(256, min(4096, 40000 // K)), 1500
    row = np.repeat(np.arange(M), d).astype(np.int32)
    col = np.concatenate([rng.permutation(N)[:d] for _ in range(M)]).astype(np.int32)
    V = (rng.normal(size=(N, K)) * K ** -0.25).astype(np.float32)
    U = (rng.normal(size=(M, K)) * K ** -0.25).astype(np.float32)
    val = ((U[row].astype(np.float64) * V[col]).sum(1) + rng.normal(size=row.size)).astype(np.float32)
    q = np.linalg.qr(rng.normal(size=(K, K)))[0]
    lam = (q * np.linspace(0.5, 2.5, K)) @ q.T
    lam, mu = 0.5 * (lam + lam.T), rng.normal(size=K)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("accuracy", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    return ds, U, V, [(lam, mu), (lam, mu)]


def rms_error(bp, K, d, hub):
    ds, U, V, hy = inputs(K, d)
    hyper = np.concatenate([np.r_[lam.ravel(), mu] for lam, mu in hy])
    with bp.Sampler(ds.M, ds.N, ds.train_row, ds.train_col, ds.train_val, K=K, alpha=2.0, seed=7,
                    path=bp.PATH_BINNED if hub else bp.PATH_PLAIN, hub_min=hub or -1) as s:
        s.set_state(U, V, hyper, it=2)
        s.sweep(0)
        got = s.get_state()[0].astype(np.float64)
        assert s.sweep_info(0)[1] == 0
    ref = oracle_sweep(ds, 0, U, V, hy, 2.0, 7, 2)
    return float(np.sqrt(np.mean((got - ref) ** 2) / np.mean(ref ** 2)))


@pytest.mark.parametrize("K,d,hub", sorted(BASE))
def test_no_further_from_fp64_than_multiply_adds(gpu_lib, K, d, hub):
    assert rms_error(gpu_lib, K, d, hub) <= 1.05 * BASE[K, d, hub]
