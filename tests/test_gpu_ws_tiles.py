"""The persistent kernel's factorisation and solves at every tile count.

Rows without ratings skip the bf16 Gram: their precision is Lambda_s alone, so
what separates their draws from the oracle's is the FP32 tile arithmetic (the
TF32-split updates, the diagonal tiles, the panels, the back substitution).
They are held to the FP32 paths' bound, at both edges of every tile row
(K + 1 = 8 g - 7 and 8 g) and in between; the few rated rows to the mixed
path's.
"""
import numpy as np
import pytest

import synth
from parity_util import TAU_FP32, oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [8, 9, 15, 16, 22, 31, 32, 36, 47, 48, 55, 63, 64, 72, 79, 87, 95, 96,
                               100, 103, 104, 111, 119, 120, 127])
def test_rows_of_the_prior_alone(gpu_lib, K):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    M, N, nnz = 400, 50, 300
    cells = rng.permutation(M // 4 * N)[:nnz]  # ratings of the first quarter of the users only
    row, col = (cells // N).astype(np.int32), (cells % N).astype(np.int32)
    val = rng.normal(size=nnz).astype(np.float32)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("prior", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=11, path=bp.PATH_MIXED,
                    heavy_kernel=1, tiny_max=-1, light_max=-1) as s:
        s.set_thresholds(0, [-1, -1, 1 << 40, 1, 0])
        s.set_state(U, V, hyper, it=3)
        s.sweep(0)
        got = s.get_state()[0]
        assert s.sweep_info(0)[1] == 0
    ref = oracle_sweep(ds, 0, U, V, hy, 2.0, 11, 3)
    err = rel_err(got, ref)
    bare = np.bincount(row, minlength=M) == 0
    assert err[bare].max() <= TAU_FP32, err[bare].max()
    assert err[~bare].max() <= 1e-3, err[~bare].max()
