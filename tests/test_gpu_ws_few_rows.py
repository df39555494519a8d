"""The persistent kernel's wide form with fewer rows than SMs: every CTA gets at
most one, and most of its consumers only the order to stop.  The prior is
well-conditioned (eigenvalues 0.5 to 2.5), so the kernel draws every row itself
and none goes to the FP64 redo.  Held to the mixed path's bound for
well-conditioned rows, 1e-3.
"""
import numpy as np
import pytest

import synth
from parity_util import oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [64, 80, 100, 127])
@pytest.mark.parametrize("M", [1, 2, 11])
def test_few_rows_are_drawn_by_the_kernel(gpu_lib, K, M):
    bp = gpu_lib
    rng = np.random.default_rng(K + M)
    N = 150
    deg = np.resize([33, 64, 16, 0, 31, 32, 1, 100, 65, 17, 5], M)
    row = np.repeat(np.arange(M), deg).astype(np.int32)
    col = np.concatenate([rng.permutation(N)[:d] for d in deg]).astype(np.int32)
    val = rng.normal(size=row.size).astype(np.float32)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("few", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    q = np.linalg.qr(rng.normal(size=(K, K)))[0]
    lam = (q * np.linspace(0.5, 2.5, K)) @ q.T
    hy[0] = (0.5 * (lam + lam.T), rng.normal(size=K))
    hyper = np.concatenate([hy[0][0].ravel(), hy[0][1], hyper[K * K + K:]])
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=17, path=bp.PATH_MIXED, heavy_kernel=1,
                    tiny_max=-1, light_max=-1) as s:
        s.set_thresholds(0, [-1, -1, 1 << 40, 1, 0])
        assert s.sweep_info(0)[0][2] == M  # all of them in the heavy bin
        s.set_state(U, V, hyper, it=3)
        s.sweep(0)
        got = s.get_state()[0]
        assert s.sweep_info(0)[1] == 0
    assert rel_err(got, oracle_sweep(ds, 0, U, V, hy, 2.0, 17, 3)).max() <= 1e-3
