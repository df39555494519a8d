"""Long rows that all rate the other side's last row, whose shadow ends the array:
where K is a multiple of eight the rating's chunk of features lies past it, and
what follows (here the statistics of the side, any bit pattern as bf16) must not
reach the product.  Every row within the mixed path's bound, none redone.
"""
import numpy as np
import pytest

import synth
from parity_util import oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 2100])  # three products a step, and two
@pytest.mark.parametrize("K", [63, 64, 65, 72, 80, 96, 100, 112, 120])
def test_last_neighbour(gpu_lib, K, n):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    M, N = 200, 2400
    deg = np.full(M, n)
    row = np.repeat(np.arange(M), deg).astype(np.int32)
    col = np.concatenate([np.r_[rng.permutation(N - 1)[:n - 1], N - 1] for _ in range(M)]).astype(np.int32)
    val = rng.normal(size=row.size).astype(np.float32)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("last", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=13, path=bp.PATH_MIXED,
                    heavy_kernel=1, tiny_max=-1, light_max=-1) as s:
        s.set_thresholds(0, [-1, -1, 1 << 40, 1, 0])
        for it in range(3):
            s.set_state(U, V * np.float32(1 + it), it=3)
            s.sample_hyper(1)
            s.set_state(U, V, hyper, it=3)
            s.sweep(0)
            assert s.sweep_info(0)[1] == 0
        got = s.get_state()[0]
    err = rel_err(got, oracle_sweep(ds, 0, U, V, hy, 2.0, 13, 3))
    assert err.max() <= 1e-3, err.max()
