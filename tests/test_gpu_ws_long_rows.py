"""Rows of more than 2,048 ratings on the persistent kernel: stages of 64
neighbours, h^T h and h^T l as one product, at both edges of its sixteen-column
steps and of the 64-feature blocks; row lengths at the edges of a stage, of a
gather warp's share of it and of the product's sixteen neighbours.  Held to the
mixed path's bound for well-conditioned rows, 1e-3.
"""
import numpy as np
import pytest

import synth
from parity_util import oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [8, 15, 16, 31, 47, 48, 63, 64, 79, 80, 95, 96, 100, 111, 112, 127])
def test_long_rows(gpu_lib, K):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    deg = np.array([2304, 2303, 2305, 2240, 2256, 2272, 2288, 2289, 2241, 2111, 64, 17, 1, 0])
    deg = np.concatenate([deg, np.full(60, 2310)])
    M, N = deg.size, 2400
    row = np.repeat(np.arange(M), deg).astype(np.int32)
    col = np.concatenate([rng.permutation(N)[:d] for d in deg]).astype(np.int32)
    val = rng.normal(size=row.size).astype(np.float32)
    assert row.size >= 2048 * M
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("long", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=13, path=bp.PATH_MIXED,
                    heavy_kernel=1, tiny_max=-1, light_max=-1) as s:
        s.set_thresholds(0, [-1, -1, 1 << 40, 1, 0])
        s.set_state(U, V, hyper, it=3)
        s.sweep(0)
        got = s.get_state()[0]
        assert s.sweep_info(0)[1] == 0
    ref = oracle_sweep(ds, 0, U, V, hy, 2.0, 13, 3)
    err = rel_err(got, ref)
    assert err.max() <= 1e-3, (err.max(), deg[int(err.max(1).argmax())])
