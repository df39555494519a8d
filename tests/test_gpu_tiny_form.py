"""A tiny row's draw does not depend on the form its products take.

Where a tiny bin's rows and ratings outnumber the other side's rows three times,
and the memory is to be had, L_s^-1 is applied to every row of the other side
once per sweep; else row by row.  A row's draw depends on its own ratings, the
other side and (seed, iteration, side, row) only, so the same rows alone (row by
row) and among many others (once per sweep) must be bitwise the same.  The
ratings are +-1 with mean exactly 0 in both.
"""
import numpy as np
import pytest

import synth
from parity_util import TAU_FP32, oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [3, 20, 32, 33, 64, 65, 96, 100, 128])
def test_same_draws_in_both_forms(gpu_lib, K):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    N = 400
    deg = np.array([0, 1, 2, 3, 4, 5, 6, 7, 8, 8, 31, 32, 1])  # the sum is even

    def data(M, degrees):
        row = np.repeat(np.arange(M), degrees).astype(np.int32)
        col = np.concatenate([rng.permutation(N)[:d] for d in degrees]).astype(np.int32)
        return row, col, np.where(np.arange(row.size) % 2 == 0, 1.0, -1.0).astype(np.float32)

    m = len(deg)
    row, col, val = data(m, deg)
    more_row, more_col, more_val = data(700, np.full(700, 2))
    few = (row, col, val)
    many = tuple(np.concatenate(p) for p in ((row, more_row + m), (col, more_col), (val, more_val)))
    assert m + row.size < 3 * N <= m + 700 + many[0].size
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("few", m, N, K, 2.0, *few, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    # a well-conditioned prior of the rows: none of them goes to the FP64 redo
    q = np.linalg.qr(rng.normal(size=(K, K)))[0]
    hy[0] = ((q * np.linspace(0.5, 2.5, K)) @ q.T, rng.normal(size=K))
    hy[0] = (0.5 * (hy[0][0] + hy[0][0].T), hy[0][1])
    hyper = np.concatenate([hy[0][0].ravel(), hy[0][1], hyper[K * K + K:]])
    got = []
    for M, (r, c, v) in ((m, few), (m + 700, many)):
        with bp.Sampler(M, N, r, c, v, K=K, alpha=2.0, seed=3, path=bp.PATH_BINNED, tiny_max=32) as s:
            assert s.sweep_info(0)[0][0] == M
            s.set_state(np.zeros((M, K), np.float32), V, hyper, it=4)
            s.sweep(0)
            got.append(s.get_state()[0][:m])
            assert s.sweep_info(0)[1] == 0
    assert np.array_equal(got[0], got[1])
    assert rel_err(got[0], oracle_sweep(ds, 0, U, V, hy, 2.0, 3, 4)).max() <= TAU_FP32
