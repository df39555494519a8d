"""Pairs outside the factors are refused wherever they stand in a warp's 32, on
the last full or ragged group, and the call after it predicts as before."""
import numpy as np
import pytest

import synth
from parity_util import random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [10, 32, 100])
@pytest.mark.parametrize("n,at", [(1, 0), (32, 31), (33, 32), (65, 31), (65, 64)])
def test_pair_out_of_range(gpu_lib, K, n, at):
    bp = gpu_lib
    ds = synth.uniform(40, 30, 200, K, seed=3)
    U, V, _, hyper = random_state(ds, K)
    rng = np.random.default_rng(n)
    row = rng.integers(0, ds.M, n).astype(np.int32)
    col = rng.integers(0, ds.N, n).astype(np.int32)
    with bp.Sampler(ds.M, ds.N, ds.train_row, ds.train_col, ds.train_val, K=K) as s:
        s.set_state(U, V, hyper)
        good = s.predict(row, col).copy()
        for r, c in ((ds.M, 0), (-1, 0), (0, ds.N), (0, -1)):
            br, bc = row.copy(), col.copy()
            br[at], bc[at] = r, c
            with pytest.raises(bp.BpmfError):
                s.predict(br, bc)
        assert np.array_equal(s.predict(row, col), good)
