"""Ratings so large that the bordered row has no pivot.

The factorisation carries b as row K of the matrix, and y = L^-1 b comes out as
that row.  Its own pivot, a corner value less y^T y (here alpha sum r^2 is about
2e33), means nothing, and neither do those of the padding rows after it: none of
them is a row of Lambda*, so none may send the row to the FP64 redo.  The draw
is linear in the ratings up to its noise, so the paths' bounds hold as for
ratings of unit size.  K = 23 has no padding row after row K; the others one to
seven.
"""
import numpy as np
import pytest

import synth
from parity_util import TAU_FP32, oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path,K,hub,tau", [
    ("plain", 3, None, TAU_FP32), ("plain", 10, None, TAU_FP32), ("plain", 23, None, TAU_FP32),
    ("plain", 32, None, TAU_FP32), ("plain", 50, None, TAU_FP32), ("plain", 60, None, TAU_FP32),
    ("binned", 20, 40, TAU_FP32), ("binned", 64, 40, TAU_FP32),
    ("mixed", 12, None, 1e-3), ("mixed", 33, None, 1e-3), ("mixed", 100, None, 1e-3),
])
def test_padding_sends_no_row_to_the_redo(gpu_lib, path, K, hub, tau):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    M, N, d = 40, 300, 130
    row = np.repeat(np.arange(M), d).astype(np.int32)
    col = np.concatenate([rng.permutation(N)[:d] for _ in range(M)]).astype(np.int32)
    val = (3e15 * rng.normal(size=row.size)).astype(np.float32)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("large", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=9,
                    path={"plain": bp.PATH_PLAIN, "binned": bp.PATH_BINNED, "mixed": bp.PATH_MIXED}[path],
                    hub_min=hub or 1 << 30) as s:
        s.set_state(U, V, hyper, it=2)
        s.sweep(0)
        got = s.get_state()[0]
        bins, redone = s.sweep_info(0)
        assert path == "plain" or (bins[3] == M) == (hub is not None)
    assert redone == 0
    assert rel_err(got, oracle_sweep(ds, 0, U, V, hy, 2.0, 9, 2)).max() <= tau
