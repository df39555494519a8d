"""FP32 rows and pieces at every tile count, against the oracle.

Rows of 0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 40 and 100 ratings (the steps of
eight and sixteen neighbours and of a 32-row stage, at, below and above their
edges), whole and as hubs split into pieces of 16, of 13 and of 3 ratings, for latent
dimensions at both edges of every tile row of the one-warp kernel, for the
three copy widths (K a multiple of four, even, odd) and on the first sizes of
the kernel that follows it.  Held to the FP32 paths' bound.
"""
import numpy as np
import pytest

import synth
from parity_util import TAU_FP32, oracle_sweep, random_state, rel_err

pytestmark = pytest.mark.gpu

DEGREES = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 40, 100]


@pytest.mark.parametrize("hub", [None, 32, 26, 7])
@pytest.mark.parametrize("K", [1, 2, 7, 8, 10, 15, 16, 20, 23, 24, 29, 31, 32, 39, 40, 47, 48, 50, 53, 54,
                               55, 56, 57, 64, 71, 100, 127, 128])
def test_rows_and_pieces(gpu_lib, K, hub):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    M, N = 3 * len(DEGREES), 160
    deg = np.tile(DEGREES, 3)
    row = np.repeat(np.arange(M), deg).astype(np.int32)
    col = np.concatenate([rng.permutation(N)[:d] for d in deg]).astype(np.int32)
    val = rng.normal(size=row.size).astype(np.float32)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("edges", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U, V, hy, hyper = random_state(ds, K)
    hub_min = hub or 1 << 30  # a piece has hub_min / 2 ratings
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=7, path=bp.PATH_BINNED, tiny_max=-1,
                    light_max=1 << 30, hub_min=hub_min) as s:
        s.set_state(U, V, hyper, it=2)
        s.sweep(0)
        got = s.get_state()[0]
        bins, redone = s.sweep_info(0)
        assert redone == 0
        assert bins[3] == (0 if hub is None else int((deg >= hub_min).sum())), bins
    ref = oracle_sweep(ds, 0, U, V, hy, 2.0, 7, 2)
    err = rel_err(got, ref)
    assert err.max() <= TAU_FP32, (err.max(), deg[int(err.max(1).argmax())])
