"""The Normal-Wishart draw at every size of its cluster and of its groups of 32
rows, against the oracle, and the rows drawn from it; W0^-1, which the same code
factors and inverts, enters through the prior.

The factor rows are +-1 over 64 rows, so the kernels' FP32 statistics are
exact (the mean is a multiple of 1/32, a centred product of 2^-10, a sum at
most 2^8) and the FP64 posterior agrees with the oracle's to rounding.  What is
left are the FP32 Box-Muller normals, off by a few 1e-7: an entry of Lambda =
B B^T by about that times the norms of its two rows of B, the draw of mu by
about that times its own spread.  The bound is 1e-5 of either.  The rows are
then held to the FP32 paths' bound (where the draw is ill-conditioned, K near or
past the 64 rows, the pivot rule sends them to the FP64 redo): they read the bordered FP32 copy and, up to
eight ratings, chol(Lambda).
"""
import numpy as np
import pytest

import oracle
import synth
from parity_util import TAU_FP32, oracle_sweep, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W0", ["identity", "dense"])
@pytest.mark.parametrize("K", [1, 2, 10, 15, 16, 17, 31, 32, 33, 50, 63, 64, 65, 95, 96, 97, 100, 127, 128])
def test_draw_matches_oracle(gpu_lib, K, W0):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    M = N = 64
    deg = np.arange(M) % 17
    row = np.repeat(np.arange(M), deg).astype(np.int32)
    col = np.concatenate([rng.permutation(N)[:d] for d in deg]).astype(np.int32)
    val = rng.normal(size=row.size).astype(np.float32)
    e = np.zeros(0, np.int32)
    ds = synth.Dataset("signs", M, N, K, 2.0, row, col, val, e, e, np.zeros(0, np.float32))
    U = rng.choice([-1.0, 1.0], size=(M, K)).astype(np.float32)
    V = rng.choice([-1.0, 1.0], size=(N, K)).astype(np.float32)
    # the dense prior has eigenvalues between 0.5 and 2.5
    q = np.linalg.qr(rng.normal(size=(K, K)))[0]
    w0 = np.eye(K) if W0 == "identity" else (q * np.linspace(0.5, 2.5, K)) @ q.T
    prior = dict(mu0=np.zeros(K), beta0=2.0, nu0=float(K), W0=w0)
    with bp.Sampler(M, N, row, col, val, K=K, alpha=2.0, seed=5, path=bp.PATH_BINNED, tiny_max=8,
                    light_max=1 << 30, hub_min=1 << 30, W0=w0) as s:
        s.set_state(U, V, it=3)
        hy = []
        for side, X in ((0, U), (1, V)):
            s.sample_hyper(side)
            hy.append(oracle.sample_hyper(X.astype(np.float64), prior, 5, 3, side))
        got = s.get_state()[2].reshape(2, K * K + K)
        for side, (lam, mu) in enumerate(hy):
            glam, gmu = got[side, :K * K].reshape(K, K), got[side, K * K:]
            d = np.sqrt(np.diag(lam))
            assert np.array_equal(glam, glam.T)
            assert np.max(np.abs(glam - lam) / np.outer(d, d)) <= 1e-5
            spread = np.sqrt(np.diag(np.linalg.inv(lam)) / (2.0 + M))
            assert np.max(np.abs(gmu - mu) / (np.abs(mu) + spread)) <= 1e-5
        s.sweep(0)
        rows = s.get_state()[0]
        ref = oracle_sweep(ds, 0, U, V, hy, 2.0, 5, 3)
        # the same rows from the same hyperparameters set, not drawn
        s.set_state(U, V, np.concatenate([np.r_[lam.ravel(), mu] for lam, mu in hy]), it=3)
        s.sweep(0)
        again = s.get_state()[0]
    assert rel_err(rows, ref).max() <= TAU_FP32
    assert rel_err(again, ref).max() <= TAU_FP32
