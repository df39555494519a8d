"""The FP64 algebra of the Normal-Wishart draw, apart from its normals.

Lambda = C G C^T with C = chol(W*) and G = A A^T, where Bartlett's A depends on
(seed, iteration, side, nu*) only.  So G, taken from one draw with the C of its
posterior, predicts another draw of the same seed and row count with other
factors and another prior: both sides of that are FP64 algebra, with the FP32
normals inside G.  The factor rows are +-1 over 64 rows, so the FP32 statistics
are exact (the mean is a multiple of 1/32, a centred product of 2^-10).  W* has
eigenvalues within a factor of 20, so each of the handful of triangular products
and solves is good to about 20 K 2^-53 < 3e-13 of the norms it combines; the
bound is 1e-11.  A pivot's reciprocal or root good to FP32 only (2^-24 = 6e-8)
would show.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 2, 10, 16, 17, 32, 33, 64, 65, 100, 128])
def test_draws_share_bartletts_factor_in_fp64(gpu_lib, K):
    bp = gpu_lib
    rng = np.random.default_rng(K)
    M = 64
    q = np.linalg.qr(rng.normal(size=(K, K)))[0]
    lams, chols = [], []
    for lo in (0.01, 0.02):
        W0 = (q * np.linspace(lo, 2 * lo, K)) @ q.T
        W0 = 0.5 * (W0 + W0.T)
        U = rng.choice([-1.0, 1.0], size=(M, K)).astype(np.float32)
        with bp.Sampler(M, 4, [0], [0], [1.0], K=K, seed=5, path=bp.PATH_BINNED, W0=W0) as s:
            s.set_state(U, np.zeros((4, K), np.float32), it=3)
            s.sample_hyper(0)
            lams.append(s.get_state()[2][:K * K].reshape(K, K))
            xbar, S = s.hyper_stats(0)
        x = U.astype(np.float64)
        assert np.array_equal(xbar, x.mean(0))
        xc = x - x.mean(0)
        assert np.array_equal(S, xc.T @ xc)
        W = oracle.nw_posterior(M, xbar, S, np.zeros(K), 2.0, float(K), W0)[3]
        assert np.linalg.cond(W) < 20
        chols.append(np.linalg.cholesky(W))
    t = np.linalg.solve(chols[0], lams[0])
    G = np.linalg.solve(chols[0], t.T)
    want = chols[1] @ G @ chols[1].T
    d = np.sqrt(np.diag(want))
    assert np.max(np.abs(lams[1] - want) / np.outer(d, d)) <= 1e-11
