"""Index arithmetic of the one-warp Cholesky and of the few-ratings Gram, on the CPU.

warp_chol.cuh factors the bordered matrix left-looking, by block columns J of
8 x 8 tiles: an update of the tiles I >= J, four (two pairs) at a time and the
rest as one pair, whose second tile and whose pairs past the last tile compute
on a tile that is there and store nothing; the diagonal tile in registers; the
panel below it, a lane a row, 64 rows at a time; and a back substitution in which
lane 2 J + h owns columns 8 J + 4 h .. + 3.  rows_small.cu's multiply-adds keep
the lower tiles in pairs of accumulators.  The loops are followed here as they
stand there: every tile is stored once per block column, every row of a panel
solved once, no address leaves the slot, and the result is the factor and the
draw, for every latent dimension; so does the map of the Gram's accumulators.
"""
import numpy as np
import pytest

TILE = 68


def tidx(i, j):
    return i * (i + 1) // 2 + j


def trow(r):
    return r * 8 + ((r >> 2) << 2)


def store(A, g):
    T = np.full(g * (g + 1) // 2 * TILE, np.nan)
    for I in range(g):
        for J in range(I + 1):
            for r in range(8):
                at = tidx(I, J) * TILE + trow(r)
                T[at:at + 8] = A[8 * I + r, 8 * J:8 * J + 8]
    return T


def tile(T, I, J):
    return np.array([T[tidx(I, J) * TILE + trow(r):][:8] for r in range(8)])


def put(T, I, J, x):
    for r in range(8):
        at = tidx(I, J) * TILE + trow(r)
        T[at:at + 8] = x[r]


def update(T, g, J, I0, pairs, ways, stored):
    for i in range(pairs):
        I = min(I0 + 2 * i, g - 1)
        both = (I, I + 1 if I + 1 < g else I)
        acc = np.zeros((ways, 2, 8, 8))
        for p in range(0, J, ways):
            for w in range(ways):
                if w > 0 and p + w >= J:
                    break
                for h in range(2):
                    acc[w, h] += tile(T, both[h], p + w) @ tile(T, J, p + w).T
        for h, real in ((0, I0 + 2 * i), (1, I0 + 2 * i + 1)):
            if real < g:
                assert real == both[h]
                put(T, real, J, tile(T, real, J) - acc.sum(0)[h])
                stored.append((real, J))


def cholesky(T, g, K, ways):
    rinv = np.zeros(8 * g)
    for J in range(g):
        stored = []
        if J > 0:
            I0 = J
            while g - I0 > 2:
                update(T, g, J, I0, 2, ways, stored)
                I0 += 4
            if g - I0 > 0:
                update(T, g, J, I0, 1, ways, stored)
            assert sorted(stored) == [(I, J) for I in range(J, g)]  # each tile once
        d = tile(T, J, J)
        for c in range(8):
            piv = d[c, c]
            assert piv > 0
            r = 0.0 if np.isinf(piv) else 1.0 / np.sqrt(piv)
            rinv[8 * J + c] = r
            d[c + 1:, c] *= r
            for j in range(c + 1, 8):
                d[j:, j] -= d[j:, c] * d[j, c]
        for i in range(1, 8):  # the strict lower triangle and what shares its 16 bytes
            at = tidx(J, J) * TILE + trow(i)
            T[at:at + (8 if i > 4 else 4)] = d[i, :8 if i > 4 else 4]
        nr, solved = 8 * (g - 1 - J), []
        for r0 in range(0, nr, 64):
            for lane in range(32):
                for k in range(2):
                    rr = r0 + lane + 32 * k
                    if rr < nr:
                        at = tidx(J + 1 + (rr >> 3), J) * TILE + trow(rr & 7)
                        x = T[at:at + 8].copy()
                        for c in range(8):
                            x[c] *= rinv[8 * J + c]
                            x[c + 1:] -= x[c] * d[c + 1:, c]
                        T[at:at + 8] = x
                        solved.append(rr)
        assert sorted(solved) == list(range(nr))
    return rinv


def back(T, rinv, z, K):
    v = np.zeros((32, 4))
    IK, pk = K >> 3, K & 7
    for lane in range(32):
        J, h4 = lane >> 1, (lane & 1) << 2
        if J <= IK:
            at = tidx(IK, J) * TILE + trow(pk) + h4
            v[lane] = T[at:at + 4] + z[8 * J + h4:8 * J + h4 + 4]
    for I in range((K - 1) >> 3, -1, -1):
        u = np.array([v[2 * I + (q >> 2), q & 3] for q in range(8)])
        d = tile(T, I, I)
        for c in range(7, -1, -1):
            u[c] = u[c] * rinv[8 * I + c] if c < K - 8 * I else 0.0
            u[:c] -= d[c, :c] * u[c]
        for lane in range(32):
            J, h4 = lane >> 1, (lane & 1) << 2
            if J < I:
                v[lane] -= u @ tile(T, I, J)[:, h4:h4 + 4]
            elif J == I:
                v[lane] = u[h4:h4 + 4]
    return np.array([v[(k >> 3) * 2 + ((k & 7) >> 2), k & 3] for k in range(K)])


@pytest.mark.parametrize("ways", [1, 2])
@pytest.mark.parametrize("K", list(range(1, 35)) + [39, 40, 47, 55, 56, 63, 64, 65, 71, 87, 88, 100, 119, 127, 128])
def test_factor_and_draw(K, ways):
    rng = np.random.default_rng(K)
    g = (K + 8) // 8
    x = rng.normal(size=(2 * K + 5, K))
    lam = x.T @ x + np.eye(K)
    b, z = rng.normal(size=K), rng.normal(size=8 * g)
    A = np.eye(8 * g)
    A[:K, :K] = lam
    A[K, :K] = b
    A[K, K] = np.inf
    T = store(np.tril(A), g)
    u = back(T, cholesky(T, g, K, ways), z, K)
    L = np.linalg.cholesky(lam)
    want = np.linalg.solve(L.T, np.linalg.solve(L, b) + z[:K])
    assert np.max(np.abs(u - want)) <= 1e-9 * np.max(np.abs(want))


@pytest.mark.parametrize("G", [1, 2, 3])
def test_accumulators_of_the_few_ratings_gram(G):
    rng = np.random.default_rng(G)
    n = 7
    X = np.zeros((8, 8 * G))
    X[:n] = rng.normal(size=(n, 8 * G))
    r = np.zeros(8)
    r[:n] = rng.normal(size=n)
    NP = (G + 1) // 2
    NA = (NP - 1) * NP + 2 * NP - 1 if G & 1 else NP * (NP + 1)
    got, s = np.zeros((8 * G, 8 * G)), np.zeros((32, G))
    for lane in range(32):
        gr, t = lane >> 2, lane & 3
        o = np.zeros((NA, 4))
        for e0 in range(0, n, 4):
            for e in range(4):
                x = [X[e0 + e, 8 * I + gr] for I in range(G)]
                for J in range(G):
                    y = X[e0 + e, 8 * J + 2 * t:8 * J + 2 * t + 2]
                    for I in range(J, G):
                        k = (I >> 1) * ((I >> 1) + 1) + J
                        o[k, 2 * (I & 1)] += x[I] * y[0]
                        o[k, 2 * (I & 1) + 1] += x[I] * y[1]
                if e == t:
                    s[lane] += r[e0 + t] * np.array(x)
        for k in range(NP):  # as the tiles are formed from them
            for J in range(G):
                for h in range(2):
                    I = 2 * k + h
                    if J <= I < G:
                        got[8 * I + gr, 8 * J + 2 * t:8 * J + 2 * t + 2] = o[k * (k + 1) + J, 2 * h:2 * h + 2]
    want = X.T @ X
    for I in range(G):
        for J in range(I + 1):
            assert np.allclose(got[8 * I:8 * I + 8, 8 * J:8 * J + 8], want[8 * I:8 * I + 8, 8 * J:8 * J + 8])
    sums = s.reshape(8, 4, G).sum(1)  # over the four lanes that share a feature
    assert np.allclose(sums.T.ravel(), r @ X)
