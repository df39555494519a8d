"""Performance cases: the calls that users of the sampler make, at the sizes they make them.

Each case is a plain dict.  `kind` says which public call a pass goes through:

* ``step``    Gibbs iterations from a given state, as a resumed chain runs them:
              set_state, then step and test_rmse per iteration, then get_state.
* ``sweep``   one half-sweep: the rows of one side given the other side, the
              unit that Algorithm 1 repeats and the place where the time goes.
* ``predict`` ratings predicted for a list of (user, movie) pairs.
* ``init``    a sampler built from rating triples, with its compressed
              structure read back.
* ``serve``   independent jobs through the job server.

Ratings are synthetic: cells placed by power-law (Chung-Lu) or uniform weights,
values from planted factors plus noise, rounded to a star scale where the data
set has one.  States are mid-chain ones: the planted factors with noise, and
hyperparameters that fit them.  `schedule` is a degree-bin schedule as
thresholds() reports it ("users;movies", five integers each), for the large
data sets the one that the autotuner settles on, which a program that runs the
same data again passes to set_thresholds(); "" keeps the defaults.
"""
import math

import numpy as np
import torch

import paper_1705_04159_gb300 as bp

PATHS = {"binned": bp.PATH_BINNED, "mixed": bp.PATH_MIXED}
NO_SPLIT = 1 << 40


def _case(name, kind, M, N, nnz, K, **more):
    c = dict(name=name, kind=kind, M=M, N=N, nnz=nnz, K=K, row_expo=0.0, col_expo=0.0, alpha=2.0,
             offset=0.0, stars=0.0, noise=1.0, path="mixed", schedule="", iterations=1, side=0,
             pairs=0, host=False, jobs=0, test=0.1)
    c.update(more)
    return c


def listed():
    return [
        # the smallest data set in use (a check of a model or a set-up): eight
        # iterations, each a chain of short launches
        _case("step_tiny_k10", "step", 1000, 500, 20_000, 10, alpha=4.0, noise=0.5, iterations=8),
        # ordinary jobs of a serving stream: uniform cells, default schedule
        _case("step_job_k32", "step", 20_000, 8_000, 500_000, 32, alpha=4.0, noise=0.5, iterations=4),
        _case("step_job_k64", "step", 50_000, 12_000, 2_500_000, 64, alpha=4.0, noise=0.5, iterations=2),
        # a MovieLens-shaped log (Zipf degrees, half stars), FP32 kernels
        _case("step_movielens_k32", "step", 138_493, 26_744, 20_000_000, 32, row_expo=1.1,
              col_expo=1.1, alpha=1.5625, offset=3.5, stars=0.5, noise=0.8, path="binned",
              schedule="-1,%d,2048,0,0;-1,%d,4096,0,0" % (NO_SPLIT, NO_SPLIT)),
        # a ChEMBL-shaped matrix: many compounds with a rating or two each
        _case("step_chembl_k64", "step", 480_000, 5_800, 1_000_000, 64, col_expo=0.78, alpha=1.0,
              offset=6.0, schedule="8,8,8192,1,0;-1,0,2048,1,0"),
        # the largest: a Netflix-shaped log, one whole iteration with its test RMSE
        _case("step_netflix_k100", "step", 480_189, 17_770, 100_000_000, 100, row_expo=0.46,
              col_expo=0.52, offset=3.6, stars=1.0,
              schedule="-1,0,%d,1,6;-1,0,%d,1,1" % (NO_SPLIT, NO_SPLIT)),
        # half-sweeps of a regional or sampled log: many rows of about 190
        # ratings, and few rows of some thousands
        _case("sweep_users_k100", "sweep", 60_000, 17_770, 12_500_000, 100, row_expo=0.5,
              col_expo=0.6, offset=3.6, stars=1.0,
              schedule="-1,0,%d,1,6;-1,0,%d,1,1" % (NO_SPLIT, NO_SPLIT)),
        _case("sweep_movies_k100", "sweep", 120_000, 4_000, 11_000_000, 100, row_expo=0.4,
              col_expo=0.5, offset=3.6, stars=1.0, side=1,
              schedule="-1,0,%d,1,6;-1,0,%d,1,1" % (NO_SPLIT, NO_SPLIT)),
        # FP32 throughout at a K that fills no tile
        _case("sweep_fp32_k50", "sweep", 30_000, 10_000, 3_000_000, 50, row_expo=0.5, col_expo=0.7,
              path="binned"),
        # candidate pairs in no order, scored from a large model on the device
        _case("predict_k100", "predict", 480_189, 17_770, 1_000_000, 100, offset=3.6, stars=1.0,
              pairs=4_000_000),
        # building a sampler from triples on the device, structure read back
        _case("init_2m", "init", 60_000, 20_000, 2_000_000, 32, row_expo=0.6, col_expo=0.8, test=0.0),
        # a burst of small jobs at the server
        _case("serve_6_jobs", "serve", 1_000, 1_000, 10_000, 64, alpha=4.0, noise=0.5, iterations=4,
              jobs=6),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes over their logarithms, any K."""
    kind = rng.choice(["step", "step", "step", "sweep", "sweep", "sweep", "predict", "init", "serve"])
    M, N = _log_between(rng, 800, 300_000), _log_between(rng, 500, 40_000)
    nnz = min(_log_between(rng, 10_000, 12_000_000), M * N // 20)
    K = rng.choice([8, 10, 16, 20, 27, 32, 33, 50, 64, 64, 77, 96, 100, 100, 117, 128])
    skew = rng.choice([0.0, rng.uniform(0.2, 0.8)])
    more = dict(row_expo=round(0.8 * skew, 3), col_expo=round(skew, 3), alpha=rng.choice([1.0, 2.0, 4.0]),
                path="binned" if rng.random() < 0.25 else "mixed")
    if rng.random() < 0.5:
        more.update(offset=3.5, stars=rng.choice([0.5, 1.0]))
    if kind == "step":
        more["iterations"] = rng.choice([1, 2])
    elif kind == "sweep":
        more["side"] = rng.choice([0, 1])
    elif kind == "predict":
        nnz = min(nnz, 500_000)
        more.update(pairs=_log_between(rng, 20_000, 4_000_000), host=rng.random() < 0.4)
        if more["host"]:
            more["pairs"] = min(more["pairs"], 300_000)
    elif kind == "init":
        nnz = min(nnz, 3_000_000)
        more.update(host=rng.random() < 0.5, test=0.0)
    else:
        M, N, nnz, K = 1_000 + rng.randrange(1_000), 1_000 + rng.randrange(1_000), 10_000, 64
        more = dict(alpha=4.0, noise=0.5, jobs=rng.randrange(3, 8), iterations=rng.choice([2, 4]))
    c = _case("", kind, M, N, nnz, K, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs --

def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))
    return g


def _ids(n, expo, count, g):
    """`count` ids below n, id of rank r weighted (r + 1)^-expo, ranks shuffled over ids."""
    if expo == 0.0:
        return torch.randint(0, n, (count,), generator=g, device="cuda")
    cdf, perm = expo
    u = torch.rand(count, generator=g, device="cuda", dtype=torch.float64)
    return perm[torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1)]


def _weights(n, expo, g):
    if expo == 0.0:
        return 0.0
    cdf = torch.arange(1, n + 1, device="cuda", dtype=torch.float64).pow_(-expo).cumsum_(0)
    return cdf / cdf[-1], torch.randperm(n, generator=g, device="cuda")


def _cells(M, N, nnz, row_expo, col_expo, g):
    """nnz distinct cells in random order."""
    rw, cw = _weights(M, row_expo, g), _weights(N, col_expo, g)
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    yields = 0.9  # share of the draws that were new cells, as seen so far
    while keys.numel() < nnz:
        had, more = keys.numel(), int((nnz - keys.numel()) / yields * 1.05) + 1024
        keys = torch.unique(torch.cat([keys, _ids(M, rw, more, g) * N + _ids(N, cw, more, g)]))
        yields = max(0.2, (keys.numel() - had) / more)
    keys = keys[torch.randperm(keys.numel(), generator=g, device="cuda")[:nnz]]
    return torch.div(keys, N, rounding_mode="floor").int(), (keys % N).int()


def _dots(U, V, r, c):
    out = torch.empty(r.numel(), dtype=U.dtype, device=U.device)
    step = max(1, (1 << 28) // U.shape[1])
    for i in range(0, r.numel(), step):
        out[i:i + step] = (U[r[i:i + step].long()] * V[c[i:i + step].long()]).sum(1)
    return out


def _data(M, N, nnz, K, seed, c):
    """(train triples, test triples, U, V): int32, int32, float32 tensors and the state."""
    g = _gen(seed)
    row, col = _cells(M, N, nnz, c["row_expo"], c["col_expo"], g)
    sd = K ** -0.25
    U = torch.randn(M, K, generator=g, device="cuda") * sd
    V = torch.randn(N, K, generator=g, device="cuda") * sd
    val = c["offset"] + _dots(U, V, row, col) + c["noise"] * torch.randn(nnz, generator=g, device="cuda")
    if c["stars"]:
        val = (torch.round(val / c["stars"]) * c["stars"]).clamp_(c["stars"], 5.0)
    nt = int(round(c["test"] * nnz))
    train = tuple(x[nt:].clone() for x in (row, col, val))
    test = tuple(x[:nt].clone() for x in (row, col, val))
    # mid-chain factors: the planted ones and the posterior's spread about them
    U = U + 0.3 * sd * torch.randn(M, K, generator=g, device="cuda")
    V = V + 0.3 * sd * torch.randn(N, K, generator=g, device="cuda")
    return train, test, U, V


def _fitting_hyper(X):
    """(Lambda, mu) about a Normal-Wishart draw for the rows X: the inverse covariance and the mean."""
    x = X.double()
    mu = x.mean(0)
    cov = ((x - mu).T @ (x - mu) / x.shape[0]).cpu().numpy()
    lam = np.linalg.inv(cov + 1e-3 * np.trace(cov) / len(cov) * np.eye(len(cov)))
    return 0.5 * (lam + lam.T), mu.cpu().numpy()


def _job_shapes(c):
    """Shapes of the jobs of a serving burst, fixed by the case: rows, columns, ratings, K."""
    rng = np.random.default_rng(1000 * c["jobs"] + c["M"] + 7 * c["N"])
    out = []
    for j in range(c["jobs"]):
        m, n, z = (int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
                   for a, b in ((1e3, 6e4), (1e3, 2e4), (1e4, 8e5)))
        out.append((m, n, min(z, m * n // 4), (16, 32, 64)[j % 3]))
    return out


def _sampler(c, train, host=False):
    arrays = tuple(x.cpu().numpy() for x in train) if host else train
    return bp.Sampler(c["M"], c["N"], *arrays, K=c["K"], alpha=c["alpha"], seed=7, path=PATHS[c["path"]])


class _State:
    pass


IT0 = 40  # iteration the resumed chain stands at


def prepare(case, seed):
    c, s = case, _State()
    s.case = c
    if c["kind"] == "serve":
        s.jobs = []
        for j, (m, n, z, k) in enumerate(_job_shapes(c)):
            train, test, _, _ = _data(m, n, z, k, seed * 64 + j, c)
            s.jobs.append((m, n, k, tuple(x.cpu().numpy() for x in train), tuple(x.cpu().numpy() for x in test)))
        s.server = bp.Server(max_resident=16)
        return s
    M, N, K = c["M"], c["N"], c["K"]
    train, test, U, V = _data(M, N, c["nnz"], K, seed, c)
    if c["kind"] == "init":
        s.train = tuple(x.cpu().numpy() for x in train) if c["host"] else train
        return s
    s.h = _sampler(c, train)
    if c["schedule"]:
        for side, part in enumerate(c["schedule"].split(";")):
            s.h.set_thresholds(side, [int(x) for x in part.split(",")])
    if c["kind"] == "predict":
        s.h.set_state(U, V, None, it=IT0)
        r, q = _pairs(c, seed)
        s.row, s.col = (r.cpu().numpy(), q.cpu().numpy()) if c["host"] else (r, q)
        s.out = None if c["host"] else torch.empty(c["pairs"], device="cuda")
        return s
    s.U0, s.V0 = U, V
    s.U, s.V = torch.empty_like(U), torch.empty_like(V)
    if c["kind"] == "step":
        s.h.set_test(*test)
    else:
        (lu, mu), (lv, mv) = _fitting_hyper(U), _fitting_hyper(V)
        hyper = np.concatenate([lu.ravel(), mu, lv.ravel(), mv])
        s.h.set_state(U, V, hyper, it=IT0)
    return s


def _pairs(c, seed):
    g = _gen(seed, 1)
    return (torch.randint(0, c["M"], (c["pairs"],), generator=g, device="cuda", dtype=torch.int32),
            torch.randint(0, c["N"], (c["pairs"],), generator=g, device="cuda", dtype=torch.int32))


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "step":
        s.h.set_state(s.U0, s.V0, None, it=IT0)
        rmse = []
        for _ in range(c["iterations"]):
            s.h.step()
            rmse.append(s.h.test_rmse()[0])  # the running mean spans passes: not returned
        _, _, hyper, _ = s.h.get_state(s.U, s.V)
        # the draw rests on statistics summed in FP32
        return {"U": s.U, "V": s.V, "hyper": hyper.astype(np.float32), "rmse": np.array(rmse, np.float32)}
    if kind == "sweep":
        s.h.sweep(c["side"])
        s.h.get_state(s.U, s.V)
        return s.U if c["side"] == 0 else s.V
    if kind == "predict":
        return s.h.predict(s.row, s.col, s.out)
    if kind == "init":
        with bp.Sampler(c["M"], c["N"], *s.train, K=c["K"], alpha=c["alpha"], seed=7,
                        path=PATHS[c["path"]]) as h:
            sides = [h.structure(side) for side in (0, 1)]
            U, V, _, _ = h.get_state()
        return {"U": U, "V": V, "mean": np.float32(sides[0][4]),
                "ptr": [x[0] for x in sides], "idx": [x[1] for x in sides],
                "val": [x[2] for x in sides], "perm": [x[3] for x in sides]}
    ids = [s.server.submit(m, n, *train, k, c["iterations"], test=test, alpha=c["alpha"], seed=7 + j,
                           path=PATHS[c["path"]], want_factors=True)
           for j, (m, n, k, train, test) in enumerate(s.jobs)]
    out = []
    for i in ids:
        r, (U, V) = s.server.result(i)
        out.append({"U": U, "V": V, "rmse": np.array([r.rmse_sample, r.rmse_mean], np.float32)})
    return out


# -------------------------------------------------------------------- work --

def _side_work(R, C, nnz, K):
    """Half-sweep: symmetric Gram and right-hand side, Cholesky and solves; each input read once."""
    return (8 * nnz + 4 * K * C + R * (4 * K + 8),
            nnz * (K * (K + 1) + 2 * K) + R * (K ** 3 / 3 + 3 * K ** 2))


def _step_work(M, N, nnz, test, K):
    b, f = 0, 0
    for R, C in ((M, N), (N, M)):
        sb, sf = _side_work(R, C, nnz, K)
        b, f = b + sb + 4 * K * R, f + sf + R * (K * (K + 1) + 2 * K)  # the statistics read the rows once more
    return b + 20 * test, f + 2 * K * test


def work(case):
    c = case
    M, N, K, nnz = c["M"], c["N"], c["K"], c["nnz"]
    test = int(round(c["test"] * nnz))
    if c["kind"] == "step":
        b, f = _step_work(M, N, nnz - test, test, K)
        return {"bytes": c["iterations"] * b, "flops": c["iterations"] * f}
    if c["kind"] == "sweep":
        b, f = _side_work(*((M, N) if c["side"] == 0 else (N, M)), nnz - test, K)
        return {"bytes": b, "flops": f}
    if c["kind"] == "predict":
        # each factor row that some pair names, once; ids in, ratings out
        rows = sum(n * -math.expm1(c["pairs"] * math.log1p(-1.0 / n)) for n in (M, N))
        return {"bytes": 12 * c["pairs"] + 4 * K * rows, "flops": 2 * K * c["pairs"]}
    if c["kind"] == "init":
        return {"bytes": (12 + 2 * 8) * nnz + (M + N) * (4 * K + 12), "flops": 2 * nnz}
    b, f = 0, 0
    for m, n, z, k in _job_shapes(c):
        t = int(round(c["test"] * z))
        sb, sf = _step_work(m, n, z - t, t, k)
        b, f = b + c["iterations"] * sb + 12 * z, f + c["iterations"] * sf
    return {"bytes": b, "flops": f}


# ------------------------------------------------- the same in 64 bits --
# The conditionals of the model with the sampler's random streams
# (Philox4x32-10, Box-Muller, Marsaglia-Tsang), in FP64 by torch.

M32 = (1 << 32) - 1


def _mul32(a, b):
    """High and low words of the product of 32-bit words (a: tensor, b: int)."""
    lo = (a * (b & 0xFFFF)) + (((a * (b >> 16)) & 0xFFFF) << 16)
    hi = (a * (b >> 16) + ((a * (b & 0xFFFF)) >> 16)) >> 16
    return hi & M32, lo & M32


def _philox(c0, c1, c2, c3, seed):
    k0, k1 = seed & M32, seed >> 32
    c = [torch.as_tensor(x, dtype=torch.int64, device="cuda") for x in (c0, c1, c2, c3)]
    c = list(torch.broadcast_tensors(*c))
    for _ in range(10):
        ha, la = _mul32(c[0], 0xD2511F53)
        hb, lb = _mul32(c[2], 0xCD9E8D57)
        c = [hb ^ c[1] ^ k0, lb, ha ^ c[3] ^ k1, la]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _unit(x):
    return (2 * (x >> 9) + 1).double() * 2.0 ** -24


def _normal_pair(a, b):
    rad, ang = torch.sqrt(-2 * torch.log(_unit(a))), 2 * math.pi * _unit(b)
    return rad * torch.cos(ang), rad * torch.sin(ang)


def _normals(ids, t, stream, side, K, seed):
    """len(ids) x K normals: number k of id i is word pair (k % 4) / 2 of counter (i, t, k / 4)."""
    q = torch.arange((K + 3) // 4, device="cuda")
    w = _philox(ids[:, None], t, q[None], (stream << 8) | side, seed)
    z = torch.stack(_normal_pair(w[0], w[1]) + _normal_pair(w[2], w[3]), dim=-1)
    return z.reshape(len(ids), -1)[:, :K]


def _exact_hyper(X, side, t, seed):
    """Normal-Wishart posterior draw with mu0 = 0, beta0 = 2, nu0 = K, W0 = I."""
    n, K = X.shape
    eye = torch.eye(K, device="cuda", dtype=torch.float64)
    xbar = X.mean(0)
    d = X - xbar
    beta = 2.0 + n
    Winv = eye + d.T @ d + (2.0 * n / beta) * torch.outer(xbar, xbar)
    C = torch.linalg.cholesky(torch.linalg.inv(Winv))
    zero = torch.zeros(1, dtype=torch.int64, device="cuda")
    flat = _normals(zero, t, 2, side, K * (K - 1) // 2 or 1, seed)[0]
    A = torch.zeros(K, K, device="cuda", dtype=torch.float64)
    i, j = torch.tril_indices(K, K, -1, device="cuda")
    A[i, j] = flat[i * (i - 1) // 2 + j] if K > 1 else 0.0
    k = torch.arange(K, device="cuda")
    shape = 0.5 * (float(K) + n - k.double())
    dd = shape - 1.0 / 3.0
    cc = 1.0 / torch.sqrt(9.0 * dd)
    gam = torch.full_like(dd, -1.0)
    for a in range(64):
        w = _philox(k, t, a, (3 << 8) | side, seed)
        zn = _normal_pair(w[0], w[1])[0]
        v = (1.0 + cc * zn) ** 3
        ok = (v > 0) & (torch.log(_unit(w[2])) < 0.5 * zn * zn + dd - dd * v + dd * torch.log(v.clamp_min(1e-300)))
        gam = torch.where((gam < 0) & ok, dd * v, gam)
        if bool((gam >= 0).all()):
            break
    A[k, k] = torch.sqrt(2.0 * gam)
    B = C @ A
    lam = B @ B.T
    z = _normals(zero, t, 1, side, K, seed)[0]
    mu = n * xbar / beta + torch.linalg.solve_triangular(B.T, z[:, None], upper=True)[:, 0] / math.sqrt(beta)
    return lam, mu


def _csr(key, other, val, R):
    order = torch.sort(key, stable=True).indices
    deg = torch.bincount(key.long(), minlength=R)
    ptr = torch.zeros(R + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = deg.cumsum(0)
    return ptr, other[order].long(), val[order]


def _exact_rows(csr, R, Vo, lam, mu, alpha, t, side, seed):
    """Every row of a side: u = L^-T (L^-1 b + z), rows of like degree together."""
    ptr, idx, val = csr
    K = Vo.shape[1]
    deg, order = torch.sort(ptr[1:] - ptr[:-1], descending=True, stable=True)
    out = torch.empty(R, K, device="cuda", dtype=torch.float64)
    b0 = lam @ mu
    q = 0
    while q < R:
        D = max(1, int(deg[q]))
        B = max(1, min(R - q, int(4e9 / (8 * D * K)), int(2e9 / (8 * K * K))))
        rows = order[q:q + B]
        at = ptr[rows][:, None] + torch.arange(D, device="cuda")
        live = at < ptr[rows + 1][:, None]
        at = torch.where(live, at, torch.zeros_like(at))
        if idx.numel():
            x = Vo[idx[at]] * live[..., None]
            r = val[at] * live
        else:
            x = torch.zeros(B, D, K, device="cuda", dtype=torch.float64)
            r = torch.zeros(B, D, device="cuda", dtype=torch.float64)
        L = torch.linalg.cholesky(lam + alpha * (x.transpose(1, 2) @ x))
        b = b0 + alpha * (r[:, None] @ x)[:, 0]
        y = torch.linalg.solve_triangular(L, b[..., None], upper=False)
        z = _normals(rows, t, 0, side, K, seed)
        out[rows] = torch.linalg.solve_triangular(L.transpose(1, 2), y + z[..., None], upper=True)[..., 0]
        q += B
    return out


def _exact_chain(M, N, K, alpha, train, test, U, V, t0, iterations, seed):
    row, col, val = train
    mean = val.double().mean()
    r = val.double() - mean
    csr = [_csr(row, col, r, M), _csr(col, row, r, N)]
    X = [U.double(), V.double()]
    hy, rmse, total = [None, None], [], 0.0
    for t in range(t0, t0 + iterations):
        for side, R in ((0, M), (1, N)):
            hy[side] = _exact_hyper(X[side], side, t, seed)
            X[side] = _exact_rows(csr[side], R, X[1 - side], *hy[side], alpha, t, side, seed)
        pred = _dots(X[0], X[1], test[0], test[1]) + mean
        total = total + pred
        truth = test[2].double()
        rmse.append(((pred - truth) ** 2).mean().sqrt())
    mean_rmse = ((total / iterations - truth) ** 2).mean().sqrt()
    hyper = torch.cat([hy[0][0].reshape(-1), hy[0][1], hy[1][0].reshape(-1), hy[1][1]])
    return X, hyper, torch.stack(rmse), mean_rmse


def _seconds64(c):
    """About what the FP64 value takes."""
    f = 0.0
    for m, n, z, k in _job_shapes(c) if c["kind"] == "serve" else [(c["M"], c["N"], c["nnz"], c["K"])]:
        sides = [(n, m)[c["side"] == 0]] if c["kind"] == "sweep" else [m, n]
        f += sum(3.0 * z * k * k / 6e11 + R * k ** 3 / 1e11 for R in sides) * c["iterations"]
    return f


def exact(case, seed):
    c = case
    M, N, K = c["M"], c["N"], c["K"]
    if c["kind"] in ("step", "sweep", "serve") and _seconds64(c) > 15:
        return None
    if c["kind"] == "serve":
        out = []
        for j, (m, n, z, k) in enumerate(_job_shapes(c)):
            train, test, _, _ = _data(m, n, z, k, seed * 64 + j, c)
            U, V = (0.1 * _normals(torch.arange(R, device="cuda"), 0, 4, side, k, 7 + j)
                    for side, R in ((0, m), (1, n)))
            X, _, rmse, mean_rmse = _exact_chain(m, n, k, c["alpha"], train, test, U, V, 0, c["iterations"], 7 + j)
            out.append({"U": X[0], "V": X[1], "rmse": torch.stack([rmse[-1], mean_rmse])})
        return out
    train, test, U, V = _data(M, N, c["nnz"], K, seed, c)
    if c["kind"] == "step":
        X, hyper, rmse, _ = _exact_chain(M, N, K, c["alpha"], train, test, U, V, IT0, c["iterations"], 7)
        return {"U": X[0], "V": X[1], "hyper": hyper, "rmse": rmse}
    mean = train[2].double().mean()
    if c["kind"] == "sweep":
        key, other = (train[0], train[1]) if c["side"] == 0 else (train[1], train[0])
        R, X, Vo = (M, U, V) if c["side"] == 0 else (N, V, U)
        lam, mu = (torch.from_numpy(x).cuda() for x in _fitting_hyper(X))
        csr = _csr(key, other, train[2].double() - mean, R)
        return _exact_rows(csr, R, Vo.double(), lam, mu, c["alpha"], IT0, c["side"], 7)
    if c["kind"] == "predict":
        return _dots(U.double(), V.double(), *_pairs(c, seed)) + mean
    sides = [_csr(train[0], train[1], train[2].double() - mean, M),
             _csr(train[1], train[0], train[2].double() - mean, N)]
    X = [0.1 * _normals(torch.arange(R, device="cuda"), 0, 4, side, K, 7) for side, R in ((0, M), (1, N))]
    return {"U": X[0], "V": X[1], "mean": mean, "ptr": [None, None], "idx": [None, None],
            "val": [x[2] for x in sides], "perm": [None, None]}
