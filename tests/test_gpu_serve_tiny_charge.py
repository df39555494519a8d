"""A job none of whose rows with ratings can be tiny is not charged for the tiny
rows' products, a buffer as large as the other side's factors: the charge decides
which jobs a server's budget admits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _job(M, N, nnz, seed=1):
    rng = np.random.default_rng(seed)
    cell = np.unique(rng.integers(0, M * N, nnz))
    return (cell // N).astype(np.int32), (cell % N).astype(np.int32), rng.normal(size=cell.size).astype(np.float32)


def _charged(bp, M, N, data, K, **cfg):
    with bp.Server(max_resident=1) as srv:
        r, _ = srv.result(srv.submit(M, N, *data, K, 1, **cfg))
        assert r.status == 0
        return r.device_bytes


def test_no_charge_for_products_that_no_row_takes(gpu_lib):
    bp = gpu_lib
    M, N, K = 300_000, 100_000, 64
    data = _job(M, N, 900_000)
    plain = _charged(bp, M, N, data, K, path=bp.PATH_BINNED)  # tiny rows: those without ratings
    tiny = _charged(bp, M, N, data, K, path=bp.PATH_BINNED, tiny_max=8)
    # the products of a row of the other side are K rounded up to 32 floats
    assert tiny - plain >= M * 64 * 4
