"""The device bytes a job is charged against what its sampler holds.

The charge is an upper estimate of what bpmf_init and the iterations hold, so it
may not be below what a sampler of the same job takes, seen from outside by the
free memory before and after.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _job(M, N, nnz, seed=1):
    rng = np.random.default_rng(seed)
    cell = np.unique(rng.integers(0, M * N, nnz))
    return (cell // N).astype(np.int32), (cell % N).astype(np.int32), rng.normal(size=cell.size).astype(np.float32)


def _charged(bp, M, N, data, K, test=None, **cfg):
    with bp.Server(max_resident=1) as srv:
        r, _ = srv.result(srv.submit(M, N, *data, K, 1, test=test, **cfg))
        assert r.status == 0
        return r.device_bytes


def _held(bp, M, N, data, K, test=None, **cfg):
    import torch

    bp.Sampler(10, 10, [0], [0], [1.0], K=K).close()  # modules loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    with bp.Sampler(M, N, *data, K=K, **cfg) as s:
        if test is not None:
            s.set_test(*test)
        s.step()
        return before - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("M,N,nnz,n_test,K,cfg", [
    (400_000, 200_000, 300_000, 0, 100, dict(path=2)),                # factors and shadows
    (400_000, 200_000, 300_000, 0, 100, dict(path=1)),
    (600_000, 300_000, 2_500_000, 0, 128, dict(path=2, tiny_max=8)),  # tiny rows' products
    (2_000, 1_000, 400_000, 0, 128, dict(path=2, hub_min=16)),        # pieces of eight ratings
    (2_000, 1_000, 300_000, 5_000_000, 16, dict(path=1)),             # a large test set
])
def test_charge_covers_what_is_held(gpu_lib, M, N, nnz, n_test, K, cfg):
    bp = gpu_lib
    data = _job(M, N, nnz)
    test = None
    if n_test:
        rng = np.random.default_rng(2)
        test = (rng.integers(0, M, n_test).astype(np.int32), rng.integers(0, N, n_test).astype(np.int32),
                rng.normal(size=n_test).astype(np.float32))
    held = _held(bp, M, N, data, K, test, **cfg)
    charged = _charged(bp, M, N, data, K, test, **cfg)
    assert charged >= held, (charged, held)
