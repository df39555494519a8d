"""The memory that building a sampler needs at its peak.

The scratch of the structure (28 bytes a rating and more) is not needed beside
the partial Grams of split rows, the largest allocation after it: a device with
room for the sampler and the larger of the two is enough.  Here the free memory
is cut down to that, and half of the smaller on top.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_scratch_is_released_before_the_pieces_are_taken(gpu_lib):
    import torch

    bp = gpu_lib
    M, N, K, hub = 20_000, 2_000, 128, 512
    nnz = M * N
    row = torch.arange(M, device="cuda", dtype=torch.int32).repeat_interleave(N)
    col = torch.arange(N, device="cuda", dtype=torch.int32).repeat(M)
    val = torch.randn(nnz, device="cuda")
    bp.Sampler(4, 4, [0], [0], [1.0], K=K).close()  # modules loaded
    torch.cuda.synchronize()

    def free():
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    before = free()
    s = bp.Sampler(M, N, row, col, val, K=K, path=bp.PATH_BINNED, hub_min=hub)
    held = before - free()
    s.close()
    scratch = 16 * nnz  # device triples: the sort's four arrays, at least
    assert held > 3 * scratch
    filler = torch.empty(free() - held - scratch // 2, dtype=torch.uint8, device="cuda")
    with bp.Sampler(M, N, row, col, val, K=K, path=bp.PATH_BINNED, hub_min=hub) as s:
        assert s.sweep_info(0)[0][3] == M
    del filler
