"""How many rows one FP32 accumulator of the centred scatter sums.

The sums move to FP64 at least every 512 rows of an accumulator (K > 32; 1,024
for K <= 32).  To count them, column 0 holds 4,096 in the first row of every
accumulator of a block and +-1 in its other rows, so that the accumulator starts
at 2^24 and every later square, 1, is lost to rounding until the next move.  The
rest is zero and the mean is exactly 0.  So at most bound - 1 ones are lost per
accumulator, and S[0, 0] is exact otherwise: every sum of what is left is a
whole number below 2^53, and the few accumulators of a block that meet in FP32
are multiples of 2^24 until the move and small whole numbers after it.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,subsets,chunk,bound", [
    (1, 288, 32, 1024), (2, 96, 32, 1024), (8, 28, 32, 1024), (32, 8, 32, 1024),
    (33, 17, 64, 512), (48, 12, 64, 512), (64, 7, 64, 512), (72, 6, 64, 512), (128, 2, 64, 512)])
def test_rows_of_an_accumulator(gpu_lib, K, subsets, chunk, bound):
    import torch

    bp = gpu_lib
    # one subset's rows of a chunk: 0, subsets, 2 subsets, ..
    per_chunk = (chunk + subsets - 1) // subsets
    chunks = 2 * bound // per_chunk + 2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = min((262144 - 128) // (K * K), 2 * sms)
    R = blocks * chunks * chunk  # every block the same rows
    block = torch.zeros(chunks, chunk)
    used = torch.zeros(chunks, chunk, dtype=torch.bool)
    used[:, ::subsets] = True
    n = int(used.sum())
    ones = torch.ones(n)
    ones[1::2] = -1.0
    block[used] = ones
    block[0, 0] = 4096.0
    X = torch.zeros(blocks, chunks * chunk, K, device="cuda")
    X[:, :, 0] = block.reshape(-1).cuda()
    X[1::2, :, 0] *= -1.0  # blocks of both signs: the mean is 0
    if blocks % 2:
        X[-1] = 0.0
        blocks -= 1
    xbar = torch.zeros(K, dtype=torch.float64, device="cuda")
    S = torch.zeros(K * K, dtype=torch.float64, device="cuda")
    bp.bpmf_hyper_stats_noalloc(X.reshape(R, K), R, K, xbar, S)
    torch.cuda.synchronize()
    assert float(xbar[0]) == 0.0
    per_block = float(S[0]) / blocks
    exact = 2.0 ** 24 + (n - 1)
    assert exact - (bound - 1) <= per_block <= exact, (per_block - exact, bound)
    S[0] = 0.0
    assert float(S.abs().max()) == 0.0
