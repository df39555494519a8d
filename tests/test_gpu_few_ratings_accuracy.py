"""Rows of few ratings and a small latent dimension against FP64, beside what FP32
multiply-adds give, as test_gpu_fp32_accuracy.py has it for large ones: here an
operand's last bit shows, which its two TF32 parts do not keep.  At and about the
sizes where the Gram goes from multiply-adds to the tensor cores: 16 ratings of a
row, 64 of a piece, K = 15 and 23.
"""
import pytest

from test_gpu_fp32_accuracy import rms_error

pytestmark = pytest.mark.gpu

# (K, ratings of a row, hub_min or 0): rms error of FP32 multiply-adds
BASE = {
    (1, 1, 0): 1.00e-07, (2, 2, 0): 1.26e-07, (3, 4, 0): 1.73e-07, (4, 9, 0): 1.94e-07,
    (7, 2, 0): 1.90e-07, (8, 3, 0): 2.21e-07, (10, 2, 0): 2.01e-07, (10, 16, 0): 3.05e-07,
    (10, 17, 0): 2.99e-07, (16, 3, 0): 2.42e-07, (20, 2, 0): 2.35e-07, (23, 4, 0): 3.19e-07,
    (24, 4, 0): 3.02e-07, (32, 3, 0): 2.95e-07, (55, 8, 0): 4.95e-07, (1, 400, 50): 1.30e-07,
    (8, 400, 50): 1.59e-07, (8, 400, 129): 1.63e-07, (16, 400, 50): 1.87e-07,
}


@pytest.mark.parametrize("K,d,hub", sorted(BASE))
def test_no_further_from_fp64_than_multiply_adds(gpu_lib, K, d, hub):
    assert rms_error(gpu_lib, K, d, hub) <= 1.05 * BASE[K, d, hub]
