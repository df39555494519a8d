"""The Normal-Wishart draw and W0^-1 on clusters of every size.

For K > 32 they take a cluster of 16 CTAs where the device has one, which is past
the portable size; where it has not (a partition of the GPU) the largest half
that fits, down to two, the warps taking their columns in rounds.  The arithmetic
of a column or a row is the same wherever it runs, so all sizes must agree bit for
bit.  wishart.cu is compiled on its own here, with the cluster's size as an
argument.
"""
import ctypes as C
import importlib
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HARNESS = r"""
#include "wishart.cu"
namespace gb {
void set_error(const char*, ...) {}
}
#define OUT extern "C" __attribute__((visibility("default")))
OUT int largest(int K) {
  int n = 0;
  return gb::wish_cluster(K, &n) == BPMF_OK ? n : -1;
}
OUT int inverse(int K, int ctas, const double* A, double* Ainv, double* scr, int* status) {
  const int rc = gb::launch_spd_inverse_f64(A, Ainv, K, ctas, scr, status, nullptr);
  return rc != BPMF_OK ? rc : (int)cudaDeviceSynchronize();
}
OUT int draw(int K, int ctas, long long n, const double* xbar, const double* S, const double* mu0,
             const double* W0inv, const uint32_t* iter, double* scr, double* lam, double* mu, float* lamaug,
             float* lchol, int* status) {
  gb::HyperArgs a;
  a.xbar = xbar; a.S = S; a.n = n; a.mu0 = mu0; a.beta0 = 2.0; a.nu0 = K; a.wmean = 2.0 * n / (2.0 + n);
  a.W0inv = W0inv; a.seed = 5; a.tp = iter; a.side = 1; a.K = K; a.scr = scr; a.lam = lam; a.mu = mu;
  a.lamaug = lamaug; a.lchol = lchol; a.status = status; a.gamma_cap = gb::kGammaCap;
  const int rc = gb::launch_wishart(a, ctas, nullptr, nullptr);
  return rc != BPMF_OK ? rc : (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def harness(gpu_lib, tmp_path_factory):
    build = importlib.import_module("paper_1705_04159_gb300.build")
    d = tmp_path_factory.mktemp("cluster")
    (d / "harness.cu").write_text(HARNESS)
    so = d / "harness.so"
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(so), str(d / "harness.cu")],
                   check=True, capture_output=True)
    return C.CDLL(str(so))


@pytest.mark.parametrize("K", [1, 10, 16, 17, 32, 33, 64, 65, 97, 128])
def test_every_size_gives_the_same_bits(harness, K):
    import torch

    rng = np.random.default_rng(K)
    q = np.linalg.qr(rng.normal(size=(K, K)))[0]
    W0 = (q * np.linspace(0.5, 2.5, K)) @ q.T
    W0 = 0.5 * (W0 + W0.T)
    x = rng.normal(size=(300, K))
    xbar = x.mean(0)
    S = (x - xbar).T @ (x - xbar)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def p(t):
        return C.c_void_p(t.data_ptr())

    dW0, dx, dS, dm = dev(W0), dev(xbar), dev(S), dev(np.zeros(K))
    it = dev(np.array([3], np.int32))
    most = harness.largest(K)
    assert most >= 2
    got = {}
    n = most
    while n >= 2:
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        scr = torch.full((6 * K * K + 8 * K,), float("nan"), dtype=torch.float64, device="cuda")
        inv = torch.full((K, K), float("nan"), dtype=torch.float64, device="cuda")
        assert harness.inverse(K, n, p(dW0), p(inv), p(scr), p(status)) == 0
        scr.fill_(float("nan"))
        lam = torch.full((K, K), float("nan"), dtype=torch.float64, device="cuda")
        mu = torch.full((K,), float("nan"), dtype=torch.float64, device="cuda")
        aug = torch.full((K + 1, K + 1), float("nan"), device="cuda")
        chol = torch.full((K * (K + 1) // 2,), float("nan"), device="cuda")
        assert harness.draw(K, n, C.c_longlong(300), p(dx), p(dS), p(dm), p(inv), p(it), p(scr), p(lam), p(mu),
                            p(aug), p(chol), p(status)) == 0
        assert int(status) == 0
        got[n] = [t.cpu().numpy() for t in (inv, lam, mu, aug, chol)]
        n //= 2
    for out in got.values():
        for a, b in zip(out, got[most]):
            assert np.all(np.isfinite(a)) and np.array_equal(a, b)
    assert np.max(np.abs(got[most][0] @ W0 - np.eye(K))) <= 1e-11
