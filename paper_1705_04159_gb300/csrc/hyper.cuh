// hyper.cuh -- arguments of the Normal-Wishart draw (wishart.cu), called from hyper.cu.
#pragma once

#include "bpmf_impl.cuh"

namespace gb {

struct HyperArgs {
  const double* xbar;
  const double* S;
  int64_t n;
  const double* mu0;
  double beta0, nu0;
  double wmean;  // beta0 n / (beta0 + n)
  const double* W0inv;
  uint64_t seed;
  const uint32_t* tp;  // iteration word on the device
  int side;
  int K;
  double* scr;  // 6 K*K + 2 K doubles
  double* lam;
  double* mu;
  float* lamaug;
  float* lchol;  // chol(Lambda) = B in FP32, packed by rows, for the rank-one row kernel
  int* status;
  int gamma_cap;  // Gamma rejection attempts per draw before kStatusRng
};

// the whole draw: one kernel, one cluster of `ctas` CTAs (wish_cluster)
int launch_wishart(const HyperArgs& a, int ctas, cudaStream_t st, int64_t* launches);

}  // namespace gb
