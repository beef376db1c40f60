// What a pivoted Cholesky factorisation (kernels.cu) reports, and what its callers make of it.
// Plain C++: read on the host, tested without a GPU.
#pragma once

namespace mpdo {

constexpr int kPcholGaveUp = -1;   // rank reported when a wait inside the kernel gave up
struct PcholOut {
  int r;
  int pad;
  double resid;   // largest remaining diagonal / trace
};
enum class PcholFit {
  fits,   // r columns represent the matrix
  zero,   // nothing to factor: a zero or non-finite matrix
  full    // more columns than rmax, or no factor at all: the caller solves the full problem
};
inline PcholFit pchol_fit(const PcholOut& o, int n, int rmax, double tol) {
  if (o.r == kPcholGaveUp) return PcholFit::full;
  if (o.r < 1) return PcholFit::zero;
  return o.r >= rmax && o.r < n && o.resid > tol ? PcholFit::full : PcholFit::fits;
}

}  // namespace mpdo
