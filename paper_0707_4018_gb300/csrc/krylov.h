// Host side of one restart cycle of a flexible GCR whose solution is formed at its end.
//
// With z_k the preconditioned vectors and w_k = A z_k made orthonormal, A Z = W R (R upper triangular:
// the Gram-Schmidt coefficients, 1 / |w_hat_k| on the diagonal) and the cycle removes sum_k alpha_k w_k
// from the residual, so x += Z y with R y = alpha. Only the w_k are orthogonalised: carrying the z_k
// along took as many FP64 multiply-adds again, which is what bounds the update.
#pragma once

#include <complex>
#include <vector>

namespace mg {

class KrylovCycle {
 public:
  explicit KrylovCycle(int restart = 0) : cap_(restart), r_((size_t)restart * restart), alpha_(restart) {}
  void reset() { used_ = 0; }
  // column k starts (its entries above the diagonal zero)
  void open(int k) {
    for (int j = 0; j < k; ++j) r_[(size_t)k * cap_ + j] = 0.0;
  }
  // w_k was projected with beta (k complex numbers)
  void project(int k, const double *beta) {
    for (int j = 0; j < k; ++j) r_[(size_t)k * cap_ + j] += std::complex<double>(beta[2 * j], beta[2 * j + 1]);
  }
  // w_k scaled by inv, alpha its coefficient in the residual
  void close(int k, double inv, double are, double aim) {
    r_[(size_t)k * cap_ + k] = 1.0 / inv;
    alpha_[k] = {are, aim};
    used_ = k + 1;
  }
  int columns() const { return used_; }
  // y (columns() complex numbers as pairs) with R y = alpha
  void solution(double *y) const {
    std::vector<std::complex<double>> t(alpha_.begin(), alpha_.begin() + used_);
    for (int k = used_ - 1; k >= 0; --k) {
      t[k] /= r_[(size_t)k * cap_ + k];
      for (int j = 0; j < k; ++j) t[j] -= r_[(size_t)k * cap_ + j] * t[k];
      y[2 * k] = t[k].real();
      y[2 * k + 1] = t[k].imag();
    }
  }

 private:
  int cap_, used_ = 0;
  std::vector<std::complex<double>> r_, alpha_;
};

}  // namespace mg
