// The row updates of one inner iteration of Algorithm 1, shared by every
// iteration kernel (row-block, pipelined, member-interleaved, one-launch
// chunk), so that their iterates agree bit for bit.
#pragma once

#include "common.cuh"

namespace pdqp {

template <typename V> __device__ __forceinline__ V step_sigma(const StepEntry& e);
template <> __device__ __forceinline__ double step_sigma<double>(const StepEntry& e) { return e.sigma_d; }
template <> __device__ __forceinline__ float step_sigma<float>(const StepEntry& e) { return e.sigma_d_f; }
template <typename V> __device__ __forceinline__ V step_tau(const StepEntry& e);
template <> __device__ __forceinline__ double step_tau<double>(const StepEntry& e) { return e.tau_p; }
template <> __device__ __forceinline__ float step_tau<float>(const StepEntry& e) { return e.tau_p_f; }
template <typename V> __device__ __forceinline__ V step_ib(const StepEntry& e);
template <> __device__ __forceinline__ double step_ib<double>(const StepEntry& e) { return e.inv_beta; }
template <> __device__ __forceinline__ float step_ib<float>(const StepEntry& e) { return e.inv_beta_f; }
template <typename V> __device__ __forceinline__ V step_ibn(const StepEntry& e);
template <> __device__ __forceinline__ double step_ibn<double>(const StepEntry& e) { return e.inv_beta_next; }
template <> __device__ __forceinline__ float step_ibn<float>(const StepEntry& e) { return e.inv_beta_next_f; }
template <typename V> __device__ __forceinline__ V step_thn(const StepEntry& e);
template <> __device__ __forceinline__ double step_thn<double>(const StepEntry& e) { return e.theta_next; }
template <> __device__ __forceinline__ float step_thn<float>(const StepEntry& e) { return e.theta_next_f; }


// The dual update of one row from its sum s = (A x_tilde)_r: y+ and y_bar+
// (shared by the row-block and the member-interleaved kernels).
template <typename V>
__device__ __forceinline__ void dual_update(V sigma, V ib, V s, V yo, V bi, V yb, V lo, bool ineq, V& yn, V& ybn) {
  yn = r_fma(-sigma, r_sub(s, bi), yo);                       // y - sigma (A x_tilde - b)
  if (ineq) yn = fmax(yn, lo);
  ybn = r_fma(ib, yn, r_mul(r_sub(V(1), ib), yb));            // (1 - 1/beta) y_bar + y+/beta
}

template <typename V>
__device__ __forceinline__ void dual_update(const StepEntry& e, V s, V yo, V bi, V yb, V lo, bool ineq, V& yn,
                                            V& ybn) {
  dual_update<V>(step_sigma<V>(e), step_ib<V>(e), s, yo, bi, yb, lo, ineq, yn, ybn);
}

// The primal update of one row from g = (Q x_md - A'y+)_r + c_r (+ the
// low-rank term): x+, x_bar+ and the next iteration's x_md and x_tilde
// (shared by the row-block and the member-interleaved kernels).
template <typename V>
__device__ __forceinline__ void primal_update(V tau, V ib, V ibn, V thn, V g, V xo, V xb0, V lr, V ur, V& xn, V& xb,
                                              V& zo, V& xtn) {
  xn = fmin(fmax(r_fma(-tau, g, xo), lr), ur);               // proj_X(x - tau g)
  xb = r_fma(ib, xn, r_mul(r_sub(V(1), ib), xb0));            // (1 - 1/beta) x_bar + x+/beta
  zo = r_fma(ibn, xn, r_mul(r_sub(V(1), ibn), xb));           // next x_md
  xtn = r_fma(thn, r_sub(xn, xo), xn);                        // next x_tilde
}

template <typename V>
__device__ __forceinline__ void primal_update(const StepEntry& e, V g, V xo, V xb0, V lr, V ur, V& xn, V& xb, V& zo,
                                              V& xtn) {
  primal_update<V>(step_tau<V>(e), step_ib<V>(e), step_ibn<V>(e), step_thn<V>(e), g, xo, xb0, lr, ur, xn, xb, zo, xtn);
}

}  // namespace pdqp
