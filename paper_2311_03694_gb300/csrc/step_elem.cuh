// BDFk/EXTk coefficients and the per-element diagonal step (Sec. 2.2,
// eq. nse_d1), shared by the step kernels.  Each translation unit that
// includes this gets its own copy of the constant tables.
#pragma once

#include "grom_internal.h"

namespace grom {

// beta_0 .. beta_k of BDFk and alpha_1 .. alpha_k of EXTk, k = 1, 2, 3
static __constant__ double c_beta[3][4] = {
    {1.0, -1.0, 0.0, 0.0},
    {1.5, -2.0, 0.5, 0.0},
    {11.0 / 6.0, -3.0, 1.5, -1.0 / 3.0},
};
static __constant__ double c_alpha[3][3] = {
    {1.0, 0.0, 0.0},
    {2.0, -1.0, 0.0},
    {3.0, -3.0, 1.0},
};

// EXTk of the newest k advection terms, g[0] the newest: g0, 2 g0 - g1 or
// 3 (g0 - g1) + g2, in at most two FP64 operations.
__device__ __forceinline__ double step_ext(int k, const double (&g)[3]) {
  return k == 1 ? g[0] : k == 2 ? fma(2.0, g[0], -g[1]) : fma(3.0, __dsub_rn(g[0], g[1]), g[2]);
}

// u^{l+1}_i of the plain diagonal step (identity mass): the BDF terms chained
// onto the extrapolation, six FP64 operations at order 3.
__device__ __forceinline__ double step_plain_elem(const double (&bdt)[3], int k, const double (&u)[3],
                                                  const double (&g)[3], double hd) {
  double y;
  if (k == 3) {  // uniform: no predicated-off FP64 instruction on the usual way
    y = fma(3.0, __dsub_rn(g[0], g[1]), g[2]);
    y = fma(bdt[2], u[2], y);
    y = fma(bdt[1], u[1], y);
  } else {
    y = step_ext(k, g);
    if (k == 2) y = fma(bdt[1], u[1], y);
  }
  y = fma(bdt[0], u[0], y);
  return __dmul_rn(-y, hd);
}

__device__ __forceinline__ int step_is_bad(double un) {  // inf or NaN, from the exponent bits
  return ((__double_as_longlong(un) >> 52) & 0x7FF) == 0x7FF;
}

// One element of the diagonal step: u^{l+1}_i from the history and n^l_i = nl.
// FP64 runs at about two operations per clock per SM on this part, so the
// terms of absent operators (mass, linear, forcing: null pointers, uniform
// branches) are skipped, beta/dt comes from the host, the energy and
// invariant terms are formed only when `sums` is set, and finiteness is
// read from the exponent bits: six FP64 operations per element in the common
// case.  PLAIN (no mass, linear or forcing term, no sums) removes
// those terms at compile time: a runtime test still issues its predicated
// FP64 instructions, which measured ~26 FP64 instructions per element on the
// batched step.
// The operands other than the newest advection term are loaded by step_load,
// which the kernels call before they sum that term, so that both loads' latencies
// pass together; a lower order leaves some unused.
struct StepElem {
  double u[3], g[3], hd, mb, ld, f;
};
// (ALL false: only the ones of order k.)
template <bool PLAIN = false, bool ALL = true>
__device__ __forceinline__ StepElem step_load(const StepArgs& a, const double* h, int64_t n, int64_t l, int k,
                                              int64_t i) {
  StepElem x;
  const int m0 = (int)(l % 3);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int m = m0 - q < 0 ? m0 - q + 3 : m0 - q;
    x.u[q] = x.g[q] = 0.0;
    if (ALL || q < k) {
      x.u[q] = h[m * n + i];
      if (q > 0) x.g[q] = h[(3 + m) * n + i];
    }
  }
  x.hd = a.hdiag[k - 1][i];
  x.mb = !PLAIN && a.mass_diag ? a.mass_diag[i] : 1.0;
  x.ld = !PLAIN && a.lin_diag ? a.lin_diag[i] : 0.0;
  x.f = !PLAIN && a.forcing ? a.forcing[i] : 0.0;
  return x;
}
template <bool PLAIN = false>
__device__ __forceinline__ double step_elem(const StepArgs& a, double* h, int64_t n, int64_t l, int k, int64_t i,
                                            const StepElem& x, double nl, double& e_part, double& i_part, int& bad,
                                            bool sums = true) {
  const bool mass = !PLAIN && a.mass_diag != nullptr;
  const bool lin = !PLAIN && a.lin_diag != nullptr;
  const bool frc = !PLAIN && a.forcing != nullptr;
  double g[3] = {nl, x.g[1], x.g[2]};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (lin) g[q] = fma(x.ld, x.u[q], g[q]);
    if (frc) g[q] += x.f;
  }
  double un;
  if (mass) {
    double bdf = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (q < k) bdf = fma(a.bdt[k - 1][q], x.u[q], bdf);
    un = fma(-x.mb, bdf, -step_ext(k, g)) * x.hd;
  } else {
    un = step_plain_elem(a.bdt[k - 1], k, x.u, g, x.hd);
  }
  e_part = 0.0;
  i_part = 0.0;
  if (sums) {
    // explicit roundings: the products must not contract into the caller's
    // sums (FMA), whose form would then depend on the kernel inlining them
    e_part = mass ? __dmul_rn(__dmul_rn(x.mb, un), un) : __dmul_rn(un, un);
    i_part = __dmul_rn(x.u[0], nl);
  }
  bad = step_is_bad(un);
  h[((l + 1) % 3) * n + i] = un;
  return un;
}

// Called by all lanes of one warp of the last block of trajectory b to
// arrive: sums the nblk per-block (energy, invariant) partials (lane q adds
// blocks q, q+32, ... in order, then a fixed shuffle tree), writes the outputs
// and advances the step count.
__device__ __forceinline__ void step_finish_last(const StepArgs& a, int b, int64_t l, int step_index) {
  const int lane = threadIdx.x & 31;
  __threadfence();
  double e = 0.0, inv = 0.0;
  const double* rr = a.red + (int64_t)b * a.nblk * 2;
  const int nsum = (a.energy || a.invariant) ? a.nblk : 0;  // no sums asked for: only the step count
  for (int q = lane; q < nsum; q += 32) {
    e += __ldcg(rr + 2 * q);
    inv += __ldcg(rr + 2 * q + 1);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, off);
    inv += __shfl_xor_sync(0xffffffffu, inv, off);
  }
  if (lane == 0) {
    if (a.energy) a.energy[(int64_t)step_index * a.batch + b] = 0.5 * e;
    if (a.invariant) a.invariant[(int64_t)step_index * a.batch + b] = inv;
    step_done(a, b, l);
    a.cnt[b] = 0u;
  }
}

}  // namespace grom
