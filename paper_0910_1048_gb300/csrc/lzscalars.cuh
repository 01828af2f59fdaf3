// Scalars that end a two-sided Lanczos step, shared by the kernels that finish it.
#pragma once

#include "devutil.cuh"
#include "kernels.h"

namespace ovl {

struct BetaVals {
  bool ok;    // false: breakdown (or a non-finite value)
  double d;   // delta_j
  double id;  // 1/delta_j = sv_{j+1}
  zd bt;      // beta_j
  zd swv;     // 1/conj(beta_j) = sw_{j+1}
  double vn;  // |v_{j+1}|
};

__device__ __forceinline__ BetaVals lz_beta_vals(const double (&sums)[4]) {
  // few FP64 operations in one dependent chain (each is slow on this GPU's FP64 pipe): with
  // r = |ip|^-1 and id = r^(1/2) = 1/delta_j, delta_j = |ip| id, beta_j = id ip, and
  // 1/conj(beta_j) = beta_j / |beta_j|^2 = id r ip (|beta_j|^2 = |ip|); the breakdown test on squares
  BetaVals b{};
  const zd ip = mk(sums[0], sums[1]);
  const double n2 = norm2(ip);
  b.ok = (n2 > 1e-28 * (sums[2] * sums[3])) && (n2 <= 1.7976931348623157e308);
  if (!b.ok) return b;
  const double r = rsqrt(n2), id = sqrt(r), idp = id * r;
  b.id = id;
  b.d = n2 * r * id;  // |ip| / delta_j = delta_j
  b.bt = id * ip;
  b.swv = mk(idp * ip.re, idp * ip.im);
  b.vn = sqrt(sums[2]) * id;
  return b;
}

// Stores the values of step j (b.ok) or marks the breakdown.
__device__ __forceinline__ void lz_beta_store(const LzDev& lz, int rhs, size_t o, int j, const BetaVals& b) {
  if (!b.ok) {
    lz.status[rhs] = 1;
    return;
  }
  lz.delta[o + j] = b.d;
  lz.beta[o + j] = make_double2(b.bt.re, b.bt.im);
  lz.sv[o + j + 1] = b.id;
  lz.sw[o + j + 1] = make_double2(b.swv.re, b.swv.im);
  lz.vnorm[o + j + 1] = b.vn;
}

}  // namespace ovl
