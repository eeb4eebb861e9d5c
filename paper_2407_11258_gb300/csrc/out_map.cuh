// Device-side addressing of a contraction's destination (OutMap, internal.h).
#pragma once
#include "internal.h"

namespace lnocc {

__device__ __forceinline__ long long out_moff(const OutMap& C, int m) {
  const int m0 = m % C.mdiv, mm = m / C.mdiv;
  const int m1 = mm % C.mdiv1, m2 = mm / C.mdiv1;
  return m2 * C.sm2 + m1 * C.sm1 + static_cast<long long>(m0) * C.sm0;
}
__device__ __forceinline__ long long out_noff(const OutMap& C, int n) {
  const int n0 = n % C.ndiv, nn = n / C.ndiv;
  const int n1 = nn % C.ndiv1, n2 = nn / C.ndiv1;
  return n2 * C.sn2 + n1 * C.sn1 + static_cast<long long>(n0) * C.sn0;
}

}  // namespace lnocc
