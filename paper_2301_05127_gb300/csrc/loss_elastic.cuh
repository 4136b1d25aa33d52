// Pointwise pieces shared by the 3-D elastic kernels.
#pragma once

#include <cuda_runtime.h>

#include "loss_line.cuh"
#include "loss_types.h"

namespace lossk {

// tau times the (stretched) derivative g along this pass's axis at line position pos.
template <typename T>
__device__ __forceinline__ T eff(int pml, const PmlAxis<T>& pa, T* mem, int64_t gi, int pos, T g, T tau, T tau_lo) {
  return (pml && pa.in(pos)) ? -pa.step(mem, gi, pos, g) : mulc(g, tau, tau_lo);
}

// Velocity-sub-step term: returns tau * (stretched derivative); in a layer with receiver corrections on, also
// stores b (X(tau/2) - X(tau)/2), the amount by which the first half of the step differs from half of it.
template <typename T>
__device__ __forceinline__ T effA(const ElArgs<T>& a, int term, int64_t gi, int pos, T g, T tau) {
  if (!(a.pml && a.pA.in(pos))) return mulc(g, tau, a.acoef_lo);
  T xh = T(0);
  const bool rec = a.dlt[term] != nullptr;
  if (rec) xh = -a.pA.half(a.memA[term], gi, pos, g);
  const T xf = -a.pA.step(a.memA[term], gi, pos, g);
  if (rec) a.dlt[term][gi] = (a.b ? a.b[gi] : a.b0) * (xh - T(0.5) * xf);
  return xf;
}

// u += delta in registers (compensated with c when KAHAN); the caller loads and stores.
template <typename T, bool KAHAN>
__device__ __forceinline__ void upd_r(T& u, T& c, T delta) {
  if constexpr (KAHAN) {
    float cc = c;
    kahan_add(u, cc, delta);
    c = cc;
  } else {
    u += delta;
  }
}

}  // namespace lossk
