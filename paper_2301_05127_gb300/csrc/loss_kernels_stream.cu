// sm_103a kernels of the 3-D elastic step on the barrier-free engines of loss_stream.cuh (FP32 and FP64).
//
// Passes of one step (X[f,a] and Y[f,a] as in loss_kernels_elastic.cu):
//   ES_BX (rows along x):  TA = X[v1,x], TB = X[v2,x], TC = X[v3,x]
//   ES_BY (y lines):       TB += X[v1,y], TD = X[v2,y], TE = X[v3,y]
//   ES_BZ (z lines):       the stress update from TA..TE and X[v1..v3, z], + source      [sub-step B]
//   ES_AZ (z lines):       UA = Y[s13,z], UB = Y[s23,z], UC = Y[s33,z]
//   ES_AX (rows along x):  UA += Y[s11,x], UB += Y[s12,x], UC += Y[s13,x]
//   ES_AY (y lines):       v_i += b (U_i + Y[s_i2, y]), + body force                     [sub-step A]
#include <cuda_runtime.h>

#include "../../include/loss.h"
#include "loss_elastic.cuh"
#include "loss_host.h"
#include "loss_stream.cuh"
#include "loss_types.h"

namespace lossk {

// REC: the receiver corrections of the three velocity terms are kept (dlt and the half-step tables are set).  Pointers
// that a launch may lack are only named under template parameters or replaced by readable ones.
template <typename T, int PASS, bool KAHAN, bool REC>
struct ElColOp {
  static constexpr int NF = 3;
  static constexpr bool SECOND = false;
  static constexpr int kBlocks = sizeof(T) == 4 ? 4 : 1;
  static constexpr int B = PASS == ES_AZ || PASS == ES_BY ? 4 : 2;
  ElArgs<T> a;
  int lam_on, mu_on, b_on;  // the coefficient is an array (its pointer is a readable one either way)
  struct Regs {
    T u[PASS == ES_BZ ? 6 : (PASS == ES_AY ? 3 : 1)], c[PASS == ES_BZ ? 6 : (PASS == ES_AY ? 3 : 1)];
    T t[PASS == ES_BZ ? 5 : (PASS == ES_AY ? 3 : 1)], m0, m1;
    T m[3];  // the memory variables of the three terms (layers only)
  };
  __device__ __forceinline__ const T* src(int f) const { return a.src[f]; }
  __device__ __forceinline__ T source_at(int dz, int dy, int dx) const {
    return (T)(a.srcp.amp * a.srcp.g[min((unsigned)dz, 24u)] * a.srcp.g[min((unsigned)dy, 24u)] *
               a.srcp.g[min((unsigned)dx, 24u)]);
  }
  static __device__ __forceinline__ constexpr int stress(int i) {  // the six stresses in the order of the updates below
    return i == 0 ? LOSS_FIELD_S11 : (i == 1 ? LOSS_FIELD_S22 : (i == 2 ? LOSS_FIELD_S12 : (i == 3 ? LOSS_FIELD_S13 :
           (i == 4 ? LOSS_FIELD_S23 : LOSS_FIELD_S33))));
  }
  static constexpr bool kStress = PASS == ES_BY || PASS == ES_BZ;
  __device__ __forceinline__ void load(Regs& r, int pos, uint32_t o) const {
    if (a.pml && a.pB.in(pos)) {
#pragma unroll
      for (int f = 0; f < 3; ++f) r.m[f] = at_off(kStress ? a.memB[f] : a.memA[f], o);
    }
    if constexpr (PASS == ES_BY) {
      r.t[0] = at_off(a.tmp[1], o);
    } else if constexpr (PASS == ES_BZ) {
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        r.u[f] = at_off(a.fld[stress(f)], o);
        if (KAHAN) r.c[f] = at_off(a.cmp[stress(f)], o);
      }
#pragma unroll
      for (int f = 0; f < 5; ++f) r.t[f] = at_off(a.tmp[f], o);
      if (lam_on) r.m0 = at_off(a.lam, o);
      if (mu_on) r.m1 = at_off(a.mu, o);
    } else if constexpr (PASS == ES_AY) {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        r.u[f] = at_off(a.fld[LOSS_FIELD_V1 + f], o);
        if (KAHAN) r.c[f] = at_off(a.cmp[LOSS_FIELD_V1 + f], o);
        r.t[f] = at_off(a.tmp[5 + f], o);
      }
      if (b_on) r.m0 = at_off(a.b, o);
    }
  }
  __device__ __forceinline__ void apply(Regs& r, const T (&e)[3], int pos, uint32_t o, int outer, int x) const {
    T* const* t = a.tmp;
    T g[3];
    if (a.pml && a.pB.in(pos)) {
#pragma unroll
      for (int f = 0; f < 3; ++f) g[f] = mulc1(e[f], a.s3h, a.s3h_lo);
      // the exact sub-flow (PmlAxis::step) on the memory values loaded ahead
      const PmlAxis<T>& pa = kStress ? a.pB : a.pA;
      const int n1 = pa.n + 1;
      const T T0 = pa.tab[pos], T1 = pa.tab[n1 + pos], T2 = pa.tab[2 * n1 + pos], T3 = pa.tab[3 * n1 + pos];
      T x[3], m1[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        m1[f] = T0 * r.m[f] - T1 * g[f];
        x[f] = -(T2 * (m1[f] - r.m[f]) - T3 * g[f]);
      }
      if constexpr (REC) {  // receiver corrections b (X(tau/2) - X(tau)/2)
        const T H0 = pa.tabh[pos], H1 = pa.tabh[n1 + pos], H2 = pa.tabh[2 * n1 + pos], H3 = pa.tabh[3 * n1 + pos];
        const T bb = b_on ? at_off(a.b, o) : a.b0;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const T xh = -(H2 * (H0 * r.m[f] - H1 * g[f] - r.m[f]) - H3 * g[f]);
          at_off(a.dlt[f], o) = bb * (xh - T(0.5) * x[f]);
        }
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        at_off(kStress ? a.memB[f] : a.memA[f], o) = m1[f];
        g[f] = x[f];
      }
    } else {
#pragma unroll
      for (int f = 0; f < 3; ++f) g[f] = mulc1(e[f], a.st, a.st_lo);
    }
    if constexpr (PASS == ES_BY) {
      at_off(t[1], o) = r.t[0] + g[0];
      at_off(t[3], o) = g[1];
      at_off(t[4], o) = g[2];
    } else if constexpr (PASS == ES_AZ) {
#pragma unroll
      for (int f = 0; f < 3; ++f) at_off(t[5 + f], o) = g[f];
    } else if constexpr (PASS == ES_BZ) {
      const T xa = r.t[0], tb = r.t[1], tc = r.t[2], xd = r.t[3], te = r.t[4];
      // constant moduli enter through mulc (their rounding errors would bias every update the same way)
      auto mlam = [&](T v) { return lam_on ? r.m0 * v : mulc1(v, a.lam0, a.lam0_lo); };
      auto mmu = [&](T v) { return mu_on ? r.m1 * v : mulc1(v, a.mu0, a.mu0_lo); };
      const T ltr = mlam(xa + xd + g[2]);
      T s11 = ltr + T(2) * mmu(xa), s22 = ltr + T(2) * mmu(xd), s33 = ltr + T(2) * mmu(g[2]);
      T s13 = mmu(tc + g[0]);
      if (a.srcp.on) {
        const int dz = pos - a.srcp.zs + 12, dy = outer - a.srcp.ys + 12, dx = x - a.srcp.xs + 12;
        if ((unsigned)dz < 25u && (unsigned)dy < 25u && (unsigned)dx < 25u) {
          const T sv = source_at(dz, dy, dx);
          if (a.src_explosive) s11 += sv, s22 += sv, s33 += sv;
          if (a.src_shear) s13 += sv;
        }
      }
      const T d[6] = {s11, s22, mmu(tb), s13, mmu(te + g[1]), s33};
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        upd_r<T, KAHAN>(r.u[f], r.c[f], d[f]);
        at_off(a.fld[stress(f)], o) = r.u[f];
        if (KAHAN) at_off(a.cmp[stress(f)], o) = r.c[f];
      }
    } else {  // ES_AY
      T force = T(0);  // body force (FORCE_X/Y/Z sources), already multiplied by the sub-step length
      if (a.srcp.on) {
        const int dz = outer - a.srcp.zs + 12, dy = pos - a.srcp.ys + 12, dx = x - a.srcp.xs + 12;
        if ((unsigned)dz < 25u && (unsigned)dy < 25u && (unsigned)dx < 25u)
          force = source_at(dz, dy, dx);
      }
      auto mb = [&](T v) { return b_on ? r.m0 * v : mulc1(v, a.b0, a.b0_lo); };
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const T ff = (a.force_mask & (1 << f)) ? force : T(0);
        upd_r<T, KAHAN>(r.u[f], r.c[f], mb(r.t[f] + g[f] + ff));
        at_off(a.fld[LOSS_FIELD_V1 + f], o) = r.u[f];
        if (KAHAN) at_off(a.cmp[LOSS_FIELD_V1 + f], o) = r.c[f];
      }
    }
  }
};

// REC as ElColOp.
template <typename T, int PASS, bool REC>
struct ElRowOp {
  static constexpr int NF = 3;
  static constexpr bool SECOND = false;
  static constexpr bool TWO = false;
  static constexpr int kBlocks = sizeof(T) == 4 ? (REC ? 3 : 4) : 2;
  ElArgs<T> a;
  int b_on;
  __device__ __forceinline__ const T* src(int f) const { return a.src[f]; }
  __device__ __forceinline__ void chunk(T (&e)[3][9], int p0, int len, int64_t gi, int) const {
    T* const* t = a.tmp;
    const PmlAxis<T>& pa = PASS == ES_BX ? a.pB : a.pA;
    T* const* mem = PASS == ES_BX ? a.memB : a.memA;
    const bool lay = a.pml && (pa.in(p0) || pa.in(p0 + len - 1));
    // every operand before the first store
    T u[3][9], m[3][9];
    if constexpr (PASS == ES_AX) {
#pragma unroll
      for (int f = 0; f < 3; ++f) ld9(t[5 + f] + gi, true, len, u[f]);
    }
    if (lay) {
#pragma unroll
      for (int f = 0; f < 3; ++f) ld9(mem[f] + gi, true, len, m[f]);
    }
    if (lay) {  // X[f,x] or Y[f,x] inside the layers: the exact sub-flow with its memory variable (PmlAxis::step)
      const int n1 = pa.n + 1;
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        const int i = min(p0 + j, pa.n);
        if (j < len && pa.in(i)) {
          const T T0 = pa.tab[i], T1 = pa.tab[n1 + i], T2 = pa.tab[2 * n1 + i], T3 = pa.tab[3 * n1 + i];
          T x[3];
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            const T g = mulc1(e[f][j], a.s3h, a.s3h_lo);
            const T m1 = T0 * m[f][j] - T1 * g;
            x[f] = -(T2 * (m1 - m[f][j]) - T3 * g);
            if constexpr (REC) {
              const T h1 = pa.tabh[i] * m[f][j] - pa.tabh[n1 + i] * g;
              const T xh = -(pa.tabh[2 * n1 + i] * (h1 - m[f][j]) - pa.tabh[3 * n1 + i] * g);
              a.dlt[f][gi + j] = (b_on ? a.b[gi + j] : a.b0) * (xh - T(0.5) * x[f]);
            }
            m[f][j] = m1;
            e[f][j] = x[f];
          }
        } else {
#pragma unroll
          for (int f = 0; f < 3; ++f) e[f][j] = mulc1(e[f][j], a.st, a.st_lo);
        }
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) st9(mem[f] + gi, true, len, m[f]);
    } else {
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int j = 0; j < 9; ++j) {
          if (j == 8 && len < 9) break;
          e[f][j] = mulc1(e[f][j], a.st, a.st_lo);
        }
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if constexpr (PASS == ES_BX) {
        st9(t[f] + gi, true, len, e[f]);
      } else {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
          if (j == 8 && len < 9) break;
          u[f][j] += e[f][j];
        }
        st9(t[5 + f] + gi, true, len, u[f]);
      }
    }
  }
};

template <typename T, class OP>
static cudaError_t launch_col(const ConvAxis& g, const ColMap& cm, const OP& op, cudaStream_t st) {
  const size_t smem = col_smem<T>(OP::NF, cm.warps);
  auto kern = k_col<T, OP>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)col_smem<T>(OP::NF, 4));
  if (e != cudaSuccess) return e;
  kern<<<col_blocks(cm, cm.warps), 32 * cm.warps, smem, st>>>(g, cm, op);
  return cudaGetLastError();
}

template <typename T, class OP>
static cudaError_t launch_row(const ConvAxis& g, const RowMap& rm, const OP& op, cudaStream_t st) {
  const size_t smem = (size_t)rm.warps * rm.wbytes;
  auto kern = k_row<T, OP>;
  if (smem > 32 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemMax);
    if (e != cudaSuccess) return e;
  }
  kern<<<row_blocks(rm, OP::kBlocks, rm.warps), 32 * rm.warps, smem, st>>>(g, rm, op);
  return cudaGetLastError();
}

// The pointers that a launch does not use, readable all the same.
template <class OP>
static void fill_unused(OP& op) {
  auto& a = op.a;
  if (!a.lam) a.lam = a.fld[0];
  if (!a.mu) a.mu = a.fld[0];
  if (!a.b) a.b = a.fld[0];
  if (!a.pml) {
    for (int f = 0; f < 3; ++f) a.memA[f] = a.memB[f] = a.fld[0];
    a.pA.tab = a.pB.tab = a.fld[0];
  }
}

template <typename T, int PASS, bool KAHAN, bool REC>
static cudaError_t launch_el_col(const ElArgs<T>& a, const ConvAxis& g, const ColMap& cm, cudaStream_t st) {
  ElColOp<T, PASS, KAHAN, REC> op{a, a.lam ? 1 : 0, a.mu ? 1 : 0, a.b ? 1 : 0};
  fill_unused(op);
  return launch_col<T>(g, cm, op, st);
}

template <typename T, int PASS, bool REC>
static cudaError_t launch_el_row(const ElArgs<T>& a, const ConvAxis& g, const RowMap& rm, cudaStream_t st) {
  ElRowOp<T, PASS, REC> op{a, a.b ? 1 : 0};
  fill_unused(op);
  return launch_row<T>(g, rm, op, st);
}

template <typename T, bool KAHAN>
cudaError_t launch_el_stream(const ElArgs<T>& a, const ConvAxis& g, const ColMap& cm, const RowMap& rm, int pass,
                             cudaStream_t st) {
  switch (pass) {
    case ES_BX: return launch_el_row<T, ES_BX, false>(a, g, rm, st);
    case ES_AX:
      if (a.pml && a.dlt[0]) return launch_el_row<T, ES_AX, true>(a, g, rm, st);
      return launch_el_row<T, ES_AX, false>(a, g, rm, st);
    case ES_BY: return launch_el_col<T, ES_BY, false, false>(a, g, cm, st);
    case ES_BZ: return launch_el_col<T, ES_BZ, KAHAN, false>(a, g, cm, st);
    case ES_AZ:
      if (a.pml && a.dlt[0]) return launch_el_col<T, ES_AZ, false, true>(a, g, cm, st);
      return launch_el_col<T, ES_AZ, false, false>(a, g, cm, st);
    default:
      if (a.pml && a.dlt[0]) return launch_el_col<T, ES_AY, KAHAN, true>(a, g, cm, st);
      return launch_el_col<T, ES_AY, KAHAN, false>(a, g, cm, st);
  }
}
template cudaError_t launch_el_stream<float, false>(const ElArgs<float>&, const ConvAxis&, const ColMap&,
                                                    const RowMap&, int, cudaStream_t);
template cudaError_t launch_el_stream<float, true>(const ElArgs<float>&, const ConvAxis&, const ColMap&,
                                                   const RowMap&, int, cudaStream_t);
template cudaError_t launch_el_stream<double, false>(const ElArgs<double>&, const ConvAxis&, const ColMap&,
                                                     const RowMap&, int, cudaStream_t);

}  // namespace lossk
