// sm_103a kernels of the stand-alone derivative operators (first and second derivative, transpose) on the barrier-free
// engines of loss_stream.cuh, dense arrays.
//
// The transpose of e = (R - L) + sum_j D_j r^|i - q_j| (D_j = sum_m w_jm f_{q_j + m}; times 3 a / h):
//   out_i = L_i - R_i (zeros beyond the ends, odd reflection transposed) + sum_j w_j,i-q_j Dbar_j,
//   Dbar_j = sum_d r^|d| g_{q_j + d}, |d| <= Q,
// so it runs on the same recursions; the weights w_j vanish but for the outer taps, as in the forward sums.
//
// Memory bound: one read and one write of the array per output (257^3 FP32: 136 MB).  The line kernel they replace
// (k_deriv, k_adj: whole lines staged in shared memory between barriers, a block's loads, elimination and stores in
// turn) took 1.75 ms for first and second derivatives and transposes along the axes of a 257^3 FP32 array that these do in
// 0.57 ms (with the host between); 129^2 FP64 operators, which launches bound, 95 us -> 80 us.  The line kernel stays for PMBC values, short patches, arrays beyond 32-bit
// offsets, arrays written over their input, and launch shapes that the caller asked for.
#include <cuda_runtime.h>

#include "../../include/loss.h"
#include "loss_host.h"
#include "loss_stream.cuh"
#include "loss_types.h"

namespace lossk {

template <typename T, bool D2>
struct DerivRowOp {
  static constexpr int NF = 1;
  static constexpr bool TWO = false, SECOND = D2;
  static constexpr int kBlocks = sizeof(T) == 4 ? 5 : 4;
  const T* f;
  T* d1;
  T* d2;
  T s1, s2;
  __device__ __forceinline__ const T* src(int) const { return f; }
  __device__ __forceinline__ void chunk(T (&e)[1][9], int, int len, int64_t gi, int) const {
#pragma unroll
    for (int j = 0; j < 9; ++j) e[0][j] *= s1;
    st9(d1 + gi, false, len, e[0]);
  }
  __device__ __forceinline__ void chunk2nd(T (&v)[9], int, int len, int64_t gi) const {
#pragma unroll
    for (int j = 0; j < 9; ++j) v[j] *= s2;
    st9(d2 + gi, false, len, v);
  }
};
template <typename T, bool D2>
struct DerivColOp {
  static constexpr int NF = 1;
  static constexpr bool SECOND = D2;
  static constexpr int kBlocks = sizeof(T) == 4 ? 6 : 4;
  static constexpr int B = 1;
  const T* f;
  T* d1;
  T* d2;
  T s1, s2;
  struct Regs {};
  __device__ __forceinline__ const T* src(int) const { return f; }
  __device__ __forceinline__ void load(Regs&, int, uint32_t) const {}
  __device__ __forceinline__ void apply(Regs&, const T (&e)[1], int, uint32_t o, int, int) const {
    at_off(d1, o) = s1 * e[0];
  }
  __device__ __forceinline__ void apply2nd(T v, uint32_t o) const { at_off(d2, o) = s2 * v; }
};

// Dbar_j as an unevaluated sum h + l (l = 0 in FP64): the sample at the junction plus the two tails, which round as the
// recursions do; their sum and the product with the junction's weights do not.  (The line kernel's form: FP32 solves
// joined, weighted and scaled in FP64.  The FP64 pipe would take 288 cycles for the products of a row window.)
template <typename T>
struct TransD {
  T h, l;
};
template <typename T>
__device__ __forceinline__ TransD<T> trans_sum(T f, T tails) {
  if constexpr (sizeof(T) == 8) {
    return {f + tails, T(0)};
  } else {
    const T h = __fadd_rn(f, tails), z = __fadd_rn(h, -f);
    return {h, __fadd_rn(__fadd_rn(f, -__fadd_rn(h, -z)), __fadd_rn(tails, -z))};
  }
}
// Weight i of the dense weights of an axis: a double, in FP32 axes a float and its rounding error.
template <typename T>
using TransW = std::conditional_t<sizeof(T) == 8, double, float2>;
template <typename T>
__device__ __forceinline__ T trans_add(T e, TransW<T> w, const TransD<T>& D) {
  if constexpr (sizeof(T) == 8) return fma(w, D.h, e);
  else return fmaf(w.x, D.h, e + fmaf(w.y, D.h, w.x * D.l));
}
// Dbar_j of the line whose samples start at byte offset o and step by sb.
template <typename T>
__device__ __forceinline__ TransD<T> trans_junction(const ConvAxis& g, int j, const T* f, uint32_t o, uint32_t sb) {
  constexpr T r = (T)kConvR;
  const int q = j * g.M;
  T a = T(0), b = T(0);
#pragma unroll 4
  for (int d = g.Q; d >= 1; --d) {
    const T va = at_off(f, o + (uint32_t)max(q - d, 0) * sb), vb = at_off(f, o + (uint32_t)min(q + d, g.n) * sb);
    a = (q - d >= 0 ? va : T(0)) + r * a;
    b = (q + d <= g.n ? vb : T(0)) + r * b;
  }
  return trans_sum(at_off(f, o + (uint32_t)q * sb), r * (a + b));
}

// out = scale * transpose along rows.
template <typename T>
__global__ void __launch_bounds__(128, 4) k_row_trans(ConvAxis g, RowMap rm, const T* __restrict__ in, T* __restrict__ out,
                                                      T scale, T scale_lo) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ T rs[kReach];
  fill_reach(rs, g);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = rm.gw, rpw = 32 / gw;
  TransD<T>* dsm = reinterpret_cast<TransD<T>*>(sm + (size_t)warp * rm.wbytes);
  const int gl = lane & (gw - 1), k = lane / gw;
  const int items = rm.groups * rm.nwin;
  const int nw = blockDim.x >> 5;
  for (int item = blockIdx.x * nw + warp; item < items; item += gridDim.x * nw) {
    const int grp = rm.nwin == 1 ? item : item / rm.nwin, win = item - grp * rm.nwin;
    const int c0 = win * (32 - 2 * Conv<T>::W);
    const int c1 = min(rm.nch, c0 + gw);
    const int o0 = win == 0 ? 0 : c0 + Conv<T>::W;
    const int o1 = c1 == rm.nch ? rm.nch : c1 - Conv<T>::W;
    auto rbase = [&](int q) {
      const int z = q / rm.ny;
      return z * rm.sz + (q - z * rm.ny) * rm.sy;
    };
    const int nrow = min(rpw, rm.rows - grp * rpw);
    const int q = grp * rpw + min(k, nrow - 1);
    const int64_t rb = rbase(q);
    const int c = c0 + gl;
    const int len = (k < nrow && c < c1) ? (c == rm.nch - 1 ? g.n + 1 - 8 * c : 8) : 0;
    const bool end = len > 0 && c == rm.nch - 1;
    const int64_t gi = rb + 8 * min(c, rm.nch - 1);
    const T rlen = end ? (T)__ldg(g.pw + len) : T(0);
    T e[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) e[j] = T(0);
    if (len > 0) ld9(in + gi, false, len, e);
    int j0 = 0, nj = 0;
    if (g.ntaps) {
      const int lo = 8 * o0, hi = o1 == rm.nch ? g.n : 8 * o1 - 1;
      j0 = lo <= g.R ? 0 : small_div(lo - g.R + g.M - 1, g.M);
      nj = min(g.p, small_div(hi + g.R, g.M)) - j0 + 1;
    }
    if (nj > 0) {  // G lanes per (row, junction)
      __syncwarp();
      const int tasks = nrow * nj, lg = tasks > 16 ? 0 : (tasks > 8 ? 1 : (tasks > 4 ? 2 : 3));
      for (int i0 = 0; i0 < tasks; i0 += 32 >> lg) {
        const int i = i0 + (lane >> lg), ii = min(i, tasks - 1);
        const int kk = small_div(ii, nj), q0 = (j0 + ii - kk * nj) * g.M;
        const T* f = in + (rpw == 1 ? rb : rbase(grp * rpw + kk));
        const int sub = lane & ((1 << lg) - 1);
        T D = T(0);
        for (int d = sub - g.Q; d <= g.Q; d += 1 << lg) {
          const int x = q0 + d;
          const T v = f[min(max(x, 0), g.n)];
          D += (x >= 0 && x <= g.n && d != 0 ? v : T(0)) * rs[64 + d];
        }
        __syncwarp();
        for (int o = 1; o < 1 << lg; o <<= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
        if (i < tasks && sub == 0) dsm[i] = trans_sum(f[q0], D);
      }
      __syncwarp();
    }
    if (end && len < 8)
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j >= len) e[j] = T(0);
    row_solve<T, kTrans>(e, c, len, end, gl, gw, rlen, T(0), T(0));
    if (len > 0 && c >= o0 && c < o1) {
      const int p0 = 8 * c;
      if (nj > 0) {
        const int ja = p0 <= g.R ? 0 : (p0 - g.R + g.M - 1) / g.M, jb = min(g.p, (p0 + 8 + g.R) / g.M);
        for (int j = ja; j <= jb; ++j) {
          const TransD<T> D = dsm[k * nj + min(max(j - j0, 0), nj - 1)];
          const TransW<T>* w = (const TransW<T>*)g.wd + (size_t)j * (2 * g.R + 1) + g.R;
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            const int m = p0 + i - j * g.M;
            const TransW<T> wi = __ldg(w + min(max(m, -g.R), g.R));
            if (m >= -g.R && m <= g.R) e[i] = trans_add<T>(e[i], wi, D);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 9; ++j) e[j] = mulc(e[j], scale, scale_lo);
      st9(out + gi, false, len, e);
    }
  }
}

// out = scale * transpose along strided lines, marched as k_col.
template <typename T>
__global__ void __launch_bounds__(128, 4) k_col_trans(ConvAxis g, ColMap cm, const T* __restrict__ in, T* __restrict__ out,
                                                      T scale, T scale_lo) {
  constexpr int W = Conv<T>::W, NR = W + 2, NJ = 4;
  constexpr T r = (T)kConvR, r8 = (T)conv_pow(8), r16 = (T)conv_pow(16);
  constexpr T i1r = (T)(2.0 / (1.0 - kConvR)), ir = (T)(1.0 / kConvR);
  extern __shared__ __align__(16) unsigned char sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t item = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  if (item >= cm.groups * cm.nseg) return;
  const int seg = (int)(item / cm.groups);
  const int64_t q0 = (item - (int64_t)seg * cm.groups) * 32 + lane;
  const bool valid = q0 < cm.lines;
  const int64_t ql = valid ? q0 : cm.lines - 1;
  const int outer = (int)(ql / cm.inner), x = (int)(ql - (int64_t)outer * cm.inner);
  const uint32_t base = (uint32_t)(((int64_t)outer * cm.so + x) * (int64_t)sizeof(T));
  const uint32_t sb = (uint32_t)(cm.stride * (int64_t)sizeof(T));
  const int n = g.n;
  const int s0 = seg * cm.seglen, s1 = min(s0 + cm.seglen, n + 1);
  const int nc = (s1 - s0 + 7) >> 3;
  const int ce = (n - s0) >> 3;
  const int le = n - s0 - 8 * ce;
  T* ring = reinterpret_cast<T*>(sm) + (size_t)warp * NR * 8 * 32 + lane;
  auto slot = [&](int c) { return ring + (size_t)(c % NR) * (8 * 32); };
  auto issue = [&](int c) {
    T* d = slot(c);
    const int p = s0 + 8 * c;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (p + j <= n) cp_async<sizeof(T)>(d + j * 32, &at_off(in, base + (uint32_t)(p + j) * sb));
    cp_async_commit();
  };
#pragma unroll
  for (int c = 0; c <= W; ++c) issue(c);
  T L = T(0);
  if (s0 > 0) {
#pragma unroll 8
    for (int k = Conv<T>::K; k >= 1; --k) L = at_off(in, base + (uint32_t)max(s0 - k, 0) * sb) + r * L;
  }
  T pb[W], Rn = T(0), endv = T(0), E0 = T(0);
  TransD<T> Dj[NJ];  // Dbar of the junctions jn - NJ .. jn - 1
#pragma unroll
  for (int i = 0; i < NJ; ++i) Dj[i] = {T(0), T(0)};
  int jn = s0 <= g.R ? 0 : (s0 - g.R + g.M - 1) / g.M;
  bool tailed = false;
  auto sums = [&](int c, int k) {
    const T* d = slot(c);
    T a = T(0);
    if (c < ce) {
#pragma unroll
      for (int j = 7; j >= 0; --j) a = d[j * 32] + r * a;
    }
    pb[k] = a;
  };
  cp_async_wait<0>();
#pragma unroll
  for (int c = 1; c < W; ++c) sums(c, c);
  for (int c = 0; c < nc; ++c) {
    issue(c + W + 1);
    cp_async_wait<1>();
#pragma unroll
    for (int k = 0; k + 1 < W; ++k) pb[k] = pb[k + 1];
    sums(c + W, W - 1);
    const T* d = slot(c);
    const int p0 = s0 + 8 * c;
    if (c == 0 && s0 == 0) {
      T a = pb[0] + r8 * pb[1];
      if (W == 4) a += r16 * (pb[W - 2] + r8 * pb[W - 1]);
      E0 = a;
#pragma unroll
      for (int j = 7; j >= 0; --j) E0 = d[j * 32] + r * E0;
      L = ir * E0;
    }
    if (!tailed && c + W >= ce) {
      tailed = true;
      T s = L;
      for (int i = 8 * c; i < n - s0; ++i) s = slot(i >> 3)[(i & 7) * 32] + r * s;
      const T* de = slot(ce);
      const T En = de[le * 32] + r * s;
      endv = s + i1r * En;
      Rn = ir * En;
      s = Rn;
      for (int j = le; j >= 0; --j) s = de[j * 32] + r * s;
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (c + 1 + k == ce) pb[k] = s;
    }
    T v[8], e[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = d[j * 32];
    T s = L;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      e[j] = s;
      s = v[j] + r * s;
    }
    L = s;
    T t = pb[0] + r8 * pb[1];
    if (W == 4) t += r16 * (pb[W - 2] + r8 * pb[W - 1]);
    if (c == ce) t = Rn;
#pragma unroll
    for (int j = 7; j >= 0; --j)
      if (c != ce || j <= le) {
        e[j] = p0 + j == 0 ? -t - i1r * E0 : (p0 + j == n ? endv : e[j] - t);
        t = v[j] + r * t;
      }
    while (g.ntaps && jn <= g.p && jn * g.M <= p0 + 7 + g.R) {
#pragma unroll
      for (int i = 0; i + 1 < NJ; ++i) Dj[i] = Dj[i + 1];
      Dj[NJ - 1] = trans_junction<T>(g, jn, in, base, sb);
      ++jn;
    }
#pragma unroll
    for (int i = 0; i < NJ; ++i) {
      const int j = jn - NJ + i;
      const int o = p0 - j * g.M;
      if (g.ntaps && j >= 0 && o <= g.R && o + 7 >= -g.R) {
        const TransW<T>* w = (const TransW<T>*)g.wd + (size_t)j * (2 * g.R + 1) + g.R;
#pragma unroll
        for (int l = 0; l < 8; ++l) {
          const int m = o + l;
          const TransW<T> wi = __ldg(w + min(max(m, -g.R), g.R));
          if (m >= -g.R && m <= g.R) e[l] = trans_add<T>(e[l], wi, Dj[i]);
        }
      }
    }
    const int len = min(8, s1 - p0);
    if (valid)
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < len) at_off(out, base + (uint32_t)(p0 + j) * sb) = mulc(e[j], scale, scale_lo);
  }
  cp_async_wait<0>();
}

// Derivatives of a dense array.  x: rows (no alignment is known), else lines.
template <typename T>
cudaError_t launch_deriv_stream(const ConvAxis& g, const ColMap& cm, const RowMap& rm, bool x, const T* f, T* d1, T* d2,
                                T s1, T s2, cudaStream_t st) {
  if (x) {
    const size_t smem = (size_t)rm.warps * rm.wbytes;
    auto go = [&](auto op, auto kern) {
      if (smem > 32 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemMax);
        if (e != cudaSuccess) return e;
      }
      kern<<<row_blocks(rm, decltype(op)::kBlocks, rm.warps), 32 * rm.warps, smem, st>>>(g, rm, op);
      return cudaGetLastError();
    };
    if (d2) return go(DerivRowOp<T, true>{f, d1, d2, s1, s2}, k_row<T, DerivRowOp<T, true>>);
    return go(DerivRowOp<T, false>{f, d1, d1, s1, s2}, k_row<T, DerivRowOp<T, false>>);
  }
  auto go = [&](auto op, auto kern, size_t smem) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)col_smem<T>(1, 4, true));
    if (e != cudaSuccess) return e;
    kern<<<col_blocks(cm, cm.warps), 32 * cm.warps, smem, st>>>(g, cm, op);
    return cudaGetLastError();
  };
  if constexpr (sizeof(T) == 4) {
    if (d2) return go(DerivColOp<T, true>{f, d1, d2, s1, s2}, k_col<T, DerivColOp<T, true>>, col_smem<T>(1, cm.warps, true));
  } else if (d2) {
    return cudaErrorNotSupported;  // not built: the line kernel takes them (run_derivative_t)
  }
  return go(DerivColOp<T, false>{f, d1, d1, s1, s2}, k_col<T, DerivColOp<T, false>>, col_smem<T>(1, cm.warps));
}

template <typename T>
cudaError_t launch_trans_stream(const ConvAxis& g, const ColMap& cm, const RowMap& rm, bool x, const T* in, T* out, T scale,
                                T scale_lo, cudaStream_t st) {
  if (x) {
    const size_t smem = (size_t)rm.warps * rm.wbytes;
    auto kern = k_row_trans<T>;
    if (smem > 32 * 1024) {
      const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemMax);
      if (e != cudaSuccess) return e;
    }
    kern<<<row_blocks(rm, 4, rm.warps), 32 * rm.warps, smem, st>>>(g, rm, in, out, scale, scale_lo);
    return cudaGetLastError();
  }
  const size_t smem = col_smem<T>(1, cm.warps);
  auto kern = k_col_trans<T>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)col_smem<T>(1, 4, true));
  if (e != cudaSuccess) return e;
  kern<<<col_blocks(cm, cm.warps), 32 * cm.warps, smem, st>>>(g, cm, in, out, scale, scale_lo);
  return cudaGetLastError();
}

template cudaError_t launch_deriv_stream<float>(const ConvAxis&, const ColMap&, const RowMap&, bool, const float*, float*,
                                                float*, float, float, cudaStream_t);
template cudaError_t launch_deriv_stream<double>(const ConvAxis&, const ColMap&, const RowMap&, bool, const double*,
                                                 double*, double*, double, double, cudaStream_t);
template cudaError_t launch_trans_stream<float>(const ConvAxis&, const ColMap&, const RowMap&, bool, const float*, float*,
                                                float, float, cudaStream_t);
template cudaError_t launch_trans_stream<double>(const ConvAxis&, const ColMap&, const RowMap&, bool, const double*, double*,
                                                 double, double, cudaStream_t);

}  // namespace lossk
