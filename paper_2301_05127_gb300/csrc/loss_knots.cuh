// Solves along lines with knots of their own.  The slopes of a patch satisfy a tridiagonal system; with the junction
// values phi_j as unknowns of their own, elimination along the whole line is two first-order recurrences
//   y_i = ra_i (f_i - f_{i-1}) + rb_i (f_{i+1} - f_i) - l_i y_{i-1},    d_i = y_i - g_i d_{i+1},
// rows scaled by their pivots, y_i = phi_j and l_i = g_i = 0 at a junction.  |l_i|, |g_i| < 2/3 (the system is
// diagonally dominant with ratio 1/2).
//
// A block holds C whole lines, a thread 8 consecutive positions of one: each thread runs its 8 positions from zero, the
// sums of its neighbours (shared memory) give the value that enters, `lf` and `lb` segments back, where the product of
// the multipliers has fallen below the precision of T (counted from the tables when they are made).  So the serial chain
// of a patch (k_nu_deriv: M positions forward and back by one thread) becomes 8 + 8 positions and three barriers.
// Bound by the latency of one block's life (load, three barriers, store), not by memory: 513^2 FP32, about 13 us a
// launch; a step with Kahan summation took 262 us (six derivative sweeps and four updates), now 60 us (four launches).
#pragma once
#include "loss_line.cuh"
#include "loss_types.h"

namespace lossk {

template <typename T>
struct KnotAxis {
  const double* W;  // [(p + 1)][2 n_nb + 1] PMBC weights
  const T* tab;     // l, g, ra, rb: 4 x 8 S (zeros beyond n)
  const T* seg;     // products of -l and -g over each segment: 2 x S
  int n, p, M, n_nb, S, lf, lb;
};
struct KnotLines {
  int64_t lines, stride, inner, inner_mul, outer_stride;  // base of line q: (q / inner) outer_stride + (q % inner) inner_mul
  int logc;                                               // log2 of the lines of a block
  int vec;                                                // rows (stride 1) on 16-byte boundaries, padded to 8
};
constexpr int kKnotThreads = 640;

// 8 positions of an array from gi on; positions beyond len repeat the last (vec rows: read the padding).
template <typename T, bool ROW>
__device__ __forceinline__ void kn_load(const T* __restrict__ p, int64_t gi, int64_t st, int vec, int len, T (&v)[8]) {
  if (ROW && vec) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int j = 0; j < 8; j += 4) {
        const float4 t = *reinterpret_cast<const float4*>(p + gi + j);
        v[j] = t.x, v[j + 1] = t.y, v[j + 2] = t.z, v[j + 3] = t.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        const double2 t = *reinterpret_cast<const double2*>(p + gi + j);
        v[j] = t.x, v[j + 1] = t.y;
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = p[gi + min(j, len - 1) * (ROW ? 1 : st)];
  }
}
template <typename T, bool ROW>
__device__ __forceinline__ void kn_store(T* __restrict__ p, int64_t gi, int64_t st, int vec, int len, const T (&v)[8]) {
  if (ROW && vec && len == 8) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int j = 0; j < 8; j += 4)
        *reinterpret_cast<float4*>(p + gi + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    } else {
#pragma unroll
      for (int j = 0; j < 8; j += 2) *reinterpret_cast<double2*>(p + gi + j) = make_double2(v[j], v[j + 1]);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < len) p[gi + j * (ROW ? 1 : st)] = v[j];
  }
}

// OP: const T* src(); void apply(const T (&d)[8], int p0, int len, int64_t gi, int64_t st, int vec, int64_t q)
// ROW: lines are rows (stride 1), a warp's lanes take consecutive segments; else a warp's lanes take the C lines of
// neighbouring columns.
template <typename T, bool ROW, class OP>
__device__ __forceinline__ void knot_block(const KnotAxis<T>& a, const KnotLines& kl, const OP& op, double* phi, int bid,
                                           unsigned char* sm) {
  const int C = 1 << kl.logc, S = a.S;
  T* fs = reinterpret_cast<T*>(sm);  // [S][C] forward sums, then
  T* bs = fs + S * C;                // [S][C] backward sums
  T* ph = bs + S * C;                // [p + 1][C]
  const int t = threadIdx.x, nt = blockDim.x;
  const bool used = t < S * C;
  const int tt = min(t, S * C - 1);
  const int c = ROW ? tt / S : tt & (C - 1), s = ROW ? tt - c * S : tt >> kl.logc;
  auto line = [&](int64_t q) { return (q / kl.inner) * kl.outer_stride + (q % kl.inner) * kl.inner_mul; };
  const int64_t q0 = (int64_t)bid << kl.logc;
  const int64_t q = min(q0 + c, kl.lines - 1);  // surplus lines repeat the last one and store nothing
  const int64_t base = line(q), st = ROW ? 1 : kl.stride;
  const int p0 = 8 * s, len = min(8, a.n + 1 - p0);
  const int64_t gi = base + p0 * st;
  const T* f = op.src();
  T e[8];
  kn_load<T, ROW>(f, gi, st, kl.vec, len, e);
  const T em = f[gi - (p0 > 0 ? st : 0)], ep = f[gi + min(8, a.n - p0) * st];
  {  // junction sums: a warp per junction, its lanes on C lines x 32 / C parts of the sum
    const int lane = t & 31, cc = lane & (C - 1), part = lane >> kl.logc, np = 32 >> kl.logc;
    const int64_t qc = min(q0 + cc, kl.lines - 1);
    const int64_t bc = line(qc);
    for (int j = t >> 5; j <= a.p; j += nt >> 5) {
      const int cj = j * a.M;
      const int mlo = max(-a.n_nb, -cj), mhi = min(a.n_nb, a.n - cj);
      const double* w = a.W + (size_t)j * (2 * a.n_nb + 1) + a.n_nb;
      double acc = 0.0;
#pragma unroll 4
      for (int m = mlo + part; m <= mhi; m += np) acc = fma(w[m], (double)f[bc + (cj + m) * st], acc);
      for (int o = 16; o >= C; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (part == 0) {
        ph[j * C + cc] = (T)acc;
        if (phi && q0 + cc < kl.lines) phi[qc * (a.p + 1) + j] = acc;
      }
    }
  }
  T l[8], y[8];
  const int n8 = 8 * S;
  {
    T ra[8], rb[8];
    kn_load<T, true>(a.tab, p0, 1, 1, 8, l);
    kn_load<T, true>(a.tab + 2 * n8, p0, 1, 1, 8, ra);
    kn_load<T, true>(a.tab + 3 * n8, p0, 1, 1, 8, rb);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const T fm = j ? e[j - 1] : em, fp = j < 7 ? e[j + 1] : ep;
      y[j] = ra[j] * (e[j] - fm) + rb[j] * (fp - e[j]);
    }
  }
  __syncthreads();
  for (int j = (p0 + a.M - 1) / a.M; j * a.M < p0 + len; ++j) {
    const int o = j * a.M - p0;
    const T v = ph[j * C + c];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i == o) y[i] = v;
  }
  // a multiplier of zero ends a patch: nothing passes it, not even a NaN
  auto step = [](T yi, T m, T x) { return m != T(0) ? yi - m * x : yi; };
  T v = T(0);
#pragma unroll
  for (int j = 0; j < 8; ++j) v = step(y[j], l[j], v);
  if (used) fs[s * C + c] = v;
  __syncthreads();
  v = T(0);
  for (int k = min(a.lf, s); k >= 1; --k) v = step(fs[(s - k) * C + c], -a.seg[s - k], v);
#pragma unroll
  for (int j = 0; j < 8; ++j) y[j] = v = step(y[j], l[j], v);
  kn_load<T, true>(a.tab + n8, p0, 1, 1, 8, l);  // g
  v = T(0);
#pragma unroll
  for (int j = 7; j >= 0; --j)
    if (j < len) v = step(y[j], l[j], v);
  if (used) bs[s * C + c] = v;
  __syncthreads();
  v = T(0);
  for (int k = min(a.lb, S - 1 - s); k >= 1; --k) v = step(bs[(s + k) * C + c], -a.seg[S + s + k], v);
#pragma unroll
  for (int j = 7; j >= 0; --j)
    if (j < len) y[j] = v = step(y[j], l[j], v);
  if (used && q0 + c < kl.lines) op.apply(y, p0, len, gi, st, kl.vec, q);
}

template <typename T, bool ROW, class OP>
__global__ void __launch_bounds__(kKnotThreads) k_knots(KnotAxis<T> a, KnotLines kl, OP op, double* phi) {
  extern __shared__ __align__(16) unsigned char sm[];
  knot_block<T, ROW>(a, kl, op, phi, blockIdx.x, sm);
}

// d1 of a field
template <typename T, bool ROW>
struct KnotDeriv {
  const T* f;
  T* d1;
  __device__ __forceinline__ const T* src() const { return f; }
  __device__ __forceinline__ void apply(const T (&d)[8], int, int len, int64_t gi, int64_t st, int vec, int64_t) const {
    kn_store<T, ROW>(d1, gi, st, vec, len, d);
  }
};

template <typename T, bool K>
__device__ __forceinline__ void kn_add(T& u, T& c, T delta) {
  if constexpr (K) kahan_add(u, c, delta);
  else u += delta;
}

// v += b X along the line, X = -tau d, or the layer's sub-flow inside it; `times` over (2: the last sub-step of one time
// step and the first of the next, which see the same sigma).
template <typename T, bool ROW, bool K>
struct KnotVel {
  const T* sigma;
  T *u, *c;
  const T* b;
  T b0, tau;
  int bc, pml, times;  // bc: b0 throughout.  Without an array or a layer its pointers name another array of the shot.
  PmlAxis<T> pa;
  T* mem;
  __device__ __forceinline__ const T* src() const { return sigma; }
  __device__ __forceinline__ void apply(const T (&d)[8], int p0, int len, int64_t gi, int64_t st, int vec, int64_t) const {
    T uv[8], cv[8], bv[8];
    kn_load<T, ROW>(u, gi, st, vec, len, uv);
    if constexpr (K) kn_load<T, ROW>(c, gi, st, vec, len, cv);
    if (!bc) kn_load<T, ROW>(b, gi, st, vec, len, bv);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (bc) bv[j] = b0;
      if (j >= len) continue;
      for (int k = 0; k < times; ++k) {
        T delta;
        if (pml) delta = bv[j] * (pa.in(p0 + j) ? pa.step(mem, gi + j * st, p0 + j, d[j]) : -tau * d[j]);
        else delta = (-tau * bv[j]) * d[j];
        kn_add<T, K>(uv[j], cv[j], delta);
      }
    }
    kn_store<T, ROW>(u, gi, st, vec, len, uv);
    if constexpr (K) kn_store<T, ROW>(c, gi, st, vec, len, cv);
  }
};

// Pressure source on knots: sigma += amp gz[oz] gx[ox] over the 25 x 25 knots around the source knot (zs, xs); gz,
// gx: the Gaussian of width 2 h on the physical distance from the source knot (0 off the grid); amp: dt f_r(t)
// times the amplitude over the cell-volume weighted sum of the profile.
struct NuSrc {
  int on, zs, xs;
  double amp;
  double gz[25], gx[25];
};

// sigma += kappa (X_x + X_z) along columns, then the source; gx: the derivative of v1 along x.
template <typename T, bool K>
struct KnotSig {
  const T* v3;
  T *u, *c;
  const T *gx, *kappa;
  T dt;
  int pml;
  PmlAxis<T> px, pz;
  T *memx, *memz;
  NuSrc q;
  __device__ __forceinline__ const T* src() const { return v3; }
  __device__ __forceinline__ void apply(const T (&d)[8], int p0, int len, int64_t gi, int64_t st, int vec,
                                        int64_t col64) const {
    const int col = (int)col64;
    T uv[8], cv[8], gv[8], kv[8];
    kn_load<T, false>(u, gi, st, vec, len, uv);
    if constexpr (K) kn_load<T, false>(c, gi, st, vec, len, cv);
    kn_load<T, false>(gx, gi, st, vec, len, gv);
    kn_load<T, false>(kappa, gi, st, vec, len, kv);
    const int ox = col - q.xs + 12;
    const double sx = q.on && ox >= 0 && ox < 25 ? q.gx[min(max(ox, 0), 24)] : 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j >= len) continue;
      T delta;
      if (pml) {
        const T Xx = px.in(col) ? px.step(memx, gi + j * st, col, gv[j]) : -dt * gv[j];
        const T Xz = pz.in(p0 + j) ? pz.step(memz, gi + j * st, p0 + j, d[j]) : -dt * d[j];
        delta = kv[j] * (Xx + Xz);
      } else {
        delta = (-dt * kv[j]) * (gv[j] + d[j]);
      }
      kn_add<T, K>(uv[j], cv[j], delta);
      if (sx != 0.0) {
        const int oz = p0 + j - q.zs + 12;
        const double sz = oz >= 0 && oz < 25 ? q.gz[min(max(oz, 0), 24)] : 0.0;
        if (sz != 0.0) kn_add<T, K>(uv[j], cv[j], (T)(q.amp * sz * sx));
      }
    }
    kn_store<T, false>(u, gi, st, vec, len, uv);
    if constexpr (K) kn_store<T, false>(c, gi, st, vec, len, cv);
  }
};

}  // namespace lossk
