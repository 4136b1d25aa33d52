// Barrier-free engines of the truncated-convolution form (loss_fir.cuh) of the LOSS derivative, FP32 and FP64.
//
// Both evaluate  e_i = (R_i - L_i) + sum_j D_j r^|i - jM|  (the scaled derivative over a; the caller multiplies by
// 3 a / h) with warps that never wait for one another:
//   - k_col: lines along a strided axis.  One thread per line, 32 neighbouring lines per warp; a thread marches along
//     its line in chunks of 8 positions.  Its samples pass through a ring of chunks in shared memory that the thread
//     fills with cp.async and reads alone, so every sample is read from global memory once and no barrier is needed.
//   - k_row: lines along the contiguous axis.  A warp (or 8 or 16 lanes of it, for short rows) takes up to 32 chunks of
//     8 positions of a row, one chunk per lane, staged in the warp's own shared memory; the warm-up sums of a
//     chunk come from its neighbour lanes by shuffles.
//
// Recursions start from sums over W whole neighbour chunks (16 terms in FP32, 32 in FP64: |r|^16 = 7e-10, |r|^32 =
// 5e-19), or, beyond a line's end, from the closed form of the odd reflection f_{-k} = 2 f_0 - f_k:
// L_0 = 2 f_0 / (1 - r) - R_0 and R_n = 2 f_n / (1 - r) - L_n.
//
// Junction corrections.  D_j = sum_m w_jm f_{jM + m} in FP64.  Away from the line ends the PMBC weights equal the
// convolution's own weights term by term up to min(n_nb, K) (both are the Toeplitz inverse), so all but the outer
// taps of a row vanish up to the rounding of their difference; the host keeps the taps that do not (ConvAxis::taps,
// 8 instead of 41 per junction at n_nb = 20, K = 16).  A correction reaches Q positions, where |r|^Q |D| is
// below the working precision (host rule conv_axis in loss_step.cu); longer patches make the second term of the
// patch-end correction, r^M D, vanish by the same rule.
//
// Accesses: loads outside a predicate have their offsets clamped to their line or row; the ring's copies and the stores
// stand under the predicate that their position lies on the line (their offsets may lie past it, and are not used
// then).  Pointers that a launch lacks are replaced on the host or excluded by a template parameter.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "loss_fir.cuh"
#include "loss_line.cuh"
#include "loss_types.h"

namespace lossk {

// Powers of r = sqrt(3) - 2 and 2 / (1 - r) in the working precision.
constexpr double kConvR = -0.26794919243112270647255365849413;
constexpr double conv_pow(int k) { return k == 0 ? 1.0 : kConvR * conv_pow(k - 1); }
template <typename T>
struct Conv {
  static constexpr int W = sizeof(T) == 4 ? 2 : 4;  // neighbour chunks of a warm-up sum
  static constexpr int K = 8 * W;
};

// Weights of a junction's correction at distance d: rs[64 + d] = r^|d| for |d| <= Q, 0 beyond, d = -64 .. 79, in
// shared memory (no barrier).
constexpr int kReach = 144;
template <typename T>
__device__ __forceinline__ void fill_reach(T* rs, const ConvAxis& g) {
  for (int i = threadIdx.x; i < kReach; i += blockDim.x) {
    const int d = abs(i - 64);
    rs[i] = d <= g.Q ? (T)__ldg(g.pw + min(d, 63)) : T(0);
  }
}

// The axis's taps in shared memory when they fit (no barrier).
constexpr int kTapsSmem = 128;
__device__ __forceinline__ const ConvTap* stage_taps(const ConvAxis& g, ConvTap* tsm) {
  if (g.ntaps > kTapsSmem) return g.taps;
  for (int i = threadIdx.x; i < g.ntaps; i += blockDim.x) tsm[i] = g.taps[i];
  return tsm;
}

// x (c + c_lo) rounded once, c_lo x aside (mulc rounds c x first, and c_lo is lost unless c_lo x exceeds half a unit of that).
template <typename T>
__device__ __forceinline__ T mulc1(T x, T c, T c_lo) {
  if constexpr (sizeof(T) == 8) return c * x;
  else return fmaf(c, x, c_lo * x);
}

// Element at a byte offset below 4 GB from a (uniform) base: one 32-bit offset serves every array of a pass.
template <typename T>
__device__ __forceinline__ T& at_off(T* p, uint32_t o) {
  using C = std::conditional_t<std::is_const_v<T>, const char, char>;
  return *reinterpret_cast<T*>(reinterpret_cast<C*>(p) + o);
}

// The sums of weight x sample over the taps of a junction are FP64, whatever T: the GPU's FP64 pipe takes 16 cycles of an
// SM per warp instruction, however few lanes are active, so several lanes of a row warp share one junction (one lane each
// had 5 of 32 at work on a row of four patches) and FP32 samples are widened on the integer units.
// Junction corrections D[f] of junction j of NF lines with their samples at byte offset o + (jM + m) * sb of src[f]; taps:
// the axis's taps (a shared-memory copy or g.taps); four taps' samples in flight at a time.
template <typename T, int NF>
__device__ __forceinline__ void conv_junction(const ConvAxis& g, const ConvTap* taps, int j, const T* const (&src)[NF],
                                              uint32_t o, uint32_t sb, T (&D)[NF]) {
  int t = __ldg(g.js + j);
  const int t1 = __ldg(g.js + j + 1);
  double s[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) s[f] = 0.0;
  for (; t < t1; t += 4) {
    ConvTap w[4];
    T v[4][NF];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      w[k] = taps[min(t + k, t1 - 1)];
      const uint32_t ot = o + (uint32_t)(j * g.M + w[k].m) * sb;
#pragma unroll
      for (int f = 0; f < NF; ++f) v[k][f] = at_off(src[f], ot);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (t + k < t1)
#pragma unroll
        for (int f = 0; f < NF; ++f) s[f] = fma(w[k].w, to_f64(v[k][f]), s[f]);
  }
#pragma unroll
  for (int f = 0; f < NF; ++f) D[f] = (T)s[f];
}
// The same for one line at f by G lanes (a power of two; sub: the lane's number among them); called by the whole warp.
template <typename T>
__device__ __forceinline__ T conv_junction_part(const ConvAxis& g, const ConvTap* taps, int j, const T* f, int sub,
                                                int G) {
  const int t1 = __ldg(g.js + j + 1);
  const T* fj = f + j * g.M;
  double s = 0.0;
  for (int t = __ldg(g.js + j) + sub; t < t1; t += 2 * G) {
    const ConvTap w0 = taps[t], w1 = taps[min(t + G, t1 - 1)];
    const T v0 = fj[w0.m], v1 = fj[w1.m];
    s = fma(w0.w, to_f64(v0), s);
    if (t + G < t1) s = fma(w1.w, to_f64(v1), s);
  }
  __syncwarp();
  for (int o = 1; o < G; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return (T)s;
}
// a / b for 0 <= a < 2^21, b > 0 (a quotient is 1 / (2 b) or more from the next integer, its error below 2^-22 of it)
__device__ __forceinline__ int small_div(int a, int b) { return (int)__fdividef((float)a + 0.5f, (float)b); }

// Block-wide copy of a launch descriptor into shared memory (no barrier).
template <class J>
__device__ __forceinline__ void copy_job(J* dst, const J* __restrict__ src) {
  static_assert(sizeof(J) % 8 == 0, "descriptor size");
  for (int i = threadIdx.x; i < (int)(sizeof(J) / 8); i += blockDim.x)
    reinterpret_cast<uint64_t*>(dst)[i] = reinterpret_cast<const uint64_t*>(src)[i];
}

// Correction of the second derivative by a junction at offset o of the chunk: slopes that differ by D r^|i - q| shift the
// scaled second derivative f_i + r (R_i + L_i) by -6 a D sgn(i - q) r^|i - q| (at the junction itself the two patches' values
// average to 0; a line end has one patch).
template <typename T, int N>
__device__ __forceinline__ void add_second(T (&v)[N], T D, int o, int j, const ConvAxis& g, const T* rs) {
  const T w = (T)(6.0 * kConvR) * D;  // a = -r
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int d = o + i;
    const T sg = d > 0 ? T(1) : (d < 0 ? T(-1) : (j == 0 ? T(1) : (j == g.p ? T(-1) : T(0))));
    v[i] += w * sg * rs[64 + d];
  }
}

// ---------------------------------------------------------------------------------------------------------------
// Strided lines.  Line q (0 .. lines - 1) starts at (q / inner) * so + q % inner and steps by `stride`; it is cut into
// segments of seglen positions (a multiple of 8, nseg of them), each marched by one thread.
//
// OP: static constexpr int NF (fields differentiated), B (positions whose pointwise operands are held in registers),
//   const T* src(int f); struct Regs; void load(Regs&, int pos, uint32_t o);
//   void apply(Regs&, const T (&e)[NF], int pos, uint32_t o, int outer, int x)
// o: byte offset of the position in every array.  Operands are loaded B positions ahead of their use, across chunks.
template <typename T, class OP>
__device__ __forceinline__ void col_block(const ConvAxis& g, const ColMap& cm, const OP& op, int bid,
                                          unsigned char* sm) {
  constexpr int NF = OP::NF, W = Conv<T>::W, LA = W + (OP::SECOND ? 1 : 0), NR = LA + 2;
  constexpr T r = (T)kConvR, r7 = (T)conv_pow(7), r8 = (T)conv_pow(8), r16 = (T)conv_pow(16);
  constexpr T i1r = (T)(2.0 / (1.0 - kConvR));
  __shared__ T rs[kReach];
  __shared__ ConvTap tsm[kTapsSmem];
  fill_reach(rs, g);
  const ConvTap* taps = stage_taps(g, tsm);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t item = (int64_t)bid * (blockDim.x >> 5) + warp;
  if (item >= cm.groups * cm.nseg) return;
  const int seg = (int)(item / cm.groups);
  const int64_t q0 = (item - (int64_t)seg * cm.groups) * 32 + lane;
  const bool valid = q0 < cm.lines;
  const int64_t q = valid ? q0 : cm.lines - 1;  // surplus lanes repeat the last line and store nothing
  const int outer = (int)(q / cm.inner), x = (int)(q - (int64_t)outer * cm.inner);
  const uint32_t base = (uint32_t)(((int64_t)outer * cm.so + x) * (int64_t)sizeof(T));
  const uint32_t sb = (uint32_t)(cm.stride * (int64_t)sizeof(T));
  const int n = g.n;
  const int s0 = seg * cm.seglen, s1 = min(s0 + cm.seglen, n + 1);
  const int nc = (s1 - s0 + 7) >> 3;      // chunks of the segment
  const int ce = (n - s0) >> 3;           // chunk that holds position n
  const int le = n - s0 - 8 * ce;         // its place there
  T* ring = reinterpret_cast<T*>(sm) + (size_t)warp * NR * 8 * NF * 32 + lane;
  auto slot = [&](int c) { return ring + (size_t)(c % NR) * (8 * NF * 32); };
  auto issue = [&](int c) {
    T* d = slot(c);
    const int p = s0 + 8 * c;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (p + j <= n)
#pragma unroll
        for (int f = 0; f < NF; ++f) cp_async<sizeof(T)>(d + (j * NF + f) * 32, &at_off(op.src(f), base + (uint32_t)(p + j) * sb));
    cp_async_commit();
  };
#pragma unroll
  for (int c = 0; c <= LA; ++c) issue(c);
  typename OP::Regs pr[OP::B];
#pragma unroll
  for (int b = 0; b < OP::B; ++b) op.load(pr[b], min(s0 + b, n), base + (uint32_t)min(s0 + b, n) * sb);
  // left sums of the segment's first position
  T L[NF];
  if (s0 > 0) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      T a = T(0);
#pragma unroll 8
      for (int k = Conv<T>::K; k >= 1; --k) a = at_off(op.src(f), base + (uint32_t)max(s0 - k, 0) * sb) + r * a;
      L[f] = a;
    }
  }
  T pb[NF][W];     // sums r^j f_j of the next W chunks
  T Rn[NF];        // R_n, from the moment chunk ce is in the ring
  T Da[NF], Db[NF];  // corrections of junctions jn - 2 and jn - 1
  int jn = s0 <= g.Q ? 0 : (s0 - g.Q + g.M - 1) / g.M;
  int ja = -1, jb = -1;
  bool tailed = false;
#pragma unroll
  for (int f = 0; f < NF; ++f) Rn[f] = Da[f] = Db[f] = T(0);
  auto sums = [&](int c, int k) {
    const T* d = slot(c);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      T a = T(0);
      if (c < ce) {
#pragma unroll
        for (int j = 7; j >= 0; --j) a = d[(j * NF + f) * 32] + r * a;
      }
      pb[f][k] = a;
    }
  };
  cp_async_wait<0>();
  // second differences (field 0): sample i of the segment, and the sums of the next chunks as for the samples
  T pb2[W], L2 = T(0), Rn2 = T(0);
  T fprev = T(0);  // the sample before the chunk
  auto val = [&](int i) { return slot(i >> 3)[(i & 7) * NF * 32]; };
  auto sums2 = [&](int c, int k) {
    T a = T(0);
    if (c < ce) {
      T fp = val(8 * c + 8), f0 = val(8 * c + 7);
#pragma unroll
      for (int j = 7; j >= 0; --j) {
        const T fm = val(8 * c + j - 1);
        a = ((fp - f0) - (f0 - fm)) + r * a;
        fp = f0;
        f0 = fm;
      }
    }
    pb2[k] = a;
  };
  if constexpr (OP::SECOND) {
    if (s0 > 0) {
      const T* f = op.src(0);
      auto at = [&](int i) { return at_off(f, base + (uint32_t)max(i, 0) * sb); };
      fprev = at(s0 - 1);
      T fm = at(s0 - Conv<T>::K - 1), f0 = at(s0 - Conv<T>::K);
#pragma unroll 8
      for (int k = Conv<T>::K; k >= 1; --k) {
        const T fp = at(s0 - k + 1);
        L2 = ((fp - f0) - (f0 - fm)) + r * L2;
        fm = f0;
        f0 = fp;
      }
    }
#pragma unroll
    for (int c = 1; c < W; ++c) sums2(c, c);
  }
#pragma unroll
  for (int c = 1; c < W; ++c) sums(c, c);  // shifted down by the first iteration
  for (int c = 0; c < nc; ++c) {
    issue(c + LA + 1);
    cp_async_wait<1>();
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int k = 0; k + 1 < W; ++k) pb[f][k] = pb[f][k + 1];
    sums(c + W, W - 1);
    if constexpr (OP::SECOND) {
#pragma unroll
      for (int k = 0; k + 1 < W; ++k) pb2[k] = pb2[k + 1];
      sums2(c + W, W - 1);
    }
    const T* d = slot(c);
    const int p0 = s0 + 8 * c;
    if (c == 0 && s0 == 0) {  // odd reflection at the line's start (n >= 40: chunks 0 .. W are whole)
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        T a = pb[f][0] + r8 * pb[f][1];
        if (W == 4) a += r16 * (pb[f][W - 2] + r8 * pb[f][W - 1]);
        T b = T(0);
#pragma unroll
        for (int j = 7; j >= 1; --j) b = d[(j * NF + f) * 32] + r * b;
        L[f] = i1r * d[f * 32] - (b + r7 * a);
      }
    }
    if constexpr (OP::SECOND) {
      if (c == 0 && s0 == 0) {
        T a = pb2[0] + r8 * pb2[1];
        if (W == 4) a += r16 * (pb2[W - 2] + r8 * pb2[W - 1]);
        T b = T(0);
#pragma unroll
        for (int j = 7; j >= 1; --j) b = ((val(j + 1) - val(j)) - (val(j) - val(j - 1))) + r * b;
        L2 = -(b + r7 * a);
      }
      if (!tailed && c + W >= ce) {
        T s = L2, fm = fprev, f0 = val(8 * c);
        for (int i = 8 * c; i < n - s0; ++i) {
          const T fp = val(i + 1);
          s = (i + s0 == 0 ? T(0) : (fp - f0) - (f0 - fm)) + r * s;
          fm = f0;
          f0 = fp;
        }
        Rn2 = -s;
        s = r * Rn2;  // position n has second difference 0
        for (int j = le - 1; j >= 0; --j) {
          const int i = 8 * ce + j;
          s = ((val(i + 1) - val(i)) - (val(i) - val(max(i - 1, 0)))) + r * s;
        }
#pragma unroll
        for (int k = 0; k < W; ++k)
          if (c + 1 + k == ce) pb2[k] = s;
      }
    }
    if (!tailed && c + W >= ce) {  // R_n, and the sum of chunk ce with its reflected continuation
      tailed = true;
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        T s = L[f];
        for (int i = 8 * c; i < n - s0; ++i) s = slot(i >> 3)[((i & 7) * NF + f) * 32] + r * s;
        const T* de = slot(ce);
        const T R = i1r * de[(le * NF + f) * 32] - s;
        Rn[f] = R;
        s = R;
        for (int j = le; j >= 0; --j) s = de[(j * NF + f) * 32] + r * s;
#pragma unroll
        for (int k = 0; k < W; ++k)
          if (c + 1 + k == ce) pb[f][k] = s;
      }
    }
    // Junctions within Q of the chunk (at most two, M >= Q + 8).  D r^|i - q| is added through the sums: L_i - D r^(i - q)
    // at positions from q on (the recursion carries it along) and R_i + D r^(q - i) before q, so a junction costs an
    // operation per chunk; only a chunk with a junction inside adds it point by point.
    while (g.ntaps && jn <= g.p && jn * g.M <= p0 + 7 + g.Q) {
      ja = jb;
      jb = jn;
      const T* fs[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        Da[f] = Db[f];
        fs[f] = op.src(f);
      }
      conv_junction<T, NF>(g, taps, jn, fs, base, sb, Db);
      const int o = p0 - jn * g.M;  // before the segment's first position
      if (o > 0)
#pragma unroll
        for (int f = 0; f < NF; ++f) L[f] -= Db[f] * rs[64 + o];
      ++jn;
    }
    const int oa = ja >= 0 ? p0 - ja * g.M : 1, ob = jb >= 0 ? p0 - jb * g.M : 1;
    const int len = min(8, s1 - p0);
    T e[NF][8];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      T v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = d[(j * NF + f) * 32];
      if (oa == 0) L[f] -= Da[f];
      if (ob == 0) L[f] -= Db[f];
      T s = L[f];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        e[f][j] = s;
        s = v[j] + r * s;
      }
      L[f] = s;
      T t = pb[f][0] + r8 * pb[f][1];
      if (W == 4) t += r16 * (pb[f][W - 2] + r8 * pb[f][W - 1]);
      if (c == ce) t = Rn[f];
      if (oa < -7) t += Da[f] * rs[64 - oa - 7];
      if (ob < -7) t += Db[f] * rs[64 - ob - 7];
#pragma unroll
      for (int j = 7; j >= 0; --j)
        if (c != ce || j <= le) {
          e[f][j] = t - e[f][j];
          t = v[j] + r * t;
        }
    }
    if constexpr (OP::SECOND) {
      T v2[8], fm = fprev, f0 = d[0];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const T fp = j < 7 ? d[(j + 1) * NF * 32] : val(8 * c + 8);
        const int i = p0 + j;
        v2[j] = i > 0 && i < n ? (fp - f0) - (f0 - fm) : T(0);
        fm = f0;
        f0 = fp;
      }
      fprev = fm;
      T e2[8], s = L2;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        e2[j] = s;
        s = v2[j] + r * s;
      }
      L2 = s;
      T t = pb2[0] + r8 * pb2[1];
      if (W == 4) t += r16 * (pb2[W - 2] + r8 * pb2[W - 1]);
      if (c == ce) t = Rn2;
#pragma unroll
      for (int j = 7; j >= 0; --j)
        if (c != ce || j <= le) {
          e2[j] = v2[j] + r * (t + e2[j]);
          t = v2[j] + r * t;
        }
      if (ja >= 0 && oa <= g.Q) add_second(e2, Da[0], oa, ja, g, rs);
      if (jb >= 0 && ob <= g.Q) add_second(e2, Db[0], ob, jb, g, rs);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < len && valid) op.apply2nd(e2[j], base + (uint32_t)(p0 + j) * sb);
    }
    if (oa < 0 && oa >= -7) {
#pragma unroll
      for (int f = 0; f < NF; ++f) {
#pragma unroll
        for (int j = 0; j < 8; ++j) e[f][j] += Da[f] * rs[64 + oa + j];
        L[f] -= Da[f] * rs[64 + oa + 8];
      }
    }
    if (ob < 0 && ob >= -7) {
#pragma unroll
      for (int f = 0; f < NF; ++f) {
#pragma unroll
        for (int j = 0; j < 8; ++j) e[f][j] += Db[f] * rs[64 + ob + j];
        L[f] -= Db[f] * rs[64 + ob + 8];
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j >= len) break;
      T ej[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) ej[f] = e[f][j];
      const uint32_t o = base + (uint32_t)(p0 + j) * sb;
      if (valid) op.apply(pr[j % OP::B], ej, p0 + j, o, outer, x);
      const int pn = min(p0 + j + OP::B, n);
      if (p0 + j + OP::B < s1) op.load(pr[j % OP::B], pn, base + (uint32_t)pn * sb);
    }
  }
  cp_async_wait<0>();
}

template <typename T, class OP>
__global__ void __launch_bounds__(128, OP::kBlocks) k_col(ConvAxis g, ColMap cm, OP op) {
  extern __shared__ __align__(16) unsigned char sm[];
  col_block<T>(g, cm, op, blockIdx.x, sm);
}

// All shots in one launch: block b does the work of block blk[b].y of shot blk[b].x's own launch.
template <typename T, class OP>
struct ColJob {
  ConvAxis g;
  ColMap cm;
  OP op;
};
template <typename T, class OP>
__global__ void __launch_bounds__(128, OP::kBlocks)
    k_col_batch(const ColJob<T, OP>* __restrict__ jobs, const int2* __restrict__ blk) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ __align__(16) unsigned char raw[sizeof(ColJob<T, OP>)];
  const int2 w = blk[blockIdx.x];
  ColJob<T, OP>& j = *reinterpret_cast<ColJob<T, OP>*>(raw);
  copy_job(&j, jobs + w.x);
  __syncthreads();
  col_block<T>(j.g, j.cm, j.op, w.y, sm);
}

// Dynamic shared memory of a k_col block.  (The kernels' limits are set to one size whatever the launch, so that threads
// with handles of their own do not lower each other's.)
constexpr int kRowSmemMax = 220 * 1024;
template <typename T>
constexpr size_t col_smem(int nf, int warps, bool second = false) {
  return (size_t)warps * (Conv<T>::W + 2 + (second ? 1 : 0)) * 8 * nf * 32 * sizeof(T);
}

// ---------------------------------------------------------------------------------------------------------------
// Contiguous rows.  Row q (0 .. rows - 1) starts at (q / ny) * sz + (q % ny) * sy.  A row has nch chunks of 8 positions,
// the last of 1 to 9 (position n joins the chunk before it when n is a multiple of 8).  Rows of at most 32 chunks are
// one window of gw = 8, 16 or 32 lanes (32 / gw rows per warp); longer rows are cut into nwin windows of 32 chunks
// that overlap by 2 W chunks, of which each owns all but the W at its inner ends.
//
// A lane loads its chunk straight into registers (two 16-byte loads in FP32, 32 bytes apart from its neighbours': the
// second finds the first's sectors in L1), so nothing is staged; samples cross lanes only in the warm-up sums.

// Eight consecutive elements (vec: p is 16-byte aligned).
template <typename T>
__device__ __forceinline__ void ld8(const T* __restrict__ p, bool vec, int len, T* v) {
  if (vec) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int j = 0; j < 8; j += 4) {
        const float4 t = *reinterpret_cast<const float4*>(p + j);
        v[j] = t.x, v[j + 1] = t.y, v[j + 2] = t.z, v[j + 3] = t.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        const double2 t = *reinterpret_cast<const double2*>(p + j);
        v[j] = t.x, v[j + 1] = t.y;
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const T u = p[min(j, max(len - 1, 0))];
      v[j] = j < len ? u : T(0);
    }
  }
}
// The first min(len, 8) of eight consecutive elements, and the ninth when len = 9.
template <typename T>
__device__ __forceinline__ void st9(T* __restrict__ p, bool vec, int len, const T* v) {
  if (vec && len >= 8) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int j = 0; j < 8; j += 4)
        *reinterpret_cast<float4*>(p + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    } else {
#pragma unroll
      for (int j = 0; j < 8; j += 2) *reinterpret_cast<double2*>(p + j) = make_double2(v[j], v[j + 1]);
    }
    if (len > 8) p[8] = v[8];
  } else {
#pragma unroll
    for (int j = 0; j < 9; ++j)
      if (j < len) p[j] = v[j];
  }
}
template <typename T>
__device__ __forceinline__ void ld9(const T* __restrict__ p, bool vec, int len, T (&v)[9]) {
  ld8(p, vec, len, v);
  const T* p8 = p + (len > 8 ? 8 : 0);
  v[8] = T(0);
  if (len > 8) v[8] = *p8;
}

// What a solve forms of the samples f of a chunk (0 beyond len), in place:
//   kFirst:  R_i - L_i (the first derivative over a, but for junctions inside the chunk);
//   kSecond: f_i + r (R_i + L_i), the second derivative's convolution of the second differences f;
//   kTrans:  L_i - R_i over zeros beyond the ends, plus the transpose of the odd reflection: with E_0 = sum r^i f_i it
//            is a r^(i-1) E_0 at i > 0 (as if L_0 were E_0 / r) and -2 E_0 / (1 - r) at i = 0; at n with the sign reversed.
// Called by all lanes of the warp; c: chunk of the row, gl: lane of the gw-lane group, end: the chunk holds position n,
// rlen = r^len; dL, dR: corrections of the junctions before and after the chunk, at its first and its last position.
enum { kFirst = 0, kSecond = 1, kTrans = 2 };
template <typename T, int MODE = kFirst>
__device__ __forceinline__ void row_solve(T (&f)[9], int c, int len, bool end, int gl, int gw, T rlen, T dL, T dR) {
  constexpr int W = Conv<T>::W;
  constexpr T r = (T)kConvR, r7 = (T)conv_pow(7), r8 = (T)conv_pow(8), r16 = (T)conv_pow(16);
  constexpr T i1r = (T)(2.0 / (1.0 - kConvR)), ir = (T)(1.0 / kConvR);
  const unsigned full = 0xffffffffu;
  T e[9];
  T pa = f[0], pb, pb1;
#pragma unroll
  for (int j = 1; j < 8; ++j) pa = f[j] + r * pa;
  if (len > 8) pb = f[7] + r * f[8];  // the ninth position of a row's last chunk
  else pb = f[7];
#pragma unroll
  for (int j = 6; j >= 1; --j) pb = f[j] + r * pb;
  pb1 = pb;
  pb = f[0] + r * pb;
  auto down = [&](T v, int d) {
    const T u = __shfl_down_sync(full, v, d, gw);
    return gl + d < gw ? u : T(0);
  };
  // left sums: chunk -1 of the row is the reflected continuation, whose whole sum is L_0
  T t = pb + r8 * down(pb, 1);
  if (W == 4) t += r16 * down(t, 2);
  const T R0 = pb1 + r7 * down(t, 1);
  const T E0 = t;
  const T l0 = c == 0 ? (MODE == kTrans ? ir * E0 : i1r * f[0] - R0) : T(0);
  const T L0 = __shfl_sync(full, l0, 0, gw);  // 0 in windows that do not start the row
  T u = __shfl_up_sync(full, pa, 1, gw);
  T s = pa + r8 * (gl == 0 ? L0 : u);
  if (W == 4) {
    u = __shfl_up_sync(full, s, 2, gw);
    s += r16 * (gl == 0 ? T(0) : (gl == 1 ? L0 : u));
  }
  u = __shfl_up_sync(full, s, 1, gw);
  s = gl == 0 ? L0 : u;
  // (the corrections enter after the sums that neighbour chunks take, and R_n is formed without them)
  T Rn = T(0), endv = T(0);
  if (end) {
    T q = s, Ln = s, fn = f[0];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      q = f[j] + r * q;
      if (j + 1 < len) Ln = q, fn = f[j + 1];
    }
    if constexpr (MODE == kTrans) {
      const T En = fn + r * Ln;
      Rn = ir * En;
      endv = Ln + i1r * En;
    } else {
      Rn = i1r * fn - Ln;
    }
    pb += rlen * Rn;
  }
  s -= dL;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    e[j] = s;
    s = f[j] + r * s;
  }
  e[8] = s;
  // right sums: the chunk that holds position n continues with R_n
  t = pb + r8 * down(pb, 1);
  if (W == 4) t += r16 * down(t, 2);
  t = down(t, 1);
  if (end) t = Rn;
  t += dR;
  auto out = [&](T fj, T lj, T rj) { return MODE == kFirst ? rj - lj : (MODE == kSecond ? fj + r * (rj + lj) : lj - rj); };
  if (len > 8) {
    const T f8 = f[8];
    f[8] = out(f8, e[8], t);
    t = f8 + r * t;
  }
#pragma unroll
  for (int j = 7; j >= 0; --j) {
    const T fj = f[j];
    f[j] = out(fj, e[j], t);
    if (MODE == kTrans && j == 0 && c == 0) f[0] = -t - i1r * E0;
    if (j < len) t = fj + r * t;
  }
  if constexpr (MODE == kTrans) {
    if (end)
#pragma unroll
      for (int j = 0; j < 9; ++j)
        if (j == len - 1) f[j] = endv;
  }
}

// OP: NF, src(f) and void chunk(T (&e)[NF][9], int p0, int len, int64_t gi, int q): the positions p0 .. p0 + len - 1 of
// row q (flat index gi of position p0).  TWO (rows of one window, NF = 1): chunk leaves the samples of a second
// derivative along the same rows, also stored at src2(), in e, and chunk2 takes that derivative.
template <typename T, class OP>
__device__ __forceinline__ void row_block(const ConvAxis& g, const RowMap& rm, const OP& op, int bid, int nblk,
                                          unsigned char* sm) {
  constexpr int NF = OP::NF;
  __shared__ T rs[kReach];
  __shared__ ConvTap tsm[kTapsSmem];
  fill_reach(rs, g);
  const ConvTap* taps = stage_taps(g, tsm);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = rm.gw, rpw = 32 / gw;
  T* dsm = reinterpret_cast<T*>(sm + (size_t)warp * rm.wbytes);
  const int gl = lane & (gw - 1), k = lane / gw;
  const int items = rm.groups * rm.nwin;
  const int nw = blockDim.x >> 5;
  for (int item = bid * nw + warp; item < items; item += nblk * nw) {
    const int grp = rm.nwin == 1 ? item : item / rm.nwin, win = item - grp * rm.nwin;
    const int c0 = win * (32 - 2 * Conv<T>::W);              // first chunk of the window
    const int c1 = min(rm.nch, c0 + gw);                     // past its last
    const int o0 = win == 0 ? 0 : c0 + Conv<T>::W;           // own chunks
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
    const int64_t gi = rb + 8 * min(c, rm.nch - 1);  // of the chunk, or for lanes beyond the row of its last one
    const T rlen = end ? (T)__ldg(g.pw + len) : T(0);
    T e[NF][9];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
#pragma unroll
      for (int j = 0; j < 9; ++j) e[f][j] = T(0);
      if (len > 0) ld9(op.src(f) + gi, rm.vec, len, e[f]);
    }
    // junctions within Q of the own positions
    int j0 = 0, nj = 0;
    if (g.ntaps) {
      const int lo = 8 * o0, hi = o1 == rm.nch ? g.n : 8 * o1 - 1;
      j0 = lo <= g.Q ? 0 : small_div(lo - g.Q + g.M - 1, g.M);
      nj = min(g.p, small_div(hi + g.Q, g.M)) - j0 + 1;
    }
    // e of the NF fields whose samples are in e and at s0 (fields 1 ..: at op.src)
    auto derive = [&](const T* s0) {
      if (nj > 0) {  // G lanes per (field, row, junction)
        __syncwarp();
        const int tasks = NF * nrow * nj;
        const int lg = tasks > 16 ? 0 : (tasks > 8 ? 1 : (tasks > 4 ? 2 : 3));
        for (int i0 = 0; i0 < tasks; i0 += 32 >> lg) {
          const int i = i0 + (lane >> lg), ii = min(i, tasks - 1);
          const int fk = small_div(ii, nj), j = ii - fk * nj;
          int f = 0;
#pragma unroll
          for (int s = 1; s < NF; ++s) f += fk >= s * nrow;
          int64_t off = rpw == 1 ? rb : rbase(grp * rpw + fk - f * nrow);
#pragma unroll
          for (int s = 1; s < NF; ++s) off += f == s ? op.src(s) - s0 : (int64_t)0;
          const T D = conv_junction_part<T>(g, taps, j0 + j, s0 + off, lane & ((1 << lg) - 1), 1 << lg);
          if (i < tasks && (lane & ((1 << lg) - 1)) == 0) dsm[i] = D;
        }
        __syncwarp();
      }
      if (end && len < 8)
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (j >= len) e[f][j] = T(0);
      // the junctions before (or at the start of) the chunk and after it; at most one of each is within Q
      const int ja = small_div(8 * c, g.M), o0j = 8 * c - ja * g.M, o1j = o0j - g.M;  // the chunk's offsets from ja and ja + 1
      const int ia = ja - j0, ib = ia + 1;
      const bool hasa = len > 0 && ia >= 0 && ia < nj && o0j <= g.Q;
      const bool hasb = len > 0 && ib >= 0 && ib < nj && -o1j - 8 <= g.Q;
      const bool inb = hasb && -o1j < len;  // junction ja + 1 inside the chunk
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        T dL = T(0), dR = T(0);
        if (hasa) dL = dsm[(f * nrow + k) * nj + ia] * rs[64 + o0j];
        if (hasb && !inb) dR = dsm[(f * nrow + k) * nj + ib] * rs[64 - o1j - (len - 1)];
        row_solve<T>(e[f], c, len, end, gl, gw, rlen, dL, dR);
        if (inb) {
          const T D = dsm[(f * nrow + k) * nj + ib];
#pragma unroll
          for (int j = 0; j < 9; ++j) e[f][j] += D * rs[64 + o1j + j];
        }
      }
    };
    const bool own = len > 0 && c >= o0 && c < o1;
    T q2[9];
    if constexpr (OP::SECOND) {  // second differences, 0 at the line's ends
      const T fm = __shfl_up_sync(0xffffffffu, e[0][7], 1, gw), fp = __shfl_down_sync(0xffffffffu, e[0][0], 1, gw);
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        const T m = j == 0 ? fm : e[0][j - 1];
        const T p = j == 8 ? T(0) : (j == 7 ? (len > 8 ? e[0][8] : fp) : e[0][j + 1]);
        const bool in = j < len && !(c == 0 && j == 0) && !(end && j == len - 1);
        q2[j] = in ? (p - e[0][j]) - (e[0][j] - m) : T(0);
      }
    }
    derive(op.src(0));
    if (own) op.chunk(e, 8 * c, len, gi, q);
    if constexpr (OP::SECOND) {
      row_solve<T, kSecond>(q2, c, len, end, gl, gw, rlen, T(0), T(0));
      if (nj > 0 && len > 0) {
        const int ja = small_div(8 * c, g.M);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const int jj = ja + s - j0, o = 8 * c - (ja + s) * g.M;
          if (jj >= 0 && jj < nj && o <= g.Q && -o - 8 <= g.Q)
            add_second(q2, dsm[k * nj + jj], o, ja + s, g, rs);
        }
      }
      if (own) op.chunk2nd(q2, 8 * c, len, gi);
    }
    if constexpr (OP::TWO) {
      if (!own)  // lanes beyond the row carry no samples into the second derivative
#pragma unroll
        for (int j = 0; j < 9; ++j) e[0][j] = T(0);
      derive(op.src2());
      if (own) op.chunk2(e, 8 * c, len, gi, q);
    }
  }
}

template <typename T, class OP>
__global__ void __launch_bounds__(128, OP::kBlocks) k_row(ConvAxis g, RowMap rm, OP op) {
  extern __shared__ __align__(16) unsigned char sm[];
  row_block<T>(g, rm, op, blockIdx.x, gridDim.x, sm);
}

// All shots in one launch, as k_col_batch; blk[b].z: blocks of the shot.
template <typename T, class OP>
struct RowJob {
  ConvAxis g;
  RowMap rm;
  OP op;
};
template <typename T, class OP>
__global__ void __launch_bounds__(128, OP::kBlocks)
    k_row_batch(const RowJob<T, OP>* __restrict__ jobs, const int4* __restrict__ blk) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ __align__(16) unsigned char raw[sizeof(RowJob<T, OP>)];
  const int4 w = blk[blockIdx.x];
  RowJob<T, OP>& j = *reinterpret_cast<RowJob<T, OP>*>(raw);
  copy_job(&j, jobs + w.x);
  __syncthreads();
  row_block<T>(j.g, j.rm, j.op, w.y, w.z, sm);
}

}  // namespace lossk
