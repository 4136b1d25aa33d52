// sm_103a kernels of the 2-D acoustic step on the barrier-free engines of loss_stream.cuh: the FP64 step and the
// x part of FP32 rows, long ones and those that the pipelined row kernel does not take (per shot and batched).
//
//   rows B:  sigma += -dt kappa (d_x v1 + d_z v3) + source          rows A:  v1 += -tau b d_x sigma
//   cols Z1: v3 += -tau b d_z sigma                                 cols Z2: tmp = d_z v3
// Rows of one window (at most 257 points) take B and A in one launch: the new sigma of a row stays in the registers of
// the lanes that computed it.
//
// The FP64 line kernels held whole lines of one block behind seven barriers per derivative and spent 11 FP64 operations
// per point and derivative; FP64 runs at 2 FMA per SM and clock here, so operations are what the step costs.  These spend
// about 5 (two warm-up sums, two recursions, one difference) plus the pointwise update: 1025^2 step 251 us -> 175 us.
// 129^2 (154 us -> 92 us) waits for the serial FP64 chain of a line's chunks.  FP32 rows are bound by issue slots and
// latency (2049^2 x part with Kahan summation 67 us on the pipelined kernel, 63 us here, 44 bytes a point).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "../../include/loss.h"
#include "loss_host.h"
#include "loss_stream.cuh"
#include "loss_types.h"

namespace lossk {

// Pointers that a launch does not use (no layer, constant density) are readable ones; b_on: the density is an array.
// TAB: the source amplitude of the step comes from the shot's device table and clock (batched launches).
template <typename T, bool KAHAN, bool REC, bool DOB, bool DOA, bool TAB>
struct AcRowOp {
  static constexpr int NF = 1;
  static constexpr bool SECOND = false;
  static constexpr bool TWO = DOB && DOA;
  static constexpr int kBlocks = sizeof(T) == 8 ? 3 : 4;
  AcXArgs<T> a;
  int b_on, pad;
  __device__ __forceinline__ const T* src(int) const { return DOB ? a.v1 : a.sigma; }
  __device__ __forceinline__ const T* src2() const { return a.sigma; }
  __device__ __forceinline__ void chunk(T (&e)[1][9], int p0, int len, int64_t gi, int q) const {
    if constexpr (DOB) stress(e[0], p0, len, gi, q);
    else velocity(e[0], p0, len, gi);
  }
  __device__ __forceinline__ void chunk2(T (&e)[1][9], int p0, int len, int64_t gi, int) const {
    velocity(e[0], p0, len, gi);
  }
  // increment -tau g, or the layer's sub-flow (PmlAxis::step) from the memory value m; m becomes the new value
  static __device__ __forceinline__ T flow(const T* tab, int n1, int i, T g, T& m) {
    const T m1 = tab[i] * m - tab[n1 + i] * g;
    const T x = tab[2 * n1 + i] * (m1 - m) - tab[3 * n1 + i] * g;
    m = m1;
    return x;
  }
  // sub-step B of a chunk; leaves the new sigma in e.  (The ninth position exists in a row's last chunk at most: every
  // loop leaves before it otherwise.)
  __device__ __forceinline__ void stress(T (&e)[9], int p0, int len, int64_t gi, int q) const {
    const bool lay = a.pml && (a.xB.in(p0) || a.xB.in(p0 + len - 1));
    const bool zlay = a.pml && a.zB.in(q);
    T sg[9], kp[9], gz[9], cs[9], mx[9], mz[9];
    ld9(a.sigma + gi, true, len, sg);
    ld9(a.kappa + gi, true, len, kp);
    ld9(a.tmp + gi, true, len, gz);
    if constexpr (KAHAN) ld9(a.csig + gi, true, len, cs);
    if (lay) ld9(a.phix + gi, true, len, mx);
    if (zlay) ld9(a.phiz + gi, true, len, mz);
    if (zlay) {
      const int n1 = a.zB.n + 1;
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        if (j == 8 && len < 9) break;
        gz[j] = -flow(a.zB.tab, n1, q, gz[j], mz[j]);
      }
      st9(a.phiz + gi, true, len, mz);
    } else {
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        if (j == 8 && len < 9) break;
        gz[j] = mulc1(gz[j], a.dt, a.dt_lo);
      }
    }
    if (lay) {
      const int n1 = a.xB.n + 1;
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        if (j == 8 && len < 9) break;
        if (j < len && a.xB.in(p0 + j)) e[j] = -flow(a.xB.tab, n1, min(p0 + j, a.xB.n), mulc1(e[j], a.s3h, a.s3h_lo), mx[j]);
        else e[j] = mulc1(e[j], a.sdt, a.sdt_lo);
      }
      st9(a.phix + gi, true, len, mx);
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        if (j == 8 && len < 9) break;
        e[j] += gz[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        if (j == 8 && len < 9) break;
        if constexpr (sizeof(T) == 8) e[j] = fma(e[j], a.sdt, gz[j]);
        else e[j] = mulc1(e[j], a.sdt, a.sdt_lo) + gz[j];
      }
    }
    // e = minus the divergence's increment: sigma += -kappa e (+ source)
    if (a.src.on && (unsigned)(q - a.src.zs + 12) < 25u) {
      double amp = a.src.amp;
      if constexpr (TAB) amp = a.src.amp_tab[a.src.clk->step];
      if (amp != 0.0)
#pragma unroll
        for (int j = 0; j < 9; ++j) {
          const int dx = p0 + j - a.src.xs + 12;
          if (j < len && (unsigned)dx < 25u) {
            const T sv = (T)(amp * a.src.g[min((unsigned)(q - a.src.zs + 12), 24u)] * a.src.g[min((unsigned)dx, 24u)]);
            if constexpr (KAHAN) {
              e[j] = -kp[j] * e[j] + sv;
              kp[j] = T(-1);
            } else {
              sg[j] += sv;
            }
          }
        }
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      if (j == 8 && len < 9) break;
      if constexpr (KAHAN) {
        float v = sg[j], c = cs[j];
        kahan_add(v, c, -kp[j] * e[j]);
        e[j] = v;
        cs[j] = c;
      } else {
        e[j] = fma(-kp[j], e[j], sg[j]);
      }
    }
    st9(a.sigma + gi, true, len, e);
    if constexpr (KAHAN) st9(a.csig + gi, true, len, cs);
    if constexpr (TWO) {  // samples of the second derivative: nothing beyond the chunk
#pragma unroll
      for (int j = 0; j < 9; ++j)
        if (j >= len) e[j] = T(0);
    }
  }
  // x part of sub-step A of a chunk
  __device__ __forceinline__ void velocity(T (&e)[9], int p0, int len, int64_t gi) const {
    const bool lay = a.pml && (a.xA.in(p0) || a.xA.in(p0 + len - 1));
    T v[9], c[9], bb[9], m[9];
    ld9(a.v1 + gi, true, len, v);
    if constexpr (KAHAN) ld9(a.cv1 + gi, true, len, c);
    if (b_on) ld9(a.b + gi, true, len, bb);
    if (lay) ld9(a.psix + gi, true, len, m);
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      if (j == 8 && len < 9) break;
      if (lay && j < len && a.xA.in(p0 + j)) {
        const int n1 = a.xA.n + 1, i = min(p0 + j, a.xA.n);
        const T g = mulc1(e[j], a.s3h, a.s3h_lo), m0 = m[j];
        e[j] = flow(a.xA.tab, n1, i, g, m[j]);
        if constexpr (REC) {
          T mh = m0;
          const T ih = flow(a.xA.tabh, n1, i, g, mh);
          a.dlt[gi + j] = (b_on ? bb[j] : a.b0) * (ih - T(0.5) * e[j]);
        }
        e[j] = b_on ? bb[j] * e[j] : mulc1(e[j], a.b0, a.b0_lo);
      } else if (b_on) {
        e[j] = bb[j] * mulc1(e[j], a.sa, a.sa_lo);
      } else if constexpr (sizeof(T) == 8) {
        v[j] = fma(e[j], a.sc, v[j]);
        e[j] = T(0);
      } else {
        e[j] = mulc1(e[j], a.sc, a.sc_lo);
      }
    }
    if (lay) st9(a.psix + gi, true, len, m);
    if (sizeof(T) == 4 || b_on || lay) {
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        if (j == 8 && len < 9) break;
        if constexpr (KAHAN) {
          float vv = v[j], cc = c[j];
          kahan_add(vv, cc, e[j]);
          v[j] = vv;
          c[j] = cc;
        } else {
          v[j] += e[j];
        }
      }
    }
    st9(a.v1 + gi, true, len, v);
    if constexpr (KAHAN) st9(a.cv1 + gi, true, len, c);
  }
};

// Columns, FP64 (the FP32 z part runs on the tiles).
template <int MODE, bool REC>
struct AcColOp {
  using T = double;
  static constexpr int NF = 1;
  static constexpr bool SECOND = false;
  static constexpr int kBlocks = 4;
  static constexpr int B = MODE == 1 ? 4 : 1;
  AcZArgs<T> a;
  int b_on, pad;
  struct Regs {
    T v, b, m;
  };
  __device__ __forceinline__ const T* src(int) const { return MODE == 1 ? a.sigma : a.v3; }
  __device__ __forceinline__ void load(Regs& r, int pos, uint32_t o) const {
    if constexpr (MODE == 1) {
      r.v = at_off(a.v3, o);
      if (b_on) r.b = at_off(a.b, o);
      if (a.pml && a.zA.in(pos)) r.m = at_off(a.psiz, o);
    }
  }
  __device__ __forceinline__ void apply(Regs& r, const T (&e)[1], int pos, uint32_t o, int, int) const {
    if constexpr (MODE == 2) {
      at_off(a.tmp, o) = mulc(e[0], a.s3h, a.s3h_lo);
    } else if (a.pml && a.zA.in(pos)) {
      const T g = mulc(e[0], a.s3h, a.s3h_lo);
      const int n1 = a.zA.n + 1;
      const T* t = a.zA.tab;
      const T m1 = t[pos] * r.m - t[n1 + pos] * g;
      const T inc = t[2 * n1 + pos] * (m1 - r.m) - t[3 * n1 + pos] * g;
      const T bb = b_on ? r.b : a.b0;
      if constexpr (REC) {
        const T* th = a.zA.tabh;
        const T mh = th[pos] * r.m - th[n1 + pos] * g;
        const T ih = th[2 * n1 + pos] * (mh - r.m) - th[3 * n1 + pos] * g;
        at_off(a.dlt, o) = bb * (ih - T(0.5) * inc);
      }
      at_off(a.psiz, o) = m1;
      at_off(a.v3, o) = r.v + bb * inc;
    } else {
      at_off(a.v3, o) = b_on ? fma(r.b * -(a.s3h * a.acoef), e[0], r.v) : fma(e[0], a.sc, r.v);
    }
  }
};

template <typename T>
static void fill_unused(AcXArgs<T>& a) {
  if (!a.b) a.b = a.v1;
  if (!a.tmp) a.tmp = a.v1;
  if (!a.kappa) a.kappa = a.v1;
  if (!a.pml) {
    a.phix = a.phiz = a.psix = a.v1;
    a.xA.tab = a.xB.tab = a.zB.tab = a.v1;
  }
}
template <typename T>
static void fill_unused(AcZArgs<T>& a) {
  if (!a.b) a.b = a.v3;
  if (!a.pml) {
    a.psiz = a.v3;
    a.zA.tab = a.v3;
  }
}

template <typename T, class OP>
static cudaError_t go_row(const ConvAxis& g, const RowMap& rm, const OP& op, cudaStream_t st) {
  const size_t smem = (size_t)rm.warps * rm.wbytes;
  auto kern = k_row<T, OP>;
  if (smem > 32 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemMax);
    if (e != cudaSuccess) return e;
  }
  kern<<<row_blocks(rm, OP::kBlocks, rm.warps), 32 * rm.warps, smem, st>>>(g, rm, op);
  return cudaGetLastError();
}
template <typename T, class OP>
static cudaError_t go_col(const ConvAxis& g, const ColMap& cm, const OP& op, cudaStream_t st) {
  const size_t smem = col_smem<T>(OP::NF, cm.warps);
  auto kern = k_col<T, OP>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)col_smem<T>(OP::NF, 4));
  if (e != cudaSuccess) return e;
  kern<<<col_blocks(cm, cm.warps), 32 * cm.warps, smem, st>>>(g, cm, op);
  return cudaGetLastError();
}

// Sub-step B (when do_B) and the x part of A: one launch for rows of one window, else two.
template <typename T, bool KAHAN>
cudaError_t launch_ac_rows(const AcXArgs<T>& a, const ConvAxis& g, const RowMap& rm, cudaStream_t st) {
  const int b_on = a.b ? 1 : 0;
  const bool rec = a.pml && a.dlt;
  AcXArgs<T> f = a;
  fill_unused(f);
  if (a.do_B && rm.nwin == 1) {
    if (rec) return go_row<T>(g, rm, AcRowOp<T, KAHAN, true, true, true, false>{f, b_on, 0}, st);
    return go_row<T>(g, rm, AcRowOp<T, KAHAN, false, true, true, false>{f, b_on, 0}, st);
  }
  if (a.do_B) {
    const cudaError_t e = go_row<T>(g, rm, AcRowOp<T, KAHAN, false, true, false, false>{f, b_on, 0}, st);
    if (e != cudaSuccess) return e;
  }
  if (rec) return go_row<T>(g, rm, AcRowOp<T, KAHAN, true, false, true, false>{f, b_on, 0}, st);
  return go_row<T>(g, rm, AcRowOp<T, KAHAN, false, false, true, false>{f, b_on, 0}, st);
}
// mode 1: Z1, mode 2: Z2.
cudaError_t launch_ac_cols(const AcZArgs<double>& a, const ConvAxis& g, const ColMap& cm, int mode, cudaStream_t st) {
  const int b_on = a.b ? 1 : 0;
  AcZArgs<double> f = a;
  fill_unused(f);
  if (mode == 2) return go_col<double>(g, cm, AcColOp<2, false>{f, b_on, 0}, st);
  if (a.pml && a.dlt) return go_col<double>(g, cm, AcColOp<1, true>{f, b_on, 0}, st);
  return go_col<double>(g, cm, AcColOp<1, false>{f, b_on, 0}, st);
}
template cudaError_t launch_ac_rows<float, false>(const AcXArgs<float>&, const ConvAxis&, const RowMap&, cudaStream_t);
template cudaError_t launch_ac_rows<float, true>(const AcXArgs<float>&, const ConvAxis&, const RowMap&, cudaStream_t);
template cudaError_t launch_ac_rows<double, false>(const AcXArgs<double>&, const ConvAxis&, const RowMap&,
                                                   cudaStream_t);

// ---------------------------------------------------------------------------------------------------------------
// Batched step.  Every shot keeps the kernels and the block-to-work mapping of its own launches (so the results are
// theirs bit for bit); one launch runs the blocks of all shots of one kind.  Kinds: 0, 1 rows B + A of one-window rows
// (without and with receiver corrections), 2 rows B, 3, 4 rows A, 5, 6 cols Z1, 7 cols Z2 (FP64).  FP32: kinds 2
// to 4, rows of at least 513 points; the columns are the batched z tiles'.
template <typename D, bool K, class F>
static void with_kind(int kind, F&& f) {
  switch (kind) {
    case 2: return f(RowJob<D, AcRowOp<D, K, false, true, false, true>>{});
    case 3: return f(RowJob<D, AcRowOp<D, K, false, false, true, true>>{});
    case 4: return f(RowJob<D, AcRowOp<D, K, true, false, true, true>>{});
  }
  if constexpr (sizeof(D) == 8) {
    switch (kind) {
      case 0: return f(RowJob<D, AcRowOp<D, K, false, true, true, true>>{});
      case 1: return f(RowJob<D, AcRowOp<D, K, true, true, true, true>>{});
      case 5: return f(ColJob<D, AcColOp<1, false>>{});
      case 6: return f(ColJob<D, AcColOp<1, true>>{});
      default: return f(ColJob<D, AcColOp<2, false>>{});
    }
  }
}
template <class J>
struct JobTraits;
template <typename T, class OP>
struct JobTraits<RowJob<T, OP>> {
  static constexpr int kInts = 4;  // ints per entry of the block table
  static RowJob<T, OP> make(const AcStreamShot<T>& s) {
    RowJob<T, OP> j{s.gx, s.rm, {s.x, s.x.b ? 1 : 0, 0}};
    fill_unused(j.op.a);
    return j;
  }
  static int blocks(const AcStreamShot<T>& s) { return row_blocks(s.rm, OP::kBlocks, 4); }
  static size_t smem(const AcStreamShot<T>& s) { return (size_t)4 * s.rm.wbytes; }
  static cudaError_t launch(const unsigned char* base, const AcBatchKind& k, cudaStream_t st) {
    auto kern = k_row_batch<T, OP>;
    if (k.smem > 32 * 1024) {
      const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemMax);
      if (e != cudaSuccess) return e;
    }
    kern<<<k.blocks, 128, k.smem, st>>>((const RowJob<T, OP>*)(base + k.jobs), (const int4*)(base + k.blk));
    return cudaGetLastError();
  }
};
template <typename T, class OP>
struct JobTraits<ColJob<T, OP>> {
  static constexpr int kInts = 2;
  static ColJob<T, OP> make(const AcStreamShot<T>& s) {
    ColJob<T, OP> j{s.gz, s.cm, {s.z, s.z.b ? 1 : 0, 0}};
    fill_unused(j.op.a);
    return j;
  }
  static int blocks(const AcStreamShot<T>& s) { return (int)col_blocks(s.cm, 4); }
  static size_t smem(const AcStreamShot<T>&) { return col_smem<T>(OP::NF, 4); }
  static cudaError_t launch(const unsigned char* base, const AcBatchKind& k, cudaStream_t st) {
    auto kern = k_col_batch<T, OP>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    if (e != cudaSuccess) return e;
    kern<<<k.blocks, 128, k.smem, st>>>((const ColJob<T, OP>*)(base + k.jobs), (const int2*)(base + k.blk));
    return cudaGetLastError();
  }
};
template <typename T>
static bool in_kind(int kind, const AcStreamShot<T>& s) {
  const bool one = s.rm.nwin == 1, rx = s.x.pml && s.x.dlt, rz = s.z.pml && s.z.dlt;
  switch (kind) {
    case 0: return one && !rx;
    case 1: return one && rx;
    case 2: return !one;
    case 3: return !one && !rx;
    case 4: return !one && rx;
    case 5: return !rz;
    case 6: return rz;
    default: return true;
  }
}

// The job and block tables of every kind in `bytes` (uploaded to a 16-byte aligned address) and where they lie.
template <typename T, bool K>
void ac_batch_tables(const std::vector<AcStreamShot<T>>& shots, std::vector<unsigned char>& bytes, AcBatchKind (&k)[8]) {
  bytes.clear();
  for (int kind = 0; kind < 8; ++kind) {
    k[kind] = AcBatchKind{};
    with_kind<T, K>(kind, [&](auto proto) {
      using J = decltype(proto);
      using Tr = JobTraits<J>;
      std::vector<J> jobs;
      std::vector<int> blk;
      AcBatchKind& q = k[kind];
      for (const AcStreamShot<T>& s : shots) {
        if (!in_kind(kind, s)) continue;
        const int nb = Tr::blocks(s);
        for (int b = 0; b < nb; ++b) {
          blk.push_back((int)jobs.size());
          blk.push_back(b);
          if (Tr::kInts == 4) blk.insert(blk.end(), {nb, 0});
        }
        q.blocks += nb;
        q.smem = std::max(q.smem, Tr::smem(s));
        jobs.push_back(Tr::make(s));
      }
      auto put = [&](const void* p, size_t n) {
        const size_t o = (bytes.size() + 15) & ~(size_t)15;
        bytes.resize(o + n);
        if (n) std::memcpy(bytes.data() + o, p, n);
        return o;
      };
      q.jobs = put(jobs.data(), jobs.size() * sizeof(J));
      q.blk = put(blk.data(), blk.size() * sizeof(int));
    });
  }
}

template <typename T, bool K>
cudaError_t launch_ac_batch(const void* base, const AcBatchKind& k, int kind, cudaStream_t st) {
  if (k.blocks == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  with_kind<T, K>(kind, [&](auto proto) { e = JobTraits<decltype(proto)>::launch((const unsigned char*)base, k, st); });
  return e;
}

template void ac_batch_tables<float, false>(const std::vector<AcStreamShot<float>>&, std::vector<unsigned char>&,
                                            AcBatchKind (&)[8]);
template void ac_batch_tables<float, true>(const std::vector<AcStreamShot<float>>&, std::vector<unsigned char>&,
                                           AcBatchKind (&)[8]);
template void ac_batch_tables<double, false>(const std::vector<AcStreamShot<double>>&, std::vector<unsigned char>&,
                                             AcBatchKind (&)[8]);
template cudaError_t launch_ac_batch<float, false>(const void*, const AcBatchKind&, int, cudaStream_t);
template cudaError_t launch_ac_batch<float, true>(const void*, const AcBatchKind&, int, cudaStream_t);
template cudaError_t launch_ac_batch<double, false>(const void*, const AcBatchKind&, int, cudaStream_t);

}  // namespace lossk
