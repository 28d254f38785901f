// Fused back-substitution epilogues shared by the SIMT and tensor-core kernels.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "mnbab_internal.h"

namespace mnbab {

// two FP32 FMAs in one instruction, each rounded as fmaf
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)),
        "l"(*reinterpret_cast<unsigned long long*>(&b)),
        "l"(*reinterpret_cast<unsigned long long*>(&c)));
  return *reinterpret_cast<float2*>(&r);
}

// x / d for 0 <= x < 2^31 by the rounded-down reciprocal m = floor((2^32 - 1) / d):
// the high product is the quotient or one less.  A convolution kernel decodes each
// of its items with several divisions by layer sizes.
struct FDiv {
  unsigned d, m;
};
__host__ __device__ inline FDiv f_div_of(int d) {
  return FDiv{(unsigned)d, 0xffffffffu / (unsigned)d};
}
__device__ __forceinline__ int f_div(int x, FDiv v) {
  const unsigned q = __umulhi((unsigned)x, v.m);
  return (int)(q + ((unsigned)x - q * v.d >= v.d ? 1u : 0u));
}
__device__ __forceinline__ int f_mod(int x, FDiv v) { return x - f_div(x, v) * (int)v.d; }

// ---------------------------------------------------------------------------
// epilogues
// ---------------------------------------------------------------------------
// ReLU back-substitution of one coefficient a on z_j (Sec. 3.1, combined ReLU
// step): a' = a + (gamma^T P)_j, D / blow from the single-neuron table with
// split precedence, ahat = a' D + beta S + (gamma^T Phat)_j.  The offset
// contribution a' blow + ahat b_j (bias of the consuming affine layer) goes to
// the row partial sum.
__device__ __forceinline__ float epi_relu(const Epi& e, int m, int j, float a, float& part) {
  const int n = e.row_node[m];
  const size_t q = (size_t)n * e.SD + e.off + j;
  const size_t qm = (size_t)m * e.SD + e.off + j;
  const float l = e.pool.L[q], u = e.pool.U[q];
  const int s = e.pool.S[q];
  float ap = a;
  if (e.GP) ap += e.GP[qm];
  float D, bl = 0.f;
  if (s == -1) D = 1.f;
  else if (s == 1) D = 0.f;
  else if (l >= 0.f) D = 1.f;
  else if (u <= 0.f) D = 0.f;
  else if (ap >= 0.f) D = e.final_mode ? e.pool.ALPHA[q] : (u >= -l ? 1.f : 0.f);
  else {
    const float den = u - l;
    D = u / den;
    bl = (-u * l) / den;
  }
  float ah = ap * D;
  if (e.final_mode) ah += e.pool.BETA[q] * (float)s;
  if (e.GPh) ah += e.GPh[qm];
  if (e.AP) e.AP[qm] = ap;
  part += ap * bl + ah * e.bias[j / e.bias_div];
  return ah;
}

// Concretisation of a coefficient on input x_j over [lo, hi] (Eq. minimum):
// x*_j = lo_j if a >= 0 else hi_j, contribution a x*_j.
__device__ __forceinline__ float epi_conc(const Epi& e, int m, int j, float a, float& part) {
  const int n = e.row_node[m];
  const PropDev& P = e.props[e.pool.prop[n]];
  const float x = a >= 0.f ? P.lo[j] : P.hi[j];
  part += a * x;
  if (e.X) e.X[(size_t)m * e.d0 + j] = x;
  return a;
}

// Adjoint of the ReLU step at pre-activation adjoint h = d lb / d ahat_j:
// d lb / d alpha_j = h a'_j on the alpha branch, d lb / d beta_j = h S_j,
// and d lb / d a'_j = h D_j + blow_j flows to the next layer.
__device__ __forceinline__ float epi_adj(const Epi& e, int m, int j, float h) {
  const int n = e.row_node[m];
  const size_t q = (size_t)n * e.SD + e.off + j;
  const size_t qm = (size_t)m * e.SD + e.off + j;
  const float l = e.pool.L[q], u = e.pool.U[q];
  const int s = e.pool.S[q];
  const float ap = e.AP[qm];
  float D, bl = 0.f;
  bool abr = false;
  if (s == -1) D = 1.f;
  else if (s == 1) D = 0.f;
  else if (l >= 0.f) D = 1.f;
  else if (u <= 0.f) D = 0.f;
  else if (ap >= 0.f) { D = e.pool.ALPHA[q]; abr = true; }
  else {
    const float den = u - l;
    D = u / den;
    bl = (-u * l) / den;
  }
  e.GA[qm] = abr ? h * ap : 0.f;
  e.GB[qm] = h * (float)s;
  const float g = h * D + bl;
  if (e.Hz) {
    e.Hz[qm] = h;
    e.Gz[qm] = g;
  }
  return g;
}

__device__ __forceinline__ float epi_apply(const Epi& e, int m, int j, float v, float& part) {
  // a node that sums two affine edges: the first edge's contribution is added
  // before the epilogue of the second
  if (e.acc_in) v += e.acc_in[(size_t)m * e.acc_ld + j];
  switch (e.kind) {
    case EPI_RELU: return epi_relu(e, m, j, v, part);
    case EPI_CONC: return epi_conc(e, m, j, v, part);
    case EPI_ADJ: return epi_adj(e, m, j, v);
    case EPI_FWD_RELU: return fmaxf(v, 0.f);
    default: return v;
  }
}

// Two-phase form of epi_apply for kernels that finish several outputs per
// thread: epi_load_node and epi_load_own issue every global load an output's
// epilogue needs (so the loads of all of a thread's outputs are in flight together),
// epi_finish does the same arithmetic as epi_apply on the loaded values.
struct EpiIn {
  float acc, l, u, al, be, gp, gph;
  float cb;  // bias of the consuming affine layer at j (ReLU step)
  int s;
};

__device__ __forceinline__ const PropDev* epi_prop(const Epi& e, int n) {
  return e.kind == EPI_CONC ? &e.props[e.pool.prop[n]] : nullptr;
}

// the part of an output's inputs that depends on its column j only
__device__ __forceinline__ float epi_colbias(const Epi& e, int j) {
  return e.kind == EPI_RELU ? e.bias[j / e.bias_div] : 0.f;
}

// every input of output (m, j) except the column bias (in.cb), in two parts: the
// inputs that depend on the node and column only
// (bounds, split, slope, multiplier; the input box), which rows of one node can
// share, and those of the row itself
__device__ __forceinline__ void epi_load_node(const Epi& e, int n, const PropDev* P, int j,
                                              EpiIn& in) {
  in.al = in.be = 0.f;
  in.s = 0;
  if (e.kind == EPI_RELU || e.kind == EPI_ADJ) {
    const size_t q = (size_t)n * e.SD + e.off + j;
    in.l = e.pool.L[q];
    in.u = e.pool.U[q];
    in.s = e.pool.S[q];
    if (e.kind == EPI_ADJ || e.final_mode) in.al = e.pool.ALPHA[q];
    if (e.kind == EPI_RELU && e.final_mode) in.be = e.pool.BETA[q];
  } else if (e.kind == EPI_CONC) {
    in.l = P->lo[j];
    in.u = P->hi[j];
  }
}

__device__ __forceinline__ void epi_load_own(const Epi& e, int m, int j, EpiIn& in) {
  in.acc = e.acc_in ? e.acc_in[(size_t)m * e.acc_ld + j] : 0.f;
  in.gp = in.gph = 0.f;
  const size_t qm = (size_t)m * e.SD + e.off + j;
  if (e.kind == EPI_RELU) {
    if (e.GP) in.gp = e.GP[qm];
    if (e.GPh) in.gph = e.GPh[qm];
  } else if (e.kind == EPI_ADJ) {
    in.gp = e.AP[qm];
  }
}

__device__ __forceinline__ float epi_finish(const Epi& e, int m, int j, float v, const EpiIn& in,
                                            float& part) {
  if (e.acc_in) v += in.acc;
  switch (e.kind) {
    case EPI_RELU: {
      const size_t qm = (size_t)m * e.SD + e.off + j;
      const float l = in.l, u = in.u;
      const int s = in.s;
      float ap = v;
      if (e.GP) ap += in.gp;
      float D, bl = 0.f;
      if (s == -1) D = 1.f;
      else if (s == 1) D = 0.f;
      else if (l >= 0.f) D = 1.f;
      else if (u <= 0.f) D = 0.f;
      else if (ap >= 0.f) D = e.final_mode ? in.al : (u >= -l ? 1.f : 0.f);
      else {
        const float den = u - l;
        D = u / den;
        bl = (-u * l) / den;
      }
      float ah = ap * D;
      if (e.final_mode) ah += in.be * (float)s;
      if (e.GPh) ah += in.gph;
      if (e.AP) e.AP[qm] = ap;
      part += ap * bl + ah * in.cb;
      return ah;
    }
    case EPI_CONC: {
      const float x = v >= 0.f ? in.l : in.u;
      part += v * x;
      if (e.X) e.X[(size_t)m * e.d0 + j] = x;
      return v;
    }
    case EPI_ADJ: {
      const size_t qm = (size_t)m * e.SD + e.off + j;
      const float l = in.l, u = in.u, ap = in.gp, h = v;
      const int s = in.s;
      float D, bl = 0.f;
      bool abr = false;
      if (s == -1) D = 1.f;
      else if (s == 1) D = 0.f;
      else if (l >= 0.f) D = 1.f;
      else if (u <= 0.f) D = 0.f;
      else if (ap >= 0.f) { D = in.al; abr = true; }
      else {
        const float den = u - l;
        D = u / den;
        bl = (-u * l) / den;
      }
      e.GA[qm] = abr ? h * ap : 0.f;
      e.GB[qm] = h * (float)s;
      const float g = h * D + bl;
      if (e.Hz) {
        e.Hz[qm] = h;
        e.Gz[qm] = g;
      }
      return g;
    }
    case EPI_FWD_RELU: return fmaxf(v, 0.f);
    default: return v;
  }
}

// The two-phase form with the kind of epilogue as a template parameter, for
// kernels that are instantiated per kind: a kernel that finishes many outputs per
// thread and switches on the kind at each is several times as long, and its CTAs
// wait for instructions more than for data.  The arithmetic is epi_finish's.
enum EpiMode { EM_RELU, EM_RELU_FINAL, EM_RELU_GAMMA, EM_CONC, EM_ADJ, EM_ADJ_GAMMA, EM_FWD, EM_STORE };

inline EpiMode epi_mode(const Epi& e) {
  switch (e.kind) {
    case EPI_RELU: return !e.final_mode ? EM_RELU : e.GP ? EM_RELU_GAMMA : EM_RELU_FINAL;
    case EPI_CONC: return EM_CONC;
    case EPI_ADJ: return e.Hz ? EM_ADJ_GAMMA : EM_ADJ;
    case EPI_FWD_RELU: return EM_FWD;
    default: return EM_STORE;
  }
}

// calls go(mode as a constant) for an epilogue of the back-substitution / of the
// forward pass
template <typename F>
inline void epi_dispatch_back(const Epi& e, F&& go) {
  switch (epi_mode(e)) {
    case EM_RELU: go(std::integral_constant<int, EM_RELU>{}); break;
    case EM_RELU_FINAL: go(std::integral_constant<int, EM_RELU_FINAL>{}); break;
    case EM_RELU_GAMMA: go(std::integral_constant<int, EM_RELU_GAMMA>{}); break;
    case EM_CONC: go(std::integral_constant<int, EM_CONC>{}); break;
    default: go(std::integral_constant<int, EM_STORE>{}); break;
  }
}
template <typename F>
inline void epi_dispatch_fwd(const Epi& e, F&& go) {
  switch (epi_mode(e)) {
    case EM_ADJ: go(std::integral_constant<int, EM_ADJ>{}); break;
    case EM_ADJ_GAMMA: go(std::integral_constant<int, EM_ADJ_GAMMA>{}); break;
    case EM_FWD: go(std::integral_constant<int, EM_FWD>{}); break;
    default: go(std::integral_constant<int, EM_STORE>{}); break;
  }
}

// calls go(mode as a constant) for any epilogue
template <typename F>
inline void epi_dispatch(const Epi& e, F&& go) {
  if (e.kind == EPI_ADJ || e.kind == EPI_FWD_RELU) epi_dispatch_fwd(e, go);
  else epi_dispatch_back(e, go);
}

// whether a zero coefficient passes the epilogue as a zero that adds nothing to
// the row's offset
template <int EM>
__device__ __forceinline__ bool epi_zero_passes(const Epi& e) {
  return !e.acc_in && ((EM == EM_RELU && !e.AP) || (EM == EM_CONC && !e.X) || EM == EM_STORE);
}

// (an earlier edge's contribution, in.acc, is loaded by epi_finish_block)
template <int EM>
__device__ __forceinline__ void epi_load_m(const Epi& e, int n, const PropDev* P, int m, int j,
                                           EpiIn& in) {
  const size_t q = (size_t)n * e.SD + e.off + j, qm = (size_t)m * e.SD + e.off + j;
  if constexpr (EM <= EM_RELU_GAMMA) {
    in.l = e.pool.L[q];
    in.u = e.pool.U[q];
    in.s = e.pool.S[q];
    in.cb = e.bias[j];
    if constexpr (EM >= EM_RELU_FINAL) {
      in.al = e.pool.ALPHA[q];
      in.be = e.pool.BETA[q];
    }
    if constexpr (EM == EM_RELU_GAMMA) {
      in.gp = e.GP[qm];
      in.gph = e.GPh[qm];
    }
  } else if constexpr (EM == EM_ADJ || EM == EM_ADJ_GAMMA) {
    in.l = e.pool.L[q];
    in.u = e.pool.U[q];
    in.s = e.pool.S[q];
    in.al = e.pool.ALPHA[q];
    in.gp = e.AP[qm];
  } else if constexpr (EM == EM_CONC) {
    in.l = P->lo[j];
    in.u = P->hi[j];
  }
}

// Finishes K outputs (m, j[i]) of one row with values v[i], in place; ok: bit i is
// set where output i counts (every j[i] is a valid index; nothing is stored or
// summed for the others).  The relaxation's two divisions are needed only where
// an unstable neuron has a negative coefficient: the outputs' other arithmetic is
// free of branches, and a lane then divides for its own such outputs one after
// another (a few of its K).  What this buys is that nothing stands between the K
// outputs' loads: issued behind a branch per output they followed one another, about
// 2000 cycles each (20 Adam steps of 128 rows of resnet_32's convolutions on the
// tensor cores, 8 outputs a block: 15.8 ms with the branches, 12.1 without).
template <int EM, int K>
__device__ __forceinline__ void epi_finish_block(const Epi& e, int m, const int (&j)[K],
                                                 float (&v)[K], const EpiIn (&in)[K], unsigned ok,
                                                 float& part) {
  if (e.acc_in) {
    float acc[K];
#pragma unroll
    for (int i = 0; i < K; ++i) acc[i] = e.acc_in[(size_t)m * e.acc_ld + j[i]];
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] += acc[i];
  }
  const size_t q0 = (size_t)m * e.SD + e.off;
  if constexpr (EM <= EM_RELU_GAMMA || EM == EM_ADJ || EM == EM_ADJ_GAMMA) {
    constexpr bool relu = EM <= EM_RELU_GAMMA;
    float ap[K], D[K], bl[K];
    unsigned need = 0, abr = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      ap[i] = relu ? v[i] : in[i].gp;
      if constexpr (EM == EM_RELU_GAMMA) ap[i] += in[i].gp;
      const float l = in[i].l, u = in[i].u;
      const int s = in[i].s;
      const bool one = s == -1 || (s != 1 && l >= 0.f);
      const bool zero = !one && (s == 1 || u <= 0.f);
      const bool up = ap[i] >= 0.f;
      const float a = EM == EM_RELU ? (u >= -l ? 1.f : 0.f) : in[i].al;
      D[i] = one ? 1.f : zero ? 0.f : a;
      bl[i] = 0.f;
      if ((ok >> i & 1u) && !one && !zero) (up ? abr : need) |= 1u << i;
    }
    while (need) {
      const int w = __ffs(need) - 1;
      need &= need - 1;
      float l = 0.f, u = 0.f;
#pragma unroll
      for (int i = 0; i < K; ++i)
        if (i == w) {
          l = in[i].l;
          u = in[i].u;
        }
      const float den = u - l;
      const float d = u / den, b = (-u * l) / den;
#pragma unroll
      for (int i = 0; i < K; ++i)
        if (i == w) {
          D[i] = d;
          bl[i] = b;
        }
    }
    const bool keep = relu && e.AP != nullptr;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const size_t qm = q0 + j[i];
      const bool st = ok >> i & 1u;
      if constexpr (relu) {
        float ah = ap[i] * D[i];
        if constexpr (EM >= EM_RELU_FINAL) ah += in[i].be * (float)in[i].s;
        if constexpr (EM == EM_RELU_GAMMA) ah += in[i].gph;
        if (keep && st) e.AP[qm] = ap[i];
        const float t = part + (ap[i] * bl[i] + ah * in[i].cb);
        part = st ? t : part;
        v[i] = ah;
      } else {
        const float h = v[i], g = h * D[i] + bl[i];
        if (st) {
          e.GA[qm] = abr >> i & 1u ? h * ap[i] : 0.f;
          e.GB[qm] = h * (float)in[i].s;
          if constexpr (EM == EM_ADJ_GAMMA) {
            e.Hz[qm] = h;
            e.Gz[qm] = g;
          }
        }
        v[i] = g;
      }
    }
  } else if constexpr (EM == EM_CONC) {
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (!(ok >> i & 1u)) continue;
      const float x = v[i] >= 0.f ? in[i].l : in[i].u;
      part += v[i] * x;
      if (e.X) e.X[(size_t)m * e.d0 + j[i]] = x;
    }
  } else if constexpr (EM == EM_FWD) {
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = fmaxf(v[i], 0.f);
  }
}

__device__ __forceinline__ bool epi_has_part(const Epi& e) {
  return e.part != nullptr && (e.kind == EPI_RELU || e.kind == EPI_CONC);
}

}  // namespace mnbab
