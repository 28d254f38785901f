// Device kernels of libmnbab: back-substitution through affine and ReLU layers
// with fused relaxation epilogues (Sec. 3.1), concretisation over the input box
// (Eq. minimum), the adjoint sweep for d lb / d (alpha, beta, gamma), projected
// Adam, ACS scoring (Sec. 3.2) and the BaB node bookkeeping (Sec. 3.2, enforcing
// splits).  All arithmetic is IEEE FP32 with FMA accumulation.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <stdint.h>

#include "epilogue.cuh"
#include "mnbab.h"
#include "mnbab_internal.h"

namespace mnbab {

// block-wide sum; every thread gets the result
__device__ float block_sum(float v) {
  __shared__ float sh[32];
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  float r = 0.f;
  for (int i = 0; i < nw; ++i) r += sh[i];
  return r;
}

// Allows a kernel `bytes` of dynamic shared memory.  The 48 KB that need no leave
// include the kernel's static shared memory (up to 9 KB here).
constexpr int SMEM_MOST = 216 * 1024;  // of any launch of this file (win_plan)
template <typename F>
static void set_smem(F f, int bytes) {
  if (bytes > 32 * 1024) allow_smem<SMEM_MOST>(f);
}

// ---------------------------------------------------------------------------
// starting rows
// ---------------------------------------------------------------------------
// Starting rows through one affine edge into node t: a = sign * A[j, :] on the
// edge's source (the folded objective rows Wf for t = R + 1), c0 = sign * (sum
// of the edge biases at j) on the first edge; the partial goes to slot_base.
// What bounds it is the latency of the epilogue's inputs (six loads per column): a
// thread takes four columns at a time and has all their loads in flight.  One column
// after another, with three divisions to find a convolution's tap, 1462 rows of 2704
// columns took 83 us and 594 of 800 17.5; now 23 and 7.2.
constexpr int INIT_U = 4;
template <int EM>
__global__ void __launch_bounds__(128) k_init_rows(NetDev net, int t, int edge, RowsDev rows,
                                                   float* out, int ld, Epi e) {
  const int m = blockIdx.x;
  if (m >= rows.M) return;
  const int n = rows.node[m];
  const int j = rows.j ? rows.j[m] : 0;
  const float sg = rows.sign ? rows.sign[m] : 1.f;
  const int src = edge == 0 ? net.src1[t] : net.src2[t];
  const int width = net.d[src];
  const PropDev* P = epi_prop(e, n);
  // a = 0 contributes nothing and maps to 0 through an intermediate ReLU step
  // (no beta / gamma terms), through concretisation (x* not kept) and as a raw
  // contribution, unless an earlier edge's contribution must be added
  const bool zero_passes = epi_zero_passes<EM>(e);
  float c0 = 0.f;
  float part = 0.f;
  // columns first, first + 128, ... below `count`: get(i, inside) returns column
  // and coefficient of entry i; inside: whether the coefficient can be nonzero
  auto walk = [&](int count, auto&& get) {
    for (int i0 = threadIdx.x; i0 < count; i0 += INIT_U * 128) {
      int col[INIT_U];
      float v[INIT_U];
      unsigned ok = 0;
#pragma unroll
      for (int u = 0; u < INIT_U; ++u) {
        const int i = i0 + u * 128;
        bool inside = true;
        v[u] = get(min(i, count - 1), col[u], inside);
        if (i < count && (inside || !zero_passes)) ok |= 1u << u;
      }
      if (ok) {
        EpiIn in[INIT_U];
#pragma unroll
        for (int u = 0; u < INIT_U; ++u) epi_load_m<EM>(e, n, P, m, col[u], in[u]);
        epi_finish_block<EM, INIT_U>(e, m, col, v, in, ok, part);
      }
      if (out) {
#pragma unroll
        for (int u = 0; u < INIT_U; ++u)
          if (i0 + u * 128 < count) out[(size_t)m * ld + col[u]] = (ok >> u & 1u) ? v[u] : 0.f;
      }
    }
  };
  if (rows.cidx) {
    // combination of three neurons of zhat_t: a = sum_k c_k W_t[j_k, :]
    const LayerDev& L = edge == 0 ? net.aff[t] : net.aff2[t];
    int jk[3];
    float ck[3];
    for (int k = 0; k < 3; ++k) {
      jk[k] = rows.cidx[3 * m + k];
      ck[k] = rows.ccoef[3 * m + k];
      if (edge == 0) {
        const float bj = net.bfull[t] ? net.bfull[t][jk[k]]
                                      : (L.kind == 1 ? L.b[jk[k]] : L.b[jk[k] / (L.ho * L.wo)]);
        c0 += ck[k] * bj;
      }
    }
    const int hw = L.ho * L.wo;
    const FDiv ihw = f_div_of(L.hi * L.wi), wi = f_div_of(L.wi);
    walk(width, [&](int i, int& col, bool&) {
      col = i;
      float a = 0.f;
      for (int k = 0; k < 3; ++k) {
        if (ck[k] == 0.f) continue;
        if (L.kind == 1) {
          a += ck[k] * L.W[(size_t)jk[k] * width + i];
        } else {
          const int co = jk[k] / hw, oh = (jk[k] % hw) / L.wo, ow = jk[k] % L.wo;
          const int ci = f_div(i, ihw), r = i - ci * (int)ihw.d, ih = f_div(r, wi);
          const int kh = ih - (oh * L.s - L.p), kw = r - ih * L.wi - (ow * L.s - L.p);
          if (kh >= 0 && kh < L.k && kw >= 0 && kw < L.k)
            a += ck[k] * L.W[(((size_t)co * L.ci + ci) * L.k + kh) * L.k + kw];
        }
      }
      return a;
    });
  } else if (t == net.R + 1) {
    const PropDev& Pr = e.props[e.pool.prop[n]];
    const float* w = Pr.Wf + (size_t)j * width;
    c0 = Pr.bf[j];
    walk(width, [&](int i, int& col, bool&) {
      col = i;
      return w[i];
    });
  } else {
    const LayerDev& L = edge == 0 ? net.aff[t] : net.aff2[t];
    if (edge == 0) {
      const float bj = net.bfull[t] ? net.bfull[t][j]
                                    : (L.kind == 1 ? L.b[j] : L.b[j / (L.ho * L.wo)]);
      c0 = sg * bj;
    }
    if (L.kind == 1) {
      const float* w = L.W + (size_t)j * width;
      walk(width, [&](int i, int& col, bool&) {
        col = i;
        return sg * w[i];
      });
    } else {
      // row j = (co, oh, ow) of the convolution's Toeplitz matrix
      const int hw = L.ho * L.wo;
      const int co = j / hw, oh = (j % hw) / L.wo, ow = j % L.wo;
      const int h0 = oh * L.s - L.p, w0 = ow * L.s - L.p;
      const int kk = L.k * L.k, ihw = L.hi * L.wi;
      const float* w = L.W + (size_t)co * L.ci * kk;
      if (!out && zero_passes) {
        // only the kernel window of neuron j is nonzero and nothing is stored: walk
        // the window (a tap outside the plane: its nearest column, left out)
        walk(L.ci * kk, [&](int q, int& col, bool& inside) {
          const int ci = q / kk, kh = (q % kk) / L.k, kw = q % L.k;
          const int ih = min(max(h0 + kh, 0), L.hi - 1), iw = min(max(w0 + kw, 0), L.wi - 1);
          inside = ih == h0 + kh && iw == w0 + kw;
          col = ci * ihw + ih * L.wi + iw;
          return sg * w[q];
        });
      } else {
        const FDiv dp = f_div_of(ihw), dw = f_div_of(L.wi);
        walk(width, [&](int i, int& col, bool& inside) {
          const int ci = f_div(i, dp), r = i - ci * ihw, ih = f_div(r, dw);
          const int kh = ih - h0, kw = r - ih * L.wi - w0;
          inside = kh >= 0 && kh < L.k && kw >= 0 && kw < L.k;
          col = i;
          // (outside the receptive field a = 0 and, without beta or gamma terms, the
          // ReLU step maps it to 0 with no offset contribution)
          return inside ? sg * w[(ci * L.k + kh) * L.k + kw] : 0.f;
        });
      }
    }
  }
  const float tot = block_sum(part);
  if (threadIdx.x == 0 && e.part) e.part[(size_t)m * e.nslot + e.slot_base] = tot + c0;
}

void launch_init_rows(const NetDev& net, int t, int edge, const RowsDev& rows, float* out, int ld,
                      const Epi& e, cudaStream_t st) {
  if (rows.M <= 0) return;
  epi_dispatch_back(e, [&](auto em) {
    k_init_rows<decltype(em)::value><<<rows.M, 128, 0, st>>>(net, t, edge, rows, out, ld, e);
  });
}

// ---------------------------------------------------------------------------
// rows of layer 1: one affine step from the input box, then concretisation
// ---------------------------------------------------------------------------
// lb = sign * b_j + sum_k min(a_k lo_k, a_k hi_k), a = sign * W_1[j, :]; a conv
// neuron touches only its k x k x ci patch (one thread per row), an FC neuron
// its whole weight row (one warp per row).
__global__ void k_first_rows_conv(NetDev net, PoolDev pool, const PropDev* props, RowsDev rows,
                                  float* lb) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= rows.M) return;
  const LayerDev& L = net.aff[1];
  const int j = rows.j[m];
  const float sg = rows.sign ? rows.sign[m] : 1.f;
  const PropDev& P = props[pool.prop[rows.node[m]]];
  const int hw = L.ho * L.wo;
  const int co = j / hw, oh = (j % hw) / L.wo, ow = j % L.wo;
  const int h0 = oh * L.s - L.p, w0 = ow * L.s - L.p;
  const float* w = L.W + (size_t)co * L.ci * L.k * L.k;
  float acc = 0.f;
  for (int ci = 0; ci < L.ci; ++ci)
    for (int kh = 0; kh < L.k; ++kh) {
      const int ih = h0 + kh;
      if (ih < 0 || ih >= L.hi) continue;
      for (int kw = 0; kw < L.k; ++kw) {
        const int iw = w0 + kw;
        if (iw < 0 || iw >= L.wi) continue;
        const float a = sg * __ldg(w + (ci * L.k + kh) * L.k + kw);
        const int x = (ci * L.hi + ih) * L.wi + iw;
        acc += a * (a >= 0.f ? P.lo[x] : P.hi[x]);
      }
    }
  lb[m] = acc + sg * (net.bfull[1] ? net.bfull[1][j] : L.b[co]);
}

__global__ void k_first_rows_fc(NetDev net, PoolDev pool, const PropDev* props, RowsDev rows,
                                float* lb) {
  const int m = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (m >= rows.M) return;
  const LayerDev& L = net.aff[1];
  const int j = rows.j[m];
  const float sg = rows.sign ? rows.sign[m] : 1.f;
  const PropDev& P = props[pool.prop[rows.node[m]]];
  const float* w = L.W + (size_t)j * L.d_in;
  float acc = 0.f;
  for (int k = lane; k < L.d_in; k += 32) {
    const float a = sg * __ldg(w + k);
    acc += a * (a >= 0.f ? P.lo[k] : P.hi[k]);
  }
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) lb[m] = acc + sg * (net.bfull[1] ? net.bfull[1][j] : L.b[j]);
}

void launch_first_rows(const NetDev& net, const PoolDev& pool, const PropDev* props,
                       const RowsDev& rows, float* lb, cudaStream_t st) {
  if (rows.M <= 0) return;
  if (net.aff[1].kind == MNBAB_CONV2D)
    k_first_rows_conv<<<(rows.M + 127) / 128, 128, 0, st>>>(net, pool, props, rows, lb);
  else
    k_first_rows_fc<<<(rows.M + 7) / 8, 256, 0, st>>>(net, pool, props, rows, lb);
}

// ---------------------------------------------------------------------------
// windowed rows (intermediate bounds of convolution neurons)
// ---------------------------------------------------------------------------
// A row at neuron (co, oh, ow) of zhat_t starts, after its first step, as the
// k x k kernel patch of output channel co with origin (oh s - p, ow s - p) at
// layer t-1.  A convolution (stride s, kernel k, padding p) maps coefficients
// on an h x w window with origin (y0, x0) to a ((h-1)s + k) x ((w-1)s + k)
// window with origin (y0 s - p, x0 s - p); relative output position yy takes
// input position Y = (yy - kh) / s wherever that is an integer in [0, h).
// Positions outside the layer (padding) carry no coefficient.
constexpr int WIN_MAX_FLOATS = 12288;  // per buffer of one row
constexpr int WIN_RB_MAX = 8;

bool win_plan(const NetDev& net, int t, WinPlan& wp) {
  if (t < 2 || t > net.R) return false;  // rows at layer 1 are direct in k_init_rows
  for (int i = 1; i <= t; ++i)
    if (net.n_edge[i] != 1 || net.src1[i] != i - 1 || net.aff[i].kind != MNBAB_CONV2D)
      return false;
  wp.t = t;
  int h = net.aff[t].k, w = net.aff[t].k;
  wp.h[t - 1] = h;
  wp.w[t - 1] = w;
  int mx = net.aff[t].ci * h * w;
  for (int i = t - 1; i >= 1; --i) {
    const LayerDev& L = net.aff[i];
    h = (h - 1) * L.s + L.k;
    w = (w - 1) * L.s + L.k;
    wp.h[i - 1] = h;
    wp.w[i - 1] = w;
    mx = std::max(mx, L.ci * h * w);
  }
  if (mx > WIN_MAX_FLOATS) return false;
  // planes of the two buffers (16-byte multiples) and the padded weights
  wp.plane[0] = wp.plane[1] = wp.wpad = 0;
  for (int i = t - 1; i >= 0; --i) {
    const int n = (net.aff[i + 1].ci * wp.h[i] * wp.w[i] + 3) / 4 * 4, side = (t - 1 - i) & 1;
    wp.plane[side] = std::max(wp.plane[side], n);
    if (i >= 1 && (net.aff[i].ci == 2 || net.aff[i].ci == 3))
      wp.wpad += net.aff[i].co * net.aff[i].k * net.aff[i].k * 4;
  }
  // rows per CTA: 8 where two CTAs still fit on an SM, else 4 or 1 (4 at most in
  // the small CTAs where a row has 256 partial sums)
  auto bytes = [&](int rb) { return (rb * (wp.plane[0] + wp.plane[1]) + wp.wpad) * 4; };
  wp.vt = mx <= 1024 ? 128 : 256;
  wp.wide = false;
  for (int i = 1; i < t; ++i) {
    const int ci = net.aff[i].ci;
    wp.wide = wp.wide || (ci & 3) == 0 || ci == 2 || ci == 3;
  }
  const int most = !wp.wide && wp.vt == 256 ? 4 : WIN_RB_MAX;
  wp.rb = bytes(most) <= 104 * 1024 ? most : bytes(4) <= SMEM_MOST ? 4 : 1;
  return bytes(wp.rb) <= SMEM_MOST;
}

// x / d for the small operands of window indices (x d < 2^32), by the rounded-up
// reciprocal `magic` = ceil(2^32 / d) (0 stands for d = 1)
__device__ __forceinline__ unsigned win_magic(int d) {
  return d == 1 ? 0u : 0xffffffffu / (unsigned)d + 1u;
}
__device__ __forceinline__ int win_div(int x, unsigned magic) {
  return magic ? (int)__umulhi((unsigned)x, magic) : x;
}

struct WinRow {
  int y0, x0;  // window origin at the current layer
};

// Output positions are enumerated phase-major (ih mod s, iw mod s) so that the
// threads of a warp share kernel taps, and with them their weight loads.
__device__ __forceinline__ void decode_phase(int pidx, int hi, int wi, int s, int& ih, int& iw) {
  for (int ph = 0; ph < s; ++ph) {
    const int nh = (hi - ph + s - 1) / s;
    for (int pw = 0; pw < s; ++pw) {
      const int nw = (wi - pw + s - 1) / s;
      const int cnt = nh * nw;
      if (pidx < cnt) {
        ih = ph + s * (pidx / nw);
        iw = pw + s * (pidx % nw);
        return;
      }
      pidx -= cnt;
    }
  }
  ih = iw = -1;
}

// the same with the divisions prepared once per thread
struct PhaseIdx {
  int s, wi, hq, hr, wq, wr;  // rows / columns of a phase: hq (+ 1 for the first hr phases)
  FDiv w0, w1;                // columns of a phase: wq + 1, wq
  __device__ __forceinline__ PhaseIdx(int hi, int wi_, int s_) : s(s_), wi(wi_) {
    hq = hi / s;
    hr = hi - hq * s;
    wq = wi / s;
    wr = wi - wq * s;
    w0 = f_div_of(wq + 1);
    w1 = f_div_of(max(wq, 1));
  }
  __device__ __forceinline__ void decode(int pidx, int& ih, int& iw) const {
    int ph = 0, nh = hq + (hr > 0);
    while (pidx >= nh * wi) {
      pidx -= nh * wi;
      ++ph;
      nh = hq + (ph < hr);
    }
    int pw = 0, nw = wq + (wr > 0);
    while (pidx >= nh * nw) {
      pidx -= nh * nw;
      ++pw;
      nw = wq + (pw < wr);
    }
    const int r = f_div(pidx, pw < wr ? w0 : w1);
    ih = ph + s * r;
    iw = pw + s * (pidx - r * nw);
  }
};

// Transposed convolution of the CTA's row windows, A (h x w) to B (h2 x w2),
// both [channel][position][RB rows].  An item is one output position x CB
// channels x four rows: a 16-byte load brings a coefficient of the four rows,
// and its CB weights serve all of them, so three loads feed 32 FMAs (CB = 8).
// SM: the weights are in shared memory, else in global memory.
template <int THREADS, int RG, int CB, bool SM>
__device__ __forceinline__ void win_conv(const LayerDev& L, const float* __restrict__ Wt, int wci,
                                         const float* A, float* B, int RB, int h, int w,
                                         const WinRow* rows) {
  const int s = L.s, k = L.k, h2 = (h - 1) * s + k, w2 = (w - 1) * s + k;
  const int hw = h * w, hw2 = h2 * w2;
  const int items = hw2 * (RB / RG) * ((L.ci + CB - 1) / CB);
  const int wco = k * k * wci;
  for (int it = threadIdx.x; it < items; it += THREADS) {
    const int px = it % hw2, rg = it / hw2 % (RB / RG) * RG, grp = it / (hw2 * (RB / RG));
    constexpr int R2 = RG == 4 ? 2 : 1;
    float2 acc[CB][R2];
#pragma unroll
    for (int c = 0; c < CB; ++c)
#pragma unroll
      for (int r = 0; r < R2; ++r) acc[c][r] = make_float2(0.f, 0.f);
    int yy, xx;
    decode_phase(px, h2, w2, s, yy, xx);
    for (int kh = yy % s, Y = yy / s; kh < k && Y >= 0; kh += s, --Y) {
      if (Y >= h) continue;
      for (int kw = xx % s, X = xx / s; kw < k && X >= 0; kw += s, --X) {
        if (X >= w) continue;
        const float* ap = A + (size_t)(Y * w + X) * RB + rg;
        const float* wp = Wt + (kh * k + kw) * wci + grp * CB;
#pragma unroll 4
        for (int o = 0; o < L.co; ++o, ap += hw * RB, wp += wco) {
          float2 v[R2];
          if (RG == 4) {
            const float4 v4 = *reinterpret_cast<const float4*>(ap);
            v[0] = make_float2(v4.x, v4.y);
            v[R2 - 1] = make_float2(v4.z, v4.w);
          } else {
            v[0] = make_float2(*ap, 0.f);
          }
          float wv[CB];
          if (CB >= 4) {
#pragma unroll
            for (int c = 0; c < CB; c += 4) {
              const float4* w4p = reinterpret_cast<const float4*>(wp + c);
              const float4 w4 = SM ? *w4p : __ldg(w4p);
              wv[c] = w4.x;
              wv[c + 1 < CB ? c + 1 : c] = w4.y;
              wv[c + 2 < CB ? c + 2 : c] = w4.z;
              wv[c + 3 < CB ? c + 3 : c] = w4.w;
            }
          } else {
            wv[0] = SM ? wp[0] : __ldg(wp);
          }
#pragma unroll
          for (int c = 0; c < CB; ++c) {
            if (RG == 4) {
              const float2 ww = make_float2(wv[c], wv[c]);
              acc[c][0] = fma2(v[0], ww, acc[c][0]);
              acc[c][R2 - 1] = fma2(v[R2 - 1], ww, acc[c][R2 - 1]);
            } else {
              acc[c][0].x = fmaf(v[0].x, wv[c], acc[c][0].x);
            }
          }
        }
      }
    }
    // positions outside the layer (padding) carry no coefficient
    bool in[RG];
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      const int y = rows[rg + r].y0 * s - L.p + yy, x = rows[rg + r].x0 * s - L.p + xx;
      in[r] = y >= 0 && y < L.hi && x >= 0 && x < L.wi;
    }
    float* bp = B + (size_t)(grp * CB * hw2 + yy * w2 + xx) * RB + rg;
#pragma unroll
    for (int c = 0; c < CB; ++c)
      if (CB < 4 || grp * CB + c < L.ci) {
        if constexpr (RG == 4)
          *reinterpret_cast<float4*>(bp + (size_t)c * hw2 * RB) =
              make_float4(in[0] ? acc[c][0].x : 0.f, in[1] ? acc[c][0].y : 0.f,
                          in[2] ? acc[c][1].x : 0.f, in[3] ? acc[c][1].y : 0.f);
        else
          bp[c * hw2] = in[0] ? acc[c][0].x : 0.f;
      }
  }
}

// RB = 8, 4 or (where four rows' windows and weights exceed 216 KB) 1 rows per CTA, their
// windows in shared memory with the rows of a position adjacent.  Bound by the latency
// of the weight and bound loads (FMA pipe 34% busy) and FP32 FMAs: on the 3x32x32
// network's layers 3 and 4 (32768 and 8192 rows, 31 GFLOP) 1.2 and 2.9 ms; a thread per output element of one
// row took 16.3 ms together.  Few items leave threads idle in the deep layers'
// first steps; splitting their reductions over lanes gained 0.7 ms and changed the
// order of the sums, which stays that of one row alone.  Four columns of one row
// per thread instead of four rows took 149 against 101 us for the 25600 rows of 16
// 1x28x28 properties (112 us before): its columns are ragged in small windows.
// WIDE: some layer of the chain has several input channels to a thread; without
// one (a one-channel image below a single convolution) smaller CTAs of fewer
// registers hide the latency of its short steps.
template <bool WIDE, int RG, int NA>
__global__ void __launch_bounds__(WIDE ? 512 : 256, WIDE ? 2 : 6)
    k_win_rows(NetDev net, WinPlan wp, RowsDev rows, Epi e, float* __restrict__ lb) {
  constexpr int THREADS = WIDE ? 512 : 256;
  extern __shared__ __align__(16) float wsm[];
  __shared__ WinRow s_row[WIN_RB_MAX];
  __shared__ float s_sum[WIN_RB_MAX][256], s_c0[WIN_RB_MAX];
  // A row's offset terms are summed as wp.vt interleaved partial sums (element x of
  // a layer to sum x mod vt), then in a tree over each 32 of them, then in order:
  // the same sum for any number of rows per CTA.  A thread holds NA of them.
  const int t = wp.t, RB = wp.rb, tpr = wp.vt / NA;
  const LayerDev& Lt = net.aff[t];
  // buffers of the layers t - 1, t - 3, ... and t - 2, t - 4, ...; then the
  // padded weights of layers with 2 or 3 input channels
  float* buf[2] = {wsm, wsm + RB * wp.plane[0]};
  float* wpad = wsm + RB * (wp.plane[0] + wp.plane[1]);
  if (WIDE) {
    float* d = wpad;
    for (int i = 1; i < t; ++i) {
      const LayerDev& L = net.aff[i];
      if (L.ci != 2 && L.ci != 3) continue;
      const int n = L.co * L.k * L.k * 4;
      for (int q = threadIdx.x; q < n; q += THREADS)
        d[q] = (q & 3) < L.ci ? __ldg(L.Wb + (q >> 2) * L.ci + (q & 3)) : 0.f;
      d += n;
    }
  }
  const int q = threadIdx.x % RB, tl = threadIdx.x / RB, nthr = THREADS / RB;
  const int m = min(blockIdx.x * RB + q, rows.M - 1);  // absent rows repeat the last (dropped)
  const int j = rows.j[m], node = rows.node[m];
  const float sg = rows.sign ? rows.sign[m] : 1.f;
  const int hwt = Lt.ho * Lt.wo;
  const int co = j / hwt, oh = (j % hwt) / Lt.wo, ow = j % Lt.wo;
  int y0 = oh * Lt.s - Lt.p, x0 = ow * Lt.s - Lt.p;
  if (tl == 0) s_row[q] = WinRow{y0, x0};
  {
    const int n0 = Lt.ci * Lt.k * Lt.k;
    for (int i = tl; i < n0; i += nthr) buf[0][i * RB + q] = sg * __ldg(Lt.W + (size_t)co * n0 + i);
  }
  const PropDev& P = e.props[e.pool.prop[node]];
  float part[NA];
#pragma unroll
  for (int v = 0; v < NA; ++v) part[v] = 0.f;
  const bool on = tl < tpr;
  int h = Lt.k, w = Lt.k;
  for (int i = t - 1, side = 0; i >= 0; --i, side ^= 1) {
    const LayerDev& Ln = net.aff[i + 1];  // layer i is this edge's input
    const int C = Ln.ci, H = Ln.hi, W = Ln.wi, hw = h * w, n = C * hw;
    const unsigned mhw = win_magic(hw), mw = win_magic(w);
    float* A = buf[side] + q;
    __syncthreads();
    if (i == 0) {
      // concretisation over the input box
      for (int r0 = on ? tl : n; r0 < n; r0 += NA * tpr)
#pragma unroll
        for (int v = 0; v < NA; ++v) {
          const int rr = r0 + v * tpr;
          const int c = win_div(rr, mhw), r = rr - c * hw, yr = win_div(r, mw);
          const int y = y0 + yr, x = x0 + r - yr * w;
          if (rr >= n || y < 0 || y >= H || x < 0 || x >= W) continue;
          const int jx = (c * H + y) * W + x;
          const float a = A[rr * RB];
          part[v] += a * (a >= 0.f ? P.lo[jx] : P.hi[jx]);
        }
      break;
    }
    // ReLU step of layer i (DeepPoly slopes, splits enforced); the bounds of
    // four elements are loaded before the first is used
    const size_t nb = (size_t)node * e.SD + net.off[i];
    const float* bias = net.bfull[i];
    for (int r0 = on ? tl : n; r0 < n; r0 += 4 * tpr) {
      int jx[4];
      float l[4], u[4], b[4];
      int sp[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int rr = r0 + v * tpr;
        const int c = win_div(rr, mhw), r = rr - c * hw, yr = win_div(r, mw);
        const int y = y0 + yr, x = x0 + r - yr * w;
        jx[v] = rr < n && y >= 0 && y < H && x >= 0 && x < W ? (c * H + y) * W + x : -1;
        l[v] = u[v] = b[v] = 0.f;
        sp[v] = 0;
        if (jx[v] >= 0) {
          l[v] = e.pool.L[nb + jx[v]];
          u[v] = e.pool.U[nb + jx[v]];
          sp[v] = e.pool.S[nb + jx[v]];
          b[v] = bias[jx[v]];
        }
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int rr = r0 + v * tpr;
        if (rr >= n) break;
        if (jx[v] < 0) {
          A[rr * RB] = 0.f;
          continue;
        }
        const float a = A[rr * RB];
        float D, bl = 0.f;
        if (sp[v] == -1) D = 1.f;
        else if (sp[v] == 1) D = 0.f;
        else if (l[v] >= 0.f) D = 1.f;
        else if (u[v] <= 0.f) D = 0.f;
        else if (a >= 0.f) D = u[v] >= -l[v] ? 1.f : 0.f;
        else {
          const float den = u[v] - l[v];
          D = u[v] / den;
          bl = (-u[v] * l[v]) / den;
        }
        const float ah = a * D;
        part[v % NA] += a * bl + ah * b[v];
        A[rr * RB] = ah;
      }
    }
    __syncthreads();
    // transposed convolution through layer i's edge
    const LayerDev& Li = net.aff[i];
    const float* in = buf[side];
    float* out = buf[side ^ 1];
    if (!WIDE) {
      win_conv<THREADS, RG, 1, false>(Li, Li.Wb, Li.ci, in, out, RB, h, w, s_row);
    } else if ((Li.ci & 7) == 0) {
      win_conv<THREADS, RG, 8, false>(Li, Li.Wb, Li.ci, in, out, RB, h, w, s_row);
    } else if ((Li.ci & 3) == 0) {
      win_conv<THREADS, RG, 4, false>(Li, Li.Wb, Li.ci, in, out, RB, h, w, s_row);
    } else if (Li.ci == 2 || Li.ci == 3) {
      const float* wt = wpad;
      for (int v = 1; v < i; ++v)
        if (net.aff[v].ci == 2 || net.aff[v].ci == 3)
          wt += net.aff[v].co * net.aff[v].k * net.aff[v].k * 4;
      win_conv<THREADS, RG, 4, true>(Li, wt, 4, in, out, RB, h, w, s_row);
    } else {
      win_conv<THREADS, RG, 1, false>(Li, Li.Wb, Li.ci, in, out, RB, h, w, s_row);
    }
    h = (h - 1) * Li.s + Li.k;
    w = (w - 1) * Li.s + Li.k;
    y0 = y0 * Li.s - Li.p;
    x0 = x0 * Li.s - Li.p;
    __syncthreads();
    if (tl == 0) s_row[q] = WinRow{y0, x0};
  }
  if (on)
#pragma unroll
    for (int v = 0; v < NA; ++v) s_sum[q][v * tpr + tl] = part[v];
  if (tl == 0) s_c0[q] = sg * (net.bfull[t] ? net.bfull[t][j] : Lt.b[co]);
  __syncthreads();
  const int wq = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wq < RB && blockIdx.x * RB + wq < rows.M) {
    float tot = 0.f;
    for (int v = 0; v < wp.vt / 32; ++v) {
      float x = s_sum[wq][v * 32 + lane];
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      tot += x;
    }
    if (lane == 0) lb[blockIdx.x * RB + wq] = tot + s_c0[wq];
  }
}

void launch_win_rows(const NetDev& net, const WinPlan& wp, const RowsDev& rows, const Epi& e,
                     float* lb, cudaStream_t st) {
  if (rows.M <= 0) return;
  const int smem = (wp.rb * (wp.plane[0] + wp.plane[1]) + wp.wpad) * (int)sizeof(float);
  const int grid = (rows.M + wp.rb - 1) / wp.rb;
  auto go = [&](auto kern, int threads) {
    set_smem(kern, smem);
    kern<<<grid, threads, smem, st>>>(net, wp, rows, e, lb);
  };
  if (wp.rb == 1) go(k_win_rows<true, 1, 1>, 512);
  else if (!wp.wide) go(k_win_rows<false, 4, 4>, 256);
  else if (wp.vt * wp.rb == 4 * 512) go(k_win_rows<true, 4, 4>, 512);
  else if (wp.vt * wp.rb == 2 * 512) go(k_win_rows<true, 4, 2>, 512);
  else go(k_win_rows<true, 4, 1>, 512);
}

// ---------------------------------------------------------------------------
// dense GEMM C = A B (+ bias) with a fused epilogue; SIMT FP32
// ---------------------------------------------------------------------------
constexpr int GBK = 16;
constexpr int GLA = GBK + 4;  // stride of a staged row of A (float4 reads without bank conflicts)

// A BM x BN tile over the reduction range [kb, ke): TM x TN outputs per thread
// (rows ty + TY i, columns TN tx + j), each summed over k in order.  Steps of GBK go
// through a ring of ST stages filled by asynchronous copies: the small products of
// a few rows are bound by the latency of their loads (about 2 us for each step of
// 16 when a step waited for its own loads), so ST - 1 steps are in flight, and a
// thread takes 8 or 16 outputs (with four, shared-memory reads fed one FMA each).
// Measured before and now: 64 x 512 x 4096 split in ten 56 and 18 us, 64 x 4096 x 512
// split in two 36 and 14; 32 x 32 tiles, 256 x 4096 x 512 126 and 46, 9 x 100 x 100
// 16.7 and 7.5; 64 x 64 tiles, 1024 x 4096 x 512 273 and 123.
template <int BM, int BN, int TM, int TN, int ST>
__device__ __forceinline__ void gemm_tile(int M, int N, int kb, int ke, const float* __restrict__ A,
                                          int lda, const float* __restrict__ B, int ldb, int m0,
                                          int n0, float* sm, float (&acc)[TM][TN]) {
  constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
  constexpr int STAGE = BM * GLA + GBK * BN;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const bool va = ((reinterpret_cast<uintptr_t>(A) | (uintptr_t)lda * 4) & 15) == 0;
  const bool vb = ((reinterpret_cast<uintptr_t>(B) | (uintptr_t)ldb * 4) & 15) == 0;
  const unsigned s0 = static_cast<unsigned>(__cvta_generic_to_shared(sm));
  // `n` of four floats (the others zero); one by one where 16-byte copies are not aligned
  auto copy4 = [](unsigned d, const float* s, const float* base, int n, bool vec) {
    if (vec) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(n > 0 ? s : base),
                   "r"(n * 4)
                   : "memory");
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 4u * u),
                     "l"(u < n ? s + u : base), "r"(u < n ? 4 : 0)
                     : "memory");
    }
  };
  auto load = [&](int it) {
    const int k0 = kb + it * GBK;
    const unsigned sa = s0 + (unsigned)(it % ST * STAGE) * 4u, sb = sa + (unsigned)(BM * GLA) * 4u;
#pragma unroll
    for (int c = tid; c < BM * GBK / 4; c += NT) {
      const int r = c / (GBK / 4), k = c % (GBK / 4) * 4, gm = m0 + r;
      const int n = gm < M ? max(0, min(4, ke - (k0 + k))) : 0;
      copy4(sa + (unsigned)(r * GLA + k) * 4u, A + (size_t)gm * lda + k0 + k, A, n, va);
    }
#pragma unroll
    for (int c = tid; c < GBK * BN / 4; c += NT) {
      const int r = c / (BN / 4), q = c % (BN / 4) * 4, gk = k0 + r;
      const int n = gk < ke ? max(0, min(4, N - (n0 + q))) : 0;
      copy4(sb + (unsigned)(r * BN + q) * 4u, B + (size_t)gk * ldb + n0 + q, B, n, vb);
    }
  };
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  const int nk = (ke - kb + GBK - 1) / GBK;
#pragma unroll
  for (int it = 0; it < ST - 1; ++it) {
    if (it < nk) load(it);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int it = 0; it < nk; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();
    if (it + ST - 1 < nk) load(it + ST - 1);  // into the stage of step it - 1
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* as = sm + it % ST * STAGE + ty * GLA;
    const float* bs = sm + it % ST * STAGE + BM * GLA + tx * TN;
#pragma unroll
    for (int k = 0; k < GBK; k += 4) {
      float a[TM][4], b[4][TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(as + i * TY * GLA + k);
        a[i][0] = v.x;
        a[i][1] = v.y;
        a[i][2] = v.z;
        a[i][3] = v.w;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if constexpr (TN == 4) {
          const float4 v = *reinterpret_cast<const float4*>(bs + (k + u) * BN);
          b[u][0] = v.x;
          b[u][1] = v.y;
          b[u][2] = v.z;
          b[u][3] = v.w;
        } else {
          const float2 v = *reinterpret_cast<const float2*>(bs + (k + u) * BN);
          b[u][0] = v.x;
          b[u][1] = v.y;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i][u], b[u][j], acc[i][j]);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

constexpr int gemm_smem(int BM, int BN, int ST) { return ST * (BM * GLA + GBK * BN) * 4; }

// BM x BN tile, BM BN / (TM TN) threads.  The outputs pass through shared memory to
// the epilogue's threads: 16 per row, columns tx + 16 j, so that a row's offset
// partial is summed in that order whatever tile computed it.
template <int BM, int BN, int TM, int TN, int ST, int EM>
__global__ void __launch_bounds__(BM * BN / (TM * TN)) k_gemm(
    int M, int N, int K, const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
    const float* __restrict__ bias, int bias_div, float* C, int ldc, Epi e) {
  extern __shared__ __align__(16) float gsm[];
  constexpr int NT = BM * BN / (TM * TN), TX = BN / TN, TY = BM / TM, LC = BN + 1;
  constexpr int RPT = BM * 16 / NT, NJ = BN / 16;  // epilogue: rows and columns per thread
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN, tid = threadIdx.x;
  {
    float acc[TM][TN];
    gemm_tile<BM, BN, TM, TN, ST>(M, N, 0, K, A, lda, B, ldb, m0, n0, gsm, acc);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        gsm[(tid / TX + TY * i) * LC + tid % TX * TN + j] = acc[i][j];
    __syncthreads();
  }
  const int tx = tid & 15, ty = tid >> 4;
  int cn[NJ];
  float cb[NJ];
  unsigned okn = 0;
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const int n = n0 + tx + 16 * j;
    cn[j] = min(n, N - 1);
    if (n < N) okn |= 1u << j;
    cb[j] = bias ? bias[cn[j] / bias_div] : 0.f;
  }
#pragma unroll 2
  for (int i = 0; i < RPT; ++i) {
    const int r = ty + NT / 16 * i, m = m0 + r;
    float part = 0.f;
    if (m < M) {
      const int rn = EM == EM_STORE || EM == EM_FWD ? 0 : e.row_node[m];
      const PropDev* rp = epi_prop(e, rn);
      float v[NJ];
      EpiIn in[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        epi_load_m<EM>(e, rn, rp, m, cn[j], in[j]);
        v[j] = gsm[r * LC + tx + 16 * j];
        if (bias) v[j] += cb[j];
      }
      epi_finish_block<EM, NJ>(e, m, cn, v, in, okn, part);
      if (C) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          if (okn >> j & 1u) C[(size_t)m * ldc + cn[j]] = v[j];
      }
    }
    if (epi_has_part(e)) {
      for (int o = 8; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o, 16);
      if (tx == 0 && m < M) e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = part;
    }
  }
}

// Split-K partial products: CTA z computes K range [z*kc, (z+1)*kc) of a
// 32 x 32 tile into ws[z][m][n] (no epilogue).
__global__ void __launch_bounds__(128) k_gemm_splitk(int M, int N, int K, int kc,
                                                     const float* __restrict__ A, int lda,
                                                     const float* __restrict__ B, int ldb,
                                                     float* __restrict__ ws) {
  extern __shared__ __align__(16) float gsm[];
  const int m0 = blockIdx.y * 32, n0 = blockIdx.x * 32, tid = threadIdx.x;
  const int kb = blockIdx.z * kc, ke = min(K, kb + kc);
  float acc[4][2];
  gemm_tile<32, 32, 4, 2, 6>(M, N, kb, ke, A, lda, B, ldb, m0, n0, gsm, acc);
  float* w = ws + (size_t)blockIdx.z * M * N;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int m = m0 + tid / 16 + 8 * i, n = n0 + tid % 16 * 2 + j;
      if (m < M && n < N) w[(size_t)m * N + n] = acc[i][j];
    }
}

// Sum of the split-K partials (fixed order) + bias, then the epilogue; a CTA
// covers 8 rows x 32 columns, one warp per row, and writes one offset partial
// per (row, 32-column tile).  An output's partials (at most 16) and its epilogue's
// inputs are loaded together.
template <int EM>
__global__ void __launch_bounds__(256) k_splitk_epi(int M, int N, int S, const float* __restrict__ ws,
                                                    const float* __restrict__ bias, int bias_div,
                                                    float* C, int ldc, Epi e) {
  const int m = blockIdx.y * 8 + (threadIdx.x >> 5);
  const int n = blockIdx.x * 32 + (threadIdx.x & 31);
  float part = 0.f;
  if (m < M && n < N) {
    const int rn = EM == EM_STORE || EM == EM_FWD ? 0 : e.row_node[m];
    float w[16];
#pragma unroll
    for (int z = 0; z < 16; ++z) w[z] = z < S ? ws[((size_t)z * M + m) * N + n] : 0.f;
    const float b = bias ? bias[n / bias_div] : 0.f;
    EpiIn in[1];
    const int j[1] = {n};
    epi_load_m<EM>(e, rn, epi_prop(e, rn), m, n, in[0]);
    float v[1] = {0.f};
#pragma unroll
    for (int z = 0; z < 16; ++z)
      if (z < S) v[0] += w[z];
    if (bias) v[0] += b;
    epi_finish_block<EM, 1>(e, m, j, v, in, 1u, part);
    if (C) C[(size_t)m * ldc + n] = v[0];
  }
  if (epi_has_part(e)) {
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0 && m < M)
      e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = part;
  }
}

// 64 x 64 tiles unless that grid would leave most of the 152 SMs idle; then
// 32 x 32 tiles, split along K when the K loop is long and the workspace fits.
// SIMT GEMM variants: V_SPLITK (reduction split over up to 16 CTAs per tile
// so that small products fill the SMs; -1 when no split is possible), V_G64,
// V_G32.
static int gemm_variant(int v, int M, int N, int K, const float* A, int lda, const float* B,
                        int ldb, const float* bias, int bias_div, float* C, int ldc, const Epi& e,
                        cudaStream_t st) {
  if (v == V_SPLITK) {
    if (K < 256 || !e.ws) return -1;
    const long small = (long)((N + 31) / 32) * ((M + 31) / 32);
    int S = (int)std::min<long>(16, std::max<long>(2, (2 * 152 + small - 1) / small));
    S = std::min(S, K / 64);
    while (S > 1 && (size_t)S * M * N > e.ws_floats) --S;
    if (S <= 1) return -1;
    const int kc = ((K + S - 1) / S + GBK - 1) / GBK * GBK;
    S = (K + kc - 1) / kc;
    dim3 g1((N + 31) / 32, (M + 31) / 32, S);
    constexpr int sm = gemm_smem(32, 32, 6);
    k_gemm_splitk<<<g1, 128, sm, st>>>(M, N, K, kc, A, lda, B, ldb, e.ws);
    dim3 g2((N + 31) / 32, (M + 7) / 8);
    epi_dispatch(e, [&](auto em) {
      k_splitk_epi<decltype(em)::value><<<g2, 256, 0, st>>>(M, N, S, e.ws, bias, bias_div, C, ldc, e);
    });
    return g2.x;
  }
  if (v == V_G64) {
    dim3 grid((N + 63) / 64, (M + 63) / 64);
    constexpr int sm = gemm_smem(64, 64, 4);
    epi_dispatch(e, [&](auto em) {
      k_gemm<64, 64, 4, 4, 4, decltype(em)::value>
          <<<grid, 256, sm, st>>>(M, N, K, A, lda, B, ldb, bias, bias_div, C, ldc, e);
    });
    return grid.x;
  }
  if (v == V_G32) {
    dim3 grid((N + 31) / 32, (M + 31) / 32);
    constexpr int sm = gemm_smem(32, 32, 6);
    epi_dispatch(e, [&](auto em) {
      k_gemm<32, 32, 4, 2, 6, decltype(em)::value>
          <<<grid, 128, sm, st>>>(M, N, K, A, lda, B, ldb, bias, bias_div, C, ldc, e);
    });
    return grid.x;
  }
  return -1;
}

// built-in choice: split-K when neither tiling fills two waves, else 64 x 64
// tiles when they do, else 32 x 32
static int gemm_launch(int M, int N, int K, const float* A, int lda, const float* B, int ldb,
                       const float* bias, int bias_div, float* C, int ldc, const Epi& e,
                       cudaStream_t st) {
  const long big = (long)((N + 63) / 64) * ((M + 63) / 64);
  const long small = (long)((N + 31) / 32) * ((M + 31) / 32);
  if (big < 2 * 152 && small < 2 * 152) {
    const int r = gemm_variant(V_SPLITK, M, N, K, A, lda, B, ldb, bias, bias_div, C, ldc, e, st);
    if (r >= 0) return r;
  }
  return gemm_variant(big >= 2 * 152 ? V_G64 : V_G32, M, N, K, A, lda, B, ldb, bias, bias_div, C,
                      ldc, e, st);
}

// ---------------------------------------------------------------------------
// convolution: transposed (back-substitution) and forward (adjoint / forward)
// ---------------------------------------------------------------------------
template <int CB>
__global__ void __launch_bounds__(128) k_convT(int M, const float* __restrict__ in, int ld_in,
                                               float* out, int ld_out, LayerDev L, Epi e) {
  extern __shared__ float Ws[];
  const int nW = L.co * L.ci * L.k * L.k;
  for (int i = threadIdx.x; i < nW; i += blockDim.x) Ws[i] = L.W[i];
  __syncthreads();
  const int m = blockIdx.y;
  const int Pin = L.hi * L.wi;
  const int pidx = blockIdx.x * blockDim.x + threadIdx.x;
  float part = 0.f;
  if (pidx < Pin) {
    int ih, iw;
    decode_phase(pidx, L.hi, L.wi, L.s, ih, iw);
    const float* lam = in + (size_t)m * ld_in;
    const int kk = L.k * L.k;
    const int hwo = L.ho * L.wo;
    const int kh0 = (ih + L.p) % L.s, kw0 = (iw + L.p) % L.s;
    for (int cb = 0; cb < L.ci; cb += CB) {
      float acc[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) acc[c] = 0.f;
      for (int kh = kh0; kh < L.k; kh += L.s) {
        const int th = ih + L.p - kh;
        if (th < 0) break;
        const int oh = th / L.s;
        if (oh >= L.ho) continue;
        for (int kw = kw0; kw < L.k; kw += L.s) {
          const int tw = iw + L.p - kw;
          if (tw < 0) break;
          const int ow = tw / L.s;
          if (ow >= L.wo) continue;
          const float* lp = lam + oh * L.wo + ow;
          const float* wp = Ws + (size_t)cb * kk + kh * L.k + kw;
          for (int co = 0; co < L.co; ++co) {
            const float v = lp[(size_t)co * hwo];
            const float* w = wp + (size_t)co * L.ci * kk;
#pragma unroll
            for (int c = 0; c < CB; ++c)
              if (CB == 1 || cb + c < L.ci) acc[c] = fmaf(v, w[c * kk], acc[c]);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const int ci = cb + c;
        if (ci >= L.ci) break;
        const int j = ci * Pin + ih * L.wi + iw;
        const float o = epi_apply(e, m, j, acc[c], part);
        if (out) out[(size_t)m * ld_out + j] = o;
      }
    }
  }
  if (epi_has_part(e)) {
    const float tot = block_sum(part);
    if (threadIdx.x == 0) e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = tot;
  }
}

template <int CB>
__global__ void __launch_bounds__(128) k_conv_fwd(int M, const float* __restrict__ in, int ld_in,
                                                  float* out, int ld_out, LayerDev L, Epi e) {
  extern __shared__ float Ws[];
  const int nW = L.co * L.ci * L.k * L.k;
  for (int i = threadIdx.x; i < nW; i += blockDim.x) Ws[i] = L.W[i];
  __syncthreads();
  // rows_per: rows sharing one CTA (output planes smaller than the CTA)
  const int Pout = L.ho * L.wo;
  const int rows_per = Pout >= (int)blockDim.x ? 1 : (int)blockDim.x / Pout;
  const int m = rows_per == 1 ? (int)blockIdx.y : (int)blockIdx.y * rows_per + (int)threadIdx.x / Pout;
  const int pos = rows_per == 1 ? (int)(blockIdx.x * blockDim.x + threadIdx.x) : (int)threadIdx.x % Pout;
  float part = 0.f;
  if (pos < Pout && m < M && (rows_per == 1 || (int)threadIdx.x < rows_per * Pout)) {
    const int oh = pos / L.wo, ow = pos % L.wo;
    const float* x = in + (size_t)m * ld_in;
    const int kk = L.k * L.k;
    const int hwi = L.hi * L.wi;
    for (int cb = 0; cb < L.co; cb += CB) {
      float acc[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) acc[c] = 0.f;
      for (int ci = 0; ci < L.ci; ++ci) {
        for (int kh = 0; kh < L.k; ++kh) {
          const int ih = oh * L.s - L.p + kh;
          if (ih < 0 || ih >= L.hi) continue;
          for (int kw = 0; kw < L.k; ++kw) {
            const int iw = ow * L.s - L.p + kw;
            if (iw < 0 || iw >= L.wi) continue;
            const float v = x[(size_t)ci * hwi + ih * L.wi + iw];
            const float* w = Ws + ((size_t)cb * L.ci + ci) * kk + kh * L.k + kw;
#pragma unroll
            for (int c = 0; c < CB; ++c)
              if (CB == 1 || cb + c < L.co) acc[c] = fmaf(v, w[(size_t)c * L.ci * kk], acc[c]);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const int co = cb + c;
        if (co >= L.co) break;
        const int j = co * Pout + pos;
        const float o = epi_apply(e, m, j, acc[c] + L.b[co], part);
        if (out) out[(size_t)m * ld_out + j] = o;
      }
    }
  }
  // forward epilogues (adjoint, ReLU) produce no offset partials; the partial
  // slot layout below assumes one row per CTA
  if (epi_has_part(e) && rows_per == 1) {
    const float tot = block_sum(part);
    if (threadIdx.x == 0) e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = tot;
  }
}

// Staging into shared memory with all of a thread's loads in flight: rows of
// `width` floats taken at src + r * stride (r < nrows), written densely.  float4
// loads when every row start is 16-byte aligned, 4 per thread per round.
__device__ __forceinline__ void stage_rows(float* __restrict__ dst, const float* __restrict__ src,
                                           int nrows, int width, size_t stride, int valid) {
  const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst) |
                     (stride * 4)) & 15) == 0 &&
                   (width & 3) == 0 && (valid & 3) == 0;
  if (vec) {
    const int w4 = width >> 2, n4 = nrows * w4;
    const FDiv dw = f_div_of(w4);
    float4* d4 = reinterpret_cast<float4*>(dst);
    const int bd = blockDim.x;
    for (int i = threadIdx.x; i < n4; i += 4 * bd) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int ii = min(i + u * bd, n4 - 1), r = f_div(ii, dw), c = (ii - r * w4) * 4;
        v[u] = c < valid ? __ldg(reinterpret_cast<const float4*>(src + r * stride + c))
                         : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + u * bd < n4) d4[i + u * bd] = v[u];
    }
    return;
  }
  const int n = nrows * width;
  const FDiv dw = f_div_of(width);
  const int bd = blockDim.x;
  for (int i = threadIdx.x; i < n; i += 4 * bd) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int ii = min(i + u * bd, n - 1), r = f_div(ii, dw), c = ii - r * width;
      v[u] = c < valid ? __ldg(src + r * stride + c) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * bd < n) dst[i + u * bd] = v[u];
  }
}

// one row of n floats
__device__ __forceinline__ void stage_row(float* __restrict__ dst, const float* __restrict__ src,
                                          int n) {
  const int bd = blockDim.x;
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
    const int n4 = n >> 2;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    float4* d4 = reinterpret_cast<float4*>(dst);
#pragma unroll 4
    for (int i = threadIdx.x; i < n4; i += bd) d4[i] = __ldg(s4 + i);
    for (int i = n4 * 4 + threadIdx.x; i < n; i += bd) dst[i] = __ldg(src + i);
    return;
  }
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += bd) dst[i] = __ldg(src + i);
}

// Row-resident convolution kernels.  A CTA takes one row, one chunk of output
// positions and one group of channel blocks.  It stages the input rows it reads and
// its slice of the weights (pre-arranged in global memory so that a channel
// block is contiguous, float4 loads) in shared memory; each thread computes
// CB channels of one output position.  Few rows are spread over more CTAs
// (position chunks x channel groups) so that a launch fills the GPU.
// What bounds them is latency and instructions, not bandwidth: the epilogue's
// inputs of an item are loaded together (they were issued one output after another,
// each behind its branches), indices are decoded by reciprocal, and registers are
// kept to 5 to 7 CTAs per SM.  Measured before and now: transposed, 594 rows of
// conv_small_28's second layer 77 and 37 us, its first layer 29 and 21 (dense rows),
// 65 and 29 (1462 rows that start at a neuron); resnet_32's first layer, 128 rows,
// 42 and 19.  Forward: 1462 rows of the first layer 50 and 26, 594 of the second 45
// and 22; resnet_32's layers, 128 rows, 36 and 22 on average.
struct ConvSplit {
  int ppc;   // positions per chunk
  int npc;   // position chunks
  int bpg;   // channel blocks per group
  int ngrp;  // channel groups
};

// smem_of(channel width) gives the staged floats for a slice of that width;
// groups are added until the slice fits in `limit` floats.
template <typename F>
static ConvSplit conv_split(int M, int P, int nblk, int CB, F smem_of, int limit) {
  const int per_row = std::max(1, std::min(32, (4 * 152 + M - 1) / M));
  ConvSplit cs;
  int min_grp = 1;
  while (min_grp < nblk && smem_of(((nblk + min_grp - 1) / min_grp) * CB) > limit) ++min_grp;
  cs.ngrp = std::max(min_grp, std::min(nblk, per_row));
  cs.bpg = (nblk + cs.ngrp - 1) / cs.ngrp;
  cs.ngrp = (nblk + cs.bpg - 1) / cs.bpg;
  cs.npc = std::max(1, std::min((per_row + cs.ngrp - 1) / cs.ngrp, (P + 31) / 32));
  cs.npc = std::max(cs.npc, (P + 1023) / 1024);
  cs.ppc = (P + cs.npc - 1) / cs.npc;
  cs.npc = (P + cs.ppc - 1) / cs.ppc;
  return cs;
}

static int convT_row_smem(const LayerDev& L, int cwidth) {
  return L.co * L.ho * L.wo + L.co * L.k * L.k * cwidth;
}

// acc += v w over CB adjacent channels
template <int CB>
__device__ __forceinline__ void row_fma(float v, const float* w, float2 (&acc)[(CB + 1) / 2]) {
  if constexpr (CB % 4 == 0) {
    const float2 vv = make_float2(v, v);
#pragma unroll
    for (int c = 0; c < CB; c += 4) {
      const float4 w4 = *reinterpret_cast<const float4*>(w + c);
      acc[c / 2] = fma2(vv, make_float2(w4.x, w4.y), acc[c / 2]);
      acc[c / 2 + 1] = fma2(vv, make_float2(w4.z, w4.w), acc[c / 2 + 1]);
    }
  } else {
    acc[0].x = fmaf(v, w[0], acc[0].x);
  }
}

// CTAs per SM that the registers allow: as many as leave the epilogue's inputs of
// CB outputs in registers
constexpr int convT_row_ctas(int CB, int EM) {
  return CB == 1 ? 6 : EM > EM_RELU_GAMMA ? 7 : CB == 8 ? 4 : 5;
}

template <int CB, int EM>
__global__ void __launch_bounds__(128, convT_row_ctas(CB, EM)) k_convT_row(int M, const float* __restrict__ in, int ld_in,
                                                   float* out, int ld_out, LayerDev L, Epi e,
                                                   ConvSplit cs) {
  extern __shared__ __align__(16) float sm[];
  const int kk = L.k * L.k;
  const int chunk = blockIdx.x % cs.npc, grp = blockIdx.x / cs.npc;
  const int nblk = (L.ci + CB - 1) / CB;
  const int b0 = grp * cs.bpg, b1 = min(nblk, b0 + cs.bpg);
  const int c0 = b0 * CB, c1 = min(L.ci, b1 * CB);
  const int cw = cs.bpg * CB;       // stride of the staged channel slice
  float* Ws = sm;                   // [co][kh][kw][cw]
  float* Ls = sm + L.co * kk * cw;  // input rows r_lo .. r_hi of every channel
  const int m = blockIdx.y;
  const int Pin = L.hi * L.wi;
  const int p0 = chunk * cs.ppc;
  const int np = min(cs.ppc, Pin - p0);
  // the input rows that the chunk's positions read (stride 1: its positions are
  // consecutive rows; the phase-major order of a larger stride reaches all of them)
  const int r_lo = L.s == 1 ? max(0, p0 / L.wi + L.p - L.k + 1) : 0;
  const int r_hi = L.s == 1 ? min(L.ho - 1, (p0 + np - 1) / L.wi + L.p) : L.ho - 1;
  const int plane = max(0, r_hi - r_lo + 1) * L.wo, nIn = L.co * plane;
  // weight slice: rows (co, kh, kw) of Wb [co][kh][kw][ci], channels c0 .. c0 + cw
  stage_rows(Ws, L.Wb + c0, L.co * kk, cw, (size_t)L.ci, c1 - c0);
  const float* lam = in + (size_t)m * ld_in;
  if (plane == L.ho * L.wo) stage_row(Ls, lam, nIn);
  else if (plane > 0) stage_rows(Ls, lam + r_lo * L.wo, L.co, plane, (size_t)L.ho * L.wo, plane);
  // bounding box (over all channels) of the row's nonzero coefficients: rows
  // that start at a convolution neuron are nonzero only in its receptive field
  // (and at split neurons), and only taps inside the box are summed
  __shared__ int box[4];
  if (threadIdx.x == 0) {
    const bool s = e.sparse_rows != 0;
    box[0] = s ? L.ho : r_lo;
    box[1] = s ? -1 : r_hi;
    box[2] = s ? L.wo : 0;
    box[3] = s ? -1 : L.wo - 1;
  }
  __syncthreads();
  if (e.sparse_rows && plane > 0) {
    const FDiv dhw = f_div_of(plane), dwo = f_div_of(L.wo);
    int bh0 = L.ho, bh1 = -1, bw0 = L.wo, bw1 = -1;
    for (int i = threadIdx.x; i < nIn; i += blockDim.x) {
      if (Ls[i] != 0.f) {
        const int r = f_mod(i, dhw), orow = f_div(r, dwo), ow = r - orow * L.wo, oh = r_lo + orow;
        bh0 = min(bh0, oh); bh1 = max(bh1, oh); bw0 = min(bw0, ow); bw1 = max(bw1, ow);
      }
    }
    bh0 = __reduce_min_sync(0xffffffffu, bh0);
    bh1 = __reduce_max_sync(0xffffffffu, bh1);
    bw0 = __reduce_min_sync(0xffffffffu, bw0);
    bw1 = __reduce_max_sync(0xffffffffu, bw1);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&box[0], bh0);
      atomicMax(&box[1], bh1);
      atomicMin(&box[2], bw0);
      atomicMax(&box[3], bw1);
    }
    __syncthreads();
  }
  const int oh_lo = box[0], oh_hi = box[1], ow_lo = box[2], ow_hi = box[3];
  // a zero coefficient maps to 0 with no offset contribution through these
  // epilogues, so positions that no tap reaches are written as 0 directly
  const bool zero_passes = e.sparse_rows && epi_zero_passes<EM>(e);
  const FDiv dnp = f_div_of(np), ds = f_div_of(L.s);
  const PhaseIdx phases(L.hi, L.wi, L.s);
  const int rn = e.row_node[m];
  const PropDev* rp = epi_prop(e, rn);
  float part = 0.f;
  // U items of a thread together; their epilogue inputs, where they are few, are in
  // flight during the taps
  constexpr int U = CB == 1 ? 4 : 1;
  constexpr bool EARLY = CB == 1 || (CB == 4 && EM == EM_CONC);
  const int items = np * (b1 - b0), bd = blockDim.x;
  for (int i0 = threadIdx.x; i0 < items; i0 += U * bd) {
    float v[U * CB];
    int j[U * CB];
    unsigned ok = 0, have = 0;
    EpiIn pin[U * CB];
    int ihs[U], iws[U], cbs[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int it = min(i0 + u * bd, items - 1), b = f_div(it, dnp), cb = b0 + b;
      int ih, iw;
      if (CB == 1) phases.decode(p0 + it - b * np, ih, iw);
      else decode_phase(p0 + it - b * np, L.hi, L.wi, L.s, ih, iw);
      ihs[u] = ih;
      iws[u] = iw;
      cbs[u] = cb;
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        j[u * CB + c] = min(cb * CB + c, L.ci - 1) * Pin + ih * L.wi + iw;
        if (i0 + u * bd < items && cb * CB + c < L.ci) have |= 1u << (u * CB + c);
        if (EARLY) epi_load_m<EM>(e, rn, rp, m, j[u * CB + c], pin[u * CB + c]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u > 0 && i0 + u * bd >= items) {
#pragma unroll
        for (int c = 0; c < CB; ++c) v[u * CB + c] = 0.f;
        continue;
      }
      // taps kh = kh0 + a s meet input row oh0 - a; columns alike
      const int oh0 = f_div(ihs[u] + L.p, ds), ow0 = f_div(iws[u] + L.p, ds);
      const int kh0 = ihs[u] + L.p - oh0 * L.s, kw0 = iws[u] + L.p - ow0 * L.s;
      const int a0 = max(0, oh0 - oh_hi), a1 = min(f_div(L.k - 1 - kh0 + L.s, ds) - 1, oh0 - oh_lo);
      const int e0 = max(0, ow0 - ow_hi), e1 = min(f_div(L.k - 1 - kw0 + L.s, ds) - 1, ow0 - ow_lo);
      const int coff = (cbs[u] - b0) * CB;
      float2 acc[(CB + 1) / 2];
#pragma unroll
      for (int c = 0; c < (CB + 1) / 2; ++c) acc[c] = make_float2(0.f, 0.f);
      if (!zero_passes || (a0 <= a1 && e0 <= e1)) ok |= ((1u << CB) - 1u) << (u * CB);
      for (int a = a0; a <= a1; ++a)
        for (int q = e0; q <= e1; ++q) {
          const float* lp = Ls + (oh0 - a - r_lo) * L.wo + ow0 - q;
          const float* wp = Ws + ((kh0 + a * L.s) * L.k + kw0 + q * L.s) * cw + coff;
#pragma unroll 4
          for (int co = 0; co < L.co; ++co, lp += plane, wp += kk * cw) row_fma<CB>(*lp, wp, acc);
        }
#pragma unroll
      for (int c = 0; c < CB; ++c) v[u * CB + c] = c & 1 ? acc[c / 2].y : acc[c / 2].x;
    }
    ok &= have;
    if (ok) {
      if (!EARLY) {
#pragma unroll
        for (int c = 0; c < U * CB; ++c) epi_load_m<EM>(e, rn, rp, m, j[c], pin[c]);
      }
      epi_finish_block<EM, U * CB>(e, m, j, v, pin, ok, part);
    }
    if (out) {
#pragma unroll
      for (int c = 0; c < U * CB; ++c)
        if (have >> c & 1u) out[(size_t)m * ld_out + j[c]] = (ok >> c & 1u) ? v[c] : 0.f;
    }
  }
  if (epi_has_part(e)) {
    const float tot = block_sum(part);
    if (threadIdx.x == 0) e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = tot;
  }
}

static int conv_fwd_row_smem(const LayerDev& L, int cwidth) {
  return L.ci * L.hi * L.wi + L.ci * L.k * L.k * cwidth;
}

// acc += v w where `on` (a tap outside the plane is left out, not multiplied by 0)
template <int CB>
__device__ __forceinline__ void row_fma_if(unsigned on, float v, const float (&w)[CB],
                                           float2 (&acc)[CB / 2]) {
  const float2 vv = make_float2(v, v);
  const unsigned long long x = *reinterpret_cast<const unsigned long long*>(&vv);
#pragma unroll
  for (int c = 0; c < CB / 2; ++c) {
    const float2 ww = make_float2(w[2 * c], w[2 * c + 1]);
    unsigned long long r = *reinterpret_cast<unsigned long long*>(&acc[c]);
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p fma.rn.f32x2 %0, %1, %2, %0;\n\t}"
        : "+l"(r)
        : "l"(x), "l"(*reinterpret_cast<const unsigned long long*>(&ww)), "r"(on));
    acc[c] = *reinterpret_cast<float2*>(&r);
  }
}

// The taps of one output position, in (ci, kh, kw) order, CB channels.  xp: its
// input at tap (0, 0), channels `plane` apart; [y0, y1), [x0, x1): the tap rows / columns that lie in the
// plane.  K: the kernel size where it is a constant (the taps are unrolled then).
template <int CB, int K>
__device__ __forceinline__ void fwd_taps(const LayerDev& L, const float* xp, int plane,
                                         const float* wp, int cw, int y0, int y1, int x0, int x1,
                                         float2 (&acc)[CB / 2]) {
  const int k = K ? K : L.k;
  auto weights = [&](const float* w, float (&wv)[CB]) {
#pragma unroll
    for (int c = 0; c < CB; c += 4) {
      const float4 w4 = *reinterpret_cast<const float4*>(w + c);
      wv[c] = w4.x;
      wv[c + 1] = w4.y;
      wv[c + 2] = w4.z;
      wv[c + 3] = w4.w;
    }
  };
  if (K > 0 && L.p == 0) {  // every tap of every position lies in the plane
    for (int ci = 0; ci < L.ci; ++ci, xp += plane, wp += k * k * cw) {
      constexpr int KK = K ? K * K : 1;
      float v[KK];
#pragma unroll
      for (int t = 0; t < KK; ++t) v[t] = xp[t / (K ? K : 1) * L.wi + t % (K ? K : 1)];
#pragma unroll
      for (int t = 0; t < KK; ++t) row_fma<CB>(v[t], wp + t * cw, acc);
    }
  } else if constexpr (K > 0) {
    const unsigned vy = (1u << y1) - (1u << y0), vx = (1u << x1) - (1u << x0);
    unsigned on[K];  // bit kw of on[kh]: the tap lies in the plane
#pragma unroll
    for (int kh = 0; kh < K; ++kh) on[kh] = vy >> kh & 1u ? vx : 0u;
    for (int ci = 0; ci < L.ci; ++ci, xp += plane, wp += K * K * cw) {
      float v[K * K];
#pragma unroll
      for (int t = 0; t < K * K; ++t)
        v[t] = on[t / K] >> t % K & 1u ? xp[t / K * L.wi + t % K] : 0.f;
#pragma unroll
      for (int t = 0; t < K * K; ++t) {
        float wv[CB];
        weights(wp + t * cw, wv);
        row_fma_if<CB>(on[t / K] >> t % K & 1u, v[t], wv, acc);
      }
    }
  } else {
    for (int ci = 0; ci < L.ci; ++ci, xp += plane, wp += k * k * cw)
      for (int kh = y0; kh < y1; ++kh)
#pragma unroll 4
        for (int kw = x0; kw < x1; ++kw) {
          float wv[CB];
          weights(wp + (kh * k + kw) * cw, wv);
          row_fma_if<CB>(1u, xp[kh * L.wi + kw], wv, acc);
        }
  }
}

// The position chunks and channel groups of a row: about 4 x 152 CTAs over all rows,
// and of the ways to split a row that many times the one whose CTAs stage the least
// (a chunk stages only the input rows it reads, a group only its channels' weights).
constexpr int FWD_CTAS = 4;  // (8: 594 rows 30 us instead of 25 on average)
static ConvSplit fwd_split(const LayerDev& L, int M, int CB, int* smem_floats) {
  const int per_row = std::max(1, std::min(32, (FWD_CTAS * 152 + M - 1) / M));
  const int P = L.ho * L.wo, nblk = (L.co + CB - 1) / CB;
  ConvSplit best{};
  long bs = 0;
  for (int g = 1; g <= nblk; ++g) {
    ConvSplit cs;
    cs.bpg = (nblk + g - 1) / g;
    cs.ngrp = (nblk + cs.bpg - 1) / cs.bpg;
    cs.npc = std::max((P + 1023) / 1024,
                      std::max(1, std::min((per_row + cs.ngrp - 1) / cs.ngrp, (P + 31) / 32)));
    cs.ppc = (P + cs.npc - 1) / cs.npc;
    cs.npc = (P + cs.ppc - 1) / cs.ppc;
    const int orows = std::min(L.ho, (cs.ppc + L.wo - 2) / L.wo + 1);  // output rows of a chunk
    const int irows = std::min(L.hi, (orows - 1) * L.s + L.k);
    const long fl = (long)L.ci * (irows * L.wi + (long)L.k * L.k * cs.bpg * CB);
    if (g == 1 || fl < bs) {
      best = cs;
      bs = fl;
    }
    if (g >= per_row && bs <= 40 * 1024) break;
  }
  *smem_floats = (int)std::min<long>(bs, 1 << 28);
  return best;
}

// CB = 4: with eight channels per thread the epilogue's inputs took 118 registers,
// and four CTAs per SM left the loads' latency uncovered (1462 rows: 52 us, now 26;
// two or four positions per thread, which share the weights' loads, 60 and more).
template <int CB, int EM>
__global__ void __launch_bounds__(128, 6) k_conv_fwd_row(int M, const float* __restrict__ in,
                                                      int ld_in, float* out, int ld_out,
                                                      LayerDev L, Epi e, ConvSplit cs) {
  extern __shared__ __align__(16) float sm[];
  const int kk = L.k * L.k;
  const int chunk = blockIdx.x % cs.npc, grp = blockIdx.x / cs.npc;
  const int nblk = (L.co + CB - 1) / CB;
  const int b0 = grp * cs.bpg, b1 = min(nblk, b0 + cs.bpg);
  const int c0 = b0 * CB, c1 = min(L.co, b1 * CB);
  const int cw = cs.bpg * CB;
  float* Ws = sm;                   // [ci][kh][kw][cw]
  float* Xs = sm + L.ci * kk * cw;  // input rows r_lo .. r_hi of every channel
  const int m = blockIdx.y;
  const int P = L.ho * L.wo;
  const int p0 = chunk * cs.ppc;
  const int np = min(cs.ppc, P - p0);
  const int r_lo = max(0, p0 / L.wo * L.s - L.p);
  const int r_hi = min(L.hi - 1, (p0 + np - 1) / L.wo * L.s - L.p + L.k - 1);
  const int plane = max(0, r_hi - r_lo + 1) * L.wi;
  // weight slice: rows (ci, kh, kw) of Wf [ci][kh][kw][co], channels c0 .. c0 + cw
  stage_rows(Ws, L.Wf + c0, L.ci * kk, cw, (size_t)L.co, c1 - c0);
  if (plane > 0)
    stage_rows(Xs, in + (size_t)m * ld_in + r_lo * L.wi, L.ci, plane, (size_t)L.hi * L.wi, plane);
  __syncthreads();
  const FDiv dnp = f_div_of(np), dwo = f_div_of(L.wo);
  const int rn = (EM == EM_ADJ || EM == EM_ADJ_GAMMA) ? e.row_node[m] : 0;
  float part = 0.f;  // forward epilogues (adjoint, ReLU) produce no offset partials
  for (int item = threadIdx.x; item < np * (b1 - b0); item += blockDim.x) {
    const int b = f_div(item, dnp), cb = b0 + b, pos = p0 + item - b * np;
    const int oh = f_div(pos, dwo), ow = pos - oh * L.wo;
    const int ih0 = oh * L.s - L.p, iw0 = ow * L.s - L.p;
    // the item's epilogue inputs are in flight during its taps
    float v[CB];
    int j[CB];
    unsigned ok = 0;
    EpiIn pin[CB];
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int co = min(cb * CB + c, L.co - 1);
      if (cb * CB + c < L.co) ok |= 1u << c;
      j[c] = co * P + pos;
      epi_load_m<EM>(e, rn, nullptr, m, j[c], pin[c]);
    }
    const int y0 = max(0, -ih0), y1 = max(y0, min(L.k, L.hi - ih0));
    const int x0 = max(0, -iw0), x1 = max(x0, min(L.k, L.wi - iw0));
    const float* xp = Xs + (ih0 - r_lo) * L.wi + iw0;
    const float* wp = Ws + b * CB;
    float2 acc[CB / 2];
#pragma unroll
    for (int c = 0; c < CB / 2; ++c) acc[c] = make_float2(0.f, 0.f);
    if (L.k == 3) fwd_taps<CB, 3>(L, xp, plane, wp, cw, min(y0, 3), y1, min(x0, 3), x1, acc);
    else if (L.k == 4) fwd_taps<CB, 4>(L, xp, plane, wp, cw, min(y0, 4), y1, min(x0, 4), x1, acc);
    else fwd_taps<CB, 0>(L, xp, plane, wp, cw, y0, y1, x0, x1, acc);
#pragma unroll
    for (int c = 0; c < CB; ++c)
      v[c] = (c & 1 ? acc[c / 2].y : acc[c / 2].x) + L.b[min(cb * CB + c, L.co - 1)];
    epi_finish_block<EM, CB>(e, m, j, v, pin, ok, part);
    if (out) {
#pragma unroll
      for (int c = 0; c < CB; ++c)
        if (ok >> c & 1u) out[(size_t)m * ld_out + j[c]] = v[c];
    }
  }
}

// ---------------------------------------------------------------------------
// implicit-GEMM convolutions for dense rows
// ---------------------------------------------------------------------------
// Forward: out[m, n, oy, ox] = sum over (ci, kh, kw) of
//   in[m, ci, oy s - p + kh, ox s - p + kw] W[n, ci, kh, kw]  (+ b[n]);
// GEMM rows (m, oy, ox), columns n = co, reduction (ci, kh, kw), weights Wf.
// Transposed (back-substitution): out[m, n, y, x] = sum over (o, kh, kw) with
//   (y + p - kh) and (x + p - kw) divisible by s of
//   in[m, o, (y + p - kh) / s, (x + p - kw) / s] W[o, n, kh, kw].
// Output positions with (y + p) mod s = ry, (x + p) mod s = rx (a parity
// class) take exactly the taps kh = ry + s a, kw = rx + s b, so each class is
// a dense GEMM with reduction (o, a, b) and weights Wb; no masked taps.
// A CTA computes RB rows x one chunk of pc positions of one class x tn
// channels; each row has its own group of tpr threads, so a row's outputs and
// its partial sum do not depend on which rows share the CTA.
struct IgCfg {
  int dir;     // 0 forward, 1 transposed
  int N;       // output channels (co forward, ci transposed)
  int RB, tpr, pc, nchunk, ncls, tn, ngrp, KC;
};

struct IgClass {
  int P, K;             // positions and reduction length of the class
  int y0, x0, ny, nx;   // first output row / column of the class and their counts
  int ry, rx, na, nb;   // residues and tap counts (transposed)
};

__device__ __forceinline__ IgClass ig_class(const LayerDev& L, int dir, int cls) {
  IgClass c;
  if (dir == 0) {
    c.P = L.ho * L.wo;
    c.K = L.ci * L.k * L.k;
    c.y0 = c.x0 = 0;
    c.ny = L.ho;
    c.nx = L.wo;
    c.ry = c.rx = 0;
    c.na = c.nb = L.k;
    return c;
  }
  const int s = L.s;
  c.ry = cls / s;
  c.rx = cls % s;
  c.y0 = ((c.ry - L.p) % s + s) % s;
  c.x0 = ((c.rx - L.p) % s + s) % s;
  c.ny = c.y0 < L.hi ? (L.hi - c.y0 + s - 1) / s : 0;
  c.nx = c.x0 < L.wi ? (L.wi - c.x0 + s - 1) / s : 0;
  c.na = c.ry < L.k ? (L.k - c.ry + s - 1) / s : 0;
  c.nb = c.rx < L.k ? (L.k - c.rx + s - 1) / s : 0;
  c.P = c.ny * c.nx;
  c.K = L.co * c.na * c.nb;
  return c;
}

template <int TN>
__global__ void __launch_bounds__(256) k_conv_igemm(int M, const float* __restrict__ in, int ld_in,
                                                    float* out, int ld_out, LayerDev L, Epi e,
                                                    IgCfg g) {
  extern __shared__ __align__(16) float ism[];
  constexpr int TM = 4;
  constexpr int PPT = 4;  // (row, position) pairs a thread gathers: RB pc <= 4 RB tpr
  __shared__ int t_off[32], t_dy[32], t_dx[32], t_row[32];
  const int nthr = blockDim.x;
  float* As = ism;                              // [KC][RB][pc]
  float* Bs = ism + (size_t)g.KC * g.RB * g.pc;  // [KC][tn]
  const int bx = blockIdx.x;
  const int grp = bx % g.ngrp;
  const int chunk = (bx / g.ngrp) % g.nchunk;
  const int cls = bx / (g.ngrp * g.nchunk);
  const IgClass c = ig_class(L, g.dir, cls);
  const int m0 = blockIdx.y * g.RB;
  const int p0 = chunk * g.pc;
  const int np = max(0, min(g.pc, c.P - p0));
  const int n0 = grp * g.tn;
  const int nn = min(g.tn, g.N - n0);
  const int q = threadIdx.x / g.tpr, tl = threadIdx.x % g.tpr;
  const int npg = g.pc / TM, nng = g.tn / TN;
  const int pg = tl % npg, ng = tl / npg;
  const bool act = q < g.RB && ng < nng;
  const int rpc = g.RB * g.pc;
  const float* Wsrc = g.dir == 0 ? L.Wf : L.Wb;
  // source plane of the gather (input of the forward conv, coefficients of the
  // transposed one) and this thread's gather pairs, decoded once
  const int Hs = g.dir == 0 ? L.hi : L.ho, Ws_ = g.dir == 0 ? L.wi : L.wo;
  int pr_base[PPT], pr_y[PPT], pr_x[PPT];
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    const int pr = threadIdx.x + i * nthr;
    const int qq = pr / g.pc, pos = pr % g.pc;
    pr_base[i] = -1;
    pr_y[i] = pr_x[i] = 0;
    if (pr < rpc && m0 + qq < M && pos < np) {
      const int pi = p0 + pos;
      const int iy = pi / c.nx, ix = pi % c.nx;
      int y, x;
      if (g.dir == 0) {
        y = iy * L.s - L.p;
        x = ix * L.s - L.p;
      } else {
        y = (c.y0 + L.s * iy + L.p - c.ry) / L.s;
        x = (c.x0 + L.s * ix + L.p - c.rx) / L.s;
      }
      pr_y[i] = y;
      pr_x[i] = x;
      pr_base[i] = 0;  // valid pair; the row offset is added at the load
    }
  }
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int jn = 0; jn < TN; ++jn) acc[i][jn] = 0.f;
  const int Kc = np > 0 ? c.K : 0;
  const int KC = min(g.KC, 32);
  for (int k0 = 0; k0 < Kc; k0 += KC) {
    const int kcn = min(KC, Kc - k0);
    __syncthreads();
    // reduction-index table of this chunk: channel-plane offset, tap shifts, weight row
    if (threadIdx.x < kcn) {
      const int kidx = k0 + threadIdx.x;
      if (g.dir == 0) {
        const int kk2 = L.k * L.k;
        const int ci = kidx / kk2, kh = (kidx / L.k) % L.k, kw = kidx % L.k;
        t_dy[threadIdx.x] = kh;
        t_dx[threadIdx.x] = kw;
        t_off[threadIdx.x] = ci * L.hi * L.wi;
        t_row[threadIdx.x] = kidx;  // Wf [ci][kh][kw][co]
      } else {
        const int nab = c.na * c.nb;
        const int o = kidx / nab, a = (kidx / c.nb) % c.na, b = kidx % c.nb;
        t_dy[threadIdx.x] = -a;
        t_dx[threadIdx.x] = -b;
        t_off[threadIdx.x] = o * L.ho * L.wo;
        t_row[threadIdx.x] = (o * L.k + c.ry + L.s * a) * L.k + c.rx + L.s * b;  // Wb [co][kh][kw][ci]
      }
    }
    __syncthreads();
    // gather the A chunk: consecutive threads take consecutive positions
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
      const int pr = threadIdx.x + i * nthr;
      if (pr >= rpc) break;
      const float* src = in + (size_t)(m0 + pr / g.pc) * ld_in;
      for (int kk = 0; kk < kcn; ++kk) {
        float v = 0.f;
        if (pr_base[i] == 0) {
          const int yy = pr_y[i] + t_dy[kk], xx = pr_x[i] + t_dx[kk];
          if (yy >= 0 && yy < Hs && xx >= 0 && xx < Ws_) v = __ldg(src + t_off[kk] + yy * Ws_ + xx);
        }
        As[kk * rpc + pr] = v;
      }
    }
    // the B chunk: weight rows of the reduction indices, channels n0 .. n0 + tn
    for (int el = threadIdx.x; el < kcn * g.tn; el += nthr) {
      const int kk = el / g.tn, n = el % g.tn;
      Bs[kk * g.tn + n] = n < nn ? __ldg(Wsrc + (size_t)t_row[kk] * g.N + n0 + n) : 0.f;
    }
    __syncthreads();
    if (act) {
      const float* ap = As + q * g.pc + pg * TM;
      const float* bp = Bs + ng * TN;
#pragma unroll 4
      for (int kk = 0; kk < kcn; ++kk) {
        const float4 a4 = *reinterpret_cast<const float4*>(ap + (size_t)kk * rpc);
        float bv[TN];
        if constexpr (TN == 4) {
          const float4 b4 = *reinterpret_cast<const float4*>(bp + kk * g.tn);
          bv[0] = b4.x;
          bv[1] = b4.y;
          bv[2] = b4.z;
          bv[3] = b4.w;
        } else {
#pragma unroll
          for (int jn = 0; jn < TN; ++jn) bv[jn] = bp[kk * g.tn + jn];
        }
        const float av[TM] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int jn = 0; jn < TN; ++jn) acc[i][jn] = fmaf(av[i], bv[jn], acc[i][jn]);
      }
    }
  }
  // epilogue
  float part = 0.f;
  const int m = m0 + q;
  if (act && m < M) {
    const int plane = g.dir == 0 ? L.ho * L.wo : L.hi * L.wi;
    const int W2 = g.dir == 0 ? L.wo : L.wi;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int pos = pg * TM + i;
      if (pos >= np) break;
      const int pi = p0 + pos;
      const int iy = pi / c.nx, ix = pi % c.nx;
      const int y = g.dir == 0 ? iy : c.y0 + L.s * iy;
      const int x = g.dir == 0 ? ix : c.x0 + L.s * ix;
#pragma unroll
      for (int jn = 0; jn < TN; ++jn) {
        const int n = ng * TN + jn;
        if (n >= nn) break;
        const int j = (n0 + n) * plane + y * W2 + x;
        float v = acc[i][jn];
        if (g.dir == 0) v += L.b[n0 + n];
        const float o = epi_apply(e, m, j, v, part);
        if (out) out[(size_t)m * ld_out + j] = o;
      }
    }
  }
  if (g.dir == 1 && epi_has_part(e)) {
    // per-row sum in a fixed order: warps of the row group, then their sums
    __shared__ float wsum[32];
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = part;
    __syncthreads();
    const int wpr = g.tpr >> 5;
    if (tl == 0 && q < g.RB && m < M) {
      float tot = 0.f;
      for (int w = 0; w < wpr; ++w) tot += wsum[q * wpr + w];
      e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = tot;
    }
  }
}

static IgCfg ig_plan(const LayerDev& L, int dir, int M) {
  IgCfg g;
  g.dir = dir;
  g.N = dir == 0 ? L.co : L.ci;
  const int TN = g.N % 4 == 0 ? 4 : 1;
  g.tn = TN == 4 ? std::min(g.N, 64) : std::min(g.N, 8);
  g.ncls = dir == 0 ? 1 : L.s * L.s;
  int pmax = 0;
  if (dir == 0) {
    pmax = L.ho * L.wo;
  } else {
    for (int r = 0; r < L.s; ++r) {
      const int y0 = ((r - L.p) % L.s + L.s) % L.s;
      const int ny = y0 < L.hi ? (L.hi - y0 + L.s - 1) / L.s : 0;
      for (int r2 = 0; r2 < L.s; ++r2) {
        const int x0 = ((r2 - L.p) % L.s + L.s) % L.s;
        const int nx = x0 < L.wi ? (L.wi - x0 + L.s - 1) / L.s : 0;
        pmax = std::max(pmax, ny * nx);
      }
    }
  }
  const int cap = TN == 4 ? 64 : 128;
  g.pc = std::max(4, std::min((pmax + 3) / 4 * 4, cap));
  // few rows: fewer rows per CTA, then narrower channel groups and shorter
  // position chunks, so that the grid covers the SMs (at most the ig_slots blocks)
  g.RB = 8;
  for (;;) {
    g.ngrp = (g.N + g.tn - 1) / g.tn;
    g.nchunk = std::max(1, (pmax + g.pc - 1) / g.pc);
    g.tpr = ((g.pc / 4) * (g.tn / TN) + 31) / 32 * 32;
    g.RB = std::max(1, std::min(g.RB, 256 / g.tpr));
    const long blocks = (long)((M + g.RB - 1) / g.RB) * g.ncls * g.nchunk * g.ngrp;
    if (blocks >= 2 * 152) break;
    if (g.RB > 1) g.RB >>= 1;
    else if (TN == 4 && g.tn > 16) g.tn = (g.tn / 2 + 3) / 4 * 4;
    else if (g.pc > 16) g.pc = std::max(16, (g.pc / 2 + 3) / 4 * 4);
    else break;
  }
  g.KC = g.RB * g.pc <= 512 ? 32 : 16;  // at most 32 (reduction-index table)
  return g;
}

static int ig_smem(const IgCfg& g) { return g.KC * (g.RB * g.pc + g.tn) * (int)sizeof(float); }

static bool ig_supported(const LayerDev& L, int dir) {
  const IgCfg g = ig_plan(L, dir, 1 << 20);
  return g.tpr <= 256 && ig_smem(g) <= 96 * 1024 && (dir == 0 ? L.Wf : L.Wb) != nullptr;
}

static int ig_slots(const LayerDev& L) {
  // the finest split of ig_plan (one row: position chunks of 16, channel groups of 16)
  const IgCfg g = ig_plan(L, 1, 1);
  return g.ncls * g.nchunk * g.ngrp;
}

// Per-row work above which the implicit GEMM beats the row-resident kernels
// (whose per-row CTAs then serialise too much work)
static bool ig_preferred(const LayerDev& L) {
  return (double)L.co * L.ho * L.wo * L.ci * L.k * L.k >= 512.0 * 1024.0;
}

// Transposed convolution of stride 1 to at most three channels (a network's input):
// a warp computes 128 consecutive positions of one row, a thread four of them and
// all N channels, in the implicit GEMM's order of taps (o, kh, kw) and of offset
// sums (a channel's four positions, the 32 lanes, then the channels), so that both
// give the same bits.  G warps share the source rows they read, which are staged
// OC channels at a time by asynchronous copies while the previous ones are summed.
// The implicit GEMM gives such a layer one channel per thread and gathers each tap's
// coefficients into shared memory: nine copies of the row for three FMAs each.  Here
// six loaded coefficients serve 36 FMAs.  Measured, 32 channels of 32 x 32 through a
// 3x3 kernel to three: 64 rows 102 us with the implicit GEMM, 14.5 here; 256 rows 214
// and 24, 1024 rows 657 and 74 (reading the coefficients once would take 20).  What
// is left is instructions: 108 of a channel's 130 or so per thread are the FMAs.
constexpr int NARROW_OC = 8;   // source channels per stage
constexpr int NARROW_ST = 2;   // stages

struct NarrowCfg {
  int G;       // warps (128 positions each) per CTA
  int nchunk;  // 128-position chunks of a row
  int rows;    // staged source rows of a CTA (at most)
  int sw;      // their stride
  int smem;
};

template <int K, int N, int EM>
__global__ void __launch_bounds__(128) k_convT_narrow(const float* __restrict__ in, int ld_in,
                                                      float* out, int ld_out, LayerDev L, Epi e,
                                                      NarrowCfg g) {
  extern __shared__ __align__(16) float nsm[];
  const int stage = NARROW_OC * g.rows * g.sw;
  float* Wn = nsm + NARROW_ST * stage;  // [o][kh][kw][4]
  const int m = blockIdx.y, nthr = blockDim.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int P = L.hi * L.wi, hwo = L.ho * L.wo;
  const int p_lo = blockIdx.x * g.G * 128, p_hi = min(P, p_lo + g.G * 128) - 1;
  const FDiv dw = f_div_of(L.wi);
  const int y_lo = f_div(p_lo, dw), y_hi = f_div(p_hi, dw);
  // staged source rows: yb .. ye of the plane, yb + i at row i; columns shifted by
  // K - 1 - p; what lies outside the plane stays zero
  const int yb = y_lo + L.p - K + 1, v_lo = max(0, yb), v_hi = min(L.ho - 1, y_hi + L.p);
  const int nrow = max(0, v_hi - v_lo + 1);
  for (int i = threadIdx.x; i < NARROW_ST * stage / 4; i += nthr)
    reinterpret_cast<float4*>(nsm)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = threadIdx.x; i < L.co * K * K * 4; i += nthr)
    Wn[i] = (i & 3) < N ? __ldg(L.Wb + (i >> 2) * N + (i & 3)) : 0.f;
  __syncthreads();
  const float* src = in + (size_t)m * ld_in + v_lo * L.wo;
  const int nel = nrow * L.wo;  // staged elements of a channel: consecutive in memory
  const FDiv dwo = f_div_of(L.wo);
  auto load = [&](int c) {  // channels c OC .. of the row into stage c mod ST
    const int o0 = c * NARROW_OC, no = min(NARROW_OC, L.co - o0);
    const unsigned base = static_cast<unsigned>(__cvta_generic_to_shared(
        nsm + c % NARROW_ST * stage + (v_lo - yb) * g.sw + K - 1 - L.p));
    const float* s0 = src + (size_t)o0 * hwo;
    const unsigned dstep = (unsigned)(g.rows * g.sw) * 4u;
    for (int q = threadIdx.x; q < nel; q += nthr) {
      const int r = f_div(q, dwo);
      unsigned d = base + (unsigned)(r * g.sw + q - r * L.wo) * 4u;
      const float* s = s0 + q;
#pragma unroll 4
      for (int o = 0; o < no; ++o, d += dstep, s += hwo)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(s) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int nc = (L.co + NARROW_OC - 1) / NARROW_OC;
  const int chunk = blockIdx.x * g.G + warp, pos = chunk * 128 + lane * 4;
  const bool act = pos < P;  // (P is a multiple of four)
  const int y = act ? f_div(pos, dw) : y_lo, x = act ? pos - y * L.wi : 0;
  float acc[N][4];
#pragma unroll
  for (int n = 0; n < N; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[n][i] = 0.f;
  load(0);
  for (int c = 0; c < nc; ++c) {
    if (c + 1 < nc) {
      load(c + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* sp = nsm + c % NARROW_ST * stage + (y - y_lo + K - 1) * g.sw + x;
    const float* wp = Wn + c * NARROW_OC * K * K * 4;
    const int no = min(NARROW_OC, L.co - c * NARROW_OC);
#pragma unroll 1
    for (int o = 0; o < no; ++o, sp += g.rows * g.sw, wp += K * K * 4) {
#pragma unroll
      for (int a = 0; a < K; ++a) {
        // coefficient x + i + p - b lies at column x + i + K - 1 - b
        constexpr int NV = (K + 3 + 1) / 2 * 2;
        float v[NV];
#pragma unroll
        for (int u = 0; u < NV; u += 4) {
          if (u + 4 <= NV) {
            const float4 q = *reinterpret_cast<const float4*>(sp - a * g.sw + u);
            v[u] = q.x;
            v[u + 1] = q.y;
            v[u + 2] = q.z;
            v[u + 3] = q.w;
          } else {
            const float2 q = *reinterpret_cast<const float2*>(sp - a * g.sw + u);
            v[u] = q.x;
            v[u + 1] = q.y;
          }
        }
#pragma unroll
        for (int b = 0; b < K; ++b) {
          const float4 w4 = *reinterpret_cast<const float4*>(wp + (a * K + b) * 4);
          const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
          for (int n = 0; n < N; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[n][i] = fmaf(v[i + K - 1 - b], w[n], acc[n][i]);
        }
      }
    }
    __syncthreads();
  }
  float tot = 0.f;
  const int rn = e.row_node[m];
  const PropDev* rp = epi_prop(e, rn);
#pragma unroll
  for (int n = 0; n < N; ++n) {
    float part = 0.f;
    if (act) {
      int j[4];
      EpiIn pin[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        j[i] = n * P + pos + i;
        epi_load_m<EM>(e, rn, rp, m, j[i], pin[i]);
      }
      epi_finish_block<EM, 4>(e, m, j, acc[n], pin, 15u, part);
      if (out) {
#pragma unroll
        for (int i = 0; i < 4; ++i) out[(size_t)m * ld_out + j[i]] = acc[n][i];
      }
    }
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    tot += part;
  }
  if (epi_has_part(e) && lane == 0 && chunk < g.nchunk)
    e.part[(size_t)m * e.nslot + e.slot_base + chunk] = tot;
}

// Whether k_convT_narrow takes what the implicit GEMM's plan g would do: whole
// 128-position chunks (from 38 rows of 1024 positions on; with fewer rows the plan's
// shorter chunks spread a row over more SMs).
static bool narrow_plan(const LayerDev& L, int dir, int M, const IgCfg& g, NarrowCfg* c) {
  if (dir != 1 || L.s != 1 || (L.k != 3 && L.k != 5) || L.ci > 3 || (L.wi & 3) || L.p > L.k - 1 ||
      g.pc != 128 || g.ngrp != 1)
    return false;
  c->nchunk = g.nchunk;
  // CTAs of four warps while they fill the SMs, else of two (one: 15.8 us for 64 rows)
  c->G = 4;
  while (c->G > 2 && (long)M * ((c->nchunk + c->G - 1) / c->G) < 2 * 152) c->G >>= 1;
  c->rows = (c->G * 128 + L.wi - 2) / L.wi + L.k;
  c->sw = (L.wi + L.k - 1 + 3) / 4 * 4;
  c->smem = (NARROW_ST * NARROW_OC * c->rows * c->sw + L.co * L.k * L.k * 4) * 4;
  return c->smem <= 96 * 1024;
}

static void launch_narrow(const LayerDev& L, int M, const float* in, int ld_in, float* out,
                          int ld_out, const Epi& e, const NarrowCfg& c, cudaStream_t st) {
  dim3 grid((c.nchunk + c.G - 1) / c.G, M);
  epi_dispatch_back(e, [&](auto em) {
    constexpr int EM = decltype(em)::value;
    auto go = [&](auto kern) {
      set_smem(kern, c.smem);
      kern<<<grid, 32 * c.G, c.smem, st>>>(in, ld_in, out, ld_out, L, e, c);
    };
    auto by_n = [&](auto k) {
      constexpr int K = decltype(k)::value;
      if (L.ci == 1) go(k_convT_narrow<K, 1, EM>);
      else if (L.ci == 2) go(k_convT_narrow<K, 2, EM>);
      else go(k_convT_narrow<K, 3, EM>);
    };
    if (L.k == 3) by_n(std::integral_constant<int, 3>{});
    else by_n(std::integral_constant<int, 5>{});
  });
}

// launches the implicit-GEMM kernel; returns the partial-sum slots (transposed)
static int launch_ig(const LayerDev& L, int dir, int M, const float* in, int ld_in, float* out,
                     int ld_out, const Epi& e, cudaStream_t st) {
  const IgCfg g = ig_plan(L, dir, M);
  NarrowCfg nc;
  if (narrow_plan(L, dir, M, g, &nc)) {
    launch_narrow(L, M, in, ld_in, out, ld_out, e, nc, st);
    return g.nchunk;
  }
  const int smem = ig_smem(g);
  dim3 grid(g.ncls * g.nchunk * g.ngrp, (M + g.RB - 1) / g.RB);
  const int thr = g.RB * g.tpr;
  if (g.N % 4 == 0) {
    set_smem(k_conv_igemm<4>, smem);
    k_conv_igemm<4><<<grid, thr, smem, st>>>(M, in, ld_in, out, ld_out, L, e, g);
  } else {
    set_smem(k_conv_igemm<1>, smem);
    k_conv_igemm<1><<<grid, thr, smem, st>>>(M, in, ld_in, out, ld_out, L, e, g);
  }
  return grid.x;
}

// Tensor-core path: always when forced, and automatically when the problem
// fills at least two waves of 128 x BN tiles on the 152 SMs.
static bool use_tc(const Epi& e, int M, int N) {
  if (e.gemm_path == 2) return true;
  if (e.gemm_path != 0 || !e.err) return false;
  const int bn = N <= 64 ? 64 : (N <= 128 ? 128 : 256);
  return (long)((M + 127) / 128) * ((N + bn - 1) / bn) >= 2 * 152;
}

// Whether the row-resident conv kernels can stage this layer (input row plus the
// narrowest weight slice within 40 K floats = 160 KB of shared memory).
bool conv_supported(const LayerDev& L) {
  const int cbT = L.ci <= 1 ? 1 : (L.ci <= 4 ? 4 : 8);
  return convT_row_smem(L, cbT) <= 40 * 1024 && conv_fwd_row_smem(L, 4) <= 40 * 1024;
}

// Tensor-core convolutions: always with gemm_path 2, never with 1, and with 0
// where the SIMT kernels would take the implicit GEMM (large per-row work);
// dense rows only (rows started at one neuron skip their zero region in the
// row-resident kernels)
static bool use_tc_conv(const LayerDev& L, int dir, const Epi& e) {
  if (e.gemm_path == 1 || !tc_conv_usable(L, dir)) return false;
  if (dir == 1 && e.sparse_rows) return false;
  return e.gemm_path == 2 || (double)L.co * L.ho * L.wo * L.ci * L.k * L.k >= 512.0 * 1024.0;
}

static int tuned_variant(const LayerDev& L, int dir, int M, const Epi& e);

bool conv_tc_chosen(const LayerDev& L, int dir, const Epi& e, int M) {
  if (L.kind != MNBAB_CONV2D) return false;
  const int tv = tuned_variant(L, dir, M, e);
  if (tv > 0) return tv == V_TC && tc_conv_usable(L, dir);
  return use_tc_conv(L, dir, e);
}

int backsub_slots(const LayerDev& L) {
  if (L.kind == 1) return (L.d_in + 31) / 32;  // upper bound over the tile shapes
  // upper bound over the implicit-GEMM blocks, the row-resident splits (<= 32
  // CTAs per row, more for large planes) and the fallback tiling (128 positions
  // per CTA)
  const int P = L.hi * L.wi;
  return std::max(std::max(std::max(32 * ((P + 1023) / 1024), (P + 127) / 128), ig_slots(L)),
                  tc_conv_slots(L));
}

// One variant of the transposed convolution (back-substitution, dir 1) or the
// convolution (forward, dir 0); -1 when it does not take this layer.
static int conv_variant(int v, int dir, const LayerDev& L, int M, const float* in, int ld_in,
                        float* out, int ld_out, const Epi& e, cudaStream_t st) {
  if (v == V_TC) {
    if (!tc_conv_usable(L, dir) || (dir == 1 && e.sparse_rows)) return -1;
    const int slots = launch_tc_conv(L, dir, M, in, ld_in, out, ld_out, e, st);
    return dir == 1 ? slots : 0;
  }
  if (v == V_IG) {
    if (!ig_supported(L, dir) || (dir == 1 && e.sparse_rows)) return -1;
    const int slots = launch_ig(L, dir, M, in, ld_in, out, ld_out, e, st);
    return dir == 1 ? slots : 0;
  }
  if (v == V_ROW && dir == 1) {
    const int CBv = L.ci <= 1 ? 1 : (L.ci <= 4 ? 4 : 8);
    const ConvSplit cs = conv_split(M, L.hi * L.wi, (L.ci + CBv - 1) / CBv, CBv,
                                    [&](int cw) { return convT_row_smem(L, cw); }, 40 * 1024);
    // (stride 1: a chunk's input rows only)
    const int irows = std::min(L.ho, L.s == 1 ? (cs.ppc + L.wi - 2) / L.wi + L.k : L.ho);
    const int rsm = (convT_row_smem(L, cs.bpg * CBv) - L.co * (L.ho - irows) * L.wo) * 4;
    if (rsm > 160 * 1024 || !L.Wb || cs.npc * cs.ngrp > backsub_slots(L)) return -1;
    dim3 grid(cs.npc * cs.ngrp, M);
    epi_dispatch_back(e, [&](auto em) {
      auto go = [&](auto kern) {
        set_smem(kern, rsm);
        kern<<<grid, 128, rsm, st>>>(M, in, ld_in, out, ld_out, L, e, cs);
      };
      constexpr int EM = decltype(em)::value;
      if (CBv == 1) go(k_convT_row<1, EM>);
      else if (CBv == 4) go(k_convT_row<4, EM>);
      else go(k_convT_row<8, EM>);
    });
    return grid.x;
  }
  if (v == V_ROW && dir == 0) {
    constexpr int CB = 4;
    int fl;
    const ConvSplit cs = fwd_split(L, M, CB, &fl);
    const int rsm = fl * 4;
    if (rsm > 160 * 1024 || !L.Wf) return -1;
    dim3 grid(cs.npc * cs.ngrp, M);
    epi_dispatch_fwd(e, [&](auto em) {
      auto kern = k_conv_fwd_row<CB, decltype(em)::value>;
      set_smem(kern, rsm);
      kern<<<grid, 128, rsm, st>>>(M, in, ld_in, out, ld_out, L, e, cs);
    });
    return 0;
  }
  if (v == V_PLAIN) {
    const int smem = L.co * L.ci * L.k * L.k * 4;
    if (smem > 200 * 1024) return -1;
    if (dir == 1) {
      dim3 grid((L.hi * L.wi + 127) / 128, M);
      if (L.ci <= 1) {
        set_smem(k_convT<1>, smem);
        k_convT<1><<<grid, 128, smem, st>>>(M, in, ld_in, out, ld_out, L, e);
      } else if (L.ci <= 4) {
        set_smem(k_convT<4>, smem);
        k_convT<4><<<grid, 128, smem, st>>>(M, in, ld_in, out, ld_out, L, e);
      } else if (L.ci <= 16) {
        set_smem(k_convT<16>, smem);
        k_convT<16><<<grid, 128, smem, st>>>(M, in, ld_in, out, ld_out, L, e);
      } else {
        set_smem(k_convT<32>, smem);
        k_convT<32><<<grid, 128, smem, st>>>(M, in, ld_in, out, ld_out, L, e);
      }
      return grid.x;
    }
    const int Pout = L.ho * L.wo;
    const int rows_per = Pout >= 128 ? 1 : 128 / Pout;
    dim3 grid(rows_per == 1 ? (Pout + 127) / 128 : 1, (M + rows_per - 1) / rows_per);
    if (L.co <= 16) {
      set_smem(k_conv_fwd<16>, smem);
      k_conv_fwd<16><<<grid, 128, smem, st>>>(M, in, ld_in, out, ld_out, L, e);
    } else {
      set_smem(k_conv_fwd<32>, smem);
      k_conv_fwd<32><<<grid, 128, smem, st>>>(M, in, ld_in, out, ld_out, L, e);
    }
    return 0;
  }
  return -1;
}

int launch_affine_variant(int v, int dir, const LayerDev& L, int M, const float* in, int ld_in,
                          float* out, int ld_out, const Epi& e, cudaStream_t st) {
  if (M <= 0) return -1;
  if (L.kind == 1) {
    if (v == V_TC) {
      const int slots =
          dir == 1 ? launch_gemm_tc(M, L.d_in, L.d_out, in, ld_in, nullptr, 1, out, ld_out, e,
                                    e.err, st, L.tc, 1)
                   : launch_gemm_tc(M, L.d_out, L.d_in, in, ld_in, L.b, 1, out, ld_out, e, e.err,
                                    st, L.tc, 0);
      return slots < 0 ? -1 : (dir == 1 ? slots : 0);
    }
    // back-substitution Lambda [M][d_out] x W [d_out][d_in]; forward G [M][d_in] x W^T + b
    const int slots =
        dir == 1 ? gemm_variant(v, M, L.d_in, L.d_out, in, ld_in, L.W, L.d_in, nullptr, 1, out,
                                ld_out, e, st)
                 : gemm_variant(v, M, L.d_out, L.d_in, in, ld_in, L.Wt, L.d_out, L.b, 1, out,
                                ld_out, e, st);
    return slots < 0 ? -1 : (dir == 1 ? slots : 0);
  }
  return conv_variant(v, dir, L, M, in, ld_in, out, ld_out, e, st);
}

// the autotuner's variant for this launch, if it applies: not under a forced
// GEMM path, and not for rows that the built-in choice serves with the
// sparse-row kernels
static int tuned_variant(const LayerDev& L, int dir, int M, const Epi& e) {
  if (e.gemm_path != 0 || (dir == 1 && e.sparse_rows && L.kind != 1)) return 0;
  return L.tune[dir][tune_bucket(M)];
}

int launch_backsub(const LayerDev& L, int M, const float* in, int ld_in, float* out, int ld_out,
                   const Epi& e, cudaStream_t st) {
  if (M <= 0) return backsub_slots(L);
  const int tv = tuned_variant(L, 1, M, e);
  if (tv > 0) {
    const int slots = launch_affine_variant(tv, 1, L, M, in, ld_in, out, ld_out, e, st);
    if (slots >= 0) return slots;
  }
  if (L.kind == 1) {
    // Lambda [M][d_out] x W [d_out][d_in]; the tensor-core kernel takes W as [d_in][d_out] = W^T
    if (use_tc(e, M, L.d_in)) {
      const int slots = launch_affine_variant(V_TC, 1, L, M, in, ld_in, out, ld_out, e, st);
      if (slots >= 0) return slots;
    }
    return gemm_launch(M, L.d_in, L.d_out, in, ld_in, L.W, L.d_in, nullptr, 1, out, ld_out, e, st);
  }
  if (use_tc_conv(L, 1, e)) return launch_tc_conv(L, 1, M, in, ld_in, out, ld_out, e, st);
  // dense rows: implicit GEMM per parity class; rows that start at a neuron
  // (nonzero only near it) skip the zero region in the row-resident kernel
  if (!e.sparse_rows && ig_supported(L, 1) && (ig_preferred(L) || !conv_supported(L)))
    return launch_ig(L, 1, M, in, ld_in, out, ld_out, e, st);
  const int slots = conv_variant(V_ROW, 1, L, M, in, ld_in, out, ld_out, e, st);
  if (slots >= 0) return slots;
  return conv_variant(V_PLAIN, 1, L, M, in, ld_in, out, ld_out, e, st);
}

void launch_forward(const LayerDev& L, int M, const float* in, int ld_in, float* out, int ld_out,
                    const Epi& e, cudaStream_t st) {
  if (M <= 0) return;
  const int tv = tuned_variant(L, 0, M, e);
  if (tv > 0 && launch_affine_variant(tv, 0, L, M, in, ld_in, out, ld_out, e, st) >= 0) return;
  if (L.kind == 1) {
    // G [M][d_in] x W^T + b; the tensor-core kernel takes W [d_out][d_in] as is
    if (use_tc(e, M, L.d_out) &&
        launch_affine_variant(V_TC, 0, L, M, in, ld_in, out, ld_out, e, st) >= 0)
      return;
    gemm_launch(M, L.d_out, L.d_in, in, ld_in, L.Wt, L.d_out, L.b, 1, out, ld_out, e, st);
    return;
  }
  if (use_tc_conv(L, 0, e)) {
    launch_tc_conv(L, 0, M, in, ld_in, out, ld_out, e, st);
    return;
  }
  if (ig_supported(L, 0) && (ig_preferred(L) || !conv_supported(L))) {
    launch_ig(L, 0, M, in, ld_in, out, ld_out, e, st);
    return;
  }
  if (conv_variant(V_ROW, 0, L, M, in, ld_in, out, ld_out, e, st) >= 0) return;
  conv_variant(V_PLAIN, 0, L, M, in, ld_in, out, ld_out, e, st);
}

// ---------------------------------------------------------------------------
// reductions and bookkeeping
// ---------------------------------------------------------------------------
// The CTA loads a row's partials together and one thread adds them in slot
// order (the sum does not depend on how they were loaded).
__global__ void __launch_bounds__(128) k_reduce_lb(int M, const float* part, int nslot, int used,
                                                   const float* gp0, float* lb, int track,
                                                   const int* row_node, PoolDev pool,
                                                   const float* X, int d0) {
  const int m = blockIdx.x;
  __shared__ int imp;
  __shared__ int node;
  __shared__ __align__(16) float s[1024];
  const float* p = part + (size_t)m * nslot;
  float acc = 0.f;
  for (int i0 = 0; i0 < used; i0 += 1024) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 128 * u + threadIdx.x;
      if (i0 + i < used) s[i] = p[i0 + i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const int n = min(1024, used - i0);
      int i = 0;
      for (; i + 8 <= n; i += 8) {
        const float4 a = *reinterpret_cast<const float4*>(s + i);
        const float4 b = *reinterpret_cast<const float4*>(s + i + 4);
        acc += a.x;
        acc += a.y;
        acc += a.z;
        acc += a.w;
        acc += b.x;
        acc += b.y;
        acc += b.z;
        acc += b.w;
      }
      for (; i < n; ++i) acc += s[i];
    }
  }
  if (threadIdx.x < 32) {
    float g = gp0 && threadIdx.x < GP_SPLIT ? gp0[(size_t)m * GP_SPLIT + threadIdx.x] : 0.f;
    for (int o = 16; o; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    if (threadIdx.x == 0) {
      if (gp0) acc -= g;
      lb[m] = acc;
      imp = 0;
      node = row_node ? row_node[m] : 0;
      if (track && acc > pool.BEST[node]) {
        pool.BEST[node] = acc;
        imp = 1;
      }
    }
  }
  __syncthreads();
  if (!imp) return;
  // the minimiser: eight loads in flight per thread (one by one, the 3072 values of
  // a 3x32x32 input were most of the launch)
  const float* x = X + (size_t)m * d0;
  float* bx = pool.BESTX + (size_t)node * d0;
  for (int k0 = threadIdx.x; k0 < d0; k0 += 8 * 128) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k0 + 128 * u < d0) v[u] = x[k0 + 128 * u];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k0 + 128 * u < d0) bx[k0 + 128 * u] = v[u];
  }
}

void launch_reduce_lb(int M, const float* part, int nslot, int used, const float* gp0, float* lb,
                      bool track, const int* row_node, PoolDev pool, const float* X, int d0,
                      cudaStream_t st) {
  if (M <= 0) return;
  k_reduce_lb<<<M, 128, 0, st>>>(M, part, nslot, used, gp0, lb, track ? 1 : 0, row_node, pool,
                                  X, d0);
}

// Rows (+e_j, -e_j) for every unstable (l < 0 < u) unsplit neuron of a layer,
// ascending j within a node.  One CTA per node (its rows lie together), bound by the
// latency of its loads: a thread has COLLECT_U neurons in flight, 32 consecutive ones
// per warp, and a tile's segments of 32 are numbered by one scan.  One node of 32768
// neurons took 65 us with 256 threads and two barriers for each 256 neurons, now 15.6.
constexpr int COLLECT_T = 1024, COLLECT_U = 8;
__global__ void __launch_bounds__(COLLECT_T) k_collect_rows(const int* nodes, PoolDev pool, int off,
                                                            int d, int* counter, int* row_node,
                                                            int* row_j, float* row_sign) {
  constexpr int NW = COLLECT_T / 32, SEG = NW * COLLECT_U;  // segments of a tile
  const int n = nodes[blockIdx.x];
  const size_t base = (size_t)n * pool.SD + off;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ int s_seg[SEG], s_cnt[NW], s_start, s_run;
  // bit u: neuron j0 + 32 (NW u + w) + lane gets rows
  auto flags = [&](int j0) {
    float l[COLLECT_U], u[COLLECT_U];
    int sp[COLLECT_U];
#pragma unroll
    for (int v = 0; v < COLLECT_U; ++v) {
      const size_t q = base + min(j0 + 32 * (NW * v + w) + lane, d - 1);
      l[v] = pool.L[q];
      u[v] = pool.U[q];
      sp[v] = pool.S[q];
    }
    unsigned f = 0;
#pragma unroll
    for (int v = 0; v < COLLECT_U; ++v)
      if (j0 + 32 * (NW * v + w) + lane < d && l[v] < 0.f && u[v] > 0.f && sp[v] == 0) f |= 1u << v;
    return f;
  };
  int cnt = 0;
  for (int j0 = 0; j0 < d; j0 += COLLECT_T * COLLECT_U) cnt += __popc(flags(j0));
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) s_cnt[w] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int i = 0; i < NW; ++i) tot += s_cnt[i];
    s_start = atomicAdd(counter, 2 * tot);
    s_run = 0;
  }
  for (int j0 = 0; j0 < d; j0 += COLLECT_T * COLLECT_U) {
    const unsigned f = flags(j0);
    unsigned bal[COLLECT_U];
#pragma unroll
    for (int v = 0; v < COLLECT_U; ++v) {
      bal[v] = __ballot_sync(0xffffffffu, f >> v & 1u);
      if (lane == 0) s_seg[NW * v + w] = __popc(bal[v]);
    }
    __syncthreads();
    if (w == 0) {  // exclusive scan of the segments, 8 per lane
      constexpr int PL = SEG / 32;
      int c[PL], sum = 0;
#pragma unroll
      for (int i = 0; i < PL; ++i) {
        c[i] = s_seg[lane * PL + i];
        sum += c[i];
      }
      int inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
      }
      int run = s_run + inc - sum;
      __syncwarp();
#pragma unroll
      for (int i = 0; i < PL; ++i) {
        s_seg[lane * PL + i] = run;
        run += c[i];
      }
      if (lane == 31) s_run = run;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < COLLECT_U; ++v)
      if (f >> v & 1u) {
        const int j = j0 + 32 * (NW * v + w) + lane;
        const int r = s_start + 2 * (s_seg[NW * v + w] + __popc(bal[v] & ((1u << lane) - 1u)));
        row_node[r] = n; row_j[r] = j; row_sign[r] = 1.f;
        row_node[r + 1] = n; row_j[r + 1] = j; row_sign[r + 1] = -1.f;
      }
    __syncthreads();
  }
}

void launch_collect_rows(int nb, const int* nodes, PoolDev pool, int off, int d, int* counter,
                         int* row_node, int* row_j, float* row_sign, cudaStream_t st) {
  if (nb <= 0) return;
  k_collect_rows<<<nb, COLLECT_T, 0, st>>>(nodes, pool, off, d, counter, row_node, row_j, row_sign);
}

__global__ void k_update_bounds(int npairs, const int* row_node, const int* row_j,
                                const float* lb, PoolDev pool, int off) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= npairs) return;
  const int n = row_node[2 * q], j = row_j[2 * q];
  const size_t i = (size_t)n * pool.SD + off + j;
  pool.L[i] = fmaxf(pool.L[i], lb[2 * q]);
  pool.U[i] = fminf(pool.U[i], -lb[2 * q + 1]);
}

void launch_update_bounds(int npairs, const int* row_node, const int* row_j, const float* lb,
                          PoolDev pool, int off, cudaStream_t st) {
  if (npairs <= 0) return;
  k_update_bounds<<<(npairs + 255) / 256, 256, 0, st>>>(npairs, row_node, row_j, lb, pool, off);
}

__device__ __forceinline__ int layer_of(const NetDev& net, int f) {
  int i = 1;
  while (i < net.R && f >= net.off[i + 1]) ++i;
  return i;
}

// gamma^T P and gamma^T Phat per neuron (CSR by neuron), and gamma^T p per row.
// A CTA serves RB consecutive rows.  The CTAs of such a group: RB x GP_SPLIT that sum
// a share of one row's gamma^T p each (k_reduce_lb adds the shares in a tree: another
// order than that of one CTA for the row, about 5e-8 of the sum apart), RB x `nzero`
// that write the zeros of neurons without entries, and the others, which take eight
// of the layers' listed neurons (those with entries) at a time: each warp brings
// one neuron's entries to shared memory, all loads in flight (a neuron in three
// groups of 150 rows has 450), then two lanes per neuron and row sum them, gamma^T P
// and gamma^T Phat, in entry order.  Rows of one property share the entries: an
// entry's index and two coefficients are loaded once for the RB rows (of a group
// of different properties, a CTA takes one row).  Bound by the latency of those
// loads and the chain of FMAs.  64 rows of the 3x32x32 network with 135k constraint
// rows: 113 us with one row per CTA, 70 with four; 9 rows of the 784-100-100-10 one
// 7.4 with one (their CTAs would not fill the SMs in groups).  20 steps of 64 such
// rows, with the gradients' kernel below: 13.4 and 11.8 ms; 14.0 where two properties
// alternate row by row, the order that groups gain nothing from.
constexpr int GP_THREADS = 256;
constexpr int GP_GROUP = 4;        // rows of a group
constexpr int GP_GROUP_MIN = 32;   // rows from which on they are grouped

// The sums of `rows` rows (at most R; all of one property) from row m on: CTA b of nb
// takes listed neurons NW b .., NW nb further on.  s_ent: a warp's staged entries (P,
// Phat, the rows' gamma; CHUNK + 4 floats each).
template <int R, int CHUNK>
__device__ __forceinline__ void gamma_proj_rows(int m, int rows, int b, int nb,
                                                const int* __restrict__ row_node,
                                                const PoolDev& pool,
                                                const PropDev* __restrict__ props,
                                                const NetDev& net, float* s_ent, int* s_len,
                                                int* s_f, float* __restrict__ GP,
                                                float* __restrict__ GPh) {
  constexpr int NW = GP_THREADS / 32, LD = CHUNK + 4, WS = (2 + R) * LD;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PropDev& P = props[pool.prop[row_node[m]]];
  const float* gam[R];
#pragma unroll
  for (int r = 0; r < R; ++r)
    gam[r] = pool.GAM + (size_t)row_node[m + (r < rows ? r : 0)] * pool.EC;
  float* own = s_ent + warp * WS;
  int total = 0;
  for (int i = 1; i <= net.R; ++i) total += P.mnc[i].n_act;
  for (int a0 = b * NW; a0 < total; a0 += nb * NW) {
    // this warp's neuron and its entries
    int q0 = 0, len = 0, goff = 0;
    const int *ce_ = nullptr;
    const float *cP_ = nullptr, *cPh_ = nullptr;
    if (a0 + warp < total) {
      int i = 1, a = a0 + warp;
      while (a >= P.mnc[i].n_act) a -= P.mnc[i++].n_act;
      const MncDev& mc = P.mnc[i];
      const int j = mc.act[a];
      q0 = mc.cptr[j];
      len = mc.cptr[j + 1] - q0;
      ce_ = mc.ce + q0;
      cP_ = mc.cP + q0;
      cPh_ = mc.cPh + q0;
      goff = mc.goff;
      if (lane == 0) s_f[warp] = net.off[i] + j;
    }
    if (lane == 0) s_len[warp] = len;
    __syncthreads();
    int most = 0;
    for (int w = 0; w < NW; ++w) most = max(most, s_len[w]);
    // lanes of the sums: row, P or Phat, neuron
    const int row = threadIdx.x % R, which = threadIdx.x / R & 1;
    const int mine = threadIdx.x / (2 * R) % NW;
    float acc = 0.f;
    for (int c0 = 0; c0 < most; c0 += CHUNK) {
      int ce[CHUNK / 32];
      float cp[CHUNK / 32], cph[CHUNK / 32];
#pragma unroll
      for (int v = 0; v < CHUNK / 32; ++v) {
        const int k = c0 + 32 * v + lane;
        ce[v] = k < len ? ce_[k] : -1;
        cp[v] = k < len ? cP_[k] : 0.f;
        cph[v] = k < len ? cPh_[k] : 0.f;
      }
#pragma unroll
      for (int v = 0; v < CHUNK / 32; ++v) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          own[(2 + r) * LD + 32 * v + lane] =
              ce[v] >= 0 && (R == 1 || r < rows) ? gam[r][goff + ce[v]] : 0.f;
        own[32 * v + lane] = cp[v];
        own[LD + 32 * v + lane] = cph[v];
      }
      __syncthreads();
      if (threadIdx.x < 2 * R * NW) {
        const float* eg = s_ent + mine * WS + (2 + row) * LD;
        const float* ec = s_ent + mine * WS + which * LD;
        const int num = min(CHUNK, s_len[mine] - c0);
        int k = 0;
        for (; k + 8 <= num; k += 8) {
          const float4 x0 = *reinterpret_cast<const float4*>(eg + k);
          const float4 x1 = *reinterpret_cast<const float4*>(eg + k + 4);
          const float4 y0 = *reinterpret_cast<const float4*>(ec + k);
          const float4 y1 = *reinterpret_cast<const float4*>(ec + k + 4);
          acc = fmaf(x0.x, y0.x, acc);
          acc = fmaf(x0.y, y0.y, acc);
          acc = fmaf(x0.z, y0.z, acc);
          acc = fmaf(x0.w, y0.w, acc);
          acc = fmaf(x1.x, y1.x, acc);
          acc = fmaf(x1.y, y1.y, acc);
          acc = fmaf(x1.z, y1.z, acc);
          acc = fmaf(x1.w, y1.w, acc);
        }
        for (; k < num; ++k) acc = fmaf(eg[k], ec[k], acc);
      }
      __syncthreads();
    }
    if (threadIdx.x < 2 * R * NW && a0 + mine < total && row < rows)
      (which ? GPh : GP)[(size_t)(m + row) * net.SD + s_f[mine]] = acc;
    __syncthreads();
  }
}

template <int RB>
__global__ void __launch_bounds__(GP_THREADS, 4) k_gamma_proj(
    int M, const int* __restrict__ row_node, PoolDev pool, const PropDev* __restrict__ props,
    NetDev net, int nzero, float* __restrict__ GP, float* __restrict__ GPh,
    float* __restrict__ gp0) {
  const int mg = blockIdx.y * RB;
  if (blockIdx.x < GP_SPLIT * RB) {
    const int m = mg + blockIdx.x / GP_SPLIT, share = blockIdx.x % GP_SPLIT;
    if (m >= M) return;
    const int n = row_node[m];
    const PropDev& P = props[pool.prop[n]];
    const float* gam = pool.GAM + (size_t)n * pool.EC;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    constexpr int step = GP_THREADS * GP_SPLIT;
    for (int i = 1; i <= net.R; ++i) {
      const MncDev& mc = P.mnc[i];
      const float* g = gam + mc.goff;
      const float* pv = mc.p;
      const int e1 = mc.e;
      for (int e = share * GP_THREADS + threadIdx.x; e < e1; e += 4 * step) {
        float gv[4], p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = e + u * step < e1;
          gv[u] = in ? g[e + u * step] : 0.f;
          p[u] = in ? pv[e + u * step] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = fmaf(gv[u], p[u], acc[u]);
      }
    }
    const float tot = block_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
    if (threadIdx.x == 0) gp0[(size_t)m * GP_SPLIT + share] = tot;
    return;
  }
  if (blockIdx.x < (GP_SPLIT + nzero) * RB) {
    const int z = blockIdx.x - GP_SPLIT * RB, m = mg + z / nzero;
    if (m >= M) return;
    const PropDev& P = props[pool.prop[row_node[m]]];
    for (int f = z % nzero * GP_THREADS + threadIdx.x; f < net.SD; f += nzero * GP_THREADS) {
      const int i = layer_of(net, f), j = f - net.off[i];
      const int* cptr = P.mnc[i].e > 0 ? P.mnc[i].cptr : nullptr;
      if (!cptr || cptr[j + 1] == cptr[j]) {
        GP[(size_t)m * net.SD + f] = 0.f;
        GPh[(size_t)m * net.SD + f] = 0.f;
      }
    }
    return;
  }
  // (RB = 4: rows of different properties get longer chunks in the same space)
  constexpr int NW = GP_THREADS / 32, C1 = RB == 1 ? 480 : 448, CG = 224;
  constexpr int W1 = 3 * (C1 + 4), WG = RB == 1 ? 0 : (2 + RB) * (CG + 4);
  __shared__ __align__(16) float s_ent[NW * (W1 > WG ? W1 : WG)];
  __shared__ int s_len[NW], s_f[NW];
  const int nother = (GP_SPLIT + nzero) * RB;
  const int nb = gridDim.x - nother, b = blockIdx.x - nother;
  const int nr = min(RB, M - mg);
  if (RB > 1) {
    bool same = true;
    const int prop0 = pool.prop[row_node[mg]];
    for (int r = 1; r < nr; ++r) same = same && pool.prop[row_node[mg + r]] == prop0;
    if (same) {
      gamma_proj_rows<RB, CG>(mg, nr, b, nb, row_node, pool, props, net, s_ent, s_len, s_f, GP, GPh);
      return;
    }
  }
  const int r = b % nr;  // (nb >= RB)
  gamma_proj_rows<1, C1>(mg + r, 1, b / nr, (nb - r + nr - 1) / nr, row_node, pool, props, net,
                         s_ent, s_len, s_f, GP, GPh);
}

void launch_gamma_proj(int M, const int* row_node, PoolDev pool, const PropDev* props,
                       const NetDev& net, float* GP, float* GPh, float* gp0, cudaStream_t st) {
  if (M <= 0) return;
  const int per = GP_THREADS / 32;
  const int nact = std::min(128, (net.SD + per - 1) / per);
  const int nzero = (net.SD + 4 * GP_THREADS - 1) / (4 * GP_THREADS);
  auto go = [&](auto kern, int rb) {
    dim3 grid((GP_SPLIT + nzero) * rb + std::max(nact, rb), (M + rb - 1) / rb);
    kern<<<grid, GP_THREADS, 0, st>>>(M, row_node, pool, props, net, nzero, GP, GPh, gp0);
  };
  if (M >= GP_GROUP_MIN) go(k_gamma_proj<GP_GROUP>, GP_GROUP);
  else go(k_gamma_proj<1>, 1);
}

// d lb / d gamma_e = sum_k P_ek (d lb / d a')_idx + Phat_ek (d lb / d ahat)_idx - p_e.
// A CTA serves RB consecutive rows; rows of one property share a constraint row's
// neurons and coefficients (28 bytes of 52 per row, at three neurons), which were
// two thirds of the time at one row per CTA.  64 rows, 135k constraint rows: 63 us,
// 32 in groups of four.
constexpr int GAMMA_NPT = 4;
template <int RB>
__global__ void __launch_bounds__(256) k_gamma_grad(
    int M, const int* __restrict__ row_node, PoolDev pool, const PropDev* __restrict__ props,
    NetDev net, const float* __restrict__ Gz, const float* __restrict__ Hz, float* __restrict__ GG) {
  constexpr int NPT = GAMMA_NPT / (RB == 1 ? 1 : 2);  // constraint rows per thread
  const int mg = blockIdx.y * RB, nr = min(RB, M - mg);
  __shared__ const PropDev* s_P[RB];
  __shared__ int s_goff[RB][MNBAB_MAXR + 1], s_e[RB][MNBAB_MAXR + 1];
  if (threadIdx.x < RB)
    s_P[threadIdx.x] = props + pool.prop[row_node[mg + min((int)threadIdx.x, nr - 1)]];
  __syncthreads();
  for (int q = threadIdx.x; q < RB * (net.R + 1); q += blockDim.x) {
    const int r = q / (net.R + 1), t = q % (net.R + 1);
    s_goff[r][t] = t >= 1 ? s_P[r]->mnc[t].goff : 0;
    s_e[r][t] = t >= 1 ? s_P[r]->mnc[t].e : 0;
  }
  __syncthreads();
  bool same = true;
#pragma unroll
  for (int r = 1; r < RB; ++r) same = same && s_P[r] == s_P[0];
  const int e0 = blockIdx.x * (blockDim.x * NPT) + threadIdx.x;
  // the gradients at constraint row ef of `rows` rows (at most R) from row r0 of the group on
  auto grad = [&](int r0, int rows, int ef, auto rc) {
    constexpr int R = decltype(rc)::value;
    const PropDev& P = *s_P[r0];
    if (ef >= P.E) return;
    int i = 0;
    for (int t = 1; t <= net.R; ++t)
      if (s_e[r0][t] > 0 && ef >= s_goff[r0][t] && ef < s_goff[r0][t] + s_e[r0][t]) i = t;
    if (i == 0) return;
    const MncDev& mc = P.mnc[i];
    const int e = ef - s_goff[r0][i];
    const size_t z0 = (size_t)(mg + r0) * net.SD + net.off[i];
    const int k = mc.k;
    const float p = mc.p[e];
    if (k == 3) {
      int j[3];
      float pc[3], hc[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        j[q] = mc.idx[(size_t)e * 3 + q];
        pc[q] = mc.P[(size_t)e * 3 + q];
        hc[q] = mc.Ph[(size_t)e * 3 + q];
      }
      float z[R][3], y[R][3];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const size_t o = z0 + (size_t)(r < rows ? r : 0) * net.SD;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          z[r][q] = Gz[o + j[q]];
          y[r][q] = Hz[o + j[q]];
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float g = -p;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          g = fmaf(pc[q], z[r][q], g);
          g = fmaf(hc[q], y[r][q], g);
        }
        if (r < rows) GG[(size_t)(mg + r0 + r) * pool.EC + ef] = g;
      }
    } else {
      for (int r = 0; r < rows; ++r) {
        const size_t o = z0 + (size_t)r * net.SD;
        float g = -p;
        for (int kk = 0; kk < k; ++kk) {
          const int j = mc.idx[(size_t)e * k + kk];
          g = fmaf(mc.P[(size_t)e * k + kk], Gz[o + j], g);
          g = fmaf(mc.Ph[(size_t)e * k + kk], Hz[o + j], g);
        }
        GG[(size_t)(mg + r0 + r) * pool.EC + ef] = g;
      }
    }
  };
  if (RB > 1 && same) {
#pragma unroll
    for (int u = 0; u < NPT; ++u)
      grad(0, nr, e0 + u * blockDim.x, std::integral_constant<int, RB>{});
    return;
  }
  // (gridDim.x >= RB)
  const int r = blockIdx.x % nr, nb = ((int)gridDim.x - r + nr - 1) / nr;
  const int E = s_P[r]->E, tile = blockDim.x * GAMMA_NPT;
  for (int t0 = (int)blockIdx.x / nr * tile + (int)threadIdx.x; t0 < E; t0 += nb * tile)
#pragma unroll
    for (int u = 0; u < GAMMA_NPT; ++u)
      grad(r, 1, t0 + u * blockDim.x, std::integral_constant<int, 1>{});
}

void launch_gamma_grad(int M, const int* row_node, PoolDev pool, const PropDev* props,
                       const NetDev& net, const float* Gz, const float* Hz, float* GG,
                       cudaStream_t st) {
  if (M <= 0 || pool.EC <= 0) return;
  auto go = [&](auto kern, int rb, int npt) {
    dim3 grid(std::max((pool.EC + 256 * npt - 1) / (256 * npt), rb), (M + rb - 1) / rb);
    kern<<<grid, 256, 0, st>>>(M, row_node, pool, props, net, Gz, Hz, GG);
  };
  if (M >= GP_GROUP_MIN) go(k_gamma_grad<GP_GROUP>, GP_GROUP, GAMMA_NPT / 2);
  else go(k_gamma_grad<1>, 1, GAMMA_NPT);
}

// Projected Adam ascent step (Sec. 3.1): alpha in [0, 1], beta, gamma >= 0.
__device__ __forceinline__ void adam1(float& th, float& mo, float& ve, float g, float lr, float b1,
                                      float b2, float eps, float bc1, float bc2) {
  mo = b1 * mo + (1.f - b1) * g;
  ve = b2 * ve + (1.f - b2) * g * g;
  const float mh = mo / bc1;
  const float vh = ve / bc2;
  th = th + lr * mh / (sqrtf(vh) + eps);
}

// largest |gradient component| of each row over alpha, beta and gamma: CTA s of
// a row covers elements s, s + gridDim.x, ... of 4 * 256-element tiles and writes
// gmax[m][s].  One CTA per row read the 260k components of the 3x32x32 network
// with 135k constraint rows at 0.2 TB/s (362 us for 64 rows).
__global__ void __launch_bounds__(256) k_grad_max(int SD, int EC, const int* row_node,
                                                  const PoolDev pool, const PropDev* props,
                                                  const float* GA, const float* GB,
                                                  const float* GG, float* gmax) {
  const int m = blockIdx.y;
  const int E = props[pool.prop[row_node[m]]].E;
  const float* src[3] = {GA + (size_t)m * SD, GB + (size_t)m * SD, GG + (size_t)m * EC};
  const int len[3] = {SD, SD, E};
  float mx = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    for (int i = blockIdx.x * 1024 + threadIdx.x; i < len[k]; i += gridDim.x * 1024) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = i + 256 * u < len[k] ? src[k][i + 256 * u] : 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) mx = fmaxf(mx, fabsf(v[u]));
    }
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  __shared__ float sh[8];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float r = sh[0];
    for (int i = 1; i < 8; ++i) r = fmaxf(r, sh[i]);
    gmax[(size_t)m * GMAX_SPLIT + blockIdx.x] = r;
  }
}

// The alpha of a neuron that is not unstable and unsplit, and the beta of an
// unsplit one, have a zero gradient at every step of an optimisation (its
// bounds and splits are fixed), and their moments start at zero: their
// updates are identities and are skipped.  A thread takes one neuron (its alpha
// or its beta, by its split) or one multi-neuron multiplier.  gmax (nsplit
// shares a row) is read only when the dead-zone or the gradient-scaled eps is on.
__global__ void __launch_bounds__(256) k_adam(
    int M, const int* __restrict__ row_node, PoolDev pool, const PropDev* __restrict__ props,
    int SD, const float* __restrict__ GA, const float* __restrict__ GB,
    const float* __restrict__ GG, const float* __restrict__ gmax, int nsplit, float floor,
    float lr_a, float lr_b, float lr_g, float b1, float b2, float eps_abs, float eps_rel,
    float bc1, float bc2) {
  const int m = blockIdx.y;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = row_node[m];
  float gm = 0.f;
  if (nsplit) {
    const int lane = threadIdx.x & 31;
    if (lane < nsplit) gm = gmax[(size_t)m * GMAX_SPLIT + lane];
    for (int o = 16; o; o >>= 1) gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  }
  const float thr = floor * gm;
  const float eps = fmaxf(eps_abs, eps_rel * gm);
  auto dz = [thr](float g) { return fabsf(g) <= thr ? 0.f : g; };
  if (idx < SD) {
    const size_t q = (size_t)n * SD + idx;
    if (pool.S[q] == 0) {
      if (!(pool.L[q] < 0.f) || !(pool.U[q] > 0.f)) return;
      float th = pool.ALPHA[q], mo = pool.MA[q], ve = pool.VA[q];
      adam1(th, mo, ve, dz(GA[(size_t)m * SD + idx]), lr_a, b1, b2, eps, bc1, bc2);
      pool.ALPHA[q] = fminf(fmaxf(th, 0.f), 1.f);
      pool.MA[q] = mo; pool.VA[q] = ve;
    } else {
      float th = pool.BETA[q], mo = pool.MB[q], ve = pool.VB[q];
      adam1(th, mo, ve, dz(GB[(size_t)m * SD + idx]), lr_b, b1, b2, eps, bc1, bc2);
      pool.BETA[q] = fmaxf(th, 0.f);
      pool.MB[q] = mo; pool.VB[q] = ve;
    }
  } else {
    const int e = idx - SD;
    if (e >= props[pool.prop[n]].E) return;
    const size_t q = (size_t)n * pool.EC + e;
    float th = pool.GAM[q], mo = pool.MG[q], ve = pool.VG[q];
    adam1(th, mo, ve, dz(GG[(size_t)m * pool.EC + e]), lr_g, b1, b2, eps, bc1, bc2);
    pool.GAM[q] = fmaxf(th, 0.f);
    pool.MG[q] = mo; pool.VG[q] = ve;
  }
}

void launch_adam(int M, const int* row_node, PoolDev pool, const PropDev* props, int SD,
                 const float* GA, const float* GB, const float* GG, float* gmax, float floor,
                 float lr_a, float lr_b, float lr_g, float b1, float b2, float eps, float eps_rel,
                 float bc1, float bc2, cudaStream_t st) {
  if (M <= 0) return;
  int nsplit = 0;
  if (floor != 0.f || eps_rel != 0.f) {
    nsplit = std::min(GMAX_SPLIT, (std::max(SD, pool.EC) + 1023) / 1024);
    k_grad_max<<<dim3(nsplit, M), 256, 0, st>>>(SD, pool.EC, row_node, pool, props, GA, GB, GG,
                                                gmax);
  }
  const int tot = SD + pool.EC;
  dim3 grid((tot + 255) / 256, M);
  k_adam<<<grid, 256, 0, st>>>(M, row_node, pool, props, SD, GA, GB, GG, gmax, nsplit, floor,
                               lr_a, lr_b, lr_g, b1, b2, eps, eps_rel, bc1, bc2);
}

__global__ void k_zero_adam(const int* row_node, PoolDev pool) {
  const int n = row_node[blockIdx.y];
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < pool.SD) {
    const size_t q = (size_t)n * pool.SD + idx;
    pool.MA[q] = 0.f; pool.VA[q] = 0.f; pool.MB[q] = 0.f; pool.VB[q] = 0.f;
  } else if (idx < pool.SD + pool.EC) {
    const size_t q = (size_t)n * pool.EC + idx - pool.SD;
    pool.MG[q] = 0.f; pool.VG[q] = 0.f;
  }
}

void launch_zero_adam(int M, const int* row_node, PoolDev pool, cudaStream_t st) {
  if (M <= 0) return;
  dim3 grid((pool.SD + pool.EC + 255) / 256, M);
  k_zero_adam<<<grid, 256, 0, st>>>(row_node, pool);
}

__global__ void k_set_best(int M, const int* row_node, PoolDev pool, float v) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < M) pool.BEST[row_node[m]] = v;
}

void launch_set_best(int M, const int* row_node, PoolDev pool, float v, cudaStream_t st) {
  if (M <= 0) return;
  k_set_best<<<(M + 255) / 256, 256, 0, st>>>(M, row_node, pool, v);
}

// ACS (Sec. 3.2) with the intercept fallback; with CAB the score is divided by
// the cost of a split in the neuron's layer (the fallback decision is taken on
// the raw scores).  Ties within 1e-5 of the maximum go to the lowest
// (layer, neuron).
__global__ void k_acs(int M, const int* row_node, PoolDev pool, const PropDev* props, NetDev net,
                      const float* GP, const float* GPh, const float* AP, int has_gamma,
                      int* out_layer, int* out_neuron, float* out_score, int* out_fallback) {
  const int m = blockIdx.x;
  const int n = row_node[m];
  const PropDev& P = props[pool.prop[n]];
  const size_t nb = (size_t)n * pool.SD, mb = (size_t)m * net.SD;
  __shared__ float smax[32];
  __shared__ int sany[32];
  __shared__ int smin[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto bmax = [&](float v) {
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) smax[w] = v;
    __syncthreads();
    float r = -INFINITY;
    for (int i = 0; i < nw; ++i) r = fmaxf(r, smax[i]);
    return r;
  };
  // candidates and whether any active-constraint score is positive
  float raw = -INFINITY;
  int any = 0;
  for (int f = threadIdx.x; f < net.SD; f += blockDim.x) {
    const float l = pool.L[nb + f], u = pool.U[nb + f];
    if (l < 0.f && u > 0.f && pool.S[nb + f] == 0) {
      any = 1;
      const float sc = has_gamma ? fabsf(GP[mb + f]) + fabsf(GPh[mb + f]) : 0.f;
      raw = fmaxf(raw, sc);
    }
  }
  raw = bmax(raw);
  for (int o = 16; o; o >>= 1) any |= __shfl_xor_sync(0xffffffffu, any, o);
  if (lane == 0) sany[w] = any;
  __syncthreads();
  any = 0;
  for (int i = 0; i < nw; ++i) any |= sany[i];
  if (!any) {
    if (threadIdx.x == 0) {
      out_layer[m] = 0; out_neuron[m] = -1; out_score[m] = 0.f; out_fallback[m] = 0;
    }
    return;
  }
  const int fallback = !(raw > 0.f);
  auto score = [&](int f, float l, float u) {
    float sc = fallback ? fabsf(AP[mb + f]) * ((-l * u) / (u - l))
                        : fabsf(GP[mb + f]) + fabsf(GPh[mb + f]);
    if (P.cab) sc *= P.cab_inv[layer_of(net, f)];
    return sc;
  };
  float mx = -INFINITY;
  for (int f = threadIdx.x; f < net.SD; f += blockDim.x) {
    const float l = pool.L[nb + f], u = pool.U[nb + f];
    if (l < 0.f && u > 0.f && pool.S[nb + f] == 0) mx = fmaxf(mx, score(f, l, u));
  }
  mx = bmax(mx);
  const float thr = mx - 1e-5f * fabsf(mx);
  int best = 0x7fffffff;
  for (int f = threadIdx.x; f < net.SD; f += blockDim.x) {
    const float l = pool.L[nb + f], u = pool.U[nb + f];
    if (l < 0.f && u > 0.f && pool.S[nb + f] == 0 && score(f, l, u) >= thr && f < best) best = f;
  }
  for (int o = 16; o; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
  __syncthreads();
  if (lane == 0) smin[w] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    int b = 0x7fffffff;
    for (int i = 0; i < nw; ++i) b = min(b, smin[i]);
    const int i = layer_of(net, b);
    out_layer[m] = i;
    out_neuron[m] = b - net.off[i];
    out_score[m] = mx;
    out_fallback[m] = fallback;
  }
}

void launch_acs(int M, const int* row_node, PoolDev pool, const PropDev* props, const NetDev& net,
                const float* GP, const float* GPh, const float* AP, int has_gamma, int* out_layer,
                int* out_neuron, float* out_score, int* out_fallback, cudaStream_t st) {
  if (M <= 0) return;
  k_acs<<<M, 256, 0, st>>>(M, row_node, pool, props, net, GP, GPh, AP, has_gamma, out_layer,
                            out_neuron, out_score, out_fallback);
}

// Children of a split (Sec. 3.2, enforcing splits): copies of the parent with
// S = +1 (zhat <= 0, u <- min(u, 0)) for the first child and S = -1 (zhat >= 0,
// l <- max(l, 0)) for the second; the split neuron's beta starts at 0.
__global__ void k_children(const int* parents, const int* kids, const int* layer,
                           const int* neuron, PoolDev pool, NetDev net) {
  const int b = blockIdx.y;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int par = parents[b];
  const int f_split = net.off[layer[b]] + neuron[b];
  for (int c = 0; c < 2; ++c) {
    const int kid = kids[2 * b + c];
    if (idx < pool.SD) {
      const size_t qs = (size_t)par * pool.SD + idx, qd = (size_t)kid * pool.SD + idx;
      float l = pool.L[qs], u = pool.U[qs];
      int8_t s = pool.S[qs];
      float be = pool.BETA[qs];
      if (idx == f_split) {
        be = 0.f;
        if (c == 0) { s = 1; u = fminf(u, 0.f); }
        else { s = -1; l = fmaxf(l, 0.f); }
      }
      pool.L[qd] = l; pool.U[qd] = u; pool.S[qd] = s;
      pool.ALPHA[qd] = pool.ALPHA[qs];
      pool.BETA[qd] = be;
    } else if (idx < pool.SD + pool.EC) {
      const int e = idx - pool.SD;
      pool.GAM[(size_t)kid * pool.EC + e] = pool.GAM[(size_t)par * pool.EC + e];
    }
    if (idx == 0) {
      pool.prop[kid] = pool.prop[par];
      pool.row[kid] = pool.row[par];
    }
  }
}

void launch_children(int nb, const int* parents, const int* kids, const int* layer,
                     const int* neuron, PoolDev pool, const NetDev& net, cudaStream_t st) {
  if (nb <= 0) return;
  dim3 grid((pool.SD + pool.EC + 255) / 256, nb);
  k_children<<<grid, 256, 0, st>>>(parents, kids, layer, neuron, pool, net);
}

// ---------------------------------------------------------------------------
// Optimised intermediate bounds (Sec. 3.1, parameter sharing): the parameter
// set of one (node, target layer, side) lives in a scratch pool slot.
// ---------------------------------------------------------------------------
// Set slot dst[b] from node src[b]: bounds and splits, DeepPoly slopes
// (alpha = 1 if u >= -l else 0), beta = 0, gamma = 0, zero Adam moments.
__global__ void k_set_init(const int* src, const int* dst, PoolDev pool) {
  const int b = blockIdx.y;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = src[b], d = dst[b];
  if (i < pool.SD) {
    const size_t qs = (size_t)s * pool.SD + i, qd = (size_t)d * pool.SD + i;
    const float l = pool.L[qs], u = pool.U[qs];
    pool.L[qd] = l;
    pool.U[qd] = u;
    pool.S[qd] = pool.S[qs];
    pool.ALPHA[qd] = u >= -l ? 1.f : 0.f;
    pool.BETA[qd] = 0.f;
    pool.MA[qd] = 0.f;
    pool.VA[qd] = 0.f;
    pool.MB[qd] = 0.f;
    pool.VB[qd] = 0.f;
  }
  if (i < pool.EC) {
    // multi-neuron multipliers start at 0 with zero moments
    const size_t qd = (size_t)d * pool.EC + i;
    pool.GAM[qd] = 0.f;
    pool.MG[qd] = 0.f;
    pool.VG[qd] = 0.f;
  }
  if (i == 0) {
    pool.prop[d] = pool.prop[s];
    pool.row[d] = pool.row[s];
  }
}

void launch_set_init(int nsets, const int* src, const int* dst, PoolDev pool, cudaStream_t st) {
  if (nsets <= 0) return;
  dim3 grid((std::max(pool.SD, pool.EC) + 255) / 256, nsets);
  k_set_init<<<grid, 256, 0, st>>>(src, dst, pool);
}

// best[m] = lb[m] on the first iterate, max(best[m], lb[m]) after.
__global__ void k_rows_best(int M, const float* lb, float* best, int first) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < M) best[m] = first ? lb[m] : fmaxf(best[m], lb[m]);
}

void launch_rows_best(int M, const float* lb, float* best, int first, cudaStream_t st) {
  if (M <= 0) return;
  k_rows_best<<<(M + 255) / 256, 256, 0, st>>>(M, lb, best, first);
}

// Adds the per-row gradients GA, GB ([row][SD], rows of one chunk) of each
// set's rows to the set's gradients IGA, IGB ([set][SD]), entries k < lim.
// seg holds (set, first row, end row) per block row, rows relative to the
// chunk; the rows of a set are summed in order.
__global__ void k_set_grad(const int* seg, int SD, int lim, const float* GA, const float* GB,
                           float* IGA, float* IGB) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= lim) return;
  const int s = seg[3 * blockIdx.y], r0 = seg[3 * blockIdx.y + 1], r1 = seg[3 * blockIdx.y + 2];
  float ga = 0.f, gb = 0.f;
  for (int m = r0; m < r1; ++m) {
    ga += GA[(size_t)m * SD + k];
    gb += GB[(size_t)m * SD + k];
  }
  IGA[(size_t)s * SD + k] += ga;
  IGB[(size_t)s * SD + k] += gb;
}

void launch_set_grad(int nseg, const int* seg, int SD, int lim, const float* GA, const float* GB,
                     float* IGA, float* IGB, cudaStream_t st) {
  if (nseg <= 0 || lim <= 0) return;
  dim3 grid((lim + 255) / 256, nseg);
  k_set_grad<<<grid, 256, 0, st>>>(seg, SD, lim, GA, GB, IGA, IGB);
}

// Adds the per-row gradients GG ([row][EC]) w.r.t. the multi-neuron
// multipliers of each set's rows to the set's gradient IGG ([set][EC]), rows
// in order; only constraints of ReLU layers below t (the layers the rows pass)
// get a gradient, every other entry stays 0 (those multipliers stay 0).
__global__ void k_set_grad_gamma(const int* seg, const int* set_slot, PoolDev pool,
                                 const PropDev* props, int t, const float* GG, float* IGG) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = seg[3 * blockIdx.y], r0 = seg[3 * blockIdx.y + 1], r1 = seg[3 * blockIdx.y + 2];
  const PropDev& P = props[pool.prop[set_slot[s]]];
  if (e >= P.E) return;
  bool below = false;
  for (int i = 1; i < t && i <= MNBAB_MAXR; ++i)
    if (e >= P.mnc[i].goff && e < P.mnc[i].goff + P.mnc[i].e) below = true;
  if (!below) return;
  float g = 0.f;
  for (int m = r0; m < r1; ++m) g += GG[(size_t)m * pool.EC + e];
  IGG[(size_t)s * pool.EC + e] += g;
}

void launch_set_grad_gamma(int nseg, const int* seg, const int* set_slot, PoolDev pool,
                           const PropDev* props, int t, const float* GG, float* IGG,
                           cudaStream_t st) {
  if (nseg <= 0 || pool.EC <= 0) return;
  dim3 grid((pool.EC + 255) / 256, nseg);
  k_set_grad_gamma<<<grid, 256, 0, st>>>(seg, set_slot, pool, props, t, GG, IGG);
}

// Intersects the bounds of neuron j[m] of the layer at offset off of node
// orig[m] with row m's best bound: sign +1 bounds zhat_j from below, -1 is
// the lower bound of -zhat_j, so -best bounds it from above.
__global__ void k_set_update(int M, const int* orig, const int* j, const float* sign,
                             const float* best, PoolDev pool, int off) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  const size_t q = (size_t)orig[m] * pool.SD + off + j[m];
  if (sign[m] > 0.f) pool.L[q] = fmaxf(pool.L[q], best[m]);
  else pool.U[q] = fminf(pool.U[q], -best[m]);
}

void launch_set_update(int M, const int* orig, const int* j, const float* sign, const float* best,
                       PoolDev pool, int off, cudaStream_t st) {
  if (M <= 0) return;
  k_set_update<<<(M + 255) / 256, 256, 0, st>>>(M, orig, j, sign, best, pool, off);
}

// Root nodes from their property's root-bound slot: DeepPoly slopes
// (alpha = 1 if u >= -l else 0), beta = gamma = 0, no splits.
__global__ void k_root_init(const int* slots, const int* srcs, const int* rows, PoolDev pool) {
  const int dst = slots[blockIdx.y];
  const int src = srcs[blockIdx.y];
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < pool.SD) {
    const size_t qs = (size_t)src * pool.SD + idx, qd = (size_t)dst * pool.SD + idx;
    const float l = pool.L[qs], u = pool.U[qs];
    pool.L[qd] = l; pool.U[qd] = u; pool.S[qd] = 0;
    pool.ALPHA[qd] = (u >= -l) ? 1.f : 0.f;
    pool.BETA[qd] = 0.f;
  } else if (idx < pool.SD + pool.EC) {
    pool.GAM[(size_t)dst * pool.EC + idx - pool.SD] = 0.f;
  }
  if (idx == 0) {
    pool.prop[dst] = pool.prop[src];
    pool.row[dst] = rows[blockIdx.y];
  }
}

void launch_root_init(int nb, const int* slots, const int* srcs, const int* rows, PoolDev pool,
                      cudaStream_t st) {
  if (nb <= 0) return;
  dim3 grid((pool.SD + pool.EC + 255) / 256, nb);
  k_root_init<<<grid, 256, 0, st>>>(slots, srcs, rows, pool);
}

// f_r(z_R) through the property's folded last layer, one warp per row.
__global__ void k_final_dot(int M, const int* row_node, PoolDev pool, const PropDev* props,
                            const float* z, int ld, int dR, float* f) {
  const int m = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (m >= M) return;
  const int n = row_node[m];
  const PropDev& P = props[pool.prop[n]];
  const int r = pool.row[n];
  const float* w = P.Wf + (size_t)r * dR;
  const float* x = z + (size_t)m * ld;
  float acc = 0.f;
  for (int k = lane; k < dR; k += 32) acc = fmaf(w[k], x[k], acc);
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) f[m] = acc + P.bf[r];
}

void launch_final_dot(int M, const int* row_node, PoolDev pool, const PropDev* props,
                      const float* z, int ld, int dR, float* f, cudaStream_t st) {
  if (M <= 0) return;
  k_final_dot<<<(M + 7) / 8, 256, 0, st>>>(M, row_node, pool, props, z, ld, dR, f);
}

// Concrete forward pass f_r(x) in FP64 (one CTA per row), used to confirm
// counterexamples: the sign of f_r at x* decides FALSIFIED (Sec. 2.2), so it is
// evaluated in double precision from the FP32 weights.  The row buffer holds
// x and every ReLU output (layer t at offset d0 + off[t]), so residual edges
// can read any earlier layer.
__device__ double f64_edge(const LayerDev& L, const double* z, int o) {
  if (L.kind == 1) {
    double acc = (double)L.b[o];
    const float* w = L.W + (size_t)o * L.d_in;
    for (int k = 0; k < L.d_in; ++k) acc = fma((double)w[k], z[k], acc);
    return acc;
  }
  const int hw = L.ho * L.wo;
  const int co = o / hw, oh = (o % hw) / L.wo, ow = o % L.wo;
  double acc = (double)L.b[co];
  for (int ci = 0; ci < L.ci; ++ci)
    for (int kh = 0; kh < L.k; ++kh) {
      const int ih = oh * L.s - L.p + kh;
      if (ih < 0 || ih >= L.hi) continue;
      for (int kw = 0; kw < L.k; ++kw) {
        const int iw = ow * L.s - L.p + kw;
        if (iw < 0 || iw >= L.wi) continue;
        acc = fma((double)L.W[(((size_t)co * L.ci + ci) * L.k + kh) * L.k + kw],
                  z[((size_t)ci * L.hi + ih) * L.wi + iw], acc);
      }
    }
  return acc;
}

// FP64 forward pass of counterexample candidates (Sec. 3.1, upper bounding):
// one launch per layer, one thread per (candidate, neuron), then the objective
// row per candidate.
// With dcount set, only the first *dcount of the M rows are live (a count the
// device computed; the grid covers M).
__global__ void k_f64_input(int M, const int* dcount, const float* X, int ldx, double* buf, int ldb,
                            int d0) {
  const int m = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (dcount && m >= *dcount) return;
  if (m < M && k < d0) buf[(size_t)m * ldb + k] = (double)X[(size_t)m * ldx + k];
}

__global__ void k_f64_layer(int M, const int* dcount, NetDev net, int t, double* buf, int ldb) {
  const int m = blockIdx.y;
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M || o >= net.d[t] || (dcount && m >= *dcount)) return;
  double* z = buf + (size_t)m * ldb;
  const int d0 = net.d[0];
  auto seg = [&](int s) { return s == 0 ? z : z + d0 + net.off[s]; };
  double v = f64_edge(net.aff[t], seg(net.src1[t]), o);
  if (net.n_edge[t] > 1) v += f64_edge(net.aff2[t], seg(net.src2[t]), o);
  seg(t)[o] = v > 0.0 ? v : 0.0;
}

__global__ void k_f64_objective(int M, const int* dcount, const int* row_node, PoolDev pool,
                                const PropDev* props, NetDev net, const double* buf, int ldb,
                                double* fout) {
  const int m = blockIdx.x;
  if (dcount && m >= *dcount) return;
  const double* z = buf + (size_t)m * ldb;
  const int n = row_node[m];
  const PropDev& P = props[pool.prop[n]];
  const int r = pool.row[n];
  const int sR = net.src1[net.R + 1];
  const int dR = net.d[sR];
  const double* h = sR == 0 ? z : z + net.d[0] + net.off[sR];
  double acc = 0.0;
  for (int k = threadIdx.x; k < dR; k += blockDim.x) acc = fma((double)P.Wf[(size_t)r * dR + k], h[k], acc);
  __shared__ double sh[32];
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tt = (double)P.bf[r];
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tt += sh[i];
    fout[m] = tt;
  }
}

void launch_forward_f64(int M, const int* row_node, PoolDev pool, const PropDev* props,
                        const NetDev& net, const float* X, int ldx, double* buf, int ldb,
                        double* fout, cudaStream_t st, const int* dcount) {
  if (M <= 0) return;
  k_f64_input<<<dim3((net.d[0] + 255) / 256, M), 256, 0, st>>>(M, dcount, X, ldx, buf, ldb,
                                                                net.d[0]);
  for (int t = 1; t <= net.R; ++t)
    k_f64_layer<<<dim3((net.d[t] + 127) / 128, M), 128, 0, st>>>(M, dcount, net, t, buf, ldb);
  k_f64_objective<<<M, 256, 0, st>>>(M, dcount, row_node, pool, props, net, buf, ldb, fout);
}

// Counterexample candidates of a batch (Sec. 3.1, upper bounding), in batch
// order: rows m < M whose FP32 objective at the node's best minimiser is
// negative and whose best bound is not positive.  One CTA of up to 1024
// threads, a thread per row and rounds of 1024 rows; writes the rows' batch
// indices and slots and their count.
__global__ void __launch_bounds__(1024) k_select_cand(int M, const float* __restrict__ fout,
                                                      const int* __restrict__ slots,
                                                      const float* __restrict__ best,
                                                      int* cand_idx, int* cand_slot, int* count) {
  __shared__ int warp_tot[32];
  __shared__ int base;
  if (threadIdx.x == 0) base = 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int m0 = 0; m0 < M; m0 += blockDim.x) {
    const int m = m0 + threadIdx.x;
    bool c = false;
    if (m < M) c = fout[m] < 0.f && !(best[slots[m]] > 0.f);
    const unsigned bal = __ballot_sync(0xffffffffu, c);
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    int before = base;
    for (int w = 0; w < warp; ++w) before += warp_tot[w];
    before += __popc(bal & ((1u << lane) - 1u));
    if (c) {
      cand_idx[before] = m;
      cand_slot[before] = slots[m];
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 0; w < nw; ++w) base += warp_tot[w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *count = base;
}

void launch_select_cand(int M, const float* fout, const int* slots, const float* best,
                        int* cand_idx, int* cand_slot, int* count, cudaStream_t st) {
  const int thr = std::max(32, std::min(1024, (M + 31) / 32 * 32));
  k_select_cand<<<1, thr, 0, st>>>(M, fout, slots, best, cand_idx, cand_slot, count);
}

__global__ void k_fill(float* p, size_t n, float v) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

// Root-bound slots of newly started properties: l = -inf, u = +inf, no splits,
// and the slot's property index.
__global__ void k_root_slot_init(int nb, const int* slots, const int* prop, PoolDev pool) {
  const int b = blockIdx.x;
  if (b >= nb) return;
  const size_t o = (size_t)slots[b] * pool.SD;
  for (int j = threadIdx.x; j < pool.SD; j += blockDim.x) {
    pool.L[o + j] = -INFINITY;
    pool.U[o + j] = INFINITY;
    pool.S[o + j] = 0;
  }
  if (threadIdx.x == 0) pool.prop[slots[b]] = prop[b];
}

void launch_root_slot_init(int nb, const int* slots, const int* prop, PoolDev pool,
                           cudaStream_t st) {
  if (nb > 0) k_root_slot_init<<<nb, 256, 0, st>>>(nb, slots, prop, pool);
}

void launch_fill(float* p, size_t n, float v, cudaStream_t st) {
  if (n == 0) return;
  k_fill<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, n, v);
}

// ---------------------------------------------------------------------------
// Pre-attack in the per-layer form (Sec. 4, experimental setup): candidate m
// is a scratch node slot whose bounds hold the pre-activations at its point
// (l = u = zhat), so that a DeepPoly back-substitution of the objective row
// through it is the gradient of the margin (ReLU' = 1 where zhat >= 0).
// ---------------------------------------------------------------------------
// Slot m of the chunk: no splits, zero parameters, property `prop`, row
// (q0 + m) / n_starts; its point, start (q0 + m) mod n_starts clipped to the
// box (starts null: left as is); best margin +inf.
__global__ void k_attack_init(int M, int q0, int n_starts, const int* slots, PoolDev pool,
                              int prop, const PropDev* props, const float* starts, float* X,
                              float* best) {
  const int m = blockIdx.y;
  const int slot = slots[m];
  const int q = q0 + m;
  const PropDev& P = props[prop];
  const int lim = max(pool.SD, pool.d0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < lim; i += gridDim.x * blockDim.x) {
    if (i < pool.SD) {
      const size_t o = (size_t)slot * pool.SD + i;
      pool.L[o] = 0.f;
      pool.U[o] = 0.f;
      pool.S[o] = 0;
      pool.ALPHA[o] = 0.f;
      pool.BETA[o] = 0.f;
    }
    if (starts && i < pool.d0)
      X[(size_t)m * pool.d0 + i] =
          fminf(fmaxf(starts[(size_t)(q % n_starts) * pool.d0 + i], P.lo[i]), P.hi[i]);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    pool.prop[slot] = prop;
    pool.row[slot] = q / n_starts;
    if (best) best[m] = INFINITY;
  }
}

void launch_attack_init(int M, int q0, int n_starts, const int* slots, PoolDev pool, int prop,
                        const PropDev* props, const float* starts, float* X, float* best,
                        cudaStream_t st) {
  if (M <= 0) return;
  const int lim = std::max(pool.SD, pool.d0);
  dim3 grid((unsigned)std::min(64, (lim + 255) / 256), (unsigned)M);
  k_attack_init<<<grid, 256, 0, st>>>(M, q0, n_starts, slots, pool, prop, props, starts, X, best);
}

// z [M][d] holds the pre-activations zhat of ReLU layer (offset off): they go
// to the bounds of each row's slot (l = u = zhat) and z becomes max(zhat, 0)
__global__ void k_pattern_relu(int M, const int* slots, PoolDev pool, int off, int d, float* z) {
  const size_t total = (size_t)M * d;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(i / d), j = (int)(i % d);
    const float v = z[i];
    const size_t q = (size_t)slots[m] * pool.SD + off + j;
    pool.L[q] = v;
    pool.U[q] = v;
    z[i] = fmaxf(v, 0.f);
  }
}

void launch_pattern_relu(int M, const int* slots, PoolDev pool, int off, int d, float* z,
                         cudaStream_t st) {
  if (M <= 0 || d <= 0) return;
  const size_t total = (size_t)M * d;
  const int blocks = (int)std::min<size_t>(152 * 8, (total + 255) / 256);
  k_pattern_relu<<<blocks, 256, 0, st>>>(M, slots, pool, off, d, z);
}

// best[m] and its point bx[m] <- f[m] and X[m] when f[m] is smaller (the
// first minimiser is kept on ties; NaN never replaces it)
__global__ void k_attack_best(const float* f, const float* X, int d0, float* best, float* bx) {
  const int m = blockIdx.x;
  const bool better = f[m] < best[m];
  if (better)
    for (int j = threadIdx.x; j < d0; j += blockDim.x) bx[(size_t)m * d0 + j] = X[(size_t)m * d0 + j];
  __syncthreads();
  if (better && threadIdx.x == 0) best[m] = f[m];
}

void launch_attack_best(int M, const float* f, const float* X, int d0, float* best, float* bx,
                        cudaStream_t st) {
  if (M <= 0) return;
  k_attack_best<<<M, 128, 0, st>>>(f, X, d0, best, bx);
}

// x <- clip(x - alpha sign(g), lo, hi), alpha_j = 2.5 (hi_j - lo_j) / (2 steps),
// sign(0) = 0, with g [M][ld] the margin's gradient
__global__ void k_attack_step(int M, const float* g, int ld, float* X, int d0,
                              const PropDev* props, int prop, int steps) {
  const PropDev& P = props[prop];
  const size_t total = (size_t)M * d0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(i / d0), j = (int)(i % d0);
    const float gj = g[(size_t)m * ld + j];
    const float sg = gj > 0.f ? 1.f : (gj < 0.f ? -1.f : 0.f);
    const float alpha = 2.5f * (P.hi[j] - P.lo[j]) / (2.0f * (float)steps);
    X[i] = fminf(fmaxf(X[i] - alpha * sg, P.lo[j]), P.hi[j]);
  }
}

void launch_attack_step(int M, const float* g, int ld, float* X, int d0, const PropDev* props,
                        int prop, int steps, cudaStream_t st) {
  if (M <= 0) return;
  const size_t total = (size_t)M * d0;
  const int blocks = (int)std::min<size_t>(152 * 8, (total + 255) / 256);
  k_attack_step<<<blocks, 256, 0, st>>>(M, g, ld, X, d0, props, prop, steps);
}

}  // namespace mnbab
