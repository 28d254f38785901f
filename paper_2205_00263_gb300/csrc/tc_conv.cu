// Tensor-core (tcgen05) implicit-GEMM convolutions for the back-substitution
// sweeps (Sec. 3.1: the affine step through a convolution is its transposed
// convolution) and the adjoint / forward passes, with 3xTF32 split products
// and the fused epilogues of epilogue.cuh.
//
// Forward (dir 0): out[m, n, oy, ox] = sum over (ci, kh, kw) of
//   in[m, ci, oy s - p + kh, ox s - p + kw] W[n, ci, kh, kw] (+ b[n]).
// Transposed (dir 1), output positions with (y + p) mod s = ry and
// (x + p) mod s = rx (one stride class) take exactly the taps kh = ry + s a,
// kw = rx + s b: out[m, n, y, x] = sum over (o, a, b) of
//   in[m, o, (y + p - kh) / s, (x + p - kw) / s] W[o, n, kh, kw].
// Each class is a dense GEMM: rows = (objective row m, position), columns =
// channels n, reduction (ci, kh, kw) or (o, a, b).
//
// A CTA computes 128 GEMM rows = 4 objective rows x 32 positions of one class
// (warp w owns row m0 + w, lane = position), all N channels:
//  - B (weights) is pre-split into TF32 hi / lo once per layer, arranged per
//    class as [K / 4][N][4] in HBM and staged by TMA (a 3-D tiled tensor map,
//    cp.async.bulk.tensor), which lands it in the canonical no-swizzle K-major
//    layout (core matrices along K N x 16 B apart, along N 128 B apart);
//  - A is the implicit im2col operand and lives in tensor memory (a GEMM row is a
//    TMEM lane): each of the 256 gather threads takes 16 of a K block's 32 reduction
//    values of its position from the coefficient rows (L2), splits them into hi / lo
//    and stores them with tcgen05.st into one of TC_AST stages; block k + 1's loads
//    are in flight meanwhile;
//  - one thread of a control warp streams the weights through a ring of TC_WST
//    stages and issues each block's MMAs (3 of K = 8 per K step: lo.hi + hi.lo +
//    hi.hi, FP32 accumulation in tensor memory, in that order);
//  - the epilogue reads each warp's 32 TMEM lanes (one objective row) with
//    tcgen05.ld, eight channels at a time whose inputs are loaded together, one
//    instantiation per kind of epilogue and rolled: unrolled with a switch on the kind
//    at every output, the CTAs waited for instructions, and loads behind a branch per
//    output followed one another;
//    a row's offset partial is a warp reduction in a fixed order, written to
//    slot (class, position chunk), so it does not depend on the other rows.
// What bounds a CTA now is its chain of accumulating MMAs: about 125 cycles each
// whatever N <= 64 is, twelve to a K block.  Measured, 20 Adam steps: 64 rows of
// conv_big_32's convolutions 10.0 ms at first, 6.6 with the rolled epilogues, 5.4
// now; 128 rows of resnet_32's 10.2, 6.3 and 5.1.  Splitting the chain over two
// accumulators would change the order of the sums; more CTAs per SM do not fit beside
// two of 256 TMEM columns.
// Every wait is bounded; on timeout the kernel sets the device error flag,
// gives its MMAs one more bounded wait, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "epilogue.cuh"
#include "mnbab.h"
#include "mnbab_internal.h"
#include "tc_common.cuh"

namespace mnbab {

struct TcConv {
  bool ok[2] = {false, false};  // dir 0 forward, dir 1 transposed
  int N[2] = {0, 0}, NP[2] = {0, 0}, Kp[2] = {0, 0}, ncls[2] = {0, 0}, nchunk[2] = {0, 0};
  CUtensorMap hi[2], lo[2];
};

namespace {

constexpr int KC = 32;    // reduction values per staged block
constexpr int TROWS = 4;  // objective rows per CTA (one warp each)
constexpr int TC_KMAX = 1024;  // longest reduction (padded to KC) the kernel takes

struct ConvClass {
  int P, K;            // positions and reduction length of the class
  int y0, x0, nx;      // first output row / column of the class, columns of the class
  int ry, rx, na, nb;  // residues and tap counts (transposed)
};

__host__ __device__ inline ConvClass conv_class(const LayerDev& L, int dir, int cls) {
  ConvClass c;
  if (dir == 0) {
    c.P = L.ho * L.wo;
    c.K = L.ci * L.k * L.k;
    c.y0 = c.x0 = 0;
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
  const int ny = c.y0 < L.hi ? (L.hi - c.y0 + s - 1) / s : 0;
  c.nx = c.x0 < L.wi ? (L.wi - c.x0 + s - 1) / s : 0;
  c.na = c.ry < L.k ? (L.k - c.ry + s - 1) / s : 0;
  c.nb = c.rx < L.k ? (L.k - c.rx + s - 1) / s : 0;
  c.P = ny * c.nx;
  c.K = L.co * c.na * c.nb;
  return c;
}

// pre-split weights of one direction: buf_hi / buf_lo [ncls][Kp / 4][NP][4]
__global__ void k_tc_conv_split(LayerDev L, int dir, int Kp, int NP, float* hi, float* lo) {
  const int cls = blockIdx.y;
  const ConvClass c = conv_class(L, dir, cls);
  const int N = dir == 0 ? L.co : L.ci;
  const int total = Kp * NP;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) {
    const int kk = q / NP, n = q % NP;
    float w = 0.f;
    if (n < N && kk < c.K) {
      if (dir == 0) {
        w = L.W[(size_t)n * c.K + kk];  // W [co][ci][kh][kw]: the reduction is contiguous
      } else {
        const int nab = c.na * c.nb;
        const int o = kk / nab, a = (kk / c.nb) % c.na, b = kk % c.nb;
        const int kh = c.ry + L.s * a, kw = c.rx + L.s * b;
        w = L.W[(((size_t)o * L.ci + n) * L.k + kh) * L.k + kw];
      }
    }
    const uint32_t h = tc::to_tf32(w);
    const uint32_t l = tc::to_tf32(w - __uint_as_float(h));
    const size_t o = (((size_t)cls * (Kp / 4) + kk / 4) * NP + n) * 4 + (kk & 3);
    hi[o] = __uint_as_float(h);
    lo[o] = __uint_as_float(l);
  }
}

constexpr int TC_GATHER = 256;   // 8 warps: two threads per GEMM row gather a K block
constexpr int TC_THREADS = 288;  // and a control warp
constexpr int TC_WST = 4;        // weight stages
constexpr int TC_AST = 3;        // A stages in tensor memory, 2 KC columns each
constexpr uint32_t TC_COLS = 256;  // tensor-memory columns of a CTA: D (64) and the A stages

// one instantiation per kind of epilogue (EM); NP: channels padded to 16
template <int EM>
__global__ void __launch_bounds__(TC_THREADS, 2)
    k_conv_tc(const __grid_constant__ CUtensorMap tm_hi, const __grid_constant__ CUtensorMap tm_lo,
              LayerDev L, int dir, int NP, int M, int nchunk, const float* __restrict__ in,
              int ld_in, float* out, int ld_out, Epi e, int* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int B_BYTES = NP * KC * 4;
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* wring = base;  // TC_WST stages of hi and lo weights
  // reduction table of the whole K range, computed once: source offset (channel
  // plane + tap shift) and tap, of which each thread knows which are in range
  int2* t_tab = reinterpret_cast<int2*>(wring + TC_WST * 2 * B_BYTES);
  // A stage written, its MMAs done [TC_AST], weights there [TC_WST]
  __shared__ __align__(8) uint64_t bars[2 * TC_AST + TC_WST];
  __shared__ uint32_t tmem_holder;
  __shared__ int s_fail;
  __shared__ float s_part[2][TROWS];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rq = warp & 3;         // objective row of this warp (TMEM lane quarter)
  const int kh = warp >> 2;        // which half of a K block this warp gathers
  const int cls = blockIdx.x / nchunk, chunk = blockIdx.x % nchunk;
  const ConvClass c = conv_class(L, dir, cls);
  const int m = blockIdx.y * TROWS + rq;
  const int pos = chunk * 32 + lane;
  const bool rowv = m < M;
  const bool pv = rowv && pos < c.P;
  const int N = dir == 0 ? L.co : L.ci;
  const bool has_part = dir == 1 && epi_has_part(e);
  if (chunk * 32 >= c.P) {
    // no position of this class in the chunk: only the row partials (zero)
    if (has_part && warp < 4 && lane == 0 && rowv)
      e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = 0.f;
    return;
  }
  // this thread's position and the source plane of its gather
  const int iy = pv ? pos / c.nx : 0, ix = pv ? pos % c.nx : 0;
  int gy, gx;
  if (dir == 0) {
    gy = iy * L.s - L.p;
    gx = ix * L.s - L.p;
  } else {
    gy = (c.y0 + L.s * iy + L.p - c.ry) / L.s;
    gx = (c.x0 + L.s * ix + L.p - c.rx) / L.s;
  }
  const int Hs = dir == 0 ? L.hi : L.ho, Wsrc = dir == 0 ? L.wi : L.wo;
  const float* src = in + (size_t)(rowv ? m : 0) * ld_in + gy * Wsrc + gx;

  const uint32_t bar0 = tc::smem_u32(bars);
  auto a_full = [&](int i) { return bar0 + 8u * i; };
  auto mma_done = [&](int i) { return bar0 + 8u * (TC_AST + i); };
  auto w_full = [&](int i) { return bar0 + 8u * (2 * TC_AST + i); };
  if (warp == TC_GATHER / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     tc::smem_u32(&tmem_holder)),
                 "r"(TC_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < TC_AST; ++i) {
      tc::mbar_init(a_full(i), TC_GATHER / 32);
      tc::mbar_init(mma_done(i), 1);
    }
    for (int i = 0; i < TC_WST; ++i) tc::mbar_init(w_full(i), 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_holder;
  const uint32_t idesc = tc::idesc_tf32_m128(NP);

  const int nk = (c.K + KC - 1) / KC;
  for (int kidx = tid; kidx < nk * KC; kidx += TC_THREADS) {
    int delta = 0, ta = 31, tb = 31;  // past K: a tap that is never in range
    if (kidx < c.K) {
      int off, dy, dx;
      if (dir == 0) {
        const int kk2 = L.k * L.k;
        off = (kidx / kk2) * L.hi * L.wi;
        dy = (kidx / L.k) % L.k;
        dx = kidx % L.k;
      } else {
        const int nab = c.na * c.nb;
        off = (kidx / nab) * L.ho * L.wo;
        dy = -((kidx / c.nb) % c.na);
        dx = -(kidx % c.nb);
      }
      delta = off + dy * Wsrc + dx;
      ta = abs(dy);
      tb = abs(dx);
    }
    t_tab[kidx] = make_int2(delta, ta | tb << 8);
  }
  // tap rows and columns whose source position lies in the plane, for this
  // thread's position (a class has at most 32 of each: K <= TC_KMAX; all 32 x 32
  // leave no padding past K)
  unsigned vy = 0, vx = 0;
  if (pv) {
    for (int a = 0; a < c.na; ++a) {
      const int yy = dir == 0 ? gy + a : gy - a;
      if (yy >= 0 && yy < Hs) vy |= 1u << a;
    }
    for (int b = 0; b < c.nb; ++b) {
      const int xx = dir == 0 ? gx + b : gx - b;
      if (xx >= 0 && xx < Wsrc) vx |= 1u << b;
    }
  }
  auto in_range = [&](int tap) { return (vy >> (tap & 31)) & (vx >> (tap >> 8)) & 1u; };
  __syncthreads();
  // implicit im2col: the 16 reduction values of this thread's GEMM row in K
  // block kb (half kh of the block)
  auto gather = [&](int kb, float (&v)[16]) {
    const int4* tt = reinterpret_cast<const int4*>(t_tab + kb * KC + kh * 16);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int4 t2 = tt[u];  // two entries: source offset, tap
      v[2 * u] = in_range(t2.y) ? __ldg(src + t2.x) : 0.f;
      v[2 * u + 1] = in_range(t2.w) ? __ldg(src + t2.z) : 0.f;
    }
  };
  bool ok = true;
  if (warp == TC_GATHER / 32) {
    // control: one thread streams the weights through their ring (block kb in
    // stage kb mod TC_WST, refilled when the MMAs that read the stage are done) and
    // issues each block's MMAs once its A tile and weights are there
    if (lane == 0) {
      auto load = [&](int kb) {
        const uint32_t b = w_full(kb % TC_WST);
        const uint32_t d = tc::smem_u32(wring + kb % TC_WST * 2 * B_BYTES);
        tc::mbar_expect_tx(b, 2 * B_BYTES);
        tc::tma_load_3d(d, &tm_hi, 0, kb * (KC / 4), cls, b);
        tc::tma_load_3d(d + B_BYTES, &tm_lo, 0, kb * (KC / 4), cls, b);
      };
      const uint32_t b_lo0 = tc::desc_lo(tc::smem_u32(wring), (uint32_t)NP * 16u);
      const uint32_t b_hi = tc::desc_hi(128);
      int loaded = 0, kb = 0;
      for (; loaded < min(nk, TC_WST); ++loaded) load(loaded);
      for (; kb < nk; ++kb) {
        const int st = kb % TC_AST;
        if (!tc::mbar_wait(a_full(st), (uint32_t)((kb / TC_AST) & 1)) ||
            !tc::mbar_wait(w_full(kb % TC_WST), (uint32_t)((kb / TC_WST) & 1))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ah = tmem + 64u + (uint32_t)st * (2 * KC), al = ah + KC;
        const uint32_t bh = b_lo0 + (uint32_t)(kb % TC_WST) * (uint32_t)(2 * B_BYTES / 16);
        const uint32_t bl = bh + (uint32_t)(B_BYTES / 16), bstep = (uint32_t)NP * 2u;
        if (kb == 0) tc::mma_tf32_tmem_lo<false>(tmem, al, bh, b_hi, idesc);
        else tc::mma_tf32_tmem_lo<true>(tmem, al, bh, b_hi, idesc);
        tc::mma_tf32_tmem_lo<true>(tmem, ah, bl, b_hi, idesc);
        tc::mma_tf32_tmem_lo<true>(tmem, ah, bh, b_hi, idesc);
#pragma unroll
        for (int ks = 1; ks < KC / 8; ++ks) {
          const uint32_t ao = ks * 8, bo = ks * bstep;
          tc::mma_tf32_tmem_lo<true>(tmem, al + ao, bh + bo, b_hi, idesc);
          tc::mma_tf32_tmem_lo<true>(tmem, ah + ao, bl + bo, b_hi, idesc);
          tc::mma_tf32_tmem_lo<true>(tmem, ah + ao, bh + bo, b_hi, idesc);
        }
        tc::mma_commit(mma_done(st));
        if (kb >= 1 && loaded < nk) {
          // the weight stage of block kb - 1 is free once its MMAs are done
          if (!tc::mbar_wait(mma_done((kb - 1) % TC_AST), (uint32_t)(((kb - 1) / TC_AST) & 1))) {
            ok = false;
            break;
          }
          load(loaded++);
        }
      }
      if (!ok) {
        // copies and MMAs in flight get one more bounded wait
        s_fail = 1;
        for (int i = kb; i < loaded; ++i)
          tc::mbar_wait(w_full(i % TC_WST), (uint32_t)((i / TC_WST) & 1));
        for (int i = max(0, kb - 1); i <= kb; ++i)
          tc::mbar_wait(mma_done(i % TC_AST), (uint32_t)((i / TC_AST) & 1));
      }
    }
  } else {
    // gather: block kb + 1's loads are in flight while block kb is split and
    // written to tensor memory (a GEMM row is a lane: no shared memory, no fence
    // between proxies)
    float v[16];
    if (nk > 0) gather(0, v);
    const uint32_t arow = tmem + ((uint32_t)(rq * 32) << 16) + 64u + (uint32_t)(kh * 16);
    for (int kb = 0; kb < nk; ++kb) {
      const int st = kb % TC_AST;
      uint32_t h[16], l[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        h[u] = tc::to_tf32(v[u]);
        l[u] = tc::to_tf32(v[u] - __uint_as_float(h[u]));
      }
      if (kb + 1 < nk) gather(kb + 1, v);
      // the MMAs of block kb - TC_AST read this A stage
      const bool free_ = kb < TC_AST || tc::mbar_wait(mma_done(st), (uint32_t)((kb / TC_AST - 1) & 1));
      if (!__all_sync(0xffffffffu, free_)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tc::tmem_st16(arow + (uint32_t)st * (2 * KC), h);
      tc::tmem_st16(arow + (uint32_t)st * (2 * KC) + KC, l);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(a_full(st));
    }
    // the last commit covers every MMA issued before it
    if (ok && nk > 0)
      ok = tc::mbar_wait(mma_done((nk - 1) % TC_AST), (uint32_t)(((nk - 1) / TC_AST) & 1));
  }
  ok = __syncthreads_and(ok && s_fail == 0) != 0;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!ok) {
    if (tid == 0) atomicExch(err, 1);
  } else if (warp < TC_GATHER / 32) {
    // epilogue: every warp reads its TMEM lane quarter (objective row rq); warp
    // group kh takes the 16-column chunks 16 (2 i + kh), eight columns at a time,
    // whose inputs are loaded together before any of them is finished.
    float part = 0.f;
    const int y = dir == 0 ? iy : c.y0 + L.s * iy;
    const int x = dir == 0 ? ix : c.x0 + L.s * ix;
    const int plane = dir == 0 ? L.ho * L.wo : L.hi * L.wi;
    const int W2 = dir == 0 ? L.wo : L.wi;
    const int pj = y * W2 + x;
    const uint32_t trow = tmem + ((uint32_t)(rq * 32) << 16);
    const int nrow = pv ? e.row_node[m] : 0;
    const PropDev* Pp = pv ? epi_prop(e, nrow) : nullptr;
#pragma unroll 1
    for (int it = 2 * kh; it < NP / 8; it += (it & 1) ? 3 : 1) {
      const int c0 = 8 * it;
      float v[8];
      __syncwarp();
      if (nk > 0) {
        tc::tmem_ld8(trow + (uint32_t)c0, v);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.f;  // a class without taps
      }
      if (pv) {
        EpiIn ein[8];
        int j[8];
        unsigned okm = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          // (a padded channel loads the last one's inputs: loads under a branch per
          // output were issued one output after another, 2000 cycles each)
          const int n = min(c0 + i, N - 1);
          j[i] = n * plane + pj;
          epi_load_m<EM>(e, nrow, Pp, m, j[i], ein[i]);
          if (dir == 0) v[i] += L.b[n];
          if (c0 + i < N) okm |= 1u << i;
        }
        epi_finish_block<EM, 8>(e, m, j, v, ein, okm, part);
        if (out) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (okm >> i & 1u) out[(size_t)m * ld_out + j[i]] = v[i];
        }
      }
    }
    if (has_part) {
      for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lane == 0) s_part[kh][rq] = part;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // a row's offset partial: the two warp groups' sums, in that order
  if (ok && has_part && warp < 4 && lane == 0 && rowv)
    e.part[(size_t)m * e.nslot + e.slot_base + blockIdx.x] = s_part[0][rq] + s_part[1][rq];
  if (warp == TC_GATHER / 32) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_COLS));
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

constexpr int conv_tc_smem(int NP, int Kp) {
  return 1024 + TC_WST * 2 * NP * KC * 4 + Kp * (int)sizeof(int2);
}

}  // namespace

size_t tc_conv_floats(const LayerDev& L) {
  if (L.kind != MNBAB_CONV2D) return 0;
  size_t tot = 0;
  for (int dir = 0; dir < 2; ++dir) {
    const int N = dir == 0 ? L.co : L.ci;
    const int NP = (N + 15) / 16 * 16;
    const int ncls = dir == 0 ? 1 : L.s * L.s;
    int K = 0;
    for (int cl = 0; cl < ncls; ++cl) K = std::max(K, conv_class(L, dir, cl).K);
    const int Kp = std::max(KC, (K + KC - 1) / KC * KC);
    if (N < 8 || NP > 64 || Kp > TC_KMAX) continue;
    tot += 2 * (size_t)ncls * Kp * NP;
  }
  return tot;
}

TcConv* tc_conv_create(const LayerDev& L, float* buf, cudaStream_t st) {
  if (L.kind != MNBAB_CONV2D || !buf) return nullptr;
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return nullptr;
  TcConv* t = new TcConv();
  size_t at = 0;
  for (int dir = 0; dir < 2; ++dir) {
    const int N = dir == 0 ? L.co : L.ci;
    const int NP = (N + 15) / 16 * 16;
    const int ncls = dir == 0 ? 1 : L.s * L.s;
    int K = 0, pmax = 0;
    for (int cl = 0; cl < ncls; ++cl) {
      const ConvClass c = conv_class(L, dir, cl);
      K = std::max(K, c.K);
      pmax = std::max(pmax, c.P);
    }
    const int Kp = std::max(KC, (K + KC - 1) / KC * KC);
    // too few or too many channels for these tiles, or a reduction longer than the table
    if (N < 8 || NP > 64 || Kp > TC_KMAX) continue;
    float* hi = buf + at;
    float* lo = hi + (size_t)ncls * Kp * NP;
    at += 2 * (size_t)ncls * Kp * NP;
    dim3 grid((unsigned)std::min(1024, (Kp * NP + 255) / 256), ncls);
    k_tc_conv_split<<<grid, 256, 0, st>>>(L, dir, Kp, NP, hi, lo);
    // [ncls][Kp / 4][NP][4] floats as a 3-D tensor {4 NP, Kp / 4, ncls}; one box
    // = one K block of 32 of one class, all NP channels
    const cuuint64_t gdim[3] = {(cuuint64_t)4 * NP, (cuuint64_t)Kp / 4, (cuuint64_t)ncls};
    const cuuint64_t gstr[2] = {(cuuint64_t)4 * NP * 4, (cuuint64_t)(Kp / 4) * 4 * NP * 4};
    const cuuint32_t box[3] = {(cuuint32_t)4 * NP, (cuuint32_t)KC / 4, 1};
    const cuuint32_t es[3] = {1, 1, 1};
    bool good = true;
    for (int part = 0; part < 2 && good; ++part)
      good = enc(part == 0 ? &t->hi[dir] : &t->lo[dir], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                 part == 0 ? hi : lo, gdim, gstr, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                 CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    if (!good) continue;
    t->ok[dir] = true;
    t->N[dir] = N;
    t->NP[dir] = NP;
    t->Kp[dir] = Kp;
    t->ncls[dir] = ncls;
    t->nchunk[dir] = (pmax + 31) / 32;
  }
  return t;
}

void tc_conv_destroy(TcConv* t) { delete t; }

bool tc_conv_usable(const LayerDev& L, int dir) {
  const TcConv* t = static_cast<const TcConv*>(L.tc);
  return t && t->ok[dir];
}

int tc_conv_slots(const LayerDev& L) {
  const TcConv* t = static_cast<const TcConv*>(L.tc);
  return t && t->ok[1] ? t->ncls[1] * t->nchunk[1] : 0;
}

int launch_tc_conv(const LayerDev& L, int dir, int M, const float* in, int ld_in, float* out,
                   int ld_out, const Epi& e, cudaStream_t st) {
  const TcConv* t = static_cast<const TcConv*>(L.tc);
  const dim3 grid(t->ncls[dir] * t->nchunk[dir], (M + TROWS - 1) / TROWS);
  const int NP = t->NP[dir], smem = conv_tc_smem(NP, t->Kp[dir]);
  auto go = [&](auto kern) {
    allow_smem<conv_tc_smem(64, TC_KMAX)>(kern);  // 73 KB; layers take 17 KB and more
    kern<<<grid, TC_THREADS, smem, st>>>(t->hi[dir], t->lo[dir], L, dir, NP, M, t->nchunk[dir], in,
                                         ld_in, out, ld_out, e, e.err);
  };
  switch (epi_mode(e)) {
    case EM_RELU: go(k_conv_tc<EM_RELU>); break;
    case EM_RELU_FINAL: go(k_conv_tc<EM_RELU_FINAL>); break;
    case EM_RELU_GAMMA: go(k_conv_tc<EM_RELU_GAMMA>); break;
    case EM_CONC: go(k_conv_tc<EM_CONC>); break;
    case EM_ADJ: go(k_conv_tc<EM_ADJ>); break;
    case EM_ADJ_GAMMA: go(k_conv_tc<EM_ADJ_GAMMA>); break;
    case EM_FWD: go(k_conv_tc<EM_FWD>); break;
    default: go(k_conv_tc<EM_STORE>); break;
  }
  return grid.x;
}

}  // namespace mnbab
