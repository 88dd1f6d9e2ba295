// The learned correction of the condensed-system preconditioner: a 128 -> 256 -> 256 -> 25
// network with ReLU hidden layers, BF16 weights and FP32 arithmetic (not in the paper; a
// learned part of the condensed-system preconditioner of Sec. 2.2/4), with its training loop
// (shuffled mini-batch Adam) and a file format for its parameters.
//
// The forward pass is one tensor-core kernel, 128 samples per CTA through all layers with the
// activations in TMEM.  The backward pass runs through a SIMT tile kernel, C (+)= op(A) op(B), K
// chunks staged in shared memory (BF16 operands widened to FP32 on the way):
//   backward dX  dZ_prev = (dZ W) * [Z_prev > 0]      (A = dZ, B = W)
//   backward dW  gW += dZ^T X, split over samples     (A = dZ stored n x out)
// plus the loss, bias-gradient and Adam kernels.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "sc_internal.cuh"
#include "sc_tcgen.cuh"

namespace {

constexpr int NI = sc::kMlpInputs, NH = 256, NO = 25;
constexpr int OFF_W2 = NH * NI, OFF_W3 = OFF_W2 + NH * NH, N_W = OFF_W3 + NO * NH;  // 104,704
constexpr int OFF_B2 = NH, OFF_B3 = 2 * NH, N_B = 2 * NH + NO;                     // 537

template <class T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return __ldg(p); }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}

enum Epi { EPI_MASK = 0, EPI_ATOMIC = 1 };

// C[M x N] from op(A)[M x K] op(B)[K x N], B stored K x N (ldb); A stored M x K (lda) or K x M
// when TA.  gridDim.z splits K (EPI_ATOMIC only).  BT x BT tiles, BK deep; the next K chunk is
// loaded while the current one is multiplied.  A training batch is latency bound: with 64 x 64
// tiles a layer of 256 samples has 16 CTAs, so small products take 32 x 32 tiles.
template <class TB_, bool TA, int EPI, int BT, int BK>
__global__ void __launch_bounds__(256) k_mlp_gemm(int M, int N, int K, const float* __restrict__ A, int lda,
                                                  const TB_* __restrict__ B, int ldb, float* __restrict__ C, int ldc,
                                                  const float* __restrict__ mask, int kchunk) {
  constexpr int PT = BT / 16, LD = BT * BK / 256;  // outputs per thread and direction, loads per thread
  __shared__ float As[BK][BT + 4];
  __shared__ float Bs[BK][BT + 4];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int m0 = blockIdx.y * BT, n0 = blockIdx.x * BT;
  const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
  float acc[PT][PT] = {}, ra[LD], rb[LD];
  // A stored M x K is contiguous in k, everything else in the tile's rows
  auto a_pos = [&](int i, int& kk, int& mm) {
    const int t = threadIdx.x + 256 * i;
    if (TA) { kk = t / BT; mm = t % BT; } else { kk = t % BK; mm = t / BK; }
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      int kk, mm;
      a_pos(i, kk, mm);
      const int ga = k0 + kk, gm = m0 + mm;
      ra[i] = ga < ke && gm < M ? (TA ? ldf(A + (size_t)ga * lda + gm) : ldf(A + (size_t)gm * lda + ga)) : 0.f;
      const int t = threadIdx.x + 256 * i, gk = k0 + t / BT, gn = n0 + t % BT;
      rb[i] = gk < ke && gn < N ? ldf(B + (size_t)gk * ldb + gn) : 0.f;
    }
  };
  load(kb);
  for (int k0 = kb; k0 < ke; k0 += BK) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      int kk, mm;
      a_pos(i, kk, mm);
      As[kk][mm] = ra[i];
      const int t = threadIdx.x + 256 * i;
      Bs[t / BT][t % BT] = rb[i];
    }
    __syncthreads();
    if (k0 + BK < ke) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[PT], b[PT];
#pragma unroll
      for (int i = 0; i < PT; ++i) { a[i] = As[kk][ty + 16 * i]; b[i] = Bs[kk][tx + 16 * i]; }
#pragma unroll
      for (int i = 0; i < PT; ++i)
#pragma unroll
        for (int j = 0; j < PT; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < PT; ++i) {
    const int r = m0 + ty + 16 * i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < PT; ++j) {
      const int cc = n0 + tx + 16 * j;
      if (cc >= N) continue;
      float v = acc[i][j];
      if (EPI == EPI_ATOMIC) {
        atomicAdd(C + (size_t)r * ldc + cc, v);
      } else {
        if (!(mask[(size_t)r * ldc + cc] > 0.f)) v = 0.f;
        C[(size_t)r * ldc + cc] = v;
      }
    }
  }
}

// ---- forward pass on the tensor cores -------------------------------------------------
// One CTA takes 128 samples through all three layers: C = A W^T as tcgen05.mma (kind::f16, BF16
// operands, M = 128).  The FP32 inputs of a layer are split exactly into three BF16 parts of 8
// significand bits each (cut, not rounded) and the weights are BF16 already, so every product is
// exact.  The tensor cores' FP32 accumulation cuts where FMA rounds: over a whole layer that
// costs four times the error of an FMA chain (1.4e-6 against 3.5e-7 of the largest output), so
// the accumulator (TMEM columns 0 .. 255) is started anew for every 64 inputs, the small parts first, and the
// partial sums are added up in registers.  An infinite weight meets the zero parts of an exactly split
// input as NaN, which the first pass carries to the outputs; a tile whose outputs hold one is done again,
// carefully: the small parts times the finite weights, then the first parts, which have the inputs'
// signs, times all of them (167 us per 100,352 samples with and without that second look).  The
// activations wait in TMEM columns 256 .. 511 for the next layer and leave the SM only if the caller asks
// for them (z1 .. h2).  Inputs and weights are
// staged in two shared-memory buffers (three 128 x 64 parts and a 256 x 64 piece of the weights,
// K-major core matrices of 8 rows x 16 bytes): while the tensor cores work on one chunk, the threads split
// and store the next and load the one after.  Thread t holds row t % 128 (its TMEM lane) and of every
// 64 columns the half t / 128.  A wait that runs out leaves SC_TC_TIMEOUT in *status and NaN in its samples' outputs.
// 100,352 samples: 0.17 ms a call against 2.43 ms for three SIMT products and their temporaries; a
// training batch of 256: about 50 us against 82.  Bound by the instruction stream of a CTA's eight warps
// (split, store, collect), not by the tensor cores.  Tried: pieces of eight rows per warp load (0.21 ms
// when the split cost more), activations written through shared memory (no gain).
constexpr int kFwStage = 3 * 128 * 64 * 2 + 256 * 64 * 2;  // bytes
constexpr int kCoreLbo = 128, kCoreSbo = 8 * kCoreLbo;
__device__ __forceinline__ uint32_t bf16_core(int row, int k) {
  return (uint32_t)((row >> 3) * kCoreSbo + (k >> 3) * kCoreLbo + (row & 7) * 16);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D = F32, A = B = BF16, both K-major, M = 128.
constexpr uint32_t idesc_bf16(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// Polls of the forward pass's waits before it gives up (a build with -1 gives up at once).
#ifndef SC_MLP_WAIT_POLLS
#define SC_MLP_WAIT_POLLS kWaitLimit
#endif
// The same for all lanes of a warp.
__device__ __forceinline__ bool wait_bounded(uint64_t* bar, uint32_t parity, long long limit) {
  bool done = false;
  for (long long it = 0; it <= limit && !done; ++it) done = mbar_try_wait(bar, parity);
  return __all_sync(0xffffffffu, done);
}
// x = p[0] + p[1] + p[2] in BF16 (bit patterns); infinities and NaN stay in the first part.
__device__ __forceinline__ void split3(float x, uint32_t p[3]) {
  const uint32_t b = __float_as_uint(x);
  p[0] = b >> 16;
  if ((b & 0x7f800000u) == 0x7f800000u) {
    if (b & 0x007fffffu) p[0] |= 0x40u;
    p[1] = p[2] = 0u;
    return;
  }
  const float r1 = x - __uint_as_float(b & 0xffff0000u);
  p[1] = __float_as_uint(r1) >> 16;
  p[2] = __float_as_uint(r1 - __uint_as_float(__float_as_uint(r1) & 0xffff0000u)) >> 16;
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
               "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
               "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
               "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
               : "memory");
}
// 32 accumulator columns added to acc.
__device__ __forceinline__ void tmem_add32(uint32_t taddr, float* acc) {
  uint32_t r[4][8];
#pragma unroll
  for (int g = 0; g < 4; ++g) tmem_ld8_async(taddr + 8 * g, r[g]);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] += __uint_as_float(r[i >> 3][i & 7]);
}

// The three parts of eight values, packed in pairs: two subtractions and one byte permutation per pair
// and part.  The remainders of a finite value are exact, so the sum of the last ones is NaN only if a
// value is infinite or NaN; those take the careful split (100,352 samples: 209 us with it for all, now 167).
__device__ __forceinline__ void split3x8(const float* x, uint32_t q[3][4]) {
  float bad = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float r[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float v = x[2 * j + h];
      r[h][0] = v - __uint_as_float(__float_as_uint(v) & 0xffff0000u);
      r[h][1] = r[h][0] - __uint_as_float(__float_as_uint(r[h][0]) & 0xffff0000u);
      bad += r[h][1];
    }
    q[0][j] = __byte_perm(__float_as_uint(x[2 * j]), __float_as_uint(x[2 * j + 1]), 0x7632);
    q[1][j] = __byte_perm(__float_as_uint(r[0][0]), __float_as_uint(r[1][0]), 0x7632);
    q[2][j] = __byte_perm(__float_as_uint(r[0][1]), __float_as_uint(r[1][1]), 0x7632);
  }
  if (bad != bad) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t lo[3], hi[3];
      split3(x[2 * j], lo);
      split3(x[2 * j + 1], hi);
#pragma unroll
      for (int s = 0; s < 3; ++s) q[s][j] = lo[s] | hi[s] << 16;
    }
  }
}

struct FwLane {  // what a thread of k_mlp_forward works on
  const __nv_bfloat16* W;
  const float* X;
  unsigned char* stage;
  uint64_t* bar;
  uint32_t tmem, lanes;
  int tid, row, half, gr, n, flags, step;
};

// Products of 64 inputs, parts s = hi .. lo of them, with `fresh` into a new accumulator (small parts
// first), by one thread.
template <int L>
__device__ __forceinline__ void fw_issue(const FwLane& f, const unsigned char* As, const unsigned char* Bs, int hi, int lo,
                                         bool fresh) {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
  for (int s = 2; s >= 0; --s)
    if (s <= hi && s >= lo)
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        mma_bf16(f.tmem, smem_desc(smem_u32(As) + s * 16384 + kk * 2 * kCoreLbo, kCoreLbo, kCoreSbo),
                 smem_desc(smem_u32(Bs) + kk * 2 * kCoreLbo, kCoreLbo, kCoreSbo), idesc_bf16(L < 2 ? 256 : 32),
                 !fresh || s < hi || kk > 0);
  mma_commit(f.bar);
}
// Two BF16 weights with infinities and NaN cleared.
__device__ __forceinline__ uint32_t finite_pair(uint32_t v) {
  if ((v & 0x7f80u) == 0x7f80u) v &= 0xffff0000u;
  if ((v & 0x7f800000u) == 0x7f800000u) v &= 0xffffu;
  return v;
}

// Piece k0 .. k0 + 63 of a layer's weights: one row per thread (256 rows), or one 16-byte piece
// (32 rows, 25 of them real).
template <int L>
__device__ __forceinline__ void fw_load_w(const FwLane& f, int k0, uint4 w[8]) {
  constexpr int K = L == 0 ? NI : NH;
  const __nv_bfloat16* Wl = f.W + (L == 0 ? 0 : L == 1 ? OFF_W2 : OFF_W3);
  auto piece = [&](int r, int k) {
    const __nv_bfloat16* p = Wl + (size_t)r * K + k0 + k;
    if (f.flags & 2) return __ldg(reinterpret_cast<const uint4*>(p));
    const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
    return make_uint4(q[0] | (uint32_t)q[1] << 16, q[2] | (uint32_t)q[3] << 16, q[4] | (uint32_t)q[5] << 16,
                      q[6] | (uint32_t)q[7] << 16);
  };
  if (L < 2) {
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = piece(f.tid, 8 * i);
  } else {
    w[0] = (f.tid & 31) < NO ? piece(f.tid & 31, 8 * (f.tid >> 5)) : make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ void fw_load_x(const FwLane& f, int k0, float a[32]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (f.gr < f.n) {
      const float* p = f.X + (size_t)f.gr * NI + k0 + 32 * f.half + 4 * i;
      if (f.flags & 1) v = __ldg(reinterpret_cast<const float4*>(p));
      else v = make_float4(p[0], p[1], p[2], p[3]);
    }
    a[4 * i] = v.x; a[4 * i + 1] = v.y; a[4 * i + 2] = v.z; a[4 * i + 3] = v.w;
  }
}

// Products of one layer: acc[32 q + i] = sum over the layer's inputs for column 64 q + 32 half + i
// (layer 3: the 32 columns, first half of the threads only).  w holds the first weights on entry
// and the next layer's first ones on return, a the first inputs of layer 1.  False: a wait ran out.
template <int L, bool CAREFUL>
__device__ __forceinline__ bool fw_layer(FwLane& f, float a[32], uint4 w[8], float acc[128]) {
  constexpr int NC = (L == 0 ? NI : NH) / 64, NQ = L < 2 ? 4 : 1;
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 32 * NQ; ++i) acc[i] = 0.f;
  auto collect = [&]() {  // the products of the chunk before
    ok = ok && wait_bounded(f.bar, (f.step - 1) & 1, SC_MLP_WAIT_POLLS);
    if (!ok) return;  // as a condition of the loads below: 2.5 us of 167 per 100,352 samples
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (L < 2 || f.half == 0)
#pragma unroll
      for (int q = 0; q < NQ; ++q) tmem_add32(f.tmem + f.lanes + 64 * q + (L < 2 ? 32 * f.half : 0), acc + 32 * q);
  };
#pragma unroll 1
  for (int ch = 0; ch < NC; ++ch) {
    unsigned char* As = f.stage + (f.step & 1) * kFwStage;
    unsigned char* Bs = As + 3 * 128 * 64 * 2;
    if (CAREFUL && ch > 0) {  // nothing overlaps in the careful pass
      collect();
      if (!__syncthreads_and(ok)) return false;
    }
    if (L > 0) {
      uint32_t r[4][8];
#pragma unroll
      for (int g = 0; g < 4; ++g) tmem_ld8_async(f.tmem + f.lanes + 256 + 64 * ch + 32 * f.half + 8 * g, r[g]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int i = 0; i < 32; ++i) a[i] = __uint_as_float(r[i >> 3][i & 7]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t q[3][4];
      split3x8(a + 8 * i, q);
#pragma unroll
      for (int s = 0; s < 3; ++s)
        *reinterpret_cast<uint4*>(As + s * 16384 + bf16_core(f.row, 32 * f.half + 8 * i)) =
            make_uint4(q[s][0], q[s][1], q[s][2], q[s][3]);
    }
    auto put_w = [&](bool finite) {
      auto put = [&](int row, int k, uint4 v) {
        if (finite) v = make_uint4(finite_pair(v.x), finite_pair(v.y), finite_pair(v.z), finite_pair(v.w));
        *reinterpret_cast<uint4*>(Bs + bf16_core(row, k)) = v;
      };
      if (L < 2) {
#pragma unroll
        for (int i = 0; i < 8; ++i) put(f.tid, 8 * i, w[i]);
      } else {
        put(f.tid & 31, 8 * (f.tid >> 5), w[0]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };
    if (CAREFUL) {  // the small parts meet the finite weights only
      put_w(true);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      if (f.tid == 0) fw_issue<L>(f, As, Bs, 2, 1, true);
      ++f.step;
      ok = ok && wait_bounded(f.bar, (f.step - 1) & 1, SC_MLP_WAIT_POLLS);
      if (!__syncthreads_and(ok)) return false;
    }
    put_w(false);
    if (ch + 1 < NC) {
      fw_load_w<L>(f, 64 * (ch + 1), w);
      if (L == 0) fw_load_x(f, 64 * (ch + 1), a);
    } else if (L < 2) {
      fw_load_w<L < 2 ? L + 1 : 2>(f, 0, w);
    }
    if (ch > 0 && !CAREFUL) collect();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    ok = __syncthreads_and(ok);
    if (!ok) return false;
    if (f.tid == 0) {
      fw_issue<L>(f, As, Bs, CAREFUL ? 0 : 2, 0, !CAREFUL);
    }
    ++f.step;
  }
  collect();
  return __syncthreads_and(ok);
}

// Bias, pre-activations (z, may be null), ReLU, activations (h, may be null), and the activations to TMEM.
template <bool CAREFUL>
__device__ __forceinline__ void fw_activate(const FwLane& f, const float* bias, float acc[128], float* z, float* h) {
  auto put = [&](float* o) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float* p = o + (size_t)f.gr * NH + 64 * q + 32 * f.half;
      if (f.flags & 4) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          reinterpret_cast<float4*>(p)[i] = make_float4(acc[32 * q + 4 * i], acc[32 * q + 4 * i + 1],
                                                       acc[32 * q + 4 * i + 2], acc[32 * q + 4 * i + 3]);
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) p[i] = acc[32 * q + i];
      }
    }
  };
#pragma unroll
  for (int i = 0; i < 128; ++i) acc[i] += bias[64 * (i >> 5) + 32 * f.half + (i & 31)];
  if (z && f.gr < f.n) put(z);
  // NaN passes the first pass's ReLU, so that the outputs show it, and gives 0 in the careful one
#pragma unroll
  for (int i = 0; i < 128; ++i) {
    if (CAREFUL) acc[i] = fmaxf(acc[i], 0.f);
    else asm("max.NaN.f32 %0, %0, 0f00000000;" : "+f"(acc[i]));
  }
  if (h && f.gr < f.n) put(h);
#pragma unroll
  for (int i = 0; i < 16; ++i) tmem_st8(f.tmem + f.lanes + 256 + 64 * (i >> 2) + 32 * f.half + 8 * (i & 3), acc + 8 * i);
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// All three layers; acc: the products of the last one.
template <bool CAREFUL>
__device__ __forceinline__ bool fw_network(FwLane& f, float a[32], uint4 w[8], float acc[128], const float* bias, float* z1,
                                           float* h1, float* z2, float* h2) {
  if (!fw_layer<0, CAREFUL>(f, a, w, acc)) return false;
  fw_activate<CAREFUL>(f, bias, acc, z1, h1);
  if (!fw_layer<1, CAREFUL>(f, a, w, acc)) return false;
  fw_activate<CAREFUL>(f, bias + OFF_B2, acc, z2, h2);
  return fw_layer<2, CAREFUL>(f, a, w, acc);
}

// The careful pass: the outputs' products to y.  A function of its own: inlined, it makes the kernel's body
// spill (177 us instead of 167).
__device__ __noinline__ bool fw_careful(FwLane* f, const float* bias, float* z1, float* h1, float* z2, float* h2, float* y) {
  float a[32], acc[128];
  uint4 w[8];
  fw_load_x(*f, 0, a);
  fw_load_w<0>(*f, 0, w);
  const bool ok = fw_network<true>(*f, a, w, acc, bias, z1, h1, z2, h2);
#pragma unroll
  for (int i = 0; i < NO; ++i) y[i] = acc[i];
  return ok;
}

// flags: bit 0 X is 16-byte aligned, bit 1 W, bit 2 the activations' rows.
__global__ void __launch_bounds__(256, 1) k_mlp_forward(int n, const __nv_bfloat16* __restrict__ W,
                                                        const float* __restrict__ bias, const float* __restrict__ X,
                                                        float* __restrict__ Y, float* __restrict__ z1,
                                                        float* __restrict__ h1, float* __restrict__ z2,
                                                        float* __restrict__ h2, int flags, int* status) {
  extern __shared__ __align__(1024) unsigned char stage_mem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_s;
  __shared__ float bias_s[N_B + 7];
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) tmem_alloc(&tmem_s, 512);
  if (tid == 0) {
    mbar_init(&mbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  FwLane f{W, X, stage_mem, &mbar, 0u, (uint32_t)(32 * (warp & 3)) << 16, tid, tid & 127, tid >> 7,
           (int)blockIdx.x * 128 + (tid & 127), n, flags, 0};
  float a[32], acc[128];
  uint4 w[8];
  fw_load_x(f, 0, a);
  fw_load_w<0>(f, 0, w);
  for (int i = tid; i < N_B + 7; i += 256) bias_s[i] = i < N_B ? bias[i] : 0.f;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  f.tmem = tmem_s;
  bool ok = fw_network<false>(f, a, w, acc, bias_s, z1, h1, z2, h2);
  bool nan = false;
  if (ok && f.half == 0 && f.gr < n)
#pragma unroll
    for (int i = 0; i < NO; ++i) nan = nan || acc[i] != acc[i];
  if (__syncthreads_or(nan)) {
    FwLane g = f;
    float y[NO];
    ok = fw_careful(&g, bias_s, z1, h1, z2, h2, y);
    f.step = g.step;
#pragma unroll
    for (int i = 0; i < NO; ++i) acc[i] = y[i];
  }
  if (!ok) {
    if (f.step > 0) wait_bounded(&mbar, (f.step - 1) & 1, kWaitLimit);  // products still in flight
    if (tid == 0) {  // device memory or a mapped host word
      *reinterpret_cast<volatile int*>(status) = SC_TC_TIMEOUT;
      __threadfence_system();
    }
  }
  if (f.half == 0 && f.gr < n)
#pragma unroll
    for (int i = 0; i < NO; ++i)
      Y[(size_t)f.gr * NO + i] = ok ? acc[i] + bias_s[OFF_B3 + i] : __int_as_float(0x7fc00000);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tmem_dealloc(f.tmem, 512);
}

cudaError_t forward(cudaStream_t st, const __nv_bfloat16* W, const float* bias, const float* X, int n, float* Y,
                    float* z1, float* h1, float* z2, float* h2, int* status) {
  auto a16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const int flags = (a16(X) ? 1 : 0) | (a16(W) ? 2 : 0) | (a16(z1) && a16(h1) && a16(z2) && a16(h2) ? 4 : 0);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kFwStage);
  if (e != cudaSuccess) return e;
  k_mlp_forward<<<(unsigned)((n + 127) / 128), 256, 2 * kFwStage, st>>>(n, W, bias, X, Y, z1, h1, z2, h2, flags,
                                                                         status);
  return cudaGetLastError();
}

// gb[c] += sum_s dZ[s][c]
__global__ void k_mlp_colsum(int n, int m, const float* __restrict__ dZ, float* __restrict__ gb) {
  const int c = blockIdx.x;
  float s = 0.f;
  for (int r = threadIdx.x; r < n; r += blockDim.x) s += dZ[(size_t)r * m + c];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ float part[32];
  if (threadIdx.x % 32 == 0) part[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < blockDim.x / 32 ? part[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) gb[c] += s;
  }
}

// Mean squared relative Frobenius error of the 25-entry outputs, and its gradient.
__global__ void k_mlp_loss(int n, const float* __restrict__ Y, const float* __restrict__ T, float* __restrict__ dY,
                           float* __restrict__ loss_sum) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  float l = 0.f;
  if (s < n) {
    float num = 0.f, den = 1e-12f;
    for (int j = 0; j < NO; ++j) {
      const float d = Y[(size_t)s * NO + j] - T[(size_t)s * NO + j];
      const float t = T[(size_t)s * NO + j];
      num = fmaf(d, d, num);
      den = fmaf(t, t, den);
    }
    l = num / den / (float)n;
    if (dY)
      for (int j = 0; j < NO; ++j)
        dY[(size_t)s * NO + j] = 2.f * (Y[(size_t)s * NO + j] - T[(size_t)s * NO + j]) / den / (float)n;
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (loss_sum && threadIdx.x % 32 == 0) atomicAdd(loss_sum, l);
}

// Adam (bias-corrected moments) over the FP32 master parameters; refreshes the BF16
// weight copy and clears the gradient it consumed.
__global__ void k_mlp_adam(int nw, int nbias, float* __restrict__ W, __nv_bfloat16* __restrict__ Wh,
                           float* __restrict__ bias, float* __restrict__ gW, float* __restrict__ gb,
                           float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                           float c1, float c2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nw + nbias) return;
  float* p = t < nw ? W + t : bias + (t - nw);
  float* g = t < nw ? gW + t : gb + (t - nw);
  const float gv = *g;
  const float mv = b1 * m[t] + (1.f - b1) * gv;
  const float vv = b2 * v[t] + (1.f - b2) * gv * gv;
  m[t] = mv;
  v[t] = vv;
  const float upd = lr * (mv / c1) / (sqrtf(vv / c2) + eps);
  const float np = *p - upd;
  *p = np;
  if (t < nw) Wh[t] = __float2bfloat16_rn(np);
  *g = 0.f;
}

template <class TB_, bool TA, int EPI>
cudaError_t gemm(cudaStream_t st, int M, int N, int K, const float* A, int lda, const TB_* B, int ldb, float* C,
                 int ldc, const float* mask, int splits = 1) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  const int kchunk = ((K + splits - 1) / splits + 31) / 32 * 32;
  const int nz = (K + kchunk - 1) / kchunk;
  auto grid = [&](int bt) { return dim3((N + bt - 1) / bt, (M + bt - 1) / bt, nz); };
  const dim3 g = grid(64);
  // 32 x 32 tiles until the 64 x 64 ones fill the 152 SMs
  if ((long long)g.x * g.y * g.z < 152)
    k_mlp_gemm<TB_, TA, EPI, 32, 32><<<grid(32), 256, 0, st>>>(M, N, K, A, lda, B, ldb, C, ldc, mask, kchunk);
  else
    k_mlp_gemm<TB_, TA, EPI, 64, 16><<<g, 256, 0, st>>>(M, N, K, A, lda, B, ldb, C, ldc, mask, kchunk);
  return cudaGetLastError();
}

// Rows perm[i0 .. i0 + nb) of X (64 wide) and T (25 wide) into contiguous batch buffers.
__global__ void k_gather_batch(const int* __restrict__ perm, int i0, int nb, const float* __restrict__ X,
                               const float* __restrict__ T, float* __restrict__ Xb, float* __restrict__ Tb) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nb * (NI + NO)) return;
  const int r = t / (NI + NO), c = t % (NI + NO);
  const long long src = __ldg(perm + i0 + r);
  if (c < NI) Xb[(long long)r * NI + c] = X[src * NI + c];
  else Tb[(long long)r * NO + c - NI] = T[src * NO + c - NI];
}

__global__ void k_to_bf16(const float* __restrict__ W, __nv_bfloat16* __restrict__ Wh, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) Wh[t] = __float2bfloat16_rn(W[t]);
}

// splitmix64 step (Steele, Lea and Flood 2014): the shuffles' random stream.
uint64_t splitmix64_next(uint64_t& state) {
  uint64_t z = (state += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// The word in which a forward pass of this host thread reports a wait that ran out: mapped host memory, so
// that reading it after the call's synchronisation costs no copy; given back with the thread.
struct StatusWord {
  int* p = nullptr;
  ~StatusWord() { if (p) cudaFreeHost(p); }
};
cudaError_t status_word(int** host, int** device) {
  static thread_local StatusWord w;
  void* d = nullptr;
  if (w.p && cudaHostGetDevicePointer(&d, w.p, 0) != cudaSuccess) {  // gone with a device reset
    (void)cudaGetLastError();
    w.p = nullptr;
  }
  if (!w.p) {
    // another thread may be capturing a graph
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    void* q = nullptr;
    e = cudaHostAlloc(&q, sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped);
    const cudaError_t back = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess || back != cudaSuccess) return e != cudaSuccess ? e : back;
    w.p = static_cast<int*>(q);
    e = cudaHostGetDevicePointer(&d, w.p, 0);
    if (e != cudaSuccess) return e;
  }
  *host = w.p;
  *device = static_cast<int*>(d);
  return cudaSuccess;
}

constexpr char kMlpMagic[8] = {'S', 'C', 'M', 'L', 'P', '0', '0', '1'};

}  // namespace

namespace sc {

// Inference: Y = net(X); *status (device) <- SC_TC_TIMEOUT if a wait runs out.
cudaError_t mlp_forward(cudaStream_t st, const uint16_t* Wbf16, const float* bias, const float* X, int n, float* Y,
                        int* status) {
  if (n <= 0) return cudaSuccess;
  return forward(st, reinterpret_cast<const __nv_bfloat16*>(Wbf16), bias, X, n, Y, nullptr, nullptr, nullptr, nullptr,
                 status);
}

}  // namespace sc

extern "C" {

sc_status sc_mlp_forward(const uint16_t* Wbf16, const float* bias, const float* X, int n, float* Y, float* cache,
                         void* cuda_stream) {
  if (!Wbf16 || !bias || !X || !Y || n < 0) return SC_ERR_ARG;
  if (n == 0) return SC_OK;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const __nv_bfloat16* W = reinterpret_cast<const __nv_bfloat16*>(Wbf16);
  // cache: [z1 | h1 | z2 | h2], each n x 256 (pre- and post-activations)
  auto part = [&](int i) { return cache ? cache + (size_t)i * n * NH : nullptr; };
  int *word = nullptr, *dword = nullptr;
  cudaError_t e = status_word(&word, &dword);
  if (e != cudaSuccess) return SC_ERR_CUDA;
  *word = 0;
  e = forward(st, W, bias, X, n, Y, part(0), part(1), part(2), part(3), dword);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess && *static_cast<volatile int*>(word) == 0 ? SC_OK : SC_ERR_CUDA;
}

sc_status sc_mlp_backward(const uint16_t* Wbf16, const float* X, const float* cache, const float* dY, int n,
                          float* gW, float* gb, float* work, void* cuda_stream) {
  if (!Wbf16 || !X || !cache || !dY || !gW || !gb || !work || n <= 0) return SC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const __nv_bfloat16* W = reinterpret_cast<const __nv_bfloat16*>(Wbf16);
  const float* z1 = cache;
  const float* h1 = cache + (size_t)n * NH;
  const float* z2 = cache + 2 * (size_t)n * NH;
  const float* h2 = cache + 3 * (size_t)n * NH;
  float* dz2 = work;                      // n x 256
  float* dz1 = work + (size_t)n * NH;     // n x 256
  const int splits = (n + 2047) / 2048;   // sample chunks of the weight gradients
  cudaError_t e;
  // layer 3: gW3 += dY^T h2, gb3 += colsum dY, dz2 = (dY W3) * [z2 > 0]
  e = gemm<float, true, EPI_ATOMIC>(st, NO, NH, n, dY, NO, h2, NH, gW + OFF_W3, NH, nullptr,
                                    splits);
  if (e == cudaSuccess) { k_mlp_colsum<<<NO, 256, 0, st>>>(n, NO, dY, gb + OFF_B3); e = cudaGetLastError(); }
  if (e == cudaSuccess)
    e = gemm<__nv_bfloat16, false, EPI_MASK>(st, n, NH, NO, dY, NO, W + OFF_W3, NH, dz2, NH, z2);
  // layer 2
  if (e == cudaSuccess)
    e = gemm<float, true, EPI_ATOMIC>(st, NH, NH, n, dz2, NH, h1, NH, gW + OFF_W2, NH, nullptr,
                                    splits);
  if (e == cudaSuccess) { k_mlp_colsum<<<NH, 256, 0, st>>>(n, NH, dz2, gb + OFF_B2); e = cudaGetLastError(); }
  if (e == cudaSuccess)
    e = gemm<__nv_bfloat16, false, EPI_MASK>(st, n, NH, NH, dz2, NH, W + OFF_W2, NH, dz1, NH, z1);
  // layer 1
  if (e == cudaSuccess)
    e = gemm<float, true, EPI_ATOMIC>(st, NH, NI, n, dz1, NH, X, NI, gW, NI, nullptr,
                                    splits);
  if (e == cudaSuccess) { k_mlp_colsum<<<NH, 256, 0, st>>>(n, NH, dz1, gb); e = cudaGetLastError(); }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? SC_OK : SC_ERR_CUDA;
}

sc_status sc_mlp_loss(const float* Y, const float* T, int n, float* dY, float* loss_sum, void* cuda_stream) {
  if (!Y || !T || n <= 0) return SC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  k_mlp_loss<<<(n + 255) / 256, 256, 0, st>>>(n, Y, T, dY, loss_sum);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? SC_OK : SC_ERR_CUDA;
}

sc_status sc_mlp_adam(float* W, uint16_t* Wbf16, float* bias, float* gW, float* gb, float* m, float* v, int step,
                      float lr, void* cuda_stream) {
  if (!W || !Wbf16 || !bias || !gW || !gb || !m || !v || step < 1) return SC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  const int tot = N_W + N_B;
  k_mlp_adam<<<(tot + 255) / 256, 256, 0, st>>>(N_W, N_B, W, reinterpret_cast<__nv_bfloat16*>(Wbf16), bias, gW, gb,
                                                 m, v, lr, b1, b2, eps, c1, c2);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? SC_OK : SC_ERR_CUDA;
}

sc_status sc_mlp_bf16(const float* W, uint16_t* Wbf16, int n, void* cuda_stream) {
  if (!W || !Wbf16 || n < 0) return SC_ERR_ARG;
  if (n == 0) return SC_OK;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  k_to_bf16<<<(n + 255) / 256, 256, 0, st>>>(W, reinterpret_cast<__nv_bfloat16*>(Wbf16), n);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? SC_OK : SC_ERR_CUDA;
}

sc_status sc_mlp_train(float* W, uint16_t* Wbf16, float* bias, float* m, float* v, int* step, const float* X,
                       const float* T, int n, int epochs, int batch, float lr, uint64_t seed, float* loss_hist,
                       void* cuda_stream) {
  if (!W || !Wbf16 || !bias || !m || !v || !step || !X || !T || n < 1 || epochs < 0 || batch < 1 || *step < 0)
    return SC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int bmax = batch < n ? batch : n;
  float *gW = nullptr, *gb = nullptr, *cache = nullptr, *work = nullptr, *Y = nullptr, *dY = nullptr;
  float *Xb = nullptr, *Tb = nullptr, *acc = nullptr;
  int* perm = nullptr;
  cudaError_t e = cudaSuccess;
  auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  A(cudaMalloc(&gW, (size_t)N_W * sizeof(float))); A(cudaMalloc(&gb, (size_t)N_B * sizeof(float)));
  A(cudaMalloc(&cache, (size_t)4 * bmax * NH * sizeof(float))); A(cudaMalloc(&work, (size_t)2 * bmax * NH * sizeof(float)));
  A(cudaMalloc(&Y, (size_t)bmax * NO * sizeof(float))); A(cudaMalloc(&dY, (size_t)bmax * NO * sizeof(float)));
  A(cudaMalloc(&Xb, (size_t)bmax * NI * sizeof(float))); A(cudaMalloc(&Tb, (size_t)bmax * NO * sizeof(float)));
  A(cudaMalloc(&acc, sizeof(float))); A(cudaMalloc(&perm, (size_t)n * sizeof(int)));
  sc_status s = e == cudaSuccess ? SC_OK : SC_ERR_OOM;
  if (s == SC_OK) {
    A(cudaMemsetAsync(gW, 0, (size_t)N_W * sizeof(float), st));
    A(cudaMemsetAsync(gb, 0, (size_t)N_B * sizeof(float), st));
    if (e != cudaSuccess) s = SC_ERR_CUDA;
  }
  std::vector<int> hp(n);
  uint64_t rs = seed;
  const int nbatch = (n + bmax - 1) / bmax;
  for (int ep = 0; ep < epochs && s == SC_OK; ++ep) {
    // Fisher-Yates shuffle of all samples: batches mix systems, elements and nodes
    for (int i = 0; i < n; ++i) hp[i] = i;
    for (int i = n - 1; i > 0; --i) {
      const int j = (int)(splitmix64_next(rs) % (uint64_t)(i + 1));
      std::swap(hp[i], hp[j]);
    }
    A(cudaMemcpyAsync(perm, hp.data(), (size_t)n * sizeof(int), cudaMemcpyHostToDevice, st));
    A(cudaMemsetAsync(acc, 0, sizeof(float), st));
    if (e != cudaSuccess) { s = SC_ERR_CUDA; break; }
    for (int b = 0; b < nbatch && s == SC_OK; ++b) {
      const int i0 = b * bmax, nb = (n - i0) < bmax ? (n - i0) : bmax;
      k_gather_batch<<<(nb * (NI + NO) + 255) / 256, 256, 0, st>>>(perm, i0, nb, X, T, Xb, Tb);
      if (cudaGetLastError() != cudaSuccess) { s = SC_ERR_CUDA; break; }
      s = sc_mlp_forward(Wbf16, bias, Xb, nb, Y, cache, st);
      if (s == SC_OK) s = sc_mlp_loss(Y, Tb, nb, dY, acc, st);
      if (s == SC_OK) s = sc_mlp_backward(Wbf16, Xb, cache, dY, nb, gW, gb, work, st);
      if (s == SC_OK) s = sc_mlp_adam(W, Wbf16, bias, gW, gb, m, v, ++*step, lr, st);
    }
    if (s == SC_OK && loss_hist) {
      float a = 0.f;
      if (cudaMemcpyAsync(&a, acc, sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess) s = SC_ERR_CUDA;
      loss_hist[ep] = a / (float)nbatch;
    }
  }
  cudaFree(gW); cudaFree(gb); cudaFree(cache); cudaFree(work); cudaFree(Y); cudaFree(dY); cudaFree(Xb); cudaFree(Tb);
  cudaFree(acc); cudaFree(perm);
  return s;
}

sc_status sc_mlp_save(const char* path, const float* W, const float* bias) {
  if (!path || !W || !bias) return SC_ERR_ARG;
  std::vector<float> hw(N_W), hb(N_B);
  if (cudaMemcpy(hw.data(), W, (size_t)N_W * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(hb.data(), bias, (size_t)N_B * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return SC_ERR_CUDA;
  FILE* f = std::fopen(path, "wb");
  if (!f) return SC_ERR_ARG;
  const int32_t counts[2] = {N_W, N_B};
  bool ok = std::fwrite(kMlpMagic, 1, 8, f) == 8 && std::fwrite(counts, sizeof(int32_t), 2, f) == 2 &&
            std::fwrite(hw.data(), sizeof(float), N_W, f) == (size_t)N_W &&
            std::fwrite(hb.data(), sizeof(float), N_B, f) == (size_t)N_B;
  ok = (std::fclose(f) == 0) && ok;
  return ok ? SC_OK : SC_ERR_ARG;
}

sc_status sc_mlp_load(const char* path, float* W, uint16_t* Wbf16, float* bias) {
  if (!path || !W || !Wbf16 || !bias) return SC_ERR_ARG;
  FILE* f = std::fopen(path, "rb");
  if (!f) return SC_ERR_ARG;
  char magic[8];
  int32_t counts[2] = {0, 0};
  std::vector<float> hw(N_W), hb(N_B);
  bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kMlpMagic, 8) == 0 &&
            std::fread(counts, sizeof(int32_t), 2, f) == 2 && counts[0] == N_W && counts[1] == N_B &&
            std::fread(hw.data(), sizeof(float), N_W, f) == (size_t)N_W &&
            std::fread(hb.data(), sizeof(float), N_B, f) == (size_t)N_B;
  std::fclose(f);
  if (!ok) return SC_ERR_ARG;
  if (cudaMemcpy(W, hw.data(), (size_t)N_W * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(bias, hb.data(), (size_t)N_B * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess)
    return SC_ERR_CUDA;
  return sc_mlp_bf16(W, Wbf16, N_W, nullptr);
}

}  // extern "C"
