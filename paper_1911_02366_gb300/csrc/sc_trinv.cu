// Element block solves with inverted triangular factors (Sec. 2.2: the block-Jacobi solves
// with the factors of S_ee).
//
// With P S_ee = L U, z = S_ee^-1 v = U^-1 (L^-1 (P v)).  The partitioned-inverse solve of
// sc_dense.cu inverts only the 32 x 32 diagonal blocks of L and U, so a solve walks through
// 2 n / 32 dependent block rows; with fewer elements than the chip holds warps that chain, not
// memory, sets the time (0.18 to 0.4 of the HBM rate).  Here the whole triangles are inverted
// once per factorisation: a solve is two triangular matrix-vector products without any chain,
// which spread over as many CTAs as the rows allow and read the same n^2 entries.
//
//   k_tri_inv      L^-1 and U^-1 of every element, one CTA per element, 32-column block and
//                  triangle (block substitution, the column block of the inverse in shared memory)
//   k_tri_apply    x = L^-1 P v, then z = U^-1 x, one CTA per element and pair of block rows
//   k_tri_product  S_ee^-1 = U^-1 L^-1 P as a dense column-major matrix (red elements of the
//                  Schur-corrected sweep)
//   k_inv_gemv     z = S_ee^-1 v with that matrix
//
// Storage is the solve layout of sc_dense.cu (row 32 b + r, column c at [b][c / 4][r][c % 4]):
// U^-1 on and above the diagonal, L^-1 (unit diagonal not stored) below it.
#include <algorithm>
#include <type_traits>

#include "sc_internal.cuh"

namespace {

// Four consecutive values as 16-byte pieces.
template <class T> struct Four { T v[4]; };
__device__ __forceinline__ Four<float> ld4(const float* p) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p));
  return {{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ Four<double> ld4(const double* p) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
  return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ Four<float> ld4(const __half* p) {  // the FP16 copy of FP32 factors
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ Four<float> lds4(const float* p) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  return {{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ Four<double> lds4(const double* p) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4(float* p, const Four<float>& a) {
  *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}
__device__ __forceinline__ void st4(double* p, const Four<double>& a) {
  reinterpret_cast<double2*>(p)[0] = make_double2(a.v[0], a.v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(a.v[2], a.v[3]);
}

// Warps per CTA of k_tri_inv: the column block (32 (nblk - 1) x 32), one 32 x 32 partial sum per
// warp and a diagonal block have to fit 227 KB at the largest n_b of each precision (FP64 760,
// FP32 1090).
template <class T> struct TiWarps { static constexpr int v = 8; };
template <> struct TiWarps<double> { static constexpr int v = 4; };
constexpr int kTbLd = 33;
template <class T>
constexpr size_t tri_inv_smem(int blocks) {
  return ((size_t)(blocks > 1 ? blocks - 1 : 1) * 1024 + TiWarps<T>::v * 1024 + 32 * kTbLd) * sizeof(T);
}

// Column block of L^-1 (upper = false) or U^-1 of one element.  M: the LU factors with the
// diagonal blocks replaced by their triangles' inverses (k_diag_inv).  The len blocks of the
// column are numbered s = 0 .. len - 1 from the diagonal outwards: block row c + s of L^-1,
// c - s of U^-1, and X_s = -D_b sum_{t < s} M_(b, block t) X_t with D_b the inverted diagonal
// triangle of block row b.  FP32/FP64 FMA bound (2/3 n^3 flops per element for both
// triangles): the warps split the sum over t, every lane holds a 4 x 8 tile of the 32 x 32
// block, so 4 global and 8 shared 16-byte loads feed 128 FMAs.  With out16 (FP32 only) the inverse is
// also written in FP16; an entry beyond the FP16 range sets *ovf.
template <class T>
__device__ void tri_inv_body(int n, int x, bool upper, const T* __restrict__ M, int lda, T* __restrict__ out,
                             int npad, __half* __restrict__ out16, int* __restrict__ ovf) {
  constexpr int NW = TiWarps<T>::v;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nblk = (n + 31) / 32, nq = npad / 4;
  const int len = nblk - x;                    // blocks of this column, diagonal one included
  const int c = upper ? nblk - 1 - x : x;      // block column; the long columns come first in the grid
  T* red = reinterpret_cast<T*>(smem_raw);     // [NW][32][32]
  T* Tb = red + NW * 1024;                     // [32][kTbLd] inverted diagonal triangle
  T* X = Tb + 32 * kTbLd;                      // [32 (len - 1)][32]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ly = lane >> 2, lx = lane & 3;
  // the diagonal block: X_0, and (from the lower CTA) the stored tile with both triangles
  for (int t = tid; t < 1024; t += 32 * NW) {
    const int r = t >> 5, k = t & 31, gr = 32 * c + r, gk = 32 * c + k;
    const T d = (gr < n && gk < n) ? M[(long long)gr * lda + gk] : T(0);
    if (len > 1) X[r * 32 + k] = upper ? (k >= r ? d : T(0)) : (k < r ? d : (k == r ? T(1) : T(0)));
    if (!upper && 8 * c + (k >> 2) < nq) {
      const long long o = (long long)c * 32 * npad + (8 * c + (k >> 2)) * 128 + r * 4 + (k & 3);
      out[o] = d;
      if (out16) {
        out16[o] = __float2half_rn((float)d);
        if (!(fabs((double)d) <= 65000.0)) atomicExch(ovf, 1);
      }
    }
  }
  for (int s = 1; s < len; ++s) {
    const int b = upper ? c - s : c + s;
    __syncthreads();
    for (int t = tid; t < 1024; t += 32 * NW) {
      const int r = t >> 5, k = t & 31, gr = 32 * b + r, gk = 32 * b + k;
      const T d = (gr < n && gk < n) ? M[(long long)gr * lda + gk] : T(0);
      Tb[r * kTbLd + k] = upper ? (k >= r ? d : T(0)) : (k < r ? d : (k == r ? T(1) : T(0)));
    }
    T acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = T(0);
    for (int ch = warp; ch < 8 * s; ch += NW) {
      const int kk = 4 * ch;
      const int col = upper ? 32 * (c - (kk >> 5)) + (kk & 31) : 32 * c + kk;
      Four<T> a[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = 32 * b + 4 * ly + i;
        const T* p = M + (long long)row * lda + col;
        if (row < n && col + 3 < n) {
          a[i] = ld4(p);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) a[i].v[j] = (row < n && col + j < n) ? p[j] : T(0);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const Four<T> x0 = lds4(X + (kk + j) * 32 + 8 * lx), x1 = lds4(X + (kk + j) * 32 + 8 * lx + 4);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[i][q] = fma(a[i].v[j], x0.v[q], acc[i][q]);
            acc[i][4 + q] = fma(a[i].v[j], x1.v[q], acc[i][4 + q]);
          }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      T* r = red + warp * 1024 + (4 * ly + i) * 32 + 8 * lx;
      st4(r, Four<T>{{acc[i][0], acc[i][1], acc[i][2], acc[i][3]}});
      st4(r + 4, Four<T>{{acc[i][4], acc[i][5], acc[i][6], acc[i][7]}});
    }
    __syncthreads();
    for (int t = tid; t < 1024; t += 32 * NW) {
      T v = red[t];
#pragma unroll
      for (int w = 1; w < NW; ++w) v += red[w * 1024 + t];
      red[t] = v;
    }
    __syncthreads();
    // X_s = -D_b (sum): lane = row, four columns per thread and pass
    for (int cq = warp; cq < 8; cq += NW) {
      Four<T> y{{T(0), T(0), T(0), T(0)}};
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const T d = Tb[lane * kTbLd + k];
        const Four<T> v = lds4(red + k * 32 + 4 * cq);
#pragma unroll
        for (int q = 0; q < 4; ++q) y.v[q] = fma(-d, v.v[q], y.v[q]);
      }
      if (s + 1 < len) st4(X + (32 * s + lane) * 32 + 4 * cq, y);
      if (8 * c + cq < nq) {
        const long long o = (long long)b * 32 * npad + (long long)(8 * c + cq) * 128 + lane * 4;
        st4(out + o, y);
        if (out16) {
          bool big = false;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            out16[o + q] = __float2half_rn((float)y.v[q]);
            big = big || !(fabs((double)y.v[q]) <= 65000.0);
          }
          if (big) atomicExch(ovf, 1);
        }
      }
    }
  }
}

template <class T>
__global__ void __launch_bounds__(32 * TiWarps<T>::v) k_tri_inv(int n, int x0, const T* __restrict__ LU,
                                                                long long stride, int lda, T* __restrict__ LS,
                                                                long long lsstride, int npad,
                                                                __half* __restrict__ LS16, int* __restrict__ ovf) {
  const int e = blockIdx.y;
  tri_inv_body<T>(n, x0 + blockIdx.x, blockIdx.z != 0, LU + (long long)e * stride, lda, LS + (long long)e * lsstride,
                  npad, LS16 ? LS16 + (long long)e * lsstride : nullptr, ovf);
}

__global__ void __launch_bounds__(32 * TiWarps<float>::v) k_tri_inv_grouped(const CondItem* __restrict__ items, int x0) {
  const CondItem it = items[blockIdx.y];
  tri_inv_body<float>(it.nb, x0 + blockIdx.x, blockIdx.z != 0, it.See, it.lds, it.Sls, (it.nb + 3) & ~3,
                      nullptr, nullptr);
}

// x = L^-1 P (v - vsub) (UPPER = false, x compact per list entry) or z = U^-1 x: CTA (p, i) forms
// the block rows p and nblk - 1 - p of list entry i, which together read the same number of
// entries for every p; its warps share the 4-column groups and meet in shared memory.
// HBM bound where the factors exceed L2: 364 elements of n_b = 760 (0.84 GB) take 0.155 ms
// (0.84 of HBM) against 0.38 ms for the chain of block rows, 216 of n_b = 1090 (1.03 GB) 0.178 (0.89) against 0.62 ms.
constexpr int kTaWarps = 8;  // one per 4-column group of a diagonal block
// T: arithmetic, TS: storage of the factors.
template <class T, class TS, bool UPPER>
__global__ void __launch_bounds__(32 * kTaWarps) k_tri_apply(int n, int nblk, const TS* __restrict__ LS,
                                                             long long lsstride, int npad,
                                                             const int* __restrict__ rowperm,
                                                             const double* __restrict__ v,
                                                             const double* __restrict__ vsub, T* __restrict__ x,
                                                             double* __restrict__ z, T* __restrict__ zt,
                                                             const int* __restrict__ elist, int compact) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);  // [32 nblk]
  __shared__ T red[kTaWarps][64];
  const int i = blockIdx.y, e = elist ? __ldg(elist + i) : i, f = compact ? i : e;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nq = npad / 4, ls = 32 * nblk;
  const int b0 = blockIdx.x, b1 = nblk - 1 - b0;  // b0 <= b1
  T* xe = x + (long long)i * ls;
  const int lo = UPPER ? 32 * b0 : 0, hi = UPPER ? ls : 32 * (b1 + 1);
  for (int t = lo + threadIdx.x; t < hi; t += blockDim.x) {
    T val = T(0);
    if (UPPER) {
      val = xe[t];
    } else if (t < n) {
      const long long r = (long long)e * n + __ldg(rowperm + (long long)f * n + t);
      val = vsub ? (T)(v[r] - vsub[r]) : (T)v[r];
    }
    s[t] = val;
  }
  __syncthreads();
  const TS* Le = LS + (long long)f * lsstride + 4 * lane;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int b = h ? b1 : b0;
    T a0 = T(0), a1 = T(0);
    if (h == 0 || b1 != b0) {
      const TS* row = Le + (long long)b * 32 * npad;
      const int R = 32 * b + lane;
      // the diagonal block's groups, entries of the other triangle left out
      const int qd = 8 * b + warp;
      if (qd < nq && R < n) {
        const Four<T> m = ld4(row + (long long)qd * 128);
        const Four<T> y = lds4(s + 4 * qd);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (UPPER ? 4 * qd + j >= R : 4 * qd + j < R) a0 = fma(m.v[j], y.v[j], a0);
      }
      const int q0 = UPPER ? 8 * b + 8 : 0, q1 = UPPER ? nq : 8 * b;
      if (R < n) {
#pragma unroll 8
        for (int q = q0 + warp; q < q1; q += kTaWarps) {
          const Four<T> m = ld4(row + (long long)q * 128);
          const Four<T> y = lds4(s + 4 * q);
          a0 = fma(m.v[0], y.v[0], a0);
          a1 = fma(m.v[1], y.v[1], a1);
          a0 = fma(m.v[2], y.v[2], a0);
          a1 = fma(m.v[3], y.v[3], a1);
        }
      }
    }
    red[warp][32 * h + lane] = a0 + a1;
  }
  __syncthreads();
  if (threadIdx.x < 64) {
    const int b = threadIdx.x < 32 ? b0 : b1, R = 32 * b + lane;
    if (threadIdx.x < 32 || b1 != b0) {
      T sum = T(0);
#pragma unroll
      for (int w = 0; w < kTaWarps; ++w) sum += red[w][threadIdx.x];
      if (!UPPER) {
        xe[R] = R < n ? s[R] + sum : T(0);
      } else if (R < n) {
        if (z) z[(long long)e * n + R] = (double)sum;
        if (zt) zt[(long long)e * n + R] = sum;
      }
    }
  }
}

// Dense inverse S_ee^-1 = U^-1 L^-1 P of compact list entry blockIdx.z, column-major with
// leading dimension ldz (rows n .. ldz - 1 zero): 128 x 64 tiles, 8 x 4 outputs per thread, the
// sum over k starting where both triangles have entries.  FP32 FMA bound, 2/3 n^3 flops.
constexpr int kTpM = 128, kTpN = 64;
__global__ void __launch_bounds__(256) k_tri_product(int n, const float* __restrict__ LS, long long lsstride, int npad,
                                                     const int* __restrict__ rowperm, int ldz,
                                                     float* __restrict__ Zinv) {
  __shared__ __align__(16) float As[32][kTpM + 4];  // U^-1 tile, transposed
  __shared__ __align__(16) float Bs[32][kTpN + 4];  // L^-1 tile
  const int i = blockIdx.z, nq = npad / 4, nblk = (n + 31) / 32;
  const int m0 = blockIdx.y * kTpM, n0 = blockIdx.x * kTpN;
  const float* Le = LS + (long long)i * lsstride;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
  for (int k0 = max(m0, n0); k0 < 32 * nblk; k0 += 32) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {  // U^-1: rows m0 .. m0 + 127, columns k0 .. k0 + 31
      const int t = tid + 256 * u, r = (t & 31) + 32 * (t >> 8), q = (t >> 5) & 7;
      const int R = m0 + r, C = k0 + 4 * q;
      Four<float> a{{0.f, 0.f, 0.f, 0.f}};
      if (R < n && C + 3 >= R && C / 4 < nq) a = ld4(Le + (long long)(R >> 5) * 32 * npad + (long long)(C / 4) * 128 + (R & 31) * 4);
#pragma unroll
      for (int j = 0; j < 4; ++j) As[4 * q + j][r] = (C + j >= R && C + j < n) ? a.v[j] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {  // L^-1: rows k0 .. k0 + 31, columns n0 .. n0 + 63
      const int t = tid + 256 * u, k = t & 31, q = t >> 5;
      const int R = k0 + k, C = n0 + 4 * q;
      Four<float> a{{0.f, 0.f, 0.f, 0.f}};
      if (R < n && C < R) a = ld4(Le + (long long)(R >> 5) * 32 * npad + (long long)(C / 4) * 128 + (R & 31) * 4);
#pragma unroll
      for (int j = 0; j < 4; ++j) a.v[j] = C + j < R ? a.v[j] : ((C + j == R && R < n) ? 1.f : 0.f);
      st4(&Bs[k][4 * q], a);
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const Four<float> a0 = lds4(&As[k][8 * ty]), a1 = lds4(&As[k][8 * ty + 4]), b = lds4(&Bs[k][4 * tx]);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[a][j] = fmaf(a0.v[a], b.v[j], acc[a][j]);
          acc[4 + a][j] = fmaf(a1.v[a], b.v[j], acc[4 + a][j]);
        }
    }
    __syncthreads();
  }
  const int row = m0 + 8 * ty;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int cc = n0 + 4 * tx + j;
    if (cc >= n) continue;
    float* o = Zinv + ((long long)i * n + __ldg(rowperm + (long long)i * n + cc)) * ldz + row;
    if (row < ldz) st4(o, Four<float>{{acc[0][j], acc[1][j], acc[2][j], acc[3][j]}});
    if (row + 4 < ldz) st4(o + 4, Four<float>{{acc[4][j], acc[5][j], acc[6][j], acc[7][j]}});
  }
}

// z = S_ee^-1 v with the dense inverses: CTA (t, i) forms rows 128 t .. of list entry i, each lane
// four rows, the warps sharing the columns.  HBM bound: 2048 elements of n_b = 490 (1.98 GB)
// take 0.294 ms (0.99 of HBM) against 0.35 ms (0.87) for the partitioned-inverse solve with the factors.
constexpr int kIgWarps = 8;
__global__ void __launch_bounds__(32 * kIgWarps) k_inv_gemv(int n, int ldz, const float* __restrict__ Zinv,
                                                            const double* __restrict__ v, double* __restrict__ z,
                                                            float* __restrict__ zt, const int* __restrict__ elist) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* s = reinterpret_cast<float*>(smem_raw);  // [n]
  __shared__ __align__(16) float red[kIgWarps][128];
  const int i = blockIdx.y, e = __ldg(elist + i);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < n; t += blockDim.x) s[t] = (float)v[(long long)e * n + t];
  __syncthreads();
  const int row = 128 * blockIdx.x + 4 * lane;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
  if (row < ldz) {
    const float* Z = Zinv + (long long)i * n * ldz + row;
    int c = warp;
#pragma unroll 4
    for (; c + kIgWarps < n; c += 2 * kIgWarps) {
      const float4 m = __ldg(reinterpret_cast<const float4*>(Z + (long long)c * ldz));
      const float4 k = __ldg(reinterpret_cast<const float4*>(Z + (long long)(c + kIgWarps) * ldz));
      const float y = s[c], w = s[c + kIgWarps];
      a.x = fmaf(m.x, y, a.x); a.y = fmaf(m.y, y, a.y); a.z = fmaf(m.z, y, a.z); a.w = fmaf(m.w, y, a.w);
      b.x = fmaf(k.x, w, b.x); b.y = fmaf(k.y, w, b.y); b.z = fmaf(k.z, w, b.z); b.w = fmaf(k.w, w, b.w);
    }
    if (c < n) {
      const float4 m = __ldg(reinterpret_cast<const float4*>(Z + (long long)c * ldz));
      const float y = s[c];
      a.x = fmaf(m.x, y, a.x); a.y = fmaf(m.y, y, a.y); a.z = fmaf(m.z, y, a.z); a.w = fmaf(m.w, y, a.w);
    }
  }
  *reinterpret_cast<float4*>(&red[warp][4 * lane]) = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
  __syncthreads();
  const int r = 128 * blockIdx.x + threadIdx.x;
  if (threadIdx.x < 128 && r < n) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kIgWarps; ++w) sum += red[w][threadIdx.x];
    if (z) z[(long long)e * n + r] = (double)sum;
    if (zt) zt[(long long)e * n + r] = sum;
  }
}

// Diagonal node blocks [S_ee^-1]_kk of every (element, boundary node) sample from the inverted
// triangles: one warp per sample, lanes over the inner index.
__global__ void __launch_bounds__(128) k_tri_node_blocks(int n, const float* __restrict__ LS, long long lsstride,
                                                         int npad, const int* __restrict__ rowperm, int nsmp,
                                                         float* __restrict__ out) {
  const int lane = threadIdx.x & 31, smp = blockIdx.x * 4 + (threadIdx.x >> 5);
  __shared__ int pos[4][5];  // permuted column of each variable
  if (smp >= nsmp) return;
  const int nbn = n / 5, e = smp / nbn, a = smp % nbn, w = threadIdx.x >> 5;
  const int* rp = rowperm + (long long)e * n;
  if (lane < 5) pos[w][lane] = n;  // a column that no row maps to meets no entry below
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    const int d = __ldg(rp + i) - 5 * a;
    if (d >= 0 && d < 5) pos[w][d] = i;
  }
  __syncwarp();
  const float* Le = LS + (long long)e * lsstride;
  auto at = [&](int r, int c) { return __ldg(Le + (long long)(r >> 5) * 32 * npad + (long long)(c >> 2) * 128 + (r & 31) * 4 + (c & 3)); };
  float acc[5][5] = {};
  for (int k = lane; k < n; k += 32) {
    float l[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int c = pos[w][j];
      l[j] = c < k ? at(k, c) : (c == k ? 1.f : 0.f);
    }
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      const float u = 5 * a + r <= k ? at(5 * a + r, k) : 0.f;
#pragma unroll
      for (int j = 0; j < 5; ++j) acc[r][j] = fmaf(u, l[j], acc[r][j]);
    }
  }
#pragma unroll
  for (int r = 0; r < 5; ++r)
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      float v = acc[r][j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) out[(long long)smp * 25 + 5 * r + j] = v;
    }
}

// Launch x = 0 .. nblk - 1 in two halves: the second one's columns are at most half as long and
// leave room for more CTAs per SM.
template <class F>
cudaError_t tri_inv_halves(int nblk, F&& launch) {
  const int half = nblk / 2;
  cudaError_t e = cudaSuccess;
  if (half > 0) e = launch(0, half, nblk);
  if (e == cudaSuccess) e = launch(half, nblk - half, nblk - half);
  return e;
}

}  // namespace

namespace sc {

// Triangle inverses of `count` factorised n x n blocks (diagonal blocks inverted) into LS.
template <class T>
cudaError_t tri_inverse(sc_ctx* c, int n, const T* LU, long long stride, int lda, T* LS, int count, __half* LS16,
                        int* ovf) {
  if (count <= 0) return cudaSuccess;
  const int nblk = (n + 31) / 32, npad = (n + 3) & ~3;
  const long long ls = (long long)nblk * 32 * npad;
  cudaError_t e = cudaFuncSetAttribute(k_tri_inv<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)tri_inv_smem<T>((kMaxNb<T> + 31) / 32));
  if (e != cudaSuccess) return e;
  return tri_inv_halves(nblk, [&](int x0, int nx, int blocks) {
    count_launch(c);
    k_tri_inv<T><<<dim3(nx, count, 2), 32 * TiWarps<T>::v, tri_inv_smem<T>(blocks), c->stream>>>(n, x0, LU, stride, lda,
                                                                                                LS, ls, npad, LS16, ovf);
    return cudaGetLastError();
  });
}
template cudaError_t tri_inverse<float>(sc_ctx*, int, const float*, long long, int, float*, int, __half*, int*);
template cudaError_t tri_inverse<double>(sc_ctx*, int, const double*, long long, int, double*, int, __half*, int*);

// The same for consecutive batched items of one block size.
cudaError_t grouped_tri_inverse(cudaStream_t st, const CondItem* items, int count, int nb) {
  if (count <= 0) return cudaSuccess;
  const int nblk = (nb + 31) / 32;
  cudaError_t e = cudaFuncSetAttribute(k_tri_inv_grouped, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)tri_inv_smem<float>((kMaxNb<float> + 31) / 32));
  if (e != cudaSuccess) return e;
  return tri_inv_halves(nblk, [&](int x0, int nx, int blocks) {
    k_tri_inv_grouped<<<dim3(nx, count, 2), 32 * TiWarps<float>::v, tri_inv_smem<float>(blocks), st>>>(items, x0);
    return cudaGetLastError();
  });
}

// z (double) and / or zt = S_ee^-1 (v - vsub) for a list of elements (all when elist is null) with
// the inverted triangles; factors by element, or compact by list position.
template <class T, class TS>
cudaError_t tri_solve(sc_ctx* c, const TS* LS, const int* rowperm, int compact, const int* elist, int count,
                      const double* v, const double* vsub, double* z, T* zt) {
  if (count <= 0) return cudaSuccess;
  const int n = c->G.nb, nblk = (n + 31) / 32, npad = (n + 3) & ~3;
  const long long ls = (long long)nblk * 32 * npad;
  const size_t smem = (size_t)nblk * 32 * sizeof(T);
  const dim3 grid((nblk + 1) / 2, count);
  T* x = static_cast<T*>(c->tri_x);
  count_launch(c);  // the profiled span counts one
  k_tri_apply<T, TS, false><<<grid, 32 * kTaWarps, smem, c->stream>>>(n, nblk, LS, ls, npad, rowperm, v, vsub, x, nullptr,
                                                                  (T*)nullptr, elist, compact);
  k_tri_apply<T, TS, true><<<grid, 32 * kTaWarps, smem, c->stream>>>(n, nblk, LS, ls, npad, rowperm, nullptr, nullptr, x, z,
                                                                 zt, elist, compact);
  return cudaGetLastError();
}
template cudaError_t tri_solve<float, __half>(sc_ctx*, const __half*, const int*, int, const int*, int, const double*,
                                              const double*, double*, float*);
template cudaError_t tri_solve<float, float>(sc_ctx*, const float*, const int*, int, const int*, int, const double*,
                                      const double*, double*, float*);
template cudaError_t tri_solve<double, double>(sc_ctx*, const double*, const int*, int, const int*, int, const double*,
                                       const double*, double*, double*);

// Dense column-major inverses (leading dimension lds) of `count` compact entries.
cudaError_t tri_dense_inverse(sc_ctx* c, const float* LS, const int* rowperm, int count, float* out) {
  if (count <= 0) return cudaSuccess;
  const int n = c->G.nb, nblk = (n + 31) / 32, npad = (n + 3) & ~3;
  count_launch(c);
  k_tri_product<<<dim3((n + kTpN - 1) / kTpN, (n + kTpM - 1) / kTpM, count), 256, 0, c->stream>>>(
      n, LS, (long long)nblk * 32 * npad, npad, rowperm, c->G.lds, out);
  return cudaGetLastError();
}

cudaError_t dense_inverse_apply(sc_ctx* c, const float* inv, const int* elist, int count, const double* v, double* z,
                                float* zt) {
  if (count <= 0) return cudaSuccess;
  const int n = c->G.nb, ldz = c->G.lds;
  k_inv_gemv<<<dim3((ldz + 127) / 128, count), 32 * kIgWarps, (size_t)n * sizeof(float), c->stream>>>(n, ldz, inv, v, z,
                                                                                                   zt, elist);
  return cudaGetLastError();
}

// out: of `count` elements, 25 values per boundary node.
cudaError_t tri_node_blocks(sc_ctx* c, const float* LS, const int* rowperm, int count, float* out) {
  const Geo& G = c->G;
  const int nblk = (G.nb + 31) / 32, npad = (G.nb + 3) & ~3, nsmp = count * G.nbn;
  count_launch(c);
  k_tri_node_blocks<<<(nsmp + 3) / 4, 128, 0, c->stream>>>(G.nb, LS, (long long)nblk * 32 * npad, npad, rowperm, nsmp,
                                                         out);
  return cudaGetLastError();
}

}  // namespace sc
