// Condensed-operator application and Krylov vector kernels.
//
// The condensed operator (Sec. 2.2 eq. SC_step1, Sec. 3.2) is applied without ever
// forming S:  S x_b = A_bb x_b - A_bi (A_ii^-1 (A_ib x_b)).  Two element-parallel
// passes do it:
//   interior pass   u_e = A_ii,e^-1 ( alpha B_i,e + beta (A_ib x_b)_e )
//   boundary pass   y_e = gamma B_b,e + delta (A_bb x_b)_e - (A_bi u)_e
// from the pattern-packed rows of sc_packed.cu (own entries and neighbour couplings).  The same
// two passes give the condensed right-hand side (x_b = 0) and the back-substitution of eq.
// SC_step2.
#include <algorithm>

#include "sc_internal.cuh"

namespace {

__device__ __forceinline__ double warp_sum(double s) {
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

__device__ __forceinline__ void fma16(const double2& a, const double2& b, double& s0, double& s1) {
  s0 = fma(a.x, b.x, s0); s1 = fma(a.y, b.y, s1);
}

// Dot product of a row segment (global, 16-byte aligned) with a vector in shared memory (16-byte
// aligned), one warp, 16-byte loads; returns this lane's partial sum.
__device__ __forceinline__ double warp_dot(const double* __restrict__ row, const double* v, int len, int lane) {
  const double2* r = reinterpret_cast<const double2*>(row);
  const double2* x = reinterpret_cast<const double2*>(v);
  const int nv = len / 2;
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
  for (int i = lane; i < nv; i += 32) fma16(__ldg(r + i), x[i], s0, s1);
  for (int i = nv * 2 + lane; i < len; i += 32) s0 = fma(__ldg(row + i), v[i], s0);
  return s0 + s1;
}

// y = A x on the full system, natural global dof order: one warp per row, gridDim.y CTAs per
// element.  FP64-pipe bound on large meshes; one CTA per element left a mesh of 64 elements on 64
// SMs (216 elements of order 6: 2.5 ms, now 1.36).
__global__ void __launch_bounds__(256) k_global_apply(Geo G, const double* __restrict__ Aown,
    const double* __restrict__ X, const int* __restrict__ nbr, const int* __restrict__ pptr,
    const int* __restrict__ pinfo, const int* __restrict__ pcol, const int* __restrict__ iperm,
    const double* __restrict__ x, double* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* v = reinterpret_cast<double*>(smem_raw);  // lda, own-column order
  __shared__ int nbr_s[18];
  const int e = blockIdx.x, ne = G.ne, nn = G.nn, lda = G.lda;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  if (threadIdx.x < 18) nbr_s[threadIdx.x] = nbr[e * 18 + threadIdx.x];
  for (int i = threadIdx.x; i < lda; i += blockDim.x) v[i] = 0.0;
  __syncthreads();
  for (int t = threadIdx.x; t < ne; t += blockDim.x) {
    const int pos = t / 5, k = t % 5;
    v[own_col(G, pos, k)] = x[((size_t)e * nn + iperm[pos]) * 5 + k];
  }
  __syncthreads();
  const double* Ae = Aown + (size_t)e * own_stride(G);
  for (int ri = blockIdx.y * nw + warp; ri < ne; ri += nw * gridDim.y) {
    const int j = __ldg(iperm + ri / 5), k = ri % 5;
    double s = warp_dot(Ae + (size_t)ri * lda, v, lda, lane);
    const int q0 = __ldg(pptr + j), q1 = __ldg(pptr + j + 1);
    const double* Xr = X + (((size_t)e * 5 + k) * G.NP + q0) * 5;
    for (int f = lane; f < 5 * (q1 - q0); f += 32) {
      const int q = q0 + f / 5, l = f % 5;
      const int nbe = nbr_s[pinfo_slot(__ldg(pinfo + q))];
      s = fma(__ldg(Xr + f), x[((size_t)nbe * nn + __ldg(pcol + q)) * 5 + l], s);
    }
    s = warp_sum(s);
    if (lane == 0) y[((size_t)e * nn + j) * 5 + k] = s;
  }
}

template <class TI>
__global__ void k_scatter(Geo G, const int* __restrict__ iperm, const double* __restrict__ xb,
                          const TI* __restrict__ xi, double* __restrict__ x) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= (size_t)G.K * G.ne) return;
  const int e = (int)(t / G.ne), r = (int)(t % G.ne);
  const int pos = r / 5, k = r % 5;
  const double v = pos < G.nin ? (double)xi[(size_t)e * G.ni + r] : xb[(size_t)e * G.nb + r - G.ni];
  x[((size_t)e * G.nn + iperm[pos]) * 5 + k] = v;
}

// Gram-Schmidt sweeps over the basis vectors V[0 .. nvec), each n long, against w:
//   GS_DOTS     out[i] = <V_i, w>
//   GS_UPDATE   w -= sum_i coef[i] V_i, then out[i] = <V_i, w>
//   GS_NORM     w -= sum_i coef[i] V_i, then out[0] = <w, w>
// The CTAs take tiles of 512 entries; the updated tile of w sits in shared memory and the second use of
// the vectors' tiles hits L1, so CGS2 reads the basis three times from memory, not four.  A warp
// takes a vector (or a part of the tile, while there are fewer than eight vectors) and
// keeps its lanes' sums in shared memory; the last CTA to finish adds up the CTAs' partial sums, in a
// fixed order.  HBM and L2 bound on large systems (16^3 elements of order 4, 15 vectors of 16 MB on
// average: 0.07 + 0.13 + 0.08 ms, as long as separate products and updates), launch bound on
// small ones: three launches per iteration in place of eight.  Tried: half a tile per unit for an
// even load of the warps (16^3: 0.29 ms in all), 2 CTAs per SM (0.32 ms).
using sc::kGsBlocks;
enum { GS_DOTS = 0, GS_UPDATE = 1, GS_NORM = 2 };
constexpr int kGsTile = 512;
__device__ __forceinline__ double2 gs_load(const double* __restrict__ v, size_t t, size_t n, bool vec2) {
  if (vec2) return t < n ? *reinterpret_cast<const double2*>(v + t) : make_double2(0.0, 0.0);
  return make_double2(t < n ? v[t] : 0.0, t + 1 < n ? v[t + 1] : 0.0);
}
// Parts of a tile that a vector's dot product is split into: 8, 4, 2 for 1, 2, 3 .. 4 vectors, else 1.
__host__ __device__ __forceinline__ int gs_parts(int nvec) { return nvec == 1 ? 8 : nvec == 2 ? 4 : nvec <= 4 ? 2 : 1; }

template <int MODE>
__global__ void __launch_bounds__(256) k_gs(const double* __restrict__ V, int nvec, size_t n, double* w,
                                            const double* __restrict__ coef, double* __restrict__ partial,
                                            double* __restrict__ out, unsigned* __restrict__ ticket, int vec2) {
  extern __shared__ __align__(16) double gsm[];
  double* ws = gsm;             // [512] the tile of w
  double* cs = ws + kGsTile;    // [nvec]
  double* acc = cs + nvec;      // [units][32] the lanes' sums
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nout = MODE == GS_NORM ? 1 : nvec, parts = MODE == GS_NORM ? 8 : gs_parts(nvec);
  const int units = nout * parts, span = 8 / parts;  // 64-entry pieces of a unit
  if (MODE != GS_DOTS)
    for (int i = tid; i < nvec; i += 256) cs[i] = coef[i];
  for (int i = tid; i < units * 32; i += 256) acc[i] = 0.0;
  for (size_t t0 = (size_t)blockIdx.x * kGsTile; t0 < n; t0 += (size_t)gridDim.x * kGsTile) {
    __syncthreads();
    {
      const size_t t = t0 + 2 * tid;
      double2 x = gs_load(w, t, n, vec2);
      if (MODE != GS_DOTS) {
        double2 s0 = make_double2(0.0, 0.0), s1 = s0;
        int i = 0;
        for (; i + 8 <= nvec; i += 8) {
          double2 a[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) a[q] = gs_load(V + (size_t)(i + q) * n, t, n, vec2);
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            s0.x = fma(cs[i + q], a[q].x, s0.x); s0.y = fma(cs[i + q], a[q].y, s0.y);
            s1.x = fma(cs[i + q + 1], a[q + 1].x, s1.x); s1.y = fma(cs[i + q + 1], a[q + 1].y, s1.y);
          }
        }
        for (; i + 2 <= nvec; i += 2) {
          const double2 a = gs_load(V + (size_t)i * n, t, n, vec2), b = gs_load(V + (size_t)(i + 1) * n, t, n, vec2);
          s0.x = fma(cs[i], a.x, s0.x); s0.y = fma(cs[i], a.y, s0.y);
          s1.x = fma(cs[i + 1], b.x, s1.x); s1.y = fma(cs[i + 1], b.y, s1.y);
        }
        for (; i < nvec; ++i) {
          const double2 a = gs_load(V + (size_t)i * n, t, n, vec2);
          s0.x = fma(cs[i], a.x, s0.x); s0.y = fma(cs[i], a.y, s0.y);
        }
        x.x -= s0.x + s1.x;
        x.y -= s0.y + s1.y;
        if (t < n) w[t] = x.x;
        if (t + 1 < n) w[t + 1] = x.y;
      }
      ws[2 * tid] = x.x;
      ws[2 * tid + 1] = x.y;
    }
    __syncthreads();
    for (int u = warp; u < units; u += 8) {
      const int i = u / parts, q = u % parts;
      double s0 = 0.0, s1 = 0.0;
      if (MODE != GS_NORM && parts == 1) {  // all eight pieces' loads in flight
        double2 a[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) a[p] = gs_load(V + (size_t)i * n, t0 + 64 * p + 2 * lane, n, vec2);
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          const double2 y = *reinterpret_cast<const double2*>(ws + 64 * p + 2 * lane);
          s0 = fma(a[p].x, y.x, s0);
          s1 = fma(a[p].y, y.y, s1);
        }
      } else {
        for (int p = 0; p < span; ++p) {
          const int l = 64 * (q * span + p) + 2 * lane;
          const double2 y = *reinterpret_cast<const double2*>(ws + l);
          const double2 a = MODE == GS_NORM ? y : gs_load(V + (size_t)i * n, t0 + l, n, vec2);
          s0 = fma(a.x, y.x, s0);
          s1 = fma(a.y, y.y, s1);
        }
      }
      acc[u * 32 + lane] += s0 + s1;
    }
  }
  __syncthreads();
  for (int i = warp; i < nout; i += 8) {
    double s = 0.0;
    for (int q = 0; q < parts; ++q) s += acc[(i * parts + q) * 32 + lane];
    s = warp_sum(s);
    if (lane == 0) partial[(size_t)i * gridDim.x + blockIdx.x] = s;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = warp; i < nout; i += 8) {
    constexpr int kPer = (kGsBlocks + 31) / 32;
    double v[kPer], s = 0.0;  // all loads in flight: a serial sum of them took most of a small sweep's time
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int b = lane + 32 * q;
      v[q] = b < (int)gridDim.x ? __ldcg(partial + (size_t)i * gridDim.x + b) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) s += v[q];
    s = warp_sum(s);
    if (lane == 0) out[i] = s;
  }
  if (tid == 0) *ticket = 0u;  // for the next launch on the stream
}

// dst = w / sqrt(norm2)
__global__ void k_normalize(double* __restrict__ dst, const double* __restrict__ w, size_t n,
                            const double* __restrict__ norm2) {
  const double a = 1.0 / sqrt(norm2[0]);
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    dst[t] = a * w[t];
}

// w -= or += sum_i coef[i] v_i (sign); with vec2 (n even, pointers 16-byte aligned) double2
// accesses and the vectors taken four at a time into independent accumulators.
__global__ void __launch_bounds__(256) k_vec_update(double* __restrict__ w, const double* __restrict__ V, int nvec,
                                                    size_t n, const double* __restrict__ coef, double sign,
                                                    int vec2) {
  __shared__ double cs[64];
  for (int i = threadIdx.x; i < nvec && i < 64; i += blockDim.x) cs[i] = coef[i];
  __syncthreads();
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  if (vec2 && nvec <= 64) {
    const size_t n2 = n / 2;
    double2* w2 = reinterpret_cast<double2*>(w);
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n2; t += stride) {
      double2 a0 = make_double2(0.0, 0.0), a1 = a0, a2 = a0, a3 = a0;
      int i = 0;
      for (; i + 4 <= nvec; i += 4) {
        const double2 v0 = __ldg(reinterpret_cast<const double2*>(V + (size_t)i * n) + t);
        const double2 v1 = __ldg(reinterpret_cast<const double2*>(V + (size_t)(i + 1) * n) + t);
        const double2 v2 = __ldg(reinterpret_cast<const double2*>(V + (size_t)(i + 2) * n) + t);
        const double2 v3 = __ldg(reinterpret_cast<const double2*>(V + (size_t)(i + 3) * n) + t);
        a0.x = fma(cs[i], v0.x, a0.x); a0.y = fma(cs[i], v0.y, a0.y);
        a1.x = fma(cs[i + 1], v1.x, a1.x); a1.y = fma(cs[i + 1], v1.y, a1.y);
        a2.x = fma(cs[i + 2], v2.x, a2.x); a2.y = fma(cs[i + 2], v2.y, a2.y);
        a3.x = fma(cs[i + 3], v3.x, a3.x); a3.y = fma(cs[i + 3], v3.y, a3.y);
      }
      for (; i < nvec; ++i) {
        const double2 v0 = __ldg(reinterpret_cast<const double2*>(V + (size_t)i * n) + t);
        a0.x = fma(cs[i], v0.x, a0.x); a0.y = fma(cs[i], v0.y, a0.y);
      }
      double2 o = w2[t];
      o.x = fma(sign, (a0.x + a1.x) + (a2.x + a3.x), o.x);
      o.y = fma(sign, (a0.y + a1.y) + (a2.y + a3.y), o.y);
      w2[t] = o;
    }
    return;
  }
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += stride) {
    double s = 0.0;
    for (int i = 0; i < nvec; ++i) s = fma(coef[i], V[(size_t)i * n + t], s);
    w[t] = fma(sign, s, w[t]);
  }
}

__global__ void k_scale_copy(double* __restrict__ dst, const double* __restrict__ src, size_t n,
                             const double* __restrict__ scal, int invert) {
  const double a = invert ? 1.0 / scal[0] : scal[0];
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    dst[t] = a * src[t];
}

__global__ void k_vec_to_float(float* __restrict__ y, const double* __restrict__ x, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    y[t] = (float)x[t];
}

// y = a x + b y; with b = 0 y is not read (it may hold anything, NaN included, e.g. a fresh
// Krylov basis vector in memory another context used before).
__global__ void k_axpby(double* __restrict__ y, double a, const double* __restrict__ x, double b, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    y[t] = b == 0.0 ? a * x[t] : a * x[t] + b * y[t];
}

constexpr int kDotBlocks = 608;  // 4 x 152 SMs

}  // namespace

namespace sc {

// The condensed operator's passes on the pattern-packed blocks.
template <class T>
cudaError_t cond_interior_t(sc_ctx* c, const T* Apk, const T* Ainv, const T* xb, double beta, const double* Bfull,
                            double alpha, T* u, int black_zero) {
  if (c->G.ni == 0) return cudaSuccess;
  ProfScope ps(c, SCK_COND_INTERIOR);
  return cond_interior_pk<T>(c, Apk, Ainv, xb, beta, Bfull, alpha, u, black_zero);
}

cudaError_t cond_interior(sc_ctx* c, const double* xb, double beta, const double* Bfull, double alpha, double* u) {
  return cond_interior_t<double>(c, c->Apk, c->Ainv, xb, beta, Bfull, alpha, u, 0);
}

cudaError_t cond_boundary(sc_ctx* c, const double* xb, double delta, const double* Bfull, double gamma_,
                          const double* u, double* y) {
  ProfScope ps(c, SCK_COND_BOUNDARY);
  return cond_boundary_pk<double>(c, c->Apk, xb, delta, Bfull, gamma_, u, y);
}

cudaError_t cond_interior32(sc_ctx* c, const float* xb, double beta, const double* Bfull, double alpha, float* u) {
  return cond_interior_t<float>(c, c->Apk32, c->Ainv32, xb, beta, Bfull, alpha, u, 0);
}

// Interior pass of the red-black sweep: u = A_ii^-1 (A_ib x_b) with x_b zero on the black
// elements, whose own part is then skipped.
cudaError_t cond_interior_sweep(sc_ctx* c, const double* xb, double* u) {
  return cond_interior_t<double>(c, c->Apk, c->Ainv, xb, 1.0, nullptr, 0.0, u, 1);
}

cudaError_t cond_interior_sweep32(sc_ctx* c, const float* xb, float* u) {
  return cond_interior_t<float>(c, c->Apk32, c->Ainv32, xb, 1.0, nullptr, 0.0, u, 1);
}

cudaError_t cond_boundary32(sc_ctx* c, const float* xb, double delta, const double* Bfull, double gamma_,
                            const float* u, double* y) {
  ProfScope ps(c, SCK_COND_BOUNDARY);
  return cond_boundary_pk<float>(c, c->Apk32, xb, delta, Bfull, gamma_, u, y);
}

cudaError_t global_apply(sc_ctx* c, const double* x, double* y) {
  const Geo& G = c->G;
  const size_t smem = (size_t)G.lda * sizeof(double);
  ProfScope ps(c, SCK_GLOBAL_APPLY);
  const int split = std::max(1, std::min((G.ne + 7) / 8, (4 * 6 * 152 + G.K - 1) / G.K));
  k_global_apply<<<dim3(G.K, split), 256, smem, c->stream>>>(G, c->Aown, c->X, c->d_nbr, c->d_pptr, c->d_pinfo, c->d_pcol,
                                                c->d_iperm, x, y);
  return cudaGetLastError();
}

cudaError_t scatter_solution(sc_ctx* c, const double* xb, const double* xi, double* x) {
  const Geo& G = c->G;
  const size_t n = (size_t)G.K * G.ne;
  count_launch(c);
  k_scatter<double><<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(G, c->d_iperm, xb, xi, x);
  return cudaGetLastError();
}

cudaError_t scatter_solution32(sc_ctx* c, const double* xb, const float* xi, double* x) {
  const Geo& G = c->G;
  const size_t n = (size_t)G.K * G.ne;
  count_launch(c);
  k_scatter<float><<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(G, c->d_iperm, xb, xi, x);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t gs_launch(sc_ctx* c, const double* V, int nvec, size_t n, double* w, const double* coef,
                             double* out_dev) {
  if (nvec < 1 || nvec > c->restart_alloc + 1) return cudaErrorInvalidValue;
  const int vec2 = n % 2 == 0 && ((reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(w)) & 15) == 0;
  const int blocks = (int)std::max<size_t>(1, std::min<size_t>(kGsBlocks, (n + kGsTile - 1) / kGsTile));
  const int units = MODE == GS_NORM ? 8 : nvec * gs_parts(nvec);
  const size_t smem = ((size_t)kGsTile + nvec + 32 * units) * sizeof(double);
  if (smem > 48 * 1024) {  // restart lengths above 170
    constexpr int most = (kGsTile + (kMaxRestart + 1) * 33) * (int)sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_gs<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
  }
  count_launch(c);
  k_gs<MODE><<<blocks, 256, smem, c->stream>>>(V, nvec, n, w, coef, c->partial, out_dev,
                                             reinterpret_cast<unsigned*>(c->partial + (size_t)kGsBlocks * (c->restart_alloc + 2)),
                                             vec2);
  return cudaGetLastError();
}

cudaError_t multidot(sc_ctx* c, const double* V, int nvec, size_t n, const double* w, double* out_dev) {
  return gs_launch<GS_DOTS>(c, V, nvec, n, const_cast<double*>(w), nullptr, out_dev);  // w is only read
}

// Classical Gram-Schmidt twice: w is made orthogonal to V[0 .. nvec), the coefficients of the two
// passes go to h1 and h2, <w, w> of the result to hn2 (all on the device).
cudaError_t gram_schmidt(sc_ctx* c, const double* V, int nvec, size_t n, double* w, double* h1, double* h2, double* hn2) {
  cudaError_t e = gs_launch<GS_DOTS>(c, V, nvec, n, w, nullptr, h1);
  if (e == cudaSuccess) e = gs_launch<GS_UPDATE>(c, V, nvec, n, w, h1, h2);
  if (e == cudaSuccess) e = gs_launch<GS_NORM>(c, V, nvec, n, w, h2, hn2);
  return e;
}

cudaError_t vec_normalize(sc_ctx* c, double* dst, const double* w, size_t n, const double* norm2_dev) {
  count_launch(c);
  k_normalize<<<kDotBlocks, 256, 0, c->stream>>>(dst, w, n, norm2_dev);
  return cudaGetLastError();
}

// Partial sums, the CTAs' ticket and the pinned copy of the Gram-Schmidt results for a restart length.
cudaError_t alloc_gs(sc_ctx* c, int restart) {
  const size_t np = (size_t)kGsBlocks * (restart + 2);
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&c->partial), (np + 1) * sizeof(double));
  if (e == cudaSuccess) e = cudaMemset(c->partial + np, 0, sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&c->Hd), (3 * (size_t)(restart + 2) + 16) * sizeof(double));
  if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&c->h_gs), (2 * (size_t)(restart + 1) + 1) * sizeof(double));
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_gs, cudaEventDisableTiming);
  return e;
}

void free_gs(sc_ctx* c) {
  if (c->partial) cudaFree(c->partial);
  if (c->Hd) cudaFree(c->Hd);
  if (c->h_gs) cudaFreeHost(c->h_gs);
  if (c->ev_gs) cudaEventDestroy(c->ev_gs);
  c->partial = c->Hd = c->h_gs = nullptr;
  c->ev_gs = nullptr;
}

cudaError_t vec_update(sc_ctx* c, double* w, const double* V, int nvec, size_t n, const double* coef_dev,
                       double sign) {
  count_launch(c);
  const int vec2 = n % 2 == 0 && ((reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(w)) & 15) == 0;
  k_vec_update<<<kDotBlocks, 256, 0, c->stream>>>(w, V, nvec, n, coef_dev, sign, vec2);
  return cudaGetLastError();
}

cudaError_t vec_scale_copy(sc_ctx* c, double* dst, const double* src, size_t n, const double* scal_dev, int invert) {
  count_launch(c);
  k_scale_copy<<<kDotBlocks, 256, 0, c->stream>>>(dst, src, n, scal_dev, invert);
  return cudaGetLastError();
}

cudaError_t vec_to_float(sc_ctx* c, float* y, const double* x, size_t n) {
  count_launch(c);
  k_vec_to_float<<<kDotBlocks, 256, 0, c->stream>>>(y, x, n);
  return cudaGetLastError();
}

cudaError_t vec_axpby(sc_ctx* c, double* y, double a, const double* x, double b, size_t n) {
  count_launch(c);
  k_axpby<<<kDotBlocks, 256, 0, c->stream>>>(y, a, x, b, n);
  return cudaGetLastError();
}

}  // namespace sc

// ---------------------------------------------------------------------------------
// Allocation-free condensed operator.
//
// sc_condensed_matvec_static applies S with the same operator passes as
// sc_condensed_matvec, but the vectors that link its passes (the interior vector
// u = A_ii^-1 A_ib x_b, and on the mixed arm also the FP32 copy of x_b) live in the static
// device array below instead of context-owned memory, so the call itself never
// allocates.  The array holds 8 MiB on every GPU that loads this library, for the life
// of the process.
// ---------------------------------------------------------------------------------
namespace {
constexpr size_t kStaticScratchBytes = size_t(8) << 20;
}  // namespace

static __device__ __align__(256) unsigned char g_condensed_scratch[kStaticScratchBytes];

namespace {
// Device address of the scratch array on the current device.  Looked up on every call
// with that device current: the lookup allocates nothing, and it stays valid across a
// cudaDeviceReset, which reloads the module at a possibly different address.
cudaError_t static_scratch_address(unsigned char** out) {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_condensed_scratch);
  if (e != cudaSuccess) return e;
  *out = static_cast<unsigned char*>(p);
  return cudaSuccess;
}
}  // namespace

extern "C" sc_status sc_condensed_matvec_static(sc_ctx* c, const double* xb, double* yb) {
  if (!c || !xb || !yb) return SC_ERR_ARG;
  if (!c->has_mesh) {
    c->err = "condensed_matvec_static before set_mesh";
    return SC_ERR_STATE;
  }
  const Geo& G = c->G;
  const bool mixed = c->cfg.precision == SC_PREC_MIXED;
  const bool expl = mixed && c->cfg.explicit_schur;
  const size_t n1 = (size_t)G.K * G.nb, nint = (size_t)G.K * G.ni;
  // FP64 arm: u in doubles; mixed arm: the FP32 copy of x_b (aligned to 256 bytes), then u
  // in floats (the explicit operator needs no u)
  const size_t xf_bytes = mixed ? ((n1 * sizeof(float) + 255) & ~size_t(255)) : 0;
  const size_t need = mixed ? xf_bytes + (expl ? 0 : nint * sizeof(float)) : nint * sizeof(double);
  if (need > kStaticScratchBytes) {
    c->err = "condensed_matvec_static: this mesh needs " + std::to_string(need) +
             " bytes of scratch (FP64 arm: 8 x elements x interior dofs; mixed arm: 4 x elements x"
             " (boundary + interior dofs)), more than the " + std::to_string(kStaticScratchBytes) +
             " bytes of the static buffer; use sc_condensed_matvec";
    return SC_ERR_ARG;
  }
  if (!c->condensed) {
    c->err = "condensed_matvec_static before condense";
    return SC_ERR_STATE;
  }
  unsigned char* scratch = nullptr;
  cudaError_t e = static_scratch_address(&scratch);
  if (e != cudaSuccess) {
    c->err = std::string("condensed_matvec_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e);
    return SC_ERR_CUDA;
  }
  // Every pass writes the entries it later reads (x_b's FP32 copy, then u) before reading
  // them, so nothing left in the array by an earlier call is ever read.
  if (mixed) {
    float* xf = reinterpret_cast<float*>(scratch);
    float* uf = reinterpret_cast<float*>(scratch + xf_bytes);
    e = sc::vec_to_float(c, xf, xb, n1);
    if (e == cudaSuccess) {
      if (expl) {
        e = sc::explicit_matvec32(c, xf, yb);
      } else {
        e = sc::cond_interior32(c, xf, 1.0, nullptr, 0.0, uf);
        if (e == cudaSuccess) e = sc::cond_boundary32(c, xf, 1.0, nullptr, 0.0, uf, yb);
      }
    }
  } else {
    double* u = reinterpret_cast<double*>(scratch);
    e = sc::cond_interior(c, xb, 1.0, nullptr, 0.0, u);
    if (e == cudaSuccess) e = sc::cond_boundary(c, xb, 1.0, nullptr, 0.0, u, yb);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    c->err = std::string("condensed_matvec_static: ") + cudaGetErrorString(e);
    return SC_ERR_CUDA;
  }
  return SC_OK;
}
