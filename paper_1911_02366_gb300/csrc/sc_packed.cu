// Pattern-packed element blocks for the condensed operator (Sec. 2.2, eq. SC_step1 with
// the implicit Schur product; Sec. 3.1 on the sparsity of the element blocks).
//
// On a tensor-product GL element the own block couples node j only to the nodes that
// share at least one of its three GL indices: the inviscid volume terms run along the
// three grid lines through j, and the BR1 viscous terms differentiate a lifted gradient
// that itself runs along lines, so they reach the three planes through j.  The operator
// passes need A_ib (interior rows, boundary columns) and [A_bi A_bb] (boundary rows): of
// these dense blocks only 43-50 % of the 5 x 5 node blocks can be nonzero.
//
// Packed layout, per element and shared by all elements: row r of the own block keeps
// the entries of its node's column list (the column nodes sharing an index, interior
// columns first, in own-column order), 5 per column node, padded with zeros to a multiple of 4
// entries, then the row's neighbour couplings (5 per node pair, in pair order), padded the same
// way: everything an operator pass reads for a row is one stream of 16-byte pieces.  Two code
// tables, also shared by all elements, name the vector entries of every four matrix entries
// (which belong to at most two column nodes).  The packing kernel also checks that every entry
// left out is exactly zero and reports the element otherwise.
#include <algorithm>
#include <type_traits>

#include "sc_internal.cuh"

namespace {

// Resident CTAs per SM asked of the operator passes.  FP32: 5 (48 registers) measured best at every
// order; 4 and 6 make the boundary pass 1 and 10 % slower at 16^3, N = 4.  The FP64 passes are
// FP64-ALU bound and keep their natural allocation (3 CTAs allow the 64-74 registers they use).
template <class T> struct PkOcc { static constexpr int v = 3; };
template <> struct PkOcc<float> { static constexpr int v = 5; };

template <class T> struct PkVec;
template <> struct PkVec<float> { using type = float4; static constexpr int n = 4; };
template <> struct PkVec<double> { using type = double2; static constexpr int n = 2; };

// Sums of 5 values over the warp by halving exchanges (8 shuffles instead of 25): afterwards lane
// writer_lane(k) holds the sum of value k.
template <class T>
__device__ __forceinline__ T wsum5(const T a[5], int lane) {
  constexpr unsigned M = 0xffffffffu;
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
  T p = h16 ? a[1] : a[0], q = h16 ? a[3] : a[2], e = a[4];
  p += __shfl_xor_sync(M, h16 ? a[0] : a[1], 16);
  q += __shfl_xor_sync(M, h16 ? a[2] : a[3], 16);
  e += __shfl_xor_sync(M, e, 16);
  T k = h8 ? q : p;
  k += __shfl_xor_sync(M, h8 ? p : q, 8);
  e += __shfl_xor_sync(M, e, 8);
  T r = h4 ? e : k;
  r += __shfl_xor_sync(M, h4 ? k : e, 4);
  r += __shfl_xor_sync(M, r, 2);
  r += __shfl_xor_sync(M, r, 1);
  return r;
}
// The value whose sum this lane holds after wsum5, or -1 (lanes 0, 16, 8, 24, 4 hold 0 .. 4).
__device__ __forceinline__ int wsum5_owner(int lane) {
  if (lane & 3) return -1;
  if (lane & 4) return lane == 4 ? 4 : -1;
  return ((lane >> 4) & 1) + 2 * ((lane >> 3) & 1);
}

// Entry w (0..3) of a group of four: the first node's entries come before position t.
__device__ __forceinline__ int group_split(int i) {  // i: group index in the row
  const int r = i % 5;
  return r == 0 ? 5 : r;
}

// The 5 rows of a node (variables k = 0..4): row k starts at P0 + k * rs with `own` packed own
// entries, of which the first n_own count (both multiples of 4), and n_cross coupling entries.
// Own entries meet the own-column-ordered vector v in shared memory: own_code[j / 4] holds the
// positions of a group of four (low half: of the entries before the split, less their index;
// high half: of those from it on).  Couplings meet the neighbours' boundary (vb, coefficient cb)
// or interior (vi, coefficient ci) vectors: cross_code[j / 4] names for both parts of a group the
// neighbour slot (31: padding), the interior flag and the offset (biased by 8, less the entry's
// index).  One loop covers both, so that a row's tail and its couplings share a step.
template <class T>
__device__ __forceinline__ void node_rows5(const T* __restrict__ P0, int rs, int own, int n_own, int n_cross,
                                           const int* __restrict__ own_code, const int2* __restrict__ cross_code,
                                           const T* __restrict__ v, const int* nbr_s, int nb, int ni,
                                           const T* __restrict__ vb, T cb, const T* __restrict__ vi, T ci, int lane,
                                           T acc[5]) {
  using V = typename PkVec<T>::type;
  constexpr int W = PkVec<T>::n;
  const int n = n_own + n_cross, skip = own - n_own;
  auto use = [&](int j, const V a[5]) {
    T x[W];
    if (j < n_own) {
      const int i = j >> 2, code = __ldg(own_code + i), t = group_split(i), w0 = j & 3;
#pragma unroll
      for (int w = 0; w < W; ++w) x[w] = v[(w0 + w < t ? (code & 0xffff) : (code >> 16)) + w0 + w];
    } else {
      const int i = (j - n_own) >> 2, t = group_split(i), w0 = j & 3;
      const int2 code = __ldg(cross_code + i);
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const int f = w0 + w < t ? code.x : code.y, slot = pinfo_slot(f);
        T g = T(0);
        if (slot != 31) {
          const int off = pinfo_offset(f) - 8 + w0 + w;
          if (pinfo_interior(f)) {
            if (vi) g = ci * __ldg(vi + (size_t)nbr_s[slot] * ni + off);
          } else {
            if (vb) g = cb * __ldg(vb + (size_t)nbr_s[slot] * nb + off);
          }
        }
        x[w] = g;
      }
    }
#pragma unroll
    for (int w = 0; w < W; ++w)
#pragma unroll
      for (int k = 0; k < 5; ++k) acc[k] = fma(reinterpret_cast<const T*>(&a[k])[w], x[w], acc[k]);
  };
  for (int j = lane * W; j < n; j += 32 * W) {
    V a[5];
    const T* p = P0 + (j < n_own ? j : j + skip);
#pragma unroll
    for (int k = 0; k < 5; ++k) a[k] = __ldg(reinterpret_cast<const V*>(p + (size_t)k * rs));
    use(j, a);
  }
}

// Per node slot p of the packed pattern: offset of its first row, row stride, own entries (padded),
// own entries in interior columns (padded; they come first), coupling entries (padded), and the
// positions of its codes in the two tables.
struct PkNode { int off, rs, own, own_int, cross, oc, cc; };
__device__ __forceinline__ PkNode pk_node(const int* __restrict__ tab, int p) {
  const int4 a = __ldg(reinterpret_cast<const int4*>(tab) + 2 * p), b = __ldg(reinterpret_cast<const int4*>(tab) + 2 * p + 1);
  return {a.x, a.y, a.z, a.w, b.x, b.y, b.z};
}

// Dense FP64 own blocks and FP64 couplings -> packed rows of type T; own entries outside the
// pattern must be zero (status <- SC_PACK_VIOLATION): a row's count of nonzero entries has to
// equal that of its packed ones.  With dense32 non-null (mixed arm) the same pass also writes the
// FP32 copy of the dense block (padding included) that the condensation products read.  One warp
// per row: the row goes through shared memory, so that both outputs are written in 16-byte
// pieces (9.5 ms for 25 GB at 16^3, N = 4; 8^3 meshes and smaller spread a block over several CTAs).
template <class T>
__global__ void __launch_bounds__(256) k_pack(Geo G, const double* __restrict__ Aown, const double* __restrict__ X,
                                              const int* __restrict__ node_tab, const int* __restrict__ own_code,
                                              const int* __restrict__ pptr, const int* __restrict__ iperm,
                                              T* __restrict__ Apk, long long pstride, int* __restrict__ status,
                                              float* __restrict__ dense32) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int e = blockIdx.x, lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  double* row = reinterpret_cast<double*>(smem_raw) + (size_t)warp * (G.lda + 4);
  const double* Ae = Aown + (size_t)e * own_stride(G);
  T* Pe = Apk + (size_t)e * pstride;
  bool bad = false;
  if (lane < 4) row[G.lda + lane] = 0.0;  // what the codes of padding entries name
  for (int r = blockIdx.y * nw + warp; r < G.ne; r += nw * gridDim.y) {
    const int p = r / 5, k = r - 5 * p;
    const PkNode nd = pk_node(node_tab, p);
    const int first = r < G.ni ? G.cb0 : 0;  // A_ii is not packed
    int nz = 0;
    __syncwarp();
    for (int c0 = 4 * lane; c0 < G.lda; c0 += 128) {
      const double2 a = __ldg(reinterpret_cast<const double2*>(Ae + (size_t)r * G.lda + c0));
      const double2 b = __ldg(reinterpret_cast<const double2*>(Ae + (size_t)r * G.lda + c0) + 1);
      reinterpret_cast<double2*>(row + c0)[0] = a;
      reinterpret_cast<double2*>(row + c0)[1] = b;
      if (c0 >= first) nz += (a.x != 0.0) + (a.y != 0.0) + (b.x != 0.0) + (b.y != 0.0);
      if (dense32)
        *reinterpret_cast<float4*>(dense32 + (size_t)e * own_stride(G) + (size_t)r * G.lda + c0) =
            make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    }
    __syncwarp();
    T* prow = Pe + nd.off + (size_t)k * nd.rs;
    auto put4 = [&](T* dst, const double v[4]) {
      if constexpr (std::is_same<T, float>::value) {
        *reinterpret_cast<float4*>(dst) = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
      } else {
        reinterpret_cast<double2*>(dst)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2*>(dst)[1] = make_double2(v[2], v[3]);
      }
    };
    for (int i = lane; 4 * i < nd.own; i += 32) {
      const int code = __ldg(own_code + nd.oc + i), t = group_split(i);
      double v[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        v[w] = row[(w < t ? (code & 0xffff) : (code >> 16)) + w];
        nz -= v[w] != 0.0;
      }
      put4(prow + 4 * i, v);
    }
    const int j = __ldg(iperm + p), q0 = __ldg(pptr + j), m = 5 * (__ldg(pptr + j + 1) - q0);
    const double* Xr = X + (((size_t)e * 5 + k) * G.NP + q0) * 5;
    for (int i = lane; 4 * i < nd.cross; i += 32) {
      double v[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) v[w] = 4 * i + w < m ? __ldg(Xr + 4 * i + w) : 0.0;
      put4(prow + nd.own + 4 * i, v);
    }
    bad = bad || __reduce_add_sync(0xffffffffu, nz) != 0;
  }
  if (bad && lane == 0) atomicCAS(status, -1, SC_PACK_VIOLATION);
}

// t = alpha B_i,e + beta (A_ib x_b)_e at the interior nodes warp, warp + step, ...; one warp per node.
template <class T>
__device__ __forceinline__ void interior_rows(const Geo& G, const T* __restrict__ Apk, long long pstride,
                                              const int* __restrict__ node_tab, const int* __restrict__ own_code,
                                              const int2* __restrict__ cross_code, const int* nbr_s,
                                              const int* __restrict__ iperm, const T* __restrict__ xb, double beta,
                                              const double* __restrict__ Bfull, double alpha, const T* v, T* t, bool own,
                                              int e, int first, int step, int lane) {
  const T* Pe = Apk + (size_t)e * pstride;
  const int mine = wsum5_owner(lane);
  for (int p = first; p < G.nin; p += step) {
    T sum = T(0);
    if (xb) {
      const PkNode nd = pk_node(node_tab, p);
      T acc[5] = {T(0), T(0), T(0), T(0), T(0)};
      node_rows5(Pe + nd.off, nd.rs, nd.own, own ? nd.own : 0, nd.cross, own_code + nd.oc, cross_code + nd.cc, v, nbr_s,
                 G.nb, G.ni, xb, T(1), (const T*)nullptr, T(0), lane, acc);
      sum = wsum5(acc, lane);
    }
    if (mine >= 0) {
      T val = T(beta) * sum;
      if (Bfull) val += T(alpha * Bfull[((size_t)e * G.nn + __ldg(iperm + p)) * 5 + mine]);
      t[5 * p + mine] = val;
    }
  }
}

// u rows = A_ii^-1 t, t (ldi values, zero padded) in shared memory: eight lanes per row, four rows
// per warp, rows 4 first .. of a stride of 4 step.
template <class T>
__device__ __forceinline__ void interior_apply(const Geo& G, const T* __restrict__ Ie, const T* t, T* __restrict__ ue,
                                               int first, int step, int lane) {
  using V = typename PkVec<T>::type;
  constexpr int W = PkVec<T>::n;
  const int sub = lane & 7;
  for (int r0 = 4 * first; r0 < G.ni; r0 += 4 * step) {
    const int r = r0 + (lane >> 3);
    T s0 = T(0), s1 = T(0);
    if (r < G.ni) {
      const T* row = Ie + (size_t)r * G.ldi;
#pragma unroll 5
      for (int j = sub * W; j < G.ldi; j += 8 * W) {
        const V a = __ldg(reinterpret_cast<const V*>(row + j));
        const V x = *reinterpret_cast<const V*>(t + j);
#pragma unroll
        for (int w = 0; w < W; w += 2) {
          s0 = fma(reinterpret_cast<const T*>(&a)[w], reinterpret_cast<const T*>(&x)[w], s0);
          s1 = fma(reinterpret_cast<const T*>(&a)[w + 1], reinterpret_cast<const T*>(&x)[w + 1], s1);
        }
      }
    }
    s0 += s1;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    if (sub == 0 && r < G.ni) ue[r] = s0;
  }
}

// black_zero: x_b is zero on the black elements (the red-black sweep), so their own A_ib x_b part
// is skipped and only the neighbour couplings feed their interior solve
__device__ __forceinline__ bool own_part(const Geo& G, int e, int black_zero) {
  return !(black_zero && ((e % G.n + (e / G.n) % G.n + e / (G.n * G.n)) & 1));
}

// Interior pass: u_e = A_ii,e^-1 (alpha B_i,e + beta (A_ib x_b)_e), both steps in one CTA per
// element.  HBM bound; meshes whose elements do not fill the chip take the two kernels below.
template <class T>
__global__ void __launch_bounds__(256, PkOcc<T>::v) k_cond_interior_pk(Geo G, const T* __restrict__ Apk,
    long long pstride, const int* __restrict__ node_tab, const int* __restrict__ own_code,
    const int2* __restrict__ cross_code, const int* __restrict__ nbr, const T* __restrict__ Ainv,
    const int* __restrict__ iperm, const T* __restrict__ xb, double beta, const double* __restrict__ Bfull,
    double alpha, T* __restrict__ u, int black_zero) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int e = blockIdx.x, ni = G.ni, nb = G.nb, lda = G.lda, ldi = G.ldi;
  T* v = reinterpret_cast<T*>(smem_raw);  // lda + 4: x_e at the boundary columns, zeros for padding
  T* t = v + lda + 4;                     // ldi: right-hand side of the interior solve
  __shared__ int nbr_s[18];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  if (threadIdx.x < 18) nbr_s[threadIdx.x] = nbr[e * 18 + threadIdx.x];
  for (int i = threadIdx.x; i < lda + 4; i += blockDim.x)
    v[i] = (xb && i >= G.cb0 && i < G.cb0 + nb) ? xb[(size_t)e * nb + i - G.cb0] : T(0);
  for (int i = ni + threadIdx.x; i < ldi; i += blockDim.x) t[i] = T(0);
  __syncthreads();
  interior_rows(G, Apk, pstride, node_tab, own_code, cross_code, nbr_s, iperm, xb, beta, Bfull, alpha, v, t,
                own_part(G, e, black_zero), e, warp, nw, lane);
  __syncthreads();
  interior_apply(G, Ainv + (size_t)e * ni * ldi, t, u + (size_t)e * ni, warp, nw, lane);
}

// The two steps of the interior pass spread over gridDim.x CTAs per element, t through memory
// (K x ldi).  gridDim.z vectors at once (the columns of a dense S): vector z is zx, zt, zu, zy
// entries behind the first.
template <class T>
__global__ void __launch_bounds__(256, PkOcc<T>::v) k_interior_rows(Geo G, const T* __restrict__ Apk, long long pstride,
    const int* __restrict__ node_tab, const int* __restrict__ own_code, const int2* __restrict__ cross_code,
    const int* __restrict__ nbr, const int* __restrict__ iperm, const T* __restrict__ xb, double beta,
    const double* __restrict__ Bfull, double alpha, T* __restrict__ t, int black_zero, long long zx, long long zt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int e = blockIdx.y, nb = G.nb;
  if (xb) xb += blockIdx.z * zx;
  t += blockIdx.z * zt;
  T* v = reinterpret_cast<T*>(smem_raw);
  __shared__ int nbr_s[18];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  if (threadIdx.x < 18) nbr_s[threadIdx.x] = nbr[e * 18 + threadIdx.x];
  for (int i = threadIdx.x; i < G.lda + 4; i += blockDim.x)
    v[i] = (xb && i >= G.cb0 && i < G.cb0 + nb) ? xb[(size_t)e * nb + i - G.cb0] : T(0);
  __syncthreads();
  interior_rows(G, Apk, pstride, node_tab, own_code, cross_code, nbr_s, iperm, xb, beta, Bfull, alpha, v,
                t + (size_t)e * G.ldi, own_part(G, e, black_zero), e, blockIdx.x * nw + warp, gridDim.x * nw, lane);
}

template <class T>
__global__ void __launch_bounds__(256, PkOcc<T>::v) k_interior_apply(Geo G, const T* __restrict__ Ainv,
                                                                     const T* __restrict__ t, T* __restrict__ u,
                                                                     long long zt, long long zu) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  t += blockIdx.z * zt;
  u += blockIdx.z * zu;
  T* ts = reinterpret_cast<T*>(smem_raw);
  const int e = blockIdx.y, lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  for (int i = threadIdx.x; i < G.ldi; i += blockDim.x) ts[i] = i < G.ni ? t[(size_t)e * G.ldi + i] : T(0);
  __syncthreads();
  interior_apply(G, Ainv + (size_t)e * G.ni * G.ldi, ts, u + (size_t)e * G.ni, blockIdx.x * nw + warp, gridDim.x * nw,
                 lane);
}

// Boundary pass: y_e = gamma B_b,e + delta (A_bb x_b)_e - (A_bi u)_e from the packed rows (delta
// x_b of boundary neighbours, -u of interior ones); one warp per boundary node (its 5 rows),
// gridDim.x CTAs per element.  HBM bound: at 16^3, N = 4 the passes over all elements and over the
// black ones average 0.38 ms (0.46 with scalar coupling loads, a decoded column list and 25
// shuffles per node; 9^3, N = 5: 0.15 against 0.22).
template <class T>
__global__ void __launch_bounds__(256, PkOcc<T>::v) k_cond_boundary_pk(Geo G, const T* __restrict__ Apk,
    long long pstride, const int* __restrict__ node_tab, const int* __restrict__ own_code,
    const int2* __restrict__ cross_code, const int* __restrict__ nbr, const int* __restrict__ iperm,
    const T* __restrict__ xb, double delta, const double* __restrict__ Bfull, double gamma_, const T* __restrict__ u,
    double* __restrict__ y, const int* __restrict__ elist, int own_zero, long long zx, long long zu, long long zy) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (xb) xb += blockIdx.z * zx;
  if (u) u += blockIdx.z * zu;
  y += blockIdx.z * zy;
  // CTA row i serves element elist[i] (one colour of the red-black sweep), or element i
  const int e = elist ? __ldg(elist + blockIdx.y) : blockIdx.y, ni = G.ni, nb = G.nb, lda = G.lda, cb0 = G.cb0;
  T* v = reinterpret_cast<T*>(smem_raw);  // lda + 4: [-u_e | 0 | delta x_e | 0]
  __shared__ int nbr_s[18];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  const T dT = T(delta);
  if (threadIdx.x < 18) nbr_s[threadIdx.x] = nbr[e * 18 + threadIdx.x];
  for (int i = threadIdx.x; i < lda + 4; i += blockDim.x) {
    T val = T(0);
    if (i < ni) { if (u) val = -u[(size_t)e * ni + i]; }
    else if (i >= cb0 && i < cb0 + nb) { if (xb) val = dT * xb[(size_t)e * nb + i - cb0]; }
    v[i] = val;
  }
  __syncthreads();
  const T* Pe = Apk + (size_t)e * pstride;
  const bool need = xb || u;
  const int mine = wsum5_owner(lane);
  for (int p = G.nin + blockIdx.x * nw + warp; p < G.nn; p += gridDim.x * nw) {
    T sum = T(0);
    if (need) {
      const PkNode nd = pk_node(node_tab, p);
      T acc[5] = {T(0), T(0), T(0), T(0), T(0)};
      // own_zero: the element's own boundary values are zero, only the interior columns count
      node_rows5(Pe + nd.off, nd.rs, nd.own, own_zero ? nd.own_int : nd.own, nd.cross, own_code + nd.oc,
                 cross_code + nd.cc, v, nbr_s, nb, ni, xb, dT, u, T(-1), lane, acc);
      sum = wsum5(acc, lane);
    }
    if (mine >= 0) {
      double val = (double)sum;
      if (Bfull) val += gamma_ * Bfull[((size_t)e * G.nn + __ldg(iperm + p)) * 5 + mine];
      y[(size_t)e * nb + 5 * (p - G.nin) + mine] = val;
    }
  }
}

// CTAs per element of a pass over `count` elements and `nodes` nodes (8 per CTA at a time): enough
// for four waves of the CTAs that reside at once, so that small meshes fill the chip and the last
// wave is short.  With one CTA per element the boundary pass took 0.32 ms for 216 elements of order
// 6 and 65 us for 64 of order 3 in FP64, now 0.137 ms (0.83 of HBM) and 19 us.
int pk_splits(int count, int nodes) {
  constexpr int kTarget = 4 * 6 * 152;
  return std::max(1, std::min((nodes + 7) / 8, (kTarget + count - 1) / count));
}

}  // namespace

namespace sc {

// Host tables of the packed layout (per mesh): per node slot the row geometry, and the codes of
// its own and coupling entries (see node_rows5).
void build_packed_pattern(sc_ctx* c) {
  const Geo& G = c->G;
  const int nn = G.nn, p1 = G.p;
  auto up4 = [](int x) { return (x + 3) & ~3; };
  auto nat = [&](int slot, int d) {
    const int m = c->iperm[slot];
    return d == 0 ? m % p1 : d == 1 ? (m / p1) % p1 : m / (p1 * p1);
  };
  c->pk_node.assign((size_t)8 * nn, 0);
  c->pk_own_code.clear();
  c->pk_cross_code.clear();
  c->pk_nnz_int = c->pk_nnz_bnd = 0;
  int off = 0;
  for (int p = 0; p < nn; ++p) {
    std::vector<int> cols;  // own column of variable 0 of every column node, interior nodes first
    int nint = 0;
    for (int q = 0; q < nn; ++q) {
      if (p < G.nin && q < G.nin) continue;  // A_ii: not packed
      if (!(nat(p, 0) == nat(q, 0) || nat(p, 1) == nat(q, 1) || nat(p, 2) == nat(q, 2))) continue;
      cols.push_back(own_col(G, q, 0));
      if (cols.back() < G.ni) nint += 5;
    }
    const int j = c->iperm[p], q0 = c->pat.ptr[j], nq = c->pat.ptr[j + 1] - q0;
    const int own = up4(5 * (int)cols.size()), cross = up4(5 * nq);
    int* nd = &c->pk_node[(size_t)8 * p];
    nd[0] = off; nd[1] = own + cross; nd[2] = own; nd[3] = up4(nint); nd[4] = cross;
    nd[5] = (int)c->pk_own_code.size(); nd[6] = (int)c->pk_cross_code.size() / 2;
    off += 5 * (own + cross);
    (p < G.nin ? c->pk_nnz_int : c->pk_nnz_bnd) += 25 * (long long)cols.size();
    // a group of four starts in variable l0 of node n0 and enters the next node at entry 5 - l0
    for (int i = 0; 4 * i < own; ++i) {
      const int n0 = 4 * i / 5, l0 = 4 * i % 5, t = 5 - l0;
      const int b0 = cols[n0] + l0;
      const int b1 = (n0 + 1 < (int)cols.size() ? cols[n0 + 1] : G.lda) - t;  // lda: the zeros for padding
      c->pk_own_code.push_back((int)((unsigned)b1 << 16 | (unsigned)b0));
    }
    auto pair_code = [&](int q, int shift) {
      if (q >= nq) return 31 << 26;
      const int pos = c->perm[c->pat.col[q0 + q]], interior = pos < G.nin ? 1 : 0;
      const int o = (interior ? 5 * pos : 5 * (pos - G.nin)) + shift + 8;
      return (c->pat.slot[q0 + q] << 26) | (interior << 25) | o;
    };
    for (int i = 0; 4 * i < cross; ++i) {
      const int n0 = 4 * i / 5, l0 = 4 * i % 5;
      c->pk_cross_code.push_back(pair_code(n0, l0));
      c->pk_cross_code.push_back(pair_code(n0 + 1, l0 - 5));
    }
  }
  c->pk_stride = off;
}

cudaError_t upload_packed_pattern(sc_ctx* c) {
  auto up = [](int* d, const std::vector<int>& h) {
    return cudaMemcpy(d, h.data(), h.size() * sizeof(int), cudaMemcpyHostToDevice);
  };
  cudaError_t e = up(c->d_pk_node, c->pk_node);
  if (e == cudaSuccess) e = up(c->d_pk_own_code, c->pk_own_code);
  if (e == cudaSuccess) e = up(c->d_pk_cross_code, c->pk_cross_code);
  return e;
}

// Pack the FP64 own blocks and couplings into the operator's precision (mixed arm: and write the
// dense blocks' FP32 copy).
template <class T>
static cudaError_t pack_t(sc_ctx* c, T* Apk, float* dense32) {
  const Geo& G = c->G;
  const size_t smem = (size_t)8 * (G.lda + 4) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_pack<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       8 * (kMaxLda + 4) * (int)sizeof(double));
  if (e != cudaSuccess) return e;
  count_launch(c);
  const int split = std::max(1, std::min((G.ne + 7) / 8, (4 * 152 * 4 + G.K - 1) / G.K));
  k_pack<T><<<dim3(G.K, split), 256, smem, c->stream>>>(G, c->Aown, c->X, c->d_pk_node, c->d_pk_own_code, c->d_pptr,
                                                        c->d_iperm, Apk, c->pk_stride, c->d_status, dense32);
  return cudaGetLastError();
}

cudaError_t pack_own(sc_ctx* c) {
  return c->cfg.precision == SC_PREC_MIXED ? pack_t<float>(c, c->Apk32, c->Aown32) : pack_t<double>(c, c->Apk, nullptr);
}

template <class T>
cudaError_t cond_interior_pk(sc_ctx* c, const T* Apk, const T* Ainv, const T* xb, double beta, const double* Bfull,
                             double alpha, T* u, int black_zero) {
  const Geo& G = c->G;
  const int2* cc = reinterpret_cast<const int2*>(c->d_pk_cross_code);
  // the rows have nin nodes, A_ii^-1 ni / 4 groups of rows: split by the larger need
  const int s1 = pk_splits(G.K, G.nin), s2 = pk_splits(G.K, (G.ni + 3) / 4);
  if (s2 == 1) {
    const size_t smem = (size_t)(G.lda + 4 + G.ldi) * sizeof(T);
    k_cond_interior_pk<T><<<G.K, 256, smem, c->stream>>>(G, Apk, c->pk_stride, c->d_pk_node, c->d_pk_own_code, cc,
                                                         c->d_nbr, Ainv, c->d_iperm, xb, beta, Bfull, alpha, u,
                                                         black_zero);
    return cudaGetLastError();
  }
  T* t = static_cast<T*>(c->row_t);
  count_launch(c);  // the profiled span counts one
  k_interior_rows<T><<<dim3(s1, G.K), 256, (size_t)(G.lda + 4) * sizeof(T), c->stream>>>(
      G, Apk, c->pk_stride, c->d_pk_node, c->d_pk_own_code, cc, c->d_nbr, c->d_iperm, xb, beta, Bfull, alpha, t,
      black_zero, 0, 0);
  k_interior_apply<T><<<dim3(s2, G.K), 256, (size_t)G.ldi * sizeof(T), c->stream>>>(G, Ainv, t, u, 0, 0);
  return cudaGetLastError();
}

template <class T>
static cudaError_t boundary_launch(sc_ctx* c, const T* Apk, const T* xb, double delta, const double* Bfull,
                                   double gamma_, const T* u, double* y, const int* elist, int count, int own_zero) {
  const Geo& G = c->G;
  k_cond_boundary_pk<T><<<dim3(pk_splits(count, G.nbn), count), 256, (size_t)(G.lda + 4) * sizeof(T), c->stream>>>(
      G, Apk, c->pk_stride, c->d_pk_node, c->d_pk_own_code, reinterpret_cast<const int2*>(c->d_pk_cross_code), c->d_nbr,
      c->d_iperm, xb, delta, Bfull, gamma_, u, y, elist, own_zero, 0, 0, 0);
  return cudaGetLastError();
}

template <class T>
cudaError_t cond_boundary_pk(sc_ctx* c, const T* Apk, const T* xb, double delta, const double* Bfull, double gamma_,
                             const T* u, double* y) {
  return boundary_launch<T>(c, Apk, xb, delta, Bfull, gamma_, c->G.ni ? u : nullptr, y, nullptr, c->G.K, 0);
}

// y_z = S x_z for m vectors at once (each K nb long, one behind the other; t: m K ldi, u: m K ni values
// of scratch): a single vector's passes leave the chip mostly idle on the small meshes whose S is
// formed densely (27 elements of order 3: 26 us and five launches per column, one vector at a time).
template <class T>
cudaError_t cond_columns_pk(sc_ctx* c, const T* Apk, const T* Ainv, const T* xb, T* t, T* u, double* y, int m) {
  const Geo& G = c->G;
  const int2* cc = reinterpret_cast<const int2*>(c->d_pk_cross_code);
  const long long zx = (long long)G.K * G.nb, zt = (long long)G.K * G.ldi, zu = (long long)G.K * G.ni;
  const int work = m * G.K;
  if (G.ni > 0) {
    count_launch(c, 2);
    k_interior_rows<T><<<dim3(pk_splits(work, G.nin), G.K, m), 256, (size_t)(G.lda + 4) * sizeof(T), c->stream>>>(
        G, Apk, c->pk_stride, c->d_pk_node, c->d_pk_own_code, cc, c->d_nbr, c->d_iperm, xb, 1.0, nullptr, 0.0, t, 0, zx, zt);
    k_interior_apply<T><<<dim3(pk_splits(work, (G.ni + 3) / 4), G.K, m), 256, (size_t)G.ldi * sizeof(T), c->stream>>>(
        G, Ainv, t, u, zt, zu);
  }
  count_launch(c);
  k_cond_boundary_pk<T><<<dim3(pk_splits(work, G.nbn), G.K, m), 256, (size_t)(G.lda + 4) * sizeof(T), c->stream>>>(
      G, Apk, c->pk_stride, c->d_pk_node, c->d_pk_own_code, cc, c->d_nbr, c->d_iperm, xb, 1.0, nullptr, 0.0,
      G.ni ? u : nullptr, y, nullptr, 0, zx, zu, zx);
  return cudaGetLastError();
}
template cudaError_t cond_columns_pk<float>(sc_ctx*, const float*, const float*, const float*, float*, float*, double*, int);
template cudaError_t cond_columns_pk<double>(sc_ctx*, const double*, const double*, const double*, double*, double*,
                                             double*, int);

// y_e = (A_bb x_b)_e - (A_bi u)_e for the elements of a list only (rows of one colour), whose
// own boundary values in x_b are zero (the black elements in the red-black sweep): their packed
// rows are read in the interior columns and the couplings only.
template <class T>
cudaError_t cond_boundary_pk_list(sc_ctx* c, const T* Apk, const T* xb, const T* u, double* y, const int* elist,
                                  int nlist) {
  if (nlist <= 0) return cudaSuccess;
  ProfScope ps(c, SCK_COND_BOUNDARY, nlist);
  return boundary_launch<T>(c, Apk, xb, 1.0, nullptr, 0.0, c->G.ni ? u : nullptr, y, elist, nlist, 1);
}
template cudaError_t cond_boundary_pk_list<float>(sc_ctx*, const float*, const float*, const float*, double*, const int*,
                                                  int);
template cudaError_t cond_boundary_pk_list<double>(sc_ctx*, const double*, const double*, const double*, double*,
                                                   const int*, int);
template cudaError_t cond_interior_pk<float>(sc_ctx*, const float*, const float*, const float*, double, const double*,
                                             double, float*, int);
template cudaError_t cond_interior_pk<double>(sc_ctx*, const double*, const double*, const double*, double,
                                              const double*, double, double*, int);
template cudaError_t cond_boundary_pk<float>(sc_ctx*, const float*, const float*, double, const double*, double,
                                             const float*, double*);
template cudaError_t cond_boundary_pk<double>(sc_ctx*, const double*, const double*, double, const double*, double,
                                              const double*, double*);

}  // namespace sc
