// Residual and Jacobian assembly of the GL-DGSEM Newton system on the GPU.
//
// Residual (Sec. 2.1, eq. DGSEMsystem, in the strong form that summation by parts
// gives on Gauss-Lobatto nodes):
//   g_a(m) = (2/h) [ sum_b D[m_a][b] q(m with coord a = b)
//                    + (1/w_N) (1/2)(q_nb - q_m)  on the +a face, - on the -a face ]   (BR1)
//   R_j = c0 J W_j (q_j - q_hist)/dt + Jf W_j sum_a sum_b D[j_a][b] F_a(m_b)
//         + sum_{faces f of j} Jf W^f_j [ fhat_f(j) - s_f F_{d_f}(j) ]
// with F = f^a - f^nu, fhat = Roe(q+, q-) - (1/2) s (f^nu_d(+) + f^nu_d(-)), J = (h/2)^3,
// Jf = (h/2)^2, W_j the tensor GL weight.  With the symmetric interior penalty (the paper's
// experiment, Sec. 4) the face flux takes f^nu at each side's own unlifted gradient
// Dq = (2/h) sum_b D[m_a][b] q(...) instead of the lifted one and adds sigma (q+ - q-); the
// volume flux F keeps the lifted gradient (qhat = {{q}}), which supplies the symmetrising
// term.  The unlifted gradients depend on their own element only, so the edge-neighbour
// couplings of BR1 vanish.
//
// Jacobian (Sec. 2.1.1-2.1.2, eqs. AdvImpDG, DiffImpDGouter, GradDGImp): the point flux
// Jacobians dF_d/dq, df^nu_d/dq and df^nu_d/dg_a, and the Roe derivatives, are
// evaluated per node with a five-direction dual number; the element blocks then follow
// from the chain rule through the (linear) lifting operator, which is non-zero only
// along grid lines:
//   dR_j/dq_r = delta_jr c0 J W_j/dt
//     + sum_d sum_{m on the d-line of j} Jf W_j D[j_d][m_d] [ delta_mr dF_d/dq(m)
//                                            + sum_a L_a(m, r) dF_d/dg_a(m) ]
//     + surface terms of the faces of j (own and neighbour lifting, Roe derivatives).
// L_a(m, r) = (2/h) D[m_a][r_a] (r on the a-line of m) + 1/(h w_N) (-[m_a = N] + [m_a = 0])
// for r = m, and +- 1/(h w_N) for the neighbour node across the a-face.
#include "sc_internal.cuh"

namespace {

constexpr int NJC = 375;  // node Jacobian components: Fq(3x25) | fvq(3x25) | fvg(9x25)

SC_HD inline void node_coords(int m, int p, int c[3]) {
  c[0] = m % p; c[1] = (m / p) % p; c[2] = m / (p * p);
}
SC_HD inline int node_index(const int c[3], int p) { return c[0] + p * (c[1] + p * c[2]); }

__global__ void k_history(Geo G, const double* __restrict__ Qs, const double* __restrict__ Qsm1,
                          double* __restrict__ Qh, size_t n, int bdf) {
  size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  Qh[t] = (bdf == 2) ? (4.0 * Qs[t] - Qsm1[t]) / 3.0 : Qs[t];
}

// ---- residual ---------------------------------------------------------------------------
// Two kernels, one thread per node, CTAs of whole elements (four of order 2, two of order 3, else
// one) whose values sit in shared memory:
//   k_point  lifted gradients and point fluxes F_d = f^a_d - f^nu_d, and the dissipation of the
//            numerical flux on the element's three faces in positive direction
//   k_rows   rows of the residual: divergence lines, face terms, and what becomes of them
// Face terms: with the central part of the numerical flux s (f^a(+) + f^a(-)) / 2 and the viscous
// average s (f^nu(+) + f^nu(-)) / 2, fhat = s (F(+) + F(-)) / 2 - diss / 2 with the point fluxes
// that are there already, and diss changes its sign with the side: a pair of face nodes costs one
// dissipation and no viscous flux.  Face nodes are their own work items, summed by their nodes
// afterwards.  FP64-pipe bound: 61 + 30 us per Runge-Kutta stage at 8^3, N = 4 (the
// stage's update included; 46 + 54 us with a dissipation per side, evaluated in k_rows) against 22 + 22 +
// 215 + 16 us in five kernels with one thread per node doing its up to three faces (Roe and two
// viscous fluxes each, 16 % of the warps resident).
inline int group_elems(const Geo& G) { return G.nn <= 32 ? 4 : G.nn <= 64 ? 2 : 1; }
inline int group_threads(const Geo& G) { return (group_elems(G) * G.nn + 31) / 32 * 32; }

// Fluxes F_d = f^a_d - f^nu_d of one node along all directions.
__device__ __forceinline__ void point_fluxes(const Geo& G, const double q[5], const double g[3][5], double F[3][5]) {
  flux_viscous_all(G, q, g, F);
  const double ir = 1.0 / q[0];
  const double u[3] = {q[1] * ir, q[2] * ir, q[3] * ir};
  const double pr = (G.gamma - 1.0) * (q[4] - 0.5 * (q[1] * u[0] + q[2] * u[1] + q[3] * u[2]));
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    F[d][0] = q[1 + d] - F[d][0];
#pragma unroll
    for (int i = 0; i < 3; ++i) F[d][1 + i] = q[1 + i] * u[d] + (i == d ? pr : 0.0) - F[d][1 + i];
    F[d][4] = (q[4] + pr) * u[d] - F[d][4];
  }
}

__device__ __forceinline__ double warp_max_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// Non-negative doubles order like their bit patterns; NaN is mapped to +inf.
__device__ __forceinline__ void warp_max_into(double v, unsigned long long* out) {
  v = warp_max_d(v == v ? v : INFINITY);
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(v));
}

// Values of each thread (n per node) through shared memory to out[node][n], coalesced.
template <int n>
__device__ __forceinline__ void store_nodes(const double (&v)[n], double* buf, double* __restrict__ out, size_t first,
                                            int nodes, bool live) {
  __syncthreads();
  if (live)
#pragma unroll
    for (int i = 0; i < n; ++i) buf[threadIdx.x * n + i] = v[i];
  __syncthreads();
  for (int i = threadIdx.x; i < nodes * n; i += blockDim.x) out[first * n + i] = buf[i];
}

// Face node ia = a + p b of the faces normal to d: node m at the lower end, sd from one layer to the next.
struct FaceNode {
  int m, sd;
  __device__ __forceinline__ FaceNode(int p, int d, int ia) {
    sd = d == 0 ? 1 : d == 1 ? p : p * p;
    m = ia % p * (d == 0 ? p : 1) + ia / p * (d == 2 ? p : p * p);
  }
};

// spd (or null): the largest signal speed |v| + c and the largest diffusivity
// max(4/3, gamma/Pr) mu / (rho Re) of all nodes, folded in as bit patterns.
template <bool IP>
__global__ void __launch_bounds__(352) k_point(Geo G, int ge, const double* __restrict__ Q, const int* __restrict__ nbr,
                                               double* __restrict__ F, double* __restrict__ grad,
                                               double* __restrict__ Floc, double* __restrict__ gloc,
                                               double* __restrict__ diss, unsigned long long* __restrict__ spd) {
  extern __shared__ __align__(16) double sm[];
  const int p = G.p, N = G.N, nn = G.nn, e0 = blockIdx.x * ge, ne = min(ge, G.K - e0), nodes = ne * nn;
  double* Ds = sm;               // p x p
  double* qs = Ds + 64;          // [nodes][5]
  double* buf = qs + ge * nn * 5;  // [nodes][15]
  const size_t first = (size_t)e0 * nn;
  for (int i = threadIdx.x; i < p * p; i += blockDim.x) Ds[i] = G.D[i / p][i % p];
  for (int i = threadIdx.x; i < nodes * 5; i += blockDim.x) qs[i] = Q[first * 5 + i];
  __syncthreads();
  for (int i = threadIdx.x; i < ne * 3 * p * p; i += blockDim.x) {  // diss[e][d][face node]
    const int el = i / (3 * p * p), d = i / (p * p) % 3, ia = i % (p * p);
    const FaceNode fn(p, d, ia);
    const int m = fn.m + N * fn.sd;
    const size_t tn = (size_t)__ldg(nbr + (e0 + el) * 18 + 2 * d + 1) * nn + fn.m;
    const int kk[5] = {0, 1 + d, d == 0 ? 2 : 1, d == 2 ? 2 : 3, 4};  // normal momentum first
    double ra[5], rb[5], o[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) { ra[k] = qs[(el * nn + m) * 5 + kk[k]]; rb[k] = __ldg(Q + tn * 5 + kk[k]); }
    adv_dissipation_x(G, ra, rb, 1.0, o);
#pragma unroll
    for (int k = 0; k < 5; ++k) diss[(((size_t)e0 * 3) * p * p + i) * 5 + kk[k]] = o[k];
  }
  const bool live = threadIdx.x < nodes;
  const int t = live ? threadIdx.x : 0, el = t / nn, m = t - el * nn, e = e0 + el;
  const double* qe = qs + el * nn * 5;
  const int c[3] = {m % p, (m / p) % p, m / (p * p)};
  double q[5], g[15], gl[15];
#pragma unroll
  for (int k = 0; k < 5; ++k) q[k] = qe[m * 5 + k];
  const int stride[3] = {1, p, p * p};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double acc[5] = {0, 0, 0, 0, 0};
    const double* line = qe + (m - c[a] * stride[a]) * 5;
    for (int b = 0; b < p; ++b) {
      const double Dab = Ds[c[a] * p + b];
#pragma unroll
      for (int k = 0; k < 5; ++k) acc[k] = fma(Dab, line[b * stride[a] * 5 + k], acc[k]);
    }
    if (IP)
#pragma unroll
      for (int k = 0; k < 5; ++k) gl[a * 5 + k] = G.dx * acc[k];
    if (live && (c[a] == N || c[a] == 0)) {
      const int s = c[a] == N ? 1 : -1;
      const int nb = __ldg(nbr + e * 18 + face_slot(a, s));
      const double* qn = Q + ((size_t)nb * nn + m + (N - 2 * c[a]) * stride[a]) * 5;
      const double coef = 0.5 * s / G.w[0];  // the end weights are equal
#pragma unroll
      for (int k = 0; k < 5; ++k) acc[k] = fma(coef, __ldg(qn + k) - q[k], acc[k]);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) g[a * 5 + k] = G.dx * acc[k];
  }
  if (grad) store_nodes(g, buf, grad, first, nodes, live);
  double f[15];
  point_fluxes(G, q, reinterpret_cast<const double(*)[5]>(g), reinterpret_cast<double(*)[5]>(f));
  store_nodes(f, buf, F, first, nodes, live);
  if (IP) {
    store_nodes(gl, buf, gloc, first, nodes, live);
    point_fluxes(G, q, reinterpret_cast<const double(*)[5]>(gl), reinterpret_cast<double(*)[5]>(f));
    store_nodes(f, buf, Floc, first, nodes, live);
  }
  if (spd) {
    const double ir = 1.0 / q[0];
    const double u = q[1] * ir, v = q[2] * ir, w = q[3] * ir, vv = u * u + v * v + w * w;
    const double pr = (G.gamma - 1.0) * (q[4] - 0.5 * q[0] * vv);
    double mu = 1.0;
    if (G.sutherland) {
      const double T = G.gamma * G.Ma * G.Ma * pr * ir;
      mu = (1.0 + G.Ts) * T * sqrt(T) / (T + G.Ts);
    }
    warp_max_into(sqrt(vv) + sqrt(G.gamma * pr * ir), spd);
    warp_max_into(fmax(4.0 / 3.0, G.gamma / G.Pr) / G.Re * mu * ir, spd + 1);
  }
}

// Rows of the residual.  RK = false: out = -R(Q); RK = true: the Runge-Kutta stage st with
// rhs = -M^-1 H(Q), out the stage's new state.
template <bool IP, bool RK>
__global__ void __launch_bounds__(352) k_rows(Geo G, int ge, const double* __restrict__ Q, const double* __restrict__ Qh,
                                              const double* __restrict__ F, const double* __restrict__ Floc,
                                              const double* __restrict__ diss, const int* __restrict__ nbr,
                                              double* __restrict__ out, sc::RkStage st) {
  extern __shared__ __align__(16) double sm[];
  const int p = G.p, N = G.N, nn = G.nn, pp = p * p, e0 = blockIdx.x * ge, ne = min(ge, G.K - e0), nodes = ne * nn;
  double* Ds = sm;                   // p x p
  double* qs = Ds + 64;              // [nodes][5]
  double* Fs = qs + ge * nn * 5;     // [nodes][15]
  double* fs = Fs + ge * nn * 15;    // [ge][6][pp][5]: face terms fhat - s F_d
  const size_t first = (size_t)e0 * nn;
  for (int i = threadIdx.x; i < p * p; i += blockDim.x) Ds[i] = G.D[i / p][i % p];
  for (int i = threadIdx.x; i < nodes * 5; i += blockDim.x) qs[i] = Q[first * 5 + i];
  for (int i = threadIdx.x; i < nodes * 15; i += blockDim.x) Fs[i] = F[first * 15 + i];
  __syncthreads();
  for (int i = threadIdx.x; i < ne * 6 * pp; i += blockDim.x) {
    const int el = i / (6 * pp), f = i / pp % 6, ia = i % pp, d = f >> 1, s = (f & 1) ? 1 : -1;
    const FaceNode fn(p, d, ia);
    const int m = fn.m + (s > 0 ? N : 0) * fn.sd, nb = __ldg(nbr + (e0 + el) * 18 + f);
    const size_t tn = (size_t)nb * nn + fn.m + (s > 0 ? 0 : N) * fn.sd;
    const double* Fa = Fs + (el * nn + m) * 15 + d * 5;
    const double* Fb = (IP ? Floc : F) + tn * 15 + d * 5;
    const double* ds = diss + (((size_t)(s > 0 ? e0 + el : nb) * 3 + d) * pp + ia) * 5;
    double* o = fs + (size_t)i * 5;
    double fb[5], dk[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) { fb[k] = __ldg(Fb + k); dk[k] = __ldg(ds + k); }
    if (IP) {
      const double* Fl = Floc + (first + el * nn + m) * 15 + d * 5;
      const double* qa = qs + (el * nn + m) * 5;
#pragma unroll
      for (int k = 0; k < 5; ++k)
        o[k] = 0.5 * s * (__ldg(Fl + k) + fb[k] - dk[k]) + G.sigma * (qa[k] - __ldg(Q + tn * 5 + k)) - s * Fa[k];
    } else {
#pragma unroll
      for (int k = 0; k < 5; ++k) o[k] = 0.5 * s * (fb[k] - Fa[k] - dk[k]);
    }
  }
  __syncthreads();
  const bool live = threadIdx.x < nodes;
  const int t = live ? threadIdx.x : 0, el = t / nn, m = t - el * nn;
  const int c[3] = {m % p, (m / p) % p, m / pp};
  const int stride[3] = {1, p, pp};
  const double Wj = G.w[c[0]] * G.w[c[1]] * G.w[c[2]];
  double r[5] = {0, 0, 0, 0, 0};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double* line = Fs + (el * nn + m - c[d] * stride[d]) * 15 + d * 5;
    for (int b = 0; b < p; ++b) {
      const double coef = Ds[c[d] * p + b];
#pragma unroll
      for (int k = 0; k < 5; ++k) r[k] = fma(coef, line[b * stride[d] * 15 + k], r[k]);
    }
    if (c[d] == 0 || c[d] == N) {
      const int f = face_slot(d, c[d] == N ? 1 : -1);
      const int ia = d == 0 ? c[1] + p * c[2] : d == 1 ? c[0] + p * c[2] : c[0] + p * c[1];
      const double* o = fs + ((size_t)(el * 6 + f) * pp + ia) * 5;
      const double iw = 1.0 / G.w[0];
#pragma unroll
      for (int k = 0; k < 5; ++k) r[k] = fma(iw, o[k], r[k]);
    }
  }
  // r is now the strong-form divergence over (h/2)^2 W_j per row: R = (h/2)^2 W_j r + time term
  const double* q = qs + t * 5;
  double y[5];
  if (!RK) {
    const double tcoef = G.c0 * G.Jf * 0.5 * G.h * Wj / G.dt, JW = G.Jf * Wj;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double h = G.c0 != 0.0 ? __ldg(Qh + (first + t) * 5 + k) : q[k];
      y[k] = -fma(JW, r[k], tcoef * (q[k] - h));
    }
  } else {
    double dt;
    if (st.first) {
      const double smax = __longlong_as_double((long long)st.spd[0]), nmax = __longlong_as_double((long long)st.spd[1]);
      const double dx = G.h / G.N;
      dt = st.cfl * dx / smax;
      if (st.dfl > 0.0 && nmax > 0.0) dt = fmin(dt, st.dfl * dx * dx / nmax);
      if (blockIdx.x == 0 && threadIdx.x == 0) *st.dt = dt;
    } else {
      dt = *st.dt;
    }
    double mx = 0.0;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double rhs = -G.dx * r[k];  // M_jj = (h/2)^3 W_j
      mx = rhs == rhs ? fmax(mx, fabs(rhs)) : INFINITY;
      const size_t i = (first + t) * 5 + k;
      double dq = dt * rhs;
      if (st.a != 0.0 && live) dq = fma(st.a, st.dq[i], dq);
      if (live) st.dq[i] = dq;
      y[k] = fma(st.b, dq, q[k]);
    }
    if (st.rmax) warp_max_into(live ? mx : 0.0, st.rmax);
  }
  store_nodes(y, Fs, out, first, nodes, live);
}

SC_HD inline void load_node(const double* __restrict__ Q, const double* __restrict__ grad,
                                          size_t t, double q[5], double g[3][5]) {
  for (int k = 0; k < 5; ++k) q[k] = Q[t * 5 + k];
  for (int a = 0; a < 3; ++a)
    for (int k = 0; k < 5; ++k) g[a][k] = grad[t * 15 + a * 5 + k];
}

// Point flux Jacobians of every node: NJ[e][comp][m].
SC_HD void nodejac_body(const Geo& G, const double* Q, const double* grad, int t, double* NJ) {
  const int e = t / G.nn, m = t % G.nn;
  double q[5], g[3][5];
  load_node(Q, grad, t, q, g);
  double* out = NJ + (size_t)e * NJC * G.nn + m;
  const size_t cs = G.nn;  // component stride
  {
    D5 qd[5], gd[3][5], fa[5], fv[3][5];
    for (int k = 0; k < 5; ++k) { qd[k] = D5(q[k]); qd[k].d[k] = 1.0; }
    for (int a = 0; a < 3; ++a)
      for (int k = 0; k < 5; ++k) gd[a][k] = D5(g[a][k]);
    flux_viscous_all(G, qd, gd, fv);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      flux_inviscid(G, qd, d, fa);
      for (int k = 0; k < 5; ++k)
        for (int l = 0; l < 5; ++l) {
          out[(size_t)(d * 25 + k * 5 + l) * cs] = fa[k].d[l] - fv[d][k].d[l];
          out[(size_t)(75 + d * 25 + k * 5 + l) * cs] = fv[d][k].d[l];
        }
    }
  }
#pragma unroll
  for (int ap = 0; ap < 3; ++ap) {
    D5 qd[5], gd[3][5], fv[3][5];
    for (int k = 0; k < 5; ++k) qd[k] = D5(q[k]);
    for (int a = 0; a < 3; ++a)
      for (int k = 0; k < 5; ++k) {
        gd[a][k] = D5(g[a][k]);
        if (a == ap) gd[a][k].d[k] = 1.0;
      }
    flux_viscous_all(G, qd, gd, fv);
    for (int d = 0; d < 3; ++d)
      for (int k = 0; k < 5; ++k)
        for (int l = 0; l < 5; ++l) out[(size_t)(150 + (d * 3 + ap) * 25 + k * 5 + l) * cs] = fv[d][k].d[l];
  }
}

__global__ void k_nodejac(Geo G, const double* __restrict__ Q, const double* __restrict__ grad,
                          double* __restrict__ NJ) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < G.K * G.nn) nodejac_body(G, Q, grad, t, NJ);
}

// Numerical-flux (Roe or Lax-Friedrichs) derivatives at every face node of every element: RJ[e][f][comp][fidx],
// comp < 25: d fhat/d q+, comp >= 25: d fhat/d q-; fidx = a + p*b over the in-face
// coordinates ((d+1)%3, (d+2)%3).
SC_HD void roejac_body(const Geo& G, const double* Q, const int* nbr, int t, double* RJ) {
  const int pp = G.p * G.p;
  const int e = t / (6 * pp), f = (t / pp) % 6, fidx = t % pp;
  const int d = f / 2, s = (f & 1) ? 1 : -1, N = G.N, p = G.p;
  int c[3]; c[d] = s > 0 ? N : 0; c[(d + 1) % 3] = fidx % p; c[(d + 2) % 3] = fidx / p;
  const int j = node_index(c, p);
  int cn[3] = {c[0], c[1], c[2]}; cn[d] = N - c[d];
  const int nb = nbr[e * 18 + f];
  const double* qa = Q + ((size_t)e * G.nn + j) * 5;
  const double* qb = Q + ((size_t)nb * G.nn + node_index(cn, p)) * 5;
  double* out = RJ + ((size_t)e * 6 + f) * 50 * pp + fidx;
  for (int side = 0; side < 2; ++side) {
    D5 a[5], b[5], fh[5];
    for (int k = 0; k < 5; ++k) { a[k] = D5(qa[k]); b[k] = D5(qb[k]); }
    for (int k = 0; k < 5; ++k) (side == 0 ? a : b)[k].d[k] = 1.0;
    flux_adv(G, a, b, d, s, fh);
    for (int k = 0; k < 5; ++k)
      for (int l = 0; l < 5; ++l) out[(size_t)(side * 25 + k * 5 + l) * pp] = fh[k].d[l];
  }
}

__global__ void k_roejac(Geo G, const double* __restrict__ Q, const int* __restrict__ nbr,
                         double* __restrict__ RJ) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < G.K * 6 * G.p * G.p) roejac_body(G, Q, nbr, t, RJ);
}

// ---- assembly helpers (all data of one element e) --------------------------------
struct ElemView {
  const double* nj;  // NJ of the element
  int nn;
  SC_HD inline double Fq(int d, int m, int kl) const { return nj[(size_t)(d * 25 + kl) * nn + m]; }
  SC_HD inline double fvq(int d, int m, int kl) const { return nj[(size_t)(75 + d * 25 + kl) * nn + m]; }
  SC_HD inline double fvg(int d, int a, int m, int kl) const {
    return nj[(size_t)(150 + (d * 3 + a) * 25 + kl) * nn + m];
  }
};

// Own-lifting coefficient L_a(m, r) for r on the a-line of m (same element).
SC_HD inline double lift_own(const Geo& G, const int cm[3], const int cr[3], int a, bool same) {
  double v = G.dx * G.D[cm[a]][cr[a]];
  if (same) {
    if (cm[a] == G.N) v -= G.inv_hw;
    if (cm[a] == 0) v += G.inv_hw;
  }
  return v;
}

SC_HD inline double wprod(const Geo& G, const int c[3]) { return G.w[c[0]] * G.w[c[1]] * G.w[c[2]]; }

// acc += coef * M where M is a 5x5 component set read through fn(kl)
#define ACC25(coef, EXPR)                                  \
  do {                                                     \
    const double _c = (coef);                              \
    if (_c != 0.0) {                                       \
      _Pragma("unroll") for (int kl = 0; kl < 25; ++kl)    \
        acc[kl] = fma(_c, (EXPR), acc[kl]);                \
    }                                                      \
  } while (0)

// Own element block: rows j, columns r (both in element e).  NJL: the point-flux Jacobians at
// the unlifted gradients (interior penalty only; null with BR1).
template <bool IP>
SC_HD void own_entry(const Geo& G, const double* NJ, const double* NJL, const double* RJ, const int* nbr, int e,
                     int j, int r, double acc[25]) {
  const int nn = G.nn, p = G.p, N = G.N;
  ElemView V{NJ + (size_t)e * NJC * nn, nn};
  constexpr bool ip = IP;
  ElemView VL{ip ? NJL + (size_t)e * NJC * nn : nullptr, nn};
  const int pp = p * p;
  {
    int cj[3], cr[3];
    node_coords(j, p, cj); node_coords(r, p, cr);
    int ndiff = 0, dc[3];
    for (int a = 0; a < 3; ++a) if (cj[a] != cr[a]) dc[ndiff++] = a;
#pragma unroll
    for (int kl = 0; kl < 25; ++kl) acc[kl] = 0.0;
    if (ndiff < 3) {
      const double Wj = wprod(G, cj);
      const double Dwj = G.Jf * Wj;  // Dw_d(j, m) = Dwj * D[j_d][m_d]
      if (ndiff == 0) {
        const double tc = G.c0 * G.Jf * 0.5 * G.h * Wj / G.dt;
        for (int k = 0; k < 5; ++k) acc[k * 6] += tc;
        for (int d = 0; d < 3; ++d) {
          ACC25(Dwj * G.D[cj[d]][cj[d]], V.Fq(d, j, kl));
          int cm[3] = {cj[0], cj[1], cj[2]};
          for (int b = 0; b < p; ++b) {  // (d, d): m along the d-line
            cm[d] = b;
            const int m = node_index(cm, p);
            ACC25(Dwj * G.D[cj[d]][b] * lift_own(G, cm, cj, d, b == cj[d]), -V.fvg(d, d, m, kl));
          }
          for (int a = 0; a < 3; ++a) {  // (d, a != d): m = j
            if (a == d) continue;
            ACC25(Dwj * G.D[cj[d]][cj[d]] * lift_own(G, cj, cj, a, true), -V.fvg(d, a, j, kl));
          }
        }
      } else if (ndiff == 1) {
        const int cdir = dc[0];
        ACC25(Dwj * G.D[cj[cdir]][cr[cdir]], V.Fq(cdir, r, kl));
        int cm[3] = {cj[0], cj[1], cj[2]};
        for (int b = 0; b < p; ++b) {  // (c, c): m along the c-line
          cm[cdir] = b;
          const int m = node_index(cm, p);
          ACC25(Dwj * G.D[cj[cdir]][b] * lift_own(G, cm, cr, cdir, b == cr[cdir]), -V.fvg(cdir, cdir, m, kl));
        }
        for (int a = 0; a < 3; ++a) {
          if (a == cdir) continue;
          // (c, a): m = r
          ACC25(Dwj * G.D[cj[cdir]][cr[cdir]] * lift_own(G, cr, cr, a, true), -V.fvg(cdir, a, r, kl));
          // (a, c): m = j
          ACC25(Dwj * G.D[cj[a]][cj[a]] * lift_own(G, cj, cr, cdir, false), -V.fvg(a, cdir, j, kl));
        }
      } else {  // ndiff == 2
        const int c1 = dc[0], c2 = dc[1];
        for (int o = 0; o < 2; ++o) {
          const int d = o ? c2 : c1, a = o ? c1 : c2;
          int cm[3] = {cj[0], cj[1], cj[2]}; cm[d] = cr[d];
          const int m = node_index(cm, p);
          ACC25(Dwj * G.D[cj[d]][cr[d]] * lift_own(G, cm, cr, a, false), -V.fvg(d, a, m, kl));
        }
      }
      // surface terms of the faces containing j
      if (ndiff <= 1) {
        for (int df = 0; df < 3; ++df) {
          if (cj[df] != 0 && cj[df] != N) continue;
          const int sf = (cj[df] == N) ? 1 : -1;
          const double Sf = G.Jf * Wj / G.w[cj[df]];
          if constexpr (ip) {
            // fhat - s F_d(j): the strong-form term -s F_d(j) keeps the lifted gradient at j
            // (full weight), the face average -s/2 f^nu(q_j, Dq_j) takes the unlifted one
            // (Dq_a(j) = dx D[j_a][r_a] q_r along the a-line), and sigma (q_j - q_jm) adds
            // sigma on the diagonal
            if (ndiff == 0) {
              const int f = face_slot(df, sf);
              const int fidx = cj[(df + 1) % 3] + p * cj[(df + 2) % 3];
              const double* rj = RJ + ((size_t)e * 6 + f) * 50 * pp + fidx;
              ACC25(Sf, rj[(size_t)kl * pp] - sf * V.Fq(df, j, kl) - 0.5 * sf * VL.fvq(df, j, kl)
                            + (kl % 6 == 0 ? G.sigma : 0.0));
              for (int a = 0; a < 3; ++a) {
                ACC25(Sf * sf * lift_own(G, cj, cj, a, true), V.fvg(df, a, j, kl));
                ACC25(-0.5 * Sf * sf * G.dx * G.D[cj[a]][cj[a]], VL.fvg(df, a, j, kl));
              }
            } else {
              const int a = dc[0];
              ACC25(Sf * sf * lift_own(G, cj, cr, a, false), V.fvg(df, a, j, kl));
              ACC25(-0.5 * Sf * sf * G.dx * G.D[cj[a]][cr[a]], VL.fvg(df, a, j, kl));
            }
          } else if (ndiff == 0) {
            const int f = face_slot(df, sf);
            const int fidx = cj[(df + 1) % 3] + p * cj[(df + 2) % 3];
            const double* rj = RJ + ((size_t)e * 6 + f) * 50 * pp + fidx;
            const int nb = nbr[e * 18 + f];
            int cn[3] = {cj[0], cj[1], cj[2]}; cn[df] = N - cj[df];
            ElemView Vn{NJ + (size_t)nb * NJC * nn, nn};
            const int jm = node_index(cn, p);
            ACC25(Sf, rj[(size_t)kl * pp] - sf * V.Fq(df, j, kl) - 0.5 * sf * V.fvq(df, j, kl)
                          + 0.5 * G.inv_hw * Vn.fvg(df, df, jm, kl));
            for (int a = 0; a < 3; ++a)
              ACC25(Sf * 0.5 * sf * lift_own(G, cj, cj, a, true), V.fvg(df, a, j, kl));
          } else {
            const int a = dc[0];
            ACC25(Sf * 0.5 * sf * lift_own(G, cj, cr, a, false), V.fvg(df, a, j, kl));
          }
        }
      }
    }
  }
}

// Pairs sharing no GL index are structurally zero: they are not in the pair list and keep the
// zeros written when the mesh was set.
template <bool IP>
__global__ void __launch_bounds__(256, 3) k_asm_own(Geo G, const double* __restrict__ NJ,
                                                 const double* __restrict__ NJL,
                                                 const double* __restrict__ RJ,
                                                 const int* __restrict__ nbr, const int* __restrict__ iperm,
                                                 const int* __restrict__ pairs, int npairs,
                                                 double* __restrict__ Aown) {
  const int e = blockIdx.x;
  const int lda = G.lda;
  for (int t = threadIdx.x; t < npairs; t += blockDim.x) {
    const int code = pairs[t];
    const int pj = code >> 16, pr = code & 0xffff;
    double acc[25];
    own_entry<IP>(G, NJ, NJL, RJ, nbr, e, iperm[pj], iperm[pr], acc);
    double* out = Aown + (size_t)e * own_stride(G) + (size_t)(5 * pj) * lda + own_col(G, pr, 0);
    for (int k = 0; k < 5; ++k)
      for (int l = 0; l < 5; ++l) out[(size_t)k * lda + l] = acc[k * 5 + l];
  }
}

// Neighbour couplings: X[e][pair][5x5] = dR_{e, row}/dq_{nbr(e, slot), col}.
// With the interior penalty (NJL non-null) the neighbour enters the face rows through its
// state and its unlifted gradient only, and the edge slots stay zero.
template <bool IP>
SC_HD void cross_entry(const Geo& G, const double* NJ, const double* NJL, const double* RJ, const int* nbr, int e,
                       int j, int slot, int r, double acc[25]) {
  const int nn = G.nn, p = G.p, N = G.N, pp = p * p;
  int cj[3], cr[3];
  node_coords(j, p, cj); node_coords(r, p, cr);
  ElemView V{NJ + (size_t)e * NJC * nn, nn};
  constexpr bool ip = IP;
#pragma unroll
  for (int kl = 0; kl < 25; ++kl) acc[kl] = 0.0;
  const double Wj = wprod(G, cj);
  if (slot < 6) {
    const int df = slot / 2, sf = (slot & 1) ? 1 : -1;
    const int jend = sf > 0 ? N : 0, nend = N - jend;
    const int nb = nbr[e * 18 + slot];
    ElemView Vn{NJ + (size_t)nb * NJC * nn, nn};
    ElemView VnL{ip ? NJL + (size_t)nb * NJC * nn : nullptr, nn};
    // (V) volume rows through e's own lifted gradient at the face node m co-located with r
    if (cr[df] == nend) {
      int cm[3] = {cr[0], cr[1], cr[2]}; cm[df] = jend;
      const int m = node_index(cm, p);
      for (int d = 0; d < 3; ++d) {
        bool online = true;
        for (int a = 0; a < 3; ++a) if (a != d && cj[a] != cm[a]) online = false;
        if (!online) continue;
        ACC25(G.Jf * Wj * G.D[cj[d]][cm[d]] * sf * G.inv_hw, -V.fvg(d, df, m, kl));
      }
    }
    if (cj[df] == jend) {
      int cn[3] = {cj[0], cj[1], cj[2]}; cn[df] = nend;
      const int jm = node_index(cn, p);
      const double Sf = G.Jf * Wj / G.w[cj[df]];
      if (r == jm) {
        const int fidx = cj[(df + 1) % 3] + p * cj[(df + 2) % 3];
        const double* rj = RJ + ((size_t)e * 6 + slot) * 50 * pp + fidx;
        if (ip)                                                                  // (S1)
          ACC25(Sf, rj[(size_t)(25 + kl) * pp] - 0.5 * sf * VnL.fvq(df, jm, kl) - (kl % 6 == 0 ? G.sigma : 0.0));
        else
          ACC25(Sf, rj[(size_t)(25 + kl) * pp] - 0.5 * sf * Vn.fvq(df, jm, kl));
        // (S2) e's lifted gradient at j reaches across the face: in every face term of j,
        // at half weight (BR1 average) or at the full weight of -s F_d(j) (interior penalty)
        const double w2 = ip ? 1.0 : 0.5;
        for (int d2 = 0; d2 < 3; ++d2) {
          if (cj[d2] != 0 && cj[d2] != N) continue;
          const int s2 = (cj[d2] == N) ? 1 : -1;
          const double Sf2 = G.Jf * Wj / G.w[cj[d2]];
          ACC25(Sf2 * w2 * s2 * sf * G.inv_hw, V.fvg(d2, df, j, kl));
        }
      }
      // (S3) the neighbour's gradient at jm (lifted, or unlifted with the interior penalty),
      // along its grid lines through jm
      int nd = 0, dd = -1;
      for (int a = 0; a < 3; ++a) if (cn[a] != cr[a]) { ++nd; dd = a; }
      if (ip) {
        if (nd == 0) {
          for (int a = 0; a < 3; ++a)
            ACC25(-0.5 * sf * Sf * G.dx * G.D[cn[a]][cn[a]], VnL.fvg(df, a, jm, kl));
        } else if (nd == 1) {
          ACC25(-0.5 * sf * Sf * G.dx * G.D[cn[dd]][cr[dd]], VnL.fvg(df, dd, jm, kl));
        }
      } else if (nd == 0) {
        for (int a = 0; a < 3; ++a)
          ACC25(-0.5 * sf * Sf * lift_own(G, cn, cn, a, true), Vn.fvg(df, a, jm, kl));
      } else if (nd == 1) {
        ACC25(-0.5 * sf * Sf * lift_own(G, cn, cr, dd, false), Vn.fvg(df, dd, jm, kl));
      }
    }
  } else if (!ip) {
    const int q = slot - 6, pi = q / 4;
    const int d1 = pi == 2 ? 1 : 0, d2 = pi == 0 ? 1 : 2;
    const int s1 = (q & 2) ? 1 : -1, s2 = (q & 1) ? 1 : -1;
    const int e1 = s1 > 0 ? N : 0, e2 = s2 > 0 ? N : 0;
    if (cj[d1] == e1 && cj[d2] == e2) {
      int cx[3] = {cj[0], cj[1], cj[2]}; cx[d1] = N - e1; cx[d2] = N - e2;
      if (node_index(cx, p) == r) {
        for (int o = 0; o < 2; ++o) {
          const int da = o ? d2 : d1, sa = o ? s2 : s1, db = o ? d1 : d2, sb = o ? s1 : s2;
          const int nb = nbr[e * 18 + face_slot(da, sa)];
          ElemView Vn{NJ + (size_t)nb * NJC * nn, nn};
          int cn[3] = {cj[0], cj[1], cj[2]}; cn[da] = N - cj[da];
          const double Sfa = G.Jf * Wj / G.w[cj[da]];
          ACC25(-0.5 * sa * Sfa * sb * G.inv_hw, Vn.fvg(da, db, node_index(cn, p), kl));
        }
      }
    }
  }
}

template <bool IP>
__global__ void k_asm_cross(Geo G, const double* __restrict__ NJ, const double* __restrict__ NJL,
                            const double* __restrict__ RJ,
                            const int* __restrict__ nbr, const int* __restrict__ prow,
                            const int* __restrict__ pslot, const int* __restrict__ pcol,
                            double* __restrict__ X) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= (size_t)G.K * G.NP) return;
  const int e = (int)(t / G.NP), pr = (int)(t % G.NP);
  double acc[25];
  cross_entry<IP>(G, NJ, NJL, RJ, nbr, e, prow[pr], pslot[pr], pcol[pr], acc);
  // layout X[e][k][pair][l]: the couplings of one row variable are contiguous
  for (int k = 0; k < 5; ++k)
    for (int l = 0; l < 5; ++l) X[(((size_t)e * 5 + k) * G.NP + pr) * 5 + l] = acc[k * 5 + l];
}

inline unsigned blocks_for(size_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

namespace sc {

// Shared memory of the residual kernels per CTA, and what order 6 takes (one element per CTA, the most of all).
constexpr int kPointSmemMax = (64 + kMaxNodes * 20) * (int)sizeof(double);
constexpr int kRowsSmemMax = (64 + kMaxNodes * 20 + 30 * kMaxP * kMaxP) * (int)sizeof(double);
static size_t point_smem(const Geo& G) { return (64 + (size_t)group_elems(G) * G.nn * 20) * sizeof(double); }
static size_t rows_smem(const Geo& G) {
  return (64 + (size_t)group_elems(G) * (G.nn * 20 + 30 * G.p * G.p)) * sizeof(double);
}

template <bool IP>
static cudaError_t launch_point(sc_ctx* c, const Geo& G, const double* Q, bool store_grad, unsigned long long* spd) {
  const int ge = group_elems(G);
  cudaError_t e = cudaFuncSetAttribute(k_point<IP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPointSmemMax);
  if (e != cudaSuccess) return e;
  count_launch(c);
  k_point<IP><<<(G.K + ge - 1) / ge, group_threads(G), point_smem(G), c->stream>>>(
      G, ge, Q, c->d_nbr, c->F, store_grad ? c->grad : nullptr, c->Floc, c->gloc, c->diss, spd);
  return cudaGetLastError();
}

template <bool IP, bool RK>
static cudaError_t launch_rows(sc_ctx* c, const Geo& G, const double* Q, const double* Qh, double* out, const RkStage& st) {
  const int ge = group_elems(G);
  cudaError_t e = cudaFuncSetAttribute(k_rows<IP, RK>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmemMax);
  if (e != cudaSuccess) return e;
  count_launch(c);
  k_rows<IP, RK><<<(G.K + ge - 1) / ge, group_threads(G), rows_smem(G), c->stream>>>(G, ge, Q, Qh, c->F, c->Floc, c->diss, c->d_nbr,
                                                                                     out, st);
  return cudaGetLastError();
}

cudaError_t launch_residual_geo(sc_ctx* c, const Geo& G, const double* Q, const double* Qh, double* out) {
  const bool ip = G.visc_flux == 1;
  const cudaError_t e = ip ? launch_point<true>(c, G, Q, true, nullptr) : launch_point<false>(c, G, Q, true, nullptr);
  if (e != cudaSuccess) return e;
  return ip ? launch_rows<true, false>(c, G, Q, Qh, out, RkStage{}) : launch_rows<false, false>(c, G, Q, Qh, out, RkStage{});
}

cudaError_t launch_rk_stage(sc_ctx* c, const Geo& G, const double* q, double* qout, const RkStage& st) {
  const bool ip = G.visc_flux == 1;
  unsigned long long* spd = st.first ? st.spd : nullptr;
  const cudaError_t e = ip ? launch_point<true>(c, G, q, false, spd) : launch_point<false>(c, G, q, false, spd);
  if (e != cudaSuccess) return e;
  return ip ? launch_rows<true, true>(c, G, q, nullptr, qout, st) : launch_rows<false, true>(c, G, q, nullptr, qout, st);
}

cudaError_t launch_residual(sc_ctx* c) { return launch_residual_geo(c, c->G, c->Q, c->Qh, c->B); }

cudaError_t launch_history(sc_ctx* c, const double* Qs, const double* Qsm1) {
  const size_t n = (size_t)c->G.K * c->G.nn * 5;
  count_launch(c);
  k_history<<<blocks_for(n, 256), 256, 0, c->stream>>>(c->G, Qs, Qsm1, c->Qh, n, c->bdf);
  return cudaGetLastError();
}

cudaError_t launch_assembly(sc_ctx* c) {
  const Geo& G = c->G;
  const size_t nodes = (size_t)G.K * G.nn;
  const bool ip = G.visc_flux == 1;
  count_launch(c, ip ? 4 : 3);
  k_nodejac<<<blocks_for(nodes, 64), 64, 0, c->stream>>>(G, c->Q, c->grad, c->NJ);
  // the unlifted gradients are those of the last residual evaluation of this state
  if (ip) k_nodejac<<<blocks_for(nodes, 64), 64, 0, c->stream>>>(G, c->Q, c->gloc, c->NJL);
  const size_t fn = (size_t)G.K * 6 * G.p * G.p;
  k_roejac<<<blocks_for(fn, 64), 64, 0, c->stream>>>(G, c->Q, c->d_nbr, c->RJ);
  {
    ProfScope ps(c, SCK_ASM_OWN);
    if (ip)
      k_asm_own<true><<<G.K, 256, 0, c->stream>>>(G, c->NJ, c->NJL, c->RJ, c->d_nbr, c->d_iperm, c->d_own_pairs,
                                                  (int)c->own_pairs.size(), c->Aown);
    else
      k_asm_own<false><<<G.K, 256, 0, c->stream>>>(G, c->NJ, nullptr, c->RJ, c->d_nbr, c->d_iperm, c->d_own_pairs,
                                                   (int)c->own_pairs.size(), c->Aown);
  }
  const size_t np = (size_t)G.K * G.NP;
  if (ip)
    k_asm_cross<true><<<blocks_for(np, 128), 128, 0, c->stream>>>(G, c->NJ, c->NJL, c->RJ, c->d_nbr, c->d_prow,
                                                                  c->d_pslot, c->d_pcol, c->X);
  else
    k_asm_cross<false><<<blocks_for(np, 128), 128, 0, c->stream>>>(G, c->NJ, nullptr, c->RJ, c->d_nbr, c->d_prow,
                                                                   c->d_pslot, c->d_pcol, c->X);
  return cudaGetLastError();
}

}  // namespace sc
