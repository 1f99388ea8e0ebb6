// Discrete adjoint of the clustered-LTS time loop, elastic equations, one or fused
// simulations (one cluster is the global-time-stepping case: a macro step is one step).
//
// One step of an element maps Q to Q' = Q + V(T) + S_L(T) + S_N(X of the face neighbours),
// with D_0 = Q, D_{d+1} = sum_c S_c D_d K_c^T (S_c the star matrices of the time kernel),
// T = sum_d c_d D_d, V = -sum_c S_c T K_c, S_L = sum_i A-_i (T F~_i) F^_i and
// S_N = sum_i A+_i (X_i F-_{j,h}) F^_i (A-_i, A+_i the 9 x 9 flux solvers of face i, X_i the
// neighbour's buffer that the cluster relation selects). For the adjoint lambda = dJ/dQ'
// the reverse passes below compute, per element,
//   mu = dJ/dT = -sum_c S_c^T lambda K_c^T + sum_i ((A-_i^T lambda) F^_i^T) F~_i^T
//        + the adjoints of the buffers the step wrote,
//   G_{O-1} = c_{O-1} mu, G_d = c_d mu + sum_c S_c^T G_{d+1} K_c,   dJ/dQ = lambda + G_0,
// the transposed neighbour fluxes into the adjoints of the buffers they read, and, for the
// material derivatives, what is left of the correlations
//   W_c  = sum_{d<O-1} G_{d+1} (D_d K_c^T)^T - lambda (T K_c)^T,
//   W-_i = lambda (T F~_i F^_i)^T,   W+_i = lambda_k (X F-_{j,h} F^_i)^T
// of S_c, A-_i, A+_i once they are contracted with everything that does not depend on the
// material: the matrices are linear in (lambda_e, mu_e, 1/rho_e) (star matrices, three sums)
// and in their products with the eight Riemann coefficients (flux solvers, ten sums a face
// and side, face_products). Each sum is a scalar product per (face) mode, so the threads
// that hold the columns form it: the 3 x 3 tiles of the 9 x 9 correlations cost k_adj_pred_sp
// a pass over shared memory per derivative and 567 FP64 additions per element (204 us a launch,
// 126 with the sums; 3 % more with the star matrices' entries as StarGeo holds them; 47,040
// elements, order 4), k_adj_nbr another 324.
// The flux solvers are explicit (FP32, from the same closed forms as the forward kernels'
// flux code), the star matrices are applied by their physical form (StarGeo); CUDA cores. The sums
// are FP32 within a pass, with the normals and the star entries rounded to FP32, and FP64 over the
// passes (the correlations were contracted with FP64 geometry once, at the end): against the FP64
// gradient of 48 to 64 seeded cases each (1,008 elements, 12 steps) the errors are those of the
// correlations times 1.05, 0.98, 1.00 (dJ/dlambda, orders 3, 4, 5), 1.03, 0.99, 0.98 (mu) and 0.91, 0.87,
// 0.79 (rho), with a standard error of 2 to 4 %; with the normals as two FP32 numbers each 1.01 instead
// of 1.05, and the gradient of 47,040 elements 6 % slower: not kept.
#pragma once
#include "kernels.cuh"

namespace ltsdev {

// operators of an element (floats)
constexpr int AM_LOC = 0;        // A-_i, i = 0..3: [out][in]
constexpr int AM_NBR = 324;      // A+_i, i = 0..3
constexpr int AM_GEO = 648;      // the star matrices' entries (StarGeo), the four unit normals
constexpr int AM_NRM = 28, AM_NGEO = 40;
constexpr int AM_SIZE = AM_GEO + AM_NGEO;
// material sums of an element (doubles)
constexpr int WG_STAR = 0;       // of lambda, mu, 1/rho
constexpr int WG_LOC = 3;        // A-_i: ten sums a face (face_products)
constexpr int WG_NBR = 43;       // A+_i
constexpr int WG_SIZE = 83;

// Threads per element group: one warp up to order 4, two at order 5 (every phase needs at
// least one thread per mode column).
template <int O>
struct AdjNT {
  static constexpr int value = (nbasis(O) <= 32) ? 32 : 64;
};

// Transposed copies of the operator tables, so that every loop over a table reads it with
// consecutive threads on consecutive entries:
//   KT[c][j][i] = K[c][i][j],  FtT[i][f][b] = F~_i[b][f],  FhT[i][b][f] = F^_i[f][b],
//   FbT[jh][f][b] = F-_{jh}[b][f].
// Velocity at the receivers from Q^n: out[f][r][q] = sum_b Q_f[elem_r][6+q][b] phi_r[b] for
// the nsim simulations of an (elastic) state in groups of G (simulation f of element k, row
// q, mode b at k qs + (f / G) 9 B G + (q B + b) G + f % G; G = 1 for one simulation).
template <int O>
__global__ void k_adj_sample(const float* Q, long long qs, int nsim, int G, const int* elem, const float* phi,
                             int nrec, float* out) {
  constexpr int B = nbasis(O);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 3 * nrec * nsim) return;
  const int f = t / (3 * nrec), r = (t / 3) % nrec, q = t % 3;
  const float* row = Q + (size_t)elem[r] * qs + (size_t)(f / G) * (9 * B * G) + f % G + (size_t)(6 + q) * B * G;
  float v = 0.f;
  for (int b = 0; b < B; ++b) v = fmaf(row[(size_t)b * G], phi[r * B + b], v);
  out[t] = v;
}

// The misfit's source: lambda_f[elem_r][6+q][b] += res[f][r][q] phi_r[b], lambda laid out
// [element][simulation][9][B]. One CTA per simulation, a thread per (component, mode) that takes
// the receivers in order (receivers that share an element add in a fixed order) and reads no
// result back (one CTA of B threads waiting for each addition: 21 us for 16 receivers, now 4 us).
template <int O>
__global__ void k_adj_source(float* lam, int nsim, const int* elem, const float* phi, const float* res, int nrec) {
  constexpr int B = nbasis(O);
  const int t = threadIdx.x, f = blockIdx.x;
  if (t >= 3 * B) return;
  for (int r = 0; r < nrec; ++r)
    atomicAdd(lam + ((size_t)elem[r] * nsim + f) * 9 * B + 6 * B + t, res[(f * nrec + r) * 3 + t / B] * phi[r * B + t % B]);
}


// Moment-tensor gradient of the point sources one neighbour pass added:
// g[src][r] += c_s sum_b lambda_f[elem][r][b] phi_src[b], with c_s = -m0 (int s dt) / |det J|
// of item s and lambda the adjoint of Q after the pass ([element][simulation][9][B]). One
// thread per (item, stress component); a pass holds at most one item per source, so every
// entry has one writer.
template <int O>
__global__ void k_adj_src_grad(const float* lam, int nsim, const SrcItem* items, const double* c, int n,
                               const float* phi, double* g) {
  constexpr int B = nbasis(O);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 6 * n) return;
  const int s = t / 6, r = t % 6;
  const SrcItem it = items[s];
  const float* row = lam + ((size_t)it.elem * nsim + it.sim) * 9 * B + (size_t)r * B;
  float v = 0.f;
  for (int b = 0; b < B; ++b) v = fmaf(row[b], phi[it.phi_off + b], v);
  g[(size_t)(it.phi_off / B) * 6 + r] += c[s] * (double)v;
}

// ------------------------------------------------------------------ clustered LTS adjoint
// The LTS state is (Q, B1, B2, B3). Taken backwards, a neighbour pass of cluster l (step n)
// that added S_N(X_i) to Q_k sends ((A+_i^T lambda_Q_k) F^_i^T) F-_{j,h}^T to the adjoint
// of the buffer it read (B1 same cluster, B3 the neighbour finer, B2 / B1 - B2 the
// neighbour coarser in the first / second half); a predict pass that wrote B1 = T,
// B2 = T(dt/2) (finer neighbour), B3 = T or B3 += T (coarser neighbour, even / odd n) and
// added V(T) + S_L(T) to Q collects mu = V^T + S_L^T + lambda_B1 (+ lambda_B3) and
// mu_half = lambda_B2, resets the buffer adjoints it overwrote (lambda_B3 survives an
// accumulation) and runs the transposed time kernel with both Taylor weights.
struct AdjLtsArgs {
  const float* Qs;                    // Q before this predict pass (element stride qs)
  const float *B1s, *B2s, *B3s;       // buffers before this neighbour pass (element stride bufs): B1 of
                                      // every owner, B2 and B3 of the elements that have one, at
  const int *slot2, *slot3;           // their rows slot2, slot3
  float* lq;                          // [K][9B] adjoint of Q
  float *lb1, *lb2, *lb3;             // [K][9B] adjoints of B1, B2, B3
  const float* amat;
  const int* fwd;
  const int* back;
  const int* owners;                  // neighbour reverse: the pass's buffer owners with an active
                                      // receiver (one CTA each), or null: owner = CTA index
  const int* meta;
  double* W;                          // [K][WG_SIZE], per-pass sums in FP32 added in FP64
  const float *KT, *FtT, *FhT, *FbT;  // transposed operator tables (see AdjTables)
  long long qs, bufs;
  int end;                            // active elements [0, end)
  // simulations of a fused run, in groups of G in the state and buffer snapshots (element k,
  // simulation f, row r, mode b at k qs + (f / G) 9 B G + (r B + b) G + f % G; one
  // simulation: nsim = G = 1); the adjoints are [element][simulation][9][B] and W sums the
  // simulations
  int nsim, G;
};

// The nine rows of a [9][LD] block, entries j .. j + 3 (16-byte aligned; the same address in
// every lane, so each load is one broadcast).
template <int LD>
__device__ __forceinline__ void load_cols4(const float* src, int j, float4 x[9]) {
#pragma unroll
  for (int r = 0; r < 9; ++r) x[r] = *reinterpret_cast<const float4*>(src + r * LD + j);
}
__device__ __forceinline__ float lane4(const float4& v, int u) { return u == 0 ? v.x : u == 1 ? v.y : u == 2 ? v.z : v.w; }

// v[r] = sum_{j < N} src[r * LD + j] * tab[j * ts + t] for the 9 rows r, the broadcast
// operand four entries at a time (LD = rup(N, 4), pad entries of src zero; the table is not
// read past row NT - 1, so that it needs no pad rows).
template <int NT, int LD>
__device__ __forceinline__ void rows9v(const float* src, const float* tab, int ts, int t, float v[9]) {
#pragma unroll
  for (int r = 0; r < 9; ++r) v[r] = 0.f;
#pragma unroll 1
  for (int j = 0; j < LD; j += 4) {
    float4 x[9];
    load_cols4<LD>(src, j, x);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int ju = NT % 4 == 0 ? j + u : min(j + u, NT - 1);
      const float w = tab[ju * ts + t];
#pragma unroll
      for (int r = 0; r < 9; ++r) v[r] = fmaf(lane4(x[r], u), w, v[r]);
    }
  }
}

// An element's star matrices S_c (AM_GEO, 16-byte aligned): mu dxi_c/dx_d at 3 c + d, kappa
// dxi_c/dx_d and dxi_c/dx_d / rho, and lambda / kappa, kappa = lambda (1 where lambda vanishes).
// Every entry is rounded once, by itself: with dxi/dx, lambda, mu and 1/rho apart, the roundings of
// the three factors scale the whole matrix alike in every step, which showed in the results
// (dJ/dsigma at the start 5 % further from the FP64 gradient, dJ/dmu at order 3 13 %).
struct StarGeo {
  float M[9], L[9], R[9], lf;
  __device__ __forceinline__ explicit StarGeo(const float* p) {
    float v[28];
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      const float4 a = reinterpret_cast<const float4*>(p)[i];
      v[4 * i] = a.x; v[4 * i + 1] = a.y; v[4 * i + 2] = a.z; v[4 * i + 3] = a.w;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      M[i] = v[i];
      L[i] = v[9 + i];
      R[i] = v[18 + i];
    }
    lf = v[27];
  }
};
// v = sum_c S_c y_c: mu times the physical velocity gradient, lambda times its trace and the
// stress divergence over rho (about 70 multiply-adds and seven 16-byte loads; the matrices' nonzero
// entries take 108 and 27).
struct StarFwd {
  float g[9], l, dv[3];   // g[3 d + j] = mu d v_j / d x_d
  __device__ __forceinline__ StarFwd() {
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = 0.f;
    l = dv[0] = dv[1] = dv[2] = 0.f;
  }
  __device__ __forceinline__ void add(const StarGeo& s, int c, const float y[9]) {
    const float *M = s.M + 3 * c, *R = s.R + 3 * c;
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int j = 0; j < 3; ++j) g[3 * d + j] = fmaf(M[d], y[6 + j], g[3 * d + j]);
#pragma unroll
    for (int d = 0; d < 3; ++d) l = fmaf(s.L[3 * c + d], y[6 + d], l);
    dv[0] = fmaf(R[0], y[0], fmaf(R[1], y[3], fmaf(R[2], y[5], dv[0])));
    dv[1] = fmaf(R[0], y[3], fmaf(R[1], y[1], fmaf(R[2], y[4], dv[1])));
    dv[2] = fmaf(R[0], y[5], fmaf(R[1], y[4], fmaf(R[2], y[2], dv[2])));
  }
  __device__ __forceinline__ void get(const StarGeo& s, float v[9]) const {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      v[i] = fmaf(2.f, g[4 * i], s.lf * l);
      v[6 + i] = dv[i];
    }
    v[3] = g[1] + g[3];
    v[4] = g[5] + g[7];
    v[5] = g[2] + g[6];
  }
};
// w = sum_c S_c^T z_c, and the products of its parts with the column x: kappa, mu and 1/rho times
// this column's share in the sums of lambda, mu and 1/rho, x^T sum_c (dS_c/dp)^T z_c.
struct StarRev {
  float a[3], p[3], q[6];   // w_v = lambda / kappa a + p, w_sigma = q
  __device__ __forceinline__ StarRev() {
#pragma unroll
    for (int i = 0; i < 3; ++i) a[i] = p[i] = q[i] = q[3 + i] = 0.f;
  }
  __device__ __forceinline__ void add(const StarGeo& s, int c, const float z[9]) {
    const float *M = s.M + 3 * c, *R = s.R + 3 * c;
    const float tr = z[0] + z[1] + z[2];
#pragma unroll
    for (int j = 0; j < 3; ++j) a[j] = fmaf(s.L[3 * c + j], tr, a[j]);
    p[0] = fmaf(M[0], 2.f * z[0], fmaf(M[1], z[3], fmaf(M[2], z[5], p[0])));
    p[1] = fmaf(M[1], 2.f * z[1], fmaf(M[0], z[3], fmaf(M[2], z[4], p[1])));
    p[2] = fmaf(M[2], 2.f * z[2], fmaf(M[1], z[4], fmaf(M[0], z[5], p[2])));
#pragma unroll
    for (int d = 0; d < 3; ++d) q[d] = fmaf(R[d], z[6 + d], q[d]);
    q[3] = fmaf(R[1], z[6], fmaf(R[0], z[7], q[3]));
    q[4] = fmaf(R[2], z[7], fmaf(R[1], z[8], q[4]));
    q[5] = fmaf(R[2], z[6], fmaf(R[0], z[8], q[5]));
  }
  __device__ __forceinline__ void get(const StarGeo& s, float w[9]) const {
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = q[i];
#pragma unroll
    for (int j = 0; j < 3; ++j) w[6 + j] = fmaf(s.lf, a[j], p[j]);
  }
  __device__ __forceinline__ void sums(const float x[9], float sgn, float f[3]) const {
    float l = 0.f, m = 0.f, r = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      l = fmaf(a[j], x[6 + j], l);
      m = fmaf(p[j], x[6 + j], m);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) r = fmaf(q[i], x[i], r);
    f[0] = fmaf(sgn, l, f[0]);
    f[1] = fmaf(sgn, m, f[1]);
    f[2] = fmaf(sgn, r, f[2]);
  }
};

// u = A^T l, A a 9 x 9 flux solver with rows padded to 12 (16-byte aligned).
__device__ __forceinline__ void flux_transposed(const float* Am, const float l[9], float u[9]) {
#pragma unroll
  for (int r = 0; r < 9; ++r) u[r] = 0.f;
#pragma unroll
  for (int s = 0; s < 9; ++s) {
    const float4 a0 = *reinterpret_cast<const float4*>(Am + s * 12);
    const float4 a1 = *reinterpret_cast<const float4*>(Am + s * 12 + 4);
    const float a8 = Am[s * 12 + 8];
    u[0] = fmaf(a0.x, l[s], u[0]);
    u[1] = fmaf(a0.y, l[s], u[1]);
    u[2] = fmaf(a0.z, l[s], u[2]);
    u[3] = fmaf(a0.w, l[s], u[3]);
    u[4] = fmaf(a1.x, l[s], u[4]);
    u[5] = fmaf(a1.y, l[s], u[5]);
    u[6] = fmaf(a1.z, l[s], u[6]);
    u[7] = fmaf(a1.w, l[s], u[7]);
    u[8] = fmaf(a8, l[s], u[8]);
  }
}

// One face mode's share in the ten sums of a flux solver (face_flux_gradient in host_flux.h): l the
// adjoint's column, x the state's. The flux maps the velocity v and the traction t of x
// through normal and tangential coefficients to a state (v*, t*), and n v*^T (lambda, mu) and
// t* / rho to the result; against l these are products of (n.v, n.t, v_T, t_T) with the trace
// of l's stresses, the vector (l n + diag(l) n) and l's velocities.
__device__ __forceinline__ void face_products(const float* n, const float l[9], const float x[9], float o[10]) {
  const float n0 = n[0], n1 = n[1], n2 = n[2];
  const float tr = l[0] + l[1] + l[2];
  const float a0 = fmaf(2.f * n0, l[0], fmaf(n1, l[3], n2 * l[5]));
  const float a1 = fmaf(2.f * n1, l[1], fmaf(n0, l[3], n2 * l[4]));
  const float a2 = fmaf(2.f * n2, l[2], fmaf(n1, l[4], n0 * l[5]));
  const float t0 = fmaf(n0, x[0], fmaf(n1, x[3], n2 * x[5]));
  const float t1 = fmaf(n1, x[1], fmaf(n0, x[3], n2 * x[4]));
  const float t2 = fmaf(n2, x[2], fmaf(n1, x[4], n0 * x[5]));
  const float vn = fmaf(n0, x[6], fmaf(n1, x[7], n2 * x[8])), tn = fmaf(n0, t0, fmaf(n1, t1, n2 * t2));
  const float an = fmaf(n0, a0, fmaf(n1, a1, n2 * a2)), ln = fmaf(n0, l[6], fmaf(n1, l[7], n2 * l[8]));
  const float v0 = fmaf(-vn, n0, x[6]), v1 = fmaf(-vn, n1, x[7]), v2 = fmaf(-vn, n2, x[8]);
  const float s0 = fmaf(-tn, n0, t0), s1 = fmaf(-tn, n1, t1), s2 = fmaf(-tn, n2, t2);
  o[0] = -tr * vn;
  o[1] = -tr * tn;
  o[2] = -an * vn;
  o[3] = -an * tn;
  o[4] = -fmaf(a0, v0, fmaf(a1, v1, a2 * v2));
  o[5] = -fmaf(a0, s0, fmaf(a1, s1, a2 * s2));
  o[6] = -ln * tn;
  o[7] = -ln * vn;
  o[8] = -fmaf(l[6], s0, fmaf(l[7], s1, l[8] * s2));
  o[9] = -fmaf(l[6], v0, fmaf(l[7], v1, l[8] * v2));
}

// Polynomial degree of volume mode j (modes are ordered by degree).
__device__ __forceinline__ int mode_degree(int j) {
  int p = 0;
  while (nbasis(p + 1) <= j) ++p;
  return p;
}

// Shared-memory plan of k_adj_pred, a persistent kernel: the operator tables (K_c^T, K_c,
// F~_i, F^_i^T, F~_i^T) once per CTA, then one region per element group. A group is one warp
// (orders 3-4) or two (order 5) and takes the CTA's elements in turn; G groups fill the
// shared memory (at most 128 registers a thread, 15 named barriers for two-warp groups).
// Mode rows are padded to BP = rup(B, 4) and face-mode rows to FP = rup(F, 4), the pad entries
// zero (table rows past B or F zero as well), so that every contraction reads its broadcast
// operand four entries at a time.
template <int O>
struct AdjPredCfg {
  static constexpr int B = nbasis(O), F = nface(O), NT = AdjNT<O>::value;
  static constexpr int BP = rup(B, 4), FP = rup(F, 4), NB9 = 9 * BP;
  static constexpr int NGEO = AM_NGEO, NALOC = 4 * 9 * 12;       // geometry; A-_i rows padded to 12
  static constexpr int NSCR = 19 * 4 * FP;
  static constexpr int ELEM = NGEO + NALOC + (4 + O) * NB9 + NSCR;   // sS, sA, sL, sT, sG[2], sD[O], scratch
  static constexpr int TAB = 6 * BP * B + 8 * BP * F + 4 * FP * B;
  static constexpr int G_SMEM = (227 * 1024 / 4 - TAB) / ELEM;
  static constexpr int G_REG = 65536 / (128 * NT);
  static constexpr int G_BAR = (NT == 32) ? 32 : 15;
  static constexpr int G0 = G_SMEM < G_REG ? G_SMEM : G_REG;
  static constexpr int G = G0 < G_BAR ? G0 : G_BAR;
  static constexpr int THREADS = G * NT;
  static constexpr int SMEM_BYTES = 4 * (TAB + G * ELEM);
  static_assert(G >= 1 && SMEM_BYTES <= 227 * 1024, "k_adj_pred shared-memory plan");
  static_assert(TAB % 4 == 0 && ELEM % 4 == 0 && NB9 % 4 == 0, "16-byte aligned regions");
};

// Barrier of one element group: the warp itself, or a named barrier over its two warps.
template <int NT>
__device__ __forceinline__ void gsync(int g) {
  if constexpr (NT == 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(NT) : "memory");
}

// dst[(q / B) BP + q % B] = src[q G] for q < 9 B: a [9][B] block (stride G between entries)
// into the padded [9][BP] layout, every load issued before the first store.
template <int B, int BP, int NT>
__device__ __forceinline__ void stage_pad(float* dst, const float* __restrict__ src, int G, int t) {
  constexpr int N = 9 * B, R = (N + NT - 1) / NT;
  float v[R];
#pragma unroll
  for (int j = 0; j < R; ++j)
    if (t + j * NT < N) v[j] = __ldg(src + (size_t)(t + j * NT) * G);
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int q = t + j * NT;
    if (q < N) dst[(q / B) * BP + q % B] = v[j];
  }
}

// Reverse of a predict pass over the active elements [0, end).
//
// Degree structure used throughout (exact): K_c[i][j] vanishes unless deg i < deg j, so
// D_d is a polynomial of degree O-1-d and lives on the first nbasis(O-d) modes; only those
// modes of its adjoint G_d matter. With Z_c = G_{d+1} K_c the reverse time kernel is
// G_d = c_d mu + c'_d mu_half + sum_c S_c^T Z_c and the star matrices' sums of level d are
// Z_c's against D_d; with V_c = lambda K_c^T the volume term is mu = -sum_c S_c^T V_c and its
// sums are -V_c's against T. The contractions run over a multiple of four entries; the extra
// entries multiply structural zeros of K_c or zero pads, so the sums are those of the
// unpadded loops, term for term.
template <int O>
__global__ void __launch_bounds__(AdjPredCfg<O>::THREADS, 1) k_adj_pred(DevOps ops, AdjLtsArgs a, PhaseArgs ph) {
  using C = AdjPredCfg<O>;
  constexpr int B = C::B, F = C::F, BP = C::BP, FP = C::FP, NB9 = C::NB9, NT = C::NT;
  extern __shared__ __align__(16) float smem[];
  float* tKT = smem;                  // [3][BP][B]   K_c^T[j][i] at (c BP + j) B + i
  float* tK = tKT + 3 * BP * B;       // [3][BP][B]   K_c[j][i]
  float* tFt = tK + 3 * BP * B;       // [4][BP][F]   F~_i[b][f] at (i BP + b) F + f
  float* tFhT = tFt + 4 * BP * F;     // [4][BP][F]   F^_i[f][b] at (i BP + b) F + f
  float* tFtT = tFhT + 4 * BP * F;    // [4][FP][B]   F~_i[b][f] at (i FP + f) B + b
  // K_c[i][j] vanishes unless deg i < deg j (phi_i is orthogonal to the derivative of phi_j
  // otherwise); those entries are set to exact zeros, so that the padded loops below add
  // exact zeros only
  for (int i = threadIdx.x; i < 3 * BP * B; i += C::THREADS) {
    const int c = i / (BP * B), j = (i / B) % BP, x = i % B;
    const bool in = j < B;
    tKT[i] = (in && mode_degree(x) < mode_degree(j)) ? a.KT[(c * B + j) * B + x] : 0.f;
    tK[i] = (in && mode_degree(j) < mode_degree(x)) ? ops.K[(c * B + j) * B + x] : 0.f;
  }
  for (int i = threadIdx.x; i < 4 * BP * F; i += C::THREADS) {
    const int fi = i / (BP * F), j = (i / F) % BP, f = i % F;
    tFt[i] = (j < B) ? ops.Ft[(fi * B + j) * F + f] : 0.f;
    tFhT[i] = (j < B) ? a.FhT[(fi * B + j) * F + f] : 0.f;
  }
  for (int i = threadIdx.x; i < 4 * FP * B; i += C::THREADS) {
    const int fi = i / (FP * B), f = (i / B) % FP, x = i % B;
    tFtT[i] = (f < F) ? a.FtT[(fi * F + f) * B + x] : 0.f;
  }
  // every group region starts zero: the pad entries are never written afterwards
  for (int i = threadIdx.x; i < C::G * C::ELEM; i += C::THREADS) smem[C::TAB + i] = 0.f;
  __syncthreads();
  const int g = threadIdx.x / NT, t = threadIdx.x % NT;
  float* sS = smem + C::TAB + g * C::ELEM;   // geometry and material
  float* sA = sS + C::NGEO;       // A-_i [4][9][12]: row s of face i at (i 9 + s) 12
  float* sL = sA + C::NALOC;      // [9][BP] lambda
  float* sT = sL + NB9;
  float* sG0 = sT + NB9;          // G ping-pong [2][9][BP]
  float* sDb = sG0 + 2 * NB9;     // D_0 .. D_{O-1} [O][9][BP]
  float* sScr = sDb + O * NB9;    // transposed fluxes and face products; star sums
  for (int k = blockIdx.x * C::G + g; k < a.end; k += gridDim.x * C::G) {
    const int meta = a.meta[k];
    const int cl = meta & 0xff;
    const bool finer = meta & FLAG_FINER, coarser = meta & FLAG_COARSER;
    const bool even = ph.parity[cl] == 0;
    {
      const float* am = a.amat + (size_t)k * AM_SIZE;
      for (int q = t; q < C::NGEO; q += NT) sS[q] = __ldg(am + AM_GEO + q);
      for (int q = t; q < 4 * 81; q += NT) sA[(q / 9) * 12 + q % 9] = __ldg(am + AM_LOC + q);
    }
    double* Wk = a.W + (size_t)k * WG_SIZE;
    float wst[3] = {0.f, 0.f, 0.f};   // this column's star sums over the simulations
    for (int sim = 0; sim < a.nsim; ++sim) {
      const size_t kf = (size_t)k * a.nsim + sim;
      stage_pad<B, BP, NT>(sL, a.lq + kf * (9 * B), 1, t);
      stage_pad<B, BP, NT>(sDb, a.Qs + (size_t)k * a.qs + (size_t)(sim / a.G) * (9 * B * a.G) + sim % a.G, a.G, t);
      {
        // the adjoints of the buffers this pass wrote: lambda_B1 (+ lambda_B3) into sG0[0],
        // lambda_B2 into sG0[1]; reset here (lambda_B3 survives an accumulation)
        constexpr int N = 9 * B, R = (N + NT - 1) / NT;
        const size_t o = kf * N;
        float v1[R], v2[R], v3[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int q = t + j * NT;
          v1[j] = v2[j] = v3[j] = 0.f;
          if (q < N) {
            v1[j] = a.lb1[o + q];
            if (coarser) v3[j] = a.lb3[o + q];
            if (finer) v2[j] = a.lb2[o + q];
          }
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int q = t + j * NT;
          if (q < N) {
            const int qp = (q / B) * BP + q % B;
            sG0[qp] = v1[j] + v3[j];
            sG0[NB9 + qp] = v2[j];
            a.lb1[o + q] = 0.f;
            if (coarser && even) a.lb3[o + q] = 0.f;
            if (finer) a.lb2[o + q] = 0.f;
          }
        }
      }
      gsync<NT>(g);
      // ---- forward time kernel: D_{d+1} = sum_c S_c D_d K_c^T on the support of D_{d+1}
#pragma unroll
      for (int d = 0; d < O - 1; ++d) {
        const int nin = nbasis(O - d), nout = nbasis(O - 1 - d);
        if (t < B) {
          float Y[3][9];
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int s = 0; s < 9; ++s) Y[c][s] = 0.f;
          if (t < nout)
#pragma unroll 1
            for (int kk = 0; kk < nin; kk += 4) {
              float4 x[9];
              load_cols4<BP>(sDb + d * NB9, kk, x);
#pragma unroll
              for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  const float kc = tKT[(c * BP + kk + u) * B + t];
#pragma unroll
                  for (int s = 0; s < 9; ++s) Y[c][s] = fmaf(lane4(x[s], u), kc, Y[c][s]);
                }
            }
          const StarGeo geo(sS);
          StarFwd st;
#pragma unroll
          for (int c = 0; c < 3; ++c) st.add(geo, c, Y[c]);
          float v[9];
          st.get(geo, v);
#pragma unroll
          for (int r = 0; r < 9; ++r) sDb[(d + 1) * NB9 + r * BP + t] = v[r];
        }
        gsync<NT>(g);
      }
      float mu[9], muh[9];
#pragma unroll
      for (int r = 0; r < 9; ++r) mu[r] = muh[r] = 0.f;
      if (t < B) {
        float T[9];
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          float v = 0.f;
          for (int d = 0; d < O; ++d) v = fmaf(ph.coef[cl][d], sDb[d * NB9 + r * BP + t], v);
          sT[r * BP + t] = T[r] = v;
        }
        // V_c = lambda K_c^T and the volume term
        float V[3][9];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int s = 0; s < 9; ++s) V[c][s] = 0.f;
#pragma unroll 1
        for (int b = 0; b < BP; b += 4) {
          float4 x[9];
          load_cols4<BP>(sL, b, x);
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const float kc = tKT[(c * BP + b + u) * B + t];
#pragma unroll
              for (int s = 0; s < 9; ++s) V[c][s] = fmaf(lane4(x[s], u), kc, V[c][s]);
            }
        }
        const StarGeo geo(sS);
        StarRev st;
#pragma unroll
        for (int c = 0; c < 3; ++c) st.add(geo, c, V[c]);
        float w[9];
        st.get(geo, w);
        st.sums(T, -1.f, wst);
#pragma unroll
        for (int r = 0; r < 9; ++r) mu[r] = -w[r];
      }
      gsync<NT>(g);
      // local surface: LF_i = lambda F^_i^T, TF_i = T F~_i, U_i = A-_i^T LF_i, per (face, f);
      // the pad columns f >= F are written zero
      float* sU = sScr;               // [4][9][FP]
      float* sP = sScr + 36 * FP;     // [4][10][FP]
      for (int p = t; p < 4 * FP; p += NT) {
        const int i = p / FP, f = p % FP;
        float u[9], o[10];
        if (f < F) {
          float lf[9], tf[9];
          rows9v<BP, BP>(sL, tFhT + i * BP * F, F, f, lf);
          rows9v<BP, BP>(sT, tFt + i * BP * F, F, f, tf);
          flux_transposed(sA + i * 108, lf, u);
          face_products(sS + AM_NRM + 3 * i, lf, tf, o);
        } else {
#pragma unroll
          for (int r = 0; r < 9; ++r) u[r] = o[r] = 0.f;
          o[9] = 0.f;
        }
#pragma unroll
        for (int r = 0; r < 9; ++r) sU[(i * 9 + r) * FP + f] = u[r];
#pragma unroll
        for (int q = 0; q < 10; ++q) sP[(i * 10 + q) * FP + f] = o[q];
      }
      gsync<NT>(g);
      if (t < B)
#pragma unroll 1
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int f = 0; f < FP; f += 4) {
            float4 x[9];
            load_cols4<FP>(sU + i * 9 * FP, f, x);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float w = tFtT[(i * FP + f + u) * B + t];
#pragma unroll
              for (int r = 0; r < 9; ++r) mu[r] = fmaf(lane4(x[r], u), w, mu[r]);
            }
          }
      for (int p = t; p < 40; p += NT) {
        float acc = 0.f;
#pragma unroll
        for (int f = 0; f < F; ++f) acc += sP[p * FP + f];
        atomicAdd(Wk + WG_LOC + p, (double)acc);
      }
      // the buffers this pass wrote
      if (t < B) {
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          mu[r] += sG0[r * BP + t];
          muh[r] = sG0[NB9 + r * BP + t];
        }
#pragma unroll
        for (int r = 0; r < 9; ++r)
          sG0[((O - 1) & 1) * NB9 + r * BP + t] = ph.coef[cl][O - 1] * mu[r] + ph.hcoef[cl][O - 1] * muh[r];
      }
      gsync<NT>(g);
      // ---- reverse time kernel
#pragma unroll
      for (int d = O - 2; d >= 0; --d) {
        const int nk = nbasis(O - 1 - d), nout = nbasis(O - d);
        const float* Gn = (sG0 + ((d + 1) & 1) * NB9);
        if (t < B) {
          float Z[3][9];
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int r = 0; r < 9; ++r) Z[c][r] = 0.f;
          // entries kk >= nk of G_{d+1} meet K_c[kk][t] = 0 for t < nout (degree structure)
          if (t < nout)
#pragma unroll 1
            for (int kk = 0; kk < nk; kk += 4) {
              float4 x[9];
              load_cols4<BP>(Gn, kk, x);
#pragma unroll
              for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  const float kc = tK[(c * BP + kk + u) * B + t];
#pragma unroll
                  for (int r = 0; r < 9; ++r) Z[c][r] = fmaf(lane4(x[r], u), kc, Z[c][r]);
                }
            }
          float gv[9];
#pragma unroll
          for (int r = 0; r < 9; ++r) gv[r] = ph.coef[cl][d] * mu[r] + ph.hcoef[cl][d] * muh[r];
          // entries t >= nout of Z_c are zero and those of D_d not part of the sums
          if (t < nout) {
            const StarGeo geo(sS);
            StarRev st;
#pragma unroll
            for (int c = 0; c < 3; ++c) st.add(geo, c, Z[c]);
            float w[9], x[9];
            st.get(geo, w);
#pragma unroll
            for (int r = 0; r < 9; ++r) {
              x[r] = sDb[d * NB9 + r * BP + t];
              gv[r] += w[r];
            }
            st.sums(x, 1.f, wst);
          }
#pragma unroll
          for (int r = 0; r < 9; ++r) sG0[(d & 1) * NB9 + r * BP + t] = gv[r];
        }
        gsync<NT>(g);
      }
      if (t < B)
#pragma unroll
        for (int r = 0; r < 9; ++r) a.lq[kf * (9 * B) + r * B + t] = sL[r * BP + t] + sG0[r * BP + t];
      gsync<NT>(g);   // the group's region is refilled for the next simulation or element
    }
    // the star sums over the columns, in order
    if (t < B)
#pragma unroll
      for (int q = 0; q < 3; ++q) sScr[q * B + t] = wst[q];
    gsync<NT>(g);
    if (t < 3) {
      double acc = 0.0;
      for (int x = 0; x < B; ++x) acc += (double)sScr[t * B + x];
      atomicAdd(Wk + WG_STAR + t, acc);
    }
    gsync<NT>(g);
  }
}

// Reverse of a neighbour pass, one CTA per buffer owner (every element): for each face
// whose neighbour (the receiver) was active, the receiver's transposed flux goes to the
// adjoint of the buffer it read, and the receiver's ten sums with that buffer are
// accumulated. Every (receiver, face) pair is visited by exactly one owner. The four faces
// are handled together: with LF = lambda_k F^_ip^T and XF = X F-_jh (9 x F each), the
// transposed flux is (A+^T LF) F-_jh^T and the sums are face_products of LF and XF. Bound by
// instruction issue (59 % of the issue slots, two fifths of the stalls on operator-table loads), so
// the CTA has a thread for every (side, face, face mode), then (face, face mode), (face, mode) and
// (row, mode), and blocks of a multiple of 16 bytes (order 4) move four entries at a time: 147 us
// a launch; 167 with single entries, 187 with one warp an owner (47,040 elements, order 4, two
// clusters, mean of both).
template <int O>
struct AdjNbrNT {
  static constexpr int value = rup(8 * nface(O), 32);
};
template <int O>
__global__ void __launch_bounds__(AdjNbrNT<O>::value) k_adj_nbr(DevOps ops, AdjLtsArgs a, PhaseArgs ph) {
  constexpr int B = nbasis(O), F = nface(O), BP = rup(B, 4), FP = rup(F, 4), NB9 = 9 * B;
  __shared__ __align__(16) float sA[4][108];
  __shared__ __align__(16) float sLk[4][9 * BP], sX[4][9 * BP];
  __shared__ __align__(16) float sLF[4][9 * FP];   // then A+^T LF
  __shared__ float sXF[4][9 * FP], sP9[4][FP];     // then the ten products
  __shared__ float sN[4][3];
  __shared__ int sF[8], sBk[8];
  const int kn = a.owners ? a.owners[blockIdx.x] : (int)blockIdx.x, t = threadIdx.x;
  if (t < 8) {
    sF[t] = a.fwd[kn * 8 + t];
    sBk[t] = a.back[kn * 8 + t];
  }
  __syncthreads();
  // buffer each active receiver read: 0 B1 (same cluster), 1 B3 (receiver coarser),
  // 2 B2 / 3 B1 - B2 (receiver finer, first / second half); -1 receiver not active
  const int lo = a.meta[kn] & 0xff, s2 = a.slot2[kn], s3 = a.slot3[kn];
  // modes packed 3 bits per face as mode + 1, so that a runtime face index needs no stack
  int modes = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = sF[2 * i];
    if (k < 0 || k >= a.end) continue;
    const int lr = a.meta[k] & 0xff;
    const int m = (lo == lr - 1) ? 1 : (lo == lr + 1) ? ((ph.parity[lr] == 0) ? 2 : 3) : 0;
    modes |= (m + 1) << (3 * i);
  }
  if (modes == 0) return;   // the same for every thread of the CTA
  auto mode = [modes](int i) { return ((modes >> (3 * i)) & 7) - 1; };
  constexpr int NT = AdjNbrNT<O>::value, R = (NB9 + NT - 1) / NT;
  // order 4: rows without pads and blocks of a multiple of 16 bytes, moved four entries at a time
  constexpr bool V4 = B % 4 == 0;
  constexpr int V = V4 ? NB9 / 4 : 1;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (mode(i) >= 0) {
      const float* am = a.amat + (size_t)sF[2 * i] * AM_SIZE;
      for (int q = t; q < 81; q += NT) sA[i][(q / 9) * 12 + q % 9] = __ldg(am + AM_NBR + sBk[2 * i] * 81 + q);
      if (t < 3) sN[i][t] = __ldg(am + AM_GEO + AM_NRM + 3 * sBk[2 * i] + t);
    }
  // pad entries of the rows: zero, never written afterwards
  for (int q = t; q < 36; q += NT) {
#pragma unroll
    for (int x = B; x < BP; ++x) sLk[q / 9][(q % 9) * BP + x] = sX[q / 9][(q % 9) * BP + x] = 0.f;
#pragma unroll
    for (int x = F; x < FP; ++x) sLF[q / 9][(q % 9) * FP + x] = 0.f;
  }
  for (int sim = 0; sim < a.nsim; ++sim) {
    // this simulation's block of the owner's buffers (stride G between modes)
    const size_t so = (size_t)(sim / a.G) * (NB9 * a.G) + sim % a.G;
    const float* b1 = a.B1s + (size_t)kn * a.bufs + so;
    const float* b2 = a.B2s + (size_t)s2 * a.bufs + so;
    const float* b3 = a.B3s + (size_t)s3 * a.bufs + so;
    if (V4 && a.G == 1) {   // (fused simulations: G apart)
      for (int p = t; p < 4 * V; p += NT) {
        const int i = p / V, q = p % V, m = mode(i);
        if (m < 0) continue;
        const float* b0 = (m == 1) ? b3 : (m == 2) ? b2 : b1;
        const float4 l = __ldg(reinterpret_cast<const float4*>(a.lq + ((size_t)sF[2 * i] * a.nsim + sim) * NB9) + q);
        float4 x = __ldg(reinterpret_cast<const float4*>(b0) + q);
        if (m == 3) {
          const float4 x2 = __ldg(reinterpret_cast<const float4*>(b2) + q);
          x.x -= x2.x;
          x.y -= x2.y;
          x.z -= x2.z;
          x.w -= x2.w;
        }
        reinterpret_cast<float4*>(sLk[i])[q] = l;
        reinterpret_cast<float4*>(sX[i])[q] = x;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int m = mode(i);
        if (m < 0) continue;
        const int k = sF[2 * i];
        stage_pad<B, BP, NT>(sLk[i], a.lq + ((size_t)k * a.nsim + sim) * NB9, 1, t);
        const float* b0 = (m == 1) ? b3 : (m == 2) ? b2 : b1;
        float x[R], x2[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int q = t + j * NT;
          x[j] = x2[j] = 0.f;
          if (q < NB9) {
            x[j] = __ldg(b0 + (size_t)q * a.G);
            if (m == 3) x2[j] = __ldg(b2 + (size_t)q * a.G);
          }
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int q = t + j * NT;
          if (q < NB9) sX[i][(q / B) * BP + q % B] = x[j] - x2[j];
        }
      }
    }
    __syncthreads();
    for (int p = t; p < 8 * F; p += NT) {
      const int i = (p / F) % 4, f = p % F;
      if (mode(i) < 0) continue;
      const int ip = sBk[2 * i], jh = sBk[2 * i + 1];
      const bool state = p >= 4 * F;
      float v[9];
      rows9v<B, BP>(state ? sX[i] : sLk[i], state ? ops.Fb + jh * B * F : a.FhT + ip * B * F, F, f, v);
      float* dst = state ? sXF[i] : sLF[i];
#pragma unroll
      for (int r = 0; r < 9; ++r) dst[r * FP + f] = v[r];
    }
    __syncthreads();
    for (int p = t; p < 4 * F; p += NT) {
      const int i = p / F, f = p % F;
      if (mode(i) < 0) continue;
      float lf[9], xf[9], u[9], o[10];
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        lf[r] = sLF[i][r * FP + f];
        xf[r] = sXF[i][r * FP + f];
      }
      flux_transposed(sA[i], lf, u);
      face_products(sN[i], lf, xf, o);
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        sLF[i][r * FP + f] = u[r];
        sXF[i][r * FP + f] = o[r];
      }
      sP9[i][f] = o[9];
    }
    __syncthreads();
    // the transposed fluxes, in place of the receivers' adjoints
    for (int p = t; p < 4 * B; p += NT) {
      const int i = p / B, b = p % B;
      if (mode(i) < 0) continue;
      float y[9];
      rows9v<F, FP>(sLF[i], a.FbT + sBk[2 * i + 1] * F * B, B, b, y);
#pragma unroll
      for (int r = 0; r < 9; ++r) sLk[i][r * BP + b] = y[r];
    }
    for (int p = t; p < 40; p += NT) {
      const int i = p / 10, q = p % 10;
      if (mode(i) < 0) continue;
      float acc = 0.f;
#pragma unroll
      for (int f = 0; f < F; ++f) acc += q < 9 ? sXF[i][q * FP + f] : sP9[i][f];
      atomicAdd(a.W + (size_t)sF[2 * i] * WG_SIZE + WG_NBR + sBk[2 * i] * 10 + q, (double)acc);
    }
    __syncthreads();
    // the faces' contributions summed per buffer in order, then one update of each adjoint touched
    if constexpr (V4) {
      for (int p = t; p < V; p += NT) {
        float4 y1 = make_float4(0.f, 0.f, 0.f, 0.f), y2 = y1, y3 = y1;
        bool u1 = false, u2 = false, u3 = false;
        auto add = [](float4& d, const float4& y, float sgn) {
          d.x = fmaf(sgn, y.x, d.x);
          d.y = fmaf(sgn, y.y, d.y);
          d.z = fmaf(sgn, y.z, d.z);
          d.w = fmaf(sgn, y.w, d.w);
        };
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int m = mode(i);
          if (m < 0) continue;
          const float4 y = reinterpret_cast<const float4*>(sLk[i])[p];
          if (m == 1) add(y3, y, 1.f);
          if (m == 2) add(y2, y, 1.f);
          if (m == 0 || m == 3) add(y1, y, 1.f);
          if (m == 3) add(y2, y, -1.f);
          u1 |= (m == 0 || m == 3);
          u2 |= (m == 2 || m == 3);
          u3 |= (m == 1);
        }
        const size_t o = ((size_t)kn * a.nsim + sim) * V + p;
        if (u1) atomicAdd(reinterpret_cast<float4*>(a.lb1) + o, y1);
        if (u2) atomicAdd(reinterpret_cast<float4*>(a.lb2) + o, y2);
        if (u3) atomicAdd(reinterpret_cast<float4*>(a.lb3) + o, y3);
      }
    } else {
      for (int p = t; p < NB9; p += NT) {
        float y1 = 0.f, y2 = 0.f, y3 = 0.f;
        bool u1 = false, u2 = false, u3 = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int m = mode(i);
          if (m < 0) continue;
          const float y = sLk[i][(p / B) * BP + p % B];
          if (m == 1) y3 += y;
          if (m == 2) y2 += y;
          if (m == 0 || m == 3) y1 += y;
          if (m == 3) y2 -= y;
          u1 |= (m == 0 || m == 3);
          u2 |= (m == 2 || m == 3);
          u3 |= (m == 1);
        }
        const size_t o = ((size_t)kn * a.nsim + sim) * NB9 + p;
        if (u1) atomicAdd(a.lb1 + o, y1);
        if (u2) atomicAdd(a.lb2 + o, y2);
        if (u3) atomicAdd(a.lb3 + o, y3);
      }
    }
    __syncthreads();   // the staged blocks are refilled for the next simulation
  }
}

}  // namespace ltsdev
