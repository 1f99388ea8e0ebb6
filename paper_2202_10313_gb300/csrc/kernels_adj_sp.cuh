// k_adj_pred_sp: the reverse of a predict pass of the clustered-LTS adjoint (elastic, one or
// fused simulations) with the operator products in generated sparse form, the counterpart of
// k_predict_sp for the transposed scheme. The arithmetic is that of k_adj_pred (see there
// and kernels_adj.cuh for the derivation); only the organisation differs:
//   row phase:    thread = (part, pair), pair = (element e, quantity row r); the thread keeps
//                 one row of its operand in registers and forms one part of the generated
//                 products with the nonzero entries of K_c and F~_i as immediate operands
//                 (sparse_ops.cuh): the time kernel D_d K_c^T (forward recomputation, and
//                 V_c = lambda K_c^T), the face traces lambda F~_i and T F~_i (F^_i = F~_i^T in
//                 the orthonormal face basis), the summed transposed traces sum_i U_i F~_i^T
//                 and the reverse time kernel Z_c = G_{d+1} K_c on the support of level d;
//   column phase: thread = (element e, mode b): star matrices (S_c, S_c^T) and this mode's
//                 share of their three sums, Taylor weights, the buffer adjoints, and the next
//                 row operand;
//   face phase:   thread = (element, face, face mode): U_i = A-_i^T (lambda F~_i) and the ten
//                 products of lambda F~_i and T F~_i, in place of T F~_i; summed over the
//                 face modes per (element, face, product) while the time kernel starts.
// Staging arrays are [mode or output][pair] with an odd pair stride XP, as in k_predict_sp.
#pragma once
#include "kernels_adj.cuh"
#include "sparse_ops.cuh"

namespace ltsdev {

// elements per CTA and parts of the row phase (NT = rup(9 NE, 32) NPART threads, NE B <= NT)
template <int O>
struct AdjSpShape;
template <>
struct AdjSpShape<5> {
  static constexpr int NE = 7, NPART = 4;
};
template <>
struct AdjSpShape<4> {
  static constexpr int NE = 12, NPART = 2;
};
template <>
struct AdjSpShape<3> {
  static constexpr int NE = 12, NPART = 1;
};

// rows of D_0 .. D_{d-1}, D_j kept on its nbasis(O - j) modes
__host__ __device__ constexpr int adj_drow(int O, int d) {
  int r = 0;
  for (int j = 0; j < d; ++j) r += nbasis(O - j);
  return r;
}

template <int O>
struct AdjSpCfg {
  static constexpr int B = nbasis(O), F = nface(O);
  static constexpr int NE = AdjSpShape<O>::NE, NPART = AdjSpShape<O>::NPART;
  static constexpr int NPAIR = 9 * NE;
  static constexpr int RT = rup(NPAIR, 32);
  static constexpr int NT = RT * NPART;
  static_assert(NE * B <= NT, "column phase needs one thread per (element, mode)");
  static constexpr int XP = NPAIR | 1;                      // odd pair stride
  static constexpr int DROWS = adj_drow(O, O - 1);          // D_0 .. D_{O-2}
  static constexpr int WROWS = (3 * B > 8 * F) ? 3 * B : 8 * F;
  static_assert(3 * B * NE <= WROWS * XP, "star sums of a batch fit into the row outputs");
  static constexpr int S_X = 0;                             // [B] row operand
  static constexpr int S_T = S_X + B * XP;                  // [B] T
  static constexpr int S_D = S_T + B * XP;                  // [DROWS] D_d
  static constexpr int S_W = S_D + DROWS * XP;              // [3B] Y_c, V_c, Z_c or [8F] LF_i (U_i), TF_i
  static constexpr int S_GEO = rup(S_W + WROWS * XP, 4);    // [NE][AM_NGEO] geometry and material
  static constexpr int S_AL = S_GEO + NE * AM_NGEO;         // [NE][4][9][12] A-_i, rows padded to 12
  static constexpr int S_P9 = S_AL + NE * 432;              // [4F][NE] the tenth product
  static constexpr int S_META = S_P9 + 4 * F * NE;          // [NE] ints
  static constexpr int TOTAL = rup(S_META + NE, 4);
};

template <int O, int XP>
__device__ __forceinline__ void sp_trace(int part, const float* x, float* g) {
  if constexpr (O == 5) ltssp::sp_trace_o5<XP>(part, x, g);
  if constexpr (O == 4) ltssp::sp_trace_o4<XP>(part, x, g);
  if constexpr (O == 3) ltssp::sp_trace_o3<XP>(part, x, g);
}
template <int O, int XP>
__device__ __forceinline__ void sp_tproj(int part, const float* x, float* y) {
  if constexpr (O == 5) ltssp::sp_tproj_o5<XP>(part, x, y);
  if constexpr (O == 4) ltssp::sp_tproj_o4<XP>(part, x, y);
  if constexpr (O == 3) ltssp::sp_tproj_o3<XP>(part, x, y);
}
template <int O, int XP>
__device__ __forceinline__ void sp_kvol(int part, int variant, const float* x, float* y) {
  if constexpr (O == 5) ltssp::sp_kvol_o5<XP>(part, variant, x, y);
  if constexpr (O == 4) ltssp::sp_kvol_o4<XP>(part, variant, x, y);
  if constexpr (O == 3) ltssp::sp_kvol_o3<XP>(part, variant, x, y);
}
template <int O, int XP>
__device__ __forceinline__ void sp_time_adj(int part, int variant, const float* x, float* y) {
  if constexpr (O == 5) ltssp::sp_time_o5<XP>(part, variant, x, y);
  if constexpr (O == 4) ltssp::sp_time_o4<XP>(part, variant, x, y);
  if constexpr (O == 3) ltssp::sp_time_o3<XP>(part, variant, x, y);
}

template <int O>
__global__ void __launch_bounds__(AdjSpCfg<O>::NT, 2) k_adj_pred_sp(AdjLtsArgs a, PhaseArgs ph) {
  using S = AdjSpCfg<O>;
  constexpr int B = S::B, F = S::F, NE = S::NE, NT = S::NT, XP = S::XP;
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  float* sX = smem + S::S_X;
  float* sT = smem + S::S_T;
  float* sD = smem + S::S_D;
  float* sW = smem + S::S_W;
  float* sGeo = smem + S::S_GEO;
  float* sAl = smem + S::S_AL;
  float* sP9 = smem + S::S_P9;
  int* sMeta = reinterpret_cast<int*>(smem + S::S_META);
  const int tid = threadIdx.x;
  // column task (element, mode), modes fastest
  const bool act = tid < NE * B;
  const int es = act ? tid / B : 0, b = act ? tid % B : 0;
  const int col = 9 * es;
  // row task (part, pair): warp w takes part w mod NPART, as in k_predict_sp
  const int part = (tid >> 5) % S::NPART, pair = ((tid >> 5) / S::NPART) * 32 + (tid & 31);
  const bool ract = pair < S::NPAIR;
  const int nbatch = (a.end + NE - 1) / NE;

  for (int batch = blockIdx.x; batch < nbatch; batch += gridDim.x) {
    const int k0 = batch * NE;
    __syncthreads();   // the previous batch is done with shared memory
    const int k = k0 + es;
    const bool valid = act && k < a.end;
    // the batch's geometry, A-_i (rows padded)
    if (tid < NE) sMeta[tid] = (k0 + tid < a.end) ? a.meta[k0 + tid] : 0;
    for (int q = tid; q < NE * AM_NGEO; q += NT) {
      const int e = q / AM_NGEO, x = q % AM_NGEO;
      sGeo[q] = (k0 + e < a.end) ? __ldg(a.amat + (size_t)(k0 + e) * AM_SIZE + AM_GEO + x) : 0.f;
    }
    for (int q = tid; q < NE * 324; q += NT) {
      const int e = q / 324, x = q % 324;
      sAl[e * 432 + (x / 9) * 12 + x % 9] = (k0 + e < a.end) ? __ldg(a.amat + (size_t)(k0 + e) * AM_SIZE + AM_LOC + x) : 0.f;
    }
    float wst[3] = {0.f, 0.f, 0.f};   // this column's star sums over the simulations
    const int meta = valid ? a.meta[k] : 0;
    const int cl = meta & 0xff;
    // fused runs take the simulations of the batch in turn: the operator matrices are staged
    // once, the star sums run over the simulations and the faces' sums receive one addition
    // per simulation, in order
    for (int sim = 0; sim < a.nsim; ++sim) {
      // this simulation's adjoints [element][simulation][9][B]
      const size_t ao = ((size_t)k * a.nsim + sim) * (9 * B) + b;
      // D_0 = Q before the pass (this column; simulation-blocked state, groups of G)
      float T[9];
      {
        float v[9];
#pragma unroll
        for (int r = 0; r < 9; ++r) v[r] = 0.f;
        if (valid) {
          const float* q = a.Qs + (size_t)k * a.qs + (size_t)(sim / a.G) * (9 * B * a.G) + sim % a.G + (size_t)b * a.G;
#pragma unroll
          for (int r = 0; r < 9; ++r) v[r] = __ldg(q + (size_t)r * B * a.G);
        }
        if (act) {
#pragma unroll
          for (int r = 0; r < 9; ++r) {
            sX[b * XP + col + r] = v[r];
            sD[b * XP + col + r] = v[r];
            T[r] = ph.coef[cl][0] * v[r];
          }
        }
      }
      __syncthreads();
      if (sim == 0) {
        // the next batch's inputs into L2 while this batch computes: operator matrices, Q,
        // lambda and lambda_B1 of every simulation (128-byte lines)
        const int kn = k0 + gridDim.x * NE;
        if (kn < a.end) {
          const int nn = min(NE, a.end - kn);
          const long long la = (long long)nn * AM_SIZE, lqn = (long long)nn * a.nsim * 9 * B, lQ = (long long)nn * a.qs;
          const float* pa = a.amat + (size_t)kn * AM_SIZE;
          const float* pq = a.Qs + (size_t)kn * a.qs;
          const float* pl = a.lq + (size_t)kn * a.nsim * 9 * B;
          const float* pb = a.lb1 + (size_t)kn * a.nsim * 9 * B;
          for (long long off = 32LL * tid; off < la; off += 32LL * NT) asm volatile("prefetch.global.L2 [%0];" ::"l"(pa + off));
          for (long long off = 32LL * tid; off < lQ; off += 32LL * NT) asm volatile("prefetch.global.L2 [%0];" ::"l"(pq + off));
          for (long long off = 32LL * tid; off < lqn; off += 32LL * NT) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(pl + off));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(pb + off));
          }
        }
      }
      const float* Gk = sGeo + es * AM_NGEO;
      // ---- forward time kernel: D_{d+1} = sum_c S_c D_d K_c^T (variant d: D_d on nbasis(O - d)
      // modes, D_{d+1} on nbasis(O - 1 - d))
#pragma unroll 1
      for (int d = 0; d < O - 1; ++d) {
        if (ract) sp_time_adj<O, XP>(part, d, sX + pair, sW + pair);
        __syncthreads();
        const int nout = nbasis(O - 1 - d);
        if (act) {
          float v[9];
#pragma unroll
          for (int r = 0; r < 9; ++r) v[r] = 0.f;
          if (b < nout) {
            const StarGeo geo(Gk);
            StarFwd st;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              float y[9];
#pragma unroll
              for (int s = 0; s < 9; ++s) y[s] = sW[(c * B + b) * XP + col + s];
              st.add(geo, c, y);
            }
            st.get(geo, v);
          }
          const float c1 = ph.coef[cl][d + 1];
#pragma unroll
          for (int r = 0; r < 9; ++r) {
            T[r] = fmaf(c1, v[r], T[r]);
            sX[b * XP + col + r] = v[r];
          }
          if (d + 1 <= O - 2 && b < nout) {
            float* dp = sD + (adj_drow(O, d + 1) + b) * XP + col;
#pragma unroll
            for (int r = 0; r < 9; ++r) dp[r] = v[r];
          }
        }
        __syncthreads();
      }
      // ---- volume: V_c = lambda K_c^T (on nbasis(O - 1) modes), mu = -sum_c S_c^T V_c,
      // its star sums
      float lam[9], mu[9], muh[9];
#pragma unroll
      for (int r = 0; r < 9; ++r) lam[r] = 0.f;
      if (valid) {
        const float* lp = a.lq + ao;
#pragma unroll
        for (int r = 0; r < 9; ++r) lam[r] = lp[r * B];
      }
      if (act) {
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          sX[b * XP + col + r] = lam[r];
          sT[b * XP + col + r] = T[r];
        }
      }
      __syncthreads();
      if (ract) sp_time_adj<O, XP>(part, 0, sX + pair, sW + pair);
      __syncthreads();
      constexpr int NV = nbasis(O - 1);
      {
        float w[9];
#pragma unroll
        for (int r = 0; r < 9; ++r) w[r] = 0.f;
        if (act && b < NV) {
          const StarGeo geo(Gk);
          StarRev st;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            float v[9];
#pragma unroll
            for (int s = 0; s < 9; ++s) v[s] = sW[(c * B + b) * XP + col + s];
            st.add(geo, c, v);
          }
          st.get(geo, w);
          st.sums(T, -1.f, wst);
        }
#pragma unroll
        for (int r = 0; r < 9; ++r) mu[r] = -w[r];
      }
      __syncthreads();
      // ---- local surface: LF_i = lambda F~_i and TF_i = T F~_i (row phase)
      if (ract) {
        sp_trace<O, XP>(part, sX + pair, sW + pair);
        sp_trace<O, XP>(part, sT + pair, sW + 4 * F * XP + pair);
      }
      __syncthreads();
      // per (element, face, face mode): U_i = A-_i^T LF_i over LF_i, the ten products over TF_i
      for (int j = tid; j < NE * 4 * F; j += NT) {
        const int e = j / (4 * F), i = (j / F) % 4, f = j % F;
        float* lp = sW + (i * F + f) * XP + 9 * e;
        float* tp = lp + 4 * F * XP;
        float lf[9], tf[9], u[9], o[10];
#pragma unroll
        for (int s = 0; s < 9; ++s) {
          lf[s] = lp[s];
          tf[s] = tp[s];
        }
        flux_transposed(sAl + e * 432 + i * 108, lf, u);
        face_products(sGeo + e * AM_NGEO + AM_NRM + 3 * i, lf, tf, o);
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          lp[r] = u[r];
          tp[r] = o[r];
        }
        sP9[(i * F + f) * NE + e] = o[9];
      }
      // the adjoints of the buffers this pass wrote: lambda_B1 (+ lambda_B3) join mu,
      // lambda_B2 is mu_half; reset here (lambda_B3 survives an accumulation)
      float l13[9];
#pragma unroll
      for (int r = 0; r < 9; ++r) l13[r] = muh[r] = 0.f;
      if (valid) {
        const bool finer = meta & FLAG_FINER, coarser = meta & FLAG_COARSER;
        const bool even = ph.parity[cl] == 0;
        const size_t o = ao;
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          l13[r] = a.lb1[o + r * B] + (coarser ? a.lb3[o + r * B] : 0.f);
          if (finer) muh[r] = a.lb2[o + r * B];
        }
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          a.lb1[o + r * B] = 0.f;
          if (coarser && even) a.lb3[o + r * B] = 0.f;
          if (finer) a.lb2[o + r * B] = 0.f;
        }
      }
      __syncthreads();
      // mu += sum_i U_i F~_i^T (row phase, into the row operand's place)
      if (ract) sp_tproj<O, XP>(part, sW + pair, sX + pair);
      __syncthreads();
      // the faces' sums (one writer per entry, the simulations in turn); the row outputs are
      // written again after the next barrier
      for (int j = tid; j < 40 * NE; j += NT) {
        const int e = j / 40, i = (j / 10) % 4, q = j % 10;
        const float* p = q < 9 ? sW + (4 + i) * F * XP + 9 * e + q : sP9 + i * F * NE + e;
        const int ld = q < 9 ? XP : NE;
        float acc = 0.f;
#pragma unroll
        for (int f = 0; f < F; ++f) acc += p[f * ld];
        if (k0 + e < a.end) atomicAdd(a.W + (size_t)(k0 + e) * WG_SIZE + WG_LOC + 10 * i + q, (double)acc);
      }
      // ---- reverse time kernel: G_{O-1} = c_{O-1} mu + c'_{O-1} mu_half (over this column's
      // face sum: read and written by the same thread), then G_d = c_d mu + c'_d mu_half +
      // sum_c S_c^T Z_c with Z_c = G_{d+1} K_c, and the star sums against D_d
      if (act) {
#pragma unroll
        for (int r = 0; r < 9; ++r) {
          mu[r] += sX[b * XP + col + r];
          mu[r] += l13[r];
          sX[b * XP + col + r] = ph.coef[cl][O - 1] * mu[r] + ph.hcoef[cl][O - 1] * muh[r];
        }
      }
      __syncthreads();
      float g0[9];
#pragma unroll 1
      for (int d = O - 2; d >= 0; --d) {
        if (ract) sp_kvol<O, XP>(part, d, sX + pair, sW + pair);
        __syncthreads();
        const int nout = nbasis(O - d);
        if (act) {
          float gv[9];
#pragma unroll
          for (int r = 0; r < 9; ++r) gv[r] = ph.coef[cl][d] * mu[r] + ph.hcoef[cl][d] * muh[r];
          // Z_c[0] = 0 (not written)
          if (b >= 1 && b < nout) {
            const StarGeo geo(Gk);
            StarRev st;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              float z[9];
#pragma unroll
              for (int r = 0; r < 9; ++r) z[r] = sW[(c * B + b) * XP + col + r];
              st.add(geo, c, z);
            }
            float w[9], x[9];
            st.get(geo, w);
            const float* dp = sD + (adj_drow(O, d) + b) * XP + col;
#pragma unroll
            for (int r = 0; r < 9; ++r) {
              gv[r] += w[r];
              x[r] = dp[r];
            }
            st.sums(x, 1.f, wst);
          }
#pragma unroll
          for (int r = 0; r < 9; ++r) {
            sX[b * XP + col + r] = gv[r];
            g0[r] = gv[r];
          }
        }
        __syncthreads();
      }
      if (valid) {
        float* lp = a.lq + ao;
#pragma unroll
        for (int r = 0; r < 9; ++r) lp[r * B] = lam[r] + g0[r];
      }
    }  // simulations
    // the batch's star sums over the columns, in order, into the FP64 totals
    if (act)
#pragma unroll
      for (int q = 0; q < 3; ++q) sW[q * (NE * B) + tid] = wst[q];
    __syncthreads();
    for (int q = tid; q < 3 * NE; q += NT) {
      const int e = q / 3;
      const float* p = sW + (q % 3) * (NE * B) + e * B;
      double acc = 0.0;
      for (int x = 0; x < B; ++x) acc += (double)p[x];
      if (k0 + e < a.end) atomicAdd(a.W + (size_t)(k0 + e) * WG_SIZE + WG_STAR + q % 3, acc);
    }
  }
}

}  // namespace ltsdev
