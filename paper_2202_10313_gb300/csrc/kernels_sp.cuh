// k_predict_sp: the predict + local kernel (time kernel, LTS buffers, volume kernel, local
// surface kernel; Sec. III-A and Eq. lts_buffers) with the operator products in generated
// sparse form (one simulation, or (element, simulation) slots of fused simulations), and
// k_neighbour_sp, the neighbour surface kernel of the same engine (below).
//
// The products run on the rows the scheme needs and on no others. The star matrices are
// combinations A_c = sum_d A_d dxi_c/dx_d, and A_d maps velocities to stresses and the stress
// row sigma_d to velocities, so
//   sum_c A_c X K_c^T  needs  K_c v_j  for the three velocities (nine velocity gradients) and
//                             K_c tau_c with tau_c = sum_d dxi_c/dx_d sigma_d (three rows per
//                             direction c, whose sum over c is the stress divergence),
// 6 rows per K_c instead of 9: a third of the multiply-adds and of the staged results go. The
// same rows carry the surface terms: dxi_c/dx is -2|S|/|det J| times the normal of the face
// opposite to coordinate c (the fourth direction is -sum_c dxi_c/dx), so tau_c is that face's
// scaled traction, the face's interface state (v*, scaled t*) projected through F^ adds to the
// set of direction c, and one application of Hooke's law gives volume and surface terms together
// (no flux rows per face).
//
// A derivative (and the volume / trace step, and the projection) is done in two phases
// separated by a barrier:
//   row phase:    lane = (row, element), elements fastest; a warp takes one part of the
//                 generated products (immediate operands, sparse_ops.cuh) for two rows of all
//                 16 elements, reading and writing its rows four modes at a time. No operator
//                 entry is read from memory and the structural zeros of K_c and F~_i (Sec. IV-A
//                 "all sparsity") are not multiplied.
//   column phase: thread = (element e, mode b), modes fastest (fused simulations: the
//                 simulations of an element fastest): it combines the products of its mode
//                 with dxi/dx and Hooke's law, applies the anelastic coupling and relaxation,
//                 adds the Taylor terms and writes the next derivative's rows.
// Staged rows are [element][row][mode] with an odd row stride and an odd element stride in
// 16-byte units (eight lanes' 16-byte accesses fall on distinct banks), and an element stride
// equal to the padded mode count modulo 32, so that the column phase's consecutive threads do too.
// A batch's DOFs and element tables arrive in shared memory by bulk asynchronous copies (TMA),
// issued a batch ahead. Receivers and sources are those of kernels.cuh.
#pragma once
#include "kernels.cuh"
#include "sparse_ops.cuh"
#include "tc.cuh"

namespace ltsdev {

// Shape of the predict kernel: a batch of 16 elements, so that the six rows of a set are three
// full warps of (row, element) lanes. BP: padded modes of a row, GP: stride of a face-state row, GS:
// of a face's six rows, YT: of a time-kernel product's row, BBP: padded modes of top degree (column
// phase). Order 5: one CTA per SM (the straight-line code of one phase at a time in the
// instruction cache).
// What bounds it (order 5, anelastic; about 20,700 cycles per 16 elements): phases of 18 warps
// between barriers, each short of the SM's limits by its own latency. Time kernel: row phases
// 5,000 cycles over the four derivatives (staged reads, multiply-adds), column phases 6,400 (issue:
// Hooke's law, coupling and relaxation); volume and traces 3,200, interface states 2,600,
// projection 1,800, update 1,900. 57 % of the issue slots, 2,964 warp instructions and 764
// shared-memory wavefronts per element; barriers are the largest stall. Measured on one GB300,
// 138,240 elements, ns per element, with nine rows per K_c and 14-element batches (order 5) before
// and with the row form now:
//   order 5, 3 mechanisms: 6.59 -> 4.19 (one cluster), 6.95 -> 4.82 (four clusters: half-step
//   traces 0.42 of it); elastic 4.52 -> 3.19; 16 simulations 6.85 -> 4.62
//   order 4: 3.09 -> 2.14, elastic 2.24 -> 1.37; order 3: 2.27 -> 1.03, elastic 1.13 -> 0.66
// No gain from: the next batch started without a barrier after the update (-0.7 % with one cluster,
// +1.4 % with four), the interface states with a face per lane, 15 instead of 16 row parts, two
// CTAs of 8 elements per SM at order 5 (4.26 -> 4.92 when measured: instruction fetch).
template <int O>
struct SpShape;
template <>
struct SpShape<5> {
  static constexpr int BP = 36, GP = 20, GS = 144, YT = 20, BBP = 16, ESM = 20, MINB = 1;
};
template <>
struct SpShape<4> {
  static constexpr int BP = 20, GP = 12, GS = 72, YT = 12, BBP = 10, ESM = 12, MINB = 2;
};
template <>
struct SpShape<3> {
  static constexpr int BP = 12, GP = 12, GS = 72, YT = 4, BBP = 6, ESM = 4, MINB = 3;
};

// Floats of an element's row in the sparse engine's tables (16-byte aligned rows). Predict:
//   [0..8] dxi_c/dx_d, [9..11] -sum_c dxi_c/dx_d, lam, mu, 1/rho, [15 + 2l] lam Y^lam_l,
//   [16 + 2l] 2 mu Y^mu_l, [23] cluster and flags (int); [24 + 12 f] of face f: normal n, then
//   a0, a1/s, a2, s a3 of the normal and of the tangential pair, s = -2|S|/|det J|; [21] (int) two
//   bits per face: 0 no neighbour, 1 neighbour in the same cluster, 2 finer, 3 coarser.
// Neighbour: [0..14] as above, [16 + 12 f] the same for the neighbour side's trace (its theta is
//   scaled by its own s_n and its own normal): n, then an0, -an1/s_n, -s an2/s_n, s an3.
constexpr int EDS = 72, NDS = 64;

// Face traces, the LTS buffers of the sparse engine: per (element, simulation) and face the six
// rows (v, theta) in the face basis, FS floats (16-byte multiple). The neighbour kernel wants
// X F~_j of the neighbour's buffer on its face j, and the predict kernel forms just that product
// for its own surface term: storing the trace (O = 5: 4 x 368 bytes per element instead of
// 1,260) leaves the neighbour kernel 368 bytes to read per face instead of 1,260, and no face
// product. A face serves one neighbour, so it needs only the buffer that neighbour reads:
//   same cluster:     T1 = trace of B1
//   coarser neighbour: T1 = trace of B3 (set at even steps, added to at odd ones)
//   finer neighbour:  T1 = trace of B2 (first half), T2 = trace of B1 - B2 (second half)
template <int F>
struct TraceCfg {
  static constexpr int FS = rup(6 * F, 4), TS = 4 * FS;
};

// The direction whose stress rows are the tractions of face f.
__host__ __device__ constexpr int set_of_face(int f) { return f < 3 ? 2 - f : 3; }

template <int O, int M, bool FU = false>
struct SpCfg {
  using C = Cfg<O, M, 1>;
  using H = SpShape<O>;
  static constexpr int B = C::B, F = C::F, NQ = C::NQ, NA = C::NA;
  static constexpr int NE = 16;
  static constexpr int BP = H::BP, GP = H::GP, GS = H::GS, YT = H::YT;
  // column phase: threads of the modes below the top degree (BA per element) first, then those
  // of the top degree (BB, padded to BBP): the time kernel's products vanish on the latter
  static constexpr int BA = nbasis(O - 1), BB = B - BA, BBP = H::BBP;
  static constexpr int NTA = NE * BA, NT = rup(NTA + NE * BBP, 32);
  static constexpr int NW = NT / 32;
  static_assert(NE % 8 == 0, "eight lanes of a row phase share a row (NE = 14 would straddle rows: bank conflicts)");
  static_assert(NTA % 32 == 0 && BP >= B && GP >= F && GS >= 6 * GP && BBP >= BB, "shape");
  static_assert(YT >= BA && (YT / 4) % 2 == 1 && (BP / 4) % 2 == 1 && (GP / 4) % 2 == 1, "row strides");
  static constexpr bool TM = M > 0;   // part of the column state lives in tensor memory
  // tensor-memory columns: TMW per warp of a lane quarter, a power of two in all
  static constexpr int TMW = 54, TMC = (NW + 3) / 4 * TMW <= 128 ? 128 : (NW + 3) / 4 * TMW <= 256 ? 256 : 512;
  // element strides: ESM modulo 32, odd in 16-byte units
  static constexpr int es(int n) { return n + (H::ESM - n % 32 + 32) % 32; }
  static constexpr int ESX = es(15 * BP);              // v (3), tau_0, tau_1, tau_2, tau_3 (3 rows each); then
                                                       // the projections of face 3 (6 rows)
  static constexpr int ESY = es(18 * BP);              // products of the sets 0..2, 6 rows each
  static constexpr int ESG = 4 * GS + 4;               // face traces, then interface states, in place
  static constexpr int S_X = 0;
  static constexpr int S_Y = S_X + NE * ESX;
  static constexpr int S_G = S_Y + NE * ESY;
  static constexpr int QBUF_ = FU ? NE * NQ * B : NE * C::QS;
  // order 5: the updated DOFs leave through shared memory by one bulk copy (over the face states,
  // which the next batch writes late); orders 3 and 4 have no room beside their other CTAs
  static constexpr bool STAGE = O == 5;
  static constexpr int S_E = S_G + rup(STAGE && QBUF_ > NE * ESG ? QBUF_ : NE * ESG, 4);   // [2][NE][EDS], double-buffered
  // the batch's DOFs: NE elements of QS floats (one simulation), or the simulation groups of its
  // NE slots (fused: groups of 4 consecutive slots, NE and the simulation count multiples of 4)
  static constexpr int QBUF = QBUF_;
  static constexpr int S_Q = rup(S_E + 2 * NE * EDS, 4);
  static constexpr int S_F = rup(S_Q + QBUF, 4);       // [4][B][F] F~ (half-step traces)
  static constexpr int S_SLOT = rup(S_F + 4 * B * F, 4);   // fused: [2][2][NE] element, simulation of the slots
  static constexpr int S_BAR = rup(S_SLOT + (FU ? 4 * NE : 0), 4);   // mbarrier of the copies (8 bytes)
  static constexpr int TOTAL = S_BAR + 4;                             // and the tensor-memory address
};

// Jobs of the row phases: (part, third of its rows: two of the six), job j for warp j mod NW. Four
// bits each, part * 3 + third. Order 5: the 12 jobs of warps w, w + 4, w + 8 (one scheduler's) add
// up to nearly equal multiply-add counts: time kernel parts K_0 (108), K_1 (252), K_2 (144, 143);
// volume and traces: direction 3 (309), 0 (471), 1 (357), 2 (390); projection: the faces (103, 105,
// 363, 309).
template <int N>
constexpr uint64_t job_table(const int (&c)[N]) {
  uint64_t t = 0;
  for (int j = 0; j < N; ++j) t |= (uint64_t)c[j] << (4 * j);
  return t;
}
template <int O>
struct SpJobs;
template <>
struct SpJobs<5> {
  static constexpr int NT = 12, NV = 12, NP = 16;   // 15: none
  static constexpr uint64_t T = job_table({3, 4, 5, 9, 6, 7, 8, 10, 0, 1, 2, 11});
  static constexpr uint64_t V = job_table({3, 4, 5, 10, 6, 7, 9, 11, 0, 1, 2, 8});
  static constexpr uint64_t P = job_table({6, 7, 8, 11, 9, 10, 0, 2, 15, 15, 1, 4, 15, 15, 3, 5});
};
template <>
struct SpJobs<4> {   // ten warps: two of them take the light jobs of the volume phase in pairs
  static constexpr int NT = 9, NV = 12, NP = 9;
  static constexpr uint64_t T = job_table({6, 7, 8, 3, 4, 5, 0, 1, 2});
  static constexpr uint64_t V = job_table({0, 2, 3, 4, 5, 9, 10, 11, 7, 8, 1, 6});
  static constexpr uint64_t P = job_table({0, 1, 2, 3, 4, 5, 6, 7, 8});
};
template <>
struct SpJobs<3> {   // one part (five warps: several jobs each measured slower)
  static constexpr int NT = 3, NV = 3, NP = 3;
  static constexpr uint64_t T = job_table({0, 1, 2}), V = T, P = T;
};

// the generated products of order O
template <int O, int DY>
__device__ __forceinline__ void sg_time(int variant, int part, const float* x, int dx, float* y) {
  if constexpr (O == 5) ltssp::sg_time_o5<DY>(variant, part, x, dx, y);
  if constexpr (O == 4) ltssp::sg_time_o4<DY>(variant, part, x, dx, y);
  if constexpr (O == 3) ltssp::sg_time_o3<DY>(variant, part, x, dx, y);
}
template <int O, int DY, int DG>
__device__ __forceinline__ void sg_vol(int part, const float* x, int dx, float* y, float* g) {
  if constexpr (O == 5) ltssp::sg_vol_o5<DY, DG>(0, part, x, dx, y, g);
  if constexpr (O == 4) ltssp::sg_vol_o4<DY, DG>(0, part, x, dx, y, g);
  if constexpr (O == 3) ltssp::sg_vol_o3<DY, DG>(0, part, x, dx, y, g);
}
template <int O, int DY, int DG>
__device__ __forceinline__ void sg_proj(int part, const float* g, float* y, float* p) {
  if constexpr (O == 5) ltssp::sg_proj_o5<DY, DG>(0, part, g, y, p);
  if constexpr (O == 4) ltssp::sg_proj_o4<DY, DG>(0, part, g, y, p);
  if constexpr (O == 3) ltssp::sg_proj_o3<DY, DG>(0, part, g, y, p);
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// dxi_c/dx_d of an element, c = 3: -sum of the others (the first 12 floats of its table row)
struct Geo {
  float J[4][3];
  __device__ __forceinline__ explicit Geo(const float* ed) {
    const float4 a = ld4(ed), b = ld4(ed + 4), c = ld4(ed + 8);
    J[0][0] = a.x, J[0][1] = a.y, J[0][2] = a.z, J[1][0] = a.w, J[1][1] = b.x, J[1][2] = b.y;
    J[2][0] = b.z, J[2][1] = b.w, J[2][2] = c.x, J[3][0] = c.y, J[3][1] = c.z, J[3][2] = c.w;
  }
};

// Rows of one mode for the row phase: v_j, then tau_c of the first NSET directions.
template <int NSET, int BP>
__device__ __forceinline__ void put_rows(float* x, const float (&q)[9], const Geo& g) {
#pragma unroll
  for (int j = 0; j < 3; ++j) x[j * BP] = q[6 + j];
#pragma unroll
  for (int c = 0; c < NSET; ++c) {
    x[(3 + 3 * c) * BP] = g.J[c][0] * q[0] + g.J[c][1] * q[3] + g.J[c][2] * q[5];
    x[(4 + 3 * c) * BP] = g.J[c][0] * q[3] + g.J[c][1] * q[1] + g.J[c][2] * q[4];
    x[(5 + 3 * c) * BP] = g.J[c][0] * q[5] + g.J[c][1] * q[4] + g.J[c][2] * q[2];
  }
}

// Hooke's law of a velocity gradient G[d][j] = d v_j / d x_d: stress rows (the elastic Jacobians'
// velocity part) and eps = sym grad v.
__device__ __forceinline__ void hooke(const float (&G)[3][3], float lam, float mu, float (&out)[9], float (&eps)[6]) {
  const float ltr = lam * (G[0][0] + G[1][1] + G[2][2]), m2 = 2.f * mu;
  const float sxy = G[0][1] + G[1][0], syz = G[1][2] + G[2][1], sxz = G[0][2] + G[2][0];
  out[0] = fmaf(m2, G[0][0], ltr);
  out[1] = fmaf(m2, G[1][1], ltr);
  out[2] = fmaf(m2, G[2][2], ltr);
  out[3] = mu * sxy;
  out[4] = mu * syz;
  out[5] = mu * sxz;
  eps[0] = G[0][0];
  eps[1] = G[1][1];
  eps[2] = G[2][2];
  eps[3] = 0.5f * sxy;
  eps[4] = 0.5f * syz;
  eps[5] = 0.5f * sxz;
}

// Upwind (Godunov) interface state of a face state g = (v, theta), theta the traction times the
// face's s = -2|S|/|det J| (of the trace's own element), in closed form, as riemann_state of
// kernels.cuh: fd = n, then the four coefficients of the normal and of the tangential pair, with
// the factors of s folded in (EDS above). w = (v*, s t*).
__device__ __forceinline__ void interface_state(const float (&g)[6], const float* fd, float (&w)[6]) {
  const float4 f0 = ld4(fd), f1 = ld4(fd + 4), f2 = ld4(fd + 8);
  const float nx = f0.x, ny = f0.y, nz = f0.z;
  const float vn = g[0] * nx + g[1] * ny + g[2] * nz;
  const float tn = g[3] * nx + g[4] * ny + g[5] * nz;
  const float vTx = g[0] - vn * nx, vTy = g[1] - vn * ny, vTz = g[2] - vn * nz;
  const float tTx = g[3] - tn * nx, tTy = g[4] - tn * ny, tTz = g[5] - tn * nz;
  const float vsn = f0.w * vn + f1.x * tn;
  const float tsn = f1.y * tn + f1.z * vn;
  w[0] = vsn * nx + f1.w * vTx + f2.x * tTx;
  w[1] = vsn * ny + f1.w * vTy + f2.x * tTy;
  w[2] = vsn * nz + f1.w * vTz + f2.x * tTz;
  w[3] = tsn * nx + f2.y * tTx + f2.z * vTx;
  w[4] = tsn * ny + f2.y * tTy + f2.z * vTy;
  w[5] = tsn * nz + f2.y * tTz + f2.z * vTz;
}

// Slots of a phase: one simulation (FUSED false): slot = element; fused simulations: slot =
// (element, simulation), the simulations of an element consecutive, simulation f of element
// k at k * (element stride) + (f / G) * (rows x B x G) + (row x B + mode) x G + f mod G in the
// simulation-blocked layout (G = FUSED_GROUP). The per-slot arithmetic is the same either way.
// Slot counts fit 32 bits (checked when the mesh is set). Fused kernels decode a batch's
// slots once (one division each, by the first NE threads) into shared memory.
template <bool FUSED>
struct Slots {
  int nsim;
  int n;                                        // slots in the phase
  __device__ Slots(const DevState& st, const PhaseArgs& ph)
      : nsim(FUSED ? st.nsim : 1), n((ph.end - ph.begin) * (FUSED ? st.nsim : 1)) {}
  // element (offset from the phase's first) and simulation of slot t < n
  __device__ void decode(int t, int& e, int& f) const {
    if (!FUSED) {
      e = t;
      f = 0;
    } else {
      e = (int)((unsigned)t / (unsigned)nsim);
      f = t - e * nsim;
    }
  }
  // offset of (simulation f, row 0, mode 0) from its element's start in an array of `rows` rows
  __device__ static int sub(int f, int rows, int B) {
    if (!FUSED) return 0;
    return (int)((unsigned)f / FUSED_GROUP) * rows * B * FUSED_GROUP + (int)((unsigned)f % FUSED_GROUP);
  }
};

template <int O, int M, bool FUSED>
__global__ void __launch_bounds__(SpCfg<O, M, FUSED>::NT, SpShape<O>::MINB)
    k_predict_sp(DevOps ops, DevState st, PhaseArgs ph) {
  using S = SpCfg<O, M, FUSED>;
  using C = typename S::C;
  using J = SpJobs<O>;
  constexpr int B = S::B, F = S::F, NE = S::NE, NT = S::NT, NQ = S::NQ, NA = S::NA, BP = S::BP, YT = S::YT, GP = S::GP,
                GS = S::GS;
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  float* sX = smem + S::S_X;
  float* sY = smem + S::S_Y;
  float* sG = smem + S::S_G;
  float* sQ = smem + S::S_Q;
  float* sF = smem + S::S_F;
  uint64_t* sBar = reinterpret_cast<uint64_t*>(smem + S::S_BAR);
  const int tid = threadIdx.x;
  if (ph.bufs & BUFS_TRACES)
    for (int i = tid; i < 4 * B * F; i += NT) sF[i] = ops.Ft[i];

  // column task (slot, mode), modes fastest: the modes below the top degree of all slots (group A),
  // then the top-degree ones. Fused simulations: set per batch below.
  constexpr int BA = S::BA, BB = S::BB, NTA = S::NTA;
  const bool grpA = tid < NTA;
  constexpr int BBP = FUSED ? BB : S::BBP;
  const int tg = grpA ? tid : tid - NTA, bg = grpA ? BA : BBP;   // task within the group, modes per slot
  int es = FUSED ? 0 : tg / bg;
  int b = FUSED ? 0 : (grpA ? 0 : BA) + tg % bg;
  const bool act = grpA || (tg < NE * BBP && tg % BBP < BB);
  // row task: row r of the sets (velocity j = r, or stress row i = r - 3) of element re
  const int warp = tid >> 5, re = tid & 15;
  const Slots<FUSED> sl(st, ph);
  const int nbatch = (sl.n + NE - 1) / NE;
  const long long qs = FUSED ? st.qs : C::QS, bs = FUSED ? st.bs : C::BUFS;
  constexpr int RS = FUSED ? B * FUSED_GROUP : B;   // row stride of Q and the buffers
  constexpr int CS = FUSED ? FUSED_GROUP : 1;       // mode stride
  constexpr int GB = NQ * B * FUSED_GROUP, FS = TraceCfg<F>::FS;
  // A batch's DOFs and element tables arrive in shared memory by two bulk asynchronous copies
  // (TMA) that thread 0 issues for the next batch as soon as the current one has read its DOFs
  // (the tables are double-buffered), completing on an mbarrier (one phase per batch): one
  // simulation, the batch's contiguous elements (n x QS floats); fused simulations, the
  // contiguous simulation groups from the batch's first slot to its last. Every wait is
  // bounded; one that gives up sets the error word and the CTA returns.
  // A batch's first element, its elements, and its DOFs in Q (offset and bytes).
  auto span = [&](int bt, int& e0, int& ne, size_t& off, uint32_t& bytes) {
    if constexpr (!FUSED) {
      e0 = ph.begin + bt * NE;
      ne = min(NE, ph.end - e0);
      off = (size_t)e0 * C::QS;
      bytes = (uint32_t)ne * C::QS * 4;
    } else {
      int f0, e1, f1;
      sl.decode(bt * NE, e0, f0);
      sl.decode(min(sl.n, bt * NE + NE) - 1, e1, f1);
      ne = e1 - e0 + 1;
      e0 += ph.begin;
      off = (size_t)e0 * qs + (size_t)(f0 / FUSED_GROUP) * GB;
      bytes = (uint32_t)(min(NE, sl.n - bt * NE) / FUSED_GROUP) * GB * 4;
    }
  };
  auto issue = [&](int bt, int buf) {
    int e0, ne;
    size_t off;
    uint32_t bytes;
    span(bt, e0, ne, off, bytes);
    tc::bulk_load2(sQ, st.Q + off, bytes, smem + S::S_E + buf * NE * EDS, st.sdata + (size_t)e0 * EDS,
                   (uint32_t)ne * EDS * 4, sBar);
  };
  // The updated DOFs of batch bt, staged in sG, leave by one bulk copy.
  auto write_back = [&](int bt) {
    int e0, ne;
    size_t off;
    uint32_t bytes;
    span(bt, e0, ne, off, bytes);
    tc::bulk_store(st.Q + off, sG, bytes);
  };
  // Tensor memory as per-thread storage (anelastic): the time integrals and the half-step integrals
  // between the derivatives, and the update's known terms and the memory variables between the
  // volume products and the update. 18 warps of 96 registers hold the rest without spills
  // (spilling instead: 62 local-memory instructions per element, most of them missing L1).
  uint32_t* sTm = reinterpret_cast<uint32_t*>(smem + S::S_BAR + 2);
  uint32_t tm = 0;
  uint32_t qpar = 0;
  if (tid == 0) tc::mbar_init(sBar, 1);
  if constexpr (S::TM) {
    if (warp == 0) {
      tc::tmem_alloc(sTm, S::TMC);
      tc::tmem_relinquish();
    }
    tc::fence_before_sync();
  }
  __syncthreads();
  if constexpr (S::TM) {
    tc::fence_after_sync();
    tm = *sTm + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * S::TMW;
  }
  wait_for_previous_kernel();
  let_next_kernel_launch();
  if (tid == 0 && blockIdx.x < nbatch && !(ph.suppress & SUPPRESS_ALL)) issue(blockIdx.x, 0);

  int last = -1;   // the batch whose updated DOFs are staged (written back once the next has arrived)
  for (int batch = blockIdx.x; batch < nbatch; batch += gridDim.x) {
    const int t0 = batch * NE;
    const float* sE = smem + S::S_E + qpar * NE * EDS;
    // fused: element, simulation of the batch's slots
    int* sSlot = reinterpret_cast<int*>(smem + S::S_SLOT) + (FUSED ? qpar * 2 * NE : 0);
    // element of the batch's slot k (fused: decoded below, two copies in turn, as the last tasks
    // of a batch may still read theirs when the next one is decoded)
    auto elem_of = [&](int k) { return FUSED ? sSlot[k] : ph.begin + t0 + k; };
    if (FUSED && tid < NE) {
      int e = 0, f = 0;
      sl.decode(min(t0 + tid, sl.n - 1), e, f);   // slots past the end: a staged element
      sSlot[tid] = ph.begin + e;
      sSlot[NE + tid] = f;
    }
    // one simulation: the barrier of the DOF wait below follows the previous batch's update
    if constexpr (FUSED) __syncthreads();
    if (FUSED && act) {
      // fused column tasks ordered by (element, mode, simulation): the slots of the batch that
      // share an element form a segment [s0, s1), and its tasks of a group take the modes in
      // turn with the segment's simulations fastest, so that a warp's lanes read consecutive
      // floats of the simulation-blocked layout (tasks of slot m lie in segment of slot m)
      const int m = tg / bg;
      const int nval = min(NE, sl.n - t0);
      if (m < nval) {
        const int fm = sSlot[NE + m];
        const int s0 = max(0, m - fm), s1 = min(nval, m - fm + sl.nsim);
        const int local = tg - bg * s0, nf = s1 - s0;
        b = (grpA ? 0 : BA) + local / nf;
        es = s0 + local % nf;
      } else {
        es = m;
        b = (grpA ? 0 : BA) + tg % bg;
      }
    }
    const int ts = t0 + es;
    const bool valid = act && ts < sl.n;
    // (offsets into Q and the modal buffers are computed where they are needed: registers)
    // trace buffer of slot k
    auto trace_of = [&](int k) {
      return (FUSED ? (size_t)sSlot[k] * st.nsim + sSlot[NE + k] : (size_t)(ph.begin + t0 + k)) * TraceCfg<F>::TS;
    };
    // staged table row of slot k: its element's position in the batch
    auto ed_of = [&](int k) { return sE + (FUSED ? sSlot[k] - sSlot[0] : k) * EDS; };
    {
      // the batch's DOFs have arrived (or the wait gave up: every thread leaves)
      const bool ok = tc::mbar_wait(sBar, qpar, ph.wait);
      qpar ^= 1;
      if (!__syncthreads_and(ok)) {
        if (tid == 0) {
          atomicOr(ph.err, 1);
          tc::mbar_wait(sBar, qpar ^ 1, ph.wait);   // the copies in flight, if any, land first
          if (S::STAGE && last >= 0) write_back(last);   // the batch before is finished: its traces are out
        }
        break;
      }
    }
    if (S::STAGE && tid == 0 && batch != (int)blockIdx.x) write_back(batch - gridDim.x);
    // this column's DOFs in the staged copy (row stride RS, as in Q)
    int soff = es * C::QS + b;
    if constexpr (FUSED) soff = (es / FUSED_GROUP) * GB + b * CS + es % FUSED_GROUP;
    const float* ed = valid ? ed_of(es) : sE;
    const int meta = valid ? __float_as_int(ed[23]) : 0;
    const int cl = meta & 0xff;
    const bool finer = (meta & FLAG_FINER) != 0;
    const bool anyfiner = __any_sync(0xffffffffu, finer);
    float T[9], Th[9], Da[NA > 0 ? NA : 1];
    float* xo = sX + es * S::ESX + b;
    {
      float v[9];
      const float* q = sQ + soff;
#pragma unroll
      for (int r = 0; r < 9; ++r) v[r] = valid ? q[r * RS] : 0.f;
#pragma unroll
      for (int r = 0; r < NA; ++r) Da[r] = valid ? q[(9 + r) * RS] : 0.f;
      if (act) put_rows<3, BP>(xo, v, Geo(ed));
      const float c0 = ph.coef[cl][0], h0 = ph.hcoef[cl][0];
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        T[r] = c0 * v[r];
        Th[r] = h0 * v[r];
      }
      if constexpr (S::TM) {
        float ta[18];
#pragma unroll
        for (int r = 0; r < NA; ++r) ta[r] = ph.ra[cl][r / 6] * Da[r];
        tc::tmem_st18(tm, ta);
        tc::tmem_st9(tm + 18, T);
        if (anyfiner) tc::tmem_st9(tm + 27, Th);
        tc::tmem_wait_st();
      }
    }
    const bool batch_finer = __syncthreads_or(finer);
    // ---- time kernel: d^{d+1} Q from d^d Q (Cauchy-Kowalevski), Taylor sums
#pragma unroll 1
    for (int d = 0; d < O - 1; ++d) {
      // elastic: d^d Q has degree <= O-1-d, so the product is truncated (variant d); the
      // anelastic coupling keeps every degree (variant 0)
      const int variant = (M == 0) ? d : 0;
#pragma unroll 1
      for (int j = warp; j < J::NT; j += S::NW) {
        const int job = (int)(J::T >> (4 * j)) & 15, part = job / 3, r = 2 * (job % 3) + ((tid >> 4) & 1);
        sg_time<O, 6 * YT>(variant, part, sX + re * S::ESX + r * BP, r < 3 ? 0 : 3 * BP, sY + re * S::ESY + r * YT);
      }
      __syncthreads();
      const float c1 = ph.coef[cl][d + 1];
      float out[9], eps[6];
      // products of modes b >= nbasis(O-1-variant) are identically zero and not written (all of
      // the top degree: whole warps, whose memory variables follow in closed form)
      const bool has = grpA && b < nbasis(O - 1 - variant);
      if (has) {
        const float* yp = sY + es * S::ESY + b;
        float Y[3][6];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int r = 0; r < 6; ++r) Y[c][r] = yp[(6 * c + r) * YT];
        const Geo geo(ed);
        const float4 m0 = ld4(ed + 12);   // lam, mu, 1/rho, lam Y^lam_0
        float G[3][3];
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
          for (int j = 0; j < 3; ++j) G[e][j] = geo.J[0][e] * Y[0][j] + geo.J[1][e] * Y[1][j] + geo.J[2][e] * Y[2][j];
        hooke(G, m0.x, m0.y, out, eps);
#pragma unroll
        for (int i = 0; i < 3; ++i) out[6 + i] = m0.z * (Y[0][3 + i] + Y[1][3 + i] + Y[2][3 + i]);
      } else {
#pragma unroll
        for (int r = 0; r < 9; ++r) out[r] = 0.f;
      }
      if constexpr (M > 0) {
        const float4 m0 = ld4(ed + 12), m1 = ld4(ed + 16);
        const float ylam[3] = {m0.w, m1.y, m1.w}, ymu[3] = {m1.x, m1.z, ed[20]};
#pragma unroll
        for (int l = 0; l < M; ++l) coupling_add(out, Da + 6 * l, ylam[l] * ph.rp[l][d], ymu[l] * ph.rp[l][d]);
        if (grpA) {
          float ta[18];
          tc::tmem_ld18(tm, ta);
#pragma unroll
          for (int l = 0; l < M; ++l) {
            const float h = ph.rh[cl][l][d], g = ph.rg[l][d];
#pragma unroll
            for (int r = 0; r < 6; ++r) {
              ta[6 * l + r] = fmaf(h, eps[r], ta[6 * l + r]);
              Da[6 * l + r] = fmaf(g, eps[r], Da[6 * l + r]);
            }
          }
          tc::tmem_st18(tm, ta);
        }
        if (anyfiner) {
          const float h1 = ph.hcoef[cl][d + 1];
          tc::tmem_ld9(tm + 27, Th);
#pragma unroll
          for (int r = 0; r < 9; ++r) Th[r] = fmaf(h1, out[r], Th[r]);
          tc::tmem_st9(tm + 27, Th);
        }
        tc::tmem_ld9(tm + 18, T);
#pragma unroll
        for (int r = 0; r < 9; ++r) T[r] = fmaf(c1, out[r], T[r]);
        tc::tmem_st9(tm + 18, T);
        tc::tmem_wait_st();
      } else if (finer && has) {
        const float h1 = ph.hcoef[cl][d + 1];
#pragma unroll
        for (int r = 0; r < 9; ++r) Th[r] = fmaf(h1, out[r], Th[r]);
      }
      // next row operand: the next derivative, or after the last one the time integral
      if (act && (M > 0 || has || d == O - 2)) {
        if constexpr (!S::TM) {
#pragma unroll
          for (int r = 0; r < 9; ++r) T[r] = fmaf(c1, out[r], T[r]);
        }
        const Geo geo(ed);
        if (d < O - 2)
          put_rows<3, BP>(xo, out, geo);
        else
          put_rows<4, BP>(xo, T, geo);
      }
      // the previous batch's DOFs have left the face states' memory
      if (S::STAGE && tid == 0 && d == O - 2) tc::bulk_store_read_wait();
      __syncthreads();
    }
    // ---- LTS buffers as modes (Eq. lts_buffers): the adjoint and partitioned runs read those
    if (ph.bufs & BUFS_MODAL) {
      if constexpr (S::TM) {
        tc::tmem_ld9(tm + 18, T);
        if (anyfiner) tc::tmem_ld9(tm + 27, Th);
      }
      if (valid) {
        const size_t boff = (size_t)elem_of(es) * bs + Slots<FUSED>::sub(FUSED ? sSlot[NE + es] : 0, 9, B) + (size_t)b * CS;
        float* b1 = st.B1 + boff;
#pragma unroll
        for (int r = 0; r < 9; ++r) b1[r * RS] = T[r];
        if (finer) {
          float* b2 = st.B2 + boff;
#pragma unroll
          for (int r = 0; r < 9; ++r) b2[r * RS] = Th[r];
        }
        if (meta & FLAG_COARSER) {
          float* b3 = st.B3 + boff;
          if (ph.parity[cl] == 0) {
#pragma unroll
            for (int r = 0; r < 9; ++r) b3[r * RS] = T[r];
          } else {
#pragma unroll
            for (int r = 0; r < 9; ++r) b3[r * RS] += T[r];
          }
        }
      }
    }
    // the update's terms that are already known: Q + E^l T^{a,l}, and Q^{a,l}, kept apart from
    // T^{a,l} until the strain rate is known: what is added to a row of Q first costs it a rounding
    // (order 5, 34,560 elements, 4 steps against 64 bits: stress 1.26e-7 -> 1.05e-7 with the
    // mechanisms summed first, memory variables 1.13e-7 -> 1.07e-7 with one rounding; no slower)
    float acc[9];
    {
      const float* q = sQ + soff;
      if constexpr (M == 0) {
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[r] = valid ? q[r * RS] : 0.f;
      } else {
        float ta[18];
        tc::tmem_ld18(tm, ta);
        const float4 m0 = ld4(ed + 12), m1 = ld4(ed + 16);
        const float ylam[3] = {m0.w, m1.y, m1.w}, ymu[3] = {m1.x, m1.z, ed[20]};
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[r] = 0.f;
#pragma unroll
        for (int l = 0; l < M; ++l) coupling_add(acc, ta + 6 * l, ylam[l], ymu[l]);
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[r] += valid ? q[r * RS] : 0.f;
#pragma unroll
        for (int r = 0; r < NA; ++r) ta[r] = valid ? q[(9 + r) * RS] : 0.f;
        tc::tmem_st18(tm + 36, ta);
        tc::tmem_st9(tm + 18, acc);
        tc::tmem_wait_st();
      }
    }
    // ---- volume products and local face traces of T (row phase)
#pragma unroll 1
    for (int j = warp; j < J::NV; j += S::NW) {
      const int job = (int)(J::V >> (4 * j)) & 15, part = job / 3, r = 2 * (job % 3) + ((tid >> 4) & 1);
      sg_vol<O, 6 * BP, GS>(part, sX + re * S::ESX + r * BP, r < 3 ? 0 : 3 * BP, sY + re * S::ESY + r * BP,
                            sG + re * S::ESG + r * GP);
    }
    __syncthreads();
    // the batch's DOF copy has been read: the next batch's copies go out now
    if (tid == 0 && batch + (int)gridDim.x < nbatch && !ph.suppress) issue(batch + gridDim.x, qpar);
    // ---- face traces to the LTS buffers, and the local surface kernel's interface states (v*,
    // s t*) in their place; one task per element, face and face mode (face modes fastest)
#pragma unroll 1
    for (int t = tid; t < NE * 4 * F; t += NT) {
      const int fe = t / (4 * F), fi = (t / F) % 4, f = t % F;
      const float* ef = ed_of(fe);
      float* gp = sG + fe * S::ESG + fi * GS + f;
      float gv[6], w6[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) gv[r] = gp[r * GP];
      if ((ph.bufs & BUFS_TRACES) && t0 + fe < sl.n) {
        const int rel = (__float_as_int(ef[21]) >> (2 * fi)) & 3;
        const size_t o = trace_of(fe) + fi * FS + f;
        // added to in memory (no result read back: one addition per address and launch)
        if (rel == 3 && ph.parity[__float_as_int(ef[23]) & 0xff] != 0) {
#pragma unroll
          for (int r = 0; r < 6; ++r) atomicAdd(st.T1 + o + r * F, gv[r]);
        } else if (rel != 0) {
          float* tp = (rel == 2 ? st.T2 : st.T1) + o;
#pragma unroll
          for (int r = 0; r < 6; ++r) tp[r * F] = gv[r];
        }
      }
      interface_state(gv, ef + 24 + 12 * fi, w6);
#pragma unroll
      for (int r = 0; r < 6; ++r) gp[r * GP] = w6[r];
    }
    __syncthreads();
    // ---- projection through F^ (row phase): faces 0..2 onto the volume products of their
    // direction, face 3 into six rows of its own (over the time integral's rows)
#pragma unroll 1
    for (int j = warp; j < J::NP; j += S::NW) {
      const int job = (int)(J::P >> (4 * j)) & 15, part = job / 3, r = 2 * (job % 3) + ((tid >> 4) & 1);
      sg_proj<O, 6 * BP, GS>(part, sG + re * S::ESG + r * GP, sY + re * S::ESY + r * BP, sX + re * S::ESX + r * BP);
    }
    __syncthreads();
    // ---- update: volume and local surface terms of all four directions at once
    if constexpr (S::TM) tc::tmem_ld9(tm + 18, acc);
    // this column of Q (anelastic: also for the memory variables, past the branch)
    auto column = [&](int e) {
      return S::STAGE ? sG + soff : st.Q + (size_t)e * qs + Slots<FUSED>::sub(FUSED ? sSlot[NE + es] : 0, NQ, B) + (size_t)b * CS;
    };
    float* q = S::TM ? column(valid ? elem_of(es) : 0) : nullptr;
    float out[9], eps[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (valid) {
      const float* yp = sY + es * S::ESY + b;
      const Geo geo(ed);
      const float4 m0 = ld4(ed + 12);
      float G[3][3], dv[3];
      {
        float P[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) P[r] = xo[r * BP];
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
          for (int j = 0; j < 3; ++j) G[e][j] = geo.J[3][e] * P[j];
#pragma unroll
        for (int i = 0; i < 3; ++i) dv[i] = P[3 + i];
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float Z[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) Z[r] = yp[(6 * c + r) * BP];
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
          for (int j = 0; j < 3; ++j) G[e][j] = fmaf(geo.J[c][e], Z[j], G[e][j]);
#pragma unroll
        for (int i = 0; i < 3; ++i) dv[i] += Z[3 + i];
      }
      hooke(G, m0.x, m0.y, out, eps);
      if constexpr (!S::TM) q = column(elem_of(es));
#pragma unroll
      for (int r = 0; r < 6; ++r) q[r * RS] = acc[r] - out[r];
#pragma unroll
      for (int i = 0; i < 3; ++i) q[(6 + i) * RS] = fmaf(-m0.z, dv[i], acc[6 + i]);
      if (S::STAGE && !FUSED && b < C::QS - NQ * B) sG[es * C::QS + NQ * B + b] = 0.f;   // padding
    }
    if constexpr (S::TM) {
      float ta[18], qa[18];
      tc::tmem_ld18(tm, ta);
      tc::tmem_ld18(tm + 36, qa);
      if (valid) {
#pragma unroll
        for (int l = 0; l < M; ++l)
#pragma unroll
          for (int r = 0; r < 6; ++r)
            q[(9 + 6 * l + r) * RS] = fmaf(-ph.omega[l], ta[6 * l + r] + eps[r], qa[6 * l + r]);
      }
    }
    if constexpr (S::STAGE) tc::fence_smem_to_async();
    last = batch;
    // ---- half-step traces of the faces with a finer neighbour: rows of the half-step integral over
    // the projections (each thread its own column), then a warp per such face, lane = (velocity or
    // stress rows, face mode). The second half's trace is the step's (stored above) minus it.
    if ((ph.bufs & BUFS_TRACES) && batch_finer) {
      if constexpr (S::TM) {
        if (anyfiner) tc::tmem_ld9(tm + 27, Th);
      }
      if (valid && finer) put_rows<4, BP>(xo, Th, Geo(ed));
      __syncthreads();
      const int lane = tid & 31;
      unsigned faces[2];   // bit per (slot, face) of the batch
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int fe = 8 * h + lane / 4;
        faces[h] = __ballot_sync(0xffffffffu, t0 + fe < sl.n &&
                                                  ((__float_as_int(ed_of(fe)[21]) >> (2 * (lane % 4))) & 3) == 2);
      }
      const int half = lane / F, f = lane % F;
      int turn = 0;        // faces go round the warps
#pragma unroll 1
      for (int h = 0; h < 2; ++h)
#pragma unroll 1
      for (unsigned m = faces[h]; m; m &= m - 1) {
        const bool mine = turn == warp;
        turn = turn + 1 == S::NW ? 0 : turn + 1;
        if (!mine) continue;
        const int s = 32 * h + __ffs(m) - 1, fe = s / 4, fi = s % 4;
        if (half < 2) {
          const float* x = sX + fe * S::ESX + (half ? 3 + 3 * set_of_face(fi) : 0) * BP;
          const float* w = sF + fi * B * F + f;
          float gv[3] = {0.f, 0.f, 0.f};
#pragma unroll
          for (int k = 0; k < B; k += 4) {
            float4 xr[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) xr[r] = ld4(x + r * BP + k);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (k + j < B) {
                const float c = w[(k + j) * F];
#pragma unroll
                for (int r = 0; r < 3; ++r) gv[r] = fmaf(j == 0 ? xr[r].x : (j == 1 ? xr[r].y : (j == 2 ? xr[r].z : xr[r].w)), c, gv[r]);
              }
          }
          const size_t o = trace_of(fe) + fi * FS + 3 * half * F + f;
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            st.T1[o + r * F] = gv[r];
            atomicAdd(st.T2 + o + r * F, -gv[r]);
          }
        }
      }
    }
  }
  if constexpr (S::STAGE) {
    __syncthreads();
    if (tid == 0) {
      if (last >= 0 && last + (int)gridDim.x >= nbatch) write_back(last);
      tc::bulk_store_wait();
    }
  }
  if constexpr (S::TM) {
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tm, S::TMC);
  }
}

// ------------------------------------------------------------------ neighbour kernel
// k_neighbour_sp: the neighbour surface kernel (Sec. III-A, with the buffer chosen by the
// clusters' time-stepping relation, Sec. V-B) on the face traces the predict kernel stored
// (TraceCfg above). The neighbour matrices factor as F-_{j,h} = F~_j R_h (trace on the neighbour's
// face j, then the face-basis map R_h of the orientation, block diagonal by degree), and the
// trace is already there, so only R_h is left of the face product:
//   states:      thread = (element, face, face mode): H = G R_h (degree block), closed-form
//                interface state with the neighbour coefficients;
//   projection:  a warp per part of the generated F^ products (parts of equal multiply-add
//                count): 30 lanes = (row, element);
//   update:      thread = (element, mode): the faces' rows combined with dxi/dx and Hooke's law
//                once (as in k_predict_sp), Q <- Q + S^N.
// Everything a batch reads arrives by bulk asynchronous copies (TMA): a lane per face copies its
// neighbour's trace and thread 0 the element tables while the previous batch projects and
// updates, and the DOFs, which only the update reads, right after the previous update.
// Measured on one GB300 (order 5, anelastic, 138,240 elements): 1.99 ns per element (1.49 elastic)
// against 3.93 ns (3.43) with gathered buffers and face products in this kernel (4 x 1,260 bytes
// and 2,365 instructions per element). Bound by instruction issue and latency between its three
// barriers (41 % issue; DRAM 9.3 KB per element: 1.4 ns at the copy rate). Warps of two kinds that
// hand batches over through double buffers (no CTA barrier, two CTAs per SM instead of three)
// took 2.53 ns, and L2 prefetches one to four batches ahead 2.29-2.31 against 2.27 ns.
template <int O>
struct SpnShape;   // CTAs per SM, narrow and wide tile; GP: face row, BP: padded modes; ESW, ESP:
                   // element strides (conflict-free 16-byte accesses of 5 x 6 lanes)
template <>
struct SpnShape<5> {
  static constexpr int MIN1 = 3, MIN0 = 2, GP = 20, BP = 36, ESW = 484, ESP = 884;
};
template <>
struct SpnShape<4> {
  static constexpr int MIN1 = 5, MIN0 = 2, GP = 12, BP = 20, ESW = 316, ESP = 484;
};
template <>
struct SpnShape<3> {
  static constexpr int MIN1 = 7, MIN0 = 3, GP = 12, BP = 12, ESW = 316, ESP = 316;
};

// elements per CTA of a tile variant (fused: whole groups of simulations)
__host__ __device__ constexpr int spn_ne(int tile, bool fused) { return fused ? (tile ? 4 : 8) : (tile ? 5 : 10); }

template <int O, int M, int TILE, bool FU>
struct SpnCfg {
  using C = Cfg<O, M, 1>;
  using H = SpnShape<O>;
  static constexpr int B = C::B, F = C::F, NQ = C::NQ;
  static constexpr int NE = spn_ne(TILE, FU);
  static constexpr int GP = H::GP, GS = 6 * H::GP, BP = H::BP, ESW = H::ESW, ESP = H::ESP;
  static constexpr int NPP = O == 5 ? 6 : 4;                  // equal parts of the projection
  static constexpr int NL = 6 * NE, NWF = rup(NL, 32) / 32;   // its lanes, and warps per part
  static constexpr int NT = rup(NE * B, 32) > 32 * NPP * NWF ? rup(NE * B, 32) : 32 * NPP * NWF;
  static constexpr int MINB = TILE ? H::MIN1 : H::MIN0;
  static_assert(ESW >= 4 * GS && ESP >= 24 * BP && 4 * NE <= 64, "strides");
  static constexpr int FS = TraceCfg<F>::FS;
  static constexpr int S_T = 0;                        // [NE][4][FS] the neighbours' traces
  static constexpr int S_W = S_T + NE * 4 * FS;        // interface states
  static constexpr int S_P = S_W + NE * ESW;           // [4][6][BP] per element: projections
  static constexpr int S_Q = S_P + NE * ESP;           // DOFs
  static constexpr int S_D = S_Q + rup(NE * (FU ? NQ * B : C::QS), 4);   // [2][NE][NDS] tables, double-buffered
  static constexpr int S_R = S_D + 2 * NE * NDS;       // [3][F][F]
  static constexpr int S_I = rup(S_R + 3 * F * F, 4);  // [2][4 NE] ints: orientation or -1, double-buffered
  static constexpr int S_BAR = rup(S_I + 8 * NE, 4);   // two mbarriers
  static constexpr int TOTAL = S_BAR + 4;
};

template <int O, int DY, int DG>
__device__ __forceinline__ void sg_nproj(int part, const float* g, float* y) {
  if constexpr (O == 5) ltssp::sg_nproj_o5<DY, DG>(0, part, g, y);
  if constexpr (O == 4) ltssp::sg_nproj_o4<DY, DG>(0, part, g, y);
  if constexpr (O == 3) ltssp::sg_nproj_o3<DY, DG>(0, part, g, y);
}

template <int O, int M, int TILE, bool FUSED>
__global__ void __launch_bounds__(SpnCfg<O, M, TILE, FUSED>::NT, SpnCfg<O, M, TILE, FUSED>::MINB)
    k_neighbour_sp(DevOps ops, DevState st, PhaseArgs ph) {
  using S = SpnCfg<O, M, TILE, FUSED>;
  using C = typename S::C;
  constexpr int B = S::B, F = S::F, NE = S::NE, NT = S::NT, NQ = S::NQ, GP = S::GP, GS = S::GS, BP = S::BP, FS = S::FS;
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  float* sT = smem + S::S_T;
  float* sW = smem + S::S_W;
  float* sP = smem + S::S_P;
  float* sQ = smem + S::S_Q;
  float* sR = smem + S::S_R;
  uint64_t* barT = reinterpret_cast<uint64_t*>(smem + S::S_BAR);   // traces and tables
  uint64_t* barQ = barT + 1;                                       // DOFs
  const int tid = threadIdx.x;
  for (int i = tid; i < 3 * F * F; i += NT) sR[i] = ops.Rh[i];

  // column task (slot, mode): modes fastest; fused: the four simulations of a group fastest
  const bool act = tid < NE * B;
  const int es = act ? (FUSED ? tid / (4 * B) * 4 + tid % 4 : tid / B) : 0;
  const int b = act ? (FUSED ? tid % (4 * B) / 4 : tid % B) : 0;
  const int warp = tid >> 5, part = warp % S::NPP, lane6 = warp / S::NPP * 32 + (tid & 31);   // projection row
  const bool pact = warp < S::NPP * S::NWF && lane6 < S::NL;
  const int pr = lane6 / NE, pe = lane6 % NE;
  const Slots<FUSED> sl(st, ph);
  const int nbatch = (sl.n + NE - 1) / NE;
  const long long qs = FUSED ? st.qs : C::QS;
  constexpr int RS = FUSED ? B * FUSED_GROUP : B;
  constexpr int CS = FUSED ? FUSED_GROUP : 1;
  constexpr int GB = NQ * B * FUSED_GROUP;
  // first element of a batch, its simulation, and the elements the batch touches
  auto span = [&](int bt, int& e0, int& f0, int& ne) {
    if constexpr (!FUSED) {
      e0 = ph.begin + bt * NE;
      f0 = 0;
      ne = min(NE, ph.end - e0);
    } else {
      int e1, f1;
      sl.decode(bt * NE, e0, f0);
      sl.decode(min(sl.n, bt * NE + NE) - 1, e1, f1);
      ne = e1 - e0 + 1;
      e0 += ph.begin;
    }
  };
  // thread 0: the batch's DOFs (n x QS floats, or its groups of simulations)
  auto issue_q = [&](int bt) {
    int e0, f0, ne;
    span(bt, e0, f0, ne);
    const float* src = st.Q + (size_t)e0 * qs + (FUSED ? (size_t)(f0 / FUSED_GROUP) * GB : 0);
    const int n = min(NE, sl.n - bt * NE);
    tc::bulk_load(sQ, src, (uint32_t)(FUSED ? n / FUSED_GROUP * GB : n * C::QS) * 4, barQ);
  };
  // The face slots of a batch belong to the threads of the first warps (tid < 4 NE): link() reads,
  // two batches ahead, what names the neighbour's trace (one 8-byte load: with neighbour, code
  // and cluster apart, two dependent loads from memory held the first warp 3,100 of 11,000 cycles
  // a batch), fetch() issues the copies.
  auto link = [&](int bt) {
    const int t = bt * NE + tid / 4;
    if (tid >= 4 * NE || t >= sl.n) return make_int2(-1, 0);
    int e, f;
    sl.decode(t, e, f);
    return __ldg(st.nlink + 4 * ((size_t)ph.begin + e) + tid % 4);
  };
  // the first rup(4 NE, 32) threads (whole warps)
  auto fetch = [&](int bt, int buf, int2 l) {
    int* sI = reinterpret_cast<int*>(smem + S::S_I) + buf * 4 * NE;
    if (tid < 4 * NE) sI[tid] = l.x < 0 ? -1 : l.y & 3;
    const unsigned m = __ballot_sync(0xffffffffu, l.x >= 0);
    tc::fence_smem_to_async();
    int e0, f0, ne;
    span(bt, e0, f0, ne);
    if ((tid & 31) == 0) {
      uint32_t bytes = (uint32_t)__popc(m) * FS * 4;
      if (tid == 0) bytes += (uint32_t)ne * NDS * 4;
      tc::mbar_expect(barT, bytes);
      if (tid == 0 && !ph.suppress) tc::bulk_copy(smem + S::S_D + buf * NE * NDS, st.sndata + (size_t)e0 * NDS, (uint32_t)ne * NDS * 4, barT);
    }
    __syncwarp();
    if (l.x >= 0 && !ph.suppress) {
      const bool second = (l.y & 4) && ph.parity[l.y >> 8] == 1;
      const size_t face = FUSED ? ((size_t)(l.x >> 2) * st.nsim + (f0 + tid / 4) % sl.nsim) * 4 + (l.x & 3) : (size_t)l.x;
      tc::bulk_copy(sT + tid * FS, (second ? st.T2 : st.T1) + face * FS, FS * 4, barT);
    }
  };
  constexpr int NFT = rup(4 * NE, 32);   // fetching threads; one mbarrier arrival per warp
  if (tid == 0) {
    tc::mbar_init(barT, NFT / 32);
    tc::mbar_init(barQ, 1);
  }
  const int2 first = link(blockIdx.x);
  int2 ahead = link(blockIdx.x + gridDim.x);   // of the next batch
  __syncthreads();
  wait_for_previous_kernel();
  let_next_kernel_launch();
  if (!(ph.suppress & SUPPRESS_ALL) && blockIdx.x < nbatch) {
    if (tid < NFT) fetch(blockIdx.x, 0, first);
    if (tid == 0) issue_q(blockIdx.x);
  }
  __syncthreads();   // the orientations written by fetch
  uint32_t par = 0;
  for (int batch = blockIdx.x; batch < nbatch; batch += gridDim.x, par ^= 1) {
    const int t0 = batch * NE, next = batch + gridDim.x;
    const int* sI = reinterpret_cast<const int*>(smem + S::S_I) + par * 4 * NE;
    const float* sD = smem + S::S_D + par * NE * NDS;
    int e0, f0, ne;
    span(batch, e0, f0, ne);
    // element position in the batch of slot k
    auto pos_of = [&](int k) { return FUSED ? (f0 + k) / sl.nsim : k; };
    const int2 links = ahead;
    ahead = link(next + gridDim.x);
    // ---- the traces and tables have arrived (or the wait gave up). H = G R_h per face mode
    // (degree block), interface states with the neighbour coefficients; faces without a
    // neighbour contribute nothing
    bool ok = tc::mbar_wait(barT, par, ph.wait);
#pragma unroll 1
    for (int t = tid; t < NE * 4 * F; t += NT) {
      const int fs = t / F, fe = fs / 4, fi = fs % 4, f = t % F;
      float w6[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      const int h = (t0 + fe < sl.n) ? sI[fs] : -1;
      if (ok && h >= 0) {
        const int pf = face_degree(f), q0 = nface(pf);
        const float* gp = sT + fs * FS + q0;
        const float* R = sR + h * F * F + q0 * F + f;
        float hv[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < O; ++j)
          if (j <= pf) {
            const float w = R[j * F];
#pragma unroll
            for (int r = 0; r < 6; ++r) hv[r] = fmaf(gp[r * F + j], w, hv[r]);
          }
        interface_state(hv, sD + pos_of(fe) * NDS + 16 + 12 * fi, w6);
      }
      float* wp = sW + fe * S::ESW + fi * GS + f;
#pragma unroll
      for (int r = 0; r < 6; ++r) wp[r * GP] = w6[r];
    }
    // a wait that gave up: the phase is still open (its copies may land yet), so nothing more may
    // arrive on its mbarrier or be copied into its memory, and every thread leaves
    if (!__syncthreads_and(ok)) {
      if (tid == 0) {
        atomicOr(ph.err, 1);
        tc::mbar_wait(barT, par, ph.wait);         // the copies in flight, if any, land first
        tc::mbar_wait(barQ, par, ph.wait);
      }
      break;
    }
    // the batch's traces have been read: the next batch's copies go out now
    if (next < nbatch && tid < NFT) fetch(next, par ^ 1, links);
    // ---- projection of the faces' states through F^_f
    if (pact) sg_nproj<O, 6 * BP, GS>(part, sW + pe * S::ESW + pr * GP, sP + pe * S::ESP + pr * BP);
    // ---- the batch's DOFs have arrived (or the wait gave up: every thread leaves)
    ok = tc::mbar_wait(barQ, par, ph.wait);
    if (!__syncthreads_and(ok)) {
      if (tid == 0) {
        atomicOr(ph.err, 1);
        tc::mbar_wait(barQ, par, ph.wait);         // the copies in flight, if any, land first
        if (next < nbatch) tc::mbar_wait(barT, par ^ 1, ph.wait);
      }
      break;
    }
    if (act && t0 + es < sl.n) {
      const float* nd = sD + pos_of(es) * NDS;
      const Geo geo(nd);
      const float4 m0 = ld4(nd + 12);   // lam, mu, 1/rho
      const float* pp = sP + es * S::ESP + b;
      float G[3][3], dv[3];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = set_of_face(i);
        float P[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) P[r] = pp[(6 * i + r) * BP];
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
          for (int j = 0; j < 3; ++j) G[e][j] = i == 0 ? geo.J[c][e] * P[j] : fmaf(geo.J[c][e], P[j], G[e][j]);
#pragma unroll
        for (int j = 0; j < 3; ++j) dv[j] = i == 0 ? P[3 + j] : dv[j] + P[3 + j];
      }
      float out[9], eps[6];
      hooke(G, m0.x, m0.y, out, eps);
      const int g = e0 + pos_of(es), fsim = FUSED ? (f0 + es) % sl.nsim : 0;
      float* q = st.Q + (size_t)g * qs + Slots<FUSED>::sub(fsim, NQ, B) + (size_t)b * CS;
      const float* qr = sQ + (FUSED ? es / FUSED_GROUP * GB + b * CS + es % FUSED_GROUP : es * C::QS + b);
#pragma unroll
      for (int r = 0; r < 6; ++r) q[r * RS] = qr[r * RS] - out[r];
#pragma unroll
      for (int j = 0; j < 3; ++j) q[(6 + j) * RS] = fmaf(-m0.z, dv[j], qr[(6 + j) * RS]);
#pragma unroll
      for (int l = 0; l < M; ++l)
#pragma unroll
        for (int r = 0; r < 6; ++r) q[(9 + 6 * l + r) * RS] = fmaf(-ph.omega[l], eps[r], qr[(9 + 6 * l + r) * RS]);
    }
    __syncthreads();
    if (tid == 0 && next < nbatch) issue_q(next);
  }
}

}  // namespace ltsdev
