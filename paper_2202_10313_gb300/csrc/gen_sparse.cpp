// Build-time generator of the sparse operator products of k_predict_sp, k_neighbour_sp and
// k_adj_pred_sp (ahead-of-time
// specialisation, the GPU counterpart of the paper's generated sparse kernels, Sec. IV-A
// "all sparsity" and Sec. IV-B).
//
// The reference operators of one order are fixed numbers: the stiffness matrices K_c and
// the face matrices F~_i (Sec. III-A) in the orthonormal basis, computed here in FP64 by
// the library's own exact polynomial integration (host_basis.cpp) and rounded to FP32 as
// the device tables are. Their entries that vanish in exact arithmetic (the integration
// leaves them at <= 1e-10 of the largest; every true entry is >= 1e-3 of it) are left out,
// and every remaining entry becomes an immediate operand of a fused multiply-add. One GPU
// thread holds one row (one quantity of one element) of the operand in registers and
// forms all products of that row; the products are split into NPART parts of nearly equal
// multiply-add count, and a warp executes one part, so every thread of a warp runs the same
// straight-line code (no divergence) and no operator entry is read from memory. A part is a
// contiguous run of the outputs ordered by mode, so its outputs share most of their inputs
// and a thread loads only the inputs its part uses.
//
// Emitted, per order O, with one part per thread group (O = 3, 4, 5: 1, 2, 4) for the discrete
// adjoint's reverse predict pass (k_adj_pred_sp):
//   sp_time_o{O}(part, variant, x, y): Y_c[b] = sum_k x[k] K_c[b][k]        (time kernel,
//       d^{d+1}Q from d^dQ; K_c[b][k] != 0 only for deg b < deg k). Variant v takes only
//       the modes k < nbasis(O - v) and outputs b < nbasis(O - 1 - v) (the elastic time
//       kernel's degree truncation at derivative v; v = 0 is the full product).
//   sp_trace_o{O}(part, x, g): the face traces G_i[f] = sum_k x[k] F~_i[k][f].
//   sp_tproj_o{O}(part, x, y): y[b] = sum_i sum_f x[i F + f] F~_i[b][f] (the transposed face
//       traces of the four faces, summed).
//   sp_kvol_o{O}(part, variant, x, y): Z_c[b] = sum_k x[k] K_c[k][b] for 1 <= b < nbasis(O - v)
//       (the reverse time kernel at level v; K_c[k][b] != 0 only for deg k < deg b, so the
//       inputs are k < nbasis(O - 1 - v)).
// x[k * XP] is the thread's row, y[(c B + b) XP] and g[(i F + f) XP] the outputs (XP the pair
// stride of the staging arrays, a template parameter so that every address is an immediate
// offset). Every output the kernel reads is written (identically zero ones as 0); Z_c[0], which
// vanishes for every c, is not.
// The forward kernels' products come in row form (sg_*): a thread holds one row of a set,
// contiguous in memory, and reads and writes it four modes at a time. Set c (0, 1, 2: reference
// direction xi_c; 3: the direction of the fourth barycentric coordinate) has six rows: the
// velocities v_j and the direction's stress rows tau_c = sum_d dxi_c/dx_d sigma_d. One reference
// derivative is all a row of set c needs, so the products of a set use K_c alone:
//   sg_time_o{O}(variant, part, x, dx, y): y[c DY + b] = sum_k x[c dx + k] K_c[b][k], c < 3
//   sg_vol_o{O}(part, x, dx, y, g): y[c DY + b] = sum_k x[c dx + k] K_c[k][b] (c < 3) and the
//       trace of set c on its face f(c), g[f DG + m] = sum_k x[c dx + k] F~_f[k][m]
//   sg_proj_o{O}(part, g, y, p): F^_f of the face states g[f DG + m], added to y[c(f) DY + b]
//       for c < 3, written to p[b] for face 3
//   sg_nproj_o{O}(part, g, y): y[f DY + b] = F^_f of g[f DG + m] for the faces f (neighbour
//       kernel; six equal parts at order 5, else four)
// (x, y: the row of set 0; dx: the distance between a thread's rows of consecutive sets, 0 for
// the velocities, which all sets share; DY, DG template parameters). Outputs are split into parts
// by set (partition_sets).
//
// Usage: gen_sparse <out.cuh>      writes the header
//        gen_sparse --list <order> lists every product term, one line each:
//        "<kind> <part> <output> <input> <value>", kind t (time kernel, output c B + b, full
//        variant), v (volume, output c B + b), g (face trace, output i F + f), p (face
//        projection, output i B + b, input i F + f), n (neighbour face trace, output j F + f),
//        s (summed transposed traces, output b, input i F + f) or k (reverse time kernel,
//        output c B + b, full variant); for checks against other operators.
//        gen_sparse --list-rows <order> lists the terms of the row-form products likewise:
//        kind T (output c B + b, input c B + k), V (volume, the same), G (trace, output f F + m,
//        input k) or P (output f B + b, input f F + m).
//        gen_sparse --list-parts <order> lists what the other two leave out: every variant of the
//        row-form time products and the neighbour kernel's partition of the projections, a line
//        "O kind variant part output" for each output that a part writes, then its terms,
//        "kind variant part output input value" (kind T or N, output and input as for T and P).
// (The kinds v, p and n of --list have no function of their own: the forward kernels use the row form.)
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <stdexcept>
#include <string>
#include <vector>

#include "host.h"

namespace {

struct Out {
  char kind;                             // t, v, g, p, n
  int id;                                // output index within its kind
  std::string dst;                       // store expression
  std::vector<std::pair<int, float>> t;  // (input index, value), ascending input
};

using Parts = std::vector<std::vector<int>>;

// One output of a row-form product: set (or face) it belongs to, output row id, inputs.
struct RowOut {
  char kind;                             // T, V, G, P
  int set;                               // set of the input row (P: face)
  int idx, count;                        // output mode and the outputs of its row (stores in fours)
  std::vector<std::pair<int, float>> t;  // (input mode, value), ascending
};

// The face opposite barycentric coordinate c: xi_c = 0 for c < 3 (faces 2, 1, 0), face 3 for c = 3.
int face_of_set(int c) { return c < 3 ? 2 - c : 3; }

// One part per set (a part reads each row it needs whole, so a part of two sets reads twice as
// much shared memory), the outputs of set `cut` in two halves of nearly equal multiply-add count
// at a multiple of four outputs (cut < 0: none).
Parts partition_sets(const std::vector<RowOut>& outs, int cut) {
  Parts parts;
  for (size_t i = 0; i < outs.size();) {
    size_t e = i, total = 0, acc = 0;
    for (; e < outs.size() && outs[e].set == outs[i].set; ++e) total += outs[e].t.size();
    parts.emplace_back();
    bool split = outs[i].set != cut;
    for (size_t o = i; o < e; ++o) {
      size_t four = 0;
      for (size_t q = o; q < std::min(e, o + 4); ++q) four += outs[q].t.size();
      if (!split && outs[o].idx % 4 == 0 && acc + four / 2 > total / 2) {
        parts.emplace_back();
        split = true;
      }
      parts.back().push_back((int)o);
      acc += outs[o].t.size();
    }
    i = e;
  }
  return parts;
}

// Consecutive runs of the outputs with equal multiply-add shares.
Parts partition_runs(const std::vector<RowOut>& outs, int n) {
  double total = 0.0, acc = 0.0;
  for (const RowOut& u : outs) total += u.t.size();
  Parts parts(n);
  int p = 0;
  for (size_t o = 0; o < outs.size(); ++o) {
    const double w = (double)outs[o].t.size();
    while (p + 1 < n && acc + 0.5 * w > total * (p + 1) / n) ++p;
    parts[p].push_back((int)o);
    acc += w;
  }
  return parts;
}

// Parts of nearly equal multiply-add count (a store counts as one), each a contiguous run
// of the outputs in the given order.
Parts partition(const std::vector<Out>& outs, int nparts, const std::vector<int>& order) {
  size_t total = 0;
  for (int o : order) total += outs[o].t.size() + 1;
  Parts parts(nparts);
  size_t acc = 0;
  int p = 0;
  for (int o : order) {
    const size_t w = outs[o].t.size() + 1;
    // move on when this output would take the part further past its share than short of it
    if (p + 1 < nparts && acc + w / 2 > (size_t)(p + 1) * total / nparts) ++p;
    parts[p].push_back(o);
    acc += w;
  }
  return parts;
}

int nb(int o) { return o * (o + 1) * (o + 2) / 6; }

// All products of one order: time-kernel variants, volume + face traces, face projection.
struct Products {
  int O = 0, B = 0, F = 0, nparts = 1;
  std::vector<std::vector<Out>> time;    // per variant
  std::vector<Parts> time_parts;
  std::vector<Out> vol;                  // Z_c (b >= 1) then G_i
  Parts vol_parts;
  std::vector<Out> proj;
  Parts proj_parts;
  std::vector<std::vector<Out>> ntrace;  // per face j: the F outputs G_j[f]
  std::vector<Out> trace;                // G_i alone
  Parts trace_parts;
  std::vector<Out> tproj;                // sum over faces of the transposed traces
  Parts tproj_parts;
  std::vector<std::vector<Out>> kvol;    // reverse time kernel, per level
  std::vector<Parts> kvol_parts;
  size_t time_terms = 0, vol_terms = 0, face_terms = 0;
  // row-form products: outputs of set c (or face f), see RowOut
  std::vector<std::vector<RowOut>> rtime;   // per variant
  std::vector<Parts> rtime_parts;
  std::vector<RowOut> rvol, rproj;
  Parts rvol_parts, rproj_parts;

  template <typename NzK, typename NzF>
  void build_rows(const lts::RefOps& ops, const NzK& nzk, const NzF& nzf) {
    for (int v = 0; v <= O - 2; ++v) {
      const int kend = nb(O - v), bend = nb(O - 1 - v);
      std::vector<RowOut> outs;
      for (int c = 0; c < 3; ++c)
        for (int b = 0; b < bend; ++b) {
          RowOut u{'T', c, b, bend, {}};
          for (int k = 0; k < kend; ++k)
            if (nzk(ops.K[c][b * B + k])) u.t.push_back({k, (float)ops.K[c][b * B + k]});
          outs.push_back(u);
        }
      // order 5: K_2 (287 of 647 terms) in two parts, so that 12 warps share the work evenly
      rtime_parts.push_back(O == 3 ? partition_runs(outs, 1) : partition_sets(outs, O == 5 ? 2 : -1));
      rtime.push_back(outs);
    }
    for (int q = 0; q < 4; ++q) {
      const int c = (q + 3) % 4;   // set 3 has a trace only
      if (c < 3)
        for (int b = 0; b < B; ++b) {
          RowOut u{'V', c, b, B, {}};
          for (int k = 0; k < B; ++k)
            if (nzk(ops.K[c][k * B + b])) u.t.push_back({k, (float)ops.K[c][k * B + b]});
          rvol.push_back(u);
        }
      for (int m = 0; m < F; ++m) {
        RowOut u{'G', c, m, F, {}};
        const int f = face_of_set(c);
        for (int k = 0; k < B; ++k)
          if (nzf(ops.Ft[f][k * F + m])) u.t.push_back({k, (float)ops.Ft[f][k * F + m]});
        rvol.push_back(u);
      }
    }
    rvol_parts = O == 3 ? partition_runs(rvol, 1) : partition_sets(rvol, -1);
    for (int f = 0; f < 4; ++f)
      for (int b = 0; b < B; ++b) {
        RowOut u{'P', f, b, B, {}};
        for (int m = 0; m < F; ++m)
          if (nzf(ops.Ft[f][b * F + m])) u.t.push_back({m, (float)ops.Ft[f][b * F + m]});
        rproj.push_back(u);
      }
    // by face; orders 4 and 3 have warps for three parts and for one
    rproj_parts = O == 5 ? partition_sets(rproj, -1) : partition_runs(rproj, O == 4 ? 3 : 1);
  }

  void build(int order, int np) {
    O = order;
    nparts = np;
    lts::RefOps ops;
    ops.build(O);
    B = ops.B;
    F = ops.F;
    double kmax = 0.0, fmax = 0.0;
    for (int c = 0; c < 3; ++c)
      for (double v : ops.K[c]) kmax = std::max(kmax, std::fabs(v));
    for (int i = 0; i < 4; ++i)
      for (double v : ops.Ft[i]) fmax = std::max(fmax, std::fabs(v));
    auto nzk = [&](double v) { return std::fabs(v) > 1e-7 * kmax; };
    auto nzf = [&](double v) { return std::fabs(v) > 1e-7 * fmax; };
    auto dst = [](const char* arr, int idx) {
      char d[64];
      std::snprintf(d, sizeof d, "%s[%d * XP]", arr, idx);
      return std::string(d);
    };
    // time kernel variants; outputs (c, b) ordered by mode b, then c
    for (int v = 0; v <= O - 2; ++v) {
      const int kend = nb(O - v), bend = nb(O - 1 - v);
      std::vector<Out> outs;
      std::vector<int> ord;
      for (int b = 0; b < bend; ++b)
        for (int c = 0; c < 3; ++c) {
          Out u{'t', c * B + b, dst("y", c * B + b), {}};
          for (int k = 0; k < kend; ++k)
            if (nzk(ops.K[c][b * B + k])) u.t.push_back({k, (float)ops.K[c][b * B + k]});
          if (v == 0) time_terms += u.t.size();
          ord.push_back((int)outs.size());
          outs.push_back(u);
        }
      time_parts.push_back(partition(outs, nparts, ord));
      time.push_back(outs);
    }
    // volume (by mode b, then c) and face traces (by face mode f, then face i)
    std::vector<int> ord;
    for (int b = 0; b < B; ++b)
      for (int c = 0; c < 3; ++c) {
        Out u{'v', c * B + b, dst("y", c * B + b), {}};
        for (int k = 0; k < B; ++k)
          if (nzk(ops.K[c][k * B + b])) u.t.push_back({k, (float)ops.K[c][k * B + b]});
        vol_terms += u.t.size();
        if (b == 0) {   // the constant mode has no derivative: Z_c[0] = 0, not read
          if (!u.t.empty()) throw std::runtime_error("K_c[k][0] must vanish");
          continue;
        }
        ord.push_back((int)vol.size());
        vol.push_back(u);
      }
    for (int m = 0; m < F; ++m)
      for (int i = 0; i < 4; ++i) {
        Out u{'g', i * F + m, dst("g", i * F + m), {}};
        for (int k = 0; k < B; ++k)
          if (nzf(ops.Ft[i][k * F + m])) u.t.push_back({k, (float)ops.Ft[i][k * F + m]});
        face_terms += u.t.size();
        ord.push_back((int)vol.size());
        vol.push_back(u);
      }
    vol_parts = partition(vol, nparts, ord);
    // face projection, outputs (i, b) by face, then mode: F^_i[f][b] = F~_i[b][f]
    ord.clear();
    for (int i = 0; i < 4; ++i)
      for (int b = 0; b < B; ++b) {
        Out u{'p', i * B + b, dst("y", i * B + b), {}};
        for (int m = 0; m < F; ++m)
          if (nzf(ops.Ft[i][b * F + m])) u.t.push_back({i * F + m, (float)ops.Ft[i][b * F + m]});
        ord.push_back((int)proj.size());
        proj.push_back(u);
      }
    proj_parts = partition(proj, nparts, ord);
    // face traces of a neighbour's buffer on its face j (one face per thread, chosen at run
    // time): G_j[f] = sum_k x[k] F~_j[k][f]
    for (int j = 0; j < 4; ++j) {
      std::vector<Out> outs;
      for (int m = 0; m < F; ++m) {
        Out u{'n', j * F + m, dst("y", m), {}};
        for (int k = 0; k < B; ++k)
          if (nzf(ops.Ft[j][k * F + m])) u.t.push_back({k, (float)ops.Ft[j][k * F + m]});
        outs.push_back(u);
      }
      ntrace.push_back(outs);
    }
    build_rows(ops, nzk, nzf);
    // adjoint products: the face traces alone (as in vol, by face mode then face)
    ord.clear();
    for (const Out& u : vol)
      if (u.kind == 'g') {
        ord.push_back((int)trace.size());
        trace.push_back(u);
      }
    trace_parts = partition(trace, nparts, ord);
    // y[b] = sum_{i, f} x[i F + f] F~_i[b][f], by mode
    ord.clear();
    for (int b = 0; b < B; ++b) {
      Out u{'s', b, dst("y", b), {}};
      for (int i = 0; i < 4; ++i)
        for (int m = 0; m < F; ++m)
          if (nzf(ops.Ft[i][b * F + m])) u.t.push_back({i * F + m, (float)ops.Ft[i][b * F + m]});
      ord.push_back((int)tproj.size());
      tproj.push_back(u);
    }
    tproj_parts = partition(tproj, nparts, ord);
    // Z_c[b] = sum_k x[k] K_c[k][b], 1 <= b < nbasis(O - v), by mode then c
    for (int v = 0; v <= O - 2; ++v) {
      std::vector<Out> outs;
      std::vector<int> o2;
      for (int b = 1; b < nb(O - v); ++b)
        for (int c = 0; c < 3; ++c) {
          Out u{'k', c * B + b, dst("y", c * B + b), {}};
          for (int k = 0; k < B; ++k)
            if (nzk(ops.K[c][k * B + b])) {
              if (k >= nb(O - 1 - v)) throw std::runtime_error("K_c[k][b] must vanish for deg k >= deg b");
              u.t.push_back({k, (float)ops.K[c][k * B + b]});
            }
          o2.push_back((int)outs.size());
          outs.push_back(u);
        }
      kvol_parts.push_back(partition(outs, nparts, o2));
      kvol.push_back(outs);
    }
  }
};

std::string flt(float v) {
  char b[64];
  std::snprintf(b, sizeof b, "%a", (double)v);
  return std::string(b) + "f";
}

// Straight-line body of one part: loads of the needed inputs, then one fma chain per
// output (terms in ascending input index, the order of the dense kernels), then its store.
void emit_part(FILE* f, const std::vector<Out>& outs, const std::vector<int>& part) {
  std::vector<int> need;
  for (int o : part)
    for (auto& t : outs[o].t) need.push_back(t.first);
  std::sort(need.begin(), need.end());
  need.erase(std::unique(need.begin(), need.end()), need.end());
  for (int k : need) std::fprintf(f, "    const float x%d = x[%d * XP];\n", k, k);
  for (int o : part) {
    const Out& u = outs[o];
    if (u.t.empty()) {   // identically zero output that the kernel reads
      std::fprintf(f, "    %s = 0.f;\n", u.dst.c_str());
      continue;
    }
    std::fprintf(f, "    {\n      float a = x%d * %s;\n", u.t[0].first, flt(u.t[0].second).c_str());
    for (size_t i = 1; i < u.t.size(); ++i)
      std::fprintf(f, "      a = fmaf(x%d, %s, a);\n", u.t[i].first, flt(u.t[i].second).c_str());
    std::fprintf(f, "      %s = a;\n    }\n", u.dst.c_str());
  }
}

void emit_dispatch(FILE* f, const char* name, const char* args, const char* call_args,
                   const std::vector<Parts>& parts_of_variant, const std::vector<std::vector<Out>>& outs_of_variant,
                   bool has_variant) {
  const int nv = (int)parts_of_variant.size();
  for (int v = 0; v < nv; ++v) {
    const auto& parts = parts_of_variant[v];
    for (size_t p = 0; p < parts.size(); ++p) {
      std::fprintf(f, "template <int XP>\n__device__ __forceinline__ void %s_v%d_p%zu(%s) {\n", name, v, p, args);
      emit_part(f, outs_of_variant[v], parts[p]);
      std::fprintf(f, "}\n");
    }
  }
  std::fprintf(f, "template <int XP>\n__device__ __forceinline__ void %s(int part%s, %s) {\n", name,
               has_variant ? ", int variant" : "", args);
  for (int v = 0; v < nv; ++v) {
    if (has_variant) std::fprintf(f, "  if (variant == %d) {\n", v);
    std::fprintf(f, "  switch (part) {\n");
    for (size_t p = 0; p < parts_of_variant[v].size(); ++p)
      std::fprintf(f, "    case %zu: %s_v%d_p%zu<XP>(%s); break;\n", p, name, v, p, call_args);
    std::fprintf(f, "    default: break;\n  }\n");
    if (has_variant) std::fprintf(f, "  return;\n  }\n");
  }
  std::fprintf(f, "}\n");
}

// Straight-line body of one part of a row-form product: per set, the input row four modes at a
// time, one fma chain per output, stores of four outputs where the part holds all four (padding
// modes are stored as zeros).
// apart: projections are written per face instead of added to their direction's row.
void emit_row_part(FILE* f, const std::vector<RowOut>& outs, const std::vector<int>& part, bool apart) {
  size_t i = 0;
  while (i < part.size()) {
    const int set = outs[part[i]].set;
    size_t e = i;
    std::vector<int> need;
    while (e < part.size() && outs[part[e]].set == set) {
      for (auto& t : outs[part[e]].t) need.push_back(t.first / 4);
      ++e;
    }
    std::sort(need.begin(), need.end());
    need.erase(std::unique(need.begin(), need.end()), need.end());
    const bool proj = outs[part[i]].kind == 'P';
    std::fprintf(f, "    {\n");
    if (proj)
      std::fprintf(f, "      const float* xs = g + %d * DG;\n", set);
    else
      std::fprintf(f, "      const float* xs = x + %d * dx;\n", set);
    for (int g : need)
      std::fprintf(f, "      const float4 q%d = *reinterpret_cast<const float4*>(xs + %d);\n", g, 4 * g);
    while (i < e) {
      // the outputs of this group of four that the part holds
      const RowOut& u0 = outs[part[i]];
      const int grp = u0.idx / 4;
      size_t j = i;
      while (j < e && outs[part[j]].kind == u0.kind && outs[part[j]].idx / 4 == grp) ++j;
      const int have = (int)(j - i), want = std::min(4, u0.count - 4 * grp);
      char dst[64];
      if (u0.kind == 'G')
        std::snprintf(dst, sizeof dst, "g + %d * DG", face_of_set(set));
      else if (proj && apart)
        std::snprintf(dst, sizeof dst, "y + %d * DY", set);
      else if (proj && set == 3)
        std::snprintf(dst, sizeof dst, "p");
      else
        std::snprintf(dst, sizeof dst, "y + %d * DY", proj ? 2 - set : set);
      const bool add = proj && set < 3 && !apart;
      std::fprintf(f, "      {\n        float* d = %s + %d;\n", dst, 4 * grp);
      const bool whole = have == want;
      static const char* comp = "xyzw";
      if (whole && add) std::fprintf(f, "        const float4 s = *reinterpret_cast<const float4*>(d);\n");
      for (size_t o = i; o < j; ++o) {
        const RowOut& u = outs[part[o]];
        const int l = u.idx % 4;
        if (add && whole)
          std::fprintf(f, "        float a%d = s.%c;\n", l, comp[l]);
        else if (add)
          std::fprintf(f, "        float a%d = d[%d];\n", l, l);
        else if (u.t.empty())
          std::fprintf(f, "        float a%d = 0.f;\n", l);
        for (size_t k = 0; k < u.t.size(); ++k) {
          const int g = u.t[k].first / 4;
          const char cc = comp[u.t[k].first % 4];
          if (k == 0 && !add)
            std::fprintf(f, "        float a%d = q%d.%c * %s;\n", l, g, cc, flt(u.t[k].second).c_str());
          else
            std::fprintf(f, "        a%d = fmaf(q%d.%c, %s, a%d);\n", l, g, cc, flt(u.t[k].second).c_str(), l);
        }
      }
      if (whole) {
        std::fprintf(f, "        *reinterpret_cast<float4*>(d) = make_float4(");
        for (int l = 0; l < 4; ++l) std::fprintf(f, l < want ? "%sa%d" : "%s0.f", l ? ", " : "", l);
        std::fprintf(f, ");\n");
      } else {
        for (size_t o = i; o < j; ++o) std::fprintf(f, "        d[%d] = a%d;\n", outs[part[o]].idx % 4, outs[part[o]].idx % 4);
      }
      std::fprintf(f, "      }\n");
      i = j;
    }
    std::fprintf(f, "    }\n");
  }
}

void emit_row_dispatch(FILE* f, const char* name, const char* tmpl, const char* targs, const char* args,
                       const char* call, const std::vector<Parts>& parts, const std::vector<std::vector<RowOut>>& outs,
                       bool apart = false) {
  for (size_t v = 0; v < parts.size(); ++v)
    for (size_t p = 0; p < parts[v].size(); ++p) {
      std::fprintf(f, "template <%s>\n__device__ __forceinline__ void %s_v%zu_p%zu(%s) {\n", tmpl, name, v, p, args);
      emit_row_part(f, outs[v], parts[v][p], apart);
      std::fprintf(f, "}\n");
    }
  std::fprintf(f, "template <%s>\n__device__ __forceinline__ void %s(int variant, int part, %s) {\n", tmpl, name, args);
  for (size_t v = 0; v < parts.size(); ++v) {
    if (parts.size() > 1) std::fprintf(f, "  if (variant == %zu) {\n", v);
    std::fprintf(f, "  switch (part) {\n");
    for (size_t p = 0; p < parts[v].size(); ++p)
      std::fprintf(f, "    case %zu: %s_v%zu_p%zu<%s>(%s); break;\n", p, name, v, p, targs, call);
    std::fprintf(f, "    default: break;\n  }\n");
    if (parts.size() > 1) std::fprintf(f, "  return;\n  }\n");
  }
  std::fprintf(f, "}\n");
}

// The neighbour kernel's parts of the projections: one per warp, of equal multiply-add count.
Parts nproj_parts(const Products& P) { return partition_runs(P.rproj, P.O == 5 ? 6 : 4); }

void emit_rows(FILE* f, int O, const Products& P) {
  char nm[64];
  std::snprintf(nm, sizeof nm, "sg_time_o%d", O);
  emit_row_dispatch(f, nm, "int DY", "DY", "const float* __restrict__ x, int dx, float* __restrict__ y", "x, dx, y",
                    P.rtime_parts, P.rtime);
  std::snprintf(nm, sizeof nm, "sg_vol_o%d", O);
  emit_row_dispatch(f, nm, "int DY, int DG", "DY, DG",
                    "const float* __restrict__ x, int dx, float* __restrict__ y, float* __restrict__ g", "x, dx, y, g",
                    {P.rvol_parts}, {P.rvol});
  std::snprintf(nm, sizeof nm, "sg_proj_o%d", O);
  emit_row_dispatch(f, nm, "int DY, int DG", "DY, DG",
                    "const float* __restrict__ g, float* __restrict__ y, float* __restrict__ p", "g, y, p",
                    {P.rproj_parts}, {P.rproj});
  std::snprintf(nm, sizeof nm, "sg_nproj_o%d", O);
  emit_row_dispatch(f, nm, "int DY, int DG", "DY, DG", "const float* __restrict__ g, float* __restrict__ y", "g, y",
                    {nproj_parts(P)}, {P.rproj}, true);
}

void emit_order(FILE* f, int O, int nparts) {
  Products P;
  P.build(O, nparts);
  std::fprintf(f, "// ---- order %d (B = %d, F = %d), %d parts\n", O, P.B, P.F, nparts);
  std::fprintf(f, "// multiply-adds per row: time kernel %zu (full variant), volume %zu, face traces %zu\n",
               P.time_terms, P.vol_terms, P.face_terms);
  char nm[64];
  std::snprintf(nm, sizeof nm, "sp_time_o%d", O);
  emit_dispatch(f, nm, "const float* __restrict__ x, float* __restrict__ y", "x, y", P.time_parts, P.time, true);
  std::snprintf(nm, sizeof nm, "sp_trace_o%d", O);
  emit_dispatch(f, nm, "const float* __restrict__ x, float* __restrict__ g", "x, g", {P.trace_parts}, {P.trace},
                false);
  std::snprintf(nm, sizeof nm, "sp_tproj_o%d", O);
  emit_dispatch(f, nm, "const float* __restrict__ x, float* __restrict__ y", "x, y", {P.tproj_parts}, {P.tproj},
                false);
  std::snprintf(nm, sizeof nm, "sp_kvol_o%d", O);
  emit_dispatch(f, nm, "const float* __restrict__ x, float* __restrict__ y", "x, y", P.kvol_parts, P.kvol, true);
  emit_rows(f, O, P);
}

int parts_of(int O) { return O == 5 ? 4 : (O == 4 ? 2 : 1); }

int list_terms(int O) {
  Products P;
  P.build(O, parts_of(O));
  auto list = [](const std::vector<Out>& outs, const Parts& parts) {
    for (size_t p = 0; p < parts.size(); ++p)
      for (int o : parts[p])
        for (auto& x : outs[o].t)
          std::printf("%c %zu %d %d %.9e\n", outs[o].kind, p, outs[o].id, x.first, (double)x.second);
  };
  list(P.time[0], P.time_parts[0]);
  list(P.vol, P.vol_parts);
  list(P.proj, P.proj_parts);
  for (auto& outs : P.ntrace) {
    std::vector<int> all(outs.size());
    for (size_t i = 0; i < all.size(); ++i) all[i] = (int)i;
    list(outs, Parts{all});
  }
  list(P.tproj, P.tproj_parts);
  list(P.kvol[0], P.kvol_parts[0]);
  return 0;
}

int list_rows(int O) {
  Products P;
  P.build(O, parts_of(O));
  auto list = [&](const std::vector<RowOut>& outs, const Parts& parts) {
    for (size_t p = 0; p < parts.size(); ++p)
      for (int o : parts[p]) {
        const RowOut& u = outs[o];
        const int in = u.kind == 'P' ? P.F : (u.kind == 'G' ? 0 : P.B);   // input stride between sets
        const int out = u.kind == 'G' ? P.F : P.B;
        const int os = u.kind == 'G' ? face_of_set(u.set) : u.set;
        for (auto& x : u.t)
          std::printf("%c %zu %d %d %.9e\n", u.kind, p, os * out + u.idx, u.set * in + x.first, (double)x.second);
      }
  };
  list(P.rtime[0], P.rtime_parts[0]);
  list(P.rvol, P.rvol_parts);
  list(P.rproj, P.rproj_parts);
  return 0;
}

int list_parts(int O) {
  Products P;
  P.build(O, parts_of(O));
  auto list = [&](char kind, size_t variant, const std::vector<RowOut>& outs, const Parts& parts, int in) {
    for (size_t p = 0; p < parts.size(); ++p)
      for (int o : parts[p]) {
        const RowOut& u = outs[o];
        std::printf("O %c %zu %zu %d\n", kind, variant, p, u.set * P.B + u.idx);
        for (auto& x : u.t)
          std::printf("%c %zu %zu %d %d %.9e\n", kind, variant, p, u.set * P.B + u.idx, u.set * in + x.first,
                      (double)x.second);
      }
  };
  for (size_t v = 0; v < P.rtime.size(); ++v) list('T', v, P.rtime[v], P.rtime_parts[v], P.B);
  list('N', 0, P.rproj, nproj_parts(P), P.F);
  return 0;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc == 3 && std::strcmp(argv[1], "--list") == 0) {
    const int O = std::atoi(argv[2]);
    if (O < 3 || O > 5) return 2;
    return list_terms(O);
  }
  if (argc == 3 && std::strcmp(argv[1], "--list-rows") == 0) {
    const int O = std::atoi(argv[2]);
    if (O < 3 || O > 5) return 2;
    return list_rows(O);
  }
  if (argc == 3 && std::strcmp(argv[1], "--list-parts") == 0) {
    const int O = std::atoi(argv[2]);
    if (O < 3 || O > 5) return 2;
    return list_parts(O);
  }
  if (argc != 2) {
    std::fprintf(stderr, "usage: gen_sparse <out.cuh> | gen_sparse --list|--list-rows|--list-parts <order>\n");
    return 2;
  }
  FILE* f = std::fopen(argv[1], "w");
  if (!f) {
    std::perror(argv[1]);
    return 1;
  }
  std::fprintf(f, "// Generated at build time by gen_sparse.cpp from the reference operators: do not edit.\n");
  std::fprintf(f, "#pragma once\nnamespace ltssp {\n");
  for (int O = 3; O <= 5; ++O) emit_order(f, O, parts_of(O));
  std::fprintf(f, "}  // namespace ltssp\n");
  return std::fclose(f) == 0 ? 0 : 1;
}
