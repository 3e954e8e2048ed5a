// Column-partitioned sweep schedules (kernel k_sweep_cols): the flattened
// program of Alg. 3 / Alg. 4 as resident runs and global phases, every
// butterfly op written out as a dense block over its inputs, every
// sweep-leaf phase as its triangle; plus a host executor of the schedule and
// its structural check (verification without a GPU).
#include <algorithm>
#include <cstring>

#include "hb_internal.h"

namespace hb {

namespace {

inline int64_t al16(int64_t b) { return (b + 15) & ~(int64_t)15; }
inline int32_t even(int64_t v) { return (int32_t)((v + 1) & ~(int64_t)1); }

// One op of a phase as a dense block: rows (output slot, nin coefficients) over
// nin inputs.  in[]: the inputs' global slots (vector row r -> r, state entry e ->
// n + e).  Resident: in0 is the window slot of the first one; global: its position
// in the batch's slice.
struct DenseOp {
  std::vector<int32_t> in, out;
  std::vector<cplx> coef;   // [row][nin]
  int32_t in0 = 0;
  bool add = false;         // rows add to their outputs' old values
  int32_t nin() const { return (int32_t)in.size(); }
  int32_t rows() const { return (int32_t)out.size(); }
};

// inputs of a flattened op: calls fn(is_state, index) in order (first segment, then the second)
template <class Fn>
void op_inputs(const FlatOp& f, Fn fn) {
  if (f.kind == FK_LEAF) return;
  const bool vec = (f.flags & FF_SRC_VEC) != 0;
  for (int i = 0; i < f.n_s0; ++i) fn(!vec, f.src0 + i);
  for (int i = 0; i < f.n_s1; ++i) fn(true, f.src1 + i);
}
int op_nin(const FlatOp& f) { return f.kind == FK_LEAF ? 0 : f.n_s0 + f.n_s1; }

// The dense block of one flattened op (semantics of the op kinds as defined with
// FlatOp: the ID's identity entries, T or S entries, conjugated for the adjoint
// layouts, negated when the op subtracts from its outputs).
void expand_op(const PackedHost& ph, const FlatOp& f, DenseOp& B) {
  const cplx* M = ph.fpool.data() + f.moff;
  const int16_t* I = f.ioff >= 0 ? ph.ipool.data() + f.ioff : nullptr;
  const bool conj_layout = (f.flags & FF_CONJ) != 0;
  const bool two = (f.flags & FF_TWO) != 0;
  const int32_t n = (int32_t)ph.n;
  op_inputs(f, [&](bool st, int32_t e) { B.in.push_back(st ? n + e : e); });
  const int32_t nin = B.nin();
  auto out0 = [&](int i) -> int32_t { return (f.flags & FF_OUT_VEC) ? f.out0 + i : n + f.out0 + i; };
  auto row = [&](int32_t o) -> cplx* {
    B.out.push_back(o);
    B.coef.resize(B.coef.size() + (size_t)nin, cplx(0.0, 0.0));
    return B.coef.data() + B.coef.size() - (size_t)nin;
  };
  if (f.kind == FK_GATHER) {
    // out_b[i] = cand[q_i] + sum_j T(i, j) cand[p_j]
    for (int b = 0; b < (two ? 2 : 1); ++b) {
      const cplx* Mb = M + (b ? f.m1 : 0);
      const int16_t* Ib = I + (b ? f.i1 : 0);
      const int k = b ? f.k1 : f.k0, c = b ? f.c1 : f.c0, nr = c - k;
      for (int i = 0; i < k; ++i) {
        cplx* w = row(b ? n + f.out1 + i : out0(i));
        w[Ib[i]] += cplx(1.0, 0.0);
        for (int j = 0; j < nr; ++j) w[Ib[k + j]] += conj_layout ? std::conj(Mb[(int64_t)i * nr + j]) : Mb[(int64_t)j * k + i];
      }
    }
  } else if (f.kind == FK_SCATTER) {
    // candidate entry r: y[map(r)] (skeleton) or sum_i T(i, j) y[i]; both blocks add
    const double sg = (f.flags & FF_SUB) ? -1.0 : 1.0;
    B.add = (f.flags & FF_SUB) != 0;
    for (int r = 0; r < f.c0; ++r) {
      cplx* w = row((!two || r < f.split) ? out0(r) : n + f.out1 + (r - f.split));
      for (int b = 0; b < (two ? 2 : 1); ++b) {
        const cplx* Mb = M + (b ? f.m1 : 0);
        const int16_t* Ib = I + (b ? f.i1 : 0);
        const int k = b ? f.k1 : f.k0, c = b ? f.c1 : f.c0, nr = c - k;
        cplx* y = w + (b ? f.n_s0 : 0);   // y_b = inputs [ybase, ybase + k)
        const int code = Ib[c + r];
        if (code >= 0) {
          y[code] += cplx(sg, 0.0);
        } else {
          const int j = -1 - code;
          for (int i = 0; i < k; ++i) y[i] += sg * (conj_layout ? std::conj(Mb[(int64_t)j * k + i]) : Mb[(int64_t)i * nr + j]);
        }
      }
    }
  } else if (f.kind == FK_MIDDLE) {
    // y = S z (S stored [c][r]); adjoint z = S^H y
    const int kr = f.k0, kc = f.c0;
    const bool adj = (f.flags & FF_ADJ) != 0;
    const int ni = adj ? kr : kc, nout = adj ? kc : kr;
    for (int oo = 0; oo < nout; ++oo) {
      cplx* w = row(n + f.out0 + oo);
      for (int i = 0; i < ni; ++i) w[i] += adj ? std::conj(M[(int64_t)oo * kr + i]) : M[(int64_t)i * kr + oo];
    }
  }
}

// rows of a flattened op
int op_rows(const FlatOp& f) {
  const bool two = (f.flags & FF_TWO) != 0;
  if (f.kind == FK_GATHER) return f.k0 + (two ? f.k1 : 0);
  if (f.kind == FK_SCATTER) return f.c0;
  return f.kind == FK_MIDDLE ? ((f.flags & FF_ADJ) ? f.c0 : f.k0) : 0;
}
// state entries written by a flattened op
template <class Fn>
void op_state_writes(const FlatOp& f, Fn fn) {
  const bool two = (f.flags & FF_TWO) != 0;
  int n0 = 0, n1 = 0;
  if (f.kind == FK_GATHER) { n0 = f.k0; n1 = two ? f.k1 : 0; }
  else if (f.kind == FK_SCATTER) { n0 = two ? f.split : f.c0; n1 = two ? f.c0 - f.split : 0; }
  else if (f.kind == FK_MIDDLE) n0 = (f.flags & FF_ADJ) ? f.c0 : f.k0;
  if (!(f.flags & FF_OUT_VEC)) for (int i = 0; i < n0; ++i) fn(f.out0 + i);
  for (int i = 0; i < n1; ++i) fn(f.out1 + i);
}

// Consecutive stages of a butterfly multiplied out.  r stages connect blocks of 2^r
// input segments with 2^r output segments, fully: the components of the stages' graph.
// A component becomes one dense op, so that r dependent phases become one; two stages
// cost no more entries than one after the other (4 k inputs per output against 2 k
// twice), more stages trade entries for phases.
struct Fuser {
  const PackedHost& ph;
  const FlatProgram& fp;
  std::vector<int32_t> prod;     // per state entry: op that last wrote it (in planning or fusing order)
  Fuser(const PackedHost& p, const FlatProgram& f) : ph(p), fp(f), prod((size_t)p.state_len, -1) {}

  static int32_t find(std::vector<int32_t>& u, int32_t x) {
    while (u[(size_t)x] != x) x = u[(size_t)x] = u[(size_t)u[(size_t)x]];
    return x;
  }
  // components of phases [p0, p1): comp[op - base[p0]] = component (0 ..), their number returned
  int32_t components(int p0, int p1, std::vector<int32_t>& comp) {
    const int32_t ob = fp.base[p0], oe = fp.base[p1];
    std::vector<int32_t> u((size_t)(oe - ob));
    for (int32_t i = 0; i < oe - ob; ++i) u[(size_t)i] = i;
    for (int p = p0; p < p1; ++p) {
      if (p > p0)
        for (int32_t o = fp.base[p]; o < fp.base[p + 1]; ++o) {
          const FlatOp& f = fp.ops[o];
          if (f.n_s0 > 0) u[(size_t)find(u, prod[(size_t)f.src0] - ob)] = find(u, o - ob);
          if (f.n_s1 > 0) u[(size_t)find(u, prod[(size_t)f.src1] - ob)] = find(u, o - ob);
        }
      for (int32_t o = fp.base[p]; o < fp.base[p + 1]; ++o) op_state_writes(fp.ops[o], [&](int32_t e) { prod[(size_t)e] = o; });
    }
    comp.assign((size_t)(oe - ob), -1);
    int32_t nc = 0;
    for (int32_t i = 0; i < oe - ob; ++i) {
      const int32_t r = find(u, i);
      if (comp[(size_t)r] < 0) comp[(size_t)r] = nc++;
      comp[(size_t)i] = comp[(size_t)r];
    }
    return nc;
  }
  // entries of the fused phases [p0, p1); -1: a component exceeds a global batch (glob)
  int64_t entries(int p0, int p1, bool glob) {
    std::vector<int32_t> comp;
    const int32_t nc = components(p0, p1, comp), ob = fp.base[p0];
    std::vector<int64_t> nin((size_t)nc, 0), rows((size_t)nc, 0);
    bool add = false;
    for (int32_t o = fp.base[p0]; o < fp.base[p0 + 1]; ++o) nin[(size_t)comp[(size_t)(o - ob)]] += op_nin(fp.ops[o]);
    for (int32_t o = fp.base[p1 - 1]; o < fp.base[p1]; ++o) {
      rows[(size_t)comp[(size_t)(o - ob)]] += op_rows(fp.ops[o]);
      add = add || (fp.ops[o].flags & FF_SUB);
    }
    int64_t e = 0;
    for (int32_t c = 0; c < nc; ++c) {
      if (glob && nin[(size_t)c] + (add ? 64 : 0) > kSwGather) return -1;
      e += even(nin[(size_t)c]) * rows[(size_t)c];
    }
    return e;
  }
  // cut the stages [p0, p1) of one butterfly (the entry phase not among them) into fused
  // phases: the cut with the least cost, a fixed one per phase plus the entries'
  std::vector<int> plan(int p0, int p1, bool glob) {
    const int m = p1 - p0;
    // a phase costs about as much as this many entries: its dependent steps (resident), the
    // gather's round trip and a barrier of all warps (global)
    const double phase = glob ? 24000.0 : 7000.0;
    const int most = glob ? 4 : m;
    std::vector<double> best((size_t)m + 1, 1e300);
    std::vector<int> from((size_t)m + 1, 0);
    best[0] = 0;
    for (int i = 0; i < m; ++i)
      for (int j = i + 1; j <= m && j - i <= most; ++j) {
        const int64_t e = entries(p0 + i, p0 + j, glob);
        if (e < 0 && j > i + 1) break;
        if (j > i + 1 && (double)e > 40.0 * phase) break;
        const double c = best[(size_t)i] + phase + (double)std::max<int64_t>(e, 0);
        if (c < best[(size_t)j]) { best[(size_t)j] = c; from[(size_t)j] = i; }
      }
    std::vector<int> cuts;
    for (int j = m; j > 0; j = from[(size_t)j]) cuts.push_back(p0 + j);
    std::reverse(cuts.begin(), cuts.end());
    return cuts;   // ends of the fused phases
  }
  // the fused phases [p0, p1) as dense ops
  void fuse(int p0, int p1, std::vector<DenseOp>& ops) {
    ops.clear();
    if (p1 == p0 + 1) {
      for (int32_t o = fp.base[p0]; o < fp.base[p1]; ++o) {
        ops.emplace_back();
        expand_op(ph, fp.ops[o], ops.back());
      }
      return;
    }
    std::vector<int32_t> comp;
    const int32_t nc = components(p0, p1, comp), ob = fp.base[p0];
    ops.resize((size_t)nc);
    // row of coefficients (over the component's inputs) of every state entry written so far
    std::vector<std::pair<int32_t, std::vector<cplx>>> val;   // (entry, row), found through at[]
    if (at.size() != (size_t)ph.state_len) at.assign((size_t)ph.state_len, -1);
    for (int32_t o = fp.base[p0]; o < fp.base[p0 + 1]; ++o) {
      const FlatOp& f = fp.ops[o];
      op_inputs(f, [&](bool st, int32_t e) { ops[(size_t)comp[(size_t)(o - ob)]].in.push_back(st ? (int32_t)ph.n + e : e); });
    }
    std::vector<int32_t> col((size_t)nc, 0);   // first phase: the op's inputs' place in its component
    for (int p = p0; p < p1; ++p)
      for (int32_t o = fp.base[p]; o < fp.base[p + 1]; ++o) {
        const int32_t c = comp[(size_t)(o - ob)];
        DenseOp& C = ops[(size_t)c];
        DenseOp B;
        expand_op(ph, fp.ops[o], B);
        const int32_t nin = C.nin();
        for (int32_t r = 0; r < B.rows(); ++r) {
          std::vector<cplx> w((size_t)nin, cplx(0.0, 0.0));
          for (int32_t i = 0; i < B.nin(); ++i) {
            const cplx b = B.coef[(size_t)r * B.nin() + i];
            if (b == cplx(0.0, 0.0)) continue;
            if (p == p0) {
              w[(size_t)(col[(size_t)c] + i)] += b;
            } else {
              const std::vector<cplx>& v = val[(size_t)at[(size_t)(B.in[(size_t)i] - ph.n)]].second;
              for (int32_t q = 0; q < nin; ++q) w[(size_t)q] += b * v[(size_t)q];
            }
          }
          if (p + 1 < p1) {
            const int32_t e = B.out[(size_t)r] - (int32_t)ph.n;
            at[(size_t)e] = (int32_t)val.size();
            val.emplace_back(e, std::move(w));
          } else {
            C.add = B.add;
            C.out.push_back(B.out[(size_t)r]);
            C.coef.insert(C.coef.end(), w.begin(), w.end());
          }
        }
        if (p == p0) col[(size_t)c] += B.nin();
      }
  }
  std::vector<int32_t> at;
};

// window slots that a phase's inputs take when they stand op by op, each op from an even slot
int64_t stage_slots(const FlatProgram& fp, int p) {
  int64_t s = 0;
  for (int32_t o = fp.base[p]; o < fp.base[p + 1]; ++o)
    if (!(fp.ops[o].flags & FF_SRC_VEC)) s += even(op_nin(fp.ops[o]));
  return s;
}

// A part of the sweep program: a resident run (all phases of one subtree), or a
// butterfly above the runs.
struct Unit {
  bool res;
  int first, count;
  int32_t row_lo, row_hi;
};

// Cut the program at the depth of the largest subtrees that fit the window: all
// subtrees of that depth become runs (every phase of a subtree is contiguous in the
// recursion's order), the phases of the butterflies above them global phases.
// stage: the largest stage of a run's butterflies (window slots).
std::vector<Unit> cut_program(const PackedHost& ph, const std::vector<DPhase>& prog, const FlatProgram& fp,
                              int64_t win_slots, int64_t& stage) {
  const int vl = ph.depth - ph.sl_t;   // depth of the sweep leaves
  const int np = (int)prog.size();
  std::vector<int> dep(np);            // depth and node of every phase
  std::vector<int64_t> node(np);
  std::vector<int64_t> need((size_t)vl + 1, 0);   // per depth the largest stage of its butterflies
  int v = 0;
  int64_t p = 0;
  for (int q = 0; q < np; ++q) {
    if (prog[q].kind == PH_LEAF) { dep[q] = vl; node[q] = prog[q].arg0; continue; }
    if (prog[q].kind == PH_ENTER) {
      const int64_t b = prog[q].arg0 / 2 + 1;   // 2^v + p
      v = 0;
      while ((int64_t)2 << v <= b) ++v;
      p = b - ((int64_t)1 << v);
    }
    dep[q] = v;
    node[q] = p;
    need[(size_t)v] = std::max(need[(size_t)v], stage_slots(fp, q));
  }
  const int64_t m = ph.n / ph.n0, ls = sw_leaf_stride((int32_t)ph.n0);
  int d = vl;
  stage = 0;
  while (d > 0) {
    const int64_t most = std::max(stage, need[(size_t)d - 1]);
    if ((m >> (d - 1)) * ls + 2 * most > win_slots) break;
    stage = most;
    --d;
  }
  std::vector<Unit> us;
  for (int q = 0; q < np;) {
    if (dep[q] < d) {
      int e = q + 1;   // from its entry phase to its exit phase
      while (e < np && prog[e].kind != PH_ENTER && prog[e].kind != PH_LEAF) ++e;
      us.push_back(Unit{false, q, e - q, 0, 0});
      q = e;
      continue;
    }
    const int64_t root = node[q] >> (dep[q] - d);
    int e = q;
    while (e < np && dep[e] >= d && (node[e] >> (dep[e] - d)) == root) ++e;
    const int64_t rows = ph.n >> d;
    us.push_back(Unit{(m >> d) * ls <= win_slots, q, e - q, (int32_t)(root * rows), (int32_t)((root + 1) * rows)});
    q = e;
  }
  return us;
}

template <class R>
void put_pair(uint8_t* dst, cplx a, cplx b) {
  const R p[4] = {(R)a.real(), (R)b.real(), (R)a.imag(), (R)b.imag()};
  std::memcpy(dst, p, sizeof(p));
}

// A row of a phase: op and row index in it.
struct RowRef {
  int32_t op, row;
};
// A batch before layout: rows of one phase in tile order (tile t takes rows [t rpt,
// (t + 1) rpt), rpt = 32 >> glog), or a triangle.
struct PBatch {
  std::vector<RowRef> rows;
  std::vector<int32_t> gl;       // global batches: the slice's entries
  int32_t reg_lo = 0, reg_hi = 0;   // inputs of the phase (resident) or of the batch stand in [reg_lo, reg_hi)
  int glog = 0;
  bool add = false;
  bool tri = false;
  int64_t tri_off = 0, tri_n = 0;   // triangle: offset in the sweep-leaf array, order
  int32_t a0 = 0;
};

// One phase part laid out on its own: descriptors with offsets relative to the
// part's data, and the data.
struct Part {
  int32_t flags = 0;   // SWP_*
  std::vector<SwDesc> descs;
  std::vector<uint8_t> data;
};

// Entries per lane of a tile whose longest row has nin inputs.  Resident tiles: a multiple
// of four, at least eight where the phase has that many inputs (the kernel then fetches
// four pairs ahead and reads the others two by two); avail: the phase's inputs.
inline int tile_len(int64_t nin, int glog, bool res, int64_t avail) {
  const int32_t e = std::max<int32_t>(2, even((even(nin) + ((int64_t)1 << glog) - 1) >> glog));
  if (!res) return e;
  const int32_t r = std::max(8, (e + 3) & ~3);
  return r <= avail ? r : e;
}

struct Builder {
  const PackedHost& ph;
  SwSched& S;
  int cb, which;
  std::vector<DenseOp> ops;   // the current phase
  // the group being collected
  std::vector<Part> pend;
  int64_t pend_bytes = 0;
  bool pend_res = false;
  Builder(const PackedHost& p, SwSched& s, int coef_bytes, int w) : ph(p), S(s), cb(coef_bytes), which(w) {}

  void pair_at(uint8_t* dst, cplx a, cplx b) {
    if (cb == 8) put_pair<float>(dst, a, b);
    else put_pair<double>(dst, a, b);
  }

  // entries per lane of each tile of a row batch
  std::vector<int> tile_lens(const PBatch& B, bool res) const {
    const size_t rpt = (size_t)(32 >> B.glog);
    std::vector<int> e;
    for (size_t r = 0; r < B.rows.size(); r += rpt) {
      int32_t nin = 0;
      for (size_t q = r; q < std::min(B.rows.size(), r + rpt); ++q) nin = std::max(nin, ops[B.rows[q].op].nin());
      e.push_back(tile_len(nin, B.glog, res, B.reg_hi - B.reg_lo));
    }
    return e;
  }
  int64_t batch_bytes(const PBatch& B, bool res) const {
    if (B.tri) return kSwTriTab + (int64_t)sw_tri_steps((int)B.tri_n) * 32 * cb;
    int64_t ne = 0, nt = 0;
    for (int e : tile_lens(B, res)) { ne += 32 * (int64_t)e; ++nt; }
    if (res) return kSwTileCoef + cb * ne;
    return al16(4 * (int64_t)B.rows.size()) + al16(4 * (nt + 1)) + 64 * nt + cb * ne + al16(4 * (int64_t)B.gl.size());
  }

  // lay out batches bs[b0, b1) as one part
  Part make_part(const std::vector<PBatch>& bs, size_t b0, size_t b1, bool res, int32_t pflags) {
    Part pt;
    pt.flags = pflags;
    for (size_t q = b0; q < b1; ++q) {
      const PBatch& B = bs[q];
      SwDesc D{};
      D.off = (int32_t)pt.data.size();
      D.glog = (int8_t)B.glog;
      if (B.tri) {
        const int s = (int)B.tri_n;
        D.nrows = s;
        D.nent = sw_tri_steps(s) * 32;
        D.a0 = B.a0;
        pt.data.resize(pt.data.size() + kSwTriTab + (int64_t)D.nent * cb, 0);
        uint8_t* d = pt.data.data() + D.off;
        const cplx* T = ph.sl[which].data() + B.tri_off;
        const bool up = which == 1 || which == 2;
        int step = 0;
        for (int v = 0; v < sw_tri_warps(s); ++v) {
          const SwTriWarp tw = sw_tri_warp(s, v);
          ((int32_t*)d)[v] = step << 16 | tw.n1 << 8 | tw.n0;
          for (int i = 0; i < tw.n1 + tw.n0; ++i, ++step)
            for (int q = 0; q < 16; ++q) {   // row pair q / 4, column group q % 4
              const int j = 4 * v + q / 4, r = i < tw.n1 ? s - 1 - j : j, p = q % 4 + 4 * (i < tw.n1 ? i : i - tw.n1);
              cplx w[2];
              if (sw_tri_live(s, j, i < tw.n1) && p < sw_tri_len(r)) {
                const int row = up ? s - 1 - r : r, c0 = up ? s - 2 - 2 * p : 2 * p;
                for (int u = 0; u < 2; ++u) {
                  const int c = c0 + u;
                  if (c < 0 || c >= s || (up ? c < row : c > row)) continue;
                  w[u] = up ? T[tri_off_upper(row, c)] : T[tri_off_lower(s, row, c)];
                }
              }
              pair_at(d + kSwTriTab + ((int64_t)step * 32 + 2 * q) * cb, w[0], w[1]);
            }
        }
        pt.descs.push_back(D);
        S.batches++;
        continue;
      }
      const int rpt = 32 >> B.glog, G = 1 << B.glog;
      const std::vector<int> te = tile_lens(B, res);
      int64_t ne = 0;
      for (int e : te) ne += 32 * (int64_t)e;
      const int64_t nr = (int64_t)B.rows.size(), nt = (int64_t)te.size();
      D.nrows = (int32_t)nr;
      D.nent = (int32_t)ne;
      D.ngl = (int32_t)B.gl.size();
      if (res) {
        D.elen = (int16_t)te[0];
        D.trows = (int8_t)nr;
        if (nt != 1 || te[0] > INT16_MAX) { S.ok = false; S.why = "resident tile"; return pt; }
        D.off_in = kSwTileIn;
        D.off_coef = kSwTileCoef;
        D.off_e0 = D.off_gl = D.off_coef + (int32_t)(cb * ne);
      } else {
        D.a0 = B.add ? B.reg_hi : 0;
        D.off_e0 = (int32_t)al16(4 * nr);
        D.off_in = D.off_e0 + (int32_t)al16(4 * (nt + 1));
        D.off_coef = D.off_in + 64 * (int32_t)nt;
        D.off_gl = D.off_coef + (int32_t)(cb * ne);
      }
      pt.data.resize(pt.data.size() + D.off_gl + (res ? 0 : al16(4 * (int64_t)D.ngl)), 0);
      uint8_t* d = pt.data.data() + D.off;
      uint8_t* cf = d + D.off_coef;
      int32_t* out = (int32_t*)d;
      int32_t* e0 = (int32_t*)(d + D.off_e0);
      int16_t* in = (int16_t*)(d + D.off_in);
      int32_t* gl = (int32_t*)(d + D.off_gl);
      if (!res) std::copy(B.gl.begin(), B.gl.end(), gl);
      int64_t t0 = 0;
      for (int64_t t = 0; t < nt; ++t) {
        const int E = te[(size_t)t];
        if (!res) e0[t] = (int32_t)(t0 / 32);
        for (int l = 0; l < 32; ++l) {
          const int64_t ri = t * rpt + (l >> B.glog);
          int32_t b = B.reg_lo;   // a lane without a row reads the phase's first inputs (coefficients 0)
          std::vector<cplx> w((size_t)E, cplx(0.0, 0.0));
          if (ri < nr) {
            const DenseOp& o = ops[B.rows[(size_t)ri].op];
            const int32_t r = B.rows[(size_t)ri].row, nin = o.nin();
            const int32_t lo = (l & (G - 1)) * E, hi = std::min<int32_t>(nin, lo + E);   // the lane's inputs
            // within the op's own slots; a lane longer than the op goes on within the region
            b = o.in0 + std::max(0, std::min(lo, even(nin) - E));
            b = std::max(B.reg_lo, std::min(b, B.reg_hi - E));
            for (int32_t i = lo; i < hi; ++i) w[(size_t)(o.in0 + i - b)] = o.coef[(size_t)r * nin + i];
            if ((l & (G - 1)) == 0) {
              out[ri] = o.out[(size_t)r];
              if (!res && B.add) gl[B.reg_hi + ri] = out[ri];
            }
          }
          if (b < 0 || (b & 1) || b + E > B.reg_hi) { S.ok = false; S.why = "inputs of a tile"; return pt; }
          in[32 * t + l] = (int16_t)b;
          for (int e = 0; e < E; e += 2) pair_at(cf + (t0 + sw_pos(e, l)) * cb, w[(size_t)e], w[(size_t)e + 1]);
        }
        t0 += 32 * (int64_t)E;
      }
      if (!res) e0[nt] = (int32_t)(t0 / 32);
      pt.descs.push_back(D);
      S.batches++;
    }
    return pt;
  }
  static int64_t part_bytes(const Part& pt) { return 8 + 40 * (int64_t)pt.descs.size() + (int64_t)pt.data.size(); }

  // write the collected parts as one group
  void flush(bool begin, int32_t beg_lo, int32_t beg_hi) {
    if (pend.empty()) return;
    const int64_t nph = (int64_t)pend.size();
    int64_t nd = 0;
    for (const Part& pt : pend) nd += (int64_t)pt.descs.size();
    const int64_t off_desc = al16(32 + 8 * nph);
    const int64_t off_data = al16(off_desc + 40 * nd);
    int64_t bytes = off_data;
    for (const Part& pt : pend) bytes += al16((int64_t)pt.data.size());
    if (bytes > INT32_MAX / 2) { S.ok = false; S.why = "group too large"; pend.clear(); return; }
    SwGroup G{(int64_t)S.image.size(), (int32_t)bytes, 0, 0, 0};
    S.image.resize((size_t)(G.img + bytes), 0);
    uint8_t* base = S.image.data() + G.img;
    SwGroupHdr H{(int32_t)nph, pend_res ? SWG_RES : 0, 0, 0, 0, 0, (int32_t)off_desc, 0};
    if (begin) {
      H.flags |= SWG_BEGIN;
      H.beg_lo = beg_lo;
      H.beg_hi = beg_hi;
    }
    std::memcpy(base, &H, sizeof(H));
    int64_t di = 0, dat = off_data;
    for (int64_t k = 0; k < nph; ++k) {
      const Part& pt = pend[k];
      const SwPhase ph_ent{(int32_t)pt.descs.size(), pt.flags | (int32_t)(di << kSwPhaseBase)};
      if (di > kSwBaseMask) { S.ok = false; S.why = "descriptors of a group"; }
      std::memcpy(base + 32 + 8 * k, &ph_ent, sizeof(ph_ent));
      for (SwDesc D : pt.descs) {
        D.off += (int32_t)dat;
        std::memcpy(base + off_desc + 40 * di, &D, sizeof(D));
        ++di;
      }
      if (!pt.data.empty()) std::memcpy(base + dat, pt.data.data(), pt.data.size());
      dat += al16((int64_t)pt.data.size());
    }
    S.max_bytes = std::max<int64_t>(S.max_bytes, bytes);
    S.groups.push_back(G);
    pend.clear();
    pend_bytes = 0;
  }

  // Lanes per row of a resident phase: the number that minimises the estimated cycles
  // of its dependent chain: the hand-over, then the tiles of the busiest warp of the set
  // (all warps for more than kSwSetTiles tiles) -- a fixed part, the first eight entries,
  // more for those not fetched ahead, one shuffle round per doubling, more for every
  // further tile of a warp.  The tiles' bytes, which the staging ring has to bring in,
  // are charged too.
  int resident_glog(const std::vector<RowRef>& order, int64_t avail) const {
    int best = 0;
    double bc = 1e300;
    for (int g = 0; g <= 5; ++g) {
      const size_t rpt = (size_t)(32 >> g);
      const int64_t nt = (int64_t)((order.size() + rpt - 1) / rpt);
      const bool all = nt > kSwSetTiles;
      double warp[kSwWarps] = {0}, bytes = 0;
      int t = 0;
      for (size_t r = 0; r < order.size(); r += rpt, ++t) {
        const int e = tile_len(ops[order[r].op].nin(), g, true, avail);   // rows by decreasing length: the first is the longest
        double& w = warp[t % (all ? kSwWarps : kSwSet)];
        w += 200.0 + 30.0 * g + (w > 0 ? 200.0 : 0.0) + (e > 8 ? 20.0 * (e - 8) : 0.0);
        bytes += 32.0 * e * cb + 40 + kSwTileCoef;
      }
      double w = 0;
      for (double x : warp) w = std::max(w, x);
      const double c = w + (all ? 400.0 : 0.0) + bytes / 64.0;
      if (c < bc) { bc = c; best = g; }
    }
    return best;
  }

  // Ops with more inputs than a slice holds, cut by rows into ops over the inputs that those
  // rows use (an ID's row uses one of the k skeletons: the other k - 1 columns are zero).
  void split_wide_ops() {
    std::vector<DenseOp> out;
    for (DenseOp& op : ops) {
      if (even(op.nin()) + (op.add ? 2 : 0) <= kSwGatherMax) { out.push_back(std::move(op)); continue; }
      const int32_t nin = op.nin();
      std::vector<char> use((size_t)nin, 0);
      int32_t r0 = 0, nuse = 0;
      auto emit = [&](int32_t r1) {
        DenseOp B;
        B.add = op.add;
        for (int32_t i = 0; i < nin; ++i)
          if (use[(size_t)i]) B.in.push_back(op.in[(size_t)i]);
        for (int32_t r = r0; r < r1; ++r) {
          B.out.push_back(op.out[(size_t)r]);
          for (int32_t i = 0; i < nin; ++i)
            if (use[(size_t)i]) B.coef.push_back(op.coef[(size_t)r * nin + i]);
        }
        out.push_back(std::move(B));
        std::fill(use.begin(), use.end(), 0);
        nuse = 0;
        r0 = r1;
      };
      for (int32_t r = 0; r < op.rows(); ++r) {
        const cplx* w = op.coef.data() + (size_t)r * nin;
        auto fresh = [&] {
          int32_t n = 0;
          for (int32_t i = 0; i < nin; ++i) n += !use[(size_t)i] && w[i] != cplx(0.0, 0.0);
          return n;
        };
        if (r > r0 && even(nuse + fresh()) + (op.add ? 2 : 0) > kSwGatherMax) emit(r);
        nuse += fresh();
        for (int32_t i = 0; i < nin; ++i)
          if (w[i] != cplx(0.0, 0.0)) use[(size_t)i] = 1;
      }
      emit(op.rows());
    }
    ops.swap(out);
  }

  void batches_of_phase(bool res, int32_t reg_lo, int32_t reg_hi, std::vector<PBatch>& bs) {
    bs.clear();
    std::vector<RowRef> order;
    if (res) {
      // a dependent phase: one batch per tile, rows by decreasing length
      for (size_t o = 0; o < ops.size(); ++o)
        for (int32_t r = 0; r < ops[o].rows(); ++r) order.push_back(RowRef{(int32_t)o, r});
      std::stable_sort(order.begin(), order.end(), [&](const RowRef& a, const RowRef& b) { return ops[a.op].nin() > ops[b.op].nin(); });
      const int g = resident_glog(order, reg_hi - reg_lo);
      const size_t rpt = (size_t)(32 >> g);
      for (size_t r = 0; r < order.size(); r += rpt) {
        PBatch B;
        B.glog = g;
        B.reg_lo = reg_lo;
        B.reg_hi = reg_hi;
        B.rows.assign(order.begin() + r, order.begin() + std::min(order.size(), r + rpt));
        bs.push_back(std::move(B));
      }
      return;
    }
    // wide phase: consecutive ops, batches of about a forty-eighth of the phase (three per
    // compute warp; 3 to 8 KB of coefficients, so that a dozen fit the staging ring) with at
    // most kSwGather inputs (an op with more: kSwGatherMax, by itself); an op whose rows exceed
    // that is split by rows
    split_wide_ops();
    int64_t tot = 0;
    for (const DenseOp& o : ops) tot += (int64_t)o.rows() * even(o.nin()) * cb;
    const int64_t target = std::max<int64_t>(3072, std::min<int64_t>(8192, tot / (3 * kSwWarps)));
    PBatch cur;
    int64_t acc = 0;
    auto close = [&]() {
      if (cur.rows.empty()) return;
      // rows by decreasing length (equal rows share a tile); as few lanes per row as fill
      // the tile: long dot products per lane cost the fewest instructions
      std::stable_sort(cur.rows.begin(), cur.rows.end(), [&](const RowRef& a, const RowRef& b) { return ops[a.op].nin() > ops[b.op].nin(); });
      int g = 0;
      while (g < 5 && cur.rows.size() <= (size_t)(32 >> (g + 1)) && (4 << g) < ops[cur.rows[0].op].nin()) ++g;
      cur.glog = g;
      cur.reg_lo = 0;
      cur.reg_hi = (int32_t)cur.gl.size();
      // rows that add: their old values are gathered after the inputs
      if (cur.add) cur.gl.resize((size_t)even((int64_t)cur.gl.size() + (int64_t)cur.rows.size()), -1);
      bs.push_back(std::move(cur));
      cur = PBatch();
      acc = 0;
    };
    for (size_t o = 0; o < ops.size(); ++o) {
      DenseOp& op = ops[o];
      const int32_t nin = op.nin(), ne = even(nin);
      const int32_t cap = ne + (op.add ? 2 : 0) > kSwGather ? kSwGatherMax : kSwGather;
      if (nin < 1 || ne + (op.add ? 2 : 0) > cap) { S.ok = false; S.why = "an op's inputs"; return; }
      const int64_t rb = (int64_t)ne * cb + 8;
      // an op opens a new batch when its rows would overfill the current one
      const int64_t slots = (int64_t)cur.gl.size() + ne + (op.add ? (int64_t)cur.rows.size() + op.rows() + 1 : 0);
      if (!cur.rows.empty() && (acc + rb * op.rows() > target || slots > kSwGather || cur.add != op.add)) close();
      // rows per batch of a large op (every batch gathers the op's inputs again; its
      // position in the slice is 0 there)
      int32_t per = (int32_t)std::max<int64_t>(8, target / rb);
      if (op.add) per = std::min(per, (cap - ne) & ~1);
      const bool split = op.rows() > 2 * per || (op.add && ne + op.rows() + 1 > cap);
      if (split) close();
      for (int32_t r = 0; r < op.rows(); ++r) {
        if (split && (int32_t)cur.rows.size() >= per) close();
        if (cur.rows.empty() || r == 0) {
          op.in0 = (int32_t)cur.gl.size();
          cur.add = op.add;
          for (int32_t e : op.in) cur.gl.push_back(e);
          if (nin & 1) cur.gl.push_back(-1);
        }
        cur.rows.push_back(RowRef{(int32_t)o, r});
        acc += rb;
      }
      if (split) close();
    }
    close();
  }

  // add a phase's batches to the groups: parts of at most kSwGroupBytes, the last one
  // ending the phase; resident parts share groups; a global batch is a group of its own
  void add_phase(const std::vector<PBatch>& bs, bool res, int32_t pflags, bool& begin, int32_t beg_lo, int32_t beg_hi) {
    size_t b0 = 0;
    while (b0 < bs.size()) {
      size_t b1 = b0;
      int64_t acc = 0;
      while (b1 < bs.size()) {
        const int64_t add = 40 + batch_bytes(bs[b1], res);
        if (b1 > b0 && (!res || acc + add > kSwGroupBytes)) break;
        acc += add;
        ++b1;
      }
      const bool last = b1 == bs.size();
      Part pt = make_part(bs, b0, b1, res, pflags & ~(last ? 0 : SWP_END));
      if (!S.ok) return;
      const int64_t pb = part_bytes(pt);
      if (!pend.empty() && (!res || !pend_res || (pflags & SWP_TRI) || pend_bytes + pb > kSwGroupBytes ||
                            (int)pend.size() >= kSwMaxPhases)) {
        flush(begin, beg_lo, beg_hi);
        begin = false;
      }
      pend_res = res;
      pend.push_back(std::move(pt));
      pend_bytes += pb;
      if (!res || (pflags & SWP_TRI)) {   // global parts and triangles form groups of their own
        flush(begin, beg_lo, beg_hi);
        begin = false;
      }
      b0 = b1;
    }
  }
};

}  // namespace

void build_sweep_sched(const PackedHost& ph, int which, int coef_bytes, int win_slots, SwSched& S) {
  // (resident runs: their groups are counted into the first one's header below)
  S = SwSched{};
  S.coef_bytes = coef_bytes;
  S.win_slots = std::max(1, std::min(win_slots, kSwWinSlots));
  const std::vector<DPhase>* progs[4] = {&ph.prog_lower, &ph.prog_upper, &ph.prog_lower_adj, &ph.prog_upper_adj};
  const std::vector<DPhase>& prog = *progs[which];
  if (ph.fpool.empty() || ph.sl[which].empty()) { S.ok = false; S.why = "factor data released"; return; }
  const FlatProgram fp = flatten_program(ph, prog, which);
  if (!fp.ok) { S.ok = false; S.why = "flattened program"; return; }
  int64_t stage = 0;
  const std::vector<Unit> units = cut_program(ph, prog, fp, S.win_slots, stage);
  Builder bd(ph, S, coef_bytes, which);
  Fuser fu(ph, fp);
  std::vector<int32_t> slot_of((size_t)ph.state_len, -1);   // window slots of a run's live state entries
  std::vector<PBatch> bs;
  std::vector<DenseOp> next;
  const int32_t n = (int32_t)ph.n, n0 = (int32_t)ph.n0;
  if ((int64_t)n + ph.state_len > INT32_MAX - 1) { S.ok = false; S.why = "state too long"; return; }
  for (const Unit& u : units) {
    const bool res = u.res;
    const int32_t row_slots = (u.row_hi - u.row_lo) / n0 * sw_leaf_stride(n0);
    bool begin = res;   // the run's first group loads its rows
    int half = 0;       // the state half that the current phase writes (it reads the other)
    bool bad = false;
    auto slot = [&](int32_t e) -> int32_t {   // window slot of vector row e or state entry e - n
      if (e >= n) return slot_of[(size_t)(e - n)];
      if (e < u.row_lo || e >= u.row_hi) { bad = true; return 0; }
      return sw_row_slot(e - u.row_lo, n0);
    };
    if (res) S.runs++;
    const size_t run_g0 = S.groups.size();
    // the unit's phases after fusing: triangles, entry phases, fused stages
    for (int p = u.first; p < u.first + u.count;) {
      if (fp.ops[fp.base[p]].kind == FK_LEAF) {
        // a sweep leaf always lies inside a resident run (its rows alone fit the window)
        if (!res || fp.base[p + 1] - fp.base[p] != 1) { S.ok = false; S.why = "sweep leaf outside a resident run"; return; }
        const FlatOp& f = fp.ops[fp.base[p]];
        bs.assign(1, PBatch());
        bs[0].tri = true;
        bs[0].tri_off = f.moff;
        bs[0].tri_n = f.c0;
        bs[0].a0 = slot(f.src0);
        bd.add_phase(bs, res, SWP_END | SWP_TRI | ((f.flags & FF_UPPER) ? SWP_UPPER : 0), begin, u.row_lo, u.row_hi);
        if (bad || !S.ok) { S.ok = false; return; }
        S.res_phases++;
        ++p;
        continue;
      }
      // a butterfly: phases [p, e)
      int e = p + 1;
      while (e < u.first + u.count && prog[e].kind != PH_ENTER && prog[e].kind != PH_LEAF) ++e;
      if (prog[p].kind != PH_ENTER || prog[e - 1].kind != PH_EXIT) { S.ok = false; S.why = "butterfly phases"; return; }
      std::vector<int> ends = fu.plan(p + 1, e, !res);
      ends.insert(ends.begin(), p + 1);
      fu.fuse(p, p + 1, bd.ops);
      for (size_t k = 0; k < ends.size(); ++k) {
        const bool more = k + 1 < ends.size();
        if (more) fu.fuse(ends[k], ends[k + 1], next);
        int32_t reg_lo = 0, reg_hi = row_slots;
        if (res) {
          if (k > 0) {
            reg_lo = row_slots + (int32_t)(stage * (half ^ 1));
            reg_hi = reg_lo;
            for (const DenseOp& o : bd.ops) reg_hi += even(o.nin());
          }
          // slots of this phase's outputs: in the order in which the next phase reads them
          if (more) {
            int32_t w = row_slots + (int32_t)(stage * half);
            for (const DenseOp& o : next) {
              for (int32_t i = 0; i < o.nin(); ++i) slot_of[(size_t)(o.in[(size_t)i] - n)] = w + i;
              w += even(o.nin());
            }
            if (w > row_slots + stage * (half + 1)) bad = true;
          }
          for (DenseOp& o : bd.ops) {
            o.in0 = slot(o.in[0]);
            if (o.in0 & 1) bad = true;
            for (int32_t i = 1; i < o.nin(); ++i)
              if (slot(o.in[(size_t)i]) != o.in0 + i) bad = true;
            for (int32_t& w : o.out) w = slot(w) | (o.add ? kSwAcc : 0);
          }
          half ^= 1;
        }
        if (bad || (res && row_slots + 2 * stage > S.win_slots)) { S.ok = false; S.why = "slot outside the run's window"; return; }
        bd.batches_of_phase(res, reg_lo, reg_hi, bs);
        if (!S.ok) return;
        const size_t g0 = S.groups.size();
        bd.add_phase(bs, res, SWP_END, begin, u.row_lo, u.row_hi);
        if (!S.ok) return;
        if (res) {
          S.res_phases++;
        } else {
          S.glob_phases++;
          // the phase's first group tells how many it has, and whether a list exceeds half a slice
          uint8_t* hb = S.image.data() + S.groups[g0].img;
          SwGroupHdr H;
          std::memcpy(&H, hb, sizeof(H));
          H.aux = (int32_t)(S.groups.size() - g0);
          for (const PBatch& B : bs)
            if ((int64_t)B.gl.size() > kSwGather) H.flags |= SWG_WIDE;
          std::memcpy(hb, &H, sizeof(H));
        }
        if (more) bd.ops.swap(next);
      }
      p = e;
    }
    bd.flush(begin, u.row_lo, u.row_hi);
    begin = false;
    if (res && S.groups.size() > run_g0) {
      // the run's last group writes the rows back after its last phase; its first
      // group tells how many groups the run has
      SwGroupHdr H;
      uint8_t* hb = S.image.data() + S.groups.back().img;
      std::memcpy(&H, hb, sizeof(H));
      H.flags |= SWG_ENDRUN;
      H.end_lo = u.row_lo;
      H.end_hi = u.row_hi;
      std::memcpy(hb, &H, sizeof(H));
      hb = S.image.data() + S.groups[run_g0].img;
      std::memcpy(&H, hb, sizeof(H));
      if (!(H.flags & SWG_BEGIN)) { S.ok = false; S.why = "resident run without its first group"; return; }
      H.aux = (int32_t)(S.groups.size() - run_g0);
      H.flags |= (int32_t)(row_slots + 2 * stage) << kSwGroupSlots;
      std::memcpy(hb, &H, sizeof(H));
      // phase by phase: the warps that compute it, the barrier after it
      int32_t* prev = nullptr;
      int set = 0, rot = 0;
      for (size_t gi = run_g0; gi < S.groups.size(); ++gi) {
        hb = S.image.data() + S.groups[gi].img;
        std::memcpy(&H, hb, sizeof(H));
        for (int k = 0; k < H.nph; ++k) {
          SwPhase* PH = reinterpret_cast<SwPhase*>(hb + 32 + 8 * k);
          if ((PH->flags & SWP_TRI) || !(PH->flags & SWP_END) || (prev && !(*prev & SWP_END)) || PH->nb > kSwSetTiles) {
            PH->flags |= SWP_ALL | rot << kSwPhaseWarp;
            rot = (PH->flags & SWP_END) ? 0 : (rot + PH->nb) % kSwWarps;
          } else {
            set ^= 1;
            if (set) PH->flags |= SWP_SET1;
            if (prev && !(*prev & SWP_ALL)) *prev |= SWP_HAND;
          }
          prev = &PH->flags;
        }
      }
    }
  }
  // (the device stages complex-FP32 images; FP64 images serve host checks only)
  if (coef_bytes == 8 && S.max_bytes > kSwRingBytes) { S.ok = false; S.why = "group image larger than the staging ring"; return; }
  // places in the ring, one after the other, and what must be consumed before
  int32_t head = 0, need = 0;
  for (size_t g = 0; g < S.groups.size(); ++g) {
    SwGroup& G = S.groups[g];
    if (head + G.bytes > kSwRingBytes) head = 0;
    G.off = head;
    head += G.bytes;
    need = std::max(need, (int32_t)g - kSwAhead + 1);
    for (int32_t q = (int32_t)g - 1; q >= need; --q)   // the latest group that overlaps
      if (S.groups[(size_t)q].off < G.off + G.bytes && G.off < S.groups[(size_t)q].off + S.groups[(size_t)q].bytes) need = q + 1;
    G.need = need;
  }
}

void host_sweep_sched(const PackedHost& ph, const SwSched& S, cplx* vec) {
  const int64_t n = ph.n;
  const int32_t n0 = (int32_t)ph.n0;
  std::vector<cplx> st((size_t)ph.state_len, cplx(0.0, 0.0)), win(kSwWinSlots), tmp, gv;
  // entries 2i, 2i + 1 of a pair at p
  auto pair = [&](const uint8_t* p, cplx* v) {
    double d[4];
    if (S.coef_bytes == 8) {
      float f[4];
      std::memcpy(f, p, 16);
      for (int i = 0; i < 4; ++i) d[i] = f[i];
    } else {
      std::memcpy(d, p, 32);
    }
    v[0] = cplx(d[0], d[2]);
    v[1] = cplx(d[1], d[3]);
  };
  auto gslot = [&](int32_t sl) -> cplx& { return sl < n ? vec[sl] : st[sl - n]; };
  // a phase's outputs are stored when it ends (its parts never read them)
  struct Out { bool res; int32_t o; cplx v; };
  std::vector<Out> outs;
  for (const SwGroup& G : S.groups) {
    const uint8_t* gb = S.image.data() + G.img;
    SwGroupHdr H;
    std::memcpy(&H, gb, sizeof(H));
    if (H.flags & SWG_BEGIN) {
      std::fill(win.begin(), win.begin() + (H.flags >> kSwGroupSlots), cplx(0.0, 0.0));
      for (int32_t r = H.beg_lo; r < H.beg_hi; ++r) win[sw_row_slot(r - H.beg_lo, n0)] = vec[r];
    }
    const bool res = (H.flags & SWG_RES) != 0;
    for (int32_t k = 0; k < H.nph; ++k) {
      SwPhase PH;
      std::memcpy(&PH, gb + 32 + 8 * k, sizeof(PH));
      for (int32_t b = 0; b < PH.nb; ++b) {
        SwDesc D;
        std::memcpy(&D, gb + H.off_desc + 40 * (((PH.flags >> kSwPhaseBase) & kSwBaseMask) + b), sizeof(D));
        const uint8_t* base = gb + D.off;
        if (PH.flags & SWP_TRI) {
          const int s = D.nrows;
          tmp.assign((size_t)s, cplx(0.0, 0.0));
          const bool up = (PH.flags & SWP_UPPER) != 0;
          // (the leaves of a sweep leaf start at multiples of the leaf stride)
          auto slot = [&](int i) { return D.a0 + sw_row_slot(i, n0); };
          for (int v = 0; v < sw_tri_warps(s); ++v) {
            const int32_t tw = ((const int32_t*)base)[v];
            const int n1 = (tw >> 8) & 0xff, nn0 = tw & 0xff;
            for (int i = 0; i < n1 + nn0; ++i)
              for (int q = 0; q < 16; ++q) {
                const int j = 4 * v + q / 4, r = i < n1 ? s - 1 - j : j, p = q % 4 + 4 * (i < n1 ? i : i - n1);
                if (!sw_tri_live(s, j, i < n1)) continue;
                cplx w[2];
                pair(base + kSwTriTab + ((int64_t)((tw >> 16) + i) * 32 + 2 * q) * S.coef_bytes, w);
                for (int u = 0; u < 2; ++u) {
                  const int c = (up ? s - 2 - 2 * p : 2 * p) + u;
                  if (c >= 0 && c < s) tmp[up ? s - 1 - r : r] += w[u] * win[slot(c)];
                }
              }
          }
          for (int r = 0; r < s; ++r) win[slot(r)] = tmp[r];
          continue;
        }
        const int32_t* out = (const int32_t*)base;
        const int32_t* e0 = (const int32_t*)(base + D.off_e0);
        const int16_t* in = (const int16_t*)(base + D.off_in);
        const int32_t* gl = (const int32_t*)(base + D.off_gl);
        const uint8_t* cf = base + D.off_coef;
        if (!res) {
          gv.assign((size_t)D.ngl, cplx(0.0, 0.0));
          for (int32_t q = 0; q < D.ngl; ++q)
            if (gl[q] >= 0) gv[q] = gslot(gl[q]);
        }
        const int rpt = 32 >> D.glog, Gl = 1 << D.glog;
        for (int t = 0; t < sw_tiles(D.nrows, D.glog); ++t) {
          const int64_t t0 = res ? 0 : 32 * (int64_t)e0[t];
          const int elen = res ? D.elen : e0[t + 1] - e0[t];
          for (int i = 0; i < rpt && t * rpt + i < D.nrows; ++i) {
            const int32_t o = out[t * rpt + i];
            cplx acc(0.0, 0.0);
            if (!res && D.a0) acc = gv[(size_t)(D.a0 + t * rpt + i)];   // the row's old value
            for (int l = i * Gl; l < (i + 1) * Gl; ++l)
              for (int e = 0; e < elen; e += 2) {
                cplx v[2];
                pair(cf + (t0 + sw_pos(e, l)) * S.coef_bytes, v);
                // (a resident tile's inputs by the kernel's rule)
                const int e2 = res && e < 2 * kSwTilePairs ? 2 * sw_tile_pair(e / 2, elen / 2) : e;
                for (int q = 0; q < 2; ++q) {
                  const int32_t at = in[32 * t + l] + e2 + q;
                  acc += v[q] * (res ? win[at] : gv[at]);
                }
              }
            outs.push_back(Out{res, o, acc});
          }
        }
      }
      if (PH.flags & SWP_END) {
        for (const Out& ov : outs) {
          const bool add = (ov.o & kSwAcc) != 0;
          const int32_t sl = ov.o & ~kSwAcc;
          cplx* d = ov.res ? &win[sl] : &gslot(sl);
          *d = add ? *d + ov.v : ov.v;
        }
        outs.clear();
      }
    }
    if (H.flags & SWG_ENDRUN)
      for (int32_t r = H.end_lo; r < H.end_hi; ++r) vec[r] = win[sw_row_slot(r - H.end_lo, n0)];
  }
}

const char* check_sweep_sched(const PackedHost& ph, const SwSched& S) {
  const int64_t n = ph.n;
  const int32_t n0 = (int32_t)ph.n0;
  const int cb = S.coef_bytes;
  int64_t run_left = 0;   // groups of the current resident run still to come
  int64_t glob_left = 0;  // groups of the current global phase still to come
  bool wide = false;      // its lists may take a whole slice
  int32_t win_rows = 0, run_slots = 0;   // window slots of the run's rows; all that it uses
  // per window slot: the last resident phase that wrote / read it (a resident
  // phase's batches run concurrently on the compute warps, so no slot may be
  // written twice in a phase, nor written and read by the same phase)
  std::vector<int64_t> wstamp((size_t)S.win_slots, -1), rstamp((size_t)S.win_slots, -1);
  int64_t pid = 0;
  int32_t last = SWP_ALL;   // flags of the run's previous phase
  for (size_t gi = 0; gi < S.groups.size(); ++gi) {
    const SwGroup& G = S.groups[gi];
    if (G.img % 16 || G.bytes % 16 || G.bytes <= 0) return "group not 16-byte aligned";
    if (cb == 8 && G.bytes > kSwRingBytes) return "group larger than the ring";
    if (G.img + G.bytes > (int64_t)S.image.size()) return "group outside the image";
    if (cb == 8) {
      if (G.off < 0 || G.off % 16 || G.off + G.bytes > kSwRingBytes) return "place in the ring";
      if (G.need > (int32_t)gi || G.need < (int32_t)gi - kSwAhead + 1 || (gi > 0 && G.need < S.groups[gi - 1].need)) return "groups in flight";
      for (int32_t q = std::max(0, G.need); q < (int32_t)gi; ++q)
        if (S.groups[q].off < G.off + G.bytes && G.off < S.groups[q].off + S.groups[q].bytes) return "groups overlap in the ring";
    }
    const uint8_t* gb = S.image.data() + G.img;
    SwGroupHdr H;
    std::memcpy(&H, gb, sizeof(H));
    const bool res = (H.flags & SWG_RES) != 0;
    if (H.nph < 1 || 32 + 8 * (int64_t)H.nph > H.off_desc || (H.off_desc & 15)) return "phase table";
    if (res) {
      if (glob_left != 0) return "resident group inside a global phase";
      if (run_left == 0) {
        if (!(H.flags & SWG_BEGIN) || H.aux < 1) return "run start without BEGIN or length";
        run_left = H.aux;
        if (H.beg_lo < 0 || H.beg_hi <= H.beg_lo || H.beg_hi > n || H.beg_lo % n0 || H.beg_hi % n0) return "run rows";
        win_rows = (H.beg_hi - H.beg_lo) / n0 * sw_leaf_stride(n0);
        run_slots = H.flags >> kSwGroupSlots;
        if (win_rows > run_slots || run_slots > S.win_slots || (run_slots & 1)) return "run rows";
      } else if (H.flags & SWG_BEGIN) {
        return "BEGIN inside a run";
      }
      --run_left;
      if ((run_left == 0) != ((H.flags & SWG_ENDRUN) != 0)) return "ENDRUN not on the run's last group";
    } else {
      if (run_left != 0) return "global group inside a run";
      if (H.nph != 1) return "global group with several phases";
      SwPhase P0;
      std::memcpy(&P0, gb + 32, sizeof(P0));
      if (P0.nb != 1) return "global group with several batches";
      if (glob_left == 0) {
        if (H.aux < 1) return "global phase without its length";
        glob_left = H.aux;
        wide = (H.flags & SWG_WIDE) != 0;
      }
      --glob_left;
      if ((glob_left == 0) != ((P0.flags & SWP_END) != 0)) return "end of a global phase";
    }
    int64_t di = 0;
    for (int32_t k = 0; k < H.nph; ++k) {
      SwPhase PH;
      std::memcpy(&PH, gb + 32 + 8 * k, sizeof(PH));
      if (PH.nb < 1) return "empty phase part";
      if (((PH.flags >> kSwPhaseBase) & kSwBaseMask) != di) return "first descriptor of a phase";
      if ((PH.flags & SWP_TRI) && (PH.nb != 1 || !res || H.nph != 1)) return "triangle part";
      if (res && !(PH.flags & SWP_END)) {
        // a resident phase split over groups: only its last part ends it
        if (k + 1 != H.nph) return "unfinished resident phase inside a group";
      }
      for (int32_t b = 0; b < PH.nb; ++b, ++di) {
        SwDesc D;
        if (H.off_desc + 40 * (di + 1) > G.bytes) return "descriptor outside the group";
        std::memcpy(&D, gb + H.off_desc + 40 * di, sizeof(D));
        if (D.off % 16 || D.off < H.off_desc) return "batch offset";
        if (PH.flags & SWP_TRI) {
          const int64_t s = D.nrows;
          if (s < 1 || s % n0) return "triangle order";
          if (D.off + kSwTriTab + (int64_t)sw_tri_steps((int)s) * 32 * cb > G.bytes) return "triangle outside the group";
          if (sw_tri_warps((int)s) > 2 * kSwWarps) return "triangle order";   // (a warp takes two parts at most)
          int step = 0;
          for (int v = 0; v < sw_tri_warps((int)s); ++v) {
            const SwTriWarp tw = sw_tri_warp((int)s, v);
            if (((const int32_t*)(gb + D.off))[v] != (step << 16 | tw.n1 << 8 | tw.n0)) return "triangle table";
            step += tw.n1 + tw.n0;
          }
          if (D.a0 < 0 || D.a0 % sw_leaf_stride(n0) || D.a0 + s / n0 * sw_leaf_stride(n0) > win_rows)
            return "triangle rows outside the window rows";
          continue;
        }
        const int64_t end = D.off + D.off_gl + (res ? 0 : al16(4 * (int64_t)D.ngl));
        if (end > G.bytes) return "batch outside the group";
        if (D.glog < 0 || D.glog > 5) return "lanes per row";
        if (!res && (D.ngl < 0 || D.ngl > (wide ? kSwGatherMax : kSwGather) || (D.ngl & 1))) return "gather list longer than a warp slice";
        const uint8_t* bb = gb + D.off;
        const int32_t* out = (const int32_t*)bb;
        const int32_t* e0 = (const int32_t*)(bb + D.off_e0);
        const int16_t* in = (const int16_t*)(bb + D.off_in);
        const int32_t* gl = (const int32_t*)(bb + D.off_gl);
        const int nt = sw_tiles(D.nrows, D.glog);
        if (D.nrows < 1 || D.off_coef % 16) return "batch layout";
        if (D.off_gl < D.off_coef + cb * D.nent || D.off_coef < D.off_in + 64 * nt) return "batch layout";
        if (res) {
          // the kernel finds a tile's pieces at fixed places
          if (nt != 1 || D.trows != D.nrows || D.elen < 2 || (D.elen & 1) || D.nent != D.elen * 32 ||
              D.off_in != kSwTileIn || D.off_coef != kSwTileCoef)
            return "resident tile";
        } else {
          if (D.off_e0 % 16 || D.off_e0 < 4 * D.nrows || D.off_in < D.off_e0 + 4 * (nt + 1) || D.off_gl % 16) return "batch layout";
          if (e0[0] != 0 || 32 * e0[nt] != D.nent) return "tile offsets";
          for (int t = 0; t < nt; ++t)
            if (e0[t + 1] - e0[t] < 2 || ((e0[t + 1] - e0[t]) & 1)) return "tile offsets";
        }
        for (int32_t r = 0; r < D.nrows; ++r) {
          if (!res && (out[r] & kSwAcc)) return "global row that adds in place";
          const int32_t o = out[r] & ~kSwAcc;
          if (res ? (o < 0 || o >= run_slots) : (o < 0 || o >= n + ph.state_len)) return "output slot";
          if (res) {
            if (wstamp[o] == pid) return "window slot written twice in one phase";
            if (rstamp[o] == pid) return "window slot read and written in one phase";
            wstamp[o] = pid;
          }
        }
        for (int t = 0; t < nt; ++t) {
          const int elen = res ? D.elen : e0[t + 1] - e0[t];
          for (int l = 0; l < 32; ++l) {
            const int32_t i0 = in[32 * t + l];
            if (i0 < 0 || i0 + elen > (res ? run_slots : D.a0 ? D.a0 : D.ngl)) return "input slot";
            if (res)
              for (int32_t i = i0; i < i0 + elen; ++i) {
                if (wstamp[i] == pid) return "window slot read and written in one phase";
                rstamp[i] = pid;
              }
            if (i0 & 1) return "inputs from an odd slot";
          }
        }
        if (!res && D.a0) {
          if (D.a0 < 2 || (D.a0 & 1) || D.a0 + D.nrows > D.ngl) return "old values of the rows";
          for (int32_t r = 0; r < D.nrows; ++r)
            if (gl[D.a0 + r] != out[r]) return "old values of the rows";
        }
        for (int32_t q = 0; q < D.ngl && !res; ++q)
          if (gl[q] < -1 || gl[q] >= n + ph.state_len) return "gathered slot";
      }
      if (res && (PH.flags & SWP_END)) ++pid;
      if (res) {
        // who computes, and the hand-over: only from one set to the other
        const bool all = (PH.flags & SWP_ALL) != 0;
        if (!all && ((PH.flags & SWP_TRI) || !(PH.flags & SWP_END))) return "phase of one set";
        if ((PH.flags >> kSwPhaseWarp) < 0 || (PH.flags >> kSwPhaseWarp) >= kSwWarps) return "first warp of a phase";
        if (all && (PH.flags & (SWP_HAND | SWP_SET1))) return "hand-over after a phase of all warps";
        if ((H.flags & SWG_BEGIN) && k == 0) last = SWP_ALL;
        if ((last & SWP_HAND) && (all || ((last ^ PH.flags) & SWP_SET1) == 0)) return "hand-over to the same set";
        if ((H.flags & SWG_ENDRUN) && k + 1 == H.nph && (PH.flags & SWP_HAND)) return "hand-over after the run's last phase";
        last = PH.flags;
      }
    }
  }
  if (run_left != 0 || glob_left != 0) return "run not closed";
  return "";
}

}  // namespace hb
