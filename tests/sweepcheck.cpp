// Host checks of the column-partitioned sweep schedules over coarse and fine factors (test
// helper; built by tests/test_sweep_shapes.py with g++ against the library's host code).
//
//   sweepcheck CHECK arc|strip|strips8 n leaf eps     (strips8: eight parallel strips, 0.3 wavelengths apart)
//
// CHECK = region: fails unless the structural check refuses a schedule of which one tile reads past
// the slots of its run, inside the window.
//
// CHECK = wide: prints the longest gather list of a global batch with the smallest resident
// window, the number of inputs of the longest op, and the number of sweeps with a schedule;
// fails where a schedule is off the packed program's sweep by more than 1e-5.
//
// CHECK = tiles3: prints how many resident tiles have three entry pairs whose third pair is
// not zero (all four sweeps), and fails where a schedule with complex-FP32 coefficients,
// executed with the kernel's input rule, is off the packed program's sweep by more than 1e-5.
//
// CHECK = nan, nan_small (the smallest resident window): a NaN in one row of the second of a CTA's two right-hand sides, the shared
// memory of the kernel followed byte by byte (window, gather slices, entry pairs; a run whose
// rows come out non-finite once more with the zero coefficients masked).  Fails where the first
// right-hand side changes, or the second one is finite in other rows than the packed program's
// sweep.  Also with a value whose products overflow in place of the NaN: fails where the first
// right-hand side changes, or rows of the second one that do not depend on the value.  Rows: a
// few at the edges of leaves and of the resident runs.
//
//   sweepcheck triangle
//
// fails where a step of a triangle product of even order (2 .. 256, lower and upper) reads a
// column that is not the triangle's.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "hb_internal.h"

using namespace hb;

namespace {

PackedHost pack(const char* curve, int64_t n, int64_t leaf, double eps) {
  Geometry g;
  const double len = n / 20.0;
  const double arc[3] = {len / M_PI, 0.0, M_PI}, strip[4] = {0.0, 0.0, len, 0.0}, strips8[3] = {8.0, len / 8.0, 0.3};
  const bool a = !std::strcmp(curve, "arc"), s8 = !std::strcmp(curve, "strips8");
  HostFactor hf;
  PackedHost ph;
  if (build_geometry(a ? HB_ARC : s8 ? HB_PARALLEL_STRIPS : HB_STRIP, a ? arc : s8 ? strips8 : strip, a || s8 ? 3 : 4, n, g) ||
      build_factor(g, 1.0, 376.73, 1.781072, leaf, eps, 1, hf, 0)) {
    std::printf("FAIL: factor\n");
    std::exit(1);
  }
  pack_factor(hf, ph);
  return ph;
}

std::vector<cplx> vec(int64_t n) {
  std::vector<cplx> v((size_t)n);
  uint64_t s = 88172645463325252ull;
  auto u = [&] {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    return (double)(s >> 11) / (double)(1ull << 53) - 0.5;
  };
  for (cplx& e : v) { const double a = u(); e = cplx(a, u()); }
  return v;
}

// every resident row batch of a schedule: fn(descriptor, its data)
template <class Fn>
void resident_tiles(const SwSched& S, Fn fn) {
  for (const SwGroup& G : S.groups) {
    const uint8_t* gb = S.image.data() + G.img;
    SwGroupHdr H;
    std::memcpy(&H, gb, sizeof(H));
    int64_t di = 0;
    for (int k = 0; k < H.nph; ++k) {
      SwPhase PH;
      std::memcpy(&PH, gb + 32 + 8 * k, sizeof(PH));
      for (int b = 0; b < PH.nb; ++b, ++di) {
        SwDesc D;
        std::memcpy(&D, gb + H.off_desc + 40 * di, sizeof(D));
        if ((H.flags & SWG_RES) && !(PH.flags & SWP_TRI)) fn(D, gb + D.off);
      }
    }
  }
}

int region(const PackedHost& ph) {
  SwSched S;
  build_sweep_sched(ph, 0, 8, kSwWinSlots, S);
  SwGroupHdr H;
  std::memcpy(&H, S.image.data() + S.groups[0].img, sizeof(H));
  const int slots = H.flags >> kSwGroupSlots;
  bool done = false;
  resident_tiles(S, [&](const SwDesc& D, const uint8_t* data) {
    if (!done) reinterpret_cast<int16_t*>(const_cast<uint8_t*>(data) + D.off_in)[0] = (int16_t)slots;
    done = true;
  });
  const std::string got = check_sweep_sched(ph, S);
  std::printf("%s\n", got.c_str());
  return slots + 64 <= kSwWinSlots && got == "input slot" ? 0 : 1;
}

// relative distance of a schedule's sweep from the packed program's
double distance(const PackedHost& ph, const SwSched& S, int which) {
  std::vector<cplx> x = vec(ph.n), r = x;
  host_sweep_sched(ph, S, x.data());
  HostFactor none;
  host_sweep(ph, none, which, r.data());
  double e = 0, d = 0;
  for (int64_t i = 0; i < ph.n; ++i) { e += std::norm(x[i] - r[i]); d += std::norm(r[i]); }
  return std::sqrt(e / d);
}

int wide(const PackedHost& ph) {
  int longest = 0, nin = 0, sweeps = 0;
  for (const DItem& it : ph.items) nin = std::max(nin, (int)it.a_k[0] + it.a_k[1]);
  for (int which = 0; which < 4; ++which) {
    SwSched S;
    build_sweep_sched(ph, which, 8, 512, S);
    if (!S.ok) continue;
    ++sweeps;
    if (const char* bad = check_sweep_sched(ph, S); *bad) { std::printf("FAIL: %s\n", bad); return 1; }
    for (const SwGroup& G : S.groups) {
      const uint8_t* gb = S.image.data() + G.img;
      SwGroupHdr H;
      SwDesc D;
      std::memcpy(&H, gb, sizeof(H));
      std::memcpy(&D, gb + H.off_desc, sizeof(D));
      if (!(H.flags & SWG_RES)) longest = std::max(longest, D.ngl);
    }
    const double e = distance(ph, S, which);
    if (!(e <= 1e-5)) { std::printf("FAIL: sweep %d off by %.3g\n", which, e); return 1; }
  }
  std::printf("list %d inputs %d sweeps %d\n", longest, nin, sweeps);
  return 0;
}

int tiles3(const PackedHost& ph) {
  int count = 0;
  for (int which = 0; which < 4; ++which) {
    SwSched S;
    build_sweep_sched(ph, which, 8, kSwWinSlots, S);
    if (!S.ok) { std::printf("FAIL: no schedule: %s\n", S.why); return 1; }
    if (const char* bad = check_sweep_sched(ph, S); *bad) { std::printf("FAIL: %s\n", bad); return 1; }
    resident_tiles(S, [&](const SwDesc& D, const uint8_t* data) {
      if (D.elen != 6) return;
      const float* c = reinterpret_cast<const float*>(data + D.off_coef);
      bool live = false;
      for (int l = 0; l < 32; ++l)
        for (int u = 0; u < 4; ++u) live = live || c[2 * sw_pos(4, l) + u] != 0.f;
      count += live;
    });
    const double e = distance(ph, S, which);
    if (!(e <= 1e-5)) { std::printf("FAIL: sweep %d off by %.3g\n", which, e); return 1; }
  }
  std::printf("tiles %d\n", count);
  return 0;
}

// Shared memory of one CTA with two right-hand sides (window slots in pairs, slices as gathered
// and in pairs), and its sweep over x[2].
struct Cta {
  static constexpr int NC = 2;
  const PackedHost& ph;
  const SwSched& S;
  std::vector<float> win = std::vector<float>(kSwWinBytes / 4, 0.f);
  std::vector<std::complex<float>> x[NC], st[NC];
  struct Out {
    int32_t o;
    float v[NC][2];
  };
  std::vector<Out> outs;   // of the current phase, stored when it ends
  int batch = 0;           // of the current global phase
  bool wide = false;       // its lists may take a whole slice

  Cta(const PackedHost& p, const SwSched& s) : ph(p), S(s) {
    for (auto& v : st) v.assign((size_t)ph.state_len, 0.f);
  }
  float* slot(int s, int c) { return win.data() + (s >> 1) * 4 * NC + 4 * c + (s & 1); }   // im two floats further
  std::complex<float>& global(int32_t s, int c) { return s < ph.n ? x[c][(size_t)s] : st[c][(size_t)(s - ph.n)]; }

  // sums of one row: its lanes' entries over pairs that start at float `base` of the window
  void row(const SwDesc& D, const uint8_t* d, int t, int i, int64_t t0, int elen, bool res, size_t base, bool mask,
           float (&v)[NC][2]) {
    const float* cf = reinterpret_cast<const float*>(d + D.off_coef);
    const int16_t* in = reinterpret_cast<const int16_t*>(d + D.off_in);
    for (int c = 0; c < NC; ++c) {
      float re = 0, im = 0;
      for (int l = i << D.glog; l < (i + 1) << D.glog; ++l)
        for (int e = 0; e < elen; e += 2) {
          const float* m = cf + 2 * (t0 + sw_pos(e, l));
          const int e2 = res && e < 2 * kSwTilePairs ? 2 * sw_tile_pair(e / 2, elen / 2) : e;
          const float* w = win.data() + base + (size_t)(in[32 * t + l] + e2) / 2 * 4 * NC + 4 * c;
          for (int q = 0; q < 2; ++q) {
            if (mask && m[q] == 0.f && m[2 + q] == 0.f) continue;
            re += m[q] * w[q] - m[2 + q] * w[2 + q];
            im += m[q] * w[2 + q] + m[2 + q] * w[q];
          }
        }
      v[c][0] = re;
      v[c][1] = im;
    }
  }
  void triangle(const SwDesc& D, const uint8_t* d, bool up, bool mask) {
    const int s = D.nrows, n0 = (int)ph.n0;
    mask = mask || (n0 & 1);
    std::vector<float> out((size_t)s * NC * 2, 0.f);
    for (int v = 0; v < sw_tri_warps(s); ++v) {
      const int32_t tw = reinterpret_cast<const int32_t*>(d)[v];
      const int n1 = (tw >> 8) & 0xff, nn0 = tw & 0xff;
      for (int i = 0; i < n1 + nn0; ++i)
        for (int q = 0; q < 16; ++q) {
          const int j = 4 * v + q / 4, r = i < n1 ? s - 1 - j : j, p = q % 4 + 4 * (i < n1 ? i : i - n1);
          if (!sw_tri_live(s, j, i < n1)) continue;
          if (!mask && p / 4 >= sw_tri_take(s, p % 4, i < n1 ? n1 : nn0)) continue;
          const float* m = reinterpret_cast<const float*>(d + kSwTriTab) + ((int64_t)((tw >> 16) + i) * 32 + 2 * q) * 2;
          for (int u = 0; u < 2; ++u) {
            const int c0 = (up ? s - 2 - 2 * p : 2 * p) + u, row = up ? s - 1 - r : r;
            if (mask && (c0 < 0 || c0 >= s || (up ? c0 < row : c0 > row))) continue;
            for (int c = 0; c < NC; ++c) {
              const float* w = slot(D.a0 + sw_row_slot(c0, n0), c);
              out[((size_t)row * NC + c) * 2] += m[u] * w[0] - m[2 + u] * w[2];
              out[((size_t)row * NC + c) * 2 + 1] += m[u] * w[2] + m[2 + u] * w[0];
            }
          }
        }
    }
    for (int r = 0; r < s; ++r)
      for (int c = 0; c < NC; ++c) {
        float* w = slot(D.a0 + sw_row_slot(r, n0), c);
        w[0] = out[((size_t)r * NC + c) * 2];
        w[2] = out[((size_t)r * NC + c) * 2 + 1];
      }
  }
  void group(const SwGroup& G, bool mask) {
    const int n0 = (int)ph.n0;
    const uint8_t* gb = S.image.data() + G.img;
    SwGroupHdr H;
    std::memcpy(&H, gb, sizeof(H));
    const bool res = (H.flags & SWG_RES) != 0;
    if (!res && H.aux > 0) wide = (H.flags & SWG_WIDE) != 0;
    if (H.flags & SWG_BEGIN) {
      std::fill(win.begin(), win.begin() + (H.flags >> kSwGroupSlots) * 2 * NC, 0.f);
      for (int32_t r = 0; r < H.beg_hi - H.beg_lo; ++r)
        for (int c = 0; c < NC; ++c) {
          float* w = slot(sw_row_slot(r, n0), c);
          w[0] = x[c][(size_t)(H.beg_lo + r)].real();
          w[2] = x[c][(size_t)(H.beg_lo + r)].imag();
        }
    }
    int64_t di = 0;
    for (int k = 0; k < H.nph; ++k) {
      SwPhase PH;
      std::memcpy(&PH, gb + 32 + 8 * k, sizeof(PH));
      for (int b = 0; b < PH.nb; ++b, ++di) {
        SwDesc D;
        std::memcpy(&D, gb + H.off_desc + 40 * di, sizeof(D));
        const uint8_t* d = gb + D.off;
        if (PH.flags & SWP_TRI) { triangle(D, d, (PH.flags & SWP_UPPER) != 0, mask); continue; }
        const int32_t* out = reinterpret_cast<const int32_t*>(d);
        const int32_t* e0 = reinterpret_cast<const int32_t*>(d + D.off_e0);
        const int32_t* gl = reinterpret_cast<const int32_t*>(d + D.off_gl);
        const size_t raw = (size_t)(batch % kSwWarps) * (kSwGatherMax * NC * 2), pairs = raw + (wide ? 0 : kSwGather * NC * 2);
        if (!res) {
          for (int q = 0; q < D.ngl; ++q)
            for (int c = 0; c < NC; ++c) {
              const std::complex<float> v = gl[q] < 0 ? 0.f : global(gl[q], c);
              win[raw + (size_t)q * 2 * NC + 2 * c] = v.real();
              win[raw + (size_t)q * 2 * NC + 2 * c + 1] = v.imag();
            }
          for (int q = 0; 2 * q < (D.a0 > 0 ? D.a0 : D.ngl); ++q) {
            float e[2][NC][2];
            std::memcpy(e, &win[raw + (size_t)q * 4 * NC], sizeof(e));
            float* p = &win[pairs + (size_t)q * 4 * NC];
            for (int c = 0; c < NC; ++c)
              for (int u = 0; u < 2; ++u) { p[4 * c + u] = e[u][c][0]; p[4 * c + 2 + u] = e[u][c][1]; }
          }
          ++batch;
        }
        const int rpt = 32 >> D.glog;
        for (int r = 0; r < D.nrows; ++r) {
          const int t = r / rpt;
          Out o{out[r], {}};
          row(D, d, t, r % rpt, res ? 0 : 32 * (int64_t)e0[t], res ? D.elen : e0[t + 1] - e0[t], res, res ? 0 : pairs, mask, o.v);
          if (!res && D.a0)
            for (int c = 0; c < NC; ++c)
              for (int u = 0; u < 2; ++u) o.v[c][u] += win[raw + (size_t)(D.a0 + r) * 2 * NC + 2 * c + u];
          outs.push_back(o);
        }
      }
      if (!(PH.flags & SWP_END)) continue;
      for (const Out& o : outs)
        for (int c = 0; c < NC; ++c) {
          if (!res) { global(o.o, c) = {o.v[c][0], o.v[c][1]}; continue; }
          float* w = slot(o.o & ~kSwAcc, c);
          w[0] = ((o.o & kSwAcc) ? w[0] : 0.f) + o.v[c][0];
          w[2] = ((o.o & kSwAcc) ? w[2] : 0.f) + o.v[c][1];
        }
      outs.clear();
      batch = 0;
    }
  }
  void sweep() {
    size_t begin = 0;
    for (size_t g = 0; g < S.groups.size(); ++g) {
      SwGroupHdr H;
      std::memcpy(&H, S.image.data() + S.groups[g].img, sizeof(H));
      if (H.flags & SWG_BEGIN) begin = g;
      group(S.groups[g], false);
      if (!(H.flags & SWG_ENDRUN)) continue;
      const int rows = H.end_hi - H.end_lo;
      bool odd = false;
      for (int r = 0; r < rows; ++r)
        for (int c = 0; c < NC; ++c) {
          const float* w = slot(sw_row_slot(r, (int)ph.n0), c);
          odd = odd || !std::isfinite(w[0]) || !std::isfinite(w[2]);
        }
      if (odd)
        for (size_t q = begin; q <= g; ++q) group(S.groups[q], true);
      for (int r = 0; r < rows; ++r)
        for (int c = 0; c < NC; ++c) {
          const float* w = slot(sw_row_slot(r, (int)ph.n0), c);
          x[c][(size_t)(H.end_lo + r)] = {w[0], w[2]};
        }
    }
  }
};

bool finite(cplx v) { return std::isfinite(v.real()) && std::isfinite(v.imag()); }

int nan(const PackedHost& ph, int win_slots) {
  const int64_t n = ph.n, n0 = ph.n0;
  const std::vector<cplx> b = vec(n);
  for (int which = 0; which < 4; ++which) {
    SwSched S;
    build_sweep_sched(ph, which, 8, win_slots, S);
    if (!S.ok) { std::printf("FAIL: no schedule: %s\n", S.why); return 1; }
    const auto run = [&](int64_t at, float value) {
      Cta cta(ph, S);
      for (auto& v : cta.x) v.assign(b.begin(), b.end());
      if (at >= 0) cta.x[1][(size_t)at] = value;
      cta.sweep();
      return cta;
    };
    const Cta clean = run(-1, 0);
    const bool up = which == 1 || which == 2;   // rows from the last one on
    for (int64_t at : {(int64_t)5, n0 - 1, n0, n0 + 3, 5 * n0 + n0 / 2, n / 2 - 1, n / 2, n / 2 + n0 + 1, n - n0, n - 2}) {
      std::vector<cplx> ref = b;
      ref[(size_t)at] = NAN;
      HostFactor none;
      host_sweep(ph, none, which, ref.data());
      for (float value : {NAN, 3e38f}) {
        const Cta cta = run(at, value);
        int64_t first = 0, free = 0, pattern = 0;
        for (int64_t r = 0; r < n; ++r) {
          first += cta.x[0][(size_t)r] != clean.x[0][(size_t)r];
          if (up ? r > at : r < at) free += cta.x[1][(size_t)r] != clean.x[1][(size_t)r];
          if (std::isnan(value)) pattern += finite(cta.x[1][(size_t)r]) != finite(ref[(size_t)r]);
        }
        if (first || free || pattern) {
          std::printf("FAIL: sweep %d, %g at %lld: %lld rows of the other column, %lld independent rows, %lld rows\n", which,
                      (double)value, (long long)at, (long long)first, (long long)free, (long long)pattern);
          return 1;
        }
      }
    }
  }
  std::printf("OK\n");
  return 0;
}

// the kernel's walk over a triangle without masks: warp v, its rows' steps, column groups
int triangle() {
  for (int s = 2; s <= 256; s += 2)
    for (int v = 0; v < sw_tri_warps(s); ++v) {
      const SwTriWarp tw = sw_tri_warp(s, v);
      for (int n : {tw.n1, tw.n0})
        for (int g = 0; g < 4; ++g)
          for (int i = 0; i < sw_tri_take(s, g, n); ++i) {
            const int p = g + 4 * i, lower = 2 * p, upper = s - 2 - 2 * p;
            if (lower + 1 >= s || upper < 0) { std::printf("FAIL: order %d, pair %d\n", s, p); return 1; }
          }
      // and no pair of a row is left out
      for (int j = 4 * v; j < 4 * v + 4; ++j)
        for (bool hi : {true, false})
          if (sw_tri_live(s, j, hi))
            for (int p = 0; p < sw_tri_len(hi ? s - 1 - j : j); ++p)
              if (p / 4 >= sw_tri_take(s, p % 4, hi ? tw.n1 : tw.n0)) { std::printf("FAIL: order %d without pair %d\n", s, p); return 1; }
    }
  std::printf("OK\n");
  return 0;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc == 2 && !std::strcmp(argv[1], "triangle")) return triangle();
  if (argc != 6) return 2;
  const std::string what = argv[1];
  const PackedHost ph = pack(argv[2], std::atoll(argv[3]), std::atoll(argv[4]), std::atof(argv[5]));
  if (what == "tiles3") return tiles3(ph);
  if (what == "region") return region(ph);
  if (what == "wide") return wide(ph);
  if (what == "nan") return nan(ph, kSwWinSlots);
  if (what == "nan_small") return nan(ph, 512);
  return 2;
}
