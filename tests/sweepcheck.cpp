// Host checks of the column-partitioned sweep schedules over coarse and fine factors (test
// helper; built by tests/test_sweep_shapes.py with g++ against the library's host code).
//
//   sweepcheck CHECK arc|strip n leaf eps
//
// CHECK = tiles3: prints how many resident tiles have three entry pairs whose third pair is
// not zero (all four sweeps), and fails where a schedule with complex-FP32 coefficients,
// executed with the kernel's input rule, is off the packed program's sweep by more than 1e-5.
//
//   sweepcheck triangle
//
// fails where a step of a triangle product of even order (2 .. 256, lower and upper) reads a
// column that is not the triangle's.
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
  const double arc[3] = {len / M_PI, 0.0, M_PI}, strip[4] = {0.0, 0.0, len, 0.0};
  const bool a = !std::strcmp(curve, "arc");
  HostFactor hf;
  PackedHost ph;
  if (build_geometry(a ? HB_ARC : HB_STRIP, a ? arc : strip, a ? 3 : 4, n, g) ||
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
    std::vector<cplx> x = vec(ph.n), r = x;
    host_sweep_sched(ph, S, x.data());
    HostFactor none;
    host_sweep(ph, none, which, r.data());
    double e = 0, d = 0;
    for (int64_t i = 0; i < ph.n; ++i) { e += std::norm(x[i] - r[i]); d += std::norm(r[i]); }
    if (!(std::sqrt(e / d) <= 1e-5)) { std::printf("FAIL: sweep %d off by %.3g\n", which, std::sqrt(e / d)); return 1; }
  }
  std::printf("tiles %d\n", count);
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
  return 2;
}
