// Column-partitioned sweep kernel (sm_103a): x = L~^{-1} b, U~^{-1} b and
// their adjoints (Algs. 3, 4) for many right-hand sides, in place.
//
// The sweep is a long chain of small dependent phases (one sweep-leaf solve,
// then the butterfly that carries its result to the next subtree, ...).  Run
// grid-wide, every link costs a grid barrier; run by one CTA, every link is a
// shared-memory round trip.  So here each CTA runs the whole sweep for its own
// one or two right-hand sides and never waits on another CTA:
//   * a producer warp streams the schedule's group images (host-built, see
//     hb_swsched.cpp: a header, batch descriptors, the batches' data) into a
//     shared-memory ring with one cp.async.bulk each.  Every group's place in the
//     ring, and the groups that must be consumed before it may be copied there, are
//     fixed by the host, so 32 lanes issue 32 groups without any bookkeeping (a lane
//     that allocated ring space and looked at every release took about a thousand
//     cycles per group, which bounded the kernel);
//   * resident runs (subtrees whose rows and live butterfly state fit the 96 KB
//     window) start by loading their rows into shared memory, and zeros into the
//     rest of what they use, and end by writing the rows back; inside them every
//     phase reads and writes the window;
//   * global phases (stages of the large butterflies) read and write the
//     vector rows and a CTA-private butterfly state in global memory; every batch
//     belongs to one warp, which gathers its inputs (cp.async, the next batch's in
//     flight while one is computed) and never touches the other warps' groups;
//   * an op of a butterfly phase is a dense block over neighbouring inputs.  The
//     window holds entry pairs as (re, re, im, im), so 16 bytes of coefficients and 16
//     of inputs give two complex multiply-adds in four packed FP32 instructions, with
//     no index per entry;
//   * consecutive stages of a butterfly are multiplied out on the host where that is
//     cheaper than one more dependent phase (the phases of the semicircle's sweep at
//     N = 65,536: 3,058 without, 1,699 with);
//   * the resident phases alternate between two sets of eight warps: while one set
//     computes, the other has its next coefficients in registers and waits only for
//     the inputs; large phases and the sweep leaves are taken by all sixteen;
//   * tiles and triangles also multiply zeros with slots that are not theirs, so that no
//     lane needs a mask.  A run whose rows come out non-finite is repeated with every zero
//     coefficient masked: an Inf or NaN reaches only the rows that depend on it.  (In a
//     global phase it reaches what its butterfly writes, which is the same rows; a value that
//     first overflows there may reach more of them.)
// What bounds it is the dependent chain of one CTA: a phase costs 1,000 to 2,000
// cycles (descriptor and coefficient fetch, the inputs' round trip, shuffles, a
// barrier), far above its share of the 9 B/clk of staged data.
// Every wait is bounded; a warp whose wait gives up stops computing but still meets
// the barriers up to the end of its unit (a run, a global phase), where all compute
// warps learn of it and stop; the factor's error flag is raised (reported by
// hb_status / the solvers) and the CTA returns after a second bounded wait for its
// copies still in flight.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "hb_device.h"
#include "hb_sweep_launch.h"

namespace hb {

namespace {

constexpr int kSwThreads = (kSwWarps + 1) * 32;
// at most five warps per scheduler: every thread may hold 96 registers
static_assert((kSwWarps + 1 + 3) / 4 * 96 * 32 <= 16384, "registers per scheduler");
constexpr int kSwSmem = kSwRingBytes + kSwWinBytes;   // ring | window
static_assert(kSwSmem <= 225 * 1024, "dynamic shared memory of the column-partitioned sweep");

__device__ __forceinline__ unsigned su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(uint64_t* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_inval(uint64_t* b) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void mb_arrive_tx(uint64_t* b, unsigned bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(su32(b)),
               "r"(bytes) : "memory");
}
__device__ __forceinline__ void mb_arrive(uint64_t* b, int count) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mb_try_wait(uint64_t* b, unsigned parity) {
  unsigned ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
  return ok != 0;
}
// non-blocking test: the consumers count polls, so that a wait limit of one poll
// gives up at once on a batch still in flight
__device__ __forceinline__ bool mb_test_wait(uint64_t* b, unsigned parity) {
  unsigned ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
  return ok != 0;
}
// asynchronous global -> shared copy of `bytes` (8 or 16), the first `src_bytes` of
// them from src and the rest zero
__device__ __forceinline__ void cp_async(unsigned dst, const void* src, int bytes, int src_bytes) {
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(su32(dst)), "l"(src), "r"(bytes), "r"(su32(b)) : "memory");
}
// named barriers of the compute warps: 1 with an OR of a flag, 2 all warps, 3 / 4 the
// hand-over from one set of warps to the other (the writers arrive, the readers wait)
__device__ __forceinline__ bool all_red_or(bool v) {
  unsigned r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
               : "=r"(r) : "r"((unsigned)v), "n"(kSwWarps * 32) : "memory");
  return r != 0;
}
__device__ __forceinline__ void all_sync() { asm volatile("bar.sync 2, %0;\n" ::"n"(kSwWarps * 32) : "memory"); }
__device__ __forceinline__ void hand_sync(unsigned id) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "n"(kSwWarps * 32) : "memory");
}
__device__ __forceinline__ void hand_arrive(unsigned id) {
  asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "n"(kSwWarps * 32) : "memory");
}

struct SwArgs {
  const SwGroup* groups;
  int64_t ngroup;
  const uint8_t* image;
  float2* x;           // vectors, layout [row][R]
  int64_t R, n;
  int n0;              // leaf rows
  int64_t col0;        // first column of this launch
  float2* st;          // CTA-private butterfly state: [CTA][state_len][NC]
  int64_t state_len;
  int* err_out;        // the factor's sticky error flag
  long long spin_limit;
};

// ---- shared memory by 32-bit address (every operand of the hot loops lives there)
typedef unsigned long long f2x;   // two packed FP32 values
struct f2x2 {
  f2x a, b;
};
__device__ __forceinline__ f2x2 lds_2(unsigned a) {   // 16 bytes: (re, re) and (im, im) of an entry pair
  f2x2 v;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];\n" : "=l"(v.a), "=l"(v.b) : "r"(a));
  return v;
}
// the same if `on`, else the given value
__device__ __forceinline__ void lds_2_if(unsigned a, bool on, f2x2& v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %3, 0;\n @p ld.shared.v2.b64 {%0, %1}, [%2];\n}\n"
               : "+l"(v.a), "+l"(v.b) : "r"(a), "r"((int)on));
}
__device__ __forceinline__ float4 lds_f4(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ float2 lds_f2(unsigned a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ float lds_f(unsigned a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ int2 lds_i2(unsigned a) {
  int2 v;
  asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds_i(unsigned a) {
  int v;
  asm volatile("ld.shared.s32 %0, [%1];\n" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds_u16(unsigned a) {
  int v;
  asm volatile("ld.shared.u16 %0, [%1];\n" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void lds_i_if(unsigned a, bool on, int& v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %2, 0;\n @p ld.shared.s32 %0, [%1];\n}\n"
               : "+r"(v) : "r"(a), "r"((int)on));
}
__device__ __forceinline__ void sts_f(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void sts_f4(unsigned a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
// image data, staged (shared address) or where it stands in global memory
__device__ __forceinline__ f2x2 img_2(unsigned a) { return lds_2(a); }
__device__ __forceinline__ f2x2 img_2(const uint8_t* p) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
  return f2x2{v.x, v.y};
}
__device__ __forceinline__ int img_i(unsigned a) { return lds_i(a); }
__device__ __forceinline__ int img_i(const uint8_t* p) { return __ldg(reinterpret_cast<const int*>(p)); }
__device__ __forceinline__ f2x ffma2(f2x a, f2x b, f2x c) {   // two FP32 multiply-adds
  f2x d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2x fmul2(f2x a, f2x b) {
  f2x d;
  asm("mul.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float lo(f2x v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi(f2x v) { return __uint_as_float((unsigned)(v >> 32)); }

// Window and slice entries stand in pairs: slots 2i, 2i + 1 of a column as (re, re, im,
// im), the columns of a pair side by side.  So 16 bytes of coefficients and 16 of inputs
// give two complex multiply-adds in four packed instructions.
template <int NC>
__device__ __forceinline__ unsigned slot_addr(unsigned base, int s) { return base + (s >> 1) * (16 * NC) + (s & 1) * 4; }
// sums of m v over entry pairs: re re, im im, re im, im re of the even and the odd entries
struct Acc {
  f2x rr = 0, ii = 0, ri = 0, ir = 0;
  __device__ __forceinline__ void set(const f2x2& m, const f2x2& v) {
    rr = fmul2(m.a, v.a);
    ii = fmul2(m.b, v.b);
    ri = fmul2(m.a, v.b);
    ir = fmul2(m.b, v.a);
  }
  __device__ __forceinline__ void add(const f2x2& m, const f2x2& v) {
    rr = ffma2(m.a, v.a, rr);
    ii = ffma2(m.b, v.b, ii);
    ri = ffma2(m.a, v.b, ri);
    ir = ffma2(m.b, v.a, ir);
  }
  __device__ __forceinline__ float2 sum() const {
    return make_float2((lo(rr) + hi(rr)) - (lo(ii) + hi(ii)), (lo(ri) + hi(ri)) + (lo(ir) + hi(ir)));
  }
};

// inputs v as the coefficients m take them: nothing where a coefficient is zero (0 times a
// foreign Inf or NaN would be NaN)
__device__ __forceinline__ f2x2 masked(const f2x2& m, f2x2 v) {
  const f2x k = (lo(m.a) == 0.f && lo(m.b) == 0.f ? 0ull : 0xffffffffull) |
                (hi(m.a) == 0.f && hi(m.b) == 0.f ? 0ull : 0xffffffffull << 32);
  v.a &= k;
  v.b &= k;
  return v;
}

// address of a global slot: a vector row (this CTA's columns of x) or a
// CTA-private state entry
__device__ __forceinline__ float2* gaddr(const SwArgs& a, int32_t s, float2* xb, float2* stp, int nc) {
  return s < a.n ? xb + (int64_t)s * a.R : stp + (int64_t)(s - a.n) * nc;
}

// NC columns of global slot s into shared address dst (8 * NC bytes) asynchronously; the
// columns beyond this CTA's ncol read as zero.  x rows are 16-byte aligned when the
// row stride and the CTA's first column are even (vec16).
template <int NC>
__device__ __forceinline__ void slot_async(const SwArgs& a, int32_t s, unsigned dst, float2* xb, float2* stp, int ncol,
                                           bool vec16) {
  if (s < 0) {
    cp_async(dst, stp, 8 * NC, 0);   // a zero
  } else if (s < a.n) {
    const float2* src = xb + (int64_t)s * a.R;
    if (NC == 2 && vec16) {
      cp_async(dst, src, 16, 8 * ncol);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) cp_async(dst + 8 * c, c < ncol ? src + c : src, 8, c < ncol ? 8 : 0);
    }
  } else {
    const float2* src = stp + (int64_t)(s - a.n) * NC;
    cp_async(dst, src, 8 * NC, 8 * NC);
  }
}

// ---- one resident tile, one warp.  The coefficients of the lane's first four entry pairs
// are held in registers, so that they can be fetched before the inputs exist; a longer
// tile (a multiple of four entries) reads the rest as it goes.  Fewer than four pairs
// (a phase of very few inputs): the absent ones have coefficient 0 and the lane's first inputs.
constexpr int kPairBytes = 32 * 16;   // one entry pair of all lanes
template <int NC>
struct Tile {
  f2x2 cf[kSwTilePairs];
  unsigned va;              // shared address of the lane's first input
  unsigned coef;            // the lane's entries (shared memory)
  int np;                   // entry pairs per lane
  int glog;
  unsigned dst;             // shared address that this lane stores (a column of) its row's sum to; 0: none
  bool add;                 // adding to the old value
};
// this lane's part of its row's sums
template <int NC>
__device__ __forceinline__ void tile_mac(const Tile<NC>& t, float2 (&s)[NC]) {
  Acc acc[NC];
  f2x2 v[kSwTilePairs][NC];
#pragma unroll
  for (int i = 0; i < kSwTilePairs; ++i)
#pragma unroll
    for (int c = 0; c < NC; ++c) v[i][c] = lds_2(t.va + sw_tile_pair(i, t.np) * (16 * NC) + 16 * c);
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c].set(t.cf[0], v[0][c]);
#pragma unroll
  for (int i = 1; i < kSwTilePairs; ++i)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c].add(t.cf[i], v[i][c]);
  if (t.np > kSwTilePairs) {
    unsigned cp = t.coef + kSwTilePairs * kPairBytes, vp = t.va + kSwTilePairs * (16 * NC);
    int i = kSwTilePairs;
#pragma unroll 1
    for (; i + 1 < t.np; i += 2, cp += 2 * kPairBytes, vp += 2 * (16 * NC)) {
      f2x2 m[2], w[2][NC];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        m[u] = lds_2(cp + u * kPairBytes);
#pragma unroll
        for (int c = 0; c < NC; ++c) w[u][c] = lds_2(vp + u * (16 * NC) + 16 * c);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c].add(m[u], w[u][c]);
    }
    if (i < t.np) {
      const f2x2 m = lds_2(cp);
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c].add(m, lds_2(vp + 16 * c));
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) s[c] = acc[c].sum();
}
// Sums over a row's 2^glog lanes.  With two columns and more than one lane the first round
// also parts the columns: the row's first lane keeps column 0, its second column 1 (both in
// s[0]); with one lane that lane keeps both.
template <int NC>
__device__ __forceinline__ void tile_reduce(float2 (&s)[NC], int glog, int lane) {
  if (glog == 0) return;
  if constexpr (NC == 2) {
    const bool odd = lane & 1;
    const float2 keep = odd ? s[1] : s[0], send = odd ? s[0] : s[1];
    s[0].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 1);
    s[0].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 1);
  } else {
    s[0].x += __shfl_xor_sync(0xffffffffu, s[0].x, 1);
    s[0].y += __shfl_xor_sync(0xffffffffu, s[0].y, 1);
  }
#pragma unroll
  for (int g = 1; g < 5; ++g) {
    if (glog == g) return;
    s[0].x += __shfl_xor_sync(0xffffffffu, s[0].x, 1 << g);
    s[0].y += __shfl_xor_sync(0xffffffffu, s[0].y, 1 << g);
  }
}
// whether a lane stores: the row's first NC lanes (its only lane)
template <int NC>
__device__ __forceinline__ bool tile_writer(int rows, int glog, int lane) {
  return (lane >> glog) < rows && (lane & ((1 << glog) - 1)) < NC;
}
// a resident tile from the first eight bytes of its descriptor (off | elen, glog, trows)
template <int NC>
__device__ __forceinline__ void tile_open(Tile<NC>& t, unsigned gimg, int2 w, unsigned win, int lane) {
  const unsigned b = gimg + w.x;
  const int in = lds_u16(b + kSwTileIn + 2 * lane);
  t.np = (w.y & 0xffff) >> 1;
  t.glog = (w.y >> 16) & 0xff;
  const bool wr = tile_writer<NC>(w.y >> 24, t.glog, lane);
  int o = 0;
  lds_i_if(b + 4 * (lane >> t.glog), wr, o);
  t.add = o < 0;
  t.dst = wr ? slot_addr<NC>(win, o & ~kSwAcc) + (NC == 2 && t.glog > 0 ? 16 * (lane & 1) : 0) : 0;
  t.coef = b + kSwTileCoef + 16 * lane;
  t.va = win + in * (8 * NC);
  if (t.np >= kSwTilePairs) {
#pragma unroll
    for (int i = 0; i < kSwTilePairs; ++i) t.cf[i] = lds_2(t.coef + i * kPairBytes);
  } else {
#pragma unroll
    for (int i = 0; i < kSwTilePairs; ++i) {
      t.cf[i] = f2x2{0, 0};
      lds_2_if(t.coef + i * kPairBytes, i < t.np, t.cf[i]);
    }
  }
}
// A resident phase's tiles b, b + stride, ... (< nb) of one warp, the first already in `t`.
template <int NC>
__device__ __forceinline__ void run_phase(Tile<NC>& t, unsigned gimg, unsigned desc, int b, int nb, int stride, unsigned win,
                                          int lane) {
  for (;; b += stride) {
    const bool more = b + stride < nb;
    int2 w = make_int2(0, 0);
    if (more) w = lds_i2(desc + 40 * (b + stride));
    const int glog = t.glog;
    const unsigned dst = t.dst;
    const bool both = NC == 2 && glog == 0;   // the lane stores both columns
    float2 s[NC], old[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) old[c] = make_float2(0.f, 0.f);
    if (t.add) {
      old[0] = make_float2(lds_f(dst), lds_f(dst + 8));
      if (both) old[NC - 1] = make_float2(lds_f(dst + 16), lds_f(dst + 24));
    }
    tile_mac<NC>(t, s);
    if (more) tile_open<NC>(t, gimg, w, win, lane);
    tile_reduce<NC>(s, glog, lane);
    if (dst) {
      sts_f(dst, old[0].x + s[0].x);
      sts_f(dst + 8, old[0].y + s[0].y);
      if (both) {
        sts_f(dst + 16, old[NC - 1].x + s[NC - 1].x);
        sts_f(dst + 24, old[NC - 1].y + s[NC - 1].y);
      }
    }
    if (!more) break;
  }
}

// One global batch, one warp: its tiles in turn, inputs from the slice's pairs, old values
// from its entries as gathered (raw), outputs to global slots.  Few lanes per row, so that
// the work is mostly the pair loop: one load of coefficients and one of inputs per column
// for four packed multiply-adds, four pairs in flight.
template <int NC>
__device__ __forceinline__ void run_batch(const SwArgs& a, unsigned desc, unsigned gimg, unsigned pairs, unsigned raw,
                                          float2* xb, float2* stp, int ncol, bool vec16, int lane) {
  const int2 w0 = lds_i2(desc), w24 = lds_i2(desc + 24);
  const unsigned bb = gimg + w0.x, e0 = bb + w24.x, in = bb + lds_i(desc + 32) + 2 * lane;
  const int nrows = lds_i(desc + 8), old0 = lds_i(desc + 20), glog = (w0.y >> 16) & 0xff, rpt = 32 >> glog;
  const int nt = (nrows + rpt - 1) >> (5 - glog);
  const bool one = NC == 2 && glog == 0;               // a lane stores both columns
  const int c0 = NC == 2 && glog > 0 ? lane & 1 : 0;   // else this one
  unsigned cp = bb + w24.y + 16 * lane;                // the lane's next coefficients
  int ea = 0;
  for (int k = 0; k < nt; ++k) {
    const int eb = lds_i(e0 + 4 * (k + 1));
    unsigned vp = pairs + lds_u16(in + 64 * k) * (8 * NC);
    const bool wr = tile_writer<NC>(nrows - k * rpt, glog, lane);
    int32_t o = 0;
    lds_i_if(bb + 4 * (k * rpt + (lane >> glog)), wr, o);
    Acc acc[NC];
    int i = (eb - ea) >> 1;
    ea = eb;
#pragma unroll 1
    for (; i >= 4; i -= 4, cp += 4 * kPairBytes, vp += 4 * (16 * NC)) {
      f2x2 m[4], w[4][NC];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        m[u] = lds_2(cp + u * kPairBytes);
#pragma unroll
        for (int c = 0; c < NC; ++c) w[u][c] = lds_2(vp + u * (16 * NC) + 16 * c);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c].add(m[u], w[u][c]);
    }
#pragma unroll 1
    for (; i > 0; --i, cp += kPairBytes, vp += 16 * NC) {
      const f2x2 m = lds_2(cp);
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c].add(m, lds_2(vp + 16 * c));
    }
    float2 s[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) s[c] = acc[c].sum();
    tile_reduce<NC>(s, glog, lane);
    if (wr) {
      float2* d = gaddr(a, o, xb, stp, NC);
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if ((c == 0 || one) && old0 > 0) {
          const float2 w = lds_f2(raw + (old0 + k * rpt + (lane >> glog)) * (8 * NC) + 8 * (c0 + c));
          s[c] = make_float2(w.x + s[c].x, w.y + s[c].y);
        }
      if (one && (o >= a.n || (vec16 && ncol == 2))) {
        *reinterpret_cast<float4*>(d) = make_float4(s[0].x, s[0].y, s[NC - 1].x, s[NC - 1].y);
      } else {
#pragma unroll
        for (int c = 0; c < NC; ++c)
          if ((c == 0 || one) && (c0 + c < ncol || o >= a.n)) d[c0 + c] = s[c];
      }
    }
  }
}

// Sweep-leaf phase: the window rows from slot a0 on replaced by the triangle times them,
// all compute warps.  A warp's work is four row pairs (stored rows j and s-1-j): lanes =
// row pair x four column groups x column (two columns) or parity of the step (one).  So
// every lane has the same 17 steps at order 128, a step's coefficients are consecutive,
// its inputs four neighbouring column pairs that all row pairs share, and a row's sum
// needs two shuffle rounds and no other warp; one barrier separates the reads of the rows
// from their replacement.  FAST, for an even leaf size (the window's slots pair up like the
// columns): without masks; else, for any, inputs beyond a row's diagonal are masked (0 times a
// foreign row's Inf would be NaN).
template <int NC>
__device__ __forceinline__ f2x2 tri_input(unsigned win, int a0, int s, bool up, int p, int c, int n0) {
  // columns c0, c0 + 1 by themselves (a column outside the triangle is masked by the caller)
  const int c0 = up ? s - 2 - 2 * p : 2 * p;
  unsigned q[4] = {0, 0, 0, 0};
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (c0 + u >= 0 && c0 + u < s) {
      const unsigned d = slot_addr<NC>(win, a0 + sw_row_slot(c0 + u, n0)) + 16 * c;
      q[u] = __float_as_uint(lds_f(d));
      q[2 + u] = __float_as_uint(lds_f(d + 8));
    }
  f2x2 v;
  v.a = q[0] | (f2x)q[1] << 32;
  v.b = q[2] | (f2x)q[3] << 32;
  return v;
}
// row r's sum over steps [0, n) (r < 0: no such row); coef: the lane's first coefficient
template <int NC, class P>
__device__ __forceinline__ float2 tri_row(int n, P coef, int r, unsigned win, int a0, int s, bool up, int n0, int lane) {
  const int g = (lane >> 1) & 3, c = NC == 2 ? lane & 1 : 0;
  // with one column the lane takes every second step
  const int i0 = NC == 2 ? 0 : lane & 1, di = NC == 2 ? 1 : 2;
  Acc acc;
#pragma unroll 1
  for (int i = i0; i < n; i += di) {
    const int p = g + 4 * i;
    const bool in = 2 * p <= r, two = 2 * p < r;   // the pair's first / second stored column within the row
    f2x2 v{0, 0};
    if (in) v = tri_input<NC>(win, a0, s, up, p, c, n0);
    const f2x mask = two ? ~0ull : up ? 0xffffffffull << 32 : 0xffffffffull;
    v.a &= mask;
    v.b &= mask;
    acc.add(img_2(coef + i * 256), v);
  }
  return acc.sum();
}
// The same without masks (the coefficients beyond the diagonal are zero; n: the steps within
// the triangle), two steps in flight.  vp: the lane's first input, dv: bytes
// per step.
template <int NC>
__device__ __forceinline__ float2 tri_row_fast(int n, unsigned cp, unsigned vp, int dv, int lane) {
  if (NC == 1) {
    // every second step per lane
    cp += (lane & 1) * 256;
    vp += (lane & 1) * dv;
    dv *= 2;
    n = (n + 1 - (lane & 1)) >> 1;
  }
  constexpr int cs = NC == 1 ? 512 : 256;
  Acc acc;
  int i = 0;
#pragma unroll 1
  for (; i + 1 < n; i += 2, cp += 2 * cs, vp += 2 * dv) {
    const f2x2 m0 = lds_2(cp), v0 = lds_2(vp), m1 = lds_2(cp + cs), v1 = lds_2(vp + dv);
    acc.add(m0, v0);
    acc.add(m1, v1);
  }
  if (i < n) acc.add(lds_2(cp), lds_2(vp));
  return acc.sum();
}
template <int NC, bool FAST, class P>
__device__ __forceinline__ void run_tri(int s, int a0, bool up, P T, unsigned win, int n0, int warp, int lane) {
  const int dv = (up ? -64 : 64) * NC, g = (lane >> 1) & 3;
  const unsigned vp = slot_addr<NC>(win, a0 + (up ? s - 2 : 0)) + (NC == 2 ? 16 * (lane & 1) : 0) + g * (dv / 4);
  const int nv = ((s + 1) / 2 + 3) / 4;
  float val[2] = {0.f, 0.f};
  unsigned dst[2] = {0, 0};   // 0: nothing to store
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int v = warp + kSwWarps * h;
    if (v < nv) {
      const int tw = img_i(T + 4 * v), n1 = (tw >> 8) & 0xff, nn0 = tw & 0xff;
      const P coef = T + (kSwTriTab + (tw >> 16) * 256 + (lane >> 1) * 16);
      const int j = 4 * v + (lane >> 3);
      const int r1 = 2 * j <= s - 1 ? s - 1 - j : -1, r0 = 2 * j < s - 1 ? j : -1;
      float2 s1, s0;
      if constexpr (FAST) {
        s1 = tri_row_fast<NC>(sw_tri_take(s, g, n1), coef, vp, dv, lane);
        s0 = tri_row_fast<NC>(sw_tri_take(s, g, nn0), coef + n1 * 256, vp, dv, lane);
      } else {
        s1 = tri_row<NC>(n1, coef, r1, win, a0, s, up, n0, lane);
        s0 = tri_row<NC>(nn0, coef + n1 * 256, r0, win, a0, s, up, n0, lane);
      }
      // parting the sums over the lanes: a lane pair keeps one row, then one component
      constexpr int d1 = NC == 2 ? 2 : 1, d2 = 2 * d1;
      const bool b1 = lane & d1, b2 = lane & d2;
      float2 keep = b1 ? s0 : s1;
      const float2 send = b1 ? s1 : s0;
      keep.x += __shfl_xor_sync(0xffffffffu, send.x, d1);
      keep.y += __shfl_xor_sync(0xffffffffu, send.y, d1);
      float w = b2 ? keep.y : keep.x;
      w += __shfl_xor_sync(0xffffffffu, b2 ? keep.x : keep.y, d2);
      if (NC == 1) w += __shfl_xor_sync(0xffffffffu, w, 4);
      const int r = b1 ? r0 : r1;
      val[h] = w;
      if (r >= 0 && (NC == 2 || !(lane & 4))) {
        const int row = up ? s - 1 - r : r;
        dst[h] = slot_addr<NC>(win, a0 + (FAST ? row : sw_row_slot(row, n0))) + (NC == 2 ? 16 * (lane & 1) : 0) + (b2 ? 8 : 0);
      }
    }
  }
  all_sync();
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if (dst[h]) sts_f(dst[h], val[h]);
}

// Rows [lo, hi) of the CTA's columns (xb, row stride R) into the window, all compute warps, and
// zeros into its slots without a row, up to `slots` (they are read as inputs of coefficient 0).
template <int NC>
__device__ __forceinline__ void load_rows(const float2* xb, int64_t R, int lo, int hi, int slots, int n0, int ncol,
                                          unsigned win, int t) {
  const int nrow = hi - lo, leaves = (n0 & 1) ? nrow / n0 : 0;
  const unsigned z1 = win + slots * (8 * NC);
  for (unsigned d = win + (nrow + leaves) * (8 * NC) + 16 * t; d < z1; d += 16 * kSwWarps * 32) sts_f4(d, 0.f, 0.f, 0.f, 0.f);
  for (int l = t; l < leaves; l += kSwWarps * 32) {
    const unsigned d = slot_addr<NC>(win, l * (n0 + 1) + n0);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      sts_f(d + 16 * c, 0.f);
      sts_f(d + 16 * c + 8, 0.f);
    }
  }
#pragma unroll 4
  for (int r = t; r < nrow; r += kSwWarps * 32) {
    const float2* src = xb + (int64_t)(lo + r) * R;
    const unsigned d = slot_addr<NC>(win, sw_row_slot(r, n0));
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const float2 v = c < ncol ? __ldcg(src + c) : make_float2(0.f, 0.f);
      sts_f(d + 16 * c, v.x);
      sts_f(d + 16 * c + 8, v.y);
    }
  }
}

// A resident run once more from its rows, with every zero coefficient masked: for a run whose
// rows came out non-finite, since a foreign Inf or NaN times zero (a neighbour's slot, a row
// beyond the diagonal) may have made them so.  All compute warps; the groups are read where they
// stand in global memory (the ring has moved on), the sums have the order of the run proper.
template <int NC>
__device__ __forceinline__ void redo_run(const uint8_t* image, const SwGroup* groups, int ngroup, const float2* xb, int64_t R,
                                         int n0, int ncol, unsigned win, int warp, int lane) {
  for (int g = 0; g < ngroup; ++g) {
    const uint8_t* img = image + groups[g].img;
    const SwGroupHdr H = *reinterpret_cast<const SwGroupHdr*>(img);
    if (g == 0) {
      load_rows<NC>(xb, R, H.beg_lo, H.beg_hi, H.flags >> kSwGroupSlots, n0, ncol, win, 32 * warp + lane);
      all_sync();
    }
    const SwDesc* desc = reinterpret_cast<const SwDesc*>(img + H.off_desc);
    for (int k = 0; k < H.nph; ++k) {
      const SwPhase PH = reinterpret_cast<const SwPhase*>(img + 32)[k];
      if (PH.flags & SWP_TRI) {
        const uint8_t* T = img + desc->off;
        const bool up = (PH.flags & SWP_UPPER) != 0;
        run_tri<NC, false>(desc->nrows, desc->a0, up, T, win, n0, warp, lane);   // (any leaf size)
      } else {
        for (int b = warp; b < PH.nb; b += kSwWarps) {
          const SwDesc& D = desc[b];
          const uint8_t* data = img + D.off;
          const int glog = D.glog, in = reinterpret_cast<const int16_t*>(data + kSwTileIn)[lane];
          unsigned vp = win + in * (8 * NC);
          const uint8_t* cp = data + kSwTileCoef + 16 * lane;
          Acc acc[NC];
          for (int i = 0; i < D.elen / 2; ++i, cp += kPairBytes, vp += 16 * NC) {
            const f2x2 m = img_2(cp);
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c].add(m, masked(m, lds_2(vp + 16 * c)));
          }
          float2 s[NC];
#pragma unroll
          for (int c = 0; c < NC; ++c) s[c] = acc[c].sum();
          tile_reduce<NC>(s, glog, lane);
          if (tile_writer<NC>(D.trows, glog, lane)) {
            const int o = reinterpret_cast<const int32_t*>(data)[lane >> glog];
            const unsigned dst = slot_addr<NC>(win, o & ~kSwAcc) + (NC == 2 && glog > 0 ? 16 * (lane & 1) : 0);
#pragma unroll
            for (int c = 0; c < (NC == 2 && glog == 0 ? NC : 1); ++c) {
              const unsigned d = dst + 16 * c;
              const float2 old = o < 0 ? make_float2(lds_f(d), lds_f(d + 8)) : make_float2(0.f, 0.f);
              sts_f(d, old.x + s[c].x);
              sts_f(d + 8, old.y + s[c].y);
            }
          }
        }
      }
      desc += PH.nb;
      if (PH.flags & SWP_END) all_sync();
    }
  }
}

// Out of line for one column (inlined, the spiral's solve takes 12.36 ms, not 12.07), inlined for
// two (called, the spills around the call cost 1.1 ms of the 35.7 ms of 256 columns).
__device__ __noinline__ void redo_run_1(const uint8_t* image, const SwGroup* groups, int ngroup, const float2* xb, int64_t R,
                                        int n0, int ncol, unsigned win, int warp, int lane) {
  redo_run<1>(image, groups, ngroup, xb, R, n0, ncol, win, warp, lane);
}

template <int NC>
// The bound of 640 threads (above the 544 launched) caps the registers at 96 a thread, so
// that the scheduler that holds five of the 17 warps stays within its 16K registers.
__global__ void __launch_bounds__(640, 1) k_sweep_cols(SwArgs a) {
  extern __shared__ __align__(128) char smem[];
  __shared__ int s_off[kSwFlight];                 // ring offset of each group in flight
  __shared__ __align__(8) uint64_t s_mbar[kSwFlight];    // group in the slot has arrived
  __shared__ __align__(8) uint64_t s_free[kSwFlight];    // every compute warp is done with it
  __shared__ int s_abort, s_issued;
  __shared__ int s_redo;   // the compute warps are busy with a run's second pass
  const unsigned ring_a = su32(smem), win_a = ring_a + kSwRingBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t lb = a.col0 + (int64_t)blockIdx.x * NC;
  const int ncol = (int)((a.R - lb) < NC ? (a.R - lb) : NC);
  float2* xb = a.x + lb;
  float2* stp = a.st + (int64_t)blockIdx.x * a.state_len * NC;
  if (threadIdx.x == 0) {
    for (int k = 0; k < kSwFlight; ++k) {
      mb_init(&s_mbar[k], 1);
      mb_init(&s_free[k], kSwWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_abort = 0;
    s_issued = 0;
    s_redo = 0;
  }
  __syncthreads();
  if (warp == kSwWarps) {
    // ---- producer: every group of the schedule into its place in the ring, one lane each,
    // 32 groups at a time; a lane may copy once the groups before `need` (its record) are
    // consumed.  [0, done) are: advanced by looking at 32 slots at once.
    int done = 0, g0 = 0;
    const int ngroup = (int)a.ngroup;
    bool stop = false;
    for (; g0 < ngroup && !stop; g0 += 32) {
      const int g = g0 + lane;
      SwGroup G{0, 0, 0, 0, 0};
      bool todo = g < ngroup;
      if (todo) G = a.groups[g];
      long long spins = 0;
      for (;;) {
        const bool go = todo && G.need <= done;
        if (go) {
          const int slot = g % kSwFlight;
          s_off[slot] = G.off;   // published with the arrive (release) below
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
          mb_arrive_tx(&s_mbar[slot], (unsigned)G.bytes);
          bulk_copy(smem + G.off, a.image + G.img, (unsigned)G.bytes, &s_mbar[slot]);
          todo = false;
        }
        const unsigned left = __ballot_sync(0xffffffffu, todo);
        if (left == 0) break;
        // groups issued so far: those before the first one left
        const int issued = g0 + __ffs(left) - 1;
        const int q = done + lane;
        const bool free = q < issued && mb_test_wait(&s_free[q % kSwFlight], (unsigned)q / kSwFlight & 1u);
        const unsigned busy = __ballot_sync(0xffffffffu, !free);
        const int adv = busy ? __ffs(busy) - 1 : 32;
        done += adv;
        if (adv == 0) {
          if (!*(volatile int*)&s_redo) ++spins;   // (a second pass takes its time, but ends)
          if (__any_sync(0xffffffffu, spins > a.spin_limit || *(volatile int*)&s_abort)) {
            if (lane == 0) {
              atomicExch(&s_abort, 1);
              s_issued = issued;
            }
            stop = true;
            break;
          }
          __nanosleep(20);
        }
      }
    }
    if (!stop && lane == 0) s_issued = ngroup;
    __syncwarp();
  } else {
    const int t = threadIdx.x;
    // gather area of global batches: entries as gathered, then the same in pairs (a long list in place)
    const unsigned raw = win_a + warp * (kSwGatherMax * NC * 8);
    const bool vec16 = NC == 2 && (a.R % 2) == 0 && (lb % 2) == 0;
    // bounded wait for group g; its image is then at group_at(g)
    auto wait_group = [&](int g) -> bool {
      const int slot = g % kSwFlight;
      const unsigned par = (unsigned)g / kSwFlight & 1u;
      if (__all_sync(0xffffffffu, mb_test_wait(&s_mbar[slot], par))) return true;
      long long spins = 1;
      bool ok = true;
      while (!mb_test_wait(&s_mbar[slot], par)) {
        if (++spins > a.spin_limit || *(volatile int*)&s_abort) { ok = false; break; }
        if (spins > 4) __nanosleep(32);   // leave the issue slots to the producer warp
      }
      if (__any_sync(0xffffffffu, !ok)) {
        if (lane == 0) atomicExch(&s_abort, 1);
        return false;
      }
      return true;
    };
    auto group_at = [&](int g) -> unsigned { return ring_a + *(volatile int*)&s_off[g % kSwFlight]; };
    // this warp no longer reads group g's ring area; its owner alone: count kSwWarps
    auto release = [&](int g, int count) {
      __syncwarp();
      if (lane == 0) mb_arrive(&s_free[g % kSwFlight], count);
    };
    // Units: resident runs and global phases.  Every unit ends with a barrier of all compute
    // warps, before which the next unit's first group is waited for; the barrier tells all
    // warps whether a wait gave up in the unit, and then all stop.
    const int ngroup = (int)a.ngroup, n0 = a.n0;
    int g = 0;
    bool bad = all_red_or(!wait_group(0));   // warp-uniform
    while (!bad && g < ngroup) {
      unsigned gimg = group_at(g);
      int2 H = lds_i2(gimg);                 // nph, flags
      int off_desc = lds_i(gimg + 24);
      const int aux = lds_i(gimg + 28);
      if (!(H.y & SWG_RES)) {
        // ---- a global phase: groups g .. g + aux - 1, one batch each; this warp's are g + warp,
        // g + warp + kSwWarps, ...  The gather of its next batch (cp.async) is in flight while the
        // current one is computed from its regrouped inputs, if that group has arrived -- but for
        // rows that add, whose old values are still read from the gathered entries.
        const int gend = g + aux;
        const bool wide = (H.y & SWG_WIDE) != 0;   // lists regrouped in place, one at a time
        const unsigned pairs = raw + (wide ? 0 : kSwGather * NC * 8);
        if (warp > 0) release(g, 1);   // (the first group: its owner, and every warp that read its header)
        auto gather = [&](unsigned img, unsigned cd) {
          const int ngl = lds_i(cd + 16);
          const unsigned gl = img + lds_i(cd) + lds_i(cd + 36);
          for (int k = lane; k < ngl; k += 32) slot_async<NC>(a, lds_i(gl + 4 * k), raw + k * (8 * NC), xb, stp, ncol, vec16);
          cp_commit();
        };
        auto regroup = [&](int nin) {
          cp_wait<0>();
          __syncwarp();
          for (int k = lane; 2 * k < nin; k += 32) {
            const unsigned r = raw + k * (16 * NC), p = pairs + k * (16 * NC);
            const float4 v = lds_f4(r);
            if constexpr (NC == 2) {
              const float4 w = lds_f4(r + 16);
              sts_f4(p, v.x, w.x, v.y, w.y);
              sts_f4(p + 16, v.z, w.z, v.w, w.w);
            } else {
              sts_f4(p, v.x, v.z, v.y, v.w);
            }
          }
          __syncwarp();
        };
        bool fail = false, ahead = false;   // ahead: the batch's gather has been started
        for (int q = g + warp; q < gend; q += kSwWarps) {
          if (!ahead && !(q == g || wait_group(q))) { fail = true; break; }
          const unsigned img = group_at(q), cd = img + lds_i(img + 24);
          if (!ahead) gather(img, cd);
          const int old0 = lds_i(cd + 20);
          regroup(old0 > 0 ? old0 : lds_i(cd + 16));
          const int nq = q + kSwWarps;
          ahead = old0 == 0 && !wide && nq < gend &&
                  __all_sync(0xffffffffu, mb_test_wait(&s_mbar[nq % kSwFlight], (unsigned)nq / kSwFlight & 1u));
          if (ahead) {
            const unsigned ni = group_at(nq);
            gather(ni, ni + lds_i(ni + 24));
          }
          run_batch<NC>(a, cd, img, pairs, raw, xb, stp, ncol, vec16, lane);
          release(q, q == g ? 1 : kSwWarps);
        }
        g = gend;
        // (the barrier also makes every compute warp's writes visible to the next phase)
        bad = all_red_or(fail || (g < ngroup && !wait_group(g)));
        continue;
      }
      // ---- a resident run: groups g .. g + aux - 1
      const int gend = g + aux, g_first = g;
      const int2 rows = lds_i2(gimg + 8);   // the run's rows [lo, hi)
      load_rows<NC>(xb, a.R, rows.x, rows.y, H.y >> kSwGroupSlots, n0, ncol, win_a, t);
      const int set = warp >= kSwSet ? SWP_SET1 : 0, wset = warp & (kSwSet - 1);
      bool hand = false, sync = true;   // the previous phase hands over to this one's set / all warps meet
      unsigned hid = 3;       // barrier of the next hand-over (3 and 4 in turn)
      int2 P0 = lds_i2(gimg + 32), nH = H, nP = H;   // the group's first phase; the next group's header
      unsigned nimg = 0;                             // the next group's image once seen, else 0
      int noff = 0;
      while (g < gend) {
        for (int k = 0; k < H.x; ++k) {
          int2 PH;   // nb, flags
          if (!bad) {
            PH = k == 0 ? P0 : lds_i2(gimg + 32 + 8 * k);
            // the group's last phase: look whether the next group has arrived, and read its header
            if (k + 1 == H.x && g + 1 < gend &&
                __all_sync(0xffffffffu, mb_test_wait(&s_mbar[(g + 1) % kSwFlight], (unsigned)(g + 1) / kSwFlight & 1u))) {
              nimg = group_at(g + 1);
              nH = lds_i2(nimg);
              noff = lds_i(nimg + 24);
              nP = lds_i2(nimg + 32);
            }
          } else {
            // after a wait that gave up: follow the run's barriers from the schedule in global memory
            const SwPhase p = reinterpret_cast<const SwPhase*>(a.image + a.groups[g].img + 32)[k];
            PH = make_int2(p.nb, p.flags);
          }
          const bool all = (PH.y & SWP_ALL) != 0, tri = (PH.y & SWP_TRI) != 0;
          const bool mine = all || (PH.y & SWP_SET1) == set;
          const int first = all ? (warp - (PH.y >> kSwPhaseWarp)) & (kSwWarps - 1) : wset;
          const bool rowsp = mine && !tri && !bad && first < PH.x;
          const unsigned desc = gimg + off_desc + 40 * ((PH.y >> kSwPhaseBase) & kSwBaseMask);
          Tile<NC> tile;
          if (rowsp) tile_open<NC>(tile, gimg, lds_i2(desc + 40 * first), win_a, lane);   // nothing here depends on the inputs
          if (hand) {
            if (mine) hand_sync(hid);
            hid ^= 7;
          } else if (sync) {
            all_sync();
          }
          if (rowsp) {
            run_phase<NC>(tile, gimg, desc, first, PH.x, all ? kSwWarps : kSwSet, win_a, lane);
          } else if (tri) {
            if (!bad) {
              const int toff = lds_i(desc), s = lds_i(desc + 8), a0 = lds_i(desc + 20);
              const bool up = (PH.y & SWP_UPPER) != 0;
              if (n0 & 1) run_tri<NC, false>(s, a0, up, gimg + toff, win_a, n0, warp, lane);
              else run_tri<NC, true>(s, a0, up, gimg + toff, win_a, n0, warp, lane);
            } else {
              all_sync();   // the barrier inside the triangle product
            }
          }
          hand = (PH.y & SWP_HAND) != 0;
          sync = (PH.y & SWP_END) != 0;   // (a phase's parts need no barrier between them)
          if (hand && mine) hand_arrive(hid);
        }
        if (!bad) release(g, 1);
        if (++g < gend) {
          if (!bad && nimg == 0) {
            bad = !wait_group(g);
            if (!bad) {
              nimg = group_at(g);
              nH = lds_i2(nimg);
              noff = lds_i(nimg + 24);
              nP = lds_i2(nimg + 32);
            }
          }
          if (!bad) {
            gimg = nimg;
            H = nH;
            off_desc = noff;
            P0 = nP;
            nimg = 0;
          } else {
            H.x = reinterpret_cast<const SwGroupHdr*>(a.image + a.groups[g].img)->nph;
          }
        }
      }
      all_sync();   // the run's last phase is done
      // An Inf or NaN that met a zero coefficient has made rows of the run NaN: look at them all
      bool odd = false;
      for (int r = t; r < rows.y - rows.x; r += kSwWarps * 32) {
        const unsigned d = slot_addr<NC>(win_a, sw_row_slot(r, n0));
#pragma unroll
        for (int c = 0; c < NC; ++c) odd = odd || !isfinite(lds_f(d + 16 * c)) || !isfinite(lds_f(d + 16 * c + 8));
      }
      if (all_red_or(odd)) {
        if (t == 0) *(volatile int*)&s_redo = 1;
        if constexpr (NC == 1) redo_run_1(a.image, a.groups + g_first, aux, xb, a.R, n0, ncol, win_a, warp, lane);
        else redo_run<NC>(a.image, a.groups + g_first, aux, xb, a.R, n0, ncol, win_a, warp, lane);
        if (t == 0) *(volatile int*)&s_redo = 0;
      }
      if (!bad)
        for (int e = t; e < (rows.y - rows.x) * NC; e += kSwWarps * 32) {
          const int r = e / NC, c = e % NC;
          const unsigned d = slot_addr<NC>(win_a, sw_row_slot(r, n0)) + 16 * c;
          if (c < ncol) xb[(int64_t)(rows.x + r) * a.R + c] = make_float2(lds_f(d), lds_f(d + 8));
        }
      bad = all_red_or(bad || (g < ngroup && !wait_group(g)));   // (the rows are written back)
    }
    if (bad && t == 0) {
      atomicExch(&s_abort, 1);
      atomicExch(a.err_out, 1);
    }
  }
  __syncthreads();
  if (*(volatile int*)&s_abort) {
    // give the copies still in flight a second bounded wait before leaving
    const int iss = s_issued;
    for (int q = 0; q < iss; ++q) {
      if (q + kSwFlight < iss) continue;
      long long spins = 0;
      while (!mb_try_wait(&s_mbar[q % kSwFlight], (unsigned)(q / kSwFlight) & 1u) &&
             ++spins < drain_limit(a.spin_limit)) {
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < kSwFlight; ++k) {
      mb_inval(&s_mbar[k]);
      mb_inval(&s_free[k]);
    }
}

template <int NC>
int launch_nc(const DevFactor& df, const DevSched& sc, float2* vec, int64_t R, int64_t col0, int grid, float2* st,
              cudaStream_t s) {
  auto kern = k_sweep_cols<NC>;
  static bool attr_done = false;
  if (!attr_done) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSwSmem) != cudaSuccess) {
      set_error("column-partitioned sweep: shared-memory attribute failed");
      return HB_ECUDA;
    }
    attr_done = true;
  }
  SwArgs a;
  a.groups = sc.groups;
  a.ngroup = sc.ngroup;
  a.image = sc.image;
  a.x = vec;
  a.R = R;
  a.n = df.n;
  a.n0 = (int)df.n0;
  a.col0 = col0;
  a.st = st;
  a.state_len = df.state_len;
  a.err_out = &((GridBar*)df.bar)->err;
  a.spin_limit = df.spin_limit;
  kern<<<grid, kSwThreads, kSwSmem, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("column-partitioned sweep launch failed: %s", cudaGetErrorString(e));
    return HB_ECUDA;
  }
  return HB_OK;
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

}  // namespace

int64_t sweep_cols_state_entries(const DevFactor& df, int64_t R) {
  // launches cover 2 * sms columns at a time (one column per CTA when R <= sms)
  const int64_t sms = sm_count();
  if (R <= sms) return df.state_len * R;
  const int64_t cols = std::min<int64_t>(R, 2 * sms);
  return df.state_len * ((cols + 1) / 2) * 2;
}

int launch_sweep_cols(const DevFactor& df, int which, void* vec, int64_t R, void* state, cudaStream_t s) {
  if (which < 0 || which > 3 || !df.sw[which].ok) {
    set_error("column-partitioned sweep: no schedule for this sweep");
    return HB_EUNSUPPORTED;
  }
  const DevSched& sc = df.sw[which];
  const int64_t sms = sm_count();
  float2* v = static_cast<float2*>(vec);
  float2* st = static_cast<float2*>(state);
  if (R <= sms) return launch_nc<1>(df, sc, v, R, 0, (int)R, st, s);
  for (int64_t c0 = 0; c0 < R; c0 += 2 * sms) {
    const int64_t cols = std::min<int64_t>(R - c0, 2 * sms);
    const int rc = launch_nc<2>(df, sc, v, R, c0, (int)((cols + 1) / 2), st, s);
    if (rc) return rc;
  }
  return HB_OK;
}

int sweep_cols_launches(int64_t R) {
  const int64_t sms = sm_count();
  return R <= sms ? 1 : (int)((R + 2 * sms - 1) / (2 * sms));
}

}  // namespace hb
