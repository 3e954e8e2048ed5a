// Hot-path CUDA kernels (sm_103a): H-IDBF apply (Alg. 2), forward and adjoint.
// (The L~ / U~ sweeps of Algs. 3, 4 live in hb_sweep.cu.)
//
// Every butterfly factor is a set of small ID blocks (Sec. 2 / Appendix).  A
// CTA owns one block op; the packer stores every matrix with the output index
// fastest, so forward factor loads are contiguous over the outputs.
//   vlike  (V stage, column ID):  z_i  = cand[q_i] + sum_j T_ij cand[p_j]
//   ulike  (U stage, row ID):     out_r = y_{map r}            (r skeleton)
//                                 out_r = sum_i T_i,j(r) y_i   (r redundant)
//   middle:                       y = S z
// Adjoint ops swap the two shapes and conjugate the entries.
// Vectors and the butterfly state use the layout [entry][R] (RHS fastest).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "hb_device.h"

namespace hb {

template <class T> struct C2;
template <> struct C2<float> { using t = float2; };
template <> struct C2<double> { using t = double2; };

// Double-float numbers (a pair of FP32 values, about 48 significant bits): the
// FP64-accurate arithmetic of the complex-FP32 factors' refinement residual at
// FP32 instruction rates (FP64 runs at a small fraction of them on this GPU).
// The product uses the exact FMA residual of the high parts (Dekker / Knuth
// two-product with FMA), the sum the two-sum of the high parts with the low
// parts added; both renormalised.
struct Dd {
  float h, l;
  __host__ __device__ Dd(float v = 0.f) : h(v), l(0.f) {}
  __host__ __device__ Dd(float hi, float lo) : h(hi), l(lo) {}
};
struct __align__(16) DdC {
  Dd x, y;
};
template <> struct C2<Dd> { using t = DdC; };
__device__ __forceinline__ Dd dd_norm(float s, float e) {
  const float t = s + e;
  return Dd(t, e - (t - s));
}
__device__ __forceinline__ Dd operator-(const Dd& a) { return Dd(-a.h, -a.l); }
__device__ __forceinline__ Dd dd_add(const Dd& a, const Dd& b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  const float e = ((a.h - (s - bb)) + (b.h - bb)) + (a.l + b.l);
  return dd_norm(s, e);
}
__device__ __forceinline__ Dd& operator+=(Dd& a, const Dd& b) { a = dd_add(a, b); return a; }
// c + a * b with an FP32 coefficient a (the product's pair need not be normalised before the sum)
__device__ __forceinline__ Dd dd_fma(float a, const Dd& b, const Dd& c) {
  const float p = a * b.h;
  return dd_add(c, Dd(p, fmaf(a, b.l, fmaf(a, b.h, -p))));
}

template <class T> __device__ __forceinline__ typename C2<T>::t mk(T a, T b) { return {a, b}; }

// a factor coefficient as the arithmetic takes it (double-float: the FP32 values themselves)
template <class T> struct Coef { using t = typename C2<T>::t; };
template <> struct Coef<Dd> { using t = float2; };
template <class T, class F>
__device__ __forceinline__ typename Coef<T>::t ldf(const F* p) {
  F v = __ldg(p);
  using S = decltype(Coef<T>::t::x);
  return {(S)v.x, (S)v.y};
}
template <class T, class F>
__device__ __forceinline__ typename Coef<T>::t ldf_conj(const F* p) {
  F v = __ldg(p);
  using S = decltype(Coef<T>::t::x);
  return {(S)v.x, -(S)v.y};
}
// acc += a * b
template <class C>
__device__ __forceinline__ void cfma(C& acc, const C& a, const C& b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
__device__ __forceinline__ void cfma(DdC& acc, const float2& a, const DdC& b) {
  acc.x = dd_fma(a.x, b.x, acc.x);
  acc.x = dd_fma(-a.y, b.y, acc.x);
  acc.y = dd_fma(a.x, b.y, acc.y);
  acc.y = dd_fma(a.y, b.x, acc.y);
}
template <class C>
__device__ __forceinline__ void cadd(C& acc, const C& a) {
  acc.x += a.x;
  acc.y += a.y;
}

// ---------------------------------------------------------------------------
// One right-hand side, a launch per step: the directions and factors that the persistent
// kernel's plan does not hold (blocks above its staging area, as close parallel strips give
// them).  A CTA takes one op, so that an op of a hundred by a hundred coefficients does not
// sit in one warp: the product's coefficients are read along their contiguous index, outputs
// across the threads and the inputs shared out over thread groups (joined in shared memory),
// or a warp to an output with lanes along the inputs.  Bound by the launches and the largest
// op of a step.  Eight strips, 131,072 unknowns, adjoint, complex64: inner steps 616 us with
// a warp to an op, 369 us now; entry 74 us, 36 us now.
// ---------------------------------------------------------------------------
constexpr int k1Threads = 64;
constexpr int k1In = 512;   // inputs staged at a time
template <class C> struct OneStage {
  C in[k1In];
  C red[k1Threads];
};
__device__ __forceinline__ float shfl_down1(float v, int d) { return __shfl_down_sync(0xffffffffu, v, d); }
__device__ __forceinline__ double shfl_down1(double v, int d) { return __shfl_down_sync(0xffffffffu, v, d); }

// put(o, sum_j M(o, j) in(j)) for o < O.  JFAST: M(o, j) = conj(M[o * J + j]); otherwise M[j * O + o].
// Whole CTA; ends with a barrier.
template <class T, class F, bool JFAST, class In, class Put>
__device__ __forceinline__ void one_dot(OneStage<typename C2<T>::t>& sm, const F* __restrict__ M, int O, int J, In&& in,
                                        Put&& put) {
  using C = typename C2<T>::t;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  constexpr int U = 4;   // outputs of a warp at a time (JFAST)
  const int ow = JFAST ? k1Threads / 32 * U : (O <= 32 ? 32 : O <= 64 ? 64 : k1Threads);
  for (int o0 = 0; o0 < O; o0 += ow) {
    C acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) acc[u] = mk<T>(0, 0);
    for (int j0 = 0; j0 < J; j0 += k1In) {
      const int nj = min(k1In, J - j0);
      if (o0 == 0 || J > k1In) {
        for (int j = t; j < nj; j += k1Threads) sm.in[j] = in(j0 + j);
        __syncthreads();
      }
      if (JFAST) {
#pragma unroll 2
        for (int j = lane; j < nj; j += 32) {
          const C v = sm.in[j];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int o = o0 + warp * U + u;
            if (o < O) cfma(acc[u], ldf_conj<T>(M + (int64_t)o * J + j0 + j), v);
          }
        }
      } else {
        const int o = o0 + t % ow, g = t / ow, G = k1Threads / ow;
        if (o < O) {
#pragma unroll 4
          for (int j = g; j < nj; j += G) cfma(acc[0], ldf<T>(M + (int64_t)(j0 + j) * O + o), sm.in[j]);
        }
      }
      if (J > k1In) __syncthreads();
    }
    if (JFAST) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
          acc[u].x += shfl_down1(acc[u].x, d);
          acc[u].y += shfl_down1(acc[u].y, d);
        }
        const int o = o0 + warp * U + u;
        if (lane == 0 && o < O) put(o, acc[u]);
      }
    } else {
      sm.red[t] = acc[0];
      __syncthreads();
      if (t < ow && o0 + t < O) {
        C v = sm.red[t];
        for (int g = 1; g < k1Threads / ow; ++g) cadd(v, sm.red[g * ow + t]);
        put(o0 + t, v);
      }
      __syncthreads();
    }
  }
  __syncthreads();
}

template <class T, class F, bool ADJ>
__global__ void __launch_bounds__(k1Threads) k_apply_enter(const DOuter* __restrict__ ops, int64_t n0,
                                                           const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                                           const typename C2<T>::t* __restrict__ x,
                                                           typename C2<T>::t* st) {
  using C = typename C2<T>::t;
  __shared__ OneStage<C> sm;
  const DOuter o = ops[blockIdx.x];   // (leaf, depth) = (blockIdx.x / D, blockIdx.x % D)
  const C* xl = x + (int64_t)o.leaf * n0;
  C* out = st + o.seg_off;
  const int k = o.blk.k;
  const int16_t* idx = ip + o.blk.ioff;
  one_dot<T, F, ADJ>(sm, fp + o.blk.moff, k, o.blk.c - k, [&](int j) { return xl[idx[k + j]]; },
                     [&](int i, C v) {
                       cadd(v, xl[idx[i]]);
                       out[i] = v;
                     });
}

template <class T, class F, bool ADJ>
__global__ void __launch_bounds__(k1Threads) k_apply_items(const DItem* __restrict__ items,
                                                           const int32_t* __restrict__ order, const F* __restrict__ fp,
                                                           const int16_t* __restrict__ ip, typename C2<T>::t* st) {
  using C = typename C2<T>::t;
  __shared__ OneStage<C> sm;
  const DItem& it = items[order[blockIdx.x]];
  const int type = it.type;
  if (type == 1) {   // middle: y = S z (or z = S^H y)
    const int kr = it.b_k[0], kc = it.a_k[0];
    const C* in = st + (ADJ ? it.b_off[0] : it.a_off[0]);
    C* out = st + (ADJ ? it.a_off[0] : it.b_off[0]);
    one_dot<T, F, ADJ>(sm, fp + it.blk[0].moff, ADJ ? kc : kr, ADJ ? kr : kc, [&](int j) { return in[j]; },
                       [&](int o, C v) { out[o] = v; });
    return;
  }
  const int ka0 = it.a_k[0], c = ka0 + it.a_k[1];
  const int a0 = it.a_off[0], a1 = it.a_off[1] - ka0;
  const auto cand = [&](int r) { return (r < ka0 ? a0 : a1) + r; };   // candidate entry r in the state
  if ((type == 0) != ADJ) {   // candidates -> skeletons
#pragma unroll 1
    for (int sb = 0; sb < 2; ++sb) {
      const DBlk& b = it.blk[sb];
      const int k = b.k;
      const int16_t* idx = ip + b.ioff;
      C* out = st + it.b_off[sb];
      one_dot<T, F, ADJ>(sm, fp + b.moff, k, c - k, [&](int j) { return st[cand(idx[k + j])]; },
                         [&](int i, C v) {
                           cadd(v, st[cand(idx[i])]);
                           out[i] = v;
                         });
    }
    return;
  }
  // skeletons -> candidates: the rows that are skeletons of both blocks, then the rows that
  // block 0 interpolates, then those that block 1 does, each on top of the other block's value
#pragma unroll 1
  for (int sb = 0; sb < 2; ++sb) {
    const DBlk& b = it.blk[sb];
    const int k = b.k;
    const int16_t* own = ip + b.ioff;
    const int16_t* oth = ip + it.blk[1 - sb].ioff + c;
    const C* y = st + it.b_off[sb];
    const C* yx = st + it.b_off[1 - sb];
    if (sb == 0)
      for (int i = threadIdx.x; i < k; i += k1Threads) {
        const int r = own[i], code = oth[r];
        if (code < 0) continue;
        C v = y[i];
        cadd(v, yx[code]);
        st[cand(r)] = v;
      }
    one_dot<T, F, ADJ>(sm, fp + b.moff, c - k, k, [&](int j) { return y[j]; },
                       [&](int o, C v) {
                         const int r = own[k + o], code = oth[r];
                         if (code >= 0) cadd(v, yx[code]);
                         else if (sb == 1) cadd(v, st[cand(r)]);
                         st[cand(r)] = v;
                       });
  }
}

// y_leaf = sum_v U0_v y_0 + A_leaf x_leaf (adjoint: sum_v V0^H z_0 + A_leaf^H x_leaf).  Block = leaf;
// thread (row, group): a group takes every G-th depth and every G-th column of the dense leaf;
// the groups' sums join in a fixed order.
template <class T, class F, bool ADJ>
__global__ void __launch_bounds__(256) k_apply_exit(const DOuter* __restrict__ ops, int D, int64_t n0,
                                                    const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                                    const F* __restrict__ leafm,
                                                    const typename C2<T>::t* __restrict__ x,
                                                    const typename C2<T>::t* st, typename C2<T>::t* y) {
  using C = typename C2<T>::t;
  __shared__ C red[256];
  const int64_t leaf = blockIdx.x;
  const F* A = leafm + leaf * n0 * n0;
  const C* xl = x + leaf * n0;
  const int rw = n0 < 256 ? (int)((n0 + 31) / 32 * 32) : 256, G = 256 / rw, g = threadIdx.x / rw;
  for (int64_t rb = 0; rb < n0; rb += rw) {
    const int64_t r = rb + threadIdx.x % rw;
    C acc = mk<T>(0, 0);
    if (g < G && r < n0) {
      for (int v = g; v < D; v += G) {
        const DOuter o = ops[leaf * D + v];
        const C* z = st + o.seg_off;
        const F* M = fp + o.blk.moff;
        const int k = o.blk.k, nr = o.blk.c - k, code = ip[o.blk.ioff + o.blk.c + r];
        if (code >= 0) {
          cadd(acc, z[code]);
        } else {
          const int j = -1 - code;
#pragma unroll 4
          for (int i = 0; i < k; ++i)
            cfma(acc, ADJ ? ldf_conj<T>(M + (int64_t)j * k + i) : ldf<T>(M + (int64_t)i * nr + j), z[i]);
        }
      }
#pragma unroll 4
      for (int64_t cc = g; cc < n0; cc += G) cfma(acc, ADJ ? ldf_conj<T>(A + r * n0 + cc) : ldf<T>(A + cc * n0 + r), xl[cc]);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    if (g == 0 && r < n0) {
      for (int q = 1; q < G; ++q) cadd(acc, red[q * rw + threadIdx.x]);
      y[leaf * n0 + r] = acc;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Two to kFewMax right-hand sides in FP32: a warp to an op, lanes over its outputs, RC columns
// in a lane's registers.  With so few columns a staged chunk (below) is mostly barriers and idle
// threads: 16,384 unknowns, complex64, 2 / 4 / 6 columns forward 117 / 119 / 137 us here against
// 180 / 156 / 153 us, adjoint 104 / 106 / 130 against 201 / 166 / 160; at 8 columns the two meet
// (150 / 142 against 148 / 149), at 12 the chunks lead (212 against 144).  In FP64 they lead
// from 2 columns on (426 against 337 us), since here every lane repeats the column loop.
// R = row stride of the [entry][R] layout, r0 = first RHS of this pass, rc = number of valid RHS
// in the pass (<= RC).
// ---------------------------------------------------------------------------
constexpr int kFewMax = 8;

// B side (k outputs) = gather + T * rest of the candidate vector cand =
// concat(a0[0..ka0), a1[..]).  UTYPE_ADJ: the block is a row ID used in
// adjoint (entries conj(T_ij) read from the U-type layout M[i*(c-k)+j]);
// otherwise a column ID (V-type layout M[j*k+i]).
template <class T, class F, int RC, bool UTYPE_ADJ>
__device__ __forceinline__ void op_vlike(const F* __restrict__ M, const int16_t* __restrict__ idx, int k, int c,
                                         const typename C2<T>::t* a0, int ka0, const typename C2<T>::t* a1,
                                         typename C2<T>::t* out, int64_t R, int64_t r0, int rc, int lane) {
  using C = typename C2<T>::t;
  const int nr = c - k;
  for (int i = lane; i < k; i += 32) {
    C acc[RC];
    const int qi = idx[i];
    const C* src = (qi < ka0) ? a0 + (int64_t)qi * R : a1 + (int64_t)(qi - ka0) * R;
#pragma unroll
    for (int rr = 0; rr < RC; ++rr) acc[rr] = (rr < rc) ? src[r0 + rr] : mk<T>(0, 0);
#pragma unroll 4
    for (int j = 0; j < nr; ++j) {
      C mij = UTYPE_ADJ ? ldf_conj<T>(M + (int64_t)i * nr + j) : ldf<T>(M + (int64_t)j * k + i);
      const int pj = idx[k + j];
      const C* s = (pj < ka0) ? a0 + (int64_t)pj * R : a1 + (int64_t)(pj - ka0) * R;
#pragma unroll
      for (int rr = 0; rr < RC; ++rr)
        if (rr < rc) cfma(acc[rr], mij, s[r0 + rr]);
    }
#pragma unroll
    for (int rr = 0; rr < RC; ++rr)
      if (rr < rc) out[(int64_t)i * R + r0 + rr] = acc[rr];
  }
}

// Contribution of one block to candidate entry r: VTYPE_ADJ: the block is a
// column ID used in adjoint (conj(T_ij) from M[j*k+i]); otherwise a row ID
// (U-type layout M[i*(c-k)+j]).
template <class T, class F, int RC, bool VTYPE_ADJ>
__device__ __forceinline__ void row_contrib(typename C2<T>::t (&acc)[RC], const F* __restrict__ M,
                                            const int16_t* __restrict__ idx, int k, int c,
                                            const typename C2<T>::t* y, int64_t R, int64_t r0, int rc, int r) {
  using C = typename C2<T>::t;
  const int code = idx[c + r];
  if (code >= 0) {
    const C* s = y + (int64_t)code * R + r0;
#pragma unroll
    for (int rr = 0; rr < RC; ++rr)
      if (rr < rc) cadd(acc[rr], s[rr]);
  } else {
    const int j = -1 - code;
    const int nr = c - k;
#pragma unroll 4
    for (int i = 0; i < k; ++i) {
      C mij = VTYPE_ADJ ? ldf_conj<T>(M + (int64_t)j * k + i) : ldf<T>(M + (int64_t)i * nr + j);
      const C* s = y + (int64_t)i * R + r0;
#pragma unroll
      for (int rr = 0; rr < RC; ++rr)
        if (rr < rc) cfma(acc[rr], mij, s[rr]);
    }
  }
}

template <class T, class F, int RC>
__device__ __forceinline__ void op_middle(const F* __restrict__ S, int kr, int kc, bool adj,
                                          const typename C2<T>::t* in, typename C2<T>::t* out, int64_t R,
                                          int64_t r0, int rc, int lane) {
  using C = typename C2<T>::t;
  const int nout = adj ? kc : kr, nin = adj ? kr : kc;
  for (int o = lane; o < nout; o += 32) {
    C acc[RC];
#pragma unroll
    for (int rr = 0; rr < RC; ++rr) acc[rr] = mk<T>(0, 0);
#pragma unroll 4
    for (int i = 0; i < nin; ++i) {
      C s = adj ? ldf_conj<T>(S + (int64_t)o * kr + i) : ldf<T>(S + (int64_t)i * kr + o);
      const C* v = in + (int64_t)i * R + r0;
#pragma unroll
      for (int rr = 0; rr < RC; ++rr)
        if (rr < rc) cfma(acc[rr], s, v[rr]);
    }
#pragma unroll
    for (int rr = 0; rr < RC; ++rr)
      if (rr < rc) out[(int64_t)o * R + r0 + rr] = acc[rr];
  }
}

// One inner item (two ID blocks or one middle block), one warp.
template <class T, class F, int RC, bool ADJ>
__device__ __forceinline__ void op_item(const DItem& it, const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                        typename C2<T>::t* st, int64_t R, int64_t r0, int rc, int lane) {
  using C = typename C2<T>::t;
  if (it.type == 1) {
    const F* S = fp + it.blk[0].moff;
    if (!ADJ) op_middle<T, F, RC>(S, it.b_k[0], it.a_k[0], false, st + (int64_t)it.a_off[0] * R, st + (int64_t)it.b_off[0] * R, R, r0, rc, lane);
    else op_middle<T, F, RC>(S, it.b_k[0], it.a_k[0], true, st + (int64_t)it.b_off[0] * R, st + (int64_t)it.a_off[0] * R, R, r0, rc, lane);
    return;
  }
  const bool to_b = (it.type == 0) != ADJ;   // V forward or U adjoint: A (candidates) -> B (skeletons)
  if (to_b) {
    const C* a0 = st + (int64_t)it.a_off[0] * R;
    const C* a1 = st + (int64_t)it.a_off[1] * R;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const DBlk& b = it.blk[s];
      if (it.type == 0)
        op_vlike<T, F, RC, false>(fp + b.moff, ip + b.ioff, b.k, b.c, a0, it.a_k[0], a1, st + (int64_t)it.b_off[s] * R, R, r0, rc, lane);
      else
        op_vlike<T, F, RC, true>(fp + b.moff, ip + b.ioff, b.k, b.c, a0, it.a_k[0], a1, st + (int64_t)it.b_off[s] * R, R, r0, rc, lane);
    }
  } else {
    const int c = it.a_k[0] + it.a_k[1];
    for (int r = lane; r < c; r += 32) {
      C acc[RC];
#pragma unroll
      for (int rr = 0; rr < RC; ++rr) acc[rr] = mk<T>(0, 0);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const DBlk& b = it.blk[s];
        if (it.type == 2)
          row_contrib<T, F, RC, false>(acc, fp + b.moff, ip + b.ioff, b.k, b.c, st + (int64_t)it.b_off[s] * R, R, r0, rc, r);
        else
          row_contrib<T, F, RC, true>(acc, fp + b.moff, ip + b.ioff, b.k, b.c, st + (int64_t)it.b_off[s] * R, R, r0, rc, r);
      }
      C* dst = (r < it.a_k[0]) ? st + (int64_t)(it.a_off[0] + r) * R : st + (int64_t)(it.a_off[1] + r - it.a_k[0]) * R;
#pragma unroll
      for (int rr = 0; rr < RC; ++rr)
        if (rr < rc) dst[r0 + rr] = acc[rr];
    }
  }
}

// Forward: block = column leaf j; warp w handles depths v = w, w+W, ...:
// z_0 = V0 x_j.  Adjoint: block = row leaf i; y_0 = U0^H x_i.
template <class T, class F, int RC, bool ADJ>
__global__ void __launch_bounds__(256) k_few_enter(const DOuter* __restrict__ ops, int D, int64_t n0,
                                                     const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                                     const typename C2<T>::t* __restrict__ x,
                                                     typename C2<T>::t* st, int64_t R) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t leaf = blockIdx.x;
  const typename C2<T>::t* xl = x + leaf * n0 * R;
  for (int v = warp; v < D; v += nw) {
    const DOuter o = ops[leaf * D + v];
    for (int64_t r0 = 0; r0 < R; r0 += RC) {
      int rc = (int)(R - r0 < (int64_t)RC ? R - r0 : (int64_t)RC);
      op_vlike<T, F, RC, ADJ>(fp + o.blk.moff, ip + o.blk.ioff, o.blk.k, o.blk.c, xl, (int)n0, xl,
                              st + (int64_t)o.seg_off * R, R, r0, rc, lane);
    }
  }
}

template <class T, class F, int RC, bool ADJ>
__global__ void __launch_bounds__(256) k_few_items(const DItem* __restrict__ items, const int32_t* __restrict__ idx,
                                                     int count, const F* __restrict__ fp,
                                                     const int16_t* __restrict__ ip, typename C2<T>::t* st,
                                                     int64_t R) {
  const int lane = threadIdx.x & 31;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= count) return;
  const DItem it = items[idx[w]];
  for (int64_t r0 = 0; r0 < R; r0 += RC) {
    int rc = (int)(R - r0 < (int64_t)RC ? R - r0 : (int64_t)RC);
    op_item<T, F, RC, ADJ>(it, fp, ip, st, R, r0, rc, lane);
  }
}

// Forward: block = row leaf i, thread = row r: y_r = sum_v (U0 y_0)_r + (A_leaf x_i)_r,
// summed in the fixed order v = 0..D-1 then the dense leaf.  Adjoint: block =
// column leaf j: (A^H x)_j = sum_v (V0^H z_0) + A_leaf^H x_j.
template <class T, class F, int RC, bool ADJ>
__global__ void __launch_bounds__(256) k_few_exit(const DOuter* __restrict__ ops, int D, int64_t n0,
                                                    const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                                    const F* __restrict__ leafm,
                                                    const typename C2<T>::t* __restrict__ x,
                                                    const typename C2<T>::t* st, typename C2<T>::t* y,
                                                    int64_t R) {
  using C = typename C2<T>::t;
  const int64_t leaf = blockIdx.x;
  const F* A = leafm + leaf * n0 * n0;
  const C* xl = x + leaf * n0 * R;
  for (int r = threadIdx.x; r < n0; r += blockDim.x) {
    for (int64_t r0 = 0; r0 < R; r0 += RC) {
      int rc = (int)(R - r0 < (int64_t)RC ? R - r0 : (int64_t)RC);
      C acc[RC];
#pragma unroll
      for (int rr = 0; rr < RC; ++rr) acc[rr] = mk<T>(0, 0);
      for (int v = 0; v < D; ++v) {
        const DOuter o = ops[leaf * D + v];
        row_contrib<T, F, RC, ADJ>(acc, fp + o.blk.moff, ip + o.blk.ioff, o.blk.k, o.blk.c,
                                   st + (int64_t)o.seg_off * R, R, r0, rc, r);
      }
#pragma unroll 4
      for (int cc = 0; cc < n0; ++cc) {
        C a = ADJ ? ldf_conj<T>(A + (int64_t)r * n0 + cc) : ldf<T>(A + (int64_t)cc * n0 + r);
        const C* s = xl + (int64_t)cc * R + r0;
#pragma unroll
        for (int rr = 0; rr < RC; ++rr)
          if (rr < rc) cfma(acc[rr], a, s[rr]);
      }
      C* dst = y + (leaf * n0 + r) * R + r0;
#pragma unroll
      for (int rr = 0; rr < RC; ++rr)
        if (rr < rc) dst[rr] = acc[rr];
    }
  }
}

// ---------------------------------------------------------------------------
// Column-parallel apply (R >= 2; FP32: more than kFewMax).  A CTA takes one op and up to cw * NC right-hand sides;
// thread = (slot, column), and a slot owns chunks of KC outputs, which its threads keep in
// registers for NC columns each while they walk the op's inputs once.  Vector rows are read
// along the columns of the [entry][R] layout; a slot's coefficients [input][KC] and input
// rows are staged in shared memory first, zero-padded to KC, so that a chunk is one
// unguarded FMA sequence with two coefficients to a 16-byte broadcast load.
// What bounds it are the dependent loads of one op (item, index lists, coefficients, vector
// rows), so chunks are small and the warps many: KC = 4, NC = 2 for FP32 and R >= 64 (four CTAs
// of 256 threads an SM; KC = 8 at 128 registers: twice the time), KC = 2, NC = 1 otherwise, and
// more slots where a step has few ops.  The twelve inner steps of 262,144 unknowns x 256
// columns: 6.47 ms with one column a thread, 16 outputs and a guarded global load to every
// coefficient, 2.77 ms now; the ten of 50,176 x 12: 206 us with a warp to an op and lanes over
// its outputs, 192 us now (entry 130 -> 90 us); 16,384 x 40 in double-float: 319 -> 130 us.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void put_coef(float2& d, float2 v) { d = v; }
__device__ __forceinline__ void put_coef(double2& d, float2 v) { d = make_double2(v.x, v.y); }
__device__ __forceinline__ void put_coef(double2& d, double2 v) { d = v; }

// A chunk: outputs o0 .. o0+no-1 (no <= KC) of a dense product with J inputs;
// coefficient (input j, output o) = M[j * sj + o * so], conjugated where asked.
template <class F> struct WChunk {
  const F* M;
  int J, sj, so, o0, no;
  int sb;   // for the caller: which block
};

constexpr int kWStage = 2048;   // coefficients staged by a CTA (all slots)
constexpr int kWThreads = 256;
constexpr int kWSlots = 16;
constexpr int64_t kWFill = 152 * 2048;   // threads that a step should have at least
// CTAs of 256 threads an SM should hold (the kernels wait on dependent loads: warps hide them)
template <class T, int NC> constexpr int w_ctas() { return std::is_same<T, float>::value ? (NC == 2 ? 4 : 6) : 3; }
template <class T, int KC> struct WStage {
  alignas(16) typename Coef<T>::t coef[kWStage];
  int32_t row[kWStage / KC];
};

// All chunks [0, nch) of one op.  chunk(ch) describes one; row_in(w, j) is the row of input j
// (in units of R entries from `in`); init(w, o, ii, col) the value an output starts from;
// row_out(w, o) the row of an output from `out` (< 0: not written).  jmax >= every chunk's J.
template <class T, class F, int KC, int NC, bool CONJ, class ChunkF, class RowIn, class Init, class RowOut>
__device__ __forceinline__ void w_chunks(WStage<T, KC>& sm, int nch, int jmax, int cw, int ns, const typename C2<T>::t* in,
                                         typename C2<T>::t* out, int64_t R, ChunkF&& chunk, RowIn&& row_in,
                                         Init&& init, RowOut&& row_out) {
  using C = typename C2<T>::t;
  using S = typename Coef<T>::t;
  const int slot = threadIdx.x / cw, lane = threadIdx.x - slot * cw;
  const int jb = kWStage / (ns * KC);
  S* coef = sm.coef + slot * jb * KC;
  int32_t* rows = sm.row + slot * jb;
  int64_t col[NC];
  bool ok[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    col[q] = (int64_t)blockIdx.y * cw * NC + q * cw + lane;
    ok[q] = col[q] < R;
  }
  for (int c0 = 0; c0 < nch; c0 += ns) {
    const bool act = c0 + slot < nch;
    WChunk<F> w{};
    if (act) w = chunk(c0 + slot);
    C acc[NC][KC];
    int j0 = 0;
    do {
      const int nj = act ? (w.J - j0 < jb ? w.J - j0 : jb) : 0;
      if (nj > 0) {
        for (int e = lane; e < nj * KC; e += cw) {
          // along the index that is contiguous in memory
          const int j = w.so == 1 ? e / KC : e % nj, ii = w.so == 1 ? e % KC : e / nj;
          F v{0, 0};
          if (ii < w.no) {
            v = __ldg(w.M + (int64_t)(j0 + j) * w.sj + (int64_t)(w.o0 + ii) * w.so);
            if (CONJ) v.y = -v.y;
          }
          put_coef(coef[j * KC + ii], v);
        }
        for (int j = lane; j < nj; j += cw) rows[j] = row_in(w, j0 + j);
      }
      if (j0 == 0) {
#pragma unroll
        for (int q = 0; q < NC; ++q)
#pragma unroll
          for (int ii = 0; ii < KC; ++ii) {
            acc[q][ii] = mk<T>(0, 0);
            if (act && ii < w.no && ok[q]) acc[q][ii] = init(w, w.o0 + ii, col[q]);
          }
      }
      __syncthreads();
      if (nj > 0 && ok[0]) {
#pragma unroll (NC == 2 ? 2 : 4)
        for (int j = 0; j < nj; ++j) {
          const C* src = in + (int64_t)rows[j] * R;
          C v[NC];
#pragma unroll
          for (int q = 0; q < NC; ++q) v[q] = ok[q] ? src[col[q]] : mk<T>(0, 0);
          constexpr int per = 16 / (int)sizeof(S) ? 16 / (int)sizeof(S) : 1;
          struct __align__(16) Pack { S s[per]; };
#pragma unroll
          for (int i2 = 0; i2 < KC; i2 += per) {
            const Pack pk = *reinterpret_cast<const Pack*>(coef + j * KC + i2);
#pragma unroll
            for (int u = 0; u < per; ++u) {
#pragma unroll
              for (int q = 0; q < NC; ++q) cfma(acc[q][i2 + u], pk.s[u], v[q]);
            }
          }
        }
      }
      __syncthreads();
      j0 += jb;
    } while (j0 < jmax);
    if (act) {
#pragma unroll
      for (int ii = 0; ii < KC; ++ii) {
        if (ii >= w.no) continue;
        const int64_t r = row_out(w, w.o0 + ii);
        if (r < 0) continue;
#pragma unroll
        for (int q = 0; q < NC; ++q)
          if (ok[q]) out[r * R + col[q]] = acc[q][ii];
      }
    }
  }
}

template <class T, class F, bool ADJ, int KC, int NC>
__global__ void __launch_bounds__(kWThreads, w_ctas<T, NC>()) k_wapply_enter(const DOuter* __restrict__ ops, int64_t n0,
                                                            const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                                            const typename C2<T>::t* __restrict__ x,
                                                            typename C2<T>::t* st, int64_t R, int cw, int ns) {
  using C = typename C2<T>::t;
  __shared__ WStage<T, KC> sm;
  const DOuter o = ops[blockIdx.x];   // (leaf, depth) = (blockIdx.x / D, blockIdx.x % D)
  const C* xl = x + (int64_t)o.leaf * n0 * R;
  const int k = o.blk.k, nr = o.blk.c - k;
  const int16_t* idx = ip + o.blk.ioff;
  w_chunks<T, F, KC, NC, ADJ>(
        sm, (k + KC - 1) / KC, nr, cw, ns, xl, st + (int64_t)o.seg_off * R, R,
      [&](int ch) {
        return WChunk<F>{fp + o.blk.moff, nr, ADJ ? 1 : k, ADJ ? nr : 1, ch * KC, min(KC, k - ch * KC), 0};
      },
      [&](const WChunk<F>&, int j) { return (int32_t)idx[k + j]; },
      [&](const WChunk<F>&, int i, int64_t col) { return xl[(int64_t)idx[i] * R + col]; },
      [&](const WChunk<F>&, int i) { return (int64_t)i; });
}

template <class T, class F, bool ADJ, int KC, int NC>
__global__ void __launch_bounds__(kWThreads, w_ctas<T, NC>()) k_wapply_items(const DItem* __restrict__ items,
                                                            const int32_t* __restrict__ order, const F* __restrict__ fp,
                                                            const int16_t* __restrict__ ip, typename C2<T>::t* st,
                                                            int64_t R, int cw, int ns) {
  using C = typename C2<T>::t;
  __shared__ WStage<T, KC> sm;
  const DItem& it = items[order[blockIdx.x]];
  const int type = it.type;
  if (type == 1) {   // middle: y = S z (or z = S^H y)
    const int kr = it.b_k[0], kc = it.a_k[0];
    const int nout = ADJ ? kc : kr, nin = ADJ ? kr : kc;
    const F* S = fp + it.blk[0].moff;
    w_chunks<T, F, KC, NC, ADJ>(
        sm, (nout + KC - 1) / KC, nin, cw, ns, st + (int64_t)(ADJ ? it.b_off[0] : it.a_off[0]) * R,
        st + (int64_t)(ADJ ? it.a_off[0] : it.b_off[0]) * R, R,
        [&](int ch) { return WChunk<F>{S, nin, ADJ ? 1 : kr, ADJ ? kr : 1, ch * KC, min(KC, nout - ch * KC), 0}; },
        [&](const WChunk<F>&, int j) { return (int32_t)j; },
        [&](const WChunk<F>&, int, int64_t) { return mk<T>(0, 0); },
        [&](const WChunk<F>&, int o) { return (int64_t)o; });
    return;
  }
  const F *const M0 = fp + it.blk[0].moff, *const M1 = fp + it.blk[1].moff;
  const int16_t *const ix0 = ip + it.blk[0].ioff, *const ix1 = ip + it.blk[1].ioff;
  const int k0 = it.blk[0].k, k1 = it.blk[1].k;
  const int ka0 = it.a_k[0], c = ka0 + it.a_k[1];
  const int a0 = it.a_off[0], a1 = it.a_off[1] - ka0, b0 = it.b_off[0], b1 = it.b_off[1];
  if ((type == 0) != ADJ) {   // candidates -> skeletons: out_i = cand[q_i] + sum_j T_ij cand[p_j], both blocks
    const int n0 = (k0 + KC - 1) / KC, n1 = (k1 + KC - 1) / KC;
    w_chunks<T, F, KC, NC, ADJ>(
        sm, n0 + n1, c - min(k0, k1), cw, ns, st, st, R,
        [&](int ch) {
          const int sb = ch >= n0, kk = sb ? k1 : k0, o0 = (ch - (sb ? n0 : 0)) * KC, nr = c - kk;
          return WChunk<F>{sb ? M1 : M0, nr, ADJ ? 1 : kk, ADJ ? nr : 1, o0, min(KC, kk - o0), sb};
        },
        [&](const WChunk<F>& w, int j) {
          const int pj = w.sb ? ix1[k1 + j] : ix0[k0 + j];
          return (int32_t)((pj < ka0 ? a0 : a1) + pj);
        },
        [&](const WChunk<F>& w, int i, int64_t col) -> C {
          const int q = (w.sb ? ix1 : ix0)[i];
          return st[(int64_t)((q < ka0 ? a0 : a1) + q) * R + col];
        },
        [&](const WChunk<F>& w, int i) { return (int64_t)((w.sb ? b1 : b0) + i); });
    return;
  }
  // skeletons -> candidates.  First pass: the rows that block 0 interpolates (block 1's skeleton
  // value added where it has one) and the rows that are skeletons of both; second pass: the
  // rows that block 1 interpolates, on top of block 0's value.
  const auto row = [&](int r) { return (int64_t)((r < ka0 ? a0 : a1) + r); };
#pragma unroll 1
  for (int sb = 0; sb < 2; ++sb) {
    const int kk = sb ? k1 : k0, nr = c - kk, nch = (nr + KC - 1) / KC;
    const F* M = sb ? M1 : M0;
    const int16_t* own = sb ? ix1 : ix0;
    const int16_t* oth = (sb ? ix0 : ix1) + c;
    const int bo = sb ? b1 : b0, bx = sb ? b0 : b1;
    w_chunks<T, F, KC, NC, ADJ>(
        sm, nch + (sb == 0 ? (kk + KC - 1) / KC : 0), kk, cw, ns, st, st, R,
        [&](int ch) {
          if (ch < nch) return WChunk<F>{M, kk, ADJ ? 1 : nr, ADJ ? kk : 1, ch * KC, min(KC, nr - ch * KC), 0};
          return WChunk<F>{fp, 0, 1, 1, (ch - nch) * KC, min(KC, kk - (ch - nch) * KC), 1};
        },
        [&](const WChunk<F>&, int j) { return (int32_t)(bo + j); },
        [&](const WChunk<F>& w, int o, int64_t col) -> C {
          const int code = oth[own[w.sb ? o : kk + o]];
          C v = mk<T>(0, 0);
          if (w.sb) v = st[(int64_t)(bo + o) * R + col];
          if (code >= 0) cadd(v, st[(int64_t)(bx + code) * R + col]);
          else if (sb == 1) v = st[row(own[kk + o]) * R + col];
          return v;
        },
        [&](const WChunk<F>& w, int o) {
          const int r = own[w.sb ? o : kk + o];
          return w.sb && oth[r] < 0 ? (int64_t)-1 : row(r);
        });
    __syncthreads();   // the second pass reads what other slots wrote
  }
}

// Candidate entries r0 .. r0+KC-1 (< c) of one block added to acc: a skeleton
// entry copies y_{map r}; a redundant one sums T_{i,j(r)} y_i (U-type layout
// M[i*(c-k)+j]; VTYPE_ADJ: a V-type block in adjoint, conj(M[j*k+i])).
template <class T, class F, bool VTYPE_ADJ, int KC>
__device__ __forceinline__ void w_rows(typename C2<T>::t (&acc)[KC], const F* __restrict__ M,
                                       const int16_t* __restrict__ idx, int k, int c, const typename C2<T>::t* y,
                                       int64_t R, int64_t col, int r0, int nrow) {
  using C = typename C2<T>::t;
  const int nr = c - k;
  int code[KC];
  bool any_red = false;
#pragma unroll
  for (int ii = 0; ii < KC; ++ii) {
    code[ii] = (ii < nrow) ? idx[c + r0 + ii] : 0;
    if (ii < nrow) {
      if (code[ii] >= 0) cadd(acc[ii], y[(int64_t)code[ii] * R + col]);
      else any_red = true;
    }
  }
  if (!any_red) return;
  for (int i = 0; i < k; ++i) {
    const C yi = y[(int64_t)i * R + col];
#pragma unroll
    for (int ii = 0; ii < KC; ++ii)
      if (ii < nrow && code[ii] < 0) {
        const int j = -1 - code[ii];
        const auto m = VTYPE_ADJ ? ldf_conj<T>(M + (int64_t)j * k + i) : ldf<T>(M + (int64_t)i * nr + j);
        cfma(acc[ii], m, yi);
      }
  }
}

// y_leaf = sum_v U0_v y_0 + A_leaf x_leaf (fixed order: depths 0..D-1, then the leaf).
// Thread = (slot, column) as above, a slot takes every ns-th chunk of KC rows of the leaf; the
// coefficients are slot-uniform loads.  Slots, not a loop over the chunks: 256 leaves of 64
// rows x 40 columns in double-float are otherwise 512 warps (1.14 ms; 0.29 ms now).
template <class T, class F, bool ADJ, int KC>
__global__ void __launch_bounds__(kWThreads) k_wapply_exit(const DOuter* __restrict__ ops, int D, int64_t n0,
                                                           const F* __restrict__ fp, const int16_t* __restrict__ ip,
                                                           const F* __restrict__ leafm,
                                                           const typename C2<T>::t* __restrict__ x,
                                                           const typename C2<T>::t* st, typename C2<T>::t* y,
                                                           int64_t R, int cw, int ns) {
  using C = typename C2<T>::t;
  const int slot = threadIdx.x / cw;
  const int64_t col = (int64_t)blockIdx.y * cw + (threadIdx.x - slot * cw);
  if (col >= R) return;
  const int64_t leaf = blockIdx.x;
  const F* A = leafm + leaf * n0 * n0;
  const C* xl = x + leaf * n0 * R;
  for (int r0 = slot * KC; r0 < (int)n0; r0 += ns * KC) {
    const int nrow = ((int)n0 - r0) < KC ? ((int)n0 - r0) : KC;
    C acc[KC];
#pragma unroll
    for (int ii = 0; ii < KC; ++ii) acc[ii] = mk<T>(0, 0);
    for (int v = 0; v < D; ++v) {
      const DOuter o = ops[leaf * D + v];
      w_rows<T, F, ADJ, KC>(acc, fp + o.blk.moff, ip + o.blk.ioff, o.blk.k, o.blk.c, st + (int64_t)o.seg_off * R, R,
                        col, r0, nrow);
    }
    for (int cc = 0; cc < (int)n0; ++cc) {
      const C xv = xl[(int64_t)cc * R + col];
#pragma unroll
      for (int ii = 0; ii < KC; ++ii)
        if (ii < nrow) {
          const auto a = ADJ ? ldf_conj<T>(A + (int64_t)(r0 + ii) * n0 + cc) : ldf<T>(A + (int64_t)cc * n0 + r0 + ii);
          cfma(acc[ii], a, xv);
        }
    }
#pragma unroll
    for (int ii = 0; ii < KC; ++ii)
      if (ii < nrow) y[(leaf * n0 + r0 + ii) * R + col] = acc[ii];
  }
}

// ---------------------------------------------------------------------------
// Layout conversion kernels: column-major [R][ld] <-> [row][R] through a tile of
// kTileRows rows x up to kTileCols columns in shared memory, so that both sides are
// read and written along their contiguous index; few columns go element by element
// (below).  HBM-bound: 256 complex64 columns of 262,144 rows take 0.17 ms (1.07 GB:
// 6.2 TB/s); element by element, with one side in steps of ld, they took 1.1 ms.
// ---------------------------------------------------------------------------
constexpr int kTileRows = 64, kTileCols = 32;
// The tile of one CTA.  Column-major side: thread -> one row, every 4th column; row-major
// side: a warp -> one row, every 8th; all eight accesses of a thread are in flight together.
struct TileAt {
  int64_t row0, c0;
  int rows, cols;
};
template <class Fn>
__device__ __forceinline__ void tile_by_rows(const TileAt& t, Fn&& fn) {   // fn(step, row, column) along the rows
  const int r = threadIdx.x % kTileRows;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int c = threadIdx.x / kTileRows + 4 * i;
    if (r < t.rows && c < t.cols) fn(i, r, c);
  }
}
template <class Fn>
__device__ __forceinline__ void tile_by_cols(const TileAt& t, Fn&& fn) {   // along the columns
  const int c = threadIdx.x % kTileCols;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = threadIdx.x / kTileCols + 8 * i;
    if (r < t.rows && c < t.cols) fn(i, r, c);
  }
}
__device__ __forceinline__ TileAt tile_at(int64_t n, int64_t R, int64_t c0) {
  const int64_t row0 = (int64_t)blockIdx.x * kTileRows;
  return TileAt{row0, c0, (int)(n - row0 < kTileRows ? n - row0 : kTileRows),
                (int)(R - c0 < kTileCols ? R - c0 : kTileCols)};
}

template <class T>
__global__ void __launch_bounds__(256) k_gather_cols(const T* __restrict__ src, int64_t ld, int64_t n, int64_t R,
                                                     T* __restrict__ dst, double scale) {
  __shared__ T tile[kTileCols][kTileRows + 1];
  for (int64_t c0 = (int64_t)blockIdx.y * kTileCols; c0 < R; c0 += (int64_t)gridDim.y * kTileCols) {
    const TileAt t = tile_at(n, R, c0);
    T v[8];
    tile_by_rows(t, [&](int i, int r, int c) { v[i] = src[(t.c0 + c) * ld + t.row0 + r]; });
    if (scale != 1.0)
      tile_by_rows(t, [&](int i, int, int) {
        v[i] = T{(decltype(T::x))(scale * (double)v[i].x), (decltype(T::y))(scale * (double)v[i].y)};
      });
    tile_by_rows(t, [&](int i, int r, int c) { tile[c][r] = v[i]; });
    __syncthreads();
    tile_by_cols(t, [&](int, int r, int c) { dst[(t.row0 + r) * R + t.c0 + c] = tile[c][r]; });
    __syncthreads();
  }
}
template <class T>
__global__ void __launch_bounds__(256) k_scatter_cols(const T* __restrict__ src, int64_t n, int64_t R, T* __restrict__ dst,
                                                      int64_t ld) {
  __shared__ T tile[kTileCols][kTileRows + 1];
  for (int64_t c0 = (int64_t)blockIdx.y * kTileCols; c0 < R; c0 += (int64_t)gridDim.y * kTileCols) {
    const TileAt t = tile_at(n, R, c0);
    T v[8];
    tile_by_cols(t, [&](int i, int r, int c) { v[i] = src[(t.row0 + r) * R + t.c0 + c]; });
    tile_by_cols(t, [&](int i, int r, int c) { tile[c][r] = v[i]; });
    __syncthreads();
    tile_by_rows(t, [&](int, int r, int c) { dst[(t.c0 + c) * ld + t.row0 + r] = tile[c][r]; });
    __syncthreads();
  }
}
// r = b - y, b and r column-major, y [row][R]
__global__ void __launch_bounds__(256) k_residual_cols(const double2* b, int64_t ld, const double2* __restrict__ y,
                                                       int64_t n, int64_t R, double2* r) {
  __shared__ double2 tile[kTileCols][kTileRows + 1];
  for (int64_t c0 = (int64_t)blockIdx.y * kTileCols; c0 < R; c0 += (int64_t)gridDim.y * kTileCols) {
    const TileAt t = tile_at(n, R, c0);
    double2 v[8], w[8];
    tile_by_cols(t, [&](int i, int q, int c) { v[i] = y[(t.row0 + q) * R + t.c0 + c]; });
    tile_by_rows(t, [&](int i, int q, int c) { w[i] = b[(t.c0 + c) * ld + t.row0 + q]; });
    tile_by_cols(t, [&](int i, int q, int c) { tile[c][q] = v[i]; });
    __syncthreads();
    tile_by_rows(t, [&](int i, int q, int c) {
      const double2 u = tile[c][q];
      r[(t.c0 + c) * ld + t.row0 + q] = {w[i].x - u.x, w[i].y - u.y};
    });
    __syncthreads();
  }
}

// Few columns: element by element in the order of the row-major side, every thread busy (a tile
// of few columns leaves most threads of its row-major side idle).  262,144 rows, us, element by
// element against tiles: gather of complex128 3.8 / 19.8 (1 column), 15.0 / 22.1 (8), 18.5 / 23.5
// (10), 22.1 / 24.6 (12), 28.8 / 27.1 (16); of complex64 4.9 / 13.9 (2), 13.9 / 15.1 (10),
// 15.7 / 15.4 (12); the scatters meet at 16; residual 3.8 / 52.0 (1), 18.3 / 74.8 (8),
// 45.4 / 94.9 (20), 115 / 100 (24).
constexpr int kFewCols = 10, kFewResidual = 20;
template <class T>
__global__ void __launch_bounds__(256) k_gather_few(const T* __restrict__ src, int64_t ld, int64_t n, int64_t R,
                                                    T* __restrict__ dst, double scale) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * R; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / R, c = e - row * R;
    T v = src[c * ld + row];
    if (scale != 1.0) v = T{(decltype(T::x))(scale * (double)v.x), (decltype(T::y))(scale * (double)v.y)};
    dst[e] = v;
  }
}
template <class T>
__global__ void __launch_bounds__(256) k_scatter_few(const T* __restrict__ src, int64_t n, int64_t R, T* __restrict__ dst,
                                                     int64_t ld) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * R; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / R, c = e - row * R;
    dst[c * ld + row] = src[e];
  }
}
__global__ void __launch_bounds__(256) k_residual_few(const double2* b, int64_t ld, const double2* __restrict__ y, int64_t n,
                                                      int64_t R, double2* r) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * R; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / R, c = e - row * R;
    const double2 u = b[c * ld + row], w = y[e];
    r[c * ld + row] = {u.x - w.x, u.y - w.y};
  }
}
static inline unsigned few_grid(int64_t total) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 152 * 32)); }

static inline dim3 tile_grid(int64_t n, int64_t R) {
  const int64_t cb = (R + kTileCols - 1) / kTileCols;
  return dim3((unsigned)((n + kTileRows - 1) / kTileRows), (unsigned)(cb < 65535 ? cb : 65535));
}

int launch_gather_cols(const void* src, int t, int64_t ld, int64_t n, int64_t R, void* dst, double scale, cudaStream_t st) {
  if (R <= kFewCols) {
    if (t == 0) k_gather_few<<<few_grid(n * R), 256, 0, st>>>((const double2*)src, ld, n, R, (double2*)dst, scale);
    else k_gather_few<<<few_grid(n * R), 256, 0, st>>>((const float2*)src, ld, n, R, (float2*)dst, scale);
    return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
  }
  const dim3 g = tile_grid(n, R);
  if (t == 0) k_gather_cols<<<g, 256, 0, st>>>((const double2*)src, ld, n, R, (double2*)dst, scale);
  else k_gather_cols<<<g, 256, 0, st>>>((const float2*)src, ld, n, R, (float2*)dst, scale);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}
int launch_scatter_cols(const void* src, int t, int64_t n, int64_t R, void* dst, int64_t ld, cudaStream_t st) {
  if (R <= kFewCols) {
    if (t == 0) k_scatter_few<<<few_grid(n * R), 256, 0, st>>>((const double2*)src, n, R, (double2*)dst, ld);
    else k_scatter_few<<<few_grid(n * R), 256, 0, st>>>((const float2*)src, n, R, (float2*)dst, ld);
    return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
  }
  const dim3 g = tile_grid(n, R);
  if (t == 0) k_scatter_cols<<<g, 256, 0, st>>>((const double2*)src, n, R, (double2*)dst, ld);
  else k_scatter_cols<<<g, 256, 0, st>>>((const float2*)src, n, R, (float2*)dst, ld);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}
int launch_residual_cols(const void* b, int64_t ld, const void* y, int64_t n, int64_t R, void* r, cudaStream_t st) {
  if (R <= kFewResidual) k_residual_few<<<few_grid(n * R), 256, 0, st>>>((const double2*)b, ld, (const double2*)y, n, R, (double2*)r);
  else k_residual_cols<<<tile_grid(n, R), 256, 0, st>>>((const double2*)b, ld, (const double2*)y, n, R, (double2*)r);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <class T, class F>
static int apply_one(const DevFactor& df, bool adj, const void* xv, void* yv, void* stv, cudaStream_t s) {
  using C = typename C2<T>::t;
  const F* fp = (const F*)df.fpool;
  const C* x = (const C*)xv;
  C* y = (C*)yv;
  C* st = (C*)stv;
  const unsigned enter = (unsigned)(df.m * df.D), exit = (unsigned)df.m;
  if (!adj) k_apply_enter<T, F, false><<<enter, k1Threads, 0, s>>>(df.vout, df.n0, fp, df.ipool, x, st);
  else k_apply_enter<T, F, true><<<enter, k1Threads, 0, s>>>(df.uout, df.n0, fp, df.ipool, x, st);
  const std::vector<int32_t>& ptr = adj ? df.astep_ptr : df.step_ptr;
  const int32_t* idx = adj ? df.astep_idx : df.step_idx;
  for (int stp = 0; stp + 1 < (int)ptr.size(); ++stp) {
    const int cnt = ptr[stp + 1] - ptr[stp];
    if (cnt <= 0) continue;
    if (!adj) k_apply_items<T, F, false><<<cnt, k1Threads, 0, s>>>(df.items, idx + ptr[stp], fp, df.ipool, st);
    else k_apply_items<T, F, true><<<cnt, k1Threads, 0, s>>>(df.items, idx + ptr[stp], fp, df.ipool, st);
  }
  if (!adj) k_apply_exit<T, F, false><<<exit, 256, 0, s>>>(df.uout, df.D, df.n0, fp, df.ipool, (const F*)df.leaf, x, st, y);
  else k_apply_exit<T, F, true><<<exit, 256, 0, s>>>(df.vout, df.D, df.n0, fp, df.ipool, (const F*)df.leaf, x, st, y);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}

template <class T, class F, int RC>
static int apply_few(const DevFactor& df, bool adj, const void* xv, void* yv, int64_t R, void* stv,
                      cudaStream_t s) {
  using C = typename C2<T>::t;
  const F* fp = (const F*)df.fpool;
  const C* x = (const C*)xv;
  C* y = (C*)yv;
  C* st = (C*)stv;
  int wpb = df.D < 8 ? df.D : 8;
  if (!adj) k_few_enter<T, F, RC, false><<<(unsigned)df.m, 32 * wpb, 0, s>>>(df.vout, df.D, df.n0, fp, df.ipool, x, st, R);
  else k_few_enter<T, F, RC, true><<<(unsigned)df.m, 32 * wpb, 0, s>>>(df.uout, df.D, df.n0, fp, df.ipool, x, st, R);
  const std::vector<int32_t>& ptr = adj ? df.astep_ptr : df.step_ptr;
  const int32_t* idx = adj ? df.astep_idx : df.step_idx;
  for (int stp = 0; stp + 1 < (int)ptr.size(); ++stp) {
    int cnt = ptr[stp + 1] - ptr[stp];
    if (cnt <= 0) continue;
    int blocks = (cnt + 7) / 8;
    if (!adj) k_few_items<T, F, RC, false><<<blocks, 256, 0, s>>>(df.items, idx + ptr[stp], cnt, fp, df.ipool, st, R);
    else k_few_items<T, F, RC, true><<<blocks, 256, 0, s>>>(df.items, idx + ptr[stp], cnt, fp, df.ipool, st, R);
  }
  int thr = (int)((df.n0 + 31) / 32 * 32);
  if (thr > 256) thr = 256;
  if (!adj) k_few_exit<T, F, RC, false><<<(unsigned)df.m, thr, 0, s>>>(df.uout, df.D, df.n0, fp, df.ipool, (const F*)df.leaf, x, st, y, R);
  else k_few_exit<T, F, RC, true><<<(unsigned)df.m, thr, 0, s>>>(df.vout, df.D, df.n0, fp, df.ipool, (const F*)df.leaf, x, st, y, R);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}

// Column threads cw and slots ns of the CTAs of `ops` ops: two warps at least, and with few ops
// more slots, so that the step still fills the chip.
struct WideGrid {
  int cw, ns;
  unsigned cb;
  WideGrid(int64_t R, int NC, int64_t ops) {
    const int64_t need = (R + NC - 1) / NC;
    cw = (int)std::min<int64_t>(need, 128);
    cb = (unsigned)((need + cw - 1) / cw);
    const int64_t fill = kWFill / (std::max<int64_t>(ops, 1) * cb * cw);
    ns = (int)std::max<int64_t>((64 + cw - 1) / cw, fill);
    ns = std::min(ns, std::min(kWSlots, kWThreads / cw));
  }
  int threads() const { return cw * ns; }
};

template <class T, class F, int KC, int NC>
static void wide_items(const DevFactor& df, bool adj, typename C2<T>::t* st, int64_t R, cudaStream_t s) {
  const F* fp = (const F*)df.fpool;
  const std::vector<int32_t>& ptr = adj ? df.astep_ptr : df.step_ptr;
  const int32_t* idx = adj ? df.astep_idx : df.step_idx;
  for (int stp = 0; stp + 1 < (int)ptr.size(); ++stp) {
    const int cnt = ptr[stp + 1] - ptr[stp];
    if (cnt <= 0) continue;
    const WideGrid w(R, NC, cnt);
    const dim3 g((unsigned)cnt, w.cb);
    if (!adj) k_wapply_items<T, F, false, KC, NC><<<g, w.threads(), 0, s>>>(df.items, idx + ptr[stp], fp, df.ipool, st, R, w.cw, w.ns);
    else k_wapply_items<T, F, true, KC, NC><<<g, w.threads(), 0, s>>>(df.items, idx + ptr[stp], fp, df.ipool, st, R, w.cw, w.ns);
  }
}

template <class T, class F, int KC, int NC>
static int apply_wide_impl(const DevFactor& df, bool adj, const void* xv, void* yv, int64_t R, void* stv,
                           cudaStream_t s) {
  using C = typename C2<T>::t;
  const F* fp = (const F*)df.fpool;
  const C* x = (const C*)xv;
  C* y = (C*)yv;
  C* st = (C*)stv;
  const WideGrid w(R, NC, df.m * df.D), v(R, 1, df.m);
  const dim3 g_enter((unsigned)(df.m * df.D), w.cb), g_exit((unsigned)df.m, v.cb);
  if (!adj) k_wapply_enter<T, F, false, KC, NC><<<g_enter, w.threads(), 0, s>>>(df.vout, df.n0, fp, df.ipool, x, st, R, w.cw, w.ns);
  else k_wapply_enter<T, F, true, KC, NC><<<g_enter, w.threads(), 0, s>>>(df.uout, df.n0, fp, df.ipool, x, st, R, w.cw, w.ns);
  wide_items<T, F, KC, NC>(df, adj, st, R, s);
  constexpr int KE = NC == 2 ? 16 : 4;
  if (!adj) k_wapply_exit<T, F, false, KE><<<g_exit, v.threads(), 0, s>>>(df.uout, df.D, df.n0, fp, df.ipool, (const F*)df.leaf, x, st, y, R, v.cw, v.ns);
  else k_wapply_exit<T, F, true, KE><<<g_exit, v.threads(), 0, s>>>(df.vout, df.D, df.n0, fp, df.ipool, (const F*)df.leaf, x, st, y, R, v.cw, v.ns);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}
constexpr int kWidePairs = 64;   // FP32 columns from which a thread takes two
template <class T, class F>
static int apply_wide(const DevFactor& df, bool adj, const void* x, void* y, int64_t R, void* st, cudaStream_t s) {
  if constexpr (std::is_same<T, float>::value)
    if (R >= kWidePairs) return apply_wide_impl<T, F, 4, 2>(df, adj, x, y, R, st, s);
  return apply_wide_impl<T, F, 2, 1>(df, adj, x, y, R, st, s);
}

template <class T, class F>
static int apply_dispatch(const DevFactor& df, bool adj, const void* x, void* y, int64_t R, void* st,
                          cudaStream_t s) {
  if constexpr (std::is_same<T, float>::value) {
    if (R > 1 && R <= 4) return apply_few<T, F, 4>(df, adj, x, y, R, st, s);
    if (R > 1 && R <= kFewMax) return apply_few<T, F, 8>(df, adj, x, y, R, st, s);
  }
  if (R > 1) return apply_wide<T, F>(df, adj, x, y, R, st, s);
  return apply_one<T, F>(df, adj, x, y, st, s);   // (the persistent kernel is tried first, in launch_apply)
}

// Forward many-column apply of the split-BF16 form: entry and exit contractions on the
// tensor cores (hb_tc.cu), the inner butterfly items on CUDA cores in complex FP32.
static int apply_wide_tc(const DevFactor& df, const void* xv, void* yv, int64_t R, void* stv, cudaStream_t s) {
  int rc = launch_tc_jobs(df, false, xv, stv, nullptr, R, s);
  if (rc) return rc;
  if (R >= kWidePairs) wide_items<float, float2, 4, 2>(df, false, (float2*)stv, R, s);
  else wide_items<float, float2, 2, 1>(df, false, (float2*)stv, R, s);
  if (cudaGetLastError() != cudaSuccess) return HB_ECUDA;
  return launch_tc_jobs(df, true, xv, stv, yv, R, s);
}

// double2 <-> double-float vectors
__global__ void k_to_dd(const double2* __restrict__ x, DdC* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = x[i];
    const float rh = (float)v.x, ih = (float)v.y;
    y[i] = DdC{Dd(rh, (float)(v.x - (double)rh)), Dd(ih, (float)(v.y - (double)ih))};
  }
}
__global__ void k_from_dd(const DdC* __restrict__ x, double2* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const DdC v = x[i];
    y[i] = make_double2((double)v.x.h + (double)v.x.l, (double)v.y.h + (double)v.y.l);
  }
}

constexpr int kWideMin = 32;   // columns from which the FP64-accurate and the tensor-core applies pay
bool apply_dd_ready(int64_t R) { return R >= kWideMin; }

int launch_apply_dd(const DevFactor& df, bool adjoint, const void* x, void* y, int64_t R, void* state, void* xdd,
                    void* ydd, cudaStream_t st) {
  if (!apply_dd_ready(R) || df.form == HB_C128) return HB_EINVAL;
  const int64_t nn = df.n * R;
  const unsigned g = (unsigned)std::min<int64_t>((nn + 255) / 256, 152 * 16);
  k_to_dd<<<g, 256, 0, st>>>((const double2*)x, (DdC*)xdd, nn);
  int rc = apply_wide<Dd, float2>(df, adjoint, xdd, ydd, R, state, st);
  if (rc) return rc;
  k_from_dd<<<g, 256, 0, st>>>((const DdC*)ydd, (double2*)y, nn);
  return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ECUDA;
}

int launch_apply(const DevFactor& df, Prec p, bool adjoint, const void* x, void* y, int64_t R, void* state,
                 cudaStream_t st) {
  if (R == 1 && apply1_ready(df, adjoint)) return launch_apply1(df, p, adjoint, x, y, state, st);
  if (p == PREC_F32 && !adjoint && R >= kWideMin && df.form == HB_SPLIT_BF16 && df.tc_ok)
    return apply_wide_tc(df, x, y, R, state, st);
  if (p == PREC_F64) return apply_dispatch<double, double2>(df, adjoint, x, y, R, state, st);
  if (p == PREC_F32) return apply_dispatch<float, float2>(df, adjoint, x, y, R, state, st);
  return apply_dispatch<double, float2>(df, adjoint, x, y, R, state, st);
}

}  // namespace hb
