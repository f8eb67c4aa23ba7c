// One site per CTA of eight warps, one hop block per warp (FP32 / BF16 blocks, FP32 vectors): the layout of
// the half apply and of the full stencil for lattices whose sites do not fill the chip by themselves.
//
// With one or two warps per site a warp walks 9 or 4.5 blocks one after another and a site takes as many
// memory latencies; below some 10^4 sites too few warps are left to hide them.  Here every block of the site
// is on its way at once: warp w reads hop block w (w < 4: F_{x,mu} for v_{x+mu}, else F_{x-mu,mu} for
// v_{x-mu}, mu = w & 3) and its share of the diagonal block's rows, and the eight partial sums meet in shared
// memory (fixed order).  Pull only: a forward block is read a second time, from L2, by the site in front of
// it.
#pragma once

#include "apply_core.cuh"
#include "common.cuh"

namespace coarse {

constexpr int kS8 = 8;  // warps

// Sum over the 8 lanes t of a row group of R = n/4 rows per lane, 2 R floats halved at each exchange;
// every row of the group ends complete in one lane, which writes it: out[4 r + g].
template <int KR>
__device__ __forceinline__ void s8_rows(float2 (&y)[KR], float2* out, int lane) {
  const int g = lane >> 3, t = lane & 7;
  // rows are dealt over the lanes: bit 0 of t picks the row parity, then the next halves as far as they go
  constexpr int H1 = (KR + 1) / 2;
  float2 a[H1];
#pragma unroll
  for (int i = 0; i < H1; ++i) {
    const float2 lo = y[2 * i], hi = y[2 * i + 1];
    const float2 keep = (t & 1) ? hi : lo, send = (t & 1) ? lo : hi;
    a[i].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 1);
    a[i].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 1);
  }
  constexpr int H2 = H1 / 2;
  float2 b[H2];
#pragma unroll
  for (int i = 0; i < H2; ++i) {
    const float2 lo = a[2 * i], hi = a[2 * i + 1];
    const float2 keep = (t & 2) ? hi : lo, send = (t & 2) ? lo : hi;
    b[i].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 2);
    b[i].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 2);
  }
#pragma unroll
  for (int i = 0; i < H2; ++i) {
    b[i].x += __shfl_xor_sync(0xffffffffu, b[i].x, 4);
    b[i].y += __shfl_xor_sync(0xffffffffu, b[i].y, 4);
  }
  if (t < 4)
#pragma unroll
    for (int i = 0; i < H2; ++i) out[4 * (4 * i + t) + g] = b[i];  // row r = 4 i + 2 (t >> 1) + (t & 1)
}

// Products of the warp's hop block into hp[warp][n]; sigma3 flips: in = operand, out = result.
template <int N, class BT>
__device__ __forceinline__ void s8_fwd(const BT* blk, const float2* v, bool flip, float2* out, int lane) {
  constexpr int CPL = N / 8, KR = N / 4;
  const int g = lane >> 3, t = lane & 7;
  float2 w[CPL], y[KR];
  load_vec<float2, float2, CPL>(v + t * CPL, w);
  if (flip && t * CPL >= N / 2)
#pragma unroll
    for (int c = 0; c < CPL; ++c) w[c] = make_float2(-w[c].x, -w[c].y);
#pragma unroll
  for (int r = 0; r < KR; ++r) {
    float2 e[CPL];
    LoadS<float2, BT>::template row<CPL>(blk + (4 * r + g) * N + t * CPL, e);
    y[r] = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < CPL; ++c) cfma(y[r], e[c], w[c]);
  }
  if (flip)
#pragma unroll
    for (int r = 0; r < KR; ++r)
      if (4 * r + g >= N / 2) y[r] = make_float2(-y[r].x, -y[r].y);
  s8_rows<KR>(y, out, lane);
}

template <int N, class BT>
__device__ __forceinline__ void s8_bwd(const BT* blk, const float2* v, bool flip, float2* out, int lane) {
  constexpr int CPL = N / 8, KR = N / 4;
  const int g = lane >> 3, t = lane & 7;
  float2 y[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) y[c] = make_float2(0.f, 0.f);
#pragma unroll
  for (int r = 0; r < KR; ++r) {
    float2 e[CPL];
    LoadS<float2, BT>::template row<CPL>(blk + (4 * r + g) * N + t * CPL, e);
    float2 x = v[4 * r + g];
    if (flip && 4 * r + g >= N / 2) x = make_float2(-x.x, -x.y);
#pragma unroll
    for (int c = 0; c < CPL; ++c) cfma_conj(y[c], e[c], x);
  }
  // sum over the four row groups: lanes 8 apart trade column halves
  constexpr int H = CPL / 2;
  const bool o = g & 1;
  const float sg = flip && t * CPL >= N / 2 ? -1.f : 1.f;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const float2 keep = o ? y[H + i] : y[i], send = o ? y[i] : y[H + i];
    float2 a;
    a.x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 8);
    a.y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 8);
    a.x += __shfl_xor_sync(0xffffffffu, a.x, 16);
    a.y += __shfl_xor_sync(0xffffffffu, a.y, 16);
    if (g < 2) out[t * CPL + o * H + i] = cscale(a, sg);
  }
}

// The diagonal-type block (self block, inverse) split over the warps by row quads 4 q + g, q = warp,
// warp + 8: loaded early, multiplied when its operand is there.
template <int N, class BT>
struct S8Diag {
  static constexpr int CPL = N / 8, KR = N / 4, Q = (KR + kS8 - 1) / kS8;
  float2 e[Q][CPL];
  __device__ __forceinline__ void load(const BT* blk, int warp, int lane) {
    const int g = lane >> 3, t = lane & 7;
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (warp + kS8 * i < KR) LoadS<float2, BT>::template row<CPL>(blk + (4 * (warp + kS8 * i) + g) * N + t * CPL, e[i]);
  }
  // w: the operand's columns of this lane; out[row]
  __device__ __forceinline__ void mul(const float2 (&w)[CPL], float2* out, int warp, int lane) const {
    const int g = lane >> 3, t = lane & 7;
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (warp + kS8 * i < KR) {  // warp-uniform
        float2 u = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < CPL; ++c) cfma(u, e[i][c], w[c]);
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) {
          u.x += __shfl_xor_sync(0xffffffffu, u.x, off);
          u.y += __shfl_xor_sync(0xffffffffu, u.y, off);
        }
        if (t == 0) out[4 * (warp + kS8 * i) + g] = u;
      }
  }
};

// Epilogue of one entry: r = S x or D x, xs = x, ac = the accumulator's old value (POLY).
__device__ __forceinline__ void s8_finish(int mode, float2 r, float2 xs, float2 ac, const double2* coef, float2* y,
                                          float2* acc) {
  if (mode == APPLY_PLAIN) {
    *y = r;
    return;
  }
  const double2 c0d = coef[0], c1d = coef[1];
  const float2 c0 = make_float2((float)c0d.x, (float)c0d.y), c1 = make_float2((float)c1d.x, (float)c1d.y);
  if (mode == APPLY_POLY_FIRST) {
    const double2 c2d = coef[2];
    ac = cmul(make_float2((float)c2d.x, (float)c2d.y), xs);
  }
  const float2 sp = csub(xs, cmul(c0, r));
  *y = sp;
  *acc = cadd(ac, cmul(c1, sp));
}

}  // namespace coarse
