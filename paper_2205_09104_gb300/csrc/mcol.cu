// Multi-column stencil and half apply: the columns that share an operator are multiplied together, so that a block is
// read once for all of them instead of once per column.  The FP32 blocks' kernels and the full BF16 stencil run on the
// FP32 pipe (below), the half apply with BF16 blocks on the tensor cores (kb_eo_mma).
//
// With R columns the block traffic per column falls by R and the FP32 rate bounds the product from about
// four columns on (72 n^2 flops per site and column against 40 n^2 bytes of FP32 or 20 n^2 bytes of BF16
// blocks per site).  So the kernel is built around packed FP32 multiply-adds (two per instruction,
// __ffma2_rn): a warp holds a piece of a block in registers (16 rows, or 16 columns for the transposed
// product) and runs over the columns, whose entries it reads from shared memory two at a time (the
// registers that shared memory returns are the next bound: with the entries stored already duplicated for
// the packed operand, 16 bytes each, the load pipe was 81% busy and the FMA pipe 37%).  The next
// piece is loaded meanwhile.
//
// One CTA of four warps per output site: warp mu multiplies the forward block F_{x,mu} by v_{x+mu} and the
// backward block sigma3 F_{x-mu,mu}^H sigma3 by v_{x-mu}; the four partial sums meet in shared memory and
// are added in a fixed order.  The half apply then multiplies by the site's inverse block, the full
// stencil has added the self block, and the epilogue runs over the CTA.  Pull only: no scratch, no
// counters.
#include <algorithm>

#include "apply_core.cuh"
#include "common.cuh"
#include "batch.cuh"
#include "mcol.cuh"
#include "oddeven.cuh"
#include "site8.cuh"

namespace coarse {
namespace {

constexpr int kMW = 4;  // warps per site

// A piece of a block in registers: raw as loaded, entries as (re, im) pairs.
//   rows:    rows r0 + g, r0 + g + 8 (g = lane / 4), columns split over the 4 lanes t of a row
//   columns: rows 8 (k / 2) + 2 g + k % 2 (g = lane / 8), columns c0 + 2 t, c0 + 2 t + 1 (t = lane % 8)
template <int N, class BT> struct Piece;
template <int N> struct Piece<N, float2> {
  static constexpr int Q = N / 4;  // entries per row and lane (rows), rows per lane (columns)
  float4 v[Q];
  __device__ __forceinline__ void load_rows(const float2* b, int r0, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int m = 0; m < Q / 2; ++m)
        v[h * (Q / 2) + m] = __ldg(reinterpret_cast<const float4*>(b + (r0 + g + 8 * h) * N + 2 * (t + 4 * m)));
  }
  __device__ __forceinline__ void load_cols(const float2* b, int c0, int lane) {
    const int g = lane >> 3, t = lane & 7;
#pragma unroll
    for (int k = 0; k < Q; ++k) v[k] = __ldg(reinterpret_cast<const float4*>(b + (8 * (k >> 1) + 2 * g + (k & 1)) * N + c0 + 2 * t));
  }
  static __device__ __forceinline__ int col(int q, int t) { return 2 * (t + 4 * (q >> 1)) + (q & 1); }
  __device__ __forceinline__ float2 row_entry(int h, int q) const {
    const float4 e = v[h * (Q / 2) + (q >> 1)];
    return (q & 1) ? make_float2(e.z, e.w) : make_float2(e.x, e.y);
  }
  __device__ __forceinline__ float2 col_entry(int k, int j) const {
    return j ? make_float2(v[k].z, v[k].w) : make_float2(v[k].x, v[k].y);
  }
};
template <int N> struct Piece<N, cbf16> {
  static constexpr int Q = N / 4;
  uint32_t v[2 * Q];
  __device__ __forceinline__ void load_rows(const cbf16* b, int r0, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int m = 0; m < Q / 4; ++m) {
        const uint4 u = __ldg(reinterpret_cast<const uint4*>(b + (r0 + g + 8 * h) * N + 4 * (t + 4 * m)));
        uint32_t* o = v + h * Q + 4 * m;
        o[0] = u.x;
        o[1] = u.y;
        o[2] = u.z;
        o[3] = u.w;
      }
  }
  __device__ __forceinline__ void load_cols(const cbf16* b, int c0, int lane) {
    const int g = lane >> 3, t = lane & 7;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(b + (8 * (k >> 1) + 2 * g + (k & 1)) * N + c0 + 2 * t));
      v[2 * k] = u.x;
      v[2 * k + 1] = u.y;
    }
  }
  static __device__ __forceinline__ int col(int q, int t) { return 4 * (t + 4 * (q >> 2)) + (q & 3); }
  __device__ __forceinline__ float2 row_entry(int h, int q) const { return bf2f(v[h * Q + q]); }
  __device__ __forceinline__ float2 col_entry(int k, int j) const { return bf2f(v[2 * k + j]); }
};

// out[c][row] (=, += if ADD) sum_j block[row][j] w[c][j] over the piece's 16 rows, columns c0, c0 + cs, ...;
// the result's rows of the second chirality are negated if `flip`
template <int N, class BT, bool ADD>
__device__ __forceinline__ void mul_rows(const Piece<N, BT>& p, const float2* tab, float* out, int r0, int c0, int cs,
                                         int R, bool flip, int lane) {
  // sigma3 of the operand: the second chirality's columns come first, then the sums change sign once; where a lane's
  // columns do not divide so, the entries change sign
  constexpr bool kFlips = sizeof(BT) == 8;  // columns of entry q >= N/2 for every lane or for none
  constexpr int Q = N / 4;
  const int g = lane >> 2, t = lane & 3;
  float2 e[2][Q];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < Q; ++q) e[h][q] = p.row_entry(h, q);
  const int row = r0 + g + 8 * (t & 1);
  const float sg = flip && row >= N / 2 ? -1.f : 1.f;
#pragma unroll 1
  for (int c = c0; c < R; c += cs) {
    const float2* w = tab + c * N;
    float2 F1[2], F2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) F1[h] = F2[h] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < Q; i += 2) {
      const int q = kFlips ? (i + Q / 2) % Q : i;  // entries q, q + 1 are neighbours
      if (kFlips && i == Q / 2 && flip)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          F1[h] = make_float2(-F1[h].x, -F1[h].y);
          F2[h] = make_float2(-F2[h].x, -F2[h].y);
        }
      float4 ww = *reinterpret_cast<const float4*>(w + Piece<N, BT>::col(q, t));
      if (!kFlips && flip && Piece<N, BT>::col(q, t) >= N / 2) ww = make_float4(-ww.x, -ww.y, -ww.z, -ww.w);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        F1[h] = __ffma2_rn(e[h][q], make_float2(ww.x, ww.x), F1[h]);
        F2[h] = __ffma2_rn(e[h][q], make_float2(ww.y, ww.y), F2[h]);
        F1[h] = __ffma2_rn(e[h][q + 1], make_float2(ww.z, ww.z), F1[h]);
        F2[h] = __ffma2_rn(e[h][q + 1], make_float2(ww.w, ww.w), F2[h]);
      }
    }
    float re[2], im[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      re[h] = F1[h].x - F2[h].y;
      im[h] = F2[h].x + F1[h].y;
    }
    // sum over the row's four lanes: lanes t ^ 1 trade rows, lanes t ^ 2 trade parts
    const bool o1 = t & 1, o2 = t & 2;
    const float ar = (o1 ? re[1] : re[0]) + __shfl_xor_sync(0xffffffffu, o1 ? re[0] : re[1], 1);
    const float ai = (o1 ? im[1] : im[0]) + __shfl_xor_sync(0xffffffffu, o1 ? im[0] : im[1], 1);
    const float y = sg * ((o2 ? ai : ar) + __shfl_xor_sync(0xffffffffu, o2 ? ar : ai, 2));
    float* o = out + c * 2 * N + 2 * row + (t >> 1);
    *o = ADD ? *o + y : y;
  }
}

// out[c][col] += sum_i conj(block[i][col]) w[c][i] over the piece's 16 columns
template <int N, class BT>
__device__ __forceinline__ void mul_cols(const Piece<N, BT>& p, const float2* tab, float* out, int j0, int R, bool flip,
                                         int lane) {
  constexpr int Q = N / 4;
  const int g = lane >> 3, t = lane & 7;
  float2 e[Q][2];
#pragma unroll
  for (int k = 0; k < Q; ++k)
#pragma unroll
    for (int j = 0; j < 2; ++j) e[k][j] = p.col_entry(k, j);
  const int col = j0 + 2 * t + (g & 1);
  const float sg = flip && col >= N / 2 ? -1.f : 1.f;
#pragma unroll 1
  for (int c = 0; c < R; ++c) {
    const float2* w = tab + c * N + 2 * g;
    float2 B1[2], B2[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) B1[j] = B2[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < Q; i += 2) {
      const int k = (i + Q / 2) % Q;  // rows of the second chirality first (sigma3 of the operand)
      if (i == Q / 2 && flip)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          B1[j] = make_float2(-B1[j].x, -B1[j].y);
          B2[j] = make_float2(-B2[j].x, -B2[j].y);
        }
      const float4 ww = *reinterpret_cast<const float4*>(w + 4 * k);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        B1[j] = __ffma2_rn(e[k][j], make_float2(ww.x, ww.x), B1[j]);
        B2[j] = __ffma2_rn(e[k][j], make_float2(ww.y, ww.y), B2[j]);
        B1[j] = __ffma2_rn(e[k + 1][j], make_float2(ww.z, ww.z), B1[j]);
        B2[j] = __ffma2_rn(e[k + 1][j], make_float2(ww.w, ww.w), B2[j]);
      }
    }
    float re[2], im[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      re[j] = B1[j].x + B2[j].y;
      im[j] = B2[j].x - B1[j].y;
    }
    const bool o1 = g & 1, o2 = g & 2;
    const float ar = (o1 ? re[1] : re[0]) + __shfl_xor_sync(0xffffffffu, o1 ? re[0] : re[1], 8);
    const float ai = (o1 ? im[1] : im[0]) + __shfl_xor_sync(0xffffffffu, o1 ? im[0] : im[1], 8);
    const float y = sg * ((o2 ? ai : ar) + __shfl_xor_sync(0xffffffffu, o2 ? ar : ai, 16));
    out[c * 2 * N + 2 * col + (g >> 1)] += y;
  }
}

// Shared memory of one CTA: per warp the forward hop's vectors of R columns, the backward hop's, the sums.
template <int N> constexpr size_t mc_smem(int R) { return (size_t)kMW * R * N * 3 * sizeof(float2); }

// One site: nbr[mu] = {source of the forward hop, site owning the backward block, source of the backward
// hop}, sources as offsets into the columns; blk: hop blocks start at blk + (site * 5 + 1) n^2.
struct McSite {
  const void* blocks;
  int x;            // site
  int R;
  int adj;          // D^H = sigma3 D sigma3 on the forward hops' side
};

// The R columns' entries at `off` into tab[column][N], by asynchronous copies (a loop of loads and stores would
// expose one memory latency per round).
template <int N>
__device__ __forceinline__ void fill_table(float2* tab, const float2* const* vp, size_t off, int R, int lane) {
  for (int i = lane; i < R * (N / 2); i += 32) {
    const int c = i / (N / 2), e = 2 * (i % (N / 2));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(tab + c * N + e)),
                 "l"(vp[c] + off + e)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// The two hops of the warp's direction into hp[c][row] of the warp; `tail` receives the warp's piece of the
// block that is multiplied after the hops (null: none), loaded behind the last piece of the hops.
template <int N, class BT>
__device__ __forceinline__ void mc_hops(const McSite& s, int mu, const int4 rec, const float2* const* vp, float2* tab,
                                        float* hp, const BT* tail_blk, Piece<N, BT>& tail, int lane) {
  constexpr int NP = N / 16;
  constexpr size_t BSZ = (size_t)N * N;
  const BT* B = static_cast<const BT*>(s.blocks);
  const BT* fb = B + ((size_t)s.x * 5 + 1 + mu) * BSZ;
  const BT* bb = B + ((size_t)rec.y * 5 + 1 + mu) * BSZ;
  Piece<N, BT> p, nx;
  p.load_rows(fb, 0, lane);
  float2* tab2 = tab + (size_t)kMW * s.R * N;
  fill_table<N>(tab, vp, (size_t)rec.x * N, s.R, lane);
  fill_table<N>(tab2, vp, (size_t)rec.z * N, s.R, lane);
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncwarp();
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    if (k + 1 < NP) nx.load_rows(fb, 16 * (k + 1), lane);
    else nx.load_cols(bb, 0, lane);
    mul_rows<N, BT, false>(p, tab, hp, 16 * k, 0, 1, s.R, s.adj, lane);
    p = nx;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    if (k + 1 < NP) nx.load_cols(bb, 16 * (k + 1), lane);
    else if (tail_blk) tail.load_rows(tail_blk, 16 * (mu % NP), lane);
    mul_cols<N, BT>(p, tab2, hp, 16 * k, s.R, !s.adj, lane);
    if (k + 1 < NP) p = nx;
  }
  __syncwarp();
}

// block * w of all columns, the block's 16-row pieces (and the columns) dealt to the four warps: `p` is
// the warp's piece, rows 16 (warp % (N / 16))
template <int N, class BT, bool ADD>
__device__ __forceinline__ void mc_block(const Piece<N, BT>& p, const float2* tab, float* out, int R, bool flip,
                                         int warp, int lane) {
  constexpr int NP = N / 16, CS = kMW / NP;
  if (warp < NP * CS) mul_rows<N, BT, ADD>(p, tab, out, 16 * (warp % NP), warp / NP, CS, R, flip, lane);
}

// The vectors of a chunk's columns whose gate is open, gathered once per CTA in one round of loads (the
// latency of a chain of descriptor loads would otherwise be most of a small site's time).
struct McPtrs {
  const float2* v[kMcCols];
  const float2* z[kMcCols];
  const float2* base[kMcCols];
  float2* y[kMcCols];
  float2* acc[kMcCols];
  const double2* coef[kMcCols];
  float mu[kMcCols];
  int n;
};

// by the whole CTA; returns the number of columns
__device__ __forceinline__ int mc_setup(McPtrs& P, const McPhase& p, const McItem& it) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x, q = it.s0 + lane;
    const int step = *p.step;
    const bool in = lane < it.cols;
    char* base = in ? p.vbase[q] : nullptr;
    const double2* coef = in ? p.S[q].polyc : nullptr;
    const double mu = in ? p.S[q].mu : 0.0;
    const bool on = in && mc_gate(p, q);
    const uint32_t m = __ballot_sync(0xffffffffu, on);
    if (on) {
      const int at = __popc(m & ((1u << lane) - 1u));
      auto vec = [&](int sel) {
        return sel == BS_NONE ? nullptr : reinterpret_cast<float2*>(base + batch_vec_offset(sel, step, p.m, it.vb));
      };
      P.v[at] = vec(p.vsel);
      P.z[at] = vec(p.zsel);
      P.base[at] = vec(p.bsel);
      P.y[at] = vec(p.ysel);
      P.acc[at] = vec(BS_ACC);
      P.coef[at] = coef + p.coef_off;
      P.mu[at] = (float)mu;
    }
    if (lane == 0) P.n = __popc(m);
  }
  __syncthreads();
  return P.n;
}

__device__ __forceinline__ McItem load_item(const McItem* p) {
  McItem it;
  const int4 a = __ldg(reinterpret_cast<const int4*>(p));
  const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(p) + 1);
  it.s0 = a.x;
  it.cols = a.y;
  it.q = a.z;
  it.nh = a.w;
  it.rec = reinterpret_cast<const int4*>(b.x);
  it.vb = b.y;
  return it;
}

// The epilogue's operands of this thread's entries (thread + k * threads of [column][N]), loaded together.
template <int N>
struct McTail {
  static constexpr int IT = (kMcCols * N + 32 * kMW - 1) / (32 * kMW);
  float2 xs[IT], ac[IT];
  __device__ __forceinline__ void load(const McPtrs& P, const McPhase& b, size_t off, int R) {
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int i = threadIdx.x + 32 * kMW * k, c = i / N;
      xs[k] = ac[k] = make_float2(0.f, 0.f);
      if (i < R * N && b.bsel != BS_NONE) xs[k] = P.base[c][off + i % N];
      if (i < R * N && b.mode == APPLY_POLY) ac[k] = P.acc[c][off + i % N];
    }
  }
  // u[column][N]: the inverse block's product
  __device__ __forceinline__ void finish(const McPtrs& P, const McPhase& b, size_t off, int R, const float2* u) const {
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int i = threadIdx.x + 32 * kMW * k, c = i / N;
      if (i >= R * N) break;
      const size_t idx = off + i % N;
      const float2 r = b.bsel != BS_NONE ? csub(xs[k], u[i]) : u[i];
      s8_finish(b.mode, r, xs[k], ac[k], P.coef[c], P.y[c] + idx, P.acc[c] + idx);
    }
  }
};

// Batched half apply: CTA -> (operator's column chunk, output site); columns whose gate is closed drop out.
template <int N, class BT>
__global__ void __launch_bounds__(32 * kMW) kb_eo_mc(const __grid_constant__ McPhase b) {
  extern __shared__ __align__(16) unsigned char mc_sm[];
  __shared__ McPtrs P;
  const McItem it = load_item(b.items + blockIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int4 rec = __ldg(it.rec + ((size_t)b.out_par * it.nh + it.q) * 4 + warp);
  const BSolve& s0 = b.S[it.s0];
  const BT* B = static_cast<const BT*>(b.poly_blocks ? s0.blk_poly : s0.blk);
  const BT* inv = static_cast<const BT*>(b.poly_blocks ? s0.inv_poly : s0.inv) + (size_t)rec.w * N * N;
  const int R = mc_setup(P, b, it);
  if (R == 0) return;
  float2* tabs = reinterpret_cast<float2*>(mc_sm);
  float* hp = reinterpret_cast<float*>(tabs + (size_t)2 * kMW * R * N);  // [warp][column][2 row + part]
  McSite s;
  s.blocks = B;
  s.x = rec.w;
  s.R = R;
  s.adj = 0;
  Piece<N, BT> tail;
  if (b.vsel != BS_NONE) {
    mc_hops<N, BT>(s, warp, rec, P.v, tabs + (size_t)warp * R * N, hp + (size_t)warp * R * 2 * N, inv, tail, lane);
    __syncthreads();
  } else {
    tail.load_rows(inv, 16 * (warp % (N / 16)), lane);
  }
  // g = z - h (or h): the operand of the inverse block
  const size_t off = (size_t)it.q * N;
  for (int i = threadIdx.x; i < R * N; i += blockDim.x) {
    const int c = i / N, e = i % N;
    float2 g = make_float2(0.f, 0.f);
    if (b.vsel != BS_NONE) {
      const float2* h = reinterpret_cast<const float2*>(hp) + i;
      g = cadd(cadd(h[0], h[(size_t)R * N]), cadd(h[(size_t)2 * R * N], h[(size_t)3 * R * N]));
    }
    if (b.zsel != BS_NONE) g = csub(P.z[c][off + e], g);
    tabs[i] = g;
  }
  McTail<N> ends;
  ends.load(P, b, off, R);
  __syncthreads();
  mc_block<N, BT, false>(tail, tabs, hp, R, false, warp, lane);
  __syncthreads();
  ends.finish(P, b, off, R, reinterpret_cast<const float2*>(hp));
}

// ------------------------------------------------------------- BF16 blocks on the tensor cores
// Half apply with BF16 blocks for the columns of one operator: mma.sync m16n8k16, the block tile as A (real
// and imaginary planes), four complex columns as B (n = 8: re, im of each).  An FP32 entry of a column is
// the exact sum of three BF16 numbers, so three products per plane keep the columns' full precision; the
// products are exact and summed in FP32, per block, and the blocks are added on the FP32 pipe.
//
// Index orders inside a 16-tile are chosen for the loads: k = 2t, 2t+1, 2t+8, 2t+9 of the fragment are
// entries 4t .. 4t+3, rows g, g+8 are rows 2g, 2g+1; a lane reads its part of a forward tile with two
// 16-byte loads from the row-major block, of a transposed tile with four 8-byte loads.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

constexpr int kMmaTiles = kMcCols / 4;  // column tiles of one pass
// Split table of one hop: [column tile][split][8 rows (column, part)][N], rows padded to an odd number of
// 16-byte units (conflict-free ldmatrix).  A row holds the entries 4i, 4i + 1 of all i, then 4i + 2, 4i + 3, so
// that the lanes of a fill, four entries each, write neighbouring words.
template <int N> constexpr int split_row() { return 2 * N + 16; }
template <int N> constexpr int split_tile() { return 3 * 8 * split_row<N>(); }
template <int N> constexpr size_t mma_smem(int R) {
  return (size_t)kMW * (((R + 3) / 4) * split_tile<N>() + (size_t)R * N * sizeof(float2));
}

// (v0, v1) = h + m + l exactly, each part a BF16 pair.  From the largest BF16 number on (3.39e38) h overflows and the
// other parts are NaN, as for infinities: the cycle reports either as non-finite.
__device__ __forceinline__ void split3(float v0, float v1, uint32_t (&o)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
    o[k] = *reinterpret_cast<const uint32_t*>(&h);
    v0 -= __uint_as_float(o[k] << 16);
    v1 -= __uint_as_float(o[k] & 0xffff0000u);
  }
}

// entries j .. j + 3 (j a multiple of 4) of column c
template <int N>
__device__ __forceinline__ void put_split(unsigned char* tab, int c, int j, const float2 (&v)[4]) {
  unsigned char* o = tab + (c >> 2) * split_tile<N>() + 2 * (c & 3) * split_row<N>() + j;
  uint32_t a[3], b[3];
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    split3(part ? v[0].y : v[0].x, part ? v[1].y : v[1].x, a);
    split3(part ? v[2].y : v[2].x, part ? v[3].y : v[3].x, b);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      *reinterpret_cast<uint32_t*>(o + (k * 8 + part) * split_row<N>()) = a[k];
      *reinterpret_cast<uint32_t*>(o + (k * 8 + part) * split_row<N>() + N) = b[k];
    }
  }
}

template <int N>
__device__ __forceinline__ void fill_split(unsigned char* tab, const float2* const* vp, size_t off, int R, bool flip,
                                           int lane) {
  constexpr int IT = (kMcCols * (N / 4) + 31) / 32;
  float4 u[IT], w[IT];
#pragma unroll
  for (int k = 0; k < IT; ++k) {  // every load on its way before the first is used
    const int i = lane + 32 * k, c = i / (N / 4), j = 4 * (i % (N / 4));
    if (i < R * (N / 4)) {
      const float4* p = reinterpret_cast<const float4*>(vp[c] + off + j);
      u[k] = p[0];
      w[k] = p[1];
    }
  }
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int i = lane + 32 * k, c = i / (N / 4), j = 4 * (i % (N / 4));
    if (i < R * (N / 4)) {
      float2 v[4] = {make_float2(u[k].x, u[k].y), make_float2(u[k].z, u[k].w), make_float2(w[k].x, w[k].y),
                     make_float2(w[k].z, w[k].w)};
      if (flip && j >= N / 2)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = make_float2(-v[q].x, -v[q].y);
      put_split<N>(tab, c, j, v);
    }
  }
}

// Tile (rt, K) of a block, or of its transpose, in registers as loaded: words [4 h + e] of the A fragment's
// rows 2g + h and entries 4t + e.
template <int N, bool BWD>
__device__ __forceinline__ void load_tile(uint32_t (&u)[8], const cbf16* blk, int rt, int K, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const uint32_t* b = reinterpret_cast<const uint32_t*>(blk);
  if (!BWD) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(b + (16 * rt + 2 * g + h) * N + 16 * K + 4 * t));
      u[4 * h] = v.x;
      u[4 * h + 1] = v.y;
      u[4 * h + 2] = v.z;
      u[4 * h + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(b + (16 * K + 4 * t + q) * N + 16 * rt + 2 * g));
      u[q] = v.x;
      u[4 + q] = v.y;
    }
  }
}

template <int N>
__device__ __forceinline__ uint32_t lane_row(uint32_t tab, int lane) {
  return tab + (uint32_t)(((lane >> 4) * 8 + (lane & 7)) * split_row<N>() + ((lane >> 3) & 1) * N);
}

// d[ct][plane] += tile times the columns' splits (= if FIRST).  The tensor core truncates its sums, so a step's
// three products, the smallest part of the columns first, start from zero and the steps meet on the FP32 pipe: a
// chain through all steps of a block had 2.2 times the FP32 kernels' error at n = 48 (measured at the dispatch).
template <int N, bool FIRST>
__device__ __forceinline__ void mul_tile(const uint32_t (&u)[8], uint32_t lrow, int K, int T,
                                         float (&d)[kMmaTiles][2][4]) {
  uint32_t re[4], im[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // rows 2g, 2g + 1 x entries 4t, 4t + 1, then 4t + 2, 4t + 3
    const int i = 4 * (k & 1) + 2 * (k >> 1);
    re[k] = __byte_perm(u[i], u[i + 1], 0x5410);
    im[k] = __byte_perm(u[i], u[i + 1], 0x7632);
  }
#pragma unroll
  for (int ct = 0; ct < kMmaTiles; ++ct)
    if (ct < T) {
      const uint32_t addr = lrow + ct * split_tile<N>() + K * 16;
      uint32_t b[4], c[2];
      asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
                   : "=r"(c[0]), "=r"(c[1])
                   : "r"(addr + 16 * split_row<N>()));
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                   : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                   : "r"(addr));
      float e[2][4] = {};
      mma_bf16(e[0], re, c[0], c[1]);
      mma_bf16(e[1], im, c[0], c[1]);
      mma_bf16(e[0], re, b[2], b[3]);
      mma_bf16(e[1], im, b[2], b[3]);
      mma_bf16(e[0], re, b[0], b[1]);
      mma_bf16(e[1], im, b[0], b[1]);
#pragma unroll
      for (int pl = 0; pl < 2; ++pl)
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
          const float2 s = make_float2(e[pl][k], e[pl][k + 1]);
          const float2 r = FIRST ? s : __fadd2_rn(make_float2(d[ct][pl][k], d[ct][pl][k + 1]), s);
          d[ct][pl][k] = r.x;
          d[ct][pl][k + 1] = r.y;
        }
    }
}

// planes -> F x (or F^H x), rows 2g, 2g + 1 of column 4 ct + t, to out[column][row] (+= sg * ... if ADD)
template <int N, bool BWD, bool ADD>
__device__ __forceinline__ void put_sums(const float (&d)[kMmaTiles][2][4], float2* out, int rt, int R, float sg,
                                         int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int ct = 0; ct < kMmaTiles; ++ct)
    if (4 * ct + t < R) {
      float y[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // columns (re, im) = fragment columns 2t, 2t + 1
        const float* r = &d[ct][0][2 * h];
        const float* i = &d[ct][1][2 * h];
        y[2 * h] = BWD ? r[0] + i[1] : r[0] - i[1];
        y[2 * h + 1] = BWD ? r[1] - i[0] : r[1] + i[0];
      }
      float4* o = reinterpret_cast<float4*>(out + (size_t)(4 * ct + t) * N + 16 * rt + 2 * g);
      if (ADD) {
        const float4 p = *o;
        *o = make_float4(fmaf(sg, y[0], p.x), fmaf(sg, y[1], p.y), fmaf(sg, y[2], p.z), fmaf(sg, y[3], p.w));
      } else {
        *o = make_float4(y[0], y[1], y[2], y[3]);
      }
    }
}

// The warp's block (all its tile rows) times the columns of `tab`, to out; u: the tiles in flight, tile 0 and 1
// loaded by the caller.  Two tiles are always on their way.
template <int N, bool BWD>
__device__ __forceinline__ void mul_block(uint32_t (&u)[3][8], const cbf16* blk, uint32_t tab, int T, float2* out, int R,
                                          int lane) {
  constexpr int NT = N / 16;
  const uint32_t lrow = lane_row<N>(tab, lane);
  float d[kMmaTiles][2][4];
#pragma unroll
  for (int i = 0; i < NT * NT; ++i) {
    if (i + 2 < NT * NT) load_tile<N, BWD>(u[(i + 2) % 3], blk, (i + 2) / NT, (i + 2) % NT, lane);
    if (i % NT == 0) mul_tile<N, true>(u[i % 3], lrow, 0, T, d);
    else mul_tile<N, false>(u[i % 3], lrow, i % NT, T, d);
    if (i % NT == NT - 1)
      // sigma3 of a backward hop's rows (a chirality boundary falls between row pairs)
      put_sums<N, BWD, BWD>(d, out, i / NT, R, 16 * (i / NT) + 2 * (lane >> 2) < N / 2 ? 1.f : -1.f, lane);
  }
}

template <int N>
__global__ void __launch_bounds__(32 * kMW, N == 48 ? 4 : 6) kb_eo_mma(const __grid_constant__ McPhase b) {
  constexpr int NT = N / 16;
  constexpr size_t BSZ = (size_t)N * N;
  extern __shared__ __align__(16) unsigned char mc_sm[];
  __shared__ McPtrs P;
  const McItem it = load_item(b.items + blockIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int4 rec = __ldg(it.rec + ((size_t)b.out_par * it.nh + it.q) * 4 + warp);
  const BSolve& s0 = b.S[it.s0];
  const cbf16* B = static_cast<const cbf16*>(b.poly_blocks ? s0.blk_poly : s0.blk);
  const cbf16* inv = static_cast<const cbf16*>(b.poly_blocks ? s0.inv_poly : s0.inv) + (size_t)rec.w * BSZ;
  const cbf16* fb = B + ((size_t)rec.w * 5 + 1 + warp) * BSZ;
  const cbf16* bb = B + ((size_t)rec.y * 5 + 1 + warp) * BSZ;
  uint32_t u[3][8];
  if (b.vsel != BS_NONE) {  // on their way while the columns are looked up
    load_tile<N, false>(u[0], fb, 0, 0, lane);
    if (NT > 1) load_tile<N, false>(u[1], fb, 0, 1, lane);
  }
  const int R = mc_setup(P, b, it), T = (R + 3) / 4;
  if (R == 0) return;
  unsigned char* tab = mc_sm + (size_t)warp * T * split_tile<N>();
  float2* hp = reinterpret_cast<float2*>(mc_sm + (size_t)kMW * T * split_tile<N>());  // [warp][column][row]
  float2* hw = hp + (size_t)warp * R * N;
  const uint32_t ta = (uint32_t)__cvta_generic_to_shared(tab);
  if (b.vsel != BS_NONE) {
    fill_split<N>(tab, P.v, (size_t)rec.x * N, R, false, lane);
    __syncwarp();
    mul_block<N, false>(u, fb, ta, T, hw, R, lane);
    load_tile<N, true>(u[0], bb, 0, 0, lane);
    if (NT > 1) load_tile<N, true>(u[1], bb, 0, 1, lane);
    __syncwarp();
    fill_split<N>(tab, P.v, (size_t)rec.z * N, R, true, lane);
    __syncwarp();
    mul_block<N, true>(u, bb, ta, T, hw, R, lane);
  }
  if (warp < NT)  // this warp's tile row of the inverse block
#pragma unroll
    for (int K = 0; K < NT; ++K) load_tile<N, false>(u[K], inv, warp, K, lane);
  __syncthreads();
  // g = z - h (or h): the operand of the inverse block, shared by the warps
  const size_t off = (size_t)it.q * N;
  for (int i = threadIdx.x; i < R * (N / 4); i += blockDim.x) {
    const int c = i / (N / 4), j = 4 * (i % (N / 4));
    float2 v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = make_float2(0.f, 0.f);
    if (b.vsel != BS_NONE)
#pragma unroll
      for (int w = 0; w < kMW; ++w) {
        const float4* h = reinterpret_cast<const float4*>(hp + ((size_t)w * R + c) * N + j);
        const float4 h0 = h[0], h1 = h[1];
        v[0] = cadd(v[0], make_float2(h0.x, h0.y));
        v[1] = cadd(v[1], make_float2(h0.z, h0.w));
        v[2] = cadd(v[2], make_float2(h1.x, h1.y));
        v[3] = cadd(v[3], make_float2(h1.z, h1.w));
      }
    if (b.zsel != BS_NONE) {
      const float4* z = reinterpret_cast<const float4*>(P.z[c] + off + j);
      const float4 z0 = z[0], z1 = z[1];
      v[0] = csub(make_float2(z0.x, z0.y), v[0]);
      v[1] = csub(make_float2(z0.z, z0.w), v[1]);
      v[2] = csub(make_float2(z1.x, z1.y), v[2]);
      v[3] = csub(make_float2(z1.z, z1.w), v[3]);
    }
    put_split<N>(mc_sm, c, j, v);
  }
  McTail<N> ends;
  ends.load(P, b, off, R);
  __syncthreads();
  if (warp < NT) {
    const uint32_t lrow = lane_row<N>((uint32_t)__cvta_generic_to_shared(mc_sm), lane);
    float d[kMmaTiles][2][4];
    mul_tile<N, true>(u[0], lrow, 0, T, d);
#pragma unroll
    for (int K = 1; K < NT; ++K) mul_tile<N, false>(u[K], lrow, K, T, d);
    put_sums<N, false, false>(d, hp, warp, R, 1.f, lane);
  }
  __syncthreads();
  ends.finish(P, b, off, R, hp);
}

// Full stencil of one site for the columns in vp (shared memory); returns with the sums in hp.
template <int N, class BT>
__device__ __forceinline__ void mc_full_site(const McSite& s, const int* nb, const float2* const* vp, float2* tabs,
                                             float* hp, int warp, int lane) {
  const int4 rec = make_int4(__ldg(nb + s.x * 8 + warp), __ldg(nb + s.x * 8 + 4 + warp), __ldg(nb + s.x * 8 + 4 + warp),
                             s.x);
  float2* tab = tabs + (size_t)warp * s.R * N;
  float* h = hp + (size_t)warp * s.R * 2 * N;
  Piece<N, BT> tail;
  mc_hops<N, BT>(s, warp, rec, vp, tab, h, static_cast<const BT*>(s.blocks) + (size_t)s.x * 5 * N * N, tail, lane);
  fill_table<N>(tab, vp, (size_t)s.x * N, s.R, lane);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  mc_block<N, BT, true>(tail, tab, h, s.R, s.adj, warp, lane);
  __syncthreads();
}

template <int N>
__device__ __forceinline__ float2 mc_full_sum(const float* hp, int i, int R, float mu, float2 xs, int e) {
  const float2* h = reinterpret_cast<const float2*>(hp) + i;
  float2 r = cadd(cadd(h[0], h[(size_t)R * N]), cadd(h[(size_t)2 * R * N], h[(size_t)3 * R * N]));
  const float m = e < N / 2 ? mu : -mu;  // + i mu sigma3 x
  r.x -= m * xs.y;
  r.y += m * xs.x;
  return r;
}

// Batched full stencil over (operator's column chunk, site).
template <int N, class BT>
__global__ void __launch_bounds__(32 * kMW) kb_apply_mc(const __grid_constant__ McPhase b) {
  extern __shared__ __align__(16) unsigned char mc_sm[];
  __shared__ McPtrs P;
  const McItem it = load_item(b.items + blockIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const BSolve& s0 = b.S[it.s0];
  const int R = mc_setup(P, b, it);
  if (R == 0) return;
  McSite s;
  s.blocks = b.poly_blocks ? s0.blk_poly : s0.blk;
  s.x = it.q;
  s.R = R;
  s.adj = 0;
  float2* tabs = reinterpret_cast<float2*>(mc_sm);
  float* hp = reinterpret_cast<float*>(tabs + (size_t)2 * kMW * R * N);
  mc_full_site<N, BT>(s, s0.nb, P.v, tabs, hp, warp, lane);
  for (int i = threadIdx.x; i < R * N; i += blockDim.x) {
    const int c = i / N;
    const size_t idx = (size_t)s.x * N + i % N;
    const float2 xs = P.v[c][idx];
    const float2 r = mc_full_sum<N>(hp, i, R, P.mu[c], xs, i % N);
    const float2 ac = b.mode == APPLY_POLY ? P.acc[c][idx] : make_float2(0.f, 0.f);
    s8_finish(b.mode, r, xs, ac, P.coef[c], P.y[c] + idx, P.acc[c] + idx);
  }
}

// y = D x for R columns x + c * ldc of one operator.
template <int N, class BT>
__global__ void __launch_bounds__(32 * kMW) k_apply_mc(const __grid_constant__ ApplyArgs a, int R, long long ldc) {
  extern __shared__ __align__(16) unsigned char mc_sm[];
  __shared__ const float2* vp[kMcCols];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < R) vp[threadIdx.x] = static_cast<const float2*>(a.x) + threadIdx.x * ldc;
  __syncthreads();
  McSite s;
  s.blocks = a.blocks;
  s.x = blockIdx.x;
  s.R = R;
  s.adj = a.adjoint;
  float2* tabs = reinterpret_cast<float2*>(mc_sm);
  float* hp = reinterpret_cast<float*>(tabs + (size_t)2 * kMW * R * N);
  mc_full_site<N, BT>(s, a.nb, vp, tabs, hp, warp, lane);
  float2* y = static_cast<float2*>(a.y);
  for (int i = threadIdx.x; i < R * N; i += blockDim.x) {
    const size_t idx = (size_t)s.x * N + i % N;
    y[(i / N) * ldc + idx] = mc_full_sum<N>(hp, i, R, (float)a.mu, vp[i / N][idx], i % N);
  }
}

// BF16 blocks go to the tensor cores, FP32 blocks to the FP32 pipe.  A half apply of a batch of 12 operators
// (up to 12 columns each, 4^4 to 8^4), n = 16 / 32 / 48: BF16 30 / 103 / 106 us, FP32 27 / 124 / 140 us; with
// one work item per column, BF16 72 / 326 / 328 us, FP32 76 / 631 / 618 us.  Relative error against FP64 sums,
// random data at 8^4: BF16 1.05e-7 / 1.16e-7 / 1.19e-7 (column by column 1.06e-7 / 1.29e-7 / 1.32e-7), FP32
// 0.99e-7 / 1.11e-7 / 1.24e-7 (1.06e-7 / 1.53e-7 / 1.48e-7).
template <int N>
int launch_beo_mc_n(bool bf, const McPhase& b, cudaStream_t s) {
  static SmemLimit mma, mc;
  if (bf) {
    COARSE_CUDA(raise_smem_limit(mma, (const void*)kb_eo_mma<N>, mma_smem<N>(kMcCols)));
    kb_eo_mma<N><<<b.count, 32 * kMW, mma_smem<N>(b.rmax), s>>>(b);
  } else {
    COARSE_CUDA(raise_smem_limit(mc, (const void*)kb_eo_mc<N, float2>, mc_smem<N>(kMcCols)));
    kb_eo_mc<N, float2><<<b.count, 32 * kMW, mc_smem<N>(b.rmax), s>>>(b);
  }
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

template <int N, class BT>
int launch_bapply_mc_n(const McPhase& b, cudaStream_t s) {
  static SmemLimit limit;
  COARSE_CUDA(raise_smem_limit(limit, (const void*)kb_apply_mc<N, BT>, mc_smem<N>(kMcCols)));
  kb_apply_mc<N, BT><<<b.count, 32 * kMW, mc_smem<N>(b.rmax), s>>>(b);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

template <int N>
int launch_apply_mc_n(const ApplyArgs& a, int R, long long ldc, cudaStream_t s) {
  static SmemLimit limit;
  COARSE_CUDA(raise_smem_limit(limit, (const void*)k_apply_mc<N, float2>, mc_smem<N>(kMcCols)));
  k_apply_mc<N, float2><<<a.V, 32 * kMW, mc_smem<N>(R), s>>>(a, R, ldc);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

}  // namespace

int launch_beo_mc(int prec, int n, const McPhase& b, cudaStream_t s) {
  if (b.count <= 0) return COARSE_OK;
  const bool bf = prec == COARSE_PREC_BF16;
  switch (n) {
    case 16: return launch_beo_mc_n<16>(bf, b, s);
    case 32: return launch_beo_mc_n<32>(bf, b, s);
    case 48: return launch_beo_mc_n<48>(bf, b, s);
  }
  set_error("batched half apply: unsupported n = %d", n);
  return COARSE_ERR_INVALID_ARG;
}

int launch_bapply_mc(int prec, int n, const McPhase& b, cudaStream_t s) {
  if (b.count <= 0) return COARSE_OK;
  const bool bf = prec == COARSE_PREC_BF16;
  switch (n) {
    case 16: return bf ? launch_bapply_mc_n<16, cbf16>(b, s) : launch_bapply_mc_n<16, float2>(b, s);
    case 32: return bf ? launch_bapply_mc_n<32, cbf16>(b, s) : launch_bapply_mc_n<32, float2>(b, s);
    case 48: return bf ? launch_bapply_mc_n<48, cbf16>(b, s) : launch_bapply_mc_n<48, float2>(b, s);
  }
  set_error("batched apply: unsupported n = %d", n);
  return COARSE_ERR_INVALID_ARG;
}

int launch_apply_mc(int n, const ApplyArgs& a, int R, long long ldc, cudaStream_t s) {
  if (R < 1 || R > kMcCols) {
    set_error("multi-column stencil: %d columns in one pass", R);
    return COARSE_ERR_INVALID_ARG;
  }
  switch (n) {
    case 16: return launch_apply_mc_n<16>(a, R, ldc, s);
    case 32: return launch_apply_mc_n<32>(a, R, ldc, s);
    case 48: return launch_apply_mc_n<48>(a, R, ldc, s);
  }
  set_error("coarse_apply: unsupported n = %d (nv must be 8, 16 or 24)", n);
  return COARSE_ERR_INVALID_ARG;
}

}  // namespace coarse
