// FP64 stencil y = D_c x by exact products of 8-bit digits on the tensor cores.
//
// GB300 runs FP64 fused multiply-adds at about 1.25 TFLOP/s, a sixtieth of its FP32 rate, so the FP64
// stencil on the FP64 pipe is bound by that rate whatever the layout (16^4 sites, n = 48: 10.3 ms against
// 1.8 ms of block traffic).  Here each block and each site vector is written once as 64-bit fixed-point
// numbers with a common power-of-two scale, cut into eight signed 8-bit digits (radix 256, digits
// -128 .. 127), and the products of digits are summed by mma.sync m16n8k16 (FP16 operands, FP32 sums):
//   a = 2^(E-6) sum_p a_p 256^-p,  x = 2^(F-6) sum_q x_q 256^-q,  |a| < 2^E, |x| < 2^F for the whole
//   block / site vector,  sum_j a_ij x_j = 2^(E+F-12) sum_s 256^-s L_s,  L_s = sum_{p+q=s} sum_j a_p x_q.
// Every L_s is an integer below 2^23, so the FP32 sums are exact.  What is left out of one real product a x is at
// most 9.03 x 2^(E+F-62): 2 units for the fixed-point conversions, 7.03 for the levels s >= 8 (seven pairs of
// digits of up to 2^14 at s = 8).  Summed over a block row that is |error| <= 25.6 z 2^(E+F-62), z the number of
// the site vector's non-zero entries; the FP64 pipe then adds up one number per block, row and part.
//
// Rows.  That error is measured by the largest entries of the block and of the site, and a row whose products are
// all far smaller would come out with few correct bits or none.  So every row also gets a lower bound of
// sum_j |a_ij| |x_j| from the leading digits, S_0 = sum_j (|re a_0| + |im a_0|)(|re x_0| + |im x_0|) over 16 of the
// columns j (one more mma per tile row; the tiles take turns over a site's blocks): sum_j |a_ij| |x_j| >=
// 2^(E+F-15) S_0, a digit being at most twice the number it rounds.  A row keeps its digit sum if, over its nine
// blocks, sum_b 2^(E_b+F_b) (S_0b - 256 z_b / n) >= 0: then its error is at most 6.4 n 2^-53 of sum_j |a_ij| |x_j|
// (on random digits about a thirtieth of that).  Every other row, also where a scale is near the FP64 range's ends
// or an entry is not finite, is summed again on the FP64 pipe.  S_0 n / z is at least 1100 to 4400 for Gaussian
// vectors and solutions with Gaussian right-hand sides (coarse Wilson blocks of n = 48, random blocks of n = 16);
// of the solution for a point source on 8^4 sites, n = 48, two rows in 10^5 are summed again.
//
// Digits in FP16: an unsigned byte b = digit + 128 zero-extended to 16 bits is the FP16 subnormal
// b 2^-24, so a block digit becomes an MMA operand with one byte permutation.  The excess 128 is taken out
// by starting the sums at -128 2^-24 sum_{p<=s} sum_j x_{s-p,j}, which the column pack computes.
//
// Operands: A = a digit plane of a 16 x 16 tile (real or imaginary part), B = the eight levels of the
// site vector (n = 8): for block digit p, level s takes vector digit s - p, so B is the digit table
// shifted by p rows (ldmatrix row addresses; rows of zeros before digit 0).  Real and imaginary block
// planes keep separate sums and are combined per block.  A backward hop uses the transposed tiles: the
// (re, im) bytes of one entry are one 16-bit element of movmatrix.
//
// Block layout: per block n/16 x n/16 tiles, per tile [digit p][lane] uint4, words a0..a3 of the
// m16n8k16 A fragment, each the bytes {re, im of column 2t, re, im of column 2t + 1}: 8 bytes per real
// number, one 4 KB stream per tile.
//
// Two kernels: one CTA of nine warps per site, one block product per warp (small lattices, several columns), and
// the push kernel, which reads every block once (one column).
#include <cuda_fp16.h>

#include "digits.cuh"

namespace coarse {
namespace {

constexpr int kDW = 9;  // warps per site: one block product each
constexpr unsigned long long kBias = 0x8080808080808080ull;
constexpr int kMaxExp = 900;        // scales, and products of scales, beyond 2^+-900 go to the FP64 pipe
constexpr float kRowNeed = 256.f;   // S_0 per non-zero share of the site vector (see above)

// The packs look at the doubles as integers (the FP64 pipe would bound them): magnitudes by their high
// words, whose top bits are the biased exponent.
__device__ __forceinline__ uint32_t high_abs(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }

// Scale of entries whose largest high word is m: true and the biased exponent of the largest, or false where it
// is too near the range's ends or not finite.  m = 0: no entry above the subnormals.
__device__ __forceinline__ bool scale_of(uint32_t m, int& ex) {
  ex = (int)(m >> 20);
  return ex > 1023 - kMaxExp && ex < 1023 + kMaxExp;
}
// 2^(E - 6) with 2^E the next power of two above a number of biased exponent ex
__device__ __forceinline__ double scale_value(int ex) { return __hiloint2double((ex + 1 - 6) << 20, 0); }
__device__ __forceinline__ double scale_special() { return __hiloint2double(0x7ff80000, 0); }

// Scale of a block's product with a site vector: a power of two, 0 (one of them is zero) or NaN.  Products of
// scales near the range's ends would lose the low levels to underflow: NaN, for the FP64 pipe.
__device__ __forceinline__ double product_scale(double block, double vec) {
  const double sc = block * vec;
  const bool in = (high_abs(sc) >> 20) - (1023u - kMaxExp) < 2u * kMaxExp;
  return in || block == 0.0 || vec == 0.0 ? sc : scale_special();
}
// Its exponent as the rows' test uses it: 0 for a zero scale, kNoScale for NaN.
constexpr int kNoScale = 2047;
__device__ __forceinline__ int scale_exp(double sc) { return (int)(high_abs(sc) >> 20); }
// 2^(e - top), 0 for a zero scale and far below `top`
__device__ __forceinline__ float scale_weight(int e, int top) {
  return e > 0 && top - e < 126 ? __int_as_float((127 - (top - e)) << 23) : 0.f;
}

// fixed-point digits of v, |v| < 2^E, in units of 2^(E - 62): byte 7 - p = digit p + 128
__device__ __forceinline__ unsigned long long digits_of(double v, int ex) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu), d = ex - e;
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  m = (e == 0 || d > 63) ? 0ull : (m << 9) >> d;
  return ((hi >> 31) ? 0ull - m : m) + kBias;
}

// ------------------------------------------------------------------------------- operand packing
// One CTA per stored block; bound by the 32 n^2 bytes it reads and writes.
__global__ void __launch_bounds__(256) k_dig_blocks(const double2* __restrict__ blocks, int n, uint4* __restrict__ dig,
                                                    double* __restrict__ scale) {
  __shared__ uint32_t top[8];
  __shared__ int ex_sh;
  const size_t blk = blockIdx.x;
  const double2* B = blocks + blk * n * n;
  uint32_t m = 0u;
  int any = 0;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const double2 v = B[e];
    m = max(m, max(high_abs(v.x), high_abs(v.y)));
    any |= v.x != 0.0 || v.y != 0.0;
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = m;
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) m = max(m, top[i]);
    int ex;
    const bool bad = !scale_of(m, ex) && any;  // not finite: the largest exponent
    ex_sh = bad ? 4096 : ex;                   // 4096: every entry below the last digit
    scale[blk] = bad ? scale_special() : (any ? scale_value(ex) : 0.0);
  }
  __syncthreads();
  const int ex = ex_sh, NT = n / 16;
  for (int w = threadIdx.x; w < NT * NT * 32; w += blockDim.x) {
    const int lane = w & 31, tile = w >> 5, U = tile / NT, W = tile % NT;
    const int r = 16 * U + (lane >> 2), c = 16 * W + 2 * (lane & 3);
    unsigned long long d[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // fragment words: rows r, r + 8, then columns + 8
      const double2* p = B + (size_t)(r + 8 * (k & 1)) * n + c + 8 * (k >> 1);
      const double2 v0 = p[0], v1 = p[1];
      d[k][0] = digits_of(v0.x, ex);
      d[k][1] = digits_of(v0.y, ex);
      d[k][2] = digits_of(v1.x, ex);
      d[k][3] = digits_of(v1.y, ex);
    }
    uint4* out = dig + ((blk * NT * NT + tile) * 8) * 32 + lane;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      uint32_t o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        o[k] = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) o[k] |= (uint32_t)((d[k][q] >> (56 - 8 * p)) & 255ull) << (8 * q);
      }
      out[p * 32] = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// Digits, corrections, scale and the rows' demand (kRowNeed) of one site vector, by one warp (dg: 16 N shorts of
// its own).
template <int N>
__device__ __forceinline__ void dig_x_site(const double2* __restrict__ p, size_t rec, short (*dg)[N],
                                           __half* __restrict__ xd, float* __restrict__ xc, double* __restrict__ xs,
                                           float* __restrict__ xn) {
  const int lane = threadIdx.x & 31;
  constexpr int PER = (N + 31) / 32;
  double2 v[PER];
  uint32_t m = 0u;  // largest high word
  int nz = 0;       // non-zero entries
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = lane + 32 * k;
    v[k] = i < N ? p[i] : make_double2(0.0, 0.0);
    nz += __popc(__ballot_sync(0xffffffffu, v[k].x != 0.0 || v[k].y != 0.0));
    m = max(m, max(high_abs(v[k].x), high_abs(v[k].y)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  int ex;
  const bool ok = scale_of(m, ex) || nz == 0;
  if (!ok) ex = 4096;  // every entry below the last digit
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = lane + 32 * k;
    if (i < N) {
      const unsigned long long dx = digits_of(v[k].x, ex), dy = digits_of(v[k].y, ex);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        dg[q][i] = (short)((int)((dx >> (56 - 8 * q)) & 255ull) - 128);
        dg[8 + q][i] = (short)((int)((dy >> (56 - 8 * q)) & 255ull) - 128);
      }
    }
  }
  __syncwarp();
  __half2* o = reinterpret_cast<__half2*>(xd + rec * dig_x_halves(N));
  for (int w = lane; w < 8 * N; w += 32) {
    const int row = w / (N / 2), c = 2 * (w % (N / 2));
    o[w] = __floats2half2_rn((float)dg[row][c], (float)dg[row][c + 1]);
  }
  if (lane < N / 2)  // magnitudes of the leading digits
    o[8 * N + lane] = __floats2half2_rn((float)(abs(dg[0][2 * lane]) + abs(dg[8][2 * lane])),
                                        (float)(abs(dg[0][2 * lane + 1]) + abs(dg[8][2 * lane + 1])));
  // lane = (half, part, digit): sums over the half, then the corrections of the two sigma3 variants
  int sum = 0;
  {
    const int row = lane & 15, h = lane >> 4;
    for (int i = 0; i < N / 2; ++i) sum += dg[row][h * (N / 2) + i];
  }
  const int lo = __shfl_sync(0xffffffffu, sum, lane & 15), hi = __shfl_sync(0xffffffffu, sum, 16 + (lane & 15));
  int t = lane < 16 ? lo + hi : lo - hi;  // lane = (variant, part, digit)
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) {  // prefix sums over the digits: levels
    const int u = __shfl_up_sync(0xffffffffu, t, off, 8);
    if ((lane & 7) >= off) t += u;
  }
  xc[rec * kDigCorr + lane] = (float)t * -0x1p-17f;  // -128 * 2^-24
  if (lane == 0) {
    xs[rec] = ok ? (nz ? scale_value(ex) : 0.0) : scale_special();
    xn[rec] = kRowNeed / N * nz;
  }
}

template <int N>
__global__ void __launch_bounds__(128) k_dig_x(const double2* __restrict__ x, long long ldc, int V,
                                               __half* __restrict__ xd, float* __restrict__ xc,
                                               double* __restrict__ xs, float* __restrict__ xn, const int* stop) {
  if (stop != nullptr && *stop) return;
  __shared__ short dg[4][16][N];
  const int warp = threadIdx.x >> 5, site = blockIdx.x * 4 + warp, col = blockIdx.y;
  if (site >= V) return;  // warp-uniform
  dig_x_site<N>(x + col * ldc + (size_t)site * N, (size_t)col * V + site, dg[warp], xd, xc, xs, xn);
}

// The column operands of one pass in `mem` (dig_x_bytes).
struct DigX {
  __half* xd;
  float* xc;
  double* xs;
  float* xn;
};
template <int N>
__host__ __device__ __forceinline__ DigX dig_x_at(void* mem, int V, int cols) {
  char* m = static_cast<char*>(mem);
  DigX d;
  d.xd = reinterpret_cast<__half*>(m);
  m += (size_t)cols * V * dig_x_halves(N) * sizeof(__half);
  d.xc = reinterpret_cast<float*>(m);
  m += (size_t)cols * V * kDigCorr * sizeof(float);
  d.xs = reinterpret_cast<double*>(m);
  m += (size_t)cols * V * sizeof(double);
  d.xn = reinterpret_cast<float*>(m);
  return d;
}

// Batched column pack: warp w of the launch takes site w - start of the pass found through the map.
template <int N>
__global__ void __launch_bounds__(128) kb_dig_x(const DigPass* __restrict__ passes, const int* __restrict__ map,
                                                const int* __restrict__ flags) {
  __shared__ short dg[4][16][N];
  const int warp = threadIdx.x >> 5, w = blockIdx.x * 4 + warp;
  const DigPass& p = passes[__ldg(map + w / kDigMapSites)];
  const int site = w - p.start;
  if (site >= p.V) return;  // warp-uniform
  const DigX d = dig_x_at<N>(p.digx, p.V, p.cols);
  if (flags[2 * p.q0 + 1] && flags[2 * (p.q0 + p.cols - 1) + 1]) return;  // every column of the pass is done
  for (int c = 0; c < p.cols; ++c) {
    dig_x_site<N>(p.x + (size_t)c * p.ldx + (size_t)site * N, (size_t)c * p.V + site, dg[warp], d.xd, d.xc, d.xs,
                  d.xn);
    __syncwarp();
  }
}

// -------------------------------------------------------------------------------------- the stencil
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t movmatrix(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// Shared-memory digit table of one column: [part][7 zero rows + 8 digits][n], rows padded to an odd
// number of 16-byte units (conflict-free ldmatrix); behind both parts the magnitudes of the leading digits.
template <int N> constexpr int dig_row() { return 2 * N + 16; }
template <int N> constexpr int dig_part() { return 15 * dig_row<N>(); }
template <int N> constexpr int dig_slab() { return 2 * dig_part<N>() + 2 * N; }

// CTAs per SM to keep registers for, as many as measured faster with two columns: n = 16 three (8^4: 93 us against 95
// with two), n = 32 and 48 two (n = 48, 8^4: 357 us, in 96 registers with spills, against 449 with one CTA).
__host__ __device__ constexpr int dig_min_blocks(int N) { return N == 16 ? 3 : 2; }

struct DigArgs {
  const uint4* dig;
  const double* bscale;
  const __half* xd;
  const float* xc;
  const double* xs;
  const float* xn;
  void* work;  // push kernel: dig_rows_at
};

// One output tile's level sums [plane of the block][part of the column] -> this lane's (row, part) of the
// product with the block (or with its adjoint).
template <bool BWD>
__device__ __forceinline__ double dig_flush(const float (&d)[2][2][4], double sc, int lane) {
  const int t = lane & 3;
  // levels 2t, 2t + 1 of (row g, row g + 8) x (re, im) as integers; F x or F^H x from the planes
  long long q[2][2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int yr[2], yi[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const int k = 2 * h + l;
      const float fr = BWD ? d[0][0][k] + d[1][1][k] : d[0][0][k] - d[1][1][k];
      const float fi = BWD ? d[0][1][k] - d[1][0][k] : d[0][1][k] + d[1][0][k];
      yr[l] = __float2int_rn(fr * 0x1p24f);
      yi[l] = __float2int_rn(fi * 0x1p24f);
    }
    q[h][0] = (long long)yr[0] * 256 + yr[1];
    q[h][1] = (long long)yi[0] * 256 + yi[1];
  }
  // sum over the quad's levels: lanes t ^ 1 trade rows, lanes t ^ 2 trade parts
  long long u[2];
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    const long long own = (t & 1) ? q[1][part] : q[0][part];
    const long long got = __shfl_xor_sync(0xffffffffu, (t & 1) ? q[0][part] : q[1][part], 1);
    u[part] = (t & 1) ? (got << 16) + own : (own << 16) + got;
  }
  const long long own = (t & 2) ? u[1] : u[0];
  const long long got = __shfl_xor_sync(0xffffffffu, (t & 2) ? u[0] : u[1], 2);
  const double hi = (double)((t & 2) ? got : own), lo = (double)((t & 2) ? own : got);
  return fma(hi, sc * 0x1p-24, lo * (sc * 0x1p-56));
}

// A words of the magnitudes |re| + |im| of a tile's leading digits, from the words of digit 0 (bytes digit + 128: the
// excess is 128 2^-24 in both halves).
__device__ __forceinline__ void dig_mag_tile(uint4 w, uint32_t (&m)[4]) {
  const uint32_t a[4] = {w.x, w.y, w.z, w.w}, eb = 0x80808080u;
  const __half2 e = *reinterpret_cast<const __half2*>(&eb);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t re = __byte_perm(a[k], 0u, 0x4240), im = __byte_perm(a[k], 0u, 0x4341);
    const __half2 s = __hadd2(__habs2(__hadd2(*reinterpret_cast<const __half2*>(&re), e)),
                              __habs2(__hadd2(*reinterpret_cast<const __half2*>(&im), e)));
    m[k] = *reinterpret_cast<const uint32_t*>(&s);
  }
}
// d += those magnitudes times the column's (mg: its magnitudes of this tile, dig_slab).  Only column q of B is filled:
// the sums of tile row after tile row land in columns of their own.
__device__ __forceinline__ void dig_mags(const uint32_t (&m)[4], const unsigned char* mg, int q, float (&d)[4], int lane) {
  const uint32_t* v = reinterpret_cast<const uint32_t*>(mg) + (lane & 3);
  const bool on = lane >> 2 == q;
  mma_f16(d, m, on ? v[0] : 0u, on ? v[4] : 0u);
}

// One block product of the warp: the block's tiles times the columns' digit tables in `tab`, added to
// acc[tile][column] (lane (g, t): row 16 tile + g + 8 (t & 1), part t >> 1); mag[column]: the rows' magnitudes,
// tile O in column O of the fragment.  flip: sigma3 on the operand and
// the result.  w: the tile being multiplied; each of its loads is replaced by the next tile's as soon as it
// is used, so that a tile's loads are in flight during the whole of the tile before it.
template <int N, int C, bool BWD>
__device__ __forceinline__ void dig_block(const uint4* __restrict__ blk, uint4 (&w)[8], const unsigned char* tab, const float (&corr)[C][4],
                                          const double (&sc)[C], double (&acc)[N / 16][C], float (&mag)[C][4],
                                          bool flip, int turn) {
  constexpr int NT = N / 16, RS = dig_row<N>(), PS = dig_part<N>(), SL = dig_slab<N>();
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint32_t slab = (uint32_t)__cvta_generic_to_shared(tab);
  const uint32_t fmask = flip ? 0x80008000u : 0u;
  // ldmatrix row of this lane: matrix lane / 8 = (part, upper half of k), level lane % 8
  const uint32_t lrow = slab + (uint32_t)((lane >> 4) * PS + (7 + (lane & 7)) * RS + ((lane >> 3) & 1) * 16);
#pragma unroll
  for (int O = 0; O < NT; ++O) {
    // sums [column][plane of the block][part of the column]
    float d[C][2][2][4];
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int pl = 0; pl < 2; ++pl)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          d[c][pl][0][k] = corr[c][k & 1];
          d[c][pl][1][k] = corr[c][2 + (k & 1)];
        }
#pragma unroll
    for (int K = 0; K < NT; ++K) {
      const int next = O * NT + K + 1;  // in the order (output tile, inner tile)
      const uint4* tn = blk + (BWD ? (next % NT) * NT + next / NT : next) * 256 + lane;
      if ((O + turn) % NT == K) {
        uint32_t m[4];
        dig_mag_tile(w[0], m);
        const uint32_t mt[4] = {BWD ? movmatrix(m[0]) : m[0], BWD ? movmatrix(m[2]) : m[1], BWD ? movmatrix(m[1]) : m[2],
                                BWD ? movmatrix(m[3]) : m[3]};
#pragma unroll
        for (int c = 0; c < C; ++c) dig_mags(mt, tab + c * SL + 2 * PS + K * 32, O, mag[c], lane);
      }
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        uint32_t a[4];
        if (BWD) {  // transposed tile: the row and column halves trade places
          a[0] = movmatrix(w[p].x);
          a[1] = movmatrix(w[p].z);
          a[2] = movmatrix(w[p].y);
          a[3] = movmatrix(w[p].w);
        } else {
          a[0] = w[p].x;
          a[1] = w[p].y;
          a[2] = w[p].z;
          a[3] = w[p].w;
        }
        uint32_t re[4], im[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          re[k] = __byte_perm(a[k], 0u, 0x4240);
          im[k] = __byte_perm(a[k], 0u, 0x4341);
        }
        if (next < NT * NT) w[p] = __ldg(tn + p * 32);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          uint32_t b[4];
          ldsm4(lrow + (uint32_t)(c * SL + K * 32 - p * RS), b);
          if (16 * K >= N / 2) {  // sigma3: the second chirality's entries negated (N / 2 is a multiple of 8)
            b[0] ^= fmask;
            b[2] ^= fmask;
          }
          if (16 * K + 8 >= N / 2) {
            b[1] ^= fmask;
            b[3] ^= fmask;
          }
          mma_f16(d[c][0][0], re, b[0], b[1]);
          mma_f16(d[c][0][1], re, b[2], b[3]);
          mma_f16(d[c][1][0], im, b[0], b[1]);
          mma_f16(d[c][1][1], im, b[2], b[3]);
        }
      }
    }
    const bool neg = flip && (16 * O + g + 8 * (t & 1)) >= N / 2;
#pragma unroll
    for (int c = 0; c < C; ++c) acc[O][c] += dig_flush<BWD>(d[c], neg ? -sc[c] : sc[c], lane);
  }
}

// Digit table of one column from its packed digits and magnitudes (asynchronous copies), its zero rows, its corrections.
template <int N>
__device__ __forceinline__ void dig_table(unsigned char* tab, const __half* xd, int lane) {
  constexpr int CH = N / 8;  // 16-byte chunks per row
#pragma unroll
  for (int i0 = 0; i0 < 17 * CH; i0 += 32) {
    const int i = i0 + lane, row = i / CH, kc = i % CH;
    const unsigned char* to = row < 16 ? tab + (row >> 3) * dig_part<N>() + (7 + (row & 7)) * dig_row<N>() + kc * 16
                                       : tab + 2 * dig_part<N>() + kc * 16;
    if (i < 17 * CH)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)),
                   "l"(reinterpret_cast<const uint4*>(xd) + i)
                   : "memory");
  }
}
template <int N, int C>
__device__ __forceinline__ void dig_zero_rows(unsigned char* slab, int lane) {
  constexpr int U = dig_row<N>() / 16;
  for (int i = lane; i < C * 2 * 7 * U; i += 32) {
    const int q = i / U, tbl = q / 7;  // tbl = (column, part)
    *reinterpret_cast<uint4*>(slab + (tbl >> 1) * dig_slab<N>() + (tbl & 1) * dig_part<N>() + (q % 7) * dig_row<N>() +
                              (i % U) * 16) = make_uint4(0, 0, 0, 0);
  }
}
__device__ __forceinline__ void dig_corr(const float* xc, bool flip, float (&corr)[4], int lane) {
  const float* p = xc + (flip ? 16 : 0) + 2 * (lane & 3);
  const float2 r = __ldg(reinterpret_cast<const float2*>(p)), i = __ldg(reinterpret_cast<const float2*>(p + 8));
  corr[0] = r.x;
  corr[1] = r.y;
  corr[2] = i.x;
  corr[3] = i.y;
}

// Row `row` of the site's nine block products on the FP64 pipe, by eight lanes (whole warps call it: four rows at a
// time); every lane of the eight gets the sum.
template <int N>
__device__ __noinline__ double2 dig_plain_row(const double2* __restrict__ B, const int* __restrict__ nb, bool adj,
                                              int site, int row, const double2* __restrict__ x) {
  const int t = threadIdx.x & 7;
  double2 y = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int u = 0; u < 9; ++u) {
    const int src = u == 0 ? site : __ldg(nb + site * 8 + (u - 1));
    const bool flip = (u < 5) == adj;  // sigma3 on the operand and the result
    const double2* blk = B + (size_t)(u < 5 ? site * 5 + u : src * 5 + u - 4) * N * N;
    double2 e[N / 8], v[N / 8], p = make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < N / 8; ++k) {
      const int j = t + 8 * k;
      e[k] = __ldg(blk + (u < 5 ? row * N + j : j * N + row));
      v[k] = __ldg(x + (size_t)src * N + j);
    }
#pragma unroll
    for (int k = 0; k < N / 8; ++k) {
      const double2 w = flip && t + 8 * k >= N / 2 ? make_double2(-v[k].x, -v[k].y) : v[k];
      if (u < 5) cfma(p, e[k], w);
      else cfma_conj(p, e[k], w);
    }
    y = flip && row >= N / 2 ? csub(y, p) : cadd(y, p);
  }
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) {
    y.x += __shfl_xor_sync(0xffffffffu, y.x, off);
    y.y += __shfl_xor_sync(0xffffffffu, y.y, off);
  }
  return y;
}

// Entry e of column c of the site from the warps' sums `part`.
template <int N, int C>
__device__ __forceinline__ double2 dig_sum(const double* part, int c, int e) {
  const double* pc = part + c * 2 * N + 2 * e;
  double2 r = make_double2(pc[0], pc[1]);
#pragma unroll
  for (int w = 1; w < kDW; ++w) r = cadd(r, make_double2(pc[w * C * 2 * N], pc[w * C * 2 * N + 1]));
  return r;
}

// Mass term and epilogue of that entry: r the sum of the blocks, idx its index in a column.
template <int N>
__device__ __forceinline__ void dig_finish(const ApplyArgs& a, double2 r, int c, int e, size_t idx, size_t ldy,
                                           double2 xs, double2 z) {
  const double2 c0 = a.mode != APPLY_PLAIN ? a.coef[0] : make_double2(0.0, 0.0);
  const double2 c1 = a.mode != APPLY_PLAIN ? a.coef[1] : make_double2(0.0, 0.0);
  const double m = e < N / 2 ? a.mu : -a.mu;  // + i mu sigma3 x
  r.x -= m * xs.y;
  r.y += m * xs.x;
  double2* y = static_cast<double2*>(a.y) + c * ldy + idx;
  if (a.mode == APPLY_PLAIN) {
    *y = r;
  } else if (a.mode == APPLY_AXPBY) {
    *y = cadd(cmul(c0, r), cmul(c1, z));
  } else {
    // chain step: s' = s - c0 D s ; acc = acc + c1 s'  (first: acc = c2 s + c1 s')
    double2* accp = static_cast<double2*>(a.acc) + c * ldy + idx;
    const double2 ac = a.mode == APPLY_POLY_FIRST ? cmul(a.coef[2], xs) : *accp;
    r = csub(xs, cmul(c0, r));
    *y = r;
    *accp = cadd(ac, cmul(c1, r));
  }
}

// One site of the columns x + c ldx (c < ncol <= C), results y + c ldy, addend z + c ldz (AXPBY).
template <int N, int C>
__device__ __forceinline__ void dig_site(const ApplyArgs& a, const DigArgs& dgt, const int site, const int ncol,
                                         const size_t ldx, const size_t ldy, const size_t ldz) {
  constexpr int NT = N / 16, SL = dig_slab<N>();
  extern __shared__ __align__(16) unsigned char dsm[];  // [kDW][C] digit tables, then [kDW][C][2N] sums
  static_assert(SL >= 2 * N * 8 + N * 4, "the sums and magnitudes take the place of the digit tables");
  __shared__ int sexp[kDW][C];     // exponents of the products' scales
  __shared__ float sneed[kDW][C];
  __shared__ uint32_t redo[3];     // rows to sum on the FP64 pipe
  const int u = threadIdx.x >> 5, lane = threadIdx.x & 31;  // warp u: block product u
  const int V = a.V;
  const int nc = ncol < C ? ncol : C;
  const int src = u == 0 ? site : __ldg(a.nb + site * 8 + (u - 1));
  const int blk = u < 5 ? site * 5 + u : src * 5 + 1 + (u - 5);
  const bool flip = (u < 5) == (a.adjoint != 0);  // sigma3 on the operand and the result
  const uint4* bp = dgt.dig + (size_t)blk * NT * NT * 256;
  uint4 w[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) w[p] = __ldg(bp + lane + p * 32);
  unsigned char* slab = dsm + (size_t)u * C * SL;
  const double bs = __ldg(dgt.bscale + blk);
  float corr[C][4];
  double sc[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const size_t rec = (size_t)(c < nc ? c : 0) * V + src;
    dig_table<N>(slab + c * SL, dgt.xd + rec * dig_x_halves(N), lane);
    dig_corr(dgt.xc + rec * kDigCorr, flip, corr[c], lane);
    sc[c] = product_scale(bs, __ldg(dgt.xs + rec));
    if (lane == 0) {
      sexp[u][c] = scale_exp(sc[c]);
      sneed[u][c] = __ldg(dgt.xn + rec);
    }
  }
  dig_zero_rows<N, C>(slab, lane);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  double acc[NT][C];
#pragma unroll
  for (int O = 0; O < NT; ++O)
#pragma unroll
    for (int c = 0; c < C; ++c) acc[O][c] = 0.0;
  float mag[C][4];
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) mag[c][k] = 0.f;
  if (u < 5) dig_block<N, C, false>(bp, w, slab, corr, sc, acc, mag, flip, u);
  else dig_block<N, C, true>(bp, w, slab, corr, sc, acc, mag, flip, u);
  __syncthreads();  // every warp is done with its tables
  double* part = reinterpret_cast<double*>(dsm);                  // [warp][column][2 row + part]
  float* pmag = reinterpret_cast<float*>(part + kDW * C * 2 * N);  // [warp][column][row]
  {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int c = 0; c < C; ++c) {
#pragma unroll
      for (int O = 0; O < NT; ++O) part[(u * C + c) * 2 * N + 2 * (16 * O + g + 8 * (t & 1)) + (t >> 1)] = acc[O][c];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int O = 2 * t + (k & 1);
        if (O < NT) pmag[(u * C + c) * N + 16 * O + g + 8 * (k >> 1)] = mag[c][k] * 0x1p24f;
      }
    }
  }
  __syncthreads();
  // one thread per entry (the first three warps)
  static_assert(C * 48 <= 96, "one thread per entry");
  const int c = threadIdx.x / N, e = threadIdx.x % N;
  const bool mine = threadIdx.x < nc * N;
  double2 r = make_double2(0.0, 0.0);
  if (u < 3) {
    bool bad = false;
    if (mine) {
      r = dig_sum<N, C>(part, c, e);
      int top = 0;
#pragma unroll
      for (int q = 0; q < kDW; ++q) top = max(top, sexp[q][c]);
      float have = 0.f;
#pragma unroll
      for (int q = 0; q < kDW; ++q) have += scale_weight(sexp[q][c], top) * (pmag[(q * C + c) * N + e] - sneed[q][c]);
      bad = top == kNoScale || !(have >= 0.f);
    }
    const uint32_t m = __ballot_sync(0xffffffffu, bad);
    if (lane == 0) redo[u] = m;
  }
  __syncthreads();
  if (redo[0] | redo[1] | redo[2]) {  // the sums in place of warp 0's
    for (int i0 = 4 * u; i0 < nc * N; i0 += 4 * kDW) {
      const int i = i0 + (lane >> 3);  // four rows of one column (N is a multiple of 4)
      if (!(redo[i0 >> 5] >> (i0 & 31) & 15u)) continue;
      const double2 v = dig_plain_row<N>(static_cast<const double2*>(a.blocks), a.nb, a.adjoint != 0, site, i % N,
                                         static_cast<const double2*>(a.x) + (size_t)(i / N) * ldx);
      if ((lane & 7) == 0) reinterpret_cast<double2*>(part)[i] = v;
    }
    __syncthreads();
    if (mine && (redo[u] >> lane & 1u)) r = reinterpret_cast<const double2*>(part)[threadIdx.x];
  }
  if (mine) {
    const size_t idx = (size_t)site * N + e;
    const double2 xs = static_cast<const double2*>(a.x)[c * ldx + idx];
    const double2 z = a.mode == APPLY_AXPBY ? static_cast<const double2*>(a.z)[c * ldz + idx] : xs;
    dig_finish<N>(a, r, c, e, idx, ldy, xs, z);
  }
}

// One CTA per site: two columns, and small lattices.
template <int N, int C>
__global__ void __launch_bounds__(32 * kDW, dig_min_blocks(N)) k_site_digits(
    const __grid_constant__ ApplyArgs a, const __grid_constant__ DigArgs dgt, int ncol, long long ldc) {
  if (a.stop != nullptr && *a.stop) return;
  dig_site<N, C>(a, dgt, blockIdx.x, ncol, ldc, ldc, ldc);
}

// ------------------------------------------------------------------ one column: every block once
// The pull kernel reads a hop block twice, as a forward hop and transposed for the site in front: nine blocks per site
// through L2, of which about a quarter hit (16^4, n = 48: 3.4 ms).  Here the four warps of site x multiply each tile of
// F_{x,mu} both ways while it is in registers: forward with the digits of x + mu into the site's own sum, transposed
// with the site's digits into the push for x + mu,
//   P_x = A_x v_x + sum_mu F_{x,mu} v_{x+mu},   T_mu[x] = sigma3 F_{x,mu}^H sigma3 v_x,
// and k_push_finish adds y_z = P_z + sum_mu T_mu[z - mu], the mass term and the epilogue.  The self block's tile
// rows are dealt to the warps.  The rows' magnitudes less their demands travel with P and T, and the finish
// decides which rows to sum on the FP64 pipe.
constexpr int kPW = 4;

// Work memory of the push kernel behind the column's operands: the rows' magnitudes less demands of P and of the four
// T, [5][V][n], and the exponents they are relative to, [5][V].
struct DigRows {
  float* have;
  int* exp;
};
template <int N>
__device__ __forceinline__ DigRows dig_rows_at(void* work, int V) {
  DigRows r;
  r.have = reinterpret_cast<float*>(static_cast<char*>(work) + dig_x_bytes(N, V, 1));
  r.exp = reinterpret_cast<int*>(r.have + (size_t)5 * V * N);
  return r;
}

__device__ __forceinline__ void dig_start(float (&d)[2][2][4], const float (&corr)[4]) {
#pragma unroll
  for (int pl = 0; pl < 2; ++pl)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      d[pl][0][k] = corr[k & 1];
      d[pl][1][k] = corr[2 + (k & 1)];
    }
}

// planes of the four A words times the level operand at `addr`
__device__ __forceinline__ void dig_mul(const uint32_t (&a)[4], uint32_t addr, uint32_t flo, uint32_t fhi,
                                        float (&d)[2][2][4]) {
  uint32_t re[4], im[4], b[4];
  ldsm4(addr, b);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    re[k] = __byte_perm(a[k], 0u, 0x4240);
    im[k] = __byte_perm(a[k], 0u, 0x4341);
  }
  b[0] ^= flo;
  b[2] ^= flo;
  b[1] ^= fhi;
  b[3] ^= fhi;
  mma_f16(d[0][0], re, b[0], b[1]);
  mma_f16(d[0][1], re, b[2], b[3]);
  mma_f16(d[1][0], im, b[0], b[1]);
  mma_f16(d[1][1], im, b[2], b[3]);
}

template <int N>
__global__ void __launch_bounds__(32 * kPW, N == 16 ? 5 : 4) k_push_digits(const __grid_constant__ ApplyArgs a,
                                                             const __grid_constant__ DigArgs dgt) {
  constexpr int NT = N / 16, RS = dig_row<N>(), PS = dig_part<N>(), SL = dig_slab<N>();
  extern __shared__ __align__(16) unsigned char dsm[];  // digit tables (own site, x + mu per warp), tile rings
  __shared__ double part[kPW][2 * N];
  __shared__ float pmag[kPW][N], smag[N];  // magnitudes less demands: forward hops, self block
  __shared__ double scl[kPW][3];
  __shared__ float needs[1 + kPW];
  if (a.stop != nullptr && *a.stop) return;
  const int mu = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int site = blockIdx.x, V = a.V;
  const bool adj = a.adjoint != 0;
  const int src = __ldg(a.nb + site * 8 + mu);
  const uint4* self = dgt.dig + (size_t)site * 5 * NT * NT * 256 + lane;
  const uint4* hop = self + (size_t)(1 + mu) * NT * NT * 256;
  // Tiles of the warp in order: the hop's, then its tile row of the self block; two are in flight in the
  // warp's ring (registers would hold one, and leave room for three CTAs per SM instead of four).
  uint4* ring = reinterpret_cast<uint4*>(dsm + (size_t)(1 + kPW) * SL) + (size_t)mu * 2 * 256 + lane;
  const int tiles = NT * NT + (mu < NT ? NT : 0);
  auto fetch = [&](int i) {
    if (i < tiles) {
      const uint4* from = i < NT * NT ? hop + i * 256 : self + (size_t)(mu * NT + i - NT * NT) * 256;
      const uint32_t to = (uint32_t)__cvta_generic_to_shared(ring + (i & 1) * 256);
#pragma unroll
      for (int p = 0; p < 8; ++p)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + p * 512), "l"(from + p * 32) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  unsigned char* own = dsm;
  unsigned char* nbr = dsm + (size_t)(1 + mu) * SL;
  if (mu == 0) dig_table<N>(own, dgt.xd + (size_t)site * dig_x_halves(N), lane);
  dig_table<N>(nbr, dgt.xd + (size_t)src * dig_x_halves(N), lane);
  if (mu == 0) dig_zero_rows<N, 1>(own, lane);
  dig_zero_rows<N, 1>(nbr, lane);
  float cf[4], cb[4];
  dig_corr(dgt.xc + (size_t)src * kDigCorr, adj, cf, lane);
  dig_corr(dgt.xc + (size_t)site * kDigCorr, !adj, cb, lane);
  asm volatile("cp.async.commit_group;" ::: "memory");  // the tables, then the first two tiles
  fetch(0);
  fetch(1);
  // the warp's product scales (forward hop, push, self block) and demands wait in shared memory: registers are short.
  // Behind the fetches, which would otherwise start one latency later (16^4, n = 48: 2484 against 2464 us)
  if (lane == 0) {
    const double bh = __ldg(dgt.bscale + (size_t)site * 5 + 1 + mu), b0 = __ldg(dgt.bscale + (size_t)site * 5);
    const double x0 = __ldg(dgt.xs + site), xn = __ldg(dgt.xs + src);
    scl[mu][0] = product_scale(bh, xn);
    scl[mu][1] = product_scale(bh, x0);
    scl[mu][2] = product_scale(b0, x0);
    needs[1 + mu] = __ldg(dgt.xn + src);
    if (mu == 0) needs[0] = __ldg(dgt.xn + site);
  }
  asm volatile("cp.async.wait_group 2;" ::: "memory");
  __syncthreads();
  double2* P = static_cast<double2*>(a.part) + (size_t)site * N;
  double2* T = static_cast<double2*>(a.push) + ((size_t)mu * V + site) * N;
  const uint32_t off = (uint32_t)((lane >> 4) * PS + (7 + (lane & 7)) * RS + ((lane >> 3) & 1) * 16);
  const uint32_t of = (uint32_t)__cvta_generic_to_shared(nbr) + off;
  const uint32_t ob = (uint32_t)__cvta_generic_to_shared(own) + off;
  const uint32_t mf = adj ? 0x80008000u : 0u, mb = adj ? 0u : 0x80008000u;
  double pull[NT];
  float mag[4] = {};  // magnitudes: column W the push's tile W, column 3 the self block's, column 4 + U the pull's
  float db[NT][2][2][4];
#pragma unroll
  for (int W = 0; W < NT; ++W) dig_start(db[W], cb);
#pragma unroll
  for (int U = 0; U < NT; ++U) {
    float df[2][2][4];
    dig_start(df, cf);
#pragma unroll
    for (int W = 0; W < NT; ++W) {
      const int i = U * NT + W;
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
      if ((U + 1 + mu) % NT == W) {
        uint32_t m[4];
        dig_mag_tile(ring[(i & 1) * 256], m);
        dig_mags(m, nbr + 2 * PS + W * 32, 4 + U, mag, lane);
        const uint32_t mt[4] = {movmatrix(m[0]), movmatrix(m[2]), movmatrix(m[1]), movmatrix(m[3])};
        dig_mags(mt, own + 2 * PS + U * 32, W, mag, lane);
      }
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        const uint4 w = ring[(i & 1) * 256 + p * 32];
        const uint32_t af[4] = {w.x, w.y, w.z, w.w};
        const uint32_t ab[4] = {movmatrix(w.x), movmatrix(w.z), movmatrix(w.y), movmatrix(w.w)};
        const uint32_t tf = of + (uint32_t)(W * 32 - p * RS), tb = ob + (uint32_t)(U * 32 - p * RS);
        const uint32_t fl = 16 * W >= N / 2 ? mf : 0u, fh = 16 * W + 8 >= N / 2 ? mf : 0u;
        const uint32_t bl = 16 * U >= N / 2 ? mb : 0u, bh2 = 16 * U + 8 >= N / 2 ? mb : 0u;
        dig_mul(af, tf, fl, fh, df);
        dig_mul(ab, tb, bl, bh2, db[W]);
      }
      __syncwarp();  // the slot has been read
      fetch(i + 2);
    }
    const bool neg = adj && 16 * U + g + 8 * (t & 1) >= N / 2;
    pull[U] = dig_flush<false>(df, neg ? -scl[mu][0] : scl[mu][0], lane);
  }
#pragma unroll
  for (int W = 0; W < NT; ++W) {
    const int row = 16 * W + g + 8 * (t & 1);
    const bool neg = !adj && row >= N / 2;
    reinterpret_cast<double*>(T + row)[t >> 1] = dig_flush<true>(db[W], neg ? -scl[mu][1] : scl[mu][1], lane);
  }
  if (mu < NT) {  // tile row mu of the self block
    float ds[2][2][4], cs[4];
    dig_corr(dgt.xc + (size_t)site * kDigCorr, adj, cs, lane);
    dig_start(ds, cs);
#pragma unroll
    for (int W = 0; W < NT; ++W) {
      const int i = NT * NT + W;
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        const uint4 w = ring[(i & 1) * 256 + p * 32];
        const uint32_t af[4] = {w.x, w.y, w.z, w.w};
        if (p == 0 && W == mu) {
          uint32_t m[4];
          dig_mag_tile(w, m);
          dig_mags(m, own + 2 * PS + W * 32, 3, mag, lane);
        }
        const uint32_t ts = ob + (uint32_t)(W * 32 - p * RS);
        const uint32_t fl = 16 * W >= N / 2 ? mf : 0u, fh = 16 * W + 8 >= N / 2 ? mf : 0u;
        dig_mul(af, ts, fl, fh, ds);
      }
      __syncwarp();
      fetch(i + 2);
    }
    const bool neg = adj && 16 * mu + g + 8 * (t & 1) >= N / 2;
    const double v = dig_flush<false>(ds, neg ? -scl[mu][2] : scl[mu][2], lane);
#pragma unroll
    for (int U = 0; U < NT; ++U)
      if (U == mu) pull[U] += v;
  }
#pragma unroll
  for (int U = 0; U < NT; ++U) part[mu][2 * (16 * U + g + 8 * (t & 1)) + (t >> 1)] = pull[U];
  const DigRows rows = dig_rows_at<N>(dgt.work, V);
  const float need = needs[0], needn = needs[1 + mu];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int q = 2 * t + (k & 1), row = g + 8 * (k >> 1);
    const float s0 = mag[k] * 0x1p24f;
    if (q < NT) rows.have[((size_t)(1 + mu) * V + site) * N + 16 * q + row] = s0 - need;
    if (q == 3 && mu < NT) smag[16 * mu + row] = s0 - need;
    if (q >= 4 && q - 4 < NT) pmag[mu][16 * (q - 4) + row] = s0 - needn;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * N; i += blockDim.x)
    reinterpret_cast<double*>(P)[i] = (part[0][i] + part[1][i]) + (part[2][i] + part[3][i]);
  int x[kPW + 1], top = x[kPW] = scale_exp(scl[0][2]);
#pragma unroll
  for (int m = 0; m < kPW; ++m) top = max(top, x[m] = scale_exp(scl[m][0]));
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    float have = scale_weight(x[kPW], top) * smag[i];
#pragma unroll
    for (int m = 0; m < kPW; ++m) have += scale_weight(x[m], top) * pmag[m][i];
    rows.have[(size_t)site * N + i] = have;
  }
  if (lane == 0) rows.exp[(size_t)(1 + mu) * V + site] = scale_exp(scl[mu][1]);
  if (threadIdx.x == 0) rows.exp[site] = top;
}

// y_z = P_z + T_0[z-0] + .. + T_3[z-3] + i mu sigma3 x_z, then the epilogue; one thread per entry.  Rows whose
// magnitudes do not meet their demand are summed on the FP64 pipe, four of a warp's at a time.
template <int N>
__global__ void __launch_bounds__(256, 3) k_push_finish(const __grid_constant__ ApplyArgs a, void* work) {
  if (a.stop != nullptr && *a.stop) return;
  const size_t i = blockIdx.x * (size_t)256 + threadIdx.x;
  const bool in = i < (size_t)a.V * N;
  const int z = in ? (int)(i / N) : 0, e = (int)(i % N), lane = threadIdx.x & 31;
  const double2* T = static_cast<const double2*>(a.push);
  const DigRows rows = dig_rows_at<N>(work, a.V);
  double2 r = make_double2(0.0, 0.0), xs = r, zv = r;
  bool bad = false;
  if (in) {
    double2 t[4];
    float h[4];
    int x[4], from[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) from[mu] = __ldg(a.nb + z * 8 + 4 + mu);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      t[mu] = T[((size_t)mu * a.V + from[mu]) * N + e];
      h[mu] = rows.have[((size_t)(1 + mu) * a.V + from[mu]) * N + e];
      x[mu] = rows.exp[(size_t)(1 + mu) * a.V + from[mu]];
    }
    r = static_cast<const double2*>(a.part)[i];
    xs = static_cast<const double2*>(a.x)[i];
    zv = a.mode == APPLY_AXPBY ? static_cast<const double2*>(a.z)[i] : xs;
    const int x0 = rows.exp[z], top = max(max(max(x0, x[0]), max(x[1], x[2])), x[3]);
    float have = scale_weight(x0, top) * rows.have[i];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) have += scale_weight(x[mu], top) * h[mu];
    bad = top == kNoScale || !(have >= 0.f);
    r = cadd(r, cadd(cadd(t[0], t[1]), cadd(t[2], t[3])));
  }
  const uint32_t m = __ballot_sync(0xffffffffu, bad);
  const int count = __popc(m), rank = __popc(m & ((1u << lane) - 1u));
  for (int q = 0; q < count; q += 4) {  // eight lanes take the q-th such row, the next eight the one after it, ...
    const int l = __fns(m, 0, min(q + (lane >> 3), count - 1) + 1);
    double2 v = dig_plain_row<N>(static_cast<const double2*>(a.blocks), a.nb, a.adjoint != 0,
                                 __shfl_sync(0xffffffffu, z, l), __shfl_sync(0xffffffffu, e, l),
                                 static_cast<const double2*>(a.x));
    v.x = __shfl_sync(0xffffffffu, v.x, 8 * (rank & 3));
    v.y = __shfl_sync(0xffffffffu, v.y, 8 * (rank & 3));
    if (bad && rank >> 2 == q >> 2) r = v;
  }
  if (in) dig_finish<N>(a, r, 0, e, i, 0, xs, zv);
}

// Batched FP64 residual r = b - D x of every pass with an unfinished column (coef: {-1, +1}).
template <int N>
__global__ void __launch_bounds__(32 * kDW, dig_min_blocks(N)) kb_residual_digits(const DigPass* __restrict__ passes,
                                                                  const int* __restrict__ map,
                                                                  const int* __restrict__ flags,
                                                                  const double2* coef) {
  const DigPass& p = passes[__ldg(map + blockIdx.x / kDigMapSites)];
  const int site = blockIdx.x - p.start;
  if (site >= p.V) return;
  if (flags[2 * p.q0 + 1] && flags[2 * (p.q0 + p.cols - 1) + 1]) return;
  const DigX dx = dig_x_at<N>(p.digx, p.V, p.cols);
  DigArgs d;
  d.dig = static_cast<const uint4*>(p.dig);
  d.bscale = p.digscale;
  d.xd = dx.xd;
  d.xc = dx.xc;
  d.xs = dx.xs;
  d.xn = dx.xn;
  d.work = nullptr;
  ApplyArgs a{};
  a.blocks = p.blocks;
  a.nb = p.nb;
  a.x = p.x;
  a.y = p.y;
  a.z = p.z;
  a.coef = coef;
  a.mu = p.mu;
  a.V = p.V;
  a.mode = APPLY_AXPBY;
  dig_site<N, kDigCols>(a, d, site, p.cols, p.ldx, p.ldy, p.ldx);
}

// Two columns: one CTA per site (they share the block operand's loads and byte permutations; dig_columns says
// when).
template <int N>
int launch_dig_2(const ApplyArgs& a, const DigArgs& d, int ncol, long long ldc, cudaStream_t s) {
  constexpr size_t smem = (size_t)kDW * 2 * dig_slab<N>();
  static SmemLimit limit;
  COARSE_CUDA(raise_smem_limit(limit, (const void*)k_site_digits<N, 2>, smem));
  k_site_digits<N, 2><<<a.V, 32 * kDW, smem, s>>>(a, d, ncol, ldc);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

// One column.  From kPushSites sites on every block once (push kernel and its finish); below, where the lattice
// does not fill the chip, one launch of the pull kernel.  Both sides, us, pull / push: 6^4 n = 16 23 / 25, n = 32 49 / 43,
// n = 48 77 / 72; 8^4 n = 16 56 / 52, n = 32 123 / 97, n = 48 215 / 178; 16^4 n = 16 797 / 598, n = 32 1753 / 1237,
// n = 48 3351 / 2465 (1800 at the copy bandwidth).
constexpr int kPushSites = 1024;
template <int N>
int launch_dig_1(const ApplyArgs& a, const DigArgs& d, cudaStream_t s) {
  static SmemLimit push, site;
  constexpr size_t ss = (size_t)kDW * dig_slab<N>(), su = (size_t)(kPW + 1) * dig_slab<N>() + (size_t)kPW * 2 * 4096;
  if (a.V >= kPushSites) {
    COARSE_CUDA(raise_smem_limit(push, (const void*)k_push_digits<N>, su));
    k_push_digits<N><<<a.V, 32 * kPW, su, s>>>(a, d);
    note_launch();
    COARSE_CUDA(cudaGetLastError());
    const size_t total = (size_t)a.V * N;
    k_push_finish<N><<<(unsigned)((total + 255) / 256), 256, 0, s>>>(a, d.work);
  } else {
    COARSE_CUDA(raise_smem_limit(site, (const void*)k_site_digits<N, 1>, ss));
    k_site_digits<N, 1><<<a.V, 32 * kDW, ss, s>>>(a, d, 1, 0);
  }
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

template <int N>
int launch_dig_n(const ApplyArgs& a, const DigUse& use, int ncol, long long ldc, cudaStream_t s) {
  DigArgs d;
  d.dig = static_cast<const uint4*>(use.dig());
  d.bscale = use.scale();
  d.work = use.work();
  const DigX x = dig_x_at<N>(d.work, a.V, ncol);
  d.xd = x.xd;
  d.xc = x.xc;
  d.xs = x.xs;
  d.xn = x.xn;
  k_dig_x<N><<<dim3((a.V + 3) / 4, ncol), 128, 0, s>>>(static_cast<const double2*>(a.x), ldc, a.V, x.xd, x.xc, x.xs,
                                                        x.xn, a.stop);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return ncol == 1 ? launch_dig_1<N>(a, d, s) : launch_dig_2<N>(a, d, ncol, ldc, s);
}

template <int N>
int launch_bresidual_n(const DigPass* passes, const int* map, int sites, const int* flags, const double2* coef,
                       cudaStream_t s) {
  constexpr size_t smem = (size_t)kDW * kDigCols * dig_slab<N>();
  static SmemLimit limit;
  COARSE_CUDA(raise_smem_limit(limit, (const void*)kb_residual_digits<N>, smem));
  kb_dig_x<N><<<sites / 4, 128, 0, s>>>(passes, map, flags);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  kb_residual_digits<N><<<sites, 32 * kDW, smem, s>>>(passes, map, flags, coef);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

}  // namespace

int launch_dig_blocks(const double2* blocks, int V, int n, void* dig, double* scale, cudaStream_t s) {
  k_dig_blocks<<<V * 5, 256, 0, s>>>(blocks, n, static_cast<uint4*>(dig), scale);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

DigPlan dig_plan(const coarse_op* op) {
  DigPlan p;
  p.dig = dig_block_bytes(op->n, op->V);
  p.scale = dig_scale_bytes(op->V);
  p.work = dig_work_bytes(op->n, op->V, op->max_nrhs < kDigCols ? op->max_nrhs : kDigCols);
  p.ctx = op;
  p.pack = [](const void* ctx, void* dig, double* scale, cudaStream_t s) {
    const coarse_op* o = static_cast<const coarse_op*>(ctx);
    return launch_dig_blocks(static_cast<const double2*>(o->blk[COARSE_PREC_FP64].ptr), o->V, o->n, dig, scale, s);
  };
  return p;
}

int launch_apply64(const coarse_op* op, const ApplyArgs& a, cudaStream_t s) {
  const DigUse d(op->digits, dig_plan(op), s);
  if (d.rc() != COARSE_OK) return d.rc();
  return d.dig() ? launch_apply_digits(op->n, a, d, 1, 0, s) : launch_apply(COARSE_PREC_FP64, op->n, a, s);
}

int launch_bresidual_digits(int n, const DigPass* passes, const int* map, int sites, const int* flags,
                            const double2* coef, cudaStream_t s) {
  if (sites <= 0) return COARSE_OK;
  switch (n) {
    case 16: return launch_bresidual_n<16>(passes, map, sites, flags, coef, s);
    case 32: return launch_bresidual_n<32>(passes, map, sites, flags, coef, s);
    case 48: return launch_bresidual_n<48>(passes, map, sites, flags, coef, s);
  }
  set_error("batched residual: unsupported n = %d", n);
  return COARSE_ERR_INVALID_ARG;
}

// The pair kernel reads a hop block twice, the second time from L2 while the lattice is small, and pays the block
// operand's byte permutations once for two columns; the push kernel reads a block once per column.  Two columns, us,
// pair / column by column, by sites:
//           1296        2304        4096        6144        9216        20736
//   n = 16  33 / 50     53 / 66     93 / 105    136 / 142   198 / 197   437 / 412
//   n = 32  64 / 85     103 / 123   172 / 193   249 / 271   378 / 389   862 / 815
//   n = 48  118 / 143   198 / 215   357 / 357   533 / 514   798 / 747   1803 / 1624
// (The batched residual takes pairs at every size: its passes share one launch.)
int dig_columns(int n, int V) { return V >= (n == 16 ? 8192 : n == 32 ? 12288 : 4096) ? 1 : kDigCols; }

int launch_apply_digits(int n, const ApplyArgs& a, const DigUse& d, int ncol, long long ldc, cudaStream_t s) {
  if (ncol < 1 || ncol > kDigCols) {
    set_error("digit stencil: %d columns in one pass", ncol);
    return COARSE_ERR_INVALID_ARG;
  }
  switch (n) {
    case 16: return launch_dig_n<16>(a, d, ncol, ldc, s);
    case 32: return launch_dig_n<32>(a, d, ncol, ldc, s);
    case 48: return launch_dig_n<48>(a, d, ncol, ldc, s);
  }
  set_error("coarse_apply: unsupported n = %d (nv must be 8, 16 or 24)", n);
  return COARSE_ERR_INVALID_ARG;
}

}  // namespace coarse
