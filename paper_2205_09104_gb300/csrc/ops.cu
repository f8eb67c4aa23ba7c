// Block ingest (canonical FP64 Galerkin blocks -> internal 5-block storage in
// FP64 / FP32 / BF16), the sigma3 relation check and the block gradients.
#include "common.cuh"

namespace coarse {
namespace {

// out[x][b][i][j], b = 0 self, 1..4 forward hops.  One thread per complex entry.
__global__ void k_ingest(const double2* self_b, const double2* hop_b, int nhop, int V, int n, double2* o64,
                         float2* o32, cbf16* o16) {
  const size_t nn = (size_t)n * n;
  const size_t total = (size_t)V * 5 * nn;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t x = e / (5 * nn);
    const size_t r = e % (5 * nn);
    const int b = (int)(r / nn);
    const size_t ij = r % nn;
    const double2 v = (b == 0) ? self_b[x * nn + ij] : hop_b[(x * nhop + (b - 1)) * nn + ij];
    if (o64) o64[e] = v;
    if (o32) o32[e] = make_float2((float)v.x, (float)v.y);
    if (o16) {
      cbf16 c;
      c.x = __float2bfloat16_rn((float)v.x);
      c.y = __float2bfloat16_rn((float)v.y);
      o16[e] = c;
    }
  }
}

__device__ void atomic_max_nonneg(double* addr, double v) {
  // non-negative doubles order like their bit patterns
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

// out2[0] = max |defect|, out2[1] = max |entry|.  Defects: backward hop vs sigma3 F^H sigma3 of the
// forward hop of x - mu, and self block vs sigma3 A^H sigma3.
__global__ void k_gamma5_defect(const double2* self_b, const double2* hop_b, int V, int n, const int* nb,
                                double* out2) {
  const int nv = n / 2;
  const size_t nn = (size_t)n * n;
  const size_t total = (size_t)V * 5 * nn;
  double dmax = 0.0, emax = 0.0;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t x = e / (5 * nn);
    const size_t r = e % (5 * nn);
    const int b = (int)(r / nn);
    const int i = (int)((r % nn) / n), j = (int)(r % n);
    const double s = ((i < nv) == (j < nv)) ? 1.0 : -1.0;
    double2 got, ref;
    if (b == 0) {
      got = self_b[x * nn + (size_t)i * n + j];
      const double2 t = self_b[x * nn + (size_t)j * n + i];
      ref = make_double2(s * t.x, -s * t.y);
    } else {
      const int mu = b - 1;
      got = hop_b[(x * 8 + 4 + mu) * nn + (size_t)i * n + j];
      const int xm = nb[x * 8 + 4 + mu];
      const double2 t = hop_b[((size_t)xm * 8 + mu) * nn + (size_t)j * n + i];
      ref = make_double2(s * t.x, -s * t.y);
      const double2 f = hop_b[(x * 8 + mu) * nn + (size_t)i * n + j];
      emax = fmax(emax, fmax(fabs(f.x), fabs(f.y)));
    }
    dmax = fmax(dmax, fmax(fabs(got.x - ref.x), fabs(got.y - ref.y)));
    emax = fmax(emax, fmax(fabs(got.x), fabs(got.y)));
    if (!isfinite(got.x) || !isfinite(got.y)) dmax = INFINITY;
  }
  for (int off = 16; off > 0; off >>= 1) {
    dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, off));
    emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, off));
  }
  if ((threadIdx.x & 31) == 0) {
    atomic_max_nonneg(out2, dmax);
    atomic_max_nonneg(out2 + 1, emax);
  }
}

// G_self[x][i][j] = -lambda_x[i] conj(x_x[j]);  G_hop[x][d][i][j] = -lambda_x[i] conj(x_{nb(x,d)}[j]).
// nhop = 4 (gamma5-compressed input, backward hops derived as sigma3 F_{x-mu,mu}^H sigma3): the
// backward hop of y + mu depends on F_{y,mu} antilinearly, so its gradient folds onto the forward
// block as sigma3 G^H sigma3:  G4[y][mu][i][j] = -lambda_y[i] conj(x_{y+mu}[j])
//                                                 - s_i s_j x_y[i] conj(lambda_{y+mu}[j]).
//
// Bound by the FP64 pipe (four products per entry: 240 us of 8^4 sites, n = 32, nine blocks, against 90 us of
// writes, (1 + nhop) n^2 V complex128).  One CTA per site: the site's lambda (and, for the folded form, x)
// and the source vectors of its blocks are read once into shared memory, then the CTA writes the
// site's blocks in order, 16 bytes per thread and contiguous over the warp, with every index a
// compile-time division.  8^4, n = 32, nine blocks: 0.27 ms; one thread per entry that read its vectors
// through the neighbour table, 0.85 ms.
template <int N, int NHOP>
__global__ void __launch_bounds__(256) k_block_grad(const double2* __restrict__ lam, const double2* __restrict__ xv,
                                                    const int* __restrict__ nb, double2* __restrict__ g_self,
                                                    double2* __restrict__ g_hop) {
  constexpr int NN = N * N, NB = 1 + NHOP, NL = NHOP == 4 ? NB : 1;
  __shared__ double2 xs[NB][N];  // x of the site and of its NHOP neighbours
  __shared__ double2 ls[NL][N];  // lambda of the site (folded form: of its forward neighbours too)
  const size_t x = blockIdx.x;
  for (int e = threadIdx.x; e < NB * N; e += blockDim.x) {
    const int b = e / N, j = e % N;
    const size_t src = b == 0 ? x : (size_t)nb[x * 8 + (b - 1)];
    xs[b][j] = xv[src * N + j];
    if (b < NL) ls[b][j] = lam[src * N + j];
  }
  __syncthreads();
#pragma unroll 1
  for (int b = 0; b < NB; ++b) {
    double2* out = b == 0 ? g_self + x * NN : g_hop + (x * NHOP + (b - 1)) * NN;
    for (int e = threadIdx.x; e < NN; e += 256) {
      const int i = e / N, j = e % N;
      const double2 l = ls[0][i], v = xs[b][j];
      double2 g = make_double2(fma(-l.x, v.x, -l.y * v.y), fma(-l.y, v.x, l.x * v.y));
      if (NHOP == 4 && b > 0) {
        // - s_i s_j x_y[i] conj(lambda_{y+mu}[j]), y the site, y + mu its neighbour b - 1
        const double2 xi = xs[0][i], lj = ls[b < NL ? b : 0][j];
        const double sgn = ((i < N / 2) == (j < N / 2)) ? -1.0 : 1.0;
        g.x += sgn * (xi.x * lj.x + xi.y * lj.y);
        g.y += sgn * (xi.y * lj.x - xi.x * lj.y);
      }
      __stcs(out + e, g);
    }
  }
}

template <int N>
void block_grad_n(const double2* lam, const double2* x, const int* nb, int V, int nhop, double2* g_self,
                  double2* g_hop, cudaStream_t s) {
  if (nhop == 4) k_block_grad<N, 4><<<V, 256, 0, s>>>(lam, x, nb, g_self, g_hop);
  else k_block_grad<N, 8><<<V, 256, 0, s>>>(lam, x, nb, g_self, g_hop);
}

int grid_for(size_t total) {
  size_t g = (total + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  return g < 1 ? 1 : (int)g;
}

}  // namespace

int launch_ingest(const double2* self_b, const double2* hop_b, int gamma5_only, int V, int n, const int* nb,
                  void* out64, void* out32, void* out16, cudaStream_t s) {
  (void)nb;
  const size_t total = (size_t)V * 5 * n * n;
  k_ingest<<<grid_for(total), 256, 0, s>>>(self_b, hop_b, gamma5_only ? 4 : 8, V, n, (double2*)out64,
                                           (float2*)out32, (cbf16*)out16);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

int launch_gamma5_defect(const double2* self_b, const double2* hop_b, int V, int n, const int* nb, double* out2,
                         cudaStream_t s) {
  COARSE_CUDA(cudaMemsetAsync(out2, 0, 2 * sizeof(double), s));
  const size_t total = (size_t)V * 5 * n * n;
  k_gamma5_defect<<<grid_for(total), 256, 0, s>>>(self_b, hop_b, V, n, nb, out2);
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

int launch_block_grad(const double2* lam, const double2* x, const int* nb, int V, int n, int nhop, double2* g_self,
                      double2* g_hop, cudaStream_t s) {
  switch (n) {
    case 16: block_grad_n<16>(lam, x, nb, V, nhop, g_self, g_hop, s); break;
    case 32: block_grad_n<32>(lam, x, nb, V, nhop, g_self, g_hop, s); break;
    case 48: block_grad_n<48>(lam, x, nb, V, nhop, g_self, g_hop, s); break;
    default: set_error("coarse_block_grad: unsupported n = %d", n); return COARSE_ERR_INVALID_ARG;
  }
  note_launch();
  COARSE_CUDA(cudaGetLastError());
  return COARSE_OK;
}

}  // namespace coarse
