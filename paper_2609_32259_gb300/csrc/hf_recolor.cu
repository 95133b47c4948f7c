// hf_recolor_fit: the Recolor initialisation of one map (Section 3.2,
// Eq. 3-5) on the GPU, from weighted aligned sample pairs (X, Y, w):
//   r = sqrt(sum w |x|^2 / (d_S sum w))                               (Eq. 3)
//   Z = X / r; weighted means and covariances of Z and Y
//   R* = polar factor of Sigma_Z^{-1/2} Sigma_ZY Sigma_Y^{-1/2}      (Eq. 4)
//   A = Sigma_Z^{-1/2} R* Sigma_Y^{1/2},  b = mu_Y - mu_Z A           (Eq. 5)
// Any square roots of the covariances give the same A: with the triangular
// factors Sigma_Z = L L^T and Sigma_Y = C C^T (hf_factor.cu),
// Sigma_Z^{-1/2} = L^{-T} Q for an orthogonal Q, which the polar factor takes
// along, so
//   A = L^{-T} polar(L^{-1} Sigma_ZY C^{-T}) C^T,
// one factorisation instead of ~11 iterations of three dense products (at
// 32,768 x 3,072 -> 1,024 the fit took 16.5 ms with iterated roots and three
// dense moment products, 5.2 ms now; fp32 fits with d_S > d_R come out a
// quarter as far from 64 bits).  Only where a pivot is too small
// for fp32 (kPivot of the mean eigenvalue; reg is 0 or tiny and the covariance
// near singular) the symmetric roots are iterated instead, as far as they
// converge: the coupled iteration T = (3I - Z Y) / 2, Y <- Y T, Z <- T Z turns Y_0 = S / c,
// Z_0 = I into (S / c)^{1/2} and (S / c)^{-1/2}; X <- X (3I - X^T X) / 2
// turns X_0 = M into the orthogonal polar factor U Q^T of
// M = U Lambda Q^T (full column rank), which is the R* of Eq. 4.
// Offline (once per map, before folding).  The products are fp32 GEMMs on
// this library's tcgen05 kernel (hf_gemm.cu: each operand split exactly into
// three bf16 parts, six partial products in an fp32 accumulator: fp32
// accuracy); the statistics, centring and elementwise passes are this file's
// kernels.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <utility>

#include <cuda_bf16.h>

#include "hf_internal.h"

namespace hf {
namespace {

// The moments' product runs over the samples in chunks of this many, so the
// bf16 planes of its operand stay a bounded part of the workspace.
constexpr int64_t kMomentChunk = 8192;
// Atoms of 64 samples that one fp32 sum of the moments takes before it goes to
// the matrix: 32 x 16 roundings for 32,768 samples instead of 512 in a row.
constexpr int kMomentFlush = 32;
// A pivot below this share of the mean eigenvalue has lost too many of its
// digits in fp32; the ridge keeps pivots above reg of it (the paper's fits: 1e-3).
constexpr float kPivot = 1e-4f;
// Split-K partials: room for every SM pair's 256 x 256 tile twice over.
constexpr size_t kPartialBytes = static_cast<size_t>(2) * 96 * 65536 * sizeof(float);

hf_status sgemm(const GemmWork& h, cudaStream_t s, int M, int N, int K, float alpha,
                const float* A, int64_t a_i, int64_t a_k, const float* B, int64_t b_k,
                int64_t b_j, float beta, float* C, int64_t ldc, const float* Cin = nullptr,
                float diag = 0.f) {
  return gemm_f32(s, h, M, N, K, alpha, A, a_i, a_k, B, b_k, b_j, beta, C, ldc, Cin, diag);
}

__device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float ld(const float* p) { return *p; }

// Column sums of w [X | Y] and, from X, sum w and sum w |x|^2, in two passes.
// rc_stats_kernel: a warp takes every eighth row of the block's slice and
// 32 V columns per read, four reads of two rows in flight; one fp32 sum takes at
// most 128 values, the rows of a slice, up to 67 M samples (GB300's fp64 rate is a
// small fraction of fp32's), the squares of a row's 4 V values being summed before,
// and the block's partial sums go out as fp64; rc_stats_sum_kernel adds the slices.
// Bounded by reading X and Y once.  (fp64 atomics in the place of the partial
// sums took 0.36 ms for 0.27 GB.)
inline int stat_slices(int64_t N) {
  const int64_t fill = std::min<int64_t>((N + 63) / 64, 128);
  return static_cast<int>(std::min<int64_t>(std::max(fill, (N + 1023) / 1024), 65535));
}
template <typename T, int V>
struct alignas(V * sizeof(T)) StatVec {
  T x[V];
};
template <typename T, int V>
__global__ void __launch_bounds__(256)
    rc_stats_kernel(const T* X, const T* Y, const float* w, int64_t N, int dx, int dy,
                    double* part) {
  constexpr int kCols = 128 * V;  // per block: four reads of a warp
  __shared__ float sums[8][kCols];
  __shared__ double ss[8], sw[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nbx = (dx + kCols - 1) / kCols;
  const bool is_x = static_cast<int>(blockIdx.x) < nbx;
  const int b0 = (is_x ? blockIdx.x : blockIdx.x - nbx) * kCols, d = is_x ? dx : dy;
  const T* const M = is_x ? X : Y;
  const int64_t per = (N + gridDim.y - 1) / gridDim.y;
  const int64_t n0 = blockIdx.y * per, n1 = min(N, n0 + per);
  float s[4 * V], q = 0.f, wt = 0.f;
#pragma unroll
  for (int i = 0; i < 4 * V; ++i) s[i] = 0.f;
#pragma unroll 2
  for (int64_t n = n0 + warp; n < n1; n += 8) {
    const float wn = w[n];
    const T* row = M + n * d;
    StatVec<T, V> v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = b0 + (lane + 32 * i) * V;  // d is a multiple of V
      if (c < d)
        v[i] = *reinterpret_cast<const StatVec<T, V>*>(row + c);
      else
        for (int k = 0; k < V; ++k) v[i].x[k] = T(0.f);
    }
    float row_q = 0.f;
#pragma unroll
    for (int i = 0; i < 4 * V; ++i) {
      const float x = ld(&v[i / V].x[i % V]), wv = wn * x;
      s[i] += wv;
      row_q = fmaf(wv, x, row_q);
    }
    q += row_q;
    wt += wn;
  }
#pragma unroll
  for (int i = 0; i < 4 * V; ++i) sums[warp][(lane + 32 * (i / V)) * V + i % V] = s[i];
  double dq = q;
  for (int o = 16; o > 0; o >>= 1) dq += __shfl_xor_sync(0xffffffffu, dq, o);
  if (lane == 0) {
    ss[warp] = dq;
    sw[warp] = wt;
  }
  __syncthreads();
  // a slice's row: the sums of X's and Y's columns, sum w, sum w |x|^2 of each
  // of X's column blocks
  double* const out = part + static_cast<int64_t>(blockIdx.y) * (dx + dy + 1 + nbx);
  for (int c = threadIdx.x; c < kCols; c += blockDim.x) {
    if (b0 + c >= d) break;
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += sums[k][c];
    out[(is_x ? 0 : dx) + b0 + c] = t;
  }
  if (is_x && threadIdx.x == 0) {
    double t = 0.0, u = 0.0;
    for (int k = 0; k < 8; ++k) {
      t += ss[k];
      u += sw[k];
    }
    if (blockIdx.x == 0) out[dx + dy] = u;
    out[dx + dy + 1 + blockIdx.x] = t;
  }
}

// sums[c] = the slices' sums of column c, c <= d (the last one sum w): 32
// columns a block, eight threads each; the grid's last block adds up the nbx
// columns of sum w |x|^2 into sums[d + 1].
__global__ void __launch_bounds__(256)
    rc_stats_sum_kernel(const double* part, int slices, int d, int nbx, double* sums) {
  __shared__ double sh[8][33];
  const int lane = threadIdx.x & 31, y = threadIdx.x >> 5, stride = d + 1 + nbx;
  const bool ss = blockIdx.x == gridDim.x - 1;
  const int c = blockIdx.x * 32 + lane;
  double t = 0.0;
  if (ss) {
    for (int i = threadIdx.x; i < slices * nbx; i += 256)
      t += part[static_cast<int64_t>(i / nbx) * stride + d + 1 + i % nbx];
  } else if (c <= d) {
#pragma unroll 8
    for (int i = y; i < slices; i += 8) t += part[static_cast<int64_t>(i) * stride + c];
  }
  sh[y][lane] = t;
  __syncthreads();
  if (y != 0) return;
  for (int k = 1; k < 8; ++k) t += sh[k][lane];
  if (ss) {
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) sums[d + 1] = t;
  } else if (c <= d) {
    sums[c] = t;
  }
}

// fp32 means mu_x (of X, not yet divided by r), mu_y, and [1 / W, 1 / r].
__global__ void rc_mean_kernel(const double* sx, const double* sy, const double* sw_ss, int dx,
                               int dy, float* mu, float* scal) {
  const double W = sw_ss[0];
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < dx + dy; c += gridDim.x * blockDim.x)
    mu[c] = static_cast<float>((c < dx ? sx[c] : sy[c - dx]) / W);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    scal[0] = static_cast<float>(1.0 / W);
    scal[1] = static_cast<float>(1.0 / sqrt(sw_ss[1] / (static_cast<double>(dx) * W)));
  }
}

// Centred, weighted samples as the moments' operand: feature f of sample n is
// sqrt(w / W) (x - mu_x) / r (f < dx), sqrt(w / W) (y - mu_y) (np <= f <
// np + dy), 0 elsewhere and past the last sample; written as the three bf16
// planes of gemm_planes, feature-major, for the samples n0 .. n0 + k_p - 1.
// A block turns 64 features x 64 samples through shared memory, read along the
// features and written along the samples, 128 bytes each way: 6 bytes written
// per value are what bounds it (32,768 x 4,096: 0.8 GB written, 0.27 GB read),
// where an fp32 copy of the centred samples cost 0.46 ms and its split
// another 0.4 ms.
template <typename T>
__global__ void __launch_bounds__(256)
    rc_planes_kernel(const T* X, const T* Y, const float* w, int64_t N, int64_t n0, int dx, int dy,
                     int np, const float* mu, const float* scal, __nv_bfloat16* out,
                     int64_t rows_p, int64_t k_p) {
  __shared__ float tile[64][65];
  __shared__ float scale[64];
  const int f0 = blockIdx.y * 64, k0 = blockIdx.x * 64;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float inv_w = scal[0], inv_r = scal[1];
  if (threadIdx.x < 64) {
    const int64_t n = n0 + k0 + threadIdx.x;
    scale[threadIdx.x] = n < N ? sqrtf(w[n] * inv_w) : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int f = f0 + lane + 32 * h;
    const bool is_x = f < dx, is_y = f >= np && f < np + dy;
    const T* src = is_x ? X + f : Y + (f - np);
    const int64_t step = is_x ? dx : dy;
    const float m = is_x ? mu[f] : is_y ? mu[dx + f - np] : 0.f;
    const float mul = is_x ? inv_r : 1.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = warp + 8 * i;
      const int64_t n = n0 + k0 + k;
      float v = 0.f;
      if ((is_x || is_y) && n < N) v = scale[k] * (ld(src + n * step) - m) * mul;
      tile[k][lane + 32 * h] = v;
    }
  }
  __syncthreads();
  const int64_t plane = rows_p * k_p / 2;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int f = warp + 8 * i;
    const float a = tile[2 * lane][f], b = tile[2 * lane + 1][f];
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(a, b);
    const float2 g0 = __bfloat1622float2(h0);
    const float ra = a - g0.x, rb = b - g0.y;
    const __nv_bfloat162 h1 = __floats2bfloat162_rn(ra, rb);
    const float2 g1 = __bfloat1622float2(h1);
    __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(out + (f0 + f) * k_p + k0) + lane;
    o[0] = h0;
    o[plane] = h1;
    o[2 * plane] = __floats2bfloat162_rn(ra - g1.x, rb - g1.y);
  }
}

// S += reg * trace(S) / d * I for the d x d matrix at S; the diagonal of its
// padding, up to n, becomes the mean eigenvalue; *thr receives the smallest
// pivot to accept (one block of 256 threads).
__global__ void rc_ridge_kernel(float* S, int64_t ld, int d, int n, float reg, float* thr) {
  __shared__ double part[256];
  double t = 0.0;
  for (int i = threadIdx.x; i < d; i += blockDim.x) t += S[i * ld + i];
  part[threadIdx.x] = t;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
    __syncthreads();
  }
  const float mean = static_cast<float>(part[0] / d);
  const float add = reg * mean;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    if (i < d)
      S[i * ld + i] += add;
    else
      S[i * ld + i] = mean;
  }
  if (threadIdx.x == 0) *thr = kPivot * mean;
}

// out (rows x cols, dense) from the matrix at S: mode 0 as it is, 1 the
// symmetric matrix whose upper triangle S holds, 2 the lower triangle with
// zeros above it.
__global__ void rc_extract_kernel(const float* S, int64_t ld, int rows, int cols, int mode,
                                  float* out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= cols) return;
  for (int i = blockIdx.y; i < rows; i += gridDim.y) {
    float v = 0.f;
    if (mode == 1 && i > j)
      v = S[j * ld + i];
    else if (mode != 2 || j <= i)
      v = S[i * ld + j];
    out[static_cast<int64_t>(i) * cols + j] = v;
  }
}

// *out = trace(S) (one block of 256 threads).
__global__ void rc_trace_kernel(const float* S, int d, double* out) {
  __shared__ double part[256];
  double t = 0.0;
  for (int i = threadIdx.x; i < d; i += blockDim.x) t += S[static_cast<int64_t>(i) * d + i];
  part[threadIdx.x] = t;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = part[0];
}

// out = a * in + b * I (square, or the leading square of a d x e matrix when
// only scaling: b = 0).
__global__ void rc_affine_kernel(float* out, const float* in, int64_t n_el, int cols, float a,
                                 float b) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_el;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / cols, c = i - r * cols;
    out[i] = a * (in ? in[i] : 0.f) + (r == c ? b : 0.f);
  }
}

// sum of squares of x, or of (x - I) when minus_identity: fp32 per thread
// (a few dozen elements each), fp64 across threads, one atomic per block (one
// per warp made the 1,024-square pass 17 us of queueing on one address).
__global__ void __launch_bounds__(256)
    rc_sumsq_kernel(const float* x, int64_t n_el, int cols, int minus_identity, double* out) {
  __shared__ double part[8];
  float s = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_el;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / cols, c = i - r * cols;
    const float v = x[i] - (minus_identity && r == c ? 1.f : 0.f);
    s = fmaf(v, v, s);
  }
  double q = s;
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = q;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) q += part[k];
    atomicAdd(out, q);
  }
}

// W_out = A^T in the output type: 32 x 32 tiles through shared memory, read
// and written along rows.
template <typename T>
__global__ void rc_transpose_kernel(const float* A, int dx, int dy, T* W_out) {
  __shared__ float tile[32][33];
  const int k0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int k = k0 + i, j = j0 + threadIdx.x;
    if (k < dx && j < dy) tile[i][threadIdx.x] = A[static_cast<int64_t>(k) * dy + j];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int j = j0 + i, k = k0 + threadIdx.x;
    if (k < dx && j < dy) W_out[static_cast<int64_t>(j) * dx + k] = T(tile[threadIdx.x][i]);
  }
}

// b = mu_y - mu_z A, mu_z = mu_x / r.  Block (j-tile of 32 columns, slice of
// 256 rows of A): thread (j, sub) sums 32 rows in fp64, the block combines its
// eight partial sums and adds them to bacc[j] (cleared before).
__global__ void rc_bias_partial_kernel(const float* A, int dx, int dy, const double* sx,
                                       const double* sw_ss, double* bacc) {
  __shared__ double part[8][33];
  const double W = sw_ss[0];
  const double inv = 1.0 / (W * sqrt(sw_ss[1] / (static_cast<double>(dx) * W)));
  const int j = blockIdx.x * 32 + threadIdx.x;
  const int kbase = blockIdx.y * 256 + threadIdx.y * 32;
  double s = 0.0;
  if (j < dy)
    for (int k = kbase; k < min(dx, kbase + 32); ++k)
      s = fma(sx[k] * inv, static_cast<double>(A[static_cast<int64_t>(k) * dy + j]), s);
  part[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && j < dy) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += part[q][threadIdx.x];
    atomicAdd(bacc + j, t);
  }
}

__global__ void rc_bias_final_kernel(const double* sy, const double* sw_ss, const double* bacc,
                                     int dy, float* b_out) {
  const double W = sw_ss[0];
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < dy; j += gridDim.x * blockDim.x)
    b_out[j] = static_cast<float>(sy[j] / W - bacc[j]);
}

struct Rc {
  size_t stats, part, bacc, mu, gram, tt, fplanes, fplanes_y, thr, flag, sz, sy, szy, p1, p2, p3, p4, sz_ih, sy_ih,
      sy_h, m, x1, x2, xtx, a, planes_a, planes_b, partial, err, total;
  size_t planes_a_bytes, planes_b_bytes;
  int np, mp, F;     // features of X and of Y padded to whole factor blocks; their sum
  int64_t chunk;     // samples per moments product (a multiple of 64)
};

Rc rc_layout(int64_t N, int dx, int dy) {
  Rc L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 255) / 256 * 256;
    return at;
  };
  const size_t f = sizeof(float);
  const size_t dmax = static_cast<size_t>(dx > dy ? dx : dy);
  L.stats = take(sizeof(double) * (dx + dy + 4));
  L.part = take(sizeof(double) * stat_slices(N) * (dx + dy + 1 + (dx + 127) / 128));
  L.bacc = take(sizeof(double) * dy);
  L.mu = take(f * (dx + dy + 2));
  auto up = [](int64_t x, int64_t a) { return (x + a - 1) / a * a; };
  L.np = static_cast<int>(up(dx, kFactorBlock));
  L.mp = static_cast<int>(up(dy, kFactorBlock));
  L.F = L.np + L.mp;
  L.chunk = std::min<int64_t>(up(N, 64), kMomentChunk);
  L.gram = take(f * L.F * L.F);
  L.tt = take(2 * f * kFactorBlock * kFactorBlock);
  L.fplanes = take(tri_factor_planes_bytes(L.np));
  L.fplanes_y = take(tri_factor_planes_bytes(L.mp));
  L.thr = take(f * 2);
  L.flag = take(sizeof(int32_t));
  L.sz = take(f * dx * dx);
  L.sy = take(f * dy * dy);
  L.szy = take(f * dx * dy);
  L.p1 = take(f * dmax * dmax);
  L.p2 = take(f * dmax * dmax);
  L.p3 = take(f * dmax * dmax);
  L.p4 = take(f * dmax * dmax);
  L.sz_ih = take(f * dx * dx);
  L.sy_ih = take(f * dy * dy);
  L.sy_h = take(f * dy * dy);
  L.m = take(f * dx * dy);
  L.x1 = take(f * dx * dy);
  L.x2 = take(f * dx * dy);
  L.xtx = take(f * dy * dy);
  L.a = take(f * dx * dy);
  // bf16 planes of the products' operands; the moments' operand holds every
  // feature for one chunk of samples
  L.planes_b_bytes = gemm_planes_bytes(static_cast<int64_t>(dmax), static_cast<int64_t>(dmax));
  L.planes_a_bytes = std::max(L.planes_b_bytes, gemm_planes_bytes(L.F, L.chunk));
  L.planes_a = take(L.planes_a_bytes);
  L.planes_b = take(L.planes_b_bytes);
  L.partial = take(kPartialBytes);
  L.err = take(sizeof(int32_t));
  L.total = off;
  return L;
}

hf_status read_double(cudaStream_t s, const double* d, double* h) {
  HF_CUDA_TRY(cudaMemcpyAsync(h, d, sizeof(double), cudaMemcpyDeviceToHost, s), "read back");
  HF_CUDA_TRY(cudaStreamSynchronize(s), "synchronize");
  return HF_OK;
}

constexpr int kMaxIter = 80;
constexpr double kTol = 2e-5;  // |X - I|_F / sqrt(d) at convergence

// Convergence test of an iteration's residual e (checked every 4 steps):
// below the tolerance, or no longer falling once small (the fp32 floor).
bool converged(double e, double* prev) {
  const bool done = e < kTol || (e < 1e-3 && e >= 0.5 * *prev);
  *prev = e;
  return done;
}

// Newton-Schulz square root and inverse square root of the SPD matrix S
// (d x d): root = S^{1/2} (when root is not null), inv_root = S^{-1/2}; Y, Z, T, U
// are d x d work buffers distinct from both.
// The coupled iteration Y <- Y T, Z <- T Z, T = (3I - Z Y) / 2 acts on each
// eigenvalue x^2 of Z Y (x the corresponding eigenvalue of (S/c)^{1/2}
// polynomials) as the cubic sign iteration x <- x (3 - x^2) / 2, which
// lifts small x by only 1.5 per step.  With a lower bound l <= x <= 1 (the
// ridge reg * trace / d bounds the smallest eigenvalue of S from below),
// each step first scales Y and Z by b = sqrt(3 / (l^2 + l + 1)), the factor
// for which the cubic maps [b l, b] onto [p(b l), 1] with p(b l) = p(b)
// (the scaled Newton-Schulz step that maximises the new lower bound): small
// x then grow by ~2.6 per step, and b -> 1 as l -> 1.  Scaling Y and Z
// together keeps Y = (S/c) Z, so the limits are unchanged.  With reg = 0
// there is no bound and the plain iteration runs.
hf_status ns_sqrt(cudaStream_t s, const GemmWork& h, const float* S, int d, float reg, float* Y, float* Z, float* T, float* U,
                  float* root, float* inv_root, double* dscr, int* iters) {
  const int64_t n_el = static_cast<int64_t>(d) * d;
  const int grid = 1024;
  double c2 = 0.0;
  HF_CUDA_TRY(cudaMemsetAsync(dscr, 0, sizeof(double), s), "clear");
  rc_sumsq_kernel<<<2 * device_sm_count(), 256, 0, s>>>(S, n_el, d, 0, dscr);
  hf_status st = read_double(s, dscr, &c2);
  if (st != HF_OK) return st;
  const double c = sqrt(c2);
  if (!(c > 0.0)) {
    set_error("hf_recolor_fit: a covariance is zero");
    return HF_ERR_INVALID_ARGUMENT;
  }
  double l = 0.0;  // lower bound of the eigenvalues x of (Z Y)^{1/2}
  if (reg > 0.f) {
    rc_trace_kernel<<<1, 256, 0, s>>>(S, d, dscr);
    double tr = 0.0;
    if ((st = read_double(s, dscr, &tr)) != HF_OK) return st;
    // S = S0 + reg tr(S0)/d I with S0 >= 0 and tr(S) = (1 + reg) tr(S0)
    const double lam_lo = reg * tr / (static_cast<double>(d) * (1.0 + reg));
    if (lam_lo > 0.0) l = std::min(1.0, sqrt(lam_lo / c));
  }
  rc_affine_kernel<<<grid, 256, 0, s>>>(Y, S, n_el, d, static_cast<float>(1.0 / c), 0.f);
  rc_affine_kernel<<<grid, 256, 0, s>>>(Z, nullptr, n_el, d, 0.f, 1.f);
  int it = 0;
  double prev = 1e30;
  for (; it < kMaxIter; ++it) {
    const double b = l > 0.0 ? sqrt(3.0 / (l * l + l + 1.0)) : 1.0;
    // T = 1.5 I - 0.5 b^2 Z Y
    if ((st = sgemm(h, s, d, d, d, static_cast<float>(-0.5 * b * b), Z, d, 1, Y, d, 1, 0.f, T,
                    d, nullptr, 1.5f)) != HF_OK)
      return st;
    // the residual |I - Z Y| = 2 |T - I| holds for unscaled steps
    if (it % 4 == 3 && b < 1.0 + 1e-6) {
      double e2 = 0.0;
      HF_CUDA_TRY(cudaMemsetAsync(dscr, 0, sizeof(double), s), "clear");
      // |I - Z Y| = 2 |T - I|
      rc_sumsq_kernel<<<2 * device_sm_count(), 256, 0, s>>>(T, n_el, d, 1, dscr);
      if ((st = read_double(s, dscr, &e2)) != HF_OK) return st;
      if (converged(2.0 * sqrt(e2 / d), &prev)) break;
    }
    const float bf = static_cast<float>(b);
    if ((st = sgemm(h, s, d, d, d, bf, Y, d, 1, T, d, 1, 0.f, U, d)) != HF_OK) return st;  // b Y T
    std::swap(Y, U);
    if ((st = sgemm(h, s, d, d, d, bf, T, d, 1, Z, d, 1, 0.f, U, d)) != HF_OK) return st;  // b T Z
    std::swap(Z, U);
    l = std::min(1.0, b * l * (3.0 - b * b * l * l) / 2.0);
  }
  *iters = it;
  // inv_root first: root may be null (not wanted), and neither may alias the
  // work buffers, which Y and Z rotate through
  rc_affine_kernel<<<grid, 256, 0, s>>>(inv_root, Z, n_el, d, static_cast<float>(1.0 / sqrt(c)),
                                        0.f);
  if (root)
    rc_affine_kernel<<<grid, 256, 0, s>>>(root, Y, n_el, d, static_cast<float>(sqrt(c)), 0.f);
  HF_CUDA_TRY(cudaGetLastError(), "hf_recolor_fit: iteration launch");
  return HF_OK;
}

constexpr double kPolarNear = 0.5, kPolarTol = 5e-8;

// Orthogonal polar factor of M (dx x dy, dx >= dy, full column rank):
// X <- X (3I - X^T X) / 2 from X_0 = M / min(|M|_F, 1).  M is the whitened
// cross-covariance Sigma_Z^{-1/2} Sigma_ZY Sigma_Y^{-1/2} of one weighted
// sample set, so its singular values (canonical correlations; the ridges
// only lower them) are at most 1 (Cauchy-Schwarz), and the iteration needs
// no smaller scale: dividing by |M|_F = sqrt(sum of squared correlations)
// would only shrink them and add ~log_1.5 |M|_F steps.  A step takes each
// singular value's error e = 1 - x^2 to e^2 (3 + e) / 4, and |X^T X - I|_F is at
// least the largest of them: once it is below kPolarNear the steps to
// kPolarTol are counted ahead, and no check, whose result the host waits for,
// comes after (a fit of 32,768 x 3,072 -> 1,024 takes six steps and products
// X^T X; seven and eight with a check every fourth step: 5.39 ms, 5.22 now).  Result in *out (one of the two buffers).
hf_status ns_polar(cudaStream_t s, const GemmWork& h, const float* M, int dx, int dy, float* X, float* X2,
                   float* P, double* dscr, float** out, int* iters) {
  const int64_t n_el = static_cast<int64_t>(dx) * dy, p_el = static_cast<int64_t>(dy) * dy;
  const int grid = 1024;
  double m2 = 0.0;
  HF_CUDA_TRY(cudaMemsetAsync(dscr, 0, sizeof(double), s), "clear");
  rc_sumsq_kernel<<<2 * device_sm_count(), 256, 0, s>>>(M, n_el, dy, 0, dscr);
  hf_status st = read_double(s, dscr, &m2);
  if (st != HF_OK) return st;
  if (!(m2 > 0.0)) {
    set_error("hf_recolor_fit: the cross-covariance is zero");
    return HF_ERR_INVALID_ARGUMENT;
  }
  rc_affine_kernel<<<grid, 256, 0, s>>>(X, M, n_el, dy,
                                        static_cast<float>(1.0 / std::min(sqrt(m2), 1.0)), 0.f);
  int it = 0, check = 3, left = -1;  // left: the steps still to go, once that is known
  for (; it < kMaxIter && left != 0; ++it) {
    // P = X^T X
    if ((st = sgemm(h, s, dy, dy, dx, 1.f, X, 1, dy, X, dy, 1, 0.f, P, dy)) != HF_OK) return st;
    if (left > 0) {
      --left;
    } else if (it == check) {
      double e2 = 0.0;
      HF_CUDA_TRY(cudaMemsetAsync(dscr, 0, sizeof(double), s), "clear");
      rc_sumsq_kernel<<<2 * device_sm_count(), 256, 0, s>>>(P, p_el, dy, 1, dscr);
      if ((st = read_double(s, dscr, &e2)) != HF_OK) return st;
      double e = sqrt(e2);
      check += 2;
      if (e < kPolarNear)
        for (left = 0; e > kPolarTol; ++left) e = e * e * (0.75 + 0.25 * e);
      if (left == 0) break;
      if (left > 0) --left;
    }
    // X2 = 1.5 X - 0.5 X P
    if ((st = sgemm(h, s, dx, dy, dy, -0.5f, X, dy, 1, P, dy, 1, 1.5f, X2, dy, X)) != HF_OK)
      return st;
    std::swap(X, X2);
  }
  *iters = it;
  *out = X;
  HF_CUDA_TRY(cudaGetLastError(), "hf_recolor_fit: iteration launch");
  return HF_OK;
}

template <typename T>
hf_status recolor_typed(int64_t N, int dx, int dy, const void* Xv, const void* Yv, const float* w,
                        float reg, void* W_out, float* b_out, float* h_r, int32_t* h_iters,
                        char* ws, cudaStream_t s) {
  const Rc L = rc_layout(N, dx, dy);
  double* stats = reinterpret_cast<double*>(ws + L.stats);
  double* sx = stats;
  double* sy = sx + dx;
  double* sw_ss = sy + dy;    // [0] sum w, [1] sum w |x|^2
  double* dscr = sw_ss + 2;   // scratch scalar
  auto F = [&](size_t off) { return reinterpret_cast<float*>(ws + off); };
  const T* X = static_cast<const T*>(Xv);
  const T* Y = static_cast<const T*>(Yv);
  GemmWork h;
  h.planes_a = ws + L.planes_a;
  h.planes_b = ws + L.planes_b;
  h.planes_a_bytes = L.planes_a_bytes;
  h.planes_b_bytes = L.planes_b_bytes;
  h.partial = F(L.partial);
  h.partial_bytes = kPartialBytes;
  h.err = reinterpret_cast<int32_t*>(ws + L.err);
  HF_CUDA_TRY(cudaMemsetAsync(h.err, 0, sizeof(int32_t), s), "clear");
  HF_CUDA_TRY(cudaMemsetAsync(stats, 0, sizeof(double) * (dx + dy + 4), s), "clear");
  const int d = dx + dy;
  {
    double* const part = reinterpret_cast<double*>(ws + L.part);
    const int slices = stat_slices(N);
    const bool pairs = dx % 2 == 0 && dy % 2 == 0 &&
                       ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) &
                        (2 * sizeof(T) - 1)) == 0;
    const int cols = pairs ? 256 : 128;
    const int nbx = (dx + cols - 1) / cols, nby = (dy + cols - 1) / cols;
    if (pairs)
      rc_stats_kernel<T, 2><<<dim3(nbx + nby, slices), 256, 0, s>>>(X, Y, w, N, dx, dy, part);
    else
      rc_stats_kernel<T, 1><<<dim3(nbx + nby, slices), 256, 0, s>>>(X, Y, w, N, dx, dy, part);
    rc_stats_sum_kernel<<<(d + 32) / 32 + 1, 256, 0, s>>>(part, slices, d, nbx, sx);
  }
  float* mu = F(L.mu);
  rc_mean_kernel<<<(d + 255) / 256, 256, 0, s>>>(sx, sy, sw_ss, dx, dy, mu, mu + d);
  HF_CUDA_TRY(cudaGetLastError(), "hf_recolor_fit: statistics launch");
  hf_status st;
  float* const G = F(L.gram);   // [Sigma_Z Sigma_ZY; . Sigma_Y], upper 256-tiles
  float* const GY = G + static_cast<int64_t>(L.np) * L.F + L.np;
  float* const thr = F(L.thr);
  int32_t* const flag = reinterpret_cast<int32_t*>(ws + L.flag);
  const int64_t rows_p = (L.F + 255) / 256 * 256;
  // The second moments of both sides are one symmetric product, of which the
  // upper 256 x 256 tiles are computed (32,768 x (3,072 + 1,024): 2.2 ms; three
  // separate dense products took 3.65 ms)
  auto moments = [&]() -> hf_status {
    HF_CUDA_TRY(cudaMemsetAsync(G, 0, sizeof(float) * L.F * L.F, s), "clear");
    for (int64_t k0 = 0; k0 < N; k0 += L.chunk) {
      const int k_p = static_cast<int>((std::min<int64_t>(L.chunk, N - k0) + 63) / 64 * 64);
      rc_planes_kernel<T><<<dim3(k_p / 64, static_cast<unsigned>(rows_p / 64)), 256, 0, s>>>(
          X, Y, w, N, k0, dx, dy, L.np, mu, mu + d, static_cast<__nv_bfloat16*>(h.planes_a),
          rows_p, k_p);
      HF_CUDA_TRY(cudaGetLastError(), "hf_recolor_fit: moments launch");
      const GemmPlanes z{h.planes_a, rows_p, 0};
      GemmShape upper;
      upper.tri = true;
      upper.flush = kMomentFlush;
      const hf_status e = gemm_planes(s, h, L.F, L.F, k_p, 1.f, z, z, 1.f, G, L.F, upper);
      if (e != HF_OK) return e;
    }
    rc_ridge_kernel<<<1, 256, 0, s>>>(G, L.F, dx, L.np, reg, thr);
    rc_ridge_kernel<<<1, 256, 0, s>>>(GY, L.F, dy, L.mp, reg, thr + 1);
    HF_CUDA_TRY(cudaGetLastError(), "hf_recolor_fit: ridge launch");
    return HF_OK;
  };
  auto extract_ld = [&](const float* S, int64_t ld, int rows, int cols, int mode, float* out) {
    rc_extract_kernel<<<dim3((cols + 255) / 256, std::min(rows, 1024)), 256, 0, s>>>(
        S, ld, rows, cols, mode, out);
  };
  auto extract = [&](const float* S, int rows, int cols, int mode, float* out) {
    extract_ld(S, L.F, rows, cols, mode, out);
  };
  if ((st = moments()) != HF_OK) return st;
  // no pivot is below the ridge but for rounding: with a larger one the roots are not
  // to be expected, and taking the moments again (2.5 ms of a fit of 32,768 x 3,072 ->
  // 1,024 with roots, 20.5 ms) is dearer than these copies only then
  const bool kept = reg < 2.f * kPivot;
  if (kept) {
    extract(G, dx, dx, 0, F(L.p1));
    extract(GY, dy, dy, 0, F(L.p2));
  }
  HF_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(int32_t), s), "clear");
  HF_CUDA_TRY(cudaMemsetAsync(F(L.sy_h), 0, sizeof(float) * dy * dy, s), "clear");
  const TriProblem tri[2] = {
      {G, L.F, L.np, F(L.tt), ws + L.fplanes, thr, nullptr, 0},
      {GY, L.F, L.mp, F(L.tt) + kFactorBlock * kFactorBlock, ws + L.fplanes_y, thr + 1, F(L.sy_h), dy}};
  if ((st = tri_factor(s, h, tri, 2, flag)) != HF_OK) return st;
  extract(G, dx, dx, 2, F(L.sz_ih));   // L^{-1}
  extract(GY, dy, dy, 2, F(L.sy_ih));  // C^{-1}
  int32_t weak = 0;
  HF_CUDA_TRY(cudaMemcpyAsync(&weak, flag, sizeof(weak), cudaMemcpyDeviceToHost, s), "read back");
  HF_CUDA_TRY(cudaStreamSynchronize(s), "synchronize");
  int it1 = 1, it2 = 1, it3 = 0;
  const int64_t left_i = weak ? dx : 1, left_k = weak ? 1 : dx;  // left root: symmetric, or L^{-T}
  if (weak) {
    if (!kept) {
      if ((st = moments()) != HF_OK) return st;
      extract(G, dx, dx, 0, F(L.p1));
      extract(GY, dy, dy, 0, F(L.p2));
    }
    extract_ld(F(L.p1), dx, dx, dx, 1, F(L.sz));
    extract_ld(F(L.p2), dy, dy, dy, 1, F(L.sy));
    extract(G + L.np, dx, dy, 0, F(L.szy));
    if ((st = ns_sqrt(s, h, F(L.sz), dx, reg, F(L.p1), F(L.p2), F(L.p3), F(L.p4), nullptr,
                      F(L.sz_ih), dscr, &it1)) != HF_OK)
      return st;
    if ((st = ns_sqrt(s, h, F(L.sy), dy, reg, F(L.p1), F(L.p2), F(L.p3), F(L.p4), F(L.sy_h),
                      F(L.sy_ih), dscr, &it2)) != HF_OK)
      return st;
    // M = Sigma_Z^{-1/2} Sigma_ZY Sigma_Y^{-1/2}
    if ((st = sgemm(h, s, dx, dy, dx, 1.f, F(L.sz_ih), dx, 1, F(L.szy), dy, 1, 0.f, F(L.x2), dy)) !=
        HF_OK)
      return st;
    if ((st = sgemm(h, s, dx, dy, dy, 1.f, F(L.x2), dy, 1, F(L.sy_ih), dy, 1, 0.f, F(L.m), dy)) !=
        HF_OK)
      return st;
  } else {
    // M = (L^{-1} Sigma_ZY) C^{-T}, by products with the computed inverses:
    // what is off in them cancels against A's outer factors, where Sigma_ZY
    // eliminated along with Sigma_Z takes rounding errors of its own (square
    // fits came out 1.5 times as far off)
    if ((st = sgemm(h, s, dx, dy, dx, 1.f, F(L.sz_ih), dx, 1, G + L.np, L.F, 1, 0.f, F(L.x2), dy)) !=
        HF_OK)
      return st;
    if ((st = sgemm(h, s, dx, dy, dy, 1.f, F(L.x2), dy, 1, F(L.sy_ih), 1, dy, 0.f, F(L.m), dy)) !=
        HF_OK)
      return st;
  }
  float* R = nullptr;
  if ((st = ns_polar(s, h, F(L.m), dx, dy, F(L.x1), F(L.x2), F(L.xtx), dscr, &R, &it3)) != HF_OK)
    return st;
  // A = Sigma_Z^{-1/2} R* Sigma_Y^{1/2}, or L^{-T} R* C^T
  float* tmp = R == F(L.x1) ? F(L.x2) : F(L.x1);
  if ((st = sgemm(h, s, dx, dy, dx, 1.f, F(L.sz_ih), left_i, left_k, R, dy, 1, 0.f, tmp, dy)) != HF_OK)
    return st;
  if ((st = sgemm(h, s, dx, dy, dy, 1.f, tmp, dy, 1, F(L.sy_h), dy, 1, 0.f, F(L.a), dy)) != HF_OK)
    return st;
  {
    double* bacc = reinterpret_cast<double*>(ws + L.bacc);
    HF_CUDA_TRY(cudaMemsetAsync(bacc, 0, sizeof(double) * dy, s), "clear");
    rc_transpose_kernel<T><<<dim3((dy + 31) / 32, (dx + 31) / 32), dim3(32, 8), 0, s>>>(
        F(L.a), dx, dy, static_cast<T*>(W_out));
    rc_bias_partial_kernel<<<dim3((dy + 31) / 32, (dx + 255) / 256), dim3(32, 8), 0, s>>>(
        F(L.a), dx, dy, sx, sw_ss, bacc);
    rc_bias_final_kernel<<<(dy + 255) / 256, 256, 0, s>>>(sy, sw_ss, bacc, dy, b_out);
  }
  HF_CUDA_TRY(cudaGetLastError(), "hf_recolor_fit: output launch");
  double hs[2];
  int32_t gemm_err = 0;
  HF_CUDA_TRY(cudaMemcpyAsync(hs, sw_ss, sizeof(hs), cudaMemcpyDeviceToHost, s), "read back");
  HF_CUDA_TRY(cudaMemcpyAsync(&gemm_err, h.err, sizeof(gemm_err), cudaMemcpyDeviceToHost, s),
              "read back");
  HF_CUDA_TRY(cudaStreamSynchronize(s), "synchronize");
  if (gemm_err != 0) {
    set_error("hf_recolor_fit: a product kernel's pipeline wait ran out (internal error)");
    return HF_ERR_DEVICE_CHECK;
  }
  if (h_r) *h_r = static_cast<float>(std::sqrt(hs[1] / (static_cast<double>(dx) * hs[0])));
  if (h_iters) {
    h_iters[0] = it1;
    h_iters[1] = it2;
    h_iters[2] = it3;
  }
  if (it1 >= kMaxIter || it2 >= kMaxIter || it3 >= kMaxIter) {
    set_error("hf_recolor_fit: an iteration did not converge (ill-conditioned covariances: "
              "raise reg)");
    return HF_ERR_DEVICE_CHECK;
  }
  return HF_OK;
}

}  // namespace
}  // namespace hf

using namespace hf;

extern "C" hf_status hf_recolor_workspace_size(int64_t N, int32_t d_S, int32_t d_R,
                                               size_t* bytes) {
  if (!bytes || N < 2 || d_S < 1 || d_R < 1 || d_S < d_R) {
    set_error("hf_recolor_workspace_size: need N >= 2 and d_S >= d_R >= 1");
    return HF_ERR_INVALID_ARGUMENT;
  }
  *bytes = rc_layout(N, d_S, d_R).total;
  return HF_OK;
}

extern "C" hf_status hf_recolor_fit(hf_dtype dtype, int64_t N, int32_t d_S, int32_t d_R,
                                    const void* d_X, const void* d_Y, const float* d_w, float reg,
                                    void* d_W_out, float* d_b_out, float* h_r_out,
                                    int32_t* h_iters_out, void* d_workspace,
                                    size_t workspace_bytes, hf_stream_t stream_) {
  if (dtype != HF_BF16 && dtype != HF_F32) {
    set_error("hf_recolor_fit: unknown dtype");
    return HF_ERR_INVALID_ARGUMENT;
  }
  if (N < 2 || d_S < 1 || d_R < 1 || d_S < d_R || N * static_cast<int64_t>(d_S) >= (1LL << 31)) {
    set_error("hf_recolor_fit: need N >= 2, d_S >= d_R >= 1 and N x d_S < 2^31");
    return HF_ERR_INVALID_ARGUMENT;
  }
  if (!d_X || !d_Y || !d_w || !d_W_out || !d_b_out || !(reg >= 0.f)) {
    set_error("hf_recolor_fit: null pointer or negative reg");
    return HF_ERR_INVALID_ARGUMENT;
  }
  if (!d_workspace || workspace_bytes < rc_layout(N, d_S, d_R).total ||
      (reinterpret_cast<uintptr_t>(d_workspace) & 255u)) {
    set_error("hf_recolor_fit: workspace missing, too small or not 256-byte aligned");
    return HF_ERR_WORKSPACE;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream_);
  char* ws = static_cast<char*>(d_workspace);
  if (dtype == HF_BF16)
    return recolor_typed<__nv_bfloat16>(N, d_S, d_R, d_X, d_Y, d_w, reg, d_W_out, d_b_out,
                                        h_r_out, h_iters_out, ws, s);
  return recolor_typed<float>(N, d_S, d_R, d_X, d_Y, d_w, reg, d_W_out, d_b_out, h_r_out,
                              h_iters_out, ws, s);
}
