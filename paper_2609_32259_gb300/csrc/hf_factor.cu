// Triangular factors of hf_recolor_fit's covariances (Section 3.2, Eq. 4-5).
//
// tri_factor eliminates S = L L^T (L lower triangular) in place, in block rows
// of 128:
//   1. rc_diag_kernel: one CTA factors the 128 x 128 diagonal block and inverts
//      its factor, T = L_kk^{-1};
//   2. rc_panel_kernel: the block row becomes T times itself: to the right of
//      the diagonal L^T, to its left the block row of L^{-1}, on it T; it also
//      writes the row's three bf16 planes;
//   3. gemm_planes: the rows below take minus (block row)^T (block row), and the
//      eliminated block column, which the symmetric row already gave, starts
//      afresh as the next block column of L^{-1}.
// Afterwards the rows hold L^{-1} on and below the diagonal blocks.
//
// A chain of n / 128 steps bounds it (one CTA's 128 pivots, then two short
// launches), not its operations: at n = 3,072 0.17 TFLOP of bf16 products, 0.1
// ms of tensor time.  So two matrices are eliminated in the same steps, and
// each kernel is launched while the one before it drains (a fit of 32,768 x
// 3,072 -> 1,024: 6.04 ms with neither, 5.40 with both).  Blocks of 128 because
// the block and its inverse fit one CTA's shared memory and two K atoms of the
// product kernel; an iteration for the roots of S costs 33 dense products of
// the same size (7.5 ms at 3,072).
#include <cfloat>

#include <cuda_bf16.h>

#include "hf_device.cuh"
#include "hf_internal.h"

namespace hf {
namespace {

constexpr int kNb = kFactorBlock;   // 128: block rows
constexpr int kSub = 32;            // blocks of the one-CTA elimination
constexpr int kLd = kNb + 4;        // padded shared-memory row
constexpr int kDiagThreads = 512;
constexpr int kPanelCols = 32;
constexpr int kPanelThreads = 256;

// Eliminates the diagonal block at row and column r0 of W (its upper triangle
// is read), as tri_factor does with blocks of 32 instead of 128: T = L^{-1}
// (zeros above the diagonal) goes to W's block and, transposed, to Tt.  With
// upper not null the block of L^T goes to upper (leading dimension n_upper,
// rows and columns below n_upper).
// One CTA per matrix.
struct TriPair {
  TriProblem p[2];
};
__global__ void __launch_bounds__(kDiagThreads)
    rc_diag_kernel(const __grid_constant__ TriPair tp, int r0, int32_t* flag) {
  const TriProblem& pr = tp.p[blockIdx.x];
  float* const W = pr.W;
  const int64_t ld = pr.ld;
  const float* const thr = pr.thr;
  float* const Tt = pr.Tt;
  float* const upper = pr.upper;
  const int n_upper = pr.n_upper;
  depend_wait();
  depend_launch();
  extern __shared__ __align__(16) float sm[];
  float* const S = sm;               // [128][kLd]
  float* const T = sm + kNb * kLd;   // [32][kSub + 4]: the sub-block's L^{-1}
  constexpr int kTs = kSub + 4;
  float* const rows = T + kSub * kTs;  // two pivots' rows: 2 x [block 32, inverse 32]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* const Wb = W + static_cast<int64_t>(r0) * ld + r0;
  constexpr int kVecs = kNb * kNb / 4 / kDiagThreads;  // all in flight: one latency
  float4 in[kVecs];
#pragma unroll
  for (int i = 0; i < kVecs; ++i) {
    const int e = tid + i * kDiagThreads, r = e / (kNb / 4), q = e % (kNb / 4);
    in[i] = *reinterpret_cast<const float4*>(Wb + r * ld + 4 * q);
  }
  const float t0 = *thr;
#pragma unroll
  for (int i = 0; i < kVecs; ++i) {
    const int e = tid + i * kDiagThreads, r = e / (kNb / 4), q = e % (kNb / 4);
    *reinterpret_cast<float4*>(S + r * kLd + 4 * q) = in[i];
  }
  __syncthreads();
  const int c = tid % kNb, g = tid / kNb;  // this thread's column, row group 0..3
#pragma unroll 1
  for (int j0 = 0; j0 < kNb; j0 += kSub) {
    // The 32 x 32 sub-block by four warps, rows 8 warp .. + 7 of column `lane`
    // with each thread: per pivot the pivot's row of the block (which is its
    // column) and of the growing inverse go through shared memory, one barrier
    // a pivot.  What bounds it is the instructions of 128 such steps: all
    // sixteen warps taking part, or one warp with rows in registers and the
    // steps unrolled, took 57 to 60 us a block.
    if (warp < 4) {
      float a[8], v[8];
      const int rb = 8 * warp;
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        a[h] = S[(j0 + min(rb + h, lane)) * kLd + j0 + max(rb + h, lane)];
        v[h] = rb + h == lane ? 1.f : 0.f;
      }
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          const int j = 8 * q + jj;
          float* const buf = rows + (jj & 1) * 2 * kSub;
          if (warp == q) {
            buf[lane] = a[jj];
            buf[kSub + lane] = v[jj];
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
          float piv = buf[j];
          if (!(piv > t0 && piv <= FLT_MAX)) {
            if (tid == 0) *flag = 1;
            piv = 1.f;
          }
          float rs = rsqrtf(piv);
          rs = rs * fmaf(-0.5f * piv * rs, rs, 1.5f);
          const float lc = buf[lane] * rs, vc = buf[kSub + lane] * rs;
          const float4 r0v = *reinterpret_cast<const float4*>(buf + rb);
          const float4 r1v = *reinterpret_cast<const float4*>(buf + rb + 4);
          const float lr[8] = {r0v.x, r0v.y, r0v.z, r0v.w, r1v.x, r1v.y, r1v.z, r1v.w};
#pragma unroll
          for (int h = 0; h < 8; ++h) {
            // rows past the pivot; its own becomes the row of L^T and of L^{-1}
            const float f = warp > q || (warp == q && h > jj) ? lr[h] * rs : 0.f;
            a[h] = fmaf(-f, lc, a[h]);
            v[h] = fmaf(-f, vc, v[h]);
          }
          if (warp == q) {
            a[jj] = lc;
            v[jj] = vc;
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const int r = rb + h, row = r0 + j0 + r, col = r0 + j0 + lane;
        const float t = lane <= r ? v[h] : 0.f;
        T[r * kTs + lane] = t;
        S[(j0 + r) * kLd + j0 + lane] = t;
        if (upper && lane >= r && row < n_upper && col < n_upper)
          upper[static_cast<int64_t>(row) * n_upper + col] = a[h];
      }
    }
    __syncthreads();
    // the block row times T (the block itself already is T)
    const bool own = c >= j0 && c < j0 + kSub;
    float x[kSub];
#pragma unroll
    for (int k = 0; k < kSub; ++k) x[k] = S[(j0 + k) * kLd + c];
    __syncthreads();
    if (!own) {
#pragma unroll 2
      for (int i = 0; i < kSub / 4; ++i) {
        const int r = g * (kSub / 4) + i;
        float y = 0.f;
#pragma unroll
        for (int k = 0; k < kSub; k += 4) {
          const float4 t = *reinterpret_cast<const float4*>(T + r * kTs + k);
          y = fmaf(t.x, x[k], y);
          y = fmaf(t.y, x[k + 1], y);
          y = fmaf(t.z, x[k + 2], y);
          y = fmaf(t.w, x[k + 3], y);
        }
        S[(j0 + r) * kLd + c] = y;
        if (upper && c > j0 && r0 + j0 + r < n_upper && r0 + c < n_upper)
          upper[static_cast<int64_t>(r0 + j0 + r) * n_upper + r0 + c] = y;
      }
    }
    __syncthreads();
    // the rows below: minus (block row)^T (block row); the block column afresh
#pragma unroll
    for (int k = 0; k < kSub; ++k) x[k] = S[(j0 + k) * kLd + c];
    const int rest = kNb - j0 - kSub, per = rest / 4;
#pragma unroll 1
    for (int i = 0; i < per; i += 4) {
      const int r = j0 + kSub + g * per + i;
      float y[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = own ? 0.f : S[(r + q) * kLd + c];
#pragma unroll
      for (int k = 0; k < kSub; ++k) {
        const float4 u = *reinterpret_cast<const float4*>(S + (j0 + k) * kLd + r);
        y[0] = fmaf(-u.x, x[k], y[0]);
        y[1] = fmaf(-u.y, x[k], y[1]);
        y[2] = fmaf(-u.z, x[k], y[2]);
        y[3] = fmaf(-u.w, x[k], y[3]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) S[(r + q) * kLd + c] = y[q];
    }
    __syncthreads();
  }
#pragma unroll 4
  for (int i = tid; i < kNb * kNb; i += kDiagThreads) {
    const int r = i / kNb, cc = i % kNb;
    Wb[r * ld + cc] = cc <= r ? S[r * kLd + cc] : 0.f;
    Tt[i] = r <= cc ? S[cc * kLd + r] : 0.f;
  }
}

// Block row [r0, r0 + 128) of W <- T times it, columns 32 blockIdx.x ..: the
// diagonal block's own columns become T.  planes: three bf16 planes of the new
// row, plane p's element (column, row) at (p rows_p + column) 128 + row.  With
// upper not null the columns right of the block also go to upper.
__global__ void __launch_bounds__(kPanelThreads)
    rc_panel_kernel(const __grid_constant__ TriPair tp, int r0) {
  const TriProblem& pr = tp.p[blockIdx.y];
  depend_wait();
  depend_launch();
  if (static_cast<int>(blockIdx.x) * kPanelCols >= pr.n) return;
  float* const W = pr.W;
  const int64_t ld = pr.ld, rows_p = (pr.n + 255) / 256 * 256;
  const float* const Tt = pr.Tt;
  __nv_bfloat16* const planes = static_cast<__nv_bfloat16*>(pr.planes);
  float* const upper = pr.upper;
  const int n_upper = pr.n_upper;
  extern __shared__ __align__(16) float sm[];
  float* const t = sm;              // [k][row]
  float* const s = sm + kNb * kNb;  // [k][32]
  const int tid = threadIdx.x;
  const int c0 = blockIdx.x * kPanelCols;
  const bool own = c0 >= r0 && c0 < r0 + kNb;
  constexpr int kTVecs = kNb * kNb / 4 / kPanelThreads;          // 16
  constexpr int kSVecs = kNb * kPanelCols / 4 / kPanelThreads;   // 4
  float4 tin[kTVecs], sin[kSVecs];
#pragma unroll
  for (int i = 0; i < kSVecs; ++i) {
    const int e = tid + i * kPanelThreads, k = e / (kPanelCols / 4), q = e % (kPanelCols / 4);
    sin[i] = *reinterpret_cast<const float4*>(W + static_cast<int64_t>(r0 + k) * ld + c0 + 4 * q);
  }
#pragma unroll
  for (int i = 0; i < kTVecs; ++i)
    tin[i] = ld_dep(reinterpret_cast<const float4*>(Tt) + tid + i * kPanelThreads);
#pragma unroll
  for (int i = 0; i < kSVecs; ++i) {
    const int e = tid + i * kPanelThreads, k = e / (kPanelCols / 4), q = e % (kPanelCols / 4);
    const int d = r0 + k - c0 - 4 * q;  // the identity's column in this quad
    if (own) sin[i] = make_float4(d == 0 ? 1.f : 0.f, d == 1 ? 1.f : 0.f, d == 2 ? 1.f : 0.f,
                                  d == 3 ? 1.f : 0.f);
    reinterpret_cast<float4*>(s)[e] = sin[i];
  }
#pragma unroll
  for (int i = 0; i < kTVecs; ++i) reinterpret_cast<float4*>(t)[tid + i * kPanelThreads] = tin[i];
  __syncthreads();
  const int tx = tid & 7, ty = tid >> 3;  // columns 4 tx .., rows 4 ty ..
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  // T is lower triangular: rows 4 ty .. read k up to their own index
#pragma unroll 4
  for (int k = 0; k < 4 * ty + 4; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(t + k * kNb + 4 * ty);
    const float4 b = *reinterpret_cast<const float4*>(s + k * kPanelCols + 4 * tx);
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + 4 * ty + i;
    *reinterpret_cast<float4*>(W + static_cast<int64_t>(r) * ld + c0 + 4 * tx) =
        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (upper && c0 >= r0 + kNb && r < n_upper) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c0 + 4 * tx + j < n_upper)
          upper[static_cast<int64_t>(r) * n_upper + c0 + 4 * tx + j] = acc[i][j];
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float x[4] = {acc[0][j], acc[1][j], acc[2][j], acc[3][j]};
    __nv_bfloat16* o = planes + (static_cast<int64_t>(c0) + 4 * tx + j) * kNb + 4 * ty;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(x[0], x[1]);
      const __nv_bfloat162 h1 = __floats2bfloat162_rn(x[2], x[3]);
      const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
      x[0] -= f0.x;
      x[1] -= f0.y;
      x[2] -= f1.x;
      x[3] -= f1.y;
      *reinterpret_cast<uint2*>(o + p * rows_p * kNb) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    }
  }
}

}  // namespace

size_t tri_factor_planes_bytes(int n) {
  const int64_t rows_p = (n + 255) / 256 * 256;
  return static_cast<size_t>(3 * rows_p * kNb * 2);
}

hf_status tri_factor(cudaStream_t s, const GemmWork& wk, const TriProblem* problems, int count,
                     int32_t* flag) {
  const size_t diag_smem = (kNb * kLd + kSub * (kSub + 4) + 4 * kSub) * sizeof(float);
  const size_t panel_smem = (kNb * kNb + kNb * kPanelCols) * sizeof(float);
  HF_CUDA_TRY(cudaFuncSetAttribute(rc_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(diag_smem)),
              "hf_recolor_fit: factor shared memory");
  HF_CUDA_TRY(cudaFuncSetAttribute(rc_panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(panel_smem)),
              "hf_recolor_fit: panel shared memory");
  int n_max = 0;
  for (int i = 0; i < count; ++i) n_max = n_max > problems[i].n ? n_max : problems[i].n;
  for (int r0 = 0; r0 < n_max; r0 += kNb) {
    TriPair tp;  // the matrices that have this block row
    int live = 0;
    for (int i = 0; i < count; ++i)
      if (r0 < problems[i].n) tp.p[live++] = problems[i];
    if (live == 1) tp.p[1] = tp.p[0];
    HF_CUDA_TRY(launch_dependent(rc_diag_kernel, dim3(live), dim3(kDiagThreads), diag_smem, s, tp, r0,
                                 flag),
                "hf_recolor_fit: factor launch");
    HF_CUDA_TRY(launch_dependent(rc_panel_kernel, dim3(n_max / kPanelCols, live),
                                 dim3(kPanelThreads), panel_smem, s, tp, r0),
                "hf_recolor_fit: panel launch");
    for (int i = 0; i < live; ++i) {
      const TriProblem& p = tp.p[i];
      const int below = r0 + kNb;
      if (below >= p.n) continue;
      const int64_t rows_p = (p.n + 255) / 256 * 256;
      const GemmPlanes a{p.planes, rows_p, below}, b{p.planes, rows_p, 0};
      GemmShape shape;  // all of L^{-1}, and of S what is on or above the diagonal
      shape.tri = true;
      shape.diag_col = below;
      shape.fresh_lo = r0;
      shape.fresh_hi = below;
      const hf_status st = gemm_planes(s, wk, p.n - below, p.n, kNb, -1.f, a, b, 1.f,
                                       p.W + static_cast<int64_t>(below) * p.ld, p.ld, shape);
      if (st != HF_OK) return st;
    }
  }
  return HF_OK;
}

}  // namespace hf
