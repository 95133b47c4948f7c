// hf_fold: folds the output-aware low-rank correction (Eq. 7) into the
// affine maps (Eq. 9): A_final = A (I + B G), b_final = b (I + B G).
// In the ABI's layout W = A^T ([d_R][K] per map), so
//   T = B^T W                      (rho x K)
//   W_final = W + G^T T            (element [n][k] += sum_r G[r][n] T[r][k])
//   b_final = b + (b B) G.
// Two forms.  fold_mma_kernel (bf16 maps, rank <= 16, d_R <= 1,024, K a multiple
// of 8, where it is the faster: see launch_fold) reads W once: the 4 rank FLOP per element outweigh the memory time on
// the fp32 ALUs, so both contractions run on the warp-level tensor
// instructions, with every fp32 factor split exactly into three bf16 parts and
// the products above 2^-23 kept (a rank of 16 is one 16-deep step: too thin for
// an accumulator in tensor memory; 80 maps of 1,024 x 3,072, rank 16, with the
// bias: 0.25 ms, fold_kernel 0.49; the same error against 64 bits).  fold_kernel
// takes the rest with plain fp32 arithmetic; a block reads its columns of W
// twice (the second time from L2) and writes them once.
#include <algorithm>

#include <cuda_bf16.h>

#include <string>

#include "hf_device.cuh"
#include "hf_internal.h"

namespace hf {
namespace {

constexpr int kMaxRank = 32;
constexpr int kFoldThreads = 256;

// CPT consecutive columns of one row: values from shared memory, stores of
// 4 * CPT (fp32) or 2 * CPT (bf16) bytes.
template <int CPT>
__device__ __forceinline__ void smem_cols(const __nv_bfloat16* p, float* x) {
#pragma unroll
  for (int j = 0; j < CPT; j += 2) {
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p + j));
    x[j] = a.x;
    x[j + 1] = a.y;
  }
}
template <int CPT>
__device__ __forceinline__ void smem_cols(const float* p, float* x) {
#pragma unroll
  for (int j = 0; j < CPT; j += 2) {
    const float2 a = *reinterpret_cast<const float2*>(p + j);
    x[j] = a.x;
    x[j + 1] = a.y;
  }
}
template <int CPT>
__device__ __forceinline__ void store_cols(__nv_bfloat16* p, const float* x) {
  if constexpr (CPT == 4) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(x[0], x[1]), b = __floats2bfloat162_rn(x[2], x[3]);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a),
                                              *reinterpret_cast<const uint32_t*>(&b));
  } else {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(x[0], x[1]);
  }
}
template <int CPT>
__device__ __forceinline__ void store_cols(float* p, const float* x) {
  if constexpr (CPT == 4)
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  else
    *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
}

// Asynchronous copy of N (4, 8 or 16) bytes from global to shared memory.
template <int N>
__device__ __forceinline__ void fold_cp_async(void* dst, const void* src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  if constexpr (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(N) : "memory");
}
__device__ __forceinline__ void fold_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fold_cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr int kFoldSlices = kFoldThreads / 32;  // row slices (8): one warp each
constexpr int kFoldRing = 16;                    // rows of W in flight per thread

// Shared memory of one block, in floats: a region holding B [d_r][R] in
// pass 1, then the slices' partial sums [slices][R][32 CPT], then G^T
// [d_r][R + 4]; after it, each thread's ring of kFoldRing rows x CPT columns.
template <typename T>
__host__ __device__ constexpr size_t fold_region_floats(int d_r, int R, int CPT) {
  const size_t b = static_cast<size_t>(d_r) * R, g = static_cast<size_t>(d_r) * (R + 4);
  const size_t p = static_cast<size_t>(kFoldSlices) * R * 32 * CPT;
  const size_t m = g > p ? g : p;
  return m > b ? m : b;
}
template <typename T>
__host__ __device__ constexpr size_t fold_smem_bytes(int d_r, int R, int CPT) {
  return fold_region_floats<T>(d_r, R, CPT) * sizeof(float) +
         static_cast<size_t>(kFoldThreads) * kFoldRing * CPT * sizeof(T);
}

// This thread's ring of W rows: rows n = sl, sl + 8, ... < d_r of its CPT
// columns, kFoldRing in flight, each thread copying and reading only its own
// bytes (so a wait on its own copies is all the synchronisation needed).
// Slot i of thread tid is at (i * 256 + tid) * CPT elements: a warp's reads
// of one slot are consecutive.
template <typename T, int CPT>
struct FoldRing {
  static constexpr int kBytes = CPT * static_cast<int>(sizeof(T));
  static constexpr int kStride = kFoldThreads * CPT;  // slots are thread-interleaved
  const T* col0;
  int64_t K;
  int d_r, sl;
  T* ring;
  // issues the first kFoldRing rows (one commit group per row)
  __device__ __forceinline__ void start() const {
#pragma unroll 1
    for (int i = 0; i < kFoldRing; ++i) {
      const int n = sl + kFoldSlices * i;
      if (n < d_r) fold_cp_async<kBytes>(ring + i * kStride, col0 + static_cast<int64_t>(n) * K);
      fold_cp_commit();
    }
  }
  // waits for the row held in `slot` and reads it
  __device__ __forceinline__ void take(int slot, float* x) const {
    fold_cp_wait<kFoldRing - 1>();
    smem_cols<CPT>(ring + slot * kStride, x);
  }
  // refills `slot` (row n, already used) with row n + 8 kFoldRing
  __device__ __forceinline__ void refill(int n, int slot) const {
    const int nn = n + kFoldSlices * kFoldRing;
    if (nn < d_r) fold_cp_async<kBytes>(ring + slot * kStride, col0 + static_cast<int64_t>(nn) * K);
    fold_cp_commit();
  }
};

// One block folds columns [k0, k0 + 32 CPT) of one map; thread (column
// group cg = lane, row slice sl = warp) owns columns k0 + CPT cg .. + CPT - 1
// and streams them, rows n = sl (mod 8), through its shared-memory ring:
//  pass 1: T = B^T W for those columns, B from shared memory (float4
//          broadcasts); the slices' partial sums go through shared memory
//          (where B was) and every thread sums its columns' R values;
//  pass 2: W_final = W + G^T T row by row (the rows come from L2 again), G^T
//          staged in shared memory with rows padded to R + 4 floats.
// Every element of the block's columns is read in pass 1 before any is
// written in pass 2, so W_final may alias W.
template <typename T, int R, int CPT>
__global__ void __launch_bounds__(kFoldThreads) fold_kernel(const T* W, const float* __restrict__ Bm,
                                                            const float* __restrict__ Gm, T* Wf,
                                                            int d_r, int64_t K) {
  extern __shared__ __align__(16) float fsm[];
  constexpr int kGs = R + 4;            // padded G^T row
  constexpr int kCols = 32 * CPT;       // columns per block
  float* const Bs = fsm;                // [d_r][R]
  float* const Ps = fsm;                // [slices][R][kCols]
  float* const Gs = fsm;                // [d_r][kGs]
  const int map = blockIdx.y;
  const int tid = threadIdx.x;
  const int cg = tid & 31, sl = tid >> 5;
  T* const ring = reinterpret_cast<T*>(fsm + fold_region_floats<T>(d_r, R, CPT)) + tid * CPT;
  const int64_t k = static_cast<int64_t>(blockIdx.x) * kCols + CPT * cg;
  const bool live = k < K;  // K is a multiple of CPT: a group's columns all exist or none
  const T* col0 = W + static_cast<int64_t>(map) * d_r * K + k;
  T* const out0 = Wf + static_cast<int64_t>(map) * d_r * K + k;
  const float* B = Bm + static_cast<int64_t>(map) * d_r * R;
  const float* G = Gm + static_cast<int64_t>(map) * R * d_r;
  for (int i = tid; i < R * d_r / 4; i += kFoldThreads)
    reinterpret_cast<float4*>(Bs)[i] = __ldg(reinterpret_cast<const float4*>(B) + i);
  __syncthreads();
  // pass 1
  float acc[R][CPT];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < CPT; ++j) acc[r][j] = 0.f;
  const FoldRing<T, CPT> rg{col0, K, d_r, sl, ring};
  if (live) {
    rg.start();
    int slot = 0;
#pragma unroll 1
    for (int n = sl; n < d_r; n += kFoldSlices) {
      float x[CPT];
      rg.take(slot, x);
      const float4* bn = reinterpret_cast<const float4*>(Bs + n * R);
#pragma unroll
      for (int q = 0; q < R / 4; ++q) {
        const float4 b = bn[q];
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
          acc[4 * q][j] = fmaf(b.x, x[j], acc[4 * q][j]);
          acc[4 * q + 1][j] = fmaf(b.y, x[j], acc[4 * q + 1][j]);
          acc[4 * q + 2][j] = fmaf(b.z, x[j], acc[4 * q + 2][j]);
          acc[4 * q + 3][j] = fmaf(b.w, x[j], acc[4 * q + 3][j]);
        }
      }
      rg.refill(n, slot);  // after x is consumed
      if (++slot == kFoldRing) slot = 0;
    }
    fold_cp_wait<0>();
  }
  __syncthreads();  // B is no longer read: the partial sums take its place
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < CPT; ++j) Ps[(sl * R + r) * kCols + CPT * cg + j] = acc[r][j];
  __syncthreads();
  float t[R][CPT];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < CPT; ++j) t[r][j] = 0.f;
#pragma unroll 1
  for (int s2 = 0; s2 < kFoldSlices; ++s2)
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int j = 0; j < CPT; ++j) t[r][j] += Ps[(s2 * R + r) * kCols + CPT * cg + j];
  __syncthreads();  // the partial sums are read: G^T takes their place
  for (int i = tid; i < R * d_r; i += kFoldThreads) {
    const int r = i / d_r, n = i - r * d_r;
    Gs[n * kGs + r] = __ldg(G + i);
  }
  __syncthreads();
  if (!live) return;
  // pass 2
  rg.start();
  int slot = 0;
#pragma unroll 1
  for (int n = sl; n < d_r; n += kFoldSlices) {
    float v[CPT];
    rg.take(slot, v);
    const float4* g = reinterpret_cast<const float4*>(Gs + n * kGs);
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
      const float4 gq = g[q];
#pragma unroll
      for (int j = 0; j < CPT; ++j) {
        v[j] = fmaf(gq.x, t[4 * q][j], v[j]);
        v[j] = fmaf(gq.y, t[4 * q + 1][j], v[j]);
        v[j] = fmaf(gq.z, t[4 * q + 2][j], v[j]);
        v[j] = fmaf(gq.w, t[4 * q + 3][j], v[j]);
      }
    }
    store_cols<CPT>(out0 + static_cast<int64_t>(n) * K, v);
    rg.refill(n, slot);  // after the row is consumed
    if (++slot == kFoldRing) slot = 0;
  }
  fold_cp_wait<0>();
}

// ---------------------------------------------------------------------------
// bf16 maps on the tensor cores
// ---------------------------------------------------------------------------
constexpr int kMmaWarps = 16;
constexpr int kMmaCols = 32;            // columns of W per unit of work
constexpr int kMmaRows = 1024;          // d_R at most: 64 rows per warp
constexpr int kTStride = kMmaCols + 8;  // padded row of T: 80 bytes, no bank twice
constexpr int kPartStride = kMmaCols + 4;
constexpr int kMmaUnits = 8192;         // units of one CTA at most
// What sums of split products cannot give: an infinity times a part that is zero is
// NaN, and so is the residual of a value that rounds to an infinity in bf16.
// Columns whose T is not finite or above this, and maps with a G above it, take
// fp32 arithmetic (products of the rest stay below 2^124).
constexpr float kMmaRange = 0x1p60f;

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                          uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Four transposed 8 x 8 matrices: two 16 x 8 right operands (16 rows of shared
// memory, two groups of eight columns).
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p)))
               : "memory");
}
// (x, y) as three bf16 pairs that add up to it exactly (24 bits).
__device__ __forceinline__ void split3(float x, float y, uint32_t* h0, uint32_t* h1, uint32_t* h2) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(x, y);
  const float2 fa = __bfloat1622float2(a);
  x -= fa.x;
  y -= fa.y;
  const __nv_bfloat162 b = __floats2bfloat162_rn(x, y);
  const float2 fb = __bfloat1622float2(b);
  const __nv_bfloat162 c = __floats2bfloat162_rn(x - fb.x, y - fb.y);
  *h0 = *reinterpret_cast<const uint32_t*>(&a);
  *h1 = *reinterpret_cast<const uint32_t*>(&b);
  *h2 = *reinterpret_cast<const uint32_t*>(&c);
}

struct FoldMmaSmem {
  // 64-byte rows, the 16-byte piece c of row r at c ^ (r / 2 mod 4): eight rows'
  // pieces lie in different banks, and tensor copies write it out
  __nv_bfloat16 w[2][kMmaRows][kMmaCols];
  float part[kMmaWarps][16][kPartStride];
  __nv_bfloat16 t[3][16][kTStride];
  float tf[16][kMmaCols];   // fold_plain_columns' T
  unsigned plain[2];        // columns that fold_plain_columns does: this unit's, the next one's
  unsigned redo[kMmaUnits]; // and every unit's of this CTA
};
static_assert(kMmaCols == 32, "the 64-byte swizzle is over rows of 32");

__device__ __forceinline__ bool above(float x, float limit) { return !(fabsf(x) <= limit); }

// The columns `mask` of the strip at column k0 of one map, whose W_final still is
// W, with plain fp32 sums in fold_kernel's order.  All threads of the CTA.
__device__ __forceinline__ void fold_plain_columns(FoldMmaSmem& sm, __nv_bfloat16* Wf, const float* B,
                                                   const float* G, int d_r, int64_t K, int rank,
                                                   int64_t k0, unsigned mask) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool mine = mask >> lane & 1u;
  __nv_bfloat16* const col = Wf + k0 + lane;
  __syncthreads();
  if (mine && warp < rank) {
    float t = 0.f;
#pragma unroll 1
    for (int s = 0; s < kFoldSlices; ++s) {
      float acc = 0.f;
#pragma unroll 1
      for (int m = s; m < d_r; m += kFoldSlices)
        acc = fmaf(B[static_cast<int64_t>(m) * rank + warp], __bfloat162float(col[m * K]), acc);
      t += acc;
    }
    sm.tf[warp][lane] = t;
  }
  __syncthreads();
  if (!mine) return;
#pragma unroll 1
  for (int n = warp; n < d_r; n += kMmaWarps) {
    float v = __bfloat162float(col[n * K]);
#pragma unroll 1
    for (int r = 0; r < rank; ++r) v = fmaf(G[static_cast<int64_t>(r) * d_r + n], sm.tf[r][lane], v);
    col[n * K] = __float2bfloat16_rn(v);
  }
}

// A persistent CTA takes a run of units (map, 32 columns).  Warp w owns rows 16
// steps w .. of W (steps <= 4 blocks of 16): it alone copies them in, works on
// them and copies them out, so that only T takes a barrier.  Per unit:
//  1. T = B^T W: the warp's share of the contraction over the rows, with the
//     split B of its rows in registers (kept while the map stays the same);
//     W is exact in bf16, so three products per term;
//  2. the warps' shares meet in shared memory, T is split there;
//  3. W += G^T T on the warp's rows: six products, added to W in fp32, rounded
//     once, back into the buffer, which then leaves by a tensor copy; once that
//     has read it (during the next unit's step 1) the buffer takes the columns of
//     the unit after.
// The chain of these steps bounds it (64 KB in and out per unit and SM; two
// buffers of 32 columns are what fits): of 9.7K cycles a unit step 3 takes 4.4K
// (3K at the tensor instructions' rate), steps 1 and 2 1.5K and 1.2K; the memory
// rate allows 5.6K.  With the rows written out by the threads a unit took 13K
// (4.1K of them in those stores; 80 maps of 1,024 x 3,072: 358 us, 254 now).
// Step 1 of a unit before step 3 of the one before it exposed the copies.
// Columns that need fp32 arithmetic (kMmaRange) leave as they came and are done
// after the run: any of it inside the loop cost 55 us, the looking costs 1.
__global__ void __launch_bounds__(32 * kMmaWarps)
    fold_mma_kernel(const __nv_bfloat16* W, const float* __restrict__ Bm,
                    const float* __restrict__ Gm, __nv_bfloat16* Wf,
                    const __grid_constant__ CUtensorMap map_out,
                    int n_maps, int d_r, int64_t K, int rank, int steps) {
  extern __shared__ __align__(1024) uint8_t fold_smem[];
  FoldMmaSmem& sm = *reinterpret_cast<FoldMmaSmem*>(fold_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;  // fragment row and column pair
  const int per_map = static_cast<int>((K + kMmaCols - 1) / kMmaCols);
  const int64_t units = static_cast<int64_t>(n_maps) * per_map;
  depend_launch();  // the biases' kernel
  const int64_t u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
  const int row0 = warp * 16 * steps, rows = min(16 * steps, d_r - row0);  // <= 0: padding only
  for (int i = lane; i < (16 * steps - max(rows, 0)) * kMmaCols; i += 32) {
    const int r = row0 + max(rows, 0) + i / kMmaCols;  // rows past d_R: zeros
    sm.w[0][r][i % kMmaCols] = sm.w[1][r][i % kMmaCols] = __nv_bfloat16(0.f);
  }
  // the warp's rows of a unit, 16-byte pieces, four per row
  const int lr = lane >> 2, lc = (lane & 3) * 8, lswz = ((lane & 3) ^ (lane >> 3)) * 8;
  auto load = [&](int64_t u) {
    if (u < u1) {
      const int map = static_cast<int>(u / per_map), buf = static_cast<int>((u - u0) & 1);
      const int64_t k0 = (u - static_cast<int64_t>(map) * per_map) * kMmaCols;
      const __nv_bfloat16* src = W + (static_cast<int64_t>(map) * d_r + row0 + lr) * K + k0 + lc;
      if (k0 + lc < K) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (lr + 8 * i < rows)
            fold_cp_async<16>(&sm.w[buf][row0 + lr + 8 * i][lswz], src + 8 * i * K);
      }
    }
    fold_cp_commit();
  };
  load(u0);
  if (tid < 2) sm.plain[tid] = 0;
  bool big_g = false;    // this thread's part of G has a value above kMmaRange
  unsigned any = 0;      // columns left to fold_plain_columns
  uint32_t bf[4][3][4];  // B^T, rank x 16 rows per step, split
  uint32_t gf[4][3][4];  // G^T, 16 rows x rank per step, split
  int map_now = -1;
  const int lrow = lane & 15, lhalf = lane >> 4;  // ldmatrix: this lane's row and piece
  const int lsw = (lrow >> 1) & 3, gsw = (g >> 1) & 3;
  for (int64_t u = u0; u < u1; ++u) {
    const int buf = static_cast<int>((u - u0) & 1);
    const int map = static_cast<int>(u / per_map);
    const int64_t k0 = (u - static_cast<int64_t>(map) * per_map) * kMmaCols;
    auto& w = sm.w[buf];
    if (map != map_now) {
      map_now = map;
      big_g = false;
      const float* const B = Bm + static_cast<int64_t>(map) * d_r * rank;
      const float* const G = Gm + static_cast<int64_t>(map) * rank * d_r;
      auto at_b = [&](int n, int r) { return n < d_r && r < rank ? __ldg(B + n * rank + r) : 0.f; };
      auto at_g = [&](int n, int r) { return n < d_r && r < rank ? __ldg(G + r * d_r + n) : 0.f; };
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        if (s >= steps) break;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // B^T: rank row g (+8), rows 2t (+8) of W
          const int r = g + 8 * (i & 1), c = row0 + 16 * s + 2 * t + 8 * (i >> 1);
          split3(at_b(c, r), at_b(c + 1, r), &bf[s][0][i], &bf[s][1][i], &bf[s][2][i]);
          // G^T: W row g (+8), rank columns 2t (+8)
          const int n = row0 + 16 * s + g + 8 * (i & 1), q = 2 * t + 8 * (i >> 1);
          float g0 = at_g(n, q), g1 = at_g(n, q + 1);
          if (above(g0, kMmaRange) || above(g1, kMmaRange)) {
            big_g = true;
            g0 = g1 = 0.f;
          }
          split3(g0, g1, &gf[s][0][i], &gf[s][1][i], &gf[s][2][i]);
        }
      }
    }
    {
      // step 1
      fold_cp_wait<0>();
      __syncwarp();
      float d[4][4] = {};
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        if (s >= steps) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t x[4];
          ldsm_x4_t(x, &w[row0 + 16 * s + lrow][((2 * h + lhalf) ^ lsw) * 8]);
#pragma unroll
          for (int p = 2; p >= 0; --p) {
            mma_16816(d[2 * h], bf[s][p], x[0], x[1]);
            mma_16816(d[2 * h + 1], bf[s][p], x[2], x[3]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float2*>(&sm.part[warp][g][8 * i + 2 * t]) = make_float2(d[i][0], d[i][1]);
        *reinterpret_cast<float2*>(&sm.part[warp][g + 8][8 * i + 2 * t]) =
            make_float2(d[i][2], d[i][3]);
      }
      if (lane == 0) bulk_store_wait_read();  // the unit before has left its buffer
      __syncwarp();
      load(u + 1);
    }
    const bool big_map = __syncthreads_or(big_g);
    {
      // step 2
      if (tid == 0) sm.plain[buf ^ 1] = 0;
      float x = 0.f;  // T[warp][lane]
#pragma unroll
      for (int q = 0; q < kMmaWarps; ++q) x += sm.part[q][warp][lane];
      const unsigned redo =
          __ballot_sync(0xffffffffu, warp < rank && (big_map || above(x, kMmaRange)));
      if (redo && lane == 0) atomicOr(&sm.plain[buf], redo);
      const __nv_bfloat16 h0 = __float2bfloat16_rn(x);
      x -= __bfloat162float(h0);
      const __nv_bfloat16 h1 = __float2bfloat16_rn(x);
      sm.t[0][warp][lane] = h0;
      sm.t[1][warp][lane] = h1;
      sm.t[2][warp][lane] = __float2bfloat16_rn(x - __bfloat162float(h1));
    }
    __syncthreads();
    const unsigned plain = sm.plain[buf];
    if (tid == 0) sm.redo[u - u0] = plain;
    any |= plain;
    if (plain) {  // without T these columns leave as they came
      if (plain >> lane & 1u)
        sm.t[0][warp][lane] = sm.t[1][warp][lane] = sm.t[2][warp][lane] = __nv_bfloat16(0.f);
      __syncthreads();
    }
    {
      // step 3
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t x[3][4];
#pragma unroll
        for (int p = 0; p < 3; ++p) ldsm_x4_t(x[p], &sm.t[p][lrow][16 * h + 8 * lhalf]);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (s >= steps) break;
          float y[2][4] = {};
#pragma unroll
          for (int k = 0; k < 6; ++k) {  // the smallest products first
            constexpr int kG[6] = {2, 1, 0, 1, 0, 0}, kT[6] = {0, 1, 2, 0, 1, 0};
            mma_16816(y[0], gf[s][kG[k]], x[kT[k]][0], x[kT[k]][1]);
            mma_16816(y[1], gf[s][kG[k]], x[kT[k]][2], x[kT[k]][3]);
          }
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int col = ((2 * h + q) ^ gsw) * 8 + 2 * t;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const int r = 16 * s + g + 8 * k;
              if (r >= rows) continue;  // rows past d_R stay zeros, whatever T holds
              __nv_bfloat162* const o = reinterpret_cast<__nv_bfloat162*>(&w[row0 + r][col]);
              const float2 wv = __bfloat1622float2(*o);
              *o = __floats2bfloat162_rn(wv.x + y[q][2 * k], wv.y + y[q][2 * k + 1]);
            }
          }
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0 && rows > 0)
        tma_store_3d(&map_out, smem_addr(&w[row0][0]), static_cast<int32_t>(k0), row0, map);
    }
  }
  if (lane == 0) {
    bulk_store_wait_read();
    bulk_store_wait_all();
  }
  if (any) {
    fence_proxy_async_all();
    __syncthreads();  // the strips have been written
#pragma unroll 1
    for (int64_t u = u0; u < u1; ++u) {
      const int64_t map = u / per_map, k0 = (u - map * per_map) * kMmaCols;
      unsigned mask = sm.redo[u - u0];
      if (K - k0 < kMmaCols) mask &= (1u << (K - k0)) - 1u;
      if (mask)
        fold_plain_columns(sm, Wf + map * d_r * K, Bm + map * d_r * rank, Gm + map * rank * d_r, d_r,
                           K, rank, k0, mask);
    }
  }
}

// b_final = b + (b B) G for one map per block, every load of a pass in flight
// at once (one rank column at a time took 17 us for 80 maps).  It is launched
// beside the end of the maps' kernel, whose CTAs leave it no room earlier
// (with the gap between the launches 12 us of 266 at 80 maps).
template <int R>
__global__ void __launch_bounds__(256) fold_b_kernel(const float* b, const float* __restrict__ Bm,
                                                     const float* __restrict__ Gm, float* bf,
                                                     int d_r) {
  __shared__ float part[256 / 32][R];
  __shared__ float bB[R];
  const int map = blockIdx.x;
  const float* bm = b + static_cast<int64_t>(map) * d_r;
  const float* B = Bm + static_cast<int64_t>(map) * d_r * R;
  const float* G = Gm + static_cast<int64_t>(map) * R * d_r;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float s[R];
#pragma unroll
  for (int r = 0; r < R; ++r) s[r] = 0.f;
#pragma unroll 2
  for (int m = threadIdx.x; m < d_r; m += blockDim.x) {
    const float x = bm[m];
#pragma unroll
    for (int q = 0; q < R; q += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(B + static_cast<int64_t>(m) * R + q));
      s[q] = fmaf(x, v.x, s[q]);
      s[q + 1] = fmaf(x, v.y, s[q + 1]);
      s[q + 2] = fmaf(x, v.z, s[q + 2]);
      s[q + 3] = fmaf(x, v.w, s[q + 3]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
    if (lane == 0) part[warp][r] = s[r];
  }
  __syncthreads();
  if (threadIdx.x < R) {
    float t = 0.f;
    for (int w = 0; w < 256 / 32; ++w) t += part[w][threadIdx.x];
    bB[threadIdx.x] = t;
  }
  __syncthreads();
  for (int n = threadIdx.x; n < d_r; n += blockDim.x) {
    float v = bm[n];
#pragma unroll
    for (int r = 0; r < R; ++r) v = fmaf(bB[r], __ldg(G + static_cast<int64_t>(r) * d_r + n), v);
    bf[static_cast<int64_t>(map) * d_r + n] = v;
  }
  depend_wait();  // the maps, which this kernel has nothing to do with, are done
}

template <typename T, int R>
hf_status launch_fold_r(int n_maps, int d_r, int64_t K, const void* W, const float* B,
                        const float* G, void* Wf, int optin, cudaStream_t stream) {
  // four columns per thread where the accumulators fit (R <= 16), the column
  // groups tile K and shared memory allows; two otherwise
  constexpr int kWide = R <= 16 ? 4 : 2;
  const bool four = kWide == 4 && K % 4 == 0 &&
                    fold_smem_bytes<T>(d_r, R, 4) <= static_cast<size_t>(optin);
  const int cpt = four ? 4 : 2;
  const size_t smem = fold_smem_bytes<T>(d_r, R, cpt);
  if (smem > static_cast<size_t>(optin)) {
    set_error("hf_fold: unsupported: d_R x rank too large for one block's shared memory");
    return HF_ERR_UNSUPPORTED;
  }
  auto kern = four ? fold_kernel<T, R, kWide> : fold_kernel<T, R, 2>;
  HF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(smem)),
              "hf_fold: shared memory size");
  const int64_t cols = 32 * cpt;
  const unsigned kblocks = static_cast<unsigned>((K + cols - 1) / cols);
  kern<<<dim3(kblocks, n_maps), kFoldThreads, smem, stream>>>(
      static_cast<const T*>(W), B, G, static_cast<T*>(Wf), d_r, K);
  HF_CUDA_TRY(cudaGetLastError(), "hf_fold: launch");
  return HF_OK;
}

template <typename T>
hf_status launch_fold(int n_maps, int d_r, int64_t K, int rank, const void* W, const float* b,
                      const float* B, const float* G, void* Wf, float* bf, cudaStream_t stream) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  hf_status s = HF_OK;
  // the tensor-core form where its units fit and its chain of steps, about as long for
  // few rows and a low rank as for many, is the shorter way (tensor-core and fp32 form,
  // K 3,072, 80 maps: rank 16, d_R 1,024 253 and 484 us, 192 119 and 124, 128 118 and 98;
  // rank 8, 1,024 249 and 299, 640 206 and 194; rank 4, 1,024 248 and 243, 256 124 and
  // 71; one map of 1,024 x 3,072, rank 4: 14 and 26); in fp32 the maps need more than
  // bf16 products of an exact W, and two 16-deep steps of rank 32 more registers than
  // a warp's share of B and G leaves
  const int64_t units = n_maps * ((K + kMmaCols - 1) / kMmaCols);
  const int steps = (d_r + 16 * kMmaWarps - 1) / (16 * kMmaWarps);
  static constexpr int kLeast[4] = {3072, 4608, 6144, 7040};  // rank d_R, by steps
  const bool fits = sizeof(T) == 2 && (rank == 4 || rank == 8 || rank == 16) && d_r <= kMmaRows &&
                    K % 8 == 0 && sizeof(FoldMmaSmem) <= static_cast<size_t>(optin);
  const bool mma =
      fits && rank * d_r >= (units <= device_sm_count() ? 768 : kLeast[steps - 1]);
  if (mma) {
    HF_CUDA_TRY(cudaFuncSetAttribute(fold_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(sizeof(FoldMmaSmem))),
                "hf_fold: shared memory size");
    const int grid = static_cast<int>(std::max<int64_t>(
        std::min<int64_t>(units, device_sm_count()), (units + kMmaUnits - 1) / kMmaUnits));
    CUtensorMap map_out;
    s = bf16_strip_map(&map_out, Wf, n_maps, d_r, K, 16 * steps);
    if (s != HF_OK) return s;
    fold_mma_kernel<<<grid, 32 * kMmaWarps, sizeof(FoldMmaSmem), stream>>>(
        static_cast<const __nv_bfloat16*>(W), B, G, static_cast<__nv_bfloat16*>(Wf), map_out, n_maps, d_r, K, rank, steps);
    HF_CUDA_TRY(cudaGetLastError(), "hf_fold: launch");
  } else
  switch (rank) {
    case 4: s = launch_fold_r<T, 4>(n_maps, d_r, K, W, B, G, Wf, optin, stream); break;
    case 8: s = launch_fold_r<T, 8>(n_maps, d_r, K, W, B, G, Wf, optin, stream); break;
    case 16: s = launch_fold_r<T, 16>(n_maps, d_r, K, W, B, G, Wf, optin, stream); break;
    case 32: s = launch_fold_r<T, 32>(n_maps, d_r, K, W, B, G, Wf, optin, stream); break;
    default:
      set_error("hf_fold: unsupported: rank must be 4, 8, 16 or 32");
      return HF_ERR_UNSUPPORTED;
  }
  if (s != HF_OK) return s;
  auto bias = [&](auto kern) {
    return launch_dependent(kern, dim3(n_maps), dim3(256), 0, stream, b, B, G, bf, d_r);
  };
  HF_CUDA_TRY(rank == 4    ? bias(fold_b_kernel<4>)
              : rank == 8  ? bias(fold_b_kernel<8>)
              : rank == 16 ? bias(fold_b_kernel<16>)
                           : bias(fold_b_kernel<32>),
              "hf_fold: bias launch");
  return HF_OK;
}

}  // namespace
}  // namespace hf

using namespace hf;

extern "C" hf_status hf_fold(hf_dtype dtype, int32_t n_maps, int32_t d_R, int64_t K, int32_t rank,
                             const void* d_W, const float* d_b, const float* d_B,
                             const float* d_G, void* d_W_final, float* d_b_final,
                             hf_stream_t stream_) {
  if (dtype != HF_BF16 && dtype != HF_F32) {
    set_error("hf_fold: unknown dtype");
    return HF_ERR_INVALID_ARGUMENT;
  }
  if (n_maps < 1 || n_maps > 65535 || d_R < 1 || K < 1 || rank < 1 || rank > kMaxRank) {
    set_error("hf_fold: n_maps in [1, 65535], d_R >= 1, K >= 1, rank in [1, 32]");
    return HF_ERR_INVALID_ARGUMENT;
  }
  if (!d_W || !d_b || !d_B || !d_G || !d_W_final || !d_b_final) {
    set_error("hf_fold: null pointer");
    return HF_ERR_INVALID_ARGUMENT;
  }
  if ((reinterpret_cast<uintptr_t>(d_B) | reinterpret_cast<uintptr_t>(d_W) |
       reinterpret_cast<uintptr_t>(d_W_final)) & 15u || (K % 2)) {
    set_error("hf_fold: W, W_final and B must be 16-byte aligned and K even");
    return HF_ERR_INVALID_ARGUMENT;
  }
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  if (dtype == HF_BF16)
    return launch_fold<__nv_bfloat16>(n_maps, d_R, K, rank, d_W, d_b, d_B, d_G, d_W_final,
                                      d_b_final, stream);
  return launch_fold<float>(n_maps, d_R, K, rank, d_W, d_b, d_B, d_G, d_W_final, d_b_final,
                            stream);
}
