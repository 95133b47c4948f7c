// Operand rows made before the transfer.  Where a map input row is not a copy of
// one sender row (pooled alignment rows, blended or weighted layers, sender
// keys that are rotated back), this pass makes it once per receiver layer and
// role, as the value rounded to bf16 and, unless the plan rounds once, the
// bf16 rounding of what that lost; the transfer kernel then copies the rows
// like any other.  The loader warps of the transfer kernel build the same rows
// tile by tile, which repeats the work for every 512 (or 256) output columns
// with few loads in flight: an 8K interpolation took 1.12 ms and a 3K context
// with rotated sender keys 1.66 ms that way.
// Bounded by memory: at 8K interpolation 2 x 2 bytes read and 2 x 2 written per
// value.  A warp makes one row, eight values per lane and step.
#include <algorithm>

#include <cuda_bf16.h>

#include "hf_device.cuh"
#include "hf_internal.h"

namespace hf {
namespace {

constexpr int kRowWarps = 8;      // rows per block
constexpr int kRotLayers = 4;     // receiver layers per block: one row's angles serve them all

struct OperandArgs {
  const __nv_bfloat16* sender;
  __nv_bfloat16* out;
  const LayerSegs* segs;
  const int32_t* run_ptr;
  const int32_t* row_ptr;
  const int32_t* col;
  const float* w;
  const int32_t* srow;       // cache row of each aligned sender token, or null
  const int32_t* spos;       // sender position of each aligned token (rotated keys)
  const float* inv_freq_s;
  const int32_t* n_distinct;
  int64_t T_s, s_rows, rows;
  int d_s, D_s, K, l0, n_l;
  int roles, n_roles;        // made roles (bits), their number
  int split, tokens, rot;    // tokens: row r is aligned sender token r, weight 1
};

__device__ __forceinline__ void put_row_chunk(const OperandArgs& a, __nv_bfloat16* o, int64_t plane,
                                              const float* acc) {
  if (a.split) {
    uint4 hi, lo;
    pack16_split(acc, &hi, &lo);
    *reinterpret_cast<uint4*>(o) = hi;
    *reinterpret_cast<uint4*>(o + plane) = lo;
  } else {
    *reinterpret_cast<uint4*>(o) = pack16(acc, (const __nv_bfloat16*)nullptr);
  }
}

// The cache row and weight of the row's entry i (valid: inside the sender).
__device__ __forceinline__ bool row_entry(const OperandArgs& a, int64_t row, int e, int64_t* kr,
                                          int* k, float* wt) {
  *k = a.tokens ? static_cast<int>(row) : __ldg(a.col + e);
  if (*k < 0 || *k >= a.T_s) return false;  // flagged at plan creation
  *wt = a.tokens ? 1.f : __ldg(a.w + e);
  *kr = a.srow ? __ldg(a.srow + *k) : *k;
  return true;
}

// Rows of sums of weighted sender rows.
__global__ void __launch_bounds__(32 * kRowWarps) operand_sum_kernel(const __grid_constant__ OperandArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t n_rows = a.tokens ? a.T_s : *a.n_distinct;
  const int l = blockIdx.y;
  const int ri = blockIdx.z;
  const int c = a.rot ? 1 : a.n_roles == 2 ? ri : a.roles >> 1;  // rotated keys: only values here
  for (int64_t row = blockIdx.x * static_cast<int64_t>(kRowWarps) + (threadIdx.x >> 5); row < n_rows;
       row += static_cast<int64_t>(gridDim.x) * kRowWarps) {
    int e0 = 0, e1 = 1;
    if (!a.tokens) {
      const int j = __ldg(a.run_ptr + row);
      e0 = __ldg(a.row_ptr + j);
      e1 = __ldg(a.row_ptr + j + 1);
    }
    const LayerSegs* const sg = a.segs + a.l0 + l;
    const int64_t plane = a.rows * a.K;
    __nv_bfloat16* const out =
        a.out + static_cast<int64_t>(l * a.n_roles + (a.n_roles == 2 ? c : 0)) * (a.split ? 2 : 1) * plane +
        row * a.K;
    const int64_t lrows = a.s_rows * a.d_s;
    if (e1 - e0 == 1) {
      // one sender token: up to eight 16-byte reads a lane in flight
      int64_t kr = 0;
      int k;
      float wt = 0.f;
      const bool valid = row_entry(a, row, e0, &kr, &k, &wt);
      for (int el0 = 8 * lane; el0 < a.K; el0 += 4 * 256) {
        uint4 x[4][2];
        float om[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int el = el0 + 256 * i;
          om[i][0] = om[i][1] = 0.f;
          x[i][0] = x[i][1] = make_uint4(0u, 0u, 0u, 0u);
          if (el >= a.K || !valid) continue;
          const int seg = el / a.d_s;
          const __nv_bfloat16* const src = a.sender + kr * a.d_s + (el - seg * a.d_s);
          om[i][0] = a.tokens ? __ldg(&sg->w[seg][0]) : __ldg(&sg->w[seg][0]) * wt;
          x[i][0] = __ldg(reinterpret_cast<const uint4*>(src + (2 * __ldg(&sg->layer[seg][0]) + c) * lrows));
          if (__ldg(&sg->n_terms[seg]) > 1) {
            om[i][1] = a.tokens ? __ldg(&sg->w[seg][1]) : __ldg(&sg->w[seg][1]) * wt;
            x[i][1] = __ldg(reinterpret_cast<const uint4*>(src + (2 * __ldg(&sg->layer[seg][1]) + c) * lrows));
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int el = el0 + 256 * i;
          if (el >= a.K) break;
          float acc[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) acc[q] = 0.f;
          accum16(x[i][0], om[i][0], acc, (const __nv_bfloat16*)nullptr);
          accum16(x[i][1], om[i][1], acc, (const __nv_bfloat16*)nullptr);
          put_row_chunk(a, out + el, plane, acc);
        }
      }
      continue;
    }
    for (int el = 8 * lane; el < a.K; el += 256) {
      const int seg = el / a.d_s, in = el - seg * a.d_s;
      const int n_t = __ldg(&sg->n_terms[seg]);
      float acc[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = 0.f;
      for (int t = 0; t < n_t; ++t) {
        const float om = __ldg(&sg->w[seg][t]);
        const __nv_bfloat16* const base =
            a.sender + (2 * __ldg(&sg->layer[seg][t]) + c) * lrows + in;
        for (int e = e0; e < e1; ++e) {
          int64_t kr;
          int k;
          float wt;
          if (!row_entry(a, row, e, &kr, &k, &wt)) continue;
          accum16(__ldg(reinterpret_cast<const uint4*>(base + kr * a.d_s)), a.tokens ? om : om * wt, acc,
                  (const __nv_bfloat16*)nullptr);
        }
      }
      put_row_chunk(a, out + el, plane, acc);
    }
  }
}

// Rows of keys that carry RoPE: each sender row is rotated back at its own
// position, pair (x, y) = (i, i + D_s/2) of a head -> (x cos + y sin, y cos - x
// sin), before the weights.  A lane takes eight pairs a step, the same ones of
// every head, so a one-entry row's angles are formed once for kRotLayers layers.
__global__ void __launch_bounds__(32 * kRowWarps) operand_unrotate_kernel(const __grid_constant__ OperandArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t n_rows = *a.n_distinct;
  const int hs = a.D_s / 2, per_head = hs / 8;   // per_head divides 32
  const int i0 = (lane % per_head) * 8;
  float f[8], cs[8], sn[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) f[i] = __ldg(a.inv_freq_s + i0 + i);
  int at = -1;  // token whose angles cs and sn are
  const int64_t plane = a.rows * a.K, lrows = a.s_rows * a.d_s;
  const int l1 = min(a.n_l, static_cast<int>(blockIdx.y + 1) * kRotLayers);
  for (int64_t row = blockIdx.x * static_cast<int64_t>(kRowWarps) + (threadIdx.x >> 5); row < n_rows;
       row += static_cast<int64_t>(gridDim.x) * kRowWarps) {
    const int j = __ldg(a.run_ptr + row);
    const int e0 = __ldg(a.row_ptr + j), e1 = __ldg(a.row_ptr + j + 1);
    for (int l = blockIdx.y * kRotLayers; l < l1; ++l) {
      const LayerSegs* const sg = a.segs + a.l0 + l;
      __nv_bfloat16* const out =
          a.out + static_cast<int64_t>(l * a.n_roles) * (a.split ? 2 : 1) * plane + row * a.K;
      for (int pc = lane; pc < a.K / 16; pc += 32) {
        const int el = (pc / per_head) * a.D_s + i0;  // feature of the first half
        const int seg = el / a.d_s, in = el - seg * a.d_s;
        const int n_t = __ldg(&sg->n_terms[seg]);
        float ax[8], ay[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) ax[i] = ay[i] = 0.f;
        for (int t = 0; t < n_t; ++t) {
          const float om = __ldg(&sg->w[seg][t]);
          const __nv_bfloat16* const base = a.sender + 2 * __ldg(&sg->layer[seg][t]) * lrows + in;
          for (int e = e0; e < e1; ++e) {
            int64_t kr;
            int k;
            float wt;
            if (!row_entry(a, row, e, &kr, &k, &wt)) continue;
            const uint4 vx = __ldg(reinterpret_cast<const uint4*>(base + kr * a.d_s));
            const uint4 vy = __ldg(reinterpret_cast<const uint4*>(base + kr * a.d_s + hs));
            if (k != at) {
              at = k;
              const int p = __ldg(a.spos + k);
#pragma unroll
              for (int i = 0; i < 8; ++i) rope_sincos(p, f[i], &sn[i], &cs[i]);
            }
            wt *= om;
            float x[8], y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = y[i] = 0.f;
            accum16(vx, 1.f, x, (const __nv_bfloat16*)nullptr);
            accum16(vy, 1.f, y, (const __nv_bfloat16*)nullptr);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              ax[i] = fmaf(wt, fmaf(x[i], cs[i], y[i] * sn[i]), ax[i]);
              ay[i] = fmaf(wt, fmaf(y[i], cs[i], -x[i] * sn[i]), ay[i]);
            }
          }
        }
        put_row_chunk(a, out + el, plane, ax);
        put_row_chunk(a, out + el + hs, plane, ay);
      }
    }
  }
}

}  // namespace

hf_status launch_operands(const hf_plan_s* p, const void* sender, cudaStream_t stream, int l_begin,
                          int l_end) {
  const hf_plan_desc& d = p->desc;
  char* const ws = p->ws;
  auto i32 = [&](size_t off) { return reinterpret_cast<const int32_t*>(ws + off); };
  OperandArgs a;
  a.sender = static_cast<const __nv_bfloat16*>(sender);
  a.out = reinterpret_cast<__nv_bfloat16*>(ws + p->lay.xbuf);
  a.segs = reinterpret_cast<const LayerSegs*>(ws + p->lay.segs);
  a.run_ptr = i32(p->lay.run_ptr);
  a.row_ptr = d.d_row_ptr;
  a.col = d.d_col;
  a.w = d.d_w;
  a.srow = p->span ? i32(p->lay.srow) : nullptr;
  a.spos = i32(p->lay.spos);
  a.inv_freq_s = reinterpret_cast<const float*>(ws + p->lay.inv_freq_s);
  a.n_distinct = i32(p->lay.n_distinct);
  a.T_s = p->T_s;
  a.s_rows = p->s_rows;
  a.rows = p->x_rows;
  a.d_s = p->d_s;
  a.D_s = d.D_s;
  a.K = p->K;
  a.l0 = l_begin;
  a.n_l = l_end - l_begin;
  a.roles = p->made;
  a.n_roles = p->made == 3 ? 2 : 1;
  a.split = p->split ? 1 : 0;
  a.tokens = p->pam ? 1 : 0;
  a.rot = p->unrot ? 1 : 0;
  // the number of distinct rows, about a quarter of x_rows with Token Alignment,
  // is on the device: blocks beyond two an SM loop instead (idle ones cost a
  // third of the pass)
  const unsigned blocks = static_cast<unsigned>(std::min<int64_t>(
      (p->x_rows + kRowWarps - 1) / kRowWarps, 2 * device_sm_count()));
  if (p->unrot)
    operand_unrotate_kernel<<<dim3(blocks, (a.n_l + kRotLayers - 1) / kRotLayers), 32 * kRowWarps, 0,
                              stream>>>(a);
  if (!p->unrot || p->made == 3)
    operand_sum_kernel<<<dim3(blocks, a.n_l, p->unrot ? 1 : a.n_roles), 32 * kRowWarps, 0, stream>>>(a);
  HF_CUDA_TRY(cudaGetLastError(), "operand rows launch");
  return HF_OK;
}

}  // namespace hf
