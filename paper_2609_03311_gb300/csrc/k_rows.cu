// k_rows.cu -- the memory-bound per-row kernels of the decoder pass: the
//   embedding gather (with the first RMSNorm's operand and sum of squares),
//   the two-row score head, and the prefix-store layout transpose.  The other
//   RMSNorms and the q/k norm + RoPE are fused into the GEMM epilogues.
// 16-byte vector accesses; the kernels whose rows are few give a row a whole block.
#include <algorithm>

#include "device_common.cuh"
#include "internal.h"

namespace dopr {
namespace {

// Sum of v over the block's WARPS warps (every thread gets it); red: WARPS floats of shared memory.
template <int WARPS>
__device__ __forceinline__ float block_sum(float v, float* red) {
  v = warp_sum(v);
  __syncthreads();  // red is reused across calls
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) t += red[w];
  return t;
}

// Four consecutive bf16 values (8-byte aligned) as floats.
__device__ __forceinline__ void bf16x4_to_float(const bf16* p, float (&v)[4]) {
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
  v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}

// One warp per row: r = E[id] widened to fp32, ss = sum(r^2),
// xn = f16(r * rsqrt(ss/H + eps) * g).  Bound by its 8 H bytes a row, and in small calls by
// latency: EMBED_AHEAD 16-byte loads are in flight per lane (one at a time took 16 rounds for a
// 4,096-element row).  The row is read twice (the second read hits L1).  4,096 elements:
// 25 rows 9.7 -> 7.6 us, 3,800 rows 29.3 -> 26.1 us, 32,768 rows 171 -> 158 us.
constexpr int ROW_WARPS = 4, EMBED_AHEAD = 8;
__global__ void __launch_bounds__(ROW_WARPS * 32)
    k_embed(const int32_t* tok_id, int T, const bf16* __restrict__ embed, const bf16* __restrict__ gain,
            int H, float eps, float* __restrict__ r, f16* __restrict__ xn, float* __restrict__ ss_out, Extents ext) {
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x * ROW_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= T) return;
  const int64_t id = tok_id[row];
  if (!index_ok(ext.err, id, ext.table_rows) || !index_ok(ext.err, row, ext.rows)) return;
  const bf16* e = embed + id * H;
  float* rr = r + static_cast<int64_t>(row) * H;
  f16* xr = xn + static_cast<int64_t>(row) * H;
  float ss = 0.f;
  for (int c0 = lane * 8; c0 < H; c0 += 256 * EMBED_AHEAD) {
    uint4 w[EMBED_AHEAD];
#pragma unroll
    for (int q = 0; q < EMBED_AHEAD; ++q)
      if (c0 + 256 * q < H) w[q] = *reinterpret_cast<const uint4*>(e + c0 + 256 * q);
#pragma unroll
    for (int q = 0; q < EMBED_AHEAD; ++q)
      if (c0 + 256 * q < H) {
        const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(&w[q]);
        float v[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 a = __bfloat1622float2(w2[k]);
          v[2 * k] = a.x;
          v[2 * k + 1] = a.y;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) ss = fmaf(v[k], v[k], ss);
        float* dst = rr + c0 + 256 * q;
        *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
      }
  }
  ss = warp_sum(ss);
  const float inv = rsqrtf(ss / static_cast<float>(H) + eps);
  bool bad = false;
#pragma unroll 4
  for (int c = lane * 8; c < H; c += 256) {
    const uint4 w = *reinterpret_cast<const uint4*>(e + c);
    const uint4 gw = *reinterpret_cast<const uint4*>(gain + c);
    const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(&w);
    const __nv_bfloat162* g2 = reinterpret_cast<const __nv_bfloat162*>(&gw);
    uint32_t o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 a = __bfloat1622float2(w2[k]), b = __bfloat1622float2(g2[k]);
      const float x0 = a.x * inv * b.x, x1 = a.y * inv * b.y;
      bad |= !(fp16_ok(x0) && fp16_ok(x1));
      o[k] = pack_f16x2(x0, x1);
    }
    *reinterpret_cast<uint4*>(xr + c) = make_uint4(o[0], o[1], o[2], o[3]);
  }
  report_range(ext.err, bad);
  if (lane == 0) ss_out[row] = ss;
}

// In place bf16 -> fp16 over n values (n even), one 32-bit word per thread and
// step; *range |= 1 when a value is not finite or outside fp16's range.
__global__ void k_bf16_to_f16(uint32_t* __restrict__ buf, int64_t n_words, int* range) {
  bool bad = false;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n_words;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    buf[i] = bf16x2_to_f16x2(buf[i], bad);
  if (bad) atomicOr(range, 1);
}

// Score head at the score-token row of each sorted pair in [p_begin, p_end):
// s = <W[0] - W[1], RMSNorm(r_row) * g>, written to scores[perm[pair]].  One CTA per pair: a
// call has few pairs, so what counts is the latency of a row (4,096 elements: a warp per row
// walked it in 192 dependent loads, 37-40 us; a block in four rounds, 6 us).
constexpr int SCORE_THREADS = 256;
__global__ void __launch_bounds__(SCORE_THREADS)
    k_score(const float* r, int H, const int32_t* __restrict__ tok_off, int tok0, int p_begin, int compact,
            const int32_t* __restrict__ perm, const bf16* __restrict__ gain, const bf16* __restrict__ head, float eps,
            float* __restrict__ scores, Extents ext) {
  __shared__ float red[SCORE_THREADS / 32];
  pdl_trigger();
  pdl_wait();
  const int s = p_begin + blockIdx.x;
  const int64_t row = compact ? s - p_begin : tok_off[s + 1] - 1 - tok0;
  if (!index_ok(ext.err, row, ext.rows)) return;  // uniform across the block
  const float* x = r + row * H;
  float ss = 0.f;
#pragma unroll 4
  for (int c = threadIdx.x * 4; c < H; c += SCORE_THREADS * 4) {
    const float4 v = *reinterpret_cast<const float4*>(x + c);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  const float inv = rsqrtf(block_sum<SCORE_THREADS / 32>(ss, red) / static_cast<float>(H) + eps);
  float yes = 0.f, no = 0.f;
#pragma unroll 4
  for (int c = threadIdx.x * 4; c < H; c += SCORE_THREADS * 4) {
    const float4 v = *reinterpret_cast<const float4*>(x + c);
    float g[4], a[4], b[4];
    bf16x4_to_float(gain + c, g);
    bf16x4_to_float(head + c, a);
    bf16x4_to_float(head + H + c, b);
    const float h[4] = {v.x * inv * g[0], v.y * inv * g[1], v.z * inv * g[2], v.w * inv * g[3]};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      yes += h[k] * a[k];
      no += h[k] * b[k];
    }
  }
  yes = block_sum<SCORE_THREADS / 32>(yes, red);
  no = block_sum<SCORE_THREADS / 32>(no, red);
  const float sc = yes - no;
  if (threadIdx.x == 0) {
    if (!isfinite(sc) && ext.err) atomicOr(ext.err, DEV_ERR_RANGE);
    scores[perm[s]] = sc;
  }
}

// MLP scoring head (Sec. 3.2.3): act(W1 hn + b1) . w2 + b2 with hn = RMSNorm(row) * g.
// A CTA takes MLP_PAIRS pairs and, 32 at a time, its share of the hidden units, four to a warp:
// the elements of hn go through shared memory MLP_CHUNK at a time, a lane multiplies its
// elements of four W1 rows into all eight pairs (fp32), so a W1 element is read from L2 once
// for eight pairs, and not once a pair, and each pass over a pair's hn serves 32 units.  The
// sums over a CTA's units go to part[pair][split]; k_score_mlp_sum adds them in split order.
// 50 pairs, 1,024 units, 2,560 elements, cold cache: one CTA per pair 508 us, these 24 + 4 us.
constexpr int MLP_WARPS = 8, MLP_PAIRS = 8, MLP_UNITS = 4, MLP_CHUNK = 1024;
constexpr int MLP_THREADS = 32 * MLP_WARPS;
constexpr int MLP_PASS = MLP_WARPS * MLP_UNITS;  // hidden units of one pass
__device__ __forceinline__ float head_act(float z, int act) {
  switch (act) {
    case 0: return fmaxf(z, 0.f);
    case 1: return 0.5f * z * (1.f + erff(z * 0.70710678118654752f));
    case 2: return z / (1.f + expf(-z));
    default: return tanhf(z);
  }
}
__global__ void __launch_bounds__(MLP_THREADS)
    k_score_mlp(const float* r, int H, const int32_t* __restrict__ tok_off, int tok0, int p_begin,
                int p_end, int compact, const bf16* __restrict__ gain, float eps, int width, int act,
                const bf16* __restrict__ w1, const bf16* __restrict__ b1, const bf16* __restrict__ w2, int passes,
                float* __restrict__ part, Extents ext) {
  __shared__ float hn[MLP_PAIRS][MLP_CHUNK];
  __shared__ float red[MLP_WARPS][MLP_PAIRS];
  pdl_trigger();
  pdl_wait();
  const int s0 = p_begin + blockIdx.x * MLP_PAIRS, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  static_assert(MLP_WARPS == MLP_PAIRS, "a warp stages a pair");
  // this warp's pair: its row and norm factor (pairs past p_end stage zeros)
  const float* x = nullptr;
  if (s0 + warp < p_end) {
    const int64_t row = compact ? s0 + warp - p_begin : tok_off[s0 + warp + 1] - 1 - tok0;
    if (index_ok(ext.err, row, ext.rows)) x = r + row * H;
  }
  float ss = 0.f;
  if (x) {
#pragma unroll 8
    for (int c = lane * 4; c < H; c += 128) {
      const float4 v = *reinterpret_cast<const float4*>(x + c);
      ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
  }
  const float inv = rsqrtf(warp_sum(ss) / static_cast<float>(H) + eps);
  float total = 0.f;  // lane i < MLP_PAIRS: pair i's sum over this warp's units
  for (int q = 0; q < passes; ++q) {
    const int j0 = (static_cast<int>(blockIdx.y) * passes + q) * MLP_PASS + warp * MLP_UNITS;
    float z[MLP_UNITS][MLP_PAIRS];
#pragma unroll
    for (int u = 0; u < MLP_UNITS; ++u)
#pragma unroll
      for (int i = 0; i < MLP_PAIRS; ++i) z[u][i] = 0.f;
    for (int c0 = 0; c0 < H; c0 += MLP_CHUNK) {
      const int n = min(MLP_CHUNK, H - c0);  // a multiple of 256
      __syncthreads();
#pragma unroll 8
      for (int c = lane * 4; c < n; c += 128) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (x) {
          v = *reinterpret_cast<const float4*>(x + c0 + c);
          float g[4];
          bf16x4_to_float(gain + c0 + c, g);
          v = make_float4(v.x * inv * g[0], v.y * inv * g[1], v.z * inv * g[2], v.w * inv * g[3]);
        }
        *reinterpret_cast<float4*>(&hn[warp][c]) = v;
      }
      __syncthreads();
      if (j0 < width) {
#pragma unroll 2
        for (int c = lane * 4; c < n; c += 128) {
          float w[MLP_UNITS][4];
#pragma unroll
          for (int u = 0; u < MLP_UNITS; ++u)  // units past the width read its last row and are dropped
            bf16x4_to_float(w1 + static_cast<int64_t>(min(j0 + u, width - 1)) * H + c0 + c, w[u]);
#pragma unroll
          for (int i = 0; i < MLP_PAIRS; ++i) {
            const float4 h = *reinterpret_cast<const float4*>(&hn[i][c]);
#pragma unroll
            for (int u = 0; u < MLP_UNITS; ++u)
              z[u][i] += w[u][0] * h.x + w[u][1] * h.y + w[u][2] * h.z + w[u][3] * h.w;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < MLP_UNITS; ++u) {
      float mine = 0.f;
#pragma unroll
      for (int i = 0; i < MLP_PAIRS; ++i) {
        const float v = warp_sum(z[u][i]);
        if (lane == i) mine = v;
      }
      if (j0 + u < width)
        total += head_act(mine + __bfloat162float(b1[j0 + u]), act) * __bfloat162float(w2[j0 + u]);
    }
  }
  if (lane < MLP_PAIRS) red[warp][lane] = total;
  __syncthreads();
  if (threadIdx.x < MLP_PAIRS && s0 + static_cast<int>(threadIdx.x) < p_end) {
    float t = 0.f;
    for (int w = 0; w < MLP_WARPS; ++w) t += red[w][threadIdx.x];
    part[static_cast<int64_t>(s0 + threadIdx.x - p_begin) * gridDim.y + blockIdx.y] = t;
  }
}
// One warp per pair: its splits' sums in order, and b2.
__global__ void k_score_mlp_sum(const float* part, int splits, int n, const int32_t* __restrict__ perm, float b2,
                                float* __restrict__ scores, int* err) {
  pdl_trigger();
  pdl_wait();
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= n) return;
  float t = 0.f;
  for (int k = lane; k < splits; k += 32) t += part[static_cast<int64_t>(i) * splits + k];
  const float sc = warp_sum(t) + b2;
  if (lane == 0) {
    if (!isfinite(sc) && err) atomicOr(err, DEV_ERR_RANGE);
    scores[perm[i]] = sc;
  }
}

// One block per pair: copy its score-token row of r (and of the partial sums) to row i (8.1 ->
// 4.5 us at 1-100 pairs of 4,096 elements: a latency, like the score head's).
constexpr int GATHER_THREADS = 256;
__global__ void __launch_bounds__(GATHER_THREADS)
    k_gather_score_rows(const float* r, const float* ss, int H, int parts,
                        const int32_t* __restrict__ tok_off, int tok0, int p_begin, float* __restrict__ dst_r,
                        float* __restrict__ dst_ss, Extents ext) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x;
  const int64_t row = tok_off[p_begin + i + 1] - 1 - tok0;
  if (!index_ok(ext.err, row, ext.rows) || !index_ok(ext.err, i, ext.rows)) return;
  const float4* src = reinterpret_cast<const float4*>(r + row * H);
  float4* dst = reinterpret_cast<float4*>(dst_r + static_cast<int64_t>(i) * H);
#pragma unroll 4
  for (int c = threadIdx.x; c < H / 4; c += GATHER_THREADS) dst[c] = src[c];
  for (int c = threadIdx.x; c < parts; c += GATHER_THREADS) dst_ss[static_cast<int64_t>(i) * parts + c] = ss[row * parts + c];
}

// [m][Hkv][128] bf16 -> [Hkv][m][128] fp16 for K and V (8 elements per thread).
// bf16 -> fp16 is exact for every value of fp16's normal range; values beyond it
// (or not finite) are flagged in *range.
__device__ __forceinline__ uint4 bf16x8_to_f16x8(uint4 x, int& bad) {
  uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
    bad |= !(fabsf(f.x) <= 65504.f) || !(fabsf(f.y) <= 65504.f);
    w[i] = pack_f16x2(f.x, f.y);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__global__ void k_store_transpose(const uint4* __restrict__ k, const uint4* __restrict__ v, int m, int Hkv,
                                  uint4* __restrict__ dk, uint4* __restrict__ dv, int* range) {
  const int64_t n = static_cast<int64_t>(m) * Hkv * (HEAD_DIM / 8);
  int bad = 0;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(i % (HEAD_DIM / 8));
    const int64_t rest = i / (HEAD_DIM / 8);
    const int h = static_cast<int>(rest % Hkv);
    const int64_t j = rest / Hkv;
    const int64_t o = (static_cast<int64_t>(h) * m + j) * (HEAD_DIM / 8) + c;
    dk[o] = bf16x8_to_f16x8(k[i], bad);
    dv[o] = bf16x8_to_f16x8(v[i], bad);
  }
  if (bad) atomicOr(range, 1);
}

// Prefix build (Sec. 3.3): copy each token's key (after the q/k norm and RoPE) and
// raw value of every kv head from the packed QKV buffer into its document's block of
// the store pool, in the layout dopr_store_put writes: per layer, K then V, per kv
// head, m rows of 128.  One warp per (token, kv head, K|V), 8 bytes a lane.
__global__ void k_prefix_store(const f16* qkv, int ld_qkv, int T, int t0, int Hq, int Hkv,
                               const int32_t* __restrict__ tok_pair, const int32_t* __restrict__ tok_pos,
                               const int32_t* __restrict__ pair_slot, const int64_t* __restrict__ slot_row,
                               const int32_t* __restrict__ slot_m, int layer, f16* __restrict__ pool, Extents ext) {
  pdl_trigger();
  pdl_wait();
  const int64_t w = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= static_cast<int64_t>(T) * Hkv * 2) return;
  const int kv = static_cast<int>(w & 1);
  const int g = static_cast<int>((w >> 1) % Hkv);
  const int t = static_cast<int>((w >> 1) / Hkv);
  const int p = tok_pair[t0 + t], j = tok_pos[t0 + t];
  const int slot = pair_slot[p];
  const int64_t row = slot_row[slot] + (static_cast<int64_t>(layer * 2 + kv) * Hkv + g) * slot_m[slot] + j;
  if (!index_ok(ext.err, j, slot_m[slot]) || !index_ok(ext.err, row, ext.pool_rows)) return;
  const uint2* src = reinterpret_cast<const uint2*>(qkv + static_cast<int64_t>(t) * ld_qkv + (Hq + kv * Hkv + g) * HEAD_DIM);
  reinterpret_cast<uint2*>(pool + row * HEAD_DIM)[lane] = src[lane];
}

// Test kernel: a bounded wait on an mbarrier that is never completed (block 0, error word err[0])
// and one at a gate that is never opened (block 1, err[1]; the gate is err[2]).
__global__ void k_wait_timeout_probe(int* err, uint64_t timeout_ns) {
  if (blockIdx.x == 1) {
    gate_wait_warp(err + 2, 1, err + 1, timeout_ns);
    return;
  }
  __shared__ uint64_t bar;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    mbar_init(b, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(b, 0, err, timeout_ns);  // nothing arrives: gives up
  __syncthreads();
}

}  // namespace

cudaError_t launch_embed(const int32_t* tok_id, int T, const bf16* embed, const bf16* gain, int H, float eps, float* r,
                         f16* xn, float* ss, const Extents& ext, cudaStream_t st) {
  if (T <= 0) return cudaSuccess;
  return launch_dependent(k_embed, (T + ROW_WARPS - 1) / ROW_WARPS, ROW_WARPS * 32, 0, st, tok_id, T, embed, gain, H, eps,
                          r, xn, ss, ext);
}

cudaError_t launch_bf16_to_f16(void* buf, int64_t n, int* range, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t words = n / 2;
  int blocks = static_cast<int>(std::min<int64_t>((words + 255) / 256, 4096));
  k_bf16_to_f16<<<blocks, 256, 0, st>>>(static_cast<uint32_t*>(buf), words, range);
  return cudaGetLastError();
}

cudaError_t launch_score(const float* r, int H, const int32_t* tok_off, int tok0, int p_begin, int p_end, int compact,
                         const int32_t* perm, const bf16* gain, const bf16* head, float eps, float* scores,
                         const Extents& ext, cudaStream_t st) {
  if (p_end <= p_begin) return cudaSuccess;
  return launch_dependent(k_score, p_end - p_begin, SCORE_THREADS, 0, st, r, H, tok_off, tok0, p_begin, compact, perm, gain,
                          head, eps, scores, ext);
}

int mlp_splits(int width) {
  const int passes = (width + MLP_PASS - 1) / MLP_PASS;
  return passes <= MLP_MAX_SPLITS ? passes : (passes + 1) / 2;  // width <= 16,384: 512 passes
}

cudaError_t launch_score_mlp(const float* r, int H, const int32_t* tok_off, int tok0, int p_begin, int p_end,
                             int compact, const int32_t* perm, const bf16* gain, float eps, int width, int act,
                             const bf16* w1, const bf16* b1, const bf16* w2, float b2, float* part, float* scores,
                             const Extents& ext, cudaStream_t st) {
  if (p_end <= p_begin) return cudaSuccess;
  const int n = p_end - p_begin, splits = mlp_splits(width);
  const int passes = (width + MLP_PASS * splits - 1) / (MLP_PASS * splits);
  const cudaError_t e = launch_dependent(k_score_mlp, dim3((n + MLP_PAIRS - 1) / MLP_PAIRS, splits), MLP_THREADS, 0, st, r, H,
                                         tok_off, tok0, p_begin, p_end, compact, gain, eps, width, act, w1, b1, w2, passes,
                                         part, ext);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_score_mlp_sum, (n + 3) / 4, 128, 0, st, part, splits, n, perm + p_begin, b2, scores, ext.err);
}

cudaError_t launch_gather_score_rows(const float* r, const float* ss, int H, int parts, const int32_t* tok_off,
                                     int tok0, int p_begin, int p_end, float* dst_r, float* dst_ss,
                                     const Extents& ext, cudaStream_t st) {
  if (p_end <= p_begin) return cudaSuccess;
  return launch_dependent(k_gather_score_rows, p_end - p_begin, GATHER_THREADS, 0, st, r, ss, H, parts, tok_off, tok0, p_begin,
                          dst_r, dst_ss, ext);
}

cudaError_t launch_store_transpose(const bf16* k, const bf16* v, int m, int Hkv, f16* dk, f16* dv, int* range,
                                   cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  const int64_t n = static_cast<int64_t>(m) * Hkv * (HEAD_DIM / 8);
  const int blocks = static_cast<int>((n + 255) / 256);
  k_store_transpose<<<blocks, 256, 0, st>>>(reinterpret_cast<const uint4*>(k), reinterpret_cast<const uint4*>(v), m,
                                            Hkv, reinterpret_cast<uint4*>(dk), reinterpret_cast<uint4*>(dv), range);
  return cudaGetLastError();
}

cudaError_t launch_prefix_store(const f16* qkv, int ld_qkv, int T, int t0, int Hq, int Hkv, const int32_t* tok_pair,
                                const int32_t* tok_pos, const int32_t* pair_slot, const int64_t* slot_row,
                                const int32_t* slot_m, int layer, f16* pool, const Extents& ext, cudaStream_t st) {
  const int64_t threads = static_cast<int64_t>(T) * Hkv * 2 * 32;
  if (threads <= 0) return cudaSuccess;
  return launch_dependent(k_prefix_store, static_cast<unsigned>((threads + 255) / 256), 256, 0, st, qkv, ld_qkv, T, t0, Hq, Hkv,
                          tok_pair, tok_pos, pair_slot, slot_row, slot_m, layer, pool, ext);
}

cudaError_t launch_wait_timeout_probe(int* err, uint64_t timeout_ns, cudaStream_t st) {
  k_wait_timeout_probe<<<2, 32, 0, st>>>(err, timeout_ns);
  return cudaGetLastError();
}

}  // namespace dopr
