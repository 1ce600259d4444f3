// k_gemm.cu -- dense projections of the decoder (QKV, O, gate/up, down) on
// the 5th-generation tensor cores: C[M][N] = A[M][K] * B[N][K]^T, fp16
// operands, fp32 accumulate in tensor memory, fused epilogues.
//
// Design (sm_103a, CTA pairs, persistent): a cluster of two CTAs on two SMs
// computes one 256 x 256 output tile with tcgen05 cta_group::2 MMAs (M = 256,
// N = 256, K = 16).  Each CTA stages its own 128 rows of A and its own 128 of
// the tile's 256 B rows per 64-wide k-block (32 KiB a stage, 6-stage ring,
// 128-byte swizzle); the MMAs read both CTAs' shared memory, so per SM a
// third less operand data moves into shared memory and out of it into the
// tensor core per FLOP than with a 128 x 256 tile on one SM.  Roles:
//   warp 0      (both CTAs) TMA producer; the copies of both CTAs complete on
//               the leader's full barrier of the stage;
//   warp 1      allocates 512 TMEM columns in both CTAs (two accumulators of
//               256 columns); in the leader one lane issues the MMAs and
//               commits stage releases and accumulator-ready barriers to both
//               CTAs (multicast), the whole warp running the loop;
//   warps 2..9  (both CTAs) epilogue on the CTA's 128 rows of the tile:
//               tcgen05.ld the finished accumulator (one TMEM lane quarter =
//               32 rows per warp, one row per thread; two warps per quarter,
//               each taking half of the tile's 256 columns, or for two rotated
//               heads half of the frequencies), tell the leader that the
//               accumulator is free after its last read, so the next tile's
//               MMAs overlap the rest, and bring 32x32-word chunks through
//               shared memory (16-byte chunks swizzled by the row) from the
//               row-per-thread layout into one where consecutive lanes hold a
//               row segment: 8 lanes 128 bytes of a row, in the QKV rotation
//               4 lanes 32 bytes of either half of a head.
// Tiles are visited in L2 groups (pair_tile_order): blocks of activation rows (up to
// 48 MiB: 4,096 rows at K = 4,096) that stay in L2 while the weight tiles stream past
// them, or, for the residual-epilogue launches, blocks of weight columns while the
// activations stream.  Groups of 2,048 activation rows at every K streamed the weights
// twice as often from HBM (gate/up: 3.5 GB read per 26,800-row launch instead of 1.9),
// and under the power cap that traffic cost about 1 % of SM clock and throughput.
//
// Fused epilogues (the decoder's RMSNorms live here, not in separate kernels):
//   RMSNorm(r) * g = rs * (r (.) g) with rs = rsqrt(mean(r^2) + eps).  The
//   residual-add epilogue writes r' = r + C, the next GEMM's operand
//   f16(r' (.) g_next * rs_pre) -- rs_pre is the row's previous norm factor,
//   which keeps the operand near unit scale -- and, per row and 128 columns,
//   the partial sum of r'^2.  The consuming GEMM sums those partials
//   (in a fixed order) and scales its accumulator rows by rs / rs_pre.
//   QKV epilogue: row scale, then per 128-column q/k head RMSNorm with the
//   q/k gain and rotate-half RoPE at the token's position (pairs i, i+64),
//   the rotation applied in the transposed layout so RoPE-table reads coalesce.
//   SwiGLU epilogue: silu(rs * gate) * (rs * up).
//   Every value written as fp16 is checked against fp16's range (DEV_ERR_RANGE).
// Every barrier wait is bounded (DEV_ERR_TIMEOUT) and the kernel always drains
// its own MMAs and frees TMEM before returning.
#include <type_traits>

#include "device_common.cuh"
#include "internal.h"

namespace dopr {
namespace {

constexpr int BM = GEMM_BM, BN = GEMM_BN, BK = GEMM_BK;  // BM: one CTA's rows of a pair tile
static_assert(GEMM_B_BOX == BM, "each CTA of a pair stages 128 of a tile's 256 B rows");
constexpr int A_BYTES = BM * BK * 2;  // 16 KiB
constexpr int THREADS = 320;
constexpr int EPI_WARPS = 8;
constexpr int XPOSE_WORDS = 32 * 32;  // per epilogue warp: 32 rows x 32 words, 16-byte chunks swizzled by the row
constexpr int XPOSE_BYTES = EPI_WARPS * XPOSE_WORDS * 4;
constexpr int BAR_BYTES = 256;

// silu(x) = x / (1 + e^-x) with the fast division (within 2 ulp of fp32, far below the fp16
// rounding of the output; tends to 0 as x -> -inf): the exact division's instruction
// sequence made the SwiGLU epilogue outlast short main loops (K = 1,024).
__device__ __forceinline__ float silu_f(float x) { return __fdividef(x, 1.0f + __expf(-x)); }

// RMSNorm factor of a row from its partial sums of squares (one per 128 columns), added in index
// order.  When the count allows, the partials arrive as independent 16-byte
// loads (up to 32 in flight) instead of one dependent load per partial.
__device__ __forceinline__ float norm_factor(const float* ss, int parts, const GemmParams& p, int row) {
  if (!ss) return 1.f;
  const float* s = ss + static_cast<int64_t>(min(row, p.M - 1)) * parts;
  float t = 0.f;
  if ((parts & 3) == 0) {
    for (int i = 0; i < parts; i += 32) {
      float4 v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        v[q] = i + 4 * q < parts ? reinterpret_cast<const float4*>(s + i)[q] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (i + 4 * q < parts) {
          t += v[q].x;
          t += v[q].y;
          t += v[q].z;
          t += v[q].w;
        }
    }
  } else {
    for (int i = 0; i < parts; ++i) t += s[i];
  }
  return rsqrtf(t / static_cast<float>(p.norm_dim) + p.eps);
}
// Consumer-side row scale: the operand was written as r * g * rs(ss_pre).
__device__ __forceinline__ float row_scale(const GemmParams& p, int row) {
  return norm_factor(p.ss_in, p.ss_parts, p, row) / norm_factor(p.ss_pre, p.ss_pre_parts, p, row);
}

// The partial sum of squares of 128 columns of rows row0 + i*4 + lane/8 (i = 0..7) from the lanes'
// own sums over their columns.
__device__ __forceinline__ void store_square_sums(const GemmParams& p, int row0, int lane, int group,
                                                  const float (&ss)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float t = ss[i];
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 4);
    const int r = i * 4 + (lane >> 3);
    if ((lane & 7) == 0 && row0 + r < p.M) p.ss_out[static_cast<int64_t>(row0 + r) * p.ss_out_parts + group] = t;
  }
}

// A narrow tile's warp holds the lanes' sums over one 32-column chunk (of the group's four) for
// its 32 rows.  The warps that hold the group's chunks may be in different CTAs: each leaves its
// lanes' sums in global memory and counts itself in; the last to come adds the chunks up in
// column order, exactly as a wide tile's warp does with its own, and clears the count.  Nothing
// waits.
__device__ __forceinline__ void publish_square_sums(const GemmParams& p, int row0, int lane, int group, int chunk,
                                                    const float (&ss)[8]) {
  const int64_t at = static_cast<int64_t>((row0 - p.row_begin) / 32) * p.ss_out_parts + group;
  float* mine = p.ss_chunks + ((at * 4 + chunk) * 8) * 32 + lane;
#pragma unroll
  for (int i = 0; i < 8; ++i) __stcg(mine + i * 32, ss[i]);
  __threadfence();
  __syncwarp();
  int before = 0;
  if (lane == 0) before = atomicAdd(p.ss_count + at, 1);
  if (__shfl_sync(0xffffffffu, before, 0) != 3) return;
  __threadfence();
  if (lane == 0) p.ss_count[at] = 0;
  float sum[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float* c = p.ss_chunks + (at * 32 + i) * 32 + lane;  // chunk k at + k * 256
    sum[i] = ((__ldcg(c) + __ldcg(c + 256)) + __ldcg(c + 512)) + __ldcg(c + 768);
  }
  store_square_sums(p, row0, lane, group, sum);
}

// Four words (a 16-byte chunk) of a row in a warp's transpose buffer: chunk c of row r lies at
// c ^ s(r) with s a permutation of r & 7 that sends neighbours 4 apart, so that a lane writing its
// own row, eight lanes reading one row and two times four lanes reading the same half of two
// neighbouring rows all move whole 16-byte chunks without bank conflicts.
__device__ __forceinline__ uint4* xs_chunk(uint32_t* xs, int r, int c) {
  return reinterpret_cast<uint4*>(xs + r * 32 + ((c ^ ((r & 1) << 2 | (r >> 1 & 3))) << 2));
}
__device__ __forceinline__ void xs_put_row(uint32_t* xs, int lane, const uint32_t (&v)[32]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) *xs_chunk(xs, lane, c) = make_uint4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
}
__device__ __forceinline__ float4 xs_get(uint32_t* xs, int r, int c) {
  const uint4 w = *xs_chunk(xs, r, c);
  return make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
}

// The warp's 32 rows x 32 words sit in `xs` (row-per-lane layout, xs_chunk).
// Write the first WORDS words of each row out transposed: with 32 words lane L covers rows
// i*4 + L/8 (i = 0..7) and words (L%8)*4 .. +3, i.e. 8 lanes per 128-byte row segment
// (16 words: 4 lanes per 64-byte segment).  dst(r, w) is where word w of row r goes.
template <int WORDS, typename RowPtr>
__device__ __forceinline__ void store_words_transposed(uint32_t* xs, int lane, int row0, int M, RowPtr dst) {
  constexpr int LANES = WORDS / 4;  // lanes to a row segment
  static_assert(WORDS == 32 || WORDS == 16, "row segments of 128 or 64 bytes");
#pragma unroll
  for (int i = 0; i < LANES; ++i) {
    const int r = i * (32 / LANES) + lane / LANES;
    const int w = (lane % LANES) * 4;
    if (row0 + r < M) {
      const uint4 v = *xs_chunk(xs, r, w >> 2);
      *reinterpret_cast<uint4*>(dst(r, w)) = v;
    }
  }
}

// What an epilogue reads that does not depend on the accumulator: fetched while
// the tile's main loop still runs, so its load latency is off the epilogue's path.
struct EpiPre {
  float scale;  // this thread's row: the consumer row scale (QKV, SwiGLU) or the previous norm factor
  int pos[4];   // QKV: positions of the 4 rows a lane rotates in the transposed layout
  float4 res[2][8];  // residual add: the lane's values of the warp's first two 32-column chunks
  uint2 gain;        // and the next norm's gains of the lane's four columns of the first
};

__device__ __forceinline__ void bf16x4_floats(uint2 w, float (&v)[4]) {
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
  v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}

// The residual values of lane L, rows i*4 + L/8 of the warp, columns col + (L%8)*4..+3.
__device__ __forceinline__ float4* residual_at(const GemmParams& p, int row0, int i, int col, int lane) {
  return reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) +
                                   static_cast<int64_t>(row0 + i * 4 + (lane >> 3)) * p.ld_out + col + (lane & 7) * 4);
}
__device__ __forceinline__ void load_residual(const GemmParams& p, int row0, int col, int lane, float4 (&res)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    res[i] = row0 + i * 4 + (lane >> 3) < p.M ? *residual_at(p, row0, i, col, lane) : make_float4(0.f, 0.f, 0.f, 0.f);
}

__device__ __forceinline__ uint2 load_gain(const GemmParams& p, int col, int lane) {
  return p.xn_out ? __ldg(reinterpret_cast<const uint2*>(p.xn_gain + col + (lane & 7) * 4)) : make_uint2(0u, 0u);
}

template <int EPI, int BNT>
__device__ __forceinline__ void epilogue_prefetch(const GemmParams& p, int row0, int nb, int part, int lane,
                                                  EpiPre& pre) {
  if constexpr (EPI == EPI_RESID_ADD) {
    const int col = nb * BNT + part * (BNT / 2);
    load_residual(p, row0, col, lane, pre.res[0]);
    if (BNT > 64) load_residual(p, row0, col + 32, lane, pre.res[1]);
    pre.gain = load_gain(p, col, lane);
    pre.scale = p.xn_out ? norm_factor(p.ss_pre, p.ss_pre_parts, p, row0 + lane) : 1.f;
  } else if constexpr (EPI == EPI_STORE) {
    pre.scale = 1.f;
  } else {
    pre.scale = row_scale(p, row0 + lane);
  }
  if constexpr (EPI == EPI_QKV) {
    if (nb * BNT + (BNT == 256 ? part * 128 : 0) < p.q_cols + p.k_cols)
#pragma unroll
      for (int i = 0; i < 4; ++i) pre.pos[i] = p.tok_pos[min(row0 + i * 8 + (lane >> 2), p.M - 1)];
  }
}

// BNT: columns of the tile, 256 (k_gemm_pair) or 64 / 128 (k_gemm_few).  The arithmetic on a row
// is the same for every BNT, operation for operation.
// release(): called by the whole warp once it has read its last accumulator value.
// HALF: the MMAs took 64 rows of each CTA (gemm_half_m), so that a lane holds half the tile's columns.
template <int EPI, int BNT, bool HALF, typename Release>
__device__ __forceinline__ void epilogue_tile(const GemmParams& p, uint32_t taddr, int row0, int nb, int part,
                                              int lane, uint32_t* xs, EpiPre& pre, Release release) {
  // row0: first row of this warp; lane = row - row0 = TMEM lane
  float most = 0.f;  // the largest magnitude written as fp16 (track_range; reported once per tile)
  // this lane's row exists (rows past M hold whatever the operand buffers held there; never stored)
  const bool live = row0 + lane < p.M;
  if constexpr (EPI == EPI_STORE || EPI == EPI_QKV) {
    f16* out = reinterpret_cast<f16*>(p.out);
    const float rs = pre.scale;
    {
      static_assert(BNT == 256 || BNT == 128, "whole 128-column heads");
      constexpr bool ONE = BNT == 128;         // one head in the tile, its columns shared by the two parts
      const int hh = ONE ? 0 : part;           // this warp's 128-column head of the tile
      const int hc = nb * BNT + hh * 128;      // first output column of this head
      const int rope_cols = EPI == EPI_QKV ? p.q_cols + p.k_cols : 0;
      // `heads` (1 or 2) consecutive heads of the tile from `head0` on, frequencies f0 .. f0 + 16 steps
      auto norm_and_rotate = [&](auto heads, auto steps, int head0, int f0) {
        constexpr int HEADS = decltype(heads)::value, STEPS = decltype(steps)::value;
        const int col_begin = nb * BNT + head0 * 128;
        // The rotation runs in the transposed layout, 16 frequencies at a time: lane L owns rows
        // i*8 + L/4 and frequencies w4 .. w4+3 of the 16, so RoPE-table reads and the stores are
        // contiguous 4-lane row segments.  The (cos, sin) of the next 16 are fetched while these
        // are rotated (rows past M read the last row's entries and are not stored).
        const int w4 = (lane & 3) * 4;
        float4 c01[4], c23[4];
        auto fetch_rope = [&](int f) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4* cs = reinterpret_cast<const float4*>(p.rope + static_cast<int64_t>(pre.pos[i]) * 64 + f + w4);
            c01[i] = __ldg(cs);
            c23[i] = __ldg(cs + 1);
          }
        };
        fetch_rope(f0);
        // per-head RMSNorm of the row-scaled values: sum of squares in the row layout
        float inv_row[HEADS];
#pragma unroll
        for (int h = 0; h < HEADS; ++h) {
          float ss = 0.f;
#pragma unroll
          for (int c = 0; c < 128; c += 32) {
            uint32_t v[32];
            tmem_ld32(taddr + (head0 + h) * 128 + c, v);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j) ss += __uint_as_float(v[j]) * __uint_as_float(v[j]);
          }
          inv_row[h] = rs * rsqrtf(ss * rs * rs * (1.f / 128.f) + p.eps);
        }
#pragma unroll 1
        for (int s = 0; s < STEPS; ++s) {
          const int f = f0 + 16 * s;
#pragma unroll
          for (int h = 0; h < HEADS; ++h) {
            const int col0 = col_begin + h * 128;
            const bf16* wgt = col0 < p.q_cols ? p.q_norm : p.k_norm;
            const uint2 gw[2] = {__ldg(reinterpret_cast<const uint2*>(wgt + f + w4)),
                                 __ldg(reinterpret_cast<const uint2*>(wgt + 64 + f + w4))};
            uint32_t v[32];  // the row's 16 elements of the first half of the head, then those 64 further on
            const uint32_t at = taddr + (head0 + h) * 128 + f;
            tmem_ld16x2(at, at + 64, v);
            tmem_ld_wait();
            if (s + 1 == STEPS && h + 1 == HEADS) release();
            xs_put_row(xs, lane, v);
            __syncwarp();
            float g1[4], g2[4];
            bf16x4_floats(gw[0], g1);
            bf16x4_floats(gw[1], g2);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int r = i * 8 + (lane >> 2);
              const float inv = __shfl_sync(0xffffffffu, inv_row[h], r);
              const float4 x1 = xs_get(xs, r, lane & 3), x2 = xs_get(xs, r, 4 + (lane & 3));
              const float cosv[4] = {c01[i].x, c01[i].z, c23[i].x, c23[i].z};
              const float sinv[4] = {c01[i].y, c01[i].w, c23[i].y, c23[i].w};
              const float a[4] = {x1.x, x1.y, x1.z, x1.w}, b[4] = {x2.x, x2.y, x2.z, x2.w};
              float y1[4], y2[4];
              float row_most = 0.f;
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const float u = a[k] * inv * g1[k], w = b[k] * inv * g2[k];
                y1[k] = u * cosv[k] - w * sinv[k];
                y2[k] = w * cosv[k] + u * sinv[k];
                track_range(row_most, y1[k]);
                track_range(row_most, y2[k]);
              }
              if (row0 + r < p.M) track_range(most, row_most);
              if (row0 + r < p.M) {
                f16* orow = out + static_cast<int64_t>(row0 + r) * p.ld_out + col0 + f + w4;
                *reinterpret_cast<uint2*>(orow) = make_uint2(pack_f16x2(y1[0], y1[1]), pack_f16x2(y1[2], y1[3]));
                *reinterpret_cast<uint2*>(orow + 64) = make_uint2(pack_f16x2(y2[0], y2[1]), pack_f16x2(y2[2], y2[3]));
              }
            }
            if (s + 1 < STEPS && h + 1 == HEADS) fetch_rope(f + 16);
            __syncwarp();
          }
        }
      };
      using std::integral_constant;
      if (EPI == EPI_QKV && ONE && hc < rope_cols) {
        norm_and_rotate(integral_constant<int, 1>{}, integral_constant<int, 2>{}, 0, part * 32);
      } else if (EPI == EPI_QKV && !ONE && nb * BNT + 128 < rope_cols) {
        // both heads rotate: the parts share the frequencies, not the heads, so that each entry of
        // the RoPE table is read once a tile: a tile's 128 KB of entries came in beside 512 KB of
        // operands at about 64 bytes a clock.  N 4,096 K 1,024 (cold cache): 4,100 rows 33.5 -> 32.9
        // us, 6,400 rows 42.8 -> 41; with no table reads at all 29.5 and 37.4
        norm_and_rotate(integral_constant<int, 2>{}, integral_constant<int, 2>{}, 0, part * 32);
      } else if (EPI == EPI_QKV && !ONE && hc < rope_cols) {
        norm_and_rotate(integral_constant<int, 1>{}, integral_constant<int, 4>{}, part, 0);
      } else {
#pragma unroll 1
        for (int c = ONE ? part * 64 : 0; c < (ONE ? part * 64 + 64 : 128); c += 64) {
          uint32_t a[32], b[32], o[32];
          tmem_ld32(taddr + hh * 128 + c, a);
          tmem_ld32(taddr + hh * 128 + c + 32, b);
          tmem_ld_wait();
          if (c + 64 == (ONE ? part * 64 + 64 : 128)) release();
          float row_most = 0.f;
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float a0 = __uint_as_float(a[j]) * rs, a1 = __uint_as_float(a[j + 1]) * rs;
            const float b0 = __uint_as_float(b[j]) * rs, b1 = __uint_as_float(b[j + 1]) * rs;
            track_range(row_most, a0);
            track_range(row_most, a1);
            track_range(row_most, b0);
            track_range(row_most, b1);
            o[j / 2] = pack_f16x2(a0, a1);
            o[16 + j / 2] = pack_f16x2(b0, b1);
          }
          if (live) track_range(most, row_most);
          xs_put_row(xs, lane, o);
          __syncwarp();
          store_words_transposed<32>(xs, lane, row0, p.M, [&](int r, int wd) {
            return out + static_cast<int64_t>(row0 + r) * p.ld_out + hc + c + 2 * wd;
          });
          __syncwarp();
        }
      }
    }
  } else if constexpr (EPI == EPI_RESID_ADD) {
    // r += C, then (optionally) the next RMSNorm's operand f16(r * g * rs_pre) and partial sums of r^2.
    // Lane L owns rows i*4 + L/8 (i = 0..7) and columns (L%8)*4..+3 of each 32-column chunk.  The
    // residual values are fetched two chunks ahead (the first two before the main loop ends):
    // one ahead, a chunk took their latency, 2,200 clocks.
    const int w4 = (lane & 7) * 4;
    // this lane's chunk of row i*4 + lane/8 lies at cpos ^ 2 (i & 1) of the transpose buffer's row
    const int cpos = (lane & 7) ^ ((lane >> 3 & 1) << 2 | lane >> 4);
    uint32_t* xrow = xs + (lane >> 3) * 32;
    float ss[8], prev[8];
    // each lane fetched its own row's previous norm factor; the row layout below takes them by shuffle
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      ss[i] = 0.f;
      prev[i] = __shfl_sync(0xffffffffu, pre.scale, i * 4 + (lane >> 3));
    }
    constexpr int CHUNKS = BNT / 64;  // 32-column chunks of this warp's half of the columns
#pragma unroll
    for (int q = 0; q < CHUNKS; ++q) {
      const int c = part * (BNT / 2) + 32 * q;
      float4(&res)[8] = pre.res[q & 1];
      uint32_t v[32];
      tmem_ld32(taddr + c, v);
      tmem_ld_wait();
      if (q + 1 == CHUNKS) release();
      xs_put_row(xs, lane, v);
      __syncwarp();
      const int col = nb * BNT + c + w4;
      if (BNT < 256) {  // a chunk's sums stand alone here
#pragma unroll
        for (int i = 0; i < 8; ++i) ss[i] = 0.f;
      }
      float g[4];
      bf16x4_floats(pre.gain, g);
      if (q + 1 < CHUNKS) pre.gain = load_gain(p, nb * BNT + c + 32, lane);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = i * 4 + (lane >> 3);
        if (row0 + r < p.M) {
          float4 x = res[i];
          const float4 d = *reinterpret_cast<const float4*>(xrow + i * 128 + ((cpos ^ (i & 1) << 1) << 2));
          x.x += d.x;
          x.y += d.y;
          x.z += d.z;
          x.w += d.w;
          *residual_at(p, row0, i, nb * BNT + c, lane) = x;
          if (p.xn_out) {
            ss[i] += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
            const float sc = prev[i];
            const float n0 = x.x * g[0] * sc, n1 = x.y * g[1] * sc, n2 = x.z * g[2] * sc, n3 = x.w * g[3] * sc;
            track_range(most, n0);
            track_range(most, n1);
            track_range(most, n2);
            track_range(most, n3);
            uint2 o;
            o.x = pack_f16x2(n0, n1);
            o.y = pack_f16x2(n2, n3);
            *reinterpret_cast<uint2*>(p.xn_out + static_cast<int64_t>(row0 + r) * p.ld_out + col) = o;
          }
        }
      }
      if (q + 2 < CHUNKS) load_residual(p, row0, nb * BNT + c + 64, lane, res);
      __syncwarp();
      if (BNT < 256 && p.ss_out)
        publish_square_sums(p, row0, lane, (nb * BNT + c) / 128, (nb * BNT + c) / 32 % 4, ss);
    }
    if (BNT == 256 && p.ss_out) store_square_sums(p, row0, lane, nb * GEMM_SS_PER_TILE + part, ss);
  } else {  // EPI_SWIGLU: the tile's first half of the columns gate, its second half up of the same outputs
    f16* out = reinterpret_cast<f16*>(p.out);
    const float rs = pre.scale;
    constexpr int OUTS = BNT / 2;   // outputs of the tile
    constexpr int MINE = OUTS / 2;  // of this warp
    static_assert(BNT >= 128, "two chunks of 32 outputs or more");
    const int c = part * MINE;
#pragma unroll
    for (int half = 0; half < MINE / 32; ++half) {
      uint32_t g[32], u[32];
      tmem_ld32(taddr + c + 32 * half, g);
      tmem_ld32(taddr + (HALF ? MINE : OUTS) + c + 32 * half, u);
      tmem_ld_wait();
      if (half + 1 == MINE / 32) release();
      float row_most = 0.f;
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {  // eight outputs: one 16-byte chunk
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int j = c4 * 8 + 2 * k;
          const float a0 = silu_f(__uint_as_float(g[j]) * rs) * (__uint_as_float(u[j]) * rs);
          const float a1 = silu_f(__uint_as_float(g[j + 1]) * rs) * (__uint_as_float(u[j + 1]) * rs);
          track_range(row_most, a0);
          track_range(row_most, a1);
          o[k] = pack_f16x2(a0, a1);
        }
        *xs_chunk(xs, lane, 4 * half + c4) = make_uint4(o[0], o[1], o[2], o[3]);
      }
      if (live) track_range(most, row_most);
    }
    __syncwarp();
    store_words_transposed<MINE / 2>(xs, lane, row0, p.M, [&](int r, int wd) {
      return out + static_cast<int64_t>(row0 + r) * p.ld_out + nb * OUTS + c + 2 * wd;
    });
    __syncwarp();
  }
  report_range(p.err, !fp16_ok(most));
}

// ============================================================================
// The pair kernel.  Barriers:
//   full[s]   leader's: armed by the leader for both CTAs' bytes; both CTAs' copies
//             complete on it (the peer addresses it through the cluster window);
//   empty[s]  each CTA's: the leader's commit arrives on both (multicast);
//   tfull[a]  each CTA's: the leader's commit at the end of a tile, multicast;
//   tempty[a] leader's: all 16 epilogue warps of the pair arrive when TMEM is read.
constexpr int PAIR_BM = 2 * BM;                 // rows of a pair tile
constexpr int PAIR_STAGES = 6;
constexpr int PAIR_B_BYTES = BM * BK * 2;       // this CTA's 128 of the tile's 256 B rows: 16 KiB
constexpr int PAIR_STAGE_BYTES = A_BYTES + PAIR_B_BYTES;
constexpr int PAIR_SMEM_BYTES = 1024 + PAIR_STAGES * PAIR_STAGE_BYTES + XPOSE_BYTES + BAR_BYTES;
// L2 tile groups.  A 256-row block of A and a 256-row block of B hold the same bytes
// (256 K 2); a group holds as many blocks as fit GROUP_BYTES (row groups at most 16).
// Row groups keep blocks of A in L2 while B streams past (once per group); column
// groups keep blocks of B while A streams.  Measured DRAM reads per 26,800-row launch
// (row / column groups): QKV 0.76 / 0.78 GB, O 1.31 / 1.07, gate/up 1.95 / 2.74, down
// 3.93 / 3.12: the launches whose epilogue streams the fp32 residual (O, down) keep
// their weight columns better, the others their activation rows.
constexpr int64_t GROUP_BYTES = 48ll << 20;
struct TileOrder {
  int group;   // blocks per group
  bool by_n;   // column groups
};
__device__ __forceinline__ TileOrder pair_tile_order(int n_tiles, int K, bool by_n) {
  const int64_t g = GROUP_BYTES / (static_cast<int64_t>(K) * 2 * 2 * BM);
  const int64_t cap = by_n ? n_tiles : 16;
  return TileOrder{g < 1 ? 1 : g > cap ? static_cast<int>(cap) : static_cast<int>(g), by_n};
}
constexpr uint32_t PAIR_IDESC = umma_idesc_f16(PAIR_BM, BN);
// TMEM columns a pair CTA allocates, and accumulators (256 columns each) it cycles through
constexpr int PAIR_ACCS = 2;
constexpr uint32_t PAIR_TMEM_COLS = PAIR_ACCS * BN;
static_assert(PAIR_SMEM_BYTES <= 227 * 1024, "shared memory budget");

// Tile t of the launch: within a group the grouped operand's blocks vary fastest, so the
// tiles of one wave share the streamed operand's blocks too.
__device__ __forceinline__ void pair_tile_coords(int t, int m_tiles, int n_tiles, TileOrder o, int& mb, int& nb) {
  if (o.by_n) {
    const int group = o.group * m_tiles;
    const int g = t / group;
    const int first_n = g * o.group;
    const int gn = min(o.group, n_tiles - first_n);
    const int r = t - g * group;
    nb = first_n + r % gn;
    mb = r / gn;
  } else {
    const int group = o.group * n_tiles;
    const int g = t / group;
    const int first_m = g * o.group;
    const int gm = min(o.group, m_tiles - first_m);
    const int r = t - g * group;
    mb = first_m + r % gm;
    nb = r / gm;
  }
}

// A bounded wait of the whole warp: all lanes go on or give up together.
__device__ __forceinline__ bool wait_all_lanes(uint32_t bar, uint32_t parity, const GemmParams& p) {
  return __all_sync(0xffffffffu, mbar_wait_cluster(bar, parity, p.err, p.timeout_ns)) != 0;
}
// An epilogue warp has read its part of an accumulator: tell the leader.
__device__ __forceinline__ void free_accumulator(uint32_t tempty_bar, int lane) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive_cluster(mapa_shared(tempty_bar, 0));
}
// A producer that gave up: its copies in flight land within microseconds; give them that long
// before the CTA can reach its exit (no barrier to wait on: they count on the leader's).
__device__ __forceinline__ void let_copies_land() {
  const uint64_t t0 = globaltimer_ns();
  while (globaltimer_ns() - t0 < 20000ull) {
  }
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    k_gemm_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sA = smem_u32(smem);
  const uint32_t sB = sA + PAIR_STAGES * A_BYTES;
  uint32_t* xpose = reinterpret_cast<uint32_t*>(smem + PAIR_STAGES * PAIR_STAGE_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + PAIR_STAGES * PAIR_STAGE_BYTES + XPOSE_BYTES);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (PAIR_STAGES + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * PAIR_STAGES + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * PAIR_STAGES + 2 + a); };
  const uint32_t drain_bar = bar0 + 8u * (2 * PAIR_STAGES + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * PAIR_STAGES + 5);
  static_assert((2 * PAIR_STAGES + 5) * 8 + 4 <= BAR_BYTES, "barrier area");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int m_tiles = (p.M + PAIR_BM - 1) / PAIR_BM, n_tiles = p.N / BN, k_blocks = p.K / BK;
  const TileOrder order = pair_tile_order(n_tiles, p.K, EPI == EPI_RESID_ADD);
  int total = m_tiles * n_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PAIR_STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), 2 * EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), PAIR_TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before either addresses the other's
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // in this order: a few-row launch beside this one (GemmParams::beside) starts once this kernel's
  // blocks have triggered, and the gate hands it what this kernel waited for
  pdl_wait();
  if (p.gate && blockIdx.x == 0 && threadIdx.x == THREADS - 32) gate_open(p.gate, p.gate_number);  // an epilogue warp's
  pdl_trigger();
  {
    // the MMAs write both CTAs' TMEM at the leader's address: both allocations must agree
    uint32_t other;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(other) : "r"(mapa_shared(smem_u32(tmem_slot), rank ^ 1u)));
    if (other != tmem_base) {
      if (threadIdx.x == 0) atomicOr(p.err, DEV_ERR_BOUNDS);
      total = 0;  // no tile runs
    }
  }

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs): own A rows and own half of B's rows.  Here and
    // in the issuer the whole warp runs the loop and one lane issues: with the loop's state
    // warp-uniform an MMA or a copy costs its thread far fewer instructions (in a loop of one
    // diverged lane an MMA took about 78 clocks to issue).  16,000 rows: N 4,096 K 12,288
    // 993 -> 967 us, N 6,144 K 4,096 453 -> 443; 4,100 rows, gate/up N 6,144 K 1,024 44.2 -> 40.5.
    const bool one = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      int mb, nb;
      pair_tile_coords(t, m_tiles, n_tiles, order, mb, nb);
      for (int kb = 0; kb < k_blocks; ++kb) {
        ok = wait_all_lanes(empty_bar(stage), phase ^ 1u, p);
        if (!ok) break;
        if (one) {
          if (leader) mbar_arrive_expect_tx(full_bar(stage), 2 * PAIR_STAGE_BYTES);
          const uint32_t fb = mapa_shared(full_bar(stage), 0);
          tma_load_2d_pair(sA + stage * A_BYTES, &tmA, fb, kb * BK, mb * PAIR_BM + static_cast<int>(rank) * BM);
          tma_load_2d_pair(sB + stage * PAIR_B_BYTES, &tmB, fb, kb * BK, nb * BN + static_cast<int>(rank) * BM);
        }
        if (++stage == PAIR_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) let_copies_land();
  } else if (warp == 1) {
    if (leader) {
      // ---------------- MMA issuer (leader only)
      const bool one = elect_one();
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int t = pair; t < total && ok; t += n_pairs, ++local) {
        const int acc = local % PAIR_ACCS;
        ok = wait_all_lanes(tempty_bar(acc), ((local / PAIR_ACCS) & 1) ^ 1u, p);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        for (int kb = 0; kb < k_blocks; ++kb) {
          ok = wait_all_lanes(full_bar(stage), phase, p);
          if (!ok) break;
          tc_fence_after();
          if (one) {
            const uint64_t ad = umma_desc_sw128(sA + stage * A_BYTES);
            const uint64_t bd = umma_desc_sw128(sB + stage * PAIR_B_BYTES);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)  // +32 bytes along K per step, in 16-byte units
              umma_f16_pair(d_tmem, ad + 2 * k, bd + 2 * k, PAIR_IDESC, (kb | k) != 0);
            umma_commit_pair_mc(empty_bar(stage), 3);  // both CTAs' stage is free once these MMAs end
          }
          if (++stage == PAIR_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok && one) umma_commit_pair_mc(tfull_bar(acc), 3);
      }
      // All MMAs this thread issued are complete once drain_bar flips.
      if (one) umma_commit_pair_mc(drain_bar, 1);
      mbar_wait_warp(drain_bar, 0, p.err, ok ? p.timeout_ns : 100000000ull);
    }
  } else {
    // ---------------- epilogue warps 2..9 (both CTAs) on this CTA's 128 rows of the tile
    const int quarter = warp & 3;
    const int part = (warp - 2) >> 2;
    uint32_t* xs = xpose + (warp - 2) * XPOSE_WORDS;
    int local = 0;
    for (int t = pair; t < total; t += n_pairs, ++local) {
      int mb2, nb;
      pair_tile_coords(t, m_tiles, n_tiles, order, mb2, nb);
      const int row0 = (2 * mb2 + static_cast<int>(rank)) * BM + quarter * 32;  // in this CTA's 128-row block
      const int acc = local % PAIR_ACCS;
      const uint32_t acc_phase = (local / PAIR_ACCS) & 1;
      EpiPre pre;
      epilogue_prefetch<EPI, BN>(p, row0, nb, part, lane, pre);
      if (!wait_all_lanes(tfull_bar(acc), acc_phase, p)) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN;
      epilogue_tile<EPI, BN, false>(p, taddr, row0, nb, part, lane, xs, pre, [&] { free_accumulator(tempty_bar(acc), lane); });
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other may still address its barriers or TMEM
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc_pair(tmem_base, PAIR_TMEM_COLS);
  }
}

// ============================================================================
// Few rows (the last layer's score rows, small batches): the pair kernel with narrower tiles,
// 64 or 128 columns, and R = 32, 64, 96 or 128 A rows per CTA instead of 128.
//
// With few rows a launch is bound by streaming the weights, and 256-column tiles leave most
// SMs without a tile (O and down of the 8B shape: 16 tiles on 32 of 152 SMs) while each SM
// takes in operand bytes at no more than about 64 bytes a clock, of which half or more were A
// rows that hold nothing.  Narrow tiles put 2 or 4 times as many SMs to work, and a CTA copies only
// its R rows (the MMAs run 128 rows a CTA, or 64 where SHORT below holds; what they read past the R
// rows is other shared memory, in tile rows that are never stored).  A stage is KB 64-wide k-blocks,
// so that each operand is one copy of at least 8 KB a stage (a 3-D map: 64 elements, rows, k-blocks;
// gate and up rows together a 5-D one).
// The K order of a row's MMAs is the wide tiles', so its result is the same bit for bit.
constexpr int FEW_RING = 192 * 1024;
constexpr int FEW_MAX_STAGES = 12;
constexpr int FEW_SMEM_BYTES = 1024 + FEW_RING + XPOSE_BYTES + BAR_BYTES;
static_assert(FEW_SMEM_BYTES <= 227 * 1024, "shared memory budget");
static_assert((2 * FEW_MAX_STAGES + 5) * 8 + 4 <= BAR_BYTES, "barrier area");
// The B stages follow the A stages, so the 128 rows that an MMA reads from the start of the last
// R-row A block (up to 12 KB past it) lie inside the ring.

template <int EPI, int BNT, int R>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    k_gemm_few(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmParams p) {
  constexpr int KB = GEMM_FEW_KB(R);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int a_blk = R * BK * 2, b_blk = BNT / 2 * BK * 2;  // one k-block of this CTA's A rows, of its B rows
  constexpr int stage_bytes = KB * (a_blk + b_blk);
  constexpr int stages = FEW_RING / stage_bytes < FEW_MAX_STAGES ? FEW_RING / stage_bytes : FEW_MAX_STAGES;
  const uint32_t sA = smem_u32(smem);
  const uint32_t sB = sA + stages * KB * a_blk;
  uint32_t* xpose = reinterpret_cast<uint32_t*>(smem + FEW_RING);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + FEW_RING + XPOSE_BYTES);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (FEW_MAX_STAGES + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * FEW_MAX_STAGES + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * FEW_MAX_STAGES + 2 + a); };
  const uint32_t drain_bar = bar0 + 8u * (2 * FEW_MAX_STAGES + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * FEW_MAX_STAGES + 5);
  constexpr uint32_t TMEM_COLS = PAIR_ACCS * BNT;
  // With at most 64 rows a CTA the residual and gate/up launches take M = 128 MMAs, 64 rows a CTA:
  // each reads half as much of A (48 -> 32 clocks of shared memory at 64 columns).  A CTA's rows are
  // then TMEM lanes 0..63 for the tile's first half of the columns and 64..127 for its second; for
  // gate and up of an output to share a lane, each CTA stages 32 gate rows and their 32 up rows.
  // Cold cache, 25 rows: gate/up N 24,576 K 4,096 (201 MB of weights, 29.7 us at the copy's rate)
  // 40.3 -> 36.3 us.
  constexpr bool SHORT = gemm_half_m(EPI, R, BNT);
  constexpr bool MIXED = SHORT && EPI == EPI_SWIGLU;
  constexpr uint32_t IDESC = umma_idesc_f16(SHORT ? BM : PAIR_BM, BNT);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int m_tiles = (p.M - p.row_begin + 2 * R - 1) / (2 * R);
  const int k_blocks = p.K / BK, k_steps = (k_blocks + KB - 1) / KB;
  int total = m_tiles * (p.N / BNT);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), 2 * EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish_pair();
  }
  // during the set-up, which hides the acquire's latency
  const bool gate_passed = !p.beside || gate_wait_warp(p.gate, p.gate_number, p.err, p.timeout_ns);
  if (p.beside) fence_proxy_async_global();
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before either addresses the other's
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_trigger();
  // (the producer starts on the weights first; beside the wide launch of the same product the gate
  // stands for this wait)
  if (warp != 0 && !p.beside) pdl_wait();
  if (!gate_passed) total = 0;  // gave up: no tile runs
  {
    uint32_t other;  // as in k_gemm_pair: both allocations must agree
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(other) : "r"(mapa_shared(smem_u32(tmem_slot), rank ^ 1u)));
    if (other != tmem_base) {
      if (threadIdx.x == 0) atomicOr(p.err, DEV_ERR_BOUNDS);
      total = 0;  // no tile runs
    }
  }

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs): own A rows and own half of B's rows
    const bool one = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    // SwiGLU weights hold gate and up in alternating blocks of 128 rows: rank 0 takes gate rows, rank 1 up rows
    auto weight_row = [&](int nb) {
      const int o = nb * (BNT / 2);
      if constexpr (MIXED) return o + static_cast<int>(rank) * 32;
      return EPI == EPI_SWIGLU ? (o / 128) * 256 + o % 128 + static_cast<int>(rank) * 128
                               : nb * BNT + static_cast<int>(rank) * (BNT / 2);
    };
    auto load_weights = [&](int s, int brow, int ks) {  // k-blocks past K are filled with zeros and count as copied
      if (leader) mbar_arrive_expect_tx(full_bar(s), 2 * stage_bytes);
      if constexpr (MIXED)  // brow: the CTA's first output
        tma_load_5d_pair(sB + s * KB * b_blk, &tmB, mapa_shared(full_bar(s), 0), 0, brow % 128, 0, brow / 128, ks * KB);
      else
        tma_load_3d_pair(sB + s * KB * b_blk, &tmB, mapa_shared(full_bar(s), 0), 0, brow, ks * KB);
    };
    // the first stages' weights, which no kernel writes, go out while the kernel before still runs
    int ahead = 0;
    if (pair < total)
      for (; ahead < min(stages, k_steps); ++ahead)
        if (one) load_weights(ahead, weight_row(pair / m_tiles), ahead);
    if (!p.beside) pdl_wait();
    for (int t = pair; t < total && ok; t += n_pairs) {
      const int nb = t / m_tiles, row = p.row_begin + (t % m_tiles) * 2 * R + static_cast<int>(rank) * R;
      const int brow = weight_row(nb);
      for (int ks = 0; ks < k_steps; ++ks) {
        ok = wait_all_lanes(empty_bar(stage), phase ^ 1u, p);
        if (!ok) break;
        if (one) {
          if (ahead == 0) load_weights(stage, brow, ks);
          tma_load_3d_pair(sA + stage * KB * a_blk, &tmA, mapa_shared(full_bar(stage), 0), 0, row, ks * KB);
        }
        if (ahead > 0) --ahead;
        if (++stage == stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) let_copies_land();
  } else if (warp == 1) {
    if (leader) {
      // ---------------- MMA issuer (leader only): the whole warp runs the loop, so that its state
      // and the operand descriptors stay warp-uniform; one lane issues
      const bool one = elect_one();
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int t = pair; t < total && ok; t += n_pairs, ++local) {
        const int acc = local % PAIR_ACCS;
        ok = wait_all_lanes(tempty_bar(acc), ((local / PAIR_ACCS) & 1) ^ 1u, p);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BNT;
        for (int ks = 0; ks < k_steps; ++ks) {
          ok = wait_all_lanes(full_bar(stage), phase, p);
          if (!ok) break;
          tc_fence_after();
          if (one) {
            const uint64_t ad = umma_desc_sw128(sA + stage * KB * a_blk);
            const uint64_t bd = umma_desc_sw128(sB + stage * KB * b_blk);
            const int left = k_blocks - ks * KB;
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
              if (kb < left) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                  umma_f16_pair(d_tmem, ad + (kb * (a_blk / 16) + 2 * k), bd + (kb * (b_blk / 16) + 2 * k), IDESC,
                                (ks | kb | k) != 0);
              }
            umma_commit_pair_mc(empty_bar(stage), 3);  // both CTAs' stage is free once these MMAs end
          }
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok && one) umma_commit_pair_mc(tfull_bar(acc), 3);
      }
      if (one) umma_commit_pair_mc(drain_bar, 1);
      mbar_wait_warp(drain_bar, 0, p.err, ok ? p.timeout_ns : 100000000ull);
    }
  } else {
    // ---------------- epilogue warps 2..9 (both CTAs) on this CTA's R rows of the tile
    const int quarter = warp & 3;
    const int part = (warp - 2) >> 2;
    uint32_t* xs = xpose + (warp - 2) * XPOSE_WORDS;
    int local = 0;
    for (int t = pair; t < total; t += n_pairs, ++local) {
      const int block = SHORT ? quarter & 1 : quarter;   // the 32 rows of this lane quarter,
      const int cols = SHORT ? quarter >> 1 : part;      // and this warp's half of the columns
      const int nb = t / m_tiles;
      const int row0 = p.row_begin + (t % m_tiles) * 2 * R + static_cast<int>(rank) * R + block * 32;
      // a warp with rows of the tile (R is a multiple of 32)
      const bool mine = block * 32 < R && row0 < p.M && !(SHORT && part != 0);
      const int acc = local % PAIR_ACCS;
      EpiPre pre;
      if (mine) epilogue_prefetch<EPI, BNT>(p, row0, nb, cols, lane, pre);
      if (!wait_all_lanes(tfull_bar(acc), (local / PAIR_ACCS) & 1, p)) break;
      tc_fence_after();
      // (epilogue_tile adds the half's first column, which here is a lane offset)
      const uint32_t taddr =
          tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BNT - (SHORT ? cols * 32 : 0);
      if (mine)
        epilogue_tile<EPI, BNT, SHORT>(p, taddr, row0, nb, cols, lane, xs, pre, [&] { free_accumulator(tempty_bar(acc), lane); });
      else
        free_accumulator(tempty_bar(acc), lane);
    }
  }

  if (p.beside) pdl_wait();  // completion carries over: the next kernel waits for this one only
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other may still address its barriers or TMEM
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
}

// f(kernel) for the few-rows kernel of a plan.
template <int EPI, typename F>
auto few_kernel(int rows, int cols, F&& f) {
  if constexpr (EPI == EPI_RESID_ADD)
    if (cols == 64)
      return rows == 32   ? f(k_gemm_few<EPI, 64, 32>)
             : rows == 64 ? f(k_gemm_few<EPI, 64, 64>)
                          : f(k_gemm_few<EPI, 64, 96>);
  return rows == 32   ? f(k_gemm_few<EPI, 128, 32>)
         : rows == 64 ? f(k_gemm_few<EPI, 128, 64>)
         : rows == 96 ? f(k_gemm_few<EPI, 128, 96>)
                      : f(k_gemm_few<EPI, 128, 128>);
}

template <int EPI>
cudaError_t set_smem() {
  cudaError_t e = cudaFuncSetAttribute(k_gemm_pair<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, PAIR_SMEM_BYTES);
  for (int rows = 32; rows <= BM; rows += 32)
    for (int cols = 64; cols <= 128; cols *= 2)
      if (e == cudaSuccess)
        e = few_kernel<EPI>(rows, cols, [](auto* k) {
          return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, FEW_SMEM_BYTES);
        });
  return e;
}

template <int EPI>
cudaError_t launch_epi(const GemmOperandA& A, const GemmOperandB& B, const GemmParams& p, const GemmPlan& g, int num_sms,
                cudaStream_t st) {
  const int tiles = ((p.M - p.row_begin + 2 * g.rows - 1) / (2 * g.rows)) * (p.N / g.cols);
  const int grid = 2 * (tiles < num_sms / 2 ? tiles : num_sms / 2 > 0 ? num_sms / 2 : 1);
  if (!g.few) {
    return launch_dependent(k_gemm_pair<EPI>, grid, THREADS, PAIR_SMEM_BYTES, st, A.wide, B.wide, p);
  }
  const CUtensorMap& ta = A.few[g.rows / 32 - 1];
  const int four = GEMM_FEW_KB(g.rows) == 4;
  const CUtensorMap& tb =
      EPI == EPI_SWIGLU && gemm_half_m(EPI, g.rows, g.cols) ? B.gate_up[four] : B.few[g.cols == 128][four];
  return few_kernel<EPI>(g.rows, g.cols,
                         [&](auto* k) { return launch_dependent(k, grid, THREADS, FEW_SMEM_BYTES, st, ta, tb, p); });
}

}  // namespace

cudaError_t gemm_setup() {
  cudaError_t e;
  if ((e = set_smem<EPI_STORE>())) return e;
  if ((e = set_smem<EPI_RESID_ADD>())) return e;
  if ((e = set_smem<EPI_SWIGLU>())) return e;
  return set_smem<EPI_QKV>();
}

// The clocks a CTA pair needs for a 64-wide k-block of a tile of 2 R rows and n columns: its SMs
// take in R + n / 2 operand rows of 128 bytes at about 64 bytes a clock, and the four MMAs take
// 512 at n = 256 but 288 at 128 and 192 at 64 (each reads 128 A rows a CTA, whatever R is; 64-row
// MMAs, gemm_half_m, 128 at 64 columns and 192 at 128).
// Every tile adds a start and an epilogue that is not hidden, about 2,000 clocks.  The tile
// with the least clocks over the launch's rounds is taken, the wide one of two equal ones.
// Measured (cold cache, wide / taken): N 4,096 K 12,288, 25 rows 63.7 / 26 us, 180 rows
// 66.0 / 37 us; N 4,096 K 4,096, 25 rows 28.0 / 13 us; gate/up N 24,576 K 4,096, 25 rows
// 59.0 / 36 us, 180 rows (estimates 3 % apart) 50.1 / 46.4 us.
namespace {
int64_t block_clocks(int epi, int R, int n) {
  const int64_t in = 2 * (R + n / 2), mma = n == BN ? 2 * BN : gemm_half_m(epi, R, n) ? 64 + n : 96 + 3 * n / 2;
  return in > mma ? in : mma;
}
int64_t rounds(int M, int N, int R, int n, int64_t pairs) {
  return (static_cast<int64_t>((M + 2 * R - 1) / (2 * R)) * (N / n) + pairs - 1) / pairs;
}
// The few-row plan of M <= GEMM_FEW_MAX_ROWS rows with the least clocks, if below `least` (which is updated).
bool few_plan(int epi, int M, int N, int K, int64_t pairs, int64_t tile_clocks, int64_t& least, GemmPlan& plan) {
  bool found = false;
  // 64 columns for the residual launches alone, and of at most 96 rows a CTA: gate/up tiles of 128
  // columns take no more clocks than any of 64 that has as many rounds (64-row MMAs up to 64 rows,
  // the same operand bytes as 64 x 128 or 96 x 128 beyond), and 128 x 64 no fewer than 96 x 128
  const int cols[2] = {128, 64};
  for (int n : cols) {
    if (N % n || (n == 64 && epi != EPI_RESID_ADD)) continue;
    for (int R = 32; R <= (n == 64 ? 96 : BM); R += 32) {
      const int64_t c = rounds(M, N, R, n, pairs) * (K / BK * block_clocks(epi, R, n) + tile_clocks);
      if (c < least) {
        least = c;
        plan = GemmPlan{true, R, n, 0};
        found = true;
      }
    }
  }
  return found;
}
}  // namespace

GemmPlan gemm_plan(int epi, int M, int N, int K, int num_sms) {
  const int64_t pairs = num_sms / 2 > 0 ? num_sms / 2 : 1;
  GemmPlan best{false, BM, BN, 0};
  const int64_t wide = rounds(M, N, BM, BN, pairs);
  if (M <= GEMM_FEW_MAX_ROWS) {
    int64_t least = wide * (K / BK * block_clocks(epi, BM, BN) + 2000);
    few_plan(epi, M, N, K, pairs, 2000, least, best);
    if (best.few) return best;
  }
  // A last round that few tiles share: where the rows beyond the rounds before it make a single
  // round of narrow tiles, they go to a few-row launch beside the wide one.  It has a start and an
  // end of its own, about 6,000 clocks.  N 4,096, K 12,288: 3,800 rows are 240 tiles, 3.2 rounds of
  // 76 pairs, of which 3,584 rows are 2.95 and the other 216 go beside them: 3 rounds instead of 4.
  // Against the same library without it, whole calls: prefix build and scoring (8B width) 2,134 ->
  // 2,114 us, selection of long documents (4B width, 5,650 rows a product) 2,186 -> 2,136,
  // uncompressed scoring 2,665 either way; the call of these 3,800 rows, under the power cap
  // throughout, 3,145 -> 3,164.
  int64_t least = wide * (K / BK) * 2 * BN * 98 / 100;
  const int m_tiles = (M + PAIR_BM - 1) / PAIR_BM;
  for (int mt = m_tiles - 1; mt > 0 && M - mt * PAIR_BM <= GEMM_FEW_MAX_ROWS; --mt) {
    const int rest = M - mt * PAIR_BM;
    const int64_t base = rounds(mt * PAIR_BM, N, BM, BN, pairs) * (K / BK) * 2 * BN + 6000;
    int64_t few = least - base;
    GemmPlan p;
    if (few > 0 && few_plan(epi, rest, N, K, pairs, 0, few, p) && rounds(rest, N, p.rows, p.cols, pairs) == 1) {
      least = base + few;
      best = p;
      best.few = false;
      best.wide_rows = mt * PAIR_BM;
    }
  }
  return best;
}

static cudaError_t launch_one(int epi, const GemmOperandA& A, const GemmOperandB& B, const GemmParams& p, const GemmPlan& g,
                              int num_sms, cudaStream_t st) {
  switch (epi) {
    case EPI_STORE: return launch_epi<EPI_STORE>(A, B, p, g, num_sms, st);
    case EPI_RESID_ADD: return launch_epi<EPI_RESID_ADD>(A, B, p, g, num_sms, st);
    case EPI_SWIGLU: return launch_epi<EPI_SWIGLU>(A, B, p, g, num_sms, st);
    default: return launch_epi<EPI_QKV>(A, B, p, g, num_sms, st);
  }
}

cudaError_t launch_gemm(int epi, const GemmOperandA& A, const GemmOperandB& B, const GemmParams& params, int num_sms,
                        cudaStream_t st) {
  if (params.M <= 0) return cudaSuccess;
  GemmParams p = params;
  p.timeout_ns = WAIT_TIMEOUT_NS;
  const GemmPlan g = gemm_plan(epi, p.M, p.N, p.K, num_sms);
  if (g.wide_rows > 0) {  // the first rows wide, the rest beside them
    p.M = g.wide_rows;
    const cudaError_t e = launch_one(epi, A, B, p, GemmPlan{false, BM, BN, 0}, num_sms, st);
    if (e != cudaSuccess) return e;
    p.M = params.M;
    p.row_begin = g.wide_rows;
    p.beside = p.gate != nullptr;  // without a gate it waits for the wide launch like any other kernel
    return launch_one(epi, A, B, p, GemmPlan{true, g.rows, g.cols, 0}, num_sms, st);
  }
  p.gate = nullptr;
  return launch_one(epi, A, B, p, g, num_sms, st);
}

}  // namespace dopr
