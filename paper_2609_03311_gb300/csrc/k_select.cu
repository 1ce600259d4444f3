// k_select.cu -- attention-based key token selection (DoPR Sec. 3.2.1, applied
// offline as in Sec. 3.3): from a document-only pass, the last layer's
// attention weights averaged over the q heads (A-bar, n x n, causal), each
// token's salience u_i = the mean of the top-p entries of column i, the
// top-K positions, and their final-layer states after the final RMSNorm.
//
//   k_sal_tc<true>   per (128-row tile, q head): the softmax maximum and sum of
//                    every row (S = Q K^T on tcgen05, 128 keys a step);
//   k_sal_tc<false>  per (128-row tile, 128-column tile on or below the diagonal):
//                    S again, head after head, and the weights exp(s - max) / sum / Hq
//                    added up in registers over the heads (fp32), so A-bar is written
//                    once, transposed (column i's entries contiguous);
//   k_sal_colstat    one warp per column: the top-p mean by a radix search of the p-th
//                    largest value, the column in registers;
//   k_sal_topk       one CTA per document: the K-th largest salience by the same search.
//
// Both tensor-core kernels are bound by the softmax warps (an FMA, an ex2 and an add per
// score), not by the MMAs or memory: S is computed twice rather than kept, since 16-32
// heads of n x n scores would be 16-64 times the bytes of A-bar.  Both together, against
// one CTA per row with scalar dot products: 32 documents of 512 tokens, 16 heads, 83 us
// (4,402 before); 4 documents of 777-2,048 tokens, 32 heads, 140 us (8,751 before).
#include <float.h>
#include <math.h>

#include "device_common.cuh"
#include "internal.h"

namespace dopr {
namespace {

// ---------------------------------------------------------------- A-bar on the tensor cores
constexpr int TILE = SEL_TILE;              // rows and key columns of a score tile
constexpr int T_HALF = TILE * 128;          // 128 rows x 64 fp16, 128-byte swizzle
constexpr int T_BYTES = 2 * T_HALF;         // a Q or K tile: 32 KB
constexpr int Q_STAGES = 3, K_STAGES = 3, S_BUFS = 4;
constexpr int PARTS = 4;                    // softmax warpgroups: 32 of a tile's 128 columns each
constexpr int SOFT_WARPS = 4 * PARTS;
constexpr int TC_THREADS = 64 + 32 * SOFT_WARPS;
constexpr uint32_t TC_TMEM = S_BUFS * TILE;
constexpr int B_QF = 0, B_QE = B_QF + Q_STAGES, B_KF = B_QE + Q_STAGES, B_KE = B_KF + K_STAGES;
constexpr int B_SF = B_KE + K_STAGES, B_SE = B_SF + S_BUFS, B_RF = B_SE + S_BUFS, B_RE = B_RF + 1, B_DRAIN = B_RE + 1;
constexpr int N_BARS = B_DRAIN + 1;
static_assert(B_KF + K_STAGES <= 32, "the producer tracks the barriers it arms in one 32-bit mask");
constexpr int OFF_K = Q_STAGES * T_BYTES, OFF_RED = OFF_K + K_STAGES * T_BYTES;
constexpr int OFF_BAR = OFF_RED + PARTS * TILE * 8;
constexpr int TC_SMEM = 1024 + OFF_BAR + N_BARS * 8 + 16;
static_assert(TC_SMEM <= 227 * 1024, "shared memory budget");

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// STATS: units are (row tile, head), one step per key tile 0 .. rt; the row's maximum and
//   sum are kept online and go to stats[head][chunk row] = (max * scale, 1 / (sum * Hq)).
// Otherwise units are (row tile, column tile), one step per head; the thread's 32 columns
//   of its row are summed over the heads and written to A[column][row].
// Warp 0 copies Q and K tiles (TMA), warp 1 issues S = Q K^T into four TMEM buffers, warps
// 2..17 read them: TMEM lane quarter warp % 4 (one row per thread), columns 32 part .. + 31.
template <bool STATS>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_sal_tc(const __grid_constant__ CUtensorMap tm, const SelUnit* __restrict__ units, int n_units, int Hq, int Hkv,
             int n_rows, float2* stats, float* __restrict__ A, Extents ext) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t s0 = smem_u32(smem);
  auto bar = [&](int i) { return s0 + OFF_BAR + 8u * static_cast<uint32_t>(i); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + OFF_BAR + N_BARS * 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = Hq / Hkv;
  const int total = STATS ? n_units * Hq : n_units;
  int* err = ext.err;

  if (threadIdx.x == 0) {
    for (int i = 0; i < N_BARS; ++i)
      mbar_init(bar(i), (i >= B_SE && i < B_RF) || i == B_RF ? SOFT_WARPS : i == B_RE ? SOFT_WARPS / PARTS : 1);
    fence_mbar_init();
    tma_prefetch_desc(&tm);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), TC_TMEM);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();

  struct Ring {
    int stage = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next(int n) {
      if (++stage == n) {
        stage = 0;
        phase ^= 1u;
      }
    }
  };
  // the steps of unit w: which head and key tile, and where a step starts or ends its use of a Q or K tile
  auto steps_of = [&](const SelUnit& u) { return STATS ? u.rt + 1 : Hq; };
  auto new_q = [&](int s) { return STATS ? s == 0 : true; };
  auto new_k = [&](int s) { return STATS ? true : s % G == 0; };
  auto end_q = [&](int s, int n) { return STATS ? s == n - 1 : true; };
  auto end_k = [&](int s) { return STATS ? true : s % G == G - 1; };

  if (warp == 0) {
    {
      const bool one = elect_one();
      Ring rq, rk;
      uint32_t armed = 0, armed_par = 0;  // bit per barrier: ever armed / parity of the last arm
      auto load = [&](Ring& r, int full, int empty, uint32_t base, int col, int row) -> bool {
        if (!mbar_wait_warp(bar(empty + r.stage), r.phase ^ 1u, err, WAIT_TIMEOUT_NS)) return false;
        const int b = full + r.stage;
        if (one) mbar_arrive_expect_tx(bar(b), T_BYTES);
        armed |= 1u << b;
        armed_par = (armed_par & ~(1u << b)) | (r.phase << b);
        for (int h = 0; one && h < 2; ++h)
          tma_load_2d(base + r.stage * T_BYTES + h * T_HALF, &tm, bar(b), col + h * 64, row);
        return true;
      };
      bool ok = true;
      for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
        const SelUnit u = units[STATS ? w / Hq : w];
        if (kCheckedBuild) {  // report only: the tensor map bounds the copies itself
          index_ok(err, u.ts, ext.rows);
          index_ok(err, u.ts + u.n - 1, ext.rows);
        }
        const int n = steps_of(u);
        for (int s = 0; s < n && ok; ++s) {
          const int h = STATS ? w % Hq : s, ct = STATS ? s : u.ct;
          if (new_q(s)) ok = load(rq, B_QF, B_QE, s0, h * HEAD_DIM, u.ts + u.rt * TILE);
          if (ok && new_k(s)) ok = load(rk, B_KF, B_KE, s0 + OFF_K, (Hq + h / G) * HEAD_DIM, u.ts + ct * TILE);
          if (new_q(s)) rq.next(Q_STAGES);
          if (new_k(s)) rk.next(K_STAGES);
        }
      }
      if (!ok) {  // every copy this thread started lands before the CTA can exit
        for (int b = 0; b < 32; ++b)
          if (armed & (1u << b)) mbar_wait_warp(bar(b), (armed_par >> b) & 1u, err, 100000000ull);
      }
    }
  } else if (warp == 1) {
    {
      const bool one = elect_one();
      Ring rq, rk, rs;
      constexpr uint32_t idesc = umma_idesc_f16(TILE, TILE);
      bool ok = true;
      for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
        const SelUnit u = units[STATS ? w / Hq : w];
        const int n = steps_of(u);
        for (int s = 0; s < n && ok; ++s) {
          ok = (!new_q(s) || mbar_wait_warp(bar(B_QF + rq.stage), rq.phase, err, WAIT_TIMEOUT_NS)) &&
               (!new_k(s) || mbar_wait_warp(bar(B_KF + rk.stage), rk.phase, err, WAIT_TIMEOUT_NS)) &&
               mbar_wait_warp(bar(B_SE + rs.stage), rs.phase ^ 1u, err, WAIT_TIMEOUT_NS);
          if (!ok) break;
          tc_fence_after();
          const uint64_t qd = umma_desc_sw128(s0 + rq.stage * T_BYTES);
          const uint64_t kd = umma_desc_sw128(s0 + OFF_K + rk.stage * T_BYTES);
          if (one) {
#pragma unroll
            for (int ks = 0; ks < HEAD_DIM / 16; ++ks) {  // 16 elements = 32 bytes a step; halves 16 KB apart
              const uint64_t off = ((ks >> 2) * T_HALF + (ks & 3) * 32) / 16;
              umma_f16(tmem + rs.stage * TILE, qd + off, kd + off, idesc, ks > 0);
            }
            umma_commit(bar(B_SF + rs.stage));
          }
          rs.next(S_BUFS);
          if (end_q(s, n)) {
            if (one) umma_commit(bar(B_QE + rq.stage));
            rq.next(Q_STAGES);
          }
          if (end_k(s)) {
            if (one) umma_commit(bar(B_KE + rk.stage));
            rk.next(K_STAGES);
          }
        }
      }
      if (one) umma_commit(bar(B_DRAIN));  // every MMA this thread issued is complete once it flips
      mbar_wait_warp(bar(B_DRAIN), 0, err, ok ? WAIT_TIMEOUT_NS : 100000000ull);
    }
  } else {
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int r = quarter * 32 + lane;  // row of the tile
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + part * 32;
    const float scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(HEAD_DIM));
    float2* red = reinterpret_cast<float2*>(smem + OFF_RED);
    Ring rs;
    uint32_t unit_par = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < total && ok; w += gridDim.x, unit_par ^= 1u) {
      const SelUnit u = units[STATS ? w / Hq : w];
      const int n = steps_of(u);
      const int pos = u.rt * TILE + r;  // this row's position in its document
      // the row's statistics of the next head are fetched a step ahead
      auto stat_at = [&](int h) {
        return !STATS && pos < u.n ? stats[static_cast<int64_t>(h) * n_rows + u.ts + pos] : make_float2(0.f, 0.f);
      };
      float mx = -INFINITY, sum = 0.f;  // STATS
      float acc[32];                    // !STATS
      float2 st = make_float2(0.f, 0.f);
      if (!STATS) {
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = 0.f;
        st = stat_at(0);
      }
      for (int s = 0; s < n; ++s) {
        const int ct = STATS ? s : u.ct;
        const int nvis = pos - (ct * TILE + part * 32) + 1;  // visible columns among this thread's 32, if in 1..31
        const float2 nst = !STATS && s + 1 < n ? stat_at(s + 1) : st;
        if (!mbar_wait_warp(bar(B_SF + rs.stage), rs.phase, err, WAIT_TIMEOUT_NS)) {
          ok = false;
          break;
        }
        tc_fence_after();
        uint32_t v[32];
        tmem_ld32(trow + rs.stage * TILE, v);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_SE + rs.stage));
        rs.next(S_BUFS);
        if constexpr (STATS) {
          if (nvis > 0) {
            float t[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
              t[i] = fmaxf(2 * i < nvis ? __uint_as_float(v[2 * i]) : -INFINITY,
                           2 * i + 1 < nvis ? __uint_as_float(v[2 * i + 1]) : -INFINITY);
#pragma unroll
            for (int k = 8; k >= 1; k >>= 1)
#pragma unroll
              for (int i = 0; i < k; ++i) t[i] = fmaxf(t[2 * i], t[2 * i + 1]);
            const float m2 = fmaxf(mx, t[0] * scale_log2);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float a = ex2_approx(fmaf(__uint_as_float(v[2 * i]), scale_log2, -m2));
              const float b = ex2_approx(fmaf(__uint_as_float(v[2 * i + 1]), scale_log2, -m2));
              t[i] = (2 * i < nvis ? a : 0.f) + (2 * i + 1 < nvis ? b : 0.f);
            }
#pragma unroll
            for (int k = 8; k >= 1; k >>= 1)
#pragma unroll
              for (int i = 0; i < k; ++i) t[i] = t[2 * i] + t[2 * i + 1];
            sum = sum * ex2_approx(mx - m2) + t[0];
            mx = m2;
          }
        } else {
          if (nvis > 0) {
#pragma unroll
            for (int j = 0; j < 32; ++j)  // columns past the diagonal are summed too, and never stored
              acc[j] = fmaf(ex2_approx(fmaf(__uint_as_float(v[j]), scale_log2, -st.x)), st.y, acc[j]);
          }
          st = nst;
        }
      }
      if (!ok) break;
      if constexpr (STATS) {
        // the four parts of a row meet in shared memory; part 0 writes the result
        if (!mbar_wait_warp(bar(B_RE), unit_par ^ 1u, err, WAIT_TIMEOUT_NS)) break;
        red[part * TILE + r] = make_float2(mx, sum);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_RF));
        if (part == 0) {
          if (!mbar_wait_warp(bar(B_RF), unit_par, err, WAIT_TIMEOUT_NS)) break;
          float2 x[PARTS];
#pragma unroll
          for (int p = 0; p < PARTS; ++p) x[p] = red[p * TILE + r];
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B_RE));
          if (pos < u.n && index_ok(err, u.ts + pos, ext.rows)) {
            float m2 = x[0].x, z = 0.f;  // part 0 of a row sees at least its document's first key
#pragma unroll
            for (int p = 1; p < PARTS; ++p) m2 = fmaxf(m2, x[p].x);
#pragma unroll
            for (int p = 0; p < PARTS; ++p) z += x[p].y * ex2_approx(x[p].x - m2);
            stats[static_cast<int64_t>(w % Hq) * n_rows + u.ts + pos] =
                make_float2(m2, 1.f / (z * static_cast<float>(Hq)));
          }
        }
      } else {
        const int c0 = u.ct * TILE + part * 32;
        if (pos < u.n && index_ok(err, u.a_off + static_cast<int64_t>(u.n) * u.n - 1, ext.a_elems)) {
          float* dst = A + u.a_off + static_cast<int64_t>(c0) * u.n + pos;
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (c0 + j <= pos) dst[static_cast<int64_t>(j) * u.n] = acc[j];
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, TC_TMEM);
  }
}

// ---------------------------------------------------------------- salience of a column
constexpr int COL_WARPS = 8;

// One warp per token (column i of its document): u_i = mean of the top-p of its n - i entries
// A[i][i..n-1], which lie together.  They are averages of weights, never negative, so their
// bit patterns order as they do: the p-th largest is found bit by bit, the lane's NV entries
// in registers, then the larger ones are added and the ties filled up.  A bitonic sort of
// 2,048 keys per column took 466 us for 5,650 columns of 777-2,048 entries, this 30 us; the
// plain mean of 16,384 columns of 512 entries 107 us (strided reads), this 7 us.
template <int NV>
__global__ void __launch_bounds__(32 * COL_WARPS)
    k_sal_colstat(const int32_t* __restrict__ tok_pair, const int32_t* __restrict__ tok_off, int t0, int p0, int n_rows,
                  const int64_t* __restrict__ a_off, const float* A, int top_p, float* __restrict__ u,
                  Extents ext) {
  pdl_trigger();
  pdl_wait();
  const int t = blockIdx.x * COL_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= n_rows) return;
  const int p = tok_pair[t0 + t];
  const int ts = tok_off[p] - t0, n = tok_off[p + 1] - tok_off[p];
  const int i = t - ts;
  const int cnt = n - i, k = min(top_p, cnt);
  if (!index_ok(ext.err, a_off[p - p0] + static_cast<int64_t>(n) * n - 1, ext.a_elems)) return;
  const float* col = A + a_off[p - p0] + static_cast<int64_t>(i) * n + i;
  uint32_t v[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = q * 32 + lane < cnt ? __float_as_uint(col[q * 32 + lane]) : 0u;
  uint32_t thr = 0;
  int above = 0;      // entries larger than thr
  bool split = false;  // exactly k entries are not below thr: the search is over
  if (k < cnt) {
#pragma unroll 1
    for (int b = 30; b >= 0 && !split; --b) {
      const uint32_t cand = thr | (1u << b);
      int c = 0;
#pragma unroll
      for (int q = 0; q < NV; ++q) c += v[q] >= cand;
      c = static_cast<int>(__reduce_add_sync(0xffffffffu, c));
      if (c >= k) thr = cand;
      split = c == k;
    }
  }
  float sum = 0.f;
#pragma unroll
  for (int q = 0; q < NV; ++q)
    if (v[q] > thr || k == cnt || (split && v[q] == thr)) {
      sum += __uint_as_float(v[q]);
      ++above;
    }
  sum = warp_sum(sum);
  if (k < cnt && !split) sum += static_cast<float>(k - static_cast<int>(__reduce_add_sync(0xffffffffu, above))) * __uint_as_float(thr);
  if (lane == 0) u[t] = sum / static_cast<float>(k);
}

// ---------------------------------------------------------------- the most salient positions
constexpr int TOPK_THREADS = 1024;

// Exclusive scan of one count per thread over the block; *total gets the sum.
__device__ __forceinline__ int block_scan(int c, int* warp_sums, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();  // warp_sums is reused across calls
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int s = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    warp_sums[lane] = s;
  }
  __syncthreads();
  *total = warp_sums[31];
  return x - c + (warp ? warp_sums[warp - 1] : 0);
}

// One CTA per document of the chunk: the min(K, n) most salient positions,
// ties to the lower position, in ascending order; -1 after them.  Thread i holds positions
// 2i and 2i + 1; the K-th largest value is searched bit by bit over keys that order as the
// floats do, then two scans pick the ties and place the positions (8 us; a bitonic sort of
// 2,048 keys and a serial compaction took 33-40 us).
__global__ void __launch_bounds__(TOPK_THREADS) k_sal_topk(const int32_t* __restrict__ tok_off, int t0, int p0,
                                                           const float* u, int K,
                                                           int32_t* __restrict__ positions) {
  static_assert(SEL_MAX_N == 2 * TOPK_THREADS, "two positions a thread");
  __shared__ int warp_sums[32];
  pdl_trigger();
  pdl_wait();
  const int p = p0 + blockIdx.x;
  const int ts = tok_off[p] - t0, n = tok_off[p + 1] - tok_off[p];
  const int k = min(K, n);
  uint32_t key[2];
  bool in[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int r = 2 * threadIdx.x + e;
    in[e] = r < n;
    const uint32_t b = in[e] ? __float_as_uint(u[ts + r]) : 0u;
    key[e] = b & 0x80000000u ? ~b : b | 0x80000000u;
  }
  uint32_t thr = 0;
#pragma unroll 1
  for (int b = 31; b >= 0; --b) {
    const uint32_t cand = thr | (1u << b);
    const int c = __syncthreads_count(in[0] && key[0] >= cand) + __syncthreads_count(in[1] && key[1] >= cand);
    if (c >= k) thr = cand;
    if (c == k) {  // the k largest are those not below thr (which is above 0): no ties to share out
      --thr;
      break;
    }
  }
  int n_above, n_ties, n_all;
  const bool gt0 = in[0] && key[0] > thr, gt1 = in[1] && key[1] > thr;
  block_scan(gt0 + gt1, warp_sums, &n_above);
  const bool eq0 = in[0] && key[0] == thr, eq1 = in[1] && key[1] == thr;
  const int tie = block_scan(eq0 + eq1, warp_sums, &n_ties);
  const bool take0 = gt0 || (eq0 && tie < k - n_above), take1 = gt1 || (eq1 && tie + eq0 < k - n_above);
  const int at = block_scan(take0 + take1, warp_sums, &n_all);
  int32_t* out = positions + static_cast<int64_t>(p) * K;
  if (take0) out[at] = 2 * threadIdx.x;
  if (take1) out[at + take0] = 2 * threadIdx.x + 1;
  for (int j = k + threadIdx.x; j < K; j += TOPK_THREADS) out[j] = -1;
}

// One warp per (document, selected slot): x = bf16(RMSNorm(r_row) * g_final), zeros for -1.
__global__ void k_sal_gather(const float* r, int H, const int32_t* __restrict__ tok_off, int t0,
                             int p0, int n_docs, const int32_t* positions, int K,
                             const bf16* __restrict__ gain, float eps, bf16* __restrict__ x, Extents ext) {
  pdl_trigger();
  pdl_wait();
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= n_docs * K) return;
  const int p = p0 + w / K, j = w % K;
  const int pos = positions[static_cast<int64_t>(p) * K + j];
  uint2* dst = reinterpret_cast<uint2*>(x + (static_cast<int64_t>(p) * K + j) * H);
  if (pos < 0) {
    for (int c = lane; c < H / 4; c += 32) dst[c] = make_uint2(0u, 0u);
    return;
  }
  const int64_t rr = static_cast<int64_t>(tok_off[p] - t0) + pos;
  if (!index_ok(ext.err, rr, ext.rows)) return;
  const float4* row = reinterpret_cast<const float4*>(r + rr * H);  // H is a multiple of 256
  float ss = 0.f;
#pragma unroll 4
  for (int c = lane; c < H / 4; c += 32) {
    const float4 a = row[c];
    ss += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
  }
  ss = warp_sum(ss);
  const float rs = rsqrtf(ss / static_cast<float>(H) + eps);
  const uint2* g = reinterpret_cast<const uint2*>(gain);
#pragma unroll 4
  for (int c = lane; c < H / 4; c += 32) {
    const float4 a = row[c];
    const uint2 gw = g[c];
    const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gw.x));
    const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gw.y));
    dst[c] = make_uint2(pack_bf16x2(a.x * rs * g0.x, a.y * rs * g0.y), pack_bf16x2(a.z * rs * g1.x, a.w * rs * g1.y));
  }
}

}  // namespace

cudaError_t select_setup() {
  const cudaError_t e =
      cudaFuncSetAttribute(k_sal_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_sal_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
}

cudaError_t launch_select(const CUtensorMap& tm_rows, const SelectArgs& a, int num_sms, cudaStream_t st) {
  if (a.n_rows <= 0) return cudaSuccess;
  const int64_t stat_units = static_cast<int64_t>(a.n_row_tiles) * a.Hq;
  cudaError_t e = launch_dependent(k_sal_tc<true>, static_cast<int>(stat_units < num_sms ? stat_units : num_sms), TC_THREADS,
                                   TC_SMEM, st, tm_rows, a.row_tiles, a.n_row_tiles, a.Hq, a.Hkv, a.n_rows, a.stats, nullptr,
                                   a.ext);
  if (e != cudaSuccess) return e;
  e = launch_dependent(k_sal_tc<false>, a.n_tiles < num_sms ? a.n_tiles : num_sms, TC_THREADS, TC_SMEM, st, tm_rows,
                       a.row_tiles + a.n_row_tiles, a.n_tiles, a.Hq, a.Hkv, a.n_rows, a.stats, a.A, a.ext);
  if (e != cudaSuccess) return e;
  // registers for the longest document's columns (64 entries a lane at 2,048 tokens)
  auto* colstat = a.max_n <= 512 ? k_sal_colstat<16> : a.max_n <= 1024 ? k_sal_colstat<32> : k_sal_colstat<64>;
  e = launch_dependent(colstat, (a.n_rows + COL_WARPS - 1) / COL_WARPS, 32 * COL_WARPS, 0, st, a.tok_pair, a.tok_off, a.t0,
                       a.p0, a.n_rows, a.a_off, a.A, a.top_p, a.u, a.ext);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_sal_topk, a.n_docs, TOPK_THREADS, 0, st, a.tok_off, a.t0, a.p0, a.u, a.top_k, a.positions);
}

cudaError_t launch_select_gather(const SelectArgs& a, const float* r, int H, const bf16* gain, float eps,
                                 cudaStream_t st) {
  const int64_t threads = static_cast<int64_t>(a.n_docs) * a.top_k * 32;
  if (threads <= 0) return cudaSuccess;
  return launch_dependent(k_sal_gather, static_cast<unsigned>((threads + 255) / 256), 256, 0, st, r, H, a.tok_off, a.t0, a.p0,
                          a.n_docs, a.positions, a.top_k, gain, eps, a.x, a.ext);
}

}  // namespace dopr
