// k_pack.cu -- device batch packer of the online pass.
//
// DoPR's online efficiency comes from reusing a document's stored prefix
// across all queries that retrieved it (Sec. 3.4, "cross-query prefix state
// reuse").  The packer orders the batch so that all pairs of one document are
// adjacent: a stable sort on doc_id (ties keep input order), then
// lays every pair's [query tokens ; score token] end to end in that order
// with RoPE positions m_doc + j.  Steps:
//   1. k_pack_order, one cluster (which also leaves what the host plans with in pinned memory, so
//      that no copies follow it): validate pairs and look up store slots, sort by doc id
//      (radix, 10 bits a pass), exclusive scan of per-pair token counts (packed token offsets);
//   2. k_pack_tokens (after the host has sized the token buffers): token ids / positions.
#include "device_common.cuh"
#include "internal.h"

namespace dopr {
namespace {

constexpr int INPUT_ERRORS = DEV_ERR_UNKNOWN_DOC | DEV_ERR_INCOMPLETE | DEV_ERR_BAD_TOKEN | DEV_ERR_BAD_OFFSETS |
                             DEV_ERR_POSITION;

constexpr int ORDER_THREADS = 1024, ORDER_WARPS = ORDER_THREADS / 32;
constexpr int ORDER_CTAS = 8;         // CTAs of the cluster for large batches
constexpr int ORDER_ONE_CTA = 4096;   // pairs that one CTA orders by itself (4,000: 17 us, as eight CTAs take)
constexpr int DIGIT_BITS = 10;
constexpr int ORDER_SMEM = ORDER_WARPS * (1 << DIGIT_BITS) * 4;  // a digit histogram per warp: 128 KB

// Block-wide exclusive scan of one value per thread; *total gets the sum.
__device__ int32_t block_scan(int32_t v, int32_t* warp_sums, int32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();  // warp_sums is reused across calls
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int32_t w = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    warp_sums[lane] = w;
  }
  __syncthreads();
  *total = warp_sums[31];
  return x - v + (warp > 0 ? warp_sums[warp - 1] : 0);
}

// One cluster of CTAs orders the batch.  Each warp owns a contiguous segment of the pairs (of the
// previous pass's order) and a histogram of its own, so the warps need not walk the pairs in
// turn: count the segment's digits, scan over (digit, CTA, warp), then place the segment 32
// pairs at a time, lanes of equal digits taking consecutive places.  doc_bits: bits of the
// largest doc id; 1,024 documents are one pass.  The look-ups by document and by place touch a
// sector per lane, and one SM takes about one sector a clock: seven such accesses a pair cost
// one CTA 64 us at 20,000 pairs, eight CTAs 26 us.  One warp walking all pairs took 740 us,
// with the other three kernels 778.
template <int CTAS>
__global__ void __launch_bounds__(ORDER_THREADS) k_pack_order(PackArgs a, int doc_bits) {
  constexpr int AHEAD = CTAS > 1 ? 4 : 2;  // pairs a lane looks at together
  extern __shared__ int32_t hist[];  // [warp][digit]
  __shared__ int32_t digit_count[1 << DIGIT_BITS], warp_sums[32], cta_total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = a.n_pairs;
  constexpr int ctas = CTAS;
  const int rank = CTAS > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  // all threads of the cluster meet; what they wrote to global memory is visible after it
  auto meet = [] {
    if constexpr (CTAS > 1) {
      __threadfence();
      cluster_sync();
    } else {
      __syncthreads();
    }
  };
  // value `at` of CTA r's shared memory
  auto peer = [&](const int32_t* at, int r) {
    if constexpr (CTAS == 1) return *at;
    int32_t v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(mapa_shared(smem_u32(at), r)) : "memory");
    return v;
  };

  if (rank == 0) {
    for (int i = tid; i < a.n_zero; i += ORDER_THREADS) a.zero[i] = 0;
    if (tid == 0) *a.err = 0;
  }
  meet();

  // ---- validate: every pair's slot, or the batch's errors
  int flags = 0;
  for (int p0 = rank * ORDER_THREADS + tid; p0 < n; p0 += ctas * ORDER_THREADS * AHEAD) {
    // AHEAD pairs' look-ups go along together: each is three loads that wait for one another
    int64_t doc[AHEAD];
    int slot[AHEAD], len[AHEAD], m[AHEAD], ok[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int64_t p = p0 + static_cast<int64_t>(k) * ctas * ORDER_THREADS;
      doc[k] = p < n ? a.doc_ids[p] : -1;
      len[k] = p < n ? a.q_off[p + 1] - a.q_off[p] : 0;
    }
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) slot[k] = doc[k] < 0 || doc[k] > a.max_doc_id ? -1 : a.slot_of[doc[k]];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      m[k] = slot[k] < 0 ? 0 : a.slot_m[slot[k]];
      ok[k] = slot[k] < 0 ? 0 : a.slot_ok[slot[k]];
    }
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int64_t p = p0 + static_cast<int64_t>(k) * ctas * ORDER_THREADS;
      if (p >= n) break;
      int flag = slot[k] < 0 ? DEV_ERR_UNKNOWN_DOC : !ok[k] ? DEV_ERR_INCOMPLETE : 0;
      if (len[k] < 0 || (p == 0 && a.q_off[0] != 0)) flag |= DEV_ERR_BAD_OFFSETS;
      if (!flag && m[k] + len[k] + 1 > a.max_position) flag |= DEV_ERR_POSITION;
      a.pair_slot[p] = flag ? -1 : slot[k];
      flags |= flag;
    }
  }
  if (flags) atomicOr(a.err, flags);
  meet();
  const int found = ld_volatile(a.err);  // the same word for the whole cluster
  if (rank == 0 && tid == 0 && a.h_err) *a.h_err = found;
  if (found & INPUT_ERRORS) return;

  // ---- stable sort by doc id; the order goes to perm, by way of sorted_slot
  const int passes = (doc_bits + DIGIT_BITS - 1) / DIGIT_BITS, bits = (doc_bits + passes - 1) / passes;
  const int n_digits = 1 << bits, warps = ctas * ORDER_WARPS;
  const int seg = ((n + warps - 1) / warps + 31) / 32 * 32;
  const int beg = static_cast<int>(min(static_cast<int64_t>(n), static_cast<int64_t>(rank * ORDER_WARPS + warp) * seg));
  const int end = min(n, beg + seg);
  int32_t* mine = hist + warp * n_digits;
  const int32_t* src = nullptr;  // the first pass reads the pairs in input order
  for (int pass = 0; pass < passes; ++pass) {
    int32_t* dst = (passes - 1 - pass) & 1 ? a.sorted_slot : a.perm;
    const int shift = pass * bits;
    auto digit_of = [&](int p) { return static_cast<int>(a.doc_ids[p] >> shift) & (n_digits - 1); };
    for (int i = tid; i < ORDER_WARPS * n_digits; i += ORDER_THREADS) hist[i] = 0;
    __syncthreads();
    for (int i = beg; i < end; i += 32 * AHEAD) {
      int d[AHEAD];
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) {
        const int s = i + 32 * k + lane;
        d[k] = s < end ? digit_of(src ? __ldcg(src + s) : s) : -1;
      }
#pragma unroll
      for (int k = 0; k < AHEAD; ++k)
        if (d[k] >= 0) atomicAdd(&mine[d[k]], 1);
    }
    __syncthreads();
    if (tid < n_digits) {
      int32_t count = 0;
#pragma unroll 8
      for (int w = 0; w < ORDER_WARPS; ++w) count += hist[w * n_digits + tid];
      digit_count[tid] = count;
    }
    meet();
    int32_t all = 0, before = 0, total;  // of this digit: in the batch, in the CTAs before this one
    if (tid < n_digits) {
      int32_t c[CTAS];
#pragma unroll
      for (int r = 0; r < CTAS; ++r) c[r] = peer(&digit_count[tid], r);
#pragma unroll
      for (int r = 0; r < CTAS; ++r) {
        all += c[r];
        before += r < rank ? c[r] : 0;
      }
    }
    int32_t run = block_scan(all, warp_sums, &total) + before;
    if (tid < n_digits)
#pragma unroll 8
      for (int w = 0; w < ORDER_WARPS; ++w) {
        const int32_t c = hist[w * n_digits + tid];
        hist[w * n_digits + tid] = run;
        run += c;
      }
    __syncthreads();
    for (int i = beg; i < end; i += 32 * AHEAD) {
      int q[AHEAD], d[AHEAD];
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) {
        const int s = i + 32 * k + lane;
        q[k] = s < end ? (src ? __ldcg(src + s) : s) : -1;
        d[k] = s < end ? digit_of(q[k]) : -1;
      }
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) {
        // lanes with this lane's digit: one vote a bit (match_any takes its time per distinct value)
        unsigned same = __ballot_sync(0xffffffffu, d[k] >= 0);
        for (int b = 0; b < bits; ++b) {
          const unsigned v = __ballot_sync(0xffffffffu, (d[k] >> b) & 1);
          same &= (d[k] >> b) & 1 ? v : ~v;
        }
        const int place = d[k] >= 0 ? mine[d[k]] : 0;
        __syncwarp();
        if (d[k] >= 0) {
          if (lane == __ffs(same) - 1) mine[d[k]] = place + __popc(same);
          dst[place + __popc(same & ((1u << lane) - 1u))] = q[k];
        }
        __syncwarp();
      }
    }
    meet();  // the pass's order is complete, and digit_count read, before either changes
    src = dst;
  }

  // ---- slots in the sorted order, and the packed offsets: this CTA's share of the places
  const int share = ((n + ctas - 1) / ctas + 3) / 4 * 4;
  const int lo = static_cast<int>(min(static_cast<int64_t>(n), static_cast<int64_t>(rank) * share)), hi = min(n, lo + share);
  int32_t sum = 0, total;
  for (int s = lo + tid; s < hi; s += ORDER_THREADS) {
    const int p = __ldcg(a.perm + s);
    const int slot = __ldcg(a.pair_slot + p);
    a.sorted_slot[s] = slot;
    if (a.h_sorted_slot) a.h_sorted_slot[s] = slot;
    const int len = a.q_off[p + 1] - a.q_off[p] + 1;
    a.tok_off[s] = len;
    sum += len;
  }
  block_scan(sum, warp_sums, &total);
  int32_t carry = 0;
  if constexpr (CTAS > 1) {
    if (tid == 0) cta_total = total;
    cluster_sync();
    int32_t c[CTAS];
#pragma unroll
    for (int r = 0; r < CTAS; ++r) c[r] = peer(&cta_total, r);
#pragma unroll
    for (int r = 0; r < CTAS; ++r) carry += r < rank ? c[r] : 0;
  }
  for (int s0 = lo; s0 < hi; s0 += ORDER_THREADS) {
    const int s = s0 + tid;  // written by this thread above
    const int32_t len = s < hi ? a.tok_off[s] : 0;
    const int32_t at = carry + block_scan(len, warp_sums, &total);
    if (s < hi) {
      a.tok_off[s] = at;
      if (a.h_tok_off) a.h_tok_off[s] = at;
    }
    carry += total;
  }
  if (tid == 0 && rank == ctas - 1) {
    a.tok_off[n] = carry;
    if (a.h_tok_off) a.h_tok_off[n] = carry;
  }
  if constexpr (CTAS > 1) cluster_sync();  // no CTA leaves while another may read its total
}

// One warp per sorted pair.
__global__ void k_pack_tokens(PackArgs a) {
  if (ld_volatile(a.err) & INPUT_ERRORS) return;
  const int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (s >= a.n_pairs) return;
  const int p = a.perm[s];
  const int q0 = a.q_off[p], L = a.q_off[p + 1] - q0;
  const int off = a.tok_off[s];
  const int m = a.slot_m[a.sorted_slot[s]];
  for (int j = lane; j <= L; j += 32) {
    int tok = j < L ? a.q_tok[q0 + j] : a.score_token;
    if (tok < 0 || tok >= a.vocab) {
      atomicOr(a.err, DEV_ERR_BAD_TOKEN);
      tok = 0;
    }
    a.tok_id[off + j] = tok;
    a.tok_pos[off + j] = m + j;
    a.tok_pair[off + j] = s;
  }
}

__global__ void k_commit_scores(const int* err, const float* scores, float* __restrict__ out, int n) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && ld_volatile(err) == 0) out[i] = scores[i];
}

}  // namespace

cudaError_t launch_commit_scores(const int* err, const float* scores, float* out, int n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  return launch_dependent(k_commit_scores, (n + 255) / 256, 256, 0, st, err, scores, out, n);
}

cudaError_t pack_setup() {
  const cudaError_t e = cudaFuncSetAttribute(k_pack_order<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, ORDER_SMEM);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_pack_order<ORDER_CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, ORDER_SMEM);
}

cudaError_t launch_pack_order(const PackArgs& a, cudaStream_t st) {
  if (a.n_pairs <= 0) return cudaSuccess;
  int doc_bits = 1;
  while (doc_bits < 31 && (a.max_doc_id >> doc_bits)) ++doc_bits;
  if (a.n_pairs <= ORDER_ONE_CTA) {
    k_pack_order<1><<<1, ORDER_THREADS, ORDER_SMEM, st>>>(a, doc_bits);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ORDER_CTAS);
  cfg.blockDim = dim3(ORDER_THREADS);
  cfg.dynamicSmemBytes = ORDER_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ORDER_CTAS;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_pack_order<ORDER_CTAS>, a, doc_bits);
}

cudaError_t launch_pack_tokens(const PackArgs& a, cudaStream_t st) {
  if (a.n_pairs <= 0) return cudaSuccess;
  k_pack_tokens<<<(a.n_pairs + 7) / 8, 256, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace dopr
