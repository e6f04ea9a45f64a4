// Row statistics of stored logits [M][V] in one pass: max, log-sum-exp, top-n and (draft sampling)
// the Gumbel-max token of every row.
//
// A cluster of 1 to 8 blocks takes a row, so that few rows still spread over the chip; a block
// reads its contiguous share of the row once, and the blocks' results meet in the first
// block's shared memory.  What bounds it: the arithmetic of the sampler (a Philox evaluation per
// logit, about 30 multiplies), not the read, which comes from L2 right behind the LM head.  Two
// things keep the rest small:
//  - the noise G = -ln(-ln u) <= -ln(1 - u), so a logit can only beat the best y so far when
//    1 - u <= exp(x / T - y): one exponential decides, and the two logarithms are taken for the
//    few that pass.  The best y is the block's (a warp's after every vector, shared through memory
//    after every batch): against each thread's own, some lane of a warp passed nearly every time
//    (576 rows of 32000: 89 -> 75 us);
//  - top-n: the n-th largest of the threads' maxima bounds the n-th largest logit from below, so
//    only threads whose own maximum reaches it (n of them, ties aside) look at their logits
//    again and put what reaches the bound on a list that one warp ranks.
// Measured against one pass per pick and a pass of its own for the sampler (LM head with its
// statistics, 13B / 33B shapes): 80 rows, top-1 140 -> 104 us; 144 rows, top-8 901 -> 267 us; 576
// rows in five launches, top-1 760 -> 623 us.
#include <cfloat>

#include <cooperative_groups.h>

#include "ps_internal.cuh"

namespace ps {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kListCap = 512;   // candidates of a block; rows with more ties than that are ranked pass by pass
constexpr int kTop = PS_MAX_TOP_N;

struct Part {   // one block's result
  float vmax, sum;
  float gv; int gi;                      // best perturbed logit
  float tv[kTop]; int ti[kTop];          // the block's own top-n
};
struct Shared {
  Part part;
  float f[kWarps], g[kWarps];
  int i[kWarps];
  unsigned keys[kWarps][kTop];
  float bound;
  unsigned thr;      // key of the block's best perturbed logit so far
  int n_list;
  float lv[kListCap];
  int li[kListCap];
};

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Larger value first, ties to the lower id.
__device__ __forceinline__ bool ranks_before(float v, int i, float w, int j) { return v > w || (v == w && i < j); }
__device__ __forceinline__ void warp_best(float& v, int& i) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, v, o);
    const int oi = __shfl_xor_sync(0xffffffffu, i, o);
    if (ranks_before(ov, oi, v, i)) { v = ov; i = oi; }
  }
}
// Unsigned keys in the order of the floats.
__device__ __forceinline__ unsigned key_of(float x) {
  const unsigned b = __float_as_uint(x);
  return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float key_value(unsigned k) { return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu)); }

template <bool SAMPLE>
__global__ void __launch_bounds__(kThreads) k_logit_stats(const float* __restrict__ logits, int V, int R, int top_n,
                                                          int* top_ids, float* top_logit, float* row_max, float* row_lse,
                                                          SampleArgs sa) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ Shared s;
  const int nclu = gridDim.x, rank = blockIdx.x, m = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) { s.n_list = 0; s.thr = 0u; }
  __syncthreads();
  const float* row = logits + (size_t)m * V;
  const int share = ((V + nclu - 1) / nclu + 3) & ~3;          // tokens per block, whole vectors
  const int v_lo = min(V, rank * share), v_hi = min(V, v_lo + share);
  // vectors from the first 16-byte boundary on; the up to three tokens before it and after them one by one
  const int v_al = min(v_hi, v_lo + (int)((16u - ((unsigned)(uintptr_t)(row + v_lo) & 15u)) & 15u) / 4);
  const int n_vec = (v_hi - v_al) / 4, n_head = v_al - v_lo, n_one = v_hi - v_lo - 4 * n_vec;
  const float4* row4 = reinterpret_cast<const float4*>(row + v_al);
  auto one_at = [&](int i) { return i < n_head ? v_lo + i : v_al + 4 * n_vec + (i - n_head); };
  uint32_t row_id = 0;
  if (SAMPLE) {
    const int b = m / R;
    row_id = ((uint32_t)b + sa.b_base) | ((uint32_t)(m - b * R) << 8);
  }
  pdl_wait();
  pdl_launch_dependents();   // (not earlier: a dependent's blocks would wait beside the LM head's)

  // ---- the pass: per-thread running maximum and sum of exponentials, best perturbed logit
  float mx = -FLT_MAX, se = 0.f, gv = -FLT_MAX, thr = -FLT_MAX;
  int gi = 0x7fffffff;
  auto sample_one = [&](float x, int v) {
    uint32_t c[4] = {(uint32_t)v, row_id, sa.off_lo, sa.off_hi};
    philox4x32_10(sa.key0, sa.key1, c);
    const uint32_t w = c[0] >> 8;
    const float y0 = x * sa.inv_temp;
    // 1 - u up to its last bit; the margins cover the rounding of the test and of y = y0 + G
    const float rest = ((float)(16777216u - w) - 0.5f) * (1.0f / 16777216.0f);
    if (!(rest > 1.01f * __expf(y0 - thr + fabsf(y0) * 2.4e-7f))) {
      const float y = y0 + gumbel_of_word(w);
      if (ranks_before(y, v, gv, gi)) { gv = y; gi = v; }
    }
  };
  constexpr int U = 4;   // vectors in flight per thread
  const bool held = n_vec <= U * kThreads;   // one batch: its logits stay in registers for the second look
  float4 x[U];
#pragma unroll
  for (int u = 0; u < U; ++u) x[u] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  for (int i0 = tid; i0 - tid < n_vec; i0 += U * kThreads) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      x[u] = i0 + u * kThreads < n_vec ? __ldcg(row4 + i0 + u * kThreads) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    float bm = mx;
#pragma unroll
    for (int u = 0; u < U; ++u) bm = fmaxf(fmaxf(fmaxf(bm, x[u].x), fmaxf(x[u].y, x[u].z)), x[u].w);
    float add = 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) add += (__expf(x[u].x - bm) + __expf(x[u].y - bm)) + (__expf(x[u].z - bm) + __expf(x[u].w - bm));
    se = se * __expf(mx - bm) + add;
    mx = bm;
    if (SAMPLE) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (i0 + u * kThreads < n_vec) {
          const int v = v_al + 4 * (i0 + u * kThreads);
          sample_one(x[u].x, v); sample_one(x[u].y, v + 1); sample_one(x[u].z, v + 2); sample_one(x[u].w, v + 3);
        }
        const unsigned k = __reduce_max_sync(0xffffffffu, key_of(gv));
        thr = fmaxf(thr, key_value(k));
      }
      if (lane == 0) atomicMax(&s.thr, key_of(thr));
      const unsigned k = *(volatile unsigned*)&s.thr;   // (any value seen is one that some lane has reached)
      if (k) thr = fmaxf(thr, key_value(k));
    }
  }
  if (tid < n_one) {
    const int v = one_at(tid);
    const float x = __ldcg(row + v), bm = fmaxf(mx, x);
    se = se * __expf(mx - bm) + __expf(x - bm);
    mx = bm;
    if (SAMPLE) sample_one(x, v);
  }
  const float my_max = mx;

  // ---- block results
  const float wm = warp_max(mx);
  const float ws = warp_sum(se * __expf(mx - wm));
  if (SAMPLE) warp_best(gv, gi);
  unsigned key = key_of(my_max);
  for (int t = 0; t < top_n; ++t) {   // the warp's largest thread maxima, in order
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    const unsigned who = __ballot_sync(0xffffffffu, key == top);
    if (lane == __ffs(who) - 1) key = 0u;
    if (lane == 0) s.keys[warp][t] = top;
  }
  if (lane == 0) {
    s.f[warp] = wm; s.g[warp] = ws;
    if (SAMPLE) { s.lv[warp] = gv; s.li[warp] = gi; }
  }
  __syncthreads();
  if (warp == 0) {
    const float a = lane < kWarps ? s.f[lane] : -FLT_MAX;
    const float bm = warp_max(a), bs = warp_sum(lane < kWarps ? s.g[lane] * __expf(a - bm) : 0.f);
    float bg = -FLT_MAX;
    int bi = 0x7fffffff;
    if (SAMPLE) {
      if (lane < kWarps) { bg = s.lv[lane]; bi = s.li[lane]; }
      warp_best(bg, bi);
    }
    // the top_n-th largest of all thread maxima: lane w walks warp w's ordered keys
    int at = 0;
    unsigned bound = 0u;
    for (int t = 0; t < top_n; ++t) {
      const unsigned k = (lane < kWarps && at < top_n) ? s.keys[lane][at] : 0u;
      bound = __reduce_max_sync(0xffffffffu, k);
      const unsigned who = __ballot_sync(0xffffffffu, k == bound);
      if (lane == __ffs(who) - 1) ++at;
    }
    if (lane == 0) {
      s.part.vmax = bm; s.part.sum = bs; s.part.gv = bg; s.part.gi = bi;
      s.bound = bound ? key_value(bound) : -FLT_MAX;
    }
  }
  __syncthreads();
  if (top_n > 0) {
    const float bound = s.bound;
    if (my_max >= bound) {
      auto offer = [&](float x, int v) {
        if (x >= bound) {
          const int at = atomicAdd(&s.n_list, 1);
          if (at < kListCap) { s.lv[at] = x; s.li[at] = v; }
        }
      };
      if (held) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = tid + u * kThreads, v = v_al + 4 * i;
          if (i < n_vec) { offer(x[u].x, v); offer(x[u].y, v + 1); offer(x[u].z, v + 2); offer(x[u].w, v + 3); }
        }
      } else {
#pragma unroll 4
        for (int i = tid; i < n_vec; i += kThreads) {
          const float4 y = __ldcg(row4 + i);
          const int v = v_al + 4 * i;
          offer(y.x, v); offer(y.y, v + 1); offer(y.z, v + 2); offer(y.w, v + 3);
        }
      }
      if (tid < n_one) offer(__ldcg(row + one_at(tid)), one_at(tid));
    }
    __syncthreads();
    const int n_list = s.n_list;
    if (n_list <= kListCap) {
      if (warp == 0) {
        float pv = FLT_MAX;
        int pi = -1;
        for (int t = 0; t < top_n; ++t) {
          float bv = -FLT_MAX;
          int bi = 0x7fffffff;
          for (int e = lane; e < n_list; e += 32) {
            const float v = s.lv[e];
            const int i = s.li[e];
            if (ranks_before(pv, pi, v, i) && ranks_before(v, i, bv, bi)) { bv = v; bi = i; }
          }
          warp_best(bv, bi);
          if (lane == 0) { s.part.tv[t] = bv; s.part.ti[t] = bi; }
          pv = bv; pi = bi;
        }
      }
    } else {   // a row of many equal logits: one pass over the block's share per pick
      float pv = FLT_MAX;
      int pi = -1;
      for (int t = 0; t < top_n; ++t) {
        float bv = -FLT_MAX;
        int bi = 0x7fffffff;
        for (int v = v_lo + tid; v < v_hi; v += kThreads) {
          const float x = __ldcg(row + v);
          if (ranks_before(pv, pi, x, v) && ranks_before(x, v, bv, bi)) { bv = x; bi = v; }
        }
        warp_best(bv, bi);
        __syncthreads();
        if (lane == 0) { s.f[warp] = bv; s.i[warp] = bi; }
        __syncthreads();
        bv = s.f[0]; bi = s.i[0];
        for (int w = 1; w < kWarps; ++w)
          if (ranks_before(s.f[w], s.i[w], bv, bi)) { bv = s.f[w]; bi = s.i[w]; }
        if (tid == 0) { s.part.tv[t] = bv; s.part.ti[t] = bi; }
        pv = bv; pi = bi;
      }
    }
  }
  // ---- the blocks' results meet in the first block
  if (nclu > 1) cl.sync(); else __syncthreads();
  if (rank == 0 && warp == 0) {
    const Part* q = lane < nclu ? (nclu > 1 ? cl.map_shared_rank(&s.part, lane) : &s.part) : nullptr;
    const float a = q ? q->vmax : -FLT_MAX;
    const float rm = warp_max(a), rs = warp_sum(q ? q->sum * __expf(a - rm) : 0.f);
    if (lane == 0) {
      if (row_max) row_max[m] = rm;
      if (row_lse) row_lse[m] = rm + logf(rs);
    }
    if (SAMPLE) {
      float bg = q ? q->gv : -FLT_MAX;
      int bi = q ? q->gi : 0x7fffffff;
      warp_best(bg, bi);
      if (lane == 0) sa.sampled[m] = bi;
    }
    int at = 0;
    float hv = -FLT_MAX;
    int hi = 0x7fffffff;
    if (q && top_n > 0) { hv = q->tv[0]; hi = q->ti[0]; }
    for (int t = 0; t < top_n; ++t) {   // every lane offers its block's best remaining entry
      float bv = hv;
      int bi = hi;
      warp_best(bv, bi);
      if (lane == 0) { top_ids[(size_t)m * top_n + t] = bi; top_logit[(size_t)m * top_n + t] = bv; }
      if (hi == bi && q) {
        ++at;
        hv = at < top_n ? q->tv[at] : -FLT_MAX;
        hi = at < top_n ? q->ti[at] : 0x7fffffff;
      }
    }
  }
  if (nclu > 1) cl.sync();   // no block leaves while the first one reads its result
}

}  // namespace

ps_status launch_logit_stats(ps_ctx* c, const float* logits, int M, int V, int R, int top_n, int* top_ids,
                             float* top_logit, float* row_max, float* row_lse, const SampleArgs* sa, cudaStream_t st) {
  if (top_n <= 0 && !row_max && !row_lse && !sa) return PS_OK;
  // Blocks per row: the count whose waves are over first, with at least 2048 tokens a block (below that its
  // fixed cost, about 2 us of reductions, outweighs what it takes off the pass).  With the sampler two blocks
  // are resident per SM and its arithmetic is what takes time, so only the balance counts: 144 rows of
  // 32000 tokens, 2 blocks in one wave, 50 -> 30 us against 4 in two; a single full wave is worth more
  // than its share says (80 rows: 7 blocks in two waves 31 us).  Without it three are resident and a block
  // is through 32000 tokens in about 5 us, so that many rows want few blocks: 640 rows 66 -> 33 us.  The clusters of
  // a wave are as many as find room (444 blocks of their own, but 104 clusters of 4, 82 of 5, 48 of 8), where a wave
  // that needs nearly every place takes as long as two, and a later wave begins before the one ahead of it has
  // ended.  128256 tokens, 80 rows: 4 blocks (131 us for the step) instead of 5 (137), which fill 80 of 82 places; 32000
  // tokens, 85 rows 90 -> 85.  Of 48 counts of rows and tokens the choice is 0.4% behind the best one, at most 2%.
  int nclu = 1;
  double best = 1e30;
  for (int n = 1; n <= 8 && (n == 1 || V / n >= 2048); ++n) {
    double cost;
    if (sa) {
      const long slots = 2l * c->n_sm, waves = ((long)M * n + slots - 1) / slots;
      cost = (waves > 1 ? 1.15 : 1.0) * waves / n + 0.005 * n;
    } else {
      int places = clusters_at_once(c->stats_clusters[n], k_logit_stats<false>, kThreads, n);
      if (places <= 0) places = std::max(1, 3 * c->n_sm / n);
      const int room = n <= 2 ? places : places * 31 / 32;
      const double waves = M <= room ? 1.0 : std::max(2, (M + places - 1) / places);
      cost = 0.5 * (waves + std::max(1.0, (double)M / places)) * (4.0 + 5.0 * V / 32000 / n) + 0.05 * n;
    }
    if (cost < best) { best = cost; nclu = n; }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nclu, M);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nclu; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = c->prof ? 1 : 2;
  const SampleArgs none{};
  const cudaError_t e =
      sa ? cudaLaunchKernelEx(&cfg, k_logit_stats<true>, logits, V, R, top_n, top_ids, top_logit, row_max, row_lse, *sa)
         : cudaLaunchKernelEx(&cfg, k_logit_stats<false>, logits, V, R, top_n, top_ids, top_logit, row_max, row_lse, none);
  c->launches++;
  return cuda_check(c, e, "k_logit_stats");
}

}  // namespace ps
