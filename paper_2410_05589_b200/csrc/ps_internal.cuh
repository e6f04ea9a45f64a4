// Internal declarations shared by the translation units of the library.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "ps.h"

namespace ps {

constexpr int kMaxRowsPerSeq = PS_MAX_MASKS + 1;  // rows of one sequence in a draft step
constexpr int kAppendChunk = 256;                 // rows handled per pass of ps_kv_append
constexpr int kAttnMaxSplit = 32;                 // key-range splits of the fused attention
constexpr int kMaxSm = 192;                       // bound used to size per-CTA scratch
constexpr size_t kGuardBytes = 256;               // guard words behind every slice of the workspace
constexpr int kGuardFill = 0x5A;

// Which sequence each row of a launch belongs to.  Passed by value as a kernel parameter.
// Row m (0-based within the launch) belongs to the sequence b with
// row_off[b] <= m + row_base < row_off[b+1]; its index inside the sequence is
// j = m + row_base - row_off[b] and its absolute position is len[b] + j.
struct SeqMap {
  int B;
  int row_base;
  int slot[PS_MAX_BATCH];
  int len[PS_MAX_BATCH];
  int row_off[PS_MAX_BATCH + 1];
  int fit;   // 1: the rows are stored as fit_row() has them
};

// A (position, head)'s key and value, of which each of `per` neighbouring lanes (a power of two) holds a part: if the
// value is not finite the key becomes no number and the value zero.  A query that sees the key gets a score that is
// none, and with it a result that is none; one that must not, and only gives it a probability of zero, is left alone (0 times
// an infinite value is not 0).  For rows that queries of several positions meet in one product.
template <class KV>
__device__ __forceinline__ void fit_row(KV& k0, KV& k1, KV& v0, KV& v1, int per) {
  constexpr int N = sizeof(KV) / 2;
  auto *a = reinterpret_cast<unsigned short*>(&v0), *b = reinterpret_cast<unsigned short*>(&v1);
  bool bad = false;
#pragma unroll
  for (int e = 0; e < N; ++e) bad |= (a[e] & 0x7F80) == 0x7F80 || (b[e] & 0x7F80) == 0x7F80;
  const unsigned lane = threadIdx.x & 31, group = (0xFFFFFFFFu >> (32 - per)) << (lane & ~(per - 1));
  if (__ballot_sync(group, bad)) {
    auto *c = reinterpret_cast<unsigned short*>(&k0), *d = reinterpret_cast<unsigned short*>(&k1);
#pragma unroll
    for (int e = 0; e < N; ++e) { c[e] = d[e] = 0x7FFF; a[e] = b[e] = 0; }
  }
}

__device__ __forceinline__ void seq_of_row(const SeqMap& s, int m, int& b, int& j) {
  int g = m + s.row_base;
  int lo = 0, hi = s.B - 1;
  while (lo < hi) {  // last b with row_off[b] <= g (empty sequences are skipped by taking the last)
    int mid = (lo + hi + 1) >> 1;
    if (s.row_off[mid] <= g) lo = mid; else hi = mid - 1;
  }
  b = lo;
  j = g - s.row_off[lo];
}

// Programmatic dependent launch.  A kernel launched with `launch_after` (pdl = true) may start
// while the kernel before it in the stream still runs; it must call pdl_wait() before it reads
// or writes anything that kernel touches (a no-op for a plain launch), and calls
// pdl_launch_dependents() early so that its own successor may be scheduled behind it.
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... KArgs, class... Args>
cudaError_t launch_after(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                         Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Philox-4x32 with 10 rounds (Salmon et al., SC'11): counter (c0..c3), key (k0, k1).
__device__ __forceinline__ void philox4x32_10(uint32_t k0, uint32_t k1, uint32_t (&c)[4]) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    // (one wide multiply for both halves of a product)
    const uint64_t p0 = (uint64_t)0xD2511F53u * c[0], p1 = (uint64_t)0xCD9E8D57u * c[2];
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c[1] ^ k0, n2 = (uint32_t)(p0 >> 32) ^ c[3] ^ k1;
    c[0] = n0; c[1] = (uint32_t)p1; c[2] = n2; c[3] = (uint32_t)p0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// Draft sampling (Algorithm 1: the tree is drafted by sampling from the parallel drafter): the
// token of a row is the arg-max over v of logit_v / T + G(v, row), G = -ln(-ln u) (the
// Gumbel-max rule), u = ((w >> 8) + 0.5) / 2^24 with w = word 0 of Philox, key = (seed_lo ^
// 0x6D756247, seed_hi), counter = (v, row_id, offset); row_id = b | j << 8.
struct SampleArgs {
  float inv_temp;
  uint32_t key0, key1, off_lo, off_hi;
  int* sampled;   // [B][k+1]
  uint32_t b_base;   // index, in the caller's batch, of the first sequence of this launch
};
// G of the 24-bit word w: e = -ln u in single precision without losing u's distance from 1 (u can
// sit within 2^-25 of it): below one half from u itself, above from 1 - u = (2^24 - w - 0.5) / 2^24,
// which like w + 0.5 is exact in fp32 on its half of the range.
__device__ __forceinline__ float gumbel_of_word(uint32_t w) {
  float e;
  if (w < (1u << 23)) e = -__logf(((float)w + 0.5f) * (1.0f / 16777216.0f));
  else e = -log1pf(-((float)(16777216u - w) - 0.5f) * (1.0f / 16777216.0f));
  return -__logf(e);
}
__device__ __forceinline__ float gumbel_noise(const SampleArgs& sa, uint32_t v, uint32_t row_id) {
  uint32_t c[4] = {v, row_id, sa.off_lo, sa.off_hi};
  philox4x32_10(sa.key0, sa.key1, c);
  return gumbel_of_word(c[0] >> 8);
}

// Device status word values (bit flags).
constexpr int kStatNonfinite = 1;
constexpr int kStatTimeout = 2;

struct RowStat {    // softmax statistics of a row of logits (token-tree verification)
  float max;
  int arg;          // its lowest id
  int bad;          // a non-finite logit was met, or nothing lies above -inf
  int pad;
  double sum;       // of exp((logit - max) / T)
};

struct VerifyRow {  // one per (sequence, position): verdict and statistics of a row pair (streaming kernel)
  int flags;        // bit 0: accepted; bit 1: a non-finite logit was met
  int targ;         // arg-max of the target row
  float tmax, dmax;
  double st, sd;    // sums of exponentials relative to the maxima
};

struct VerifyDraw { // one per sequence: where its chain stops
  int pos, acc;     // position to draw at (-1: none), accepted drafts before it
  float tmax, dmax; // statistics of the position's row pair
  double st, sd;
};

struct VerifyRec {  // one per (sequence, position): result of the acceptance test
  int accept;       // bit 0: accepted; bit 1: a non-finite logit was met
  int token;        // token to emit if this position ends the chain
};

}  // namespace ps

struct ps_ctx {
  ps_config cfg;
  ps_weights w;
  int device;
  char* ws;
  size_t ws_bytes;
  int max_rows;    // rows the activation buffers hold
  // workspace slices
  void* kcache;    // [max_batch][n_kv_heads][max_ctx][head_dim] storage dtype, post-RoPE
  void* vcache;
  int* dev_status;
  unsigned* tickets;        // [max_batch] arrival counters of the verify kernel (zero between calls)
  ps::VerifyRec* vrec;      // [max_batch][PS_MAX_MASKS+2]
  ps::VerifyRow* vrow;      // [max_batch][PS_MAX_MASKS+2]
  ps::VerifyDraw* vdraw;    // [max_batch]
  ps::RowStat* tree_stats;  // [max_batch][2 PS_MAX_TREE_NODES + 1]
  float *x0, *q, *kv_tmp, *attn, *a, *gate, *hdn, *logits;
  // staging for ps_round_host
  void* fused_scratch;      // buffers of the fused bf16 path (see fused_kernels.cu)
  void* umma_maps = nullptr;   // tensor maps of the tensor-core GEMMs, built on first use
  bool umma_tried = false;
  int act_rows = 0;            // rows of the last draft step whose "act" exists as planes only
  double* rope_inv_freq;    // [head_dim/2] base^(-2i/d), filled once at ps_init
  int n_sm;                 // multiprocessors of the context's device
  int smem_optin;           // opt-in shared memory per block
  // answers asked of this context's device once (0 = not asked yet)
  int clusters[4][17] = {};       // [chain verify, tree walk, the same at other T than 0 and 1][cluster size]: resident at once, -1 none
  int stream_clusters[2][9] = {}; // streaming verify [T is 0 or 1, other][cluster size]
  int stats_clusters[9] = {};     // row statistics without the sampler [cluster size]
  int attn_blocks_per_sm[4][16] = {};   // [kernel variant][tile size / 16]: resident blocks, -1 none
  cudaStream_t copy_stream = nullptr;   // ps_round_host: carries the target logits beside the draft step
  cudaEvent_t copy_done = nullptr;
  int* host_res = nullptr;              // ps_round_host: pinned host copy of the round's results
  void* st_hidden; int* st_tok; float* st_tlogits; float* st_dlogits; int* st_top; int* st_res;
  std::vector<int> len;     // committed positions per slot (host is the source of truth)
  std::vector<size_t> guards;   // offsets of the guard words in the workspace
  long long launches;
  std::string err;
  // optional stage timing (ps_profile): events recorded between stages
  bool prof = false;
  bool prof_launches = false;   // events per launch: chained stages stay chained (ps_profile(ctx, 2))
  std::vector<cudaEvent_t> prof_ev;
  std::vector<const char*> prof_name;   // name of the stage that ENDS at the event
  size_t prof_used = 0;
};

namespace ps {

// Clusters of nclu blocks of this kernel that are resident on the context's device at once, -1 for none (sizes above 8
// are an opt-in of the kernel, a per-device function attribute).  Asked once per context, kernel and size.  A
// cluster lies in one group of SMs, so not every SM can be filled: with one block an SM 33 clusters of 4 (132
// SMs), 15 of 8 (120), 7 of 16 (112); with four an SM 560 blocks in clusters of 4 or of 8, not 592.
template <class... Args>
int clusters_at_once(int& cache, void (*kern)(Args...), int threads, int nclu) {
  if (cache == 0) {
    cache = -1;
    if (nclu <= 8 || cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(nclu);
      cfg.blockDim = dim3(threads);
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = nclu; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) cache = n;
    }
    (void)cudaGetLastError();
  }
  return cache;
}

ps_status fail(ps_ctx* c, ps_status s, const std::string& what);
ps_status cuda_check(ps_ctx* c, cudaError_t e, const char* what);
// Records a timing event that closes stage `name` (no-op unless profiling is on).
void prof_mark(ps_ctx* c, cudaStream_t st, const char* name);

// ---- unfused kernels with fp32 activations (all dtypes, all shapes) -----------------------
ps_status plain_kv_append(ps_ctx* c, const SeqMap& sm, int rows, const void* hidden,
                          const int* tokens, cudaStream_t st);
ps_status plain_draft_step(ps_ctx* c, const SeqMap& sm, int B, const void* hidden_last,
                           const int* token_last, int top_n, int* top_ids, float* top_logit,
                           float* row_max, float* row_lse, float* logits_out, float* feat_out,
                           const SampleArgs* sa, cudaStream_t st);
// One pass over stored logits [M][V] (R rows per sequence): max, log-sum-exp, top-n and, with sa, the
// Gumbel-max token of every row (row_stats.cu).
ps_status launch_logit_stats(ps_ctx* c, const float* logits, int M, int V, int R, int top_n, int* top_ids,
                             float* top_logit, float* row_max, float* row_lse, const SampleArgs* sa, cudaStream_t st);
// bf16 matrix [rows][cols] row-major; boxes of box_rows x 64 columns, 128-byte swizzle, zeros
// outside the matrix.  False when the driver cannot encode tensor maps (tensor_map.cu).
constexpr int kMapCols = 64;
bool make_map(CUtensorMap* m, const void* base, size_t rows, size_t cols, int box_rows);
// bf16 matrix [rows][128] seen as [2][rows][64]; boxes of both halves of box_rows rows.
bool make_halves_map(CUtensorMap* m, const void* base, size_t rows, int box_rows);
// ---- fused bf16 kernels for small M ---------------------------------------------------------
bool fused_supported(ps_ctx* c, int M);
int fused_kv_rows(ps_ctx* c);     // most rows per pass of fused_kv_append (0: not available)
int append_pass_rows(const ps_config& g, int n_sm, int total, int most);   // rows of an append's passes, at most `most`
ps_status fused_kv_append(ps_ctx* c, const SeqMap& sm, int rows, const void* hidden, const int* tokens,
                          cudaStream_t st);
// RoPE on the k half of fp32 kv rows [0, rows) and the store of k and v into the bf16 cache rows.
ps_status launch_rope_store_kv(ps_ctx* c, const SeqMap& sm, int rows, const float* kv, cudaStream_t st);
int fused_row_limit(ps_ctx* c);   // most rows fused_supported() takes for this context (0: none)
size_t fused_scratch_bytes(const ps_config& g);
cudaError_t fused_init(ps_ctx* c, cudaStream_t st);   // zeroes the fused path's counters
void fused_release(ps_ctx* c);   // frees what the fused path holds on the host
ps_status fused_debug_buffer(ps_ctx* c, const char* name, void** ptr, size_t* bytes);
ps_status launch_rope_table(ps_ctx* c, cudaStream_t st);
// Test kernel: a bounded barrier wait that runs out after `limit_cycles` and raises the status word.
ps_status launch_wait_expires(ps_ctx* c, long long limit_cycles, cudaStream_t st);
ps_status launch_late_copy(ps_ctx* c, uint32_t* dst, const uint32_t* src, size_t n, long long delay_ns, cudaStream_t st);
ps_status launch_attn_split(ps_ctx* c, const SeqMap& sm, int B, const float* qkv, float* att_ml,
                            float* att_o, unsigned* tickets, __nv_bfloat16* out_hi,
                            __nv_bfloat16* out_lo, cudaStream_t st);
ps_status fused_draft_step(ps_ctx* c, const SeqMap& sm, int B, const void* hidden_last,
                           const int* token_last, int top_n, int* top_ids, float* top_logit,
                           float* row_max, float* row_lse, float* logits_out, float* feat_out,
                           const SampleArgs* sa, cudaStream_t st);
ps_status launch_verify(ps_ctx* c, int B, int n_draft, int n_target, const int* draft_tokens,
                        const float* draft_logits, const float* target_logits, float temperature,
                        uint64_t seed, uint64_t offset, int* accept_len, int* out_tokens,
                        int* n_out, cudaStream_t st);
ps_status launch_verify_tree(ps_ctx* c, int B, int n_nodes, const int* parent, const int* tokens,
                             const float* draft_logits, const float* target_logits, float temperature,
                             uint64_t seed, uint64_t offset, int* accept_len, int* out_tokens, int* n_out,
                             int* path, int* max_depth_out, cudaStream_t st);
ps_status launch_build_tree(ps_ctx* c, int B, int n_nodes, const int* parent, const int* rank, const int* top_ids,
                            int top_n, const int* sampled_ids, int* tokens, cudaStream_t st);
ps_status launch_kv_copy(ps_ctx* c, int slot, int len, void* K, void* V, bool to_cache,
                         cudaStream_t st);
}  // namespace ps
