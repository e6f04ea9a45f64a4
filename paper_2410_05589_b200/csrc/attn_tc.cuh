// Interface of the tensor-memory attention (attn_tc.cu).
#pragma once
#include "ps_internal.cuh"

namespace ps {
namespace atc {

constexpr int kD = 128;          // head dimension
constexpr int kNewRows = 16;     // rows kept per sequence (or bundle of them) and kv head for the step's new keys / values
constexpr int kMaxRows = 32;     // query rows of a kv head's group (heads of the group x rows per sequence)

// Query rows of a kv head's group padded to a multiple of 8 (0: the kernel does not take the shape).
inline int padded_rows(const ps_config& g) {
  const int rows = (g.n_heads / g.n_kv_heads) * (g.k_masks + 1);
  return g.head_dim == kD && rows <= kMaxRows ? (rows + 7) / 8 * 8 : 0;
}

// Whether a batch has enough keys for this kernel: it reads a kv head's keys once for all query heads
// and hides everything behind the stream, but costs a launch more and the way through its warps'
// barriers, where k_attn_mma's blocks, one per query head and key split, are through at once.  What
// separates the two is the key tiles of all query heads for every SM (884 whole steps, 1 to 64 heads, 1 to
// 16 rows, contexts of 16 to 4000): with up to 16 query rows a kv head 6 of them, with more (a ring of five
// slots, scores of 24 or 32 rows a tile) 16.  Llama-3-8B shape, 4 x 512 keys, 5 rows: 40 -> 24 us.
// The groups of the training layout, which this kernel takes several to a pair, are counted one by one all the same:
// of 168 calls (3 to 128 groups of 1 to 9 rows, 6 to 40 heads, contexts of 100 to 1500) those beyond the line are up to twice as
// long with the other kernel and 5% shorter at most (128 groups of 9 rows, which are not bundled; bundled ones
// 2%), and those short of it 5% longer at most.
inline bool worth_it(const ps_config& g, const SeqMap& sm, int B, int n_sm) {
  long long tiles = 0;
  for (int b = 0; b < B; ++b) tiles += std::max(1, (sm.len[b] + 127) / 128);
  return tiles * g.n_heads >= (long long)(padded_rows(g) <= 16 ? 6 : 16) * n_sm;
}

struct Buffers {
  __nv_bfloat16* q;      // [pairs][hi, lo][NR][128] rotated, scaled query rows (pair = sequence or bundle x kv head)
  __nv_bfloat16* kv_new; // [pairs][k, v][kNewRows][128] the step's new rows, rounded as a cache row is
  float* part_o;         // [2 CTAs' segments][NR][128] partial outputs
  float2* part_ml;       // [2 CTAs' segments][NR] their (reference, sum)
};
struct CacheMaps { CUtensorMap m[2][4]; };   // K and V slabs: boxes of 32, 64, 96 and 128 rows
struct Maps { CacheMaps cache; CUtensorMap q, kv_new, q_bundle; };

size_t bytes(const ps_config& g);                 // of the buffers; 0 when padded_rows() is 0
Buffers carve(const ps_config& g, char* base);
bool build_maps(const ps_ctx* c, const Buffers& b, Maps* m);
// qkv: float [B * R][Hq + 2 Hkv] before RoPE; merged output planes [B * R][n_heads * 128].
// tickets: [B][n_heads], zero between calls.
ps_status launch(ps_ctx* c, const SeqMap& sm, int B, const float* qkv, const Buffers& b, const Maps& m,
                 unsigned* tickets, __nv_bfloat16* out_hi, __nv_bfloat16* out_lo, cudaStream_t st);

}  // namespace atc
}  // namespace ps
