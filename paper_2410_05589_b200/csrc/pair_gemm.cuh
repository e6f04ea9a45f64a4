// Interface of the CTA-pair GEMM (pair_gemm.cu): Y[m][n] = sum_k X[m][k] W[n][k] for more than 16
// activation rows, and of the kernels that finish its split tiles.
#pragma once
#include <cuda.h>

#include "ps_internal.cuh"

namespace ps {
namespace pg {

constexpr int kMaxNp = 256;       // activation rows of a tile (the widest N a tcgen05.mma takes)
constexpr int kNpStep = 32;       // rows are padded to a multiple of this (16 rows per CTA of the pair)
constexpr int kMaxNormWidth = 32768;   // features of a row that launch_row_norm takes
constexpr int kMaxSplit = 16;     // k blocks a shared tile is dealt in

// How a stage's tiles are dealt to the CTA pairs; computed on the host, read by the GEMM and by
// the kernels that add up the partial tiles.  A tile is TW = 256 * wt weight rows times Np
// activation rows.  Tile t = w * n_rt + rt (weight tile w, row tile rt), so that pairs working
// side by side share weights.  Tiles [0, n_dp) go whole, one per pair and wave; the k range of
// each of the `rem` tiles behind them is cut into `split` blocks and the S = rem * split blocks
// are dealt to the first Pe pairs as contiguous runs, so that the last wave keeps every pair busy.
// A pair that holds part of a tile's k range is its contributor number j (in k order) and
// leaves its sums in a slot.  Slots are as large as a tile: one for every whole tile that goes
// through them, then one for every (shared tile, contributor), in the order of the runs, at
// shared tile + pair (from one to the next the tile, the pair or both go up by one, so these
// numbers are distinct and below rem + Pe).  A tile's contributors lie one behind the other.
struct Plan {
  int M, Np, n_rt;          // activation rows, rows per row tile, row tiles
  int wt, tiles_w;          // 128-row sub-tiles per CTA; weight tiles over all matrices
  int comb;                 // hi and lo planes are one MMA operand of 2 Np columns
  int KB;                   // k-blocks of 64 columns
  int T, n_dp, rem, split, S, Pe;
  int slot_t0;              // first tile that has slots
  int shared;               // some tile has more than one contributor
  int n_mats, mat_tiles[3], mat_rows[3], mat_off[3];
};

__host__ __device__ inline int run_owner(const Plan& p, int x) { return ((x + 1) * p.Pe - 1) / p.S; }
__host__ __device__ inline int run_begin(const Plan& p, int c) { return p.S * c / p.Pe; }
// Contributors of tile t.
__host__ __device__ inline int tile_contributors(const Plan& p, int t) {
  if (t < p.n_dp) return 1;
  const int x = (t - p.n_dp) * p.split;
  return run_owner(p, x + p.split - 1) - run_owner(p, x) + 1;
}
// Element offset of row mi of contributor j's slot of tile t: rows of TW floats.
__host__ __device__ inline size_t slot_row(const Plan& p, int j, int t, int mi) {
  int s = t - p.slot_t0 + j;
  if (t >= p.n_dp && p.split > 1) s += run_owner(p, (t - p.n_dp) * p.split);   // (else one pair a tile: its number)
  return ((size_t)s * p.Np + mi) * (size_t)(256 * p.wt);
}
// Tiles the slots must hold.
__host__ __device__ inline int slot_tiles(const Plan& p) { return p.T - p.slot_t0 + (p.split > 1 ? p.Pe - 1 : 0); }

enum Mode {
  MODE_RAW = 0,      // every tile's sums go to slots; a row kernel finishes them
  MODE_STORE = 1,    // whole tiles go to out[m][n], shared ones to slots
  MODE_SWIGLU = 2    // the CTA's two sub-tiles are gate and up rows: silu(g) * u as hi/lo planes
};

struct Args {
  Plan p;
  int planes;                     // 2: hi and lo planes of the activations, 1: they are exact bf16
  float* part;                    // slots
  float* out; int ldo;            // MODE_STORE
  __nv_bfloat16 *hi, *lo; int ld_plane;   // MODE_SWIGLU
  int* status;
};

// Tensor maps of a plane with boxes of 16, 32, ... rows: Np / 2 of them, or Np where the planes are one operand.
struct PlaneMaps { CUtensorMap m[kMaxNp / kNpStep]; };

struct Weights { const CUtensorMap* map[3]; int rows[3]; int n_mats; bool zip; };

int smem_bytes();   // shared memory of a block
// Deals the weights over K columns; `part_floats`: capacity of the slots.
Plan make_plan(int M, const Weights& w, int K, int planes, Mode mode, size_t part_floats, int n_sm);
ps_status launch_gemm(ps_ctx* c, const Weights& w, const PlaneMaps& hi, const PlaneMaps& lo, Args& a, Mode mode,
                      cudaStream_t st);
// Adds the slots of the shared tiles of a MODE_STORE / MODE_SWIGLU stage and stores the result as the
// GEMM stores its whole tiles (nothing to do when no tile is shared).
ps_status launch_finish_shared(ps_ctx* c, const Args& a, Mode mode, cudaStream_t st);
// Row m of a MODE_RAW stage with H features: x = sum of slots + bias + res (out, optional), and the
// hi/lo planes of x * rsqrt(mean(x^2) + eps) * gain.
ps_status launch_row_norm(ps_ctx* c, const Args& a, int H, const __nv_bfloat16* bias, const float* res,
                          const __nv_bfloat16* gain, float* out, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t st);

}  // namespace pg
}  // namespace ps
