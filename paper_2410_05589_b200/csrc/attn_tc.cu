// Attention of a draft step on tcgen05, for batches whose keys and values are worth streaming at
// full HBM rate (Sec. 4.1: the k+1 rows of a sequence see the cached real positions and the new
// rows up to themselves).
//
// What bounds it: the K/V stream.  A persistent CTA per SM walks a contiguous range of (sequence,
// kv head, 128-key tile) units; the K and V tiles come by tiled TMA into a ring of 32 KB slots
// (five or six: 160-192 KB in flight per SM) that nothing but the tensor cores reads:
//   S^T[key][row] = K[key][d] Q^T[d][row]     keys on the 128 lanes, the group's query rows (hi and
//                                             lo planes side by side, N = 2 NR) on the columns
//   O^T[d][row]  += V^T[d][key] P^T[key][row] channels on the lanes; V is read MN-major, as cached
// Eight warps turn a tile's scores into probabilities, one key per thread: no reduction over the
// keys is needed, because the exponentials are taken against a reference score per row (that of
// the first key of the segment) instead of the running maximum; only when a score exceeds it by
// 2^64 are the sums so far rescaled.  The probabilities are written to shared memory as bf16 hi + lo
// planes, a key's rows side by side (MN-major), so that a thread stores 8 or 16 bytes at a time.  Four
// more warps read a finished segment's O^T back while the next one runs.  All heads that share a kv head are
// rows of one product, so its keys and values are read once; so are, up to 16 rows, the sequences of one
// slot in the training layout.
// Rows of a pair whose tiles are dealt to several CTAs: partial results, merged in CTA order by the
// last of them to finish.
// A small kernel ahead (k_attn_prep) rotates and splits the query rows and rounds the new k / v
// rows as the cache would; the ring is filled with cached tiles while it runs.
// Measured (attention alone, with the small kernel) against mma.sync blocks that stage a tile,
// synchronise and compute: 33B shape, 16 sequences of 1024-4096 keys, 9 rows: 343 -> 210 us (973 MB:
// 4.8 TB/s of K/V in the main kernel); 13B shape, 64 x 256-2048 keys, 9 rows: 459 -> 332 us (1.5 GB); 16
// sequences, 5 rows: 94 -> 82 us; 128 training groups of 300-428 keys: 273 -> 198 us.  Then, by the vector
// stores and by warps that no longer meet at a barrier in every step (both builds in turn on one GPU, events between the
// stages): 64 sequences 393 -> 369 us, 33B shape 235 and 235, 16 sequences of 5 rows 95 -> 93; by three groups a
// pair, 128 training groups 241 -> 134 us.  (The clock is what the power limit leaves: a call by itself has 334 us for the 64
// sequences and 192 for the 33B shape.)  What was worth
// most after the first version: one TMA instruction per tile (the producer thread issued sixteen:
// 351 -> 318 us on the 64-sequence case, 282 -> 179 on the groups), two MMA issuers, eight softmax
// warps.  Putting the new rows into the last cached tile was slower (more, smaller boxes).
#include <cfloat>

#include "attn_tc.cuh"
#include "umma_gemm.cuh"

namespace ps {
namespace atc {
namespace {

using umma::fence_after_sync;
using umma::fence_before_sync;
using umma::mbar_arrive;
using umma::mbar_arrive_expect_tx;
using umma::mbar_init;
using umma::mbar_wait;
using umma::smem_desc;
using umma::smem_u32;

constexpr int kTile = 128;                 // keys of a unit
constexpr int kSlotBytes = kTile * kD * 2; // a K or V tile
constexpr int kBoxRows = 32;               // a ragged tile is fetched up to a multiple of it
constexpr int kSoftWarps = 8;              // two per lane quadrant, half of the rows each
constexpr int kThreads = 96 + 32 * (kSoftWarps + 4);   // producer, two MMA issuers, softmax, 4 epilogue warps
constexpr float kSlack = 64.f;             // a score this far above the reference (log2) forces a rescale
constexpr float kNoRef = -1e30f;           // reference of a row that has seen no key yet

__host__ __device__ constexpr int op_bytes(int NR) { return 2 * NR * kD * 2; }   // Q or P planes of one buffer
__host__ __device__ constexpr int n_slots(int NR) { return NR <= 16 ? 6 : 5; }
__host__ __device__ constexpr int tmem_cols(int NR) { return NR <= 8 ? 64 : (NR <= 16 ? 128 : 256); }

template <int NR>
struct Ctl {
  uint64_t full[6], empty[6];              // ring slots
  uint64_t q_full[2], q_empty[2];          // query planes, by segment
  uint64_t s_full[2], s_empty[2];          // scores, by step
  uint64_t p_full[2], p_empty[2];          // probabilities, by step
  uint64_t o_full[2], o_empty[2];          // outputs, by segment
  uint64_t l_full[2];                      // references and sums, by segment
  uint64_t checked[2][2];                  // by half of the rows and step: its four warps have looked for outgrown scores
  uint64_t soft[2];                        // by half: its four warps have come this far
  uint32_t tmem_base;
  int abort_flag, is_last;
  int outgrown[2][2];                      // by half and step: some score has outgrown its reference
  int sees[NR];                            // what a row sees, see the softmax warps
  float ref[2][NR];
  float sum[2][4][NR];                     // per lane quadrant; new maxima while a segment is under way
};
template <int NR>
constexpr int smem_bytes() { return n_slots(NR) * kSlotBytes + 4 * op_bytes(NR) + (int)sizeof(Ctl<NR>) + 1024; }

// What a (sequence, kv head) pair is to the kernel: the query rows of the kv head's group.  Sequences that read
// the same cache rows (the groups of the training layout: one slot, each a position longer than the one before)
// go several to a pair, so that their common keys are read and multiplied once: `subs` of them, whose
// rows follow one another.  Sequence i of a pair sees len + i cached keys, where len is the first one's; the other
// cached ones and the new ones of other sequences have probability 0 to it, and values that fit_row() made finite (told
// apart in k_attn_tc, by the thread that issues the products, the attention of 128 groups of 300 keys took 30 us more).
struct Work {
  SeqMap sm;
  int off[PS_MAX_BATCH + 1];   // units before bundle b of `subs` sequences (over all its kv heads)
  int n_kv, group, R, max_ctx, n_heads;
  int subs, n_bundles;
};
__device__ __forceinline__ int units_of(int len) { return max(1, (len + kTile - 1) / kTile); }
__device__ __forceinline__ int unit_begin(int c, int U, int G) { return (int)((unsigned)U * (unsigned)c / (unsigned)G); }
__device__ __forceinline__ int unit_owner(int u, int U, int G) {
  return (int)(((unsigned)(u + 1) * (unsigned)G - 1u) / (unsigned)U);
}

// Walks a CTA's steps: the cached tiles of a segment (one pair's share of the range), then, where
// the segment holds the pair's last unit, the step of the new rows.
struct Walk {
  int u, u_end;                     // units left after the segment begin at u
  int b, hk, len, nu, t, t_end;     // the segment: bundle, kv head, its cached tiles [t, t_end)
  int cnt, len0;                    // the bundle's sequences; cached keys of the first one (len: of the last)
  bool tail, in_tail, first, ok, whole;
  int seg;
  __device__ void enter() {         // the segment that begins at tile t of (b, hk)
    ok = u < u_end;
    if (!ok) return;
    const int e = min(nu, t + u_end - u);
    u += e - t;
    tail = e == nu;
    whole = tail && t == 0;
    t_end = min(e, (len + kTile - 1) / kTile);
    in_tail = t >= t_end;
    first = true;
  }
  __device__ void sequence(const Work& w) {
    cnt = min(w.subs, w.sm.B - b * w.subs);
    len0 = w.sm.len[b * w.subs];
    len = len0 + cnt - 1;
    nu = units_of(len);
  }
  __device__ void start(const Work& w, int u0, int u1) {
    u = u0; u_end = u1; seg = 0;
    int lo = 0, hi = w.n_bundles - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (w.off[mid] <= u) lo = mid; else hi = mid - 1;
    }
    b = lo;
    sequence(w);
    const int r = u - w.off[b];
    hk = r / nu;
    t = r - hk * nu;
    enter();
  }
  __device__ void next_segment(const Work& w) {
    ++seg;
    t = 0;
    if (++hk == w.n_kv) {
      hk = 0;
      ++b;
      if (b < w.n_bundles) sequence(w);
    }
    enter();
  }
  __device__ bool last() const { return in_tail || (t + 1 == t_end && !tail); }
  __device__ bool last_of_cta() const { return u >= u_end && last(); }
  __device__ int keys(const Work& w) const { return in_tail ? cnt * w.R : min(kTile, len - t * kTile); }
  __device__ int rows(const Work& w) const { return cnt * w.group * w.R; }
  // rows of the step's box: the halves of its tile lie that many rows apart
  __device__ int box(const Work& w) const { return in_tail ? kNewRows : (keys(w) + kBoxRows - 1) & ~(kBoxRows - 1); }
  __device__ void next(const Work& w) {
    if (last()) { next_segment(w); return; }
    first = false;
    if (++t == t_end) in_tail = true;
  }
};

// One box of rows y.. of a [rows][128] matrix seen as [2][rows][64]: both 64-channel halves, one behind
// the other (the producer thread is bound by the instructions it issues, not by their size).
__device__ __forceinline__ void tma_load_rows(uint32_t dst, const CUtensorMap* map, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(map), "r"(0), "r"(y), "r"(0), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void split1(float x, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(x);
  l = __float2bfloat16_rn(x - __bfloat162float(h));
}
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4_async(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3])
               : "memory");
}
// The sums hi + lo of the NR rows of an accumulator of 2 NR columns, for this thread's lane.
template <int NR>
__device__ __forceinline__ void tmem_rows(uint32_t taddr, float (&v)[NR]) {
  uint32_t r[2 * NR / 16][16];
#pragma unroll
  for (int i = 0; i < 2 * NR / 16; ++i) tmem_ld16_async(taddr + 16 * i, r[i]);
  umma::tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < NR; ++i)
    v[i] = __uint_as_float(r[i / 16][i % 16]) + __uint_as_float(r[(NR + i) / 16][(NR + i) % 16]);
}
// V^T as the MMA's M side: channels contiguous (MN-major), 128-byte swizzle; 64-channel halves
// half_bytes apart, groups of 8 keys 1024 bytes apart.
__device__ __forceinline__ uint64_t vt_desc(uint32_t saddr, uint32_t half_bytes) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(half_bytes >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Probabilities as the MMA's N side: a key's 2 NR values (rows of the hi plane, then of the lo plane) contiguous
// (MN-major), 32-byte swizzle; 16 values at a time, the next 16 kAtomStride bytes on; groups of 8 keys 256 bytes
// apart.
constexpr int kAtomStride = kTile * 32;
__device__ __forceinline__ uint64_t p_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kAtomStride >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}
// Two values' hi and lo parts, packed.
__device__ __forceinline__ void split2(float x, float y, uint32_t& h, uint32_t& l) {
  const __nv_bfloat162 hv = __floats2bfloat162_rn(x, y);
  h = *reinterpret_cast<const uint32_t*>(&hv);
  const __nv_bfloat162 lv = __floats2bfloat162_rn(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xFFFF0000u));
  l = *reinterpret_cast<const uint32_t*>(&lv);
}
// Sums of MC values over the warp, halving the values a lane carries at each step: lane l ends with
// the sum of value l / (32 / MC).
template <int MC>
__device__ __forceinline__ float warp_sum_many(float (&v)[MC], int lane) {
#pragma unroll
  for (int n = MC, o = 16; n > 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float keep = up ? v[i + n / 2] : v[i], give = up ? v[i] : v[i + n / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  float t = v[0];
#pragma unroll
  for (int o = 16 / MC; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}
// Barrier of the 128 epilogue threads.
constexpr int kBarEpi = 1;
__device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool bar_any(int id, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, %2, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(id)
      : "memory");
  return r != 0;
}

// Query rows of a pair (rotated, scaled by log2(e) / sqrt(128), hi and lo planes, zero rows up to
// NR) and its new k (rotated) and v rows rounded to the cache's type.  Block: kPrepHeads kv heads of
// a sequence.  Bound by the read of q|k|v from L2; the rotation table is formed once per block.
constexpr int kPrepHeads = 4;
__global__ void __launch_bounds__(256) k_attn_prep(const __grid_constant__ Work w, const float* __restrict__ qkv, int ldq,
                                                   int Hq, int Hkv, const double* __restrict__ inv_freq, int NR,
                                                   __nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ kv) {
  __shared__ float cs[kMaxRowsPerSeq][kD / 2], sn[kMaxRowsPerSeq][kD / 2];
  const int b = blockIdx.y, h0 = blockIdx.x * kPrepHeads, nh = min(kPrepHeads, w.n_kv - h0), R = w.R, G = w.group;
  const int m0 = b * R, tid = threadIdx.x;
  const int u = b / w.subs, sub = b - u * w.subs;                    // its bundle, its place there
  const bool last_sub = sub == w.subs - 1 || b == w.sm.B - 1;        // the last one writes the zero rows behind it
  pdl_launch_dependents();
  for (int i = tid; i < R * (kD / 2); i += blockDim.x) {
    double ang = (double)(w.sm.len[b] + i / (kD / 2)) * inv_freq[i % (kD / 2)];
    ang -= 6.283185307179586476925 * rint(ang * 0.15915494309189533577);
    sincosf((float)ang, &sn[i / (kD / 2)][i % (kD / 2)], &cs[i / (kD / 2)][i % (kD / 2)]);
  }
  __syncthreads();
  pdl_wait();
  const float scale = rsqrtf((float)kD) * 1.4426950408889634f;
  struct alignas(8) B4 { __nv_bfloat16 v[4]; };
  // 16 threads per row: four channels i..i+3 of the lower half and their partners 64 above
  const int q_rows = last_sub ? NR - sub * G * R : G * R;
  const int n_q = nh * q_rows * 16;
  for (int it = tid; it < n_q; it += blockDim.x) {
    const int i = (it & 15) * 4, r = (it >> 4) % q_rows, hk = h0 + (it >> 4) / q_rows;
    B4 h0v{}, l0v{}, h1v{}, l1v{};
    if (r < G * R) {
      const int g = r / R, j = r - g * R;
      const float* src = qkv + (size_t)(m0 + j) * ldq + (hk * G + g) * kD + i;
      const float4 x = __ldcg(reinterpret_cast<const float4*>(src)), y = __ldcg(reinterpret_cast<const float4*>(src + kD / 2));
      const float xa[4] = {x.x, x.y, x.z, x.w}, ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float c = cs[j][i + e], s = sn[j][i + e];
        split1((xa[e] * c - ya[e] * s) * scale, h0v.v[e], l0v.v[e]);
        split1((ya[e] * c + xa[e] * s) * scale, h1v.v[e], l1v.v[e]);
      }
    }
    __nv_bfloat16* d = q + ((size_t)(u * w.n_kv + hk) * 2 * NR + sub * G * R + r) * kD + i;
    *reinterpret_cast<B4*>(d) = h0v;
    *reinterpret_cast<B4*>(d + kD / 2) = h1v;
    *reinterpret_cast<B4*>(d + (size_t)NR * kD) = l0v;
    *reinterpret_cast<B4*>(d + (size_t)NR * kD + kD / 2) = l1v;
  }
  const int kv_rows = last_sub ? kNewRows - sub * R : R;
  const int n_kv_items = nh * kv_rows * 16;
  for (int it = tid; it < n_kv_items; it += blockDim.x) {
    const int i = (it & 15) * 4, j = (it >> 4) % kv_rows, hk = h0 + (it >> 4) / kv_rows;
    B4 k0{}, k1{}, v0{}, v1{};
    if (j < R) {
      const float* src = qkv + (size_t)(m0 + j) * ldq + Hq + hk * kD + i;
      const float4 x = __ldcg(reinterpret_cast<const float4*>(src)), y = __ldcg(reinterpret_cast<const float4*>(src + kD / 2));
      const float4 a = __ldcg(reinterpret_cast<const float4*>(src + Hkv)),
                   c4 = __ldcg(reinterpret_cast<const float4*>(src + Hkv + kD / 2));
      const float xa[4] = {x.x, x.y, x.z, x.w}, ya[4] = {y.x, y.y, y.z, y.w}, va[4] = {a.x, a.y, a.z, a.w},
                  vb[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float c = cs[j][i + e], s = sn[j][i + e];
        k0.v[e] = __float2bfloat16_rn(xa[e] * c - ya[e] * s);
        k1.v[e] = __float2bfloat16_rn(ya[e] * c + xa[e] * s);
        v0.v[e] = __float2bfloat16_rn(va[e]);
        v1.v[e] = __float2bfloat16_rn(vb[e]);
      }
    }
    if (w.subs > 1) fit_row(k0, k1, v0, v1, 16);
    __nv_bfloat16* d = kv + ((size_t)(u * w.n_kv + hk) * 2 * kNewRows + sub * R + j) * kD + i;
    *reinterpret_cast<B4*>(d) = k0;
    *reinterpret_cast<B4*>(d + kD / 2) = k1;
    *reinterpret_cast<B4*>(d + (size_t)kNewRows * kD) = v0;
    *reinterpret_cast<B4*>(d + (size_t)kNewRows * kD + kD / 2) = v1;
  }
}

template <int NR>
__global__ void __launch_bounds__(kThreads, 1)
k_attn_tc(const __grid_constant__ CacheMaps t_c, const __grid_constant__ CUtensorMap t_q, const __grid_constant__ CUtensorMap t_new,
          const __grid_constant__ Work w, float* __restrict__ part_o, float2* __restrict__ part_ml, unsigned* tickets, __nv_bfloat16* __restrict__ out_hi,
          __nv_bfloat16* __restrict__ out_lo, int* status) {
  constexpr int N = 2 * NR, NS = n_slots(NR), kOp = op_bytes(NR);
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* ring_g = smem_raw + (base - raw);
  const uint32_t s_q = base + NS * kSlotBytes, s_p = s_q + 2 * kOp;
  Ctl<NR>& ctl = *reinterpret_cast<Ctl<NR>*>(ring_g + NS * kSlotBytes + 4 * kOp);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = gridDim.x, U = w.off[w.n_bundles];
  const int u0 = unit_begin(blockIdx.x, U, G), u1 = unit_begin(blockIdx.x + 1, U, G);
  volatile int* abort_flag = &ctl.abort_flag;

  if (tid == 0) {
    for (int i = 0; i < NS; ++i) { mbar_init(&ctl.full[i], 1); mbar_init(&ctl.empty[i], 1); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&ctl.q_full[i], 1); mbar_init(&ctl.q_empty[i], 1);
      mbar_init(&ctl.s_full[i], 1); mbar_init(&ctl.s_empty[i], kSoftWarps);
      mbar_init(&ctl.p_full[i], kSoftWarps); mbar_init(&ctl.p_empty[i], 1);
      mbar_init(&ctl.o_full[i], 1); mbar_init(&ctl.o_empty[i], 4);
      mbar_init(&ctl.l_full[i], kSoftWarps);
      for (int h = 0; h < 2; ++h) { mbar_init(&ctl.checked[h][i], kSoftWarps / 2); ctl.outgrown[h][i] = 0; }
      mbar_init(&ctl.soft[i], kSoftWarps / 2);
    }
    ctl.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    pdl_launch_dependents();
  }
  // A row sees new keys [first, last] of its bundle's and, of the cached ones, sub more than the first sequence
  // does: first | last << 8 | sub << 16 (rows past the last one see none of the new keys).
  if (tid >= kThreads - NR) {
    const int r = tid - (kThreads - NR), sub = r / (w.group * w.R);
    ctl.sees[r] = sub < w.subs ? sub * w.R | (sub * w.R + r % w.R) << 8 | sub << 16 : 1;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem_base)),
                 "r"(tmem_cols(NR))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *(volatile uint32_t*)&ctl.tmem_base, tmem_o = tmem + 2 * N;

  // Ring order of the loads, which is the order the MMAs use them in: K of step 0, then K of step
  // i + 1 and V of step i for every i.
  if (warp == 0) {
    if (lane == 0) {   // ---- TMA producer
      Walk wk, wv;
      wk.start(w, u0, u1);
      wv.start(w, u0, u1);
      int slot = 0, n_issued = 0;
      uint32_t use = 0;
      bool dep = false, alive = true;          // dep: the kernel before this one (the query and new rows) is complete
      auto load_q = [&](int b, int hk, int seg) {
        uint64_t* bar = &ctl.q_full[seg & 1];
        const uint32_t dst = s_q + (seg & 1) * kOp;
        mbar_arrive_expect_tx(bar, kOp);
        const int y = (b * w.n_kv + hk) * N;
        tma_load_rows(dst, &t_q, y, bar);
      };
      auto need_dep = [&]() {
        if (dep) return;
        pdl_wait();
        dep = true;
        Walk first;
        first.start(w, u0, u1);
        load_q(first.b, first.hk, 0);
      };
      // (Cached tiles are asked for before the wait: what stored them belongs to a call before this one or to
      // its append, and the first kernel of a step lets the others start only when that is complete.)
      auto load = [&](const Walk& x, int v) {
        if (n_issued >= NS || x.in_tail) need_dep();
        if (n_issued >= NS && !mbar_wait(&ctl.empty[slot], (use & 1) ^ 1, abort_flag)) { alive = false; return; }
        const uint32_t dst = base + slot * kSlotBytes;
        uint64_t* bar = &ctl.full[slot];
        const int rows = x.box(w);
        mbar_arrive_expect_tx(bar, rows * kD * 2);
        if (x.in_tail) tma_load_rows(dst, &t_new, ((x.b * w.n_kv + x.hk) * 2 + v) * kNewRows, bar);
        else tma_load_rows(dst, &t_c.m[v][rows / kBoxRows - 1], (w.sm.slot[x.b * w.subs] * w.n_kv + x.hk) * w.max_ctx + x.t * kTile, bar);
        ++n_issued;
        if (++slot == NS) { slot = 0; ++use; }
      };
      auto load_k = [&]() {
        if (wk.first && wk.seg > 0) {
          need_dep();
          if (!mbar_wait(&ctl.q_empty[wk.seg & 1], ((wk.seg >> 1) & 1) ^ 1, abort_flag)) { alive = false; return; }
          load_q(wk.b, wk.hk, wk.seg);
        }
        load(wk, 0);
        wk.next(w);
      };
      if (wk.ok) load_k();
      while (alive && wv.ok) {
        if (wk.ok) load_k();
        if (alive) { load(wv, 1); wv.next(w); }
      }
      if (alive && u0 < u1) need_dep();
    }
  } else if (warp == 1) {
    if (lane == 0) {   // ---- MMA issuer, scores (a thread issues about one MMA per 50-60 cycles: two of them keep up)
      Walk x;
      const uint32_t id = umma::idesc(N);
      // (descriptors hold addresses in units of 16 bytes: offsets are added to them)
      const uint64_t dk0 = smem_desc(base), dq0 = smem_desc(s_q);
      x.start(w, u0, u1);
      int slot = 0;            // of this step's K: ring position 0, then 2 i - 1
      uint32_t use = 0;
      for (int i = 0; x.ok; ++i) {
        const int buf = i & 1, qb = x.seg & 1;
        // In a ring of odd length the slot's use before this one was a V tile, whose arrival the other
        // issuer waits for.  A wait by parity cannot tell a use from the one two before it, so it must not
        // begin until the V tile has been consumed (which the arrival of this K implies: nothing is
        // lost).  In a ring of even length a slot's uses are all waited for by one issuer, but for the
        // first (K of step 0) and the last (V of the last step), whose neighbours have long landed.
        if ((x.first && !mbar_wait(&ctl.q_full[qb], (x.seg >> 1) & 1, abort_flag)) ||
            !mbar_wait(&ctl.s_empty[buf], ((i >> 1) & 1) ^ 1, abort_flag) ||
            ((NS & 1) && use > 0 && !mbar_wait(&ctl.empty[slot], (use - 1) & 1, abort_flag)) ||
            !mbar_wait(&ctl.full[slot], use & 1, abort_flag)) break;
        fence_after_sync();
        const uint64_t da = dk0 + (uint64_t)(slot * (kSlotBytes / 16)), db = dq0 + (uint64_t)(qb * (kOp / 16));
        const uint64_t half = (uint64_t)(x.box(w) * 128 / 16);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks)
          umma::mma_f16(tmem + buf * N, da + (ks >> 2) * half + (ks & 3) * 2,
                        db + (ks >> 2) * (kOp / 32) + (ks & 3) * 2, id, ks > 0);
        umma::mma_commit(&ctl.s_full[buf]);
        umma::mma_commit(&ctl.empty[slot]);
        if (x.last()) umma::mma_commit(&ctl.q_empty[qb]);
        slot += i == 0 ? 1 : 2;
        if (slot >= NS) { slot -= NS; ++use; }
        x.next(w);
      }
    }
  } else if (warp == 2) {
    if (lane == 0) {   // ---- MMA issuer, outputs
      Walk x;
      const uint32_t id = umma::idesc(N) | (1u << 15) | (1u << 16);   // (both operands MN-major)
      const uint64_t dv0 = vt_desc(base, 0), dp0 = p_desc(s_p);
      x.start(w, u0, u1);
      int slot = x.ok && x.last_of_cta() ? 1 : 2;   // of this step's V: ring position 2 i + 2, of the very last one 2 i + 1
      uint32_t use = 0;
      for (int i = 0; x.ok; ++i) {
        const int buf = i & 1, ob = x.seg & 1;
        if ((x.first && !mbar_wait(&ctl.o_empty[ob], ((x.seg >> 1) & 1) ^ 1, abort_flag)) ||
            !mbar_wait(&ctl.full[slot], use & 1, abort_flag) ||
            !mbar_wait(&ctl.p_full[buf], (i >> 1) & 1, abort_flag)) break;
        fence_after_sync();
        const uint64_t da = dv0 + (uint64_t)(slot * (kSlotBytes / 16)) + ((uint64_t)(x.box(w) * 128 / 16) << 16),
                       db = dp0 + (uint64_t)(buf * (kOp / 16));
        const int n_ks = (x.keys(w) + 15) >> 4;
        const uint32_t d = tmem_o + ob * N, acc = x.first ? 0u : 1u;
        if (n_ks == kTile / 16) {
#pragma unroll
          for (int ks = 0; ks < kTile / 16; ++ks)
            umma::mma_f16(d, da + ks * (2048 / 16), db + ks * (512 / 16), id, ks > 0 ? 1u : acc);
        } else {
#pragma unroll 1
          for (int ks = 0; ks < n_ks; ++ks)
            umma::mma_f16(d, da + ks * (2048 / 16), db + ks * (512 / 16), id, ks > 0 ? 1u : acc);
        }
        umma::mma_commit(&ctl.p_empty[buf]);
        umma::mma_commit(&ctl.empty[slot]);
        if (x.last()) umma::mma_commit(&ctl.o_full[ob]);
        x.next(w);
        slot += x.ok && x.last_of_cta() ? 1 : 2;
        if (slot >= NS) { slot -= NS; ++use; }
      }
    }
  } else if (warp < 3 + kSoftWarps) {
    // ---- softmax: thread = key of the tile, half of the rows.  The four warps of a half share their rows'
    // references, so they meet in every step; they do so a few hundred cycles after each has said
    // whether one of its scores has outgrown its reference, and find the others' words there.  (A barrier at that
    // point cost 500-800 cycles a step, more than the arithmetic: below the clock that the power limit
    // leaves, a step's cycles are what bounds the kernel.)  All these waits are bounded.
    constexpr int NH = NR / 2, kSoft = 32 * kSoftWarps, kPiece = NH % 8 == 0 ? 8 : 4;
    const int q = warp & 3, key = 32 * q + lane, half = (warp - 3) >> 2, r0 = half * NH;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    // this thread's key in the probabilities; the 16-byte halves of its 32 change places every four keys
    unsigned char* const p_base = ring_g + NS * kSlotBytes + 2 * kOp + key * 32;
    const int flip = ((key >> 2) & 1) << 4;
    uint32_t soft_phase = 0;
    auto meet = [&]() {   // the half's warps; what each wrote to shared memory is visible to the others
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.soft[half]);
      const bool ok = mbar_wait(&ctl.soft[half], soft_phase, abort_flag);
      soft_phase ^= 1;
      return (bool)__all_sync(0xffffffffu, ok);
    };
    Walk x;
    x.start(w, u0, u1);
    float ref[NH], l[NH];
    for (int i = 0; x.ok; ++i) {
      const int buf = i & 1, sb = x.seg & 1, n = x.keys(w);
      const bool last = x.last();
      bool ok = mbar_wait(&ctl.s_full[buf], (i >> 1) & 1, abort_flag);
      if (x.first) ok = mbar_wait(&ctl.o_empty[sb], ((x.seg >> 1) & 1) ^ 1, abort_flag) && ok;
      if (!__all_sync(0xffffffffu, ok)) break;
      fence_after_sync();
      float s[NH];
      {
        uint32_t h[NH / 4][4], lo[NH / 4][4];
        const uint32_t at = tmem + lane_off + buf * N + r0;
#pragma unroll
        for (int c = 0; c < NH / 4; ++c) { tmem_ld4_async(at + 4 * c, h[c]); tmem_ld4_async(at + NR + 4 * c, lo[c]); }
        umma::tmem_ld_wait();
#pragma unroll
        for (int r = 0; r < NH; ++r) s[r] = __uint_as_float(h[r / 4][r % 4]) + __uint_as_float(lo[r / 4][r % 4]);
      }
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.s_empty[buf]);   // read back: the next scores may be formed
      const int n0 = x.len0 - x.t * kTile;   // cached keys of the tile that the bundle's first sequence sees
      if (x.in_tail) {   // new keys of other sequences, or that a row does not see yet
#pragma unroll
        for (int r = 0; r < NH; ++r) {
          const int v = ctl.sees[r0 + r];
          if (key < (v & 255) || key > (v >> 8 & 255)) s[r] = -INFINITY;
        }
      } else if (n0 < kTile) {   // keys past the end
#pragma unroll
        for (int r = 0; r < NH; ++r)
          if (key >= n0 + (ctl.sees[r0 + r] >> 16)) s[r] = -INFINITY;
      }
      if (x.first) {   // the references: the scores of the segment's first key (a row that does not see it: below all)
        if (key == 0) {
#pragma unroll
          for (int r = 0; r < NH; ++r) ctl.ref[sb][r0 + r] = fmaxf(s[r], kNoRef);
        }
        if (!meet()) break;
#pragma unroll
        for (int r = 0; r < NH; ++r) { ref[r] = ctl.ref[sb][r0 + r]; l[r] = 0.f; }
      }
      float top = -INFINITY;
#pragma unroll
      for (int r = 0; r < NH; ++r) top = fmaxf(top, s[r] - ref[r]);
      const bool mine = __any_sync(0xffffffffu, top > kSlack);
      if (lane == 0) {
        if (mine) *(volatile int*)&ctl.outgrown[half][buf] = 1;
        mbar_arrive(&ctl.checked[half][buf]);
      }
      // (With 12 or 16 rows a thread there is no room for scores and probabilities side by side.)
      constexpr bool kAhead = NH <= 8;
      float p[NH];
      if constexpr (kAhead) {
#pragma unroll
        for (int r = 0; r < NH; ++r) p[r] = ex2(s[r] - ref[r]);   // (0 for what is masked)
      }
      if (!__all_sync(0xffffffffu, mbar_wait(&ctl.checked[half][buf], (i >> 1) & 1, abort_flag))) break;
      if (*(volatile int*)&ctl.outgrown[half][buf]) {
        // Rare: some score lies far above its reference.  New references; the sums and the outputs
        // so far are rescaled once the MMAs that form them have completed.
        for (int r = 0; r < NH; ++r) {
          float m = -INFINITY;
#pragma unroll
          for (int e = 0; e < NH; ++e) m = e == r ? s[e] : m;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
          if (lane == 0) ctl.sum[sb][q][r0 + r] = m;
        }
        if (!meet()) break;
        if (key == 0) *(volatile int*)&ctl.outgrown[half][buf] = 0;   // (everyone has read it)
        const auto& mx = ctl.sum[sb];
        float f[NH];
#pragma unroll
        for (int r = 0; r < NH; ++r) {
          const int rr = r0 + r;
          const float m = fmaxf(fmaxf(fmaxf(mx[0][rr], mx[1][rr]), fmaxf(mx[2][rr], mx[3][rr])), ref[r]);
          f[r] = ex2(ref[r] - m);
          l[r] *= f[r];
          ref[r] = m;
          if constexpr (kAhead) p[r] = ex2(s[r] - m);
          if (key == 0) ctl.ref[sb][rr] = m;
        }
        if (last && !meet()) break;   // (the sums are written below)
        if (!x.first) {
          if (!__all_sync(0xffffffffu, mbar_wait(&ctl.p_empty[(i - 1) & 1], ((i - 1) >> 1) & 1, abort_flag))) break;
          fence_after_sync();
#pragma unroll
          for (int c = 0; c < 2 * NH / 4; ++c) {   // this warp's columns: hi, then lo
            uint32_t v[4];
            const uint32_t at = tmem_o + lane_off + sb * N + (c < NH / 4 ? 0 : NR) + r0 + 4 * (c % (NH / 4));
            tmem_ld4_async(at, v);
            umma::tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * f[4 * (c % (NH / 4)) + e]);
            tmem_st4(at, v);
          }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          fence_before_sync();
        }
      }
      // ---- probabilities as hi/lo planes, the key's values side by side
#pragma unroll
      for (int r = 0; r < NH; ++r) {
        if constexpr (!kAhead) p[r] = ex2(s[r] - ref[r]);
        l[r] += p[r];
      }
      if (i >= 2) mbar_wait(&ctl.p_empty[buf], ((i >> 1) & 1) ^ 1, abort_flag);
      const int n16 = (n + 15) & ~15;
      if (key < n16) {
        unsigned char* const pp = p_base + buf * kOp;
#pragma unroll
        for (int c = 0; c < NH; c += kPiece) {
          uint32_t h[kPiece / 2], lo[kPiece / 2];
#pragma unroll
          for (int e = 0; e < kPiece / 2; ++e) split2(p[c + 2 * e], p[c + 2 * e + 1], h[e], lo[e]);
          // value v of the key: 16 values to an atom, 8 to a 16-byte half of its 32 bytes
          const int vh = r0 + c, vl = NR + vh;
          unsigned char* const ph = pp + (vh >> 4) * kAtomStride + ((((vh >> 3) & 1) << 4) ^ flip) + (vh & 7) * 2;
          unsigned char* const pl = pp + (vl >> 4) * kAtomStride + ((((vl >> 3) & 1) << 4) ^ flip) + (vl & 7) * 2;
          if constexpr (kPiece == 8) {
            *reinterpret_cast<uint4*>(ph) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(pl) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          } else {
            *reinterpret_cast<uint2*>(ph) = make_uint2(h[0], h[1]);
            *reinterpret_cast<uint2*>(pl) = make_uint2(lo[0], lo[1]);
          }
        }
      }
      if (n16 > n && !x.in_tail) {
        // rows of V between the tile's end and the next multiple of 16 meet probabilities of zero: they
        // must be finite
        const int half_bytes = x.box(w) * 128;
        const int pos = x.last_of_cta() ? 2 * i + 1 : 2 * i + 2, vs = pos % NS;   // ring position of this V
        mbar_wait(&ctl.full[vs], (pos / NS) & 1, abort_flag);
        for (int e = tid - 96; e < (n16 - n) * 16; e += kSoft) {
          const int row = n + (e >> 4), c16 = e & 15;
          *reinterpret_cast<uint4*>(ring_g + vs * kSlotBytes + (c16 >> 3) * half_bytes + row * 128 + (c16 & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.p_full[buf]);
      if (last) {
        constexpr int NP = NH <= 4 ? 4 : NH <= 8 ? 8 : 16;   // (a lane ends with the sum of row lane / (32 / NP))
        float v[NP];
#pragma unroll
        for (int r = 0; r < NP; ++r) v[r] = r < NH ? l[r < NH ? r : 0] : 0.f;
        const float t = warp_sum_many<NP>(v, lane);
        const int r = lane / (32 / NP);
        if (lane % (32 / NP) == 0 && r < NH) ctl.sum[sb][q][r0 + r] = t;
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl.l_full[sb]);
      }
      x.next(w);
    }
    fence_before_sync();
  } else {
    // ---- epilogue: thread = output channel
    const int q = warp & 3, d = 32 * q + lane;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    Walk x;
    for (x.start(w, u0, u1); x.ok;) {
      const int sb = x.seg & 1, rows = x.rows(w);
      const bool ok = mbar_wait(&ctl.o_full[sb], (x.seg >> 1) & 1, abort_flag) &&
                      mbar_wait(&ctl.l_full[sb], (x.seg >> 1) & 1, abort_flag);
      if (bar_any(kBarEpi, !ok)) break;
      fence_after_sync();
      float o[NR], l[NR];
      tmem_rows<NR>(tmem_o + lane_off + sb * N, o);
#pragma unroll
      for (int r = 0; r < NR; ++r)
        l[r] = (ctl.sum[sb][0][r] + ctl.sum[sb][1][r]) + (ctl.sum[sb][2][r] + ctl.sum[sb][3][r]);
      const float my_ref = d < NR ? ctl.ref[sb][d] : 0.f;
      float my_sum = 0.f;
      if (d < NR) my_sum = (ctl.sum[sb][0][d] + ctl.sum[sb][1][d]) + (ctl.sum[sb][2][d] + ctl.sum[sb][3][d]);
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.o_empty[sb]);
      bool write = x.whole;
      if (!x.whole) {
        const int a = w.off[x.b] + x.hk * x.nu;                     // the pair's first unit
        const int mine = blockIdx.x * 2 + (u0 >= a ? 0 : 1);        // its first segment, or its last
        float* po = part_o + (size_t)mine * NR * kD + d;
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (r < rows) po[r * kD] = o[r];
        if (d < NR) part_ml[mine * NR + d] = make_float2(my_ref, my_sum);
        bar_sync(kBarEpi);
        const int c0 = unit_owner(a, U, G), c1 = unit_owner(a + x.nu - 1, U, G);
        if (d == 0) {
          __threadfence();
          unsigned* tk = tickets + x.b * w.n_heads + x.hk;
          const int is_last = atomicAdd(tk, 1u) == (unsigned)(c1 - c0);
          if (is_last) { *tk = 0u; __threadfence(); }
          ctl.is_last = is_last;
        }
        bar_sync(kBarEpi);
        write = ctl.is_last != 0;
        if (write) {   // all contributors in CTA order
          float m[NR];
#pragma unroll
          for (int r = 0; r < NR; ++r) { m[r] = -FLT_MAX; l[r] = o[r] = 0.f; }
          for (int c = c0; c <= c1; ++c) {
            const int sl = c * 2 + (unit_begin(c, U, G) >= a ? 0 : 1);
            float ov[NR];
            float2 ml[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              ov[r] = r < rows ? __ldcg(part_o + ((size_t)sl * NR + r) * kD + d) : 0.f;
              ml[r] = r < rows ? __ldcg(part_ml + sl * NR + r) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              const float mm = fmaxf(m[r], ml[r].x), f0 = ex2(m[r] - mm), f1 = ex2(ml[r].x - mm);
              l[r] = l[r] * f0 + ml[r].y * f1;
              o[r] = o[r] * f0 + ov[r] * f1;
              m[r] = mm;
            }
          }
        }
        bar_sync(kBarEpi);   // everyone has read the flag
      }
      if (write) {
        int m0 = x.b * w.subs * w.R;
        int j = 0, g = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          if (r < rows) {
            const size_t at = (size_t)(m0 + j) * w.n_heads * kD + (size_t)(x.hk * w.group + g) * kD + d;
            split1(o[r] / l[r], out_hi[at], out_lo[at]);
          }
          if (++j == w.R) {
            j = 0;
            if (++g == w.group) { g = 0; m0 += w.R; }
          }
        }
      }
      x.next_segment(w);
    }
    fence_before_sync();
  }

  __syncthreads();
  if (ctl.abort_flag) {
    // let copies and MMAs that are still in flight finish before shared and tensor memory go
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    if (tid == 0) atomicOr(status, kStatTimeout);
    __syncthreads();
  }
  if (warp == 1) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols(NR)) : "memory");
  }
}

size_t take(size_t& off, size_t n) {
  const size_t at = off;
  off += (n + 255) & ~(size_t)255;
  return at;
}

// Sequences of one slot that share a pair's query rows, and their rows padded.  (Up to 16 rows: with 32, six
// groups of five rows instead of three, a step of the softmax takes 4900 cycles instead of 3100.)
constexpr int kBundleRows = 16;
static_assert(kBundleRows <= kNewRows, "the new keys of a bundle");
int bundle_subs(const ps_config& g) {
  return padded_rows(g) ? std::max(1, std::min(g.max_batch, kBundleRows / ((g.n_heads / g.n_kv_heads) * (g.k_masks + 1)))) : 1;
}
int bundle_rows(const ps_config& g) { return (bundle_subs(g) * (g.n_heads / g.n_kv_heads) * (g.k_masks + 1) + 7) / 8 * 8; }

Buffers layout(const ps_config& g, char* base, size_t* total) {
  Buffers b{};
  const size_t nr = padded_rows(g), pairs = (size_t)g.max_batch * g.n_kv_heads;
  size_t off = 0;
  if (nr) {
    const size_t subs = bundle_subs(g), nb = bundle_rows(g), bundles = (g.max_batch + subs - 1) / subs * g.n_kv_heads;
    const size_t q = take(off, std::max(pairs * nr, bundles * nb) * 2 * kD * 2);
    const size_t kv = take(off, pairs * kNewRows * 2 * kD * 2);
    const size_t o = take(off, (size_t)kMaxSm * 2 * nb * kD * 4), ml = take(off, (size_t)kMaxSm * 2 * nb * sizeof(float2));
    if (base) {
      b.q = (__nv_bfloat16*)(base + q); b.kv_new = (__nv_bfloat16*)(base + kv);
      b.part_o = (float*)(base + o); b.part_ml = (float2*)(base + ml);
    }
  }
  *total = off;
  return b;
}

template <int NR>
cudaError_t launch_nr(ps_ctx* c, const Work& w, int grid, const Buffers& b, const Maps& m, unsigned* tickets,
                      __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t st) {
  auto kern = k_attn_tc<NR>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<NR>());
  if (e != cudaSuccess) return e;
  return launch_after(kern, dim3(grid), dim3(kThreads), smem_bytes<NR>(), st, !c->prof, m.cache, w.subs > 1 ? m.q_bundle : m.q, m.kv_new, w,
                      b.part_o, b.part_ml, tickets, hi, lo, c->dev_status);
}

}  // namespace

size_t bytes(const ps_config& g) {
  size_t n;
  layout(g, nullptr, &n);
  return n;
}
Buffers carve(const ps_config& g, char* base) {
  size_t n;
  return layout(g, base, &n);
}

bool build_maps(const ps_ctx* c, const Buffers& b, Maps* m) {
  const ps_config& g = c->cfg;
  const size_t nr = padded_rows(g), pairs = (size_t)g.max_batch * g.n_kv_heads, rows = pairs * g.max_ctx;
  const void* slab[2] = {c->kcache, c->vcache};
  if (!nr) return false;
  for (int v = 0; v < 2; ++v)
    for (int i = 0; i < kTile / kBoxRows; ++i)
      if (!make_halves_map(&m->cache.m[v][i], slab[v], rows, (i + 1) * kBoxRows)) return false;
  const size_t subs = bundle_subs(g), nb = bundle_rows(g), bundles = (g.max_batch + subs - 1) / subs * g.n_kv_heads;
  return make_halves_map(&m->q, b.q, pairs * 2 * nr, (int)(2 * nr)) &&
         make_halves_map(&m->kv_new, b.kv_new, pairs * 2 * kNewRows, kNewRows) &&
         make_halves_map(&m->q_bundle, b.q, bundles * 2 * nb, (int)(2 * nb));
}

ps_status launch(ps_ctx* c, const SeqMap& sm, int B, const float* qkv, const Buffers& b, const Maps& m, unsigned* tickets,
                 __nv_bfloat16* out_hi, __nv_bfloat16* out_lo, cudaStream_t st) {
  const ps_config& g = c->cfg;
  const int Hq = g.n_heads * kD, Hkv = g.n_kv_heads * kD;
  Work w;
  std::memset(&w, 0, sizeof(w));
  w.sm = sm;
  w.n_kv = g.n_kv_heads; w.group = g.n_heads / g.n_kv_heads; w.R = g.k_masks + 1; w.max_ctx = g.max_ctx; w.n_heads = g.n_heads;
  w.subs = B > 1 && sm.slot[1] == sm.slot[0] ? bundle_subs(g) : 1;
  for (int i = 1; i < B; ++i)
    if (sm.slot[i] != sm.slot[0] || sm.len[i] != sm.len[0] + i) w.subs = 1;
  w.n_bundles = (B + w.subs - 1) / w.subs;
  const int nr = w.subs > 1 ? bundle_rows(g) : padded_rows(g);
  long long units = 0;
  for (int i = 0; i < w.n_bundles; ++i) {
    w.off[i] = (int)units;
    units += (long long)std::max(1, (sm.len[std::min(B, (i + 1) * w.subs) - 1] + kTile - 1) / kTile) * g.n_kv_heads;
  }
  w.off[w.n_bundles] = (int)units;
  if (units * (c->n_sm + 1) >= (1ll << 31)) return fail(c, PS_ERR_UNSUPPORTED, "too many key tiles in one call");
  cudaError_t e = launch_after(k_attn_prep, dim3((g.n_kv_heads + kPrepHeads - 1) / kPrepHeads, B), dim3(256), 0, st, !c->prof, w,
                               qkv, Hq + 2 * Hkv, Hq, Hkv, (const double*)c->rope_inv_freq, nr, b.q, b.kv_new);
  c->launches++;
  if (e != cudaSuccess) return cuda_check(c, e, "k_attn_prep");
  const int grid = (int)std::min<long long>(c->n_sm, units);
  e = nr == 8    ? launch_nr<8>(c, w, grid, b, m, tickets, out_hi, out_lo, st)
      : nr == 16 ? launch_nr<16>(c, w, grid, b, m, tickets, out_hi, out_lo, st)
      : nr == 24 ? launch_nr<24>(c, w, grid, b, m, tickets, out_hi, out_lo, st)
                 : launch_nr<32>(c, w, grid, b, m, tickets, out_hi, out_lo, st);
  c->launches++;
  return cuda_check(c, e, "k_attn_tc");
}

}  // namespace atc
}  // namespace ps
