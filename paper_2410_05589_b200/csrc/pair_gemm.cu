// GEMM of the draft step beyond 16 activation rows, and of the cache append: CTA pairs on the
// 5th-generation tensor cores.
//
// Two CTAs (one cluster, the two SMs of a TPC) work on one tile of 256 weight rows (128 per CTA;
// twice that with wt = 2) times Np <= 256 activation rows with tcgen05.mma.cta_group::2: each CTA
// brings its own weight rows and HALF of the activation rows into shared memory, the tensor
// cores read both halves.  What bounds these launches beside the weight stream is the traffic of
// the activation planes from L2: a CTA that works alone needs 2 * Np * 128 bytes of planes (hi and
// lo) beside every 16 KB weight box; in a pair it needs half of that, and with two weight
// sub-tiles per CTA a quarter.
// Activations are fp32 values split into bf16 hi + lo planes (x = hi + lo to about 2^-17).  Beyond 128
// rows both products go to the same fp32 accumulator in tensor memory, one MMA each.  Up to 128 rows
// the planes are one operand of 2 Np columns (the leader's half of it is the hi plane, the other CTA's the
// lo plane) and the epilogue adds the two halves of the accumulator: an MMA of a pair costs about 95
// cycles however narrow it is, so that two of Np <= 96 columns took 0.85 us a unit where the weights
// arrive in 0.6.  Steps of the 13B shape: 20 rows 314 -> 290 us, 80 rows 393 -> 375, 125 rows 389 -> 381;
// 33B shape, 60 rows 432 -> 413.
//
// Warp roles per CTA: warp 0 issues the TMA loads of its own shared memory (completion counted
// on the leader's barrier), warp 1 allocates tensor memory and, in the leader CTA, issues the
// MMAs for both; warps 2..9 read the accumulators back and store them (two warps per lane
// quadrant, alternating column chunks).  Accumulators are double buffered when two tiles' fit
// tensor memory (tiles of up to 256 columns: wt * Np, or twice that where the planes are one operand).
//
// A tile whose k range is shared by several pairs is left as partial sums in slots (see Plan) and
// finished by a kernel of its own: no CTA waits for another cluster, the sums are added in k
// order whoever finishes first, and for the stages whose output is normalised per row that
// kernel sees whole rows, so it forms the norm on the spot.
//
// Measured (13B shape, whole calls) against one CTA per tile of 128 weight rows and at most 128
// activation rows per pass over the weights: 80 rows 512 -> 454 us, 576 rows 2.97 -> 1.76 ms, 33B
// shape 144 rows 1.39 -> 0.96 ms, 640 training rows 2.82 -> 1.50 ms, 4000 prompt rows appended
// 5.69 -> 1.88 ms.  GEMM launches alone at 80 rows: gate|up 95 -> 59 us (4.8 TB/s of weights), at
// 576 rows 475 -> 222 us (1.47 PFLOP/s of hi + lo products).
#include <cfloat>

#include "pair_gemm.cuh"
#include "umma_gemm.cuh"

namespace ps {
namespace pg {
namespace {

using umma::fence_after_sync;
using umma::fence_before_sync;
using umma::kABytes;
using umma::kBK;
using umma::mbar_arrive_expect_tx;
using umma::mbar_init;
using umma::mbar_wait;
using umma::smem_desc;
using umma::smem_u32;

constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kRing = 222 * 1024;
constexpr int kMaxStages = 12;
constexpr int kMaxComb = 128;     // rows of a tile up to which hi and lo planes are one operand (2 Np <= 256)
constexpr uint32_t kPeerMask = 0xFEFFFFFFu;   // shared::cluster address of the same offset in the leader CTA

struct Ctl {
  uint64_t full[kMaxStages];    // leader: a stage's boxes of both CTAs have landed
  uint64_t empty[kMaxStages];   // the MMAs that read a stage have completed (one per CTA)
  uint64_t acc_full[2];         // an accumulator holds a finished segment (one per CTA)
  uint64_t acc_empty[2];        // leader: the epilogue warps of both CTAs have read it back
  uint32_t tmem_base;
  int abort_flag;
};
constexpr int kSmem = kRing + 1024 + (int)sizeof(Ctl);

__host__ __device__ constexpr int stage_bytes(int wt, int planes, int Np) {
  return wt * kABytes + planes * (Np / 2) * kBK * 2;
}
__host__ __device__ constexpr int n_stages(int bytes) {
  return kRing / bytes < kMaxStages ? kRing / bytes : kMaxStages;
}

// Instruction descriptor of kind::f16 for a CTA pair: fp32 accumulator, bf16 x bf16, both operands
// K-major, N / 8 in bits [17,23), M / 16 = 16 in bits [24,29).
__device__ __forceinline__ uint32_t pair_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (16u << 24);
}
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t leader_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(map), "r"(x), "r"(y), "r"(leader_bar)
      : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
// Arrives on the barrier of this offset in both CTAs once the MMAs issued so far have completed.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void arrive_leader(uint64_t* bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(smem_u32(bar) & kPeerMask) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// 16 accumulator columns of this thread's lane; the caller waits (tmem_ld_wait) before it uses them.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// x += y, as floats.
__device__ __forceinline__ void add16(uint32_t (&x)[16], const uint32_t (&y)[16]) {
#pragma unroll
  for (int j = 0; j < 16; ++j) x[j] = __float_as_uint(__uint_as_float(x[j]) + __uint_as_float(y[j]));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void split1(float x, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(x);
  l = __float2bfloat16_rn(x - __bfloat162float(h));
}
// Two values' hi and lo parts, packed (the conversion takes two values an instruction).
__device__ __forceinline__ void split2(float x, float y, uint32_t& h, uint32_t& l) {
  const __nv_bfloat162 hv = __floats2bfloat162_rn(x, y);
  h = *reinterpret_cast<const uint32_t*>(&hv);
  const __nv_bfloat162 lv = __floats2bfloat162_rn(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xFFFF0000u));
  l = *reinterpret_cast<const uint32_t*>(&lv);
}
// hi/lo planes of four consecutive values as 8-byte stores.
__device__ __forceinline__ void split4(const float4& v, __nv_bfloat16* hi, __nv_bfloat16* lo) {
  uint2 h, l;
  split2(v.x, v.y, h.x, l.x);
  split2(v.z, v.w, h.y, l.y);
  *reinterpret_cast<uint2*>(hi) = h;
  *reinterpret_cast<uint2*>(lo) = l;
}
// Four bf16 values (of a gain or bias vector, which the caller may have put on any 2-byte boundary).
__device__ __forceinline__ float4 load_bf4(const __nv_bfloat16* x) {
  return make_float4(__bfloat162float(x[0]), __bfloat162float(x[1]), __bfloat162float(x[2]), __bfloat162float(x[3]));
}
__device__ __forceinline__ float silu_mul(float g, float u) { return g / (1.f + __expf(-g)) * u; }

// The segments (tile, k range) of a pair, in working order: its run of shared blocks first, then
// its whole tiles.
struct Seg { int t, kb0, kb1, j; bool whole; };
struct SegWalk {
  int x, x_end, d, P;
  __device__ void start(const Plan& p, int pair, int n_pairs) {
    P = n_pairs;
    d = pair;
    x = x_end = 0;
    if (p.rem > 0 && pair < p.Pe) { x = run_begin(p, pair); x_end = run_begin(p, pair + 1); }
  }
  __device__ bool next(const Plan& p, int pair, Seg& s) {
    if (x < x_end) {
      const int tr = x / p.split, j0 = x - tr * p.split, x2 = min(x_end, (tr + 1) * p.split), j1 = x2 - tr * p.split;
      s.t = p.n_dp + tr;
      s.kb0 = j0 * p.KB / p.split;
      s.kb1 = j1 * p.KB / p.split;
      s.j = pair - run_owner(p, tr * p.split);
      s.whole = j0 == 0 && j1 == p.split;
      x = x2;
      return true;
    }
    if (d < p.n_dp) {
      s.t = d; s.kb0 = 0; s.kb1 = p.KB; s.j = 0; s.whole = true;
      d += P;
      return true;
    }
    return false;
  }
};
// Walks a pair's units (segment, k-block) in working order.
struct UnitWalk {
  SegWalk sw;
  Seg s;
  int kb, mat, row0, yb;   // matrix and first weight row of the tile, first activation row
  bool ok;
  __device__ void enter(const Plan& p, int pair, bool zip) {
    ok = sw.next(p, pair, s);
    if (!ok) return;
    kb = s.kb0;
    int w = s.t / p.n_rt;
    yb = (s.t - w * p.n_rt) * p.Np;
    mat = 0;
    if (!zip)
      while (mat + 1 < p.n_mats && w >= p.mat_tiles[mat]) { w -= p.mat_tiles[mat]; ++mat; }
    row0 = w * (zip ? 256 : 256 * p.wt);
  }
  __device__ void start(const Plan& p, int pair, int n_pairs, bool zip) {
    sw.start(p, pair, n_pairs);
    enter(p, pair, zip);
  }
  __device__ void next(const Plan& p, int pair, bool zip) {
    if (++kb == s.kb1) enter(p, pair, zip);
  }
};

template <int MODE, int WT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_pair_gemm(const __grid_constant__ CUtensorMap tA0, const __grid_constant__ CUtensorMap tA1,
            const __grid_constant__ CUtensorMap tA2, const __grid_constant__ CUtensorMap tBh,
            const __grid_constant__ CUtensorMap tBl, const __grid_constant__ Args a) {
  constexpr bool kZip = MODE == MODE_SWIGLU;
  static_assert(!kZip || WT == 2, "gate and up rows are the two sub-tiles");
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  Ctl& ctl = *reinterpret_cast<Ctl*>(smem_raw + (base - raw) + kRing);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const Plan& p = a.p;
  const int Np = p.Np, planes = a.planes;
  const int sbytes = stage_bytes(WT, planes, Np), nst = n_stages(sbytes), plane_bytes = (Np / 2) * kBK * 2;
  const bool comb = p.comb != 0;
  const int nc = comb ? 2 * Np : Np;   // accumulator columns of a sub-tile
  const bool two_buf = WT * nc <= 256;

  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) { mbar_init(&ctl.full[i], 1); mbar_init(&ctl.empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&ctl.acc_full[i], 1); mbar_init(&ctl.acc_empty[i], 2 * kEpiWarps); }
    ctl.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    pdl_launch_dependents();
  }
  __syncwarp();
  // Tensor memory is allocated by the pair together: not before both CTAs run (an allocation that one of
  // them asked for while the other was still to start left the other waiting for good), and the right
  // to allocate is given up once both have it.
  cluster_sync();   // both run, both CTAs' barriers are initialised
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem_base)), "r"(512)
                 : "memory");
    fence_before_sync();
  }
  // (the producer needs no tensor memory: it waits for this barrier's phase only when it is done)
  cluster_arrive();
  if (warp != 0) {
    cluster_wait();   // both have their tensor memory
    fence_after_sync();
  }
  if (warp == 1) asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  const uint32_t tmem = warp == 0 ? 0u : *(volatile uint32_t*)&ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;

  if (warp == 0) {
    if (lane == 0) {   // ---- TMA producer
      const uint32_t pair_bytes = 2u * (uint32_t)sbytes;
      auto load_a = [&](const UnitWalk& u, int st) {
        const uint32_t dst = base + st * sbytes, bar = smem_u32(&ctl.full[st]) & kPeerMask;
        if (rank == 0) mbar_arrive_expect_tx(&ctl.full[st], pair_bytes);
        const int x = u.kb * kBK, y = u.row0 + (int)rank * 128;
        if (kZip) {
          tma_load_pair(dst, &tA0, x, y, bar);
          tma_load_pair(dst + kABytes, &tA1, x, y, bar);
        } else {
          const CUtensorMap* m = u.mat == 0 ? &tA0 : (u.mat == 1 ? &tA1 : &tA2);
#pragma unroll
          for (int s = 0; s < WT; ++s) tma_load_pair(dst + s * kABytes, m, x, y + 256 * s, bar);
        }
      };
      auto load_b = [&](const UnitWalk& u, int st) {
        const uint32_t dst = base + st * sbytes + WT * kABytes, bar = smem_u32(&ctl.full[st]) & kPeerMask;
        const int x = u.kb * kBK;
        if (comb) {   // all rows of one plane
          tma_load_pair(dst, rank == 0 ? &tBh : &tBl, x, u.yb, bar);
          return;
        }
        const int y = u.yb + (int)rank * (Np / 2);
        tma_load_pair(dst, &tBh, x, y, bar);
        if (planes == 2) tma_load_pair(dst + plane_bytes, &tBl, x, y, bar);
      };
      // the weights do not depend on the kernel before this one, the activations do
      UnitWalk u;
      u.start(p, pair, n_pairs, kZip);
      int n_early = 0;
      for (; n_early < nst && u.ok; ++n_early) { load_a(u, n_early); u.next(p, pair, kZip); }
      pdl_wait();
      UnitWalk v;
      v.start(p, pair, n_pairs, kZip);
      for (int i = 0; i < n_early; ++i) { load_b(v, i); v.next(p, pair, kZip); }
      int st = 0;
      uint32_t parity = 0;
      while (u.ok) {
        if (!mbar_wait(&ctl.empty[st], parity, abort_flag)) break;
        load_a(u, st);
        load_b(u, st);
        u.next(p, pair, kZip);
        if (++st == nst) { st = 0; parity ^= 1; }
      }
    }
    __syncwarp();
    cluster_wait();
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {   // ---- MMA issuer of the pair
      SegWalk sw;
      sw.start(p, pair, n_pairs);
      Seg s;
      const uint32_t id = pair_idesc(nc);
      int st = 0, segc = 0;
      uint32_t parity = 0;
      bool alive = true;
      for (; alive && sw.next(p, pair, s); ++segc) {
        const int buf = two_buf ? (segc & 1) : 0;
        const uint32_t use = two_buf ? (uint32_t)(segc >> 1) : (uint32_t)segc;
        if (!mbar_wait(&ctl.acc_empty[buf], (use & 1) ^ 1, abort_flag)) break;
        fence_after_sync();
        const uint32_t d = tmem + buf * WT * nc;
        uint32_t acc = 0;
        for (int kb = s.kb0; kb < s.kb1; ++kb) {
          if (!mbar_wait(&ctl.full[st], parity, abort_flag)) { alive = false; break; }
          fence_after_sync();
          const uint32_t sa = base + st * sbytes, sb = sa + WT * kABytes;
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) {
#pragma unroll
            for (int w = 0; w < WT; ++w)
              mma_pair(d + w * nc, smem_desc(sa + w * kABytes + k * 32), smem_desc(sb + k * 32), id, acc | (k > 0));
            if (planes == 2 && !comb) {
#pragma unroll
              for (int w = 0; w < WT; ++w)
                mma_pair(d + w * nc, smem_desc(sa + w * kABytes + k * 32), smem_desc(sb + plane_bytes + k * 32), id, 1u);
            }
          }
          acc = 1;
          commit_pair(&ctl.empty[st]);
          if (++st == nst) { st = 0; parity ^= 1; }
        }
        if (alive) commit_pair(&ctl.acc_full[buf]);
      }
    }
  } else {
    // ---- epilogue warps: accumulator lane r = 32 q + lane, column chunks of 16 alternating
    const int q = warp & 3, half = (warp - 2) >> 2, r = 32 * q + lane;
    SegWalk sw;
    sw.start(p, pair, n_pairs);
    Seg s;
    pdl_wait();   // the slots and outputs written below may still be read by the kernel before this one
    for (int segc = 0; sw.next(p, pair, s); ++segc) {
      const int buf = two_buf ? (segc & 1) : 0;
      const uint32_t use = two_buf ? (uint32_t)(segc >> 1) : (uint32_t)segc;
      const bool ok = mbar_wait(&ctl.acc_full[buf], use & 1, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) break;
      fence_after_sync();
      int w = s.t / p.n_rt;
      const int rt = s.t - w * p.n_rt, m0 = rt * Np, mrows = min(Np, p.M - m0);
      const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + buf * WT * nc;
      const bool slots = MODE == MODE_RAW || !s.whole;
      if (slots || !kZip) {
        float* dst0;
        size_t ld;
        bool valid[WT];
        if (slots) {
          dst0 = a.part + slot_row(p, s.j, s.t, 0) + rank * 128 + r;
          ld = 256 * WT;
#pragma unroll
          for (int i = 0; i < WT; ++i) valid[i] = true;
        } else {
          int mat = 0;
          while (mat + 1 < p.n_mats && w >= p.mat_tiles[mat]) { w -= p.mat_tiles[mat]; ++mat; }
          const int n = w * 256 * WT + (int)rank * 128 + r;
          dst0 = a.out + (size_t)m0 * a.ldo + p.mat_off[mat] + n;
          ld = a.ldo;
#pragma unroll
          for (int i = 0; i < WT; ++i) valid[i] = n + 256 * i < p.mat_rows[mat];
        }
        for (int c0 = half * 16; c0 < mrows; c0 += 32) {
          uint32_t x[WT][16];
#pragma unroll
          for (int i = 0; i < WT; ++i) tmem_ld16_async(ta + i * nc + c0, x[i]);
          if (comb) {
            uint32_t y[WT][16];
#pragma unroll
            for (int i = 0; i < WT; ++i) tmem_ld16_async(ta + i * nc + Np + c0, y[i]);
            umma::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < WT; ++i) add16(x[i], y[i]);
          } else {
            umma::tmem_ld_wait();
          }
          float* d = dst0 + (size_t)c0 * ld;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
#pragma unroll
            for (int i = 0; i < WT; ++i)
              if (c0 + j < mrows && valid[i]) d[256 * i] = __uint_as_float(x[i][j]);
            d += ld;
          }
        }
      } else {   // a whole gate / up tile
        const int n = w * 256 + (int)rank * 128 + r;
        const bool valid = n < p.mat_rows[0];
        for (int c0 = half * 16; c0 < mrows; c0 += 32) {
          uint32_t xg[16], xu[16];
          tmem_ld16_async(ta + c0, xg);
          tmem_ld16_async(ta + nc + c0, xu);
          if (comb) {
            uint32_t yg[16], yu[16];
            tmem_ld16_async(ta + Np + c0, yg);
            tmem_ld16_async(ta + nc + Np + c0, yu);
            umma::tmem_ld_wait();
            add16(xg, yg);
            add16(xu, yu);
          } else {
            umma::tmem_ld_wait();
          }
          const size_t at = (size_t)(m0 + c0) * a.ld_plane + n;
          __nv_bfloat16 *h = a.hi + at, *l = a.lo + at;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (valid && c0 + j < mrows) split1(silu_mul(__uint_as_float(xg[j]), __uint_as_float(xu[j])), *h, *l);
            h += a.ld_plane;
            l += a.ld_plane;
          }
        }
      }
      fence_before_sync();
      __syncwarp();
      if (lane == 0) arrive_leader(&ctl.acc_empty[buf]);   // read back: the MMA warp may reuse it
    }
    fence_before_sync();
  }

  __syncthreads();
  if (ctl.abort_flag) {
    // let copies and MMAs that are still in flight finish before shared and tensor memory go
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    if (tid == 0) atomicOr(a.status, kStatTimeout);
    __syncthreads();
  }
  cluster_sync();   // neither CTA leaves while the other's copies, MMAs or arrivals may still touch it
  if (warp == 1) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// Shared tiles of a MODE_STORE / MODE_SWIGLU stage: adds the contributors' slots in k order.
// Block (tile, kFinRows rows, and of a plain tile 256 of its columns); bound by the latency of its loads.  Where
// the blocks of four rows find room at once, a thread has four rows of four contributors in flight (a tile of the
// last wave has up to 18 contributors, each of which was a round trip with eight rows: 13B, 20 rows, q|k|v 7.1 -> 3.3
// us; 33B, 144 rows 10 -> 4.7; 576 rows, LM head 10.2 -> 6.0); beyond that eight rows of two (of one, of gate and up)
// move more per instruction (2048 appended rows 17.5 -> 15.0 us, 903 rows 24 -> 9.5; four of four 16.4).
template <bool ZIP, int kFinRows, int kFinJ>
__global__ void __launch_bounds__(256) k_finish_shared(const __grid_constant__ Args a) {
  pdl_launch_dependents();
  const Plan& p = a.p;
  const int t = p.n_dp + blockIdx.x, cnt = tile_contributors(p, t);
  int w = t / p.n_rt;
  const int rt = t - w * p.n_rt, mi0 = blockIdx.y * kFinRows, m0 = rt * p.Np + mi0;
  const int rows = min(min(kFinRows, p.Np - mi0), p.M - m0);
  const int TW = 256 * p.wt, c = blockIdx.z * 256 + threadIdx.x;   // (zipped: the second half are the up features)
  const float* s = a.part + slot_row(p, 0, t, mi0) + c;
  const size_t layer = (size_t)p.Np * TW;
  constexpr int NS = ZIP ? 2 : 1;
  float v[NS][kFinRows];
#pragma unroll
  for (int h = 0; h < NS; ++h)
#pragma unroll
    for (int i = 0; i < kFinRows; ++i) v[h][i] = 0.f;
  pdl_wait();
  if (cnt < 2 || rows <= 0) return;
  for (int j = 0; j < cnt; j += kFinJ) {
    float x[kFinJ][NS][kFinRows];
#pragma unroll
    for (int b = 0; b < kFinJ; ++b)
#pragma unroll
      for (int h = 0; h < NS; ++h)
#pragma unroll
        for (int i = 0; i < kFinRows; ++i)
          x[b][h][i] = j + b < cnt && i < rows ? __ldcg(s + (j + b) * layer + (size_t)i * TW + 256 * h) : 0.f;
#pragma unroll
    for (int b = 0; b < kFinJ; ++b)
#pragma unroll
      for (int h = 0; h < NS; ++h)
#pragma unroll
        for (int i = 0; i < kFinRows; ++i) v[h][i] += x[b][h][i];
  }
  if (ZIP) {
    const int n = w * 256 + c;
    if (n < p.mat_rows[0]) {
#pragma unroll
      for (int i = 0; i < kFinRows; ++i) {
        const size_t at = (size_t)(m0 + i) * a.ld_plane + n;
        if (i < rows) split1(silu_mul(v[0][i], v[NS - 1][i]), a.hi[at], a.lo[at]);
      }
    }
  } else {
    int mat = 0;
    while (mat + 1 < p.n_mats && w >= p.mat_tiles[mat]) { w -= p.mat_tiles[mat]; ++mat; }
    const int n = w * TW + c;
    if (n < p.mat_rows[mat]) {
#pragma unroll
      for (int i = 0; i < kFinRows; ++i)
        if (i < rows) a.out[(size_t)(m0 + i) * a.ldo + p.mat_off[mat] + n] = v[0][i];
    }
  }
}

// Row m of a MODE_RAW stage: the row's slots added in k order, bias and residual, the row's sum
// of squares, the planes of its RMS-normalised values.  One block per row, NV vectors of four features a
// thread, held in registers from the loads to the stores.
// Bound by the latency of its loads from L2, which are hidden in two ways: the slots of JB = 4 contributors in flight
// together, or one contributor's in so few registers that two blocks share an SM (see launch_row_norm).  The
// divisions that find a tile's slots are made once per tile and block.
template <int NV, int JB, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_row_norm(const __grid_constant__ Args a, int H, float eps,
                                                           const __nv_bfloat16* __restrict__ bias, const float* res,
                                                           const __nv_bfloat16* __restrict__ gain, float* out,
                                                           __nv_bfloat16* hi, __nv_bfloat16* lo) {
  __shared__ float s_part[32];
  // By weight tile: how many contributors it has (6 bits: 16 k blocks at most are dealt out), and where the row's first
  // slot lies (in vectors; the slots of 2048 rows of the widest stage are 2^25).  256 bytes in all up to 8192 features:
  // beside a CTA of the GEMM that this block waits for 3.75 KB are left, so that three blocks (1 KB each belongs to the
  // system) are there when it ends.  As two arrays for the widest rows it was one, and the table of the others was formed
  // after the wait (768 features, 160 rows 93.6 -> 91.1 us, 256 rows 115 -> 112).
  __shared__ unsigned s_tile[NV * 4 * NT / 256];
  pdl_launch_dependents();
  const Plan& p = a.p;
  const int m = blockIdx.x, tid = threadIdx.x, nthr = blockDim.x;
  const int sh = p.wt == 2 ? 7 : 6;                    // vectors of a tile's row: 128 or 64
  const bool out_vec = ((uintptr_t)out & 15) == 0;     // (the caller's feature rows may sit anywhere)
  const bool gain_vec = ((uintptr_t)gain & 7) == 0;    // (and so may the gains)
  const unsigned layer = (unsigned)p.Np << sh;         // vectors between a tile's contributors
  for (int w = tid; w < p.tiles_w; w += nthr) {
    const int rt = m / p.Np, mi = m - rt * p.Np, t = w * p.n_rt + rt;
    s_tile[w] = (unsigned)tile_contributors(p, t) | (unsigned)(slot_row(p, 0, t, mi) / 4) << 6;
  }
  __syncthreads();
  const float4* part = reinterpret_cast<const float4*>(a.part);
  const int nv = H >> 2;                               // H % 8 == 0
  float4 x[NV];
  uint2 gr[NV];                                        // the gains' bits
  unsigned slot[NV];
  int cnt[NV], cmax = 0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int n = tid + i * nthr;
    cnt[i] = 0;
    slot[i] = 0;
    x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n < nv) {
      const unsigned at = s_tile[n >> sh];
      cnt[i] = (int)(at & 63u);
      cmax = max(cmax, cnt[i]);
      slot[i] = (at >> 6) + (n & ((1 << sh) - 1));
      asm volatile("" : "+r"(cnt[i]), "+r"(slot[i]));   // (taken apart once, not for every contributor)
      if (bias) x[i] = load_bf4(bias + 4 * n);
    }
  }
  pdl_wait();
  float4 rv[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int n = tid + i * nthr;
    gr[i] = make_uint2(0u, 0u);
    if (n < nv && gain_vec) {
      gr[i] = __ldg(reinterpret_cast<const uint2*>(gain) + n);
    } else if (n < nv) {
      const unsigned short* gp = reinterpret_cast<const unsigned short*>(gain) + 4 * n;
      gr[i] = make_uint2(gp[0] | (unsigned)gp[1] << 16, gp[2] | (unsigned)gp[3] << 16);
    }
    rv[i] = (res && n < nv) ? __ldcg(reinterpret_cast<const float4*>(res + (size_t)m * H) + n) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int j = 0; j < cmax; j += JB) {
    float4 v[JB][NV];
#pragma unroll
    for (int b = 0; b < JB; ++b)
#pragma unroll
      for (int i = 0; i < NV; ++i)
        v[b][i] = j + b < cnt[i] ? __ldcg(part + (slot[i] + (j + b) * layer)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int b = 0; b < JB; ++b)
#pragma unroll
      for (int i = 0; i < NV; ++i) { x[i].x += v[b][i].x; x[i].y += v[b][i].y; x[i].z += v[b][i].z; x[i].w += v[b][i].w; }
  }
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    x[i].x += rv[i].x; x[i].y += rv[i].y; x[i].z += rv[i].z; x[i].w += rv[i].w;
    ss += (x[i].x * x[i].x + x[i].y * x[i].y) + (x[i].z * x[i].z + x[i].w * x[i].w);
  }
  ss = warp_sum(ss);
  if ((tid & 31) == 0) s_part[tid >> 5] = ss;
  __syncthreads();
  const float tot = warp_sum((tid & 31) < (nthr >> 5) ? s_part[tid & 31] : 0.f);
  const float sc = rsqrtf(tot / (float)H + eps);
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int n = 4 * (tid + i * nthr);
    if (n < H) {
      if (out) {
        float* o = out + (size_t)m * H + n;
        if (out_vec) *reinterpret_cast<float4*>(o) = x[i];
        else { o[0] = x[i].x; o[1] = x[i].y; o[2] = x[i].z; o[3] = x[i].w; }
      }
      const float4 y = make_float4(x[i].x * sc * __uint_as_float(gr[i].x << 16), x[i].y * sc * __uint_as_float(gr[i].x & 0xFFFF0000u),
                                   x[i].z * sc * __uint_as_float(gr[i].y << 16), x[i].w * sc * __uint_as_float(gr[i].y & 0xFFFF0000u));
      split4(y, hi + (size_t)m * H + n, lo + (size_t)m * H + n);
    }
  }
}

// Modelled time of a launch and of what finishes it (microseconds), for the choice between plans
// only; fitted to the stage times of plans with one and two sub-tiles and 1 to 16 k blocks, 7B to 33B
// shapes, 20 to 640 rows, with two MMAs a unit throughout (the plan chosen was 1.6% behind the best one on average; a model in which
// each pair had a fixed share of HBM was 4.9% behind: 33B q|k|v at 20 rows 87 us, now 67; 13B LM head
// at 20 rows 95 us, now 83; 33B q|k|v at 288 rows 158 us, now 139).
//  - a unit of a pair (wt weight boxes and the planes beside them in both CTAs) takes the longer of
//    its way through the ring and its MMAs; idle pairs leave their share of HBM to the others, so
//    HBM bounds the launch as a whole;
//  - two sub-tiles of more than 128 rows fill the tensor memory, so the MMAs of the next tile wait
//    until this one is read: one sub-tile is the better one there unless a pair has one tile only.
//    (Where the planes are one operand, two sub-tiles of more than 64 rows fill it too.  The count leaves
//    that out: with it a few stages of 65 to 128 rows get other plans, which took as long for 33B, 8192 features and
//    128256 tokens and made steps of the 7B shape 1.2% longer.  Nor does it matter that an MMA of a pair takes 95 cycles at
//    least and not 58: such units wait for the ring.)
//  - each contributor more costs a round trip, its slots the way through L2 twice, and a stage
//    without a row norm a kernel that adds them.
double stream_cost(const Plan& p, int planes, int units) {
  const double a = p.wt * 32.768e3;
  const double ring = 0.17 + (a + planes * p.Np * 128.0) / 185e3;
  const double mma = (p.comb ? std::max(58.0, p.Np * 1.2) : planes * std::max(58.0, p.Np * 0.6)) * 4 * p.wt / 1.85e3;
  return std::max(units * std::max(ring, mma), (double)p.T * p.KB * a / p.n_rt / 7.2e6);
}
double finish_cost(const Plan& p, Mode mode, int segs, int contributors, int n_slots) {
  const double cols = (double)p.wt * p.Np;
  double t = cols * 0.021 + (cols > 256 ? cols * 0.035 * (segs - 1) : 0.0);
  if (mode == MODE_RAW || contributors > 1) t += 0.5 * (contributors - 1) + 2.0 * n_slots * cols * 1024.0 / 5e6;
  if (mode != MODE_RAW && contributors > 1) t += 5.0 + 0.008 * p.Np * p.n_rt;
  return t;
}

}  // namespace

int smem_bytes() { return kSmem; }

Plan make_plan(int M, const Weights& w, int K, int planes, Mode mode, size_t part_floats, int n_sm) {
  const int P = n_sm / 2;
  Plan best{};
  double best_cost = 1e30;
  for (int wt = mode == MODE_SWIGLU ? 2 : 1; wt <= 2; ++wt) {
    Plan p{};
    p.M = M;
    p.n_rt = (M + kMaxNp - 1) / kMaxNp;
    p.Np = ((M + p.n_rt - 1) / p.n_rt + kNpStep - 1) / kNpStep * kNpStep;
    p.wt = wt;
    p.comb = planes == 2 && p.Np <= kMaxComb;
    p.KB = (K + kBK - 1) / kBK;
    p.n_mats = w.zip ? 1 : w.n_mats;
    const int tile_rows = w.zip ? 256 : 256 * wt;
    int off = 0;
    for (int i = 0; i < p.n_mats; ++i) {
      p.mat_rows[i] = w.rows[i];
      p.mat_tiles[i] = (w.rows[i] + tile_rows - 1) / tile_rows;
      p.mat_off[i] = off;
      off += w.rows[i];
      p.tiles_w += p.mat_tiles[i];
    }
    p.T = p.tiles_w * p.n_rt;
    p.n_dp = p.T / P * P;
    p.rem = p.T - p.n_dp;
    // Several full tiles a pair, two accumulators of 256 columns: the model has them 4% shorter than two
    // sub-tiles on prompts.  They are on 7B shapes (4096 rows 676 -> 639 us), but 13B ones are 3% and 33B
    // ones 16% longer (1527 -> 1778), so these tiles always have two sub-tiles.
    if (mode != MODE_SWIGLU && wt == 1 && p.Np == kMaxNp && p.T > P) continue;
    p.slot_t0 = mode == MODE_RAW ? 0 : p.n_dp;
    const size_t slot = (size_t)p.Np * 256 * wt;
    for (int s = 1; s <= std::min(kMaxSplit, p.KB); ++s) {
      if (p.rem == 0 && s > 1) break;
      p.split = s;
      p.S = p.rem * s;
      p.Pe = std::max(1, std::min(P, p.S));
      int units = p.n_dp / P * p.KB, segs = p.n_dp / P, jmax = 1, n_slots = p.n_dp - p.slot_t0;
      if (p.rem > 0) units += (p.S + p.Pe - 1) / p.Pe * ((p.KB + s - 1) / s);
      double cost = stream_cost(p, planes, units);
      if (cost >= best_cost) continue;
      if (p.rem > 0) {
        // at least so many contributors to a tile and in all: most candidates need not be walked
        if (cost + finish_cost(p, mode, segs + 1, (p.Pe + p.rem - 1) / p.rem, n_slots + std::max(p.rem, p.Pe)) >= best_cost)
          continue;
        // one walk over the runs (run_begin without its divisions): contributors of each tile, tiles of a run
        const int q = p.S / p.Pe, r = p.S % p.Pe;
        int runs = 0, err = 0, pos = 0, j = 0;
        for (int c = 0; c < p.Pe; ++c) {
          int len = q, tiles = 0;
          if ((err += r) >= p.Pe) { err -= p.Pe; ++len; }
          while (len > 0) {
            j = pos == 0 ? 1 : j + 1;
            jmax = std::max(jmax, j);
            ++tiles;
            const int take = std::min(len, s - pos);
            len -= take;
            if ((pos += take) == s) pos = 0;
          }
          n_slots += tiles;
          runs = std::max(runs, tiles);
        }
        segs += runs;
      }
      p.shared = jmax > 1;
      if ((mode == MODE_RAW || jmax > 1) && slot_tiles(p) * slot > part_floats) continue;
      cost += finish_cost(p, mode, segs, jmax, n_slots);
      if (cost < best_cost) { best_cost = cost; best = p; }
    }
  }
  return best;   // (T == 0: the slots hold not even one contributor)
}

ps_status launch_gemm(ps_ctx* c, const Weights& w, const PlaneMaps& hi, const PlaneMaps& lo, Args& a, Mode mode,
                      cudaStream_t st) {
  const Plan& p = a.p;
  if (p.T == 0) return fail(c, PS_ERR_CAPACITY, "GEMM scratch too small for the rows of the call");
  auto kern = mode == MODE_RAW     ? (p.wt == 2 ? k_pair_gemm<MODE_RAW, 2> : k_pair_gemm<MODE_RAW, 1>)
              : mode == MODE_STORE ? (p.wt == 2 ? k_pair_gemm<MODE_STORE, 2> : k_pair_gemm<MODE_STORE, 1>)
                                   : k_pair_gemm<MODE_SWIGLU, 2>;
  a.status = c->dev_status;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return cuda_check(c, e, "pair gemm smem attribute");
  const CUtensorMap &m1 = *w.map[w.n_mats > 1 ? 1 : 0], &m2 = *w.map[w.n_mats > 2 ? 2 : 0];
  const int box = (p.comb ? 2 : 1) * p.Np / kNpStep - 1;
  e = launch_after(kern, dim3(c->n_sm & ~1), dim3(kThreads), kSmem, st, !c->prof, *w.map[0], m1, m2,
                   hi.m[box], lo.m[box], a);
  c->launches++;
  return cuda_check(c, e, "k_pair_gemm");
}

ps_status launch_finish_shared(ps_ctx* c, const Args& a, Mode mode, cudaStream_t st) {
  const Plan& p = a.p;
  if (!p.shared) return PS_OK;
  const int np = std::min(p.Np, p.M), z = mode == MODE_SWIGLU ? 1 : p.wt;
  const bool few = p.rem * ((np + 3) / 4) * z <= 3 * c->n_sm;   // (see k_finish_shared)
  const int rows = few ? 4 : 8;
  auto kern = mode == MODE_SWIGLU ? (few ? k_finish_shared<true, 4, 4> : k_finish_shared<true, 8, 1>)
                                  : (few ? k_finish_shared<false, 4, 4> : k_finish_shared<false, 8, 2>);
  const cudaError_t e = launch_after(kern, dim3(p.rem, (np + rows - 1) / rows, z), dim3(256), 0, st, !c->prof, a);
  c->launches++;
  return cuda_check(c, e, "k_finish_shared");
}

ps_status launch_row_norm(ps_ctx* c, const Args& a, int H, const __nv_bfloat16* bias, const float* res,
                          const __nv_bfloat16* gain, float* out, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t st) {
  if (H > kMaxNormWidth) return fail(c, PS_ERR_UNSUPPORTED, "hidden size beyond 32768");
  // More rows than SMs, a second block on an SM: up to 4096 features the blocks of four contributors have 512 threads
  // and share an SM as they are; of 640 threads two fit with one contributor in flight (5120 features, steps without a
  // large vocabulary: 192 rows 333.0 -> 329.5 us, 512 rows 703 -> 691, 160 rows 298.0 and 297.7; 4096 features, 160 rows 223.5,
  // with one contributor 227.3; 768 features 93.6 and 96.7).  Wider rows would not fit the registers of half an SM (6656
  // features, 320 rows: 765, with 16 features a thread, spilled, 794; 8192 features 1158 and 1179).
  const bool two = H > 4096 && H <= 5120 && a.p.M > c->n_sm;
  const int threads = H <= 8192 ? (H / 8 + 31) / 32 * 32 : 512;
  auto kern = two ? k_row_norm<2, 1, 640, 2>
              : H <= 8192 ? k_row_norm<2, 4, 1024, 1> : H <= 16384 ? k_row_norm<8, 1, 512, 1> : k_row_norm<16, 1, 512, 1>;
  const cudaError_t e = launch_after(kern, dim3(a.p.M), dim3(threads), 0, st, !c->prof, a, H, c->cfg.rms_eps, bias, res, gain,
                                     out, hi, lo);
  c->launches++;
  return cuda_check(c, e, "k_row_norm");
}

}  // namespace pg
}  // namespace ps
