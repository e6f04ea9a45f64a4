// ps_verify: speculative-sampling acceptance for a drafted chain (Eq. 1; Algorithm 1 with one
// child per node).  One thread block per (position, sequence) evaluates its row pair
// speculatively: softmax statistics of the target and draft rows, the test r < min(1, p/q),
// and -- if the test fails or the row is the extra target row -- the token that would be
// emitted there (residual max(0, p-q) normalised, or p itself).  The last block of a sequence
// to finish walks the positions in order and writes accept_len / out_tokens / n_out.
// Nothing spins: blocks only take a ticket, the last arriver does the merge.
#include <cfloat>
#include <cstdio>
#include <mutex>

#include <cooperative_groups.h>

#include "ps_internal.cuh"

namespace ps {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kSeg = 128;  // elements per warp-wide segment of the inverse-CDF search

__global__ void k_philox_fill(uint32_t k0, uint32_t k1, const uint32_t* ctr, uint32_t* out, int n) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t c[4] = {ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]};
  philox4x32_10(k0, k1, c);
  for (int j = 0; j < 4; ++j) out[4 * i + j] = c[j];
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct Scratch {
  float fmax[kWarps];
  int imax[kWarps];
  double dsum[kWarps];
  int flag[kWarps];
  float bc_f;
  int bc_i;
  double bc_d;
  int bc_flag;
};

// Max over a row with NaN treated as -inf, ties to the lower index; also reports whether the
// row holds a NaN or +inf (or nothing above -inf).  Result broadcast to all threads.
__device__ void row_argmax(const float* row, int V, Scratch& s, float& vmax, int& imax, int& bad) {
  float bv = -INFINITY;
  int bi = 0x7fffffff, bd = 0;
  for (int v = threadIdx.x; v < V; v += kThreads) {
    float x = row[v];
    if (x != x || x == INFINITY) bd = 1;
    if (x != x) x = -INFINITY;
    if (x > bv || (x == bv && v < bi)) { bv = x; bi = v; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float ov = __shfl_xor_sync(0xffffffffu, bv, o);
    int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    bd |= __shfl_xor_sync(0xffffffffu, bd, o);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { s.fmax[warp] = bv; s.imax[warp] = bi; s.flag[warp] = bd; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kWarps; ++w) {
      if (s.fmax[w] > bv || (s.fmax[w] == bv && s.imax[w] < bi)) { bv = s.fmax[w]; bi = s.imax[w]; }
      bd |= s.flag[w];
    }
    if (bv == -INFINITY) bd = 1;  // an all -inf row has no distribution
    s.bc_f = bv; s.bc_i = bi; s.bc_flag = bd;
  }
  __syncthreads();
  vmax = s.bc_f; imax = s.bc_i; bad = s.bc_flag;
  __syncthreads();
}

// sum_v exp((row[v] - vmax) / T), accumulated in double, broadcast to all threads.
__device__ double row_sumexp(const float* row, int V, float vmax, double inv_t, Scratch& s) {
  double acc = 0.0;
  for (int v = threadIdx.x; v < V; v += kThreads)
    acc += (double)expf((float)(((double)row[v] - (double)vmax) * inv_t));
  acc = warp_sum_d(acc);
  if ((threadIdx.x & 31) == 0) s.dsum[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kWarps; ++w) t += s.dsum[w];
    s.bc_d = t;
  }
  __syncthreads();
  double r = s.bc_d;
  __syncthreads();
  return r;
}

// Weight of token v in the distribution to sample: max(0, p_v - q_v), or p_v when use_q == 0.
// q is softmax(drow/T) when drow != nullptr, else the point mass on x.
__device__ __forceinline__ float weight_of(int v, const float* trow, const float* drow, int x,
                                           int use_q, float tmax, float dmax, double inv_t,
                                           float inv_st, float inv_sd) {
  float p = expf((float)(((double)trow[v] - (double)tmax) * inv_t)) * inv_st;
  if (!use_q) return p;
  float q = drow ? expf((float)(((double)drow[v] - (double)dmax) * inv_t)) * inv_sd
                 : (v == x ? 1.f : 0.f);
  return fmaxf(p - q, 0.f);
}

// Inverse-CDF draw with uniform u from the weights above: the first v whose running sum
// exceeds u * total.  seg_sum: shared array of ceil(V / kSeg) doubles.  Returns the token to
// all threads; returns -1 if the total weight is not positive.
__device__ int sample_weights(const float* trow, const float* drow, int x, int use_q, int V,
                              float tmax, float dmax, double inv_t, double st, double sd,
                              double u, double* seg_sum, Scratch& s) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nseg = (V + kSeg - 1) / kSeg;
  const float inv_st = (float)(1.0 / st), inv_sd = (float)(1.0 / sd);
  constexpr int E = kSeg / 32;
  for (int g = warp; g < nseg; g += kWarps) {
    double a = 0.0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      int v = g * kSeg + lane * E + e;
      if (v < V) a += (double)weight_of(v, trow, drow, x, use_q, tmax, dmax, inv_t, inv_st, inv_sd);
    }
    a = warp_sum_d(a);
    if (lane == 0) seg_sum[g] = a;
  }
  __syncthreads();
  if (warp == 0) {
    // lane owns segments [lane*c, lane*c + c)
    int c = (nseg + 31) / 32;
    int g_lo = min(nseg, lane * c), g_hi = min(nseg, lane * c + c);
    double mine = 0.0;
    for (int g = g_lo; g < g_hi; ++g) mine += seg_sum[g];
    double incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      double t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    double total = __shfl_sync(0xffffffffu, incl, 31);
    double target = u * total;
    int token = -1;
    if (total > 0.0) {  // uniform across the warp
      // first lane whose inclusive sum exceeds the target, else the last lane with weight
      unsigned over = __ballot_sync(0xffffffffu, incl > target);
      unsigned pos = __ballot_sync(0xffffffffu, mine > 0.0);
      int src = over ? __ffs(over) - 1 : (pos ? 31 - __clz(pos) : 0);
      int gsel = -1;
      double gbase = 0.0;
      if (lane == src) {
        double run = incl - mine;
        int last_pos = -1;
        double last_base = 0.0;
        for (int g = g_lo; g < g_hi; ++g) {
          if (seg_sum[g] > 0.0) { last_pos = g; last_base = run; }
          if (run + seg_sum[g] > target) { gsel = g; gbase = run; break; }
          run += seg_sum[g];
        }
        if (gsel < 0) { gsel = last_pos; gbase = last_base; }
      }
      gsel = __shfl_sync(0xffffffffu, gsel, src);
      gbase = __shfl_sync(0xffffffffu, gbase, src);
      // inside the segment: lane owns E consecutive tokens
      float wv[E];
      double lsum = 0.0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        int v = gsel * kSeg + lane * E + e;
        wv[e] = (gsel >= 0 && v < V) ? weight_of(v, trow, drow, x, use_q, tmax, dmax, inv_t, inv_st, inv_sd) : 0.f;
        lsum += (double)wv[e];
      }
      double linc = lsum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        double t = __shfl_up_sync(0xffffffffu, linc, o);
        if (lane >= o) linc += t;
      }
      unsigned over2 = __ballot_sync(0xffffffffu, gbase + linc > target);
      unsigned pos2 = __ballot_sync(0xffffffffu, lsum > 0.0);
      int src2 = over2 ? __ffs(over2) - 1 : (pos2 ? 31 - __clz(pos2) : 0);
      int pick = -1;
      if (lane == src2 && gsel >= 0 && (over2 | pos2)) {
        double run2 = gbase + linc - lsum;
        int lastp = -1;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (wv[e] > 0.f) lastp = e;
          run2 += (double)wv[e];
          if (pick < 0 && run2 > target) pick = e;
        }
        if (pick < 0) pick = lastp;
        pick = pick < 0 ? -1 : gsel * kSeg + lane * E + pick;
      }
      token = __shfl_sync(0xffffffffu, pick, src2);
    }
    if (lane == 0) s.bc_i = token;
  }
  __syncthreads();
  int tok = s.bc_i;
  __syncthreads();
  return tok;
}

struct VerifyArgs {
  int B, n_draft, n_target, V;
  const int* draft_tokens;
  const float* draft_logits;
  const float* target_logits;
  float temperature;
  uint32_t key0, key1, off_lo, off_hi;
  int* accept_len;
  int* out_tokens;
  int* n_out;
  VerifyRec* rec;      // [B][PS_MAX_MASKS+2]
  unsigned* tickets;   // [B], zero on entry and on exit
  int* status;
};

// Called by one thread per (position, sequence): records the speculative outcome, takes a
// ticket, and -- as the last arriver of its sequence -- walks the positions in order and writes
// accept_len / out_tokens / n_out.
__device__ void finish_position(const VerifyArgs& a, int i, int b, int accept, int bad, int token) {
  VerifyRec* recw = a.rec + (size_t)b * (PS_MAX_MASKS + 2);
  recw[i].accept = accept | (bad << 1);
  recw[i].token = token;
  __threadfence();
  unsigned t = atomicAdd(&a.tickets[b], 1u);
  if (t != (unsigned)a.n_target - 1u) return;
  __threadfence();
  volatile VerifyRec* rec = recw;
  int* out = a.out_tokens + (size_t)b * (a.n_draft + 1);
  int acc = 0, any_bad = 0, emitted = -1;
  while (acc < a.n_draft) {
    int f = rec[acc].accept;
    any_bad |= (f >> 1) & 1;
    if (!(f & 1)) { emitted = rec[acc].token; break; }
    out[acc] = a.draft_tokens[(size_t)b * a.n_draft + acc];
    ++acc;
  }
  if (acc == a.n_draft && a.n_target == a.n_draft + 1) {
    any_bad |= (rec[acc].accept >> 1) & 1;
    emitted = rec[acc].token;
  }
  int n = acc;
  if (emitted >= 0) out[n++] = emitted;
  for (int j = n; j <= a.n_draft; ++j) out[j] = -1;
  a.accept_len[b] = acc;
  a.n_out[b] = n;
  if (any_bad) atomicOr(a.status, kStatNonfinite);
  a.tickets[b] = 0u;
}

__global__ void __launch_bounds__(kThreads) k_verify(VerifyArgs a) {
  extern __shared__ double seg_sum[];
  __shared__ Scratch s;
  const int i = blockIdx.x, b = blockIdx.y, V = a.V;
  const bool bonus = i >= a.n_draft;
  const float* trow = a.target_logits + ((size_t)b * a.n_target + i) * V;
  const float* drow = (!bonus && a.draft_logits) ? a.draft_logits + ((size_t)b * a.n_draft + i) * V
                                                 : nullptr;
  int x = bonus ? -1 : a.draft_tokens[(size_t)b * a.n_draft + i];
  int accept = 0, token = -1, bad = 0;

  float tmax; int targ, tbad;
  row_argmax(trow, V, s, tmax, targ, tbad);
  if (a.temperature == 0.f) {
    accept = (!bonus && x == targ) ? 1 : 0;
    token = targ;
  } else {
    double inv_t = 1.0 / (double)a.temperature;
    float dmax = 0.f; int darg, dbad = 0;
    if (drow) row_argmax(drow, V, s, dmax, darg, dbad);
    bad = tbad | dbad;
    if (bad) {
      token = targ;
    } else {
      double st = row_sumexp(trow, V, tmax, inv_t, s);
      double sd = drow ? row_sumexp(drow, V, dmax, inv_t, s) : 1.0;
      uint32_t c[4] = {(uint32_t)i, (uint32_t)b, a.off_lo, a.off_hi};
      philox4x32_10(a.key0, a.key1, c);
      double r = (double)(c[0] >> 8) * (1.0 / 16777216.0);
      double u2 = (double)(c[1] >> 8) * (1.0 / 16777216.0);
      if (!bonus) {
        bool in_range = x >= 0 && x < V;
        double logp = in_range ? ((double)trow[x] - (double)tmax) * inv_t - log(st) : -INFINITY;
        double logq = drow ? (in_range ? ((double)drow[x] - (double)dmax) * inv_t - log(sd) : -INFINITY)
                           : 0.0;
        double diff = logp - logq;
        double ratio = (diff != diff) ? 0.0 : exp(fmin(diff, 0.0));
        accept = r < ratio ? 1 : 0;
      }
      if (!accept) {  // uniform across the block: every thread computed the same decision
        token = sample_weights(trow, drow, x, bonus ? 0 : 1, V, tmax, dmax, inv_t, st, sd, u2,
                               seg_sum, s);
        if (token < 0)
          token = sample_weights(trow, drow, x, 0, V, tmax, dmax, inv_t, st, sd, u2, seg_sum, s);
        if (token < 0) token = targ;
      }
    }
  }

  if (threadIdx.x == 0) finish_position(a, i, b, accept, bad, token);
}

// ---- cluster variant ------------------------------------------------------------------------
// A cluster of kClu thread blocks shares one (position, sequence) row pair, so that a batch of
// one still spreads its few rows over dozens of SMs.  Thread g = rank * kCluThreads + tid owns
// the contiguous tokens [g * C, g * C + C) of both rows and keeps them in registers: the logits
// are read from memory once, with all 16-byte loads in flight together.  Row statistics are
// combined through distributed shared memory (each block publishes its partials, a cluster
// barrier, every block reads all of them in rank order, so all blocks hold identical values).
// The inverse-CDF draw descends block -> warp -> lane -> token over running sums.
constexpr int kClu = 8;
constexpr int kCluThreads = 512;
constexpr int kCluWarps = kCluThreads / 32;
constexpr int kCluV4 = 4;  // float4 per thread and row: up to kClu * kCluThreads * 16 tokens
constexpr int kCluMaxVocab = kClu * kCluThreads * 4 * kCluV4;        // with the portable cluster size
constexpr int kCluMaxVocab16 = 16 * kCluThreads * 4 * kCluV4;         // with 16 blocks (opt-in size)

struct CluPart {       // one per block, read by the whole cluster
  float tmax, dmax;
  int targ, bad;
  double st, sd;
  double wsum;         // weight held by this block
  double turn[2];      // sums of successive exchanges (tree walk)
  int pick, lastp;     // token chosen inside this block / its last token with weight
};

struct CluScratch {
  float f[kCluWarps], f2[kCluWarps];
  int i[kCluWarps], flag[kCluWarps];
  double d[kCluWarps], d2[kCluWarps];
};

// 1 / T in two parts.  Temperatures below the smallest whose inverse is a float act like it: logits that differ
// at all are then 1e31 apart.
struct InvT {
  float hi, lo;
  __device__ __forceinline__ explicit InvT(double inv_t) {
    const double x = fmin(inv_t, (double)FLT_MAX);
    hi = (float)x;
    lo = (float)(x - (double)hi);
  }
};

// exp argument (t - m) / T with one rounding: in single precision with the rounding errors of the
// difference and of the product carried along.  (m may lie below t while a block looks for its reference; where
// the argument then overflows, the block takes another reference.)  UNIT: T = 1.
template <bool UNIT>
__device__ __forceinline__ float exp_arg(float t, float m, const InvT& i) {
  const float d = t - m;
  if (UNIT) return d;
  const float bv = t - d, av = d + bv;
  const float e = (t - av) + (bv - m);
  const float p = d * i.hi;
  // (where p is -infinity the errors are infinite or no number: the minimum makes any finite value of them.  It has one
  // instruction where a comparison has two: 576 rows of 32000 tokens at T = 0.7 67.6 us with one that sees to infinite
  // differences only, 66.8 so; 5 trees of 23 nodes, 128256 tokens 52.9 -> 52.5)
  return p + fminf(fmaf(d, i.hi, -p) + fmaf(e, i.hi, d * i.lo), FLT_MAX);
}

// The same by way of double precision; at T = 1 that is the difference rounded once, which single precision
// gives bit for bit without the conversions (the register-resident kernels, 8 or 16 tokens a thread and row: 13B, one
// sequence 242.5 -> 241.4 us for draft + verify).
template <bool UNIT>
__device__ __forceinline__ float exp_arg_d(float t, float m, double inv_t) {
  return UNIT ? t - m : (float)(((double)t - (double)m) * inv_t);
}

// (NCLU blocks per cluster: 8; 16 for vocabularies beyond 65536; 4 for batches of several waves.)
// (V4: 16-byte vectors a thread holds per row: 4, or 2 when the row fits in half as many -- the
// loops over a thread's tokens are unrolled, and this kernel runs its code once per launch, so
// what it is not asked to execute it should not have to fetch.)
template <int NCLU, int V4, bool UNIT>
__device__ __forceinline__ void verify_cluster_body(const VerifyArgs& a) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ CluPart part;
  __shared__ CluScratch s;
  const int rank = (int)cl.block_rank();
  constexpr int nclu = NCLU;
  const int i = blockIdx.x / nclu, b = blockIdx.y, V = a.V;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool bonus = i >= a.n_draft;
  const float* trow = a.target_logits + ((size_t)b * a.n_target + i) * V;
  const bool greedy = a.temperature == 0.f;
  const float* drow = (!bonus && !greedy && a.draft_logits)
                          ? a.draft_logits + ((size_t)b * a.n_draft + i) * V : nullptr;
  const int nv4 = ((V + nclu * kCluThreads - 1) / (nclu * kCluThreads) + 3) / 4;
  const int C = nv4 * 4, v0 = (rank * kCluThreads + tid) * C;

  // All rows may be what the kernel before this one in the stream wrote last (the target model's LM
  // head, the draft step), and that kernel may let its dependents start before it writes: nothing of
  // them is read before the wait.
  pdl_launch_dependents();
  pdl_wait();
  float t[V4 * 4], d[V4 * 4];
#pragma unroll
  for (int k = 0; k < V4; ++k) {
    const int v = v0 + 4 * k;   // V % 4 == 0: a vector lies inside the row or outside it
    float4 tv = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (k < nv4 && v < V) tv = __ldcs(reinterpret_cast<const float4*>(trow + v));
    t[4 * k] = tv.x; t[4 * k + 1] = tv.y; t[4 * k + 2] = tv.z; t[4 * k + 3] = tv.w;
  }
  const int x = bonus ? -1 : a.draft_tokens[(size_t)b * a.n_draft + i];
#pragma unroll
  for (int k = 0; k < V4; ++k) {
    const int v = v0 + 4 * k;
    float4 dv = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (drow && k < nv4 && v < V) dv = *reinterpret_cast<const float4*>(drow + v);
    d[4 * k] = dv.x; d[4 * k + 1] = dv.y; d[4 * k + 2] = dv.z; d[4 * k + 3] = dv.w;
  }

  // ---- maxima (NaN counts as -inf, ties to the lower id) and non-finite flags
  float tm = -INFINITY, dm = -INFINITY;
  int ti = 0x7fffffff, bad = 0;
#pragma unroll
  for (int e = 0; e < V4 * 4; ++e) {
    const int v = v0 + e;
    if (e < C && v < V) {
      float xt = t[e];
      if (xt != xt || xt == INFINITY) bad = 1;
      if (xt != xt) xt = -INFINITY;
      if (xt > tm || (xt == tm && v < ti)) { tm = xt; ti = v; }
      if (drow) {
        float xd = d[e];
        if (xd != xd || xd == INFINITY) bad = 1;
        if (xd != xd) xd = -INFINITY;
        dm = fmaxf(dm, xd);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, tm, o);
    const int oi = __shfl_xor_sync(0xffffffffu, ti, o);
    if (ov > tm || (ov == tm && oi < ti)) { tm = ov; ti = oi; }
    dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (lane == 0) { s.f[warp] = tm; s.i[warp] = ti; s.flag[warp] = bad; s.f2[warp] = dm; }
  __syncthreads();
  if (warp == 0) {   // the warps' values, one per lane, through a shuffle tree
    static_assert(kCluWarps == 16, "one lane per warp in the low half of warp 0");
    tm = -INFINITY; dm = -INFINITY; ti = 0x7fffffff; bad = 0;
    if (lane < kCluWarps) { tm = s.f[lane]; ti = s.i[lane]; bad = s.flag[lane]; dm = s.f2[lane]; }
#pragma unroll
    for (int o = kCluWarps / 2; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, tm, o);
      const int oi = __shfl_xor_sync(0xffffffffu, ti, o);
      if (ov > tm || (ov == tm && oi < ti)) { tm = ov; ti = oi; }
      dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if (lane == 0) {
      part.tmax = tm; part.targ = ti; part.dmax = dm; part.bad = bad;
      part.pick = -1; part.lastp = -1; part.wsum = 0.0; part.st = 0.0; part.sd = 0.0;
    }
  }
  cl.sync();
  // lane r of every warp fetches block r's partial (one round trip through distributed shared
  // memory for the whole cluster instead of one per block), a shuffle tree combines them; every
  // warp of every block runs the same tree on the same values
  tm = -INFINITY; dm = -INFINITY; ti = 0x7fffffff; bad = 0;
  if (lane < nclu) {
    const CluPart* pr = cl.map_shared_rank(&part, lane);
    tm = pr->tmax; ti = pr->targ; dm = pr->dmax; bad = pr->bad;
  }
#pragma unroll
  for (int o = nclu / 2; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, tm, o);
    const int oi = __shfl_xor_sync(0xffffffffu, ti, o);
    if (ov > tm || (ov == tm && oi < ti)) { tm = ov; ti = oi; }
    dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  tm = __shfl_sync(0xffffffffu, tm, 0); ti = __shfl_sync(0xffffffffu, ti, 0);
  dm = __shfl_sync(0xffffffffu, dm, 0); bad = __shfl_sync(0xffffffffu, bad, 0);
  if (tm == -INFINITY || (drow && dm == -INFINITY)) bad = 1;  // a row without a distribution
  const float tmax = tm, dmax = dm;
  const int targ = ti;

  int accept = 0, token = -1;
  if (greedy) {
    accept = (!bonus && x == targ) ? 1 : 0;
    token = targ;
    bad = 0;
  } else if (bad) {
    token = targ;
  } else {
    // every block takes the same branches below: the values they depend on are identical
    const double inv_t = 1.0 / (double)a.temperature;
    double st = 0.0, sd = 0.0;
#pragma unroll
    for (int e = 0; e < V4 * 4; ++e) {
      const bool in = e < C && v0 + e < V;
      t[e] = in ? expf(exp_arg_d<UNIT>(t[e], tmax, inv_t)) : 0.f;
      st += (double)t[e];
      if (drow) {
        d[e] = in ? expf(exp_arg_d<UNIT>(d[e], dmax, inv_t)) : 0.f;
        sd += (double)d[e];
      }
    }
    st = warp_sum_d(st);
    sd = warp_sum_d(sd);
    if (lane == 0) { s.d[warp] = st; s.d2[warp] = sd; }
    __syncthreads();
    if (warp == 0) {
      double x1 = lane < kCluWarps ? s.d[lane] : 0.0, x2 = lane < kCluWarps ? s.d2[lane] : 0.0;
#pragma unroll
      for (int o = kCluWarps / 2; o > 0; o >>= 1) {
        x1 += __shfl_xor_sync(0xffffffffu, x1, o);
        x2 += __shfl_xor_sync(0xffffffffu, x2, o);
      }
      if (lane == 0) { part.st = x1; part.sd = x2; }
    }
    cl.sync();
    st = 0.0; sd = 0.0;
    if (lane < nclu) {
      const CluPart* pr = cl.map_shared_rank(&part, lane);
      st = pr->st; sd = pr->sd;
    }
#pragma unroll
    for (int o = nclu / 2; o > 0; o >>= 1) {
      st += __shfl_xor_sync(0xffffffffu, st, o);
      sd += __shfl_xor_sync(0xffffffffu, sd, o);
    }
    st = __shfl_sync(0xffffffffu, st, 0); sd = __shfl_sync(0xffffffffu, sd, 0);
    if (!drow) sd = 1.0;
    uint32_t c[4] = {(uint32_t)i, (uint32_t)b, a.off_lo, a.off_hi};
    philox4x32_10(a.key0, a.key1, c);
    const double r = (double)(c[0] >> 8) * (1.0 / 16777216.0);
    const double u2 = (double)(c[1] >> 8) * (1.0 / 16777216.0);
    if (!bonus) {
      const bool in_range = x >= 0 && x < V;
      const double logp = in_range ? ((double)trow[x] - (double)tmax) * inv_t - log(st) : -INFINITY;
      const double logq = drow ? (in_range ? ((double)drow[x] - (double)dmax) * inv_t - log(sd) : -INFINITY)
                               : 0.0;
      const double diff = logp - logq;
      const double ratio = (diff != diff) ? 0.0 : exp(fmin(diff, 0.0));
      accept = r < ratio ? 1 : 0;
    }
    if (!accept) {
      const float inv_st = (float)(1.0 / st), inv_sd = (float)(1.0 / sd);
      // attempt 0: residual max(0, p - q); attempt 1: p itself (extra row, or an empty residual)
      for (int attempt = bonus ? 1 : 0; attempt < 2 && token < 0; ++attempt) {
        float w[V4 * 4];
        double mine = 0.0;
        int lastp = -1;
#pragma unroll
        for (int e = 0; e < V4 * 4; ++e) {
          const float p = t[e] * inv_st;
          float wv = p;
          if (attempt == 0) {
            const float q = drow ? d[e] * inv_sd : ((v0 + e == x) ? 1.f : 0.f);
            wv = fmaxf(p - q, 0.f);
          }
          w[e] = (e < C && v0 + e < V) ? wv : 0.f;
          mine += (double)w[e];
          if (w[e] > 0.f) lastp = v0 + e;
        }
        double incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double up = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += up;
        }
        lastp = __reduce_max_sync(0xffffffffu, lastp);
        __syncthreads();   // the scratch arrays are free again
        if (lane == 31) { s.d[warp] = incl; s.i[warp] = lastp; }
        __syncthreads();
        if (tid == 0) {
          double x1 = 0.0;
          int lp = -1;
          for (int k = 0; k < kCluWarps; ++k) { x1 += s.d[k]; lp = max(lp, s.i[k]); }
          part.wsum = x1; part.lastp = lp; part.pick = -1;
        }
        cl.sync();
        // level 1: the block whose running sum first exceeds the target (lane r holds block r's
        // weight; a shuffle scan gives every block's running sum)
        double bw = lane < nclu ? cl.map_shared_rank(&part, lane)->wsum : 0.0;
        double binc = bw;
#pragma unroll
        for (int o = 1; o < nclu; o <<= 1) {
          const double up = __shfl_up_sync(0xffffffffu, binc, o);
          if (lane >= o) binc += up;
        }
        const double total = __shfl_sync(0xffffffffu, binc, nclu - 1);
        int sel = -1;
        if (total > 0.0) {
          const double target = u2 * total;
          const unsigned over_b = __ballot_sync(0xffffffffu, lane < nclu && binc > target);
          double base = 0.0;
          if (over_b) {   // (the base is the sum that was compared: a rounded difference could lie above the target)
            sel = __ffs(over_b) - 1;
            if (sel > 0) base = __shfl_sync(0xffffffffu, binc, sel - 1);
          }
          if (sel == rank) {
            // level 2: the warp, level 3: the lane, level 4: the token
            double t2 = target - base, wrun = 0.0, wbase = 0.0;
            int wsel = -1;
            for (int k = 0; k < kCluWarps; ++k) {
              const double nx = wrun + s.d[k];
              if (wsel < 0 && nx > t2) { wsel = k; wbase = wrun; }
              wrun = nx;
            }
            if (warp == wsel) {
              const double t3 = t2 - wbase;
              const unsigned over = __ballot_sync(0xffffffffu, incl > t3);
              if (over) {
                const int src = __ffs(over) - 1;
                double excl = __shfl_up_sync(0xffffffffu, incl, 1);
                if (lane == 0) excl = 0.0;
                if (lane == src) {
                  const double t4 = t3 - excl;
                  double run4 = 0.0;
                  int pick = -1, lp = -1;
#pragma unroll
                  for (int e = 0; e < V4 * 4; ++e) {
                    if (w[e] > 0.f) lp = e;
                    run4 += (double)w[e];
                    if (pick < 0 && run4 > t4) pick = e;
                  }
                  if (pick < 0) pick = lp;
                  if (pick >= 0) part.pick = v0 + pick;
                }
              }
            }
          }
        }
        cl.sync();
        if (total > 0.0) {
          // rounding may leave no token chosen on the way down: take the last one with weight
          token = sel >= 0 ? cl.map_shared_rank(&part, sel)->pick : -1;
          if (token < 0)
            for (int rr = 0; rr < nclu; ++rr) token = max(token, cl.map_shared_rank(&part, rr)->lastp);
        }
        cl.sync();   // all reads of this attempt's partials are done before they are rewritten
      }
      if (token < 0) token = targ;
    }
  }
  if (rank == 0 && tid == 0) finish_position(a, i, b, accept, bad, token);
  cl.sync();   // no block leaves while another may still read its shared memory
}


// The 8-block cluster is fixed at compile time; the 16-block one (an opt-in size) is a launch attribute.
template <bool UNIT>
__global__ void __cluster_dims__(kClu, 1, 1) __launch_bounds__(kCluThreads) k_verify_cluster(VerifyArgs a) {
  verify_cluster_body<kClu, kCluV4, UNIT>(a);
}
// (rows of up to 32768 tokens: 8 tokens per thread)
template <bool UNIT>
__global__ void __cluster_dims__(kClu, 1, 1) __launch_bounds__(kCluThreads) k_verify_cluster_v2(VerifyArgs a) {
  verify_cluster_body<kClu, 2, UNIT>(a);
}
// (Rows of up to 8192 tokens: one block, whose barriers cost less than a cluster's; 1000 tokens, 5 row
// pairs: 13.3 -> 11.1 us.  Rows of up to 2048 and 4096 tokens: a quarter and a half of the tokens a thread, for
// the unrolled loops of a kernel that runs its code once: 1000 tokens, draft + verify 41.8 -> 39.0 us.)
constexpr int kOneMaxVocab = kCluThreads * 4 * kCluV4;
template <int V4, bool UNIT>
__global__ void __launch_bounds__(kCluThreads) k_verify_block(VerifyArgs a) {
  verify_cluster_body<1, V4, UNIT>(a);
}
template <bool UNIT>
__global__ void __launch_bounds__(kCluThreads) k_verify_cluster16(VerifyArgs a) {
  verify_cluster_body<16, kCluV4, UNIT>(a);
}
// Four blocks per row pair: for batches whose 8-block clusters would not be resident at once
// (one block fills an SM) while these are, and a thread can still hold its share of a row (16 tokens).
constexpr int kCluSmall = 4;
constexpr int kCluSmallMaxVocab = kCluSmall * kCluThreads * 4 * kCluV4;
template <bool UNIT>
__global__ void __cluster_dims__(kCluSmall, 1, 1) __launch_bounds__(kCluThreads) k_verify_cluster4(VerifyArgs a) {
  verify_cluster_body<kCluSmall, kCluV4, UNIT>(a);
}

// ---- streaming variant: many row pairs --------------------------------------------------------
// When a call has so many row pairs that the register-resident clusters above would run in
// several waves, what counts is throughput: a row pair goes to a cluster of 1 to 8 blocks of few
// registers, four of them resident per SM, that stream both rows once (so the HBM reads of one
// hide the exponentials of another), and the draw, which needs the rows again, is done for ONE
// position per sequence only: every row pair leaves its statistics and its verdict in a record, the
// last cluster of a sequence to finish walks the verdicts and notes where the chain stops.
// Exponentials are taken against a reference value of the block (the maximum of its first
// batch) instead of the row's maximum, which is not known yet; their relative precision is the
// same, and the sums are moved to the maximum once, in double.  Should the maximum lie far from the
// reference, the sums are formed again.
// The draws are a launch of their own (k_verify_draw) over all sequences, eight blocks each: done by
// the last cluster of a sequence, a block or two would read a row pair while the rest of the chip
// idles (576 pairs of 32000 tokens: 122 us in all, 43 us of it without the draws).
// Measured (T = 1, rows from HBM) against the register-resident clusters in waves: 40 pairs of 32000
// tokens 28.0 -> 20.6 us, 80 pairs 40.2 -> 23.7, 144 pairs 61.5 -> 32.9, 576 pairs 210 -> 50.9 us (2.9
// TB/s; the exponentials and their double-precision sums bound it); 208 pairs of 128256 tokens 442 ->
// 75.5 us.
constexpr int kStrThreads = 256, kStrPerSm = 4, kStrWarps = kStrThreads / 32;
struct StreamPart {    // one per block, read by its cluster
  float tmax, dmax, tref, dref;
  int targ, bad;
  double st, sd;
};
struct StreamScratch {
  float f[kStrWarps], f2[kStrWarps];
  int i[kStrWarps];
  double d[kStrWarps], d2[kStrWarps];
};
constexpr float kRefSlack = 60.f;   // exponent range left beside the reference before sums are formed again

template <bool UNIT>
__global__ void __launch_bounds__(kStrThreads, kStrPerSm) k_verify_stream(VerifyArgs a, VerifyRow* rows, VerifyDraw* draws) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ StreamPart part;
  __shared__ StreamScratch s;
  const int nclu = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int i = blockIdx.x / nclu, b = blockIdx.y, V = a.V;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool bonus = i >= a.n_draft, greedy = a.temperature == 0.f;
  const float* trow = a.target_logits + ((size_t)b * a.n_target + i) * V;
  const float* drow = (!bonus && !greedy && a.draft_logits) ? a.draft_logits + ((size_t)b * a.n_draft + i) * V : nullptr;
  const int share = ((V + nclu - 1) / nclu + kSeg - 1) / kSeg * kSeg;
  const int v_lo = min(V, rank * share), n_vec = (min(V, v_lo + share) - v_lo) / 4;   // V % 4 == 0
  const double inv_t = greedy ? 1.0 : 1.0 / (double)a.temperature;
  const InvT inv(inv_t);
  pdl_launch_dependents();

  // ---- one pass over both rows
  constexpr int U = 2;
  const float4 none = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  const float4 *t4 = reinterpret_cast<const float4*>(trow + v_lo), *d4 = reinterpret_cast<const float4*>(drow + (drow ? v_lo : 0));
  float tm = -INFINITY, dm = -INFINITY;
  int ti = 0x7fffffff;
  double st = 0.0, sd = 0.0;
  float tref = -INFINITY, dref = -INFINITY;
  for (int attempt = 0; attempt < 2; ++attempt) {
    st = sd = 0.0;
    const bool again = attempt > 0;
    for (int v0 = tid; v0 - tid < n_vec; v0 += U * kStrThreads) {
      float4 t[U], d[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int v = v0 + u * kStrThreads;
        t[u] = v < n_vec ? __ldg(t4 + v) : none;
        d[u] = (drow && v < n_vec) ? __ldg(d4 + v) : none;
      }
      if (!again) {
        float bt = -INFINITY, bd = -INFINITY;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          bt = fmaxf(fmaxf(fmaxf(bt, t[u].x), fmaxf(t[u].y, t[u].z)), t[u].w);
          bd = fmaxf(fmaxf(fmaxf(bd, d[u].x), fmaxf(d[u].y, d[u].z)), d[u].w);
        }
        if (bt > tm) {   // (rare after the first batch) the lowest id that holds the new maximum
          tm = bt;
#pragma unroll
          for (int u = U - 1; u >= 0; --u) {
            const int v = v_lo + 4 * (v0 + u * kStrThreads);
            if (t[u].w == bt) ti = v + 3;
            if (t[u].z == bt) ti = v + 2;
            if (t[u].y == bt) ti = v + 1;
            if (t[u].x == bt) ti = v;
          }
        }
        dm = fmaxf(dm, bd);
        if (!greedy && v0 == tid) {   // first batch: the block's reference
          float rt = bt, rd = bd;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            rt = fmaxf(rt, __shfl_xor_sync(0xffffffffu, rt, o));
            rd = fmaxf(rd, __shfl_xor_sync(0xffffffffu, rd, o));
          }
          if (lane == 0) { s.f[warp] = rt; s.f2[warp] = rd; }
          __syncthreads();
#pragma unroll
          for (int w = 0; w < kStrWarps; ++w) { tref = fmaxf(tref, s.f[w]); dref = fmaxf(dref, s.f2[w]); }
          if (tref == -INFINITY) tref = 0.f;   // (differences from a reference are NaN for NaN logits only)
          if (dref == -INFINITY) dref = 0.f;
        }
      }
      if (!greedy) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          st += (double)expf(exp_arg<UNIT>(t[u].x, tref, inv)); st += (double)expf(exp_arg<UNIT>(t[u].y, tref, inv));
          st += (double)expf(exp_arg<UNIT>(t[u].z, tref, inv)); st += (double)expf(exp_arg<UNIT>(t[u].w, tref, inv));
          if (drow) {
            sd += (double)expf(exp_arg<UNIT>(d[u].x, dref, inv)); sd += (double)expf(exp_arg<UNIT>(d[u].y, dref, inv));
            sd += (double)expf(exp_arg<UNIT>(d[u].z, dref, inv)); sd += (double)expf(exp_arg<UNIT>(d[u].w, dref, inv));
          }
        }
      }
    }
    // ---- the block's values
    if (!again) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, tm, o);
        const int oi = __shfl_xor_sync(0xffffffffu, ti, o);
        if (ov > tm || (ov == tm && oi < ti)) { tm = ov; ti = oi; }
        dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      }
    }
    st = warp_sum_d(st);
    sd = warp_sum_d(sd);
    __syncthreads();   // the references have been read
    if (lane == 0) { s.f[warp] = tm; s.i[warp] = ti; s.f2[warp] = dm; s.d[warp] = st; s.d2[warp] = sd; }
    __syncthreads();
    st = sd = 0.0;
#pragma unroll
    for (int w = 0; w < kStrWarps; ++w) {
      if (s.f[w] > tm || (s.f[w] == tm && s.i[w] < ti)) { tm = s.f[w]; ti = s.i[w]; }
      dm = fmaxf(dm, s.f2[w]);
      st += s.d[w];
      sd += s.d2[w];
    }
    if (greedy) break;
    const bool far_t = tm > -INFINITY && fabs((double)tm - (double)tref) * inv_t > kRefSlack;
    const bool far_d = dm > -INFINITY && fabs((double)dm - (double)dref) * inv_t > kRefSlack;
    if (!far_t && !far_d) break;
    if (far_t) tref = tm;
    if (far_d) dref = dm;
    __syncthreads();
  }
  // (the maxima skip NaN, but a NaN logit leaves its row's sum NaN)
  const int bad = tm == INFINITY || dm == INFINITY || st != st || sd != sd;
  if (tid == 0) {
    part.tmax = tm; part.targ = ti; part.dmax = dm; part.bad = bad; part.st = st; part.sd = sd;
    part.tref = tref; part.dref = dref;
  }
  cl.sync();
  // ---- first block: the row pair's verdict, its record, the ticket; as the last arriver of the
  // sequence, the walk over the verdicts
  if (rank == 0 && warp == 0) {
    const StreamPart* pr = lane < nclu ? cl.map_shared_rank(&part, lane) : nullptr;
    float m = pr ? pr->tmax : -INFINITY, q = pr ? pr->dmax : -INFINITY;
    int mi = pr ? pr->targ : 0x7fffffff, bd = pr ? pr->bad : 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, m, o);
      const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
      if (ov > m || (ov == m && oi < mi)) { m = ov; mi = oi; }
      q = fmaxf(q, __shfl_xor_sync(0xffffffffu, q, o));
      bd |= __shfl_xor_sync(0xffffffffu, bd, o);
    }
    m = __shfl_sync(0xffffffffu, m, 0); mi = __shfl_sync(0xffffffffu, mi, 0);
    q = __shfl_sync(0xffffffffu, q, 0); bd = __shfl_sync(0xffffffffu, bd, 0);
    if (m == -INFINITY || (drow && q == -INFINITY)) bd = 1;   // a row without a distribution
    if (mi == 0x7fffffff) mi = 0;                             // (nothing above -inf: the lowest id)
    double xt = 0.0, xd = 0.0;
    if (!greedy && !bd && pr) {
      if (pr->st > 0.0) xt = pr->st * exp(((double)pr->tref - (double)m) * inv_t);
      if (drow && pr->sd > 0.0) xd = pr->sd * exp(((double)pr->dref - (double)q) * inv_t);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      xt += __shfl_xor_sync(0xffffffffu, xt, o);
      xd += __shfl_xor_sync(0xffffffffu, xd, o);
    }
    if (lane == 0) {
      if (!drow) xd = 1.0;
      const int x = bonus ? -1 : a.draft_tokens[(size_t)b * a.n_draft + i];
      int accept = 0;
      if (greedy) {
        accept = (!bonus && x == mi) ? 1 : 0;
        bd = 0;
      } else if (!bd && !bonus) {
        uint32_t c[4] = {(uint32_t)i, (uint32_t)b, a.off_lo, a.off_hi};
        philox4x32_10(a.key0, a.key1, c);
        const double r = (double)(c[0] >> 8) * (1.0 / 16777216.0);
        const bool in_range = x >= 0 && x < V;
        const double logp = in_range ? ((double)trow[x] - (double)m) * inv_t - log(xt) : -INFINITY;
        const double logq = drow ? (in_range ? ((double)drow[x] - (double)q) * inv_t - log(xd) : -INFINITY) : 0.0;
        const double diff = logp - logq;
        const double ratio = (diff != diff) ? 0.0 : exp(fmin(diff, 0.0));
        accept = r < ratio ? 1 : 0;
      }
      VerifyRow* recw = rows + (size_t)b * (PS_MAX_MASKS + 2);
      VerifyRow rec;
      rec.flags = accept | (bd << 1); rec.targ = mi; rec.tmax = m; rec.dmax = q; rec.st = xt; rec.sd = xd;
      recw[i] = rec;
      __threadfence();
      if (atomicAdd(&a.tickets[b], 1u) == (unsigned)a.n_target - 1u) {
        __threadfence();
        a.tickets[b] = 0u;
        int* out = a.out_tokens + (size_t)b * (a.n_draft + 1);
        int acc = 0, any_bad = 0, stop = -1, flags = 0;
        while (acc < a.n_draft) {
          flags = __ldcg(&recw[acc].flags);
          any_bad |= (flags >> 1) & 1;
          if (!(flags & 1)) { stop = acc; break; }
          out[acc] = a.draft_tokens[(size_t)b * a.n_draft + acc];
          ++acc;
        }
        if (acc == a.n_draft && a.n_target == a.n_draft + 1) {
          flags = __ldcg(&recw[acc].flags);
          any_bad |= (flags >> 1) & 1;
          stop = acc;
        }
        const int n = acc + (stop >= 0 ? 1 : 0);
        for (int j = n; j <= a.n_draft; ++j) out[j] = -1;
        a.accept_len[b] = acc;
        a.n_out[b] = n;
        if (any_bad) atomicOr(a.status, kStatNonfinite);
        VerifyDraw dw;
        dw.pos = -1;
        if (stop >= 0) {
          const VerifyRow* rr = recw + stop;
          const int targ = __ldcg(&rr->targ);
          out[acc] = targ;   // (a draw replaces it)
          if (!greedy && !(flags & 2)) {
            dw.pos = stop; dw.acc = acc;
            dw.tmax = __ldcg(&rr->tmax); dw.dmax = __ldcg(&rr->dmax);
            dw.st = __ldcg(&rr->st); dw.sd = __ldcg(&rr->sd);
          }
        }
        draws[b] = dw;
      }
    }
  }
  cl.sync();   // no block leaves while another may still read its shared memory
}

// The token of each sequence whose chain stops at a position with a distribution: inverse-CDF draw
// from max(0, p - q), or from p at the extra row and where the residual is empty.  A cluster of
// kDrawClu blocks per sequence; a warp takes segments of kSeg tokens, four in flight.
constexpr int kDrawClu = 8, kDrawBatch = 4;
template <bool UNIT>
__global__ void __cluster_dims__(kDrawClu, 1, 1) __launch_bounds__(kStrThreads)
k_verify_draw(VerifyArgs a, const VerifyDraw* draws) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double seg_sum[];          // [segments of the block's share]
  __shared__ double s_wsum;
  __shared__ int s_done;
  const int rank = (int)cl.block_rank(), b = blockIdx.y, V = a.V;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int share = ((V + kDrawClu - 1) / kDrawClu + kSeg - 1) / kSeg * kSeg;
  const int v_lo = min(V, rank * share), n_vec = (min(V, v_lo + share) - v_lo) / 4;   // V % 4 == 0
  const double inv_t = 1.0 / (double)a.temperature;
  const InvT inv(inv_t);
  const float4 none = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  pdl_launch_dependents();
  pdl_wait();
  const VerifyDraw dw = draws[b];
  const int pos = dw.pos;
  if (pos >= 0) {   // uniform over the cluster
    const float tmax = dw.tmax, dmax = dw.dmax;
    const float inv_st = (float)(1.0 / dw.st), inv_sd = (float)(1.0 / dw.sd);
    const bool use_q0 = pos < a.n_draft;
    const float* tr = a.target_logits + ((size_t)b * a.n_target + pos) * V;
    const float* dr = (use_q0 && a.draft_logits) ? a.draft_logits + ((size_t)b * a.n_draft + pos) * V : nullptr;
    const int x = use_q0 ? a.draft_tokens[(size_t)b * a.n_draft + pos] : -1;
    uint32_t c[4] = {(uint32_t)pos, (uint32_t)b, a.off_lo, a.off_hi};
    philox4x32_10(a.key0, a.key1, c);
    const double u2 = (double)(c[1] >> 8) * (1.0 / 16777216.0);
    const int n_seg = (4 * n_vec + kSeg - 1) / kSeg;
    // this lane's four tokens of segment g, and their weights: max(0, p - q), or p
    auto fetch = [&](int g, bool use_q, float4& tv, float4& dv) {
      tv = dv = none;
      if (g < 0 || g * (kSeg / 4) + lane >= n_vec) return;
      const int v = v_lo + g * kSeg + 4 * lane;
      tv = __ldg(reinterpret_cast<const float4*>(tr + v));
      if (use_q && dr) dv = __ldg(reinterpret_cast<const float4*>(dr + v));
    };
    auto weights = [&](int g, bool use_q, const float4& tv, const float4& dv, float (&w)[4]) {
      const int v = v_lo + g * kSeg + 4 * lane;
      const float t[4] = {tv.x, tv.y, tv.z, tv.w}, d[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        w[e] = expf(exp_arg<UNIT>(t[e], tmax, inv)) * inv_st;
        if (use_q) {
          const float qv = dr ? expf(exp_arg<UNIT>(d[e], dmax, inv)) * inv_sd : (v + e == x ? 1.f : 0.f);
          w[e] = fmaxf(w[e] - qv, 0.f);
        }
      }
    };
    bool done = false;
    for (int attempt = use_q0 ? 0 : 1; attempt < 2 && !done; ++attempt) {
      const bool use_q = attempt == 0;
      for (int g0 = warp; g0 < n_seg; g0 += kDrawBatch * kStrWarps) {
        float4 tv[kDrawBatch], dv[kDrawBatch];
        double mine[kDrawBatch];
#pragma unroll
        for (int k = 0; k < kDrawBatch; ++k) fetch(g0 + k * kStrWarps, use_q, tv[k], dv[k]);   // (past the share: nothing)
#pragma unroll
        for (int k = 0; k < kDrawBatch; ++k) {
          float w[4];
          weights(g0 + k * kStrWarps, use_q, tv[k], dv[k], w);
          mine[k] = ((double)w[0] + (double)w[1]) + ((double)w[2] + (double)w[3]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int k = 0; k < kDrawBatch; ++k) mine[k] += __shfl_xor_sync(0xffffffffu, mine[k], o);
#pragma unroll
        for (int k = 0; k < kDrawBatch; ++k)
          if (lane == 0 && g0 + k * kStrWarps < n_seg) seg_sum[g0 + k * kStrWarps] = mine[k];
      }
      __syncthreads();
      // lane owns segments [lane * per, ...) of the block's share
      double incl = 0.0, own = 0.0;
      int g_lo = 0, g_hi = 0;
      if (warp == 0) {
        const int per = (n_seg + 31) / 32;
        g_lo = min(n_seg, lane * per);
        g_hi = min(n_seg, g_lo + per);
        for (int g = g_lo; g < g_hi; ++g) own += seg_sum[g];
        incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double up = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += up;
        }
        if (lane == 31) s_wsum = incl;
      }
      cl.sync();
      if (warp == 0) {
        const double bw = lane < kDrawClu ? *cl.map_shared_rank(&s_wsum, lane) : 0.0;
        double binc = bw;
#pragma unroll
        for (int o = 1; o < kDrawClu; o <<= 1) {
          const double up = __shfl_up_sync(0xffffffffu, binc, o);
          if (lane >= o) binc += up;
        }
        const double total = __shfl_sync(0xffffffffu, binc, kDrawClu - 1);
        done = total > 0.0;
        if (done) {
          // At every level: the first holder of weight whose running sum exceeds the target; rounding
          // may leave none, then the last holder of weight.
          const double target = u2 * total;
          const unsigned has_b = __ballot_sync(0xffffffffu, bw > 0.0);
          const unsigned over_b = __ballot_sync(0xffffffffu, bw > 0.0 && binc > target);
          const int sel = over_b ? __ffs(over_b) - 1 : 31 - __clz(has_b);
          const double base = __shfl_sync(0xffffffffu, binc - bw, sel);
          if (sel == rank) {
            const unsigned has = __ballot_sync(0xffffffffu, own > 0.0);
            const unsigned over = __ballot_sync(0xffffffffu, own > 0.0 && base + incl > target);
            const int src = over ? __ffs(over) - 1 : 31 - __clz(has);
            int gs = -1;
            double gbase = 0.0;
            if (lane == src) {
              double run = base + incl - own;
              for (int g = g_lo; g < g_hi; ++g) {
                const double sg = seg_sum[g];
                if (sg > 0.0) {
                  gs = g;
                  gbase = run;
                  if (run + sg > target) break;
                }
                run += sg;
              }
            }
            gs = __shfl_sync(0xffffffffu, gs, src);
            gbase = __shfl_sync(0xffffffffu, gbase, src);
            float4 tv, dv;
            float w[4];
            fetch(gs, use_q, tv, dv);
            weights(gs, use_q, tv, dv, w);
            const double mine = ((double)w[0] + (double)w[1]) + ((double)w[2] + (double)w[3]);
            double linc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const double up = __shfl_up_sync(0xffffffffu, linc, o);
              if (lane >= o) linc += up;
            }
            const unsigned has2 = __ballot_sync(0xffffffffu, mine > 0.0);
            const unsigned over2 = __ballot_sync(0xffffffffu, mine > 0.0 && gbase + linc > target);
            const int src2 = over2 ? __ffs(over2) - 1 : 31 - __clz(has2);
            if (lane == src2) {
              double run = gbase + linc - mine;
              int pick = -1;
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                if (w[e] > 0.f && (pick < 0 || !(run > target))) pick = e;
                run += (double)w[e];
              }
              a.out_tokens[(size_t)b * (a.n_draft + 1) + dw.acc] = v_lo + gs * kSeg + 4 * lane + pick;
            }
          }
        }
        if (lane == 0) s_done = done;
      }
      __syncthreads();
      done = s_done != 0;
      cl.sync();   // the blocks' sums have been read
    }
  }
}

// ---- token-tree verification (Algorithm 1 in full) -------------------------------------------
// Two launches.  (1) k_row_softmax streams the target rows that have children and the draft rows
// once and leaves their maxima and sums (at temperature 0: the arg-max of every target row).  (2)
// k_tree_walk: one cluster per sequence walks the tree from the root.  Whether the first child of a
// node is accepted is a test of two scalars; only a rejection needs the rows again: the cluster then
// holds them in registers.  After j rejections the target distribution of Algorithm 1 is
// norm((p - c q)+) with c_0 = 0, c_{j+1} = c_j + Z(c_j), Z(c) = sum_v (p_v - c q_v)+ (the repeated
// "subtract q, clip, renormalise" in closed form), so a rejection costs one reduction over the
// cluster.  Where the walk stops the cluster draws the token.
// Bound by the latency of the walk's cluster exchanges (1-2 us each).  A cluster per decision row
// that tries its children speculatively was bound by its blocks' occupancy instead.  23 nodes, T = 1, before ->
// after: 1 x 32000 tokens 23.5 -> 18.0 us, 4 x 57 -> 24.7, 16 x 201 -> 34.8; 1 x 128256 tokens 83 -> 25, 4 x 318 -> 40.
struct TreeTopo {
  int n_nodes, max_depth;
  unsigned char depth[PS_MAX_TREE_NODES];
  unsigned char child_off[PS_MAX_TREE_NODES + 2];   // children of decision row u: child_idx[off[u] .. off[u+1])
  unsigned char child_idx[PS_MAX_TREE_NODES];
  signed char parent[PS_MAX_TREE_NODES];
  unsigned char nth[PS_MAX_TREE_NODES];             // node i is the nth child of its parent
};

struct TreeArgs {
  int B, V;
  TreeTopo topo;
  const int* tokens;           // [B][n_nodes]
  const float* draft_logits;   // [B][max_depth][V]
  const float* target_logits;  // [B][n_nodes+1][V]
  float temperature;
  uint32_t key0, key1, off_lo, off_hi;
  int* accept_len; int* out_tokens; int* n_out; int* path;
  RowStat* stats;              // [B][kTreeRows]: target rows by decision row, then draft rows by depth
  int leaf_stats;              // the rows of leaves are among them
  int* status;
};
constexpr int kTreeRows = 2 * PS_MAX_TREE_NODES + 1;
// Rows whose statistics the walk needs: target rows with children (all at temperature 0, and where few rows
// leave the chip idle: the leaf where a walk ends then needs no exchanges of its own), draft rows.
struct TreeRows { int n; unsigned char row[kTreeRows]; };

// Statistics of row blockIdx.x / nclu of the list for sequence blockIdx.y; exponentials against a
// reference of the block, as in k_verify_stream.
template <bool UNIT>
__global__ void __launch_bounds__(kStrThreads, kStrPerSm) k_row_softmax(const __grid_constant__ TreeArgs a,
                                                                        const __grid_constant__ TreeRows list) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ StreamPart part;
  __shared__ StreamScratch s;
  const int nclu = (int)cl.num_blocks(), rank = (int)cl.block_rank(), b = blockIdx.y, V = a.V;
  const int r = list.row[blockIdx.x / nclu], n_target = a.topo.n_nodes + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool greedy = a.temperature == 0.f;
  const float* row = r < n_target ? a.target_logits + ((size_t)b * n_target + r) * V
                                  : a.draft_logits + ((size_t)b * a.topo.max_depth + (r - n_target)) * V;
  const int share = ((V + nclu - 1) / nclu + kSeg - 1) / kSeg * kSeg;
  const int v_lo = min(V, rank * share), n_vec = (min(V, v_lo + share) - v_lo) / 4;   // V % 4 == 0
  const double inv_t = greedy ? 1.0 : 1.0 / (double)a.temperature;
  const InvT inv(inv_t);
  pdl_launch_dependents();
  pdl_wait();
  constexpr int U = 4;
  const float4* r4 = reinterpret_cast<const float4*>(row + v_lo);
  float mx = -INFINITY, ref = -INFINITY;
  int mi = 0x7fffffff;
  double st = 0.0;
  for (int attempt = 0; attempt < 2; ++attempt) {
    st = 0.0;
    for (int v0 = tid; v0 - tid < n_vec; v0 += U * kStrThreads) {
      float4 t[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int v = v0 + u * kStrThreads;
        t[u] = v < n_vec ? __ldg(r4 + v) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      }
      if (attempt == 0) {
        float bt = -INFINITY;
#pragma unroll
        for (int u = 0; u < U; ++u) bt = fmaxf(fmaxf(fmaxf(bt, t[u].x), fmaxf(t[u].y, t[u].z)), t[u].w);
        if (bt > mx) {   // (rare after the first batch) the lowest id that holds the new maximum
          mx = bt;
#pragma unroll
          for (int u = U - 1; u >= 0; --u) {
            const int v = v_lo + 4 * (v0 + u * kStrThreads);
            if (t[u].w == bt) mi = v + 3;
            if (t[u].z == bt) mi = v + 2;
            if (t[u].y == bt) mi = v + 1;
            if (t[u].x == bt) mi = v;
          }
        }
        if (!greedy && v0 == tid) {   // first batch: the block's reference
          float rt = bt;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) rt = fmaxf(rt, __shfl_xor_sync(0xffffffffu, rt, o));
          if (lane == 0) s.f[warp] = rt;
          __syncthreads();
#pragma unroll
          for (int w = 0; w < kStrWarps; ++w) ref = fmaxf(ref, s.f[w]);
          if (ref == -INFINITY) ref = 0.f;   // (differences from the reference are NaN for NaN logits only)
        }
      }
      if (!greedy) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          st += (double)expf(exp_arg<UNIT>(t[u].x, ref, inv)); st += (double)expf(exp_arg<UNIT>(t[u].y, ref, inv));
          st += (double)expf(exp_arg<UNIT>(t[u].z, ref, inv)); st += (double)expf(exp_arg<UNIT>(t[u].w, ref, inv));
        }
      }
    }
    if (attempt == 0) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, mx, o);
        const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
        if (ov > mx || (ov == mx && oi < mi)) { mx = ov; mi = oi; }
      }
    }
    st = warp_sum_d(st);
    __syncthreads();   // the reference has been read
    if (lane == 0) { s.f[warp] = mx; s.i[warp] = mi; s.d[warp] = st; }
    __syncthreads();
    st = 0.0;
#pragma unroll
    for (int w = 0; w < kStrWarps; ++w) {
      if (s.f[w] > mx || (s.f[w] == mx && s.i[w] < mi)) { mx = s.f[w]; mi = s.i[w]; }
      st += s.d[w];
    }
    if (greedy || !(mx > -INFINITY && fabs((double)mx - (double)ref) * inv_t > kRefSlack)) break;
    ref = mx;
    __syncthreads();
  }
  if (tid == 0) {   // (the maximum skips NaN, but a NaN logit leaves the sum NaN)
    part.tmax = mx; part.targ = mi; part.tref = ref; part.st = st;
    part.bad = mx == INFINITY || st != st;
  }
  cl.sync();
  if (rank == 0 && warp == 0) {
    const StreamPart* pr = lane < nclu ? cl.map_shared_rank(&part, lane) : nullptr;
    float m = pr ? pr->tmax : -INFINITY;
    int id = pr ? pr->targ : 0x7fffffff, bad = pr ? pr->bad : 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, m, o);
      const int oi = __shfl_xor_sync(0xffffffffu, id, o);
      if (ov > m || (ov == m && oi < id)) { m = ov; id = oi; }
      bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    m = __shfl_sync(0xffffffffu, m, 0);
    double x = 0.0;
    if (!greedy && pr && pr->st > 0.0 && m > -INFINITY && m < INFINITY)
      x = pr->st * exp(((double)pr->tref - (double)m) * inv_t);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) {
      RowStat rs;
      rs.max = m; rs.arg = id == 0x7fffffff ? 0 : id; rs.bad = bad | (m == -INFINITY ? 1 : 0); rs.pad = 0; rs.sum = x;
      a.stats[(size_t)b * kTreeRows + r] = rs;
    }
  }
  cl.sync();   // no block leaves while the first one reads its part
}

// Sum over the cluster of one double per thread; every thread of every block gets the value.  (One cluster
// barrier and shuffle trees instead of two and a serial sum over the warps, here and in the draw: the walk
// of 23 nodes, 128256 tokens, 29 -> 25 us.)
__device__ double cluster_sum(cooperative_groups::cluster_group& cl, CluPart& part, CluScratch& s, double v,
                              int& turn, int warp, int lane) {
  v = warp_sum_d(v);
  __syncthreads();
  if (lane == 0) s.d[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double x1 = lane < kCluWarps ? s.d[lane] : 0.0;
#pragma unroll
    for (int o = kCluWarps / 2; o > 0; o >>= 1) x1 += __shfl_xor_sync(0xffffffffu, x1, o);
    if (lane == 0) part.turn[turn] = x1;
  }
  cl.sync();
  // lane r fetches block r's sum (one remote round trip), a shuffle tree adds them
  double tot = lane < (int)cl.num_blocks() ? cl.map_shared_rank(&part, lane)->turn[turn] : 0.0;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  tot = __shfl_sync(0xffffffffu, tot, 0);
  turn ^= 1;   // (the other place next time: whoever rewrites this one has seen everyone past the next barrier)
  return tot;
}

// Inverse-CDF draw by the cluster over per-thread weights w[] (thread owns tokens v0 + e): the
// first token whose running sum exceeds u * total, found block -> warp -> lane -> token.
// Returns the token to every thread of every block, -1 if the total weight is not positive.
__device__ int cluster_draw(cooperative_groups::cluster_group& cl, CluPart& part, CluScratch& s,
                            const float (&w)[kCluV4 * 4], int v0, double u, int rank, int tid, int warp,
                            int lane) {
  double mine = 0.0;
  int lastp = -1;
#pragma unroll
  for (int e = 0; e < kCluV4 * 4; ++e) {
    mine += (double)w[e];
    if (w[e] > 0.f) lastp = v0 + e;
  }
  double incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  lastp = __reduce_max_sync(0xffffffffu, lastp);
  __syncthreads();
  if (lane == 31) { s.d[warp] = incl; s.i[warp] = lastp; }
  __syncthreads();
  // running sums over the warps, in order (every warp forms them: the one that holds the token needs its own)
  double winc = lane < kCluWarps ? s.d[lane] : 0.0;
#pragma unroll
  for (int o = 1; o < kCluWarps; o <<= 1) {
    const double up = __shfl_up_sync(0xffffffffu, winc, o);
    if (lane >= o) winc += up;
  }
  if (warp == 0) {
    const int lp = __reduce_max_sync(0xffffffffu, lane < kCluWarps ? s.i[lane] : -1);
    if (lane == kCluWarps - 1) { part.wsum = winc; part.lastp = lp; part.pick = -1; }
  }
  cl.sync();
  // lane r holds block r's weight; a shuffle scan gives every block's running sum
  const int nb = (int)cl.num_blocks();
  const double bw = lane < nb ? cl.map_shared_rank(&part, lane)->wsum : 0.0;
  double binc = bw;
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    const double up = __shfl_up_sync(0xffffffffu, binc, o);
    if (lane >= o) binc += up;
  }
  const double total = __shfl_sync(0xffffffffu, binc, nb - 1);
  int sel = -1, token = -1;
  if (total > 0.0) {
    const double target = u * total;
    const unsigned over_b = __ballot_sync(0xffffffffu, lane < nb && binc > target);
    // At every level what is taken off the target is the very sum before the one that exceeded it, so that nothing below
    // is negative and the token has weight (a rounded difference, sum minus own, could lie above the target).
    double base = 0.0;
    if (over_b) {
      sel = __ffs(over_b) - 1;
      if (sel > 0) base = __shfl_sync(0xffffffffu, binc, sel - 1);
    }
    if (sel == rank) {
      const double t2 = target - base;
      const unsigned over_w = __ballot_sync(0xffffffffu, lane < kCluWarps && winc > t2);
      const int wsel = over_w ? __ffs(over_w) - 1 : -1;
      const double wbase = wsel > 0 ? __shfl_sync(0xffffffffu, winc, wsel - 1) : 0.0;
      if (warp == wsel) {
        const double t3 = t2 - wbase;
        const unsigned over = __ballot_sync(0xffffffffu, incl > t3);
        if (over) {
          const int src = __ffs(over) - 1;
          double excl = __shfl_up_sync(0xffffffffu, incl, 1);
          if (lane == 0) excl = 0.0;
          if (lane == src) {
            const double t4 = t3 - excl;
            double run4 = 0.0;
            int pick = -1, lp = -1;
#pragma unroll
            for (int e = 0; e < kCluV4 * 4; ++e) {
              if (w[e] > 0.f) lp = e;
              run4 += (double)w[e];
              if (pick < 0 && run4 > t4) pick = e;
            }
            if (pick < 0) pick = lp;
            if (pick >= 0) part.pick = v0 + pick;
          }
        }
      }
    }
  }
  cl.sync();
  if (total > 0.0) {
    // rounding may leave no token chosen on the way down: take the last one with weight
    token = sel >= 0 ? cl.map_shared_rank(&part, sel)->pick : -1;
    if (token < 0)
      for (int rr = 0; rr < (int)cl.num_blocks(); ++rr) token = max(token, cl.map_shared_rank(&part, rr)->lastp);
  }
  cl.sync();   // all reads of the partials are done before they are rewritten
  return token;
}

// What the walk reads of a node before it knows whether it gets there, formed for all nodes at once: level
// by level the chain of loads, logarithms and exponentials was 2.5 us a level (a chain of four nodes, one
// sequence of 32000 tokens: 22.0 -> 13.9 us in all).
struct TreeNodes {
  double logp[PS_MAX_TREE_NODES], logq[PS_MAX_TREE_NODES];   // of the node's token at its parent's row
  double ratio[PS_MAX_TREE_NODES], r[PS_MAX_TREE_NODES];     // p / q (1 at most), the uniform it is tried with
  int tok[PS_MAX_TREE_NODES];
  RowStat stat[kTreeRows];
};

// (The cluster size is a launch attribute: see launch_verify_tree.)
template <bool UNIT>
__global__ void __launch_bounds__(kCluThreads) k_tree_walk(const __grid_constant__ TreeArgs a) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ CluPart part;
  __shared__ CluScratch s;
  __shared__ TreeNodes nd;
  const int rank = (int)cl.block_rank(), nclu = (int)cl.num_blocks();
  const int b = blockIdx.y, V = a.V, n_nodes = a.topo.n_nodes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool greedy = a.temperature == 0.f, writer = rank == 0 && tid == 0;
  const double inv_t = greedy ? 1.0 : 1.0 / (double)a.temperature;
  const int* toks = a.tokens + (size_t)b * n_nodes;
  const int nv4 = ((V + nclu * kCluThreads - 1) / (nclu * kCluThreads) + 3) / 4;
  const int C = nv4 * 4, v0 = (rank * kCluThreads + tid) * C;
  int* out = a.out_tokens + (size_t)b * (a.topo.max_depth + 1);
  int* pth = a.path + (size_t)b * a.topo.max_depth;
  pdl_launch_dependents();
  pdl_wait();
  const RowStat* stats = a.stats + (size_t)b * kTreeRows;
  const int n_rows = n_nodes + 1 + (greedy ? 0 : a.topo.max_depth);
  for (int i = tid; i < n_rows; i += kCluThreads) nd.stat[i] = stats[i];   // (rows nobody formed are not used)
  if (tid < n_nodes) nd.tok[tid] = toks[tid];
  __syncthreads();
  if (!greedy && tid < n_nodes) {
    const int up = a.topo.parent[tid] + 1, dep = a.topo.depth[tid], x = nd.tok[tid], j = a.topo.nth[tid];
    const RowStat ts = nd.stat[up], ds = nd.stat[n_nodes + 1 + dep];
    uint32_t ctr[4] = {(uint32_t)up + ((uint32_t)j << 16), (uint32_t)b, a.off_lo, a.off_hi};
    philox4x32_10(a.key0, a.key1, ctr);
    const bool in_range = x >= 0 && x < V;
    const double logp = in_range ? ((double)a.target_logits[((size_t)b * (n_nodes + 1) + up) * V + x] - (double)ts.max) * inv_t -
                                       log(ts.sum) : -INFINITY;
    const double logq = in_range ? ((double)a.draft_logits[((size_t)b * a.topo.max_depth + dep) * V + x] - (double)ds.max) * inv_t -
                                       log(ds.sum) : -INFINITY;
    const double diff = logp - logq;
    nd.logp[tid] = logp;
    nd.logq[tid] = logq;
    nd.ratio[tid] = (diff != diff) ? 0.0 : exp(fmin(diff, 0.0));
    nd.r[tid] = (double)(ctr[0] >> 8) * (1.0 / 16777216.0);
  }
  __syncthreads();
  int u = 0, len = 0, any_bad = 0, token = -1, turn = 0;
  // every block takes the same branches below: the values they depend on are identical
  for (;;) {
    const int kid0 = a.topo.child_off[u], n_kids = a.topo.child_off[u + 1] - kid0;
    const float* trow = a.target_logits + ((size_t)b * (n_nodes + 1) + u) * V;
    const int dq = len;   // depth of the children of u
    const float* drow = (!greedy && n_kids > 0) ? a.draft_logits + ((size_t)b * a.topo.max_depth + dq) * V : nullptr;
    RowStat ts, ds;
    ts.max = 0.f; ts.arg = 0; ts.bad = 0; ts.sum = 1.0;
    ds = ts;
    if (greedy || n_kids > 0 || a.leaf_stats) ts = nd.stat[u];
    if (drow) ds = nd.stat[n_nodes + 1 + dq];
    int next = -1;
    if (greedy) {
      for (int j = 0; j < n_kids && next < 0; ++j)
        if (nd.tok[a.topo.child_idx[kid0 + j]] == ts.arg) next = a.topo.child_idx[kid0 + j];
      if (next < 0) token = ts.arg;
    } else if (ts.bad | ds.bad) {
      any_bad = 1;
      token = ts.arg;
    } else {
      float t[kCluV4 * 4], d[kCluV4 * 4];   // the rows' exponentials, once they are needed
      bool loaded = false;
      float tmax = ts.max;
      auto load = [&]() {
        loaded = true;
#pragma unroll
        for (int k = 0; k < kCluV4; ++k) {
          const int v = v0 + 4 * k;   // V % 4 == 0: a vector lies inside the row or outside it
          float4 tv = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), dv = tv;
          if (k < nv4 && v < V) {
            tv = *reinterpret_cast<const float4*>(trow + v);
            if (drow) dv = *reinterpret_cast<const float4*>(drow + v);
          }
          t[4 * k] = tv.x; t[4 * k + 1] = tv.y; t[4 * k + 2] = tv.z; t[4 * k + 3] = tv.w;
          d[4 * k] = dv.x; d[4 * k + 1] = dv.y; d[4 * k + 2] = dv.z; d[4 * k + 3] = dv.w;
        }
      };
      auto exponentials = [&]() {
#pragma unroll
        for (int e = 0; e < kCluV4 * 4; ++e) {
          const bool in = e < C && v0 + e < V;
          t[e] = in ? expf(exp_arg_d<UNIT>(t[e], tmax, inv_t)) : 0.f;
          d[e] = (in && drow) ? expf(exp_arg_d<UNIT>(d[e], ds.max, inv_t)) : 0.f;
        }
      };
      double st = ts.sum;
      bool bad = false;
      if (n_kids == 0 && a.leaf_stats) {
        load();
        exponentials();
      } else if (n_kids == 0) {   // a leaf: its statistics are formed here
        load();
        float tm = -INFINITY;
        int ti = 0x7fffffff, bd = 0;
#pragma unroll
        for (int e = 0; e < kCluV4 * 4; ++e) {
          const int v = v0 + e;
          if (e < C && v < V) {
            float xt = t[e];
            if (xt != xt || xt == INFINITY) bd = 1;
            if (xt != xt) xt = -INFINITY;
            if (xt > tm || (xt == tm && v < ti)) { tm = xt; ti = v; }
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float ov = __shfl_xor_sync(0xffffffffu, tm, o);
          const int oi = __shfl_xor_sync(0xffffffffu, ti, o);
          if (ov > tm || (ov == tm && oi < ti)) { tm = ov; ti = oi; }
          bd |= __shfl_xor_sync(0xffffffffu, bd, o);
        }
        __syncthreads();
        if (lane == 0) { s.f[warp] = tm; s.i[warp] = ti; s.flag[warp] = bd; }
        __syncthreads();
        if (tid == 0) {
          for (int w = 1; w < kCluWarps; ++w) {
            if (s.f[w] > tm || (s.f[w] == tm && s.i[w] < ti)) { tm = s.f[w]; ti = s.i[w]; }
            bd |= s.flag[w];
          }
          part.tmax = tm; part.targ = ti; part.bad = bd;
        }
        cl.sync();
        tm = -INFINITY; ti = 0x7fffffff; bd = 0;
        if (lane < nclu) {
          const CluPart* pr = cl.map_shared_rank(&part, lane);
          tm = pr->tmax; ti = pr->targ; bd = pr->bad;
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
          const float ov = __shfl_xor_sync(0xffffffffu, tm, o);
          const int oi = __shfl_xor_sync(0xffffffffu, ti, o);
          if (ov > tm || (ov == tm && oi < ti)) { tm = ov; ti = oi; }
          bd |= __shfl_xor_sync(0xffffffffu, bd, o);
        }
        tmax = __shfl_sync(0xffffffffu, tm, 0);
        ts.arg = __shfl_sync(0xffffffffu, ti, 0);
        bad = __shfl_sync(0xffffffffu, bd, 0) != 0 || tmax == -INFINITY;
        if (ts.arg == 0x7fffffff) ts.arg = 0;
        cl.sync();   // the partials are free again
        if (!bad) {
          exponentials();
          double mine = 0.0;
#pragma unroll
          for (int e = 0; e < kCluV4 * 4; ++e) mine += (double)t[e];
          st = cluster_sum(cl, part, s, mine, turn, warp, lane);
        }
      }
      if (bad) {
        any_bad = 1;
        token = ts.arg;
      } else {
        const float inv_st = (float)(1.0 / st), inv_sd = (float)(1.0 / ds.sum);
        double c = 0.0, Zc = 1.0;   // the target distribution at u is now (p - c q)+ / Zc
        for (int j = 0; j < n_kids; ++j) {
          const int kid = a.topo.child_idx[kid0 + j];
          double ratio;
          if (c == 0.0) {
            ratio = nd.ratio[kid];
          } else {
            const double px = exp(nd.logp[kid]), qx = exp(nd.logq[kid]);
            const double wx = fmax(px - c * qx, 0.0) / Zc;
            ratio = qx > 0.0 ? fmin(wx / qx, 1.0) : (wx > 0.0 ? 1.0 : 0.0);
          }
          if (nd.r[kid] < ratio) { next = kid; break; }
          // rejected: the target distribution becomes norm((p - (c + Zc) q)+)
          if (!loaded) { load(); exponentials(); }
          const double c_new = c + Zc;
          const float cf = (float)c_new;
          double mine = 0.0;
#pragma unroll
          for (int e = 0; e < kCluV4 * 4; ++e) mine += (double)fmaxf(t[e] * inv_st - cf * (d[e] * inv_sd), 0.f);
          const double Z = cluster_sum(cl, part, s, mine, turn, warp, lane);
          if (Z > 0.0) { c = c_new; Zc = Z; } else { c = 0.0; Zc = 1.0; }   // nothing left: back to p
        }
        if (next < 0) {
          uint32_t ctr[4] = {(uint32_t)u, (uint32_t)b, a.off_lo, a.off_hi};
          philox4x32_10(a.key0, a.key1, ctr);
          const double u2 = (double)(ctr[1] >> 8) * (1.0 / 16777216.0);
          const float cf = (float)c;
          float w[kCluV4 * 4];
#pragma unroll
          for (int e = 0; e < kCluV4 * 4; ++e) w[e] = fmaxf(t[e] * inv_st - cf * (d[e] * inv_sd), 0.f);
          token = cluster_draw(cl, part, s, w, v0, u2, rank, tid, warp, lane);
          if (token < 0 && c != 0.0) {   // the residual vanished in fp32: draw from p
#pragma unroll
            for (int e = 0; e < kCluV4 * 4; ++e) w[e] = t[e] * inv_st;
            token = cluster_draw(cl, part, s, w, v0, u2, rank, tid, warp, lane);
          }
          if (token < 0) token = ts.arg;
        }
      }
    }
    if (next < 0) break;
    if (writer) {
      out[len] = nd.tok[next];
      pth[len] = next;
    }
    ++len;
    u = next + 1;
  }
  if (writer) {
    out[len] = token;
    for (int j = len + 1; j <= a.topo.max_depth; ++j) out[j] = -1;
    for (int j = len; j < a.topo.max_depth; ++j) pth[j] = -1;
    a.accept_len[b] = len;
    a.n_out[b] = len + 1;
    if (any_bad) atomicOr(a.status, kStatNonfinite);
  }
  cl.sync();   // no block leaves while another may still read its shared memory
}

// Token tree from the top-n lists of a draft step (see ps_build_tree): one thread per node.
struct BuildArgs {
  int B, n_nodes, R, top_n;
  unsigned char depth[PS_MAX_TREE_NODES], rank[PS_MAX_TREE_NODES];
  const int* top_ids; const int* sampled; int* tokens;
};
__global__ void k_build_tree(BuildArgs a) {
  const int i = threadIdx.x, b = blockIdx.x;
  if (i >= a.n_nodes) return;
  const int t = a.depth[i], r = a.rank[i];
  const int* top = a.top_ids + ((size_t)b * a.R + t) * a.top_n;
  int tok = top[r];
  if (a.sampled) {
    const int sx = a.sampled[(size_t)b * a.R + t];
    if (r == 0) tok = sx;
    else if (tok == sx) tok = top[0];
  }
  a.tokens[(size_t)b * a.n_nodes + i] = tok;
}

}  // namespace

ps_status launch_build_tree(ps_ctx* c, int B, int n_nodes, const int* parent, const int* rank, const int* top_ids,
                            int top_n, const int* sampled_ids, int* tokens, cudaStream_t st) {
  BuildArgs a;
  a.B = B; a.n_nodes = n_nodes; a.R = c->cfg.k_masks + 1; a.top_n = top_n;
  a.top_ids = top_ids; a.sampled = sampled_ids; a.tokens = tokens;
  for (int i = 0; i < n_nodes; ++i) {
    if (parent[i] >= i || parent[i] < -1) return fail(c, PS_ERR_INVALID_ARG, "parent[i] must be -1 or a node before i");
    const int d = parent[i] < 0 ? 0 : a.depth[parent[i]] + 1;
    if (d >= a.R) return fail(c, PS_ERR_INVALID_ARG, "the tree is deeper than the k+1 rows of a draft step");
    if (rank[i] < 0 || rank[i] >= top_n) return fail(c, PS_ERR_INVALID_ARG, "rank[i] must be in [0, top_n)");
    for (int j = 0; j < i; ++j)
      if (parent[j] == parent[i] && rank[j] == rank[i])
        return fail(c, PS_ERR_INVALID_ARG, "two siblings of the same rank would carry the same token");
    a.depth[i] = (unsigned char)d;
    a.rank[i] = (unsigned char)rank[i];
  }
  k_build_tree<<<B, PS_MAX_TREE_NODES, 0, st>>>(a);
  c->launches++;
  return cuda_check(c, cudaGetLastError(), "k_build_tree");
}

// Launch with a cluster of nclu blocks along x (a launch attribute, not a compile-time one).
template <class... KArgs, class... Args>
cudaError_t launch_cluster(void (*kern)(KArgs...), dim3 grid, int nclu, int threads, size_t smem, cudaStream_t st,
                           bool pdl, const Args&... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nclu; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, a...);
}

ps_status launch_verify(ps_ctx* c, int B, int n_draft, int n_target, const int* draft_tokens,
                        const float* draft_logits, const float* target_logits, float temperature,
                        uint64_t seed, uint64_t offset, int* accept_len, int* out_tokens,
                        int* n_out, cudaStream_t st) {
  VerifyArgs a;
  a.B = B; a.n_draft = n_draft; a.n_target = n_target; a.V = c->cfg.vocab;
  a.draft_tokens = draft_tokens; a.draft_logits = draft_logits; a.target_logits = target_logits;
  a.temperature = temperature;
  a.key0 = (uint32_t)seed; a.key1 = (uint32_t)(seed >> 32);
  a.off_lo = (uint32_t)offset; a.off_hi = (uint32_t)(offset >> 32);
  a.accept_len = accept_len; a.out_tokens = out_tokens; a.n_out = n_out;
  a.rec = c->vrec; a.tickets = c->tickets; a.status = c->dev_status;
  const bool aligned = (((uintptr_t)target_logits | (uintptr_t)draft_logits) & 15u) == 0;
  const int nclu = a.V <= kCluMaxVocab ? kClu : 16, pairs = n_target * B;
  const bool unit = temperature == 1.f || temperature == 0.f;   // (no exponentials at 0)
  // More row pairs than the register-resident clusters can take at once (each of their blocks fills
  // an SM): smaller clusters where those hold a row, then the streaming kernel, with as many blocks per pair as are
  // resident together.  Below that the register-resident ones win: one launch, and no second look at the rows.
  // (Draft + verify of 32000 tokens: 15 pairs in clusters of 8 253 us, streamed 256; 16 and 18 pairs, in two
  // waves, 261 and 270, in clusters of 4 259 and 263; 32 pairs in clusters of 4 272, streamed 274; 36, in two
  // waves, 297, streamed 293.  128256 tokens: 7 pairs in clusters of 16 328, streamed 336; 8, in two waves, 343,
  // streamed 337.  144 pairs of 32000 tokens streamed by clusters of 4, in two waves, 23.3 us, of 2 18.7.)
  // Arg-max alone of many rows beyond 131072 tokens is one pass of k_verify's blocks (64 x 5 rows of 131076:
  // 48 us, streamed 54; 16 x 6 rows: 20, streamed 13).
  const bool greedy_long = temperature == 0.f && a.V > kCluMaxVocab16 && 4 * pairs > 3 * c->n_sm;
  int* const at_once = c->clusters[unit ? 0 : 2];
  auto fits = [&](auto kern, int n) {
    const int k = clusters_at_once(at_once[n], kern, kCluThreads, n);
    return pairs <= (k > 0 ? k : c->n_sm / n);
  };
  int reg = 0;   // blocks per pair of the register-resident kernel, 0: they don't all find room
  if (a.V <= kOneMaxVocab) reg = pairs <= c->n_sm ? 1 : 0;
  else if (a.V > kCluMaxVocab16) reg = pairs * 16 <= c->n_sm ? 16 : 0;   // (k_verify's)
  else if (nclu == 16) reg = fits(unit ? k_verify_cluster16<true> : k_verify_cluster16<false>, 16) ? 16 : 0;
  else if (a.V <= kClu * kCluThreads * 4 * 2 ? fits(unit ? k_verify_cluster_v2<true> : k_verify_cluster_v2<false>, kClu)
                                             : fits(unit ? k_verify_cluster<true> : k_verify_cluster<false>, kClu)) reg = kClu;
  else if (a.V <= kCluSmallMaxVocab && fits(unit ? k_verify_cluster4<true> : k_verify_cluster4<false>, kCluSmall)) reg = kCluSmall;
  if (a.V % 4 == 0 && aligned && !greedy_long && reg == 0) {
    int per = 1;
    while (per < 8) {
      const int k = clusters_at_once(c->stream_clusters[unit ? 0 : 1][2 * per], unit ? k_verify_stream<true> : k_verify_stream<false>,
                                     kStrThreads, 2 * per);
      if (pairs > (k > 0 ? k : kStrPerSm * c->n_sm / (2 * per))) break;
      per *= 2;
    }
    const size_t bytes = (size_t)(((a.V + kDrawClu - 1) / kDrawClu + kSeg - 1) / kSeg) * sizeof(double);
    if (bytes <= 40 * 1024) {
      prof_mark(c, st, "begin");
      cudaError_t e = launch_cluster(unit ? k_verify_stream<true> : k_verify_stream<false>, dim3(n_target * per, B), per,
                                     kStrThreads, 0, st, false, a, c->vrow, c->vdraw);
      c->launches++;
      if (e == cudaSuccess && temperature > 0.f) {
        e = launch_after(unit ? k_verify_draw<true> : k_verify_draw<false>, dim3(kDrawClu, B), dim3(kStrThreads), bytes, st,
                         !c->prof, a, (const VerifyDraw*)c->vdraw);
        c->launches++;
      }
      prof_mark(c, st, "verify");
      return cuda_check(c, e, "k_verify_stream");
    }
  }
  if (a.V % 4 == 0 && a.V <= kCluMaxVocab16 && aligned && (nclu == kClu || clusters_at_once(at_once[16], unit ? k_verify_cluster16<true> : k_verify_cluster16<false>, kCluThreads, 16) > 0)) {
    prof_mark(c, st, "begin");
    cudaError_t e;
    // (The 8-block clusters are plain launches: as dependents they start their loads earlier and run
    // 3 us shorter alone, but a step of one sequence gets 3-5 us longer -- clusters of 8 blocks that
    // each fill an SM are slow to place while the LM head's CTAs drain.  The 4-block ones of a batch
    // gain: four sequences 330 -> 326 us.)
    const bool pdl = !c->prof;
    // One block holds rows of up to 8192 tokens; from 6144 on, clusters that are resident together share a
    // row's exponentials to more gain than their barriers cost (8192 tokens, 5 pairs 11.2 -> 9.9 us, 30 pairs
    // 11.4 -> 10.2; 5000 tokens 9.9 against 10.0), unless an extra row's draw is among many (24: 12.6, 12.9).
    // (Clusters of 8 that need most of the chip's SMs don't all find room at once: 16 pairs 15.1, one block 10.2;
    // nor do more than 33 of 4: 36 pairs of 8000 tokens 18.0, one block 12.5.)
    const bool share = a.V > 6144 && (4 * pairs * kClu <= 3 * c->n_sm ||
                                      (n_target == n_draft && pairs * kClu > c->n_sm &&
                                       fits(unit ? k_verify_cluster4<true> : k_verify_cluster4<false>, kCluSmall)));
    if (a.V <= kOneMaxVocab && !share) {
      // (as few tokens a thread as hold the row: see verify_cluster_body)
      constexpr int kPer = kCluThreads * 4;
      e = launch_after(a.V <= kPer       ? (unit ? k_verify_block<1, true> : k_verify_block<1, false>)
                       : a.V <= 2 * kPer ? (unit ? k_verify_block<2, true> : k_verify_block<2, false>)
                                         : (unit ? k_verify_block<kCluV4, true> : k_verify_block<kCluV4, false>),
                       dim3(n_target, B), dim3(kCluThreads), 0, st, pdl, a);
    } else if (nclu == kClu && a.V <= kCluSmallMaxVocab && (reg == kCluSmall || (reg != kClu && pairs * kClu > c->n_sm))) {   // half the waves
      e = launch_after(unit ? k_verify_cluster4<true> : k_verify_cluster4<false>, dim3(n_target * kCluSmall, B), dim3(kCluThreads), 0, st, pdl, a);
    } else if (nclu == kClu) {
      e = launch_after(a.V <= kClu * kCluThreads * 4 * 2 ? (unit ? k_verify_cluster_v2<true> : k_verify_cluster_v2<false>)
                                                         : (unit ? k_verify_cluster<true> : k_verify_cluster<false>),
                       dim3(n_target * kClu, B), dim3(kCluThreads), 0, st, false, a);
    } else {
      e = launch_cluster(unit ? k_verify_cluster16<true> : k_verify_cluster16<false>, dim3(n_target * 16, B), 16, kCluThreads, 0, st, false, a);
    }
    c->launches++;
    prof_mark(c, st, "verify");
    return cuda_check(c, e, "k_verify_cluster");
  }
  size_t smem = (size_t)((a.V + kSeg - 1) / kSeg) * sizeof(double);
  if (smem > 160 * 1024) return fail(c, PS_ERR_UNSUPPORTED, "vocab too large for ps_verify");
  if (smem > 40 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_verify, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(c, e, "verify smem");
  }
  prof_mark(c, st, "begin");
  k_verify<<<dim3(n_target, B), kThreads, smem, st>>>(a);
  c->launches++;
  prof_mark(c, st, "verify");
  return cuda_check(c, cudaGetLastError(), "k_verify");
}

ps_status launch_verify_tree(ps_ctx* c, int B, int n_nodes, const int* parent, const int* tokens,
                             const float* draft_logits, const float* target_logits, float temperature,
                             uint64_t seed, uint64_t offset, int* accept_len, int* out_tokens, int* n_out,
                             int* path, int* max_depth_out, cudaStream_t st) {
  TreeArgs a;
  a.B = B; a.V = c->cfg.vocab;
  TreeTopo& tp = a.topo;
  tp.n_nodes = n_nodes;
  tp.max_depth = 0;
  for (int i = 0; i < n_nodes; ++i) {
    if (parent[i] >= i || parent[i] < -1) return fail(c, PS_ERR_INVALID_ARG, "parent[i] must be -1 or a node before i");
    tp.depth[i] = (unsigned char)(parent[i] < 0 ? 0 : tp.depth[parent[i]] + 1);
    tp.max_depth = std::max(tp.max_depth, (int)tp.depth[i] + 1);
  }
  // children of decision row u in increasing node id (comparing every node with every row was 1.5 us of a call with 60 nodes)
  unsigned char count[PS_MAX_TREE_NODES + 1] = {};
  for (int i = 0; i < n_nodes; ++i) {
    tp.parent[i] = (signed char)parent[i];
    tp.nth[i] = count[parent[i] + 1]++;
  }
  tp.child_off[0] = 0;
  for (int u = 0; u <= n_nodes; ++u) tp.child_off[u + 1] = (unsigned char)(tp.child_off[u] + count[u]);
  for (int i = 0; i < n_nodes; ++i) tp.child_idx[tp.child_off[parent[i] + 1] + tp.nth[i]] = (unsigned char)i;
  if (max_depth_out) *max_depth_out = tp.max_depth;
  if (temperature != 0.f && !draft_logits) return fail(c, PS_ERR_INVALID_ARG, "draft_logits needed at temperature > 0");
  const bool aligned = (((uintptr_t)target_logits | (uintptr_t)draft_logits) & 15u) == 0;
  if (a.V % 4 || a.V > kCluMaxVocab16 || !aligned)
    return fail(c, PS_ERR_UNSUPPORTED, "ps_verify_tree needs vocab % 4 == 0, vocab <= 131072 and 16-byte aligned logits");
  a.tokens = tokens; a.draft_logits = draft_logits; a.target_logits = target_logits;
  a.temperature = temperature;
  a.key0 = (uint32_t)seed; a.key1 = (uint32_t)(seed >> 32);
  a.off_lo = (uint32_t)offset; a.off_hi = (uint32_t)(offset >> 32);
  a.accept_len = accept_len; a.out_tokens = out_tokens; a.n_out = n_out; a.path = path;
  a.stats = c->tree_stats; a.status = c->dev_status;
  const int least = a.V <= kOneMaxVocab ? 1 : a.V <= 2 * kOneMaxVocab ? 2 : a.V <= kCluSmallMaxVocab ? kCluSmall
                  : a.V <= kCluMaxVocab ? kClu : 16;   // blocks that hold a row
  // One block for short rows (16 trees of 9 nodes, 1000 tokens: 37.7 us with clusters of 8, 17.1 with one block;
  // 8192 tokens, one tree: one block 18.4, four 16.6); no more than hold a row where larger clusters would
  // not find room at once (16 trees of 23 nodes, 32000 tokens: 47.0 with clusters of 8, 34.8 with 4).
  const int want = a.V <= kOneMaxVocab / 2 ? 1 : a.V <= kOneMaxVocab ? kCluSmall : a.V <= kCluMaxVocab ? kClu : 16;
  const int nclu = 4 * B * want > 3 * c->n_sm ? least : want;
  const bool unit = temperature == 1.f || temperature == 0.f;
  auto walk = unit ? k_tree_walk<true> : k_tree_walk<false>;
  if (nclu > 8 && clusters_at_once(c->clusters[unit ? 1 : 3][nclu], walk, kCluThreads, nclu) < 0)
    return fail(c, PS_ERR_UNSUPPORTED, "this device cannot run the 16-block clusters a vocabulary beyond 65536 needs");
  TreeRows list;
  list.n = 0;
  // (the leaves' rows too where all rows' blocks fit the chip twice over)
  a.leaf_stats = temperature != 0.f && 2 * (n_nodes + 1 + tp.max_depth) * B <= kStrPerSm * c->n_sm;
  for (int u = 0; u <= n_nodes; ++u)
    if (temperature == 0.f || a.leaf_stats || tp.child_off[u + 1] > tp.child_off[u]) list.row[list.n++] = (unsigned char)u;
  if (temperature != 0.f)
    for (int t = 0; t < tp.max_depth; ++t) list.row[list.n++] = (unsigned char)(n_nodes + 1 + t);
  int per = 1;   // blocks per row: as many as are resident together, with a vector for each of their threads
  while (per < 8 && 2 * list.n * B * per <= kStrPerSm * c->n_sm && a.V >= 2 * per * 4 * kStrThreads) per *= 2;
  prof_mark(c, st, "begin");
  cudaError_t e = launch_cluster(temperature == 1.f ? k_row_softmax<true> : k_row_softmax<false>, dim3(list.n * per, B), per,
                                 kStrThreads, 0, st, !c->prof, a, list);
  c->launches++;
  if (e == cudaSuccess) {
    e = launch_cluster(walk, dim3(nclu, B), nclu, kCluThreads, 0, st, !c->prof, a);
    c->launches++;
  }
  prof_mark(c, st, "verify_tree");
  return cuda_check(c, e, "k_tree_walk");
}

}  // namespace ps

extern "C" ps_status ps_philox_fill(const uint32_t key[2], const uint32_t* ctr, uint32_t* out, int n,
                                    void* stream) {
  if (!key || !ctr || !out || n < 0) return PS_ERR_INVALID_ARG;
  if (n == 0) return PS_OK;
  ps::k_philox_fill<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(key[0], key[1], ctr, out, n);
  return cudaGetLastError() == cudaSuccess ? PS_OK : PS_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------
// ps_verify_static: the same kernel with its scratch in a fixed device array of this library
// instead of a caller-allocated workspace, for callers that must not allocate.
namespace ps {
namespace {

struct StaticScratch {
  unsigned tickets[PS_STATIC_MAX_BATCH];                       // must be zero when a call starts
  VerifyRec rec[PS_STATIC_MAX_BATCH * (PS_MAX_MASKS + 2)];     // fully rewritten by every call
  int status_sink;                                             // takes the flag when the caller passes none
};

// About 18 KB, held by every GPU that loads the library until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[sizeof(StaticScratch)];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
void* g_static_ptr[kMaxDevices] = {nullptr};

// Device address of the array on the CURRENT device, looked up once per device.  The array's
// name is only a host-side handle here; a kernel must be given the address obtained below.
cudaError_t static_scratch_address(StaticScratch** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return e;
    g_static_ptr[dev] = p;
  }
  *out = (StaticScratch*)g_static_ptr[dev];
  return cudaSuccess;
}

ps_status static_fail(char* err, size_t cap, ps_status s, const char* text) {
  if (err && cap) std::snprintf(err, cap, "%s", text);
  return s;
}

}  // namespace
}  // namespace ps

extern "C" ps_status ps_verify_static(int vocab, int B, int n_draft, int n_target,
                                      const int* draft_tokens, const float* draft_logits,
                                      const float* target_logits, float temperature, uint64_t seed,
                                      uint64_t offset, int* accept_len, int* out_tokens, int* n_out,
                                      int* nonfinite_flag, char* err, size_t err_cap, void* stream) {
  using namespace ps;
  if (err && err_cap) err[0] = 0;
  if (!draft_tokens || !target_logits || !accept_len || !out_tokens || !n_out)
    return static_fail(err, err_cap, PS_ERR_INVALID_ARG, "ps_verify_static: null pointer");
  if (B < 1 || n_draft < 1 || vocab < 1)
    return static_fail(err, err_cap, PS_ERR_INVALID_ARG, "ps_verify_static: sizes must be positive");
  if (B > PS_STATIC_MAX_BATCH)
    return static_fail(err, err_cap, PS_ERR_CAPACITY,
                       "ps_verify_static: B exceeds PS_STATIC_MAX_BATCH (the fixed scratch holds 128 sequences)");
  if (n_draft > PS_MAX_MASKS + 1)
    return static_fail(err, err_cap, PS_ERR_CAPACITY,
                       "ps_verify_static: n_draft exceeds PS_MAX_MASKS+1 (16 positions per sequence)");
  if (vocab > PS_STATIC_MAX_VOCAB)
    return static_fail(err, err_cap, PS_ERR_CAPACITY,
                       "ps_verify_static: vocab exceeds PS_STATIC_MAX_VOCAB (262144)");
  if (n_target != n_draft && n_target != n_draft + 1)
    return static_fail(err, err_cap, PS_ERR_INVALID_ARG,
                       "ps_verify_static: n_target must be n_draft or n_draft+1");
  if (!(temperature >= 0.f))
    return static_fail(err, err_cap, PS_ERR_INVALID_ARG, "ps_verify_static: temperature must be >= 0");
  StaticScratch* sc = nullptr;
  cudaError_t e = static_scratch_address(&sc);
  if (e != cudaSuccess) return static_fail(err, err_cap, PS_ERR_CUDA, cudaGetErrorString(e));
  cudaStream_t st = (cudaStream_t)stream;
  // The arrival counters keep whatever the previous call left; they must start at zero.
  e = cudaMemsetAsync(sc->tickets, 0, sizeof(sc->tickets), st);
  if (e != cudaSuccess) return static_fail(err, err_cap, PS_ERR_CUDA, cudaGetErrorString(e));
  VerifyArgs a;
  a.B = B; a.n_draft = n_draft; a.n_target = n_target; a.V = vocab;
  a.draft_tokens = draft_tokens; a.draft_logits = draft_logits; a.target_logits = target_logits;
  a.temperature = temperature;
  a.key0 = (uint32_t)seed; a.key1 = (uint32_t)(seed >> 32);
  a.off_lo = (uint32_t)offset; a.off_hi = (uint32_t)(offset >> 32);
  a.accept_len = accept_len; a.out_tokens = out_tokens; a.n_out = n_out;
  a.rec = sc->rec; a.tickets = sc->tickets;
  a.status = nonfinite_flag ? nonfinite_flag : &sc->status_sink;
  size_t smem = (size_t)((vocab + kSeg - 1) / kSeg) * sizeof(double);   // <= 16 KB at the vocab limit
  k_verify<<<dim3(n_target, B), kThreads, smem, st>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return static_fail(err, err_cap, PS_ERR_CUDA, cudaGetErrorString(e));
  return PS_OK;
}
