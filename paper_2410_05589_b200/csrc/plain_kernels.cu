// Kernels with fp32 activations.  They cover every dtype and shape the library accepts and are the
// path for fp32 models (and for bf16 ones the tensor-core kernels do not take).  A draft step is seven
// launches, each the dependent of the one before it:
//   fc (rows gathered) -> q|k|v (RMSNorm) -> attention (RoPE) -> o (+ residual)
//   -> silu(gate) * up (RMSNorm) -> down (+ residual) -> LM head (RMSNorm)   [-> row statistics]
// (Sec. 4.1 "Inference", Sec. 4.3, Sec. 5.1 "Models".)
// What bounds them at the sizes fp32 models are used at (a few MB of weights) is launches and the
// latency of a handful of dependent loads: hence the neighbouring element-wise work inside the
// products, the first weights in flight before the wait for the kernel ahead, and no predicates in
// the inner loop.  Measured (hidden 256, 5 rows, 64 cached keys; draft + verify): 18 launches 114 us
// -> 9 launches 49 us -> 39 (attention, verify).
#include <cfloat>

#include "ps_internal.cuh"

namespace ps {
namespace {

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void store_as(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_as(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Source rows of the fc input.  Row j = 0 of a sequence: [embed[token] ; hidden]; rows j >= 1:
// [mask_embed[j-1] ; mask_feat[j-1]].  With all_real every row is a real (token, hidden) pair.
template <typename WT>
struct GatherSrc {
  const WT *embed, *mask_embed, *mask_feat, *hidden;
  const int* tokens;
  int all_real, H, V;
};
template <typename WT>
__device__ __forceinline__ void gather_row(const GatherSrc<WT>& g, const SeqMap& sm, int m, const WT*& e, const WT*& f) {
  int b, j;
  seq_of_row(sm, m, b, j);
  if (g.all_real || j == 0) {
    const int src = g.all_real ? (m + sm.row_base) : b;
    const int tok = min(max(g.tokens[src], 0), g.V - 1);
    e = g.embed + (size_t)tok * g.H;
    f = g.hidden ? g.hidden + (size_t)src * g.H : nullptr;
  } else {
    e = g.mask_embed + (size_t)(j - 1) * g.H;
    f = g.mask_feat ? g.mask_feat + (size_t)(j - 1) * g.H : nullptr;
  }
}
// Embedding-only input (PS_FLAG_NO_FC): x0 is the embedding half.
template <typename WT>
__global__ void __launch_bounds__(256) k_gather_embed(const __grid_constant__ SeqMap sm, GatherSrc<WT> g, float* x0) {
  pdl_wait();   // (first: see k_linear)
  pdl_launch_dependents();
  const WT *e, *f;
  gather_row(g, sm, blockIdx.x, e, f);
  for (int i = threadIdx.x; i < g.H; i += blockDim.x) x0[(size_t)blockIdx.x * g.H + i] = to_f32(e[i]);
}

// Y[m][n] = sum_k x[m][k] W[n][k] over up to three concatenated matrices, one warp per output
// feature, MC rows per block row.  K is a multiple of 8.  A block's warps share the activations: they
// come through shared memory, kKC columns at a time (each warp reading them from L2 for itself was
// bound by that: 64 KB per block and 256 columns), the weights of those columns in flight meanwhile.
//   LIN_GATHER  x: the gathered fc input (K = 2 H); bias
//   LIN_NORM    x = X * rsqrt(mean(X^2) + eps) * gain: the sums of squares are taken on the way into
//               shared memory, the scale is applied to the result
//   LIN_SWIGLU  LIN_NORM, and Y = silu(g) * u for matrices 0 (gate) and 1 (up)
//   LIN_RES     x = X; Y += res
enum { LIN_GATHER = 0, LIN_NORM = 1, LIN_SWIGLU = 2, LIN_RES = 3 };
template <typename WT>
struct LinArgs {
  const float* X; int ldx;
  const WT* W[3]; int n[3]; float* Y[3]; int ldy[3];
  const WT* bias;
  const WT* gain; float eps;
  const float* res; int ldr;
  int M, K, vec;      // vec: embedding, feature and gain rows are 16-byte aligned
};
// What only the gathering kind reads: the other kinds' parameters stay small (a kernel that runs for
// 2 us feels the fetch of 2 KB of them).
template <typename WT>
struct GatherArgs { GatherSrc<WT> g; SeqMap sm; };
struct NoGather {};
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
// 4 consecutive values as floats; p is 8-byte (bf16) / 16-byte (fp32) aligned.
__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 r = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xffff0000u));
}
template <typename WT>
__device__ __forceinline__ float4 load4_any(const WT* p, bool vec) {
  return vec ? load4(p) : make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
}
constexpr int kKC = 512;
template <typename WT, int KIND, int MC, typename GA>
__global__ void __launch_bounds__(256) k_linear(const __grid_constant__ LinArgs<WT> a, const __grid_constant__ GA ga) {
  // The first kernel of a call: whatever the caller enqueued before it, an update of the weights for
  // one, is complete before it reads and before any kernel behind it, which asks for weights
  // ahead of its own wait, can start.
  if (KIND == LIN_GATHER) pdl_wait();
  pdl_launch_dependents();
  constexpr bool kNorm = KIND == LIN_NORM || KIND == LIN_SWIGLU, kTwo = KIND == LIN_SWIGLU;
  constexpr int C = kKC / 128;                    // float4 groups of a warp per chunk
  constexpr int NL = MC * (kKC / 4) / 256;        // vectors a thread brings in per chunk: rows 2 j + (tid >> 7)
  static_assert(MC % 2 == 0 && kKC == 512, "a row of a chunk is half a block's vectors");
  __shared__ __align__(16) float xs[MC][kKC];
  __shared__ float s_sq[8][NL];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int n = blockIdx.x * 8 + warp, mat = 0;
  if (!kTwo) {
    while (mat < 2 && n >= a.n[mat]) { n -= a.n[mat]; ++mat; }
  }
  const bool active = n < a.n[mat];
  const int m0 = blockIdx.y * MC, K = a.K;
  const bool vec = a.vec != 0;
  const WT* w0 = active ? a.W[mat] + (size_t)n * K : a.W[0];   // (a warp without a feature follows feature 0)
  const WT* w1 = kTwo ? (active ? a.W[1] + (size_t)n * K : a.W[1]) : nullptr;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float acc[MC], acc2[kTwo ? MC : 1], sq[NL];
#pragma unroll
  for (int i = 0; i < MC; ++i) {
    acc[i] = 0.f;
    if (kTwo) acc2[i] = 0.f;
  }
#pragma unroll
  for (int j = 0; j < NL; ++j) sq[j] = 0.f;
  // the thread's place in the rows it brings in (rows past the end repeat the last one)
  const int col = (tid & 127) * 4;
  const float* xr[NL];
  const WT *xe[NL], *xf[NL];
  for (int k0 = 0; k0 < K; k0 += kKC) {
    float4 wv[C], uv[kTwo ? C : 1];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int k = k0 + c * 128 + lane * 4;
      wv[c] = k < K ? load4(w0 + k) : zero;
      if (kTwo) uv[c] = k < K ? load4(w1 + k) : zero;
    }
    float4 g = zero;
    if (kNorm && k0 + col < K) g = load4_any(a.gain + k0 + col, vec);
    if (k0 == 0) {
      pdl_wait();
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        const int m = min(m0 + 2 * j + (tid >> 7), a.M - 1);
        if constexpr (KIND == LIN_GATHER) gather_row(ga.g, ga.sm, m, xe[j], xf[j]);
        else xr[j] = a.X + (size_t)m * a.ldx;
      }
    } else {
      __syncthreads();   // the chunk before has been consumed
    }
    float4 x[NL];
    const int k = k0 + col;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      x[j] = zero;
      if (k < K) {
        if constexpr (KIND == LIN_GATHER) x[j] = load4_any(k < ga.g.H ? xe[j] + k : xf[j] + (k - ga.g.H), vec);   // (H is a multiple of 8)
        else x[j] = __ldcg(reinterpret_cast<const float4*>(xr[j] + k));
      }
    }
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      if (kNorm) {
        sq[j] += (x[j].x * x[j].x + x[j].y * x[j].y) + (x[j].z * x[j].z + x[j].w * x[j].w);
        x[j].x *= g.x; x[j].y *= g.y; x[j].z *= g.z; x[j].w *= g.w;
      }
      *reinterpret_cast<float4*>(&xs[2 * j + (tid >> 7)][col]) = x[j];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < C; ++c) {
#pragma unroll
      for (int i = 0; i < MC; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(&xs[i][c * 128 + lane * 4]);
        acc[i] += (wv[c].x * v.x + wv[c].y * v.y) + (wv[c].z * v.z + wv[c].w * v.w);
        if (kTwo) acc2[i] += (uv[c].x * v.x + uv[c].y * v.y) + (uv[c].z * v.z + uv[c].w * v.w);
      }
    }
  }
  if (kNorm) {
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const float t = warp_sum(sq[j]);
      if (lane == 0) s_sq[warp][j] = t;
    }
    __syncthreads();
  }
  const float t = warp_sum_many<MC>(acc, lane);
  float t2 = 0.f;
  if constexpr (kTwo) t2 = warp_sum_many<MC>(acc2, lane);
  const int i = lane / (32 / MC), m = m0 + i;
  if (active && lane % (32 / MC) == 0 && m < a.M) {
    float v = t;
    if (KIND == LIN_GATHER && a.bias) v += to_f32(a.bias[n]);
    if (kNorm) {
      const int w = (i & 1) * 4, j = i >> 1;   // the four warps that brought row i in
      const float sc = rsqrtf(((s_sq[w][j] + s_sq[w + 1][j]) + (s_sq[w + 2][j] + s_sq[w + 3][j])) / (float)K + a.eps);
      v *= sc;
      if (kTwo) v = v / (1.f + __expf(-v)) * (t2 * sc);
    }
    if (KIND == LIN_RES) v += __ldcg(a.res + (size_t)m * a.ldr + n);
    a.Y[mat][(size_t)m * a.ldy[mat] + n] = v;
  }
}

// RoPE on the k half of appended rows and the store of k and v into the cache slab at the row's
// absolute position.  One block per row.  kv row = [k (Hkv) ; v (Hkv)] fp32.  The pair (i, i + d/2)
// of a head is rotated by pos * base^(-2i/d); angles are formed in double.
template <typename WT>
__global__ void __launch_bounds__(128) k_rope_store(const __grid_constant__ SeqMap sm, const float* __restrict__ kv, WT* kcache,
                                                    WT* vcache, int n_kv_heads, int d, int max_ctx,
                                                    const double* __restrict__ inv_freq) {
  __shared__ float cs[64], sn[64];
  const int m = blockIdx.x, half = d >> 1;
  int b, j;
  seq_of_row(sm, m, b, j);
  const int pos = sm.len[b] + j;
  if ((int)threadIdx.x < half) {
    double s, c;
    sincos((double)pos * inv_freq[threadIdx.x], &s, &c);
    cs[threadIdx.x] = (float)c;
    sn[threadIdx.x] = (float)s;
  }
  __syncthreads();
  pdl_wait();   // (and no early launch of dependents: see k_kv_store)
  const int Hkv = n_kv_heads * d;
  const float* kr = kv + (size_t)m * 2 * Hkv;
  const float* vr = kr + Hkv;
  const size_t slab = (size_t)sm.slot[b] * n_kv_heads;
  for (int t = threadIdx.x; t < n_kv_heads * half; t += blockDim.x) {
    const int h = t / half, i = t - h * half;
    const float x = kr[h * d + i], y = kr[h * d + i + half];
    const size_t at = ((slab + h) * max_ctx + pos) * d + i;
    store_as(kcache + at, x * cs[i] - y * sn[i]);
    store_as(kcache + at + half, y * cs[i] + x * sn[i]);
    store_as(vcache + at, vr[h * d + i]);
    store_as(vcache + at + half, vr[h * d + i + half]);
  }
}

// 8 consecutive cached values in shared memory as floats; p is 16-byte aligned.
__device__ __forceinline__ void shared8(const float* p, float (&w)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}
__device__ __forceinline__ void shared8(const __nv_bfloat16* p, float (&w)[8]) {
  const uint4 r = *reinterpret_cast<const uint4*>(p);
  const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    w[2 * i] = __uint_as_float(u[i] << 16);
    w[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Attention under the parallel-draft mask: row j of a sequence sees cache rows [0, len) and the new
// rows 0..j, which come from q / kv before RoPE.  One block per (head, sequence).  A tile of keys at a
// time: one or two threads hold the scores of a key against all rows, then 256 / D groups of threads
// walk the keys, a thread per channel; running maximum and sums between tiles.
// What bounds it at the lengths fp32 models are used at is a chain of latencies, so the first tile's cached rows
// are asked for before the wait for the kernel ahead, all at once, and RC rows (4, 8 or 16) are computed
// without a branch per row, each of which waited for a shared-memory load of its own (5 rows, 64 keys:
// 11.5 -> 6.9 us; draft + verify, 5 rows 47.9 -> 41.8 us; what the rows past R hold is not kept).
// The tiles take the shared memory of an SM: one block each, which pays where there are more blocks than SMs too (draft
// steps of 32 heads, 64 channels, 5 rows against two blocks an SM without the tiles: 8 sequences of 500 keys 284 -> 271
// us, 40 of 500 1259 -> 1195, 16 of 1500 711 -> 634; 9 rows, 16 of 500 861 and 864; 128 channels, 16 of 500 1689 -> 1677).
constexpr int kAttThreads = 256;
template <typename WT, int D>
constexpr int att_pitch() { return D + 16 / (int)sizeof(WT); }
template <int D>
constexpr int att_tile() { return 16384 / D; }
template <typename WT, int D>
constexpr int att_smem() { return 2 * att_tile<D>() * att_pitch<WT, D>() * (int)sizeof(WT); }
template <typename WT, int D, int RC>
__global__ void __launch_bounds__(kAttThreads) k_attention(const __grid_constant__ SeqMap sm, const float* __restrict__ q,
                                                           const float* __restrict__ kv, const WT* __restrict__ kcache,
                                                           const WT* __restrict__ vcache, int n_heads, int n_kv_heads,
                                                           int max_ctx, const double* __restrict__ inv_freq, float* attn) {
  constexpr int HALF = D / 2, GROUPS = kAttThreads / D, WARPS = kAttThreads / 32, TK = att_tile<D>(), P = att_pitch<WT, D>();
  constexpr int PARTS = kAttThreads / TK, VEC = 16 / (int)sizeof(WT), VPR = D / VEC;
  extern __shared__ __align__(16) unsigned char att_smem_raw[];
  WT* const s_kt = reinterpret_cast<WT*>(att_smem_raw);   // [TK][P]
  WT* const s_vt = s_kt + TK * P;
  __shared__ __align__(16) float s_q[RC][D];               // rotated q (scaled)
  __shared__ __align__(16) WT s_kn[RC][D], s_vn[RC][D];    // the new rows, as the cache holds them
  __shared__ float s_p[RC][TK];
  __shared__ float s_cs[RC][HALF], s_sn[RC][HALF];
  __shared__ float s_red[WARPS][RC];
  const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = sm.row_off[b + 1] - sm.row_off[b], L = sm.len[b], m0 = sm.row_off[b] - sm.row_base;
  const int hk = h / (n_heads / n_kv_heads), Hq = n_heads * D, Hkv = n_kv_heads * D, total = L + R;
  const WT* kb = kcache + ((size_t)sm.slot[b] * n_kv_heads + hk) * max_ctx * D;
  const WT* vb = vcache + ((size_t)sm.slot[b] * n_kv_heads + hk) * max_ctx * D;
  pdl_launch_dependents();
  auto stage = [&](int t0) {   // cached rows of the tile, asynchronously
    const int n = min(TK, L - t0);
    for (int i = tid; i < n * VPR; i += kAttThreads) {
      const int r = i / VPR, c = (i % VPR) * VEC;
      cp_async16(s_kt + r * P + c, kb + (size_t)(t0 + r) * D + c);
      cp_async16(s_vt + r * P + c, vb + (size_t)(t0 + r) * D + c);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(0);   // (the cache is older than the launch before)
  for (int i = tid; i < R * HALF; i += kAttThreads) {   // rotations of the new positions
    double s, c;
    sincos((double)(L + i / HALF) * inv_freq[i % HALF], &s, &c);
    s_cs[i / HALF][i % HALF] = (float)c;
    s_sn[i / HALF][i % HALF] = (float)s;
  }
  pdl_wait();
  const float scale = rsqrtf((float)D);
  __syncthreads();
  for (int i = tid; i < R * HALF; i += kAttThreads) {
    const int j = i / HALF, e = i - j * HALF;
    const float* qr = q + (size_t)(m0 + j) * Hq + h * D + e;
    const float* kr = kv + (size_t)(m0 + j) * 2 * Hkv + hk * D + e;
    const float q0 = __ldcg(qr), q1 = __ldcg(qr + HALF), k0 = __ldcg(kr), k1 = __ldcg(kr + HALF), v0 = __ldcg(kr + Hkv),
                v1 = __ldcg(kr + Hkv + HALF), c = s_cs[j][e], s = s_sn[j][e];
    s_q[j][e] = (q0 * c - q1 * s) * scale;
    s_q[j][e + HALF] = (q1 * c + q0 * s) * scale;
    store_as(&s_kn[j][e], k0 * c - k1 * s);
    store_as(&s_kn[j][e + HALF], k1 * c + k0 * s);
    store_as(&s_vn[j][e], v0);
    store_as(&s_vn[j][e + HALF], v1);
  }
  float m[RC], l[RC], o[RC];
#pragma unroll
  for (int j = 0; j < RC; ++j) { m[j] = -FLT_MAX; l[j] = 0.f; o[j] = 0.f; }
  const int d = tid % D, grp = tid / D, key = tid / PARTS, part = tid % PARTS;
  for (int t0 = 0; t0 < total; t0 += TK) {
    const int nk = min(TK, total - t0), r_new = max(0, L - t0);
    if (t0 > 0) stage(t0);
    __syncthreads();   // the new rows are formed
    for (int i = tid; i < (nk - r_new) * D; i += kAttThreads) {   // those of them in the tile
      const int r = r_new + i / D, c = i % D, j = t0 + r - L;
      s_kt[r * P + c] = s_kn[j][c];
      s_vt[r * P + c] = s_vn[j][c];
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float s[RC];
#pragma unroll
    for (int j = 0; j < RC; ++j) s[j] = 0.f;
    if (key < nk) {
#pragma unroll 2
      for (int c0 = 0; c0 < D / PARTS; c0 += 8) {
        const int c = c0 + part * (D / PARTS);
        float k8[8];
        shared8(s_kt + key * P + c, k8);
#pragma unroll
        for (int j = 0; j < RC; ++j) {
          const float4 a = *reinterpret_cast<const float4*>(&s_q[j][c]), a2 = *reinterpret_cast<const float4*>(&s_q[j][c + 4]);
          s[j] += (k8[0] * a.x + k8[1] * a.y + k8[2] * a.z + k8[3] * a.w) + (k8[4] * a2.x + k8[5] * a2.y + k8[6] * a2.z + k8[7] * a2.w);
        }
      }
    }
    __syncwarp();
    float mx[RC];
#pragma unroll
    for (int j = 0; j < RC; ++j) {
#pragma unroll
      for (int x = 1; x < PARTS; x <<= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], x);
      if (key >= nk || t0 + key - L > j || j >= R) s[j] = -FLT_MAX;   // a new key is seen by its own row and the later ones
      mx[j] = s[j];
    }
#pragma unroll
    for (int x = 16; x > 0; x >>= 1)
#pragma unroll
      for (int j = 0; j < RC; ++j) mx[j] = fmaxf(mx[j], __shfl_xor_sync(0xffffffffu, mx[j], x));
    if (lane == 0) {
#pragma unroll
      for (int j = 0; j < RC; ++j) s_red[warp][j] = mx[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RC; ++j) {
      float t = m[j];
#pragma unroll
      for (int w = 0; w < WARPS; ++w) t = fmaxf(t, s_red[w][j]);
      const float f = __expf(m[j] - t), p = s[j] > -FLT_MAX ? __expf(s[j] - t) : 0.f;
      l[j] = l[j] * f + (part == 0 ? p : 0.f);      // (this thread's share of the row's sum)
      o[j] *= f;
      m[j] = t;
      if (part == 0) s_p[j][key] = p;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = grp; kk < nk; kk += GROUPS) {
      const float v = to_f32(s_vt[kk * P + d]);
#pragma unroll
      for (int j = 0; j < RC; ++j) o[j] += s_p[j][kk] * v;
    }
    __syncthreads();
  }
  // the rows' sums over all threads, the groups' partial outputs (in the keys' place)
  float (*const s_o)[kAttThreads] = reinterpret_cast<float (*)[kAttThreads]>(att_smem_raw);
  static_assert(RC * kAttThreads * 4 <= att_smem<WT, D>(), "they fit it");
#pragma unroll
  for (int x = 16; x > 0; x >>= 1)
#pragma unroll
    for (int j = 0; j < RC; ++j) l[j] += __shfl_xor_sync(0xffffffffu, l[j], x);
#pragma unroll
  for (int j = 0; j < RC; ++j) {
    if (lane == 0) s_red[warp][j] = l[j];
    s_o[j][tid] = o[j];
  }
  __syncthreads();
  for (int i = tid; i < R * D; i += kAttThreads) {
    const int j = i / D, e = i - j * D;
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) num += s_o[j][g * D + e];
#pragma unroll
    for (int w = 0; w < WARPS; ++w) den += s_red[w][j];
    attn[(size_t)(m0 + j) * Hq + h * D + e] = num / den;
  }
}

// k and v of appended positions, fp32 rows [k ; v], into the cache: RoPE as in k_rope_store, with the
// frequencies from the context's table.  Block: 16 heads (of 128 channels) of a row per pass; a
// thread moves four channels and their rotation partners with 16-byte loads and 8-byte stores.
// Bound by the read; the row's table (double-precision angles) is formed while the projection
// before it still runs.  2048 rows of the 13B shape: 64 -> 20 us; 9 rows: 17.9 -> 3.7 us.
__global__ void __launch_bounds__(256) k_kv_store(SeqMap sm, const float* __restrict__ kv, __nv_bfloat16* __restrict__ kcache,
                                                  __nv_bfloat16* __restrict__ vcache, int n_kv_heads, int d, int max_ctx,
                                                  const double* __restrict__ inv_freq) {
  __shared__ float cs[64], sn[64];
  const int m = blockIdx.x, half = d >> 1, per = half >> 2;
  int b, j;
  seq_of_row(sm, m, b, j);
  const int pos = sm.len[b] + j;
  if ((int)threadIdx.x < half) {
    double s, c;
    sincos((double)pos * inv_freq[threadIdx.x], &s, &c);
    cs[threadIdx.x] = (float)c;
    sn[threadIdx.x] = (float)s;
  }
  __syncthreads();
  pdl_wait();
  const int Hkv = n_kv_heads * d, n = n_kv_heads * per;
  const float* kr = kv + (size_t)m * 2 * Hkv;
  const size_t slab = (size_t)sm.slot[b] * n_kv_heads;
  struct alignas(8) B4 { __nv_bfloat16 v[4]; };
  for (int t = blockIdx.y * blockDim.x + threadIdx.x; t < n; t += gridDim.y * blockDim.x) {
    const int h = t / per, i = (t - h * per) * 4;
    const float* src = kr + h * d + i;
    const float4 x4 = __ldcg(reinterpret_cast<const float4*>(src)), y4 = __ldcg(reinterpret_cast<const float4*>(src + half));
    const float4 a4 = __ldcg(reinterpret_cast<const float4*>(src + Hkv)), b4 = __ldcg(reinterpret_cast<const float4*>(src + Hkv + half));
    const float x[4] = {x4.x, x4.y, x4.z, x4.w}, y[4] = {y4.x, y4.y, y4.z, y4.w};
    const float va[4] = {a4.x, a4.y, a4.z, a4.w}, vb[4] = {b4.x, b4.y, b4.z, b4.w};
    B4 k0, k1, v0, v1;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float c = cs[i + e], s = sn[i + e];
      k0.v[e] = __float2bfloat16_rn(x[e] * c - y[e] * s);
      k1.v[e] = __float2bfloat16_rn(y[e] * c + x[e] * s);
      v0.v[e] = __float2bfloat16_rn(va[e]);
      v1.v[e] = __float2bfloat16_rn(vb[e]);
    }
    if (sm.fit) fit_row(k0, k1, v0, v1, per);
    const size_t at = ((slab + h) * max_ctx + pos) * d + i;
    *reinterpret_cast<B4*>(kcache + at) = k0;
    *reinterpret_cast<B4*>(kcache + at + half) = k1;
    *reinterpret_cast<B4*>(vcache + at) = v0;
    *reinterpret_cast<B4*>(vcache + at + half) = v1;
  }
  // (no early launch of dependents: an attention kernel asks for cached rows before it waits for the
  // kernel ahead of it, so whatever follows this one must find the rows written)
}

// A slot's rows between the cache and [len][n_kv_heads][d] arrays, in vectors of T (16 bytes, or one
// element where the caller's arrays are not aligned); 1 << lg vectors per head and row.  A block moves
// kCopyRows passes of rows of one head, whose cache rows are contiguous, with all its loads in flight: no
// division per vector.  A dependent launch, so that a chain of small copies does not wait for its launches.
// Bound by HBM on long contexts (1250 rows of the 13B shape, 51 MB of traffic, one of four in a row: 12.7 -> 10.0
// us), by launches on short
// ones (append of 12 rows and export of the four slots: 78.8 -> 73.8 us).
constexpr int kCopyRows = 4;
template <typename T>
__global__ void __launch_bounds__(256) k_kv_copy(T* __restrict__ kcache, T* __restrict__ vcache, T* __restrict__ K,
                                                 T* __restrict__ V, int slot, int len, int n_kv_heads, int lg, int max_ctx,
                                                 int to_cache) {
  pdl_wait();   // (first: what follows a copy asks for cached rows only behind a kernel that waits before it triggers)
  pdl_launch_dependents();
  const int chunk = blockIdx.x / n_kv_heads, h = blockIdx.x - chunk * n_kv_heads;
  const int rp = 256 >> lg, c = threadIdx.x & ((1 << lg) - 1), t0 = chunk * (kCopyRows * rp) + (threadIdx.x >> lg);
  const size_t cache0 = ((((size_t)slot * n_kv_heads + h) * max_ctx) << lg) + c, flat0 = ((size_t)h << lg) + c;
  const size_t row = (size_t)n_kv_heads << lg;
  const T *ks = to_cache ? K + flat0 : kcache + cache0, *vs = to_cache ? V + flat0 : vcache + cache0;
  T *kd = to_cache ? kcache + cache0 : K + flat0, *vd = to_cache ? vcache + cache0 : V + flat0;
  const size_t sstep = to_cache ? row : (size_t)1 << lg, dstep = to_cache ? (size_t)1 << lg : row;
  T kx[kCopyRows], vx[kCopyRows];
#pragma unroll
  for (int u = 0; u < kCopyRows; ++u) {
    const int t = t0 + u * rp;
    if (t < len) { kx[u] = ks[t * sstep]; vx[u] = vs[t * sstep]; }
  }
#pragma unroll
  for (int u = 0; u < kCopyRows; ++u) {
    const int t = t0 + u * rp;
    if (t < len) { kd[t * dstep] = kx[u]; vd[t * dstep] = vx[u]; }
  }
}

// One product: rows [0, a.M) of the stage's kind.
template <typename WT, int KIND, typename GA = NoGather>
ps_status linear(ps_ctx* c, const LinArgs<WT>& a, cudaStream_t st, const GA& ga = GA()) {
  const int N = KIND == LIN_SWIGLU ? a.n[0] : a.n[0] + a.n[1] + a.n[2];
  cudaError_t e;
  if (a.M <= 4)
    e = launch_after(k_linear<WT, KIND, 4, GA>, dim3((N + 7) / 8, 1), dim3(256), 0, st, !c->prof, a, ga);
  else
    e = launch_after(k_linear<WT, KIND, 8, GA>, dim3((N + 7) / 8, (a.M + 7) / 8), dim3(256), 0, st, !c->prof, a, ga);
  c->launches++;
  return cuda_check(c, e, "k_linear");
}

template <typename WT>
bool rows_aligned(const ps_ctx* c, const void* hidden) {
  const ps_weights& w = c->w;
  return (((uintptr_t)w.embed | (uintptr_t)w.mask_embed | (uintptr_t)w.mask_feat | (uintptr_t)hidden | (uintptr_t)w.g_in |
           (uintptr_t)w.g_post | (uintptr_t)w.g_final) & 15) == 0;
}

// x0 of `rows` rows, then their k | v (and q) projections of the normalised rows.
template <typename WT>
ps_status fc_qkv(ps_ctx* c, const SeqMap& sm, int rows, int all_real, const void* hidden, const int* tokens, bool with_q,
                 cudaStream_t st) {
  const ps_config& g = c->cfg;
  const ps_weights& w = c->w;
  const int H = g.hidden, Hq = g.n_heads * g.head_dim, Hkv = g.n_kv_heads * g.head_dim;
  const bool no_fc = (g.flags & PS_FLAG_NO_FC) != 0;
  typedef const WT* P;
  ps_status s;
  prof_mark(c, st, "begin");
  LinArgs<WT> a{};
  a.M = rows; a.vec = rows_aligned<WT>(c, hidden); a.eps = g.rms_eps;
  const GatherSrc<WT> src{(P)w.embed, (P)w.mask_embed, (P)w.mask_feat, no_fc ? nullptr : (P)hidden, tokens, all_real, H, g.vocab};
  if (no_fc) {
    const cudaError_t e = launch_after(k_gather_embed<WT>, dim3(rows), dim3(256), 0, st, !c->prof, sm, src, c->x0);
    c->launches++;
    if (e != cudaSuccess) return cuda_check(c, e, "k_gather_embed");
  } else {
    LinArgs<WT> f = a;
    f.W[0] = (P)w.w_fc; f.n[0] = H; f.Y[0] = c->x0; f.ldy[0] = H; f.K = 2 * H;
    f.bias = (g.flags & PS_FLAG_FC_BIAS) ? (P)w.b_fc : nullptr;
    if ((s = linear<WT, LIN_GATHER>(c, f, st, GatherArgs<WT>{src, sm}))) return s;
  }
  prof_mark(c, st, "fc_norm");
  a.X = c->x0; a.ldx = H; a.K = H; a.gain = (P)w.g_in;
  int i = 0;
  if (with_q) { a.W[i] = (P)w.w_q; a.n[i] = Hq; a.Y[i] = c->q; a.ldy[i++] = Hq; }
  a.W[i] = (P)w.w_k; a.n[i] = Hkv; a.Y[i] = c->kv_tmp; a.ldy[i++] = 2 * Hkv;
  a.W[i] = (P)w.w_v; a.n[i] = Hkv; a.Y[i] = c->kv_tmp + Hkv; a.ldy[i++] = 2 * Hkv;
  if ((s = linear<WT, LIN_NORM>(c, a, st))) return s;
  prof_mark(c, st, "qkv_rope");
  return PS_OK;
}

template <typename WT>
ps_status kv_append_impl(ps_ctx* c, const SeqMap& sm, int rows, const void* hidden, const int* tokens, cudaStream_t st) {
  const ps_config& g = c->cfg;
  const ps_status s = fc_qkv<WT>(c, sm, rows, 1, hidden, tokens, false, st);
  if (s) return s;
  const cudaError_t e = launch_after(k_rope_store<WT>, dim3(rows), dim3(128), 0, st, !c->prof, sm, c->kv_tmp, (WT*)c->kcache,
                                     (WT*)c->vcache, g.n_kv_heads, g.head_dim, g.max_ctx, (const double*)c->rope_inv_freq);
  c->launches++;
  prof_mark(c, st, "qkv_rope");
  return cuda_check(c, e, "k_rope_store");
}

template <typename WT, int D>
cudaError_t attention(ps_ctx* c, const SeqMap& sm, int B, cudaStream_t st) {
  const ps_config& g = c->cfg;
  const int R = g.k_masks + 1;
  auto kern = R <= 4 ? k_attention<WT, D, 4> : R <= 8 ? k_attention<WT, D, 8> : k_attention<WT, D, 16>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, att_smem<WT, D>());
  if (e != cudaSuccess) return e;
  return launch_after(kern, dim3(g.n_heads, B), dim3(kAttThreads), att_smem<WT, D>(), st, !c->prof, sm, c->q, c->kv_tmp,
                      (const WT*)c->kcache, (const WT*)c->vcache, g.n_heads, g.n_kv_heads, g.max_ctx,
                      (const double*)c->rope_inv_freq, c->attn);
}

template <typename WT>
ps_status draft_impl(ps_ctx* c, const SeqMap& sm, int B, const void* hidden_last,
                     const int* token_last, int top_n, int* top_ids, float* top_logit,
                     float* row_max, float* row_lse, float* logits_out, float* feat_out,
                     const SampleArgs* sa, cudaStream_t st) {
  const ps_config& g = c->cfg;
  const ps_weights& w = c->w;
  const int H = g.hidden, Hq = g.n_heads * g.head_dim, F = g.ffn, V = g.vocab, M = B * (g.k_masks + 1);
  typedef const WT* P;
  ps_status s;
  if ((s = fc_qkv<WT>(c, sm, M, 0, hidden_last, token_last, true, st))) return s;
  cudaError_t e;
  if (g.head_dim == 64) e = attention<WT, 64>(c, sm, B, st);
  else e = attention<WT, 128>(c, sm, B, st);
  c->launches++;
  if (e != cudaSuccess) return cuda_check(c, e, "k_attention");
  prof_mark(c, st, "attention");
  LinArgs<WT> a{};
  a.M = M; a.vec = rows_aligned<WT>(c, hidden_last); a.eps = g.rms_eps;
  {
    LinArgs<WT> x = a;
    x.X = c->attn; x.ldx = Hq; x.K = Hq; x.W[0] = (P)w.w_o; x.n[0] = H; x.Y[0] = c->a; x.ldy[0] = H; x.res = c->x0; x.ldr = H;
    if ((s = linear<WT, LIN_RES>(c, x, st))) return s;
  }
  prof_mark(c, st, "o_proj");
  // (the LM head reads these rows in 16-byte vectors; the caller's feature rows may sit anywhere)
  const bool in_place = feat_out && ((uintptr_t)feat_out & 15) == 0;
  float* hdn = in_place ? feat_out : c->hdn;
  {
    LinArgs<WT> x = a;
    x.X = c->a; x.ldx = H; x.K = H; x.gain = (P)w.g_post;
    x.W[0] = (P)w.w_gate; x.W[1] = (P)w.w_up; x.n[0] = F; x.Y[0] = c->gate; x.ldy[0] = F;
    if ((s = linear<WT, LIN_SWIGLU>(c, x, st))) return s;
    x = a;
    x.X = c->gate; x.ldx = F; x.K = F; x.W[0] = (P)w.w_down; x.n[0] = H; x.Y[0] = hdn; x.ldy[0] = H; x.res = c->a; x.ldr = H;
    if ((s = linear<WT, LIN_RES>(c, x, st))) return s;
  }
  prof_mark(c, st, "ffn");
  float* logits = logits_out ? logits_out : c->logits;
  {
    LinArgs<WT> x = a;
    x.X = hdn; x.ldx = H; x.K = H; x.gain = (P)w.g_final; x.W[0] = (P)w.w_lm; x.n[0] = V; x.Y[0] = logits; x.ldy[0] = V;
    if ((s = linear<WT, LIN_NORM>(c, x, st))) return s;
  }
  if (feat_out && !in_place) {
    const cudaError_t ce = cudaMemcpyAsync(feat_out, hdn, (size_t)M * H * 4, cudaMemcpyDeviceToDevice, st);
    if (ce != cudaSuccess) return cuda_check(c, ce, "feature rows");
  }
  if ((s = launch_logit_stats(c, logits, M, V, g.k_masks + 1, top_n, top_ids, top_logit, row_max, row_lse, sa, st)))
    return s;
  prof_mark(c, st, "lm_head");
  return PS_OK;
}

}  // namespace

ps_status plain_kv_append(ps_ctx* c, const SeqMap& sm, int rows, const void* hidden,
                          const int* tokens, cudaStream_t st) {
  return c->cfg.dtype == PS_DTYPE_F32 ? kv_append_impl<float>(c, sm, rows, hidden, tokens, st)
                                      : kv_append_impl<__nv_bfloat16>(c, sm, rows, hidden, tokens, st);
}

ps_status plain_draft_step(ps_ctx* c, const SeqMap& sm, int B, const void* hidden_last,
                           const int* token_last, int top_n, int* top_ids, float* top_logit,
                           float* row_max, float* row_lse, float* logits_out, float* feat_out,
                           const SampleArgs* sa, cudaStream_t st) {
  return c->cfg.dtype == PS_DTYPE_F32
             ? draft_impl<float>(c, sm, B, hidden_last, token_last, top_n, top_ids, top_logit,
                                 row_max, row_lse, logits_out, feat_out, sa, st)
             : draft_impl<__nv_bfloat16>(c, sm, B, hidden_last, token_last, top_n, top_ids,
                                         top_logit, row_max, row_lse, logits_out, feat_out, sa, st);
}

ps_status launch_rope_store_kv(ps_ctx* c, const SeqMap& sm, int rows, const float* kv, cudaStream_t st) {
  const ps_config& g = c->cfg;
  // few rows: a block per 256 work items, so that a row's heads are in flight together; many: one
  // block per row, which forms the row's table once
  const int items = g.n_kv_heads * g.head_dim / 8;
  const int by = rows < 2 * c->n_sm ? (items + 255) / 256 : 1;
  const cudaError_t e = launch_after(k_kv_store, dim3(rows, by), dim3(256), 0, st, !c->prof, sm, kv, (__nv_bfloat16*)c->kcache,
                                     (__nv_bfloat16*)c->vcache, g.n_kv_heads, g.head_dim, g.max_ctx,
                                     (const double*)c->rope_inv_freq);
  c->launches++;
  return cuda_check(c, e, "k_kv_store");
}

ps_status launch_kv_copy(ps_ctx* c, int slot, int len, void* K, void* V, bool to_cache, cudaStream_t st) {
  const ps_config& g = c->cfg;
  if (len <= 0) return PS_OK;
  const size_t eb = g.dtype == PS_DTYPE_F32 ? 4 : 2;
  const bool vec = (((uintptr_t)K | (uintptr_t)V) & 15) == 0;
  const size_t tb = vec ? 16 : eb;
  int lg = 0;
  while (((size_t)tb << lg) < g.head_dim * eb) ++lg;   // (64 or 128 channels: a power of two of at most 128 vectors)
  const size_t blocks = (size_t)g.n_kv_heads * (((size_t)len + kCopyRows * (256 >> lg) - 1) / (kCopyRows * (256 >> lg)));
  if (blocks > 0x7fffffffu) return fail(c, PS_ERR_UNSUPPORTED, "cache row too long");
  cudaError_t e;
  auto run = [&](auto kern, auto* one) {
    typedef decltype(one) P;
    e = launch_after(kern, dim3((unsigned)blocks), dim3(256), 0, st, !c->prof, (P)c->kcache, (P)c->vcache, (P)K, (P)V, slot, len,
                     g.n_kv_heads, lg, g.max_ctx, to_cache ? 1 : 0);
  };
  if (vec) run(k_kv_copy<uint4>, (uint4*)nullptr);
  else if (eb == 4) run(k_kv_copy<float>, (float*)nullptr);
  else run(k_kv_copy<uint16_t>, (uint16_t*)nullptr);
  c->launches++;
  return cuda_check(c, e, "k_kv_copy");
}

}  // namespace ps
