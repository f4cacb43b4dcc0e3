// CUDA-core (SIMT) kernel path: fp32 accumulate everywhere, any supported geometry.  This is the path of the
// fp32 configuration (tensor-core tf32 would not hold a 1e-4 bound) and the cross-check for the tensor-core path.
// Six launches a step (seven with heads wider than 64), chained with programmatic dependent launch:
//   RMSNorm -> Q projection (+ score, stored query, rotary embedding) -> selection -> K/V projection of the refresh set
//   (+ rotary embedding, cache scatter) -> attention -> output projection.
#include "dare_internal.h"
#include "tc_ptx.cuh"

namespace dare {

using namespace ptx;

namespace {

template <typename T>
__device__ __forceinline__ T from_f(float v);
template <>
__device__ __forceinline__ float from_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Four consecutive elements global -> shared as fp32: an asynchronous 16-byte copy, or (bf16) load, widen and store.
// !ok: zeros (the source address is valid all the same).
__device__ __forceinline__ void fetch4(float* dst, const float* src, bool ok) { cp_async_16(smem_u32(dst), src, ok ? 16u : 0u); }
__device__ __forceinline__ void fetch4(float* dst, const __nv_bfloat16* src, bool ok) {
  uint2 raw = make_uint2(0u, 0u);
  if (ok) raw = *reinterpret_cast<const uint2*>(src);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
  *reinterpret_cast<float4*>(dst) = make_float4(a.x, a.y, b.x, b.y);
}

// ------------------------------------------------------------------------------------------------ projections
// C[m, n] = sum_k A[arow(m), k] * W[n, k]  (W stored [out, in]: Alg. 1 line 2).  A tile has 8 * RM rows and 64 columns:
// 32 rotary pairs, columns (j, j + head_dim / 2) of the heads they belong to, so that the rotary embedding (and, with
// heads of at most 64, the drift score) happens on the accumulators.  128 threads own RM x 4 results each; KG such groups
// share the tile, each taking 32 of every 32 * KG k-elements.  Operands lie in shared memory row by row with k innermost
// (pitch = 4 mod 32 words: the rows a quarter-warp reads start on different banks), three stages deep by cp.async; a
// thread reads four k at a time and multiplies two of them per packed instruction (fma.f32x2), even and odd k in
// accumulators of their own.  Bound by the FMA pipe and by shared-memory reads, 12 16-byte reads per 128 FMAs at RM = 8.
enum { SG_Q = 0, SG_KV = 1, SG_OUT = 2 };
struct SgemmParams {
  const void* a;
  const int* idx;        // gathered rows of A (tokens), or nullptr
  const int* count;      // device count of them
  int a_cache_rows;      // A is addressed by cache row
  StepGeom g;
  int rows;              // rows of the launch (capacity of the list if gathered)
  const void* w0;
  const void* w1;        // SG_KV: W_V
  void* out0;
  void* out1;
  const float2* rope;
  float* q_prev;
  float* scores;
  float* q_raw;          // heads wider than 64: un-rotated scoring head of every token, for score_kernel
  int has_prev;
  int* status;
};
constexpr int kStages = 3, kGroup = 128;

template <int RM, int KG>
struct Sg {
  static constexpr int BM = 8 * RM, BN = 64, BK = 32 * KG, PITCH = BK + 4, THREADS = kGroup * KG;
  static constexpr int STAGE = (BN + BM) * PITCH;                     // floats: W rows, then A rows
  static constexpr int CHUNKS = (BN + BM) * (BK / 4) / THREADS, W_CHUNKS = BN * (BK / 4) / THREADS;
  static_assert(W_CHUNKS == 4, "16 rows per chunk index");
  static constexpr int SMEM = kStages * STAGE * 4;
  static_assert((KG - 1) * BM * BN <= kStages * STAGE, "group sums fit the ring");
};

template <typename T, int EPI, int RM, int KG>
__global__ void __launch_bounds__(kGroup* KG) sgemm_kernel(const SgemmParams p) {
  using S = Sg<RM, KG>;
  constexpr int BM = S::BM, PITCH = S::PITCH;
  extern __shared__ __align__(16) float ring[];
  __shared__ int s_tok[BM];                      // token of a row, -1: no such row
  __shared__ float s_part[BM][2][3];             // partial score sums
  const int tid = threadIdx.x, K = p.g.d, half = p.g.head_dim >> 1, lh = 31 - __clz(half);
  const int n_tiles = (K / 2 + 31) / 32;
  const bool second = EPI == SG_KV && (int)blockIdx.x >= n_tiles;
  const int pair0 = ((int)blockIdx.x - (second ? n_tiles : 0)) * 32, n_pairs = K / 2;
  auto column = [&](int pair, int hi) { return (pair >> lh) * (2 * half) + (pair & (half - 1)) + hi * half; };

  // this thread's share of a stage: 16-byte chunks at (row, kc), the same ones in every stage
  const T* src[S::CHUNKS];
  bool ok[S::CHUNKS];
  const int kc = (tid % (S::BK / 4)) * 4, row_of = tid / (S::BK / 4);
  const T* w = reinterpret_cast<const T*>(second ? p.w1 : p.w0);
#pragma unroll
  for (int i = 0; i < S::W_CHUNKS; ++i) {
    const int n = i * 16 + row_of, pair = pair0 + (n & 31);
    ok[i] = pair < n_pairs;
    src[i] = w + (size_t)(ok[i] ? column(pair, n >> 5) : 0) * K + kc;
  }
  const int nk = (K + S::BK - 1) / S::BK;
  auto fetch = [&](int kb, int i0, int i1) {
    float* st = ring + (kb % kStages) * S::STAGE;
#pragma unroll
    for (int i = 0; i < S::CHUNKS; ++i) {
      if (i < i0 || i >= i1) continue;
      const bool in = ok[i] && kb * S::BK + kc < K;
      fetch4(st + (i * 16 + row_of) * PITCH + kc, src[i] + (in ? kb * S::BK : -kc), in);
    }
  };
  // the weights do not depend on the kernel before: their first stages are on their way while it drains
  // (row tiles past the first of a gathered launch are usually empty: they look at the count first)
  const bool likely = p.count == nullptr || blockIdx.y == 0;
  auto fetch_w = [&]() {
#pragma unroll
    for (int kb = 0; kb < kStages - 1; ++kb)
      if (kb < nk) fetch(kb, 0, S::W_CHUNKS);
  };
  if (likely) fetch_w();
  pdl_wait();
  pdl_launch_dependents();
  const int m0 = (int)blockIdx.y * BM;
  const int m_eff = p.count ? checked_count(*p.count, p.rows, p.status) : p.rows;
  if (m0 >= m_eff) {                             // uniform over the CTA
    cp_async_commit();
    cp_async_wait<0>();
    return;
  }
  if (!likely) fetch_w();
  for (int r = tid; r < BM; r += S::THREADS) {
    int t = m0 + r < m_eff ? (p.idx ? p.idx[m0 + r] : m0 + r) : -1;
    if (p.idx && t != -1 && !token_ok(t, p.g.tokens(), p.status)) t = -1;   // read as zeros, not written
    s_tok[r] = t;
  }
  __syncthreads();
#pragma unroll
  for (int i = S::W_CHUNKS; i < S::CHUNKS; ++i) {
    const int t = s_tok[(i - S::W_CHUNKS) * 16 + row_of];
    ok[i] = t >= 0;
    const size_t row = t < 0 ? 0 : (p.a_cache_rows ? (size_t)p.g.cache_row(t) : (size_t)t);
    src[i] = reinterpret_cast<const T*>(p.a) + row * K + kc;
  }
#pragma unroll
  for (int kb = 0; kb < kStages - 1; ++kb) {
    if (kb < nk) fetch(kb, S::W_CHUNKS, S::CHUNKS);
    cp_async_commit();                           // (the first group holds every stage's W chunks as well)
  }

  const int grp = tid / kGroup, wp = (tid >> 5) & 3, lane = tid & 31;
  const int wm = wp >> 1, wn = wp & 1, tx = lane & 7, ty = lane >> 3;
  // rows wm * BM/2 + ty + 4 i; columns 16 wn + tx + {0, 8} and their partners + 32
  float2 acc[RM][4];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int w_at = (16 * wn + tx) * PITCH + grp * 32, a_at = (64 + wm * (BM / 2) + ty) * PITCH + grp * 32;
  for (int kb = 0; kb < nk; ++kb) {
    cp_async_wait<kStages - 2>();
    __syncthreads();
    if (kb + kStages - 1 < nk) fetch(kb + kStages - 1, 0, S::CHUNKS);
    cp_async_commit();
    const float* st = ring + (kb % kStages) * S::STAGE;
#pragma unroll
    for (int k4 = 0; k4 < 8; ++k4) {
      float4 wv[4], av[RM];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        wv[j] = *reinterpret_cast<const float4*>(st + w_at + ((j & 1) * 8 + (j >> 1) * 32) * PITCH + 4 * k4);
#pragma unroll
      for (int i = 0; i < RM; ++i) av[i] = *reinterpret_cast<const float4*>(st + a_at + 4 * i * PITCH + 4 * k4);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = __ffma2_rn(make_float2(av[i].x, av[i].y), make_float2(wv[j].x, wv[j].y), acc[i][j]);
          acc[i][j] = __ffma2_rn(make_float2(av[i].z, av[i].w), make_float2(wv[j].z, wv[j].w), acc[i][j]);
        }
    }
  }
  cp_async_wait<0>();
  float v[RM][4];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = acc[i][j].x + acc[i][j].y;
  if (KG > 1) {
    // the other groups' sums through the ring, which is idle now
    __syncthreads();
    if (grp > 0) {
#pragma unroll
      for (int e = 0; e < RM * 4; ++e) ring[((grp - 1) * RM * 4 + e) * kGroup + (tid & (kGroup - 1))] = v[e >> 2][e & 3];
    }
    __syncthreads();
    if (grp > 0) return;
    for (int gi = 0; gi < KG - 1; ++gi)
#pragma unroll
      for (int e = 0; e < RM * 4; ++e) v[e >> 2][e & 3] += ring[(gi * RM * 4 + e) * kGroup + tid];
  }

  // ---- the projection's own tail
  const int pair = pair0 + 16 * wn + tx;         // and pair + 8
  const bool score_tile = EPI == SG_Q && half <= 32 && ((p.g.score_head * half) >> 5) == pair0 >> 5;
  T* out = reinterpret_cast<T*>(second ? p.out1 : p.out0);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int r = wm * (BM / 2) + ty + 4 * i, t = s_tok[r];
    const bool row_ok = t >= 0;
    const int pos = row_ok ? p.g.position(t) : 0;
    const size_t cr = row_ok ? (size_t)p.g.cache_row(t) : 0;
    float dot = 0.f, n1 = 0.f, n2 = 0.f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int pj = pair + 8 * j;
      if (!row_ok || pj >= n_pairs) continue;
      float a = v[i][j], b = v[i][j + 2];
      const int jj = pj & (half - 1), c = column(pj, 0);
      if (EPI == SG_Q && (pj >> lh) == p.g.score_head) {
        // Sec. 3.1 on the un-rotated query; the current one is kept for the next step (Sec. 3.2)
        if (score_tile) {
          float* qp = p.q_prev + cr * (2 * half) + jj;
          if (p.has_prev) {
            const float pa = qp[0], pb = qp[half];
            dot = fmaf(a, pa, fmaf(b, pb, dot)); n1 = fmaf(a, a, fmaf(b, b, n1)); n2 = fmaf(pa, pa, fmaf(pb, pb, n2));
          }
          qp[0] = a; qp[half] = b;
        } else {
          float* qr = p.q_raw + (size_t)t * (2 * half) + jj;
          qr[0] = a; qr[half] = b;
        }
      }
      if (EPI == SG_Q || (EPI == SG_KV && !second)) {
        const float2 cs = p.rope[(size_t)pos * half + jj];
        const float ra = a * cs.x - b * cs.y, rb = a * cs.y + b * cs.x;
        a = ra; b = rb;
      }
      T* dst = out + (EPI == SG_KV ? cr : (size_t)t) * K + c;
      dst[0] = from_f<T>(a);
      dst[half] = from_f<T>(b);
    }
    if (score_tile) {
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        dot += __shfl_xor_sync(0xffffffffu, dot, o);
        n1 += __shfl_xor_sync(0xffffffffu, n1, o);
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      }
      if (tx == 0) { s_part[r][wn][0] = dot; s_part[r][wn][1] = n1; s_part[r][wn][2] = n2; }
    }
  }
  if (score_tile) {
    asm volatile("bar.sync 1, %0;" ::"n"(kGroup) : "memory");
    for (int r = tid; r < BM; r += kGroup) {
      if (s_tok[r] < 0) continue;
      const float D = s_part[r][0][0] + s_part[r][1][0], A = s_part[r][0][1] + s_part[r][1][1], B = s_part[r][0][2] + s_part[r][1][2];
      const float den = sqrtf(A) * sqrtf(B);
      p.scores[s_tok[r]] = p.has_prev ? 1.f - (den > 0.f ? D / den : 0.f) : __int_as_float(0x7f800000);
    }
  }
}

// Heads wider than 64 span several tiles: the drift score from the stored un-rotated scoring head, a warp per token.
__global__ void __launch_bounds__(256) score_kernel(const float* __restrict__ q_raw, float* __restrict__ q_prev,
                                                    float* __restrict__ scores, int has_prev, StepGeom g) {
  pdl_wait();
  pdl_launch_dependents();
  const int t = (int)blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, hd = g.head_dim;
  if (t >= g.tokens()) return;
  const float4* qn = reinterpret_cast<const float4*>(q_raw + (size_t)t * hd);
  float4* qp = reinterpret_cast<float4*>(q_prev + (size_t)g.cache_row(t) * hd);
  float dot = 0.f, n1 = 0.f, n2 = 0.f;
  for (int v = lane; v < hd / 4; v += 32) {
    const float4 a = qn[v];
    if (has_prev) {
      const float4 b = qp[v];
      dot += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
      n1 += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
      n2 += b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w;
    }
    qp[v] = a;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dot += __shfl_xor_sync(0xffffffffu, dot, o);
    n1 += __shfl_xor_sync(0xffffffffu, n1, o);
    n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  }
  if (lane == 0) {
    const float den = sqrtf(n1) * sqrtf(n2);
    scores[t] = has_prev ? 1.f - (den > 0.f ? dot / den : 0.f) : __int_as_float(0x7f800000);   // +inf: nothing to compare with
  }
}

template <typename T, int EPI, int RM, int KG>
cudaError_t launch_sgemm_as(const SgemmParams& p, int n_tiles, cudaStream_t st) {
  using S = Sg<RM, KG>;
  static std::atomic<unsigned long long> attr_done{0};
  auto kern = sgemm_kernel<T, EPI, RM, KG>;
  if (cudaError_t e = ensure_dyn_smem(kern, S::SMEM, attr_done); e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(n_tiles, (p.rows + S::BM - 1) / S::BM), dim3(S::THREADS), S::SMEM, st, 1, p);
}
// rows_likely: rows that the launch is sized for (a gathered launch's count is known to the device only).
template <typename T, int EPI>
cudaError_t launch_sgemm(const SgemmParams& p, int rows_likely, cudaStream_t st) {
  if (p.rows <= 0) return cudaSuccess;
  const int n_tiles = (p.g.d / 2 + 31) / 32 * (EPI == SG_KV ? 2 : 1);
  auto tiles = [&](int bm) { return n_tiles * ((rows_likely + bm - 1) / bm); };
  // The taller tile reads less shared memory per FMA (measured rate 1 : 1.25 : 1.9), the shorter ones spread few rows over
  // more SMs: whichever leaves the busiest SM the least to do.
  auto cost = [&](int bm, float f) { return (float)((tiles(bm) + 147) / 148 * bm) * f; };
  const float c64 = cost(64, 1.f), c32 = cost(32, 1.25f), c16 = cost(16, 1.9f);
  if (c16 < c32 && c16 < c64) return launch_sgemm_as<T, EPI, 2, 4>(p, n_tiles, st);
  if (c32 < c64) return launch_sgemm_as<T, EPI, 4, 2>(p, n_tiles, st);
  return launch_sgemm_as<T, EPI, 8, 1>(p, n_tiles, st);
}
}  // namespace

// ------------------------------------------------------------------------------------------------ attention
// Eq. 4 / Alg. 2 line 8 (row-sparse) and Alg. 1 line 10 (all rows): bidirectional softmax attention, no mask, fp32.
// One CTA = one head x 32 query rows of one sequence.  Two groups of 128 threads take alternate key blocks, each with
// its own double-buffered K and V tiles (cp.async), running maxima, sums and accumulators, merged at the end.  A thread
// owns 4 rows: scores of BKV / 16 keys each, then HD / 16 output columns each; the 16 lanes of a half-warp share their
// rows, so the softmax is shuffles and the probabilities pass through shared memory within the half-warp only.
// Bound by the FMA pipe and shared-memory reads like the projections (8 16-byte reads per 64 FMAs).  The result row is
// written into the O cache; rows that are not computed keep what they hold (Alg. 2 lines 9-10).
// (One warp per row and head, a key at a time, was bound by the latency of its five-step reduction per key: 2 x 384 rows
// of 16 heads x 64 over 384 keys took about 300 us.)
namespace {
struct SattnParams {
  const void* q;
  const void* kc;
  const void* vc;
  void* oc;
  const int* idx;        // refresh set (row-sparse), or nullptr
  const int* batch_off;  // its slice per sequence
  StepGeom g;
  int* status;
};
template <int HD>
struct Sa {
  static constexpr int BQ = 32, BKV = HD <= 64 ? 64 : (HD == 128 ? 32 : 16), JN = BKV / 16;
  static constexpr int KP = HD + 4, PP = BKV + 4;                       // pitches of K / Q rows and of the probabilities
  static constexpr int VW = HD >= 64 ? 4 : 2, NC = HD / (16 * VW);      // a lane's output columns: NC vectors of VW
  static constexpr int BUF = BKV * KP + BKV * HD;                       // K and V of one block (floats)
  static constexpr int Q_OFF = 0, P_OFF = BQ * KP, KV_OFF = P_OFF + 2 * BQ * PP, FLOATS = KV_OFF + 2 * 2 * BUF;
  static constexpr int SMEM = FLOATS * 4;
  static_assert(SMEM <= 226 * 1024 && BQ * HD + 2 * BQ <= 2 * BUF, "shared memory, merge buffer");
};

template <typename T, int HD>
__global__ void __launch_bounds__(256) sattn_kernel(const SattnParams p) {
  using S = Sa<HD>;
  constexpr int BQ = S::BQ, BKV = S::BKV, JN = S::JN, KP = S::KP, PP = S::PP, VW = S::VW, NC = S::NC;
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_tok[BQ];
  const StepGeom& g = p.g;
  const int tid = threadIdx.x, grp = tid >> 7, gt = tid & 127, tx = gt & 15, ty = gt >> 4;
  const int h = blockIdx.x, b = blockIdx.y, tile = blockIdx.z, d = g.d;
  pdl_wait();
  pdl_launch_dependents();
  int row0, n_rows;
  if (p.idx) {
    const int lo = p.batch_off[b], hi = p.batch_off[b + 1];
    if (!slice_ok(lo, hi, g.tokens(), p.status) || lo + tile * BQ >= hi) return;
    row0 = lo + tile * BQ;
    n_rows = min(BQ, hi - row0);
  } else {
    row0 = b * g.seq_act + tile * BQ;
    n_rows = min(BQ, g.seq_act - tile * BQ);
  }
  const T* kbase = reinterpret_cast<const T*>(p.kc) + (size_t)b * g.max_seq * d + h * HD;
  const T* vbase = reinterpret_cast<const T*>(p.vc) + (size_t)b * g.max_seq * d + h * HD;
  const int n_blocks = (g.kv_len + BKV - 1) / BKV;
  float* kv = sm + S::KV_OFF + grp * 2 * S::BUF;
  auto fetch_block = [&](int blk, int buf) {       // keys past the last: zeros
    float* kd = kv + buf * S::BUF;
    float* vd = kd + BKV * KP;
    for (int c = gt; c < BKV * (HD / 4); c += 128) {
      const int r = c / (HD / 4), e = (c % (HD / 4)) * 4, key = blk * BKV + r;
      const bool ok = key < g.kv_len;
      const size_t off = (size_t)(ok ? key : 0) * d + e;
      fetch4(kd + r * KP + e, kbase + off, ok);
      fetch4(vd + r * HD + e, vbase + off, ok);
    }
  };
  if (grp < n_blocks) fetch_block(grp, 0);
  if (tid < BQ) {
    int t = tid < n_rows ? (p.idx ? p.idx[row0 + tid] : row0 + tid) : -1;
    if (p.idx && t != -1 && !token_ok(t, g.tokens(), p.status)) t = -1;   // neither a query row to read nor a cache row to write
    s_tok[tid] = t;
  }
  __syncthreads();
  for (int c = tid; c < BQ * (HD / 4); c += 256) {
    const int r = c / (HD / 4), e = (c % (HD / 4)) * 4, t = s_tok[r];
    fetch4(sm + S::Q_OFF + r * KP + e, reinterpret_cast<const T*>(p.q) + (size_t)(t < 0 ? 0 : t) * d + h * HD + e, t >= 0);
  }
  cp_async_commit();
  const float c = rsqrtf((float)HD) * 1.4426950408889634f;              // softmax scale folded into the exp2 argument
  float m[4], l[4], acc[4][NC][VW];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
      for (int e = 0; e < VW; ++e) acc[i][n][e] = 0.f;
  }
  const float* qs = sm + S::Q_OFF + ty * KP;                            // rows ty + 8 i
  float* ps = sm + S::P_OFF + grp * BQ * PP + ty * PP;
  cp_async_wait<0>();
  __syncthreads();                                                      // Q is both groups'
  int buf = 0;
  for (int blk = grp; blk < n_blocks; blk += 2, buf ^= 1) {
    if (blk + 2 < n_blocks) fetch_block(blk + 2, buf ^ 1);
    cp_async_commit();
    const float* ks = kv + buf * S::BUF + tx * KP;                      // keys tx + 16 j
    const float* vs = kv + buf * S::BUF + BKV * KP + tx * VW;
    float2 s2[4][JN];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < JN; ++j) s2[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int e = 0; e < HD; e += 4) {
      float4 kf[JN], qf[4];
#pragma unroll
      for (int j = 0; j < JN; ++j) kf[j] = *reinterpret_cast<const float4*>(ks + 16 * j * KP + e);
#pragma unroll
      for (int i = 0; i < 4; ++i) qf[i] = *reinterpret_cast<const float4*>(qs + 8 * i * KP + e);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) {
          s2[i][j] = __ffma2_rn(make_float2(qf[i].x, qf[i].y), make_float2(kf[j].x, kf[j].y), s2[i][j]);
          s2[i][j] = __ffma2_rn(make_float2(qf[i].z, qf[i].w), make_float2(kf[j].z, kf[j].w), s2[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float s[JN], mx = m[i];
#pragma unroll
      for (int j = 0; j < JN; ++j) {
        s[j] = blk * BKV + tx + 16 * j < g.kv_len ? (s2[i][j].x + s2[i][j].y) * c : -INFINITY;
        mx = fmaxf(mx, s[j]);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float corr = exp2f(m[i] - mx);
      m[i] = mx;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < JN; ++j) {
        const float pr = exp2f(s[j] - mx);
        sum += pr;
        ps[8 * i * PP + tx + 16 * j] = pr;
      }
      l[i] = l[i] * corr + sum;                                         // (this lane's share of the row sum)
#pragma unroll
      for (int n = 0; n < NC; ++n)
#pragma unroll
        for (int e = 0; e < VW; ++e) acc[i][n][e] *= corr;
    }
    __syncwarp();
#pragma unroll 2
    for (int k = 0; k < BKV; k += 4) {
      float4 pf[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) pf[i] = *reinterpret_cast<const float4*>(ps + 8 * i * PP + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int n = 0; n < NC; ++n) {
          float vf[VW];
          const float* vp = vs + (k + kk) * HD + n * 16 * VW;
          if constexpr (VW == 4) {
            const float4 t = *reinterpret_cast<const float4*>(vp);
            vf[0] = t.x; vf[1] = t.y; vf[2] = t.z; vf[3] = t.w;
          } else {
            const float2 t = *reinterpret_cast<const float2*>(vp);
            vf[0] = t.x; vf[1] = t.y;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float pr = kk == 0 ? pf[i].x : (kk == 1 ? pf[i].y : (kk == 2 ? pf[i].z : pf[i].w));
#pragma unroll
            for (int e = 0; e < VW; e += 2) {
              const float2 r = __ffma2_rn(make_float2(pr, pr), make_float2(vf[e], vf[e + 1]),
                                          make_float2(acc[i][n][e], acc[i][n][e + 1]));
              acc[i][n][e] = r.x; acc[i][n][e + 1] = r.y;
            }
          }
        }
    }
    cp_async_wait<0>();
    asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");        // the group is done with this buffer; the next has landed
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], o);
  // group 1 hands its part over through its own (idle) K/V buffers
  float* part = sm + S::KV_OFF + 2 * S::BUF;                            // accumulators [BQ][HD], then maxima, then sums
  if (grp == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 8 * i;
#pragma unroll
      for (int n = 0; n < NC; ++n)
#pragma unroll
        for (int e = 0; e < VW; ++e) part[r * HD + n * 16 * VW + tx * VW + e] = acc[i][n][e];
      if (tx == 0) { part[BQ * HD + r] = m[i]; part[BQ * HD + BQ + r] = l[i]; }
    }
  }
  __syncthreads();
  if (grp == 1) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = ty + 8 * i, t = s_tok[r];
    if (t < 0) continue;
    const float mo = part[BQ * HD + r], lo = part[BQ * HD + BQ + r], mx = fmaxf(m[i], mo);
    const float wa = exp2f(m[i] - mx), wb = exp2f(mo - mx), inv = 1.f / (wa * l[i] + wb * lo);
    T* dst = reinterpret_cast<T*>(p.oc) + (size_t)g.cache_row(t) * d + h * HD + tx * VW;
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
      for (int e = 0; e < VW; ++e)
        dst[n * 16 * VW + e] = from_f<T>((wa * acc[i][n][e] + wb * part[r * HD + n * 16 * VW + tx * VW + e]) * inv);
  }
}

template <typename T, int HD>
cudaError_t launch_sattn_hd(const SattnParams& p, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  auto kern = sattn_kernel<T, HD>;
  if (cudaError_t e = ensure_dyn_smem(kern, Sa<HD>::SMEM, attr_done); e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(p.g.n_heads, p.g.batch, (p.g.seq_act + 31) / 32), dim3(256), Sa<HD>::SMEM, st, 1, p);
}
}  // namespace

// ------------------------------------------------------------------------------------------------ launches
template <typename T>
cudaError_t launch_q_simt(const SimtStep& s, const T* xn, const T* w_q, T* q, cudaStream_t st, int* launches) {
  SgemmParams p = {};
  p.a = xn; p.g = s.g; p.rows = s.g.tokens(); p.w0 = w_q; p.out0 = q;
  p.rope = reinterpret_cast<const float2*>(s.rope_cs); p.q_prev = s.q_prev; p.scores = s.scores; p.q_raw = s.tmp;
  p.has_prev = s.has_prev; p.status = s.status;
  ++*launches;
  if (cudaError_t e = launch_sgemm<T, SG_Q>(p, p.rows, st); e != cudaSuccess) return e;
  if (s.g.head_dim <= 64) return cudaSuccess;
  ++*launches;
  return launch_pdl(score_kernel, dim3((p.rows + 7) / 8), dim3(256), 0, st, 1, s.tmp, s.q_prev, s.scores, p.has_prev, s.g);
}
template <typename T>
cudaError_t launch_kv_simt(const SimtStep& s, const T* xn, const int* idx, const int* count, const T* w_k, const T* w_v,
                           T* kc, T* vc, cudaStream_t st) {
  SgemmParams p = {};
  p.a = xn; p.idx = idx; p.count = count; p.g = s.g; p.rows = s.g.tokens(); p.w0 = w_k; p.w1 = w_v; p.out0 = kc; p.out1 = vc;
  p.rope = reinterpret_cast<const float2*>(s.rope_cs); p.status = s.status;
  // (a refresh set is sized for a quarter of the tokens)
  return launch_sgemm<T, SG_KV>(p, idx ? (p.rows + 3) / 4 : p.rows, st);
}
template <typename T>
cudaError_t launch_attention_simt(const SimtStep& s, const T* q, const T* kc, const T* vc, const int* idx,
                                  const int* batch_off, T* oc, cudaStream_t st) {
  SattnParams p = {q, kc, vc, oc, idx, batch_off, s.g, s.status};
  switch (s.g.head_dim) {
    case 32: return launch_sattn_hd<T, 32>(p, st);
    case 64: return launch_sattn_hd<T, 64>(p, st);
    case 128: return launch_sattn_hd<T, 128>(p, st);
    case 256: return launch_sattn_hd<T, 256>(p, st);
    default: return cudaErrorInvalidValue;       // rejected at creation
  }
}
template <typename T>
cudaError_t launch_out_simt(const SimtStep& s, const T* oc, const T* w_o, T* y, cudaStream_t st) {
  SgemmParams p = {};
  p.a = oc; p.a_cache_rows = 1; p.g = s.g; p.rows = s.g.tokens(); p.w0 = w_o; p.out0 = y; p.status = s.status;
  return launch_sgemm<T, SG_OUT>(p, p.rows, st);
}
#define SIMT_LAUNCHES(T)                                                                                                   \
  template cudaError_t launch_q_simt<T>(const SimtStep&, const T*, const T*, T*, cudaStream_t, int*);                     \
  template cudaError_t launch_kv_simt<T>(const SimtStep&, const T*, const int*, const int*, const T*, const T*, T*, T*,   \
                                         cudaStream_t);                                                                   \
  template cudaError_t launch_attention_simt<T>(const SimtStep&, const T*, const T*, const T*, const int*, const int*, T*, \
                                                cudaStream_t);                                                            \
  template cudaError_t launch_out_simt<T>(const SimtStep&, const T*, const T*, T*, cudaStream_t);
SIMT_LAUNCHES(float)
SIMT_LAUNCHES(__nv_bfloat16)

}  // namespace dare
