// CUDA-core (SIMT) kernel path: fp32 accumulate everywhere, any supported geometry.  This is the path of the
// fp32 configuration (whose larger projections go to the tensor cores in split operands, gemm_f32.cu) and the cross-check for
// the tensor-core path.
// Six launches a step (seven with heads wider than 64), chained with programmatic dependent launch:
//   RMSNorm -> Q projection (+ score, stored query, rotary embedding) -> selection -> K/V projection of the refresh set
//   (+ rotary embedding, cache scatter) -> attention -> output projection.
#include <type_traits>
#include "sgemm.h"
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
  if (ok) raw = __ldcg(reinterpret_cast<const uint2*>(src));
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
  *reinterpret_cast<float4*>(dst) = make_float4(a.x, a.y, b.x, b.y);
}

// ------------------------------------------------------------------------------------------------ projections
// C[m, n] = sum_k A[arow(m), k] * W[n, k]  (W stored [out, in]: Alg. 1 line 2).  A tile has BM rows and 64 columns: 32
// rotary pairs, columns (j, j + head_dim / 2) of the heads they belong to, so that the rotary embedding (and, with heads
// of at most 64, the drift score) happens on the accumulators.  A CTA has 512 threads, 16 warps, and an SM to itself:
// KG groups of 2 x WM warps share the tile, each taking 32 of every 32 * KG k-elements, and a thread owns RM x 4 results
// (BM = 4 * RM * WM).  Operands lie in shared memory row by row with k innermost (pitch = 4 mod 32 words: the rows a
// quarter-warp reads start on different banks), three stages deep by cp.async; a thread reads four k at a time and
// multiplies two of them per packed instruction (fma.f32x2), even and odd k in accumulators of their own.
// Bound by the FMA pipe and the registers that feed it: the inner loop alone reaches 53 TFLOP/s at RM = 6, 48 at RM = 4,
// 30 at RM = 2.  (Two CTAs of 256 threads an SM were slower: a launch of one wave filled SMs two by two and left the
// others idle.)
constexpr int kStages = 3, kSgThreads = 512;

template <int RM, int WM, int KG>
struct Sg {
  static constexpr int GROUP = 64 * WM;                               // threads of a k-group
  static_assert(GROUP * KG == kSgThreads, "16 warps");
  static constexpr int BM = 4 * RM * WM, BN = 64, BK = 32 * KG, PITCH = BK + 4, THREADS = kSgThreads;
  static constexpr int STAGE = (BN + BM) * PITCH;                     // floats: W rows, then A rows
  static constexpr int CHUNKS = (BN + BM) * (BK / 4) / THREADS, W_CHUNKS = BN * (BK / 4) / THREADS;
  static constexpr int ROWS = THREADS / (BK / 4);                     // rows per chunk index
  static_assert(W_CHUNKS * ROWS == BN && CHUNKS * ROWS == BN + BM, "whole rows per chunk index");
  static constexpr int SMEM = kStages * STAGE * 4 > 116 * 1024 ? kStages * STAGE * 4 : 116 * 1024;   // one CTA an SM
  static_assert((KG - 1) * BM * BN <= kStages * STAGE, "group sums fit the ring");
};

template <typename T, int EPI, int RM, int WM, int KG>
__global__ void __launch_bounds__(kSgThreads, 1) sgemm_kernel(const SgemmParams p) {
  using S = Sg<RM, WM, KG>;
  constexpr int kGroup = S::GROUP;
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
    const int n = i * S::ROWS + row_of, pair = pair0 + (n & 31);
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
      fetch4(st + (i * S::ROWS + row_of) * PITCH + kc, src[i] + (in ? kb * S::BK : -kc), in);
    }
  };
  // the weights do not depend on the kernel before: their first stages are on their way while it drains
  // (row tiles past the first of a gathered launch are usually empty: they look at the count first)
  const int m0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * BM;
  const bool likely = p.count == nullptr || m0 == 0;
  auto fetch_w = [&]() {
#pragma unroll
    for (int kb = 0; kb < kStages - 1; ++kb)
      if (kb < nk) fetch(kb, 0, S::W_CHUNKS);
  };
  if (likely) fetch_w();
  pdl_wait();
  pdl_launch_dependents();
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
    const int t = s_tok[(i - S::W_CHUNKS) * S::ROWS + row_of];
    ok[i] = t >= 0;
    const size_t row = t < 0 ? 0 : (p.a_cache_rows ? (size_t)p.g.cache_row(t) : (size_t)t);
    src[i] = reinterpret_cast<const T*>(p.a) + row * K + kc;
  }
#pragma unroll
  for (int kb = 0; kb < kStages - 1; ++kb) {
    if (kb < nk) fetch(kb, S::W_CHUNKS, S::CHUNKS);
    cp_async_commit();                           // (the first group holds every stage's W chunks as well)
  }

  const int grp = tid / kGroup, wp = (tid % kGroup) >> 5, lane = tid & 31;
  const int wm = wp >> 1, wn = wp & 1, tx = lane & 7, ty = lane >> 3;
  // All table reads of the tail together, one memory round trip for the rows of this thread; the shortest tiles, whose launches
  // are short chains of round trips, have the registers to start them ahead of the main loop.  (The stored query is this
  // layer's previous step's, the tables are constant.)
  constexpr bool kEarlyTables = RM == 2;
  const int pair = pair0 + 16 * wn + tx;         // and pair + 8
  const bool score_tile = EPI == SG_Q && half <= 32 && ((p.g.score_head * half) >> 5) == pair0 >> 5;
  const bool rotate = EPI == SG_Q || (EPI == SG_KV && !second);
  T* out = reinterpret_cast<T*>(second ? p.out1 : p.out0);
  float2 cs[RM][2], old[RM][2];
  auto read_tables = [&]() {
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      const int t = s_tok[wm * (4 * RM) + ty + 4 * i];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int pj = pair + 8 * j, jj = pj & (half - 1);
        cs[i][j] = old[i][j] = make_float2(0.f, 0.f);
        if (t < 0 || pj >= n_pairs) continue;
        if (rotate) cs[i][j] = p.rope[(size_t)p.g.position(t) * half + jj];
        if (score_tile && p.has_prev && (pj >> lh) == p.g.score_head) {
          const float* qp = p.q_prev + (size_t)p.g.cache_row(t) * (2 * half) + jj;
          old[i][j] = make_float2(qp[0], qp[half]);
        }
      }
    }
  };
  if (kEarlyTables && grp == 0) read_tables();
  // rows wm * 4 RM + ty + 4 i; columns 16 wn + tx + {0, 8} and their partners + 32
  float2 acc[RM][4];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int w_at = (16 * wn + tx) * PITCH + grp * 32, a_at = (64 + wm * (4 * RM) + ty) * PITCH + grp * 32;
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
  if (!kEarlyTables) read_tables();
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int r = wm * (4 * RM) + ty + 4 * i, t = s_tok[r];
    const bool row_ok = t >= 0;
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
          const float2 o = old[i][j];
          dot = fmaf(a, o.x, fmaf(b, o.y, dot)); n1 = fmaf(a, a, fmaf(b, b, n1)); n2 = fmaf(o.x, o.x, fmaf(o.y, o.y, n2));
          float* qp = p.q_prev + cr * (2 * half) + jj;
          qp[0] = a; qp[half] = b;
        } else {
          float* qr = p.q_raw + (size_t)t * (2 * half) + jj;
          qr[0] = a; qr[half] = b;
        }
      }
      if (rotate) {
        const float ra = a * cs[i][j].x - b * cs[i][j].y, rb = a * cs[i][j].y + b * cs[i][j].x;
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

template <typename T, int EPI, int RM, int WM, int KG>
cudaError_t launch_sgemm_as(const SgemmParams& p, int n_tiles, cudaStream_t st) {
  using S = Sg<RM, WM, KG>;
  static std::atomic<unsigned long long> attr_done{0};
  auto kern = sgemm_kernel<T, EPI, RM, WM, KG>;
  if (cudaError_t e = ensure_dyn_smem(kern, S::SMEM, attr_done); e != cudaSuccess) return e;
  // row tiles over y and z: one dimension of a grid stops at 65535 (a CTA past the last tile leaves)
  const int row_tiles = (p.rows + S::BM - 1) / S::BM, nz = (row_tiles + 65534) / 65535;
  return launch_pdl(kern, dim3(n_tiles, (row_tiles + nz - 1) / nz, nz), dim3(S::THREADS), S::SMEM, st, 1, p);
}
// rows_likely: rows that the launch is sized for (a gathered launch's count is known to the device only).
template <typename T, int EPI>
cudaError_t launch_sgemm(const SgemmParams& p, int rows_likely, int* forms, cudaStream_t st) {
  if (p.rows <= 0) return cudaSuccess;
  const int n_tiles = (p.g.d / 2 + 31) / 32 * (EPI == SG_KV ? 2 : 1);
  // What a launch takes is its waves of one tile an SM times the tile height over the rate of its inner loop (above), plus
  // what a tile costs whatever its height (first operands, finishing), about 12 rows: one wave of width 1024 takes 56.0 /
  // 41.8 / 35.9 / 27.7 / 23.4 us at 96 / 64 / 48 / 32 / 16 rows, 0.51-0.60 us a unit of this cost at every height.
  // Q projection in us by tile height 96 / 64 / 48 / 32 / 16, fp32, the pick in brackets: width 256, 128 rows 22.8 / 18.4 /
  // 18.4 / 14.3 / [11.4]; 768, 384 rows 45.9 / 33.9 / 30.6 / [23.6] / 31.9; 512, 768 rows 34.0 / 25.7 / [24.1] / 31.7 / 33.9;
  // 768, 768 rows 45.9 / [34.8] / 54.0 / 40.4 / 58.9; 1024, 1600 rows [107] / 114 / 125 / 133 / 189.  At all twelve sizes
  // timed (64 to 1600 rows) the pick was the fastest, for Q and for K/V.
  auto cost = [&](int bm, float f) {
    return (float)((n_tiles * ((rows_likely + bm - 1) / bm) + kSms - 1) / kSms) * (12.f + (float)bm * f);
  };
  const float c[5] = {cost(96, 1.f), cost(64, 1.1f), cost(48, 1.f), cost(32, 1.1f), cost(16, 1.8f)};
  int best = 0;
  for (int i = 1; i < 5; ++i)
    if (c[i] < c[best]) best = i;
  // fp32 on the tensor cores (gemm_f32.cu) instead?  A unit of the cost above is 0.42 us at width 1024; a tile of 128 rows takes
  // 4.5 us and 1 us a block of 64 k-elements there, 1.2 beyond width 1024, where most of the step's weights come from the HBM.
  // Dense steps in us, here / there with every projection / as the rule below picks for each:
  //   64 rows of width 384 30.4 / 41.7 / 30.4    2 x 200 of 256 33.9 / 45.5 / 33.9      4 x 1000 of 128 106 / 101 / 106
  //   2 x 384 of 384 58.1 / 59.1 / 53.8          4 x 400 of 256 73.8 / 68.1 / 68.0      4 x 2200 of 128 360 / 327 / 360
  //   4 x 400 of 384 131 / 98.7 / 98.8           2 x 128 of 512 42.8 / 53.5 / 42.8      4 x 1000 of 192 162 / 148 / 162
  //   2 x 384 of 512 89.6 / 73.7 / 73.7          300 of 640 67.4 / 68.4 / 64.0          300 of 768 81.9 / 76.4 / 73.5
  //   128 of 1024 66.6 / 77.8 / 66.6             256 of 1024 96.5 / 85.3 / 82.7         4 x 400 of 1024 498 / 275 / 275
  //   64 of 1536 95.5 / 116 / 95.6               100 of 1536 117 / 114 / 109            200 of 1536 174 / 125 / 125
  //   64 of 2048 119 / 147 / 119                 100 of 2048 165 / 140 / 136            200 of 2048 299 / 156 / 156
  //   32 of 4096 211 / 304 / 211                 64 of 4096 305 / 282 / 266             200 of 4096 1052 / 381 / 379
  // Widths below 256 stay here: little to gain, and short sums are the ones that this kernel rounds least (gemm_f32.cu).
  if constexpr (std::is_same<T, float>::value) {
    const int tiles = p.g.d / 64 * (EPI == SG_KV ? 2 : 1) * ((rows_likely + 127) / 128);
    const float there = (float)((tiles + kSms - 1) / kSms) * (4.5f + (p.g.d <= 1024 ? 1.f : 1.2f) * (float)(p.g.d / 64));
    if (p.g.d % 64 == 0 && p.g.d >= 256 && there < 0.42f * (float)p.g.d / 1024.f * c[best]) {
      *forms |= EPI == SG_Q ? DARE_FORM_SPLIT_Q : (EPI == SG_KV ? DARE_FORM_SPLIT_KV : DARE_FORM_SPLIT_OUT);
      return launch_gemm_f32(EPI, p, st);
    }
  }
  switch (best) {
    case 0: return launch_sgemm_as<T, EPI, 6, 4, 2>(p, n_tiles, st);
    case 1: return launch_sgemm_as<T, EPI, 4, 4, 2>(p, n_tiles, st);
    case 2: return launch_sgemm_as<T, EPI, 6, 2, 4>(p, n_tiles, st);
    case 3: return launch_sgemm_as<T, EPI, 4, 2, 4>(p, n_tiles, st);
    default: return launch_sgemm_as<T, EPI, 2, 2, 4>(p, n_tiles, st);
  }
}
}  // namespace

// ------------------------------------------------------------------------------------------------ attention
// Eq. 4 / Alg. 2 line 8 (row-sparse) and Alg. 1 line 10 (all rows): bidirectional softmax attention, no mask, fp32.
// One CTA = one head x 32 * RG query rows of one sequence, RG x KG groups of 128 threads: a group has 32 of the rows and
// every KG-th key block.  The RG groups of a key group share its K and V tile (cp.async: the next K block arrives while
// P V is computed, V while S is); KG partial results are merged at the end.  A thread owns 4 rows: scores of BKV / 16 keys
// each, then HD / 16 output columns each; the 16 lanes of a half-warp share their rows, so the softmax is shuffles and the
// probabilities pass through shared memory within the half-warp only.
// Bound by the FMA pipe and shared-memory reads like the projections (8 16-byte reads per 64 FMAs).  Row groups re-read
// the keys least, key groups leave more SMs with work when rows are few (launch rule below).  The result row is written
// into the O cache; rows that are not computed keep what they hold (Alg. 2 lines 9-10).
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
template <int HD, int RG, int KG>
struct Sa {
  static constexpr int BQ = 32 * RG, BKV = HD == 256 ? 16 : (HD == 128 || KG > 2 ? 32 : 64), JN = BKV / 16;
  static constexpr int THREADS = 128 * RG * KG;
  static constexpr int KP = HD + 4, PP = BKV + 4;                       // pitches of K / Q rows and of the probabilities
  static constexpr int VW = HD >= 64 ? 4 : 2, NC = HD / (16 * VW);      // a lane's output columns: NC vectors of VW
  static constexpr int BUF = BKV * KP + BKV * HD;                       // K and V of one block (floats)
  static constexpr int Q_OFF = 0, P_OFF = BQ * KP, KV_OFF = P_OFF + KG * BQ * PP, FLOATS = KV_OFF + KG * BUF;
  static constexpr int PART = BQ * HD + 2 * BQ;                         // a key group's part in the merge, over Q, P, K, V
  static constexpr int SMEM = FLOATS * 4;
  static_assert(SMEM <= 226 * 1024 && (KG - 1) * PART <= FLOATS, "shared memory, merge buffer");
};

template <typename T, int HD, int RG, int KG>
__global__ void __launch_bounds__(128 * RG * KG, 1) sattn_kernel(const SattnParams p) {
  using S = Sa<HD, RG, KG>;
  constexpr int BQ = S::BQ, BKV = S::BKV, JN = S::JN, KP = S::KP, PP = S::PP, VW = S::VW, NC = S::NC;
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_tok[BQ];
  const StepGeom& g = p.g;
  const int tid = threadIdx.x, grp = tid / (128 * RG), lt = tid % (128 * RG), tx = tid & 15, ty = lt >> 4;   // key group; row
  const int r0 = (ty >> 3) * 32 + (ty & 7);                             // this thread's rows: r0 + 8 i
  // one flat grid (the other two dimensions stop at 65535): heads fastest, then sequences, then row tiles, so that the first
  // row tile of every sequence, the one that has work when a refresh set is small, comes first
  const int lin = blockIdx.x, rest = lin / g.n_heads, h = lin - rest * g.n_heads;
  const int tile = rest / g.batch, b = rest - tile * g.batch, d = g.d;
  // The kernel before (the K/V projection) writes the caches only; queries and refresh set come from kernels further back,
  // complete by the time any CTA of this grid runs: they are read, through the L2, ahead of the wait.
  int row0, n_rows;
  if (p.idx) {
    const int lo = __ldcg(p.batch_off + b), hi = __ldcg(p.batch_off + b + 1);
    if (!slice_ok(lo, hi, g.tokens(), p.status) || lo + tile * BQ >= hi) { pdl_wait(); return; }
    row0 = lo + tile * BQ;
    n_rows = min(BQ, hi - row0);
  } else {
    row0 = b * g.seq_act + tile * BQ;
    n_rows = min(BQ, g.seq_act - tile * BQ);
  }
  const T* kbase = reinterpret_cast<const T*>(p.kc) + (size_t)b * g.max_seq * d + h * HD;
  const T* vbase = reinterpret_cast<const T*>(p.vc) + (size_t)b * g.max_seq * d + h * HD;
  const int n_blocks = (g.kv_len + BKV - 1) / BKV;
  float* kd = sm + S::KV_OFF + grp * S::BUF;
  float* vd = kd + BKV * KP;
  auto fetch_block = [&](float* dst, int pitch, const T* base, int blk) {       // keys past the last: zeros
    if (blk < n_blocks) {
#pragma unroll 4
      for (int c = lt; c < BKV * (HD / 4); c += 128 * RG) {
        const int r = c / (HD / 4), e = (c % (HD / 4)) * 4, key = blk * BKV + r;
        const bool ok = key < g.kv_len;
        fetch4(dst + r * pitch + e, base + (size_t)(ok ? key : 0) * d + e, ok);
      }
    }
    cp_async_commit();                             // (empty past the last block: the group count stays uniform)
  };
  if (tid < BQ) {
    int t = tid < n_rows ? (p.idx ? __ldcg(p.idx + row0 + tid) : row0 + tid) : -1;
    if (p.idx && t != -1 && !token_ok(t, g.tokens(), p.status)) t = -1;   // neither a query row to read nor a cache row to write
    s_tok[tid] = t;
  }
  __syncthreads();
  for (int c = tid; c < BQ * (HD / 4); c += S::THREADS) {
    const int r = c / (HD / 4), e = (c % (HD / 4)) * 4, t = s_tok[r];
    fetch4(sm + S::Q_OFF + r * KP + e, reinterpret_cast<const T*>(p.q) + (size_t)(t < 0 ? 0 : t) * d + h * HD + e, t >= 0);
  }
  pdl_wait();
  pdl_launch_dependents();
  fetch_block(kd, KP, kbase, grp);                 // (one group with Q)
  fetch_block(vd, HD, vbase, grp);
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
  const float* qs = sm + S::Q_OFF + r0 * KP;
  float* ps = sm + S::P_OFF + (grp * BQ + r0) * PP;
  const float* ks = kd + tx * KP;                                       // keys tx + 16 j
  const float* vs = vd + tx * VW;
  auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(128 * RG) : "memory"); };
  cp_async_wait<1>();
  __syncthreads();                                                      // Q is every group's
  for (int blk = grp; blk < n_blocks; blk += KG) {
    if (blk != grp) {
      cp_async_wait<1>();                                               // this K block; its V may still be on its way
      group_sync();
    }
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
    group_sync();                                                       // everybody is done with the K block
    fetch_block(kd, KP, kbase, blk + KG);
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
    cp_async_wait<1>();                                                 // this V block
    group_sync();                                                       // (and the half-warp's probabilities)
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
    group_sync();
    fetch_block(vd, HD, vbase, blk + KG);
  }
  cp_async_wait<0>();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], o);
  // key groups hand their parts to the first one through shared memory, idle once all are past their blocks
  if (KG > 1) {
    __syncthreads();
    float* part = sm + (grp - 1) * S::PART;                             // accumulators [BQ][HD], then maxima, then sums
    if (grp > 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + 8 * i;
#pragma unroll
        for (int n = 0; n < NC; ++n)
#pragma unroll
          for (int e = 0; e < VW; ++e) part[r * HD + n * 16 * VW + tx * VW + e] = acc[i][n][e];
        if (tx == 0) { part[BQ * HD + r] = m[i]; part[BQ * HD + BQ + r] = l[i]; }
      }
    }
    __syncthreads();
    if (grp > 0) return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + 8 * i, t = s_tok[r];
    if (t < 0) continue;
    float w[KG], mx = m[i], sum = 0.f;
#pragma unroll
    for (int k = 1; k < KG; ++k) mx = fmaxf(mx, sm[(k - 1) * S::PART + BQ * HD + r]);
    w[0] = exp2f(m[i] - mx);
    sum = w[0] * l[i];
#pragma unroll
    for (int k = 1; k < KG; ++k) {
      const float* pk = sm + (k - 1) * S::PART + BQ * HD;
      w[k] = exp2f(pk[r] - mx);
      sum = fmaf(w[k], pk[BQ + r], sum);
    }
    const float inv = 1.f / sum;
    T* dst = reinterpret_cast<T*>(p.oc) + (size_t)g.cache_row(t) * d + h * HD + tx * VW;
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
      for (int e = 0; e < VW; ++e) {
        float o = w[0] * acc[i][n][e];
#pragma unroll
        for (int k = 1; k < KG; ++k) o = fmaf(w[k], sm[(k - 1) * S::PART + r * HD + n * 16 * VW + tx * VW + e], o);
        dst[n * 16 * VW + e] = from_f<T>(o * inv);
      }
  }
}

template <typename T, int HD, int RG, int KG>
cudaError_t launch_sattn_as(const SattnParams& p, cudaStream_t st) {
  using S = Sa<HD, RG, KG>;
  static std::atomic<unsigned long long> attr_done{0};
  auto kern = sattn_kernel<T, HD, RG, KG>;
  if (cudaError_t e = ensure_dyn_smem(kern, S::SMEM, attr_done); e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(p.g.n_heads * p.g.batch * ((p.g.seq_act + S::BQ - 1) / S::BQ)), dim3(S::THREADS), S::SMEM, st,
                    1, p);
}
template <typename T, int HD>
cudaError_t launch_sattn_hd(const SattnParams& p, cudaStream_t st) {
  // rows a sequence is likely to have (a refresh set's size is known to the device only: a quarter of the window)
  const int rows = p.idx ? (p.g.seq_act + 3) / 4 : p.g.seq_act;
  // Waves of one CTA an SM, times the rows of one, times the keys its slowest group takes, times what a row and key cost in
  // that form beside the 2 x 2 one (heads of 64: 1.2-1.3 / 1 / 1.05-1.1 / 0.97-1.1).  Dense attention in us, row groups x key
  // groups 1 x 4 / 2 x 2 / 3 x 1 / 4 x 1, fp32, the pick in brackets: 4 heads of 64, 400 rows [24.6] / 36.9 / 51.2 / 63.5; 16
  // heads of 64, 2 x 384 rows 57.3 / 57.3 / [45.1] / 55.3; 12 heads of 64, 3 x 200 rows 28.7 / [24.6] / 32.8 / 38.9; 8 heads of
  // 64, 4 x 400 rows [63.5] / 67.6 / 94.2 / 65.5; 4 heads of 256, 4 x 400 rows 143 / [139] / 205 / 262.  Of twelve sizes timed
  // the pick was the fastest at eleven; 8 heads of 128, 4 x 400 rows: 98.3 / 117 / 176 / [115] (1.15 is too much there).
  auto cost = [&](int bq, int kg, int bkv, float f) {
    const int tiles = p.g.n_heads * p.g.batch * ((rows + bq - 1) / bq), blocks = (p.g.kv_len + bkv - 1) / bkv;
    return (float)((tiles + kSms - 1) / kSms) * (float)bq * (float)((blocks + kg - 1) / kg * kg * bkv) * f;
  };
  const int b1 = Sa<HD, 1, 4>::BKV, b2 = Sa<HD, 2, 2>::BKV, b3 = Sa<HD, 3, 1>::BKV;
  const float c1 = cost(32, 4, b1, 1.15f), c2 = cost(64, 2, b2, 1.f), c3 = cost(96, 1, b3, 1.05f), c4 = cost(128, 1, b3, 1.f);
  if (c1 <= c2 && c1 <= c3 && c1 <= c4) return launch_sattn_as<T, HD, 1, 4>(p, st);
  if (c2 <= c3 && c2 <= c4) return launch_sattn_as<T, HD, 2, 2>(p, st);
  if (c3 <= c4) return launch_sattn_as<T, HD, 3, 1>(p, st);
  return launch_sattn_as<T, HD, 4, 1>(p, st);
}
}  // namespace

// ------------------------------------------------------------------------------------------------ launches
template <typename T>
cudaError_t launch_q_simt(const SimtStep& s, const T* xn, const T* w_q, T* q, cudaStream_t st, int* launches) {
  SgemmParams p = {};
  p.a = xn; p.g = s.g; p.rows = s.g.tokens(); p.w0 = w_q; p.out0 = q;
  p.rope = reinterpret_cast<const float2*>(s.rope_cs); p.q_prev = s.q_prev; p.scores = s.scores; p.q_raw = s.q_raw;
  p.has_prev = s.has_prev; p.status = s.status;
  ++*launches;
  if (cudaError_t e = launch_sgemm<T, SG_Q>(p, p.rows, s.forms, st); e != cudaSuccess) return e;
  if (s.g.head_dim <= 64) return cudaSuccess;
  ++*launches;
  return launch_pdl(score_kernel, dim3((p.rows + 7) / 8), dim3(256), 0, st, 1, s.q_raw, s.q_prev, s.scores, p.has_prev, s.g);
}
template <typename T>
cudaError_t launch_kv_simt(const SimtStep& s, const T* xn, const int* idx, const int* count, const T* w_k, const T* w_v,
                           T* kc, T* vc, cudaStream_t st) {
  SgemmParams p = {};
  p.a = xn; p.idx = idx; p.count = count; p.g = s.g; p.rows = s.g.tokens(); p.w0 = w_k; p.w1 = w_v; p.out0 = kc; p.out1 = vc;
  p.rope = reinterpret_cast<const float2*>(s.rope_cs); p.status = s.status;
  // (a refresh set is sized for a quarter of the tokens)
  return launch_sgemm<T, SG_KV>(p, idx ? (p.rows + 3) / 4 : p.rows, s.forms, st);
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
  return launch_sgemm<T, SG_OUT>(p, p.rows, s.forms, st);
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
