// fp32 projections on the tensor cores: C[m, n] = sum_k A[m, k] * W[n, k] with fp32 operands and fp32 accuracy.
// An fp32 number is the sum of three bf16 numbers (8 + 8 + 8 bits of mantissa), here scaled: x = h + m / 2^8 + l / 2^16, the split
// of Henry, Tang and Heinecke, "Leveraging the bfloat16 Artificial Intelligence Datatype for Higher-Precision Computations" (ARITH
// 2019).  With the scales it holds exactly for every finite x that does not round up to infinity: h, m and l are multiples of 2^-133,
// bf16's smallest number, however small x is (without them the last part is lost below about 2^-110, and weights of size 1e-35 left
// 44 units of the error below).  Of the nine products of two such sums six are taken, hh, hm, mh, mm, hl, lh; the others are below
// 2^-25 of the product.  Products of bf16 are exact on the tensor core, so what is left to lose is the accumulation: the tensor
// core's adds truncate, each by up to an ulp of the running sum, and where the sum does not cancel these errors share a sign.  So
// no sum of full size is added to there: every 16 k-elements of hh have an accumulator of their own (16 products of 8 x 8 bits fit
// its 24 bits nearly always), only the small products, 2^-8 of the sum and less, add up over the whole reduction, those of scale
// 2^8 and of 2^16 apart.  The rest is added in fp32 registers, rounded to nearest: the four accumulators of a block of 64 as a
// tree, the blocks in chains of two to eight, the chains.
// Error of V against fp64 in units of 2^-24 (2-norms), CUDA-core tiles that the launch rule takes otherwise / split, by operands:
//   width                        128          192          256          384          448          512          1024
//   zero-mean normal             1.49 / 0.95  2.20 / 0.96  2.51 / 1.06  2.26 / 1.12  3.25 / 1.11  3.47 / 1.18  4.86 / 1.28
//   their magnitudes             0.75 / 0.72  1.11 / 0.72  1.10 / 0.72  0.95 / 0.87  1.46 / 0.77  1.46 / 0.76  2.01 / 0.82
//   normal + 1                   0.78 / 0.79  1.07 / 0.71  1.14 / 0.76  0.95 / 0.81  1.40 / 0.71  1.46 / 0.73  1.94 / 0.75
//   normal, every 61st x 60      1.37 / 1.24  2.32 / 1.24  2.59 / 1.32  2.27 / 1.37  3.37 / 1.36  3.58 / 1.41  4.99 / 1.51
//   +- exp(2 normal)             1.49 / 1.26  2.42 / 1.20  2.31 / 1.34  2.16 / 1.32  3.02 / 1.37  3.22 / 1.38  4.17 / 1.39
//   exp(normal)                  0.81 / 0.80  1.10 / 0.73  1.20 / 0.81  0.95 / 0.84  1.50 / 0.79  1.57 / 0.86  2.13 / 0.89
//   exp(2 normal), one sign      1.28 / 2.25  2.00 / 2.11  2.02 / 1.99  1.68 / 2.09  4.65 / 2.25  3.19 / 2.31  4.41 / 2.51
// (the last line: 16 products of one sign that span far more than 2^8, whose small ones are cut where they are lined up.  Four hh steps
// into one accumulator, as it was first: 1.39 to 1.83 on the first line, 1.45 to 1.67 on the second, 5.7 to 8.1 on the last.)
// Bound by the splitting, which the adding up beside it slows.  The products of one part of A with two parts of W that lie side by
// side are one MMA, with the accumulators of both scales side by side as well: 16 MMAs a block that read 112 KB of shared memory,
// not 24 that read 144.  A step of 2 x 384 tokens of width 1024, key and value reuse, 171.5 us on the CUDA cores, 122 here (24 MMAs:
// 124; unscaled, one accumulator a block, less accurate: 117), dense of 4 x 400 498 -> 275 us (277; 264).
// A CTA takes 128 rows x 64 columns: 32 rotary pairs, columns (j, j + head_dim / 2) of the heads they belong to, as in simt.cu.
//   warps 0-3   add up: thread <-> row, tensor memory -> registers, into the finished tile
//   warps 4-11  fetch the operands (16 bytes a lane, whole lines), a block ahead of the one they split, and write the parts
//               into a ring of two stages (72 KB each: 192 rows x 64 k x 3 parts) in the 128-byte-swizzled layout
//   warp 12     issues the 16 MMAs (M 128, N 64 or 128, K 16) of a block
#include "sgemm.h"
#include "tc_ptx.cuh"

namespace dare {

using namespace ptx;

namespace {
constexpr int BM = 128, BN = 64, BK = 64, STAGES = 2, kSplitters = 256, kThreads = 128 + kSplitters + 32;
// Tensor memory, 64 columns each: an accumulator for the hh products of every 16 k-elements of a block, the small products of the
// whole reduction by their scale (2^8: hm, mh; 2^16: hl, mm, lh), and the sums put aside.
constexpr int HH = BK / 16, ACC_MID = HH * BN, ACC_LOW = ACC_MID + BN, ACC_ASIDE = ACC_LOW + BN, TMEM_COLS = 512;
static_assert(HH == 4 && ACC_ASIDE + BN <= TMEM_COLS, "tensor memory of one CTA");
constexpr int A_PART = BM * BK * 2, W_PART = BN * BK * 2, STAGE_BYTES = 3 * (A_PART + W_PART), W_OFFSET = 3 * A_PART;
constexpr int CHUNKS = (BM + BN) * (BK / 4) / kSplitters;              // 16-byte chunks of a stage per splitting thread
constexpr int ROWS = kSplitters / (BK / 4), W_CHUNKS = BN / ROWS;      // 16 rows a chunk index
constexpr int SLOT_OFFSET = STAGES * STAGE_BYTES, SLOT_BYTES = (BM + BN) * BK * 4;   // an fp32 block on its way
constexpr int BAR_OFFSET = SLOT_OFFSET + SLOT_BYTES;
constexpr int SMEM_TOTAL = BAR_OFFSET + 256 + 1024;
constexpr int TILE_PITCH = BN + 4;                                     // floats of a row of the finished tile
static_assert(CHUNKS * kSplitters == (BM + BN) * (BK / 4) && SMEM_TOTAL + 1024 <= 232448, "shared memory of one CTA");

// Two outputs the plain way: of operands that are no finite numbers (inf times a part that is zero would be NaN), or sums that
// overflowed.
__device__ __noinline__ float2 plain_dots(const float* a, const float* w0, const float* w1, int K) {
  float2 s = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    const float4 x = *reinterpret_cast<const float4*>(a + k), y = *reinterpret_cast<const float4*>(w0 + k),
                 z = *reinterpret_cast<const float4*>(w1 + k);
    s.x = fmaf(x.x, y.x, s.x); s.x = fmaf(x.y, y.y, s.x); s.x = fmaf(x.z, y.z, s.x); s.x = fmaf(x.w, y.w, s.x);
    s.y = fmaf(x.x, z.x, s.y); s.y = fmaf(x.y, z.y, s.y); s.y = fmaf(x.z, z.z, s.y); s.y = fmaf(x.w, z.w, s.y);
  }
  return s;
}
// (volatile: a load that stays where it is written, a block ahead of its use)
__device__ __forceinline__ float4 load_now(const float* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool finite(float x) { return fabsf(x) <= 3.402823466e38f; }
}  // namespace

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1) gemm_f32_kernel(const SgemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + BAR_OFFSET);
  uint64_t* empty_bar = full_bar + STAGES;
  uint64_t* acc_full = empty_bar + STAGES;
  uint64_t* acc_empty = acc_full + 1;
  uint64_t* all_done = acc_empty + 1;          // every MMA of the tile complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(all_done + 1);
  float* tile = reinterpret_cast<float*>(smem);
  // of a row: its token (-1: no such row, or one whose token failed its check), its row of A (then that of token 0: read, and the
  // result not written), cache row and position
  __shared__ int s_tok[BM], s_pos[BM];
  __shared__ size_t s_row[BM], s_crow[BM];
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31, tid = (int)threadIdx.x;
  const int K = p.g.d, half = p.g.head_dim >> 1, lh = 31 - __clz(half), KB = K / BK;
  const int n_tiles = K / BN;
  const bool second = EPI == SG_KV && (int)blockIdx.x >= n_tiles;
  const int pair0 = ((int)blockIdx.x - (second ? n_tiles : 0)) * (BN / 2);
  const float* w = reinterpret_cast<const float*>(second ? p.w1 : p.w0);
  auto column = [&](int pair) { return (pair >> lh) * (2 * half) + (pair & (half - 1)); };
  const int m0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * BM;
  // (row tiles past the first of a gathered launch are usually empty: they look at the count first)
  if (p.count != nullptr && m0 > 0) {
    pdl_wait();
    if (m0 >= checked_count(*p.count, p.rows, p.status)) return;
  }
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full_bar[s], kSplitters / 32); mbar_init(&empty_bar[s], 1); }
    mbar_init(acc_full, 1); mbar_init(acc_empty, 4); mbar_init(all_done, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  // a splitting thread's chunks: rows row_of + 16 i of W's 64 and A's 128, elements kc .. kc + 3 of a block.  The weights do not
  // depend on the kernel before: their first chunks are on their way while it drains.
  const int st_id = tid - 128, row_of = st_id >> 4, kc = (st_id & 15) * 4;
  const bool splitter = warp >= 4 && warp < 12;
  const float* src[CHUNKS];
  float4 v0[CHUNKS];
  if (splitter) {
#pragma unroll
    for (int i = 0; i < W_CHUNKS; ++i) {
      const int row = row_of + ROWS * i;
      src[i] = w + (size_t)(column(pair0 + (row & 31)) + (row >> 5) * half) * K + kc;
      v0[i] = load_now(src[i]);
    }
  }
  pdl_wait();
  pdl_launch_dependents();
  const int m_eff = p.count ? checked_count(*p.count, p.rows, p.status) : p.rows;
  const bool active = m0 < m_eff;                // uniform over the CTA
  if (tid < BM) {
    int t = m0 + tid < m_eff ? (p.idx ? p.idx[m0 + tid] : m0 + tid) : -1;
    if (p.idx && t != -1 && !token_ok(t, p.g.tokens(), p.status)) t = -1;   // (not written)
    const int tc = max(t, 0);
    s_tok[tid] = t;
    s_pos[tid] = p.g.position(tc);
    s_crow[tid] = (size_t)p.g.cache_row(tc);
    s_row[tid] = p.a_cache_rows ? s_crow[tid] : (size_t)tc;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (active && splitter) {
#pragma unroll
    for (int i = W_CHUNKS; i < CHUNKS; ++i) {
      src[i] = reinterpret_cast<const float*>(p.a) + s_row[row_of + ROWS * i - BN] * K + kc;
      v0[i] = load_now(src[i]);
    }
    // Even blocks come into registers, odd ones into a slot of shared memory (a thread's own chunks: nobody else waits for
    // them), the next on its way while one is split.
    auto fetch = [&]() {
#pragma unroll
      for (int i = 0; i < CHUNKS; ++i) v0[i] = load_now(src[i]);
    };
    float* slot = reinterpret_cast<float*>(smem + SLOT_OFFSET) + st_id * 4;
    auto fetch_slot = [&]() {
#pragma unroll
      for (int i = 0; i < CHUNKS; ++i) {
        cp_async_16(smem_u32(slot + i * (kSplitters * 4)), src[i] + BK, 16u);
        src[i] += 2 * BK;                        // (the next even block)
      }
      cp_async_commit();
    };
    auto split2 = [](float x, float y, uint32_t (&o)[3]) {
      float2 v = make_float2(x, y);
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
        o[part] = *reinterpret_cast<const uint32_t*>(&b);
        if (part < 2)
          v = __fmul2_rn(__ffma2_rn(make_float2(__uint_as_float(o[part] << 16), __uint_as_float(o[part] & 0xffff0000u)),
                                    make_float2(-1.f, -1.f), v), make_float2(256.f, 256.f));
      }
    };
    const uint32_t thread_at = smem_u32(smem) + (uint32_t)(row_of * 128 + (((kc >> 3) ^ (row_of & 7)) << 4) + (kc & 4) * 2);
    auto put = [&](auto chunk, int kb) {
      const int s = kb % STAGES;
      mbar_wait(&empty_bar[s], ((kb / STAGES) & 1) ^ 1, p.status);
      const uint32_t stage = thread_at + (uint32_t)(s * STAGE_BYTES);
#pragma unroll
      for (int i = 0; i < CHUNKS; ++i) {
        const uint32_t dst = stage + (uint32_t)(i < W_CHUNKS ? W_OFFSET + ROWS * i * 128 : (ROWS * i - BN) * 128);
        constexpr uint32_t kPart[2] = {A_PART, W_PART};
        const uint32_t part_bytes = kPart[i < W_CHUNKS ? 1 : 0];
        uint32_t a[3], b[3];
        const float4 v = chunk(i);
        split2(v.x, v.y, a);
        split2(v.z, v.w, b);
#pragma unroll
        for (int part = 0; part < 3; ++part)
          asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + part * part_bytes), "r"(a[part]), "r"(b[part]) : "memory");
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_bar[s]);
    };
    auto from_regs = [&](int i) { return v0[i]; };
    auto from_slot = [&](int i) { return *reinterpret_cast<const float4*>(slot + i * (kSplitters * 4)); };
    if (KB > 1) fetch_slot();
    for (int kb = 0; kb < KB; kb += 2) {
      put(from_regs, kb);
      if (kb + 2 < KB) fetch();
      if (kb + 1 < KB) {
        cp_async_wait<0>();
        put(from_slot, kb + 1);
        if (kb + 3 < KB) fetch_slot();
      }
    }
  } else if (active && warp == 12) {
    constexpr uint32_t idesc = idesc_bf16(BM, BN), idesc2 = idesc_bf16(BM, 2 * BN);
    for (int kb = 0; kb < KB; ++kb) {
      const int s = kb % STAGES;
      mbar_wait(&full_bar[s], (kb / STAGES) & 1, p.status);
      mbar_wait(acc_empty, (kb & 1) ^ 1, p.status);
      tc_fence_after();
      if (elect_one()) {
        const uint32_t stage = smem_u32(smem) + (uint32_t)(s * STAGE_BYTES);
        uint64_t ad[3], wd[3];
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          ad[part] = smem_desc_k_sw128(stage + part * A_PART);
          wd[part] = smem_desc_k_sw128(stage + W_OFFSET + part * W_PART);
        }
        // hh first: while the small products run, the other warps read these four
#pragma unroll
        for (int k = 0; k < HH; ++k) umma_ss(tmem_base + k * BN, ad[0] + 2 * k, wd[0] + 2 * k, idesc, 0u);
        umma_commit(acc_full);
#pragma unroll
        for (int k = 0; k < HH; ++k) umma_ss(tmem_base + ACC_MID, ad[0] + 2 * k, wd[1] + 2 * k, idesc2, (kb | k) != 0 ? 1u : 0u);   // hm, hl
#pragma unroll
        for (int k = 0; k < HH; ++k) umma_ss(tmem_base + ACC_MID, ad[1] + 2 * k, wd[0] + 2 * k, idesc2, 1u);                        // mh, mm
#pragma unroll
        for (int k = 0; k < HH; ++k) umma_ss(tmem_base + ACC_LOW, ad[2] + 2 * k, wd[0] + 2 * k, idesc, 1u);                         // lh
        umma_commit(&empty_bar[s]);
        if (kb == KB - 1) umma_commit(all_done);
      }
      __syncwarp();
    }
  } else if (active) {
    const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
    float2 acc[BN / 2];
#pragma unroll
    for (int c = 0; c < BN / 2; ++c) acc[c] = make_float2(0.f, 0.f);
    auto pair = [](const float* v, int e) { return make_float2(v[e], v[e + 1]); };
    const float none[8] = {};
#pragma unroll
    for (int c = 0; c < BN; c += 8) tmem_st_32x8(t_lane + ACC_ASIDE + c, none);
    const int chain = KB <= 6 ? 2 : max(4, KB / 8);                          // then its sum is put aside
    int left = chain;
#pragma unroll 1
    for (int kb = 0; kb < KB; ++kb) {
      mbar_wait(acc_full, kb & 1, p.status);
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < BN; c += 8) {
        float v[HH][8];
#pragma unroll
        for (int k = 0; k < HH; ++k) tmem_ld_32x8_nowait(t_lane + k * BN + c, v[k]);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; e += 2)
          acc[(c + e) / 2] = __fadd2_rn(acc[(c + e) / 2], __fadd2_rn(__fadd2_rn(pair(v[0], e), pair(v[1], e)),
                                                                     __fadd2_rn(pair(v[2], e), pair(v[3], e))));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
      if (--left == 0) {
        left = chain;
#pragma unroll
        for (int c = 0; c < BN; c += 8) {
          float sum[8];
          tmem_ld_32x8_nowait(t_lane + ACC_ASIDE + c, sum);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            const float2 x = __fadd2_rn(pair(sum, e), acc[(c + e) / 2]);
            sum[e] = x.x; sum[e + 1] = x.y;
            acc[(c + e) / 2] = make_float2(0.f, 0.f);
          }
          tmem_st_32x8(t_lane + ACC_ASIDE + c, sum);
        }
      }
    }
    mbar_wait(all_done, 0, p.status);
    tc_fence_after();
    const float2 down = make_float2(1.f / 256.f, 1.f / 256.f);
#pragma unroll
    for (int c = 0; c < BN; c += 8) {
      float mid[8], low[8], sum[8];
      tmem_ld_32x8_nowait(t_lane + ACC_MID + c, mid);
      tmem_ld_32x8_nowait(t_lane + ACC_LOW + c, low);
      tmem_ld_32x8_nowait(t_lane + ACC_ASIDE + c, sum);
      tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 8; e += 2)
        acc[(c + e) / 2] = __fadd2_rn(__ffma2_rn(__ffma2_rn(pair(low, e), down, pair(mid, e)), down, acc[(c + e) / 2]), pair(sum, e));
    }
    // the tile through the ring, idle by now (every MMA that read it is complete)
#pragma unroll
    for (int c = 0; c < BN; c += 4)
      *reinterpret_cast<float4*>(tile + tid * TILE_PITCH + c) = make_float4(acc[c / 2].x, acc[c / 2].y, acc[c / 2 + 1].x, acc[c / 2 + 1].y);
  }
  if (active) {
    // ---- the projection's own tail: a warp a row, lane <-> rotary pair, the table reads of four rows in flight together
    constexpr int NW = kThreads / 32, RB = 5;    // rows warp, warp + 13, ...: two batches of five
    const bool rotate = EPI == SG_Q || (EPI == SG_KV && !second);
    float* out = reinterpret_cast<float*>(second ? p.out1 : p.out0);
    const int pj = pair0 + lane, jj = pj & (half - 1), col = column(pj);
    const bool scoring = EPI == SG_Q && (pj >> lh) == p.g.score_head;                 // this lane's pair is the scoring head's
    const bool score_tile = EPI == SG_Q && half <= 32 && ((p.g.score_head * half) >> 5) == pair0 >> 5;
    float2 cs[RB], old[RB];
    auto read_tables = [&](int r0) {
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        const int r = min(r0 + NW * k, BM - 1);
        cs[k] = old[k] = make_float2(0.f, 0.f);
        if (rotate) cs[k] = p.rope[(size_t)s_pos[r] * half + jj];
        if (score_tile && scoring && p.has_prev) {
          const float* qp = p.q_prev + s_crow[r] * (2 * half) + jj;
          old[k] = make_float2(qp[0], qp[half]);
        }
      }
    };
    read_tables(warp);
    __syncthreads();
    for (int r0 = warp; r0 < BM; r0 += NW * RB) {
      if (r0 != warp) read_tables(r0);
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        const int r = r0 + NW * k, t = r < BM ? s_tok[r] : -1;
        if (t < 0) continue;                       // (uniform over the warp)
        const size_t cr = s_crow[r];
        float a = tile[r * TILE_PITCH + lane], b = tile[r * TILE_PITCH + 32 + lane];
        if (!finite(a) || !finite(b)) {
          const float2 ab = plain_dots(reinterpret_cast<const float*>(p.a) + s_row[r] * K, w + (size_t)col * K,
                                       w + (size_t)(col + half) * K, K);
          if (!finite(a)) a = ab.x;
          if (!finite(b)) b = ab.y;
        }
        if (score_tile) {
          // Sec. 3.1 on the un-rotated query; the current one is kept for the next step (Sec. 3.2)
          float dot = 0.f, n1 = 0.f, n2 = 0.f;
          if (scoring) {
            dot = fmaf(a, old[k].x, b * old[k].y); n1 = fmaf(a, a, b * b); n2 = fmaf(old[k].x, old[k].x, old[k].y * old[k].y);
            float* qp = p.q_prev + cr * (2 * half) + jj;
            qp[0] = a; qp[half] = b;
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            dot += __shfl_xor_sync(0xffffffffu, dot, o);
            n1 += __shfl_xor_sync(0xffffffffu, n1, o);
            n2 += __shfl_xor_sync(0xffffffffu, n2, o);
          }
          if (lane == 0) {
            const float den = sqrtf(n1) * sqrtf(n2);
            p.scores[t] = p.has_prev ? 1.f - (den > 0.f ? dot / den : 0.f) : __int_as_float(0x7f800000);
          }
        } else if (scoring) {                      // (heads wider than 64 span several tiles: score_kernel)
          float* qr = p.q_raw + (size_t)t * (2 * half) + jj;
          qr[0] = a; qr[half] = b;
        }
        if (rotate) {
          const float ra = a * cs[k].x - b * cs[k].y, rb = a * cs[k].y + b * cs[k].x;
          a = ra; b = rb;
        }
        float* dst = out + (EPI == SG_KV ? cr : (size_t)t) * K + col;
        dst[0] = a;
        dst[half] = b;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
}

template <int EPI>
static cudaError_t launch_as(const SgemmParams& p, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  if (cudaError_t e = ensure_dyn_smem(gemm_f32_kernel<EPI>, SMEM_TOTAL, attr_done); e != cudaSuccess) return e;
  const int row_tiles = (p.rows + BM - 1) / BM, nz = (row_tiles + 65534) / 65535;
  return launch_pdl(gemm_f32_kernel<EPI>, dim3(p.g.d / BN * (EPI == SG_KV ? 2 : 1), (row_tiles + nz - 1) / nz, nz), dim3(kThreads),
                    SMEM_TOTAL, st, 1, p);
}
cudaError_t launch_gemm_f32(int epi, const SgemmParams& p, cudaStream_t st) {
  if (p.rows <= 0) return cudaSuccess;
  if (epi == SG_Q) return launch_as<SG_Q>(p, st);
  if (epi == SG_KV) return launch_as<SG_KV>(p, st);
  return launch_as<SG_OUT>(p, st);
}

}  // namespace dare
