// SwiGLU projection of few rows: act[t, n] = silu(sum_k W_G[n, k] x[t, k]) * (sum_k W_U[n, k] x[t, k]) for at most 256 rows
// (the decode window of a stack), tcgen05.  With so few rows the launch is a stream of both weight matrices, and what
// matters is that every SM pulls its share of it at the same time: the tile width is not fixed, it is the d_ff columns
// over the SMs (or SM pairs) of the device, rounded up to the step of an MMA's N (16, of two-CTA MMAs 32), so that the
// launch is ONE wave of equal tiles.
// (With tiles of 128 outputs d_ff = 12288 is 96 tiles on 74 SM pairs: a full wave and a wave of 22; 256 rows x 4096 took
// 55.7 us in that form, the second wave with its reduction split, against 31 us for the weights at the copy peak.)
//   PAIR   two CTAs share M = 256 MMAs (cta_group::2): each keeps 128 rows of x and half of the tile's weight rows
//   !PAIR  one row tile of at most 128 rows per CTA
// Gate and up projection are two MMAs of N = `width` per 16 k-elements into tensor-memory columns [0, 256) and [256, 512).
//   warp 0     TMA producer: x rows, then `width` (PAIR: width / 2) rows of each matrix per 64 k-elements; the weight
//              tiles of the first stages start before the wait on the kernel in front
//   warp 1     MMA issuer (PAIR: of the even CTA)
//   all eight  finishing pass: thread <-> row, 16 columns at a time tensor memory -> registers -> 32-byte row segments
#include "layer.h"
#include "tc.h"
#include "tc_ptx.cuh"

namespace dare {

using namespace ptx;

namespace {
constexpr int BM = 128, BK = 64;
constexpr int A_BYTES = BM * BK * 2;
constexpr int kRing = 222 * 1024;                   // bytes of operand stages (as many whole ones as fit, at most kMaxStages)
constexpr int kMaxStages = 8;
constexpr int SMEM_TOTAL = kRing + 256 + 1024;
static_assert(SMEM_TOTAL <= 227 * 1024, "shared memory of one CTA");
constexpr int kThreads = 256;

template <bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
swiglu_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_g,
              const __grid_constant__ CUtensorMap tm_u, const int width, const int rows, const int d_ff, const int K,
              __nv_bfloat16* __restrict__ act, int* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + kRing);
  uint64_t* empty_bar = full_bar + kMaxStages;
  uint64_t* accum_bar = empty_bar + kMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum_bar + 1);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int pr = PAIR ? (int)cluster_ctarank() : 0;
  const int n0 = (PAIR ? (int)blockIdx.x / 2 : (int)blockIdx.x) * width;       // first output of the tile
  const int w_rows = PAIR ? width / 2 : width;      // rows of each matrix this CTA brings: a multiple of 8, so that the
  const int w_bytes = w_rows * BK * 2;              // second matrix starts on a 1024-byte boundary as well
  const int stage_bytes = A_BYTES + 2 * w_bytes;
  const int stages = min(kMaxStages, kRing / stage_bytes), KB = K / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    mbar_init(accum_bar, 1);
    fence_mbar_init();
    prefetch_tmap(&tm_x);
    prefetch_tmap(&tm_g);
    prefetch_tmap(&tm_u);
  }
  if (warp == 1) {
    if (PAIR) { tmem_alloc2(tmem_slot, 512); tmem_relinquish2(); }
    else { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  }
  tc_fence_before();
  __syncthreads();
  uint32_t tmem_base;
  if (PAIR) {
    cluster_sync_all();              // both CTAs have their barriers and tensor memory before either touches the other's
    tc_fence_after();
    tmem_base = ld_cluster_u32(map_to_cta(smem_u32(tmem_slot), 0));
  } else {
    tc_fence_after();
    tmem_base = *tmem_slot;
  }
  auto load_w = [&](int i, int s) {                 // one thread; PAIR: the bytes of both CTAs count on the even one's barrier
    uint8_t* dst = smem + s * stage_bytes + A_BYTES;
    if (PAIR) {
      const uint32_t fb = map_to_cta(smem_u32(&full_bar[s]), 0);
      if (pr == 0) mbar_arrive_expect_tx(&full_bar[s], 2u * stage_bytes);
      tma_load_2d_pair(dst, &tm_g, i * BK, n0 + pr * w_rows, fb);
      tma_load_2d_pair(dst + w_bytes, &tm_u, i * BK, n0 + pr * w_rows, fb);
    } else {
      mbar_arrive_expect_tx(&full_bar[s], (uint32_t)stage_bytes);
      tma_load_2d(dst, &tm_g, i * BK, n0, &full_bar[s]);
      tma_load_2d(dst + w_bytes, &tm_u, i * BK, n0, &full_bar[s]);
    }
  };
  auto load_x = [&](int i, int s) {
    uint8_t* dst = smem + s * stage_bytes;
    if (PAIR) tma_load_2d_pair(dst, &tm_x, i * BK, pr * BM, map_to_cta(smem_u32(&full_bar[s]), 0));
    else tma_load_2d(dst, &tm_x, i * BK, 0, &full_bar[s]);
  };
  // Weights asked for while the kernel before (a short norm) finishes: four stages; all of them took bandwidth from it.  Decoding
  // step with every stage / four / three / two early, us: six layers of width 2048, 256 rows 500.2 / 496.9 / 497.0 / 498.1, 2 x 32
  // rows 491.6 / 485.5 / 485.5 / 483.7; eight of 4096, 256 rows 1388.7 / 1384.5 / 1385.8 / 1386.6.
  const int n_early = min(min(stages, 4), KB);
  if (warp == 0 && lane == 0)
    for (int i = 0; i < n_early; ++i) load_w(i, i);
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    if (elect_one())
      for (int i = 0; i < n_early; ++i) load_x(i, i);
    __syncwarp();
    for (int i = n_early; i < KB; ++i) {
      const int s = i % stages;
      mbar_wait(&empty_bar[s], ((i / stages) & 1) ^ 1, status);
      if (elect_one()) { load_w(i, s); load_x(i, s); }
      __syncwarp();
    }
  } else if (warp == 1 && pr == 0) {
    const uint32_t idesc = idesc_bf16(PAIR ? 2 * BM : BM, width);
    for (int i = 0; i < KB; ++i) {
      const int s = i % stages;
      mbar_wait(&full_bar[s], (i / stages) & 1, status);
      tc_fence_after();
      if (elect_one()) {
        const uint32_t a_addr = smem_u32(smem + s * stage_bytes);
        const uint64_t a = smem_desc_k_sw128(a_addr), g = smem_desc_k_sw128(a_addr + A_BYTES),
                       u = smem_desc_k_sw128(a_addr + A_BYTES + w_bytes);
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) {
          const uint32_t acc = (i | k) != 0 ? 1u : 0u;
          if (PAIR) {
            umma2_ss(tmem_base, a + 2 * k, g + 2 * k, idesc, acc);
            umma2_ss(tmem_base + 256, a + 2 * k, u + 2 * k, idesc, acc);
          } else {
            umma_ss(tmem_base, a + 2 * k, g + 2 * k, idesc, acc);
            umma_ss(tmem_base + 256, a + 2 * k, u + 2 * k, idesc, acc);
          }
        }
        if (PAIR) {
          umma2_commit(map_to_cta(smem_u32(&empty_bar[s]), 0));
          umma2_commit(map_to_cta(smem_u32(&empty_bar[s]), 1));
          if (i == KB - 1) {
            umma2_commit(map_to_cta(smem_u32(accum_bar), 0));
            umma2_commit(map_to_cta(smem_u32(accum_bar), 1));
          }
        } else {
          umma_commit(&empty_bar[s]);
          if (i == KB - 1) umma_commit(accum_bar);
        }
      }
      __syncwarp();
    }
  }
  mbar_wait(accum_bar, 0, status);
  tc_fence_after();
  {
    const int quarter = warp & 3, r = pr * BM + quarter * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const int chunks = min(width, d_ff - n0) / 16;                              // (d_ff and n0 are multiples of 16)
    const int c_half = (chunks + 1) / 2;                                        // two warps per lane quarter
    __nv_bfloat16* dst = act + (size_t)r * d_ff + n0;
    for (int c = (warp >> 2) * c_half; c < ((warp >> 2) ? chunks : c_half); ++c) {
      float g[16], u[16];
      tmem_ld_32x16_nowait(t_lane + c * 16, g);
      tmem_ld_32x16_nowait(t_lane + 256 + c * 16, u);
      tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 16; ++e) g[e] = g[e] / (1.f + __expf(-g[e])) * u[e];
      if (r < rows) {
        reinterpret_cast<uint4*>(dst + c * 16)[0] = pack8_bf16(g);
        reinterpret_cast<uint4*>(dst + c * 16)[1] = pack8_bf16(g + 8);
      }
    }
  }
  tc_fence_before();
  if (PAIR) cluster_sync_relaxed(); else __syncthreads();      // nobody frees tensor memory its partner's MMAs may still use
  if (warp == 1) {
    if (PAIR) tmem_dealloc2(*tmem_slot, 512);
    else tmem_dealloc(*tmem_slot, 512);
  }
}
}  // namespace

// One wave: the columns over the SMs (pair: SM pairs), rounded up to a step of N; at most 256, the width of an MMA.
int swiglu_width(int d_ff, int sms, bool pair) {
  const int units = pair ? sms / 2 : sms, step = pair ? 32 : 16;
  const int w = units > 0 ? ((d_ff + units - 1) / units + step - 1) / step * step : 256;
  return w < 256 ? w : 256;
}

cudaError_t launch_swiglu(const CUtensorMap& x, const CUtensorMap& gate, const CUtensorMap& up, int width, int rows, int d_ff,
                          int K, __nv_bfloat16* act, int* status, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  const bool pair = rows > BM;
  if (rows > 2 * BM || width % (pair ? 32 : 16) != 0 || width > 256 || d_ff % 16 != 0 || K % BK != 0) return cudaErrorInvalidValue;
  const int tiles = (d_ff + width - 1) / width;
  static std::atomic<unsigned long long> done1{0}, done2{0};
  if (pair) {
    if (cudaError_t e = ensure_dyn_smem(swiglu_kernel<true>, SMEM_TOTAL, done2); e != cudaSuccess) return e;
    return launch_pdl_xz(swiglu_kernel<true>, dim3(2 * tiles), dim3(kThreads), SMEM_TOTAL, st, 2, 1, x, gate, up, width, rows, d_ff,
                         K, act, status);
  }
  if (cudaError_t e = ensure_dyn_smem(swiglu_kernel<false>, SMEM_TOTAL, done1); e != cudaSuccess) return e;
  return launch_pdl(swiglu_kernel<false>, dim3(tiles), dim3(kThreads), SMEM_TOTAL, st, 1, x, gate, up, width, rows, d_ff, K, act,
                    status);
}

}  // namespace dare
