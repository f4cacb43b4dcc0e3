// Stand-alone drift score and threshold/compaction for token counts far beyond one layer step (millions of rows):
// the same arithmetic as inside the layer step, organised for HBM bandwidth.
//   drift score (Sec. 3.1): hd / 4 lanes per row, 16-byte loads of both query rows, shuffle reduction
//   compaction (Eq. 2, complement): three passes over tiles of 16384 scores; the scores are read once
//     (1) per-tile count of refreshed tokens and the decisions themselves, a plain bit array -> scratch
//     (2) exclusive scan of the tile counts (one CTA) -> scratch, total -> *count
//     (3) per-tile compaction from the decision bits, written at the tile's offset: ascending index list
// No CTA waits for another; the order of the list does not depend on scheduling.  Every kernel here is launched programmatically
// dependent, its launch latency hidden behind the kernel before: with the drift scores and pass 1 among them, scores, quantile
// and compaction of 20000 rows of 64 take 19.9 us, 22.5 before.
// A single pass (tiles handed out by ticket, every CTA publishing its tile's count and adding up the counts published
// before it back to the nearest known running total, entries staged in shared memory and written as whole lines) was
// built as well, list and count identical, and measured on the same 2^24 scores against 22.6 us for the three passes:
// 27.7-32.3 us with one tile per CTA (16384 down to 4096 scores per tile, walk by one warp), 33-40 us with the walk by
// the whole CTA, 40-65 us with resident CTAs that have the next two tiles copied into shared memory (bulk copies on
// an mbarrier) while they work.  All CTAs of a wave reach the walk at the same time, so the nearest known total is a
// whole wave back, and a CTA's loads do not overlap its walk: the chain per tile (scores -> scan -> publish -> walk
// -> write) is several microseconds long, and what a CTA has in flight during it does not cover it.
#include <math.h>
#include <algorithm>
#include <mutex>

#include "dare_internal.h"
#include "tc_ptx.cuh"

namespace dare {

namespace {
constexpr int kThreads = 1024, kVecs = 4;
constexpr int kTile = kThreads * kVecs * 4;     // 16384 scores per CTA: four 16-byte vectors per thread
constexpr int kTileWords = kTile / 32;          // 512 words of decision bits per tile

// LPR lanes to a row (hd = 4 * LPR * VPL), so that every lane of a warp has work, and U rows of each lane group in
// flight at once: the kernel is a stream of both query arrays, bound by how many bytes an SM keeps on their way (one row
// a warp: 5.3 TB/s at 2^20 rows of 128).
template <int LPR, int VPL, int U>
__global__ void __launch_bounds__(256) drift_score_kernel(const float* __restrict__ a, const float* __restrict__ b,
                                                          long long rows, float* __restrict__ scores) {
  constexpr int RPW = 32 / LPR * U, HD = 4 * LPR * VPL;      // rows a warp takes at once
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();
  const int lane = threadIdx.x & 31, sub = lane & (LPR - 1), grp = lane / LPR;
  const long long warp0 = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long r0 = warp0 * RPW; r0 < rows; r0 += nwarps * RPW) {
    float4 x[U][VPL], y[U][VPL];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long r = r0 + u * (32 / LPR) + grp, rc = r < rows ? r : rows - 1;
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        x[u][v] = __ldcs(reinterpret_cast<const float4*>(a + rc * HD) + v * LPR + sub);
        y[u][v] = __ldcs(reinterpret_cast<const float4*>(b + rc * HD) + v * LPR + sub);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float dot = 0.f, n1 = 0.f, n2 = 0.f;
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        const float4 p = x[u][v], q = y[u][v];
        dot += p.x * q.x + p.y * q.y + p.z * q.z + p.w * q.w;
        n1 += p.x * p.x + p.y * p.y + p.z * p.z + p.w * p.w;
        n2 += q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
      }
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) {
        dot += __shfl_xor_sync(0xffffffffu, dot, o);
        n1 += __shfl_xor_sync(0xffffffffu, n1, o);
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      }
      const long long r = r0 + u * (32 / LPR) + grp;
      if (sub == 0 && r < rows) {
        const float den = sqrtf(n1) * sqrtf(n2);
        scores[r] = 1.f - (den > 0.f ? dot / den : 0.f);
      }
    }
  }
}
// any other row length
__global__ void __launch_bounds__(256) drift_score_any_kernel(const float* __restrict__ a, const float* __restrict__ b,
                                                              long long rows, int hd, float* __restrict__ scores) {
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const long long warp0 = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long r = warp0; r < rows; r += nwarps) {
    const float4* pa = reinterpret_cast<const float4*>(a + r * hd);
    const float4* pb = reinterpret_cast<const float4*>(b + r * hd);
    float dot = 0.f, n1 = 0.f, n2 = 0.f;
    for (int v = lane; v < hd / 4; v += 32) {
      const float4 x = pa[v], y = pb[v];
      dot += x.x * y.x + x.y * y.y + x.z * y.z + x.w * y.w;
      n1 += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
      n2 += y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      dot += __shfl_xor_sync(0xffffffffu, dot, o);
      n1 += __shfl_xor_sync(0xffffffffu, n1, o);
      n2 += __shfl_xor_sync(0xffffffffu, n2, o);
    }
    if (lane == 0) {
      const float den = sqrtf(n1) * sqrtf(n2);
      scores[r] = 1.f - (den > 0.f ? dot / den : 0.f);
    }
  }
}

// refreshed <=> !(s <= tau): a NaN score refreshes.
// Thread t of a tile owns the four 16-byte vectors k = 0..3 at scores[base + (k * 1024 + t) * 4 ...]: every load
// instruction of a warp covers 512 contiguous bytes, and all four are in flight before the first is used.  Returns
// its 16 decisions, bit 4k + j <-> element j of vector k.
__device__ __forceinline__ unsigned tile_flags(const float* __restrict__ scores, long long n, long long base, float tau) {
  float4 v[kVecs];
  bool full[kVecs];
#pragma unroll
  for (int k = 0; k < kVecs; ++k) {
    const long long i0 = base + ((long long)k * kThreads + threadIdx.x) * 4;
    full[k] = i0 + 3 < n;
    v[k] = make_float4(0.f, 0.f, 0.f, 0.f);                 // 0 <= tau or not, a missing element is masked out below
    if (full[k]) {
      v[k] = __ldcs(reinterpret_cast<const float4*>(scores + i0));
    } else {
      if (i0 < n) v[k].x = scores[i0];
      if (i0 + 1 < n) v[k].y = scores[i0 + 1];
      if (i0 + 2 < n) v[k].z = scores[i0 + 2];
    }
  }
  unsigned bits = 0;
#pragma unroll
  for (int k = 0; k < kVecs; ++k) {
    const long long i0 = base + ((long long)k * kThreads + threadIdx.x) * 4;
    unsigned b = (!(v[k].x <= tau) ? 1u : 0u) | (!(v[k].y <= tau) ? 2u : 0u) | (!(v[k].z <= tau) ? 4u : 0u) |
                 (!(v[k].w <= tau) ? 8u : 0u);
    if (!full[k]) {
      const long long left = n - i0;                        // elements of this vector that exist: <= 3, maybe <= 0
      b &= left <= 0 ? 0u : ((1u << (int)left) - 1u);
    }
    bits |= b << (4 * k);
  }
  return bits;
}

// exclusive prefix of `v` over the threads of the CTA (whole warps, at most 32 of them); *total = sum
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* warp_sums, T* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const T w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : T(0);
    T winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T n = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += n;
    }
    warp_sums[lane] = winc - w;
    if (lane == 31) *total = winc;
  }
  __syncthreads();
  return warp_sums[warp] + inc - v;
}

// pass 1: the only pass that reads the scores.  Leaves the decisions as a plain bit array (bit i of the array <->
// score i) and the tile's count.  For one vector index k the 32 lanes of a warp hold the decisions on 128 consecutive
// scores, four bits each: eight lanes' nibbles make one 32-bit word of the array, put together with three shuffles.
__global__ void __launch_bounds__(kThreads) tile_flag_kernel(const float* __restrict__ scores, long long n, float tau,
                                                             int* __restrict__ tile_counts,
                                                             unsigned* __restrict__ flags) {
  __shared__ int total;
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();            // the scan's CTA may take its place now; it waits for this grid to complete
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  const unsigned bits = tile_flags(scores, n, (long long)blockIdx.x * kTile, tau);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned* tile_words = flags + (size_t)blockIdx.x * kTileWords;
#pragma unroll
  for (int k = 0; k < kVecs; ++k) {
    unsigned v = ((bits >> (4 * k)) & 0xfu) << (4 * (lane & 7));
    v |= __shfl_xor_sync(0xffffffffu, v, 1);
    v |= __shfl_xor_sync(0xffffffffu, v, 2);
    v |= __shfl_xor_sync(0xffffffffu, v, 4);
    // scores [(k * 1024 + 32 * warp + 8 * w) * 4, + 32) of the tile, w = lane / 8
    if ((lane & 7) == 0) tile_words[k * (kThreads / 8) + warp * 4 + (lane >> 3)] = v;
  }
  const int c = __reduce_add_sync(0xffffffffu, __popc(bits));
  if (lane == 0) atomicAdd(&total, c);
  __syncthreads();
  if (threadIdx.x == 0) tile_counts[blockIdx.x] = total;
}

// pass 2: exclusive scan of the tile counts, one CTA
__global__ void __launch_bounds__(kThreads) tile_scan_kernel(const int* __restrict__ tile_counts, int n_tiles,
                                                             int* __restrict__ tile_offsets, int* __restrict__ count) {
  __shared__ int warp_sums[32];
  __shared__ int total;
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();
  int base = 0;
  for (int start = 0; start < n_tiles; start += kThreads) {
    const int i = start + threadIdx.x;
    const int v = i < n_tiles ? tile_counts[i] : 0;
    const int ex = block_exclusive_scan<int>(v, warp_sums, &total);
    if (i < n_tiles) tile_offsets[i] = base + ex;
    base += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) *count = base;
}

// pass 3: from the decision bits alone (4 bytes per thread instead of 128 bytes of scores).  One thread per word of
// 32 consecutive scores, 512 threads per tile: one scan of the words' popcounts places every thread, which then
// writes the indices of its set bits, ascending, at consecutive places.  Every lane of such a store lands in another
// sector (ncu: 10.7 sectors per request), yet the pass is bound by the chain load -> scan -> stores of its CTAs
// rather than by the stores: two other forms measured slower on the same 2^24 scores (22.7 us per call for this one):
// lane-consecutive stores, each list entry found by a binary search over the words' first places in shared memory
// (27.5 us), and 256-thread CTAs with two words per thread so that every tile is resident at once (25.5 us).
// No store goes past entry n - 1 of the list, whatever the offsets say: if another call raced on a shared scratch
// array, the list is wrong but the caller's buffer is the only memory written.
__global__ void __launch_bounds__(kTileWords) tile_scatter_kernel(const unsigned* __restrict__ flags,
                                                                  const int* __restrict__ tile_offsets,
                                                                  int* __restrict__ idx, long long n) {
  __shared__ int warp_sums[32];
  __shared__ int total;
  ptx::pdl_wait();                         // before any read: decisions (two kernels back) and offsets (one back)
  unsigned word = flags[(size_t)blockIdx.x * kTileWords + threadIdx.x];
  long long out = tile_offsets[blockIdx.x];
  out += block_exclusive_scan<int>(__popc(word), warp_sums, &total);
  const int i0 = (int)((long long)blockIdx.x * kTile) + (int)threadIdx.x * 32;
  while (word != 0u) {
    if (out >= 0 && out < n) idx[out] = i0 + __ffs((int)word) - 1;
    ++out;
    word &= word - 1u;
  }
}

// ---- the k-th smallest of many scores, by ONE cluster of CTAs: exact selection by narrowing a range of order-preserving
// keys, 2048 bins at a time.  Every CTA counts its share of the scores that lie in the range into a histogram in its own
// shared memory; the CTAs then send one another slices of the bins (bulk copies), add up their own, tell one another the
// slices' totals, and all of them pick the bin that holds rank k: the next range.  All keys are three such passes.  A
// shared-memory atomic takes a cycle a lane whatever it meets, so the first pass costs a cycle a score of the CTA's share
// (copies of the histogram changed nothing): with many scores the range starts as a bracket around rank k from a sample of
// 256 of them, which most scores lie outside; a bracket that turns out not to hold the rank is given up for all keys.
// Where the bracket's keys fit (kth_list_keys), they are kept in shared memory as they are found, and the narrowing passes read
// them, not the scores again: a call of 2^19 to 2^21 scores 1-10 % shorter; a kernel of its own, for the code cost 20000 scores 0.6 us.
// A cluster (rather than a grid) because the call has no scratch memory to meet in: nothing is shared between calls,
// whatever streams they run on.
// A CTA that waits in vain for the others' bins records the time-out in the status word (if the caller has one), gives the
// copies still on their way to it as long again, and says so in place of its total: all CTAs then leave together, and the
// threshold is NaN, which Eq. 2 reads as "refresh everything".
constexpr int kKthBins = 2048, kKthMaxCtas = 16, kKthSample = 256;
constexpr int kKthBracket = 1 << 19;        // the sample costs about 4 us: from this many scores on
constexpr int kKthList = 48 * 1024;         // keys of the bracket that a CTA keeps in shared memory, at most (one CTA an SM)
constexpr unsigned kKeyMinusInf = 0x007fffffu, kKeyPlusInf = 0xff800000u;

// The bracket around rank k: the sample's keys four standard deviations of its rank either side.
__host__ __device__ __forceinline__ void kth_bracket(int n, int k, int* lo, int* hi) {
  const float p = (float)k / (float)n;
  const int c = (int)(p * kKthSample), w = (int)(4.f * sqrtf(p * (1.f - p) * kKthSample)) + 2;
  *lo = c - w; *hi = c + w;
}
// Keys that a CTA keeps of it: its share of the scores between those two keys (27 % at the median, 18 % for k = 0.87 n, 14 % for
// 0.93 n) and four standard deviations of that share, as far as they fit; none where not even two would, from 2.4, 3.4 and 4.1
// million scores on (collected and then of no use, they made calls of 4 to 16 million 50-65 % longer).
int kth_list_keys(int n, int k, int ctas) {
  int lo, hi;
  kth_bracket(n, k, &lo, &hi);
  const float share = (float)(std::min(hi + 1, kKthSample) - std::max(lo, 0)) / (float)kKthSample;
  const float sd = sqrtf(share * (1.f - share) / (float)kKthSample), scores = (float)n / (float)ctas;
  return (share + 2.f * sd) * scores <= (float)kKthList ? std::min(kKthList, (int)((share + 4.f * sd) * scores)) : 0;
}

constexpr int kKthLost = -2;                // s_bin: some CTA's bins never came
constexpr unsigned long long kKthLoseWaitNs = 1000000ull;

// What follows a first poll in vain.  Out of line: the kernel is a short chain, and instructions it does not run cost it
// fetches (drift scores, quantile and compaction of 20000 scores: 22.4 us with both waits inline, 22.05 so).
__device__ __noinline__ bool kth_wait(uint64_t* bar, uint32_t phase, int* status, int lose_one) {
  const unsigned long long limit = lose_one ? kKthLoseWaitNs : ptx::kWaitLimitNs;
  if (ptx::mbar_wait(bar, phase, status, limit)) return true;
  ptx::mbar_wait(bar, phase, nullptr, limit);         // (nobody leaves before what is on its way has landed)
  return false;
}
// lose_one (diagnostics): CTA 0 keeps its bins from CTA 1, whose wait for them then runs out, after a millisecond.
template <bool kBracket>       // n >= kKthBracket
__global__ void __launch_bounds__(kThreads) kth_cluster_kernel(const float* __restrict__ scores, int n, int k,
                                                               float* __restrict__ tau_out, int* status, int lose_one) {
  __shared__ __align__(16) int hist[kKthBins];
  __shared__ __align__(16) int recv[kKthBins];        // [sender][bin of this CTA's slice]
  __shared__ uint64_t recv_bar;
  __shared__ __align__(16) int red[kKthBins / 8];     // this CTA's slice of the bins over the whole cluster
  __shared__ __align__(16) unsigned sample[kKthSample];
  __shared__ int part[kKthBins / 8 / 32], totals[kKthMaxCtas], below[kKthMaxCtas], s_below, s_bin, s_rank;
  __shared__ unsigned s_lo, s_hi;
  __shared__ int s_list, s_under;
  extern __shared__ unsigned list[];                  // (bracket only, and only where the launch gave it room)
  int list_keys = kBracket ? (int)(ptx::dynamic_smem_bytes() / 4u) : 0;
  const int ctas = (int)gridDim.x, rank_cta = (int)ptx::cluster_ctarank(), lane = threadIdx.x & 31, tid = (int)threadIdx.x;
  const int slice = kKthBins / ctas;                  // 128 or 256: whole warps, four or eight bins to a lane
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();
  // 16-byte loads from the first aligned score on; the few before and after them are CTA 0's
  const int head = min(n, (int)((16u - (unsigned)(reinterpret_cast<uintptr_t>(scores) & 15u)) & 15u) / 4);
  const float4* body = reinterpret_cast<const float4*>(scores + head);
  const int n4 = (n - head) / 4, tail0 = head + 4 * n4;
  auto scan = [&](int v) {                            // inclusive, over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    return v;
  };
  // ---- the bracket, the same in every CTA
  if (kBracket && tid < kKthSample) sample[tid] = score_key(scores[(int)(((long long)tid * n) / kKthSample)]);
  if (tid == 0) {
    s_lo = kKeyMinusInf; s_hi = kKeyPlusInf;
    s_list = 0; s_under = 0;
    ptx::mbar_init(&recv_bar, 1);
    ptx::fence_mbar_init();
  }
  __syncthreads();
  if (kBracket) {
    int at_lo, at_hi;
    kth_bracket(n, k, &at_lo, &at_hi);
    const int me = tid >> 2;                          // four threads to a sample key
    const unsigned mine = sample[me];
    int r = 0;
    for (int i = (tid & 3) * 4; i < kKthSample; i += 16) {
      const uint4 v = *reinterpret_cast<const uint4*>(sample + i);
      r += (v.x < mine || (v.x == mine && i < me)) + (v.y < mine || (v.y == mine && i + 1 < me)) +
           (v.z < mine || (v.z == mine && i + 2 < me)) + (v.w < mine || (v.w == mine && i + 3 < me));
    }
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    if ((tid & 3) == 0) {
      if (r == at_lo && mine != kKeyNaN) s_lo = mine;
      if (r == at_hi && mine != kKeyNaN) s_hi = mine;
    }
  }
  __syncthreads();
  unsigned lo = s_lo, hi = s_hi;                      // keys in [lo, hi]
  int rank = k;                                       // of the wanted key: among all of them, then among those in the range
  bool found = false, numbers = true, lost = false;   // numbers: rank k falls among the scores that are numbers
  auto raw_key = [](float f) {                        // score_key of a number; NaN goes below -inf or above +inf
    const unsigned u = __float_as_uint(f);
    return u ^ ((unsigned)((int)u >> 31) | 0x80000000u);
  };
  // width of a bin of [lo, hi], as a shift
  auto shift_now = [&]() { return hi - lo < (unsigned)kKthBins ? 0 : 21 - __clz((int)(hi - lo)); };
  auto lower = [&](unsigned key) { return key - kKeyMinusInf < lo - kKeyMinusInf ? 1 : 0; };
  auto walk = [&](auto count) {
    constexpr int U = 8;                            // vectors a thread has in flight
    const int step = ctas * kThreads;
    int i = rank_cta * kThreads + tid;
    for (; i + (U - 1) * step < n4; i += U * step) {
      float4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = body[i + u * step];
#pragma unroll
      for (int u = 0; u < U; ++u) { count(v[u].x); count(v[u].y); count(v[u].z); count(v[u].w); }
    }
    for (; i < n4; i += step) {
      const float4 v = body[i];
      count(v.x); count(v.y); count(v.z); count(v.w);
    }
    if (rank_cta == 0) {
      if (tid < head) count(scores[tid]);
      if (tid < n - tail0) count(scores[tail0 + tid]);
    }
  };
  // ---- the first pass over a bracket: what lies below it, and its keys, kept for all passes that follow (a CTA whose keys turn out to
  // be more than it has room for reads the scores for them, whatever the others do), or the first pass's bins
  bool listed = false, binned = false;                // binned: the bins of [lo, hi] are there
  if (kBracket) {
    const unsigned range = hi - lo;
    const int shift = shift_now();
    int under = 0;
    for (int b = tid; b < kKthBins; b += kThreads) hist[b] = 0;
    // No keys kept where one pass is all (a bracket of one tied score, say), or where the sample says that they will not fit (a
    // tie with one of the bracket's ends)
    const int in_sample = __syncthreads_count(tid < kKthSample && sample[tid & (kKthSample - 1)] - lo <= range);
    if (shift == 0 || (float)in_sample * (float)n > (float)list_keys * (float)(kKthSample * ctas)) list_keys = 0;
    auto bin = [&](float f) {
      const unsigned key = raw_key(f);
      under += lower(key);
      if (key - lo <= range) atomicAdd(&hist[(key - lo) >> shift], 1);
    };
    auto keep = [&](float f) {
      const unsigned key = raw_key(f);
      under += lower(key);
      if (key - lo > range) return;
      const int at = atomicAdd(&s_list, 1);
      if (at < list_keys) list[at] = key;
    };
    if (list_keys > 0) {
      constexpr int U = 4;                            // vectors a thread has in flight; a warp's share of the list in one piece
      const int step = ctas * kThreads;
      for (int base = rank_cta * kThreads + (tid & ~31); base < n4; base += U * step) {
        unsigned key[U][4];
        int mine = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = base + lane + u * step;
          const float4 v = i < n4 ? body[i] : make_float4(0.f, 0.f, 0.f, 0.f);
          key[u][0] = raw_key(v.x); key[u][1] = raw_key(v.y); key[u][2] = raw_key(v.z); key[u][3] = raw_key(v.w);
          if (i >= n4) key[u][0] = key[u][1] = key[u][2] = key[u][3] = kKeyNaN;      // (neither inside nor below)
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            under += lower(key[u][e]);
            mine += key[u][e] - lo <= range ? 1 : 0;
          }
        const int inc = scan(mine);
        int at = 0;
        if (lane == 31) at = atomicAdd(&s_list, inc);
        at = __shfl_sync(0xffffffffu, at, 31) + inc - mine;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (key[u][e] - lo <= range) {
              if (at < list_keys) list[at] = key[u][e];
              ++at;
            }
      }
      if (rank_cta == 0) {
        if (tid < head) keep(scores[tid]);
        if (tid < n - tail0) keep(scores[tail0 + tid]);
      }
    } else {
      walk(bin);
      binned = true;
    }
    under = __reduce_add_sync(0xffffffffu, under);
    if (lane == 0 && under != 0) atomicAdd(&s_under, under);
    __syncthreads();
    listed = list_keys > 0 && s_list <= list_keys;
  }
  ptx::cluster_sync_all();                            // every CTA's barrier is set up
  uint32_t phase = 0;
  for (bool first = true, whole = lo == kKeyMinusInf && hi == kKeyPlusInf; !found && numbers && !lost; ) {
    const int shift = shift_now();
    if (!binned)
      for (int b = tid; b < kKthBins; b += kThreads) hist[b] = 0;
    if (tid == 0) { s_bin = -1; s_below = kBracket && first && !whole ? s_under : 0; }
    __syncthreads();
    if (!binned) {
      const unsigned range = hi - lo;
      auto bin_of = [&](unsigned key) {
        const unsigned d = key - lo;
        if (d <= range) atomicAdd(&hist[d >> shift], 1);
      };
      if (kBracket && listed)
        for (int i = tid; i < s_list; i += kThreads) bin_of(list[i]);
      else
        walk([&](float f) { bin_of(raw_key(f)); });
    }
    binned = false;
    if (tid == 0) ptx::mbar_arrive_expect_tx(&recv_bar, (uint32_t)kKthBins * 4u);
    ptx::fence_proxy_async_smem();
    __syncthreads();
    if (tid < ctas && !(lose_one && rank_cta == 0 && tid == 1))       // slice `tid` of this CTA's bins goes to CTA `tid`
      ptx::bulk_copy_to_cta(ptx::map_to_cta(ptx::smem_u32(recv + rank_cta * slice), (uint32_t)tid),
                            ptx::smem_u32(hist + tid * slice), (uint32_t)slice * 4u,
                            ptx::map_to_cta(ptx::smem_u32(&recv_bar), (uint32_t)tid));
    const bool came = ptx::mbar_try_wait(&recv_bar, phase) || kth_wait(&recv_bar, phase, status, lose_one);
    phase ^= 1;
    if (tid < slice) {
      int mine = 0;
#pragma unroll
      for (int j = 0; j < kKthMaxCtas; ++j) mine += j < ctas ? recv[j * slice + tid] : 0;
      red[tid] = mine;
      mine = __reduce_add_sync(0xffffffffu, mine);
      if (lane == 0) part[tid >> 5] = mine;
    }
    const bool all_came = __syncthreads_and(came) != 0;
    if (tid < ctas) {                                 // the slice's total goes to every CTA, and what lies below the range
      int tot = all_came ? 0 : -1;
      for (int w = 0; all_came && w < slice / 32; ++w) tot += part[w];
      ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&totals[rank_cta]), (uint32_t)tid), (uint32_t)tot);
      ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&below[rank_cta]), (uint32_t)tid), (uint32_t)s_below);
    }
    ptx::cluster_sync_all();
    if (tid < 32) {
      int want = rank;
      if (first) want -= __reduce_add_sync(0xffffffffu, lane < ctas ? below[lane] : 0);
      const int st = lane < ctas ? totals[lane] : 0, inc = scan(st);
      const unsigned hit = __ballot_sync(0xffffffffu, inc - st < want && want <= inc);
      if (__any_sync(0xffffffffu, st < 0)) {
        if (lane == 0) s_bin = kKthLost;
      } else if (hit != 0u) {
        const int sl = __ffs((int)hit) - 1, per = slice / 32;
        const int before = __shfl_sync(0xffffffffu, inc - st, sl);
        int c[8], tot = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          c[j] = j < per ? (int)ptx::ld_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&red[lane * per + j]), (uint32_t)sl)) : 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) tot += c[j];
        int cum = before + scan(tot) - tot;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (cum < want && want <= cum + c[j]) { s_bin = sl * slice + lane * per + j; s_rank = want - cum; }
          cum += c[j];
        }
      }
    }
    __syncthreads();
    const int bin = s_bin;                            // (the same in every CTA)
    if (bin >= 0) {
      lo += (unsigned)bin << shift;
      hi = min(hi, lo + ((1u << shift) - 1u));
      rank = s_rank;
      found = shift == 0;
      first = false;
    } else if (bin == kKthLost) {
      lost = true;
    } else if (first && !whole) {                     // the bracket does not hold the rank: all keys
      lo = kKeyMinusInf; hi = kKeyPlusInf; whole = true; listed = false;
    } else {
      numbers = false;
    }
    __syncthreads();
  }
  if (rank_cta == 0 && tid == 0) *tau_out = lost ? __int_as_float(0x7fc00000) : (numbers ? key_score(lo) : __int_as_float(0x7f800000));
  ptx::cluster_sync_all();                            // nobody leaves while its bins are being read
}
// ---- compaction of up to kClusterSelect scores by one cluster in one launch: every CTA decides on a contiguous share
// (kept as bits in registers), tells the others its count over distributed shared memory, and writes its part of the list
// behind the ones before it.  Below that size three launches take longer than their work (2^16 scores: 13 -> 6 us).
constexpr int kClusterIters = 8;                      // 16-byte vectors a thread decides on
constexpr int kClusterSelect = 8 * kClusterIters * kThreads * 4;       // scores that eight CTAs (the portable size) can take

__global__ void __launch_bounds__(kThreads) select_cluster_kernel(const float* __restrict__ scores, int n, float tau,
                                                                  int* __restrict__ idx, int* __restrict__ count_out) {
  __shared__ int warp_sums[32], total, totals[kKthMaxCtas];
  const int ctas = (int)gridDim.x, rank = (int)ptx::cluster_ctarank(), tid = (int)threadIdx.x;
  ptx::cluster_arrive_relaxed();                      // "this CTA runs": the others may store into its shared memory
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();
  const int iters = (n + ctas * kThreads * 4 - 1) / (ctas * kThreads * 4);   // <= kClusterIters
  const int base = rank * iters * kThreads * 4;
  unsigned bits = 0u;
#pragma unroll
  for (int it = 0; it < kClusterIters; ++it) {
    const int i0 = base + (it * kThreads + tid) * 4;
    if (it >= iters || i0 >= n) continue;
    if (i0 + 3 < n) {
      const float4 v = *reinterpret_cast<const float4*>(scores + i0);
      bits |= ((!(v.x <= tau) ? 1u : 0u) | (!(v.y <= tau) ? 2u : 0u) | (!(v.z <= tau) ? 4u : 0u) | (!(v.w <= tau) ? 8u : 0u)) << (4 * it);
    } else {
      for (int e = 0; i0 + e < n; ++e) bits |= (!(scores[i0 + e] <= tau) ? 1u : 0u) << (4 * it + e);
    }
  }
  const int mine = __reduce_add_sync(0xffffffffu, __popc(bits));
  if (tid == 0) total = 0;
  __syncthreads();
  if ((tid & 31) == 0 && mine != 0) atomicAdd(&total, mine);
  __syncthreads();
  ptx::cluster_wait();                                // every CTA of the cluster has started
  if (tid < ctas) ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&totals[rank]), (uint32_t)tid), (uint32_t)total);
  ptx::cluster_sync_all();
  int out = 0, all = 0;
  for (int c = 0; c < ctas; ++c) { out += c < rank ? totals[c] : 0; all += totals[c]; }
  if (rank == 0 && tid == 0) *count_out = all;
  for (int it = 0; it < iters; ++it) {
    const unsigned b = (bits >> (4 * it)) & 15u;
    int at = out + block_exclusive_scan<int>(__popc(b), warp_sums, &total);
    const int i0 = base + (it * kThreads + tid) * 4;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (b & (1u << e)) idx[at++] = i0 + e;
    out += total;
    __syncthreads();
  }
}
__global__ void set_float_kernel(float* dst, float value) { *dst = value; }
}  // namespace

// One cluster of 16 CTAs where the device takes one of that size (asked once per device and kernel), of the portable 8
// otherwise.
// smem(number of CTAs): dynamic shared memory of a CTA, at most max_smem.
template <bool kTag, typename Smem, typename... KArgs, typename... Args>
static cudaError_t launch_cluster(void (*kernel)(KArgs...), int max_smem, Smem smem, cudaStream_t st, Args... args) {
  static std::atomic<unsigned long long> asked{0}, wide{0};      // (per kernel: signature and tag tell them apart)
  int dev = 0;
  if (cudaError_t e = cudaGetDevice(&dev); e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  if (!(asked.load(std::memory_order_acquire) & bit)) {
    int clusters = 0;
    cfg.gridDim = dim3(kKthMaxCtas);
    attr[0].val.clusterDim.x = kKthMaxCtas;
    cfg.numAttrs = 1;
    cfg.dynamicSmemBytes = max_smem;
    if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem); e != cudaSuccess) return e;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0)
      wide.fetch_or(bit);
    else
      cudaGetLastError();
    asked.fetch_or(bit, std::memory_order_release);
  }
  const unsigned ctas = (wide.load() & bit) ? kKthMaxCtas : 8u;
  cfg.gridDim = dim3(ctas);
  attr[0].val.clusterDim.x = ctas;
  cfg.numAttrs = 2;
  cfg.dynamicSmemBytes = smem((int)ctas);
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

cudaError_t launch_kth_score_large(const float* scores, int n, int k, float* tau_out, cudaStream_t st, int* status,
                                   bool lose_one) {
  if (k <= 0 || k >= n) {
    set_float_kernel<<<1, 1, 0, st>>>(tau_out, k <= 0 ? -INFINITY : INFINITY);
    return cudaGetLastError();
  }
  if (n >= kKthBracket)
    return launch_cluster<true>(kth_cluster_kernel<true>, kKthList * 4, [&](int ctas) { return kth_list_keys(n, k, ctas) * 4; }, st,
                                scores, n, k, tau_out, status, lose_one ? 1 : 0);
  return launch_cluster<false>(kth_cluster_kernel<false>, 0, [](int) { return 0; }, st, scores, n, k, tau_out, status,
                               lose_one ? 1 : 0);
}

int select_large_tiles(long long n) { return (int)((n + kTile - 1) / kTile); }
size_t select_large_flag_bytes(long long n) { return (size_t)select_large_tiles(n) * kTileWords * sizeof(unsigned); }

cudaError_t launch_drift_scores(const float* a, const float* b, long long rows, int hd, float* scores,
                                cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  auto blocks = [&](int rows_per_warp, int per_sm) {
    const long long n = (rows + 8 * rows_per_warp - 1) / (8 * rows_per_warp);
    return (int)(n < kSms * per_sm ? n : kSms * per_sm);
  };
  auto launch = [&](auto kernel, int grid, auto... args) { return launch_pdl(kernel, dim3(grid), dim3(256), 0, st, 1, args...); };
  if (hd == 32) return launch(drift_score_kernel<8, 1, 4>, blocks(16, 8), a, b, rows, scores);
  if (hd == 64) return launch(drift_score_kernel<16, 1, 4>, blocks(8, 8), a, b, rows, scores);
  if (hd == 128) return launch(drift_score_kernel<32, 1, 4>, blocks(4, 8), a, b, rows, scores);
  if (hd == 256) return launch(drift_score_kernel<32, 2, 2>, blocks(2, 8), a, b, rows, scores);
  return launch(drift_score_any_kernel, blocks(1, 16), a, b, rows, hd, scores);
}

// tile_counts and tile_offsets: device arrays of select_large_tiles(n) ints each; flags: 512 32-bit words per tile
cudaError_t launch_select_large(const float* scores, long long n, float tau, int* idx, int* count, int* tile_counts,
                                int* tile_offsets, unsigned* flags, cudaStream_t st) {
  const int tiles = select_large_tiles(n);
  if (tiles == 0) return cudaMemsetAsync(count, 0, sizeof(int), st);
  if (n <= kClusterSelect) return launch_cluster<false>(select_cluster_kernel, 0, [](int) { return 0; }, st, scores, (int)n, tau, idx, count);
  cudaError_t e = launch_pdl(tile_flag_kernel, dim3(tiles), dim3(kThreads), 0, st, 1, scores, n, tau, tile_counts, flags);
  if (e != cudaSuccess) return e;
  e = launch_pdl(tile_scan_kernel, dim3(1), dim3(kThreads), 0, st, 1, (const int*)tile_counts, tiles,
                             tile_offsets, count);
  if (e != cudaSuccess) return e;
  e = launch_pdl(tile_scatter_kernel, dim3(tiles), dim3(kTileWords), 0, st, 1, (const unsigned*)flags,
                 (const int*)tile_offsets, idx, n);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dare

// ------------------------------------------------------------------------------------------------------------------
// Compaction without any caller-provided or allocated scratch.
//
// Some hosts of this library hand all of the device's memory to one arena at start-up and forbid every later
// cudaMalloc (an inference server with a fixed memory plan), or sit in a latency-critical loop where the device-wide
// synchronisation an allocation implies is not acceptable.  For them the per-tile counts and offsets and the decision
// bits of the three-pass compaction live in arrays that are part of the library image: 2 x 1024 ints + 1024 x 512
// 32-bit words = 2 MB + 8 KB of device memory on every GPU that loads the library, held until the process exits.
// That bounds the call at 1024 tiles = 16,777,216 scores.
//
// In host code the name `g_select_scratch` is only a stand-in for the symbol; the address a kernel may use comes from
// cudaGetSymbolAddress, asked once per device with that device current (the first call on a device does this; make
// that first call outside any stream capture).  All calls on a device share the array: it still holds the previous
// call's tile counts when the next one starts (every entry a call reads is written by that call first, so nothing
// needs clearing), and two calls that overlap on the GPU (different streams) race on it.
namespace dare {
namespace {
constexpr int kStaticTiles = 1024;
// [0, 2 * tiles) ints: counts, offsets; behind them the decision words
static __device__ __align__(256) int g_select_scratch[2 * kStaticTiles + kStaticTiles * kTileWords];
constexpr int kMaxDevices = 64;
int* g_select_scratch_addr[kMaxDevices] = {};
std::mutex g_select_scratch_mutex;

cudaError_t static_scratch_for_current_device(int** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_select_scratch_mutex);
  if (g_select_scratch_addr[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_select_scratch);
    if (e != cudaSuccess) return e;
    g_select_scratch_addr[dev] = static_cast<int*>(p);
  }
  *out = g_select_scratch_addr[dev];
  return cudaSuccess;
}
}  // namespace
}  // namespace dare

extern "C" int64_t dare_select_compact_static_max_tokens(void) { return (int64_t)dare::kStaticTiles * dare::kTile; }

extern "C" dare_status_t dare_select_compact_static(const float* scores, int64_t n_tokens, float threshold, int32_t* idx,
                                                    int32_t* count, void* cuda_stream) {
  if (!scores || !idx || !count) return DARE_ERR_INVALID_ARG;
  if (isnan(threshold)) return DARE_ERR_INVALID_ARG;
  if (n_tokens < 0 || n_tokens > dare_select_compact_static_max_tokens()) return DARE_ERR_SHAPE;   // beyond the array
  if ((reinterpret_cast<uintptr_t>(scores) & 15u) != 0) return DARE_ERR_ALIGN;
  int* scratch = nullptr;
  if (dare::static_scratch_for_current_device(&scratch) != cudaSuccess) { cudaGetLastError(); return DARE_ERR_CUDA; }
  cudaError_t e = dare::launch_select_large(scores, n_tokens, threshold, idx, count, scratch,
                                            scratch + dare::kStaticTiles,
                                            reinterpret_cast<unsigned*>(scratch + 2 * dare::kStaticTiles),
                                            (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) { cudaGetLastError(); return DARE_ERR_CUDA; }
  return DARE_OK;
}
