// Declarations of the tensor-core path (tcgen05 GEMM and attention kernels) shared between its translation units.
#pragma once

#include <cuda.h>

#include "dare_internal.h"

namespace dare {

enum { EPI_Q = 0, EPI_KV = 1, EPI_OUT = 2, EPI_SWIGLU = 3, EPI_F32 = 4,
       EPI_OUT_RES = 5,     // EPI_OUT plus a residual row (chosen by the launcher when GemmParams::resid is set)
       EPI_SCORE = 6,       // the one column tile of the scoring head: scored and kept (as in EPI_Q), no query stored
       EPI_QKV = 7 };       // EPI_KV and a third matrix: the queries of the same rows (persistent kernel)

struct GemmParams {
  int K;                 // reduction length (multiple of 64)
  int m_tiles;           // row tiles of the launch (set by the launcher; a pair launch pads its grid to an even count)
  int m_total;           // dense: tokens of the step; gathered: capacity of the row list
  int seq_act;           // dense row mapping: rows per sequence ...
  int tiles_per_seq;     // ... and 128-row tiles per sequence
  int a_seq_stride;      // rows between sequences in A's row space
  int a_row0;            // first row of the window in A's row space
  int flat;              // dense row tiles run on across sequences (one "sequence" of all the step's tokens in the mapping
                         // above): positions and cache rows come from the tokens
  int a_piece;           // ... and A is addressed by cache row, in boxes of 32 rows (windows of a multiple of 32 rows)
  const int* idx;        // gathered: token of each A row (ascending refresh set), else nullptr
  const int* count;      // gathered: device count of rows, else nullptr
  const __nv_bfloat16* gather_src;  // gathered: the matrix [*, K] whose rows idx[] the kernel fetches itself as its A
                                    // operand (Alg. 1 line 6); nullptr: A comes through the tensor map
  int gather_cache_rows; // gather_src is addressed by cache row (the O cache) instead of by flat token index
  int unit_gate;         // persistent listed launches issued as a pair of kernels: the two-CTA form runs when the count
                         // gives it at least this many (column tile, row-tile pair) units, the one-CTA form otherwise;
                         // 0: no gate
  StepGeom g;
  int n_split;           // n-tiles [0, n_split) use W0/out0, the next n_split W1/out1 and (EPI_QKV) the last n_split
                         // W2/out2: rotated, stored by token
  __nv_bfloat16* out0;
  __nv_bfloat16* out1;
  int ld_out;
  int out_is_cache;      // output rows addressed by cache row (1), by flat token index (0), or by the row's place
                         // in the gathered list (2)
  const __nv_bfloat16* resid;  // EPI_OUT: rows added to the result (indexed like a token-addressed output), or nullptr
  int ld_resid;
  union {                // (no larger: every launch carries the struct, and 8 bytes more cost short steps 0.5 %)
    float* out_f32;        // EPI_F32: fp32 output instead of out0
    __nv_bfloat16* out2;   // EPI_QKV: see n_split
  };
  int b_pair;            // the W tile is BN/2 rows of W0 followed by BN/2 rows of W1, both at row nt*BN/2 (EPI_SWIGLU:
                         // gate and up projections of the same BN/2 outputs)
  const float2* rope;    // rotary table [max_seq][head_dim/2]
  float* q_prev;         // stored scoring-head query [cache rows][head_dim], fp32
  float* scores;
  int has_prev;
  int* status;
  unsigned long long* debug;   // 8 timestamp slots of this kernel or nullptr
  // A step whose refresh set is large runs its projections and attention in their dense forms (every operand through
  // TMA straight from the step's buffers, no compact copy, two-CTA MMAs) and only keeps the results of the rows that
  // were refreshed; only the device knows the set's size, so both forms of a launch are issued and each looks at the
  // count: a launch runs when gate_lo <= *gate_count < gate_hi and leaves at once otherwise (gate_count == nullptr:
  // always runs).  store_mask (the staleness counters, by cache row): a dense-form K/V projection stores a row only
  // where the counter is 0, i.e. where this step's selection refreshed the token (Eq. 3: every other row keeps its
  // cached K and V).
  const int* gate_count;
  int gate_lo, gate_hi;
  const int* store_mask;
  int loop_rows;         // gathered launch with ONE row of CTAs in the grid: each takes the refresh set's row tiles in turn
  int late_wait;         // 1: only the finishing pass needs what the predecessor writes (store_mask): the main loop runs
                         // beside it, its operands come from two or more kernels back
  int wait_at_end;       // 1: the launch reads nothing its predecessor in the stream writes and writes nothing that one
                         // reads, so it runs beside it: its CTAs start as soon as the predecessor's have passed their own
                         // dependency wait (everything further back is then complete), and wait for the predecessor
                         // only before they leave, which keeps completion transitive along the stream
};

#ifdef __CUDACC__
// Position and cache row of the rows of a tile that runs on across sequences (GemmParams::flat): row r of the tile is the
// step's token t0 + r.  One integer division per tile; per row a multiplication, exact because the quotient is small (a
// tile spans at most 128 sequences) and (i + 0.5) / seq_act stays 0.5 / seq_act away from an integer.
struct FlatRows {
  int b0, i0, seq_act, pos_begin, max_seq;
  float inv;
  __device__ __forceinline__ FlatRows(const StepGeom& g, int t0, bool used) {
    if (!used) return;
    b0 = t0 / g.seq_act;
    i0 = t0 - b0 * g.seq_act;
    seq_act = g.seq_act; pos_begin = g.pos_begin; max_seq = g.max_seq;
    inv = 1.f / (float)g.seq_act;
  }
  __device__ __forceinline__ void at(int r, int* pos, size_t* crow) const {
    const int i = i0 + r, b = (int)(((float)i + 0.5f) * inv);
    *pos = pos_begin + i - b * seq_act;
    *crow = (size_t)(b0 + b) * max_seq + *pos;
  }
};
#endif

struct AttnParams {
  const __nv_bfloat16* q;   // [T, d] rotated queries of the step (flat token rows)
  __nv_bfloat16* oc;        // attention-output cache
  const int* idx;           // refresh set (row-sparse) or nullptr (all rows)
  const int* batch_off;     // [batch+1] slice of idx per sequence (row-sparse only)
  StepGeom g;
  int* status;
  unsigned long long* debug;
  const int* gate_count;    // as in GemmParams: the launch runs when gate_lo <= *gate_count < gate_hi
  int gate_lo, gate_hi;
  const int* store_mask;    // dense form of a row-sparse step: a row's output is stored only where the staleness counter
                            // (by cache row) is 0 (Eq. 4: every other row keeps its cached output); tiles without such
                            // a row are skipped
  int wait_first;           // 1: the queries or the refresh set come from the kernel just before this one in the stream,
                            // so nothing of the step is read ahead of the dependency wait
  int dense_from;           // > 0 (two-tile kernel, row-sparse parameters above, gate_count set): one launch carries both
  const int* dense_mask;    // forms; with *gate_count >= dense_from its CTAs run the dense form with this store mask
};

// does a launch of this geometry take the kernel with two query tiles per CTA?
bool attention_tc_two_tiles(const StepGeom& g, bool row_sparse);

// K and V caches as attention operands: boxes of 64 columns x 128 or 64 rows (keys).
struct KvMaps { CUtensorMap k128, v128, k64, v64; };
cudaError_t launch_attention_tc(const KvMaps& maps, const AttnParams& p, cudaStream_t st);

// grid = (n_tiles of bn columns, m_tiles of 128 rows, splits of the reduction dimension = cluster size: 1, 2, or 4 with
// bn = 128);
// bn = 256 (least re-reading per flop) or 128 (more CTAs where few rows make the launch a stream of the weights).
// The W tensor maps must have a box of bn rows.
// Row-major bf16 matrix [rows, cols] as a TMA tensor map with a box of 64 columns x box_rows rows, 128-byte swizzle.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows);

// Two-CTA MMAs (pairs of row tiles share their W tile: a third less operand traffic from the L2 per CTA) pay where
// the main loop is bound by that traffic: launches of at most four row tiles, or of about one wave.  Launches of
// many waves measured slower with them (they are bound by the tensor pipe under the power cap, and the pair adds two
// cluster barriers and ties two SMs' pipelines together).
inline bool pairs_pay(int n_tiles, int m_tiles, int splits) {
  const int ctas = n_tiles * ((m_tiles + 1) / 2 * 2) * splits;
  return m_tiles >= 2 && (ctas <= 160 || m_tiles <= 4);
}

// The form of a dense projection that is one wave of CTAs: tile width, two-CTA MMAs or not, reduction splits.  What a CTA
// takes is its k-blocks times what one takes it (bound by the operand bytes an SM pulls from the L2: 48, 32, 32 and 24 KB
// for wide, wide pair, narrow and narrow pair tiles), the read-out of the accumulator with the exchange of partial tiles,
// and the finishing pass over its share of the tile (measured by the kernels' own stamps).  Few row tiles want narrow
// tiles and more splits (one row tile of 4096 x 4096: 32 CTAs of 32 k-blocks -> 128 of 16), more of them wide ones.
// Clusters of four CTAs do not cover all 148 SMs, and clusters of eight wait for eight free SMs of one GPC behind the
// kernel before (a 240-row pass of a 2048-wide stack took 29 % longer with them), so there are none.
// Q projection in us with an event on either side (the first about 10 us of each figure are those), narrow / narrow split in
// two / in four / narrow pairs / narrow pairs split in two / wide / wide split in two / wide pairs / wide pairs split in two, the
// pick in brackets, - where it does not fit one wave:
//   width 1024,  128 rows: 17.5 / 15.3 / [13.3] / - / - / 19.6 / 17.4 / - / -
//   width 2048,  512 rows: 22.6 / 17.2 / - / 20.7 / [17.1] / 26.6 / 20.4 / 24.6 / 19.5   (heads of 64; of 128: 17.7 and [17.0])
//   width 2048, 1024 rows: 23.3 / - / - / 21.5 / - / 26.8 / 20.6 / 25.6 / [20.8]
//   width 4096,  128 rows: 29.4 / 21.3 / [18.6] / - / - / 38.1 / 25.8 / - / -
//   width 4096,  256 rows: 30.8 / 22.6 / - / 28.7 / [20.8] / 37.8 / 26.6 / 34.0 / 24.7
//   width 4096,  512 rows: 31.6 / - / - / 29.0 / - / 38.9 / 27.5 / 34.9 / [26.7]
//   width 4096, 1024 rows: - / - / - / - / - / 39.6 / - / [37.6] / -
// At seventeen sizes (widths 512 to 4096, 128 to 1024 rows) the pick is the fastest or within 0.2 us of it, for Q and for the
// output projection.  (Forms past one wave: two waves of clusters cost 6-8 us more.)
// `beside`: CTAs of a launch that runs at the same time and should find SMs free; such a form is taken if it takes no
// longer than `limit_us`, that launch itself.  false: no form.
struct TileForm { int bn, pair, splits; };
inline bool pick_one_wave(int d_out, int m_tiles, int kblocks, TileForm* best, int beside = 0,
                          float limit_us = 1e29f) {
  const float sms = (float)(kSms - beside);
  float best_us = 1e30f;
  for (int pair = 0; pair < 2; ++pair)
    for (int bn = 128; bn <= 256; bn += 128)
      for (int s = 1; s <= (bn == 128 && !pair ? 4 : 2); s *= 2) {
        const int cluster = (pair + 1) * s, ctas = d_out / bn * (pair ? (m_tiles + 1) / 2 * 2 : m_tiles) * s;
        if (d_out % bn != 0 || (float)ctas > (cluster >= 4 ? 0.87f : 1.f) * sms || kblocks % s != 0 || kblocks / s < 2) continue;
        if (pair && m_tiles < 2) continue;
        const float main_loop = (float)(kblocks / s) * (bn == 256 ? (pair ? 0.33f : 0.36f) : (pair ? 0.25f : 0.31f));
        const float exchange = s == 1 ? 1.f : (bn == 256 ? 2.5f : (s == 2 ? 2.f : 2.2f));
        const float finish = 1.1f + 0.5f * (float)(4 / s * (bn / 128));
        const float us = main_loop + exchange + finish + (pair ? 0.3f : 0.f);
        if (us < best_us) { best_us = us; *best = TileForm{bn, pair, s}; }
      }
  return best_us < limit_us;
}

cudaError_t launch_gemm_tc(int epi, int bn, const CUtensorMap& a, const CUtensorMap& b0, const CUtensorMap& b1,
                           const GemmParams& p, int n_tiles, int m_tiles, int splits, cudaStream_t st, int pair = 0);


// SwiGLU of at most 256 rows (gemm_swiglu.cu): x maps the rows with 128-row boxes, gate / up the matrices with boxes of
// `width` rows (rows <= 128) or width / 2 (two-CTA form, beyond); width = swiglu_width(..., rows > 128).
int swiglu_width(int d_ff, int sms, bool pair);
cudaError_t launch_swiglu(const CUtensorMap& x, const CUtensorMap& gate, const CUtensorMap& up, int width, int rows, int d_ff,
                          int K, __nv_bfloat16* act, int* status, cudaStream_t st);

// Persistent form for launches of many row tiles (dense rows, 256-wide tiles, no reduction split, epilogues Q, K/V,
// OUT): one CTA per SM walks the tiles, finishing pass overlapped with the next tile's main loop.
// pair != 0: two-CTA MMAs over pairs of row tiles, b0 / b1 / b2 with 128-row boxes.
cudaError_t launch_gemm_persist(int epi, const CUtensorMap& a, const CUtensorMap& b0, const CUtensorMap& b1, const CUtensorMap& b2,
                                const GemmParams& p, int n_tiles, int m_tiles, cudaStream_t st, int pair = 0);
inline cudaError_t launch_gemm_persist(int epi, const CUtensorMap& a, const CUtensorMap& b0, const CUtensorMap& b1,
                                       const GemmParams& p, int n_tiles, int m_tiles, cudaStream_t st, int pair = 0) {
  return launch_gemm_persist(epi, a, b0, b1, b1, p, n_tiles, m_tiles, st, pair);
}
// ... pays as soon as the tiles are more than one wave: from there on a tile's set-up, pipeline fill and finishing pass
// hide behind the next tile's main loop.
inline bool persist_pays(int n_tiles, int m_tiles, int splits) { return splits == 1 && n_tiles * m_tiles > kSms; }
// A listed launch comes with a compact copy of its rows and a second form that only looks at the count: from two waves.
inline bool persist_pays_listed(int n_tiles, int m_tiles) { return n_tiles * m_tiles >= 2 * kSms; }
// Two-CTA MMAs in it, or single CTAs?  A k-block takes a pair 0.93 of the time it takes a single CTA (644 against 667-690
// cycles), but pairs walk in waves of 74 units of two row tiles, an odd row tile being padded to a pair.
inline bool persist_pairs_pay(int n_tiles, int m_tiles) {
  const int units = n_tiles * ((m_tiles + 1) / 2), tiles = n_tiles * m_tiles;
  return 0.93f * (float)((units + kSms / 2 - 1) / (kSms / 2)) <= (float)((tiles + kSms - 1) / kSms);
}

}  // namespace dare
