// Host side of the tensor-core path: TMA tensor maps and the per-step kernel sequence.
#include <new>

#include "layer.h"
#include "tc.h"

namespace dare {

struct TcState {
  CUtensorMap a_xn, a_oc;                  // A operands, box 64 x 128 rows
  CUtensorMap a_oc32;                      // ... box 64 x 32 rows, for row tiles that run on across sequences
  CUtensorMap a_xg;                        // compact copy of a refresh set's rows (the input staging buffer, idle after RMSNorm)
  CUtensorMap w_q, w_k, w_v, w_o;          // weights, box 64 x 256 rows
  CUtensorMap w_k128, w_v128, w_q128, w_o128;   // weights, box 64 x 128 rows
  CUtensorMap w_q64, w_o64;                // weights, box 64 x 64 rows (narrow pair tiles)
  KvMaps kv;                               // K/V caches as attention operands
};

namespace {

// units (column tile x pair of row tiles) from which the two-CTA form of a listed launch runs: two rounds of the 74 clusters
constexpr int kPairUnitGate = 2 * (kSms / 2);

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Reduction splits for a launch with `tiles` output tiles: enough CTAs to cover the SMs, never more than the
// k-blocks or the scratch allow.
int pick_splits(int tiles, int kblocks) {
  int s = 1;
  while (s < 2 && tiles * s * 2 <= 160 && s * 2 <= kblocks) s *= 2;
  return s;
}

// ... of narrow K/V tiles: up to four
int kv_splits(int tiles, int kblocks) {
  int s = pick_splits(tiles, kblocks);
  return s == 2 && tiles * 4 <= 128 && kblocks % 4 == 0 && kblocks >= 16 ? 4 : s;
}

}  // namespace

// Row-major bf16 matrix [rows, cols]; box = 64 columns (128 bytes, the swizzle span) x box_rows rows.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool tc_supported(const dare_layer_config_t& c) {
  return c.dtype == DARE_BF16 && (c.head_dim == 128 || c.head_dim == 64) && c.d_model % 256 == 0;
}

dare_status_t tc_create(dare_layer* L) {
  TcState* s = new (std::nothrow) TcState();
  if (!s) return DARE_ERR_INVALID_ARG;
  const uint64_t Tm = (uint64_t)L->cfg.max_batch * L->cfg.max_seq, d = L->cfg.d_model;
  bool ok = make_map(&s->a_xn, L->buf.xn, Tm, d, 128) && make_map(&s->a_xg, L->buf.x_stage, Tm, d, 128) &&
            make_map(&s->a_oc, L->buf.oc, Tm, d, 128) && make_map(&s->a_oc32, L->buf.oc, Tm, d, 32) && make_map(&s->w_q, L->w.w_q, d, d, 256) &&
            make_map(&s->w_k, L->w.w_k, d, d, 256) && make_map(&s->w_v, L->w.w_v, d, d, 256) &&
            make_map(&s->w_o, L->w.w_o, d, d, 256) && make_map(&s->w_k128, L->w.w_k, d, d, 128) &&
            make_map(&s->w_v128, L->w.w_v, d, d, 128) && make_map(&s->w_q128, L->w.w_q, d, d, 128) &&
            make_map(&s->w_o128, L->w.w_o, d, d, 128) && make_map(&s->w_q64, L->w.w_q, d, d, 64) &&
            make_map(&s->w_o64, L->w.w_o, d, d, 64) && make_map(&s->kv.k128, L->buf.kc, Tm, d, 128) &&
            make_map(&s->kv.v128, L->buf.vc, Tm, d, 128) && make_map(&s->kv.k64, L->buf.kc, Tm, d, 64) &&
            make_map(&s->kv.v64, L->buf.vc, Tm, d, 64);
  if (!ok) { delete s; return DARE_ERR_CUDA; }
  L->tc = s;
  return DARE_OK;
}

void tc_destroy(dare_layer* L) {
  delete L->tc;
  L->tc = nullptr;
}

dare_status_t step_tc(dare_layer* L, const void* x, const StepGeom& g, int mode, float tau, void* y, cudaStream_t st,
                      bool add_input) {
  typedef __nv_bfloat16 bf16;
  const Buffers& B = L->buf;
  const TcState& S = *L->tc;
  const int T_ = g.tokens(), d = g.d;
  const bool has_prev = L->has_prev;
  const bool kv_sparse = has_prev && (mode & DARE_MODE_KV);
  const bool o_sparse = has_prev && (mode & DARE_MODE_O);
  // the input staging buffer doubles as the compact copy of a refresh set's rows once x has been normalised; not
  // when x is still needed later (the residual of a transformer block reads it in the output projection)
  const bool compact_ok = !add_input || x != B.x_stage;
  // Row tiles of the projections run on across sequences: x_norm is compact over the step's tokens, and the O cache is
  // too where the step covers all of every sequence, or can be fetched in boxes of 32 rows.  Otherwise a sequence's last
  // tile may be partly filled (eight windows of 32 rows are two tiles, not eight).
  const int tiles_per_seq = (g.seq_act + 127) / 128, m_tiles_seq = g.batch * tiles_per_seq;
  const bool run_on = (T_ + 127) / 128 < m_tiles_seq;
  const int m_tiles_dense = run_on ? (T_ + 127) / 128 : m_tiles_seq;
  const bool oc_compact = g.seq_act == g.max_seq, oc_flat = run_on && (oc_compact || g.seq_act % 32 == 0);
  const int m_tiles_out = oc_flat ? m_tiles_dense : m_tiles_seq;
  const int kblocks = d / 64;
  int launches = 0;
  cudaError_t e;

  GemmParams base;
  base.K = d; base.m_total = T_; base.seq_act = g.seq_act; base.tiles_per_seq = tiles_per_seq;
  base.a_seq_stride = g.seq_act; base.a_row0 = 0; base.flat = 0; base.a_piece = 0;
  if (run_on) { base.seq_act = base.a_seq_stride = T_; base.tiles_per_seq = m_tiles_dense; base.flat = 1; }
  base.idx = nullptr; base.count = nullptr; base.g = g;
  base.gather_src = nullptr; base.gather_cache_rows = 0; base.unit_gate = 0;
  base.n_split = 1 << 30; base.out0 = nullptr; base.out1 = nullptr; base.ld_out = d;
  base.out_is_cache = 0; base.resid = nullptr; base.ld_resid = 0; base.out_f32 = nullptr; base.b_pair = 0;
  base.rope = reinterpret_cast<const float2*>(B.rope_cs); base.q_prev = B.q_prev;
  base.scores = B.scores; base.has_prev = has_prev ? 1 : 0; base.status = B.status;
  base.debug = nullptr; base.wait_at_end = 0; base.late_wait = 0; base.loop_rows = 0;
  base.gate_count = nullptr; base.gate_lo = 0; base.gate_hi = 1 << 30; base.store_mask = nullptr;
  // Steps of many row tiles: from these refresh-set sizes on the dense forms of the K/V projection, of attention and of
  // the output projection (results kept for the refreshed rows only) are faster than the listed forms.  Measured on
  // the long-context sweep (batch 4 x 4096): the listed K/V projection with its compact copy passes the dense form's
  // time at about 78 % of the tokens, row-sparse attention + gathered output projection with its copy of the reused
  // rows at about 80 %, all of them together at about 85 %.
  const int gate_kv = (int)(0.75 * T_), gate_o = (int)(0.80 * T_);
  unsigned long long* dbg = L->debug_on ? B.debug : nullptr;
  // (no clearing between steps: a copy or memset in the stream would break the kernels' launch overlap; the stamps
  // are plain stores or maxima of a clock that only grows)

  // A dense K/V projection (Alg. 2 line 7, or the full forward of Appendix E.2) needs nothing from the Q projection
  // or the selection.  On a short step (launches of about one wave, where fixed costs and the hand-off between
  // kernels decide) it is issued right behind the Q projection and runs beside it: the two launches are one fused
  // Q/K/V projection of the step's rows, spread over two grids because the Q tiles take a split reduction and the
  // K/V tiles do not.  The selection then follows both.
  // (K/V tiles that are more than one wave may be better off in the persistent kernel behind the Q projection: a round of
  // CTAs of both launches takes about 9 us + 0.36 us a k-block, the persistent kernel 0.33 us a k-block and round of pairs)
  bool kv_beside_q = !kv_sparse && m_tiles_dense <= 8;
  if (kv_beside_q && persist_pays(2 * d / 256, m_tiles_dense, pick_splits(2 * d / 256 * m_tiles_dense, kblocks))) {
    const int q_ctas = d / 256 * ((m_tiles_dense + 1) / 2 * 2), units = 2 * d / 256 * ((m_tiles_dense + 1) / 2);
    const float beside = (float)((q_ctas + 2 * d / 256 * m_tiles_dense + kSms - 1) / kSms) * (9.f + 0.36f * (float)kblocks);
    const float behind = 20.f + 0.33f * (float)(kblocks * (1 + (units + 73) / 74));
    kv_beside_q = beside < behind;
  }
  // A projection of the refresh set's rows of x_norm (p.idx, p.count): a compact copy of them, then the launch in three forms,
  // each of which looks at the count (launches counted here): listed in two-CTA and in one-CTA tiles; from gate_kv refreshed tokens on dense, every row
  // of the step projected and the refresh set's stored.
  auto listed_projection = [&](int epi, GemmParams p, const CUtensorMap& b0, const CUtensorMap& b1, const CUtensorMap& b2, const CUtensorMap& b0h,
                               const CUtensorMap& b1h, const CUtensorMap& b2h, int n_tiles) {
    const int m_tiles = (T_ + 127) / 128;
    const bool dense_form = persist_pays_listed(n_tiles, m_tiles_dense);
    const int hi = dense_form ? gate_kv : 1 << 30;
    launch_gather_step_rows((const bf16*)B.xn, B.idx, B.count, (bf16*)B.x_stage, g, false, st, B.status, hi); ++launches;
    p.gather_src = nullptr;
    p.unit_gate = kPairUnitGate;
    p.gate_count = B.count; p.gate_hi = hi;
    cudaError_t err = launch_gemm_persist(epi, S.a_xg, b0h, b1h, b2h, p, n_tiles, m_tiles, st, 1); ++launches;
    if (err == cudaSuccess) { err = launch_gemm_persist(epi, S.a_xg, b0, b1, b2, p, n_tiles, m_tiles, st, 0); ++launches; }
    if (dense_form && err == cudaSuccess) {
      p.idx = nullptr; p.count = nullptr; p.unit_gate = 0;
      p.gate_lo = gate_kv; p.gate_hi = 1 << 30; p.store_mask = B.delta;
      err = launch_gemm_persist(epi, S.a_xn, b0h, b1h, b2h, p, n_tiles, m_tiles_dense, st, 1); ++launches;
    }
    return err;
  };
  prof_begin(L);
  // Alg. 1/2 line 1
  prof_mark(L, SLOT_NORM, st);
  launch_rmsnorm<bf16>((const bf16*)x, L->w.rms_gain, (bf16*)B.xn, T_, d, L->cfg.rms_eps, st, dbg ? dbg + 40 : nullptr);
  ++launches;
  // A step of many tokens that reuses attention outputs needs the scoring head of every token (the score, the stored query),
  // and of the other heads only the queries that attend, the refresh set's (Alg. 2 line 8): the scoring head's 128 columns are
  // projected first, and the refresh set's queries behind the selection, beside its K and V where those are listed as well.
  // 4 x 4096 tokens of width 4096, both rules, 15 % refreshed: 1019 -> 684 us; 8 x 1024, output reuse, 13 %: 783 -> 627 us.
  // With (nearly) all tokens refreshed the scoring head is projected twice and launches are added that only look at the count, which
  // costs up to 4 % of a step; hence a query projection of some size, and of some width: the scoring head's launch streams x_norm,
  // 360 / d of the time of the whole query projection.  In us, one projection of all queries / scoring head first, at 15 %, 50 %
  // and all tokens refreshed:
  //   both:   4 x 4096 of 4096  954 / 656, 1737 / 1543, 2808 / 2770    16 x 288 of 2048 (34 GFLOP) 144 / 122, 207 / 193, 243 / 251
  //           8 x 1700 of 1536  220 / 171, 339 / 294, 489 / 496        32 x 1024 of 1024 300 / 246, 432 / 389, 579 / 595
  //   output: 4 x 4096 of 4096  1574 / 1186, 2250 / 1905, 2799 / 2764  2 x 1250 of 4096 (84 GFLOP) 324 / 282, 388 / 373, 417 / 416
  //           4 x 4096 of 2048  593 / 542, 980 / 905, 1046 / 1035      4 x 2300 of 2048 (77 GFLOP) 349 / 315, -, 496 / 507
  //   widths below the rule's, both: 32 x 1024 of 768 247 / 211, -, 432 / 450    64 x 1100 of 512 396 / 352, -, 826 / 875
  //           128 x 2100 of 256 964 / 934, -, 2128 / 2247
  // A step that is given its reuse rate knows when more than three quarters will be refreshed, one with a threshold below every
  // score that all will.  (Up to eight row tiles the projections are streams of the weights whatever the rows: 90 us this way
  // against 78 at 512 tokens of width 4096.)
  const int n_listed = (kv_sparse ? 3 : 1) * (d / 256);
  const double q_flop = 2.0 * T_ * (double)d * d;
  const bool many_known = L->reuse_count >= 0 ? 4ll * (T_ - L->reuse_count) > 3ll * T_ : tau < 0.f;
  const bool q_pays = !many_known && d >= 1024 && q_flop >= (kv_sparse ? 34e9 : 80e9);
  const bool q_listed = o_sparse && m_tiles_dense > 8 && compact_ok && q_pays && persist_pays_listed(n_listed, (T_ + 127) / 128);
  if (q_listed) {
    GemmParams p = base;
    p.debug = dbg;
    prof_mark(L, SLOT_Q_GEMM, st);
    TileForm f;
    if (!pick_one_wave(128, m_tiles_dense, kblocks, &f)) f = TileForm{128, 0, 1};
    const CUtensorMap& wq = f.pair ? S.w_q64 : S.w_q128;
    e = launch_gemm_tc(EPI_SCORE, 128, S.a_xn, wq, wq, p, 1, m_tiles_dense, f.splits, st, f.pair);
    ++launches;
    if (e != cudaSuccess) return DARE_ERR_CUDA;
  } else {
    // line 2 + line 3 + stored-query update + rotary embedding, one kernel
    GemmParams p = base;
    p.out0 = (bf16*)B.q;
    p.debug = dbg;
    prof_mark(L, SLOT_Q_GEMM, st);
    TileForm f;
    // (a K/V projection beside it: both launches resident at once where they fit and this one does not become the longer)
    int kv_ctas = 0;
    float kv_us = 0.f;
    if (kv_beside_q) {
      const int n_kv = 2 * d / 256, sp = pick_splits(n_kv * m_tiles_dense, kblocks);
      kv_ctas = m_tiles_dense == 1 ? 2 * n_kv * kv_splits(2 * n_kv, kblocks)
                                   : n_kv * (pairs_pay(n_kv, m_tiles_dense, sp) ? (m_tiles_dense + 1) / 2 * 2 : m_tiles_dense) * sp;
      kv_us = 0.33f * (float)(kblocks / sp) + 6.f;
    }
    if ((kv_ctas > 0 && pick_one_wave(d, m_tiles_dense, kblocks, &f, kv_ctas, kv_us)) ||
        pick_one_wave(d, m_tiles_dense, kblocks, &f)) {
      const int box = f.pair ? f.bn / 2 : f.bn;
      const CUtensorMap& wq = box == 256 ? S.w_q : (box == 128 ? S.w_q128 : S.w_q64);
      e = launch_gemm_tc(EPI_Q, f.bn, S.a_xn, wq, wq, p, d / f.bn, m_tiles_dense, f.splits, st, f.pair);
    } else {
      const int pair = persist_pairs_pay(d / 256, m_tiles_dense) ? 1 : 0;
      const CUtensorMap& wq = pair ? S.w_q128 : S.w_q;
      e = launch_gemm_persist(EPI_Q, S.a_xn, wq, wq, p, d / 256, m_tiles_dense, st, pair);
    }
    ++launches;
    if (e != cudaSuccess) return DARE_ERR_CUDA;
  }
  // lines 4-5 + Sec. 4
  const bool select_all = !has_prev || mode == DARE_MODE_DENSE;
  auto select_now = [&]() {
    prof_mark(L, SLOT_SELECT, st);
    // (a selection that refreshes everything reads no scores: behind the two projections it runs beside them)
    select_step(L, g, mode, tau, kv_beside_q && select_all, st, &launches);
  };
  const bool injected = L->inject != 0;          // (diagnostics: the projection then has to read the list)
  if (!kv_beside_q) select_now();
  // K/V projection with rotary embedding and cache scatter
  {
    GemmParams p = base;
    p.n_split = d / 256;
    p.out0 = (bf16*)B.kc; p.out1 = (bf16*)B.vc; p.out_is_cache = 1;
    p.debug = dbg ? dbg + 8 : nullptr;
    const int n_tiles = 2 * d / 256;
    if (kv_sparse) {
      // Alg. 1 line 6: the projection fetches the refresh set's rows of x_norm by index as its A operand
      p.idx = B.idx; p.count = B.count; p.gather_src = (const bf16*)B.xn;
      const int m_tiles = (T_ + 127) / 128;
      prof_mark(L, SLOT_KV_GEMM, st);
      if (T_ <= 128 && !injected) {
        // One row tile holds every token of the step, refreshed or not: it is projected as it lies, by TMA, while the
        // selection is still at work, and the rows of the refresh set are stored.  No list, and the main loop is over by
        // the time the selection is (2 windows of 32 rows, width 4096: step 68.5 -> 61.0 us).
        p.idx = nullptr; p.count = nullptr; p.gather_src = nullptr;
        p.n_split = d / 128;
        p.store_mask = B.delta; p.late_wait = 1;
        e = launch_gemm_tc(EPI_KV, 128, S.a_xn, S.w_k128, S.w_v128, p, 2 * d / 128, m_tiles_dense, kv_splits(2 * d / 128, kblocks), st);
        ++launches;
      } else if (m_tiles <= 8) {
        // Few tokens: the refresh set fits one or two row tiles and the projection is a stream of the weights.
        // Narrower tiles put twice as many CTAs on it; the reduction split is sized for one row tile.
        p.n_split = d / 128;
        const int n_tiles128 = 2 * d / 128;
        p.loop_rows = 1;                         // one row of CTAs: no CTA that only looks at the count and leaves
        e = launch_gemm_tc(EPI_KV, 128, S.a_xn, S.w_k128, S.w_v128, p, n_tiles128, 1, kv_splits(n_tiles128, kblocks), st);
        ++launches;
      } else {
        // Many tokens: even a small refreshed fraction fills the GPU with 256-wide tiles, which re-read the least.
        const int n_listed_tiles = q_listed ? n_listed : n_tiles;
        if (persist_pays_listed(n_listed_tiles, m_tiles) && compact_ok) {
          // a compact copy of the refresh set's rows first (a stream of n x d elements), then the projection with
          // every operand through TMA and two-CTA MMAs; beyond gate_kv refreshed tokens the dense form instead: every
          // row of the step projected, the rows of the refresh set stored (the others keep their cached K and V)
          if (q_listed) p.out2 = (bf16*)B.q;
          e = listed_projection(q_listed ? EPI_QKV : EPI_KV, p, S.w_k, S.w_v, S.w_q, S.w_k128, S.w_v128, S.w_q128, n_listed_tiles);
        } else {
          e = launch_gemm_tc(EPI_KV, 256, S.a_xn, S.w_k, S.w_v, p, n_tiles, m_tiles, 1, st);
          ++launches;
        }
      }
    } else {
      prof_mark(L, SLOT_KV_GEMM, st);
      if (q_listed) {
        GemmParams pq = base;
        pq.out0 = (bf16*)B.q;
        pq.idx = B.idx; pq.count = B.count;
        e = listed_projection(EPI_KV, pq, S.w_q, S.w_q, S.w_q, S.w_q128, S.w_q128, S.w_q128, n_listed);
        if (e != cudaSuccess) return DARE_ERR_CUDA;
      }
      p.wait_at_end = kv_beside_q ? 1 : 0;
      const int sp = pick_splits(n_tiles * m_tiles_dense, kblocks);
      if (!kv_beside_q && persist_pays(n_tiles, m_tiles_dense, sp)) {
        const int pair = persist_pairs_pay(n_tiles, m_tiles_dense) ? 1 : 0;
        e = launch_gemm_persist(EPI_KV, S.a_xn, pair ? S.w_k128 : S.w_k, pair ? S.w_v128 : S.w_v, p, n_tiles, m_tiles_dense,
                                st, pair);
      }
      else if (m_tiles_dense == 1) {             // few rows: a stream of the weights, narrow tiles put twice as many CTAs on it
        p.n_split = d / 128;
        e = launch_gemm_tc(EPI_KV, 128, S.a_xn, S.w_k128, S.w_v128, p, 2 * d / 128, 1, kv_splits(2 * d / 128, kblocks), st);
      }
      else if (pairs_pay(n_tiles, m_tiles_dense, sp))
        e = launch_gemm_tc(EPI_KV, 256, S.a_xn, S.w_k128, S.w_v128, p, n_tiles, m_tiles_dense, sp, st, 1);
      else
        e = launch_gemm_tc(EPI_KV, 256, S.a_xn, S.w_k, S.w_v, p, n_tiles, m_tiles_dense, sp, st);
      ++launches;
    }
    if (e != cudaSuccess) return DARE_ERR_CUDA;
  }
  if (kv_beside_q) select_now();
  // attention (row-sparse over the refresh set when O reuse is on)
  prof_mark(L, SLOT_ATTN, st);
  {
    AttnParams p;
    p.q = (const bf16*)B.q; p.oc = (bf16*)B.oc; p.idx = o_sparse ? B.idx : nullptr;
    p.batch_off = o_sparse ? B.batch_off : nullptr; p.g = g; p.status = B.status;
    p.debug = dbg ? dbg + 16 : nullptr;
    // the refresh set then comes from the kernel right before; or the two kernels before ran beside the Q projection
    // without waiting for it, so the queries are not known to be complete before this kernel's own wait
    // (or the kernel before wrote the queries themselves)
    p.wait_first = kv_beside_q || (q_listed && kv_sparse) ? 1 : 0;
    p.gate_count = nullptr; p.gate_lo = 0; p.gate_hi = 1 << 30; p.store_mask = nullptr;
    // a long row-sparse step is issued in both forms: over the refresh set's rows, and dense with only the refreshed
    // rows stored (tiles without one skipped); the size of the set decides on the device which of them runs
    const bool both_forms = o_sparse && m_tiles_dense > 8 && persist_pays_listed(d / 256, m_tiles_dense);
    // (one launch carries both when both take the kernel with two query tiles per CTA: its CTAs pick the form; a
    // launch that only looks at the count and leaves still costs a wave of CTAs per 148 of them)
    const bool one_launch = both_forms && attention_tc_two_tiles(g, true) && attention_tc_two_tiles(g, false);
    p.dense_from = 0; p.dense_mask = nullptr;
    if (both_forms) {
      p.gate_count = B.count;
      if (one_launch) { p.dense_from = gate_o; p.dense_mask = B.delta; }
      else p.gate_hi = gate_o;
    }
    e = launch_attention_tc(S.kv, p, st); ++launches;
    if (both_forms && !one_launch && e == cudaSuccess) {
      AttnParams pd = p;
      pd.idx = nullptr; pd.batch_off = nullptr; pd.debug = nullptr;
      pd.gate_lo = gate_o; pd.gate_hi = 1 << 30; pd.store_mask = B.delta;
      e = launch_attention_tc(S.kv, pd, st); ++launches;
    }
    if (e != cudaSuccess) return DARE_ERR_CUDA;
  }
  // Output projection, read from the O cache.  Alg. 2 line 11 projects every row of the window.  A row whose
  // attention output was reused projects to what it projected to before (W_O acts row by row), so with many tokens
  // the library keeps those projections by cache row and, on a step that reuses attention outputs, projects the
  // refresh set's rows only (fetched from the O cache by index, like the rows of the gathered K/V projection) and
  // copies the others.  With few tokens the projection is a stream of W_O whatever the row count, and stays dense.
  {
    const bool many = m_tiles_dense > 8 && !add_input;
    const CUtensorMap& a_oc = oc_flat && !oc_compact ? S.a_oc32 : S.a_oc;
    const bool y_sparse = o_sparse && many && L->yc_valid;
    GemmParams p = base;
    if (oc_flat) {
      p.a_piece = oc_compact ? 0 : 1;
    } else {
      p.seq_act = g.seq_act; p.tiles_per_seq = tiles_per_seq; p.a_seq_stride = g.max_seq; p.a_row0 = g.pos_begin; p.flat = 0;
    }
    p.out0 = (bf16*)y;
    if (many) p.out1 = (bf16*)B.yc;                                   // kept by cache row for later steps
    if (add_input) { p.resid = (const bf16*)x; p.ld_resid = d; }      // y = x + W_O O (residual block)
    p.debug = dbg ? dbg + 24 : nullptr;
    const int n_tiles = d / 256;
    prof_mark(L, SLOT_OUT_GEMM, st);
    if (y_sparse) {
      const int a_piece = p.a_piece;
      p.idx = B.idx; p.count = B.count; p.gather_src = (const bf16*)B.oc; p.gather_cache_rows = 1; p.a_piece = 0;
      bool dense_form = false;
      if (persist_pays_listed(n_tiles, (T_ + 127) / 128) && compact_ok) {
        // (beyond gate_o refreshed tokens the dense projection of every row instead: Alg. 2 line 11 as written)
        dense_form = persist_pays_listed(n_tiles, m_tiles_out);
        const int hi = dense_form ? gate_o : 1 << 30;
        launch_gather_step_rows((const bf16*)B.oc, B.idx, B.count, (bf16*)B.x_stage, g, true, st, B.status, hi); ++launches;
        p.gather_src = nullptr;
        p.unit_gate = kPairUnitGate;
        p.gate_count = B.count; p.gate_hi = hi;
        e = launch_gemm_persist(EPI_OUT, S.a_xg, S.w_o128, S.w_o128, p, n_tiles, (T_ + 127) / 128, st, 1); ++launches;
        if (e == cudaSuccess) e = launch_gemm_persist(EPI_OUT, S.a_xg, S.w_o, S.w_o, p, n_tiles, (T_ + 127) / 128, st, 0);
        if (dense_form && e == cudaSuccess) {
          GemmParams pd = p;
          pd.idx = nullptr; pd.count = nullptr; pd.unit_gate = 0; pd.gather_cache_rows = 0; pd.a_piece = a_piece;
          pd.gate_lo = gate_o; pd.gate_hi = 1 << 30;
          ++launches;
          e = launch_gemm_persist(EPI_OUT, a_oc, S.w_o128, S.w_o128, pd, n_tiles, m_tiles_out, st, 1);
        }
      } else
        e = launch_gemm_tc(EPI_OUT, 256, S.a_oc, S.w_o, S.w_o, p, n_tiles, (T_ + 127) / 128, 1, st);
      ++launches;
      if (e != cudaSuccess) return DARE_ERR_CUDA;
      launch_copy_reused_rows((const bf16*)B.yc, (bf16*)y, B.delta, g, st, dense_form ? B.count : nullptr, gate_o); ++launches;
    } else {
      TileForm f;
      if (pick_one_wave(d, m_tiles_out, kblocks, &f)) {
        const int box = f.pair ? f.bn / 2 : f.bn;
        const CUtensorMap& wo = box == 256 ? S.w_o : (box == 128 ? S.w_o128 : S.w_o64);
        e = launch_gemm_tc(EPI_OUT, f.bn, a_oc, wo, wo, p, d / f.bn, m_tiles_out, f.splits, st, f.pair);
      } else {
        const int pair = persist_pairs_pay(n_tiles, m_tiles_out) ? 1 : 0;
        const CUtensorMap& wo = pair ? S.w_o128 : S.w_o;
        e = launch_gemm_persist(EPI_OUT, a_oc, wo, wo, p, n_tiles, m_tiles_out, st, pair);
      }
      ++launches;
      if (e != cudaSuccess) return DARE_ERR_CUDA;
      // the cache is complete once a dense projection has covered every cached row, and stays so while every
      // later step maintains it
      if (many) {
        if (g.pos_begin == 0 && g.seq_act == g.kv_len) L->yc_valid = true;
      } else {
        L->yc_valid = false;
      }
    }
  }
  prof_end(L, st);
  L->last_launches = launches;
  L->last_forms = q_listed ? DARE_FORM_SCORE_FIRST : 0;
  if (cudaGetLastError() != cudaSuccess) return DARE_ERR_CUDA;
  return DARE_OK;
}

}  // namespace dare
