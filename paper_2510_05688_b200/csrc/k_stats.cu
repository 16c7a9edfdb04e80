// Deterministic sums and base-sample statistics.
//
// For each (batch row, query head) the rows of I_f = sink + I_t + window and of the base sample I_bs
// are gathered (K and V), rescored in fp64 and reduced:
//     D_f = sum_{I_f} w_i,  N_f = sum_{I_f} w_i V[i]                       (Sec. 4.1, N_f and D_f)
//     sum w, sum w^2, sum r, sum r.r over I_bs with r_i = w_i V[i]           (Algorithm 2, get-stats)
// with w_i = exp(s_i - m).  Every CTA leaves one partial; the last CTA of a head to finish (a counter) adds them in
// split order and evaluates the budget (Algorithm 2, Theorem 4.3 / Corollaries D.2):
//     sigma^2, Tr(Sigma), D_hat, |N_hat|,  b_D, b_N, b_SDPA,  b = clamp(ceil(b_X), b0, n_s)
// in fp64 (the two square-root / division chains on two lanes, the 15 split points of b_SDPA on 15 lanes).  Nearly
// every head is then done: its I_dyn is the unmarked entries of a prefix of the final sample's walk, laid out or (beyond the walk
// array) computed by the gather, or every residual token.  Only a head with more than 1,024 marked entries in the array, whose
// positions are not all known, has its final sample (Algorithm 1 line 7) listed by the same CTA: the array's entries without
// the marked ones, then further positions, or, when b is the whole residual, every residual token in token order.
//
// Everything that decides the integer budget is fp64: the same inputs must give the same ceil() as a
// plain fp64 evaluation.  Variances are accumulated around a pivot (the first base-sample row), which
// removes the cancellation of the one-pass formula and makes a constant population give exactly 0.
//
// Grid: per head, `stat_splits` CTAs take the deterministic rows and `stat_splits` CTAs the base-sample
// rows (two code paths with disjoint accumulators, which halves the register footprint of either).
// What bounds it: instruction issue (fp64 products, bf16 -> fp64 conversions, reductions across lanes) as much as memory.
// A row group (LPR lanes) works in batches of four rows: one read of q from shared memory, one exp and one
// handing-over butterfly per batch; K elements become doubles by integer moves; a row's address is one multiply-add from
// its 32-bit index; rows arrive by asynchronous copies two batches ahead (see the main loop).
#include "rows_stats.cuh"

namespace {

// CTAS: CTAs per SM (see stat_ctas_per_sm)
template <typename T, int D, bool SPLIT, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) k_stats(const __grid_constant__ Prob p) {
  constexpr int NE = D + 3;               // det CTA: N_f[D], D_f;  base CTA: Sr[D], Sw, Sww, Srr
  using R = StatRows<T, D, SPLIT>;
  __shared__ typename R::Sm sm;

  const int tid = threadIdx.x;
  // Grid (S, Hq, 2 B).  In dispatch order a batch row's base-row CTAs follow its deterministic-row CTAs, so that the first rows'
  // heads have their budgets while later rows' CTAs are still to come (202.2 -> 199.2 us per step at 8 x 32,768, 141.6 ->
  // 140.1 at 5 x 12,100 to 48,401; base-row CTAs first: 201.2).  With one CTA of either kind per head (many heads) those of all
  // rows come first: they are short, and the others' words are there by then (57.6 against 61.7 at 480 heads x 178 to 1,427).
  const bool base_cta = p.stat_by_row ? (blockIdx.z & 1u) != 0u : (int)blockIdx.z >= p.B;
  const int h = blockIdx.y, b = p.stat_by_row ? blockIdx.z >> 1 : base_cta ? blockIdx.z - p.B : blockIdx.z, g = h / p.G;
  const int bh = b * p.Hq + h;
  const int split = blockIdx.x;
  const int vx = (base_cta ? MAXS : 0) + split;    // position among the head's 2 MAXS partial slots
  const int n = head_len(p, b, h);
  const Geo geo = head_geometry(p, n);
  const int s0 = geo.s0, l_start = geo.l_start, kk = geo.kk, b0 = geo.b0;
  const int n_f = s0 + kk + (n - l_start);
  // CTAs of either kind that this head uses: the grid is sized for the longest sequence a plan takes
  const int Sd = stat_ctas(n_f, p.stat_splits, p.stat_rows), Sb = stat_ctas(b0, p.stat_splits_base, p.stat_rows);
  const int S = base_cta ? Sb : Sd;
  if (split >= S) return;
  __shared__ double s_pre[3];                      // for the budget: n_s / b0, 1 / b0, 1 / (b0 - 1)
  if (tid == NT - 1) {
    s_pre[0] = b0 > 0 ? (double)geo.n_s / (double)b0 : 0.0;
    s_pre[1] = b0 > 0 ? 1.0 / (double)b0 : 0.0;
    s_pre[2] = b0 > 1 ? 1.0 / (double)(b0 - 1) : 0.0;
  }
  TICK_BEGIN(p, VATTN_K_STATS);
  pdl_trigger();
  R::load_q(p, sm, b, h);
  // What a CTA needs of its head comes from the step's inputs (the head's geometry), from the score pass (the
  // largest score) and, for the base sample, from one 64-bit word that the selection kernel publishes when I_t is
  // written and marked in the walk arrays: 2 | K not finite << 2 | base_J << 3 | the pivot row's index << 32.  This grid's CTAs
  // were launched after every CTA of that kernel had started (programmatic dependent launch), so the producer of a
  // word is running or done when a CTA here polls it: the wait cannot starve.  It is bounded all the same; when it
  // runs out the CTA falls back to the grid-level dependency wait, which is always sufficient.
  __shared__ unsigned long long s_word;
  __shared__ int s_flag;
  __shared__ int s_misc[8];
  // deterministic-row CTAs wait for a 32-bit word of their own, base-row CTAs for the 64-bit one (the selection kernel
  // stores both together, once I_t is marked in the base walk)
  HeadWords* hw = p.words + bh;
  if (tid == 0) {
    const unsigned long long v = base_cta ? wait_word64(&hw->sample, VATTN_WORD_SPINS)
                                          : (unsigned long long)wait_word32(&hw->topk, VATTN_WORD_SPINS);
    s_word = v;
  }
  const float m_f = unord_f32(__ldcg(p.m_ord + bh));
  __syncthreads();
  unsigned long long word = s_word;
  if (word == 0ull) {                              // the bounded wait ran out
    pdl_wait();
    __syncthreads();                               // (every thread has seen the zero before it is replaced)
    if (tid == 0) s_word = base_cta ? __ldcg(&hw->sample) : (unsigned long long)__ldcg(&hw->topk);
    __syncthreads();
    word = s_word;
  }
  if (base_cta) DBGT(36);
  if (base_cta && split == 0) DBGH(bh, 6);
  const bool odd = ((word >> (base_cta ? 2 : 1)) & 1ull) != 0;       // the KV head's K holds elements that are not finite
  const int base_J = (int)((word >> 3) & 0x3FFFFFull), word_piv = (int)(unsigned)(word >> 32);
  if (n == 0) {                                    // an empty row: no sums, budget 0
    if (base_cta && split == 0) {
      pdl_wait();
      if (tid == 0) {
        publish_budget(p, bh, GMeta{0, 0, 0.f, 0, 0, 0, 0, 0});
        if (p.dbg.dyn_cnt) p.dbg.dyn_cnt[bh] = 0;
        if (p.dbg.budgets) for (int e = 0; e < 4; ++e) p.dbg.budgets[bh * 4 + e] = 0;
        if (p.dbg.stats) for (int e = 0; e < 8; ++e) p.dbg.stats[bh * 8 + e] = 0.0;
      }
    }
    return;
  }
  // base sample: the unmarked entries among the first base_J of its walk array
  const int total = base_cta ? (b0 > 0 ? base_J : 0) : n_f;
  const int chunk = (total + S - 1) / S;
  const int r_begin = min(total, split * chunk), r_end = min(total, r_begin + chunk);
  R::run(p, sm, bh, g, base_cta, odd, word_piv, m_f, r_begin, r_end);
  double* gpart = p.stat_part + ((long long)bh * 2 * MAXS + vx) * NE;
  for (int e = tid; e < NE; e += NT) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < NWARP; ++w) s += sm.u.part[w][e];
    gpart[e] = s;
  }
  if (base_cta && split == 0 && b0 > 0)              // the pivot travels with this CTA's partial
    for (int e = tid; e <= D; e += NT) p.stat_piv[(long long)bh * (D + 1) + e] = sm.piv[e];
  // ---- the last CTA of the head to arrive here evaluates the budget
  // (the barrier orders every thread's writes before thread 0's fence, which is cumulative; likewise on the way in)
  __syncthreads();
  DBGT(34);
  if (tid == 0) {
    s_flag = ticket(&hw->stat_ticket) == (unsigned)(Sd + Sb - 1);
  }
  __syncthreads();
  if (base_cta && split == 0) DBGH(bh, 2);              // (one base CTA's rows are done)
  if (s_flag) {
    DBGH(bh, 3);
    // the rest of the list needs the selection kernel's last words (how far it listed the walk): wait for that
    // grid as a whole, which also makes "this grid has completed" imply "the selection kernel has" for the gather
    // kernel behind
    pdl_wait();
    DBGT(35);
    TICK_BEGIN(p, VATTN_T_BUDGET);
    const double* src = p.stat_part + (long long)bh * 2 * MAXS * NE;
    const double* gpiv = p.stat_piv + (long long)bh * (D + 1);
    const HeadBudget hb = head_budget<D>(p, bh, Sd, Sb, s_pre, sm.pivT, true,
                                         [&](int kind, int s, int e) { return __ldcg(src + (kind * MAXS + s) * NE + e); },
                                         [&](int e) { return __ldcg(gpiv + e); });
    // N_f and D_f for the gather kernel's last finisher, then the head's record, which is "the budget is known" at the same
    // time.  The barrier orders every thread's writes before thread 0's release, which is cumulative.
    double* det = p.det_sums + (long long)bh * (D + 1);
    if (tid < D) det[tid] = hb.det;
    if (tid == 0) det[D] = hb.det_den;
    if (hb.g.list) list_sample(p, b, h, bh, hb.g.b, s_misc);
    __syncthreads();
    if (tid == 0) publish_budget(p, bh, hb.g);
    if (!hb.g.list && p.dbg.dyn_idx) list_sample(p, b, h, bh, hb.g.b, s_misc);
    if (tid == 0) p.m_ord[bh] = 0u;                  // (every CTA of the head has read it: ready for the next step)
    DBGH(bh, 4);
    TICK_END(p, VATTN_T_BUDGET);
  }
  TICK_END(p, VATTN_K_STATS);
}

}  // namespace

template <typename T, int D, bool SPLIT, int CTAS>
static cudaError_t launch_stats_n(const Prob& p, cudaStream_t s) {
  static size_t have[VATTN_MAXDEV];
  cudaError_t e = optin_smem(k_stats<T, D, SPLIT, CTAS>, 0, have, true);
  if (e != cudaSuccess) return e;
  const dim3 grid(p.stat_splits > p.stat_splits_base ? p.stat_splits : p.stat_splits_base, p.Hq, 2 * p.B);
  return launch_pdl(k_stats<T, D, SPLIT, CTAS>, grid, dim3(NT), 0, s, p);
}
template <typename T, int D>
static cudaError_t launch_stats_t(const Prob& p, cudaStream_t s) {
  if (p.row_unit == 0u) return launch_stats_n<T, D, true, 5>(p, s);      // (rare: one form)
  return stat_ctas_per_sm(p.B * p.Hq) == 4 ? launch_stats_n<T, D, false, 4>(p, s) : launch_stats_n<T, D, false, 5>(p, s);
}

cudaError_t launch_stats(const Prob& p, cudaStream_t s) {
  if (p.stat_splits < 1 || p.stat_splits > MAXS || p.stat_splits_base < 1 || p.stat_splits_base > MAXS) return cudaErrorInvalidValue;
  if (p.dtype == VATTN_DTYPE_BF16) return p.D == 128 ? launch_stats_t<bf16_t, 128>(p, s) : launch_stats_t<bf16_t, 64>(p, s);
  return p.D == 128 ? launch_stats_t<float, 128>(p, s) : launch_stats_t<float, 64>(p, s);
}
