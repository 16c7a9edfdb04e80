// The statistics of a head's rows and the budget they give: shared by the kernels that work on rows (k_stats.cu, k_rows.cu).
#pragma once
#include "vattn_internal.cuh"
#include <math_constants.h>

namespace {

constexpr int NT = 128;
constexpr int NWARP = NT / 32;
constexpr int UN = 4;            // rows per batch of a row group
constexpr int SEC = 256;         // entries staged at a time
constexpr int MAXS = VATTN_STAT_MAXS;   // most split CTAs per head and kind
constexpr unsigned FULLMASK = 0xFFFFFFFFu;

template <typename T> __device__ __forceinline__ float slice_elem(const uint4& v, int e);
template <> __device__ __forceinline__ float slice_elem<float>(const uint4& v, int e) {
  return __uint_as_float(e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w);
}
template <> __device__ __forceinline__ float slice_elem<bf16_t>(const uint4& v, int e) {
  const unsigned w = (e >> 1) == 0 ? v.x : (e >> 1) == 1 ? v.y : (e >> 1) == 2 ? v.z : v.w;
  return __uint_as_float((e & 1) ? (w & 0xFFFF0000u) : (w << 16));
}
// A finite bf16 element times 2^-896 as a double, exactly, by moving its bits: the fp32 pattern shifted right by three
// under its sign is the upper half of that double's pattern (zeros and denormals included).  Two integer instructions
// instead of a conversion, which has a quarter of their rate; the factor is taken up by q.  (Infinities and NaNs would
// come out finite: the caller takes the conversion for caches that hold any.)
constexpr double Q_SCALE = 0x1p896;
template <typename T> __device__ __forceinline__ double scaled_elem(const uint4& v, int e) {
  const unsigned t = __float_as_uint(slice_elem<T>(v, e));
  return __hiloint2double((int)(((unsigned)((int)t >> 3)) & 0x8FFFFFFFu), 0);
}
__device__ __forceinline__ double shfl_xor_d(double v, int mask) { return __shfl_xor_sync(FULLMASK, v, mask); }

// fp64 weights exp(scale <q, K[row]> - m) of the UN = 4 rows whose K slices a row group's LPR lanes hold.  The lanes'
// partial inner products are added by a butterfly that hands rows over while it adds (two exchanges, one exchange,
// then plain additions): lane j ends with one row's product, evaluates ONE exp, and the four weights are handed
// round: 4 + log2(LPR) + 1 double shuffles per four rows instead of 4 log2(LPR) + 4.  q (times Q_SCALE) is read from
// shared memory once per element and batch.  odd: some K element of the KV head is not finite.
template <typename T, int D>
__device__ __forceinline__ void weights64(const double* qs, const uint4 (&k)[UN], bool odd, double scale, double m, int j, double (&w)[UN]) {
  constexpr int EPL = Elem<T>::EPL, LPR = D / EPL;
  static_assert(UN == 4 && LPR >= 8, "two hand-over levels");
  double d[UN] = {0.0, 0.0, 0.0, 0.0};
  if (sizeof(T) == 2 && !odd) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const double q = qs[e * LPR];
#pragma unroll
      for (int u = 0; u < UN; ++u) d[u] = fma(q, scaled_elem<T>(k[u], e), d[u]);
    }
  } else {
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const double q = qs[e * LPR] * (1.0 / Q_SCALE);
#pragma unroll
      for (int u = 0; u < UN; ++u) d[u] = fma(q, (double)slice_elem<T>(k[u], e), d[u]);
    }
  }
  const bool a = (j & (LPR / 2)) != 0, b = (j & (LPR / 4)) != 0;
  const double x0 = (a ? d[2] : d[0]) + shfl_xor_d(a ? d[0] : d[2], LPR / 2);
  const double x1 = (a ? d[3] : d[1]) + shfl_xor_d(a ? d[1] : d[3], LPR / 2);
  double y = (b ? x1 : x0) + shfl_xor_d(b ? x0 : x1, LPR / 4);
#pragma unroll
  for (int mask = LPR / 8; mask >= 1; mask >>= 1) y += shfl_xor_d(y, mask);
  const double mine = exp(y * scale - m);
#pragma unroll
  for (int u = 0; u < UN; ++u) w[u] = __shfl_sync(FULLMASK, mine, (u >> 1) * (LPR / 2) + (u & 1) * (LPR / 4), LPR);
}
constexpr int WPT = 8;                 // walk positions (or tokens) per thread and round of the list extension

__device__ __forceinline__ int ceil_sat(double x) {
  if (!isfinite(x) || x >= 2147483647.0) return 2147483647;
  return (int)ceil(x);
}
__device__ __forceinline__ int block_scan_reg(int val, int* wtot, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = val;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(FULLMASK, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) wtot[warp] = incl;
  __syncthreads();
  int before = 0;
  total = 0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) {
    const int t = wtot[w];
    if (w < warp) before += t;
    total += t;
  }
  __syncthreads();
  return before + incl - val;
}

// CTAs that share `rows` rows: a share of less than stat_rows does not pay for a CTA's fixed costs
__device__ __forceinline__ int stat_ctas(int rows, int most, int share) { return min(most, max(1, (rows + share - 1) / share)); }

// I_dyn as a list: budgets beyond what the known positions serve (unusual: saturated budgets), and for the debug buffer
__device__ __noinline__ void list_sample(const Prob& p, int b, int h, int bh, int bfin, int* misc) {
  const HeadMeta mt = ld_meta(p.meta + bh);
  const int tid = threadIdx.x, n_s = mt.n_s, b0 = mt.b0;
  int* dl = p.dyn_idx + (long long)bh * 3 * p.npad;
  if (bfin > 0) {
    __shared__ unsigned rkeys[8];
    if (tid < 2) walk_keys(p, b, h, 1, tid, rkeys);
    __syncthreads();
    const int s0 = mt.s0, l_start = mt.l_start;
    const int* vt = p.vtab + (long long)bh * VATTN_BANDCAP;
    const float* sc = p.scores + (long long)bh * p.npad;
    const unsigned* gbitmap = p.bitmap + (long long)bh * p.nwords;
    const bool whole = bfin >= n_s;                    // every residual token, in token order
    const Walk wk = make_walk(rkeys, l_start - s0);
    // the walk's laid-out entries are read, not computed again (522 -> 438 us per step of 32 heads x 131,071 tokens, a tenth of
    // them top-k; 1,165 -> 763 at 64 x 65,536 with nearly all of them read)
    const int W1 = walk_region(dyn_listed_want(p, n_s, b0), n_s, l_start - s0, mt.kk);
    const int* wt = p.walk_tok + ((long long)bh * 4 + 2) * p.npad;
    // (the inner loop's parameters in registers: the function gets them by reference, and the list's stores might change what
    // that refers to; 340 -> 288 us per step at 16 heads x 40,000 tokens, all of them sampled from a list)
    const int* bt = p.bt + (long long)b * p.max_blocks;
    const int blocks = p.num_blocks, npad = p.npad;
    const unsigned row_pg = p.row_pg, row_tk = p.row_tk;
    int have = 0;
    int cur = whole ? s0 : 0;
    const int end = whole ? l_start : (l_start - s0);
#pragma unroll 1
    while (have < bfin && cur < end) {
      int tokc[WPT];
      int nres = 0;
#pragma unroll
      for (int q_ = 0; q_ < WPT; ++q_) {
        tokc[q_] = -1;
        const int x = cur + tid * WPT + q_;
        if (x < end) {
          const bool laid = !whole && x < W1;          // (an entry of the array: marked if it is a member)
          const int tok = whole ? x : laid ? __ldcg(wt + x) : s0 + walk_at(wk, x);
          if (laid ? tok >= 0 : !in_topk(mt, vt, gbitmap, tok, __ldg(sc + tok))) { tokc[q_] = tok; ++nres; }
        }
      }
      int tot1;
      int rank = have + block_scan_reg(nres, misc, tot1);
#pragma unroll
      for (int q_ = 0; q_ < WPT; ++q_) {
        if (tokc[q_] >= 0) {
          if (rank < bfin) {
            int pg = bt[tokc[q_] >> 4];
            if ((unsigned)pg >= (unsigned)blocks) pg = checked_page(p, pg);
            dl[rank] = tokc[q_];
            dl[npad + rank] = row_of(row_pg, row_tk, pg, tokc[q_]);
          }
          ++rank;
        }
      }
      have += tot1;
      cur += NT * WPT;
    }
  }
  __syncthreads();
  if (p.dbg.dyn_idx) {
    int* dbg = p.dbg.dyn_idx + (long long)bh * p.max_seq_len;
    for (int i = tid; i < bfin; i += NT) dbg[i] = __ldcg(dl + i);
  }
}

// The least J with bfin unmarked positions below it, for budgets beyond the walk array and more members of I_t out there than
// the threads hold in registers (see head_budget): every step reads the positions again.
__device__ __noinline__ int far_prefix(int bfin, const int* near, int n_near, const int* far, int n_far, int most, int* cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int turn = 0;
  auto marked_below = [&](int Jq) {                        // (uniform over the CTA)
    int c = 0;
    for (int i = threadIdx.x; i < n_near; i += NT) c += __ldcg(near + i) < Jq;
#pragma unroll 8
    for (int i = threadIdx.x; i < n_far; i += NT) c += __ldcg(far + i) < Jq;
    c = __reduce_add_sync(FULLMASK, c);
    if (lane == 0) cnt[turn * NWARP + warp] = c;
    __syncthreads();
    int t = 0;
#pragma unroll
    for (int w = 0; w < NWARP; ++w) t += cnt[turn * NWARP + w];
    turn ^= 1;
    return t;
  };
  int J = bfin;
  for (int it = 0; it < 8; ++it) {
    const int c = marked_below(J);
    if (bfin + c == J) return J;
    J = bfin + c;
  }
  int hi = most, lo = min(J, hi);
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (mid - marked_below(mid) >= bfin) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// Budget of head bh from the partials of its S0 + S1 CTAs, by the last of them.  It stands between the rows and the
// gather of every head, so it is a short chain: everything it reads is requested at once (one round trip), thread e
// adds element e of both kinds in split order, warp k the k-th scalar sum, one barrier, and every warp evaluates the
// budgets for itself (no broadcast).  What does not depend on the rows is computed elsewhere: coefficients on the
// host, pre[0..2] = n_s / b0, 1 / b0, 1 / (b0 - 1) before the CTA's waits.  scal: 16 doubles and 2 NWARP ints of shared memory.
// (7 us from a head's last row to its published budget before, one head of 1,024 tokens.)  Inlined into the kernel, so that
// the parameters are constants of the launch: as a function of its own it read each of them through memory, and the chain
// took 5.0 instead of 3.8 us at 32 heads x 32,768 tokens; only the list is one.
// part(kind, s, e): element e of partial s of a kind; piv(e): the pivot.  lead: this CTA reports (status, introspection).
struct HeadBudget {
  GMeta g;                 // what the gather needs
  double det, det_den;     // thread e: element e of N_f; D_f (with the base sample's share where that is folded in)
};
template <int D, class Part, class Piv>
__device__ __forceinline__ HeadBudget head_budget(const Prob& p, int bh, int S0, int S1, const double* pre, double* scal, bool lead, Part part, Piv piv) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const HeadMeta mt = ld_meta(p.meta + bh);
  // the marked positions of the final sample's walk array, eight per thread (what lies behind the last one is ignored)
  const int* hd = p.hole_pos + (long long)bh * VATTN_BANDCAP;
  static_assert(VATTN_BANDCAP == 8 * NT, "eight positions per thread");
  int hp[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) hp[i] = __ldcg(hd + i * NT + tid);
  // scalar sums: kind 0 (deterministic rows): D_f; kind 1 (base-sample rows): Sw, Sww, Srr
  double sv = 0.0;
  if (lane < (warp == 0 ? S0 : S1)) sv = part(warp == 0 ? 0 : 1, lane, D + (warp == 0 ? 0 : warp - 1));
  double a0 = 0.0, a1 = 0.0, pv = 0.0;
  const double pvD = piv(D);
  if (tid < D) {
    pv = piv(tid);
#pragma unroll 1
    for (int s0 = 0; s0 < MAXS; s0 += 8) {             // eight of either kind in flight
      if (s0 >= S0 && s0 >= S1) break;
      double v0[8], v1[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        v0[i] = s0 + i < S0 ? part(0, s0 + i, tid) : 0.0;
        v1[i] = s0 + i < S1 ? part(1, s0 + i, tid) : 0.0;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) { a0 += v0[i]; a1 += v1[i]; }
    }
  }
  const int n_s = mt.n_s, b0 = mt.b0;
  const double ratio = pre[0], rb0 = pre[1], rb1 = pre[2], db0 = (double)b0;
  const double c1 = lane < 17 ? p.c1[lane] : 0.0, c2 = lane < 17 ? p.c2[lane] : 0.0;      // lane's coefficients of A and B
  const double pivD = b0 > 0 ? pvD : 0.0;              // (the pivot the base-row CTAs used: all of them computed the same numbers)
  if (b0 <= 0) pv = 0.0;
  const double nh = a0 + ratio * (a1 + db0 * pv);
  double nn = nh * nh, sr2 = a1 * a1;                  // |N_hat|^2 and sum_j (sum_i r'_ij)^2
#pragma unroll
  for (int mask = 16; mask >= 1; mask >>= 1) {
    nn += __shfl_xor_sync(FULLMASK, nn, mask);
    sr2 += __shfl_xor_sync(FULLMASK, sr2, mask);
    if (mask < MAXS) sv += __shfl_xor_sync(FULLMASK, sv, mask);
  }
  static_assert(MAXS == 16, "sv sums 16 lanes");
  if (lane == 0) { scal[warp] = sv; scal[4 + warp] = nn; scal[8 + warp] = sr2; }
  __syncthreads();
  const double Dfv = scal[0], Swv = scal[1], Swwv = scal[2], Srrv = scal[3];
  nn = (scal[4] + scal[5]) + (scal[6] + scal[7]);
  sr2 = (scal[8] + scal[9]) + (scal[10] + scal[11]);
  double sigma2 = 0.0, trace = 0.0, Dhat = Dfv;
  int bD = 0, bN = 0, bS = 0, bfin = 0;
  if (n_s > 0) {
    // lane 0: the denominator chain A = n_s sigma / D_hat, lane 1: the numerator chain B = n_s sqrt(Tr) / |N_hat|,
    // both as n_s sqrt(variance / squared norm): one division and one square root deep
    const double sq = lane == 0 ? Swwv : Srrv, lin2 = lane == 0 ? Swv * Swv : sr2;
    double var = 0.0;
    if (b0 >= 2) var = fmax(0.0, (sq - lin2 * rb0) * rb1);
    Dhat = Dfv + ratio * (Swv + db0 * pivD);
    const double den2 = lane == 0 ? Dhat * Dhat : nn;
    const double ab = (double)n_s * sqrt(var / den2);
    const double A = __shfl_sync(FULLMASK, ab, 0), Bn = __shfl_sync(FULLMASK, ab, 1);
    sigma2 = __shfl_sync(FULLMASK, var, 0);
    trace = __shfl_sync(FULLMASK, var, 1);
    // lanes 0..14: the split points of b_SDPA; lane 15: b_D; lane 16: b_N (one body: (c1 A + c2 B)^2)
    const double x = c1 * A + c2 * Bn;
    const double x2 = lane <= 16 ? x * x : CUDART_INF;
    const bool nan = __any_sync(FULLMASK, lane < 15 && x2 != x2);
    double mn = lane < 15 ? x2 : CUDART_INF;
#pragma unroll
    for (int mask = 8; mask >= 1; mask >>= 1) mn = fmin(mn, __shfl_xor_sync(FULLMASK, mn, mask));
    const double b_D = __shfl_sync(FULLMASK, x2, 15), b_N = __shfl_sync(FULLMASK, x2, 16);
    const double b_S = nan ? CUDART_NAN : __shfl_sync(FULLMASK, mn, 0);
    bD = ceil_sat(b_D); bN = ceil_sat(b_N); bS = ceil_sat(b_S);
    const double bx = p.mode == 1 ? b_D : (p.mode == 2 ? b_N : b_S);
    if (p.force_budget >= 0) bfin = min(p.force_budget, n_s);
    else {
      if (!isfinite(bx) && tid == 0 && lead) atomicOr(p.status, VATTN_STATUS_NONFINITE);
      bfin = min(max(ceil_sat(bx), b0), n_s);
    }
  }
  if (tid == 0 && lead) {
    if (p.dbg.dyn_cnt) p.dbg.dyn_cnt[bh] = bfin;
    if (p.dbg.budgets) {
      int* o = p.dbg.budgets + bh * 4;
      o[0] = bD; o[1] = bN; o[2] = bS; o[3] = bfin;
    }
    if (p.dbg.stats) {
      double* o = p.dbg.stats + bh * 8;
      o[0] = Dfv; o[1] = sigma2; o[2] = trace; o[3] = Dhat; o[4] = sqrt(nn); o[5] = (double)n_s; o[6] = (double)b0;
      o[7] = (double)mt.m;
    }
  }
  // I_dyn = the unmarked entries among the first J of the final sample's walk, J = bfin + the marked positions below J:
  // the least fixed point of that map, reached in a few steps in the usual case; with nearly every position marked the
  // steps are as short as the runs of marked positions, so after eight a bisection takes over.  All threads count.
  // (Budgets beyond what the known positions serve take a list: list_sample.)
  const bool listed = bfin > mt.dyn_listed;
  int J = bfin, start = 0;
  if (!listed && bfin >= n_s) J = mt.l_start - mt.s0;      // the whole residual: every middle token, in token order
  else if (!listed) {
    const int nholes = min(max(mt.holes1, 0), VATTN_BANDCAP), nholes2 = min(max(mt.holes2, 0), p.npad);
    const int* hd2 = p.dyn_idx + ((long long)bh * 3 + 2) * p.npad;
    const bool far = bfin > mt.dyn_J - nholes;             // reaches beyond the walk array: the members there count too
    int hf[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i * NT + tid >= nholes) hp[i] = 0x7FFFFFFF;
      hf[i] = far && i * NT + tid < nholes2 ? __ldcg(hd2 + i * NT + tid) : 0x7FFFFFFF;
    }
    int* cnt = reinterpret_cast<int*>(scal + 16);          // [2][NWARP], taken in turn
    int turn = 0;
    auto marked_below = [&](int Jq) {                      // (uniform over the CTA)
      int c = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) c += (hp[i] < Jq) + (hf[i] < Jq);
      c = __reduce_add_sync(FULLMASK, c);
      if (lane == 0) cnt[turn * NWARP + warp] = c;
      __syncthreads();
      int t = 0;
#pragma unroll
      for (int w = 0; w < NWARP; ++w) t += cnt[turn * NWARP + w];
      turn ^= 1;
      return t;
    };
    if (far && nholes2 > 8 * NT) J = far_prefix(bfin, hd, nholes, hd2, nholes2, mt.l_start - mt.s0, cnt);
    else {
      bool conv = false;
      for (int it = 0; it < 8; ++it) {
        const int c = marked_below(J);
        if (bfin + c == J) { conv = true; break; }
        J = bfin + c;
      }
      if (!conv) {
        int hi_ = far ? mt.l_start - mt.s0 : mt.dyn_J, lo_ = min(J, hi_);
        while (lo_ < hi_) {
          const int mid = (lo_ + hi_) >> 1;
          if (mid - marked_below(mid) >= bfin) hi_ = mid; else lo_ = mid + 1;
        }
        J = lo_;
      }
    }
    // nested samples: the base sample's rows are the first b0 rows of I_dyn and their sums are known here (in fp64, from
    // rescored weights): they are folded into the deterministic sums (scaled like the sample), and the gather kernel
    // starts behind them.  Not for lists, nor when the whole residual is visited in token order.
    if (p.nested_base && b0 > 0 && mt.base_J <= J) start = mt.base_J;
  }
  const double f = (start > 0) ? (double)n_s / (double)bfin : 0.0;
  return HeadBudget{GMeta{bfin, n_s, mt.m, 1, J, listed ? 1 : 0, mt.dyn_J, start}, a0 + (start > 0 ? f * (a1 + db0 * pv) : 0.0),
                    Dfv + (start > 0 ? f * (Swv + db0 * pivD) : 0.0)};
}

// The rows of one CTA: entries [r_begin, r_end) of the head's deterministic rows (sink, I_t, window) or of its base
// sample's walk array.  Leaves the warps' sums in sm.u.part (behind a barrier): det: N_f slice, D_f; base: Sr, Sw, Sww, Srr.
template <typename T, int D, bool SPLIT>
struct StatRows {
  static constexpr int EPL = Elem<T>::EPL, LPR = D / EPL, RPI = 32 / LPR;
  static constexpr int NE = D + 3;
  static constexpr int WB = RPI * UN, CB = NWARP * WB;   // rows per warp and per CTA of a batch
  static_assert(SEC % CB == 0 && CB <= NT, "whole batches per section");
  struct Sm {
    union U {
      uint4 ring[NWARP][2][2][UN][32];      // per lane: two batches of K and of V slices
      double part[NWARP][NE];               // the warps' sums, when the rows are done
      __device__ U() {}
    } u;
    alignas(16) int idx[SEC];               // row indices of the section
    int cell[SEC / 32];
    double piv[D + 1];
    double pivT[D];                         // the pivot's w*V, element-major per lane: pivT[e * LPR + j]
    double qT[D];                           // q (times Q_SCALE), likewise: read where it is used instead of living in 16 registers
    __device__ Sm() {}
  };
  // q in fp64 to shared memory (one warp; the caller's barrier)
  static __device__ __forceinline__ void load_q(const Prob& p, Sm& sm, int b, int h) {
    const int lane = threadIdx.x & 31, rsub = lane / LPR, j = lane % LPR;
    if (threadIdx.x < 32 && rsub == 0) {
      float qf[EPL];
      Elem<T>::load(reinterpret_cast<const T*>(p.q) + q_row(p, b, h) + j * EPL, qf);
#pragma unroll
      for (int e = 0; e < EPL; ++e) sm.qT[e * LPR + j] = (double)qf[e] * Q_SCALE;
    }
  }
  static __device__ __forceinline__ void run(const Prob& p, Sm& sm, int bh, int g, bool base_cta, bool odd, int word_piv, float m_f, int r_begin, int r_end) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double m = (double)m_f, scale = (double)p.scale;
    const int rsub = lane / LPR, j = lane % LPR;
    const int first = warp * WB + rsub * UN;                 // this row group's first row of a batch
    // entries: row indices (and, for the base sample, tokens: a marked entry, token -1, is a member of I_t and not a sample)
    const int* etok = p.walk_tok + (long long)bh * 4 * p.npad;
    const int* erow = base_cta ? etok + p.npad : p.topk_idx + (long long)bh * 2 * p.npad + p.npad;
    const char* kb = head_rows<T>(p, p.kc, g) + j * 16;
    const char* vb = head_rows<T>(p, p.vc, g) + j * 16;

    const double* qs = sm.qT + j;

    double acc[EPL], s1 = 0.0, s2 = 0.0, s3 = 0.0;           // det: N_f slice, D_f;  base: Sr slice, Sw, Sww, Srr
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.0;

    // The CTA's entries are staged in sections: row indices to shared memory, without the marked ones (members of I_t are
    // no samples).  Then every warp streams its rows, WB at a time: each lane copies its 16 bytes of K and V rows into
    // slots of its own (asynchronous copies, two batches of K and of V in flight; nothing to synchronise), so the
    // fp64 arithmetic of one batch hides the round trips of the next two without holding their rows in registers.
    double cw = 0.0;
    if (base_cta && r_begin < r_end) {
      // the pivot (the first base-sample row): every CTA of the head computes the same numbers
      uint4 pk[UN];
      pk[0] = __ldg(reinterpret_cast<const uint4*>(row_at<SPLIT>(p, kb, word_piv)));
      const uint4 pv = __ldg(reinterpret_cast<const uint4*>(row_at<SPLIT>(p, vb, word_piv)));
#pragma unroll
      for (int u = 1; u < UN; ++u) pk[u] = pk[0];
      double w4[UN];
      weights64<T, D>(qs, pk, odd, scale, m, j, w4);
      cw = w4[0];
      if (warp == 0 && rsub == 0) {
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
          const double c = cw * (double)slice_elem<T>(pv, e);
          sm.piv[j * EPL + e] = c;
          sm.pivT[e * LPR + j] = c;
        }
        if (j == 0) sm.piv[D] = cw;
      }
    }
#pragma unroll 1
    for (int x0 = r_begin; x0 < r_end; x0 += SEC) {
      const int cnt = min(SEC, r_end - x0);
      __syncthreads();                                       // the section before this one has been used (and pivT written)
      int rows = cnt;                                        // rows that count
      if (!base_cta) {
#pragma unroll
        for (int i = 0; i < SEC / NT; ++i) sm.idx[i * NT + tid] = __ldcg(erow + x0 + min(i * NT + tid, cnt - 1));
      } else {
        int row[SEC / NT];
        unsigned on[SEC / NT];
#pragma unroll
        for (int i = 0; i < SEC / NT; ++i) {
          const int x = x0 + min(i * NT + tid, cnt - 1);
          row[i] = __ldcg(erow + x);
          on[i] = (unsigned)(i * NT + tid < cnt && __ldcg(etok + x) >= 0);
        }
#pragma unroll
        for (int i = 0; i < SEC / NT; ++i) {
          on[i] = __ballot_sync(FULLMASK, on[i] != 0u);
          if (lane == 0) sm.cell[i * NWARP + warp] = __popc(on[i]);
        }
        __syncthreads();
        int before[SEC / NT];
        rows = 0;
#pragma unroll
        for (int c = 0; c < SEC / 32; ++c) {
          if (c % NWARP == warp) before[c / NWARP] = rows;
          rows += sm.cell[c];
        }
#pragma unroll
        for (int i = 0; i < SEC / NT; ++i)
          if ((on[i] >> lane) & 1u) sm.idx[before[i] + __popc(on[i] & ((1u << lane) - 1u))] = row[i];
        if (tid < CB && rows + tid < SEC) sm.idx[rows + tid] = word_piv;      // (padding of the last batch: a real row)
      }
      __syncthreads();
      const int nbat = (rows + CB - 1) / CB;
      auto issue = [&](int k, int kv, const char* base) {
        if (k < nbat) {
          const int4 id = *reinterpret_cast<const int4*>(sm.idx + k * CB + first);
          uint4 (&dst)[UN][32] = sm.u.ring[warp][k & 1][kv];
          cp_async16(&dst[0][lane], row_at<SPLIT>(p, base, id.x));
          cp_async16(&dst[1][lane], row_at<SPLIT>(p, base, id.y));
          cp_async16(&dst[2][lane], row_at<SPLIT>(p, base, id.z));
          cp_async16(&dst[3][lane], row_at<SPLIT>(p, base, id.w));
        }
        cp_async_commit();
      };
      issue(0, 0, kb); issue(0, 1, vb); issue(1, 0, kb); issue(1, 1, vb);
#pragma unroll 1
      for (int k = 0; k < nbat; ++k) {
        double w[UN];
        uint4 r[UN];
        cp_async_wait<3>();                                  // K of batch k
#pragma unroll
        for (int u = 0; u < UN; ++u) r[u] = sm.u.ring[warp][k & 1][0][u][lane];
        weights64<T, D>(qs, r, odd, scale, m, j, w);
        issue(k + 2, 0, kb);
        cp_async_wait<3>();                                  // V of batch k
#pragma unroll
        for (int u = 0; u < UN; ++u) r[u] = sm.u.ring[warp][k & 1][1][u][lane];
        const int left = rows - (k * CB + first);            // rows of this group that exist (4 but at the end)
        if (!base_cta) {
          if (left < UN) {
#pragma unroll
            for (int u = 0; u < UN; ++u) if (u >= left) { w[u] = 0.0; r[u] = make_uint4(0u, 0u, 0u, 0u); }
          }
#pragma unroll
          for (int u = 0; u < UN; ++u) s1 += w[u];
#pragma unroll
          for (int e = 0; e < EPL; ++e) {
#pragma unroll
            for (int u = 0; u < UN; ++u) acc[e] = fma(w[u], (double)slice_elem<T>(r[u], e), acc[e]);
          }
        } else if (left >= UN) {
#pragma unroll
          for (int u = 0; u < UN; ++u) { const double dw = w[u] - cw; s1 += dw; s2 = fma(dw, dw, s2); }
#pragma unroll
          for (int e = 0; e < EPL; ++e) {
            const double c = sm.pivT[e * LPR + j];
#pragma unroll
            for (int u = 0; u < UN; ++u) {
              const double dr = fma(w[u], (double)slice_elem<T>(r[u], e), -c);
              acc[e] += dr;
              s3 = fma(dr, dr, s3);
            }
          }
        } else {
#pragma unroll
          for (int u = 0; u < UN; ++u) {
            if (u < left) {
              const double dw = w[u] - cw;
              s1 += dw;
              s2 = fma(dw, dw, s2);
#pragma unroll
              for (int e = 0; e < EPL; ++e) {
                const double dr = fma(w[u], (double)slice_elem<T>(r[u], e), -sm.pivT[e * LPR + j]);
                acc[e] += dr;
                s3 = fma(dr, dr, s3);
              }
            }
          }
        }
        issue(k + 2, 1, vb);
      }
      cp_async_wait<0>();
    }
    __syncthreads();                                         // (the partials lie over the rows)
    // across the row groups of the warp
#pragma unroll
    for (int mask = LPR; mask < 32; mask <<= 1) {
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] += __shfl_xor_sync(0xFFFFFFFFu, acc[e], mask);
      s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, mask);
      s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, mask);
    }
#pragma unroll
    for (int mask = 1; mask < 32; mask <<= 1) s3 += __shfl_xor_sync(0xFFFFFFFFu, s3, mask);
    if (rsub == 0) {
#pragma unroll
      for (int e = 0; e < EPL; ++e) sm.u.part[warp][j * EPL + e] = acc[e];
      if (j == 0) { sm.u.part[warp][D] = s1; sm.u.part[warp][D + 1] = s2; sm.u.part[warp][D + 2] = s3; }
    }
    __syncthreads();
  }
};

}  // namespace
