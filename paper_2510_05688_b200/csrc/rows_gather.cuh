// The gather of a chunk of a head's sampled V rows: shared by the kernels that work on rows (k_gather.cu, k_rows.cu).
//
// A gather of V rows.  Work unit = a chunk of consecutive entries of one head's I_dyn, taken by a CTA; its warps work for
// themselves, without barriers, each on every fourth batch of rows.  A warp takes its entries in stages of 32 (64 for short
// bf16 rows):
//   1  one lane per entry: token and row index (from the walk array or the list; computed for entries beyond the array and
//      for whole-residual budgets), requested while the stage before is streamed; the row indices go to shared memory;
//   2  again one lane per entry, the weight expf(s - m) from the stored fp32 score (no K re-read; members of I_t weigh
//      nothing; the scores are requested three batches ahead) to shared memory;
//   3  the rows: LPR lanes fetch one row with one 16-byte asynchronous copy each into a ring of S batches that belongs to
//      the lane alone (a lane reads what it copied itself, so nothing is synchronised), and add weight times row.  The ring
//      runs on from one stage to the next.
// What bounds it: DRAM and L2 at large batch (scattered rows), dependent round trips (budget, entries, rows, partials) for
// one sequence.
// (Sections of 256 entries per CTA, staged between barriers, drained the ring at the end of each: 619 instead of 594 us per
// step at 1,024 heads of 4,096 to 32,768 tokens, 205.7 instead of 202.5 at 256 x 32,768, 109.3 instead of 106.2 at 128 x
// 32,768.  A version that kept rows in registers, with entries, scores, exps and validity tests handled by the lanes of a
// row, issued about 250 instructions per eight rows and reached half the bandwidth.)
#pragma once
#include "vattn_internal.cuh"
#include <stddef.h>

namespace {

template <typename T, int D, bool KV, bool SPLIT>
struct Gather {
  static constexpr int NT = 128, NWARP = NT / 32;
  static constexpr int UN = 4;                              // rows per batch of a row group
  static constexpr unsigned FULL = 0xFFFFFFFFu;
  static constexpr int EPL = Elem<T>::EPL, LPR = D / EPL, RPI = 32 / LPR, NE = D + 1;
  static constexpr int WB = RPI * UN, CB = NWARP * WB;      // rows per warp and per CTA of a batch
  static constexpr int S = 3;                               // batches in flight
  static constexpr int EN = WB > 8 ? 2 : 1;                 // entries per lane of a stage ...
  static constexpr int NB = 32 * EN / WB;                   // ... which is this many of the warp's batches
  static constexpr int AHEAD = EN == 1 ? 8 : 4;             // entries per lane whose sigma is computed in one go
  static_assert(AHEAD % EN == 0, "whole stages");
  static_assert(NB > S && NB * WB == 32 * EN && LPR >= 8, "a stage is opened after the one before it has its weights; two hand-over levels of the K+V variant");
  union WarpMem {
    uint4 ring[S][UN][32];
    float part[NE];                                         // the warp's sums, when its rows are done
    __device__ WarpMem() {}
  };
  struct Stages {
    alignas(16) int idx[NWARP][2][32 * EN];                 // row indices of two stages
    alignas(16) float w[NWARP][2][32 * EN];                 // weights
    unsigned keys[8];
    HeadMeta mt;
    GMeta meta;
    float den;
    int flag;
    unsigned ahead[NWARP][AHEAD][32];                       // sigma of the next entries beyond the walk array
    __device__ Stages() {}
  };
  // (the rings first: behind the stages their rows cost the kernel 1 % at 1,024 heads)
  struct Rings {
    WarpMem warp[NWARP];
    __device__ Rings() {}
  };
  struct Sm : Rings, Stages {
    __device__ Sm() {}
  };
  // (a user of the stages declares them alone, and a lane reads four row indices or weights as one 16-byte word)
  static_assert(alignof(Stages) >= 16 && offsetof(Stages, idx) % 16 == 0 && offsetof(Stages, w) % 16 == 0, "four indices or weights per read");
  static __device__ __forceinline__ void unpack(const uint4& r, float (&v)[EPL]) {
    if (EPL == 8) {
      v[0] = __uint_as_float(r.x << 16); v[1] = __uint_as_float(r.x & 0xFFFF0000u);
      v[2] = __uint_as_float(r.y << 16); v[3] = __uint_as_float(r.y & 0xFFFF0000u);
      v[4 % EPL] = __uint_as_float(r.z << 16); v[5 % EPL] = __uint_as_float(r.z & 0xFFFF0000u);
      v[6 % EPL] = __uint_as_float(r.w << 16); v[7 % EPL] = __uint_as_float(r.w & 0xFFFF0000u);
    } else {
      v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y); v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
    }
  }

  // The rows of a chunk: this lane's share of the sums to acc and dd.  Where the entries come from is decided outside: with all
  // three in one loop, the tests cost 1 % of a step at 1,024 heads of 4,096 to 32,768 tokens.
  enum { ARRAY, WALK, ALL };                                // the walk array or the list; entries from W1 on computed; every middle token
  template <int KIND>
  static __device__ __forceinline__ void stream(const Prob& p, WarpMem* wm, Stages& sm, int bh, float m, const int* dyn, int W1,
                                                int r_begin, int r_end, bool careful, float (&acc)[EPL], float& dd) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int h = bh % p.Hq, b = bh / p.Hq, g = h / p.G;
    const int* drow = dyn + p.npad;
    const float* sc = p.scores + (long long)bh * p.npad;
    const int rsub = lane / LPR, j = lane % LPR;
    const char* vb = head_rows<T>(p, p.vc, g) + j * 16;
    // Every warp works for itself, without a barrier.  Its share of the chunk (WB of every CB entries) is taken in stages
    // of 32 EN entries: a stage is opened (its row indices go to shared memory, its scores and the next stage's entries are
    // requested) when its first rows are wanted, S batches before its weights are.
    const int nbat = (r_end - r_begin + CB - 1) / CB;
    const int from = careful ? 0 : nbat - 1;                // the first batch whose entries of no weight must not count (see sums)
    int tok_n[EN], row_n[EN];                               // the next stage's entries
    float sc_n[EN];                                         // the open stage's scores
    int tok_o[EN];                                          // ... and tokens (-1: weighs nothing)
    auto entry = [&](int t, int i) { const int at = i * 32 + lane; return r_begin + (t * NB + at / WB) * CB + warp * WB + at % WB; };
    // sigma of a lane's next AHEAD entries.  Cycle walking repeats the network until the value falls below |M|, up to twice on
    // average: a lane goes on to its next entry as soon as one is finished and waits for the warp's slowest once in AHEAD
    // entries.  (Once in every entry: 92 instead of 85 us per step at 17 heads x 33,200 tokens with budgets of 40 base budgets,
    // 160 instead of 148 at 24 x 66,000, 265 instead of 239 at 40 x 66,000; all of a chunk's entries laid out before its rows:
    // 650 instead of 634 at 1,024 heads of 4,096 to 32,768.)
    const int nstages = (nbat + NB - 1) / NB;
    auto far = [&](int t) {
      const Walk wk = make_walk(sm.keys, sm.mt.l_start - sm.mt.s0);
      const int todo = min(AHEAD, (nstages - t) * EN);
      auto pos = [&](int a) { return min(entry(t + a / EN, a % EN), r_end - 1); };
      int a = 0;
      while (a < todo && pos(a) < W1) ++a;                  // (these are in the array)
      unsigned cur = (unsigned)pos(a);
      while (a < todo) {
        cur = walk_pass(wk, cur);
        if (cur < wk.mlen) { sm.ahead[warp][a][lane] = cur; cur = (unsigned)pos(++a); }
      }
      __syncwarp();
    };
    auto load = [&](int t) {
      if (KIND == WALK && t * EN % AHEAD == 0) far(t);
#pragma unroll
      for (int i = 0; i < EN; ++i) {
        const int x = min(entry(t, i), r_end - 1);          // (the padding of the last batch repeats a real row)
        if (KIND == ALL) { tok_n[i] = sm.mt.s0 + x; row_n[i] = row_of(p, page_of(p, b, tok_n[i] >> 4), tok_n[i]); }
        else if (KIND == ARRAY || x < W1) { tok_n[i] = __ldcg(dyn + x); row_n[i] = __ldcg(drow + x); }
        else {
          tok_n[i] = sm.mt.s0 + (int)sm.ahead[warp][(t * EN + i) % AHEAD][lane];
          row_n[i] = table_entry(p, b, tok_n[i] >> 4);      // (looked at when the stage is opened)
        }
      }
    };
    auto open = [&](int t) {
#pragma unroll
      for (int i = 0; i < EN; ++i) {
        if (KIND == WALK && min(entry(t, i), r_end - 1) >= W1) row_n[i] = row_of(p, checked_page(p, row_n[i]), tok_n[i]);
        sm.idx[warp][t & 1][i * 32 + lane] = row_n[i];
        tok_o[i] = entry(t, i) < r_end ? tok_n[i] : -1;
        if (!KV || KIND != ARRAY) sc_n[i] = tok_o[i] >= 0 ? __ldg(sc + tok_o[i]) : 0.f;
      }
      __syncwarp();
      if ((t + 1) * NB < nbat) load(t + 1);
    };
    auto weigh = [&](int t) {                               // the open stage's weights
      if (KV) dots(p, sm, bh, t, nbat);
#pragma unroll
      for (int i = 0; i < EN; ++i) {
        bool on = tok_o[i] >= 0;
        if (on && (KIND == ALL || (KIND == WALK && entry(t, i) >= W1)))       // (computed entries carry no marks)
          on = !in_topk(sm.mt, p.vtab + (long long)bh * VATTN_BANDCAP, p.bitmap + (long long)bh * p.nwords, tok_o[i], sc_n[i]);
        const float w = on ? expf((KV ? sm.w[warp][t & 1][i * 32 + lane] : sc_n[i]) - m) : 0.f;
        sm.w[warp][t & 1][i * 32 + lane] = w;
        dd += w;
      }
      __syncwarp();
    };
    auto issue = [&](int k, int slot_) {                    // batch k into a slot of the ring
      if (k < nbat) {
        const int4 id = *reinterpret_cast<const int4*>(&sm.idx[warp][(k / NB) & 1][(k % NB) * WB + rsub * UN]);
        uint4 (&dst)[UN][32] = wm[warp].ring[slot_];
        cp_async16(&dst[0][lane], row_at<SPLIT>(p, vb, id.x));
        cp_async16(&dst[1][lane], row_at<SPLIT>(p, vb, id.y));
        cp_async16(&dst[2][lane], row_at<SPLIT>(p, vb, id.z));
        cp_async16(&dst[3][lane], row_at<SPLIT>(p, vb, id.w));
      }
      cp_async_commit();
    };
    if (nbat > 0) {
      load(0);
      open(0);
#pragma unroll
      for (int k = 0; k < S; ++k) issue(k, k);
      int slot_ = 0;
#pragma unroll 1
      for (int k = 0; k < nbat; ++k) {
        if (k % NB == 0) weigh(k / NB);
        const float4 w4 = *reinterpret_cast<const float4*>(&sm.w[warp][(k / NB) & 1][(k % NB) * WB + rsub * UN]);
        const float w[UN] = {w4.x, w4.y, w4.z, w4.w};
        cp_async_wait<S - 1>();
        uint4 raw[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) raw[u] = wm[warp].ring[slot_][u][lane];
        if (k >= from) {                                    // (uniform) whatever its row holds
#pragma unroll
          for (int u = 0; u < UN; ++u) if (w[u] == 0.f) raw[u] = make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          float v[EPL];
          unpack(raw[u], v);
#pragma unroll
          for (int e = 0; e < EPL; ++e) acc[e] = fmaf(w[u], v[e], acc[e]);
        }
        if ((k + S) % NB == 0 && k + S < nbat) open((k + S) / NB);
        issue(k + S, slot_);                                // (into the slot that has just been read)
        slot_ = slot_ == S - 1 ? 0 : slot_ + 1;
      }
      cp_async_wait<0>();
    }
  }
  // entries [r_begin, r_end) of head bh: the warps' sums to wm[].part, behind a barrier
  static __device__ __forceinline__ void sums(const Prob& p, WarpMem* wm, Stages& sm, int bh, const GMeta& meta, int r_begin, int r_end) {
    const int tid = threadIdx.x;
    // I_dyn: the unmarked entries of a prefix of the final sample's walk array (a marked entry, token -1, is a
    // member of I_t: its row is fetched like the others and weighs nothing), the head's list, entries beyond the array
    // (sigma; membership in I_t decided from the score like the selection kernel would), or, for a budget equal to the
    // whole residual, every middle token in token order
    const bool ident = !meta.list && meta.b >= meta.n_s && meta.b > 0;
    const int W1 = meta.list ? r_end : ident ? 0 : meta.W1;
    const bool computed = r_end > W1;                       // this chunk has entries that are computed here
    if (computed) {
      if (tid < 8) sm.keys[tid] = __ldcg(p.wkeys + (long long)bh * 8 + tid);
      if (tid == 32) sm.mt = ld_meta(p.meta + bh);
      __syncthreads();
    }
    const int* dyn = meta.list ? p.dyn_idx + (long long)bh * 3 * p.npad : p.walk_tok + ((long long)bh * 4 + 2) * p.npad;
    // Rows of no weight (members of I_t, the last batch's padding) are fetched like the others, and an infinite element of one
    // would make the sum a NaN.  The padding is left out as it comes; where a sum has come out infinite or a NaN, the warp goes
    // over its rows once more without any of them.
    if (!warp_sums(p, wm, sm, bh, meta.m, dyn, W1, computed, ident, r_begin, r_end, false)) again(p, wm, sm, bh, meta.m, dyn, W1, computed, ident, r_begin, r_end);
    __syncthreads();
  }
  // (a function of its own: as a second round of a loop in sums, 638.6 instead of 634.8 us at 1,024 heads)
  static __device__ __noinline__ void again(const Prob& p, WarpMem* wm, Stages& sm, int bh, float m, const int* dyn, int W1, bool computed, bool ident,
                                            int r_begin, int r_end) {
    warp_sums(p, wm, sm, bh, m, dyn, W1, computed, ident, r_begin, r_end, true);
  }
  // one warp's sums to its part; false: one of them is not finite
  static __device__ __forceinline__ bool warp_sums(const Prob& p, WarpMem* wm, Stages& sm, int bh, float m, const int* dyn, int W1, bool computed, bool ident,
                                                   int r_begin, int r_end, bool careful) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rsub = lane / LPR, j = lane % LPR;
    float acc[EPL], dd = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
    if (!computed) stream<ARRAY>(p, wm, sm, bh, m, dyn, W1, r_begin, r_end, careful, acc, dd);
    else if (ident) stream<ALL>(p, wm, sm, bh, m, dyn, W1, r_begin, r_end, careful, acc, dd);
    else stream<WALK>(p, wm, sm, bh, m, dyn, W1, r_begin, r_end, careful, acc, dd);
#pragma unroll
    for (int mask = LPR; mask < 32; mask <<= 1) {
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] += __shfl_xor_sync(FULL, acc[e], mask);
    }
#pragma unroll
    for (int mask = 16; mask >= 1; mask >>= 1) dd += __shfl_xor_sync(FULL, dd, mask);
    bool finite = true;
#pragma unroll
    for (int e = 0; e < EPL; ++e) finite &= (bool)isfinite(acc[e]);
    finite = __all_sync(FULL, finite);
    __syncwarp();                                           // (the warp's sums lie over its rows)
    if (rsub == 0) {
#pragma unroll
      for (int e = 0; e < EPL; ++e) wm[warp].part[j * EPL + e] = acc[e];
      if (j == 0) wm[warp].part[D] = dd;
    }
    __syncwarp();
    return finite;
  }
  // entries [r_begin, r_end) of head bh -> partial `slot`; the last of `nslots` finishers combines
  static __device__ __forceinline__ void run(const Prob& p, Sm& sm, int bh, const GMeta& meta, int r_begin, int r_end, int slot, int nslots) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h = bh % p.Hq, b = bh / p.Hq, g = h / p.G;
    T* out = reinterpret_cast<T*>(p.out) + q_row(p, b, h);
    if (meta.n == 0) {
      if (slot == 0) for (int e = tid; e < D; e += NT) out[e] = Elem<T>::from_float(0.f);
      return;
    }
    sums(p, sm.warp, sm, bh, meta, r_begin, r_end);
    float* gpart = p.gat_part + ((long long)bh * p.gat_slots + slot) * NE;
    for (int e = tid; e < NE; e += NT) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < NWARP; ++w) s += sm.warp[w].part[e];
      gpart[e] = s;
    }
    // (the barrier orders every thread's writes before thread 0's fence, which is cumulative; likewise on the way in)
    __syncthreads();
    if (tid == 0) sm.flag = ticket(&p.words[bh].gather_ticket) == (unsigned)(nslots - 1);
    __syncthreads();
    if (!sm.flag) return;
    if (tid == 0) p.kabsmax[bh / p.Hq * p.Hkv + g] = 0u;      // (the selection has completed: ready for the next step)
    DBGH(bh, 5);

    // last finisher of the head: every thread requests all partials of its element at once (one memory
    // round trip), adds them in slot order, scales by n_s/b and divides
    const int nb = meta.b;
    const double* det = p.det_sums + (long long)bh * (D + 1);
    const double f = (nb > 0) ? (double)meta.n_s / (double)nb : 0.0;
    const float* src0 = p.gat_part + (long long)bh * p.gat_slots * NE;
    float num_s[(D + NT - 1) / NT];
    double det_e[(D + NT - 1) / NT];
    const double det_d = __ldcg(det + D);             // N_f, D_f of the statistics kernel, requested with the partials
#pragma unroll
    for (int it = 0; it < (D + NT - 1) / NT; ++it) det_e[it] = (tid + it * NT < D) ? __ldcg(det + tid + it * NT) : 0.0;
#pragma unroll
    for (int it = 0; it < (D + NT - 1) / NT; ++it) {
      const int e = tid + it * NT;
      float s = 0.f;
      for (int s0 = 0; s0 < nslots; s0 += 32) {       // 32 partials per round trip, added in slot order
        float vv[32];
#pragma unroll
        for (int sp = 0; sp < 32; ++sp) vv[sp] = (s0 + sp < nslots && e < D) ? __ldcg(src0 + (long long)(s0 + sp) * NE + e) : 0.f;
#pragma unroll
        for (int sp = 0; sp < 32; ++sp) s += vv[sp];
      }
      num_s[it] = s;
    }
    if (warp == 0) {                                  // the denominator: lane sp holds slot s0 + sp
      float s = 0.f;
      for (int s0 = 0; s0 < nslots; s0 += 32) {
        const float vd = (s0 + lane < nslots) ? __ldcg(src0 + (long long)(s0 + lane) * NE + D) : 0.f;
#pragma unroll
        for (int sp = 0; sp < 32; ++sp) s += __shfl_sync(FULL, vd, sp);
      }
      if (lane == 0) sm.den = s;
    }
    __syncthreads();
    const double den = det_d + f * (double)sm.den;
#pragma unroll
    for (int it = 0; it < (D + NT - 1) / NT; ++it) {
      const int e = tid + it * NT;
      if (e < D) out[e] = Elem<T>::from_float((float)((det_e[it] + f * (double)num_s[it]) / den));
    }
  }
  // K+V variant: scale <q, K[row]> of a stage's rows to sm.w (what a selector that leaves no scores for the whole
  // context behind would need), from rows in registers; one warp
  static __device__ __forceinline__ void dots(const Prob& p, Stages& sm, int bh, int t, int nbat) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane % LPR, rsub = lane / LPR;
    const int h = bh % p.Hq, b = bh / p.Hq, g = h / p.G;
    const char* kb = head_rows<T>(p, p.kc, g) + j * 16;
    float qf[EPL];
    Elem<T>::load(reinterpret_cast<const T*>(p.q) + q_row(p, b, h) + j * EPL, qf);
    uint4 r[UN];
    auto load = [&](int k) {
      const int4 id = *reinterpret_cast<const int4*>(&sm.idx[warp][t & 1][k * WB + rsub * UN]);
      r[0] = __ldcs(reinterpret_cast<const uint4*>(row_at<SPLIT>(p, kb, id.x)));
      r[1] = __ldcs(reinterpret_cast<const uint4*>(row_at<SPLIT>(p, kb, id.y)));
      r[2] = __ldcs(reinterpret_cast<const uint4*>(row_at<SPLIT>(p, kb, id.z)));
      r[3] = __ldcs(reinterpret_cast<const uint4*>(row_at<SPLIT>(p, kb, id.w)));
    };
    const int batches = min(NB, nbat - t * NB);
    load(0);
#pragma unroll 1
    for (int k = 0; k < batches; ++k) {
      float d[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        float x[EPL];
        unpack(r[u], x);
        d[u] = 0.f;
#pragma unroll
        for (int e = 0; e < EPL; ++e) d[u] = fmaf(qf[e], x[e], d[u]);
      }
      if (k + 1 < batches) load(k + 1);
      // a butterfly that hands rows over while it adds: lane j ends with the product of row own
      const bool a = (j & (LPR / 2)) != 0, c = (j & (LPR / 4)) != 0;
      const float y0 = (a ? d[2] : d[0]) + __shfl_xor_sync(FULL, a ? d[0] : d[2], LPR / 2);
      const float y1 = (a ? d[3] : d[1]) + __shfl_xor_sync(FULL, a ? d[1] : d[3], LPR / 2);
      float y = (c ? y1 : y0) + __shfl_xor_sync(FULL, c ? y0 : y1, LPR / 4);
#pragma unroll
      for (int mask = LPR / 8; mask >= 1; mask >>= 1) y += __shfl_xor_sync(FULL, y, mask);
      if (j % (LPR / 4) == 0) sm.w[warp][t & 1][k * WB + rsub * UN + (a ? 2 : 0) + (c ? 1 : 0)] = p.scale * y;
    }
    __syncwarp();
  }
};

}  // namespace
