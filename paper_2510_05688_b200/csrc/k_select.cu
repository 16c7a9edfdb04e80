// Index selection:
//
//   I_t   = the k middle tokens with the largest score, ties to the lowest index (Algorithm 1 line 3, the
//           "oracle top-k" of Sec. 3), as a list with row indices and as a membership rule for the row kernels;
//   I_bs  = uniform-sample of b0 residual tokens (Algorithm 2 line 1): how long a prefix of its walk holds b0 of them;
//   the members of I_t marked in the walk of the final sample (Algorithm 1 line 7).
//
// One CTA per head (256 to 1024 threads).  What bounds it is a chain of block-wide phases of a few hundred ns each and,
// at large batch, how many heads an SM works on at once; so it keeps little in shared memory and in registers, reads
// the scores where they are (L2), and takes few phases:
//   A  a lower bound of the k-th largest score from a sample (every 32nd token): the sample's key of rank
//      rs + 4 sqrt(rs) + 9, rs = k * samples / |M|, four standard deviations below where rank k is expected (one histogram
//      of the top 12 key bits, a second one of the next 12 where the bin is crowded);
//   B  every score is compared with it: the candidates, one and a half times k or so, go to a list in an order that
//      depends on the data only (thread order, one prefix sum);
//   C  the exact rank-k key T among the candidates: a 12-bit histogram, then the few keys of the bin ranked directly.
// The stored scores differ from the exact inner products by at most gamma (a bound from the summation structure
// of the score kernel), so candidates above T + 2 gamma are certainly selected, candidates below T - 2 gamma
// certainly not, and the few in between are rescored in fp64 from their K rows and ranked exactly.
// Anything unusual (fewer than k candidates, too many candidates or near-ties, a k too large for the list, every middle
// token selected) takes the general path: a 32-bit radix select over the whole range with re-read scores, and for more than 1,024 near-ties
// (constant keys, a zero query) an exact 64-bit radix select over fp64 scores.
// (A version with one 1024-thread CTA per head that held all keys in 227 KB of shared memory: 193 us instead of 95 at
// 1,024 heads of 4,096 to 32,768 tokens, 55 instead of 35 at 256 heads of 32,768, 45 instead of 23 at 256 heads of
// 2,049, and beyond 32,768 tokens it only had the general path: 213 us instead of 59 at 32 heads of 131,071.)
//
// Samples.  A sample of c residual tokens is "the entries of a walk that are not in I_t, up to the c-th".  For the
// base sample the CTA looks its walk's first entries up in the scores (requested before the threshold is known),
// marks the members (token = -1; the row index stays valid) and counts: ballots and one scan of 32 counts.  For the final
// sample, whose length is not known yet, each member's walk position is sigma^-1(token): it is marked there and the
// positions are left for the budget.
#include "vattn_internal.cuh"
#include <math_constants.h>



namespace {

constexpr int HB = 4096;               // histogram bins: the sample's top 12 key bits, then the candidates'
constexpr int GBINS = 2048;            // bins of one radix level of the general path
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int SPT = 4;                 // samples per thread, at most
constexpr int PGCAP = 2048;            // physical pages of a head held in shared memory (longer contexts look them up)

struct Sm {
  int* hist;                   // [HB]; after the exact selection: near-tie arrays band_s and vtab
  unsigned* candk;             // [cap] candidate keys
  int* candt;                  // [cap] candidate tokens
  int* pages;                  // [PGCAP] physical pages of the head's context
  int* vtab;                   // [BANDCAP] near-tie tokens, bit 31 = member of I_t
  double* band_s;              // [BANDCAP] exact scores of the near-ties
  int* misc;                   // [16]
  int* wtot, * wtot2;          // [32] each: scratch of the block scans
  int* cell;                   // [32] residual tokens per 32 walk positions
  unsigned* rkeys;             // [2][8] round keys of the two walks
  float* gamma;                // [1]
};
constexpr size_t smem_bytes(int cap) { return HB * 4 + (size_t)cap * 8 + PGCAP * 4 + 64 + 3 * 128 + 64 + 16; }
static_assert(VATTN_BANDCAP * 12 <= HB * 4 && VATTN_SEL_MINCAP * 8 + PGCAP * 4 + HB * 4 >= VATTN_MAX_SEQ / 8 && GBINS <= HB, "overlaid arrays");
__device__ __forceinline__ Sm carve(unsigned char* base, int cap) {
  Sm s;
  s.hist = reinterpret_cast<int*>(base);
  s.band_s = reinterpret_cast<double*>(base);
  s.vtab = reinterpret_cast<int*>(base) + 2 * VATTN_BANDCAP;
  base += HB * 4;
  s.candk = reinterpret_cast<unsigned*>(base);  base += cap * 4;
  s.candt = reinterpret_cast<int*>(base);       base += cap * 4;
  s.pages = reinterpret_cast<int*>(base);       base += PGCAP * 4;
  s.misc = reinterpret_cast<int*>(base);        base += 64;
  s.wtot = reinterpret_cast<int*>(base);        base += 128;
  s.wtot2 = reinterpret_cast<int*>(base);       base += 128;
  s.cell = reinterpret_cast<int*>(base);        base += 128;
  s.rkeys = reinterpret_cast<unsigned*>(base);  base += 64;
  s.gamma = reinterpret_cast<float*>(base);
  return s;
}
// order-reversed key of a score (smaller key = larger score)
__device__ __forceinline__ unsigned key_of(unsigned u) { return u ^ (~((int)u >> 31) & 0x7FFFFFFFu); }

// ---------------------------------------------------------------------------------------------
// block-level scans (NT threads); `wtot`: NWARP words that no thread touches until the caller's next barrier
template <int NT, typename V>
__device__ __forceinline__ V block_scan(V val, V* wtot, V& total) {
  constexpr int NWARP = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  V incl = val;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const V v = __shfl_up_sync(FULL, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) wtot[warp] = incl;
  __syncthreads();
  const V mine = lane < NWARP ? wtot[lane] : (V)0;
  V winc = mine;
#pragma unroll
  for (int off = 1; off < NWARP; off <<= 1) {
    const V v = __shfl_up_sync(FULL, winc, off);
    if (lane >= off) winc += v;
  }
  total = __shfl_sync(FULL, winc, NWARP - 1);
  const V before = __shfl_sync(FULL, winc - mine, warp);
  return before + incl - val;
}
// exclusive prefix sum of a[0..nw) in place; returns the total.
template <int NT>
__device__ __noinline__ int block_excl_scan(int* a, int nw, int* wtot) {
  const int tid = threadIdx.x;
  const int ipt = (nw + NT - 1) / NT;
  const int start = min(nw, tid * ipt), end = min(nw, start + ipt);
  int local = 0;
  for (int i = start; i < end; ++i) local += a[i];
  __syncthreads();                       // the scratch may still be read by an earlier call
  int total;
  int run = block_scan<NT>(local, wtot, total);
  for (int i = start; i < end; ++i) { const int v = a[i]; a[i] = run; run += v; }
  __syncthreads();
  return total;
}
// One level of a selection by histogram: thread t holds bins [t * PER, (t + 1) * PER); the bin of rank `rem` (1-based)
// goes to out[0], the keys before it to out[1], the keys in it to out[2].  Nothing is written when there is no such
// rank.  One barrier inside; the caller's next barrier publishes the result.
template <int NT, int NB>
__device__ __forceinline__ void block_pick(const int* h, int rem, int* wtot, int* out) {
  constexpr int PER = NB / NT;
  const int tid = threadIdx.x;
  int c[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; i += 4) {
    const int4 v = *reinterpret_cast<const int4*>(h + tid * PER + i);
    c[i] = v.x; c[i + 1] = v.y; c[i + 2] = v.z; c[i + 3] = v.w;
  }
#pragma unroll
  for (int i = 0; i < PER; ++i) sum += c[i];
  int total;
  int cum = block_scan<NT>(sum, wtot, total);
  if (cum < rem && rem <= cum + sum) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (rem > cum && rem <= cum + c[i]) { out[0] = tid * PER + i; out[1] = cum; out[2] = c[i]; }
      cum += c[i];
    }
  }
}

// Radix select over the keys `loop` delivers (loop(body) calls body(key) for every key): the rank-th smallest
// key (rank >= 1) and how many keys equal to it are among the rank smallest.
template <int NT, typename KeyT, class Loop>
__device__ KeyT radix_select(const Sm& sm, int rank, int& need_eq, Loop loop) {
  constexpr int KB = (int)sizeof(KeyT) * 8;
  constexpr int NLEV = (KB + 10) / 11;
  const int tid = threadIdx.x;
  KeyT prefix = 0;
  int rem = rank, used = 0;
#pragma unroll 1
  for (int l = 0; l < NLEV; ++l) {
    const int bits = (KB - used) < 11 ? KB - used : 11;   // 11 + 11 + 10 bits, or 5 x 11 + 9
    const int shift = KB - used - bits;
    int* h = sm.hist;
    for (int i = tid; i < GBINS; i += NT) h[i] = 0;
    __syncthreads();
    loop([&](KeyT key) {
      if (l == 0 || (key >> (shift + bits)) == prefix) atomicAdd(&h[(unsigned)(key >> shift) & (unsigned)((1 << bits) - 1)], 1);
    });
    __syncthreads();
    block_pick<NT, GBINS>(h, rem, sm.wtot, sm.misc);
    __syncthreads();
    prefix = (prefix << bits) | (KeyT)(unsigned)sm.misc[0];
    rem -= sm.misc[1];
    used += bits;
    __syncthreads();
  }
  need_eq = rem;
  return prefix;
}

// exact fp64 score of one token, computed by a whole warp from global memory (all lanes return it)
template <typename T, int D>
__device__ __noinline__ double score64_warp(const T* krow, const T* qrow, float scale) {
  const int lane = threadIdx.x & 31;
  double acc = 0.0;
#pragma unroll
  for (int t = 0; t < D / 32; ++t) {
    const int e = lane + 32 * t;
    acc = fma((double)Elem<T>::to_float(qrow[e]), (double)Elem<T>::to_float(krow[e]), acc);
  }
#pragma unroll
  for (int mask = 16; mask >= 1; mask >>= 1) acc += __shfl_xor_sync(FULL, acc, mask);
  return acc * (double)scale;
}
// the same number, by one thread (identical summation tree, so identical bits)
template <typename T, int D>
__device__ __noinline__ double score64_thread(const T* krow, const T* qrow, float scale) {
  double part[32];
  for (int l = 0; l < 32; ++l) {
    double acc = 0.0;
    for (int t = 0; t < D / 32; ++t) {
      const int e = l + 32 * t;
      acc = fma((double)Elem<T>::to_float(qrow[e]), (double)Elem<T>::to_float(krow[e]), acc);
    }
    part[l] = acc;
  }
  for (int mask = 16; mask >= 1; mask >>= 1)
    for (int l = 0; l < mask; ++l) part[l] = part[l] + part[l | mask];
  return part[0] * (double)scale;
}

// "I_t is written and marked in the base sample's walk array" (thread 0, behind a barrier): one cumulative fence, then
// both words of the head, which are stored together
__device__ __forceinline__ void publish(const Prob& p, int bh, unsigned long long word) {
  __threadfence();
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&p.words[bh].sample), "l"(word) : "memory");
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(&p.words[bh].topk), "r"(1u | ((unsigned)(word >> 1) & 2u)) : "memory");
}

// Selection, general case: a radix select over the whole middle range with re-read scores (and, for more near-ties than
// the list holds, an exact one over fp64 scores).  A function of its own: it is seldom taken, and the usual case keeps
// its registers.
struct Found { float hi, lo; int nbt, band_mode, path; };
template <typename T, int D, int NT>
__device__ __noinline__ Found select_general(const Prob& p, unsigned char* smem, int b, int bh, int g, int n, int s0, int l_start, int kk,
                                             const T* qrow, int* tk, int* tkrow, int path) {
  constexpr int NWARP = NT / 32;
  const Sm sm = carve(smem, p.sel_cap);                // (not a reference: the caller's copy stays in registers)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int mlen = l_start - s0;
  const float* sc = p.scores + (long long)bh * p.npad;
  unsigned* gbitmap = p.bitmap + (long long)bh * p.nwords;
  float hi, lo;
  int nbt, band_mode = 0;
  const int PT = (mlen + NT - 1) / NT;               // keys per thread
  // every key of the middle range, in token order per thread: f(u, token, valid, key); uniform trip count, four scores
  // requested at a time
  auto for_slice = [&](auto f) {
#pragma unroll 1
    for (int u0 = 0; u0 < PT; u0 += 1) {
      float s[1];
#pragma unroll
      for (int e = 0; e < 1; ++e) { const int i = s0 + tid + NT * (u0 + e); s[e] = i < l_start ? __ldg(sc + i) : 0.f; }
#pragma unroll
      for (int e = 0; e < 1; ++e) {
        const int u = u0 + e, i = s0 + tid + NT * u;
        if (u >= PT) break;
        const bool v = i < l_start;
        // (a NaN score ranks below everything: the lists stay complete whatever the inputs hold)
        f(u, i, v, v ? ~ord_f32(s[e] == s[e] ? s[e] : -CUDART_INF_F) : 0xFFFFFFFFu);
      }
    }
  };
  __syncthreads();
  const float gamma = sm.gamma[0] >= 0.f ? sm.gamma[0] : 0.f;      // (NaN: non-finite inputs)
  int* cntM = p.sel_cnt + (long long)bh * 2 * (p.npad / 16 + 32);                                 // [PT * NWARP] tokens above the band per (u, warp), then its scan
  int* cntB = cntM + p.npad / 16 + 32;                         // the same for the band
  if (kk == mlen) { hi = -CUDART_INF_F; lo = -CUDART_INF_F; }
  else {
    int need_eq;
    const unsigned Tk = radix_select<NT, unsigned>(sm, kk, need_eq, [&](auto body) {
#pragma unroll 1
      for (int i0 = s0 + tid; i0 < l_start; i0 += 4 * NT) {      // (four scores requested at a time)
        float s[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = i0 + e * NT < l_start ? __ldg(sc + i0 + e * NT) : 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) if (i0 + e * NT < l_start) body(~ord_f32(s[e] == s[e] ? s[e] : -CUDART_INF_F));
      }
    });
    const float Tf = unord_f32(~Tk);
    hi = __fadd_ru(Tf, 2.f * gamma); lo = __fadd_rd(Tf, -2.f * gamma);
  }
  // ---- classify: above the band (ordered counts per (u, warp)), inside it
  for_slice([&](int u, int, bool v, unsigned key) {
    const float s = unord_f32(~key);
    const unsigned bm = __ballot_sync(FULL, v && s > hi), bb = __ballot_sync(FULL, v && !(s > hi) && s >= lo);
    if (lane == 0) { cntM[u * NWARP + warp] = __popc(bm); cntB[u * NWARP + warp] = __popc(bb); }
  });
  __syncthreads();
  const int n_in = block_excl_scan<NT>(cntM, PT * NWARP, sm.wtot);
  nbt = block_excl_scan<NT>(cntB, PT * NWARP, sm.wtot);
  for_slice([&](int u, int i, bool v, unsigned key) {
    const float s = unord_f32(~key);
    const bool mem = v && s > hi, bnd = v && !(s > hi) && s >= lo;
    const unsigned bm = __ballot_sync(FULL, mem), bb = __ballot_sync(FULL, bnd);
    if (mem) {
      const int pos = cntM[u * NWARP + warp] + __popc(bm & lt);
      tk[pos] = i;
      tkrow[pos] = row_of(p, page_of(p, b, i >> 4), i);
    }
    const int posb = cntB[u * NWARP + warp] + __popc(bb & lt);
    if (bnd && posb < VATTN_BANDCAP) sm.vtab[posb] = i;
  });
  __syncthreads();
  const int need = kk - n_in;
  if (nbt <= VATTN_BANDCAP) {
    if (need >= nbt) {
      for (int c = tid; c < nbt; c += NT) sm.vtab[c] |= (int)0x80000000;
    } else {
      path |= 2;
      for (int c = warp; c < nbt; c += NWARP) {
        const double s64 = score64_warp<T, D>(row_ptr<T>(p, p.kc, b, g, sm.vtab[c]), qrow, p.scale);
        if (lane == 0) sm.band_s[c] = s64;
      }
      __syncthreads();
      for (int c = tid; c < nbt; c += NT) {
        const double mine = sm.band_s[c];
        int rank = 0;
        for (int u = 0; u < nbt; ++u) {
          const double o = sm.band_s[u];
          rank += (o > mine) || (o == mine && u < c);
        }
        if (rank < need) sm.vtab[c] |= (int)0x80000000;
      }
    }
    __syncthreads();
    for (int c = tid; c < nbt; c += NT) {            // the band's members behind the tokens above it, ascending too
      const int e = sm.vtab[c];
      if (e < 0) {
        int ord = 0;
        for (int u = 0; u < c; ++u) ord += sm.vtab[u] < 0;
        const int tok = e & 0x7FFFFFFF;
        tk[n_in + ord] = tok;
        tkrow[n_in + ord] = row_of(p, page_of(p, b, tok >> 4), tok);
      }
    }
  } else {
    // too many near-ties for a list: exact fp64 scores as ordered 64-bit keys (smaller key = larger score), an
    // exact radix select of the `need` smallest, equal keys to the lowest indices; verdicts go to the bitmap
    path |= 4;
    band_mode = 1;
    if (tid == 0) atomicOr(p.status, VATTN_STATUS_BAND_OVERFLOW);
    for (int w = tid; w < ((n + 31) >> 5); w += NT) gbitmap[w] = 0u;      // (only this path sets and reads bits)
    unsigned long long* k64 = reinterpret_cast<unsigned long long*>(p.dyn_idx + (long long)bh * 3 * p.npad);
    for_slice([&](int, int i, bool v, unsigned key) {
      const float s = unord_f32(~key);
      if (v && !(s > hi) && s >= lo) k64[i] = ~ord_f64(score64_thread<T, D>(row_ptr<T>(p, p.kc, b, g, i), qrow, p.scale));
    });
    __syncthreads();
    int need_eq;
    const unsigned long long T64 = radix_select<NT, unsigned long long>(sm, need, need_eq, [&](auto body) {
      for_slice([&](int, int i, bool v, unsigned key) {
        const float s = unord_f32(~key);
        if (v && !(s > hi) && s >= lo) body(k64[i]);
      });
    });
    // ordered counts of the keys below T64 and equal to it
    for_slice([&](int u, int i, bool v, unsigned key) {
      const float s = unord_f32(~key);
      const bool bnd = v && !(s > hi) && s >= lo;
      const unsigned long long kx = bnd ? k64[i] : 0ull;
      const unsigned bl = __ballot_sync(FULL, bnd && kx < T64), be = __ballot_sync(FULL, bnd && kx == T64);
      if (lane == 0) { cntM[u * NWARP + warp] = __popc(bl); cntB[u * NWARP + warp] = __popc(be); }
    });
    __syncthreads();
    block_excl_scan<NT>(cntM, PT * NWARP, sm.wtot);
    block_excl_scan<NT>(cntB, PT * NWARP, sm.wtot);
    for_slice([&](int u, int i, bool v, unsigned key) {
      const float s = unord_f32(~key);
      const bool bnd = v && !(s > hi) && s >= lo;
      const unsigned long long kx = bnd ? k64[i] : 0ull;
      const bool isl = bnd && kx < T64, ise = bnd && kx == T64;
      const unsigned bl = __ballot_sync(FULL, isl), be = __ballot_sync(FULL, ise);
      const int lt_before = cntM[u * NWARP + warp] + __popc(bl & lt);
      const int eq_before = cntB[u * NWARP + warp] + __popc(be & lt);
      if (isl || (ise && eq_before < need_eq)) {
        const int pos = n_in + lt_before + min(eq_before, need_eq);
        tk[pos] = i;
        tkrow[pos] = row_of(p, page_of(p, b, i >> 4), i);
        atomicOr(&gbitmap[i >> 5], 1u << (i & 31));
      }
    });
  }
  __threadfence();                                   // the bitmap's bits are read back below through L2
  __syncthreads();
  return Found{hi, lo, nbt, band_mode, path};
}

// ---------------------------------------------------------------------------------------------
template <typename T, int D, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_select(const __grid_constant__ Prob p) {
  constexpr int NWARP = NT / 32;
  constexpr int JQ = 1024 / NT;          // walk positions per thread in a round of the base sample's count
  constexpr int SAMPLES = SPT * NT;      // samples of a head, at most
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bh = blockIdx.x;
  const int b = bh / p.Hq, h = bh % p.Hq, g = h / p.G;
  const unsigned lt = (1u << lane) - 1u;
  const int cap = p.sel_cap;             // candidates the list holds
  const Sm sm = carve(smem_raw, cap);
  TICK_BEGIN(p, VATTN_K_SELECT);

  // ------------------------------------------------------------------ before the wait: the step's inputs only
  const int n = head_len(p, b, h);
  const Geo geo = head_geometry(p, n);
  const int s0 = geo.s0, l_start = geo.l_start, kk = geo.kk, n_s = geo.n_s, b0 = geo.b0;
  const int mlen = l_start - s0;
  const T* qrow = reinterpret_cast<const T*>(p.q) + q_row(p, b, h);
  const float* sc = p.scores + (long long)bh * p.npad;
  int* tk = p.topk_idx + (long long)bh * 2 * p.npad;   // I_t, and the rows of I_f: sink, I_t, window
  int* tkrow = tk + p.npad + s0;                       // (rows of I_t)
  unsigned* gbitmap = p.bitmap + (long long)bh * p.nwords;
  // The words that this step's later kernels count and publish with are cleared here: the step before has completed,
  // and those kernels start only after this one has let them (pdl_trigger).  The fence makes the clears visible first.
  if (tid < (int)(sizeof(HeadWords) / sizeof(uint4))) {
    reinterpret_cast<uint4*>(p.words + bh)[tid] = make_uint4(0u, 0u, 0u, 0u);
    __threadfence();
  }
  __syncthreads();
  if (n == 0) {
    pdl_wait();
    if (bh == 0 && tid == 0) *p.unit_ctr = 0u;
    pdl_trigger();
    if (tid == 0) {
      p.meta[bh] = HeadMeta{};
      if (p.dbg.topk_cnt) p.dbg.topk_cnt[bh] = 0;
      if (p.dbg.base_cnt) p.dbg.base_cnt[bh] = 0;
      if (p.dbg.paths) p.dbg.paths[bh] = 0;
      publish(p, bh, 2ull);
    }
    return;
  }
  const int npg = (n + 15) >> 4;
  const bool pages_cached = npg <= PGCAP;
  for (int i = tid; i < HB / 4; i += NT) reinterpret_cast<int4*>(sm.hist)[i] = make_int4(0, 0, 0, 0);
  if (pages_cached) for (int i = tid; i < npg; i += NT) sm.pages[i] = page_of(p, b, i);
  if (tid < 4) walk_keys(p, b, h, tid >> 1, tid & 1, sm.rkeys + (tid >> 1) * 8);
  if (tid == 0) { sm.misc[13] = 0; sm.misc[14] = mlen; }         // (the base sample's pivot and prefix, should scores be NaN)
  double gfac = 0.0;                                   // (warp NWARP - 1) gamma / max|K|
  if (warp == NWARP - 1) {
    // gamma: bound on |fp32 score - exact score|.  fp32 path: at most 13 roundings (x16 = margin).  bf16
    // tensor-core path: at most 8 accumulation steps of 16 exact products each, every step assumed to lose up
    // to 17 units of 2^-23 of the running magnitude (truncating adder) -> 8*17*2 = 272, taken as 512.
    double sa = 0.0;                                   // sum |q_e|
    for (int e = lane; e < D; e += 32) sa += fabs((double)Elem<T>::to_float(qrow[e]));
#pragma unroll
    for (int mk = 16; mk >= 1; mk >>= 1) sa += __shfl_xor_sync(FULL, sa, mk);
    const double roundings = (p.dtype == VATTN_DTYPE_BF16) ? 512.0 : 16.0;
    gfac = roundings * 5.9604644775390625e-8 * fabs((double)p.scale) * sa * 1.000001;
  }
  int* wa0 = p.walk_tok + (long long)bh * 4 * p.npad;            // base sample's walk: tokens (row indices at + npad)
  int* wa1 = wa0 + 2 * p.npad;                                   // final sample's walk
  const int W0 = walk_region(n_s > 0 ? b0 : 0, n_s, mlen, kk);   // entries the walk kernel wrote
  const int W1 = walk_region(dyn_listed_want(p, n_s, b0), n_s, mlen, kk);
  auto row_idx = [&](int tok) {
    return row_of(p, pages_cached ? sm.pages[tok >> 4] : page_of(p, b, tok >> 4), tok);
  };
  for (int i = tid; i < s0; i += NT) tk[p.npad + i] = row_of(p, page_of(p, b, i >> 4), i);
  for (int i = l_start + tid; i < n; i += NT) tkrow[kk + i - l_start] = row_of(p, page_of(p, b, i >> 4), i);
  __syncthreads();                                     // the histogram is clear

  pdl_wait();                                          // the score pass and the walk are complete
  TICK_BEGIN(p, VATTN_T_TOPK);
  // requested here, wanted later: the largest score, max|K|, the first entries of the base sample's walk (position
  // q * NT + tid) and the row indices of the first 32 of them
  const float m = unord_f32(__ldcg(p.m_ord + bh));
  const unsigned kmax_bits = __ldcg(p.kabsmax + b * p.Hkv + g);
  int jt[JQ];
#pragma unroll
  for (int q_ = 0; q_ < JQ; ++q_) jt[q_] = q_ * NT + tid < W0 ? __ldcg(wa0 + q_ * NT + tid) : -1;
  const int jph = (warp == 0 && lane < W0) ? __ldcg(wa0 + p.npad + lane) : 0;

  int path = 0;
  float hi = CUDART_INF_F, lo = CUDART_INF_F;          // members: s > hi; near-tie band: lo <= s <= hi
  int nbt = 0, band_mode = 0;
  // there is a threshold to find, and the list is likely to hold what the bound lets through (see sel_kmax in api.cu)
  const bool usual = kk > 0 && kk < mlen && (mlen <= cap || kk <= p.sel_kmax);
  bool general = kk > 0 && !usual;
  if (!usual && warp == NWARP - 1 && lane == 0)
    sm.gamma[0] = __double2float_ru(gfac * (double)__uint_as_float(kmax_bits));

  // scores of the base walk's first entries (wanted at the very end)
  float js[JQ];
  auto load_js = [&]() {
#pragma unroll
    for (int q_ = 0; q_ < JQ; ++q_) js[q_] = jt[q_] >= 0 ? __ldg(sc + jt[q_]) : 0.f;
  };
  if (!usual) { pdl_trigger(); load_js(); }
  // ------------------------------------------------------------------ selection, usual case
  if (usual) {
    // ---- the candidates: every middle token whose score is at least the head's bound
    float s_dn = -CUDART_INF_F;
    int ncand = 0;
    // The head's own sample (every 32nd token, or every 64th, ...), one histogram of the top 12 key bits (sign, exponent,
    // three bits of the mantissa) and, where the bin of the wanted rank is crowded, one of the next 12: logits that share an
    // offset fall into one bin.  Then every score is compared, 64 per thread and round.  (Ranking a crowded bin's keys
    // against one another took 106 instead of 72 us per step at 32 heads x 32,768 tokens with logits around 20, and 780 instead
    // of 176 at 131,071.)
    if (mlen > cap) {
      const int stride = sample_stride(n, SAMPLES), ns_all = (n + stride - 1) / stride;
      unsigned kept[SAMPLES / NT];             // (all ones: not a middle token)
#pragma unroll
      for (int e = 0; e < SAMPLES / NT; ++e) {
        const int i = e * NT + tid, tok = sample_token(i, stride);
        kept[e] = i < ns_all && tok >= s0 && tok < l_start ? key_of(__ldg(reinterpret_cast<const unsigned*>(sc) + tok)) : 0xFFFFFFFFu;
      }
#pragma unroll
      for (int e = 0; e < SAMPLES / NT; ++e) if (kept[e] != 0xFFFFFFFFu) atomicAdd(&sm.hist[kept[e] >> 20], 1);
      if (tid == 0) sm.misc[0] = -1;
      __syncthreads();
      constexpr int PER = HB / NT;
      int c[PER], sum = 0, ns;
#pragma unroll
      for (int i = 0; i < PER; i += 4) {
        const int4 v = *reinterpret_cast<const int4*>(sm.hist + tid * PER + i);
        c[i] = v.x; c[i + 1] = v.y; c[i + 2] = v.z; c[i + 3] = v.w;
        *reinterpret_cast<int4*>(sm.hist + tid * PER + i) = make_int4(0, 0, 0, 0);       // (used again below)
      }
#pragma unroll
      for (int i = 0; i < PER; ++i) sum += c[i];
      int cum = block_scan<NT>(sum, sm.wtot, ns);
      const int rank = bound_rank(kk, ns, mlen);
      if (cum < rank && rank <= cum + sum) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
          if (rank > cum && rank <= cum + c[i]) { sm.misc[0] = tid * PER + i; sm.misc[1] = cum; sm.misc[2] = c[i]; }
          cum += c[i];
        }
      }
      __syncthreads();
      const int bin = sm.misc[0], before = sm.misc[1], inb = sm.misc[2];
      if (bin >= 0) {
        unsigned kend_ = ((unsigned)bin << 20) | 0xFFFFFu;
        if (before + inb > rank + (rank >> 3)) {     // (uniform over the CTA) the bin's keys by their next 12 bits
#pragma unroll
          for (int e = 0; e < SAMPLES / NT; ++e)
            if (kept[e] != 0xFFFFFFFFu && (kept[e] >> 20) == (unsigned)bin) atomicAdd(&sm.hist[(kept[e] >> 8) & 0xFFFu], 1);
          __syncthreads();
          block_pick<NT, HB>(sm.hist, rank - before, sm.wtot2, sm.misc + 8);
#pragma unroll
          for (int i = 0; i < PER; i += 4) *reinterpret_cast<int4*>(sm.hist + tid * PER + i) = make_int4(0, 0, 0, 0);
          __syncthreads();
          kend_ = ((unsigned)bin << 20) | ((unsigned)sm.misc[8] << 8) | 0xFFu;
        }
        const float v = unord_f32(~kend_);
        if (v > -CUDART_INF_F) s_dn = v;             // (not for NaN codes)
      }
    }
#pragma unroll 1
    for (int r0 = 0; r0 < l_start; r0 += 64 * NT) {
      unsigned cm[2] = {0u, 0u};                     // word w, bit 4 q + e: token r0 + ((8 w + q) * NT + tid) * 4 + e
      float4 kv[2][4];
      auto fetch = [&](int hf) {
#pragma unroll
        for (int q_ = 0; q_ < 4; ++q_) {
          const int i0 = r0 + ((4 * hf + q_) * NT + tid) * 4;
          kv[hf & 1][q_] = i0 < l_start ? __ldg(reinterpret_cast<const float4*>(sc + i0))
                                        : make_float4(CUDART_NAN_F, CUDART_NAN_F, CUDART_NAN_F, CUDART_NAN_F);
        }
      };
      fetch(0);
#pragma unroll
      for (int hf = 0; hf < 4; ++hf) {
        if (hf < 3) fetch(hf + 1);
        if (r0 + hf * 16 * NT >= l_start) break;     // (uniform)
#pragma unroll
        for (int q_ = 0; q_ < 4; ++q_) {
          const float4 x = kv[hf & 1][q_];
          const int i0 = r0 + ((4 * hf + q_) * NT + tid) * 4;
          unsigned c = (x.x >= s_dn ? 1u : 0u) | (x.y >= s_dn ? 2u : 0u) | (x.z >= s_dn ? 4u : 0u) | (x.w >= s_dn ? 8u : 0u);
          if (i0 < s0 || i0 + 4 > l_start)             // (an edge of the middle range)
            c &= i0 + 3 >= s0 && i0 < l_start ? (15u << max(0, s0 - i0)) & (15u >> max(0, i0 + 4 - l_start)) : 0u;
          cm[hf >> 1] |= c << (16 * (hf & 1) + 4 * q_);
        }
      }
      int tot;
      int cpos = ncand + block_scan<NT>(__popc(cm[0]) + __popc(cm[1]), sm.wtot2, tot);
      ncand += tot;
#pragma unroll 1
      for (int w = 0; w < 2; ++w) {
        const int t0 = r0 + (8 * w * NT + tid) * 4;
        unsigned c = w ? cm[1] : cm[0];
        while (c) {
          const int e = __ffs(c) - 1;
          c &= c - 1;
          if (cpos < cap) sm.candt[cpos] = t0 + (e >> 2) * (4 * NT) + (e & 3);
          ++cpos;
        }
      }
      __syncthreads();
    }
    if (warp == NWARP - 1 && lane == 0) sm.gamma[0] = __double2float_ru(gfac * (double)__uint_as_float(kmax_bits));
    // their keys, relative to that of the largest score (no candidate has a smaller one), and the first level of the
    // exact selection among them; scores of the base walk's first entries
    general = ncand < kk || ncand > cap;
    const unsigned kbase = key_of(__float_as_uint(m)), kend = key_of(__float_as_uint(s_dn));
    const int kbits = 32 - __clz(max(kend - kbase, 1u)), sh1 = max(0, kbits - 12);
    load_js();
#pragma unroll 1
    for (int c0 = tid; c0 < min(ncand, cap); c0 += 8 * NT) {
      unsigned u[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int c = c0 + e * NT;
        u[e] = c < min(ncand, cap) ? __ldg(reinterpret_cast<const unsigned*>(sc) + sm.candt[c]) : 0u;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int c = c0 + e * NT;
        if (c < min(ncand, cap)) {
          // (a key outside [kbase, kend] is a zero of the other sign, which compares equal)
          const unsigned key = max(min(key_of(u[e]), kend), kbase);
          sm.candk[c] = key;
          atomicAdd(&sm.hist[(key - kbase) >> sh1], 1);
        }
      }
    }
    pdl_trigger();                                     // (not earlier: the dependents' prologues would share this SM)
    __syncthreads();
    if (!general) {
      const float gamma = sm.gamma[0];
      // ---- C: the kk-th smallest candidate key.  Levels of 12 bits until at most NT keys share the prefix
      // (the first level leaves a handful), which are then ranked directly.
      int rem = kk, shift = sh1, inbin;
      unsigned pref;
      block_pick<NT, HB>(sm.hist, rem, sm.wtot, sm.misc + 8);
      if (tid == 0) sm.misc[11] = 0;
      __syncthreads();
      pref = (unsigned)sm.misc[8]; rem -= sm.misc[9]; inbin = sm.misc[10];
      while (inbin > NT && shift > 0) {                // (uniform over the CTA)
        const int nsh = max(0, shift - 12), wid = shift - nsh;
        __syncthreads();
        for (int i = tid; i < HB / 4; i += NT) reinterpret_cast<int4*>(sm.hist)[i] = make_int4(0, 0, 0, 0);
        __syncthreads();
        for (int c = tid; c < ncand; c += NT) {
          const unsigned rel = sm.candk[c] - kbase;
          if ((rel >> shift) == pref) atomicAdd(&sm.hist[(rel >> nsh) & ((1u << wid) - 1u)], 1);
        }
        __syncthreads();
        block_pick<NT, HB>(sm.hist, rem, sm.wtot, sm.misc + 8);
        __syncthreads();
        pref = (pref << wid) | (unsigned)sm.misc[8]; rem -= sm.misc[9]; inbin = sm.misc[10];
        shift = nsh;
      }
      unsigned Tk;
      if (shift == 0 || inbin > NT) Tk = kbase + (pref << shift);       // all keys of the bin are equal (shift is 0)
      else {
        unsigned* fin = reinterpret_cast<unsigned*>(sm.hist);           // (the histogram has been read)
        for (int c = tid; c < ncand; c += NT) {
          const unsigned key = sm.candk[c];
          if (((key - kbase) >> shift) == pref) fin[atomicAdd(&sm.misc[11], 1)] = key;
        }
        __syncthreads();
        if (tid < inbin) {
          const unsigned key = fin[tid];
          int less = 0, eq = 0;
          for (int u = 0; u < inbin; ++u) { const unsigned o = fin[u]; less += o < key; eq += o == key; }
          if (less < rem && rem <= less + eq) sm.misc[12] = (int)key;         // (equal keys write the same value)
        }
        __syncthreads();
        Tk = (unsigned)sm.misc[12];
      }
      const float Tf = unord_f32(~Tk);
      hi = __fadd_ru(Tf, 2.f * gamma); lo = __fadd_rd(Tf, -2.f * gamma);
      const bool dn_ok = lo >= s_dn;                   // the band must not reach below the bound (tokens there are not listed)
      // classify the candidates: thread t takes a run of consecutive entries, so ordinals are one prefix sum
      const int per = (ncand + NT - 1) / NT;
      const int c_lo = min(ncand, tid * per), c_hi = min(ncand, c_lo + per);
      int na = 0, nbd = 0;
      for (int c = c_lo; c < c_hi; ++c) {
        const float sv = unord_f32(~sm.candk[c]);
        na += sv > hi; nbd += sv <= hi && sv >= lo;
      }
      unsigned tot;
      const unsigned ex = block_scan<NT>((unsigned)na | ((unsigned)nbd << 16), reinterpret_cast<unsigned*>(sm.wtot2), tot);
      const int n_above = (int)(tot & 0xFFFFu);
      nbt = (int)(tot >> 16);
      general = !dn_ok || nbt > VATTN_BANDCAP;
      if (!general) {
        // those above the band are members; the near-ties go to their list
        int pos = (int)(ex & 0xFFFFu), bo = (int)(ex >> 16);
        for (int c = c_lo; c < c_hi; ++c) {
          const float sv = unord_f32(~sm.candk[c]);
          const int tok = sm.candt[c];
          if (sv > hi) { tk[pos] = tok; tkrow[pos] = row_idx(tok); ++pos; }
          else if (sv >= lo) sm.vtab[bo++] = tok;
        }
        __syncthreads();
        const int need = kk - n_above;         // near-ties that belong to I_t (at least the rank-k key itself)
        const bool all = need >= nbt;
        if (!all) {
          path |= 2;
          for (int c = warp; c < nbt; c += NWARP) {
            const double s64 = score64_warp<T, D>(row_ptr<T>(p, p.kc, b, g, sm.vtab[c]), qrow, p.scale);
            if (lane == 0) sm.band_s[c] = s64;
          }
          __syncthreads();
        }
        for (int c = tid; c < nbt; c += NT) {
          const int tok = sm.vtab[c] & 0x7FFFFFFF;
          int rank = 0;                                // (equal scores: the lower token first)
          if (all) rank = c;
          else {
            const double mine = sm.band_s[c];
            for (int u = 0; u < nbt; ++u) {
              const double o = sm.band_s[u];
              rank += (o > mine) || (o == mine && (sm.vtab[u] & 0x7FFFFFFF) < tok);
            }
          }
          if (rank < need) {
            const int at = n_above + rank;
            tk[at] = tok; tkrow[at] = row_idx(tok);
            sm.vtab[c] = tok | (int)0x80000000;
          }
        }
        path |= mlen <= cap || n <= 32 * SAMPLES ? 1 : 16;       // (16: a bound from fewer tokens than every 32nd)
      }
      __syncthreads();
    }
  }

  if (kk > 0 && general) {
    const Found f = select_general<T, D, NT>(p, smem_raw, b, bh, g, n, s0, l_start, kk, qrow, tk, tkrow, path);
    hi = f.hi; lo = f.lo; nbt = f.nbt; band_mode = f.band_mode; path = f.path;
  }
  if (bh == 0 && tid == 0) *p.unit_ctr = 0u;           // (the score pass is complete: ready for the next step)
  if (band_mode) nbt = 0;                              // (their verdicts are in the bitmap)
  TICK_END(p, VATTN_T_TOPK);
  DBGH(bh, 0);

  // the final walk's round keys for the gather kernel (it extends the walk array for long budgets)
  if (tid < 8) p.wkeys[(long long)bh * 8 + tid] = sm.rkeys[8 + tid];
  // the near-tie list for the budget's list path and the gather kernel
  int* gvtab = p.vtab + (long long)bh * VATTN_BANDCAP;
  for (int c = tid; c < nbt; c += NT) gvtab[c] = sm.vtab[c];

  // ------------------------------------------------------------------ the base sample
  // Its first b0 residual tokens: rounds of 1,024 walk positions (q * NT + tid, so a ballot is 32 consecutive ones),
  // J = the position behind the b0-th entry that is not in I_t.  The walk kernel wrote the entries that are expected
  // to be needed and four standard deviations more; further ones are computed (and written) here.
  int base_J = 0, piv_ph = 0;
  if (n_s > 0) {
    int have = 0;
#pragma unroll 1
    for (int j0 = 0, je; j0 < mlen && have < b0; j0 = je) {
      je = min(j0 + JQ * NT, j0 < W0 ? W0 : mlen);     // (the round [j0, je): entries of the array, or entries beyond it)
      unsigned bal[JQ];
#pragma unroll
      for (int q_ = 0; q_ < JQ; ++q_) {
        const int j = j0 + q_ * NT + tid;
        if (j0 > 0) {
          int tok = -1;
          float sv = 0.f;
          if (j < je) {
            if (j < W0) tok = __ldcg(wa0 + j);
            else {
              tok = s0 + walk_at(make_walk(sm.rkeys + (p.nested_base ? 8 : 0), mlen), j);
              wa0[j] = tok;
              wa0[p.npad + j] = row_idx(tok);
            }
            sv = __ldg(sc + tok);
          }
          jt[q_] = tok; js[q_] = sv;
        }
        const bool mem = jt[q_] >= 0 && (js[q_] > hi || (js[q_] >= lo && near_tie_member(nbt, band_mode, sm.vtab, gbitmap, jt[q_])));
        if (mem) wa0[j] = -1;
        bal[q_] = __ballot_sync(FULL, jt[q_] >= 0 && !mem);
        if (lane == 0) sm.cell[q_ * NWARP + warp] = __popc(bal[q_]);
      }
      __syncthreads();
      // cell c = position range [j0 + 32 c, j0 + 32 c + 32), counted by warp c % NWARP
      const int mine = sm.cell[lane];
      int incl = mine;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) { const int v = __shfl_up_sync(FULL, incl, off); if (lane >= off) incl += v; }
      const int total = __shfl_sync(FULL, incl, 31);
      auto word = [&](int c) {                         // this warp's ballot of cell c
        unsigned w = bal[0];
#pragma unroll
        for (int q_ = 1; q_ < JQ; ++q_) w = c / NWARP == q_ ? bal[q_] : w;
        return w;
      };
      if (have == 0 && total > 0) {                    // the pivot: the first residual token
        const int c = __ffs(__ballot_sync(FULL, mine > 0)) - 1;
        if (warp == c % NWARP) {
          const int bit = __ffs(word(c)) - 1, j = j0 + c * 32 + bit;
          int ph = __shfl_sync(FULL, jph, bit);
          if (lane == 0) {
            if (j0 > 0 || j >= 32) ph = __ldcg(wa0 + p.npad + j);      // (jph: positions 0..31, of the first round)
            sm.misc[13] = ph;
          }
        }
      }
      if (have + total >= b0) {
        const int c = __ffs(__ballot_sync(FULL, have + incl >= b0)) - 1;
        const int before = have + __shfl_sync(FULL, incl - mine, c);
        if (warp == c % NWARP) {
          // the lane whose residual token is the (b0 - before)-th of the word
          const unsigned w = word(c);
          if (((w >> lane) & 1u) && __popc(w & lt) == b0 - before - 1) sm.misc[14] = j0 + c * 32 + lane + 1;
        }
      }
      have += total;
      __syncthreads();
    }
    base_J = sm.misc[14]; piv_ph = sm.misc[13];
  } else __syncthreads();
  // the head's record, then "I_t is written (and marked in the base sample's walk)" for the statistics kernel.  The
  // barrier above orders every thread's writes before thread 0's release, which is cumulative: one fence.
  if (tid == 0) {
    HeadMeta mt = {};
    mt.n = n; mt.s0 = s0; mt.l_start = l_start; mt.kk = kk; mt.n_s = n_s; mt.b0 = b0;
    mt.nbt = nbt; mt.band_mode = band_mode; mt.m = m; mt.hi = hi; mt.lo = lo; mt.path = path; mt.base_J = base_J;
    p.meta[bh] = mt;
    if (p.dbg.topk_cnt) p.dbg.topk_cnt[bh] = kk;
    if (p.dbg.base_cnt) p.dbg.base_cnt[bh] = b0;
    if (p.dbg.paths) p.dbg.paths[bh] = path;
    publish(p, bh, 2ull | ((kmax_bits & 0x7F800000u) == 0x7F800000u ? 4ull : 0ull) | ((unsigned long long)(unsigned)base_J << 3) | ((unsigned long long)(unsigned)piv_ph << 32));
    DBGH(bh, 1);
  }
  // ---- the final walk: marks in its array, positions of all members (read by the budget code and the gather
  //      kernel, which start after this kernel has completed)
  if (n_s > 0) {
    int* cnts = sm.misc;                               // members inside the walk array, beyond it
    int* hp1 = p.hole_pos + (long long)bh * VATTN_BANDCAP;         // positions inside the walk array
    int* hp2 = p.dyn_idx + ((long long)bh * 3 + 2) * p.npad;       // ... and beyond it
    const Walk wk1 = make_walk(sm.rkeys + 8, mlen);
    if (tid < 2) cnts[tid] = 0;
    __syncthreads();
    for (int a = tid; a < kk; a += NT) {
      const int x1 = walk_inv(wk1, __ldcg(tk + a) - s0);
      if (x1 < W1) {
        wa1[x1] = -1;
        const int i1 = atomicAdd(&cnts[0], 1);
        if (i1 < VATTN_BANDCAP) hp1[i1] = x1;
      } else {                                         // (budgets that reach beyond the array need these)
        hp2[atomicAdd(&cnts[1], 1)] = x1;
      }
    }
    __syncthreads();
    if (tid == 0) {
      const int holes1 = cnts[0], holes2 = cnts[1];
      // every member's position is known: any budget can be served as "the non-members among the first J positions"
      // (entries beyond the array are computed by the gather).  More marks in the array than the list holds: none can.
      HeadMeta* gm = p.meta + bh;
      gm->holes1 = min(holes1, VATTN_BANDCAP); gm->holes2 = holes2;
      if (holes1 <= VATTN_BANDCAP) { gm->dyn_J = W1; gm->dyn_listed = n_s; }
    }
  }
  // ---- introspection: I_t ascending (a bitmap of the tokens in shared memory), I_bs in walk order
  if (p.dbg.topk_idx) {
    unsigned* bits = reinterpret_cast<unsigned*>(smem_raw);          // over the histogram, the candidate list and the pages
    const int nw = (n + 31) >> 5;
    __syncthreads();
    for (int w = tid; w < nw; w += NT) bits[w] = 0u;
    __syncthreads();
    for (int a = tid; a < kk; a += NT) { const int tok = __ldcg(tk + a); atomicOr(&bits[tok >> 5], 1u << (tok & 31)); }
    __syncthreads();
    const int per = (nw + NT - 1) / NT, w_lo = min(nw, tid * per), w_hi = min(nw, w_lo + per);
    int c = 0;
    for (int w = w_lo; w < w_hi; ++w) c += __popc(bits[w]);
    int tot1;
    int pos = block_scan<NT>(c, sm.wtot, tot1);
    int* dst = p.dbg.topk_idx + (long long)bh * p.max_seq_len;
    for (int w = w_lo; w < w_hi; ++w)
      for (unsigned v = bits[w]; v; v &= v - 1) dst[pos++] = w * 32 + __ffs(v) - 1;
  }
  if (p.dbg.base_idx && n_s > 0) {
    int* dst = p.dbg.base_idx + (long long)bh * p.max_seq_len;
    int at = 0;
    for (int j0 = 0; j0 < base_J; j0 += NT) {
      const int tok = j0 + tid < base_J ? __ldcg(wa0 + j0 + tid) : -1;
      int tot1;
      __syncthreads();
      const int r = block_scan<NT>(tok >= 0 ? 1 : 0, sm.wtot, tot1);
      if (tok >= 0) dst[at + r] = tok;
      at += tot1;
    }
  }
  TICK_END(p, VATTN_K_SELECT);
}

// The tokens of the first walk positions of both walks, for every head.  sigma depends on (seed, layer, step, batch
// row, head, stream, sequence length) only, not on K or the scores, so it is evaluated here, beside the score pass
// (which is bound by HBM and leaves the integer pipes idle); the selection kernel then only looks tokens up.
// Grid: at most eight CTAs per SM, which share the (head, part) units (a CTA per 1,024 positions that the longest sequence
// could need: most of them found nothing to do on short ones, 15 us for 8 x 2,049 tokens on a 32K plan instead of 7).  A part takes positions [1024 part, + 1024), and every parts * 1024 further, of the head's two
// walks laid end to end.
__global__ void __launch_bounds__(256, 6) k_walk(const __grid_constant__ Prob p, int parts) {
  constexpr int PER = 1024, WT = 256;
  __shared__ unsigned keys[16];
  __shared__ int s_tok[PER];
  pdl_trigger();
  TICK_BEGIN(p, VATTN_K_WALK);
  const int tid = threadIdx.x;
#pragma unroll 1
  for (int u = blockIdx.x; u < p.B * p.Hq * parts; u += gridDim.x) {
    const int bh = u / parts, part = u % parts;
    const int b = bh / p.Hq, h = bh % p.Hq;
    const Geo geo = head_geometry(p, head_len(p, b, h));
    const int mlen = geo.l_start - geo.s0;
    const int J0 = walk_region(geo.b0, geo.n_s, mlen, geo.kk);
    const int J1 = walk_region(dyn_listed_want(p, geo.n_s, geo.b0), geo.n_s, mlen, geo.kk);
    if (geo.n_s <= 0 || part * PER >= J0 + J1) continue;
    __syncthreads();                                   // (the keys of the unit before have been used)
    if (tid < 4) walk_keys(p, b, h, tid >> 1, tid & 1, keys + (tid >> 1) * 8);
    int* out0 = p.walk_tok + (long long)bh * 4 * p.npad;       // [walk][tokens, row indices][npad]
    // Cycle walking repeats the network until the value falls below |M|; with |M| just above a power of two that is two
    // passes on average and four or five for the slowest lane of a warp, so a lane does not wait for its neighbours: it
    // has several positions to do and goes on to its next one as soon as one is finished (one pass per loop iteration).
    // The tokens go to shared memory; their pages are looked up afterwards, four per thread at a time.
#pragma unroll 1
    for (int x_lo = part * PER; x_lo < J0 + J1; x_lo += parts * PER) {
      const int x_hi = min(x_lo + PER, J0 + J1);
      __syncthreads();                                 // (the keys; s_tok of the round before has been read)
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {        // the part of this range in the base walk, then in the final walk
        const int a = which == 0 ? x_lo : max(x_lo, J0), e = which == 0 ? min(x_hi, J0) : x_hi;
        if (a >= e) continue;
        const Walk w = make_walk(keys + ((which == 1 || p.nested_base) ? 8 : 0), mlen);
        const int off = which == 0 ? 0 : J0;
        int x = a + tid;
        unsigned cur = (unsigned)(x - off);
        while (x < e) {
          cur = walk_pass(w, cur);
          if (cur < w.mlen) {
            s_tok[x - x_lo] = geo.s0 + (int)cur;
            x += WT;
            cur = (unsigned)(x - off);
          }
        }
      }
      __syncthreads();
      int tok[PER / WT], pg[PER / WT];
#pragma unroll
      for (int i = 0; i < PER / WT; ++i) tok[i] = x_lo + i * WT + tid < x_hi ? s_tok[i * WT + tid] : geo.s0;
#pragma unroll
      for (int i = 0; i < PER / WT; ++i) pg[i] = page_of(p, b, tok[i] >> 4);
#pragma unroll
      for (int i = 0; i < PER / WT; ++i) {
        const int x = x_lo + i * WT + tid;
        if (x < x_hi) {
          int* dst = out0 + (x < J0 ? x : 2 * p.npad + x - J0);
          dst[0] = tok[i];
          dst[p.npad] = row_of(p, pg[i], tok[i]);
        }
      }
    }
  }
  TICK_END(p, VATTN_K_WALK);
  // This grid does not wait for the score kernel before it, so one of its CTAs does at the end: "this grid has completed"
  // then implies "the score kernel has" for the selection kernel behind it.
  if (blockIdx.x == 0) pdl_wait();
}

}  // namespace

// positions per head: about 1.03 (b0 + 8 b0), or the whole middle range under a forced budget; 1024 positions per CTA
static int walk_ctas(const Prob& p) {
  const double b0max = (double)p.base_rate * (double)p.max_seq_len + 2.0;
  double pos = p.force_budget >= 0 ? (double)p.max_seq_len + 1.1 * b0max : (1.2 + 1.05 * VATTN_WALK_B0S) * b0max + 64.0;
  if (pos > 2.0 * p.max_seq_len) pos = 2.0 * p.max_seq_len;
  const int gx = (int)(pos / 1024.0) + 1;
  return gx > 65535 ? 65535 : gx;
}
cudaError_t launch_walk(const Prob& p, cudaStream_t s) {
  static size_t have[VATTN_MAXDEV];
  cudaError_t e = optin_smem(k_walk, 0, have, true);
  if (e != cudaSuccess) return e;
  const long long heads = (long long)p.B * p.Hq, fit = 8ll * device_sm_count();
  const int parts = (int)max(1ll, min((long long)walk_ctas(p), fit / heads));
  const unsigned grid = (unsigned)min(heads * parts, fit);
  return launch_pdl(k_walk, dim3(grid), dim3(256), 0, s, p, parts);
}

template <typename T, int D, int NT>
static cudaError_t launch_select_n(const Prob& p, cudaStream_t s) {
  static size_t have[VATTN_MAXDEV];
  cudaError_t e = optin_smem(k_select<T, D, NT>, smem_bytes(p.sel_cap), have, true);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_select<T, D, NT>, dim3((unsigned)(p.B * p.Hq)), dim3(NT), smem_bytes(p.sel_cap), s, p);
}
// Threads per CTA: with few heads every SM has at most one and the phases are as long as a thread's share of the
// scores, so long contexts get 1024 (82.6 -> 80.8 us per step at 32 heads of 32,768 tokens) and short ones, where
// barriers weigh more, 512; with more heads than two CTAs of 512 per SM hold, small CTAs overlap better.
int select_threads(const Prob& p) {
  // (a 1,024-thread CTA has its SM to itself: from half the SMs' number of heads on, and unless the context is very long, 512
  // leave room for the row kernel's CTAs: 63.3 -> 61.7 us per step at 96 heads x 8,192 tokens, 128.8 -> 127.0 at 128 x 32,768,
  // but 406 -> 420 at 128 x 131,071)
  const int heads = p.B * p.Hq, sms = device_sm_count();
  if (heads <= sms && p.max_seq_len > (heads <= sms / 2 ? 16384 : 65536)) return 1024;
  return heads <= 2 * sms ? 512 : 256;
}
template <typename T, int D>
static cudaError_t launch_select_t(const Prob& p, cudaStream_t s) {
  switch (select_threads(p)) {
    case 1024: return launch_select_n<T, D, 1024>(p, s);
    case 512: return launch_select_n<T, D, 512>(p, s);
    default: return launch_select_n<T, D, 256>(p, s);
  }
}

cudaError_t launch_select(const Prob& p, cudaStream_t s) {
  if (p.dtype == VATTN_DTYPE_BF16) {
    if (p.D == 128) return launch_select_t<bf16_t, 128>(p, s);
    return launch_select_t<bf16_t, 64>(p, s);
  }
  if (p.D == 128) return launch_select_t<float, 128>(p, s);
  return launch_select_t<float, 64>(p, s);
}
