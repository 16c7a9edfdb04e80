// Sampled part of the estimator and the final combination (Sec. 4.1 of the paper):
//     N = N_f + (n_s/b) * sum_{I_dyn} w_i V[i],   D = D_f + (n_s/b) * sum_{I_dyn} w_i,   out = N / D
// which is SDPA_{S,p} of Sec. 3 with p = 1 on I_f and p = b/n_s on I_dyn.
//
// (The work on a chunk: rows_gather.cuh.)
// Partials are added in chunk order by the last CTA of the head ("ticket"), so results are reproducible.
//
// Two decompositions:
//  * flat (batch * heads <= 32): budgets differ a lot between heads, so the chunks of all heads form one
//    list that the CTAs walk with a grid stride.  A chunk is a whole number of CTA batches (32 rows of 128 bf16) and a
//    head uses up to 32 chunks (64 to 128 when no more than 16 heads share the grid): the short chunks fill the SMs.
//    (With up to 128 single-batch chunks per head the last finisher needed three dependent rounds of partial loads
//    and long lists overflowed the grid.)
//  * per head (larger problems): grid (16, heads); a head with budget b uses ceil(b / chunk) of its CTAs,
//    chunk = max(least, ceil(b / 16)) rows, the others exit at once.  A CTA's wait, its first round trips, its partial and
//    its ticket cost about as much as a few hundred rows, so `least` grows with the heads that fill the SMs anyway:
//    128 rows up to 160 heads (where 16 x 148 chunks are about two waves), 256 below 512, 512 from there on.
//    (The flat form up to 128 heads: 120.8 instead of 110.6 us per step at 128 heads x 32,768 tokens, 73.7 instead of 67
//    at 96 x 8,192, but 63.4 instead of 68 at 32 x 32,768.  32 CTAs per head: 643 instead of 628 us at 1,024 heads of 4,096
//    to 32,768 tokens, 69 instead of 63 at 256 x 2,049; 8: 393 instead of 389 at 512 x 32,768.  With the heads'
//    first chunks first in dispatch order: 279 instead of 238 us at 1,024 heads, the CTAs that run at the same
//    time then touch the whole cache.)
#include "rows_gather.cuh"

namespace {

constexpr int NT = 128;
constexpr int MAXS = VATTN_GATHER_SLOTS;
constexpr int FLAT_MAX_HEADS = VATTN_GATHER_FLAT_HEADS;
__host__ __device__ constexpr int min_chunk(int heads) { return heads >= 512 ? 512 : heads > 160 ? 256 : 128; }   // per-head decomposition

template <typename T, int D, bool KV, bool SPLIT>
__global__ void __launch_bounds__(NT, VATTN_GATHER_CTAS) k_gather(const __grid_constant__ Prob p) {
  using G = Gather<T, D, KV, SPLIT>;
  __shared__ __align__(16) typename G::Sm sm;
  pdl_trigger();                                        // (the next step's first kernel waits before it touches anything)
  TICK_BEGIN(p, VATTN_K_GATHER);
  const int bh = blockIdx.y, ci = blockIdx.x;      // (the chunks of a head are neighbours: one region of the cache)
  // A head's CTAs start when that head's budget is published (the statistics kernel's last CTA of the head
  // releases a word), not when the whole statistics kernel has completed: heads finish over tens of microseconds
  // at large batch.  Every CTA of the statistics kernel had started before this grid was launched, so the wait
  // cannot starve; it is bounded and falls back to the grid-level wait.  CTAs leave as soon as they are done (a CTA
  // that waited for the grid at its end would hold its slot against the CTAs behind it); one CTA does wait, so
  // that "this grid has completed" implies "the statistics kernel has".
  const bool anchor = bh == 0 && ci == 0;
  const int least = min_chunk(p.B * p.Hq);
  {
    // more chunks than the whole residual would need: nothing to wait for
    const Geo geo = head_geometry(p, head_len(p, bh / p.Hq, bh % p.Hq));
    if (ci > 0 && ci * least >= geo.l_start - geo.s0) return;
  }
  if (threadIdx.x == 0) sm.flag = wait_budget(p, bh, sm.meta, VATTN_WORD_SPINS);
  __syncthreads();
  const bool waited = sm.flag == 0;
  if (waited) {                                         // uniform over the CTA
    pdl_wait();
    if (threadIdx.x == 0) wait_budget(p, bh, sm.meta, 1u);
    __syncthreads();
  }
  const GMeta meta = sm.meta;
  const int nb = meta.n > 0 ? meta.L - meta.start : 0; // entries to visit: [start, L)
  // chunks of at least `least` rows, at most MAXS of them; CTAs beyond the head's chunk count leave at once
  const int chunk = max(least, (nb + MAXS - 1) / MAXS);
  const int nslots = max(1, (nb + chunk - 1) / chunk);
  if (ci < nslots) {
    const int r_begin = meta.start + min(nb, ci * chunk), r_end = min(meta.L, r_begin + chunk);
    G::run(p, sm, bh, meta, r_begin, r_end, ci, nslots);
    TICK_END(p, VATTN_K_GATHER);
  }
  if (anchor && !waited) pdl_wait();
}

template <typename T, int D, bool KV>
__global__ void __launch_bounds__(NT, VATTN_GATHER_CTAS) k_gather_flat(const __grid_constant__ Prob p) {
  using G = Gather<T, D, KV, false>;
  __shared__ __align__(16) typename G::Sm sm;
  pdl_trigger();                                        // (the next step's first kernel waits before it touches anything)
  TICK_BEGIN(p, VATTN_K_GATHER);
  const int tid = threadIdx.x;
  const int BH = p.B * p.Hq;
  // Work unit u = chunk u / BH of head u % BH: neighbouring CTAs (which tend to share an SM) serve different heads,
  // whose chunks differ in length.  A head's units start as soon as its budget is published (a per-head word that
  // the statistics kernel's last CTA of the head releases), not when all budgets are known.  Every CTA of the
  // statistics kernel had started before this grid was launched (programmatic dependent launch), so the wait
  // cannot starve; it is bounded all the same and falls back to the grid-level dependency wait.
  bool waited = false;
  for (int u = blockIdx.x; u < BH * p.gat_slots; u += gridDim.x) {
    const int bh = u % BH, ci = u / BH;
    if (tid == 0) sm.flag = wait_budget(p, bh, sm.meta, waited ? 1u : VATTN_WORD_SPINS);
    __syncthreads();
    if (!waited && sm.flag == 0) {                      // uniform over the CTA
      pdl_wait();
      waited = true;
      if (tid == 0) wait_budget(p, bh, sm.meta, 1u);
      __syncthreads();
    }
    const GMeta meta = sm.meta;
    const int nb = meta.n > 0 ? meta.L - meta.start : 0;       // entries to visit: [start, L)
    const int batches = (nb + G::CB - 1) / G::CB;
    const int rows = G::CB * max(1, (batches + p.gat_slots - 1) / p.gat_slots);
    const int nslots = max(1, (nb + rows - 1) / rows); // a head without samples still writes its output
    if (ci < nslots) {
      const int r_begin = meta.start + min(nb, ci * rows), r_end = min(meta.L, r_begin + rows);
      G::run(p, sm, bh, meta, r_begin, r_end, ci, nslots);
    }
    __syncthreads();
  }
  TICK_END(p, VATTN_K_GATHER);
  if (!waited) pdl_wait();                             // "this grid has completed" implies "the one before has"
}

}  // namespace

template <typename T, int D, bool KV, bool SPLIT>
static cudaError_t launch_per_head(const Prob& p, cudaStream_t s) {
  static size_t have[VATTN_MAXDEV];
  if (p.gat_slots < MAXS) return cudaErrorInvalidValue;
  cudaError_t e = optin_smem(k_gather<T, D, KV, SPLIT>, 0, have, true);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_gather<T, D, KV, SPLIT>, dim3(MAXS, p.B * p.Hq), dim3(NT), 0, s, p);
}
template <typename T, int D, bool KV>
static cudaError_t launch_gather_t(const Prob& p, cudaStream_t s) {
  const int BH = p.B * p.Hq;
  if (p.row_unit == 0u) return launch_per_head<T, D, KV, true>(p, s);      // (rare: no flat variant)
  if (BH > FLAT_MAX_HEADS) return launch_per_head<T, D, KV, false>(p, s);
  // at most gat_slots chunks per head; one wave of CTAs walks them with a grid stride
  static size_t have[VATTN_MAXDEV];
  if (p.gat_slots < VATTN_GATHER_FLAT_SLOTS) return cudaErrorInvalidValue;
  cudaError_t e = optin_smem(k_gather_flat<T, D, KV>, 0, have, true);
  if (e != cudaSuccess) return e;
  const long long most = (long long)BH * p.gat_slots, cap = (long long)VATTN_GATHER_CTAS * device_sm_count();
  return launch_pdl(k_gather_flat<T, D, KV>, dim3((unsigned)(most < cap ? most : cap)), dim3(NT), 0, s, p);
}

cudaError_t launch_gather(const Prob& p, cudaStream_t s) {
  if (p.dtype == VATTN_DTYPE_BF16) {
    if (p.D == 128) return p.gather_kv ? launch_gather_t<bf16_t, 128, true>(p, s) : launch_gather_t<bf16_t, 128, false>(p, s);
    return p.gather_kv ? launch_gather_t<bf16_t, 64, true>(p, s) : launch_gather_t<bf16_t, 64, false>(p, s);
  }
  if (p.D == 128) return p.gather_kv ? launch_gather_t<float, 128, true>(p, s) : launch_gather_t<float, 128, false>(p, s);
  return p.gather_kv ? launch_gather_t<float, 64, true>(p, s) : launch_gather_t<float, 64, false>(p, s);
}
