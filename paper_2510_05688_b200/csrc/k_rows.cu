// Statistics, budget and gather of a head in one kernel, for few heads.
//
// A cluster of C CTAs serves a head.  Some of them take the deterministic rows, the others the base sample's (rows_stats.cuh);
// behind a cluster barrier every CTA adds the partial sums of all of them out of their shared memory and evaluates the budget
// for itself (the same numbers in the same order, so the same bits); then each gathers its chunk of the sampled V rows
// (rows_gather.cuh), hands its sums to the first CTA's shared memory, and that one, behind a second barrier, divides.
// What bounds it: the chain of memory round trips.  The two kernels it stands for exchange partials and the budget through
// global memory, by fences, tickets and polled words (1.5 to 3 us each: partials to their last finisher twice, the budget to
// the gather); a cluster barrier takes 0.2 us and a read of another CTA's shared memory 0.2 to 0.4.
#include "rows_gather.cuh"
#include "rows_stats.cuh"

namespace {

__device__ __forceinline__ unsigned cluster_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned map_rank(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ double ld_cluster(unsigned addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster(unsigned addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

// CTAS: CTAs per SM.  Four (128 registers) up to 16 heads: 24.6 -> 24.2 us per step at one fp32 head of 1,024 tokens, 35.8 -> 34.9
// at 16 x 4,096; 32 clusters need five (41.7 against 50.6 at 32 fp32 heads of 64 elements).
template <typename T, int D, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) k_rows(const __grid_constant__ Prob p) {
  using R = StatRows<T, D, false>;
  using G = Gather<T, D, false, false>;
  constexpr int NE = D + 3, NG = D + 1, C = VATTN_ROWS_CLUSTER;
  __shared__ typename R::Sm sm;
  __shared__ typename G::Stages stages;
  __shared__ double s_sum[NE];                     // this CTA's partial of the statistics
  __shared__ double s_scal[16 + NWARP];
  __shared__ double s_pre[3];                      // for the budget: n_s / b0, 1 / b0, 1 / (b0 - 1)
  __shared__ unsigned long long s_word;
  __shared__ int s_misc[8];
  // over the rows of the statistics, when their sums have been taken: the gather's rows, and (in the first CTA) the sums that
  // the others hand over
  typename G::WarpMem* wm = reinterpret_cast<typename G::WarpMem*>(&sm.u);
  float* slots = reinterpret_cast<float*>(wm + NWARP);
  static_assert(sizeof(typename G::WarpMem) * NWARP + (C - 1) * NG * sizeof(float) <= sizeof(sm.u), "overlaid arrays");

  const int tid = threadIdx.x;
  const int rank = (int)cluster_rank(), bh = blockIdx.x / C;
  const int b = bh / p.Hq, h = bh % p.Hq, g = h / p.G;
  const int n = head_len(p, b, h);
  const Geo geo = head_geometry(p, n);
  const int s0 = geo.s0, l_start = geo.l_start, kk = geo.kk, b0 = geo.b0;
  const int n_f = s0 + kk + (n - l_start);
  // the CTAs of either kind: a base row costs about a quarter more than a deterministic one
  const int Sd = min(C - 1, max(1, (8 * C * n_f + 4 * n_f + 5 * b0) / max(1, 8 * n_f + 10 * b0)));
  const bool base_cta = rank >= Sd;
  const int split = base_cta ? rank - Sd : rank, S = base_cta ? C - Sd : Sd;
  if (tid == NT - 1) {
    s_pre[0] = b0 > 0 ? (double)geo.n_s / (double)b0 : 0.0;
    s_pre[1] = b0 > 0 ? 1.0 / (double)b0 : 0.0;
    s_pre[2] = b0 > 1 ? 1.0 / (double)(b0 - 1) : 0.0;
  }
  TICK_BEGIN(p, VATTN_K_STATS);
  pdl_trigger();                                   // (the next step's first kernel waits before it touches anything)
  R::load_q(p, sm, b, h);
  // (the words and the bounded wait: as in the statistics kernel)
  HeadWords* hw = p.words + bh;
  if (tid == 0) s_word = base_cta ? wait_word64(&hw->sample, VATTN_WORD_SPINS) : (unsigned long long)wait_word32(&hw->topk, VATTN_WORD_SPINS);
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
  if (base_cta && split == 0) DBGH(bh, 6);
  T* out = reinterpret_cast<T*>(p.out) + q_row(p, b, h);
  if (n == 0) {                                    // an empty row (uniform over the cluster): zeros
    pdl_wait();
    if (rank == 0) {
      for (int e = tid; e < D; e += NT) out[e] = Elem<T>::from_float(0.f);
      if (tid == 0) {
        if (p.dbg.dyn_cnt) p.dbg.dyn_cnt[bh] = 0;
        if (p.dbg.budgets) for (int e = 0; e < 4; ++e) p.dbg.budgets[bh * 4 + e] = 0;
        if (p.dbg.stats) for (int e = 0; e < 8; ++e) p.dbg.stats[bh * 8 + e] = 0.0;
      }
    }
    return;
  }
  // ---- the rows of the statistics
  {
    const bool odd = ((word >> (base_cta ? 2 : 1)) & 1ull) != 0;       // the KV head's K holds elements that are not finite
    const int base_J = (int)((word >> 3) & 0x3FFFFFull), word_piv = (int)(unsigned)(word >> 32);
    const int total = base_cta ? (b0 > 0 ? base_J : 0) : n_f;
    const int chunk = (total + S - 1) / S;
    const int r_begin = min(total, split * chunk), r_end = min(total, r_begin + chunk);
    R::run(p, sm, bh, g, base_cta, odd, word_piv, m_f, r_begin, r_end);
    for (int e = tid; e < NE; e += NT) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < NWARP; ++w) s += sm.u.part[w][e];
      s_sum[e] = s;
    }
  }
  if (base_cta && split == 0) DBGH(bh, 2);
  cluster_sync();                                  // (every CTA's sums and pivot are there; the rows' memory is free)
  if (rank == 0) DBGH(bh, 3);
  // ---- the budget, by every CTA
  // (what the selection kernel writes behind its words: the members' walk positions, the record)
  pdl_wait();
  if (rank == 0) TICK_BEGIN(p, VATTN_T_BUDGET);
  const unsigned sums = smem_u32(s_sum), pivot = map_rank(smem_u32(sm.piv), (unsigned)Sd);
  HeadBudget hb = head_budget<D>(p, bh, Sd, C - Sd, s_pre, s_scal, rank == 0,
                                 [&](int kind, int s, int e) { return ld_cluster(map_rank(sums, (unsigned)(kind * Sd + s)) + 8u * (unsigned)e); },
                                 [&](int e) { return ld_cluster(pivot + 8u * (unsigned)e); });
  if (rank == 0) {
    TICK_END(p, VATTN_T_BUDGET);
    DBGH(bh, 4);
    if (tid == 0) p.m_ord[bh] = 0u;                // (every CTA of the head has read it: ready for the next step)
    if (tid == 0) p.kabsmax[b * p.Hkv + g] = 0u;   // (the selection has completed)
    if (hb.g.list || p.dbg.dyn_idx) list_sample(p, b, h, bh, hb.g.b, s_misc);
  }
  if (hb.g.list) cluster_sync();                   // (uniform over the cluster: the list is complete)
  TICK_END(p, VATTN_K_STATS);
  // ---- the sampled rows
  TICK_BEGIN(p, VATTN_K_GATHER);
  const int nb = hb.g.L - hb.g.start, batches = (nb + G::CB - 1) / G::CB;
  const int rows = G::CB * ((batches + C - 1) / C);
  const int x0 = hb.g.start + min(nb, rank * rows), x1 = min(hb.g.L, x0 + rows);
  G::sums(p, wm, stages, bh, hb.g, x0, x1);
  float own[2] = {0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int e = i * NT + tid;
    if (e < NG) {
#pragma unroll
      for (int w = 0; w < NWARP; ++w) own[i] += wm[w].part[e];
      if (rank > 0) st_cluster(map_rank(smem_u32(slots + (rank - 1) * NG + e), 0u), own[i]);
      else if (e == D) stages.den = own[i];
    }
  }
  cluster_sync();
  if (rank == 0) {
    // the chunks' sums in their order, scaled by n_s / b, on top of the deterministic ones
    const double f = hb.g.b > 0 ? (double)hb.g.n_s / (double)hb.g.b : 0.0;
    float den = stages.den, num = own[0];
#pragma unroll
    for (int r = 0; r < C - 1; ++r) {
      den += slots[r * NG + D];
      if (tid < D) num += slots[r * NG + tid];
    }
    if (tid < D) out[tid] = Elem<T>::from_float((float)((hb.det + f * (double)num) / (hb.det_den + f * (double)den)));
    DBGH(bh, 5);
    TICK_END(p, VATTN_K_GATHER);
  }
}

template <typename T, int D, int CTAS>
cudaError_t launch_rows_n(const Prob& p, cudaStream_t s, int* fit) {
  constexpr int C = VATTN_ROWS_CLUSTER;
  static_assert(C > 8, "more than the portable cluster size");
  static size_t have[VATTN_MAXDEV];
  cudaError_t e = optin_smem(k_rows<T, D, CTAS>, 0, have, true);
  if (e != cudaSuccess) return e;
  static int wide[VATTN_MAXDEV];                   // clusters beyond the portable size are allowed
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (!__atomic_load_n(&wide[dev], __ATOMIC_ACQUIRE)) {
    if ((e = cudaFuncSetAttribute(k_rows<T, D, CTAS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
    __atomic_store_n(&wide[dev], 1, __ATOMIC_RELEASE);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.B * p.Hq * C)); cfg.blockDim = dim3(NT); cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  if (fit) {
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(fit, k_rows<T, D, CTAS>, &cfg);
  }
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_rows<T, D, CTAS>, p);
}
template <typename T, int D>
cudaError_t launch_rows_t(const Prob& p, cudaStream_t s, int* fit) {
  if constexpr (sizeof(T) == 4 && D == 64)
    if (p.B * p.Hq > 16) return launch_rows_n<T, D, 5>(p, s, fit);
  return launch_rows_n<T, D, 4>(p, s, fit);
}
cudaError_t launch_rows_any(const Prob& p, cudaStream_t s, int* fit) {
  if (p.dtype == VATTN_DTYPE_BF16) return p.D == 128 ? launch_rows_t<bf16_t, 128>(p, s, fit) : launch_rows_t<bf16_t, 64>(p, s, fit);
  return p.D == 128 ? launch_rows_t<float, 128>(p, s, fit) : launch_rows_t<float, 64>(p, s, fit);
}

}  // namespace

cudaError_t launch_rows(const Prob& p, cudaStream_t s) { return launch_rows_any(p, s, nullptr); }

// Whether a call takes the fused kernel; else the statistics and the gather run as two.  Up to 16 heads a cluster of 16
// per head leaves most SMs to themselves: 28.3 -> 23.7 us per step at one fp32 head of 1,024 tokens, 33.9 -> 28.9 at one bf16
// head that samples a fifth of 4,096, 41.2 -> 33.6 at a fifth of 12,800.  Beyond that the clusters, which need 16 places in one
// GPC, load the SMs unevenly and a head waits for its slowest CTA: 62.5 -> 64.9 at 32 x 32,768, 43.8 -> 45.5 at 32 x 8,192.
// fp32 rows of 64 elements have them up to 32 heads where the selection's CTAs (512 threads then, see select_threads) leave
// room on their SMs: 32.6 -> 29.8 at 17 x 4,096, 36.8 -> 35.3 at 32 x 4,096, but at rows of 128 elements 35.9 -> 37.1 at 32 x
// 2,048 and 45.7 -> 48.6 at 24 x 9,001.
// More deterministic and base rows than 256 per CTA: two kernels, which have up to 32 CTAs per head for the statistics (104.2 ->
// 106.8 at 8 heads x 100,001 tokens).  The sampled rows count as well, as many as the call may take, for the budget is known on
// the GPU only: 16 CTAs keep 384 KB of a head's rows in flight, where the two kernels spread them over up to 128 CTAs.  With
// every residual token sampled, at rows of 256 bytes: one head 40.8 -> 39.8 at 12,800 tokens, 42.3 -> 42.3 at 16,384, 48.8 ->
// 57.8 at 32,768; four heads 42.1 -> 43.5 and eight 44.8 -> 46.3 at 16,384, 54.1 -> 59.5 at 24,000; 12 heads 46.5 -> 47.1 at
// 12,800, 47.0 -> 49.6 at 16,384; 16 heads 40.5 -> 41.6 at 8,192, 47.7 -> 51.5 at 16,384; 32 fp32 heads 42.3 -> 42.0 at 8,192,
// 55.9 -> 58.1 at 16,000.  At 512 bytes one head 37.7 -> 35.6 at 8,192 and 39.2 -> 42.6 at 12,800, 16 heads 44.6 -> 44.2 at
// 8,192; at 128 bytes one head 41.0 -> 37.8 at 16,384 and 45.5 -> 47.5 at 32,768, 16 heads 43.4 -> 43.1 at 16,384 and 52.2 ->
// 57.9 at 24,000.  Hence at most 16,384 rows and 4 MB of a head and 16 Mi elements of all heads; with budgets of a tenth it
// then gains 39.0 -> 33.4 at four heads x 16,384, 40.3 -> 36.3 at eight.  (Kept beyond that for budgets that turn out small it
// would save up to 5 us more.  Both ways to leave only the large ones to more CTAs cost what they saved: a gather kernel behind
// it 2 us, 46.7 -> 46.5 and 50.6 -> 53.2 at 8 and 16 heads x 32,768; clusters without a head of their own that wait for the
// budgets 3 to 12 us.)
bool rows_in_one(const Prob& p) {
  if (p.row_unit == 0u || p.gather_kv) return false;
  const int heads = p.B * p.Hq;
  if (heads > (p.dtype == VATTN_DTYPE_FP32 && p.D == 64 && p.max_seq_len <= 16384 ? 32 : 16)) return false;
  const double msl = (double)p.max_seq_len, kmax = p.topk_frac > 0.f ? (double)p.topk_frac * msl : (double)p.k;
  if ((double)p.sink + (double)p.window + kmax + (double)p.base_rate * msl > 256.0 * VATTN_ROWS_CLUSTER) return false;
  const int sampled = p.force_budget >= 0 && p.force_budget < p.max_seq_len ? p.force_budget : p.max_seq_len;
  const long long elements = (long long)sampled * p.D;
  if (sampled > 16384 || elements * (p.dtype == VATTN_DTYPE_BF16 ? 2 : 4) > 4ll << 20 || heads * elements > 16ll << 20) return false;
  // (a device that cannot hold such a cluster takes the two kernels)
  static signed char ok[VATTN_MAXDEV][2][2][2];
  int dev = 0, fit = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= VATTN_MAXDEV) { cudaGetLastError(); return false; }
  signed char* known = &ok[dev][p.dtype == VATTN_DTYPE_BF16][p.D == 128][heads <= 16];
  signed char k = __atomic_load_n(known, __ATOMIC_ACQUIRE);
  if (k == 0) {
    k = launch_rows_any(p, nullptr, &fit) == cudaSuccess && fit >= 1 ? 1 : -1;
    if (k < 0) cudaGetLastError();
    __atomic_store_n(known, k, __ATOMIC_RELEASE);
  }
  return k > 0;
}
