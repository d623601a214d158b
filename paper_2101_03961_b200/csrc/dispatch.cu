// Capacity-limited dispatch of the Switch FFN layer (Section 2.2, Eq. 3 and Fig. 3) and the load-balancing loss
// (Eq. 4-6), as integer index work: no one-hot dispatch / combine tensor is ever built.
//   plan   : count_i, pos_t = number of earlier tokens with the same expert, keep_t = pos_t < C,
//            slot_t = e_t * C + pos_t, token_of_slot, kept_i = min(count_i, C), token-tile list for the grouped GEMMs,
//            P-sums and aux = alpha . E . sum_i (count_i / T)(Psum_i / T)
//   gather : X_d[slot] = x[token]   (forward)        dY_d[slot] = g_token . dy[token], dgate_token (backward)
// Positions are deterministic (token order): block histograms -> column scan -> stable in-block rank. No atomics
// decide a position.
#include "switch_common.cuh"

namespace swmoe {
namespace {

// hist[b][e] = number of tokens of block b routed to expert e
__global__ void __launch_bounds__(kPlanBlockTokens)
plan_hist_kernel(const int* __restrict__ expert_index, int T, int E, int* __restrict__ hist) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int h[kMaxExperts];
  for (int e = threadIdx.x; e < E; e += blockDim.x) h[e] = 0;
  __syncthreads();
  const int t = blockIdx.x * kPlanBlockTokens + threadIdx.x;
  const int e = t < T ? expert_index[t] : -1;
  if ((unsigned)e < (unsigned)E) atomicAdd(&h[e], 1);        // integer counts: order-independent; negative or >= E: no vote
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += blockDim.x) hist[(size_t)blockIdx.x * E + e] = h[e];
}

// Tile lists, shared by the scan kernels: 128-row token tiles (single-CTA GEMM; skipped where `tile_expert` is null) and,
// for the paired-CTA GEMM, each expert's kept rows cut into the fewest pieces of at most kPairTileTokens rows, equal up to
// rounding each piece to a multiple of 16 (the MMA's N granularity).  Thread e < 256 owns expert e: the tiles of earlier
// experts and the loss terms come from warp scans and the eight warps' totals, in a fixed order (the loss is the same
// number on every run).  `term` and `kept_s` are shared-memory arrays filled before the call, at the cost of one barrier;
// log2 steps over the whole block cost sixteen, in a kernel of one block that others wait for.
__device__ __forceinline__ void write_tile_lists(const float* term, const int* kept_s, int E, float loss_scale,
                                                 float* __restrict__ aux_loss, int* __restrict__ tile_expert,
                                                 int* __restrict__ tile_row0, int4* __restrict__ ntile) {
  constexpr int kWarps = kMaxExperts / 32;
  __shared__ int tot128[kWarps], totn[kWarps];
  __shared__ float totl[kWarps];
  const int e = threadIdx.x, lane = e & 31, w = e >> 5;
  __syncthreads();
  int k = 0, n128 = 0, npair = 0, start128 = 0, startn = 0;
  if (e < kMaxExperts) {
    k = e < E ? kept_s[e] : 0;
    n128 = (k + kTileM - 1) / kTileM;
    npair = (k + kPairTileTokens - 1) / kPairTileTokens;
    float l = e < E ? term[e] : 0.f;
    int a = n128, b = npair;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {                   // inclusive scans within the warp
      const int ua = __shfl_up_sync(0xffffffffu, a, off), ub = __shfl_up_sync(0xffffffffu, b, off);
      if (lane >= off) { a += ua; b += ub; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if (lane == 31) { tot128[w] = a; totn[w] = b; totl[w] = l; }
    start128 = a - n128;
    startn = b - npair;
  }
  __syncthreads();
  if (e >= kMaxExperts) return;
  int n_all = 0, m_all = 0;
  float loss = 0.f;
#pragma unroll
  for (int i = 0; i < kWarps; ++i) {
    if (i < w) { start128 += tot128[i]; startn += totn[i]; }
    n_all += tot128[i];
    m_all += totn[i];
    loss += totl[i];
  }
  if (e == 0) {
    if (aux_loss != nullptr) *aux_loss = loss_scale * loss;                           // Eq. 4
    ntile[0] = make_int4(m_all, 0, 0, 0);
    if (tile_expert != nullptr) { tile_expert[0] = n_all; tile_row0[0] = n_all; }
  }
  if (k > 0) {
    if (tile_expert != nullptr) {
      int n = start128;
      for (int r = 0; r < k; r += kTileM, ++n) { tile_expert[1 + n] = e; tile_row0[1 + n] = r; }
    }
    const int rows = ((k + npair - 1) / npair + 15) / 16 * 16;
    int m = startn;
    for (int r = 0; r < k; r += rows, ++m) ntile[1 + m] = make_int4(e, r, min(rows, (k - r + 15) / 16 * 16), 0);
  }
}

// One block of 1024 threads = G groups x Ew columns (Ew = E rounded up to a power of two, at least 32; G = 1024 / Ew):
// thread (g, e) owns slice g of the rows of column e.  Column scan of the histograms, counts, kept, P-sums (all in a
// fixed order), the auxiliary loss and the token-tile list.  A thread's rows are loaded once, all loads in flight
// together, and kept in registers for the scan (up to kScanRows rows per thread; longer slices are re-read).
constexpr int kScanThreads = 1024;
constexpr int kScanRows = 16;
__global__ void __launch_bounds__(kScanThreads)
plan_scan_kernel(const int* __restrict__ hist, int plan_blocks, int loss_blocks, const float* __restrict__ psum_partial,
                 int router_blocks, int T, int E, int Ew, int C, float alpha, int* __restrict__ hist_base,
                 int* __restrict__ count, int* __restrict__ kept, float* __restrict__ psum,
                 float* __restrict__ aux_loss, int* __restrict__ tile_expert, int* __restrict__ tile_row0,
                 int4* __restrict__ ntile, int* __restrict__ count_g, int* __restrict__ group_base) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int qsum[kScanThreads];                         // [g][e], Ew columns per row
  __shared__ int qfirst[kScanThreads];                       // the same over rows < loss_blocks (top-2: first choices)
  __shared__ float qps[kScanThreads];
  __shared__ float term[kMaxExperts];
  __shared__ int kept_s[kMaxExperts];
  const int G = kScanThreads / Ew;
  const int e = threadIdx.x % Ew, g = threadIdx.x / Ew;
  const int hq = (plan_blocks + G - 1) / G, h0 = g * hq, h1 = min(plan_blocks, h0 + hq);
  const int rq = (router_blocks + G - 1) / G, r0 = g * rq, r1 = min(router_blocks, r0 + rq);
  int hv[kScanRows];
  if (e < E) {
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) hv[j] = h0 + j < h1 ? hist[(size_t)(h0 + j) * E + e] : 0;
    float pv[kScanRows];
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) pv[j] = r0 + j < r1 ? psum_partial[(size_t)(r0 + j) * E + e] : 0.f;
    int sum = 0, first = 0;
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) { sum += hv[j]; if (h0 + j < loss_blocks) first += hv[j]; }
    for (int b = h0 + kScanRows; b < h1; ++b) {
      const int v = hist[(size_t)b * E + e];
      sum += v;
      if (b < loss_blocks) first += v;
    }
    float ps = 0.f;
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) ps += pv[j];                                   // fixed order
    for (int b = r0 + kScanRows; b < r1; ++b) ps += psum_partial[(size_t)b * E + e];
    qsum[g * Ew + e] = sum;
    qfirst[g * Ew + e] = first;
    qps[g * Ew + e] = ps;
  }
  __syncthreads();
  if (e < E) {
    int run = 0;
    for (int q = 0; q < g; ++q) run += qsum[q * Ew + e];
#pragma unroll
    for (int j = 0; j < kScanRows; ++j)
      if (h0 + j < h1) { hist_base[(size_t)(h0 + j) * E + e] = run; run += hv[j]; }
    for (int b = h0 + kScanRows; b < h1; ++b) { hist_base[(size_t)b * E + e] = run; run += hist[(size_t)b * E + e]; }
    if (g == 0) {
      int total = 0, first = 0;
      float ps = 0.f;
      for (int q = 0; q < G; ++q) { total += qsum[q * Ew + e]; first += qfirst[q * Ew + e]; ps += qps[q * Ew + e]; }
      count[e] = first;                                                                // f counts the argmax (Eq. 5)
      count_g[e] = first;                                                              // one routing group
      group_base[e] = 0;
      const int k = min(total, C);
      kept[e] = k;
      kept_s[e] = k;
      psum[e] = ps;
      term[e] = ((float)first / (float)T) * (ps / (float)T);                           // f_i . P_i  (Eq. 5, 6)
    }
  }
  write_tile_lists(term, kept_s, E, alpha * (float)E, aux_loss, tile_expert, tile_row0, ntile);
}

// Several routing groups (the pseudo-code's leading cores dimension): every group has its own counts, its own
// capacity cut and its own f and P; an expert's rows are numbered group by group.  One block of 1024 threads;
// thread (q, e) handles groups q, q + Q, ... of column e (Q = 1024 / Ew).  hist_base[b][e] is the position base of
// block b inside its own group; group_base[g][e] = kept tokens of expert e in groups before g; the loss is the mean
// of the groups' losses: (alpha E / G) sum_g sum_i (count_gi / Tg)(Psum_gi / Tg).
constexpr int kScanGroupCells = 8192;                        // G x Ew counters kept in shared memory
__global__ void __launch_bounds__(kScanThreads)
plan_scan_groups_kernel(const int* __restrict__ hist, int blocks_per_group, const float* __restrict__ psum_partial,
                        int rows_per_group, int NG, int Tg, int E, int Ew, int Cg, float alpha,
                        int* __restrict__ hist_base, int* __restrict__ count, int* __restrict__ kept,
                        float* __restrict__ psum, float* __restrict__ aux_loss, int* __restrict__ tile_expert,
                        int* __restrict__ tile_row0, int4* __restrict__ ntile, int* __restrict__ count_g,
                        int* __restrict__ group_base) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int cnt_s[kScanGroupCells];                     // [g][e], Ew columns per row
  __shared__ float qps[kScanThreads], qterm[kScanThreads];   // [q][e]
  __shared__ float term[kMaxExperts];
  __shared__ int kept_s[kMaxExperts];
  const int Q = kScanThreads / Ew;
  const int e = threadIdx.x % Ew, q = threadIdx.x / Ew;
  float ps_tot = 0.f, t_tot = 0.f;
  if (e < E) {
    for (int g = q; g < NG; g += Q) {
      int run = 0;
      for (int b = g * blocks_per_group; b < (g + 1) * blocks_per_group; ++b) {
        hist_base[(size_t)b * E + e] = run;
        run += hist[(size_t)b * E + e];
      }
      float ps = 0.f;
      for (int r = g * rows_per_group; r < (g + 1) * rows_per_group; ++r) ps += psum_partial[(size_t)r * E + e];
      cnt_s[g * Ew + e] = run;
      count_g[(size_t)g * E + e] = run;
      ps_tot += ps;                                                                    // fixed order
      t_tot += ((float)run / (float)Tg) * (ps / (float)Tg);                            // f_gi . P_gi  (Eq. 5, 6)
    }
  }
  qps[threadIdx.x] = ps_tot;
  qterm[threadIdx.x] = t_tot;
  __syncthreads();
  if (q == 0 && e < E) {
    int base = 0, total = 0;
    for (int g = 0; g < NG; ++g) {
      const int c = cnt_s[g * Ew + e];
      group_base[(size_t)g * E + e] = base;
      base += min(c, Cg);
      total += c;
    }
    float ps = 0.f, tm = 0.f;
    for (int k = 0; k < Q; ++k) { ps += qps[k * Ew + e]; tm += qterm[k * Ew + e]; }
    count[e] = total;
    kept[e] = base;
    kept_s[e] = base;
    psum[e] = ps;
    term[e] = tm;
  }
  write_tile_lists(term, kept_s, E, alpha * (float)E / (float)NG, aux_loss, tile_expert, tile_row0, ntile);
}

// pos_t = base[block][e] + (tokens of earlier warps with e) + (earlier lanes with e); slot, token_of_slot.
__global__ void __launch_bounds__(kPlanBlockTokens)
plan_assign_kernel(const int* __restrict__ expert_index, const int* __restrict__ hist_base,
                   const int* __restrict__ kept, const int* __restrict__ group_base, int blocks_per_group, int T,
                   int E, int C, int Cg, int* __restrict__ slot, int* __restrict__ token_of_slot) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int warp_cnt[kPlanBlockTokens / 32][kMaxExperts];
  constexpr int kWarps = kPlanBlockTokens / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < kWarps * kMaxExperts; i += blockDim.x) (&warp_cnt[0][0])[i] = 0;
  __syncthreads();
  const int t = blockIdx.x * kPlanBlockTokens + tid;
  int e = t < T ? expert_index[t] : -1;                       // negative: no expert (takes no slot)
  if (e >= E) e = -1;                                         // an index no expert has is treated the same way
  const unsigned same = __match_any_sync(0xffffffffu, e >= 0 ? e : -1 - lane);   // distinct dummies for those lanes
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (e >= 0 && rank == 0) warp_cnt[warp][e] = __popc(same);
  __syncthreads();
  if (t < T && e < 0) slot[t] = -1;
  if (e >= 0) {
    int pos = hist_base[(size_t)blockIdx.x * E + e] + rank;                  // position inside the token's own group
    for (int w = 0; w < warp; ++w) pos += warp_cnt[w][e];
    const int grp = blockIdx.x / blocks_per_group;
    const int s = pos < Cg ? e * C + group_base[(size_t)grp * E + e] + pos : -1;
    slot[t] = s;
    if (s >= 0) token_of_slot[s] = t;
  }
  // empty slots of every expert: -1 (disjoint from the kept slots written above)
  const int total = E * C;
  for (int s = blockIdx.x * blockDim.x + tid; s < total; s += gridDim.x * blockDim.x) {
    const int ex = s / C, pos = s - ex * C;
    if (pos >= kept[ex]) token_of_slot[s] = -1;
  }
}

// The plan of one routing group from block histograms, hist[r][e] = tokens of the r-th block of `hist_tokens` tokens routed to
// expert e (the tensor-core router's forward kernel leaves them, plan_hist_kernel counts them otherwise), in two kernels that
// both start from that table.
//
// Slots: every block of 1024 tokens adds up the histogram columns itself -- all rows for the totals (kept_i =
// min(count_i, C), Eq. 3), the rows before its own tokens for its position base -- instead of waiting for a scan kernel:
// the table is small (64 KB at 128 x 128) and stays in L2.  Then, as in plan_assign_kernel, pos_t = base + (tokens of
// earlier warps with the same expert) + (earlier lanes with it), in token order, with no atomics deciding a position.
//
// Summary (one block): counts, P-sums, the auxiliary loss (Eq. 4-6) and the tile lists.  It runs beside the slots kernel:
// that kernel lets its successor start only once its own wait on the router is over, so the router has completed and its
// tables are in L2 when the summary starts.  It reads them from there (__ldcg), past the L1 lines that an earlier call may
// have left on its SM: its own wait, which comes last, has not vouched for those yet.  (Waiting first, the plan took 13.3
// us instead of 9.2 at 256 tokens and 128 experts, 19.5 instead of 13.4 at 20011 and 200.  As one more block of the slots
// kernel it did the same work in code and registers that every block had to carry: 96 tokens, d 256, E 8, whole forward
// pass 29.1 us against 28.4.  Launched after the gather instead, to run beside that, it was no faster and delayed GEMM1
// where the gather is short.)
// Every block reads the whole table, so the work grows with the square of T, and from some T on one scan kernel and its
// wait cost less.  Plan, us, these kernels / scan and assignment, at 64, 128, 200 experts: 131072 tokens 13, 17, 28 / 19, 26,
// 42; 262144 28, 44, 75 / 28, 48, 81; 524288 75, 130, 239 / 50, 85, 153; 1048576 214, 396, 712 / 91, 161, 296.
constexpr int kFusedTokens = 1024, kFusedMaxTokens = 262144;

// Column sums of the histogram table by the whole block: tot over all rows, pre over rows below row_end, as partial sums
// per thread (column e = tid % Ew, slice q = tid / Ew of the rows, every Q-th one).
__device__ __forceinline__ void hist_column_sums(const int* __restrict__ hist, int hist_rows, int row_end, int E, int e,
                                                 int q, int Q, int* pre_out, int* tot_out) {
  int pre = 0, tot = 0;
  if (e < E) {
    for (int r0 = q; r0 < hist_rows; r0 += 16 * Q) {           // 16 rows in flight
      int v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = r0 + j * Q < hist_rows ? hist[(size_t)(r0 + j * Q) * E + e] : 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) { tot += v[j]; if (r0 + j * Q < row_end) pre += v[j]; }
    }
  }
  *pre_out = pre;
  *tot_out = tot;
}

__global__ void __launch_bounds__(kFusedTokens)
plan_slots_kernel(const int* __restrict__ expert_index, const int* __restrict__ hist, int hist_rows, int hist_tokens, int T,
                  int E, int Ew, int C, int* __restrict__ slot, int* __restrict__ token_of_slot, int* __restrict__ kept) {
  pdl_wait();
  pdl_launch_dependents();                                      // (in this order: see above)
  __shared__ int part_pre[kFusedTokens], part_tot[kFusedTokens];    // [slice][column]
  __shared__ int base_s[kMaxExperts], kept_s[kMaxExperts];
  constexpr int kWarps = kFusedTokens / 32;
  __shared__ int warp_cnt[kMaxExperts][kWarps];                // [expert][warp of the block]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int Q = kFusedTokens / Ew;
  const int t = (int)blockIdx.x * kFusedTokens + tid;
  int et = t < T ? expert_index[t] : -1;                      // negative: no expert (takes no slot)
  hist_column_sums(hist, hist_rows, min(hist_rows, (int)blockIdx.x * (kFusedTokens / hist_tokens)), E, tid % Ew, tid / Ew, Q,
                   &part_pre[tid], &part_tot[tid]);
  for (int i = tid; i < kWarps * E; i += kFusedTokens) (&warp_cnt[0][0])[i] = 0;
  __syncthreads();
  if (tid < E) {
    int b = 0, total = 0;
    for (int k = 0; k < Q; ++k) { b += part_pre[k * Ew + tid]; total += part_tot[k * Ew + tid]; }
    base_s[tid] = b;
    kept_s[tid] = min(total, C);
    if (blockIdx.x == 0) kept[tid] = min(total, C);
  }
  if (et >= E) et = -1;
  const unsigned same = __match_any_sync(0xffffffffu, et >= 0 ? et : -1 - lane);   // distinct dummies for those lanes
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (et >= 0 && rank == 0) warp_cnt[et][warp] = __popc(same);
  __syncthreads();
  for (int ex = warp; ex < E; ex += kWarps) {                  // exclusive scan over the block's warps, per expert
    const int c = warp_cnt[ex][lane];
    int incl = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += up;
    }
    warp_cnt[ex][lane] = incl - c;
  }
  __syncthreads();
  if (t < T) {
    int sl = -1;
    if (et >= 0) {
      const int pos = base_s[et] + warp_cnt[et][warp] + rank;
      if (pos < C) { sl = et * C + pos; token_of_slot[sl] = t; }
    }
    slot[t] = sl;
  }
  // empty slots of every expert: -1 (disjoint from the kept slots written above)
  const int total_slots = E * C;
  for (int sidx = (int)blockIdx.x * kFusedTokens + tid; sidx < total_slots; sidx += (int)gridDim.x * kFusedTokens) {
    const int ex = sidx / C, pos = sidx - ex * C;
    if (pos >= kept_s[ex]) token_of_slot[sidx] = -1;
  }
}

// Launched after plan_slots_kernel.  Reads only what the kernels before that one wrote (the router its P-sums and, on the
// tensor cores, the histograms; plan_hist_kernel those of the other calls), past L1, and writes what no kernel in flight reads;
// plan_slots_kernel has waited for all of them before it lets this one start.  Its own wait comes last, so that the next kernel's wait covers everything before this one.
__global__ void __launch_bounds__(kFusedTokens)
plan_summary_kernel(const int* hist, int hist_rows, const float* psum_partial, int psum_rows, int T, int E, int Ew, int C,
                    float alpha, int* __restrict__ count, float* __restrict__ psum, float* __restrict__ aux_loss,
                    int* __restrict__ tile_expert, int* __restrict__ tile_row0, int4* __restrict__ ntile,
                    int* __restrict__ count_g, int* __restrict__ group_base) {
  pdl_launch_dependents();
  __shared__ int part_tot[kFusedTokens];
  __shared__ float part_ps[kFusedTokens], term[kMaxExperts];
  __shared__ int kept_s[kMaxExperts];
  const int tid = threadIdx.x, Q = kFusedTokens / Ew, q = tid / Ew, e = tid % Ew;
  // column sums of the histograms and of p, the latter in a fixed order (slice by slice, rows ascending inside a slice)
  int tot = 0;
  float ps = 0.f;
  if (e < E) {
    for (int r0 = q; r0 < max(hist_rows, psum_rows); r0 += 16 * Q) {   // 16 rows of each table in flight, added in row order
      int v[16];
      float f[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = r0 + j * Q < hist_rows ? __ldcg(hist + (size_t)(r0 + j * Q) * E + e) : 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) f[j] = r0 + j * Q < psum_rows ? __ldcg(psum_partial + (size_t)(r0 + j * Q) * E + e) : 0.f;
#pragma unroll
      for (int j = 0; j < 16; ++j) { tot += v[j]; ps += f[j]; }
    }
  }
  part_tot[tid] = tot;
  part_ps[tid] = ps;
  __syncthreads();
  if (tid < E) {
    int total = 0;
    float sum = 0.f;
    for (int k = 0; k < Q; ++k) { total += part_tot[k * Ew + tid]; sum += part_ps[k * Ew + tid]; }
    count[tid] = total;                                                                // f counts the argmax (Eq. 5)
    count_g[tid] = total;
    group_base[tid] = 0;
    kept_s[tid] = min(total, C);
    psum[tid] = sum;
    term[tid] = ((float)total / (float)T) * (sum / (float)T);                          // f_i . P_i  (Eq. 5, 6)
  }
  write_tile_lists(term, kept_s, E, alpha * (float)E, aux_loss, tile_expert, tile_row0, ntile);
  pdl_wait();
}

// ---- further stages of No-Token-Left-Behind routing (Appendix B) ---------------------------------------------
// alt[t] = the expert that follows prev[t] in the token's ranking of the experts (probability, highest first; equal
// probabilities by index, lowest first) for a token that has no slot yet; -1 for a token that has one, and when no
// expert is left.  With prev = the argmax this is the second choice (stage 2), with prev = the previous stage's
// choices the third, and so on.  One warp per token.
__global__ void __launch_bounds__(256)
reroute_choice_kernel(const float* __restrict__ probs, const int* __restrict__ prev, const int* __restrict__ slot,
                      int T, int E, int* __restrict__ alt) {
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (t >= T) return;
  const int e1 = prev[t];
  if (slot[t] >= 0 || e1 < 0 || e1 >= E) {
    if (lane == 0) alt[t] = -1;
    return;
  }
  const float v1 = probs[(size_t)t * E + e1];
  float best = -1.f;
  int arg = 0x7fffffff;
  for (int e = lane; e < E; e += 32) {
    const float v = probs[(size_t)t * E + e];
    const bool later = v < v1 || (v == v1 && e > e1);         // ranked after prev[t]
    if (later && v > best) { best = v; arg = e; }             // ascending e: the first maximum wins
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int oa = __shfl_xor_sync(0xffffffffu, arg, off);
    if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
  }
  if (lane == 0) alt[t] = arg < E ? arg : -1;                  // nothing ranked after prev[t]
}

// Position bases of a further stage: the rerouted tokens of expert e queue up behind the kept[e] tokens it has so far.
// Also rewrites kept[] and the tile lists for the grown experts.  Thread (g, e) of the one block owns slice g of the rows of
// column e, as in plan_scan_kernel (a thread per expert walking all rows waited for one batch of loads after another: 13.6
// us from the previous kernel's end to its own at 32768 tokens and 64 experts; with slices 6.7).
__global__ void __launch_bounds__(kScanThreads)
reroute_scan_kernel(const int* __restrict__ hist, int plan_blocks, int E, int Ew, int C, int* __restrict__ hist_base,
                    int* __restrict__ kept, int* __restrict__ tile_expert, int* __restrict__ tile_row0,
                    int4* __restrict__ ntile) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int qsum[kScanThreads];                         // [g][e], Ew columns per row
  __shared__ float term[kMaxExperts];
  __shared__ int kept_s[kMaxExperts];
  const int G = kScanThreads / Ew;
  const int e = threadIdx.x % Ew, g = threadIdx.x / Ew;
  const int hq = (plan_blocks + G - 1) / G, h0 = g * hq, h1 = min(plan_blocks, h0 + hq);
  int hv[kScanRows], run = 0;
  if (e < E) {
    run = kept[e];
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) hv[j] = h0 + j < h1 ? hist[(size_t)(h0 + j) * E + e] : 0;
    int sum = 0;
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) sum += hv[j];
    for (int b = h0 + kScanRows; b < h1; ++b) sum += hist[(size_t)b * E + e];
    qsum[g * Ew + e] = sum;
  }
  __syncthreads();                                             // (also: kept[] has been read by every slice)
  if (e < E) {
    for (int q = 0; q < g; ++q) run += qsum[q * Ew + e];
#pragma unroll
    for (int j = 0; j < kScanRows; ++j)
      if (h0 + j < h1) { hist_base[(size_t)(h0 + j) * E + e] = run; run += hv[j]; }
    for (int b = h0 + kScanRows; b < h1; ++b) { hist_base[(size_t)b * E + e] = run; run += hist[(size_t)b * E + e]; }
    if (g == G - 1) {
      const int k = min(run, C);
      kept[e] = k;
      kept_s[e] = k;
      term[e] = 0.f;
    }
  }
  write_tile_lists(term, kept_s, E, 0.f, nullptr, tile_expert, tile_row0, ntile);
}

// Slots of the rerouted tokens (same stable in-block rank as the first stage), their gate (the probability of the
// expert that now processes them, Eq. 2) and, for every token, the expert that processes it.
__global__ void __launch_bounds__(kPlanBlockTokens)
reroute_assign_kernel(const int* __restrict__ alt, const int* __restrict__ expert_index,
                      const int* __restrict__ hist_base, const float* __restrict__ probs, int T, int E, int C,
                      int* __restrict__ slot, int* __restrict__ token_of_slot, float* __restrict__ gate,
                      int* __restrict__ expert_proc, int first_stage) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int warp_cnt[kPlanBlockTokens / 32][kMaxExperts];
  constexpr int kWarps = kPlanBlockTokens / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < kWarps * kMaxExperts; i += blockDim.x) (&warp_cnt[0][0])[i] = 0;
  __syncthreads();
  const int t = blockIdx.x * kPlanBlockTokens + tid;
  int a = t < T ? alt[t] : -1;
  if (a >= E) a = -1;
  const int key = a >= 0 ? a : -1 - lane;                     // distinct dummies for tokens that do not move
  const unsigned same = __match_any_sync(0xffffffffu, key);
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (a >= 0 && rank == 0) warp_cnt[warp][a] = __popc(same);
  __syncthreads();
  if (t < T) {
    bool moved = false;
    if (a >= 0) {
      int pos = hist_base[(size_t)blockIdx.x * E + a] + rank;
      for (int w = 0; w < warp; ++w) pos += warp_cnt[w][a];
      if (pos < C) {
        const int s = a * C + pos;
        slot[t] = s;
        token_of_slot[s] = t;
        gate[t] = probs[(size_t)t * E + a];
        moved = true;
      }
    }
    // the expert that processes the token: its first choice until a stage moves it
    if (moved) expert_proc[t] = a;
    else if (first_stage) expert_proc[t] = expert_index[t];
  }
}

// ---- top-2 routing ------------------------------------------------------------------------------------------
// Second choice of every token: the expert with the second-highest probability (lowest index on ties) and its
// probability, stored as assignment T + t.  One warp per token.
__global__ void __launch_bounds__(256)
top2_choice_kernel(const float* __restrict__ probs, int T, int E, int* __restrict__ expert_index,
                   float* __restrict__ gate) {
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (t >= T) return;
  const int e1 = expert_index[t];
  float best = -1.f;
  int arg = 0x7fffffff;
  for (int e = lane; e < E; e += 32) {
    const float v = probs[(size_t)t * E + e];
    if (e != e1 && v > best) { best = v; arg = e; }          // ascending e: the first maximum wins
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int oa = __shfl_xor_sync(0xffffffffu, arg, off);
    if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
  }
  if (lane == 0) {
    expert_index[T + t] = arg < E ? arg : -1;                 // E == 1: no second choice (a negative index takes no slot)
    gate[T + t] = arg < E ? best : 0.f;
  }
}

// out[t] = rows[t] + rows[T + t] (+ skip[t]), a dropped assignment (slot < 0) counting as zero: y from the weighted
// expert outputs of the two choices, dx from their input gradients; `skip` is the layer's input (or dy) when the
// layer carries its own residual connection.  One warp per token, float32 sum, one rounding.
template <bool kBf16>
__global__ void __launch_bounds__(256)
top2_sum_kernel(const uint4* __restrict__ rows, const uint4* __restrict__ skip, const int* __restrict__ slot, int T,
                int row_vec, uint4* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (t >= T) return;
  const bool k1 = slot[t] >= 0, k2 = slot[T + t] >= 0;
  const uint4* r1 = rows + (size_t)t * row_vec;
  const uint4* r2 = rows + (size_t)(T + t) * row_vec;
  const uint4* r3 = skip != nullptr ? skip + (size_t)t * row_vec : nullptr;
  uint4* dst = out + (size_t)t * row_vec;
  const uint4 zero = make_uint4(0, 0, 0, 0);
  for (int v = lane; v < row_vec; v += 32) {
    const uint4 a = k1 ? r1[v] : zero, b = k2 ? r2[v] : zero, c = r3 != nullptr ? r3[v] : zero;
    uint4 o;
    if (kBf16) {
      const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
      const __nv_bfloat162* pc = reinterpret_cast<const __nv_bfloat162*>(&c);
      __nv_bfloat162* po = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 fa = __bfloat1622float2(pa[i]), fb = __bfloat1622float2(pb[i]), fc = __bfloat1622float2(pc[i]);
        po[i] = __floats2bfloat162_rn((fa.x + fb.x) + fc.x, (fa.y + fb.y) + fc.y);
      }
    } else {
      const float* fa = reinterpret_cast<const float*>(&a);
      const float* fb = reinterpret_cast<const float*>(&b);
      const float* fc = reinterpret_cast<const float*>(&c);
      float* fo = reinterpret_cast<float*>(&o);
#pragma unroll
      for (int i = 0; i < 4; ++i) fo[i] = (fa[i] + fb[i]) + fc[i];
    }
    dst[v] = o;
  }
}

// ---- gathers --------------------------------------------------------------------------------------------------
// Bound by HBM; a warp per slot row at a time, and no more blocks than are resident at once: a grid of one row per warp
// spends its time on launching blocks.  The forward gather takes four rows at a time, their loads in flight together
// (65536 tokens, d_model 256, 128 experts: 18 us, 27 with one row; 32768 x 768: 21 and 24); the backward gather, whose rows
// end in a reduction, is faster with twice the warps and one row each (32768 x 768: 31 us; two rows on half the warps 35).
constexpr int kGatherBlocksPerSm = 4, kGatherDyBlocksPerSm = 8;   // x 256 threads

// Slot row s of the buffers: the token it holds (>= 0), -1: a row to zero-fill (up to a multiple of `pad` rows past the
// expert's last token, so that tensor-core tiles never read stale rows), -2: leave alone.
__device__ __forceinline__ int slot_source(int s, int slots, int C, int pad, const int* __restrict__ token_of_slot,
                                           const int* __restrict__ kept) {
  if (s >= slots) return -2;
  const int ex = s / C, pos = s - ex * C, k = kept[ex];
  if (pos < k) return token_of_slot[s];
  return pos < (k + pad - 1) / pad * pad ? -1 : -2;
}

// Rows of dropped tokens: dst[t] = src[t], or zero where src is null.  A warp looks at tokens gw, gw + n_warps, ...: an
// overflowing expert drops the last of its tokens, so neighbours are dropped together and must not fall to one warp
// (with 32 neighbours each, copied piece by piece, 4686 tokens of 3.5 KB, 5 skewed experts at capacity factor 1, skip path:
// x gather 31 us, dy gather 117; dealt out 12 and 17).
__device__ __forceinline__ void dropped_rows(const int* __restrict__ slot, int T, int row_vec, const uint4* __restrict__ src,
                                             uint4* __restrict__ dst, int gw, int n_warps, int lane) {
  for (long long t0 = gw; t0 < T; t0 += 32ll * n_warps) {
    const long long mine = t0 + (long long)lane * n_warps;
    unsigned dropped = __ballot_sync(0xffffffffu, mine < T && slot[mine] < 0);
    while (dropped != 0) {
      const size_t at = (size_t)(t0 + (long long)(__ffs(dropped) - 1) * n_warps) * row_vec;
      dropped &= dropped - 1;
      for (int v = lane; v < row_vec; v += 128) {              // four pieces in flight
        uint4 r[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          r[j] = src != nullptr && v + 32 * j < row_vec ? src[at + v + 32 * j] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (v + 32 * j < row_vec) dst[at + v + 32 * j] = r[j];
      }
    }
  }
}

// Forward: kept slots copy the token's row.  Dropped tokens get a zero output row (their representation reaches the next
// layer only through the residual connection, Section 2.2), or, when the layer itself adds the skip path (`residual`),
// their input row; `y` is null for top-2 routing, whose outputs are formed per assignment.  Top-2: slot s may hold
// assignment T + t (the second choice of token t): its source row is still x[t].
__global__ void __launch_bounds__(256, kGatherBlocksPerSm)
gather_x_kernel(const uint4* __restrict__ x, const int* __restrict__ token_of_slot, const int* __restrict__ kept,
                const int* __restrict__ slot, int T, int slots, int C, int row_vec, int pad, int residual,
                uint4* __restrict__ xd, uint4* __restrict__ y) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr int kRows = 4;
  const int lane = threadIdx.x & 31, gw = blockIdx.x * 8 + (threadIdx.x >> 5), n_warps = gridDim.x * 8;
  for (int s0 = gw * kRows; s0 < slots; s0 += n_warps * kRows) {
    const uint4* src[kRows];
    int tok[kRows];
#pragma unroll
    for (int j = 0; j < kRows; ++j) tok[j] = slot_source(s0 + j, slots, C, pad, token_of_slot, kept);
#pragma unroll
    for (int j = 0; j < kRows; ++j) src[j] = x + (size_t)max(tok[j] >= T ? tok[j] - T : tok[j], 0) * row_vec;
    uint4* dst = xd + (size_t)s0 * row_vec;
    for (int v = lane; v < row_vec; v += 32) {
      uint4 r[kRows];
#pragma unroll
      for (int j = 0; j < kRows; ++j) r[j] = tok[j] >= 0 ? src[j][v] : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int j = 0; j < kRows; ++j)
        if (tok[j] != -2) dst[(size_t)j * row_vec + v] = r[j];
    }
  }
  if (y != nullptr) dropped_rows(slot, T, row_vec, residual ? x : nullptr, y, gw, n_warps, lane);
}

// The whole plan and the forward gather in one launch, for one routing group of at most kSmallTokens tokens.  Such a call is
// latency from end to end: three dependent launches of about 5 us each (slots, summary beside them, gather) for work that
// takes one.  Every block ranks all tokens itself (a token per thread, in token order as in plan_slots_kernel, no atomics) and
// then moves its share of the rows; block 0 also leaves what the summary leaves.  96 tokens, d 256, E 8, whole forward pass
// 26.7 us before, 24.2 with this; 256 tokens, d 768, E 128 187.5 and 184.4.
__host__ __device__ inline int small_plan_parts(int C, int pad) { return ((C < pad ? C : pad) + 15) / 16; }
__global__ void __launch_bounds__(kSmallTokens)
plan_gather_small_kernel(const int* __restrict__ expert_index, const float* __restrict__ psum_partial, int psum_rows, int T,
                         int E, int C, float alpha, int row_vec, int pad, int residual, const uint4* __restrict__ x,
                         uint4* __restrict__ xd, uint4* __restrict__ y, int* __restrict__ slot,
                         int* __restrict__ token_of_slot, int* __restrict__ count, int* __restrict__ kept,
                         float* __restrict__ psum, float* __restrict__ aux_loss, int* __restrict__ tile_expert,
                         int* __restrict__ tile_row0, int4* __restrict__ ntile, int* __restrict__ count_g,
                         int* __restrict__ group_base) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr int kWarps = kSmallTokens / 32;
  static_assert(kSmallTokens >= kMaxExperts, "a thread per token and per expert");
  __shared__ int warp_cnt[kWarps][kMaxExperts];
  __shared__ int kept_s[kMaxExperts], slot_s[kSmallTokens];
  __shared__ float term[kMaxExperts];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int e = tid < T ? expert_index[tid] : -1;                   // negative or >= E: no expert (takes no slot)
  if (e >= E) e = -1;
  float ps = 0.f;                                             // thread i < E: Psum_i, rows in order
  if (blockIdx.x == 0 && tid < E)
    for (int r = 0; r < psum_rows; ++r) ps += psum_partial[(size_t)r * E + tid];
  for (int i = tid; i < kWarps * kMaxExperts; i += kSmallTokens) (&warp_cnt[0][0])[i] = 0;
  __syncthreads();
  const unsigned same = __match_any_sync(0xffffffffu, e >= 0 ? e : -1 - lane);   // distinct dummies for those lanes
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (e >= 0 && rank == 0) warp_cnt[warp][e] = __popc(same);
  __syncthreads();
  if (tid < E) {
    int total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) total += warp_cnt[w][tid];
    const int k = min(total, C);
    kept_s[tid] = k;
    if (blockIdx.x == 0) {
      kept[tid] = k;
      count[tid] = total;                                                              // f counts the argmax (Eq. 5)
      count_g[tid] = total;
      group_base[tid] = 0;
      psum[tid] = ps;
      term[tid] = ((float)total / (float)T) * (ps / (float)T);                         // f_i . P_i  (Eq. 5, 6)
    }
  }
  if (tid < T) {
    int sl = -1;
    if (e >= 0) {
      int pos = rank;
      for (int w = 0; w < warp; ++w) pos += warp_cnt[w][e];
      if (pos < C) sl = e * C + pos;
    }
    slot_s[tid] = sl;
    if (blockIdx.x == 0) {
      slot[tid] = sl;
      if (sl >= 0) token_of_slot[sl] = tid;
    }
  }
  __syncthreads();
  // rows: kept tokens to their slots, dropped tokens' output rows, a token per warp at a time
  const int gw = (int)blockIdx.x * kWarps + warp, n_warps = (int)gridDim.x * kWarps;
  for (int t = gw; t < T; t += n_warps) {
    const int sl = slot_s[t];
    const uint4* src = x + (size_t)t * row_vec;
    uint4* dst = sl >= 0 ? xd + (size_t)sl * row_vec : y + (size_t)t * row_vec;
    const bool copy = sl >= 0 || residual;
    for (int v = lane; v < row_vec; v += 128) {                // four pieces in flight
      uint4 r[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) r[j] = copy && v + 32 * j < row_vec ? src[v + 32 * j] : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (v + 32 * j < row_vec) dst[v + 32 * j] = r[j];
    }
  }
  // empty slots, and the zero rows that a tile may read past an expert's last token (see slot_source)
  // 16 of them per warp at a time
  const int parts = small_plan_parts(C, pad);
  for (int i = gw; i < E * parts; i += n_warps) {
    const int ex = i / parts, part = i - ex * parts, k = kept_s[ex], r0 = k + 16 * part;
    const int r1 = min(min(C, (k + pad - 1) / pad * pad), r0 + 16);
    if (part == 0)
      for (int pos = k + lane; pos < C; pos += 32) token_of_slot[ex * C + pos] = -1;
    uint4* rows = xd + (size_t)ex * C * row_vec;
    for (int v = r0 * row_vec + lane; v < r1 * row_vec; v += 32) rows[v] = make_uint4(0, 0, 0, 0);
  }
  if (blockIdx.x == 0)
    write_tile_lists(term, kept_s, E, alpha * (float)E, aux_loss, tile_expert, tile_row0, ntile);
}

__device__ __forceinline__ float dot_scale8(const uint4& a, const uint4& b, float g, uint4* out) {
  const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
  const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
  __nv_bfloat162* po = reinterpret_cast<__nv_bfloat162*>(out);
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 fa = __bfloat1622float2(pa[i]), fb = __bfloat1622float2(pb[i]);
    s = fmaf(fa.x, fb.x, s);
    s = fmaf(fa.y, fb.y, s);
    po[i] = __floats2bfloat162_rn(g * fa.x, g * fa.y);
  }
  return s;
}
__device__ __forceinline__ float dot_scale4(const uint4& a, const uint4& b, float g, uint4* out) {
  const float* fa = reinterpret_cast<const float*>(&a);
  const float* fb = reinterpret_cast<const float*>(&b);
  float* fo = reinterpret_cast<float*>(out);
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) { s = fmaf(fa[i], fb[i], s); fo[i] = g * fa[i]; }
  return s;
}

// Backward: dY_d[slot] = g . dy[token] (derivative of Eq. 2 w.r.t. the expert output) and dgate[token] = <dy, o> with
// o = y / g (derivative w.r.t. the gate).  With the skip path inside the layer (`dx` not null) the dropped tokens' dx rows
// start at dy: the router's gradient is added to them later, and no expert ever writes them.
template <bool kBf16>
__global__ void __launch_bounds__(256, kGatherDyBlocksPerSm)
gather_dy_kernel(const uint4* __restrict__ dy, const uint4* __restrict__ y, const float* __restrict__ gate,
                 const int* __restrict__ token_of_slot, const int* __restrict__ kept, const int* __restrict__ slot,
                 int T, int slots, int C, int row_vec, int pad, uint4* __restrict__ dyd,
                 float* __restrict__ dgate, uint4* __restrict__ dx) {
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31, gw = blockIdx.x * 8 + (threadIdx.x >> 5), n_warps = gridDim.x * 8;
  for (int s = gw; s < slots; s += n_warps) {
    const int tok = slot_source(s, slots, C, pad, token_of_slot, kept);
    if (tok == -2) continue;
    uint4* dst = dyd + (size_t)s * row_vec;
    if (tok < 0) {
      for (int v = lane; v < row_vec; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
      continue;
    }
    const float g = gate[tok];                                 // top-2 routing: assignment t or T + t of token t mod T
    const uint4* src = dy + (size_t)(tok >= T ? tok - T : tok) * row_vec;
    const uint4* ysrc = y + (size_t)tok * row_vec;
    float dot = 0.f;
    for (int v = lane; v < row_vec; v += 32) {
      uint4 o;
      dot += kBf16 ? dot_scale8(src[v], ysrc[v], g, &o) : dot_scale4(src[v], ysrc[v], g, &o);
      dst[v] = o;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    // (a second or rerouted choice may have lost its probability to underflow: its gate's gradient enters dh times that 0)
    if (lane == 0) dgate[tok] = g != 0.f ? dot / g : 0.f;
  }
  if (dx != nullptr) dropped_rows(slot, T, row_vec, dy, dx, gw, n_warps, lane);
}

}  // namespace

int launch_reroute(const Shape& s, const Plan& p, void* ws, cudaStream_t st);

namespace {
// Columns of a plan block's [slice][expert] layout: E rounded up to a power of two, at least 32.
int column_width(int E) {
  int w = 32;
  while (w < E) w *= 2;
  return w;
}
// The 128-row tile list, for the path that reads it.
int* list128(const Shape& s, const Plan& p, void* ws) {
  return s.gemm_path == SWITCH_MOE_GEMM_TC_1CTA ? ws_ptr<int>(ws, p.tile_expert) : nullptr;
}
}  // namespace

int launch_dispatch_plan(const Shape& s, const Plan& p, const int32_t* expert_index, bool after_router, float* aux_loss,
                         void* ws, cudaStream_t st) {
  int* ei = ws_ptr<int>(ws, p.expert_index);
  if (expert_index != nullptr && expert_index != ei) {
    if (cudaMemcpyAsync(ei, expert_index, (size_t)s.Tv * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
      return SWITCH_MOE_CUDA_ERROR;
  }
  // The tensor-core router's forward kernel leaves the histograms of its own expert choices in the workspace.  They are
  // good only right after it: the counting kernel below and every rerouting stage put tables of another layout in their
  // place, and the expert indices may have been edited since.
  const bool have_hist = after_router && s.router_hist;
  if (!have_hist)
    launch_k(plan_hist_kernel, dim3(s.plan_blocks), dim3(kPlanBlockTokens), 0, st, ei, s.Tv, s.E, ws_ptr<int>(ws, p.hist));
  // Slots and summary each read whole tables (every block the counts, one block those and the router's P-sums), the scan reads
  // them once and serially.  Where the router has left the counts that is the faster form up to kFusedMaxTokens; where they are
  // counted first, up to 2^21 cells of tokens x experts and 2^15 of P-sums (of at most 1024 rows).  Staged plan, us, so / by scan: bf16
  // 32768 tokens, 64 experts 13.1 / 13.6; 49152, 128 18.9 / 16.9; 32768, 256 19.4 / 17.5; float32 4096, 128 13.0 / 14.9; 4096, 256
  // 17.2 / 17.0; 65536, 8 13.5 / 15.1; 131072, 8 19.3 / 17.5; 262144, 256 155 / 111.
  const bool counted_small = (long long)s.T * s.E <= 1 << 21 && s.router_blocks <= 1024 && s.router_blocks * s.E <= 1 << 15;
  if (s.G == 1 && !s.top2 && s.T <= kFusedMaxTokens && (have_hist || counted_small)) {
    const int token_blocks = (s.T + kFusedTokens - 1) / kFusedTokens;
    const int hist_rows = have_hist ? s.router_blocks : s.plan_blocks;
    launch_k(plan_slots_kernel, dim3(token_blocks), dim3(kFusedTokens), 0, st, ei, ws_ptr<int>(ws, p.hist), hist_rows,
             have_hist ? s.router_block_tokens : kPlanBlockTokens, s.T, s.E, column_width(s.E), s.Cg, ws_ptr<int>(ws, p.slot),
             ws_ptr<int>(ws, p.token_of_slot), ws_ptr<int>(ws, p.kept));
    launch_k(plan_summary_kernel, dim3(1), dim3(kFusedTokens), 0, st, ws_ptr<int>(ws, p.hist), hist_rows,
             ws_ptr<float>(ws, p.psum_partial), s.router_blocks, s.T, s.E, column_width(s.E), s.Cg, s.alpha,
             ws_ptr<int>(ws, p.count), ws_ptr<float>(ws, p.psum), aux_loss, list128(s, p, ws), ws_ptr<int>(ws, p.tile_row0),
             ws_ptr<int4>(ws, p.ntile), ws_ptr<int>(ws, p.count_g), ws_ptr<int>(ws, p.group_base));
    return launch_reroute(s, p, ws, st);
  }
  const int Ew = column_width(s.E);
  const int blocks_per_group = s.plan_blocks / s.G;
  int* count_g = ws_ptr<int>(ws, p.count_g);
  int* group_base = ws_ptr<int>(ws, p.group_base);
  if (s.G == 1) {
    launch_k(plan_scan_kernel, dim3(1), dim3(kScanThreads), 0, st, ws_ptr<int>(ws, p.hist), s.plan_blocks,
             s.top2 ? s.plan_blocks / 2 : s.plan_blocks, ws_ptr<float>(ws, p.psum_partial), s.router_blocks, s.T, s.E, Ew,
             s.Cg, s.alpha,
             ws_ptr<int>(ws, p.hist_base), ws_ptr<int>(ws, p.count), ws_ptr<int>(ws, p.kept),
             ws_ptr<float>(ws, p.psum), aux_loss, list128(s, p, ws), ws_ptr<int>(ws, p.tile_row0),
             ws_ptr<int4>(ws, p.ntile), count_g, group_base);
  } else {
    if (s.G * Ew > kScanGroupCells || s.router_blocks % s.G != 0) return SWITCH_MOE_UNSUPPORTED_SHAPE;
    launch_k(plan_scan_groups_kernel, dim3(1), dim3(kScanThreads), 0, st, ws_ptr<int>(ws, p.hist), blocks_per_group,
             ws_ptr<float>(ws, p.psum_partial), s.router_blocks / s.G, s.G, s.Tg, s.E, Ew, s.Cg, s.alpha,
             ws_ptr<int>(ws, p.hist_base), ws_ptr<int>(ws, p.count), ws_ptr<int>(ws, p.kept),
             ws_ptr<float>(ws, p.psum), aux_loss, list128(s, p, ws), ws_ptr<int>(ws, p.tile_row0),
             ws_ptr<int4>(ws, p.ntile), count_g, group_base);
  }
  launch_k(plan_assign_kernel, dim3(s.plan_blocks), dim3(kPlanBlockTokens), 0, st, ei, ws_ptr<int>(ws, p.hist_base),
           ws_ptr<int>(ws, p.kept), group_base, blocks_per_group, s.Tv, s.E, s.C, s.Cg, ws_ptr<int>(ws, p.slot),
           ws_ptr<int>(ws, p.token_of_slot));
  return launch_reroute(s, p, ws, st);
}

// The further stages of No-Token-Left-Behind routing, after either form of the first-stage plan: per stage the next
// choices of the tokens still without a slot, their block histograms, the position bases behind the rows every
// expert already holds, and the slots.
int launch_reroute(const Shape& s, const Plan& p, void* ws, cudaStream_t st) {
  int* ei = ws_ptr<int>(ws, p.expert_index);
  for (int stage = 0; stage < s.reroute_stages; ++stage) {
    int* alt = ws_ptr<int>(ws, p.alt) + (size_t)stage * s.T;
    const int* prev = stage == 0 ? ei : alt - s.T;
    launch_k(reroute_choice_kernel, dim3((s.T + 7) / 8), dim3(256), 0, st, ws_ptr<float>(ws, p.probs), prev,
             ws_ptr<int>(ws, p.slot), s.T, s.E, alt);
    launch_k(plan_hist_kernel, dim3(s.plan_blocks), dim3(kPlanBlockTokens), 0, st, alt, s.T, s.E,
             ws_ptr<int>(ws, p.hist));
    launch_k(reroute_scan_kernel, dim3(1), dim3(kScanThreads), 0, st, ws_ptr<int>(ws, p.hist), s.plan_blocks, s.E,
             column_width(s.E), s.C, ws_ptr<int>(ws, p.hist_base), ws_ptr<int>(ws, p.kept), list128(s, p, ws),
             ws_ptr<int>(ws, p.tile_row0), ws_ptr<int4>(ws, p.ntile));
    launch_k(reroute_assign_kernel, dim3(s.plan_blocks), dim3(kPlanBlockTokens), 0, st, alt, ei,
             ws_ptr<int>(ws, p.hist_base), ws_ptr<float>(ws, p.probs), s.T, s.E, s.C, ws_ptr<int>(ws, p.slot),
             ws_ptr<int>(ws, p.token_of_slot), ws_ptr<float>(ws, p.gate), ws_ptr<int>(ws, p.expert_proc),
             stage == 0 ? 1 : 0);
  }
  return launch_status();
}

namespace {
dim3 gather_grid(long long warps, int per_sm) {
  const long long blocks = (warps + 7) / 8, most = (long long)sm_count_or_default() * per_sm;
  return dim3((unsigned)(blocks < most ? blocks : most));
}
// Rows to deal out over a gather's warps: the slots', and where it also writes the dropped tokens' rows at least the tokens'
// (65536 tokens of 1.5 KB, 8 experts of one slot each: x gather
// 31 us, dy gather with the skip path 37; with warps for the slots alone, a block each, 5.2 and 8.5 ms).
long long gathered_rows(const Shape& s, bool dropped) {
  const long long slots = (long long)s.E * s.C;
  return dropped && s.T > slots ? s.T : slots;
}
// Rows past an expert's last token that the GEMMs' tiles may read: the CTA-pair path's tiles end at a multiple of 16.
int pad_rows(const Shape& s) { return s.gemm_path == 0 ? 16 : kTileM; }
}  // namespace

int launch_gather_x(const Shape& s, const Plan& p, const void* x, void* y, void* ws, cudaStream_t st) {
  const int row_vec = (int)((size_t)s.d * s.elt / 16);
  // top-2 routing: the output rows of dropped assignments are skipped by the kernel that sums the two choices
  launch_k(gather_x_kernel, gather_grid((gathered_rows(s, !s.top2) + 3) / 4, kGatherBlocksPerSm), dim3(256), 0, st,
      static_cast<const uint4*>(x), ws_ptr<int>(ws, p.token_of_slot), ws_ptr<int>(ws, p.kept),
      ws_ptr<int>(ws, p.slot), s.T, s.E * s.C, s.C, row_vec, pad_rows(s), s.residual, ws_ptr<uint4>(ws, p.xd),
      s.top2 ? nullptr : static_cast<uint4*>(y));
  return launch_status();
}

// launch_dispatch_plan and launch_gather_x in one launch, where `s.plan_gather` says so.
int launch_plan_gather(const Shape& s, const Plan& p, const void* x, void* y, float* aux_loss, void* ws, cudaStream_t st) {
  const int row_vec = (int)((size_t)s.d * s.elt / 16);
  const int zero_parts = s.E * small_plan_parts(s.C, pad_rows(s)), rows = s.T > zero_parts ? s.T : zero_parts;
  const int warps = kSmallTokens / 32, blocks = (rows + warps - 1) / warps;
  launch_k(plan_gather_small_kernel, dim3((unsigned)(blocks < kChipSms ? blocks : kChipSms)), dim3(kSmallTokens), 0, st,
           ws_ptr<int>(ws, p.expert_index), ws_ptr<float>(ws, p.psum_partial), s.router_blocks, s.T, s.E, s.C, s.alpha, row_vec,
           pad_rows(s), s.residual, static_cast<const uint4*>(x), ws_ptr<uint4>(ws, p.xd), static_cast<uint4*>(y),
           ws_ptr<int>(ws, p.slot), ws_ptr<int>(ws, p.token_of_slot), ws_ptr<int>(ws, p.count), ws_ptr<int>(ws, p.kept),
           ws_ptr<float>(ws, p.psum), aux_loss, list128(s, p, ws), ws_ptr<int>(ws, p.tile_row0), ws_ptr<int4>(ws, p.ntile),
           ws_ptr<int>(ws, p.count_g), ws_ptr<int>(ws, p.group_base));
  return launch_status();
}

int launch_gather_dy(const Shape& s, const Plan& p, const void* dy, const void* y, void* dx, void* ws, cudaStream_t st) {
  const int row_vec = (int)((size_t)s.d * s.elt / 16);
  // (top-2 routing: dx rows are formed by the kernel that sums the two assignments, and `y` is the per-assignment
  // output buffer already)
  const bool skip = s.residual && !s.top2;
  // with the skip path inside the layer, y holds x + g . E(x): the gate's gradient needs the copy without x
  const void* ysrc = skip ? ws_ptr<char>(ws, p.layer_y) : y;
  auto kernel = s.dtype == SWITCH_MOE_BF16 ? gather_dy_kernel<true> : gather_dy_kernel<false>;
  launch_k(kernel, gather_grid(gathered_rows(s, skip), kGatherDyBlocksPerSm), dim3(256), 0, st, static_cast<const uint4*>(dy),
           static_cast<const uint4*>(ysrc), ws_ptr<float>(ws, p.gate), ws_ptr<int>(ws, p.token_of_slot),
           ws_ptr<int>(ws, p.kept), ws_ptr<int>(ws, p.slot), s.T, s.E * s.C, s.C, row_vec, pad_rows(s),
           ws_ptr<uint4>(ws, p.dyd), ws_ptr<float>(ws, p.dgate), skip ? static_cast<uint4*>(dx) : nullptr);
  return launch_status();
}

int launch_top2_choice(const Shape& s, const Plan& p, void* ws, cudaStream_t st) {
  launch_k(top2_choice_kernel, dim3((s.T + 7) / 8), dim3(256), 0, st, ws_ptr<float>(ws, p.probs), s.T, s.E,
           ws_ptr<int>(ws, p.expert_index), ws_ptr<float>(ws, p.gate));
  return launch_status();
}

int launch_top2_sum(const Shape& s, const Plan& p, const void* per_assignment, const void* skip, void* out, void* ws,
                    cudaStream_t st) {
  const int row_vec = (int)((size_t)s.d * s.elt / 16);
  if (s.dtype == SWITCH_MOE_BF16)
    launch_k(top2_sum_kernel<true>, dim3((s.T + 7) / 8), dim3(256), 0, st, static_cast<const uint4*>(per_assignment),
             static_cast<const uint4*>(skip), ws_ptr<int>(ws, p.slot), s.T, row_vec, static_cast<uint4*>(out));
  else
    launch_k(top2_sum_kernel<false>, dim3((s.T + 7) / 8), dim3(256), 0, st, static_cast<const uint4*>(per_assignment),
             static_cast<const uint4*>(skip), ws_ptr<int>(ws, p.slot), s.T, row_vec, static_cast<uint4*>(out));
  return launch_status();
}

}  // namespace swmoe
