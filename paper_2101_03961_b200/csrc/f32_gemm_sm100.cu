// Grouped expert GEMMs of the float32 layer on the B200 tensor cores (tcgen05 + TMEM, operands staged by TMA): the expert
// FFN h = x W_in, y = ReLU(h) W_out (Section 5, FFN review) and its derivatives, float32 in, float32 out, with the fused
// epilogues of the FMA kernels in simt_gemm.cu.
//
// Arithmetic.  A float32 times 2^24 is the exact sum of three bfloat16 parts, h + m + l (8 + 8 + 8 significand bits, each
// rounded to nearest), from the smallest subnormal up to 2^104 (unscaled, l of an operand below 2^-110 would reach under
// bfloat16's smallest subnormal: 2^-118 came out exact to 1e-5 only), and a product of two bfloat16 is exact in float32; the
// sums are scaled back by 2^-48.  Of the nine cross products six are formed (h.h, h.m, m.h, m.m, h.l, l.h); the other three
// are below 2^-25 of the product (contractions of at most 16 steps form them too).  The tensor pipe adds into its float32 accumulator with
// truncation, so a long sum left there would drift: here an accumulator lives for kK = 32 steps of the contraction only.
// Within such a chunk the five correction products (at most 2^-8 of the sum) go first and h.h last, then the chunk is read
// out of tensor memory and added to a float32 sum in registers, round to nearest.  A chain of one fused multiply-add per step
// rounds at the size of the running sum K times, this one K / 32 times (and twice inside a chunk): the error against
// float64 is smaller than the FMA kernels' at every contraction length (tests/test_gpu_f32_products.py holds it to that).
// Values that the parts cannot hold (infinities, NaN, |x| from 2^104 on) and sums from 2^80 on turn up as a non-finite result;
// that element, and no other, is then formed again by a plain chain of fused multiply-adds from the float32 operands (redo).
//
// Layout.  All six products are written out[n][m], m contiguous: m = weight columns or rows on the MMA's M side (tiles of
// 128, TMEM lanes), n = an expert's tokens, or the other index of a weight gradient, on the N side, at most 128 wide (64 sums
// per thread of the eight warps that add the chunks up; two accumulators and three stages of the A parts take 2 x 128 + 3 x 48
// columns of tensor memory).  Roles of the warps: one issues TMA loads of float32 tiles into a ring (A 128 x 32, B up to
// 128 x 32); two groups of four convert a staged tile into its parts -- A into tensor memory, where a lane is a row and no
// transposition of the contiguous axis is needed, B into 64-byte-swizzled shared memory; two issue the MMAs; eight read
// finished chunks and write the results, a lane per m, so that a warp's store is a full line.  A in tensor memory is what
// makes this pay: from shared memory every one of the six products would read 4 KB more per 16 steps, and the 128 B per
// clock of shared memory also carry the staging of the float32 tiles and the parts.
//
// What bounds it: instructions.  Of a stage's 1100 to 1300 cycles the MMAs take 770 at 128 columns and 390 at 64; conversion,
// adding up and the waits between the roles issue in 60% of all slots, and the code of all roles together streams through the
// instruction caches.  Taking out any one of conversion of A, of B, the correction MMAs, or the adding up shortened a product by
// 6 to 14%.  4096 tokens, 512 x 2048, 16 experts, between stage events, FMA kernels / here: GEMM1 187 / 80 us, GEMM2 233 / 86,
// dgrad2 213 / 78, wgrad2 170 / 69, dgrad1 242 / 84, wgrad1 170 / 69 (100 to 125 TFLOP/s; the FMA pipes' peak is 74.5).
#include <cfloat>
#include <cmath>

#include "tc_common.cuh"

namespace swmoe {
using namespace tc;
namespace {

constexpr int kBoxRows = 32;                         // token rows per TMA box
constexpr int kK = 32;                               // contraction steps per stage, and life of an accumulator
constexpr int kM = 128, kNMax = 128, kNFix = kNMax;    // output tile: m, most tokens, columns of a weight gradient's tile
constexpr int kLoadStages = 4, kPartStages = 3;
constexpr int kALoad = kM * kK * 4, kBLoad = kNMax * kK * 4, kLoadBytes = kALoad + kBLoad;      // 16 KB each
constexpr int kPartBytes = kNMax * kK * 2, kPartStage = 3 * kPartBytes;                          // 3 x 8 KB
constexpr int kAPartCols = kK / 2, kAStageCols = 3 * kAPartCols;                                 // TMEM columns
constexpr int kGroups = 2, kConvWarps = 4 * kGroups, kMmaWarps = 2, kEpiWarps = 8;
// Stages alternate between the groups, between the issuing warps and between the accumulators.  A barrier's parity tells two
// phases apart, so its next phase must not be able to complete before every waiter has seen this one: each barrier has one
// group or warp waiting for it, and the next phase needs what that one does after its wait.  The ring of parts has three
// buffers, hence two barriers per buffer, used in turn (stage s: barriers s % 6, buffer s % 3).
constexpr int kPartBars = 2 * kPartStages;
static_assert(kGroups == 2 && kMmaWarps == 2 && kLoadStages % 2 == 0 && kPartStages % 2 == 1, "fixed owners");
constexpr int kTmaWarp = kConvWarps + kEpiWarps, kMmaWarp = kTmaWarp + 1;
constexpr int kF32Threads = 32 * (kMmaWarp + kMmaWarps);
constexpr int kHalf = kNMax / 2;                     // columns per epilogue warp
constexpr int kSums = (kHalf + 15) / 16 * 8;            // pairs of columns, read 16 columns at a time
constexpr int kTabBytes = kEpiWarps * kHalf * 8;     // output row and scale per column
constexpr int kCumBytes = (2 * kMaxExperts + 1 + 2 * 10) * 4;
constexpr int kF32Smem = 1024 + kLoadStages * kLoadBytes + kPartStages * kPartStage + kTabBytes + 256 + kCumBytes;
constexpr int kWidths = kNMax / 16;                  // candidate tile widths: 16, 32 .. kNMax

constexpr float kUp = 16777216.f, kDown = 1.f / (kUp * kUp);    // scale of the operands, of the sums

struct F32Problem {
  const float* A; long long a_es, a_ms, a_ks;        // A(e, m, k) element strides (the loads go through the tensor maps)
  const float* B; long long b_es, b_ns, b_ks;        // B(e, n, k)
  int M, N, K;                                       // N < 0: kept[e] tokens;  K < 0: kept[e] tokens
  int E, C, n_mtiles, n_ntiles;                      // n_ntiles: weight gradients
  const int* kept; const int* token_of_slot; const float* gate;
  float* out; int ld_out;
  // ReLU'(u) = [u > 0]: a byte per hidden unit and 8 slot rows, [E][rows / 8][units], from GEMM1 to dgrad2
  uint8_t* hmask; int hrows, hcols;
  const float* res; float* out2;                     // skip path: row added to the output; second copy without it
  int plain;                                         // GEMM1 / dgrad2 without ReLU and mask (GEGLU experts gate elsewhere)
  int* status;
};

struct F32Tile {
  int e, m0, n0, n_valid, n_mma, K;
  // A contraction of one step of the MMA is two chunks, the corrections and the high parts: what the pipe truncates there
  // is all the error there is, and the products of the high parts alone rarely reach past the accumulator's last bit.  All
  // eight corrections then: a single product comes out rounded once, like an FMA's (without the three smallest 2% less exact).
  __device__ __forceinline__ bool apart() const { return K <= kUmmaK; }
};

__device__ __forceinline__ void tc_mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tm)) : "memory");
}
__device__ __forceinline__ void tc_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tc_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major tile with rows of 64 bytes, 64-byte swizzle: atoms of 8 rows.
__device__ __forceinline__ uint64_t part_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// Two float32 in one register pair: packed instructions round each half like the scalar ones and take half the issue slots.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// x minus the packed bfloat16 pair h (exact: h is x rounded to bfloat16).
__device__ __forceinline__ float2 minus_pair(float2 x, uint32_t h) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r)
      : "l"(pack2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u))), "l"(pack2(-1.f, -1.f)), "l"(pack2(x.x, x.y)));
  return unpack2(r);
}
__device__ __forceinline__ uint32_t bf16_pair(float2 v) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&b);
}
// Two consecutive floats of the contraction -> packed bfloat16 pairs of the three parts of x 2^24.
__device__ __forceinline__ void split3(float x0, float x1, uint32_t* h, uint32_t* m, uint32_t* l) {
  float2 x = unpack2(mul2(pack2(x0, x1), pack2(kUp, kUp)));
  *h = bf16_pair(x);
  x = minus_pair(x, *h);
  *m = bf16_pair(x);
  *l = bf16_pair(minus_pair(x, *m));
}

// The element-wise end of a product for one output.  `live`: ReLU'(u) of this output (dgrad2); `skip`: the row added on the
// skip path (combine, scatter).  What is not finite is left so in the output, for redo to find, unless it is `final`.
template <int OP>
__device__ __forceinline__ void finish(const F32Problem& p, long long at, float scale, float v, bool live, float skip,
                                       bool final = false) {
  if (OP == kGemm2Combine) v *= scale;
  if (OP == kGemm1Relu && !p.plain && (final || v >= -FLT_MAX)) v = fmaxf(v, 0.f);
  if (OP == kDgrad2Mask && !p.plain) v = live ? v : 0.f;
  if (OP == kGemm2Combine && p.out2 != nullptr) p.out2[at] = v;
  if ((OP == kGemm2Combine || OP == kDgrad1Scatter) && p.res != nullptr) v += skip;
  p.out[at] = v;
}

// The results of one m over a warp's columns that are not finite in the output, by a chain of fused multiply-adds each, in
// ascending order of the contraction.  Four columns share the loads of A, four steps of them are in flight, 16 bytes at a time
// along whichever axis is contiguous; eight columns at a time were up to a quarter faster, but spilled registers of the kernel.  A
// step of 8192 tokens, 256 x 1024, 4 experts, every element of dy, W_in or W_out NaN: 8.8, 2.8, 7.2 ms, on the FMA kernels 0.84.
// `progress` changes as it goes: the other warps of the block wait for this one under a limit, and start that anew whenever it
// has, so that the limit holds for a contraction of any length.
template <int OP>
__device__ __noinline__ void redo(const F32Problem& p, int e, int n0, int K, int m, int mine, const int2* tab,
                                  volatile int* progress) {
  constexpr bool kToken = OP != kWgrad2 && OP != kWgrad1;              // B contiguous along the contraction, else along n
  constexpr bool kAKMajor = OP == kDgrad2Mask || OP == kDgrad1Scatter; // A contiguous along the contraction, else along m
  const float* a = p.A + e * p.a_es + m * p.a_ms;
  for (int c0 = 0; c0 < mine; c0 += 4) {
    uint32_t cols = 0;
    for (int c = 0; c < min(4, mine - c0); ++c)
      cols |= fabsf(p.out[(long long)tab[c0 + c].x * p.ld_out + m]) <= FLT_MAX ? 0u : 1u << c;
    if (cols == 0) continue;
    const float* b[4];                                        // token products: a row per column, rows of good ones not touched
#pragma unroll
    for (int c = 0; c < 4; ++c)
      b[c] = p.B + e * p.b_es + (n0 + c0 + (kToken ? (cols >> c & 1u ? c : __ffs(cols) - 1) : 0)) * p.b_ns;
    float s[4] = {};
    for (int k = 0; k < K; k += 4) {
      float av[4], bv[4][4];
      if (kAKMajor) {
        *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(a + k);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) av[j] = k + j < K ? a[(k + j) * p.a_ks] : 0.f;
      }
      if (kToken) {
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<float4*>(bv[c]) = *reinterpret_cast<const float4*>(b[c] + k);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 row = *reinterpret_cast<const float4*>(b[0] + min(k + j, K - 1) * p.b_ks);
          bv[0][j] = row.x; bv[1][j] = row.y; bv[2][j] = row.z; bv[3][j] = row.w;
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (kToken || k + j < K) {                            // (token products: K is a multiple of 8)
#pragma unroll
          for (int c = 0; c < 4; ++c) s[c] = fmaf(av[j], bv[c][j], s[c]);
        }
      }
      if ((k & 1023) == 0) *progress = (int)clock64();
    }
    uint8_t* byte = p.hmask + ((long long)e * p.hrows + (n0 + c0) / 8) * p.hcols + m;
    const uint32_t sh = c0 & 4, old = (OP == kDgrad2Mask || OP == kGemm1Relu) && !p.plain ? *byte : 0u, live = old >> sh;
    uint32_t bits = old & ~(cols << sh);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if ((cols >> c & 1u) == 0) continue;
      const int2 r = tab[c0 + c];
      const long long at = (long long)r.x * p.ld_out + m;
      const bool skip = (OP == kGemm2Combine || OP == kDgrad1Scatter) && p.res != nullptr;
      finish<OP>(p, at, __int_as_float(r.y), s[c], live >> c & 1u, skip ? p.res[at] : 0.f, true);
      bits |= s[c] > 0.f ? 1u << (c + sh) : 0u;
    }
    if (OP == kGemm1Relu && !p.plain) *byte = (uint8_t)bits;
  }
}

template <int OP>
__global__ void __launch_bounds__(kF32Threads, 1)
f32_expert_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ F32Problem p) {
  constexpr bool kToken = OP != kWgrad2 && OP != kWgrad1;              // n = tokens, contraction contiguous in B
  constexpr bool kAKMajor = OP == kDgrad2Mask || OP == kDgrad1Scatter; // contraction contiguous in A
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t parts = base + kLoadStages * kLoadBytes;
  uint8_t* parts_gen = gen + kLoadStages * kLoadBytes;
  uint8_t* tab_gen = parts_gen + kPartStages * kPartStage;
  uint8_t* bar_gen = tab_gen + kTabBytes;
  const uint32_t bars = smem_u32(bar_gen);
  auto lfull = [&](int s) { return bars + 8u * s; };
  auto lempty = [&](int s) { return bars + 8u * (kLoadStages + s); };
  auto pfull = [&](int s) { return bars + 8u * (2 * kLoadStages + s); };
  auto pempty = [&](int s) { return bars + 8u * (2 * kLoadStages + kPartBars + s); };
  auto dfull = [&](int s) { return bars + 8u * (2 * (kLoadStages + kPartBars) + s); };
  auto dempty = [&](int s) { return bars + 8u * (2 * (kLoadStages + kPartBars) + 2 + s); };
  constexpr int kBars = 2 * (kLoadStages + kPartBars) + 4;
  static_assert(8 * kBars + 12 <= 256, "barrier block");
  volatile uint32_t* tmem_ptr_s = reinterpret_cast<volatile uint32_t*>(bar_gen + 8 * kBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_gen + 8 * kBars + 4);     // and, behind it, redo's progress
  int* kept_s = reinterpret_cast<int*>(bar_gen + 256);       // tokens per expert
  int* cum_s = kept_s + kMaxExperts;                         // [E + 1] token tiles of earlier experts
  float* cost_s = reinterpret_cast<float*>(cum_s + kMaxExperts + 1);

  const int warp = uniform_warp_id(), lane = threadIdx.x & 31;
  if (warp == kTmaWarp && elect_one()) {
    prefetch_map(&tmA);
    prefetch_map(&tmB);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kLoadStages; ++s) { mbar_init(lfull(s), 1); mbar_init(lempty(s), 4); }
    for (int s = 0; s < kPartBars; ++s) { mbar_init(pfull(s), 4); mbar_init(pempty(s), 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(dfull(s), 1); mbar_init(dempty(s), kEpiWarps); }
    abort_flag[0] = abort_flag[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_ptr_s))), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();                                                 // the previous kernel's results are needed from here on
  for (int e = threadIdx.x; e < p.E; e += kF32Threads) kept_s[e] = p.kept[e];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_s;
  const uint32_t a_tmem = tmem_base + 2 * kNMax;

  // Token products: the width of a token tile.  A block's time is its rounds of tiles times the time of a tile: stages that
  // take no less below 96 columns (the A tile and the waits are the same), and a result that grows with the width.  Experts are
  // cut into the fewest tiles of at most the chosen width, equal up to rounding to 16.  (Weighting the result four times as much
  // and letting stages shrink down to 64 columns chose the same widths or times within 1%.)
  int cap = kNFix, n_tiles;
  if (kToken) {
    if (warp < kWidths) {
      const int w = 16 * (warp + 1);
      int n = 0, widest = 0;
      for (int e = lane; e < p.E; e += 32) {
        const int k = kept_s[e];
        if (k > 0) {
          const int nt = (k + w - 1) / w;
          n += nt;
          widest = max(widest, ((k + nt - 1) / nt + 15) / 16 * 16);
        }
      }
      n = __reduce_add_sync(0xffffffffu, n);
      widest = __reduce_max_sync(0xffffffffu, widest);
      const int rounds = (n * p.n_mtiles + (int)gridDim.x - 1) / (int)gridDim.x;
      const float stages = (float)((p.K + kK - 1) / kK);
      if (lane == 0) cost_s[warp] = (float)rounds * (stages * (float)max(96, widest) + 170.f + (float)widest);
    }
    __syncthreads();
    float best = cost_s[kWidths - 1];
    cap = kNMax;
    for (int i = kWidths - 2; i >= 0; --i)
      if (cost_s[i] < best) { best = cost_s[i]; cap = 16 * (i + 1); }
    if (warp == 0) {                                          // token tiles of earlier experts
      int run = 0;
      for (int e0 = 0; e0 < p.E; e0 += 32) {
        const int n = e0 + lane < p.E ? (kept_s[e0 + lane] + cap - 1) / cap : 0;
        int incl = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int up = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += up;
        }
        if (e0 + lane < p.E) cum_s[e0 + lane] = run + incl - n;
        run += __shfl_sync(0xffffffffu, incl, 31);
      }
      if (lane == 0) cum_s[p.E] = run;
    }
    __syncthreads();
    n_tiles = cum_s[p.E] * p.n_mtiles;
  } else {
    n_tiles = p.E * p.n_mtiles * p.n_ntiles;
  }
  auto decode = [&](int id) {
    F32Tile t;
    if (kToken) {
      int lo = 0, hi = p.E;                                   // last expert whose first tile is at or before id
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cum_s[mid] * p.n_mtiles <= id) lo = mid; else hi = mid;
      }
      const int nt = cum_s[lo + 1] - cum_s[lo], rem = id - cum_s[lo] * p.n_mtiles, kept = kept_s[lo];
      const int width = ((kept + nt - 1) / nt + 15) / 16 * 16, mt = rem / nt;
      t.e = lo;
      t.m0 = mt * kM;
      t.n0 = (rem - mt * nt) * width;
      t.n_valid = min(width, kept - t.n0);
      t.K = p.K;
    } else {
      const int per_e = p.n_mtiles * p.n_ntiles, rem = id % per_e;
      t.e = id / per_e;
      t.m0 = rem % p.n_mtiles * kM;
      t.n0 = rem / p.n_mtiles * kNFix;
      t.n_valid = min(kNFix, p.N - t.n0);
      t.K = kept_s[t.e];
    }
    t.n_mma = (t.n_valid + 15) & ~15;
    return t;
  };

  if (warp == kTmaWarp) {
    // ------------------------------------------------------------------------------------------ TMA producer
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const F32Tile t = decode(id);
      const int boxes = (t.n_mma + kBoxRows - 1) / kBoxRows;
      const uint32_t bytes = kALoad + (kToken ? boxes * kBoxRows : kNFix) * kK * 4;
      for (int k0 = 0; k0 < t.K; k0 += kK) {
        ok = mbar_wait_warp<true>(lempty(stage), phase ^ 1u, abort_flag, p.status, 51);
        if (!ok) break;
        if (elect_one()) {
          const uint32_t a_dst = base + stage * kLoadBytes, b_dst = a_dst + kALoad;
          mbar_arrive_expect_tx(lfull(stage), bytes);
          if (kAKMajor) tma_load_3d(a_dst, &tmA, lfull(stage), k0, t.m0, t.e);
          else tma_load_3d(a_dst, &tmA, lfull(stage), t.m0, k0, t.e);
          if (kToken) {
            for (int j = 0; j < boxes; ++j)
              tma_load_3d(b_dst + j * kBoxRows * kK * 4, &tmB, lfull(stage), k0, t.n0 + kBoxRows * j, t.e);
          } else {
            tma_load_3d(b_dst, &tmB, lfull(stage), t.n0, k0, t.e);
          }
        }
        __syncwarp();
        if (++stage == kLoadStages) { stage = 0; phase ^= 1u; }
      }
    }
    if (*abort_flag != 0) {
      // give copies that are still in flight a bounded time to land before the CTA's shared memory is released
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
  } else if (warp >= kMmaWarp) {
    // ------------------------------------------------------------------------------------------ MMA issuers
    // Two warps take turns: twelve short MMAs per stage keep the pipe busy for as long as their issue takes, and the waits
    // between two stages (about 400 cycles for a warp) would leave it idle.
    const int w = warp - kMmaWarp;
    int pbar = 0, turn = 0;
    uint32_t pphase = 0, dphase = 0;                          // dphase: of this warp's accumulator
    bool ok = true;
    const uint64_t b_desc0 = part_desc(parts);
    constexpr uint32_t kPartStep = kPartBytes >> 4, kStep = (kUmmaK * 2) >> 4;      // descriptor address units
    for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const F32Tile t = decode(id);
      const bool apart = t.apart();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(t.n_mma >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
#pragma unroll 1
      for (int k0 = 0; k0 < t.K; k0 += kK, turn ^= 1) {
        if (turn == w) {                                      // this warp's accumulator is number w
          ok = mbar_wait_warp<true>(dempty(w), dphase ^ 1u, abort_flag, p.status, 52) &&
               mbar_wait_warp<true>(pfull(pbar), pphase, abort_flag, p.status, 53);
          if (!ok) break;
          tc_fence_after();
          const int ps = pbar < kPartStages ? pbar : pbar - kPartStages;
          const uint32_t dt = tmem_base + (uint32_t)w * kNMax, at = a_tmem + (uint32_t)ps * kAStageCols;
          const uint64_t bd = b_desc0 + (uint64_t)(ps * (kPartStage >> 4));
          // part pairs (A, B), 0 = high, 1 = middle, 2 = low: the corrections from the smallest up, then high . high; the first
          // three in contractions of one step only
          constexpr int pa[9] = {2, 1, 2, 2, 0, 1, 1, 0, 0}, pb[9] = {2, 2, 1, 0, 2, 1, 0, 1, 0};
          if (!apart) {
            if (elect_one()) {
#pragma unroll
              for (int q = 3; q < 9; ++q)
#pragma unroll
                for (int ks = 0; ks < kK / kUmmaK; ++ks)
                  tc_mma_bf16_ts(dt, at + pa[q] * kAPartCols + ks * (kUmmaK / 2), bd + pb[q] * kPartStep + ks * kStep, idesc,
                                 q + ks > 3 ? 1u : 0u);
              tc_commit(pempty(pbar));                          // frees the parts once these MMAs have read them
              tc_commit(dfull(w));
            }
          } else {                                            // one step in two chunks, see F32Tile::apart
            if (elect_one()) {
#pragma unroll
              for (int q = 0; q < 8; ++q)
                tc_mma_bf16_ts(dt, at + pa[q] * kAPartCols, bd + pb[q] * kPartStep, idesc, q > 0 ? 1u : 0u);
              tc_commit(dfull(w));
            }
            __syncwarp();
            dphase ^= 1u;
            ok = mbar_wait_warp<true>(dempty(w), dphase ^ 1u, abort_flag, p.status, 52);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
              tc_mma_bf16_ts(dt, at, bd, idesc, 0u);
              tc_commit(pempty(pbar));
              tc_commit(dfull(w));
            }
          }
          __syncwarp();
          dphase ^= 1u;
        }
        if (++pbar == kPartBars) { pbar = 0; pphase ^= 1u; }
      }
    }
  } else if (warp < kConvWarps) {
    // ------------------------------------------------------------------------------------------ float32 -> parts
    // Two groups of four warps take turns: while one waits for its tensor-memory stores, the other converts.
    const int group = warp >> 2, lg = warp & 3;               // lg: A's TMEM lane group; B's group of 8 steps
    const int m = lg * 32 + lane;
    int ls = 0, pbar = 0, turn = 0;
    uint32_t lphase = 0, pphase = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const F32Tile t = decode(id);
      for (int k0 = 0; k0 < t.K; k0 += kK, turn ^= 1) {
        if (turn == group) {
          ok = mbar_wait_warp<true>(lfull(ls), lphase, abort_flag, p.status, 54) &&
               (pbar < kPartStages                            // the buffer's previous stage was three stages ago
                    ? mbar_wait_warp<true>(pempty(pbar + kPartStages), pphase ^ 1u, abort_flag, p.status, 55)
                    : mbar_wait_warp<true>(pempty(pbar - kPartStages), pphase, abort_flag, p.status, 55));
          if (!ok) break;
          tc_fence_after();
          const int ps = pbar < kPartStages ? pbar : pbar - kPartStages;
          const uint8_t* a_src = gen + ls * kLoadBytes;
          const uint8_t* b_src = a_src + kALoad;
          const int live = t.K - k0;                          // steps of this stage inside the contraction
          const uint32_t at = a_tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(ps * kAStageCols);
#pragma unroll
          for (int kh = 0; kh < kK / 16; ++kh) {
            float v[16];
            if (kAKMajor) {                                   // rows of 128 bytes, 128-byte swizzle
#pragma unroll
              for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float4*>(v + 4 * j) =
                    *reinterpret_cast<const float4*>(a_src + m * 128 + (((kh * 4 + j) ^ (m & 7)) << 4));
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] = reinterpret_cast<const float*>(a_src)[(kh * 16 + j) * kM + m];
            }
            if (!kToken && live < kK) {                       // slot rows past the expert's last token hold anything
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] = kh * 16 + j < live ? v[j] : 0.f;
            }
            uint32_t h[8], md[8], lo[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) split3(v[2 * j], v[2 * j + 1], &h[j], &md[j], &lo[j]);
            tc_st8(at + kh * (kUmmaK / 2), h);
            tc_st8(at + kAPartCols + kh * (kUmmaK / 2), md);
            tc_st8(at + 2 * kAPartCols + kh * (kUmmaK / 2), lo);
          }
          uint8_t* b_dst = parts_gen + ps * kPartStage;
#pragma unroll 2
          for (int n = lane; n - lane < t.n_mma; n += 32) {
            float v[8];
            if (kToken) {
#pragma unroll
              for (int j = 0; j < 2; ++j)
                *reinterpret_cast<float4*>(v + 4 * j) =
                    *reinterpret_cast<const float4*>(b_src + n * 128 + (((lg * 2 + j) ^ (n & 7)) << 4));
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) v[j] = reinterpret_cast<const float*>(b_src)[(lg * 8 + j) * kNFix + n];
              if (live < kK) {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = lg * 8 + j < live ? v[j] : 0.f;
              }
            }
            uint32_t bh[4], bm[4], bl[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) split3(v[2 * j], v[2 * j + 1], &bh[j], &bm[j], &bl[j]);
            uint8_t* dst = b_dst + n * 64 + ((lg ^ ((n >> 1) & 3)) << 4);
            *reinterpret_cast<uint4*>(dst) = make_uint4(bh[0], bh[1], bh[2], bh[3]);
            *reinterpret_cast<uint4*>(dst + kPartBytes) = make_uint4(bm[0], bm[1], bm[2], bm[3]);
            *reinterpret_cast<uint4*>(dst + 2 * kPartBytes) = make_uint4(bl[0], bl[1], bl[2], bl[3]);
          }
          tc_wait_st();
          tc_fence_before();
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(lempty(ls));
            mbar_arrive(pfull(pbar));
          }
        }
        if (++ls == kLoadStages) { ls = 0; lphase ^= 1u; }
        if (++pbar == kPartBars) { pbar = 0; pphase ^= 1u; }
      }
    }
  } else {
    // ------------------------------------------------------------------------------------------ epilogue warps
    const int lg = warp & 3, hf = (warp - kConvWarps) >> 2;   // TMEM lane group, half of the tile's columns
    int2* tab = reinterpret_cast<int2*>(tab_gen) + (warp - kConvWarps) * kHalf;   // {output row, scale} per column
    int d = 0;                                                // a stage's accumulator: the parity of its running number
    uint32_t dphase0 = 0, dphase1 = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const F32Tile t = decode(id);
      const int cols = t.n_mma >> 1, c0 = hf * cols;          // this warp's columns: c0 .. c0 + cols - 1
      const int mine = min(cols, t.n_valid - c0);             // of which inside the problem (may be <= 0)
      const int tab_row0 = t.e * (kToken ? p.C : p.N) + t.n0 + c0;
      for (int j = lane; j < mine; j += 32) {
        int row;
        float scale = 1.f;
        if (OP == kGemm2Combine || OP == kDgrad1Scatter) {
          row = p.token_of_slot[tab_row0 + j];
          if (OP == kGemm2Combine) scale = p.gate[row];       // Eq. 2: y = p_i(x) E_i(x)
        } else {
          row = tab_row0 + j;
        }
        tab[j] = make_int2(row, __float_as_int(scale));
      }
      __syncwarp();
      const int m = t.m0 + lg * 32 + lane;
      // (Read back from the hidden activations, a float per element, the mask made dgrad2 take 101 us where GEMM1 took 66; as a
      // word per column and 32 units, collected and spread by votes and shuffles, it cost either product another 15: 4096 tokens,
      // 512 x 2048, 16 experts.)
      const bool relu = (OP == kGemm1Relu || OP == kDgrad2Mask) && !p.plain, m_in = m < p.M;
      uint8_t* const mask_bytes = p.hmask + ((long long)t.e * p.hrows + (t.n0 + c0) / 8) * p.hcols + m;
      uint32_t live[kHalf / 32] = {};                         // a byte per 8 columns
      if (OP == kDgrad2Mask && relu && m_in) {
#pragma unroll
        for (int g = 0; g < kHalf / 8; ++g)
          if (8 * g < mine) live[g / 4] |= (uint32_t)mask_bytes[(long long)g * p.hcols] << (8 * (g % 4));
      }
      uint64_t sum[kSums];                                    // two columns each
#pragma unroll
      for (int j = 0; j < kSums; ++j) sum[j] = 0;
      const bool twice = t.apart() && t.K > 0;                // two chunks, both in the same accumulator
      const int chunks = twice ? 2 : (t.K + kK - 1) / kK;
      for (int c = 0; c < chunks; ++c) {
        ok = mbar_wait_warp<true>(dfull(d), d ? dphase1 : dphase0, abort_flag, p.status, 56);
        if (!ok) break;
        tc_fence_after();
        const uint32_t ta = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(d * kNMax + c0);
#pragma unroll
        for (int g = 0; g < (kHalf + 15) / 16; ++g) {
          if (16 * g < cols) {
            uint32_t v[16];
            tc_ld8(ta + 16 * g, v);
            tc_ld8(ta + 16 * g + 8, v + 8);
            tc_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j)
              sum[8 * g + j] = add2(sum[8 * g + j], pack2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(dempty(d));
        if (d) dphase1 ^= 1u; else dphase0 ^= 1u;
        if (!twice || c == 1) d ^= 1;
      }
      if (!ok) break;
      // Eight columns at a time, left where a tile has no more: the code is straight-line, the sums are registers, and fetching
      // it costs as much as executing it.  (Through shared memory and a loop over groups of 4 or 16 columns the weight gradients
      // of 4096 tokens, 512 x 2048, 16 experts took 83 us, like this 68.)
      constexpr bool kRows = OP == kGemm2Combine || OP == kDgrad1Scatter;        // a token's row per column
      float check = 0.f;                                      // NaN once a result is not finite
      auto group = [&](int g) {
        if (8 * g >= mine) return false;
        float v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 a = unpack2(mul2(sum[4 * g + j], pack2(kDown, kDown)));
          v[2 * j] = a.x; v[2 * j + 1] = a.y;
        }
        const int left = mine - 8 * g;
        const uint32_t on = live[g / 4] >> (8 * (g % 4));
        if (m_in) {
          float skip[8];
          if (kRows) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              skip[j] = p.res != nullptr && j < left ? p.res[(long long)tab[8 * g + j].x * p.ld_out + m] : 0.f;
          }
          if (OP == kGemm1Relu && relu) {
            uint32_t bits = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) bits |= v[j] > 0.f ? 1u << j : 0u;
            mask_bytes[(long long)g * p.hcols] = (uint8_t)bits;
          }
          long long at = (long long)(tab_row0 + 8 * g) * p.ld_out + m;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (j >= left) continue;
            float scale = 1.f;
            if (kRows) {
              const int2 r = tab[8 * g + j];
              at = (long long)r.x * p.ld_out + m;
              scale = __int_as_float(r.y);
            }
            check = fmaf(v[j], 0.f, check);
            finish<OP>(p, at, scale, v[j], on >> j & 1u, kRows ? skip[j] : 0.f);
            at += p.ld_out;
          }
        }
        return true;
      };
      static_assert(kHalf == 64, "eight groups of 8 columns");
      (void)(group(0) && group(1) && group(2) && group(3) && group(4) && group(5) && group(6) && group(7));
      if (check != check) redo<OP>(p, t.e, t.n0 + c0, t.K, m, mine, tab, abort_flag + 1);
      __syncwarp();
    }
  }

  // ---------------------------------------------------------------------------------------------- teardown
  // Dependents are let in only now.  No block fits beside one of these, so a trigger at the start overlaps nothing: it packs the
  // next kernel's blocks onto the few SMs that finish first.  Training steps with the trigger at the start / here, us: 4096 tokens,
  // 512 x 2048, 16 experts 557 / 530; 1024, 256 x 768, 8 125.2 / 121.1; 1024, 768 x 256, 8 148 / 136; 512, 512 x 2048, 8 with
  // expert dropout 230 / 214.
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

template <int OP>
int launch_op(const CUtensorMap& tmA, const CUtensorMap& tmB, const F32Problem& pr, cudaStream_t st) {
  if (cudaFuncSetAttribute(f32_expert_gemm_kernel<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kF32Smem) != cudaSuccess)
    return SWITCH_MOE_CUDA_ERROR;
  launch_k(f32_expert_gemm_kernel<OP>, dim3((unsigned)sm_count_or_default()), dim3(kF32Threads), kF32Smem, st, tmA, tmB, pr);
  return launch_status();
}

}  // namespace

// Which float32 products run here: those of at least 0.07 GFLOP (weight gradients 0.09; 2 rows d f), below which the 3 us that a
// launch has more to set up than an FMA kernel's (tensor memory, barriers, cold code) decide, and of them
// - token products with enough steps per tile to pay for its two ends.  Whole forward passes with the product here / on FMA,
//   medians over shapes of 16 to 65536 tokens, 1 to 256 experts, by contraction: GEMM1 8..15 1.21, 32..47 1.08, 64..71 1.03, 72..79
//   0.99, 96..127 0.94; GEMM2 8..15 1.16, 32..47 1.06, 80..95 0.97 (steps: up to 1.07), 96..111 0.97 (1.00), 128..191 0.90.  An output
//   no wider than half a tile leaves the rest of its MMAs idle: 64..95 1.06, 144..191 0.99 (up to 1.11), 192..255 0.94.  Tiles of
//   few tokens whose contraction is short, or output narrower still, are nothing but their ends: GEMM1 of 25 tokens per expert, 72 x
//   96, 226 experts 18.4 / 12.6 us; 22, 528 x 16, 194 30.7 / 22.5.
// - weight gradients of enough tokens to be more than writing the output: whole steps, tokens per expert 4..7 1.12, 12..15 1.07,
//   20..31 1.01, 32..47 0.99, 64..127 0.96, more 0.82.  (A tile walks its contraction on one SM at the rate of one FMA block of
//   64 x 64.  Where outputs have few tiles the FMA kernels are up to a fifth faster by themselves, but in a row of launches their
//   few blocks crowd onto the first free SMs: 13764 tokens, 16 x 472, 2 GEGLU experts, a step 463 us here, 836 there.)
// On 660 shapes no call is slower by more than 2% than with all products on FMA; forward passes take 0.73, steps 0.70 of its time
// in the mean.  GEMM1 and dgrad2 always go together: the mask that one leaves is the one that the other reads.
bool f32_on_tensor_cores(GemmOp op, const Shape& s) {
  if (!s.f32_tc) return false;
  const double rows = s.Tv < (double)s.E * s.C ? s.Tv : (double)s.E * s.C, flops = 2.0 * rows * s.d * s.f;
  if (op == kWgrad2 || op == kWgrad1) return flops >= 9e7 && rows >= 24.0 * s.E;
  const bool first = op == kGemm1Relu || op == kDgrad2Mask;            // d deep, f wide; the other token products f deep, d wide
  const int steps = first ? s.d : op == kGemm2Combine ? s.f : s.fin, width = first ? s.f : s.d;
  const double tiles = (double)s.E * ceil(rows / s.E / kNMax) * ((width + kM - 1) / kM), tile_flops = 2.0 * rows * width * steps / tiles;
  return flops >= 7e7 && steps >= (width <= 64 ? 192 : first ? 72 : 96) && (tile_flops >= 5e5 || (steps >= 128 && width >= 32));
}

int launch_f32_gemm(GemmOp op, const Shape& s, const Plan& p, const GemmArgs& a, void* ws, cudaStream_t st) {
  if (!f32_on_tensor_cores(op, s)) return launch_simt_gemm(op, s, p, a, ws, st);
  const long long C = s.C, d = s.d, f = s.f, fin = s.fin;      // fin: columns of W_in, f or 2 f for GEGLU experts
  float* xd = ws_ptr<float>(ws, p.xd); float* h = ws_ptr<float>(ws, p.h);
  float* dyd = ws_ptr<float>(ws, p.dyd); float* dh = ws_ptr<float>(ws, p.dh);
  float* ab = ws_ptr<float>(ws, p.ab);
  float* du = s.geglu ? ws_ptr<float>(ws, p.dab) : dh;         // gradient of the pre-activation(s)
  const float* W_in = static_cast<const float*>(a.W_in); const float* W_out = static_cast<const float*>(a.W_out);
  F32Problem pr{};
  pr.E = s.E; pr.C = s.C;
  pr.kept = ws_ptr<int>(ws, p.kept);
  pr.token_of_slot = ws_ptr<int>(ws, p.token_of_slot);
  pr.gate = ws_ptr<float>(ws, p.gate);
  pr.status = ws_ptr<int>(ws, p.status);
  pr.plain = s.geglu;
  pr.hmask = ws_ptr<uint8_t>(ws, p.hmask); pr.hrows = (s.C + 15) / 16 * 2; pr.hcols = (s.f + 31) / 32 * 32;
  // operand [E][rows][cols], which of the two axes is the contraction, and the output
  auto A = [&](const float* q, long long rows, long long cols, bool k_major) {
    pr.A = q; pr.a_es = rows * cols; pr.a_ms = k_major ? cols : 1; pr.a_ks = k_major ? 1 : cols;
    pr.M = (int)(k_major ? rows : cols);
  };
  auto B = [&](const float* q, long long cols, bool k_major) {
    pr.B = q; pr.b_es = C * cols; pr.b_ns = k_major ? cols : 1; pr.b_ks = k_major ? 1 : cols;
    pr.N = k_major ? -1 : (int)cols;
    pr.K = k_major ? (int)cols : -1;
  };
  auto out = [&](void* q, long long ld) { pr.out = static_cast<float*>(q); pr.ld_out = (int)ld; };
  switch (op) {
    case kGemm1Relu: A(W_in, d, fin, false); B(xd, d, true); out(s.geglu ? ab : h, fin); break;
    case kGemm2Combine: A(W_out, f, d, false); B(h, f, true); out(a.y, d); break;
    case kDgrad2Mask: A(W_out, f, d, true); B(dyd, d, true); out(dh, f); break;
    case kDgrad1Scatter: A(W_in, d, fin, true); B(du, fin, true); out(a.dx, d); break;
    case kWgrad2: A(dyd, C, d, false); B(h, f, false); out(a.dW_out, d); break;
    case kWgrad1: A(du, C, fin, false); B(xd, d, false); out(a.dW_in, fin); break;
    default: return SWITCH_MOE_INVALID_ARGUMENT;
  }
  // (top-2 routing adds the skip path where the two assignments' rows are summed, not here)
  if (s.residual && !s.top2 && op == kGemm2Combine) {
    pr.res = static_cast<const float*>(a.x);
    pr.out2 = ws_ptr<float>(ws, p.layer_y);
  }
  if (s.residual && !s.top2 && op == kDgrad1Scatter) pr.res = static_cast<const float*>(a.dy);
  pr.n_mtiles = (pr.M + kM - 1) / kM;
  pr.n_ntiles = pr.N < 0 ? 0 : (pr.N + kNFix - 1) / kNFix;
  const bool a_k = pr.a_ks == 1;
  CUtensorMap tmA, tmB;
  const long long a_cols = a_k ? pr.a_ms : pr.a_ks, b_cols = pr.N < 0 ? pr.b_ns : pr.b_ks;
  if (make_map_f32(&tmA, pr.A, s.E, pr.a_es / a_cols, a_cols, a_k ? kK : kM, a_k ? kM : kK) != SWITCH_MOE_OK ||
      make_map_f32(&tmB, pr.B, s.E, C, b_cols, pr.N < 0 ? kK : kNFix, pr.N < 0 ? kBoxRows : kK) != SWITCH_MOE_OK)
    return SWITCH_MOE_CUDA_ERROR;
  switch (op) {
    case kGemm1Relu: return launch_op<kGemm1Relu>(tmA, tmB, pr, st);
    case kGemm2Combine: return launch_op<kGemm2Combine>(tmA, tmB, pr, st);
    case kDgrad2Mask: return launch_op<kDgrad2Mask>(tmA, tmB, pr, st);
    case kDgrad1Scatter: return launch_op<kDgrad1Scatter>(tmA, tmB, pr, st);
    case kWgrad2: return launch_op<kWgrad2>(tmA, tmB, pr, st);
    default: return launch_op<kWgrad1>(tmA, tmB, pr, st);
  }
}

}  // namespace swmoe
