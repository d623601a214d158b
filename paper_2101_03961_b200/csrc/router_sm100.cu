// Router of the Switch FFN layer on the B200 tensor cores with float32-grade accuracy (Section 2.4: the router is the
// part of the layer that must not run in bfloat16).
//
// x is bfloat16, hence exact in float32.  A float32 operand w is written as the sum of two bfloat16 numbers
// (w = hi + mid up to 2^-18 relative: each part carries 8 significant bits and a third part would add what the 1e-5
// tolerance of the router never sees), every bf16 x bf16 product is exact in float32, and tcgen05 accumulates in
// float32.  So
//   logits   h = x W_r            = x (W_hi + W_mid)                              (Section 2.1; Eq. 1 follows in the epilogue)
//   dW_r       = x^T dh           = x^T (dh_hi + dh_mid)                          (contraction over tokens, split over CTAs)
//   dx_router  = dh W_r^T         ~ dh_hi W_hi^T + dh_hi W_mid^T + dh_mid W_hi^T  (the output is bfloat16: 2^-16 suffices)
// are bfloat16 tensor-core products whose results agree with the float32 definition to a few 1e-6 relative, and the
// router stops being bound by the FP32 FMA pipes (E flop per byte of x) and becomes a streaming kernel.
//
// The forward epilogue keeps one token per thread (a TMEM lane holds all E logits of a token): softmax, top-1 with
// lowest-index ties and the gate need no cross-thread traffic; the column sums of p for Eq. 6 use warp shuffles.
#include "tc_common.cuh"

namespace swmoe {
using namespace tc;
namespace {

// ------------------------------------------------------------------------------------------------------------------
// Forward router.  A CTA works on one or two 128-token tiles at a time that share every staged k-block of W_r; these
// tokens are one row of the dispatch plan's histogram table and of the P-sum partials, which the epilogue leaves: the
// block's histogram of expert choices (Section 2.2: the counts behind Eq. 3's capacity cut and Eq. 5's f) and its
// column sums of the probabilities (Eq. 6's P), both in a fixed order.
//
// What bounds it: the k-loop streams x and W_r into one CTA per SM (memory latency for few tokens, bandwidth for many),
// and the epilogue runs once or a few times per launch, so its instructions come cold from memory: straight-line code
// over all E logits of a token paid more for fetching instructions than for executing them.  It is therefore three short
// loops over chunks of 32 logits, with the logits (and then their exponentials) kept in tensor memory between the
// passes, which also leaves no limit on E short of the accumulator's 256 columns.  Straight-line code took 39 us where this
// takes 19 (256 tokens, d_model 768, 128 experts).
//
// Probabilities and noise cross between memory order and token-per-lane order through shared memory.  With every lane
// storing its own row, 16 bytes of 32 different rows at a time, the stores alone cost 6 of 25 us (32768 tokens, d_model
// 768, 128 experts) and 12 of 29 (65536, 256, 128), the noise 10 of 40 (20011, 512, 200); this way all takes 22, 23 and 38
// (7 of the last for expf).  Twice as many epilogue warps, each with half of the experts, gained nothing.
struct RouterFwdParams {
  int T, d, E, Epad64, n_blocks, k_blocks, b_atoms, stages, stage_bytes;
  int tiles;                 // 128-token tiles per block: 1 or 2
  int stage_parts;           // parts of W_r staged with each x block: both (E <= 128), or one at a time
  int rot_wrap;              // E <= 128: the contraction of a 256-token block starts at k-block (block % rot_wrap) % k_blocks
  int acc_step, n_acc;       // TMEM columns of one accumulator set (all tiles), and how many sets fit (1 or 2)
  const float* bias; const float* noise; float* probs; int* expert_index; float* gate;
  float* psum_partial;       // [n_blocks][E]: column sums of p over each block's tokens
  int* hist;                 // [n_blocks][E]: tokens of each block per expert
  int* status;
};
constexpr int kRFParts = 2;                                    // W_r = hi + mid (bfloat16 each): exact to 2^-18 relative
constexpr int kRFMaxStages = 6;
constexpr int kRFRingBytes = 196608;                           // 192 KB of operand stages
constexpr int kRFOutBytes = 8 * kMaxExperts * 4;               // the epilogue warps' column sums
constexpr int kRFTailBytes = 256 + kMaxExperts * 4;            // barriers, TMEM pointer, flags; the block's histogram
constexpr int kRFTurnBytes = 8 * 32 * 16 * 4;                  // per epilogue warp: 32 tokens x 16 experts
constexpr int kRFSmemBytes = 1024 + kRFRingBytes + kRFOutBytes + kRFTailBytes + kRFTurnBytes;
constexpr int kRFThreads = 64 + 2 * 128;                       // TMA warp, MMA warp, 4 epilogue warps per token tile

__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <bool kWide>                                          // more than 128 experts
__global__ void __launch_bounds__(kRFThreads, 1)
router_fwd_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const RouterFwdParams p) {
  pdl_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + kRFRingBytes + kRFOutBytes;
  uint8_t* bar_gen = smem_gen + kRFRingBytes + kRFOutBytes;
  const uint32_t full0 = bar_base, empty0 = bar_base + 8u * kRFMaxStages;
  const uint32_t tfull0 = bar_base + 16u * kRFMaxStages, tempty0 = tfull0 + 16u;
  volatile uint32_t* tmem_ptr_s = reinterpret_cast<volatile uint32_t*>(bar_gen + 16 * kRFMaxStages + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_gen + 16 * kRFMaxStages + 36);
  volatile int* fail_s = reinterpret_cast<volatile int*>(bar_gen + 16 * kRFMaxStages + 40);   // an epilogue warp gave up
  int* hist_s = reinterpret_cast<int*>(bar_gen + 256);         // kMaxExperts counters
  const int warp = uniform_warp_id(), lane = threadIdx.x & 31;
  const int n_epi = 128 * p.tiles;                             // epilogue threads of this launch

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRFMaxStages; ++s) { mbar_init(full0 + 8u * s, 1); mbar_init(empty0 + 8u * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull0 + 8u * a, 1); mbar_init(tempty0 + 8u * a, 4 * p.tiles); }
    *abort_flag = 0;
    *fail_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_ptr_s))), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = threadIdx.x; i < kMaxExperts; i += blockDim.x) hist_s[i] = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_s;
  pdl_wait();                                                 // the previous kernel's results are needed from here on
  const int n_blocks = p.n_blocks, kbs = p.k_blocks, b_atoms = p.b_atoms, tiles = p.tiles, stage_parts = p.stage_parts;
  const int n_iter = stage_parts == kRFParts ? kbs : kRFParts * kbs;   // staged blocks per tile
  const uint32_t n_stages = (uint32_t)p.stages, stage_bytes = (uint32_t)p.stage_bytes;

  if (warp == 0) {
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < n_blocks && ok; id += gridDim.x) {
      const int m0 = id * tiles * kTileM;
      // Blocks walk the contraction in rotated order: otherwise all CTAs would ask the same L2 lines of W_r at the same
      // moment.  The order decides the last bit of a logit, hence near-ties of the top-1: it depends on the token alone,
      // not on how many tiles a CTA has.
      const int rot = p.rot_wrap > 0 ? (m0 / (2 * kTileM)) % p.rot_wrap % kbs : 0;
#pragma unroll 1
      for (int it = 0; it < n_iter; ++it) {
        ok = mbar_wait_warp(empty0 + 8u * stage, phase ^ 1u, abort_flag, p.status, 31);
        if (!ok) break;
        const uint32_t a_dst = smem_base + stage * stage_bytes, fb = full0 + 8u * stage;
        const int part0 = it >= kbs ? 1 : 0;                   // one part at a time: all of hi, then all of mid
        int kr = it - part0 * kbs + rot;
        if (kr >= kbs) kr -= kbs;
        if (elect_one()) {
          mbar_arrive_expect_tx(fb, stage_bytes);
          tma_load_3d(a_dst, &tmA, fb, kr * kBK, m0, 0);                              // x tiles [128 tok][64 k]
          if (tiles > 1) tma_load_3d(a_dst + kABytes, &tmA, fb, kr * kBK, m0 + kTileM, 0);
          uint32_t b_dst = a_dst + tiles * kABytes;
          for (int part = part0; part < part0 + stage_parts; ++part)
            for (int j = 0; j < b_atoms; ++j, b_dst += kAtomBytes)                     // W part [64 k][64 e]
              tma_load_3d(b_dst, &tmB, fb, 64 * j, kr * kBK, part);
        }
        if (++stage == n_stages) { stage = 0; phase ^= 1u; }
      }
    }
    if (*abort_flag != 0) {
      const long long t0 = clock64();
      while (clock64() - t0 < 4000000ll) __nanosleep(1000);
    }
  } else if (warp == 1) {
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(p.Epad64 >> 3) << 17) |
                           ((uint32_t)(kTileM >> 4) << 24);
    const uint64_t a_desc0 = make_smem_desc(smem_base, 16u, 1024u);
    const uint64_t b_desc0 = make_smem_desc(smem_base + tiles * kABytes, kAtomBytes, 1024u);
    const uint32_t part_step = (uint32_t)(b_atoms * kAtomBytes) >> 4;
    const uint32_t tile_step = (uint32_t)(p.acc_step / tiles);
    uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < n_blocks && ok; id += gridDim.x) {
      ok = mbar_wait_warp(tempty0 + 8u * acc, acc_phase ^ 1u, abort_flag, p.status, 32);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + acc * (uint32_t)p.acc_step;
#pragma unroll 1
      for (int it = 0; it < n_iter; ++it) {
        ok = mbar_wait_warp(full0 + 8u * stage, phase, abort_flag, p.status, 33);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ad = a_desc0 + (uint64_t)(stage * (stage_bytes >> 4));
        const uint64_t bd0 = b_desc0 + (uint64_t)(stage * (stage_bytes >> 4));
        if (elect_one()) {
#pragma unroll 1
          for (int tile = 0; tile < tiles; ++tile) {
            uint64_t bd = bd0;
#pragma unroll 1
            for (int part = 0; part < stage_parts; ++part, bd += part_step) {
#pragma unroll
              for (int ks = 0; ks < kBK / kUmmaK; ++ks)
                tc_mma_bf16(d_tmem + tile * tile_step, ad + (uint64_t)(tile * (kABytes >> 4) + ks * ((kUmmaK * 2) >> 4)),
                            bd + (uint64_t)(ks * ((kUmmaK * 128) >> 4)), idesc, (it > 0 || part > 0 || ks > 0) ? 1u : 0u);
            }
          }
          tc_commit(empty0 + 8u * stage);
          if (it == n_iter - 1) tc_commit(tfull0 + 8u * acc);
        }
        if (++stage == n_stages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      if (++acc == (uint32_t)p.n_acc) { acc = 0; acc_phase ^= 1u; }
    }
  } else {
    const int lg = warp & 3, ti = (warp - 2) >> 2;            // TMEM lane group; which of the token tiles
    const int et = threadIdx.x - 64;                          // 0 .. n_epi - 1 over the epilogue warps
    const int nch = (p.E + 31) >> 5;                          // chunks of 32 logits
    const bool vec_rows = (p.E & 3) == 0;
    const bool vec_noise = vec_rows && (reinterpret_cast<uintptr_t>(p.noise) & 15u) == 0;   // (the caller's own array)
    float* sums = reinterpret_cast<float*>(smem_gen + kRFRingBytes);
    // Rows of probabilities and noise move between memory and the lanes that own them through this warp's tile of 32 tokens x
    // 16 experts (64 bytes per row, 16-byte pieces exchanged by the row): lane l owns row l, and in memory order it handles
    // piece l % 4 of rows l / 4, l / 4 + 8, ...
    float* turn = reinterpret_cast<float*>(bar_gen + kRFTailBytes) + (warp - 2) * 512;
    float4* own = reinterpret_cast<float4*>(turn + lane * 16);
    const int own_x = (lane >> 1) & 3, row0 = lane >> 2, piece = lane & 3;
    float4* mem = reinterpret_cast<float4*>(turn + row0 * 16) + (piece ^ ((lane >> 3) & 3));     // row row0 + 8 k: mem[32 k]
    uint32_t acc = 0, acc_phase = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < n_blocks; id += gridDim.x) {
      const int tok = (id * tiles + ti) * kTileM + lg * 32 + lane;       // the token whose logits this lane holds
      const int tok0 = tok - lane + row0;                     // this lane's first row in memory order
      float4 z[8];                                            // a chunk of noise, requested one chunk ahead
      auto load_noise = [&](int c) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int e = c * 32 + (k >> 2) * 16 + piece * 4, t = tok0 + 8 * (k & 3);
          const float* src = p.noise + (size_t)t * p.E + e;
          z[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (t < p.T && vec_noise) {
            if (e < p.E) z[k] = *reinterpret_cast<const float4*>(src);
          } else if (t < p.T) {
            if (e < p.E) z[k].x = src[0];
            if (e + 1 < p.E) z[k].y = src[1];
            if (e + 2 < p.E) z[k].z = src[2];
            if (e + 3 < p.E) z[k].w = src[3];
          }
        }
      };
      if (p.noise != nullptr) load_noise(0);
      ok = mbar_wait_warp(tfull0 + 8u * acc, acc_phase, abort_flag, p.status, 34);
      // the epilogue warps meet at barriers below: all of them leave together if the bounded wait of any gave up
      if (!ok && lane == 0) *fail_s = 1;
      asm volatile("bar.sync 1, %0;" ::"r"(n_epi) : "memory");
      if (*fail_s != 0) break;
      tc_fence_after();
      const uint32_t t_addr = tmem_base + ((uint32_t)(lg * 32) << 16) + acc * (uint32_t)p.acc_step +
                              (uint32_t)(ti * (p.acc_step / tiles));
      const bool live = tok < p.T;
      // Pass 1: Eq. 1's maximum and top-1 (first maximum wins) as four interleaved chains, all within this lane.
      float mq[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      int aq[4] = {0, 1, 2, 3};
#pragma unroll 1
      for (int c = 0; c < nch; ++c) {
        uint32_t v[32];
        tc_ld32(t_addr + c * 32, v);
        tc_wait_ld();
        if (p.bias != nullptr || p.noise != nullptr) {        // a constant per expert; exploration noise (an input)
          if (p.bias != nullptr) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (c * 32 + i < p.E) v[i] = __float_as_uint(__uint_as_float(v[i]) + p.bias[c * 32 + i]);
          }
          if (p.noise != nullptr) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
              for (int k = 0; k < 4; ++k) mem[32 * k] = z[4 * h + k];
              __syncwarp();
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float4 n = own[q ^ own_x];
                const int i = 16 * h + 4 * q;
                v[i] = __float_as_uint(__uint_as_float(v[i]) + n.x);
                v[i + 1] = __float_as_uint(__uint_as_float(v[i + 1]) + n.y);
                v[i + 2] = __float_as_uint(__uint_as_float(v[i + 2]) + n.z);
                v[i + 3] = __float_as_uint(__uint_as_float(v[i + 3]) + n.w);
              }
              __syncwarp();
            }
            if (c + 1 < nch) load_noise(c + 1);
          }
          tc_st32(t_addr + c * 32, v);
          tc_wait_st();
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int e = c * 32 + i;
          const float h = __uint_as_float(v[i]);
          if (e < p.E && h > mq[i & 3]) { mq[i & 3] = h; aq[i & 3] = e; }
        }
      }
      float m = mq[0];
      int am = aq[0];
#pragma unroll
      for (int u = 1; u < 4; ++u)
        if (mq[u] > m || (mq[u] == m && aq[u] < am)) { m = mq[u]; am = aq[u]; }
      // Pass 2: exponentials, back into tensor memory, and their sum.  Up to 128 experts the hardware's exp2 of an argument
      // scaled in the same multiply-add: relative error below 1e-6 for h within 10 of m, whatever m is, because the rounding
      // of m log2(e) is one factor of the whole row and leaves with the sum -- it has to be in the gate's numerator too, so
      // the gate is formed like the probability it is, from the maximum's own exponential.  Above 128 experts expf of the
      // difference and one running sum: 2e-7 of the exponential instead of 1e-6, for 7 us (20011 tokens, d_model 512, 200
      // experts: training step 562 us with the first form, 569 with this one).
      float sum, top;                                          // top: the maximum's own exponential
      if constexpr (kWide) {
        sum = 0.f;
        top = 1.f;
#pragma unroll 1
        for (int c = 0; c < nch; ++c) {
          uint32_t v[32];
          tc_ld32(t_addr + c * 32, v);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float ex = c * 32 + i < p.E ? expf(__uint_as_float(v[i]) - m) : 0.f;
            sum += ex;
            v[i] = __float_as_uint(ex);
          }
          tc_st32(t_addr + c * 32, v);
        }
      } else {
        const float kLog2e = 1.4426950408889634f;
        const float ms = m * kLog2e;
        auto exp_minus_m = [&](float h) {
          float ex;
          asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(fmaf(h, kLog2e, -ms)));
          return ex;
        };
        float sq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int c = 0; c < nch; ++c) {
          uint32_t v[32];
          tc_ld32(t_addr + c * 32, v);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float ex = c * 32 + i < p.E ? exp_minus_m(__uint_as_float(v[i])) : 0.f;
            sq[i & 3] += ex;
            v[i] = __float_as_uint(ex);
          }
          tc_st32(t_addr + c * 32, v);
        }
        sum = (sq[0] + sq[1]) + (sq[2] + sq[3]);
        top = exp_minus_m(m);
      }
      tc_wait_st();
      const float inv = 1.f / sum;
      if (live) {
        p.expert_index[tok] = am;
        p.gate[tok] = top * inv;
        atomicAdd(&hist_s[am], 1);                            // integer counts: the order does not matter
      }
      // Pass 3: the probabilities, in memory order, and their column sums over the warp's 32 tokens (Eq. 6's sum over tokens):
      // over the four rows of a lane, then over the lanes with the same columns, in a fixed order.
      const float scale = live ? inv : 0.f;                    // rows past the last token add nothing to the sums
#pragma unroll 1
      for (int c = 0; c < p.E; c += 16) {
        uint32_t v[16];
        tc_ld16(t_addr + c, v);
        tc_wait_ld();
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q)
          own[q ^ own_x] = make_float4(__uint_as_float(v[4 * q]) * scale, __uint_as_float(v[4 * q + 1]) * scale,
                                       __uint_as_float(v[4 * q + 2]) * scale, __uint_as_float(v[4 * q + 3]) * scale);
        __syncwarp();
        const int e = c + piece * 4;
        float4 w[4], sum4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          w[k] = mem[32 * k];
          float* dst = p.probs + (size_t)(tok0 + 8 * k) * p.E + e;
          if (tok0 + 8 * k < p.T && vec_rows) {
            if (e < p.E) *reinterpret_cast<float4*>(dst) = w[k];
          } else if (tok0 + 8 * k < p.T) {
            if (e < p.E) dst[0] = w[k].x;
            if (e + 1 < p.E) dst[1] = w[k].y;
            if (e + 2 < p.E) dst[2] = w[k].z;
            if (e + 3 < p.E) dst[3] = w[k].w;
          }
        }
        sum4.x = (w[0].x + w[1].x) + (w[2].x + w[3].x);
        sum4.y = (w[0].y + w[1].y) + (w[2].y + w[3].y);
        sum4.z = (w[0].z + w[1].z) + (w[2].z + w[3].z);
        sum4.w = (w[0].w + w[1].w) + (w[2].w + w[3].w);
#pragma unroll
        for (int step = 4; step <= 16; step <<= 1) {
          sum4.x += __shfl_xor_sync(0xffffffffu, sum4.x, step);
          sum4.y += __shfl_xor_sync(0xffffffffu, sum4.y, step);
          sum4.z += __shfl_xor_sync(0xffffffffu, sum4.z, step);
          sum4.w += __shfl_xor_sync(0xffffffffu, sum4.w, step);
        }
        if (row0 == 0) *reinterpret_cast<float4*>(sums + (warp - 2) * kMaxExperts + e) = sum4;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8u * acc);         // the accumulator is free
      asm volatile("bar.sync 1, %0;" ::"r"(n_epi) : "memory");   // the epilogue warps: histogram and column sums complete
      for (int e = et; e < p.E; e += n_epi) {
        float v = sums[e];                                     // the warps' sums, added in warp order
        for (int w = 1; w < 4 * tiles; ++w) v += sums[w * kMaxExperts + e];
        p.psum_partial[(size_t)id * p.E + e] = v;
        p.hist[(size_t)id * p.E + e] = hist_s[e];
        hist_s[e] = 0;
      }
      asm volatile("bar.sync 1, %0;" ::"r"(n_epi) : "memory");   // before the next round reuses the sums and the counters
      if (++acc == (uint32_t)p.n_acc) { acc = 0; acc_phase ^= 1u; }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// ------------------------------------------------------------------------------------------------------------------
// Backward router: dW_r = x^T dh and dx += dh W_r^T in one pass over the tokens.
//
// A CTA owns a block of 128 columns of d_model and walks its share of the 128-token tiles.  Per tile it stages the x
// block [128 tokens][128 columns] and, one 16 KB block of 64 experts at a time, both bfloat16 parts of the logit
// gradients; the parts of W_r for its columns stay in shared memory for the CTA's life.  A staged block of dh serves both
// products (as the K-major A operand of dh W_r^T and the N-major B operand of x^T dh: the same bytes).  dW_r accumulates
// in tensor memory over all the CTA's tiles and leaves once, as one partial per CTA; dx has two accumulators, so the
// epilogue of a tile (read dx, add, round, store) overlaps the next tile's products.
//
// What bounds it: every column block reads all of dh from L2 (211 MB into the SMs at 32768 tokens, d 768, E 128; with the
// stores, the dx reads and most MMAs taken out the kernel still took 24 of its 37 us, i.e. 9 TB/s).  More x stages, a longer
// ring or x requested into L2 ahead changed nothing (one x stage: 47 us).  With its neighbours (logit gradients before,
// reduction of the partials after), and in brackets with one kernel per product: 32768 tokens, d 768, E 128 67 us (82); 65536
// tokens, d 256, E 128, jitter 63 (83); 16384 tokens, d 768, E 64 34 (45); 20011 tokens, d 512, E 200 63 (61).
struct RouterBwdParams {
  int T, d, E, ka;           // ka: blocks of 64 experts (1..4)
  int n_mtiles, n_cols, splits, x_stages, ring;
  float* partial; __nv_bfloat16* dx; const int* slot; int accumulate; const __nv_bfloat16* jitter_u;
  int* status;
};
constexpr int kRBThreads = 320;                                // TMA warp, MMA warp, 8 epilogue warps
constexpr int kRBBlock = kTileM * 128;                         // 128 rows of 128 bytes: a block of dh, of W_r, half of x
constexpr int kRBStageOut = 8 * 16 * 128;                      // epilogue transposition, 16 rows of 128 bytes per warp
constexpr int kRBOperandBytes = 208 * 1024;                    // W_r parts, x stages, ring of dh blocks
constexpr int kRBMaxRing = 6;
constexpr int kRBSmemBytes = 1024 + kRBOperandBytes + kRBStageOut + 256;
constexpr int kRBDwrCol = 256;                                 // first TMEM column of the dW_r accumulator

template <bool kJitter>
__global__ void __launch_bounds__(kRBThreads, 1)
router_bwd_tc_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmH,
                     const __grid_constant__ CUtensorMap tmW, const RouterBwdParams p) {
  pdl_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + kRBOperandBytes + kRBStageOut;
  uint8_t* bar_gen = smem_gen + kRBOperandBytes + kRBStageOut;
  // barriers: ring full[6] | ring empty[6] | x full[2] | x empty[2] | dx full[2] | dx empty[2] | W_r full | dW_r full
  const uint32_t rfull0 = bar_base, rempty0 = rfull0 + 8u * kRBMaxRing, xfull0 = rempty0 + 8u * kRBMaxRing;
  const uint32_t xempty0 = xfull0 + 16u, tfull0 = xfull0 + 32u, tempty0 = xfull0 + 48u, wfull = xfull0 + 64u, dfull = xfull0 + 72u;
  volatile uint32_t* tmem_ptr_s = reinterpret_cast<volatile uint32_t*>(bar_gen + 16 * kRBMaxRing + 80);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_gen + 16 * kRBMaxRing + 84);
  const int warp = uniform_warp_id(), lane = threadIdx.x & 31;
  const int col_block = (int)(blockIdx.x % (unsigned)p.n_cols), split = (int)(blockIdx.x / (unsigned)p.n_cols);
  const int n0 = col_block * 128, ka = p.ka;
  const uint32_t w_s = smem_base, x_s = w_s + 2u * ka * kRBBlock, ring_s = x_s + 2u * p.x_stages * kRBBlock;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRBMaxRing; ++s) { mbar_init(rfull0 + 8u * s, 1); mbar_init(rempty0 + 8u * s, 1); }
    for (int s = 0; s < 2; ++s) {
      mbar_init(xfull0 + 8u * s, 1); mbar_init(xempty0 + 8u * s, 1);
      mbar_init(tfull0 + 8u * s, 1); mbar_init(tempty0 + 8u * s, 8);
    }
    mbar_init(wfull, 1);
    mbar_init(dfull, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_ptr_s))), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_s;
  pdl_wait();                                                 // the previous kernel's results are needed from here on

  if (warp == 0) {
    // ------------------------------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      mbar_arrive_expect_tx(wfull, 2u * (uint32_t)ka * kRBBlock);
      for (int part = 0; part < 2; ++part)
        for (int kk = 0; kk < ka; ++kk) tma_load_3d(w_s + (uint32_t)(part * ka + kk) * kRBBlock, &tmW, wfull, kk * 64, n0, part);
    }
    __syncwarp();
    uint32_t slot_i = 0, slot_phase = 0, xs = 0, x_phase = 0;
    bool ok = true;
    for (int tile = split; tile < p.n_mtiles && ok; tile += p.splits) {
      const int m0 = tile * kTileM;
      ok = mbar_wait_warp(xempty0 + 8u * xs, x_phase ^ 1u, abort_flag, p.status, 11);
      if (!ok) break;
      if (elect_one()) {
        mbar_arrive_expect_tx(xfull0 + 8u * xs, 2u * kRBBlock);
        tma_load_3d(x_s + 2u * xs * kRBBlock, &tmX, xfull0 + 8u * xs, n0, m0, 0);              // x [128 tok][64 columns]
        tma_load_3d(x_s + (2u * xs + 1u) * kRBBlock, &tmX, xfull0 + 8u * xs, n0 + 64, m0, 0);
      }
      if (++xs == (uint32_t)p.x_stages) { xs = 0; x_phase ^= 1u; }
#pragma unroll 1
      for (int b = 0; b < 2 * ka; ++b) {
        ok = mbar_wait_warp(rempty0 + 8u * slot_i, slot_phase ^ 1u, abort_flag, p.status, 12);
        if (!ok) break;
        const int part = b >= ka ? 1 : 0;
        if (elect_one()) {
          mbar_arrive_expect_tx(rfull0 + 8u * slot_i, kRBBlock);
          tma_load_3d(ring_s + slot_i * kRBBlock, &tmH, rfull0 + 8u * slot_i, (b - part * ka) * 64, m0, part);
        }
        if (++slot_i == (uint32_t)p.ring) { slot_i = 0; slot_phase ^= 1u; }
      }
    }
    if (*abort_flag != 0) {
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------------------------ MMA issuer
    constexpr uint32_t idesc_dx = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
    constexpr uint32_t idesc_dw = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((64u >> 3) << 17) |
                                  ((uint32_t)(kTileM >> 4) << 24);
    uint32_t slot_i = 0, slot_phase = 0, xs = 0, x_phase = 0, acc = 0, acc_phase = 0;
    bool first = true;
    bool ok = mbar_wait_warp(wfull, 0u, abort_flag, p.status, 15);
    for (int tile = split; tile < p.n_mtiles && ok; tile += p.splits) {
      ok = mbar_wait_warp(tempty0 + 8u * acc, acc_phase ^ 1u, abort_flag, p.status, 13) &&
           mbar_wait_warp(xfull0 + 8u * xs, x_phase, abort_flag, p.status, 16);
      if (!ok) break;
      tc_fence_after();
      const uint64_t xd = make_smem_desc(x_s + 2u * xs * kRBBlock, kRBBlock, 1024u);           // x^T: two 64-column atoms
#pragma unroll 1
      for (int b = 0; b < 2 * ka; ++b) {
        ok = mbar_wait_warp(rfull0 + 8u * slot_i, slot_phase, abort_flag, p.status, 17);
        if (!ok) break;
        tc_fence_after();
        const int part = b >= ka ? 1 : 0, kk = b - part * ka;
        const uint32_t blk = ring_s + slot_i * kRBBlock;
        if (elect_one()) {
          // dx: dh_hi meets W_hi and W_mid, dh_mid meets W_hi (the output is bfloat16: 2^-16 suffices)
          const uint64_t ad = make_smem_desc(blk, 16u, 1024u);
#pragma unroll 1
          for (int wp = 0; wp < 2 - part; ++wp) {
            const uint64_t bd = make_smem_desc(w_s + (uint32_t)(wp * ka + kk) * kRBBlock, 16u, 1024u);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              tc_mma_bf16(tmem_base + acc * 128u, ad + ks * 2, bd + ks * 2, idesc_dx, (b > 0 || wp > 0 || ks > 0) ? 1u : 0u);
          }
          // dW_r, columns 64 kk ..: contraction over the tile's 128 tokens, 16 at a time
          const uint64_t hd = make_smem_desc(blk, kRBBlock, 1024u);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            tc_mma_bf16(tmem_base + kRBDwrCol + 64u * kk, xd + ks * 128, hd + ks * 128, idesc_dw,
                        (!first || part > 0 || ks > 0) ? 1u : 0u);
          tc_commit(rempty0 + 8u * slot_i);
          if (b == 2 * ka - 1) {
            tc_commit(xempty0 + 8u * xs);
            tc_commit(tfull0 + 8u * acc);
          }
        }
        if (++slot_i == (uint32_t)p.ring) { slot_i = 0; slot_phase ^= 1u; }
      }
      if (!ok) break;
      first = false;
      if (++xs == (uint32_t)p.x_stages) { xs = 0; x_phase ^= 1u; }
      acc ^= 1u;
      if (acc == 0) acc_phase ^= 1u;
    }
    if (ok && elect_one()) tc_commit(dfull);
    __syncwarp();
  } else {
    // ------------------------------------------------------------------------------------------ epilogue warps
    const int lg = warp & 3, half = (warp - 2) >> 2;          // TMEM lane group (32 tokens); which 64 columns
    uint8_t* stage_gen = smem_gen + kRBOperandBytes + (warp - 2) * 2048;
    const int col = n0 + half * 64 + (lane & 7) * 8;          // this lane's 8 columns in every store
    const bool col_ok = col < p.d;
    const uint32_t t_lane = tmem_base + ((uint32_t)(lg * 32) << 16);
    uint32_t acc = 0, acc_phase = 0;
    bool ok = true;
    // Store `it` of this lane writes token tok0 + 4 it + lane / 8.  What those rows hold so far is requested a tile ahead:
    // the loads of the next tile are in flight while this one's sums are formed and its accumulator is awaited.  (Under
    // jitter the factors take those registers: requested at the tile's start.)
    unsigned add_rows = 0;
    uint4 prev[8], uu[kJitter ? 8 : 1];
    auto fetch_rows = [&](int tile) {
      const int tok0 = tile * kTileM + lg * 32, mine = tok0 + lane;
      add_rows = __ballot_sync(0xffffffffu, p.accumulate != 0 && mine < p.T && (p.accumulate == 2 || p.slot[mine] >= 0));
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int row = it * 4 + (lane >> 3);
        const size_t off = (size_t)(tok0 + row) * p.d + col;
        prev[it] = ((add_rows >> row) & 1u) && col_ok ? *reinterpret_cast<const uint4*>(p.dx + off) : make_uint4(0, 0, 0, 0);
        if (kJitter)
          uu[kJitter ? it : 0] = tok0 + row < p.T && col_ok ? *reinterpret_cast<const uint4*>(p.jitter_u + off)
                                                            : make_uint4(0, 0, 0, 0);
      }
    };
    if (!kJitter) fetch_rows(split);
    for (int tile = split; tile < p.n_mtiles && ok; tile += p.splits) {
      if (kJitter) fetch_rows(tile);
      const int tok0 = tile * kTileM + lg * 32;
      ok = mbar_wait_warp(tfull0 + 8u * acc, acc_phase, abort_flag, p.status, 14);
      if (!ok) break;
      tc_fence_after();
      uint32_t v[64];
      tc_ld32(t_lane + acc * 128u + (uint32_t)half * 64u, v);
      tc_ld32(t_lane + acc * 128u + (uint32_t)half * 64u + 32u, v + 32);
      tc_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8u * acc);
      // transposed through shared memory as bfloat16 (one extra rounding of the small router term); the sum is formed
      // afterwards, with coalesced rows (a bfloat16 add or multiply-add rounds the exact result once)
      uint32_t pk[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
        pk[j] = *reinterpret_cast<const uint32_t*>(&h2);
      }
      uint4 old[8];
      const unsigned add_now = add_rows;
#pragma unroll
      for (int it = 0; it < 8; ++it) old[it] = prev[it];
      if (!kJitter && tile + p.splits < p.n_mtiles) fetch_rows(tile + p.splits);
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        if ((it & 3) == 0) {                                   // 16 rows at a time
          if (it > 0) __syncwarp();
          if ((lane >> 4) == (it >> 2)) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              *reinterpret_cast<uint4*>(stage_gen + (lane & 15) * 128 + ((j ^ (lane & 7)) << 4)) =
                  make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
          }
          __syncwarp();
        }
        const int row = it * 4 + (lane >> 3);
        uint4 val = *reinterpret_cast<const uint4*>(stage_gen + (row & 15) * 128 + (((lane & 7) ^ (row & 7)) << 4));
        const bool add = (add_now >> row) & 1u;
        __nv_bfloat162* vp = reinterpret_cast<__nv_bfloat162*>(&val);
        const __nv_bfloat162* pp = reinterpret_cast<const __nv_bfloat162*>(&old[it]);
        if (kJitter) {                                         // d(x . u)/dx = u; one rounding for (router term . u) + dx
          const __nv_bfloat162* up = reinterpret_cast<const __nv_bfloat162*>(&uu[kJitter ? it : 0]);
#pragma unroll
          for (int q = 0; q < 4; ++q) vp[q] = add ? __hfma2(vp[q], up[q], pp[q]) : __hmul2(vp[q], up[q]);
        } else if (add) {
#pragma unroll
          for (int q = 0; q < 4; ++q) vp[q] = __hadd2(vp[q], pp[q]);
        }
        if (tok0 + row < p.T && col_ok) *reinterpret_cast<uint4*>(p.dx + (size_t)(tok0 + row) * p.d + col) = val;
      }
      __syncwarp();
      acc ^= 1u;
      if (acc == 0) acc_phase ^= 1u;
    }
    // float32 partial of x^T dh over this CTA's tokens: row = an index into d_model
    if (ok) ok = mbar_wait_warp(dfull, 0u, abort_flag, p.status, 18);
    if (ok) {
      tc_fence_after();
      const int row = n0 + lg * 32 + lane, nch = (p.E + 31) >> 5;
#pragma unroll 1
      for (int c = half; c < nch; c += 2) {
        uint32_t v[32];
        tc_ld32(t_lane + kRBDwrCol + (uint32_t)c * 32u, v);
        tc_wait_ld();
        if (row < p.d) {
          float* dst = p.partial + ((size_t)split * p.d + row) * p.E + c * 32;
          if ((p.E & 3) == 0) {
#pragma unroll
            for (int i = 0; i < 32; i += 4)
              if (c * 32 + i < p.E)
                *reinterpret_cast<float4*>(dst + i) = make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]),
                                                                  __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (c * 32 + i < p.E) dst[i] = __uint_as_float(v[i]);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// wsplit[part][k][e] for e < Epad64 (zero beyond E): W_r = hi + mid up to 2^-18 relative.  The layer's first kernel: it also
// clears the status words (`status` may be null).
__global__ void split_w_kernel(const float* __restrict__ W_r, int d, int E, int Epad64,
                               __nv_bfloat16* __restrict__ wsplit, int* __restrict__ status) {
  pdl_launch_dependents();
  pdl_wait();
  if (status != nullptr && blockIdx.x == 0 && threadIdx.x < kStatusWords) status[threadIdx.x] = 0;
  const size_t n = (size_t)d * Epad64;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int k = (int)(i / Epad64), e = (int)(i - (size_t)k * Epad64);
  split2(e < E ? W_r[(size_t)k * E + e] : 0.f, &wsplit[i], &wsplit[n + i]);
}

}  // namespace

// Up to 128 experts both parts of W_r are staged with the x block they multiply; beyond that a stage holds one part (three
// stages of 64 KB instead of two of 96) and x comes from L2 a second time.
int launch_router_tc_fwd(const Shape& s, const Plan& p, const void* x, const float* W_r, const float* bias,
                         const float* noise, bool clear_status, void* ws, cudaStream_t st) {
  __nv_bfloat16* wsplit = ws_ptr<__nv_bfloat16>(ws, p.wsplit);
  const size_t n = (size_t)s.d * s.Epad64;
  launch_k(split_w_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, W_r, s.d, s.E, s.Epad64, wsplit,
           clear_status ? ws_ptr<int>(ws, p.status) : nullptr);
  CUtensorMap tmA, tmB;
  if (make_map(&tmA, x, 1, s.T, s.d, kTileM) != SWITCH_MOE_OK) return SWITCH_MOE_CUDA_ERROR;
  if (make_map(&tmB, wsplit, 2, s.d, s.Epad64, 64) != SWITCH_MOE_OK) return SWITCH_MOE_CUDA_ERROR;
  RouterFwdParams q{};
  q.T = s.T; q.d = s.d; q.E = s.E; q.Epad64 = s.Epad64;
  q.tiles = s.router_block_tokens / kTileM;
  q.n_blocks = s.router_blocks;
  q.k_blocks = s.d / kBK;
  q.b_atoms = s.Epad64 / 64;
  q.acc_step = q.tiles * (s.Epad64 <= 128 ? 128 : 256);
  q.n_acc = 2 * q.acc_step <= kTmemCols ? 2 : 1;
  q.stage_parts = s.Epad64 <= 128 ? kRFParts : 1;
  q.rot_wrap = s.Epad64 <= 128 ? sm_count_or_default() : 0;
  q.stage_bytes = q.tiles * kABytes + q.stage_parts * q.b_atoms * kAtomBytes;
  q.stages = kRFRingBytes / q.stage_bytes < kRFMaxStages ? kRFRingBytes / q.stage_bytes : kRFMaxStages;
  q.bias = bias; q.noise = noise; q.probs = ws_ptr<float>(ws, p.probs); q.expert_index = ws_ptr<int>(ws, p.expert_index);
  q.gate = ws_ptr<float>(ws, p.gate); q.status = ws_ptr<int>(ws, p.status);
  q.psum_partial = ws_ptr<float>(ws, p.psum_partial); q.hist = ws_ptr<int>(ws, p.hist);
  const int sms = sm_count_or_default(), grid = q.n_blocks < sms ? q.n_blocks : sms;
  auto kernel = s.E > 128 ? router_fwd_tc_kernel<true> : router_fwd_tc_kernel<false>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRFSmemBytes) != cudaSuccess)
    return SWITCH_MOE_CUDA_ERROR;
  launch_k(kernel, dim3(grid), dim3(64 + 128 * q.tiles), kRFSmemBytes, st, tmA, tmB, q);
  return launch_status();
}

int launch_router_tc_bwd(const Shape& s, const Plan& p, const void* x, const float* W_r, void* ws, void* dx,
                         bool accumulate_dx, cudaStream_t st) {
  __nv_bfloat16* wsplit = ws_ptr<__nv_bfloat16>(ws, p.wsplit);
  __nv_bfloat16* dhsplit = ws_ptr<__nv_bfloat16>(ws, p.dhsplit);
  if (!accumulate_dx) {
    // staged call: split W_r here.  The whole-layer backward (accumulate_dx) reuses the parts its forward pass left
    // in the workspace: W_r must be unchanged between the two calls anyway.
    const size_t nw = (size_t)s.d * s.Epad64;
    launch_k(split_w_kernel, dim3((unsigned)((nw + 255) / 256)), dim3(256), 0, st, W_r, s.d, s.E, s.Epad64, wsplit,
             static_cast<int*>(nullptr));
  }
  RouterBwdParams q{};
  q.T = s.T; q.d = s.d; q.E = s.E; q.ka = s.Epad64 / 64;
  q.n_mtiles = (s.T + kTileM - 1) / kTileM; q.n_cols = (s.d + 127) / 128; q.splits = s.dwr_chunks;
  // 208 KB of operands: W_r parts (32 KB per block of 64 experts), then two x stages if they leave at least four blocks
  // of the dh ring (up to 128 experts), else one
  const int left = kRBOperandBytes / kRBBlock - 2 * q.ka;
  q.x_stages = left - 4 >= 4 ? 2 : 1;
  q.ring = left - 2 * q.x_stages < kRBMaxRing ? left - 2 * q.x_stages : kRBMaxRing;
  q.partial = ws_ptr<float>(ws, p.dwr_partial);
  q.dx = static_cast<__nv_bfloat16*>(dx); q.slot = ws_ptr<int>(ws, p.slot);
  q.accumulate = accumulate_dx ? ((s.residual || s.top2) ? 2 : 1) : 0;   // 2: every row already holds a value
  q.jitter_u = static_cast<const __nv_bfloat16*>(s.jitter_u);
  q.status = ws_ptr<int>(ws, p.status);
  CUtensorMap tmX, tmH, tmW;
  if (make_map(&tmX, x, 1, s.T, s.d, kTileM) != SWITCH_MOE_OK ||
      make_map(&tmH, dhsplit, 2, s.T, s.Epad64, kTileM) != SWITCH_MOE_OK ||
      make_map(&tmW, wsplit, 2, s.d, s.Epad64, kTileM) != SWITCH_MOE_OK)
    return SWITCH_MOE_CUDA_ERROR;
  auto kernel = s.jitter ? router_bwd_tc_kernel<true> : router_bwd_tc_kernel<false>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRBSmemBytes) != cudaSuccess)
    return SWITCH_MOE_CUDA_ERROR;
  launch_k(kernel, dim3(q.n_cols * q.splits), dim3(kRBThreads), kRBSmemBytes, st, tmX, tmH, tmW, q);
  return launch_status();
}

}  // namespace swmoe
