// Grouped expert GEMMs on pairs of SMs (tcgen05 cta_group::2, M = 256), bfloat16 in, float32 accumulate, bfloat16
// out: the expert FFN h = x W_in, y = ReLU(h) W_out (Section 5, FFN review) and its derivatives, with the layer's
// element-wise steps fused into the epilogues (ReLU, the gate of Eq. 2 with the scatter back to token order, the
// ReLU mask of the backward pass; for GEGLU experts the gating GELU(a) . b in GEMM1's epilogue and its derivative in
// dgrad2's, two more instantiations of the same kernel).
//
// Orientation.  An expert has about 256 tokens but thousands of weight rows, so the weight matrix sits on the MMA's
// M side (256 rows per CTA pair, 128 per CTA) and the expert's tokens on the N side, whose granularity is 16:
//   H^T  [f, tok] = W_in^T  [f, d] . X_d^T  [d, tok]      y^T  [d, tok] = W_out^T [d, f] . H^T  [f, tok]
//   dH^T [f, tok] = W_out   [f, d] . dY_d^T [d, tok]      dx^T [d, tok] = W_in    [d, f] . dH^T [f, tok]
// so no 128-row token tile is padded, every weight element enters shared memory exactly once, and the epilogue
// transposes 32x32 blocks through shared memory to write token-major rows.  The weight gradients keep the natural
// orientation (dW_out = H^T dY_d, dW_in = X_d^T dH: M = weight rows, N = weight columns, contraction over tokens).
//
// A CTA pair shares the B operand: each CTA stages its own 128 A rows and half of B per 64-deep k-block, the leader
// CTA's MMA warp issues M=256 instructions that read both CTAs' shared memory, and tcgen05.commit with a
// cluster mask releases stages and publishes accumulators in both CTAs.  TMA loads carry no multicast.  Each CTA
// drains its own 128 TMEM lanes with 8 epilogue warps while the next tile's MMAs run.
//
// One pass per expert.  A token tile holds up to 320 tokens (the capacity of the paper's layers at capacity factor
// 1.25), so an expert's weights cross shared memory once; a tile wider than the MMA's N limit of 256 is two column
// segments, i.e. two MMAs per k-step that read the same A block.  The token operand's TMA box is exactly the rows
// the tile has (one tensor map per box height), so no byte enters shared memory that no MMA reads.
// Two accumulators of up to 320 columns do not fit 512 TMEM columns side by side, so they overlap in the middle:
// even tiles of a CTA pair use columns [0, n), odd tiles [512 - n, 512).  The epilogue drains a tile starting from
// the middle columns and tells the MMA thread (barrier `tmid`) once the columns the next tile also uses have been
// read; the next tile's MMAs then start while the rest of the tile is still being drained.
//
// Epilogue of the token products.  It has to turn lanes (weight rows) x columns (tokens) into token rows; with few k-blocks
// per tile (small d_model) it is what a tile waits for, so it is kept to few instructions: the accumulator is read as matrix
// fragments, scaled, rounded and masked in that order, transposed by stmatrix, and what dgrad2 needs from GEMM1 (ReLU bits,
// GEGLU factors) is saved in fragment order and never transposed at all.  Against packing token pairs through 32-bit
// shared-memory words: 65536 tokens, 256 x 512, 128 experts GEMM1 45 -> 35 us, dgrad2 42 -> 38; GEGLU 32768 tokens, 768 x
// 2048, 128 experts GEMM1 260 -> 232, dgrad2 197 -> 170; 32768 x 768 x 3072 (ReLU) unchanged, HBM bounds it there.
//
// Every mbarrier wait is bounded in time (status word + abort flag); both CTAs always reach the final cluster
// barrier, so tensor memory is freed and no CTA exits while its peer can still address its shared memory.
#include "tc_common.cuh"

namespace swmoe {
using namespace tc;
namespace {

constexpr int kPStages = 6;                            // weight gradients: six blocks of A and six of half of B
constexpr int kPMaxStages = 8;                         // token products: as many stages as fit, at most this
constexpr int kPHalfBytes = 16384;                     // A tile (128 x 64) and B half tile (<= 128 x 64)
constexpr int kPStageBytes = 2 * kPHalfBytes;
constexpr int kPRingBytes = kPStages * kPStageBytes;   // 192 KB of operand stages
constexpr int kPWgradA = kPStages, kPWgradB = kPStages;   // weight gradients: A and B blocks of 16 KB in rings of their own
constexpr int kPTransWarp = 32 * 64;                   // per epilogue warp: 32 tokens x 32 weight rows of bfloat16
constexpr int kPTransBytes = 8 * kPTransWarp;
constexpr int kPAuxBytes = 8 * 128;                    // 8 epilogue warps x 32 gates
constexpr int kPKeptCache = kMaxExperts;                 // kept[e] for every expert
constexpr int kPTileCache = 448;                        // first token tiles of the list ({expert, row, rows})
constexpr int kPCacheBytes = kPKeptCache * 4 + kPTileCache * 16;
constexpr int kPSmemBytes = 1024 + kPRingBytes + kPTransBytes + kPAuxBytes + 256 + kPCacheBytes;
constexpr int kPThreads = 320;
constexpr uint32_t kPeerMask = 0xFEFFFFFFu;            // clears the CTA-rank bit of a shared::cluster address
// GEMM1 of GEGLU experts with the gating in its epilogue (a seventh instantiation beside the six GemmOp products):
// a CTA's 128 weight rows are 64 columns of W_0 and the same 64 columns of W_1, so a_j and b_j of one hidden unit sit
// in TMEM lanes j and 64 + j of one CTA, i.e. with epilogue warps two lane groups apart.
constexpr int kGemm1Gated = 6;
// dgrad2 of GEGLU experts with the derivative of the gating in its epilogue: d a = dH . (b GELU'(a)), d b = dH . GELU(a),
// the two factors read back from what the gated GEMM1 saved.
constexpr int kDgrad2Gated = 7;

struct PairParams {
  int op;                  // GemmOp
  int token_op;            // 1: tokens on N (transposed epilogue); 0: weight gradient (contraction over tokens)
  int a_mn_major;
  int Mw;                  // rows of the M-side operand per expert (d_ff or d_model)
  int Nfix;                // weight gradients: output columns
  int k_blocks_fixed;      // token ops: K / 64
  int n_mpairs, n_ntiles_fixed;
  int tokens_per_expert;   // average, at most the capacity
  int strips;              // weight gradients: strips that a row of column tiles (256 output rows) is cut into
  int C, E;
  const int4* ntile;       // [0].x = number of token tiles; then {expert, first slot row, rows (multiple of 16)}
  const int* kept;
  const int* token_of_slot;
  const float* gate;
  __nv_bfloat16* out;
  uint16_t* hmask;          // [block][lane]: [H > 0] of a thread's 16 elements of a block of 16 tokens x 32 hidden units, in
                            // fragment order (bits 0-7 the even tokens, 8-15 the odd ones); written by GEMM1, read by
                            // dgrad2; block = (expert * cb + row / 16) * (hid / 32) + unit / 32
  int cb, hid;              // 16-row blocks per expert, d_ff
  long long ld_out;
  int* status;
  const __nv_bfloat16* res;   // combine / scatter with the skip path inside the layer: rows added to the output (x or dy)
  __nv_bfloat16* out2;        // combine with the skip path: second copy of the output without it
  int gate_f;                 // gated products: d_ff.  Gated GEMM1: W_in has 2 d_ff columns [W_0 | W_1], out = hidden.
                              // Gated dgrad2: out = d[a | b] (2 d_ff columns).
  uint4* gate_buf;            // what the gated GEMM1 saves: [block][4][lane] of 4 words {GELU(a), b GELU'(a)}, in fragment order
  // expert dropout (Section 2.4) in the epilogues: GEMM1 multiplies the hidden activations by keep / (1 - rate) before
  // it rounds them and takes the mask bits (the gated GEMM1: the hidden activations and both saved factors); dgrad2
  // multiplies by 1 / (1 - rate), its mask bits already say "kept and positive".
  const uint32_t* keep_bits;  // [E * C][d_ff / 32]: bit i of word [row][w] = keep hidden unit 32 w + i; or null
  int keep_words;             // d_ff / 32
  float keep_scale;           // 1 / (1 - rate); 1 without dropout
  int stages, stage_bytes;    // operand ring: token products size a stage for the widest tile the capacity allows
  // ceil(2^32 / divisor) for the three divisions of the tile decode (n_mpairs; n_mpairs * n_ntiles_fixed;
  // n_ntiles_fixed): id / d = umulhi(id, magic) as long as id * d < 2^32
  uint32_t magic_mpairs, magic_per_e, magic_strips;
};

__device__ __forceinline__ int fast_div(int id, uint32_t magic, int divisor) {
  return divisor == 1 ? id : (int)__umulhi((uint32_t)id, magic);
}

// Token products: the token operand's TMA box is exactly this CTA's share of the tile (n / 2 rows, a multiple of 8):
// one tensor map per height 8, 16, .., 128.  Weight gradients use entry 0 (a 64-row box of the token contraction).
constexpr int kBMaps = 16;
struct BMapSet {
  CUtensorMap m[kBMaps];
};

struct PTile {
  int e, m0, n0, row0, n, n1, k_blocks, last_mmas;   // n1: columns of the first segment (n if n <= 256)
  int tiles;                                         // weight gradients: column tiles of the strip that starts at n0
};

// Tile decode reads the plan through shared-memory copies made at kernel start: a dependent global load per tile
// would stall the producer warp for longer than a short tile's whole k-loop.
__device__ __forceinline__ PTile p_decode(const PairParams& p, int id, const int* kept_s, const int4* tile_s) {
  PTile t;
  if (p.token_op) {
    const int nt = fast_div(id, p.magic_mpairs, p.n_mpairs);
    const int4 q = nt < kPTileCache ? tile_s[nt] : p.ntile[1 + nt];
    t.e = q.x; t.row0 = q.y; t.n = q.z; t.n0 = 0;
    t.n1 = t.n <= 256 ? t.n : ((t.n >> 1) + 15) & ~15;         // two segments: both multiples of 16, both <= 256
    t.m0 = (id - nt * p.n_mpairs) * 256;
    t.k_blocks = p.k_blocks_fixed; t.tiles = 1;
    t.last_mmas = kBK / kUmmaK;
  } else {
    const int per_e = p.n_mpairs * p.strips;
    t.e = fast_div(id, p.magic_per_e, per_e);
    const int rem = id - t.e * per_e;
    const int mp = fast_div(rem, p.magic_strips, p.strips);
    const int strip = rem - mp * p.strips;                      // strips of a row differ by at most one tile
    int first = strip, last = strip + 1;
    if (p.strips < p.n_ntiles_fixed) {
      first = (int)((unsigned)strip * (unsigned)p.n_ntiles_fixed / (unsigned)p.strips);
      last = (int)((unsigned)(strip + 1) * (unsigned)p.n_ntiles_fixed / (unsigned)p.strips);
    }
    t.m0 = mp * 256;
    t.n0 = first * 256;
    t.tiles = last - first;
    t.row0 = 0; t.n = 256; t.n1 = 256;
    const int k = kept_s[t.e];
    t.k_blocks = (k + kBK - 1) / kBK;
    const int rem_rows = k - (t.k_blocks - 1) * kBK;          // rows of the last k-block that hold tokens
    t.last_mmas = (rem_rows + kUmmaK - 1) / kUmmaK;            // rows beyond them are never multiplied
  }
  return t;
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t local_bar, uint32_t cta) {
  asm volatile(
      "{\n\t.reg .b32 ra;\n\t"
      "mapa.shared::cluster.u32 ra, %0, %1;\n\t"
      "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}"
      ::"r"(local_bar), "r"(cta)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* tm, uint32_t leader_bar, int c0,
                                                 int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(leader_bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
// 16 lanes x 32 columns of the accumulator as matrix fragments: registers 4 j .. 4 j + 3 of a thread are columns
// 8 j + 2 (lane % 4), + 1 of TMEM lane lane / 4, then of lane lane / 4 + 8.
__device__ __forceinline__ void tc_ld_16x256b_x4(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Waits for this thread's loads; the registers pass through so that no use of them can move ahead of the wait.
__device__ __forceinline__ void tc_wait_ld_regs(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                 "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
// Four 8 x 8 matrices of bfloat16, transposed: lane l's address is row l % 8 of matrix l / 8.
__device__ __forceinline__ void stmatrix_trans(uint32_t addr, const uint32_t* w) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3])
               : "memory");
}
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, const uint32_t* w) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3])
               : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h2);
}
__device__ __forceinline__ uint32_t relu_bf16x2(uint32_t w) {
  const __nv_bfloat162 z = __floats2bfloat162_rn(0.f, 0.f);
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&w), z);
  return *reinterpret_cast<const uint32_t*>(&r);
}
// 0xFFFF in each half that is positive.
__device__ __forceinline__ uint32_t positive_bf16x2(uint32_t w) {
  return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&w), __floats2bfloat162_rn(0.f, 0.f));
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// One instantiation per product (OP is a GemmOp): each kernel carries only its own epilogue, and the operand
// orientations are compile-time constants, which keeps the code footprint of every role small.
//
// `pair` of `n_pairs` is this CTA pair's place among the pairs that work on this product: the whole grid for a
// launch of one product, a share of it when two products run side by side in one launch (below).
template <int OP, bool DROP = false>                          // DROP: expert dropout in this product's epilogue
__device__ __forceinline__ void pair_body(const CUtensorMap& tmA, const BMapSet& bm, const PairParams& p,
                                          const int pair, const int n_pairs) {
  constexpr bool kGated = OP == kGemm1Gated, kDGated = OP == kDgrad2Gated;
  constexpr bool kTok = OP <= kDgrad1Scatter || kGated || kDGated;   // tokens on N, transposed epilogue
  constexpr bool kAMn = (OP == kGemm1Relu || kGated || OP == kGemm2Combine || OP == kWgrad2 || OP == kWgrad1);
  constexpr bool kBMn = !kTok;
  pdl_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  uint8_t* trans_gen = smem_gen + kPRingBytes;
  uint8_t* aux_gen = trans_gen + kPTransBytes;
  uint8_t* bar_gen = aux_gen + kPAuxBytes;
  const uint32_t bar_base = smem_base + kPRingBytes + kPTransBytes + kPAuxBytes;
  // barrier block: full[S] | empty[S] | tmem_full[2] | tmem_empty[2] | tmem_mid[2] | tmem_ptr | abort | gate[4]
  // (S = kPMaxStages; gate[i] at byte 192 + 8 i: the handshake of the two epilogue warps that hold a and b of the
  // same hidden units, gated GEMM1 only; there a weight gradient has aempty[kPWgradA], the release of its A blocks)
  const uint32_t full0 = bar_base, empty0 = bar_base + 8u * kPMaxStages;
  const uint32_t tfull0 = bar_base + 16u * kPMaxStages, tempty0 = tfull0 + 16u, tmid0 = tfull0 + 32u;
  const uint32_t gate0 = bar_base + 192u, aempty0 = gate0;
  volatile uint32_t* tmem_ptr_s = reinterpret_cast<volatile uint32_t*>(bar_gen + 8 * (2 * kPMaxStages + 6));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_gen + 8 * (2 * kPMaxStages + 6) + 4);
  int* kept_s = reinterpret_cast<int*>(bar_gen + 256);
  int4* tile_s = reinterpret_cast<int4*>(bar_gen + 256 + kPKeptCache * 4);

  const int warp = uniform_warp_id(), lane = threadIdx.x & 31;
  const uint32_t rank = __shfl_sync(0xffffffffu, cluster_ctarank(), 0);   // 0 = leader (issues the MMAs)
  const uint32_t n_stages = kTok ? (uint32_t)p.stages : (uint32_t)kPWgradB;
  const uint32_t stage_bytes = kTok ? (uint32_t)p.stage_bytes : (uint32_t)kPHalfBytes;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPMaxStages; ++s) { mbar_init(full0 + 8u * s, 1); mbar_init(empty0 + 8u * s, 1); }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8u * a, 1); mbar_init(tempty0 + 8u * a, 16); mbar_init(tmid0 + 8u * a, 16);
    }
    if (kGated)
      for (int a = 0; a < 4; ++a) mbar_init(gate0 + 8u * a, 2);
    if (!kTok)
      for (int a = 0; a < kPWgradA; ++a) mbar_init(aempty0 + 8u * a, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_ptr_s))), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  pdl_wait();                                                 // the previous kernel's results are needed from here on
  const int n_ntiles_listed = kTok ? p.ntile[0].x : 0;
  for (int i = threadIdx.x; i < p.E; i += kPThreads) kept_s[i] = p.kept[i];
  for (int i = threadIdx.x; i < min(n_ntiles_listed, kPTileCache); i += kPThreads) tile_s[i] = p.ntile[1 + i];
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_s;
  const int n_tiles = kTok ? n_ntiles_listed * p.n_mpairs : p.E * p.n_mpairs * p.strips;

  // Weight gradients: A blocks are released by barriers of their own where a strip has several tiles.  With single tiles
  // both rings, equally long, move in step, and a stage's release is its A block's too (512 tokens per expert, 768 x 3072, 64
  // experts: wgrad2 107 us, dgrad1 with wgrad1 214; with the second wait and commit per k-block 111 and 227).
  static_assert(kPWgradA == kPWgradB, "single tiles: one release per stage");
  const bool a_ring = !kTok && p.strips < p.n_ntiles_fixed;

  // Accumulator columns of this pair's `it`-th tile: even tiles [0, n), odd tiles [512 - n, 512).  Consecutive tiles
  // share the middle columns when n + n_next > 512.
  if (warp == 0) {
    // ------------------------------------------------------------------------------------------ TMA producer (both CTAs)
    uint32_t stage = 0, phase = 0, a_slot = 0, a_phase = 0;
    bool ok = true;
    for (int id = pair; id < n_tiles && ok; id += n_pairs) {
      const PTile t = p_decode(p, id, kept_s, tile_s);
      // coordinates of this CTA's boxes; only the contraction coordinate moves inside the tile
      // gated GEMM1: 64 columns of W_0 and the same 64 columns of W_1 (a pair covers 128 hidden units)
      const int a_m = kGated ? (t.m0 >> 1) + 64 * (int)rank : t.m0 + 128 * (int)rank;
      const int a_m2 = kGated ? p.gate_f + a_m : a_m + 64;
      const int e = t.e, kbs = t.k_blocks;
      // token products: this CTA's half of each column segment's token rows, in boxes of exactly that height;
      // weight gradients: this CTA's 128 of the 256 output columns
      const int h1 = t.n1 >> 1, h2 = (t.n - t.n1) >> 1;
      const int b_r = kTok ? t.row0 + (int)rank * h1 : t.n0 + 128 * (int)rank;
      const int b_r2 = t.row0 + t.n1 + (int)rank * h2;
      const CUtensorMap* tmB = kTok ? &bm.m[(h1 >> 3) - 1] : &bm.m[0];
      const CUtensorMap* tmB2 = (kTok && h2 > 0) ? &bm.m[(h2 >> 3) - 1] : tmB;
      // both CTAs' bytes land on the leader's barrier
      const uint32_t tx_bytes = kTok ? 2u * (uint32_t)(kPHalfBytes + (t.n >> 1) * 128) : 2u * (uint32_t)kPHalfBytes;
      // weight gradients: the tiles of a strip multiply the same A; it is loaded with the first of them and kept to the
      // last if its k-blocks fit the A ring.  A block's full barrier counts the A bytes that come with it.
      const bool resident = !kTok && kbs <= kPWgradA;
#pragma unroll 1
      for (int j = 0; j < (kTok ? 1 : t.tiles) && ok; ++j) {
        const bool load_a = kTok || j == 0 || !resident;
#pragma unroll 1
        for (int kb = 0; kb < kbs; ++kb) {
          if (load_a && a_ring) {
            ok = mbar_wait_warp(aempty0 + 8u * a_slot, a_phase ^ 1u, abort_flag, p.status, 28);
            if (!ok) break;
          }
          const uint32_t eb = empty0 + 8u * stage;
          ok = mbar_wait_warp(eb, phase ^ 1u, abort_flag, p.status, 21);
          if (!ok) break;
          const uint32_t a_dst = smem_base + (kTok ? stage * stage_bytes : a_slot * (uint32_t)kPHalfBytes);
          const uint32_t b_dst = kTok ? a_dst + kPHalfBytes : smem_base + (kPWgradA + stage) * (uint32_t)kPHalfBytes;
          const uint32_t fb = full0 + 8u * stage;
          const uint32_t lead_full = fb & kPeerMask;
          const int k0 = kb * kBK;
          if (elect_one()) {
            if (rank == 0) mbar_arrive_expect_tx(fb, !kTok && load_a ? 2u * tx_bytes : tx_bytes);
            if (kAMn) {
              if (load_a) {
                tma_load_3d_pair(a_dst, &tmA, lead_full, a_m, k0, e);
                tma_load_3d_pair(a_dst + kAtomBytes, &tmA, lead_full, a_m2, k0, e);
              }
            } else {
              tma_load_3d_pair(a_dst, &tmA, lead_full, k0, a_m, e);
            }
            if (kBMn) {
              const int col = b_r + 256 * j;
              tma_load_3d_pair(b_dst, tmB, lead_full, col, k0, e);
              tma_load_3d_pair(b_dst + kAtomBytes, tmB, lead_full, col + 64, k0, e);
            } else {
              tma_load_3d_pair(b_dst, tmB, lead_full, k0, b_r, e);
              if (h2 > 0) tma_load_3d_pair(b_dst + (uint32_t)h1 * 128u, tmB2, lead_full, k0, b_r2, e);
            }
          }
          if (++stage == n_stages) { stage = 0; phase ^= 1u; }
          if (!kTok && load_a && ++a_slot == (uint32_t)kPWgradA) { a_slot = 0; a_phase ^= 1u; }
        }
      }
    }
    if (*abort_flag != 0) {
      const long long t0 = clock64();
      while (clock64() - t0 < 4000000ll) __nanosleep(1000);  // let copies in flight land (about 2 ms)
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------------------------ MMA issuer (leader CTA)
    if (rank == 0) {
      constexpr uint32_t idesc_base = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)kAMn << 15) |
                                      ((uint32_t)kBMn << 16) | ((uint32_t)(256 >> 4) << 24);
      // descriptors differ between stages and k-steps only in the start-address field (units of 16 bytes)
      constexpr uint32_t a_kstep = (kAMn ? kUmmaK * 128u : kUmmaK * 2u) >> 4;
      constexpr uint32_t b_kstep = (kBMn ? kUmmaK * 128u : kUmmaK * 2u) >> 4;
      const uint64_t a_desc0 = make_smem_desc(smem_base, kAMn ? kAtomBytes : 16u, 1024u);
      const uint64_t b_desc0 = make_smem_desc(smem_base + (kTok ? 1 : kPWgradA) * kPHalfBytes, kBMn ? kAtomBytes : 16u, 1024u);
      uint32_t stage = 0, phase = 0, it = 0, a_first = 0;
      int n_prev = 0;
      bool ok = true;
      for (int id = pair; id < n_tiles && ok; id += n_pairs) {
        const PTile t = p_decode(p, id, kept_s, tile_s);
        const bool resident = !kTok && t.k_blocks <= kPWgradA;
#pragma unroll 1
        for (int j = 0; j < (kTok ? 1 : t.tiles) && ok; ++j, ++it) {
          const bool free_a = !kTok && (j == t.tiles - 1 || !resident);
          uint32_t a_slot = a_first;
          const uint32_t side = it & 1u, use = it >> 1;          // this side's `use`-th tile
          const uint32_t idesc1 = idesc_base | ((uint32_t)(t.n1 >> 3) << 17);
          const int n2 = t.n - t.n1;
          const uint32_t idesc2 = idesc_base | ((uint32_t)(n2 >> 3) << 17);
          const uint32_t b2_off = ((uint32_t)(t.n1 >> 1) * 128u) >> 4;    // second segment's rows in this CTA's half of B
          const int kbs = t.k_blocks, last_mmas = t.last_mmas;
          // the side's previous tile has been read out completely ...
          ok = mbar_wait_warp(tempty0 + 8u * side, (use & 1u) ^ 1u, abort_flag, p.status, 22);
          if (!ok) break;
          // ... and so have the middle columns of the other side's tile, if this tile reaches into them
          if (kTok && it > 0 && n_prev + t.n > kTmemCols) {
            ok = mbar_wait_warp(tmid0 + 8u * (side ^ 1u), ((it - 1u) >> 1) & 1u, abort_flag, p.status, 25);
            if (!ok) break;
          }
          n_prev = t.n;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (side ? (uint32_t)(kTmemCols - t.n) : 0u);
          const uint32_t d_tmem2 = d_tmem + (uint32_t)t.n1;
#pragma unroll 1
          for (int kb = 0; kb < kbs; ++kb) {
            ok = mbar_wait_warp(full0 + 8u * stage, phase, abort_flag, p.status, 23);
            if (!ok) break;
            tc_fence_after();
            const uint64_t ad = a_desc0 + (uint64_t)((kTok ? stage : a_slot) * (stage_bytes >> 4));
            const uint64_t bd = b_desc0 + (uint64_t)(stage * (stage_bytes >> 4));
            const int n_mma = (!kTok && kb == kbs - 1) ? last_mmas : kBK / kUmmaK;
            const uint32_t acc0 = kb > 0 ? 1u : 0u;
            if (elect_one()) {
              if (kTok && n2 > 0) {
#pragma unroll
                for (int ks = 0; ks < kBK / kUmmaK; ++ks) {
                  tc_mma_bf16_pair(d_tmem, ad + ks * a_kstep, bd + ks * b_kstep, idesc1, ks > 0 ? 1u : acc0);
                  tc_mma_bf16_pair(d_tmem2, ad + ks * a_kstep, bd + b2_off + ks * b_kstep, idesc2, ks > 0 ? 1u : acc0);
                }
              } else {
#pragma unroll
                for (int ks = 0; ks < kBK / kUmmaK; ++ks)
                  if (ks == 0 || ks < n_mma)
                    tc_mma_bf16_pair(d_tmem, ad + ks * a_kstep, bd + ks * b_kstep, idesc1, ks > 0 ? 1u : acc0);
              }
              tc_commit_pair(empty0 + 8u * stage);              // frees this stage in both CTAs
              if (free_a && a_ring) tc_commit_pair(aempty0 + 8u * a_slot);
              if (kb == kbs - 1) tc_commit_pair(tfull0 + 8u * side);   // accumulator complete, in both CTAs
            }
            if (++stage == n_stages) { stage = 0; phase ^= 1u; }
            if (!kTok && ++a_slot == (uint32_t)kPWgradA) a_slot = 0;
          }
          if (!ok) break;
          if (free_a) a_first = a_slot;
          if (kbs <= 0 && lane == 0) {                          // nothing to contract: epilogues write zeros
            mbar_arrive(tfull0 + 8u * side);
            mbar_arrive_remote(tfull0 + 8u * side, 1);
          }
        }
      }
    }
  } else if constexpr (!kTok) {
    // --------------------------------------------------------------- epilogue warps (both CTAs), weight gradients
    // Rows of the output are lanes of the accumulator.  A warp drains its 32 rows x 2 chunks of 64 columns in four units
    // of 16 rows: read as matrix fragments, rounded, stored as 8 x 8 matrices into 128-byte rows (16-byte pieces
    // exchanged by the row), written to memory as whole lines; the next unit's accumulator is in flight meanwhile.  The
    // stores bound it: without them a 768 x 3072 x 128 launch takes 130 us, with them 172 (with 32-lane row reads and half
    // warps storing in turn 154 and 172); 604 MB of output alone are 82 us of pure writes.
    const int lg = warp & 3, half = (warp - 2) >> 2;
    uint8_t* tr = trans_gen + (warp - 2) * kPTransWarp;
    const uint32_t sa = smem_u32(tr) + (uint32_t)((lane & 15) * 128), sx = lane & 7, sq = lane >> 4;
    const int rr0 = lane >> 3, chunk = lane & 7;
    uint32_t it = 0;
    bool ok = true;
    for (int id = pair; id < n_tiles && ok; id += n_pairs) {
      const PTile t = p_decode(p, id, kept_s, tile_s);
      const int m_warp = t.m0 + 128 * (int)rank + 32 * lg;
      const bool have_acc = t.k_blocks > 0, m_ok = m_warp < p.Mw;
#pragma unroll 1
      for (int j = 0; j < t.tiles; ++j, ++it) {
        const uint32_t side = it & 1u, use = it >> 1;
        const uint32_t t_addr = tmem_base + ((uint32_t)(lg * 32) << 16) + (side ? 256u : 0u);
        uint32_t v[32];
        auto load_unit = [&](int u) {
          const uint32_t at = t_addr + ((uint32_t)(16 * (u & 1)) << 16) + (uint32_t)((half + (u & 2)) * 64);
          tc_ld_16x256b_x4(at, v);
          tc_ld_16x256b_x4(at + 32u, v + 16);
        };
        ok = mbar_wait_warp(tfull0 + 8u * side, use & 1u, abort_flag, p.status, 24);
        if (!ok) break;
        tc_fence_after();
        if (have_acc) load_unit(0);
        else {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = 0u;
        }
        const int n0 = t.n0 + 256 * j + half * 64;              // (rows and columns come in multiples of 64)
        __nv_bfloat16* o = p.out + ((long long)t.e * p.Mw + m_warp + rr0) * p.ld_out + n0 + chunk * 8;
#pragma unroll 2
        for (int u = 0; u < 4; ++u) {
          if (have_acc) tc_wait_ld_regs(v);
          if (u == 3) {                                         // accumulator read out
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty0 + 8u * side, 0);
          }
          uint32_t pk[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
          if (have_acc && u < 3) load_unit(u + 1);
          __syncwarp();
#pragma unroll
          for (int g = 0; g < 4; ++g)                           // 16-byte pieces 2 g and 2 g + 1 of rows 0-7 and 8-15
            stmatrix_x4(sa + (((2u * g + sq) ^ sx) << 4), pk + 4 * g);
          __syncwarp();
          const bool inside = m_ok && n0 + (u & 2) * 64 < p.Nfix;
          __nv_bfloat16* ou = o + (long long)(16 * (u & 1)) * p.ld_out + (u & 2) * 64;
#pragma unroll
          for (int st = 0; st < 4; ++st) {
            const int rr = st * 4 + rr0;
            const uint4 val = *reinterpret_cast<const uint4*>(tr + rr * 128 + ((chunk ^ (rr & 7)) << 4));
            if (inside) *reinterpret_cast<uint4*>(ou + (long long)(4 * st) * p.ld_out) = val;
          }
        }
      }
    }
  } else {
    // --------------------------------------------------------------- epilogue warps (both CTAs), token products
    const int lg = warp & 3;
    const int half = (warp - 2) >> 2;
    uint8_t* tr = trans_gen + (warp - 2) * kPTransWarp;       // this warp's transpose tile
    float* gate_s = reinterpret_cast<float*>(aux_gen + (warp - 2) * 128);
    uint32_t it = 0;
    bool ok = true;
    // gated GEMM1: lane groups 0, 1 hold a = x W_0, lane groups 2, 3 hold b = x W_1 of the same 32 hidden units
    const int role = lg >> 1;
    const uint8_t* tr_other = trans_gen + (half * 4 + lg) * kPTransWarp;   // the transpose tile of the warp two lane groups away
    const uint32_t gate_bar = gate0 + 8u * (uint32_t)(half * 2 + (lg & 1));
    uint32_t gate_phase = 0;
    // Token products.  A chunk of 32 accumulator columns (tokens) x the warp's 32 lanes (weight rows) is read as matrix
    // fragments: word [4 g + i] of a thread = weight row 8 i + lane / 4 of tokens 8 g + 2 (lane % 4), + 1.  stmatrix with
    // transposition turns that into token rows of 64 bytes in this warp's tile; a store then writes 16 bytes per lane,
    // eight tokens at a time.  16-byte pieces are exchanged within a row by the row so that neither side conflicts.
    const uint32_t st_addr = smem_u32(tr) + (uint32_t)((lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4));
    const uint8_t* ld_addr = tr + (lane >> 2) * 64 + (((lane & 3) ^ ((lane >> 3) & 3)) << 4);
    for (int id = pair; id < n_tiles && ok; id += n_pairs, ++it) {
      const PTile t = p_decode(p, id, kept_s, tile_s);
      const uint32_t side = it & 1u, use = it >> 1;
      const int unit0 = (t.m0 >> 1) + 64 * (int)rank + 32 * (lg & 1);        // gated GEMM1: first hidden unit of this warp
      // first M row (weight row = output column) this warp holds
      const int m_warp = kGated ? role * p.gate_f + unit0 : t.m0 + 128 * (int)rank + 32 * lg;
      const int c0 = side ? kTmemCols - t.n : 0;              // first accumulator column of the tile
      const uint32_t t_addr = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)c0;
      // Chunks are numbered so that chunk j of an even tile holds the tile's tokens [32 j, 32 j + 32) and chunk j of an
      // odd tile its tokens [n - 32 (j + 1), n - 32 j): a chunk is then always inside the 512 columns, and counting j
      // down from the last chunk starts in the middle columns, the ones the next tile may also use.  This warp's chunks
      // are j = n_chunks - 1 - half, then every second one down to 0.
      constexpr bool kSlotRows = (OP == kGemm1Relu || kGated || OP == kDgrad2Mask || kDGated);
      constexpr int kQueue = 5;                              // (320 / 32) chunks over two warps
      const int n_chunks = (t.n + 31) >> 5;
      const bool m_ok = kGated ? unit0 < p.gate_f : m_warp < p.Mw;   // (weight rows come in multiples of 64)
      const int kept_e = kept_s[t.e];
      const int row_limit = kSlotRows ? min(p.C, (kept_e + 15) / 16 * 16) : kept_e;
      const int id_next = id + n_pairs;
      const int n_next = id_next < n_tiles ? p_decode(p, id_next, kept_s, tile_s).n : 0;
      const int j_mid = (t.n - max(0, t.n + n_next - kTmemCols)) >> 5;   // chunks j >= j_mid: columns the next tile uses too
      __nv_bfloat16* out_rows = p.out + ((long long)t.e * p.C + t.row0) * p.ld_out;   // slot-row products: the tile's first row
      auto chunk_tok0 = [&](int j) { return side ? t.n - 32 * (j + 1) : 32 * j; };
      auto row_ok = [&](int col) { return col >= 0 && col < t.n && t.row0 + col < row_limit; };
      // 16-token blocks of 32 hidden units: what GEMM1 saves for dgrad2 is kept per block in fragment order.  block0 is the
      // block of the tile's first token; 16 tokens further is hid / 32 blocks further.
      const int words = p.hid >> 5;
      const long long block0 = ((long long)t.e * p.cb + (t.row0 >> 4)) * words + ((kGated ? unit0 : m_warp) >> 5);
      auto block_ok = [&](int col) { return m_ok && col >= 0 && col < t.n; };
      // Everything the epilogue needs from global memory is requested here, before the accumulator is awaited; head of a
      // queue = next chunk to process.  Lane i of a chunk describes its token column i: the token (scatter products), its
      // gate, its dropout word.  dgrad2: ReLU mask bits of this thread's fragment, two blocks of 16 tokens.
      int q_tok[kQueue] = {-1, -1, -1, -1, -1};
      float q_gate[kQueue] = {1.f, 1.f, 1.f, 1.f, 1.f};
      uint32_t q_mw[kQueue] = {0u, 0u, 0u, 0u, 0u};
      if constexpr (!kSlotRows) {
        const int* tos = p.token_of_slot + (long long)t.e * p.C + t.row0;
#pragma unroll
        for (int k = 0; k < kQueue; ++k) {
          const int j = n_chunks - 1 - half - 2 * k, col = chunk_tok0(j) + lane;
          q_tok[k] = j >= 0 && row_ok(col) ? tos[col] : -1;
        }
        if (OP == kGemm2Combine) {                            // Eq. 2: y = p_i(x) E_i(x)
#pragma unroll
          for (int k = 0; k < kQueue; ++k) q_gate[k] = p.gate[max(q_tok[k], 0)];
        }
      }
      if constexpr (DROP && (OP == kGemm1Relu || kGated)) {   // 32 hidden units are one word per row
        const uint32_t* keep = p.keep_bits + ((long long)t.e * p.C + t.row0) * p.keep_words + ((kGated ? unit0 : m_warp) >> 5);
#pragma unroll
        for (int k = 0; k < kQueue; ++k) {
          const int j = n_chunks - 1 - half - 2 * k, col = chunk_tok0(j) + lane;
          q_mw[k] = j >= 0 && m_ok && row_ok(col) ? keep[(long long)col * p.keep_words] : 0u;
        }
      }
      if constexpr (OP == kDgrad2Mask) {
        const uint16_t* hm = p.hmask + block0 * 32 + lane;
#pragma unroll
        for (int k = 0; k < kQueue; ++k) {
          const int j = n_chunks - 1 - half - 2 * k, tok0 = chunk_tok0(j);
          const uint32_t b0 = j >= 0 && block_ok(tok0) ? hm[(long long)(tok0 >> 4) * p.hid] : 0u;
          const uint32_t b1 = j >= 0 && block_ok(tok0 + 16) ? hm[(long long)((tok0 >> 4) + 1) * p.hid] : 0u;
          q_mw[k] = b0 | (b1 << 16);
        }
      }
      // gated dgrad2: the saved factors of this thread's fragment ({GELU(a), b GELU'(a)} as two bfloat16 per element)
      uint4 gg[kDGated ? 8 : 1];
      auto fetch_factors = [&](int j) {
        if constexpr (kDGated) {
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            const int col = chunk_tok0(j) + 16 * b;
            const bool valid = j >= 0 && block_ok(col);
            const uint4* src = p.gate_buf + (valid ? (block0 + (long long)(col >> 4) * words) * 128 + lane : 0);
#pragma unroll
            for (int q = 0; q < 4; ++q) gg[4 * b + q] = valid ? src[32 * q] : make_uint4(0, 0, 0, 0);
          }
        }
      };
      fetch_factors(n_chunks - 1 - half);
      ok = mbar_wait_warp(tfull0 + 8u * side, use & 1u, abort_flag, p.status, 24);
      if (!ok) break;
      tc_fence_after();
      bool released = false, mid_sent = false;
      uint32_t v[32];                                         // [16 h + 4 g + ..]: weight rows 16 h .., tokens 8 g ..
      auto load_acc = [&](int j) {
        const uint32_t at = t_addr + (uint32_t)chunk_tok0(j);  // (-16 in an odd tile's last chunk: the columns before it)
        tc_ld_16x256b_x4(at, v);
        tc_ld_16x256b_x4(at + (16u << 16), v + 16);
      };
      auto value = [&](int g, int i, int b) { return __uint_as_float(v[16 * (i >> 1) + 4 * g + 2 * (i & 1) + b]); };
      if (m_ok && n_chunks - 1 - half >= 0) load_acc(n_chunks - 1 - half);
#pragma unroll 1
      for (int j = n_chunks - 1 - half; j >= 0 && m_ok; j -= 2) {
        const int tok0 = chunk_tok0(j);
        tc_wait_ld_regs(v);
        if (!mid_sent && j - 2 < j_mid) {                     // this warp's share of the middle columns is read out
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(tmid0 + 8u * side, 0);
          mid_sent = true;
        }
        if (j - 2 < 0) {                                      // last chunk of this warp: accumulator read out
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(tempty0 + 8u * side, 0);
          released = true;
        }
        if constexpr (kGated) {
          // GEGLU gating.  Both warps of a pair round their values (a or b of 32 hidden units x 32 tokens); the a warp
          // gates the chunk's first 16 tokens, the b warp the others: each hands the other its half through its tile,
          // between two handshakes.
          uint32_t mine[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {                       // word 4 g + i of this warp's block, and of the other's
            const int g = k >> 2, i = k & 3;
            const uint32_t w0 = pack_bf16(value(g, i, 0), value(g, i, 1)), w1 = pack_bf16(value(g + 2, i, 0), value(g + 2, i, 1));
            mine[k] = role ? w1 : w0;
            *reinterpret_cast<uint32_t*>(tr + k * 128 + lane * 4) = role ? w0 : w1;
          }
          if (j - 2 >= 0) load_acc(j - 2);
          __syncwarp();
          if (lane == 0) mbar_arrive(gate_bar);
          ok = mbar_wait_warp(gate_bar, gate_phase, abort_flag, p.status, 26);     // both tiles are written
          gate_phase ^= 1u;
          if (!ok) break;
          uint32_t other[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) other[k] = *reinterpret_cast<const uint32_t*>(tr_other + k * 128 + lane * 4);
          __syncwarp();
          if (lane == 0) mbar_arrive(gate_bar);
          ok = mbar_wait_warp(gate_bar, gate_phase, abort_flag, p.status, 27);     // both tiles have been read
          gate_phase ^= 1u;
          if (!ok) break;
          const int col0 = tok0 + 16 * role;                  // this warp's block of 16 tokens
          uint32_t fac[16], hw[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int g = k >> 2, i = k & 3;
            const uint32_t aw = role ? other[k] : mine[k], bw = role ? mine[k] : other[k];
            const float2 af = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw));
            const float2 bf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw));
            float cdf0, pdf0, cdf1, pdf1;
            gelu_cdf_pdf(af.x, &cdf0, &pdf0);
            gelu_cdf_pdf(af.y, &cdf1, &pdf1);
            float ga0 = af.x * cdf0, ga1 = af.y * cdf1;
            float gp0 = bf.x * fmaf(af.x, pdf0, cdf0), gp1 = bf.y * fmaf(af.y, pdf1, cdf1);
            if (DROP) {                                       // expert dropout: the hidden unit's factor on all three
              const int tk = 16 * role + 8 * g + 2 * (lane & 3), unit = 8 * i + (lane >> 2);
              const uint32_t kw0 = __shfl_sync(0xffffffffu, q_mw[0], tk), kw1 = __shfl_sync(0xffffffffu, q_mw[0], tk + 1);
              const float f0 = (kw0 >> unit) & 1u ? p.keep_scale : 0.f, f1 = (kw1 >> unit) & 1u ? p.keep_scale : 0.f;
              ga0 *= f0; gp0 *= f0; ga1 *= f1; gp1 *= f1;
            }
            fac[2 * k] = pack_bf16(ga0, gp0);
            fac[2 * k + 1] = pack_bf16(ga1, gp1);
            hw[k] = pack_bf16(ga0 * bf.x, ga1 * bf.y);
          }
          if (block_ok(col0)) {
            uint4* dst = p.gate_buf + (block0 + (long long)(col0 >> 4) * words) * 128 + lane;
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[32 * q] = make_uint4(fac[4 * q], fac[4 * q + 1], fac[4 * q + 2], fac[4 * q + 3]);
          }
#pragma unroll
          for (int g = 0; g < 2; ++g) stmatrix_trans(st_addr + 512u * g, hw + 4 * g);
          __syncwarp();
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const uint4 val = *reinterpret_cast<const uint4*>(ld_addr + 512 * g);
            const int col = col0 + 8 * g + (lane >> 2);
            if (row_ok(col)) *reinterpret_cast<uint4*>(out_rows + (long long)col * p.ld_out + unit0 + (lane & 3) * 8) = val;
          }
        } else {
          constexpr int kSets = kDGated ? 2 : 1;              // gated dgrad2 writes d a and d b from one accumulator
          uint32_t pk[kSets][16];
          // dgrad2: a block's bits with the even tokens' in the low half, the odd ones' in the high half
          const uint32_t mask[2] = {__byte_perm(q_mw[0], 0, 0x4140), __byte_perm(q_mw[0], 0, 0x4342)};
          if (OP == kGemm2Combine) { gate_s[lane] = q_gate[0]; __syncwarp(); }
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            float2 ga = make_float2(1.f, 1.f);
            if (OP == kGemm2Combine) ga = *reinterpret_cast<const float2*>(gate_s + 8 * g + 2 * (lane & 3));
            uint32_t kw0 = 0u, kw1 = 0u;
            if (DROP && OP == kGemm1Relu) {                   // expert dropout before the rounding and the mask bits
              kw0 = __shfl_sync(0xffffffffu, q_mw[0], 8 * g + 2 * (lane & 3));
              kw1 = __shfl_sync(0xffffffffu, q_mw[0], 8 * g + 2 * (lane & 3) + 1);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              float x = value(g, i, 0), y = value(g, i, 1);
              if (OP == kGemm2Combine) { x *= ga.x; y *= ga.y; }
              if (DROP && OP == kGemm1Relu) {
                const int unit = 8 * i + (lane >> 2);
                x = (kw0 >> unit) & 1u ? x * p.keep_scale : 0.f;
                y = (kw1 >> unit) & 1u ? y * p.keep_scale : 0.f;
              }
              if (DROP && OP == kDgrad2Mask) { x *= p.keep_scale; y *= p.keep_scale; }
              if constexpr (kDGated) {                        // high half: b GELU'(a); low half: GELU(a)
                const uint4 f4 = gg[4 * (g >> 1) + 2 * (g & 1) + (i >> 1)];
                const uint32_t f0 = i & 1 ? f4.z : f4.x, f1 = i & 1 ? f4.w : f4.y;
                pk[0][4 * g + i] = pack_bf16(x * __uint_as_float(f0 & 0xFFFF0000u), y * __uint_as_float(f1 & 0xFFFF0000u));
                pk[kSets - 1][4 * g + i] = pack_bf16(x * __uint_as_float(f0 << 16), y * __uint_as_float(f1 << 16));
              } else {
                uint32_t w = pack_bf16(x, y);
                if (OP == kGemm1Relu) w = relu_bf16x2(w);
                if (OP == kDgrad2Mask)                        // ReLU'(u) = [u > 0]: bits saved by the forward GEMM
                  w &= ((mask[g >> 1] >> (4 * (g & 1) + i)) & 0x00010001u) * 0xFFFFu;
                pk[0][4 * g + i] = w;
              }
            }
          }
          if (j - 2 >= 0) load_acc(j - 2);                    // in flight while this chunk is stored
          fetch_factors(j - 2);
          if (OP == kGemm1Relu) {                             // save [H > 0], one bit per element, in fragment order
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              uint32_t bits = 0;
#pragma unroll
              for (int k = 0; k < 8; ++k) bits |= positive_bf16x2(pk[0][8 * b + k]) & (0x00010001u << k);
              if (block_ok(tok0 + 16 * b))
                p.hmask[block0 * 32 + (long long)((tok0 >> 4) + b) * p.hid + lane] = (uint16_t)((bits & 0xFFu) | (bits >> 8));
            }
          }
#pragma unroll
          for (int set = 0; set < kSets; ++set) {
            if (set > 0) __syncwarp();                        // the tile's readers of the first set are done
#pragma unroll
            for (int g = 0; g < 4; ++g) stmatrix_trans(st_addr + 512u * g, pk[set] + 4 * g);
            __syncwarp();
            const int mcol = m_warp + (lane & 3) * 8 + set * p.gate_f;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              uint4 val = *reinterpret_cast<const uint4*>(ld_addr + 512 * g);
              if (kSlotRows) {
                const int col = tok0 + 8 * g + (lane >> 2);
                if (row_ok(col)) *reinterpret_cast<uint4*>(out_rows + (long long)col * p.ld_out + mcol) = val;
              } else {
                const int tok = __shfl_sync(0xffffffffu, q_tok[0], 8 * g + (lane >> 2));
                if (tok >= 0) {
                  const long long off = (long long)tok * p.ld_out + mcol;
                  if (p.res != nullptr) {
                    // skip path inside the layer: y = x + g E(x), dx = dy + dH W_in^T (the expert term is already bf16)
                    if (OP == kGemm2Combine) *reinterpret_cast<uint4*>(p.out2 + off) = val;
                    const uint4 r = *reinterpret_cast<const uint4*>(p.res + off);
                    const __nv_bfloat162* rv = reinterpret_cast<const __nv_bfloat162*>(&r);
                    __nv_bfloat162* vv = reinterpret_cast<__nv_bfloat162*>(&val);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                      const float2 a2 = __bfloat1622float2(vv[q]), b2 = __bfloat1622float2(rv[q]);
                      vv[q] = __floats2bfloat162_rn(a2.x + b2.x, a2.y + b2.y);
                    }
                  }
                  *reinterpret_cast<uint4*>(p.out + off) = val;
                }
              }
            }
          }
        }
#pragma unroll
        for (int k = 0; k < kQueue - 1; ++k) {                // advance the queue
          q_tok[k] = q_tok[k + 1];
          q_gate[k] = q_gate[k + 1];
          q_mw[k] = q_mw[k + 1];
        }
        __syncwarp();
      }
      if (!ok) break;
      if (!mid_sent) {                                        // this warp had no chunk in this tile
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(tmid0 + 8u * side, 0);
      }
      if (!released) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(tempty0 + 8u * side, 0);
      }
    }
  }

  // ---------------------------------------------------------------------------------------------- teardown
  __syncwarp();                                               // lanes of the last arrivals rejoin their warps
  tc_fence_before();
  cluster_sync_all();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

template <int OP, bool DROP = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPThreads, 1)
expert_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ BMapSet bm,
                        const PairParams p) {
  pair_body<OP, DROP>(tmA, bm, p, (int)(blockIdx.x >> 1), (int)(gridDim.x >> 1));
}

// Two products that read the same activations, side by side in one launch: the first `split` CTA pairs work on
// product A, the others on product B, each walking the experts in the same order.  dgrad1 (dx = dH W_in^T) and wgrad1
// (dW_in = X_d^T dH) both read dH and nothing of each other; run one after the other each reads its 0.2 GB from HBM,
// run together the expert's rows that one of them fetched are still in L2 when the other asks for them (whichever
// runs ahead pays the HBM latency and so falls back: the two stay within a few experts of each other).
template <int OPA, int OPB>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPThreads, 1)
expert_gemm_pair_dual_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ BMapSet tmB0,
                             const PairParams p0, const __grid_constant__ CUtensorMap tmA1,
                             const __grid_constant__ BMapSet tmB1, const PairParams p1, const int split) {
  const int cl = (int)(blockIdx.x >> 1), n = (int)(gridDim.x >> 1);
  if (cl < split) pair_body<OPA>(tmA0, tmB0, p0, cl, split);
  else pair_body<OPB>(tmA1, tmB1, p1, cl - split, n - split);
}

// persistent grid: as many CTA pairs as can be resident at once (at most one CTA per SM).  The occupancy query
// costs tens of microseconds of host time, so its answer is kept per device and kernel.
template <typename Kernel>
int pair_grid(Kernel kernel, int* cached_grid, int dev, int sm_count, cudaStream_t st, int* grid_out) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmemBytes) != cudaSuccess)
    return SWITCH_MOE_CUDA_ERROR;
  int grid = (dev >= 0 && dev < 64) ? cached_grid[dev] : 0;
  if (grid == 0) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(sm_count & ~1), 1, 1);
    lc.blockDim = dim3(kPThreads, 1, 1);
    lc.dynamicSmemBytes = kPSmemBytes;
    lc.stream = st;
    int max_clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&max_clusters, kernel, &lc) != cudaSuccess || max_clusters < 1) {
      (void)cudaGetLastError();
      max_clusters = sm_count / 2;
    }
    grid = 2 * (max_clusters < sm_count / 2 ? max_clusters : sm_count / 2);
    if (grid < 2) return SWITCH_MOE_CUDA_ERROR;
    if (dev >= 0 && dev < 64) cached_grid[dev] = grid;
  }
  *grid_out = grid;
  return SWITCH_MOE_OK;
}

uint32_t magic(int d) { return d > 1 ? (uint32_t)((0x100000000ull + (uint64_t)d - 1) / (uint64_t)d) : 0u; }

// Weight gradients: into how many strips a row of `nt` column tiles is cut.  A strip's A operand is loaded once if its
// k-blocks fit the ring, so longer strips read less (up to 12% of a tile's time at the power limit); but the pairs' shares
// are whole strips, and experts differ in size, so the last one leaves half a strip idle on average.  Experts that on
// average do not fit the ring gain nothing and are balanced tile by tile.  Strips are for the power limit, where training
// runs; before it sets in they cost a little.  Whole training steps, us, tile by tile / strips, at the limit and in bursts at
// full clock: 16384 tokens, 4096 x 10240, 64 experts 9287 / 8898 (always at the limit); 32768 tokens, 768 x 3072, 128 experts
// (strips of 3 and 6) 1291 / 1263, burst 1114 / 1120; top-2 on 64 experts 780 / 764, burst 682 / 682; GEGLU 768 x 2048, 128
// experts (3 and 8) 1433 / 1427, burst 1255 / 1269; 20011 tokens, 512 x 1536, 200 experts 585 / 578, burst 610 / 611.
int set_strips(PairParams* q, int n_pairs) {
  const int nt = q->n_ntiles_fixed;
  const long long rows = (long long)q->E * q->n_mpairs;
  int best = nt;
  float best_cost = 0.f;
  for (int S = q->tokens_per_expert > kPWgradA * kBK ? nt : 1; S <= nt; ++S) {
    const int L = (nt + S - 1) / S;
    const float tiles = (float)((rows * S + n_pairs - 1) / n_pairs * L);
    const float cost = tiles * (1.f + 0.12f * (float)S / (float)nt) + 0.5f * (float)L;
    if (best_cost == 0.f || cost < best_cost) { best = S; best_cost = cost; }
  }
  q->strips = best;
  const uint64_t per_e = (uint64_t)q->n_mpairs * best;        // the decode is exact while id * divisor < 2^32
  if ((uint64_t)q->E * per_e * per_e >= 0x100000000ull) return SWITCH_MOE_UNSUPPORTED_SHAPE;
  q->magic_per_e = magic((int)per_e);
  q->magic_strips = magic(best);
  return SWITCH_MOE_OK;
}

template <int OP, bool DROP = false>
int launch_pair_op(const CUtensorMap& tmA, const BMapSet& tmB, PairParams q, int dev, int sm_count,
                   cudaStream_t st) {
  static int cached_grid[64] = {0};
  int grid = 0;
  const int rc = pair_grid(expert_gemm_pair_kernel<OP, DROP>, cached_grid, dev, sm_count, st, &grid);
  if (rc != SWITCH_MOE_OK) return rc;
  if (!q.token_op && set_strips(&q, grid / 2) != SWITCH_MOE_OK) return SWITCH_MOE_UNSUPPORTED_SHAPE;
  launch_k(expert_gemm_pair_kernel<OP, DROP>, dim3(grid), dim3(kPThreads), kPSmemBytes, st, tmA, tmB, q);
  return launch_status();
}

// Widest token tile: what the capacity allows, rounded up to the MMA's granularity.
int widest_tile(const Shape& s) { return s.C < kPairTileTokens ? (s.C + 15) / 16 * 16 : kPairTileTokens; }

// The token operand's maps: one per box height (8 j rows) up to half of the widest tile or segment.
int make_token_maps(BMapSet* bm, const Shape& s, const void* base, long long cols) {
  const int most = widest_tile(s) / 16 < kBMaps ? widest_tile(s) / 16 : kBMaps;
  for (int j = 1; j <= most; ++j)
    if (make_map(&bm->m[j - 1], base, s.E, s.C, cols, 8 * j) != SWITCH_MOE_OK) return SWITCH_MOE_CUDA_ERROR;
  return SWITCH_MOE_OK;
}

// Operands, output and tile counts of one product.
int pair_problem(GemmOp op, const Shape& s, const Plan& p, const GemmArgs& a, void* ws, PairParams* out,
                 CUtensorMap* tmA_out, BMapSet* tmB_out) {
  const void* xd = ws_ptr<char>(ws, p.xd);
  const void* h = ws_ptr<char>(ws, p.h);
  const void* dyd = ws_ptr<char>(ws, p.dyd);
  const void* dh = ws_ptr<char>(ws, p.dh);
  const int fin = s.fin;                                      // columns of W_in: f, or 2 f for GEGLU experts
  const void* du = s.geglu ? ws_ptr<char>(ws, p.dab) : dh;    // gradient of the pre-activation(s)

  PairParams q{};
  q.op = (int)op;
  q.C = s.C; q.E = s.E;
  q.ntile = ws_ptr<int4>(ws, p.ntile);
  q.kept = ws_ptr<int>(ws, p.kept);
  q.token_of_slot = ws_ptr<int>(ws, p.token_of_slot);
  q.gate = ws_ptr<float>(ws, p.gate);
  q.status = ws_ptr<int>(ws, p.status);
  q.hmask = ws_ptr<uint16_t>(ws, p.hmask);
  q.cb = (s.C + 15) / 16; q.hid = s.f;
  q.keep_scale = 1.f;
  CUtensorMap& tmA = *tmA_out;
  BMapSet& bm = *tmB_out;
  CUtensorMap& tmB = bm.m[0];
  int rc = SWITCH_MOE_OK, rc2 = SWITCH_MOE_OK;
  int K = 0;
  switch (op) {
    case kGemm1Relu:       // A = W_in [E][d (k)][f (m)]: m contiguous -> MN-major; B = X_d [E][C][d] K-major
      q.token_op = 1; q.a_mn_major = 1; q.Mw = fin; K = s.d;   // GEGLU: 2 f weight columns [W_0 | W_1], no ReLU
      rc = make_map(&tmA, a.W_in, s.E, s.d, fin, 64); rc2 = make_token_maps(&bm, s, xd, s.d);
      q.out = ws_ptr<__nv_bfloat16>(ws, p.h); q.ld_out = s.f;
      if (s.geglu) { q.gate_f = s.f; q.gate_buf = ws_ptr<uint4>(ws, p.ab); }   // gating in the epilogue
      if (s.dropout) {
        if (s.keep_bits == nullptr || (reinterpret_cast<uintptr_t>(s.keep_bits) & 3u) != 0) return SWITCH_MOE_INVALID_ARGUMENT;
        q.keep_bits = s.keep_bits; q.keep_words = s.f / 32; q.keep_scale = s.keep_scale;
      }
      break;
    case kGemm2Combine:    // A = W_out [E][f (k)][d (m)] MN-major; B = H [E][C][f] K-major
      q.token_op = 1; q.a_mn_major = 1; q.Mw = s.d; K = s.f;
      rc = make_map(&tmA, a.W_out, s.E, s.f, s.d, 64); rc2 = make_token_maps(&bm, s, h, s.f);
      q.out = static_cast<__nv_bfloat16*>(a.y); q.ld_out = s.d;
      if (s.residual && !s.top2) {   // (top-2 routing adds the skip path where the two assignments' rows are summed)
        q.res = static_cast<const __nv_bfloat16*>(a.x); q.out2 = ws_ptr<__nv_bfloat16>(ws, p.layer_y);
      }
      break;
    case kDgrad2Mask:      // A = W_out [E][f (m)][d (k)] K-major; B = dY_d [E][C][d] K-major
      q.token_op = 1; q.a_mn_major = 0; q.Mw = s.f; K = s.d;
      rc = make_map(&tmA, a.W_out, s.E, s.f, s.d, 128); rc2 = make_token_maps(&bm, s, dyd, s.d);
      q.out = ws_ptr<__nv_bfloat16>(ws, p.dh); q.ld_out = s.f;
      if (s.dropout && !s.geglu) q.keep_scale = s.keep_scale;   // (GEGLU: the saved factors carry the dropout factor)
      if (s.geglu) {   // the derivative of the gating in the epilogue: d[a | b] is written, dH never is
        q.out = ws_ptr<__nv_bfloat16>(ws, p.dab); q.ld_out = fin; q.gate_f = s.f;
        q.gate_buf = ws_ptr<uint4>(ws, p.ab);
      }
      break;
    case kDgrad1Scatter:   // A = W_in [E][d (m)][f (k)] K-major; B = dH [E][C][f] K-major  (GEGLU: d[a | b], K = 2 f)
      q.token_op = 1; q.a_mn_major = 0; q.Mw = s.d; K = fin;
      rc = make_map(&tmA, a.W_in, s.E, s.d, fin, 128); rc2 = make_token_maps(&bm, s, du, fin);
      q.out = static_cast<__nv_bfloat16*>(a.dx); q.ld_out = s.d;
      if (s.residual && !s.top2) q.res = static_cast<const __nv_bfloat16*>(a.dy);
      break;
    case kWgrad2:          // dW_out [f][d] = H^T dY_d: A = H [E][C (k)][f (m)] MN-major; B = dY_d [E][C (k)][d (n)]
      q.token_op = 0; q.a_mn_major = 1; q.Mw = s.f; q.Nfix = s.d;
      rc = make_map(&tmA, h, s.E, s.C, s.f, 64); rc2 = make_map(&tmB, dyd, s.E, s.C, s.d, 64);
      q.out = static_cast<__nv_bfloat16*>(a.dW_out); q.ld_out = s.d; break;
    case kWgrad1:          // dW_in [d][f] = X_d^T dH  (GEGLU: X_d^T d[a | b], 2 f columns)
      q.token_op = 0; q.a_mn_major = 1; q.Mw = s.d; q.Nfix = fin;
      rc = make_map(&tmA, xd, s.E, s.C, s.d, 64); rc2 = make_map(&tmB, du, s.E, s.C, fin, 64);
      q.out = static_cast<__nv_bfloat16*>(a.dW_in); q.ld_out = fin; break;
    default: return SWITCH_MOE_INVALID_ARGUMENT;
  }
  if (rc != SWITCH_MOE_OK || rc2 != SWITCH_MOE_OK) return SWITCH_MOE_CUDA_ERROR;
  q.tokens_per_expert = s.Tv / s.E < s.C ? s.Tv / s.E : s.C;
  q.n_mpairs = (q.Mw + 255) / 256;
  // operand ring of the token products: a stage holds A (16 KB) and this CTA's half of the widest token tile the
  // capacity allows (at most kPairTileTokens / 2 rows of 128 bytes, rounded up to whole 1 KB swizzle atoms)
  const int widest = widest_tile(s);
  q.stage_bytes = kPHalfBytes + ((widest / 2) * 128 + 1023) / 1024 * 1024;
  q.stages = kPRingBytes / q.stage_bytes < kPMaxStages ? kPRingBytes / q.stage_bytes : kPMaxStages;
  q.n_ntiles_fixed = q.token_op ? 0 : (q.Nfix + 255) / 256;
  q.k_blocks_fixed = q.token_op ? K / kBK : 0;
  q.magic_mpairs = magic(q.n_mpairs);
  // (weight gradients: set_strips)
  if (q.token_op && (uint64_t)s.max_mtiles * q.n_mpairs * q.n_mpairs >= 0x100000000ull) return SWITCH_MOE_UNSUPPORTED_SHAPE;
  *out = q;
  return SWITCH_MOE_OK;
}

int device_and_sms(int* dev, int* sm_count) {
  if (cudaGetDevice(dev) != cudaSuccess) return SWITCH_MOE_CUDA_ERROR;
  if (cudaDeviceGetAttribute(sm_count, cudaDevAttrMultiProcessorCount, *dev) != cudaSuccess)
    return SWITCH_MOE_CUDA_ERROR;
  return SWITCH_MOE_OK;
}

}  // namespace

int launch_pair_gemm(GemmOp op, const Shape& s, const Plan& p, const GemmArgs& a, void* ws, cudaStream_t st) {
  int dev = 0, sm_count = 0;
  if (device_and_sms(&dev, &sm_count) != SWITCH_MOE_OK) return SWITCH_MOE_CUDA_ERROR;
  PairParams q;
  CUtensorMap tmA;
  BMapSet tmB;
  const int rc = pair_problem(op, s, p, a, ws, &q, &tmA, &tmB);
  if (rc != SWITCH_MOE_OK) return rc;
  switch (op) {
    case kGemm1Relu:
      if (s.geglu) return s.dropout ? launch_pair_op<kGemm1Gated, true>(tmA, tmB, q, dev, sm_count, st)
                                    : launch_pair_op<kGemm1Gated>(tmA, tmB, q, dev, sm_count, st);
      return s.dropout ? launch_pair_op<kGemm1Relu, true>(tmA, tmB, q, dev, sm_count, st)
                       : launch_pair_op<kGemm1Relu>(tmA, tmB, q, dev, sm_count, st);
    case kGemm2Combine: return launch_pair_op<kGemm2Combine>(tmA, tmB, q, dev, sm_count, st);
    case kDgrad2Mask:
      if (s.geglu) return launch_pair_op<kDgrad2Gated>(tmA, tmB, q, dev, sm_count, st);
      return s.dropout ? launch_pair_op<kDgrad2Mask, true>(tmA, tmB, q, dev, sm_count, st)
                       : launch_pair_op<kDgrad2Mask>(tmA, tmB, q, dev, sm_count, st);
    case kDgrad1Scatter: return launch_pair_op<kDgrad1Scatter>(tmA, tmB, q, dev, sm_count, st);
    case kWgrad2: return launch_pair_op<kWgrad2>(tmA, tmB, q, dev, sm_count, st);
    default: return launch_pair_op<kWgrad1>(tmA, tmB, q, dev, sm_count, st);
  }
}

// dgrad1 and wgrad1 in one launch (see expert_gemm_pair_dual_kernel).  The two products have the same flops, but a weight
// gradient's tile contracts over the expert's tokens only, so with few of them its epilogue (256 x 256 outputs for a few
// k-blocks) weighs more and it gets the larger share of the CTA pairs.  Measured on 74 pairs, pairs for dgrad1: 32 to 256
// tokens per expert 33 is best (768 x 3072, 128 experts: 256 tokens 322 us against 329 with 35 and 347 with 37; 32 tokens
// 211 / 214 / 225; 1792 x 4864, 113 tokens 154 / 162 / 169), 512 tokens and more an even split (512 x 1536, 2048 tokens 77 us
// against 85 with 33; 256 x 512, 512 tokens 46 / 50).
int launch_pair_dgrad1_wgrad1(const Shape& s, const Plan& p, const GemmArgs& a, void* ws, cudaStream_t st) {
  int dev = 0, sm_count = 0;
  if (device_and_sms(&dev, &sm_count) != SWITCH_MOE_OK) return SWITCH_MOE_CUDA_ERROR;
  PairParams q0, q1;
  CUtensorMap tmA0, tmA1;
  BMapSet tmB0, tmB1;
  int rc = pair_problem(kDgrad1Scatter, s, p, a, ws, &q0, &tmA0, &tmB0);
  if (rc != SWITCH_MOE_OK) return rc;
  rc = pair_problem(kWgrad1, s, p, a, ws, &q1, &tmA1, &tmB1);
  if (rc != SWITCH_MOE_OK) return rc;
  static int cached_grid[64] = {0};
  int grid = 0;
  auto kernel = expert_gemm_pair_dual_kernel<kDgrad1Scatter, kWgrad1>;
  rc = pair_grid(kernel, cached_grid, dev, sm_count, st, &grid);
  if (rc != SWITCH_MOE_OK) return rc;
  const int n_pairs = grid / 2;
  if (n_pairs < 2) {                                          // nothing to share a launch with: one after the other
    rc = launch_pair_op<kDgrad1Scatter>(tmA0, tmB0, q0, dev, sm_count, st);
    return rc != SWITCH_MOE_OK ? rc : launch_pair_op<kWgrad1>(tmA1, tmB1, q1, dev, sm_count, st);
  }
  const bool few_tokens = s.Tv < 384 * s.E;                   // per expert, before the capacity cut
  int split = few_tokens ? (n_pairs * 33 + 37) / 74 : n_pairs / 2;
  if (split < 1) split = 1;
  if (split > n_pairs - 1) split = n_pairs - 1;
  if (set_strips(&q1, n_pairs - split) != SWITCH_MOE_OK) return SWITCH_MOE_UNSUPPORTED_SHAPE;
  launch_k(kernel, dim3(grid), dim3(kPThreads), kPSmemBytes, st, tmA0, tmB0, q0, tmA1, tmB1, q1, split);
  return launch_status();
}

}  // namespace swmoe
