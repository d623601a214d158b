// Grouped expert GEMMs on the plain FP32 FMA pipes (no tensor cores): the expert FFN h = x W_in, y = ReLU(h) W_out
// (Section 5, FFN review) and its derivatives, one problem per expert, with the same fused epilogues as the
// tensor-core path.  These are the small products of the float32 layer (f32_gemm_sm100.cu has the rule and the others) and a
// validation path for either type; accumulation is float32, one fused multiply-add per term in ascending order of the
// contraction index, whatever the tile.
//
// What bounds it is the FMA pipes: 128 multiply-adds per SM and clock, 74.5 TFLOP/s.  A plain FFMA takes an issue slot
// per multiply-add and leaves none for the operand loads; the packed form (fma.rn.f32x2, two independent IEEE
// multiply-adds) halves the slots.  In the large tile a thread keeps 8 x 8 outputs (two groups of 4 rows x two groups of
// 4 columns), so four 16-byte shared-memory loads feed 64 multiply-adds, and the next k-chunk travels from global memory
// to registers while the current one is multiplied; three blocks of four warps per SM leave it 168 registers.  Warps whose rows lie past an expert's last token multiply nothing.
// Measured at 4096 tokens, 512 x 2048, 16 experts (on this path; by default that layer runs on the tensor cores): weight gradients 168 us each (51 TFLOP/s) where 64 x 64 tiles with plain
// FFMA and no prefetch took 330; GEMM1 187 (377), dgrad2 214 (385).
#include "switch_common.cuh"

namespace swmoe {
namespace {

struct SimtProblem {
  const void* A; long long a_es, a_ms, a_ks;   // A(e, m, k) element strides; one of a_ms, a_ks is 1
  const void* B; long long b_es, b_ks, b_ns;   // B(e, k, n) element strides; one of b_ks, b_ns is 1
  int M, K, N;                                  // M < 0: M_e = kept[e];  K < 0: K_e = kept[e]
  int C;                                        // expert capacity (rows per expert of the slot buffers)
  const int* kept; const int* token_of_slot; const float* gate;
  void* out; const void* mask_src; int ld_out;
  const void* res;   // combine / scatter with the skip path inside the layer: row added to the output (x or dy)
  void* out2;        // combine with the skip path: second copy of the output without it
  int plain;         // GEMM1 / dgrad2 without ReLU and mask (GEGLU experts gate elsewhere)
};

// Four consecutive elements as float4 (16-byte aligned float32, 8-byte aligned bfloat16).
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}
__device__ __forceinline__ float rnd(const float*, float v) { return v; }
__device__ __forceinline__ float rnd(const __nv_bfloat16*, float v) { return __bfloat162float(__float2bfloat16(v)); }

__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// BM x BN outputs and BK contraction steps per round and block, WM x WN warps of (BM / WM) x (BN / WN) outputs; the
// 4 x 8 lanes of a warp hold RG groups of 4 rows and CG groups of 4 columns each.
template <int BM_, int BN_, int BK_, int WM_, int WN_, int kMinBlocks_>
struct Tile {
  static constexpr int BM = BM_, BN = BN_, BK = BK_, WM = WM_, WN = WN_, kThreads = 32 * WM_ * WN_;
  static constexpr int kMinBlocks = kMinBlocks_;
  static constexpr int RG = BM / WM / 16, CG = BN / WN / 32;
};
using BigTile = Tile<64, 128, 16, 2, 2, 3>;
using MidTile = Tile<64, 64, 32, 2, 2, 4>;
using SmallTile = Tile<32, 32, 64, 2, 1, 6>;

// A k-contiguous operand is transposed on its way into shared memory: eight lanes write the same rows of eight different
// steps, rows of R + 4 floats that start in only two banks.  Exchanging groups of four rows by the step spreads them over
// all banks and keeps 16-byte reads whole.
// (4096 tokens, 512 x 2048, 16 experts: dgrad1 254 -> 242 us, GEMM2 240 -> 233 with rounds of 32 steps; with rounds of 16,
// four steps to a row, the extra address arithmetic costs what the conflicts did.)
template <bool kKFast, int BK>
__device__ __forceinline__ int swizzle(int k) {
  return kKFast && BK > 16 ? ((k >> 2) & 7) << 2 : 0;
}

// One operand tile of R rows (m or n) x BK contraction steps: global -> registers -> shared memory [k][row].
template <typename ET, int R, int BK, int kThreads, bool kKFast>
struct Stager {
  static constexpr int kVecs = R * BK / 4 / kThreads;          // 4-element loads per thread
  static_assert(kVecs >= 1, "tile too small for the block");
  float4 v[kVecs];
  __device__ __forceinline__ static int row_of(int i) {
    const int idx = (int)threadIdx.x + i * kThreads;
    return kKFast ? idx / (BK / 4) : idx % (R / 4) * 4;
  }
  __device__ __forceinline__ static int k_of(int i) {
    const int idx = (int)threadIdx.x + i * kThreads;
    return kKFast ? idx % (BK / 4) * 4 : idx / (R / 4);
  }
  __device__ __forceinline__ void fetch(const ET* base, long long rs, long long ks, int r0, int rows, int k0, int K) {
#pragma unroll
    for (int i = 0; i < kVecs; ++i) {
      // Extents along a contiguous axis are multiples of 8, so a group of 4 is inside or outside -- except a
      // contraction over an expert's tokens, which is never the contiguous axis.
      const int r = r0 + row_of(i), k = k0 + k_of(i);
      v[i] = r < rows && k < K ? ld4(base + (long long)r * (kKFast ? rs : 1) + (long long)k * (kKFast ? 1 : ks))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void put(float (*s)[R + 4]) const {
#pragma unroll
    for (int i = 0; i < kVecs; ++i) {
      const int k = k_of(i), r = row_of(i) ^ swizzle<kKFast, BK>(k);
      if (kKFast) {
        s[k][r] = v[i].x; s[k + 1][r] = v[i].y; s[k + 2][r] = v[i].z; s[k + 3][r] = v[i].w;
      } else {
        *reinterpret_cast<float4*>(&s[k][r]) = v[i];
      }
    }
  }
};

template <typename ET, int OP, typename TL>
__global__ void __launch_bounds__(TL::kThreads, TL::kMinBlocks) simt_grouped_gemm_kernel(const SimtProblem pr) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr bool kAKFast = OP != kWgrad2 && OP != kWgrad1;             // token rows: the contraction is contiguous
  constexpr bool kBKFast = OP == kDgrad2Mask || OP == kDgrad1Scatter;  // transposed weights
  constexpr int BM = TL::BM, BN = TL::BN, BK = TL::BK, RG = TL::RG, CG = TL::CG;
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ __align__(16) float Bs[2][BK][BN + 4];
  const int e = blockIdx.z;
  const int kept_e = pr.kept[e];
  const int M = pr.M < 0 ? kept_e : pr.M;
  const int K = pr.K < 0 ? kept_e : pr.K;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= M) return;
  const ET* A = static_cast<const ET*>(pr.A) + (long long)e * pr.a_es;
  const ET* B = static_cast<const ET*>(pr.B) + (long long)e * pr.b_es;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wm = warp / TL::WN * (BM / TL::WM), wn = warp % TL::WN * (BN / TL::WN);
  const int row = wm + (lane >> 3) * 4, col = wn + (lane & 7) * 4;     // + 16 per row group, + 32 per column group
  const bool busy = m0 + wm < M && n0 + wn < pr.N;                     // any output of this warp inside the problem

  unsigned long long acc[RG * 4][CG * 2];
#pragma unroll
  for (int i = 0; i < RG * 4; ++i)
#pragma unroll
    for (int j = 0; j < CG * 2; ++j) acc[i][j] = 0ull;

  Stager<ET, BM, BK, TL::kThreads, kAKFast> sa;
  Stager<ET, BN, BK, TL::kThreads, kBKFast> sb;
  auto fetch = [&](int k0) {
    sa.fetch(A, pr.a_ms, pr.a_ks, m0, M, k0, K);
    sb.fetch(B, pr.b_ns, pr.b_ks, n0, pr.N, k0, K);
  };
  fetch(0);
  sa.put(As[0]);
  sb.put(Bs[0]);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < K;
    if (more) fetch(k0 + BK);
    if (busy) {
#pragma unroll 16
      for (int kk = 0; kk < BK; ++kk) {
        float4 a[RG];
        unsigned long long b[CG * 2];
#pragma unroll
        for (int g = 0; g < RG; ++g) a[g] = *reinterpret_cast<const float4*>(&As[buf][kk][(row + 16 * g) ^ swizzle<kAKFast, BK>(kk)]);
#pragma unroll
        for (int g = 0; g < CG; ++g) {
          const float4 t = *reinterpret_cast<const float4*>(&Bs[buf][kk][(col + 32 * g) ^ swizzle<kBKFast, BK>(kk)]);
          b[2 * g] = pack2(t.x, t.y);
          b[2 * g + 1] = pack2(t.z, t.w);
        }
#pragma unroll
        for (int g = 0; g < RG; ++g) {
          const unsigned long long a0 = pack2(a[g].x, a[g].x), a1 = pack2(a[g].y, a[g].y);
          const unsigned long long a2 = pack2(a[g].z, a[g].z), a3 = pack2(a[g].w, a[g].w);
#pragma unroll
          for (int j = 0; j < CG * 2; ++j) {
            fma2(acc[4 * g][j], a0, b[j]);
            fma2(acc[4 * g + 1][j], a1, b[j]);
            fma2(acc[4 * g + 2][j], a2, b[j]);
            fma2(acc[4 * g + 3][j], a3, b[j]);
          }
        }
      }
    }
    if (more) {                                                // the other buffer was last read before the last barrier
      sa.put(As[buf ^ 1]);
      sb.put(Bs[buf ^ 1]);
      __syncthreads();
    }
  }

#pragma unroll
  for (int i = 0; i < RG * 4; ++i) {
    const int m = m0 + row + 16 * (i >> 2) + (i & 3);
    if (m >= M) continue;
    long long orow;
    float scale = 1.f;
    if (OP == kGemm2Combine || OP == kDgrad1Scatter) {
      const int tok = pr.token_of_slot[(long long)e * pr.C + m];
      orow = (long long)tok * pr.ld_out;
      if (OP == kGemm2Combine) scale = pr.gate[tok];                 // Eq. 2: y = p_i(x) E_i(x)
    } else if (OP == kGemm1Relu || OP == kDgrad2Mask) {
      orow = ((long long)e * pr.C + m) * pr.ld_out;
    } else {
      orow = ((long long)e * M + m) * pr.ld_out;
    }
#pragma unroll
    for (int g = 0; g < CG; ++g) {
      const int n = n0 + col + 32 * g;                         // N is a multiple of 8: a group of 4 is inside or outside
      if (n >= pr.N) continue;
      const float2 lo = unpack2(acc[i][2 * g]), hi = unpack2(acc[i][2 * g + 1]);
      float4 v = make_float4(lo.x * scale, lo.y * scale, hi.x * scale, hi.y * scale);
      if (OP == kGemm1Relu && !pr.plain) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
      if (OP == kDgrad2Mask && !pr.plain) {
        const float4 h = ld4(static_cast<const ET*>(pr.mask_src) + orow + n);
        v = make_float4(h.x > 0.f ? v.x : 0.f, h.y > 0.f ? v.y : 0.f, h.z > 0.f ? v.z : 0.f, h.w > 0.f ? v.w : 0.f);
      }
      if (OP == kGemm2Combine && pr.out2 != nullptr) st4(static_cast<ET*>(pr.out2) + orow + n, v);
      if ((OP == kGemm2Combine || OP == kDgrad1Scatter) && pr.res != nullptr) {   // the expert term is rounded first
        const float4 r = ld4(static_cast<const ET*>(pr.res) + orow + n);
        const ET* t = nullptr;
        v = make_float4(rnd(t, v.x) + r.x, rnd(t, v.y) + r.y, rnd(t, v.z) + r.z, rnd(t, v.w) + r.w);
      }
      st4(static_cast<ET*>(pr.out) + orow + n, v);
    }
  }
}

template <typename ET, int OP, typename TL>
void launch_tile(const SimtProblem& pr, int max_m, int E, cudaStream_t st) {
  const dim3 grid((unsigned)((pr.N + TL::BN - 1) / TL::BN), (unsigned)((max_m + TL::BM - 1) / TL::BM), (unsigned)E);
  launch_k(simt_grouped_gemm_kernel<ET, OP, TL>, grid, dim3(TL::kThreads), 0, st, pr);
}

template <typename ET, int OP>
void launch_op(const SimtProblem& pr, int max_m, int E, cudaStream_t st) {
  // The largest tile that still occupies the chip: below that a launch waits for the few blocks there are, each walking
  // its whole contraction, and smaller tiles spread the outputs over more SMs.  64 x 128 tiles (three blocks per SM) want
  // as many blocks as are resident: at 4096 tokens, 512 x 2048, 16 experts (SWITCH_MOE_GEMM_SIMT) GEMM2's 320 blocks took 299 us, 64 x 64 tiles
  // 240, while GEMM1 (1280 blocks) takes 187 and 221.  128 x 128 tiles: 371 and 215 (a third of their rows lie past the
  // experts' last tokens).  GEMM2 of 512 tokens, 64 x 256, 8 experts: 27 us with 64 x 64 tiles and 16 steps per round, 13
  // with 32 x 32 and 64 steps.
  constexpr long long kEnoughBig = BigTile::kMinBlocks * kChipSms, kEnough = kChipSms * 3 / 2;
  auto blocks = [&](int bm, int bn) { return (long long)((pr.N + bn - 1) / bn) * ((max_m + bm - 1) / bm) * E; };
  if (blocks(BigTile::BM, BigTile::BN) >= kEnoughBig) launch_tile<ET, OP, BigTile>(pr, max_m, E, st);
  else if (blocks(MidTile::BM, MidTile::BN) >= kEnough) launch_tile<ET, OP, MidTile>(pr, max_m, E, st);
  else launch_tile<ET, OP, SmallTile>(pr, max_m, E, st);
}

template <typename ET>
int launch_t(GemmOp op, const Shape& s, const Plan& p, const GemmArgs& a, void* ws, cudaStream_t st) {
  SimtProblem pr{};
  const long long C = s.C, d = s.d, f = s.f;
  pr.C = s.C;
  pr.kept = ws_ptr<int>(ws, p.kept);
  pr.token_of_slot = ws_ptr<int>(ws, p.token_of_slot);
  pr.gate = ws_ptr<float>(ws, p.gate);
  void* xd = ws_ptr<char>(ws, p.xd); void* h = ws_ptr<char>(ws, p.h);
  void* dyd = ws_ptr<char>(ws, p.dyd); void* dh = ws_ptr<char>(ws, p.dh);
  const long long fin = s.fin;                               // columns of W_in: f, or 2 f for GEGLU experts
  void* ab = ws_ptr<char>(ws, p.ab);
  void* du = s.geglu ? ws_ptr<char>(ws, p.dab) : dh;         // gradient of the pre-activation(s)
  int max_m;
  switch (op) {
    case kGemm1Relu:      // H[e] (C x f) = ReLU(X_d[e] (C x d) . W_in[e] (d x f));  GEGLU: [a | b] (C x 2f), no ReLU
      pr = SimtProblem{xd, C * d, d, 1, a.W_in, d * fin, fin, 1, -1, s.d, s.fin, s.C, pr.kept, pr.token_of_slot,
                       pr.gate, s.geglu ? ab : h, nullptr, s.fin};
      pr.plain = s.geglu;
      max_m = s.C; break;
    case kGemm2Combine:   // y[token] = g . (H[e] (C x f) . W_out[e] (f x d))
      pr = SimtProblem{h, C * f, f, 1, a.W_out, f * d, d, 1, -1, s.f, s.d, s.C, pr.kept, pr.token_of_slot, pr.gate,
                       a.y, nullptr, s.d};
      max_m = s.C; break;
    case kDgrad2Mask:     // dH[e] = (dY_d[e] (C x d) . W_out[e]^T (d x f)) * [H > 0];  GEGLU: no mask
      pr = SimtProblem{dyd, C * d, d, 1, a.W_out, f * d, 1, d, -1, s.d, s.f, s.C, pr.kept, pr.token_of_slot, pr.gate,
                       dh, h, s.f};
      pr.plain = s.geglu;
      max_m = s.C; break;
    case kDgrad1Scatter:  // dx[token] = dH[e] (C x f) . W_in[e]^T (f x d);  GEGLU: d[a | b] (C x 2f)
      pr = SimtProblem{du, C * fin, fin, 1, a.W_in, d * fin, 1, fin, -1, s.fin, s.d, s.C, pr.kept, pr.token_of_slot,
                       pr.gate, a.dx, nullptr, s.d};
      max_m = s.C; break;
    case kWgrad2:         // dW_out[e] (f x d) = H[e]^T (f x kept) . dY_d[e] (kept x d)
      pr = SimtProblem{h, C * f, 1, f, dyd, C * d, d, 1, s.f, -1, s.d, s.C, pr.kept, pr.token_of_slot, pr.gate,
                       a.dW_out, nullptr, s.d};
      max_m = s.f; break;
    case kWgrad1:         // dW_in[e] (d x f) = X_d[e]^T (d x kept) . dH[e] (kept x f);  GEGLU: d[a | b], 2f columns
      pr = SimtProblem{xd, C * d, 1, d, du, C * fin, fin, 1, s.d, -1, s.fin, s.C, pr.kept, pr.token_of_slot, pr.gate,
                       a.dW_in, nullptr, s.fin};
      max_m = s.d; break;
    default: return SWITCH_MOE_INVALID_ARGUMENT;
  }
  // (top-2 routing adds the skip path where the two assignments' rows are summed, not here)
  if (s.residual && !s.top2 && op == kGemm2Combine) { pr.res = a.x; pr.out2 = ws_ptr<char>(ws, p.layer_y); }
  if (s.residual && !s.top2 && op == kDgrad1Scatter) pr.res = a.dy;
  switch (op) {
    case kGemm1Relu: launch_op<ET, kGemm1Relu>(pr, max_m, s.E, st); break;
    case kGemm2Combine: launch_op<ET, kGemm2Combine>(pr, max_m, s.E, st); break;
    case kDgrad2Mask: launch_op<ET, kDgrad2Mask>(pr, max_m, s.E, st); break;
    case kDgrad1Scatter: launch_op<ET, kDgrad1Scatter>(pr, max_m, s.E, st); break;
    case kWgrad2: launch_op<ET, kWgrad2>(pr, max_m, s.E, st); break;
    case kWgrad1: launch_op<ET, kWgrad1>(pr, max_m, s.E, st); break;
  }
  return launch_status();
}

}  // namespace

int launch_simt_gemm(GemmOp op, const Shape& s, const Plan& p, const GemmArgs& a, void* ws, cudaStream_t st) {
  return s.dtype == SWITCH_MOE_BF16 ? launch_t<__nv_bfloat16>(op, s, p, a, ws, st)
                                    : launch_t<float>(op, s, p, a, ws, st);
}

}  // namespace swmoe
