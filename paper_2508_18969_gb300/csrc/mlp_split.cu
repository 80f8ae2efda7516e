// FP32 network layers on the 5th-generation tensor cores: out = act(A W^T + b) with every FP32
// operand held as three BF16 planes, v = v0 + v1 + v2 (v0 = bf16(v), v1 = bf16(v - v0), v2 the rest:
// 8 + 8 + 8 significant bits, so the sum is v exactly), and the product summed as
//   A0 W2 + A2 W0 + A1 W1 + A1 W0 + A0 W1 + A0 W0
// by tcgen05.mma kind::f16 into FP32 accumulators. The three products left out (A1 W2, A2 W1,
// A2 W2) are below 2^-24 of |a||w|, less than the rounding of one FP32 multiplication.
//
// Accumulation. The tensor core truncates as it adds, so a long chain in one accumulator would
// drift. Each k-block of 64 therefore starts its own accumulator, adds the small products before
// the large ones (their truncations are 2^-8 and less of the result's ulp), and the epilogue warps
// add the k-blocks' sums into FP32 registers, rounding to nearest. On rows of the 32-1600-800-400-30
// network the outputs are 2.3e-7 off the FP64 ones (2-norm), against 8.2e-7 with a chain of FP32 FMAs
// (11-256-128-64-9: 2.1e-7 against 3.5e-7; 32-2048-1024-512-4: 3.4e-7 against 1.5e-6).
//
// What bounds it: six BF16 MMAs per product, so a sixth of the tensor rate (323 TFLOP/s of the
// measured 1939) against the ~70 TFLOP/s of the FP32 pipes. Wide tiling: 256 rows x 256 columns on CTA
// pairs (cta_group::2): per k-block an SM loads 96 KB for 24 MMAs of 256 columns. A stage is one plane
// of one k-block (A 16 KB + W 16 KB), two per plane: with plane 2 freed after the first two products,
// plane 1 after the next three and plane 0 at the end, each load has between one and one and two thirds
// k-blocks of time to land, in the 192 KB that two whole k-blocks take. Small tiling: 128 x 64 on single
// CTAs, two epilogue groups that take tiles in turn, so the end of one tile (activation, planes, stores)
// overlaps the sums of the next: best where a batch is short or the epilogue is most of the work (rule
// in launch_split). On 131,072 rows of that network, us per layer (FP32 FMAs / wide / small):
//   32 -> 1600: 739 / 361 / 272 (1.26 GB of planes written: 4.6 TB/s);  1600 -> 800: 8012 / 1261 / 3204
//   (wide: 266 TFLOP/s, 0.82 of the bound);  800 -> 400: 2302 / 400 / 899;  400 -> 30: 301 / 93 / 79.
// (128-column pair tiles with two groups took 410, 1889, 593 and 100 us.)
//
// Results that are not finite: products of an infinite operand with the other's planes would give
// NaN (inf x 0) where FP32 arithmetic gives an infinity, and a sum near the end of the FP32 range
// may overflow in another order. A CTA that met such a sum goes over its tiles once more when its
// pipeline has ended (redo_nonfinite): elements whose result is not finite are recomputed as chains of
// FP32 FMAs over k, in blocks through shared memory. Nothing waits for that pass inside the kernel, so
// its length cannot run out a pipeline wait: one infinite gradient row, which touches every weight of a
// layer, makes a backward pass of 65,536 rows 16 ms instead of 2.8, of 262,145 rows 77 instead of 10.6.
// (As a chain per element in the epilogue it held up the other roles for as long, past their limit.)
//
// Warp roles (one CTA per SM): warp 0 TMA producer, warp 1 tensor memory and MMAs, then groups of
// eight epilogue warps (two per TMEM lane quarter, each holding every other 32-column chunk of its 32
// rows: up to 128 FP32 accumulators a thread). Waits are bounded and drains complete as in mlp_tc.cu.
#include "dfgb_internal.cuh"
#include "pdl.cuh"
#include "planes.cuh"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>

namespace dfgb {
namespace {

constexpr int kGroupWarps = 8;                  // epilogue warps working on one tile
constexpr int kPlanes = 3;
constexpr int kRing = 2;                        // stages per plane
constexpr int kStgBytes = 4096;                 // staging per epilogue warp: 32 x 32 FP32
constexpr int kABytes = BM * kRowBytes;         // one A plane of a stage
constexpr int kBadWords = 64;                   // bits of marked m units, by m unit modulo their number

enum { kSActNone = 0, kSActTanh = 1, kSActTable = 2 };
enum { kSPlain = 0, kSStoreG = 1, kSRowG = 2 };
// Operands read along their other dimension: the reduction index is the matrix's row and the product's
// row or column index runs along memory (MN-major), so the backward pass needs no transposed copy of
// the activations, output gradients or weights. 10,007 rows of 32-1600-800-400-30, forward and backward:
// 7.95 -> 1.01 ms (the FMA GEMM ran a weight gradient on 4 to 91 blocks, 1.5 ms each, after transposes).
constexpr int kTrA = 1, kTrW = 2;

// The two tilings. Wide: 256-column tiles on CTA pairs, one epilogue group of up to 128 accumulators
// a thread. Small: 64-column tiles on single CTAs, two groups.
enum { kWide = 0, kSmall = 1 };

template <int CFG>
struct SCfg {
  static constexpr bool kPair = CFG == kWide;
  static constexpr int kBN = CFG == kWide ? 256 : 64;   // widest tile
  static constexpr int kGroups = CFG == kWide ? 1 : 2;
  static constexpr int kEpiWarps = kGroups * kGroupWarps;
  static constexpr int kThreads = 64 + 32 * kEpiWarps;
  static constexpr int kBRows = kPair ? kBN / 2 : kBN;   // rows of W this CTA holds per stage
  static constexpr int kSlot = kABytes + kBRows * kRowBytes;
  static constexpr int kChunks = kBN / 64;               // 32-column chunks per epilogue warp
  static constexpr int kTmemCols = 2 * kGroups * kBN;    // two accumulators per group
  static constexpr int kSmem = kPlanes * kRing * kSlot + kEpiWarps * kStgBytes + 1024 + 512;
};
static_assert(std::max(SCfg<kWide>::kSmem, SCfg<kSmall>::kSmem) + 4 * kBadWords + 64 <= kSmemLimit, "stages must fit");

struct SplitArgs {
  RowMap rows;
  int N, K;
  int tw;                  // tile width, a multiple of 32
  const float* bias;       // [N], zero padded to 32
  const float4* gtab;
  float* G;                // GELU'(z) written (kSStoreG) or read (kSRowG), [cells x ldg]
  int64_t ldg;
  int ntan;
  int ksplit;
  int64_t split_rows;
  // the planes, for elements recomputed in FP32: entry (r, k) of A at r a_rs + k a_ks, likewise W
  const __nv_bfloat16 *A, *W;
  int64_t a_rs, a_ks, a_plane, w_rs, w_ks, w_plane;
  void* out;               // and the output they go to
  int64_t ldo, o_plane;
  int* err;
  long long budget;
  uint32_t suspend;
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map,
                                                 uint32_t bar_cluster, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar_cluster)
      : "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(src)
               : "memory");
}

// tanh-form GELU, 0.5 z (1 + tanh u) = z / (1 + exp(-2 u)), u = c (z + a z^3): one exponential and
// one division, and no cancellation for negative z. e returns exp(-2 u).
constexpr float kGc = 0.7978845608028654f, kGa = 0.044715f;
constexpr float kG2 = (float)(-2.0 * 1.4426950408889634 * 0.79788456080286535588);
constexpr float kG3 = (float)(-2.0 * 1.4426950408889634 * 0.79788456080286535588 * 0.044715);

__device__ __forceinline__ float gelu_exp(float z) {
  float e;
  const float x = z * fmaf(z * z, kG3, kG2);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x));
  return e;
}

// GELU'(z) = s (1 + 2 c z (1 - s) (1 + 3 a z^2)) with s = 1 / (1 + exp(-2 u)).
__device__ __forceinline__ float gelu_grad_exp(float z, float e) {
  const float s = __fdividef(1.0f, 1.0f + e);
  return s * fmaf(2.0f * kGc * z * (1.0f - s), fmaf(3.0f * kGa * z, z, 1.0f), 1.0f);
}

// Whether any of the 32 values times scale is infinite or NaN: x * 0 is NaN exactly then. One test for
// the chunk, so that the epilogue is straight-line code (a test per element kept the elements' chains
// of exponential and division from overlapping: the 32 -> 1600 layer took
// 697 us on 131,072 rows instead of 361).
__device__ __forceinline__ bool any_nonfinite(const float (&v)[32], float scale) {
  float2 a = make_float2(0.f, 0.f), c = a;
  const float2 z = a, k = make_float2(scale, scale);
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    a = __ffma2_rn(__fmul2_rn(make_float2(v[i], v[i + 1]), k), z, a);
    c = __ffma2_rn(__fmul2_rn(make_float2(v[i + 2], v[i + 3]), k), z, c);
  }
  const float t = (a.x + a.y) + (c.x + c.y);
  return t != t;
}

// Writes 32 FP32 values of this thread's row to the warp's staging buffer (128-byte swizzle) and
// stores the box.
__device__ __forceinline__ void store_f32(const float (&v)[32], const CUtensorMap* map, uint8_t* stg,
                                          int col0, int64_t m0, int lane) {
  if (lane == 0) bulk_wait_read0();
  __syncwarp();
  const int sw = swz<128>(lane);
#pragma unroll
  for (int u = 0; u < 8; ++u)
    *reinterpret_cast<float4*>(stg + lane * 128 + ((u ^ sw) * 16)) =
        make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0) {
    tma_store_3d(map, smem_u32(stg), col0, (int)m0, 0);
    bulk_commit();
  }
}

// One 32-column chunk of the epilogue on this thread's row: bias and activation (or the row-group
// scale), then the three planes, or the FP32 values, through the warp's staging buffer and out by TMA.
// A sum that is not finite leaves a result that is not (the activations and the scale keep it so), or
// one to be looked at because it is large: either marks the m unit mu in `bad`.
template <bool PLANES, int ACT, int MODE>
__device__ __forceinline__ void split_chunk(float (&v)[32], const SplitArgs& g, const CUtensorMap* tmO,
                                            const CUtensorMap* tmG, int64_t M, int64_t mrow, int64_t m0,
                                            int col0, uint32_t mu, uint32_t* bad, uint8_t* stg, int& buf,
                                            int lane) {
  const int64_t row = mrow + lane;          // row of A
  const bool row_ok = row < M;
  if constexpr (MODE == kSRowG) {
    const float4* gr = reinterpret_cast<const float4*>(g.G + ((row_ok ? row : M - 1) / g.ntan) * g.ldg + col0);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float4 x = gr[u];
      v[4 * u] *= x.x; v[4 * u + 1] *= x.y; v[4 * u + 2] *= x.z; v[4 * u + 3] *= x.w;
    }
  } else {
    const float4* b4 = reinterpret_cast<const float4*>(g.bias + col0);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float4 b = __ldg(b4 + u);
      v[4 * u] += b.x; v[4 * u + 1] += b.y; v[4 * u + 2] += b.z; v[4 * u + 3] += b.w;
    }
    if constexpr (MODE == kSStoreG) {
      // GELU'(z) first, while the pre-activations are still there
      float gp[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) gp[i] = gelu_grad_exp(v[i], gelu_exp(v[i]));
      store_f32(gp, tmG, stg, col0, m0, lane);
      if (lane == 0) bulk_wait_read0();   // the planes take either half of the buffer
      __syncwarp();
    }
    if constexpr (ACT == kSActTanh) {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = __fdividef(v[i], 1.0f + gelu_exp(v[i]));
    } else if constexpr (ACT == kSActTable) {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = gelu_from_table(v[i], g.gtab);
    }
  }
  const bool big = any_nonfinite(v, PLANES ? 4.0f : 1.0f);   // not finite, or too large for plain rounding (rare)
  if (big && row_ok) {
    atomicOr(bad + (mu >> 5) % kBadWords, 1u << (mu & 31));
    bad[kBadWords] = 1;
  }
  if constexpr (PLANES) {
    // the planes one after the other through two staging halves of 32 rows x 64 bytes (64-byte
    // swizzle); plane p + 1 is formed from what plane p leaves
    const int sw = swz<64>(lane);
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
      uint32_t w[16];
      if (p == 0 && big) {
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          __nv_bfloat16 a0, a1, a2, c0, c1, c2;
          split_one(v[i], a0, a1, a2);
          split_one(v[i + 1], c0, c1, c2);
          const __nv_bfloat162 h = __halves2bfloat162(a0, c0);
          memcpy(&w[i / 2], &h, 4);
          v[i] = isfinite(v[i]) ? v[i] - __bfloat162float(a0) : 0.0f;
          v[i + 1] = isfinite(v[i + 1]) ? v[i + 1] - __bfloat162float(c0) : 0.0f;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(v[i], v[i + 1]);
          memcpy(&w[i / 2], &h, 4);
          if (p < kPlanes - 1) {
            const float2 f = __bfloat1622float2(h);
            const float2 r = __fadd2_rn(make_float2(v[i], v[i + 1]), make_float2(-f.x, -f.y));
            v[i] = r.x;
            v[i + 1] = r.y;
          }
        }
      }
      uint8_t* sp = stg + buf * 2048;
      if (lane == 0) bulk_wait_read1();   // the store before last has read this half
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 4; ++u)
        *reinterpret_cast<uint4*>(sp + lane * 64 + ((u ^ sw) * 16)) =
            make_uint4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        tma_store_3d(tmO, smem_u32(sp), col0, (int)m0, p);
        bulk_commit();
      }
      buf ^= 1;
    }
  } else {
    store_f32(v, tmO, stg, col0, m0, lane);
  }
}

// Recomputes the non-finite results of the 128 x 32 outputs at rows m0 (of A; o0 of the output) and
// columns col0 as chains of FP32 FMAs over k in [k0, k1), ascending, and stores those elements. All
// threads of the block; the first 256 hold 4 x 4 elements each. Blocks of 32 k of both operands, summed
// from their planes, go through shared memory; the loop ends once every such element is NaN, which is
// the first block for the rows of a cell that is not finite.
constexpr int kRedoK = 32;
constexpr int kRedoA = BM + 4, kRedoW = 32 + 4;   // pitches
template <bool PLANES, int ACT, int MODE>
__device__ void redo_nonfinite(const SplitArgs& g, float* sm, int64_t M, int64_t m0, int64_t o0,
                                            int col0, int k0, int k1) {
  const int t = threadIdx.x, ty = t >> 3, tx = t & 7;
  unsigned todo = 0;   // bit 4 i + j: element (4 ty + i, 4 tx + j)
  if (t < 256) {
#pragma unroll 1
    for (int e = 0; e < 16; ++e) {
      const int64_t r = m0 + 4 * ty + (e >> 2);
      const int c = col0 + 4 * tx + (e & 3);
      if (r >= M || c >= g.N) continue;
      const int64_t o = (r - m0 + o0) * g.ldo + c;
      const float v = PLANES ? __bfloat162float(((const __nv_bfloat16*)g.out)[o]) : ((const float*)g.out)[o];
      if (!isfinite(v)) todo |= 1u << e;
    }
  }
  if (!__syncthreads_or(todo != 0)) return;
  float *sA = sm, *sW = sm + kRedoK * kRedoA;
  float acc[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e] = 0.0f;
  auto value = [](const __nv_bfloat16* p, int64_t plane) {
    return __bfloat162float(__ldg(p)) + (__bfloat162float(__ldg(p + plane)) + __bfloat162float(__ldg(p + 2 * plane)));
  };
  // the operand's contiguous index runs along the threads
  const bool ka = g.a_ks == 1, kw = g.w_ks == 1;
  for (int kb = k0; kb < k1; kb += kRedoK) {
#pragma unroll 1
    for (int i = t; i < BM * kRedoK; i += blockDim.x) {
      const int r = ka ? i / kRedoK : i % BM, k = ka ? i % kRedoK : i / BM;
      const bool in = m0 + r < M && kb + k < k1;
      sA[k * kRedoA + r] = in ? value(g.A + (m0 + r) * g.a_rs + (kb + k) * g.a_ks, g.a_plane) : 0.0f;
    }
#pragma unroll 1
    for (int i = t; i < 32 * kRedoK; i += blockDim.x) {
      const int c = kw ? i / kRedoK : i % 32, k = kw ? i % kRedoK : i / 32;
      const bool in = col0 + c < g.N && kb + k < k1;
      sW[k * kRedoW + c] = in ? value(g.W + (col0 + c) * g.w_rs + (kb + k) * g.w_ks, g.w_plane) : 0.0f;
    }
    __syncthreads();
    bool more = false;
    if (todo) {
      const int nk = min(kRedoK, k1 - kb);
#pragma unroll 1
      for (int k = 0; k < nk; ++k) {
        const float4 a = *reinterpret_cast<const float4*>(sA + k * kRedoA + 4 * ty);
        const float4 w = *reinterpret_cast<const float4*>(sW + k * kRedoW + 4 * tx);
        const float av[4] = {a.x, a.y, a.z, a.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = fmaf(av[e >> 2], wv[e & 3], acc[e]);
      }
#pragma unroll
      for (int e = 0; e < 16; ++e) more = more || (((todo >> e) & 1u) && acc[e] == acc[e]);
    }
    if (!__syncthreads_or(more)) break;
  }
  // the sums go through this thread's slots of shared memory, so that the stores are one loop body (the
  // code of all sixteen made every launch 0.5 us longer, used or not)
  float* mine = sW + kRedoK * kRedoW + t;
  if (!todo) return;
#pragma unroll
  for (int e = 0; e < 16; ++e) mine[256 * e] = acc[e];
#pragma unroll 1
  for (int e = 0; e < 16; ++e) {
    if (!((todo >> e) & 1u)) continue;
    const int64_t r = m0 + 4 * ty + (e >> 2), ro = r - m0 + o0;
    const int c = col0 + 4 * tx + (e & 3);
    float v = mine[256 * e];
    if constexpr (MODE == kSRowG) {
      v *= g.G[(r / g.ntan) * g.ldg + c];
    } else {
      v += g.bias[c];
      if constexpr (MODE == kSStoreG) g.G[ro * g.ldg + c] = gelu_grad_exp(v, gelu_exp(v));
      if constexpr (ACT == kSActTanh) v = __fdividef(v, 1.0f + gelu_exp(v));
      else if constexpr (ACT == kSActTable) v = gelu_from_table(v, g.gtab);
    }
    if constexpr (PLANES) {
      __nv_bfloat16* o = (__nv_bfloat16*)g.out + ro * g.ldo + c;
      split_one(v, o[0], o[g.o_plane], o[2 * g.o_plane]);
    } else {
      ((float*)g.out)[ro * g.ldo + c] = v;
    }
  }
}

// redo_nonfinite over this CTA's tiles whose m unit is marked in `bad`. Out of line, with everything formed anew: what it needs
// must not take registers from the epilogue.
template <int CFG, bool PLANES, int ACT, int MODE>
__device__ __noinline__ void redo_tiles(const SplitArgs& g, const WalkStep& step, const uint32_t* bad) {
  constexpr bool PAIR = SCfg<CFG>::kPair;
  extern __shared__ uint8_t smem_raw[];
  float* sm = (float*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  asm volatile("fence.proxy.async;" ::: "memory");
  const int64_t M = valid_rows(g.rows), tiles_m = (M + BM - 1) / BM;
  const uint32_t units_m = (uint32_t)(PAIR ? (tiles_m + 1) / 2 : tiles_m);
  const int tiles_n = (g.N + g.tw - 1) / g.tw;
  const int kbs = ((g.K + 63) / 64 + g.ksplit - 1) / g.ksplit;
  for (ItemWalk w(PAIR ? blockIdx.x >> 1 : blockIdx.x, units_m, tiles_n); w.split < g.ksplit;
       w.next(step, units_m, tiles_n)) {
    if (!((bad[(w.mu >> 5) % kBadWords] >> (w.mu & 31)) & 1u)) continue;
    const int k0 = w.split * kbs * 64, k1 = min(g.K, k0 + kbs * 64), n0 = w.nt(tiles_n) * g.tw;
    const int64_t m0 = (PAIR ? w.mu * 2 + cluster_rank() : (int64_t)w.mu) * BM;
    for (int c = n0; c < n0 + g.tw && c < g.N && m0 < M; c += 32) {
      redo_nonfinite<PLANES, ACT, MODE>(g, sm, M, m0, m0 + w.split * g.split_rows, c, k0, k1);
      __syncthreads();
    }
  }
}

template <int CFG, bool PLANES, int ACT, int MODE, int TR>
__global__ void __launch_bounds__(SCfg<CFG>::kThreads, 1) split_gemm_kernel(
    const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
    const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmG,
    const __grid_constant__ SplitArgs g) {
  using C = SCfg<CFG>;
  constexpr bool PAIR = C::kPair;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sOut = smem + kPlanes * kRing * C::kSlot;
  uint64_t* bars = (uint64_t*)(sOut + C::kEpiWarps * kStgBytes);
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  __shared__ uint32_t bad_sh[kBadWords + 1];   // m units with sums that are not finite; whether any is
  __shared__ WalkStep walk_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // stage (plane p, slot s) = p * kRing + s
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kPlanes * kRing;
  // accumulator b of group gr: 2 gr + b
  const uint32_t tfull0 = empty0 + 8 * kPlanes * kRing, tempty0 = tfull0 + 16 * C::kGroups;
  const uint32_t drain = tempty0 + 16 * C::kGroups;
  const uint32_t rank = PAIR ? cluster_rank() : 0;
  const int tiles_n = (g.N + g.tw - 1) / g.tw;

  if (threadIdx.x == 0) {
    abort_sh = 0;
    const uint32_t step = PAIR ? (gridDim.x >> 1) : gridDim.x, tn = (uint32_t)tiles_n;
    walk_sh.q = step / tn;
    walk_sh.r = (int)(step - walk_sh.q * tn);
    walk_sh.rot = (int)(walk_sh.q % tn);
    for (int s = 0; s < kPlanes * kRing; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2 * C::kGroups; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, PAIR ? 2 * kGroupWarps : kGroupWarps);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  for (int i = threadIdx.x; i <= kBadWords; i += C::kThreads) bad_sh[i] = 0;
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(&tmem_base_sh)), "r"((uint32_t)C::kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(&tmem_base_sh)), "r"((uint32_t)C::kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  volatile int* abort = &abort_sh;
  pdl_begin();

  const int64_t M = valid_rows(g.rows);
  const int64_t tiles_m = (M + BM - 1) / BM;
  const int64_t units_m = PAIR ? (tiles_m + 1) / 2 : tiles_m;
  const uint32_t units_m32 = (uint32_t)units_m;
  const int kblocks = (g.K + 63) / 64;
  const int kbs = (kblocks + g.ksplit - 1) / g.ksplit;
  const uint32_t t_first = PAIR ? (blockIdx.x >> 1) : blockIdx.x;
  auto tile_m0 = [&](int64_t mu) -> int64_t { return PAIR ? (mu * 2 + rank) * BM : mu * BM; };
  // MMA width of n tile nt: the columns left, rounded up to the N granule of 16
  auto tile_w = [&](int nt) -> int { return min(g.tw, (g.N - nt * g.tw + 15) & ~15); };

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmW) : "memory");
    const uint32_t bytes = kABytes + ((TR & kTrW) ? (uint32_t)C::kBRows * kRowBytes
                                                  : (uint32_t)(PAIR ? g.tw / 2 : g.tw) * kRowBytes);
    uint32_t it = 0, issued[kPlanes] = {0, 0, 0};
    bool ok = true;
    for (ItemWalk w(t_first, units_m32, tiles_n); w.split < g.ksplit && ok;
         w.next(walk_sh, units_m32, tiles_n)) {
      const int kb0 = w.split * kbs, kb1 = min(kblocks, kb0 + kbs);
      const int m0 = (int)tile_m0(w.mu);
      const int nt = w.nt(tiles_n);
      const int n0 = nt * g.tw + (PAIR ? (int)rank * (tile_w(nt) >> 1) : 0);
      for (int kb = kb0; kb < kb1 && ok; ++kb, ++it) {
        const uint32_t ph = (it / kRing) & 1;
        // in the order in which the MMAs free the stages
#pragma unroll
        for (int p = kPlanes - 1; p >= 0; --p) {
          const int s = p * kRing + it % kRing;
          if (!mbar_wait(empty0 + 8 * s, ph ^ 1, abort, g.err, g.budget, g.suspend)) {
            ok = false;
            break;
          }
          const uint32_t dA = smem_u32(smem + s * C::kSlot), dB = dA + kABytes;
          const uint32_t bar = PAIR ? map_shared(full0 + 8 * s, 0) : full0 + 8 * s;
          if (!PAIR || rank == 0) mbar_arrive_expect_tx(full0 + 8 * s, PAIR ? 2 * bytes : bytes);
          auto load = [&](uint32_t dst, const CUtensorMap* map, int x, int y) {
            if constexpr (PAIR) tma_load_3d_pair(dst, map, bar, x, y, p);
            else tma_load_3d(dst, map, bar, x, y, p);
          };
          // an MN-major operand comes as boxes of 64 of its columns x the 64 rows of the k-block
          if constexpr (TR & kTrA) {
#pragma unroll
            for (int i = 0; i < BM / 64; ++i) load(dA + i * kMnBox, &tmA, m0 + 64 * i, kb * 64);
          } else {
            load(dA, &tmA, kb * 64, m0);
          }
          if constexpr (TR & kTrW) {
#pragma unroll
            for (int i = 0; i < C::kBRows / 64; ++i) load(dB + i * kMnBox, &tmW, n0 + 64 * i, kb * 64);
          } else {
            load(dB, &tmW, kb * 64, n0);
          }
          ++issued[p];
        }
      }
    }
    // Drain: the last loads of every stage land before the CTA exits; in a pair also the commits
    // that free this CTA's stages (as in tc_gemm_kernel).
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
      const uint32_t n = issued[p], first = n > (uint32_t)kRing ? n - kRing : 0;
      for (uint32_t j = first; j < n; ++j) {
        const uint32_t s = p * kRing + j % kRing, ph = (j / kRing) & 1;
        if (!PAIR || rank == 0) {
          const long long t0 = clock64();
          while (!mbar_try(full0 + 8 * s, ph) && clock64() - t0 < kWaitBudget) {
          }
        }
        if constexpr (PAIR) {
          const long long t0 = clock64();
          while (!mbar_try_cluster(empty0 + 8 * s, ph) && clock64() - t0 < kWaitBudget) {
          }
        }
      }
    }
  } else if (warp == 1 && lane == 0 && rank == 0) {
    // ---------------- MMA issuer ----------------
    constexpr uint32_t id0 = idesc<false, 0, PAIR ? 2 * BM : BM>() |
                             ((TR & kTrA) ? kIdescMnA : 0u) | ((TR & kTrW) ? kIdescMnB : 0u);
    // descriptor step of one instruction's K = 16: 32 bytes of a K-major row, or 16 rows of 128 bytes
    constexpr uint32_t stepA = (TR & kTrA) ? 128 : 2, stepW = (TR & kTrW) ? 128 : 2;
    uint32_t it = 0, done0 = 0, done1 = 0;   // k-blocks issued: in all, and by group
    int gr = 0;
    bool ok = true;
    for (ItemWalk w(t_first, units_m32, tiles_n); w.split < g.ksplit && ok;
         w.next(walk_sh, units_m32, tiles_n), gr ^= C::kGroups - 1) {
      const int kb0 = w.split * kbs, kb1 = min(kblocks, kb0 + kbs);
      const uint32_t id = id0 | ((uint32_t)(tile_w(w.nt(tiles_n)) >> 3) << 17);
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        const uint32_t n = gr ? done1++ : done0++;
        const int a = 2 * gr + (n & 1), r = it % kRing;
        const uint32_t ph = (it / kRing) & 1;
        if (PAIR ? !mbar_wait_cluster(tempty0 + 8 * a, ((n >> 1) & 1) ^ 1, abort, g.err, g.budget, g.suspend)
                 : !mbar_wait(tempty0 + 8 * a, ((n >> 1) & 1) ^ 1, abort, g.err, g.budget, g.suspend)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dt = tmem + a * C::kBN;
        const int steps = min(4, (g.K - kb * 64 + 15) >> 4);   // K = 16 per instruction
        uint64_t da[kPlanes], db[kPlanes];
#pragma unroll
        for (int p = 0; p < kPlanes; ++p) {
          const uint32_t sa = smem_u32(smem + (p * kRing + r) * C::kSlot);
          da[p] = (TR & kTrA) ? desc_mn128(sa) : desc_sw128(sa);
          db[p] = (TR & kTrW) ? desc_mn128(sa + kABytes) : desc_sw128(sa + kABytes);
        }
        auto full = [&](int p) {
          return mbar_wait(full0 + 8 * (p * kRing + r), ph, abort, g.err, g.budget, g.suspend);
        };
        auto mma = [&](int i, int j, bool first) {
          for (int kk = 0; kk < steps; ++kk) {
            if constexpr (PAIR)
              mma_issue_pair<false>(dt, da[i] + stepA * kk, db[j] + stepW * kk, id, (first && kk == 0) ? 0u : 1u);
            else
              mma_issue<false>(dt, da[i] + stepA * kk, db[j] + stepW * kk, id, (first && kk == 0) ? 0u : 1u);
          }
        };
        auto free_plane = [&](int p) {
          if constexpr (PAIR) mma_commit_pair_both(empty0 + 8 * (p * kRing + r));
          else mma_commit(empty0 + 8 * (p * kRing + r));
        };
        if (!full(2) || !full(0)) {
          ok = false;
          break;
        }
        tc_fence_after();
        mma(2, 0, true);
        mma(0, 2, false);
        free_plane(2);
        if (!full(1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        mma(1, 1, false);
        mma(1, 0, false);
        mma(0, 1, false);
        free_plane(1);
        mma(0, 0, false);
        free_plane(0);
        if constexpr (PAIR) mma_commit_pair_both(tfull0 + 8 * a);
        else mma_commit(tfull0 + 8 * a);
      }
    }
    if constexpr (PAIR) mma_commit_pair_local(drain);
    else mma_commit(drain);
    const long long t0 = clock64();
    while (!mbar_try(drain, 0) && clock64() - t0 < kWaitBudget) {
    }
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int q = warp & 3, slot = ((warp - 2) >> 2) & 1, group = (warp - 2) / kGroupWarps;
    int buf = 0, gr = 0;
    uint8_t* stg = sOut + (warp - 2) * kStgBytes;
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmO) : "memory");
    uint32_t it = 0;
    bool ok = true;
    for (ItemWalk w(t_first, units_m32, tiles_n); w.split < g.ksplit && ok;
         w.next(walk_sh, units_m32, tiles_n), gr ^= C::kGroups - 1) {
      if (gr != group) continue;   // the other group's tile
      const int kb0 = w.split * kbs, kb1 = min(kblocks, kb0 + kbs);
      const int nt = w.nt(tiles_n);
      const int width = tile_w(nt);
      float acc[C::kChunks][32];
#pragma unroll
      for (int c = 0; c < C::kChunks; ++c)
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[c][i] = 0.0f;
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        const int a = 2 * group + (it & 1);
        if (!mbar_wait(tfull0 + 8 * a, (it >> 1) & 1, abort, g.err, g.budget, g.suspend)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + a * C::kBN;
#pragma unroll
        for (int c = 0; c < C::kChunks; ++c) {
          const int c0 = 32 * (slot + 2 * c);
          if (c0 < width) {
            uint32_t r[32];
            tmem_ld32(tbase + c0, r);
            tmem_wait(r);
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
              const float2 s = __fadd2_rn(make_float2(acc[c][i], acc[c][i + 1]),
                                          make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])));
              acc[c][i] = s.x;
              acc[c][i + 1] = s.y;
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR && rank != 0) mbar_arrive_cluster(map_shared(tempty0 + 8 * a, 0));
          else mbar_arrive(tempty0 + 8 * a);
        }
      }
      if (!ok) break;
      const int64_t mt = tile_m0(w.mu);
      if (PAIR && mt >= M) continue;   // the odd CTA of a pair whose tile lies past the rows
      const int64_t mrow = mt + q * 32;
      const int64_t m0 = mrow + w.split * g.split_rows;
#pragma unroll
      for (int c = 0; c < C::kChunks; ++c) {
        const int col0 = nt * g.tw + 32 * (slot + 2 * c);
        if (32 * (slot + 2 * c) < width && col0 < g.N)
          split_chunk<PLANES, ACT, MODE>(acc[c], g, &tmO, &tmG, M, mrow, m0, col0, w.mu, bad_sh, stg, buf, lane);
      }
    }
    if (lane == 0) bulk_wait_all();
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();
  tc_fence_after();
  if (warp == 1) {
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"((uint32_t)C::kTmemCols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"((uint32_t)C::kTmemCols) : "memory");
  }
  // the stores above have completed, and so have all copies into and MMA reads of shared memory
  if (bad_sh[kBadWords] && !abort_sh) redo_tiles<CFG, PLANES, ACT, MODE>(g, walk_sh, bad_sh);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// A 3-D map [planes][rows][cols] of `elem` bytes with box {box_c, box_r, 1}.
bool encode_3d(CUtensorMap* m, const void* base, int elem, int64_t cols, int64_t rows, int64_t planes,
               int64_t ld, int64_t plane, uint32_t box_c, uint32_t box_r, CUtensorMapSwizzle sw,
               char* err, size_t errlen) {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                            &q) == cudaSuccess && q == cudaDriverEntryPointSuccess
               ? (EncodeTiledFn)p : nullptr;
  }();
  if (!fn) {
    snprintf(err, errlen, "cuTensorMapEncodeTiled is not available from the driver");
    return false;
  }
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * elem, (cuuint64_t)plane * elem};
  if (((uintptr_t)base & 15) || (strides[0] & 15) || (strides[1] & 15)) {
    snprintf(err, errlen, "tensor map: base or pitch not 16-byte aligned");
    return false;
  }
  const cuuint32_t box[3] = {box_c, box_r, 1}, es[3] = {1, 1, 1};
  const CUresult r = fn(m, elem == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                        3, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                        box_r == 32 && box_c == 32 ? CU_TENSOR_MAP_L2_PROMOTION_NONE
                                                   : CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    snprintf(err, errlen, "cuTensorMapEncodeTiled (planes) failed (%d)", (int)r);
    return false;
  }
  return true;
}

// The kernel's dynamic shared memory, once per device; for CTA pairs also how many fit at once.
template <int CFG, bool PLANES, int ACT, int MODE, int TR>
cudaError_t split_attr(int* max_clusters) {
  using C = SCfg<CFG>;
  static bool done[64] = {false};
  static int clusters[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!done[dev]) {
    auto kern = split_gemm_kernel<CFG, PLANES, ACT, MODE, TR>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem);
    if (e != cudaSuccess) return e;
    if (C::kPair) {
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 2;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(2, 1, 1);
      cfg.blockDim = dim3(C::kThreads, 1, 1);
      cfg.dynamicSmemBytes = C::kSmem;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      e = cudaOccupancyMaxActiveClusters(&n, (const void*)kern, &cfg);
      if (e != cudaSuccess) return e;
      if (n <= 0) return cudaErrorInvalidConfiguration;
      clusters[dev] = n;
    }
    done[dev] = true;
  }
  if (max_clusters) *max_clusters = clusters[dev];
  return cudaSuccess;
}

template <int CFG, bool PLANES, int ACT, int MODE, int TR = 0>
cudaError_t split_go(const SplitLayer& L, SplitArgs a, int num_sms, cudaStream_t st) {
  using C = SCfg<CFG>;
  auto kern = split_gemm_kernel<CFG, PLANES, ACT, MODE, TR>;
  int max_clusters = 0;
  cudaError_t e = split_attr<CFG, PLANES, ACT, MODE, TR>(&max_clusters);
  if (e != cudaSuccess || num_sms <= 0) return e;   // num_sms 0: attribute set-up only
  a.tw = L.tw[CFG];
  const int64_t per = C::kPair ? 2 * BM : BM;
  const int64_t items = (a.rows.nmax + per - 1) / per * ((a.N + a.tw - 1) / a.tw) * a.ksplit;
  if (items > 0x7FFFFFFF) return cudaErrorInvalidValue;
  if constexpr (C::kPair) {
    const int64_t nc = std::max<int64_t>(1, std::min<int64_t>(items, std::min(max_clusters, num_sms / 2)));
    return pdl_launch(kern, (unsigned)(2 * nc), C::kThreads, C::kSmem, st, 2, L.tmA, L.tmW[CFG], L.tmO, L.tmG, a);
  } else {
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(items, num_sms));
    return pdl_launch(kern, grid, C::kThreads, C::kSmem, st, 1, L.tmA, L.tmW[CFG], L.tmO, L.tmG, a);
  }
}

template <int CFG>
cudaError_t split_pick(const SplitLayer& L, const SplitArgs& a, int num_sms, cudaStream_t st) {
  if (L.mode == kSRowG) {
    if (!L.planes || L.gelu || (L.tr & kTrA)) return cudaErrorInvalidValue;
    return L.tr ? split_go<CFG, true, kSActNone, kSRowG, kTrW>(L, a, num_sms, st)
                : split_go<CFG, true, kSActNone, kSRowG>(L, a, num_sms, st);
  }
  if (!L.planes) {
    if (L.gelu || L.tr == kTrA) return cudaErrorInvalidValue;
    return L.tr == 0      ? split_go<CFG, false, kSActNone, kSPlain>(L, a, num_sms, st)
           : L.tr == kTrW ? split_go<CFG, false, kSActNone, kSPlain, kTrW>(L, a, num_sms, st)
                          : split_go<CFG, false, kSActNone, kSPlain, kTrA | kTrW>(L, a, num_sms, st);
  }
  if (L.tr) return cudaErrorInvalidValue;
  if (L.mode == kSStoreG) {
    if (!L.planes || !L.gelu || L.gtab) return cudaErrorInvalidValue;
    return split_go<CFG, true, kSActTanh, kSStoreG>(L, a, num_sms, st);
  }
  if (!L.gelu) return cudaErrorInvalidValue;
  return L.gtab ? split_go<CFG, true, kSActTable, kSPlain>(L, a, num_sms, st)
                : split_go<CFG, true, kSActTanh, kSPlain>(L, a, num_sms, st);
}

// planes [3][.][ldo] of the FP32 matrix in [rows x ldi], columns cols..ldo-1 zero; eight columns
// (16 bytes of each plane) per thread.
__global__ void split_rows_kernel(RowMap rm, int cols, const float* __restrict__ in, int64_t ldi,
                                  __nv_bfloat16* __restrict__ out, int64_t ldo, int64_t plane) {
  pdl_begin();
  const int64_t rows = valid_rows(rm);
  const int groups = (int)(ldo >> 3);
  const int64_t total = rows * groups;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / groups;
    const int c0 = (int)(t - r * groups) * 8;
    __align__(16) __nv_bfloat16 h[kPlanes][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float v = c0 + i < cols ? in[r * ldi + c0 + i] : 0.0f;
      split_one(v, h[0][i], h[1][i], h[2][i]);
    }
#pragma unroll
    for (int p = 0; p < kPlanes; ++p)
      *reinterpret_cast<uint4*>(out + p * plane + r * ldo + c0) = *reinterpret_cast<const uint4*>(h[p]);
  }
}

}  // namespace

// Tile widths: columns cut into the fewest tiles of at most the tiling's width, all equal up to the
// rounding to whole 32-column chunks, so that no tile is much narrower than the rest.
bool split_encode(SplitLayer& L, int64_t a_rows, void* out, int64_t o_rows, int64_t ldo, float* G,
                  char* err, size_t errlen) {
  const CUtensorMapSwizzle s128 = CU_TENSOR_MAP_SWIZZLE_128B, s64 = CU_TENSOR_MAP_SWIZZLE_64B;
  static const int most[2] = {SCfg<kWide>::kBN, SCfg<kSmall>::kBN};
  L.g = G;
  L.out = out;
  L.ldo = ldo;
  if (L.tr & kTrA) {   // columns 0..M-1 of the L.K rows; rows past them read as zero
    if (!encode_3d(&L.tmA, L.A, 2, L.M, L.K, kPlanes, L.lda, L.a_plane, 64, 64, s128, err, errlen)) return false;
  } else if (!encode_3d(&L.tmA, L.A, 2, L.K, a_rows, kPlanes, L.lda, L.a_plane, 64, BM, s128, err, errlen)) {
    return false;
  }
  for (int c = 0; c < 2; ++c) {
    const int nt = (L.N + most[c] - 1) / most[c];
    L.tw[c] = ((L.N + nt - 1) / nt + 31) / 32 * 32;
    const bool ok = (L.tr & kTrW)
        ? encode_3d(&L.tmW[c], L.W, 2, L.N, L.K, kPlanes, L.ldw, L.w_plane, 64, 64, s128, err, errlen)
        : encode_3d(&L.tmW[c], L.W, 2, L.K, L.N, kPlanes, L.ldw, L.w_plane, 64,
                    (uint32_t)(c == kSmall ? L.tw[c] : L.tw[c] / 2), s128, err, errlen);
    if (!ok) return false;
  }
  if (L.planes ? !encode_3d(&L.tmO, out, 2, L.N, o_rows, kPlanes, ldo, L.o_plane, 32, 32, s64, err, errlen)
               : !encode_3d(&L.tmO, out, 4, L.N, o_rows, 1, ldo, o_rows * ldo, 32, 32, s128, err, errlen))
    return false;
  L.tmG = L.tmO;
  if (L.mode == kSStoreG)
    return encode_3d(&L.tmG, G, 4, L.N, o_rows, 1, L.ldg, o_rows * L.ldg, 32, 32, s128, err, errlen);
  return true;
}

cudaError_t prepare_split(const SplitLayer& L) {
  SplitArgs a{};
  const cudaError_t e = split_pick<kWide>(L, a, 0, nullptr);
  return e == cudaSuccess ? split_pick<kSmall>(L, a, 0, nullptr) : e;
}

cudaError_t launch_split(const SplitLayer& L, const RowMap& rows, int num_sms, int* err, cudaStream_t st) {
  if (rows.nmax <= 0) return cudaSuccess;
  SplitArgs a;
  a.rows = rows;
  a.N = L.N;
  a.K = L.K;
  a.tw = 0;
  a.bias = L.bias;
  a.gtab = L.gtab;
  a.G = L.g;
  a.ldg = L.ldg;
  a.ntan = L.ntan > 0 ? L.ntan : 1;
  a.ksplit = L.ksplit > 0 ? L.ksplit : 1;
  a.split_rows = L.split_rows;
  a.A = (const __nv_bfloat16*)L.A;
  a.W = (const __nv_bfloat16*)L.W;
  a.a_rs = (L.tr & kTrA) ? 1 : L.lda;
  a.a_ks = (L.tr & kTrA) ? L.lda : 1;
  a.a_plane = L.a_plane;
  a.w_rs = (L.tr & kTrW) ? 1 : L.ldw;
  a.w_ks = (L.tr & kTrW) ? L.ldw : 1;
  a.w_plane = L.w_plane;
  a.out = L.out;
  a.ldo = L.ldo;
  a.o_plane = L.o_plane;
  a.err = err;
  a.budget = kWaitBudget;
  a.suspend = kSuspendNs;
  // The cheaper tiling by the time of its waves of tiles. Both take about 1.5 us per k-block of a
  // tile (the wide one for its 24 MMAs of 256 columns, the small one for the latency of its loads); a
  // wide tile pays about 8 us more for its epilogue, which nothing overlaps (fits to the times above).
  const int64_t kb = ((L.K + 63) / 64 + a.ksplit - 1) / a.ksplit;
  auto waves = [&](int cfg, int64_t rows_per, int64_t slots) {
    const int64_t items = (rows.nmax + rows_per - 1) / rows_per * ((L.N + L.tw[cfg] - 1) / L.tw[cfg]) * a.ksplit;
    return (items + slots - 1) / slots;
  };
  const int64_t wide = waves(kWide, 2 * BM, std::max(1, num_sms / 2)) * (3 * kb + 16);
  const int64_t small = waves(kSmall, BM, num_sms) * 3 * kb;
  return wide < small ? split_pick<kWide>(L, a, num_sms, st) : split_pick<kSmall>(L, a, num_sms, st);
}

cudaError_t launch_split_rows(const RowMap& rows, int cols, const float* in, int64_t ldi, void* out,
                              int64_t ldo, int64_t plane, int num_sms, cudaStream_t st) {
  if (rows.nmax <= 0) return cudaSuccess;
  if (ldo & 7) return cudaErrorInvalidValue;
  const int64_t total = rows.nmax * (ldo >> 3);
  const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, (int64_t)num_sms * 16));
  return pdl_launch(split_rows_kernel, g, 256, 0, st, 1, rows, cols, in, ldi, (__nv_bfloat16*)out, ldo, plane);
}

}  // namespace dfgb
