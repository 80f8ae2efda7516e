// Equation-of-state kernels of the reaction step: a1-a5 (eos_pre), a8-a10 (eos_post) and
// the real-fluid property evaluation. One thread per cell; species-major (SoA) field reads
// are coalesced across the threads of a warp.
//
// Peng-Robinson (Sec. 2 names the EoS; equations from Peng & Robinson 1976):
//   sqrt(a_k(T)) = sqrt(a_c,k) [1 + kappa_k (1 - sqrt(T / Tc_k))] = s_k - r_k sqrt(T),
//   a_m = sum_ij X_i X_j sqrt(a_i a_j) (1 - k_ij) = A0 - 2 A1 sqrt(T) + A2 T
// with three quadratic forms A0, A1, A2 of the composition, computed once per composition,
// so each Newton iteration of the T-from-h solve is O(1) in the species count.
//
// Precision plan (FP64 runs at 1/64 of the FP32 rate on this GPU, so FP64 instructions --
// arithmetic, compares and conversions alike -- are the scarce resource):
//   * every sum over species and species pairs (W_mix, b_m, the three forms, the mixture
//     NASA-7 coefficients) is accumulated in double-float on the FP32 pipes (~1e-14), from a
//     per-thread shared-memory column of the mass fractions in double-float;
//   * Y' = Y (1 + delta), its sum and the renormalisation are double-float too; delta itself
//     is FP32 (it only scales Y' - Y);
//   * finiteness and threshold tests look at the bits of the FP64 values, and the FP32 <-> FP64
//     conversions are integer operations (ddfloat.cuh);
//   * the state -- cubic, root, departure enthalpy, c_p, the Newton solve for T -- is double-float in
//     the step and Jacobian kernels; the property kernel takes the cubic's coefficients, the last
//     step of its root and the density in FP64, the transport kernel its whole state; reciprocals and
//     square roots start from FP32 values and take one or two Newton refinements;
//   * the Box-Cox features that feed the network are FP32 (they are quantised anyway).
#include "dfgb_internal.cuh"
#include "ddfloat.cuh"
#include "pdl.cuh"

#include <algorithm>
#include <atomic>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

namespace dfgb {
namespace {

constexpr double kSQ2 = 1.41421356237309504880;
constexpr double kInvR = 1.0 / kR;
// The step's EoS kernels run blocks of 256 threads, three per SM (80 registers): the constant
// tables in shared memory are then shared by more threads than with five blocks of 128, and the
// SM holds 24 warps instead of 20 (eos_pre 0.71 -> 0.66 ms, eos_post 0.69 -> 0.66 ms on the
// 2^20-cell step).
constexpr int kThreads = 256;
constexpr int kPreBlocks = 3;    // resident blocks per SM the register budget is sized for
constexpr int kPostBlocks = 3;
// Launches that one wave of smaller blocks holds run blocks of 64 threads without a register cap instead:
// four times the blocks, so that no SM is idle while another has eight warps, and room for the compiler
// to overlap a thread's chains (rule in small_blocks).
constexpr int kSmallThreads = 64;
constexpr int kPropThreads = 128;  // the transport and Jacobian state kernels
constexpr int kPropBlocks = 5;
constexpr int kCellNotConverged = 1;
constexpr int kCellNoRoot = 2;
constexpr int kCellNonfinite = 4;
constexpr double kTLo = 50.0, kTHi = 5000.0;

struct Mixture {
  double inv;        // sum_k Y_k / W_k = 1 / W_mix
  double e[6];       // ideal-gas mass-specific enthalpy: h_ig(T) = sum_j e_j T^j, J/kg
  double A0, A1, A2; // a_m(T) = A0 - 2 A1 sqrt(T) + A2 T
  double bm;
  double kb;         // 1 / (2 sqrt2 b_m)
};

// The same coefficients in double-float, for the kernels that evaluate the state in double-float.
struct MixDF {
  f2 inv;
  f2 e[6];
  f2 A0, A1, A2;
  f2 bm;
  f2 kb;
};

// The raw double-float sums of one composition (before the 1/W_mix scalings).
struct MixSums {
  f2 inv, bs, e[6], F0, F1, F2;
};

struct SharedConsts {
  const float4* spc4;  // [5 n] EosParams::spc4
  const float4* K4;    // EosParams::K4
  const float4* qabs;  // EosParams::qabs
  const float2* kf2;   // pairs j > i: (k_ij s_j / W_j, k_ij r_j / W_j) in FP32 (T-from-h only)
  const double* lnt;   // [256] log table (ln c_j, then 1 / c_j); FP64 kernels only
  const f2* lt2;       // the same table in double-float, in the same words; DF kernels only
  const float* normf;  // normalisation constants [2 K0 + 2 n] in FP32
  const float* smax;   // [kSpcStride] EosParams::spcmax (T-from-h kernel only)
};

// 8-byte words of shared memory the constants take (an even number: 16-byte columns follow): the log
// table, then the species, pair and bound tables, then the normalisation in FP32.
__host__ __device__ inline int consts_words(const EosParams& P) {
  return (256 + 10 * P.n + 4 * pair_blocks(P.n) + 6 * (P.n + (P.n & 1)) + (P.K0 + P.n) + 1) & ~1;
}

// Copies `floats` floats (a multiple of four, both 16-byte aligned).
__device__ __forceinline__ void copy_table(float* dst, const float* src, int floats) {
  for (int i = threadIdx.x; i < floats / 4; i += blockDim.x)
    reinterpret_cast<float4*>(dst)[i] = __ldg(reinterpret_cast<const float4*>(src) + i);
}

// DF: the first 256 words hold the double-float log table (the kernels that evaluate the state
// in double-float) instead of the FP64 one.
template <bool DF = false>
__device__ SharedConsts load_consts(const EosParams& P, double* sm0) {
  const int nspc = 20 * P.n, nk = 8 * pair_blocks(P.n), na = 12 * (P.n + (P.n & 1)), nn = 2 * P.K0 + 2 * P.n;
  if (DF) {
    copy_table(reinterpret_cast<float*>(sm0), P.lntab2, 512);
  } else {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) sm0[i] = P.lntab[i];
  }
  // 16-byte aligned, like every table after it (their sizes are multiples of four floats)
  float* fs = reinterpret_cast<float*>(sm0 + 256);
  copy_table(fs, P.spc4, nspc);
  copy_table(fs + nspc, P.K4, nk);
  copy_table(fs + nspc + nk, P.qabs, na);
  float* nf = fs + nspc + nk + na;
  for (int i = threadIdx.x; i < nn; i += blockDim.x) nf[i] = (float)P.norm[i];
  __syncthreads();
  return SharedConsts{reinterpret_cast<const float4*>(fs), reinterpret_cast<const float4*>(fs + nspc),
                      reinterpret_cast<const float4*>(fs + nspc + nk), nullptr, DF ? nullptr : sm0,
                      DF ? reinterpret_cast<const f2*>(sm0) : nullptr, nf, nullptr};
}

// A thread's column of mass fractions in shared memory for mixture_sums: species pairs (2q, 2q + 1) as
// float4 (hi, hi', lo, lo'), entry q at y4[q * STRIDE] (STRIDE the block's threads); a zero pads an odd n.
template <int STRIDE>
struct PairCol {
  float4* y4;
  __device__ __forceinline__ float* at(int k) const {
    return reinterpret_cast<float*>(y4 + (k >> 1) * STRIDE) + (k & 1);
  }
  __device__ __forceinline__ f2 get(int k) const {
    const float* p = at(k);
    return f2{p[0], p[2]};
  }
  __device__ __forceinline__ void set(int k, f2 v) const {
    float* p = at(k);
    p[0] = v.h;
    p[2] = v.l;
  }
  __device__ __forceinline__ void set_pair(int q, f2 a, f2 b) const {
    y4[q * STRIDE] = make_float4(a.h, b.h, a.l, b.l);
  }
};

// The layout of the T-from-h kernel: double-float log table, species table, the FP32 k_ij pair table,
// FP32 normalisation (no double-float pair tables).
__host__ __device__ inline int consts_words_post(const EosParams& P) {
  return 256 + 10 * P.n + P.n * (P.n - 1) / 2 + 1 + (P.K0 + P.n) + kSpcStride / 2;
}

__device__ SharedConsts load_consts_post(const EosParams& P, double* sm0) {
  const int nspc = 20 * P.n, nn = 2 * P.K0 + 2 * P.n;
  copy_table(reinterpret_cast<float*>(sm0), P.lntab2, 512);
  float* fs = reinterpret_cast<float*>(sm0 + 256);
  copy_table(fs, P.spc4, nspc);
  float* ks = fs + nspc;   // 16-byte aligned
  const int nkf = P.n * (P.n - 1) + 2;
  for (int i = threadIdx.x; i < nkf; i += blockDim.x) ks[i] = P.kf2[i];
  float* nf = ks + nkf;
  for (int i = threadIdx.x; i < nn; i += blockDim.x) nf[i] = (float)P.norm[i];
  float* mx = nf + nn;
  for (int i = threadIdx.x; i < kSpcStride; i += blockDim.x) mx[i] = P.spcmax[i];
  __syncthreads();
  return SharedConsts{reinterpret_cast<const float4*>(fs), nullptr, nullptr,
                      reinterpret_cast<const float2*>(ks), nullptr,
                      reinterpret_cast<const f2*>(sm0), nf, mx};
}

// FP64 reciprocal: FP32 seed, two FP64 Newton steps (relative error ~1 ulp).
__device__ __forceinline__ double drcp(double x) {
  double r = f_to_d(__frcp_rn(d_to_f_trunc(x)));
  double e = fma(-x, r, 1.0);
  r = fma(r, e, r);
  e = fma(-x, r, 1.0);
  return fma(r, e, r);
}

// Mixture coefficients of one composition (a1, a2 and the ideal-gas part of a4), all sums in
// double-float, two at a time with the packed FP32x2 instructions and 16-byte loads of species pairs.
// The FP32 pipe takes a packed instruction in the time of two, so the gain is the loads, the broadcasts
// and the issue slots: eos_pre 617 -> 599 us, eos_post 644 -> 616 us on 2^20 cells of 30 species, the
// property kernel 211 -> 195 us on 2^18.
// Symmetric quadratic forms with K_ii = 1, ys_i = Y_i s_i / W_i, yr_i = Y_i r_i / W_i:
//   F0 = sum_ij K_ij ys_i ys_j = sum_i ys_i (ys_i + 2 P_i),  P_i = sum_{j>i} Ks_ij Y_j,
//   F1 = sum_ij K_ij ys_i yr_j = sum_i ys_i (yr_i + Q_i) + yr_i P_i,  Q_i = sum_{j>i} Kr_ij Y_j,
//   F2 = sum_ij K_ij yr_i yr_j = sum_i yr_i (yr_i + 2 Q_i).
// The O(n^2) sums P_i and Q_i use offset accumulators (acc_off_fma), one for the even and one for the
// odd species j, with one offset for all rows: B = sum_j |Y_j| max_l |Ks_lj| (summed rounding up) bounds
// every partial sum of every P_i (likewise for Q_i), and the offset is the power of two above B, or above
// 4 B when some Y_j is negative. The two accumulators' sums less their offsets are multiples of the same
// 2^-23 (2^-24) of the offset and bounded by it, so their sum is exact. A row's error is then a few units
// of 2^-48 B rather than of its own suffix bound, which the forms F weigh by ys_i <= B: the forms stay
// within ~2^-42 B^2, far inside the 1e-10 the state is held to, for 16 fewer operations per row than
// per-row offsets.
template <int STRIDE>
__device__ void mixture_sums(const PairCol<STRIDE> ycol, int n, const SharedConsts& c, MixSums& ms) {
  const float4* y4 = ycol.y4;
  const int nq = (n + 1) >> 1;
  // The O(n) sums (1/W, b/W and the six enthalpy coefficients, species-table columns 0 and 3..9)
  // take offset accumulators too, with bounds Bq = sum_j |Y_j| |q_j| from the same pass.
  const float2 zero = make_float2(0.f, 0.f);
  float2 Bsr = zero, Bq[4] = {zero, zero, zero, zero};
  unsigned neg = 0u;
#pragma unroll 2
  for (int q = 0; q < nq; ++q) {
    const float4 v = y4[q * STRIDE];
    neg |= __float_as_uint(v.x) | __float_as_uint(v.y);
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const float y = fabsf(o ? v.y : v.x);
      const float2 yy = make_float2(y, y);
      const float4* t = c.qabs + 3 * (2 * q + o);
      const float4 a = t[0], b = t[1], k = t[2];
      Bsr = __ffma2_ru(yy, make_float2(k.x, k.y), Bsr);
      Bq[0] = __ffma2_ru(yy, make_float2(a.x, a.y), Bq[0]);
      Bq[1] = __ffma2_ru(yy, make_float2(a.z, a.w), Bq[1]);
      Bq[2] = __ffma2_ru(yy, make_float2(b.x, b.y), Bq[2]);
      Bq[3] = __ffma2_ru(yy, make_float2(b.z, b.w), Bq[3]);
    }
  }
  const float Bs = Bsr.x, Br = Bsr.y;
  // the bounds are rounded up throughout; |Y_j| <= |hi| (1 + 2^-23) is inside the column maxima's margin,
  // and the 2^-10 margin of the O(n) offsets covers the low parts of Y and of the table. The
  // terms are non-negative for Y >= 0 except in the enthalpy columns, whose coefficients have
  // either sign: those take the offset for terms of both signs.
  const float sgf = (neg >> 31) ? 4.0f : 1.0f;
  float2 sq[4], hq[4], lq[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float f = k == 0 ? sgf : 4.0f;
    sq[k] = make_float2(pow2_up(__fmul_ru(f * Bq[k].x, 1.0009765625f)), pow2_up(__fmul_ru(f * Bq[k].y, 1.0009765625f)));
    hq[k] = sq[k];
    lq[k] = zero;
  }
  // The forms themselves: F0 += ys_i ys_i + ys_i (2 P_i), F1 += ys_i yr_i + ys_i Q_i + yr_i P_i,
  // F2 += yr_i yr_i + yr_i (2 Q_i), each into an offset accumulator (F0 and F2 as a pair). The absolute
  // values of the terms of F0 sum to sum_ij |K_ij| |ys_i| |ys_j| <= S_s Bs <= Bs^2, since S_s = sum_i
  // |ys_i| <= Bs (K_jj = 1) and sum_j |K_ij| |ys_j| <= Bs for every i; likewise Bs Br bounds F1 and
  // Br^2 bounds F2.
  const float2 sF02 = make_float2(pow2_up(__fmul_ru(sgf, __fmul_ru(Bs, Bs))), pow2_up(__fmul_ru(sgf, __fmul_ru(Br, Br))));
  const float sF1 = pow2_up(__fmul_ru(sgf, __fmul_ru(Bs, Br)));
  float2 F02h = sF02, F02l = zero;
  float F1h = sF1, F1l = 0.f;
  const float sgs = pow2_up(sgf * Bs), sgr = pow2_up(sgf * Br);   // the rows' common offsets
  const float4* kp = c.K4;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const float4 v = y4[(i >> 1) * STRIDE];
    const float yh = (i & 1) ? v.y : v.x, yl = (i & 1) ? v.w : v.z;
    const float2 yh2 = make_float2(yh, yh), yl2 = make_float2(yl, yl);
    // the O(n) sums and ys_i = Y_i s_i / W_i, yr_i = Y_i r_i / W_i as a pair
    const float4* t = c.spc4 + 5 * i;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 a = t[k];
      acc_off_fma2(hq[k], lq[k], yh2, yl2, make_float2(a.x, a.y), make_float2(a.z, a.w));
    }
    const float4 sr = t[4];
    float2 ysh, ysl;   // (ys, yr)
    mul2(yh2, yl2, make_float2(sr.x, sr.y), make_float2(sr.z, sr.w), ysh, ysl);
    float2 ph = make_float2(sgs, sgs), pl = zero, qh = make_float2(sgr, sgr), ql = zero;
#pragma unroll 4
    for (int q = (i + 1) >> 1; q < nq; ++q, kp += 2) {
      const float4 yj = y4[q * STRIDE], a = kp[0], b = kp[1];
      const float2 jh = make_float2(yj.x, yj.y), jl = make_float2(yj.z, yj.w);
      acc_off_fma2(ph, pl, make_float2(a.x, a.y), make_float2(a.z, a.w), jh, jl);
      acc_off_fma2(qh, ql, make_float2(b.x, b.y), make_float2(b.z, b.w), jh, jl);
    }
    float2 PQh, PQl;   // (P, Q)
    norm2(make_float2(__fadd_rn(__fsub_rn(ph.x, sgs), __fsub_rn(ph.y, sgs)),
                      __fadd_rn(__fsub_rn(qh.x, sgr), __fsub_rn(qh.y, sgr))),
          make_float2(__fadd_rn(pl.x, pl.y), __fadd_rn(ql.x, ql.y)), PQh, PQl);
    acc_off_fma2(F02h, F02l, ysh, ysl, ysh, ysl);
    acc_off_fma2(F02h, F02l, ysh, ysl, __fadd2_rn(PQh, PQh), __fadd2_rn(PQl, PQl));
    const f2 ys = f2{ysh.x, ysl.x}, yr = f2{ysh.y, ysl.y};
    acc_off_fma(F1h, F1l, ys, yr);
    acc_off_fma(F1h, F1l, ys, f2{PQh.y, PQl.y});
    acc_off_fma(F1h, F1l, yr, f2{PQh.x, PQl.x});
    if ((i & 3) == 3) {  // every fourth species: keep the low parts small
#pragma unroll
      for (int k = 0; k < 4; ++k) acc_renorm2(hq[k], lq[k]);
      acc_renorm2(F02h, F02l);
      acc_renorm(F1h, F1l);
    }
  }
  auto fin = [](float h, float sig, float l) { return f2_norm(__fsub_rn(h, sig), l); };
  ms.F0 = fin(F02h.x, sF02.x, F02l.x);
  ms.F1 = fin(F1h, sF1, F1l);
  ms.F2 = fin(F02h.y, sF02.y, F02l.y);
  ms.inv = fin(hq[0].x, sq[0].x, lq[0].x);
  ms.bs = fin(hq[0].y, sq[0].y, lq[0].y);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ms.e[2 * k] = fin(hq[k + 1].x, sq[k + 1].x, lq[k + 1].x);
    ms.e[2 * k + 1] = fin(hq[k + 1].y, sq[k + 1].y, lq[k + 1].y);
  }
}

template <int STRIDE>
__device__ void mixture(const PairCol<STRIDE> ycol, int n, const SharedConsts& c, Mixture& m) {
  MixSums s;
  mixture_sums<STRIDE>(ycol, n, c, s);
  const double invd = f2_to(s.inv);
  const double Wm = drcp(invd);
  const double W2 = Wm * Wm;
  m.inv = invd;
#pragma unroll
  for (int k = 0; k < 6; ++k) m.e[k] = f2_to(s.e[k]);
  m.A0 = W2 * f2_to(s.F0);
  m.A1 = W2 * f2_to(s.F1);
  m.A2 = W2 * f2_to(s.F2);
  m.bm = Wm * f2_to(s.bs);
  m.kb = drcp(2.0 * kSQ2 * m.bm);
}

// Double-float constants (hi, lo) of the state evaluation.
constexpr float kRh = (float)kR, kRl = (float)(kR - (double)(float)kR);
constexpr float kIRh = (float)(1.0 / kR), kIRl = (float)(1.0 / kR - (double)(float)(1.0 / kR));
constexpr float kS2h = (float)(2.0 * kSQ2), kS2l = (float)(2.0 * kSQ2 - (double)(float)(2.0 * kSQ2));
constexpr float kSPh = (float)(1.0 + kSQ2), kSPl = (float)(1.0 + kSQ2 - (double)(float)(1.0 + kSQ2));
constexpr float kSMh = (float)(1.0 - kSQ2), kSMl = (float)(1.0 - kSQ2 - (double)(float)(1.0 - kSQ2));
constexpr float k3h = (float)(1.0 / 3.0), k3l = (float)(1.0 / 3.0 - (double)(float)(1.0 / 3.0));
constexpr float kL2h = (float)0.69314718055994530942,
                kL2l = (float)(0.69314718055994530942 - (double)(float)0.69314718055994530942);

// W_mix scalings of the sums, in double-float.
__device__ __forceinline__ void mix_df_final(const MixSums& s, MixDF& m) {
  const f2 Wm = f2_rcp(s.inv);
  const f2 W2 = f2_mul(Wm, Wm);
  m.inv = s.inv;
#pragma unroll
  for (int k = 0; k < 6; ++k) m.e[k] = s.e[k];
  m.A0 = f2_mul(W2, s.F0);
  m.A1 = f2_mul(W2, s.F1);
  m.A2 = f2_mul(W2, s.F2);
  m.bm = f2_mul(Wm, s.bs);
  m.kb = f2_rcp(f2_mul(m.bm, f2{kS2h, kS2l}));
}

template <int STRIDE>
__device__ void mixture_df(const PairCol<STRIDE> ycol, int n, const SharedConsts& c, MixDF& m) {
  MixSums s;
  mixture_sums<STRIDE>(ycol, n, c, s);
  mix_df_final(s, m);
}

// ln(x) for a positive normal x from the shared table: x = 2^e m, m in [1, 2); with c the
// midpoint of m's 1/128 interval, ln x = e ln2 + ln c + ln(1 + r), r = m / c - 1, |r| < 2^-8,
// ln(1 + r) by its series to r^5 (truncation below 4e-16). Other x take the library log.
__device__ __forceinline__ double dlog_tab(double x, const double* lnt) {
  const int hi = __double2hiint(x);
  const int be = (hi >> 20) & 0x7FF;
  if (hi <= 0 || be == 0 || be == 0x7FF) return log(x);
  const int j = (hi >> 13) & 127;
  const double m = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, __double2loint(x));
  const double r = fma(m, lnt[128 + j], -1.0);
  const double poly = r * fma(r, fma(r, fma(r, fma(r, 0.2, -0.25), 1.0 / 3.0), -0.5), 1.0);
  const double e = f_to_d((float)(be - 1023));
  constexpr double kLn2Hi = 6.93147180369123816490e-01, kLn2Lo = 1.90821492927058770002e-10;
  return fma(e, kLn2Hi, lnt[j] + fma(e, kLn2Lo, poly));
}

// sqrt(x) for a positive normal x: t0 = x rsqrt_32(x), then one Newton step
// t = t0 + (x - t0^2) r / 2 with the FP32 r = rsqrt_32(x) (relative error ~2^-44).
__device__ __forceinline__ double dsqrt_pos(double x) {
  const float r = rsqrtf(d_to_f_trunc(x));
  const double rd = f_to_d(r);
  const double t0 = x * rd;
  return fma(fma(-t0, t0, x), 0.5 * rd, t0);
}

// mixture() for the T-from-h solve, where h(T) needs ~1e-8 relative accuracy (T' to ~1e-6 K):
// with K = 1 - k the forms split into squares of O(n) sums, kept in double-float, and k_ij
// corrections (k <= 0.1 of the squares) summed in FP32,
//   F0 = S_s^2 - 2 sum_i ys_i Pk_i,  F1 = S_s S_r - sum_i (ys_i Qk_i + yr_i Pk_i),
//   F2 = S_r^2 - 2 sum_i yr_i Qk_i,  Pk_i = sum_{j>i} k_ij ys_j,  Qk_i = sum_{j>i} k_ij yr_j.
template <int STRIDE>
__device__ void mixture_post(const f2* ycol, int n, const SharedConsts& c, MixDF& m) {
  constexpr int stride = STRIDE;
  // the ten O(n) sums over the species table take offset accumulators, as in mixture(), here
  // with the looser bounds (sum_j |Y_j|) max_j |q_j|: h(T) is needed to ~1e-8 only, and the
  // bounds then cost one addition per species instead of ten
  float S = 0.f;
  unsigned neg = 0u;
#pragma unroll 2
  for (int j = 0; j < n; ++j) {
    const float yh = ycol[j * stride].h;
    neg |= __float_as_uint(yh);
    S = __fadd_ru(S, fabsf(yh));
  }
  // columns 0..3 (1/W, s/W, r/W, b/W) are non-negative; the enthalpy columns have either sign
  const float sgf = (neg >> 31) ? 4.0f : 1.0f;
  auto sigma = [&](int col) {
    return pow2_up(__fmul_ru((col < 4 ? sgf : 4.0f) * __fmul_ru(S, c.smax[col]), 1.0009765625f));
  };
  // the sums two at a time (packed), in the order of the species table's pairs
  constexpr int colA[5] = {0, 4, 6, 8, 1}, colB[5] = {3, 5, 7, 9, 2};
  float2 sq[5], hq[5], lq[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    sq[k] = make_float2(sigma(colA[k]), sigma(colB[k]));
    hq[k] = sq[k];
    lq[k] = make_float2(0.f, 0.f);
  }
  float C0 = 0.f, C1 = 0.f, C2 = 0.f;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const f2 y = ycol[i * stride];
    const float2 yh2 = make_float2(y.h, y.h), yl2 = make_float2(y.l, y.l);
    const float4* t = c.spc4 + 5 * i;
    float4 a;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      a = t[k];
      acc_off_fma2(hq[k], lq[k], yh2, yl2, make_float2(a.x, a.y), make_float2(a.z, a.w));
    }
    float Pk = 0.f, Qk = 0.f;
    const float2* R = c.kf2 + (i * n - i * (i + 1) / 2) - (i + 1);   // R[j], j > i
#pragma unroll 4
    for (int j = i + 1; j < n; ++j) {
      const float yj = ycol[j * stride].h;
      const float2 k = R[j];
      Pk = fmaf(k.x, yj, Pk);
      Qk = fmaf(k.y, yj, Qk);
    }
    if ((i & 3) == 3) {  // every fourth species: keep the low parts small
#pragma unroll
      for (int k = 0; k < 5; ++k) acc_renorm2(hq[k], lq[k]);
    }
    const float ysi = y.h * a.x, yri = y.h * a.y;   // s/W and r/W: the last pair
    C0 = fmaf(ysi, Pk, C0);
    C1 = fmaf(ysi, Qk, fmaf(yri, Pk, C1));
    C2 = fmaf(yri, Qk, C2);
  }
  f2 r[kSpcStride];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    r[colA[k]] = f2_norm(__fsub_rn(hq[k].x, sq[k].x), lq[k].x);
    r[colB[k]] = f2_norm(__fsub_rn(hq[k].y, sq[k].y), lq[k].y);
  }
  const f2 inv = r[0], Ss = r[1], Sr = r[2], bs = r[3];
  const f2 Wm = f2_rcp(inv);
  const f2 W2 = f2_mul(Wm, Wm);
  m.inv = inv;
#pragma unroll
  for (int k = 0; k < 6; ++k) m.e[k] = r[4 + k];
  m.A0 = f2_mul(W2, f2_addf(f2_mul(Ss, Ss), -2.0f * C0));
  m.A1 = f2_mul(W2, f2_addf(f2_mul(Ss, Sr), -C1));
  m.A2 = f2_mul(W2, f2_addf(f2_mul(Sr, Sr), -2.0f * C2));
  m.bm = f2_mul(Wm, bs);
  m.kb = f2_rcp(f2_mul(m.bm, f2{kS2h, kS2l}));
}

__device__ __forceinline__ double h_ig(const Mixture& m, double T) {
  return fma(fma(fma(fma(fma(m.e[5], T, m.e[4]), T, m.e[3]), T, m.e[2]), T, m.e[1]), T, m.e[0]);
}

__device__ __forceinline__ double cp_ig(const Mixture& m, double T) {
  return fma(fma(fma(fma(5.0 * m.e[5], T, 4.0 * m.e[4]), T, 3.0 * m.e[3]), T, 2.0 * m.e[2]), T,
             m.e[1]);
}

// One Newton step on the cubic. The step uses an FP32 reciprocal of f'(Z): that scales the
// correction by (1 + O(1e-7)), so a step from an FP32-accurate seed still gains ~7 digits.
__device__ __forceinline__ double cubic_step(double Z, double c2, double c1, double c0) {
  const double f = fma(fma(Z + c2, Z, c1), Z, c0);
  const double fp = fma(fma(3.0, Z, 2.0 * c2), Z, c1);
  const float fpf = d_to_f_trunc(fp);
  return fpf != 0.0f ? fma(-f, f_to_d(__frcp_rn(fpf)), Z) : Z;
}

__device__ __forceinline__ double cubic_polish(double Z, double c2, double c1, double c0) {
  return cubic_step(cubic_step(Z, c2, c1, c0), c2, c1, c0);
}

__device__ __forceinline__ double g_dep(double Z, double A, double B, const double* lnt) {
  return Z - 1.0 - dlog_tab(Z - B, lnt) -
         A * drcp(2.0 * kSQ2 * B) * dlog_tab((Z + (1.0 + kSQ2) * B) * drcp(Z + (1.0 - kSQ2) * B), lnt);
}

// Compressibility (a3): the real root of
//   Z^3 - (1 - B) Z^2 + (A - 3B^2 - 2B) Z - (AB - B^2 - B^3) = 0
// above B with least departure Gibbs energy (ties within 1e-12 keep the larger root).
// Seeds come from the FP32 closed form (Cardano for one real root, the trigonometric form
// for three), each polished by two FP64 Newton steps on the cubic.
// The three-real-root case of select_Z: seeds from the trigonometric form, each polished, the
// root above B with least departure Gibbs energy kept. Out of line: it is the rarer branch,
// and keeping it out of the Newton loop's body keeps that loop's code small.
__device__ __noinline__ double select_Z3(double A, double B, double c2, double c1, double c0,
                                         double P, double Q, const double* lnt, int& status);

__device__ double select_Z(double A, double B, const double* lnt, int& status) {
  const double c2 = B - 1.0;
  const double c1 = A - 3.0 * B * B - 2.0 * B;
  const double c0 = B * B + B * B * B - A * B;
  const double P = c1 - c2 * c2 * (1.0 / 3.0);
  const double Q = 2.0 * c2 * c2 * c2 * (1.0 / 27.0) - c2 * c1 * (1.0 / 3.0) + c0;
  const double disc = 0.25 * Q * Q + P * P * P * (1.0 / 27.0);
  if (disc > 0.0) {
    const float qf = d_to_f_trunc(Q), pf = d_to_f_trunc(P);
    const float sq = sqrtf(d_to_f_trunc(disc));
    const float u = cbrtf(-0.5f * qf - copysignf(sq, qf));
    const float t = (u != 0.0f) ? u - pf / (3.0f * u) : 0.0f;
    const double Z0 = f_to_d(t) - c2 * (1.0 / 3.0);
    const double Z = cubic_polish(Z0, c2, c1, c0);
    if (!(Z > B)) status |= kCellNoRoot;
    return Z;
  }
  return select_Z3(A, B, c2, c1, c0, P, Q, lnt, status);
}

__device__ __noinline__ double select_Z3(double A, double B, double c2, double c1, double c0,
                                         double P, double Q, const double* lnt, int& status) {
  const float pf = d_to_f_trunc(P);
  const float m = (pf < 0.0f) ? 2.0f * sqrtf(-pf / 3.0f) : 0.0f;
  float cphi = (pf < 0.0f) ? (3.0f * d_to_f_trunc(Q) / (2.0f * pf)) * sqrtf(-3.0f / pf) : 0.0f;
  cphi = fminf(fmaxf(cphi, -1.0f), 1.0f);
  const float phi = acosf(cphi) * (1.0f / 3.0f);
  double best = __longlong_as_double(0x7ff8000000000000LL);
  double gbest = __longlong_as_double(0x7ff0000000000000LL);
#pragma unroll
  for (int k = 0; k < 3; ++k) {  // k = 0, 1, 2 give descending seeds
    const float tk = m * cosf(phi - 2.0943951023931955f * (float)k);
    const double Z = cubic_polish(cubic_polish(f_to_d(tk) - c2 * (1.0 / 3.0), c2, c1, c0), c2,
                                  c1, c0);
    if (Z > B) {
      const double g = g_dep(Z, A, B, lnt);
      if (g < gbest - 1e-12) {
        gbest = g;
        best = Z;
      }
    }
  }
  if (!(best > B)) status |= kCellNoRoot;
  return best;
}

struct PRPoint {
  double Z, h_dep, cp_dep;  // molar departure enthalpy and its T-derivative at fixed p
};

// Real-fluid state at (T, p) of a composition (a2-a4), with the departure cp if asked.
__device__ PRPoint pr_point(const Mixture& m, double T, double p, bool want_cp, const double* lnt,
                            int& status) {
  const double iT = drcp(T);
  const double t = dsqrt_pos(T);
  const double it = t * iT;                       // 1 / sqrt(T)
  const double am = fma(-2.0 * m.A1, t, fma(m.A2, T, m.A0));
  const double dam = fma(-m.A1, it, m.A2);
  const double RT = kR * T;
  const double iRT = iT * kInvR;
  const double A = am * p * iRT * iRT;
  const double B = m.bm * p * iRT;
  PRPoint r;
  r.Z = select_Z(A, B, lnt, status);
  const double Zp = r.Z + (1.0 + kSQ2) * B;
  const double Zm = r.Z + (1.0 - kSQ2) * B;
  const double iZm = drcp(Zm);
  const double L = dlog_tab(Zp * iZm, lnt);
  const double tdam_am = fma(T, dam, -am);
  r.h_dep = fma(RT, r.Z - 1.0, tdam_am * m.kb * L);
  r.cp_dep = 0.0;
  if (want_cp) {
    const double d2am = 0.5 * m.A1 * it * iT;
    const double dB = -B * iT;
    const double dA = A * fma(dam, drcp(am), -2.0 * iT);
    const double Z = r.Z;
    const double FZ = fma(3.0 * Z, Z, -2.0 * (1.0 - B) * Z) + (A - 3.0 * B * B - 2.0 * B);
    const double FA = Z - B;
    const double FB = Z * Z - (6.0 * B + 2.0) * Z - (A - 2.0 * B - 3.0 * B * B);
    const double dZ = -(FA * dA + FB * dB) / FZ;
    const double dL = (dZ + (1.0 + kSQ2) * dB) * drcp(Zp) - (dZ + (1.0 - kSQ2) * dB) * iZm;
    r.cp_dep = kR * (Z - 1.0) + RT * dZ + m.kb * (T * d2am * L + tdam_am * dL);
  }
  return r;
}

// ---------------------------------------------------------------- double-float state
// The real-fluid point of eos_pre and every Newton iteration of eos_post in double-float on
// the FP32 pipes (~2^-46 relative per operation). On this GPU one FP64 instruction costs the
// issue time of ~30 FP32 instructions (measured in the T-from-h kernel), and a double-float
// operation takes 4 to 15. The steps are those of pr_point above.

// ln x for a positive normal double-float x from the double-float table lt (ln c_j, then
// 1 / c_j): x = 2^e m, m in [1, 2); r = m / c_j - 1 (|r| < 2^-8) formed exactly to first order;
// ln(1 + r) = r - r^2/2 in double-float plus r^3 (1/3 - r/4 + r^2/5) in FP32 (below 2^-25).
__device__ __noinline__ f2 f2_log_slow(f2 x) { return f2_from(log(f2_to(x))); }

__device__ __forceinline__ f2 f2_log_tab(f2 x, const f2* lt) {
  const unsigned u = __float_as_uint(x.h);
  const int be = (int)((u >> 23) & 0xFFu);
  if ((int)u <= 0 || be == 0 || be >= 254) return f2_log_slow(x);
  const int j = (int)((u >> 16) & 127u);
  const float sc = __uint_as_float((unsigned)(254 - be) << 23);   // 2^-(be - 127), exact
  const float mh = __fmul_rn(x.h, sc), ml = __fmul_rn(x.l, sc);
  const f2 ic = lt[128 + j];
  const float p = __fmul_rn(mh, ic.h);
  const float pe = __fmaf_rn(mh, ic.h, -p);
  const f2 r = f2_norm(__fsub_rn(p, 1.0f), __fmaf_rn(mh, ic.l, __fmaf_rn(ml, ic.h, pe)));
  const float r2 = __fmul_rn(r.h, r.h);
  const float r2e = __fmaf_rn(2.0f * r.h, r.l, __fmaf_rn(r.h, r.h, -r2));
  const float tail =
      __fmul_rn(__fmul_rn(r2, r.h), __fmaf_rn(r.h, __fmaf_rn(r.h, 0.2f, -0.25f), 0.33333334f));
  const f2 l1p = f2_addf(f2_add(r, f2{-0.5f * r2, -0.5f * r2e}), tail);
  const float E = (float)(be - 127);
  const float q = __fmul_rn(E, kL2h);
  const f2 el2 = f2_norm(q, __fmaf_rn(E, kL2l, __fmaf_rn(E, kL2h, -q)));
  return f2_add(f2_add(el2, lt[j]), l1p);
}

// x^(1/3) in FP32 for a seed: 2^(log2|x| / 3) with the sign of x, then one Newton step
// t <- t - (t^3 - x) / (3 t^2) (~1 ulp).
__device__ __forceinline__ float cbrt_seed(float x) {
  if (x == 0.0f) return 0.0f;
  const float t = copysignf(exp2f(log2f(fabsf(x)) * (1.0f / 3.0f)), x);
  return t - (t - __fdividef(x, t * t)) * (1.0f / 3.0f);
}

// One Newton step on the cubic, f(Z) and f'(Z) in double-float, the step with an approximate
// FP32 reciprocal of f'(Z) (it scales the correction by 1 + O(1e-7)).
__device__ __forceinline__ f2 cubic_step_df(f2 Z, f2 c2, f2 c1, f2 c0) {
  const f2 f = f2_fma(f2_fma(f2_add(Z, c2), Z, c1), Z, c0);
  const f2 fp = f2_fma(f2_add(f2_mulf(Z, 3.0f), f2_scale2(c2)), Z, c1);
  return fp.h != 0.0f ? f2_add(Z, f2_mulf(f, -__fdividef(1.0f, fp.h))) : Z;
}

__device__ __forceinline__ f2 g_dep_df(f2 Z, f2 A, f2 B, const f2* lt) {
  const f2 Zp = f2_fma(B, f2{kSPh, kSPl}, Z), Zm = f2_fma(B, f2{kSMh, kSMl}, Z);
  const f2 L = f2_log_tab(f2_mul(Zp, f2_rcp(Zm)), lt);
  const f2 a = f2_mul(A, f2_rcp(f2_mul(B, f2{kS2h, kS2l})));
  return f2_sub(f2_sub(f2_addf(Z, -1.0f), f2_log_tab(f2_sub(Z, B), lt)), f2_mul(a, L));
}

// Departure Gibbs energy in FP32 (for choosing among the three roots when the choice is clear).
__device__ __forceinline__ float g_dep_f(float Z, float A, float B) {
  const float s2 = 1.41421356f;
  return Z - 1.0f - __logf(Z - B) -
         __fdividef(A, 2.0f * s2 * B) * __logf(__fdividef(Z + (1.0f + s2) * B, Z + (1.0f - s2) * B));
}

// The distance from B beyond which the Gibbs energy at an FP32 seed ranks its root: a hundred times the
// seed's error (3e-7, and 2e-7 over the sine of phi, which goes to 0 at a double root). The roots are
// stationary points of the Gibbs energy, so that error enters as (error / (Z - B))^2 / 2 = 5e-5.
__device__ __forceinline__ float seed_distance(float cphi) {
  return fmaf(2e-5f, rsqrtf(fmaxf(fmaf(-cphi, cphi, 1.0f), 1e-6f)), 3e-5f);
}

// Three real roots (select_Z3 in double-float). Out of line, as there. The roots above B are
// first ranked by their FP32 seeds and FP32 departure Gibbs energies; when one root is lower
// by more than 1e-4 (the FP32 energies are good to 2e-5) and no seed is too close to B
// (seed_distance), only that root is polished. Otherwise every root is polished and compared in
// double-float: next to a saturation line, where the energies nearly agree, or at low pressure, where
// a liquid's root lies as near to B as its FP32 seed is off.
__device__ __noinline__ f2 select_Z3_df(f2 A, f2 B, f2 c2, f2 c1, f2 c0, f2 c23, float Pf,
                                        float Qf, const f2* lt, int& status) {
  const float m = (Pf < 0.0f) ? 2.0f * sqrtf(-Pf / 3.0f) : 0.0f;
  float cphi = (Pf < 0.0f) ? (3.0f * Qf / (2.0f * Pf)) * sqrtf(-3.0f / Pf) : 0.0f;
  cphi = fminf(fmaxf(cphi, -1.0f), 1.0f);
  const float phi = acosf(cphi) * (1.0f / 3.0f);
  {
    float tbest = 0.0f, g1 = __int_as_float(0x7f800000), g2 = g1;
    bool clear = true;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
      const float tk = m * cosf(phi - 2.0943951023931955f * (float)k);
      const float zk = tk - c23.h;
      if (fabsf(zk - B.h) < seed_distance(cphi)) clear = false;
      if (zk > B.h) {
        const float g = g_dep_f(zk, A.h, B.h);
        if (!(g == g)) clear = false;
        if (g < g1) {
          g2 = g1;
          g1 = g;
          tbest = tk;
        } else if (g < g2) {
          g2 = g;
        }
      }
    }
    if (clear && g1 < g2 - 1e-4f) {
      f2 Z = f2_sub(f2{tbest, 0.0f}, c23);
#pragma unroll 1
      for (int q = 0; q < 4; ++q) Z = cubic_step_df(Z, c2, c1, c0);
      if (!f2_gt(Z, B)) status |= kCellNoRoot;
      return Z;
    }
  }
  f2 best = f2{__int_as_float(0x7fc00000), 0.0f};
  f2 gbest = f2{__int_as_float(0x7f800000), 0.0f};
  bool have = false;
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {  // k = 0, 1, 2 give descending seeds
    const float tk = m * cosf(phi - 2.0943951023931955f * (float)k);
    f2 Z = f2_sub(f2{tk, 0.0f}, c23);
#pragma unroll 1
    for (int q = 0; q < 4; ++q) Z = cubic_step_df(Z, c2, c1, c0);
    if (f2_gt(Z, B)) {
      const f2 g = g_dep_df(Z, A, B, lt);
      if (!have || f2_lt(g, f2_addf(gbest, -1e-12f))) {
        gbest = g;
        best = Z;
        have = true;
      }
    }
  }
  if (!have) status |= kCellNoRoot;
  return best;
}

// select_Z in double-float: the coefficients, P, Q and the discriminant in double-float, the
// seeds in FP32, one or two double-float Newton polishes as in select_Z.
template <bool FAST>
__device__ __forceinline__ f2 select_Z_df(f2 A, f2 B, const f2* lt, int& status) {
  const f2 c2 = f2_addf(B, -1.0f);
  const f2 c1 = f2_sub(A, f2_mul(B, f2_addf(f2_mulf(B, 3.0f), 2.0f)));  // A - 3B^2 - 2B
  const f2 c0 = f2_mul(B, f2_sub(f2_fma(B, B, B), A));                 // B^2 + B^3 - AB
  const f2 c23 = f2_mul(c2, f2{k3h, k3l});                              // c2 / 3
  const f2 P = f2_sub(c1, f2_mul(c2, c23));                             // c1 - c2^2 / 3
  // Q = 2 c2^3 / 27 - c2 c1 / 3 + c0 = 2 (c2/3)^3 - (c2/3) c1 + c0
  const f2 Q = f2_add(f2_sub(f2_scale2(f2_mul(c23, f2_mul(c23, c23))), f2_mul(c23, c1)), c0);
  const f2 P3 = f2_mul(P, f2{k3h, k3l});
  const f2 Qh = f2{0.5f * Q.h, 0.5f * Q.l};
  const f2 disc = f2_fma(Qh, Qh, f2_mul(P3, f2_mul(P3, P3)));          // Q^2/4 + P^3/27
  if (disc.h > 0.0f) {
    const float qf = Q.h, pf = P.h;
    const float sq = sqrtf(disc.h);
    const float u = cbrt_seed(-0.5f * qf - copysignf(sq, qf));
    const float t = (u != 0.0f) ? u - __fdividef(pf, 3.0f * u) : 0.0f;
    const f2 Z0 = f2_sub(f2{t, 0.0f}, c23);
    f2 Z = cubic_step_df(Z0, c2, c1, c0);
    if (!FAST || fabsf(Z.h - Z0.h) > 1e-6f * fabsf(Z.h)) Z = cubic_step_df(Z, c2, c1, c0);
    if (!f2_gt(Z, B)) status |= kCellNoRoot;
    return Z;
  }
  return select_Z3_df(A, B, c2, c1, c0, c23, P.h, Q.h, lt, status);
}

struct PRPointDF {
  f2 Z, h_dep;    // compressibility, molar departure enthalpy
  float cp_dep;   // its T-derivative in FP32 (FAST with want_cp only)
};

// pr_point in double-float; with FAST the departure cp (the chord slope of the T-from-h
// solve) in FP32 as there.
template <bool FAST>
__device__ PRPointDF pr_point_df(const MixDF& m, f2 T, f2 p, bool want_cp, const f2* lt,
                                 int& status) {
  const f2 iT = f2_rcp(T);
  const f2 t = f2_sqrt_pos(T);
  const f2 it = f2_mul(t, iT);                                   // 1 / sqrt(T)
  const f2 am = f2_fma(m.A1, f2{-2.0f * t.h, -2.0f * t.l}, f2_fma(m.A2, T, m.A0));
  const f2 dam = f2_fma(f2_neg(m.A1), it, m.A2);
  const f2 RT = f2_mul(T, f2{kRh, kRl});
  const f2 iRT = f2_mul(iT, f2{kIRh, kIRl});
  const f2 piRT = f2_mul(p, iRT);
  const f2 A = f2_mul(f2_mul(am, piRT), iRT);
  const f2 B = f2_mul(m.bm, piRT);
  PRPointDF r;
  r.Z = select_Z_df<FAST>(A, B, lt, status);
  const f2 Zp = f2_fma(B, f2{kSPh, kSPl}, r.Z), Zm = f2_fma(B, f2{kSMh, kSMl}, r.Z);
  const f2 L = f2_log_tab(f2_mul(Zp, f2_rcp(Zm)), lt);
  const f2 tdam_am = f2_fma(T, dam, f2_neg(am));
  r.h_dep = f2_fma(RT, f2_addf(r.Z, -1.0f), f2_mul(f2_mul(tdam_am, m.kb), L));
  r.cp_dep = 0.0f;
  if (FAST && want_cp) {
    // FP32: dA/dT = p (dam - 2 am / T) / (RT)^2 needs no division by am
    const float Tf = T.h, iTf = __fdividef(1.0f, Tf), itf = rsqrtf(Tf);
    const float Z = r.Z.h, Af = A.h, Bf = B.h;
    const float pf = p.h, iRTf = iTf * (float)kInvR;
    const float d2am = 0.5f * m.A1.h * itf * iTf;
    const float dB = -Bf * iTf;
    const float dA = pf * iRTf * iRTf * (dam.h - 2.0f * am.h * iTf);
    const float FZ = fmaf(3.0f * Z, Z, -2.0f * (1.0f - Bf) * Z) + (Af - 3.0f * Bf * Bf - 2.0f * Bf);
    const float FA = Z - Bf;
    const float FB = Z * Z - (6.0f * Bf + 2.0f) * Z - (Af - 2.0f * Bf - 3.0f * Bf * Bf);
    // (a chord slope: approximate FP32 divisions suffice)
    const float dZ = -__fdividef(FA * dA + FB * dB, FZ);
    const float s2 = (float)kSQ2;
    const float dL = __fdividef(dZ + (1.0f + s2) * dB, Zp.h) - __fdividef(dZ + (1.0f - s2) * dB, Zm.h);
    r.cp_dep = (float)kR * (Z - 1.0f) + (float)kR * Tf * dZ +
               m.kb.h * (Tf * d2am * L.h + tdam_am.h * dL);
  }
  return r;
}

__device__ __forceinline__ f2 h_ig_df(const MixDF& m, f2 T) {
  f2 a = m.e[5];
#pragma unroll
  for (int k = 4; k >= 0; --k) a = f2_fma(a, T, m.e[k]);
  return a;
}

__device__ __forceinline__ float cp_ig_f(const MixDF& m, float T) {
  return fmaf(fmaf(fmaf(fmaf(5.0f * m.e[5].h, T, 4.0f * m.e[4].h), T, 3.0f * m.e[3].h), T,
                   2.0f * m.e[2].h), T, m.e[1].h);
}

// a9: T from h(T, p, Y') = h0 for the composition of m, safeguarded Newton inside a bracket that
// starts at [50, 5000] K and shrinks with the sign of h - h0, the residual and the iterates in
// double-float. Adds flags to st and the iteration count to iters; returns the last iterate. Chord
// steps: the slope of the first iteration is reused while the iterates stay close (each step contracts
// the error by ~|1 - cp(T)/cp(T0)| ~ 1e-5 there). A step within tolerance has converged; only a longer
// step that leaves the bracket (or is not finite) is replaced by bisection, after which the slope is
// evaluated afresh.
__device__ f2 solve_T_df(const MixDF& m, f2 p, f2 h0, double Told, const EosParams& P,
                         const f2* lt, int& iters, int& st) {
  f2 lo = f2{(float)kTLo, 0.0f}, hi = f2{(float)kTHi, 0.0f};
  f2 Tn = f2_from(Told);
  if (f2_lt(Tn, lo)) Tn = lo;
  if (f2_gt(Tn, hi)) Tn = hi;
  bool conv = false, need_cp = true;
  float icp = 0.0f;
  const float tolf = (float)P.newton_tol;
  for (int it = 0; it < P.newton_max_iter; ++it) {
    ++iters;
    int s2 = 0;
    const PRPointDF q = pr_point_df<true>(m, Tn, p, need_cp, lt, s2);
    if (s2) {
      st |= s2;
      break;
    }
    const f2 f = f2_sub(f2_fma(q.h_dep, m.inv, h_ig_df(m, Tn)), h0);
    // an FP32 reciprocal slope scales the step by 1 + O(1e-7)
    if (need_cp) icp = __fdividef(1.0f, fmaf(q.cp_dep, m.inv.h, cp_ig_f(m, Tn.h)));
    if (__float_as_int(f.h) >= 0) hi = Tn; else lo = Tn;
    const f2 step = f2_mulf(f, -icp);
    f2 Tx = f2_add(Tn, step);
    const bool done = fabsf(step.h) <= tolf * Tn.h;
    need_cp = false;
    if (!done && !(f2_gt(Tx, lo) && f2_lt(Tx, hi))) {
      const f2 mid = f2_add(lo, hi);
      Tx = f2{0.5f * mid.h, 0.5f * mid.l};
      need_cp = true;
    }
    Tn = Tx;
    if (done) {
      conv = true;
      break;
    }
  }
  if (!conv && st == 0) st |= kCellNotConverged;
  if (!isfinite(Tn.h)) st |= kCellNonfinite;
  return Tn;
}

template <typename XT>
__device__ __forceinline__ XT to_x(float v, float scale);
template <>
__device__ __forceinline__ float to_x<float>(float v, float) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_x<__nv_bfloat16>(float v, float) {
  return __float2bfloat16_rn(v);
}
template <>
__device__ __forceinline__ __nv_fp8_e4m3 to_x<__nv_fp8_e4m3>(float v, float scale) {
  return __nv_fp8_e4m3(v * scale);
}

// Raw bits of a network-input element, for packing a row into 16-byte stores.
__device__ __forceinline__ uint32_t x_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t x_bits(__nv_bfloat16 v) { return __bfloat16_as_ushort(v); }
__device__ __forceinline__ uint32_t x_bits(__nv_fp8_e4m3 v) { return v.__x; }

template <typename XT, int RW>
__device__ __forceinline__ void x_put(uint32_t (&w)[RW], int e, XT v) {
  constexpr int EPW = 4 / (int)sizeof(XT);
  w[e / EPW] |= x_bits(v) << (8 * (int)sizeof(XT) * (e % EPW));
}

// Y^lambda of a Box-Cox feature. Features rounded to BF16 or FP8 (8 or 4 significant bits)
// take the hardware approximations of log2 and exp2 (a relative error of a few 1e-7, far below
// that rounding); FP32 features take the library's accurate functions.
template <typename XT>
__device__ __forceinline__ float boxcox_pow(float y, float lam) {
  if constexpr (sizeof(XT) < 4) return __powf(y, lam);
  else return exp2f(lam * log2f(y));
}

// Species whose mass fractions a thread loads before using any (NM is a multiple of it).
constexpr int kLoadBatch = 16;

// a1-a5 for the valid rows of a batch.
template <int NM, typename XT, int TH>
__global__ void __launch_bounds__(TH, TH == kThreads ? kPreBlocks : 1) eos_pre_kernel(EosParams P, RowMap rows,
    const double* __restrict__ T, const double* __restrict__ p, const double* __restrict__ Y,
    int64_t ldY, double* __restrict__ h0, double* __restrict__ Zout, XT* __restrict__ x,
    int64_t ldx, float x_scale, int32_t* __restrict__ status, double* __restrict__ rho) {
  extern __shared__ __align__(16) double sm[];
  const SharedConsts c = load_consts<true>(P, sm);
  const PairCol<TH> ycol{reinterpret_cast<float4*>(sm + consts_words(P)) + threadIdx.x};
  pdl_begin();   // the constants above do not change; the cells and rows do
  const int64_t nrow = valid_rows(rows);
  const int n = P.n, K0 = P.K0;
  const float lam = (float)P.lambda;
  const float ilam = 1.0f / lam;
  const float* mf = c.normf;        // in_mean
  const float* isf = c.normf + K0;  // 1 / in_std
  // Network-input rows go out as 16-byte stores from registers when the row pitch allows:
  // RW words hold the NM + 2 entries a row can have, EPC elements make one 16-byte chunk.
  constexpr int EPC = 16 / (int)sizeof(XT);
  constexpr int RW = ((NM + 2 + EPC - 1) / EPC) * 4;
  const int64_t row_bytes = ldx * (int64_t)sizeof(XT);
  const bool xvec = x && (row_bytes & 15) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const int nch = (int)(row_bytes >> 4);
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nrow;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cell = row_cell(rows, r);
    const double Tc = T[cell], pc = p[cell];
    bool finite = d_finite(Tc) && d_finite(pc) && d_pos(pc) && d_pos(Tc);
    XT* xr = x ? x + r * ldx : nullptr;
    // the double-float column of Y (and, without packed rows, the a5 features), sixteen
    // species at a time with all their loads issued first: one memory latency per batch
#pragma unroll
    for (int k0 = 0; k0 < NM; k0 += kLoadBatch) {
      double yv[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) yv[u] = k0 + u < n ? Y[(k0 + u) * ldY + cell] : 0.0;
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int k = k0 + u;
        if (k < n) {
          const double yd = yv[u];
          finite = finite && d_finite(yd);
          if (xr && !xvec) {
            const float y = fmaxf(d_to_f_trunc(yd), 0.0f);
            const float bc = (y > 0.0f) ? (boxcox_pow<XT>(y, lam) - 1.0f) * ilam : -ilam;
            xr[2 + k] = to_x<XT>((bc - mf[2 + k]) * isf[2 + k], x_scale);
          }
          if ((u & 1) == 0) ycol.set_pair(k >> 1, f2_from(yd), f2_from(yv[u + 1]));
        }
      }
    }
    if (xr && !xvec) {
      xr[0] = to_x<XT>(finite ? (d_to_f_trunc(Tc) - mf[0]) * isf[0] : 0.0f, x_scale);
      xr[1] = to_x<XT>(finite ? (d_to_f_trunc(pc) - mf[1]) * isf[1] : 0.0f, x_scale);
      if (!finite)
        for (int k = 0; k < n; ++k) xr[2 + k] = to_x<XT>(0.0f, x_scale);
      for (int k = K0; k < ldx; ++k) xr[k] = to_x<XT>(0.0f, x_scale);
    }
    int st = 0;
    double h = __longlong_as_double(0x7ff8000000000000LL), Z = h;
    if (finite) {
      MixDF m;
      mixture_df<TH>(ycol, n, c, m);
      const f2 Td = f2_from(Tc), pd = f2_from(pc);
      const PRPointDF q = pr_point_df<false>(m, Td, pd, false, c.lt2, st);
      Z = f2_to_int(q.Z);
      const f2 hd = f2_fma(q.h_dep, m.inv, h_ig_df(m, Td));
      h = f2_to_int(hd);
      if (!isfinite(hd.h)) st |= kCellNonfinite;
      // rho = p W_mix / (Z R T)
      if (rho) rho[r] = f2_to_int(f2_mul(pd, f2_rcp(f2_mul(f2_mul(m.inv, q.Z), f2_mul(Td, f2{kRh, kRl})))));
    } else {
      st = kCellNonfinite;
    }
    if (xvec) {
      // a5 features from the column (its high parts are Y rounded to FP32), packed into
      // registers and written as 16-byte stores: a row of RW words covers any n <= NM
      uint32_t w[RW];
#pragma unroll
      for (int q = 0; q < RW; ++q) w[q] = 0u;
      if (finite) {
#pragma unroll
        for (int k = 0; k < NM; ++k) {
          if (k < n) {
            const float y = fmaxf(*ycol.at(k), 0.0f);
            const float bc = (y > 0.0f) ? (boxcox_pow<XT>(y, lam) - 1.0f) * ilam : -ilam;
            x_put(w, 2 + k, to_x<XT>((bc - mf[2 + k]) * isf[2 + k], x_scale));
          }
        }
      }
      x_put(w, 0, to_x<XT>(finite ? (d_to_f_trunc(Tc) - mf[0]) * isf[0] : 0.0f, x_scale));
      x_put(w, 1, to_x<XT>(finite ? (d_to_f_trunc(pc) - mf[1]) * isf[1] : 0.0f, x_scale));
      uint4* xo = reinterpret_cast<uint4*>(xr);
#pragma unroll
      for (int q = 0; q < RW / 4; ++q)
        if (q < nch) xo[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
      for (int q = RW / 4; q < nch; ++q) xo[q] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (h0) h0[r] = h;
    if (Zout) Zout[r] = Z;
    if (status) status[r] = st;
  }
}

__device__ __forceinline__ double ipow(double b, int m) {
  double r = 1.0;
  while (m) {
    if (m & 1) r *= b;
    b *= b;
    m >>= 1;
  }
  return r;
}

// Y' = Y (1 + eps)^m for a growth (1 + eps)^m beyond e^80, in FP64. Out of line (rare).
__device__ __noinline__ f2 yprime_large(double y, float eps, int mpow) {
  return f2_from(y * ipow(1.0 + f_to_d(eps), mpow));
}

// Y' = Y (1 + eps)^m by log1p and expm1, for |eps| > 1/16 or 1/lambda > 16 (out of line: the
// common case takes the binomial sum).
__device__ __noinline__ f2 yprime_log(double y, float eps, float mf, int mpow) {
  const f2 yf = f2_from(y);
  const float lg = mf * log1pf(eps);
  return (lg < 80.0f) ? f2_add(yf, f2_mulf(yf, expm1f(lg))) : yprime_large(y, eps, mpow);
}

// Y' for Y below 1e-30 (or not positive): the closed form (Y^lambda + lambda du)^(1/lambda).
// Y^lambda (< 1e-30^lambda) in FP32, lambda du is FP32 already, the power in double-float: an
// absolute error of ~1e-7 Y^lambda in the base moves Y' by less than m 1e-7 Y^lambda base^(m-1).
__device__ __forceinline__ f2 yprime_small(double y, float lamf, float ldu, int mpow) {
  const float yf = d_to_f_trunc(y);
  const float base = ((yf > 0.0f) ? exp2f(lamf * log2f(yf)) : 0.0f) + ldu;
  if (!(base > 0.0f)) return f2{0.f, 0.f};
  f2 r = f2{1.0f, 0.0f}, b = f2{base, 0.0f};
  for (int m = mpow; m; m >>= 1) {
    if (m & 1) r = f2_mul(r, b);
    b = f2_mul(b, b);
  }
  return r;
}

// a8-a10 for the valid rows of a batch. Y' lives in this thread's shared-memory column (double-
// float) from the increment to the write-back, which happens only once the Newton solve for T
// has succeeded.
template <int NM, int TH>
__global__ void __launch_bounds__(TH, TH == kThreads ? kPostBlocks : 1) eos_post_kernel(EosParams P, RowMap rows,
    const float* __restrict__ O, int64_t ldo, const double* __restrict__ h0,
    double* __restrict__ T, const double* __restrict__ p, double* __restrict__ Y, int64_t ldY,
    const int32_t* __restrict__ pre_status, int32_t* __restrict__ cell_status, Source src) {
  extern __shared__ __align__(16) double sm[];
  const SharedConsts c = load_consts_post(P, sm);
  f2* ycol = reinterpret_cast<f2*>(sm + consts_words_post(P)) + threadIdx.x;
  constexpr int stride = TH;
  pdl_begin();
  const int64_t nrow = valid_rows(rows);
  const int n = P.n, K0 = P.K0;
  const float* out_mean = c.normf + 2 * K0;
  const float* out_std = c.normf + 2 * K0 + n;
  const float lamf = (float)P.lambda;
  const int mpow = P.inv_lambda;
  const float mf = (float)P.inv_lambda;
  const bool binom = P.binom[0] != 0.0f;
  const bool ovec = (ldo & 3) == 0 && (reinterpret_cast<uintptr_t>(O) & 15) == 0;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nrow;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cell = row_cell(rows, r);
    const double Told = T[cell], pc = p[cell], h0c = h0[r];
    int st = pre_status ? pre_status[r] : 0;  // flags eos_pre raised for this row
    bool finite = d_finite(Told) && d_finite(pc) && d_pos(pc) && d_finite(h0c);
    f2 S = {0.f, 0.f};
    const float* Or = O + r * ldo;
    // Y's column into this thread's column slots as FP64 bit patterns, sixteen loads in flight
    // at a time; each slot is overwritten by Y'_k below
#pragma unroll
    for (int k0 = 0; k0 < NM; k0 += kLoadBatch) {
      double yv[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) yv[u] = k0 + u < n ? Y[(k0 + u) * ldY + cell] : 0.0;
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u)
        if (k0 + u < n)
          ycol[(k0 + u) * stride] = f2{__int_as_float(__double2loint(yv[u])),
                                       __int_as_float(__double2hiint(yv[u]))};
    }
    // the row's outputs four at a time (one 16-byte load when the row pitch allows, the next
    // group's load issued before this group's arithmetic)
    float4 onext = ovec ? *reinterpret_cast<const float4*>(Or) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < n; k0 += 4) {
      float o4[4];
      if (ovec) {
        const float4 v = onext;
        if (k0 + 4 < n) onext = *reinterpret_cast<const float4*>(Or + k0 + 4);
        o4[0] = v.x;
        o4[1] = v.y;
        o4[2] = v.z;
        o4[3] = v.w;
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) o4[q] = (k0 + q < n) ? Or[k0 + q] : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = k0 + q;
        if (k >= n) break;
        const f2 yraw = ycol[k * stride];
        const double y = __hiloint2double(__float_as_int(yraw.l), __float_as_int(yraw.h));
        finite = finite && d_finite(y);
        const float ldu = lamf * fmaf(out_std[k], o4[q], out_mean[k]);  // lambda du
        f2 yn = {0.f, 0.f};
        if (d_ge_pos(y, 1e-30)) {
          // Y' = (Y^lambda + lambda du)^(1/lambda) = Y (1 + eps)^m, eps = lambda du Y^-lambda;
          // the increment delta = (1 + eps)^m - 1 only scales Y' - Y, so FP32 suffices.
          const f2 yf = f2_from(y);
          const float eps = ldu * exp2f(-lamf * log2f(yf.h));
          if (binom && fabsf(eps) <= 0.0625f) {
            // delta = sum_{j=1..m} C(m, j) eps^j by Horner; for |eps| <= 1/16 the terms fall
            // off at least like (m eps)^j / j!, so the FP32 sum is good to a few ulp
            float b = 1.0f;
#pragma unroll 4
            for (int j = mpow - 1; j >= 1; --j) b = fmaf(b, eps, P.binom[j]);
            yn = f2_add(yf, f2_mulf(yf, b * eps));
          } else if (eps > -1.0f) {
            yn = yprime_log(y, eps, mf, mpow);
          }
        } else if (d_finite(y)) {
          yn = yprime_small(y, lamf, ldu, mpow);
        }
        ycol[k * stride] = yn;
        acc_add(S, yn);
      }
    }
    S = f2_fin(S);
    if (!finite || !(S.h > 0.0f) || !isfinite(S.h)) st |= kCellNonfinite;
    double Tn = Told;
    int iters = 0;
    if (st == 0) {
      const f2 iS = f2_rcp(S);
      for (int k = 0; k < n; ++k) ycol[k * stride] = f2_mul(ycol[k * stride], iS);
      MixDF m;
      mixture_post<TH>(ycol, n, c, m);
      Tn = f2_to_int(solve_T_df(m, f2_from(pc), f2_from(h0c), Told, P, c.lt2, iters, st));
    }
    if (st == 0 && src.omega) {
      // source terms rho (Y' - Y) / dt; Y' - Y in double-float
      const f2 sc = f2_from(src.rho[r] * src.inv_dt);
#pragma unroll 2
      for (int k = 0; k < n; ++k) {
        const f2 d = f2_add(ycol[k * stride], f2_from(-Y[k * ldY + cell]));
        src.omega[k * src.ldw + cell] = f2_to_int(f2_mul(d, sc));
      }
      if (src.T_new) src.T_new[cell] = Tn;
    } else if (st == 0) {
      T[cell] = Tn;
#pragma unroll 2
      for (int k = 0; k < n; ++k) Y[k * ldY + cell] = f2_to_int(ycol[k * stride]);
    }
    if (cell_status) cell_status[cell] = st;
    if (st && P.flagged) atomicAdd((unsigned long long*)P.flagged, 1ull);
    if (P.newton_iters) {  // one atomic per warp
      const unsigned mask = __activemask();
      const int tot = __reduce_add_sync(mask, iters);
      if ((threadIdx.x & 31) == __ffs(mask) - 1)
        atomicAdd((unsigned long long*)P.newton_iters, (unsigned long long)tot);
    }
  }
}

// Compressibility, the cubic's slope there and the density from the mixing sums, for the properties: the
// root is told and found in double-float, then takes a Newton step on the cubic in FP64, whose coefficients
// are FP64 from the sums on. Near critical points and where roots merge the slope goes to zero and a root
// is off by the coefficients' error divided by it; a dilute gas's Z is 1 less a small number.
struct Root64 {
  double Z, slope, rho;
};
__device__ __forceinline__ Root64 root64(const MixSums& s, double T, double p, const f2* lt, int& status) {
  const double Wm = drcp(f2_to(s.inv)), W2 = Wm * Wm, iT = drcp(T), t = dsqrt_pos(T);
  const double am = W2 * fma(-2.0 * f2_to(s.F1), t, fma(f2_to(s.F2), T, f2_to(s.F0)));
  const double iRT = iT * kInvR, pRT = p * iRT;
  const double A = am * pRT * iRT, B = Wm * f2_to(s.bs) * pRT;
  const double c2 = B - 1.0, c1 = fma(B, fma(-3.0, B, -2.0), A), c0 = B * (fma(B, B, B) - A);
  Root64 r;
  r.Z = cubic_step(f2_to(select_Z_df<false>(f2_from(A), f2_from(B), lt, status)), c2, c1, c0);
  r.slope = fma(fma(3.0, r.Z, 2.0 * c2), r.Z, c1);
  r.rho = pRT * Wm * drcp(r.Z);
  return r;
}

// Real-fluid c_p of the state q = pr_point_df(m, T, p) and the coefficients of dh/dY_k at fixed T, p.
// (Without GRAD: c_p and the departure enthalpy at the root q.Z, where the cubic's slope is given.)
// With u_k = y_k sqrt(a_k), yr_k = y_k r_k (y = Y / W), v = K u, w = K yr, sigma = sum y = 1 / W:
//   a = W^2 u.v,  a' = -(W^2 / sqrt T) yr.v,  b = W sum y_k b_k,
//   da/dy_k = 2 W^2 sqrt(a_k) v_k - 2 W a,  db/dy_k = W (b_k - b),
//   da'/dy_k = -2 W a' - (W^2 / sqrt T)(r_k v_k + sqrt(a_k) w_k),
//   dZ from the implicit cubic, h = sum y_k h_k(T) + sigma h_dep,
//   dh/dY_k = (h_k(T) + h_dep + sigma dh_dep/dy_k) / W_k.
// h_dep depends on the composition through a, a' and b alone; with alpha, beta, gamma its derivatives,
//   dh/dY_k = h_k/W_k + c0 / W_k + (c1 A_k - c2 R_k) v_k - c2 A_k w_k + c3 b_k / W_k,
//   A_k = (s_k - r_k sqrt T) / W_k,  R_k = r_k / W_k,  c1 = 2 W alpha,  c2 = W beta / sqrt T,  c3 = gamma,
//   c0 = h_dep - 2 a alpha - 2 a' beta - b gamma.
struct HGrad {
  f2 T, t, c0, c1, c2, c3;
};

template <bool GRAD>
__device__ __noinline__ void state_grad(const MixDF& m, f2 T, f2 p, PRPointDF& q, f2 slope, const f2* lt, f2& cp,
                                        HGrad& g) {
  const f2 iT = f2_rcp(T), t = f2_sqrt_pos(T), it = f2_mul(t, iT);
  const f2 am = f2_fma(m.A1, f2{-2.0f * t.h, -2.0f * t.l}, f2_fma(m.A2, T, m.A0));
  const f2 dam = f2_fma(f2_neg(m.A1), it, m.A2);
  const f2 RT = f2_mul(T, f2{kRh, kRl}), iRT = f2_mul(iT, f2{kIRh, kIRl});
  const f2 pRT = f2_mul(p, iRT), pRT2 = f2_mul(pRT, iRT);
  const f2 A = f2_mul(am, pRT2), B = f2_mul(m.bm, pRT), Z = q.Z;
  const f2 c1s = f2{kSPh, kSPl}, c2s = f2{kSMh, kSMl};
  const f2 iZp = f2_rcp(f2_fma(B, c1s, Z)), iZm = f2_rcp(f2_fma(B, c2s, Z));
  const f2 L = f2_log_tab(f2_mul(f2_fma(B, c1s, Z), iZm), lt);
  const f2 tda = f2_fma(T, dam, f2_neg(am));
  const f2 kbL = f2_mul(m.kb, L);
  // f_Z, f_A, f_B of the cubic: 3 Z^2 - 2 (1 - B) Z + A - 3 B^2 - 2 B, Z - B, Z^2 - (6 B + 2) Z - (A - 2 B - 3 B^2)
  const f2 B3 = f2_mul(B, f2_addf(f2_mulf(B, 3.0f), 2.0f));
  const f2 FZ = GRAD ? f2_add(f2_mul(Z, f2_add(f2_mulf(Z, 3.0f), f2_scale2(f2_addf(B, -1.0f)))), f2_sub(A, B3)) : slope;
  const f2 FA = f2_sub(Z, B);
  const f2 FB = f2_add(f2_mul(Z, f2_sub(Z, f2_addf(f2_mulf(B, 6.0f), 2.0f))), f2_sub(B3, A));
  const f2 iFZ = f2_rcp(FZ);
  const f2 e1 = f2_sub(iZp, iZm), e2 = f2_sub(f2_mul(c1s, iZp), f2_mul(c2s, iZm));
  const f2 tk = f2_mul(tda, m.kb);
  // dh_dep = gz dZ + kb L d(T a' - a) + T a' terms; dZ = -(FA dA + FB dB) / FZ
  const f2 gz = f2_fma(tk, e1, RT);
  // c_p: d/dT at fixed composition, dA = A (a'/a - 2/T) = p (a' - 2 a / T) / (RT)^2, dB = -B / T
  const f2 d2am = f2_mul(f2_mulf(m.A1, 0.5f), f2_mul(it, iT));
  const f2 dA = f2_mul(pRT2, f2_sub(dam, f2_scale2(f2_mul(am, iT))));
  const f2 dB = f2_neg(f2_mul(B, iT));
  const f2 dZ = f2_neg(f2_mul(iFZ, f2_fma(FA, dA, f2_mul(FB, dB))));
  const f2 dL = f2_fma(dZ, e1, f2_mul(dB, e2));
  const f2 Rf = f2{kRh, kRl};
  f2 cpd = f2_mul(Rf, f2_addf(Z, -1.0f));
  cpd = f2_fma(RT, dZ, cpd);
  cpd = f2_fma(f2_mul(T, d2am), kbL, cpd);
  cpd = f2_fma(tk, dL, cpd);
  f2 cpi = f2_mulf(m.e[5], 5.0f);
  cpi = f2_fma(cpi, T, f2_mulf(m.e[4], 4.0f));
  cpi = f2_fma(cpi, T, f2_mulf(m.e[3], 3.0f));
  cpi = f2_fma(cpi, T, f2_scale2(m.e[2]));
  cpi = f2_fma(cpi, T, m.e[1]);
  cp = f2_fma(cpd, m.inv, cpi);
  if constexpr (!GRAD) {
    q.h_dep = f2_fma(RT, f2_addf(Z, -1.0f), f2_mul(tk, L));
    return;
  }
  const f2 W = f2_rcp(m.inv);
  const f2 gi = f2_mul(gz, iFZ);
  const f2 al = f2_neg(f2_fma(f2_mul(gi, FA), pRT2, kbL));
  const f2 be = f2_mul(kbL, T);
  f2 ga = f2_neg(f2_mul(f2_mul(gi, FB), pRT));
  ga = f2_sub(ga, f2_mul(f2_mul(tda, kbL), f2_rcp(m.bm)));
  ga = f2_fma(f2_mul(tk, e2), pRT, ga);
  g.T = T;
  g.t = t;
  g.c1 = f2_scale2(f2_mul(W, al));
  g.c2 = f2_mul(f2_mul(be, W), it);
  g.c3 = ga;
  f2 c0 = f2_sub(q.h_dep, f2_scale2(f2_mul(am, al)));
  c0 = f2_sub(c0, f2_scale2(f2_mul(dam, be)));
  g.c0 = f2_sub(c0, f2_mul(m.bm, ga));
}

// Density, enthalpy, c_p and compressibility of every cell (outputs may be NULL), in double-float but for
// the cubic's coefficients, the last step of its root and the density (Root64). 2^18 cells of 30 species:
// 195 us with all of the state in FP64 (its pipe busy half of the time) and mass fractions loaded two at a
// time, 153 us so, 147 us without FP64, whose roots near critical points were twice as far off. Errors
// against FP64 on ordinary states: 1.7e-13 in density and 1.4e-13 in c_p, set by the mixing sums.
template <int NM>
__global__ void __launch_bounds__(kThreads, kPreBlocks) props_kernel(EosParams P, int64_t ncell,
    const double* __restrict__ T, const double* __restrict__ p, const double* __restrict__ Y,
    int64_t ldY, double* rho, double* h, double* cp, double* Zo) {
  extern __shared__ __align__(16) double sm[];
  const SharedConsts c = load_consts<true>(P, sm);
  const PairCol<kThreads> ycol{reinterpret_cast<float4*>(sm + consts_words(P)) + threadIdx.x};
  const int n = P.n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncell;
       i += (int64_t)gridDim.x * blockDim.x) {
    const f2 Td = f2_from(T[i]), pd = f2_from(p[i]);
#pragma unroll
    for (int k0 = 0; k0 < NM; k0 += kLoadBatch) {
      double yv[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) yv[u] = k0 + u < n ? Y[(k0 + u) * ldY + i] : 0.0;
#pragma unroll
      for (int u = 0; u < kLoadBatch; u += 2)
        if (k0 + u < n) ycol.set_pair((k0 + u) >> 1, f2_from(yv[u]), f2_from(yv[u + 1]));
    }
    MixSums ms;
    mixture_sums<kThreads>(ycol, n, c, ms);
    int st = 0;
    const Root64 z = root64(ms, T[i], p[i], c.lt2, st);
    if (rho) rho[i] = z.rho;
    if (Zo) Zo[i] = z.Z;
    if (!h && !cp) continue;
    MixDF m;
    mix_df_final(ms, m);
    PRPointDF q;
    q.Z = f2_from(z.Z);
    f2 cpv;
    HGrad g;
    state_grad<false>(m, Td, pd, q, f2_from(z.slope), c.lt2, cpv, g);
    if (h) h[i] = f2_to_int(f2_fma(q.h_dep, m.inv, h_ig_df(m, Td)));
    if (cp) cp[i] = f2_to_int(cpv);
  }
}


// ---------------------------------------------------------------- transport properties
// Chung, Ajlan, Lee & Starling (1988), the high-pressure viscosity and thermal conductivity of
// a mixture from its pseudo-critical constants (Chung's mixing rules over the mole fractions)
// and its molar density, here the Peng-Robinson density; the ideal-gas Cv and the real-fluid c_p
// come from the same NASA-7 / Peng-Robinson state. The correlation is accurate to a few percent,
// so it is evaluated in FP32 (the PR state and the outer mixing sums stay FP64).

// Chung's coefficients E_i = a_i + b_i omega (viscosity) and B_i (conductivity), nonpolar,
// non-associating species
__constant__ float kChungE[10][2] = {
    {6.324f, 50.412f}, {1.210e-3f, -1.154e-3f}, {5.283f, 254.209f}, {6.623f, 38.096f},
    {19.745f, 7.630f}, {-1.900f, -12.537f}, {24.275f, 3.450f}, {0.7972f, 1.117f},
    {-0.2382f, 0.06770f}, {0.06863f, 0.3479f}};
__constant__ float kChungB[7][2] = {
    {2.4166f, 0.74824f}, {-0.50924f, -1.5094f}, {6.6107f, 5.6207f}, {14.543f, -8.9139f},
    {0.79274f, 0.82019f}, {-5.8634f, 12.801f}, {91.089f, 128.73f}};

// Chung's G2 with coefficients C1..C5 at reduced density y (G1 the Carnahan-Starling contact
// value); (1 - exp(-C4 y)) / y by expm1 so that dilute cells keep their digits
__device__ __forceinline__ float chung_g2(const float (&C)[10], float y, float G1) {
  const float t = y > 0.0f ? -expm1f(-C[3] * y) / y : C[3];
  return (C[0] * t + C[1] * G1 * __expf(C[4] * y) + C[2] * G1) / (C[0] * C[3] + C[1] + C[2]);
}

// mu (Pa s) and lambda (W/(m K)) of a pseudo-pure fluid (Tc K, Vc cm^3/mol, omega, M g/mol) at
// temperature T, molar density rho (mol/cm^3) and ideal-gas molar Cv (J/(mol K))
__device__ void chung(float T, float rho, float Tc, float Vc, float om, float M, float cv,
                      float& mu, float& lam) {
  const float Ts = 1.2593f * T / Tc;
  // collision integral of Neufeld, Janzen & Aziz (1972)
  const float Om = 1.16145f * __powf(Ts, -0.14874f) + 0.52487f * __expf(-0.77320f * Ts) +
                   2.16178f * __expf(-2.43787f * Ts);
  const float y = rho * Vc * (1.0f / 6.0f);
  const float omy = 1.0f - y;
  const float G1 = (1.0f - 0.5f * y) / (omy * omy * omy);
  float E[10], B[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) E[i] = kChungE[i][0] + kChungE[i][1] * om;
#pragma unroll
  for (int i = 0; i < 7; ++i) B[i] = kChungB[i][0] + kChungB[i][1] * om;
  const float G2 = chung_g2(E, y, G1);
  const float Fc = 1.0f - 0.2756f * om;
  const float c = cbrtf(Vc);
  const float vc23 = c * c;
  const float eta_k = sqrtf(Ts) / Om * Fc * (1.0f / G2 + E[5] * y);
  const float eta_p = E[6] * y * y * G2 * __expf(E[7] + E[8] / Ts + E[9] / (Ts * Ts));
  mu = (eta_k + eta_p) * 36.344f * sqrtf(M * Tc) / vc23 * 1e-7f;
  // thermal conductivity: dilute viscosity (Pa s), Cv correction Psi, dense terms
  const float Mk = M * 1e-3f;
  const float eta0 = 40.785f * Fc * sqrtf(M * T) / (vc23 * Om) * 1e-7f;
  const float a = cv * (float)kInvR - 1.5f;
  const float b = 0.7862f - 0.7109f * om + 1.3168f * om * om;
  const float Tr = T / Tc;
  const float Zp = 2.0f + 10.5f * Tr * Tr;
  const float psi = 1.0f + a * (0.215f + 0.28288f * a - 1.061f * b + 0.26665f * Zp) /
                               (0.6366f + b * Zp + 1.061f * a * b);
  const float H2 = chung_g2(B, y, G1);
  const float q = 3.586e-3f * sqrtf(Tc / Mk) / vc23;
  lam = 31.2f * eta0 * psi / Mk * (1.0f / H2 + B[5] * y) + q * B[6] * y * y * sqrtf(Tr) * H2;
}

template <int NM>
__global__ void __launch_bounds__(kPropThreads, kPropBlocks) transport_kernel(EosParams P, int64_t ncell,
    const double* __restrict__ T, const double* __restrict__ p, const double* __restrict__ Y,
    int64_t ldY, double* mu, double* lam, double* alpha) {
  extern __shared__ __align__(16) double sm[];
  const SharedConsts c = load_consts(P, sm);
  const PairCol<kPropThreads> ycol{reinterpret_cast<float4*>(sm + consts_words(P)) + threadIdx.x};
  const int n = P.n, nn = P.n * P.n;
  const float* __restrict__ tp = P.tpair;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncell;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double Tk = T[i], pk = p[i];
    bool finite = d_finite(Tk) && d_finite(pk) && d_pos(pk) && d_pos(Tk);
    for (int k = 0; k < n; k += 2) {
      const double ya = Y[k * ldY + i], yb = k + 1 < n ? Y[(k + 1) * ldY + i] : 0.0;
      finite = finite && d_finite(ya) && d_finite(yb);
      ycol.set_pair(k >> 1, f2_from(ya), f2_from(yb));
    }
    double m_out = __longlong_as_double(0x7ff8000000000000LL), l_out = m_out, a_out = m_out;
    if (finite) {
      Mixture m;
      mixture<kPropThreads>(ycol, n, c, m);
      int st = 0;
      const PRPoint q = pr_point(m, Tk, pk, true, c.lnt, st);
      const double rho = pk / (m.inv * q.Z * kR * Tk);            // kg/m^3
      const double cpm = cp_ig(m, Tk) + q.cp_dep * m.inv;           // J/(kg K)
      const double Wm = 1.0 / m.inv;
      // mole fractions x_k = (Y_k / W_k) W_mix, kept in the column's high words
      const float Wmf = (float)Wm;
      for (int k = 0; k < n; ++k) *ycol.at(k) = *ycol.at(k) * c.spc4[5 * k].x * Wmf;
      // Chung's mixing sums, symmetric: sum_ij x_i x_j A_ij = sum_i x_i (A_ii x_i + 2 sum_{j>i} A_ij x_j)
      double S[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
      for (int a = 0; a < n; ++a) {
        const float xa = *ycol.at(a);
        float R4[4];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) R4[qq] = 0.5f * __ldg(tp + qq * nn + a * n + a) * xa;
        for (int b = a + 1; b < n; ++b) {
          const float xb = *ycol.at(b);
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) R4[qq] = fmaf(__ldg(tp + qq * nn + a * n + b), xb, R4[qq]);
        }
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) S[qq] = fma(2.0 * (double)xa, (double)R4[qq], S[qq]);
      }
      const double eps_m = S[1] / S[0];
      const double sig2 = cbrt(S[0] * S[0]);                        // sigma_m^2
      const double Mr = S[3] / (eps_m * sig2);
      const float Tcm = (float)(1.2593 * eps_m);
      const float Vcm = (float)(S[0] / (0.809 * 0.809 * 0.809));
      const float omm = (float)(S[2] / S[0]);
      const float cv = (float)(cp_ig(m, Tk) * Wm - kR);             // ideal-gas molar Cv
      float muf, lamf;
      chung((float)Tk, (float)(rho * m.inv * 1e-6), Tcm, Vcm, omm, (float)(Mr * Mr), cv, muf, lamf);
      if (st == 0) {
        m_out = (double)muf;
        l_out = (double)lamf;
        a_out = (double)lamf / (rho * cpm);
      }
    }
    if (mu) mu[i] = m_out;
    if (lam) lam[i] = l_out;
    if (alpha) alpha[i] = a_out;
  }
}


// ---------------------------------------------------------------- Jacobian of the step

// b^m for an integer m >= 0 by squaring, in double-float.
__device__ __forceinline__ f2 f2_ipow(f2 b, int m) {
  f2 r = f2{1.0f, 0.0f};
  for (; m; m >>= 1) {
    if (m & 1) r = f2_mul(r, b);
    if (m > 1) b = f2_mul(b, b);
  }
  return r;
}

// y^lambda for a normal FP32 y > 0 and lambda = 1/m to within dl: r0 = FP32 power (relative error
// ~1e-6), then r = r0 (1 + e)^(-1/m) with e = r0^m / y - 1 by its series to e^3 (|e| ~ 1e-5,
// truncation below 1e-19), in double-float.
__device__ __forceinline__ f2 f2_root(f2 y, float lamf, int m, float dl) {
  const float r0 = exp2f(lamf * log2f(y.h));
  const f2 e = f2_addf(f2_mul(f2_ipow(f2{r0, 0.0f}, m), f2_rcp(y)), -1.0f);
  const float im = 1.0f / (float)m;
  // (1 + e)^(-1/m) - 1 = -e/m + (1/m)(1/m + 1) e^2 / 2 - (1/m)(1/m + 1)(1/m + 2) e^3 / 6
  const float q = im * (im + 1.0f) * 0.5f * e.h * e.h * (1.0f - (im + 2.0f) * (1.0f / 3.0f) * e.h);
  f2 c = f2_mul(e, f2_rcp(f2{-(float)m, 0.0f}));
  c = f2_addf(c, dl != 0.0f ? q + dl * logf(y.h) : q);
  return f2_add(f2{r0, 0.0f}, f2_mulf(c, r0));
}

// y^lambda for 0 < y < 1e-30, whose double-float low part, or itself, falls out of FP32's range: the root
// of y 2^(sm), which lies in it, times 2^-s. (Such species count as much as any other: the root of 1e-300
// is 1e-30 for lambda = 0.1 and 2e-5 for 1/64.)
__device__ __forceinline__ f2 root_small(double y, float lamf, int m, float dl) {
  const int s = (m - 71 - max((__double2hiint(y) >> 20) - 1023, -1023)) / m;   // y 2^(sm) >= 2^-70 (normal y)
  if (s > 120) return f2{0.0f, 0.0f};
  const f2 r = f2_root(f2_from(y * __hiloint2double((1023 + s * m) << 20, 0)), lamf, m, dl);
  return f2_mulf(r, __int_as_float((127 - s) << 23) * fmaf(-0.6931472f * dl, (float)(s * m), 1.0f));
}

// Input scales of the tangent directions (T, Y_1..Y_n): dx_0/dT = 1/std_T and
// dx_{2+j}/dY_j = BC'(Y_j) / std_{2+j}, BC'(y) = max(y, 1e-12)^(lambda - 1) in FP64: for lambda = 1/m
// the m-th root by the series of f2_root in FP64 (about 20 FP64 operations against the hundred of pow:
// 106 -> 42 us for 20,000 cells x 31 directions), else pow.
__global__ void jac_scale_kernel(EosParams P, int64_t ncell, const double* __restrict__ Y,
                                 int64_t ldY, const double* __restrict__ norm,
                                 float* __restrict__ sc) {
  const int ntan = P.n + 1, K0 = P.K0, m = P.inv_lambda;
  const bool root = P.lambda == 1.0 / m;
  const float lamf = (float)P.lambda;
  const double im = 1.0 / m, i2 = im * (im + 1.0) * 0.5, i3 = i2 * (im + 2.0) * (1.0 / 3.0);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ncell * ntan;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = e / ntan;
    const int t = (int)(e % ntan);
    double v;
    if (t == 0) {
      v = norm[K0];
    } else {
      const double y = fmax(Y[(int64_t)(t - 1) * ldY + c], 1e-12);
      if (root && y < 1e30) {
        const double r0 = f_to_d(exp2f(lamf * log2f(d_to_f_trunc(y)))), iy = drcp(y);
        double q = 1.0, b = r0;
        for (int k = m; k; k >>= 1) {
          if (k & 1) q *= b;
          if (k > 1) b *= b;
        }
        const double d = fma(q, iy, -1.0);
        v = r0 * iy * fma(d, fma(d, fma(-d, i3, i2), -im), 1.0) * norm[K0 + 1 + t];
      } else {
        v = pow(y, P.lambda - 1.0) * norm[K0 + 1 + t];
      }
    }
    sc[e] = (float)v;
  }
}

// Layer-1 tangents: dH1[c ntan + t, j] = sc[c, t] * W1[j, col(t)] * G1[c, j], col(0) = 0 (T),
// col(t) = t + 1 (Y_{t-1}); W1T is W1 transposed [K0 x N1]. A block takes kTanCells cells; each thread
// holds eight G1 values of each of them as they are stored, reads eight weights of a direction
// once (two 16-byte loads when N1 is a multiple of four) and writes the scaled products into
// the cells' tangent rows as 16-byte (BF16) or 32-byte (FP32) groups. Pitches ldg and ldh are
// multiples of eight elements. Bound by the writes (1.99 GB for 20,011 cells of 30 species); a direction's
// weights and scales are read one direction ahead of their use, the cells' G1 takes half the registers
// in BF16, and a block per cell group leaves no partial round: 475 -> 360 us (5.5 TB/s).
constexpr int kTanCells = 4;

// Eight consecutive values, converted to FP32 when used.
template <typename GT>
struct Eight;
template <>
struct Eight<__nv_bfloat16> {
  uint4 q;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { q = __ldg(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ float get(int e) const {   // BF16 is the upper half of FP32
    const uint32_t x = (e >> 1) == 0 ? q.x : (e >> 1) == 1 ? q.y : (e >> 1) == 2 ? q.z : q.w;
    return __uint_as_float((e & 1) ? x & 0xFFFF0000u : x << 16);
  }
};
template <>
struct Eight<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = __ldg(reinterpret_cast<const float4*>(p));
    b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  }
  __device__ __forceinline__ float get(int e) const {
    const float4& v = e < 4 ? a : b;
    return (e & 3) == 0 ? v.x : (e & 3) == 1 ? v.y : (e & 3) == 2 ? v.z : v.w;
  }
};

template <typename OT, typename GT>
__global__ void __launch_bounds__(256) jac_tangent0_kernel(int64_t ncell, int ntan, int N1,
    const float* __restrict__ sc, const float* __restrict__ W1T, const GT* __restrict__ G1, int64_t ldg,
    OT* __restrict__ dH, int64_t ldh) {
  const int groups = (N1 + 7) / 8;
  const bool vec_w = (N1 & 3) == 0;
  const int64_t c0 = (int64_t)blockIdx.x * kTanCells;
  const int nc = (int)(ncell - c0 < kTanCells ? ncell - c0 : kTanCells);
  for (int g = threadIdx.x; g < groups; g += blockDim.x) {
    const int j0 = 8 * g;
    const int m = min(8, N1 - j0);
    Eight<GT> gv[kTanCells];
#pragma unroll
    for (int q = 0; q < kTanCells; ++q) gv[q].load(G1 + (c0 + min(q, nc - 1)) * ldg + j0);
    float w[8], s[kTanCells];
    auto load = [&](int t, float (&wt)[8], float (&st)[kTanCells]) {
      const float* wp = W1T + (int64_t)(t == 0 ? 0 : t + 1) * N1 + j0;
      if (vec_w && m == 8) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(wp));
        const float4 b = __ldg(reinterpret_cast<const float4*>(wp) + 1);
        wt[0] = a.x; wt[1] = a.y; wt[2] = a.z; wt[3] = a.w;
        wt[4] = b.x; wt[5] = b.y; wt[6] = b.z; wt[7] = b.w;
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) wt[e] = e < m ? __ldg(wp + e) : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < kTanCells; ++q) st[q] = __ldg(sc + (c0 + min(q, nc - 1)) * ntan + t);
    };
    load(0, w, s);
    for (int t = 0; t < ntan; ++t) {
      float wn[8], sn[kTanCells];
      load(min(t + 1, ntan - 1), wn, sn);
#pragma unroll
      for (int q = 0; q < kTanCells; ++q) {
        if (q >= nc) break;
        const int64_t row = (c0 + q) * ntan + t;
        __align__(16) OT o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) o[e] = (OT)(s[q] * w[e] * gv[q].get(e));
        OT* dst = dH + row * ldh + j0;
        if (m == 8) {
          // 8 elements at an offset that is a multiple of 8: 16 or 32 aligned bytes
          if constexpr (sizeof(OT) == 2) {
            *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(o);
          } else {
            reinterpret_cast<uint4*>(dst)[0] = reinterpret_cast<const uint4*>(o)[0];
            reinterpret_cast<uint4*>(dst)[1] = reinterpret_cast<const uint4*>(o)[1];
          }
        } else {
          for (int e = 0; e < m; ++e) dst[e] = o[e];
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) w[e] = wn[e];
#pragma unroll
      for (int q = 0; q < kTanCells; ++q) s[q] = sn[q];
    }
  }
}

// Jacobian of the step of every cell (treated as reacting): J[c][k][t] = d(Y'_k - Y_k)/dv_t and
// dTn[c][t] = dT'/dv_t, v = (T, Y_1..Y_n), from the network output O, its tangents dO
// ([c ntan + t][k] = dO_k/dv_t) and the implicit function h(T', p, Y') = h0(T, p, Y).
// Two kernels, both in double-float (FP64 arithmetic took 1.35 ms for 20,000 cells: jac_post 834 us at
// four warps per SM, each a chain of FP64 sums over species pairs; assembly 513 us on the FP64 pipe):
// jac_state_kernel, a thread per cell, takes what is scalar in the cell: Y', the mixture sums and states
// at (T, Y) and (T', Y'), T' by Newton; it leaves in the cell's scratch row, as double-float pairs,
//   [dZ_k/du_k / S (n), Y'_k (n), c_p(T, Y), c_p(T', Y'), HGrad at (T, Y), HGrad at (T', Y')];
// jac_columns_kernel, a warp per cell, takes the rest: lane k the sums over species of dh/dY_k at both
// states, then lane t the column of direction t. 114 and 188 us for those cells. The first is bound by
// the chains of its four warps an SM; the second by L1: lane t reads its direction's tangents one float
// at a time from a row of its own, 25 sectors a request (L1 data pipe 77 %, FP32 pipes 33 %).
constexpr int kJacRow = 2 + 2 * 6;   // scalars per cell after the two columns

template <int NM>
__global__ void __launch_bounds__(kPropThreads) jac_state_kernel(EosParams P, int64_t ncell, int64_t cell0,
    const double* __restrict__ T, const double* __restrict__ p, const double* __restrict__ Y,
    int64_t ldY, const float* __restrict__ O, int64_t ldo, const double* __restrict__ h0,
    bool want_dT, float2* __restrict__ scr, int32_t* __restrict__ cst) {
  extern __shared__ __align__(16) double sm[];
  const SharedConsts c = load_consts<true>(P, sm);
  constexpr int stride = kPropThreads;
  const PairCol<stride> ycol{reinterpret_cast<float4*>(sm + consts_words(P)) + threadIdx.x};
  const int n = P.n, K0 = P.K0;
  const float* out_mean = c.normf + 2 * K0;
  const float* out_std = c.normf + 2 * K0 + n;
  const float lamf = (float)P.lambda;
  const int mpow = P.inv_lambda;
  const float dl = (float)(P.lambda - 1.0 / mpow);
  auto put = [](float2* d, f2 v) { *d = make_float2(v.h, v.l); };
  auto put_grad = [&](float2* d, const HGrad& g) {
    put(d, g.T); put(d + 1, g.t); put(d + 2, g.c0); put(d + 3, g.c1); put(d + 4, g.c2); put(d + 5, g.c3);
  };
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < ncell;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cell = cell0 + r;
    const double Tc = T[cell], pc = p[cell], h0c = h0[r];
    bool finite = d_finite(Tc) && d_finite(pc) && d_pos(pc) && d_finite(h0c);
#pragma unroll
    for (int k0 = 0; k0 < NM; k0 += kLoadBatch) {
      double yv[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) yv[u] = k0 + u < n ? Y[(k0 + u) * ldY + cell] : 0.0;
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u)
        if (k0 + u < n) {
          finite = finite && d_finite(yv[u]);
          if ((u & 1) == 0) ycol.set_pair((k0 + u) >> 1, f2_from(yv[u]), f2_from(yv[u + 1]));
        }
    }
    int st = finite && d_pos(Tc) ? 0 : kCellNonfinite;
    float2* q = scr + r * (int64_t)(2 * n + kJacRow);
    const f2 pd = f2_from(pc);
    if (st == 0) {
      MixDF m;
      mixture_df<stride>(ycol, n, c, m);
      const f2 Td = f2_from(Tc);
      PRPointDF s0 = pr_point_df<false>(m, Td, pd, false, c.lt2, st);
      if (want_dT) {
        f2 cp;
        HGrad g;
        state_grad<true>(m, Td, pd, s0, f2{0.0f, 0.0f}, c.lt2, cp, g);
        put(q + 2 * n, cp);
        put_grad(q + 2 * n + 2, g);
      }
    }
    if (st == 0) {
      // Y' and dZ_k/du_k = Z_k^(1 - lambda) = base^(m - 1), base = Y_k^lambda + lambda du_k
      f2 S = f2{0.0f, 0.0f};
      const float* Or = O + r * ldo;
      for (int k = 0; k < n; ++k) {
        const float ldu = lamf * fmaf(out_std[k], Or[k], out_mean[k]);
        const f2 yk = ycol.get(k);
        f2 root = f2{0.0f, 0.0f};
        if (yk.h >= 1e-30f) {
          root = f2_root(yk, lamf, mpow, dl);
        } else if (yk.h >= 0.0f) {
          const double y = Y[k * ldY + cell];
          if (y > 0.0) root = root_small(y, lamf, mpow, dl);
        }
        const f2 base = f2_addf(root, ldu);
        f2 zl = f2{0.0f, 0.0f}, z = zl;
        if (base.h > 0.0f) {
          zl = f2_ipow(base, mpow - 1);
          z = f2_mul(zl, base);
        }
        put(q + k, zl);
        ycol.set(k, z);
        acc_add(S, z);
      }
      S = f2_fin(S);
      if (!(S.h > 0.0f) || !isfinite(S.h)) st |= kCellNonfinite;
      if (st == 0) {
        const f2 iS = f2_rcp(S);
        for (int k = 0; k < n; ++k) {
          const f2 z = f2_mul(ycol.get(k), iS);
          ycol.set(k, z);
          put(q + n + k, z);
          const float2 zl = q[k];
          put(q + k, f2_mul(f2{zl.x, zl.y}, iS));
        }
        MixDF m;
        mixture_df<stride>(ycol, n, c, m);
        int iters = 0;
        const f2 Tn = solve_T_df(m, pd, f2_from(h0c), Tc, P, c.lt2, iters, st);
        if (st == 0) {
          PRPointDF s1 = pr_point_df<false>(m, Tn, pd, false, c.lt2, st);
          if (want_dT) {
            f2 cp;
            HGrad g;
            state_grad<true>(m, Tn, pd, s1, f2{0.0f, 0.0f}, c.lt2, cp, g);
            put(q + 2 * n + 1, cp);
            put_grad(q + 2 * n + 8, g);
          }
        }
      }
    }
    cst[r] = st;
  }
}

// Columns of the Jacobian from jac_state_kernel's per-cell results: ju_k = out_std_k dO_k/dv_t +
// [t = k + 1] BC'(Y_k), jy_k = (dZ_k/du_k ju_k - Y'_k sum_j dZ_j/du_j ju_j) / S, J[k][t] = jy_k -
// [t = k + 1], dT'/dv_t = (dh/dv_t - sum_k dh/dY'_k jy_k) / c_p. The BC' term enters linearly, so the
// loops over k run without it and its share is added at k = t - 1. Cells whose status is not 0 get NaN.
constexpr int kColWarps = 8;
template <int NM>
__global__ void __launch_bounds__(32 * kColWarps) jac_columns_kernel(EosParams P, int64_t ncell,
    int64_t cell0, const double* __restrict__ Y, int64_t ldY, const float* __restrict__ dO,
    int64_t lddo, const float2* __restrict__ scr, const int32_t* __restrict__ cst,
    float* __restrict__ J, double* __restrict__ dTn) {
  const int n = P.n, K0 = P.K0, ntan = n + 1;
  // K transposed (lane k reads K[k][j] at j * NM + k) and, per warp, columns that all lanes read
  __shared__ float2 Ksh[NM * NM];
  __shared__ float2 col[kColWarps][5][NM];
  __shared__ float sdf[NM];
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const f2 v = f2_from(P.Kmat[e]);
    Ksh[(e % n) * NM + e / n] = make_float2(v.h, v.l);
  }
  for (int k = threadIdx.x; k < n; k += blockDim.x) sdf[k] = (float)P.norm[2 * K0 + n + k];
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float2 *zl = col[w][0], *yp = col[w][1], *hg = col[w][2], *cu = col[w][3], *cr = col[w][4];
  const int kl = lane < n ? lane : n - 1;
  // this lane's species constants over W: 1/W, s/W, r/W, b/W, enthalpy coefficients
  const float2* sp = reinterpret_cast<const float2*>(P.spcw2) + kl * kSpcStride;
  auto ld = [](const float2* a) { const float2 v = *a; return f2{v.x, v.y}; };
  auto st2 = [](float2* d, f2 v) { *d = make_float2(v.h, v.l); };
  const float lamf = (float)P.lambda;
  const int mpow = P.inv_lambda;
  const float dl = (float)(P.lambda - 1.0 / mpow);
  const int64_t warps = (int64_t)gridDim.x * kColWarps;
  // dh/dY_k of lane k at the state of coefficients g (6 pairs) and mass fraction y
  auto h_grad = [&](const float2* g, f2 y) -> f2 {
    const f2 Tg = ld(g), t = ld(g + 1);
    const f2 rw = ld(sp + 2), A = f2_sub(ld(sp + 1), f2_mul(rw, t));
    __syncwarp();
    if (lane < n) {
      st2(cu + lane, f2_mul(y, A));
      st2(cr + lane, f2_mul(y, rw));
    }
    __syncwarp();
    f2 v = f2{0.0f, 0.0f}, x = v;
#pragma unroll 2
    for (int j = 0; j < n; ++j) {
      const f2 K = ld(Ksh + j * NM + kl);
      acc_fma(v, K, ld(cu + j));
      acc_fma(x, K, ld(cr + j));
    }
    v = f2_fin(v);
    x = f2_fin(x);
    f2 h = ld(sp + 9);
#pragma unroll
    for (int k = 8; k >= 4; --k) h = f2_fma(h, Tg, ld(sp + k));
    const f2 c2 = ld(g + 4);
    h = f2_fma(ld(g + 2), ld(sp), h);
    h = f2_fma(f2_sub(f2_mul(ld(g + 3), A), f2_mul(c2, rw)), v, h);
    h = f2_sub(h, f2_mul(f2_mul(c2, A), x));
    return f2_fma(ld(g + 5), ld(sp + 3), h);
  };
  for (int64_t r = blockIdx.x * (int64_t)kColWarps + w; r < ncell; r += warps) {
    const int64_t cell = cell0 + r;
    float* Jc = J + cell * (int64_t)n * ntan;
    double* dTc = dTn ? dTn + cell * (int64_t)ntan : nullptr;
    if (cst[r] != 0) {
      const float nanf = __int_as_float(0x7fc00000);
      for (int e = lane; e < n * ntan; e += 32) Jc[e] = nanf;
      if (dTc)
        for (int t = lane; t < ntan; t += 32) dTc[t] = __longlong_as_double(0x7ff8000000000000LL);
      continue;
    }
    const float2* q = scr + r * (int64_t)(2 * n + kJacRow);
    const f2 y0 = lane < n ? f2_from(Y[(int64_t)lane * ldY + cell]) : f2{0.0f, 0.0f};
    const f2 y1 = ld(q + n + kl), z1 = ld(q + kl);
    f2 g0 = f2{0.0f, 0.0f}, g1 = g0, cp0 = g0, icp = g0;
    if (dTc) {
      g0 = h_grad(q + 2 * n + 2, y0);
      g1 = h_grad(q + 2 * n + 8, y1);
      cp0 = ld(q + 2 * n);
      icp = f2_rcp(ld(q + 2 * n + 1));
    }
    __syncwarp();
    if (lane < n) {
      st2(zl + lane, z1);
      st2(yp + lane, y1);
      st2(hg + lane, g1);
    }
    __syncwarp();
    // BC'(Y_k) of lane k; direction t = k + 1 sits one lane further (direction n of 32 species in lane 0's
    // second pass)
    const f2 ym = y0.h > 1e-12f ? y0 : f2_from(1e-12);
    const f2 bc = f2_mul(f2_root(ym, lamf, mpow, dl), f2_rcp(ym));
    for (int t0 = 0; t0 < ntan; t0 += 32) {
      const int t = t0 + lane;
      const int src = (t - 1) & 31;
      const f2 bcp = f2{__shfl_sync(0xffffffffu, bc.h, src), __shfl_sync(0xffffffffu, bc.l, src)};
      const f2 dh = f2{__shfl_sync(0xffffffffu, g0.h, src), __shfl_sync(0xffffffffu, g0.l, src)};
      if (t >= ntan) continue;
      const float* dOr = dO + (r * ntan + t) * lddo;
      f2 sj = f2{0.0f, 0.0f};
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        const float d = dOr[k], u = __fmul_rn(sdf[k], d);
        acc_fma(sj, ld(zl + k), f2{u, __fmaf_rn(sdf[k], d, -u)});
      }
      f2 zt = f2{0.0f, 0.0f};   // (dZ/du BC') / S of species t - 1
      if (t > 0) {
        zt = f2_mul(ld(zl + t - 1), bcp);
        acc_add(sj, zt);
      }
      sj = f2_neg(f2_fin(sj));
      f2 acc = f2{0.0f, 0.0f};
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        const float d = dOr[k], u = __fmul_rn(sdf[k], d);
        f2 jy = f2_fma(ld(yp + k), sj, f2_mul(ld(zl + k), f2{u, __fmaf_rn(sdf[k], d, -u)}));
        float o = jy.h;
        if (t == k + 1) {
          jy = f2_add(jy, zt);
          o = f2_addf(jy, -1.0f).h;
        }
        Jc[k * ntan + t] = o;
        if (dTc) acc_fma(acc, ld(hg + k), jy);
      }
      if (dTc) dTc[t] = f2_to_int(f2_mul(f2_sub(t == 0 ? cp0 : dh, f2_fin(acc)), icp));
    }
  }
}

// Dynamic shared memory of an EoS block of `threads` threads: constants and the per-thread
// double-float column of mass fractions (n words per thread, rounded up to whole pairs).
size_t eos_smem(const EosParams& P, int threads = kThreads) {
  return sizeof(double) * ((size_t)consts_words(P) + (size_t)(P.n + (P.n & 1)) * threads);
}

size_t eos_smem_post(const EosParams& P, int threads) {
  return sizeof(double) * ((size_t)consts_words_post(P) + (size_t)P.n * threads);
}

// Opts a kernel into more than 48 KB of dynamic shared memory, once per device.
template <auto Kern>
cudaError_t smem_optin() {
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!done[dev]) {
    e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    // these kernels are bound by their shared-memory columns: ask for the largest carveout
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(Kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    done[dev] = true;
  }
  return cudaSuccess;
}

// Blocks of Kern (threads threads, smem bytes) that fit on the device at once. Kept per device and
// species count, which fixes an instance's shared memory: it is what the block's size is chosen by.
template <auto Kern>
int64_t resident_blocks(int n, size_t smem, int threads) {
  static std::atomic<int> per_sm[64][kMaxSpecies + 1];
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int nb = (dev >= 0 && dev < 64) ? per_sm[dev][n].load(std::memory_order_relaxed) : 0;
  if (nb <= 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, Kern, threads, smem) != cudaSuccess ||
        nb <= 0) {
      cudaGetLastError();
      nb = 4;
    }
    if (dev >= 0 && dev < 64) per_sm[dev][n].store(nb, std::memory_order_relaxed);
  }
  return (int64_t)sms * nb;
}

// Grid of a grid-stride kernel: one wave of its resident blocks, fewer when there is less work.
template <auto Kern>
int grid_resident(int n, int64_t nmax, size_t smem, int threads = kThreads) {
  const int64_t need = std::max<int64_t>(1, (nmax + threads - 1) / threads);
  return (int)std::min(need, resident_blocks<Kern>(n, smem, threads));
}

int grid_for(int64_t nmax, int threads = kThreads) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t need = (nmax + threads - 1) / threads;
  int64_t cap = (int64_t)sms * 8;
  if (need < 1) need = 1;
  return (int)(need < cap ? need : cap);
}

// Whether an eos_pre or eos_post launch of at most nmax rows takes small blocks: while one wave of them
// holds the rows (a second one would cost more than the large blocks' fuller SMs save). Step of 20,011
// cells of 30 species 218 -> 192 us, of 50,021 cells 336 -> 285 us, of 4,096 cells of 9 species 82.6 ->
// 77.7 us; at 77,003 cells, beyond the wave, small blocks took 427 us against 408.
template <auto Kern>
bool small_blocks(int n, int64_t nmax, size_t smem) {
  return nmax <= resident_blocks<Kern>(n, smem, kSmallThreads) * kSmallThreads;
}

template <int NM, typename XT, int TH>
cudaError_t pre_launch(const EosParams& P, const RowMap& rows, const double* T, const double* p,
                       const double* Y, int64_t ldY, double* h0, double* Z, XT* x, int64_t ldx,
                       float xs, int32_t* status, cudaStream_t st, double* rho) {
  constexpr auto kern = eos_pre_kernel<NM, XT, TH>;
  cudaError_t e = smem_optin<kern>();
  if (e != cudaSuccess) return e;
  const size_t smem = eos_smem(P, TH);
  return pdl_launch(kern, grid_resident<kern>(P.n, rows.nmax, smem, TH), TH, smem, st, 1, P, rows, T, p, Y, ldY, h0, Z, x,
                    ldx, xs, status, rho);
}

template <int NM, typename XT>
cudaError_t pre_th(const EosParams& P, const RowMap& rows, const double* T, const double* p,
                   const double* Y, int64_t ldY, double* h0, double* Z, XT* x, int64_t ldx,
                   float xs, int32_t* status, cudaStream_t st, double* rho) {
  return small_blocks<eos_pre_kernel<NM, XT, kSmallThreads>>(P.n, rows.nmax, eos_smem(P, kSmallThreads))
             ? pre_launch<NM, XT, kSmallThreads>(P, rows, T, p, Y, ldY, h0, Z, x, ldx, xs, status, st, rho)
             : pre_launch<NM, XT, kThreads>(P, rows, T, p, Y, ldY, h0, Z, x, ldx, xs, status, st, rho);
}

template <int NM>
cudaError_t pre_nm(const EosParams& P, const RowMap& rows, const double* T, const double* p,
                   const double* Y, int64_t ldY, double* h0, double* Z, void* x, int xkind,
                   int64_t ldx, float xs, int32_t* status, cudaStream_t st, double* rho) {
  switch (xkind) {
    case kXBF16:
      return pre_th<NM>(P, rows, T, p, Y, ldY, h0, Z, (__nv_bfloat16*)x, ldx, xs, status, st, rho);
    case kXFP8:
      return pre_th<NM>(P, rows, T, p, Y, ldY, h0, Z, (__nv_fp8_e4m3*)x, ldx, xs, status, st, rho);
    default:
      return pre_th<NM>(P, rows, T, p, Y, ldY, h0, Z, (float*)x, ldx, xs, status, st, rho);
  }
}

template <int NM, int TH>
cudaError_t post_launch(const EosParams& P, const RowMap& rows, const float* O, int64_t ldo,
                        const double* h0, double* T, const double* p, double* Y, int64_t ldY,
                        const int32_t* pre_status, int32_t* cell_status, cudaStream_t st,
                        const Source& src) {
  constexpr auto kern = eos_post_kernel<NM, TH>;
  cudaError_t e = smem_optin<kern>();
  if (e != cudaSuccess) return e;
  const size_t smem = eos_smem_post(P, TH);
  return pdl_launch(kern, grid_resident<kern>(P.n, rows.nmax, smem, TH), TH, smem, st, 1, P, rows, O, ldo, h0, T, p, Y,
                    ldY, pre_status, cell_status, src);
}

template <int NM>
cudaError_t post_nm(const EosParams& P, const RowMap& rows, const float* O, int64_t ldo,
                    const double* h0, double* T, const double* p, double* Y, int64_t ldY,
                    const int32_t* pre_status, int32_t* cell_status, cudaStream_t st,
                    const Source& src) {
  return small_blocks<eos_post_kernel<NM, kSmallThreads>>(P.n, rows.nmax, eos_smem_post(P, kSmallThreads))
             ? post_launch<NM, kSmallThreads>(P, rows, O, ldo, h0, T, p, Y, ldY, pre_status, cell_status, st, src)
             : post_launch<NM, kThreads>(P, rows, O, ldo, h0, T, p, Y, ldY, pre_status, cell_status, st, src);
}

template <int NM>
cudaError_t transport_nm(const EosParams& P, int64_t n, const double* T, const double* p,
                         const double* Y, int64_t ldY, double* mu, double* lam, double* alpha,
                         cudaStream_t st) {
  cudaError_t e = smem_optin<transport_kernel<NM>>();
  if (e != cudaSuccess) return e;
  transport_kernel<NM><<<grid_for(n, kPropThreads), kPropThreads, eos_smem(P, kPropThreads), st>>>(
      P, n, T, p, Y, ldY, mu, lam, alpha);
  return cudaGetLastError();
}

template <int NM>
cudaError_t props_nm(const EosParams& P, int64_t n, const double* T, const double* p,
                     const double* Y, int64_t ldY, double* rho, double* h, double* cp, double* Z,
                     cudaStream_t st) {
  cudaError_t e = smem_optin<props_kernel<NM>>();
  if (e != cudaSuccess) return e;
  props_kernel<NM><<<grid_resident<props_kernel<NM>>(P.n, n, eos_smem(P)), kThreads, eos_smem(P), st>>>(
      P, n, T, p, Y, ldY, rho, h, cp, Z);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_eos_pre(const EosParams& P, const RowMap& rows, const double* T,
                           const double* p, const double* Y, int64_t ldY, double* h0,
                           double* Z, void* x, int xkind, int64_t ldx, float x_scale,
                           int32_t* status, cudaStream_t st, double* rho) {
  if (rows.nmax <= 0) return cudaSuccess;
  if (P.n <= 16)
    return pre_nm<16>(P, rows, T, p, Y, ldY, h0, Z, x, xkind, ldx, x_scale, status, st, rho);
  return pre_nm<32>(P, rows, T, p, Y, ldY, h0, Z, x, xkind, ldx, x_scale, status, st, rho);
}

template <int NM, int TH>
cudaError_t prepare_step(int xkind) {
  cudaError_t e = xkind == kXBF16  ? smem_optin<eos_pre_kernel<NM, __nv_bfloat16, TH>>()
                  : xkind == kXFP8 ? smem_optin<eos_pre_kernel<NM, __nv_fp8_e4m3, TH>>()
                                   : smem_optin<eos_pre_kernel<NM, float, TH>>();
  if (e == cudaSuccess) e = smem_optin<eos_pre_kernel<NM, float, TH>>();  // stage entry point
  return e == cudaSuccess ? smem_optin<eos_post_kernel<NM, TH>>() : e;
}

template <int NM>
cudaError_t prepare_nm(int xkind) {
  cudaError_t e = prepare_step<NM, kThreads>(xkind);
  if (e == cudaSuccess) e = prepare_step<NM, kSmallThreads>(xkind);
  if (e == cudaSuccess) e = smem_optin<props_kernel<NM>>();
  if (e == cudaSuccess) e = smem_optin<transport_kernel<NM>>();
  return e;
}

cudaError_t prepare_eos(const EosParams& P, int xkind) {
  cudaError_t e = P.n <= 16 ? prepare_nm<16>(xkind) : prepare_nm<32>(xkind);
  if (e == cudaSuccess) e = P.n <= 16 ? smem_optin<jac_state_kernel<16>>() : smem_optin<jac_state_kernel<32>>();
  return e;
}

cudaError_t launch_jac_scale(const EosParams& P, int64_t ncell, const double* Y, int64_t ldY,
                             float* sc, cudaStream_t st) {
  if (ncell <= 0) return cudaSuccess;
  jac_scale_kernel<<<grid_for(ncell * (P.n + 1)), kThreads, 0, st>>>(P, ncell, Y, ldY, P.norm, sc);
  return cudaGetLastError();
}

cudaError_t launch_jac_tangent0(int64_t ncell, int ntan, int N1, const float* sc, const float* W1T,
                                const void* G1, int64_t ldg, bool bf16, void* dH, int64_t ldh,
                                cudaStream_t st) {
  if (ncell <= 0) return cudaSuccess;
  if ((ldg & 7) || (ldh & 7)) return cudaErrorInvalidValue;
  // kTanCells cells per block, a thread per group of eight columns
  const int groups = (N1 + 7) / 8;
  const int threads = std::min(256, (groups + 31) / 32 * 32);
  const int64_t g = (ncell + kTanCells - 1) / kTanCells;
  if (g > 0x7FFFFFFF) return cudaErrorInvalidValue;
  if (bf16)
    jac_tangent0_kernel<__nv_bfloat16, __nv_bfloat16><<<(unsigned)g, threads, 0, st>>>(
        ncell, ntan, N1, sc, W1T, (const __nv_bfloat16*)G1, ldg, (__nv_bfloat16*)dH, ldh);
  else
    jac_tangent0_kernel<float, float><<<(unsigned)g, threads, 0, st>>>(ncell, ntan, N1, sc, W1T,
                                                             (const float*)G1, ldg, (float*)dH, ldh);
  return cudaGetLastError();
}

cudaError_t launch_jac_post(const EosParams& P, int64_t ncell, int64_t cell0, const double* T,
                            const double* p, const double* Y, int64_t ldY, const float* O,
                            int64_t ldo, const float* dO, int64_t lddo, const double* h0, float* J,
                            double* dTn, double* scr, int32_t* cst, cudaStream_t st) {
  if (ncell <= 0) return cudaSuccess;
  const size_t smem = eos_smem(P, kPropThreads);
  const int g = grid_for(ncell, kPropThreads);
  float2* row = reinterpret_cast<float2*>(scr);
  const unsigned cg = (unsigned)std::min<int64_t>((ncell + kColWarps - 1) / kColWarps, grid_for(INT64_MAX / 2));
  if (P.n <= 16) {
    jac_state_kernel<16><<<g, kPropThreads, smem, st>>>(P, ncell, cell0, T, p, Y, ldY, O, ldo, h0, dTn != nullptr,
                                                        row, cst);
    jac_columns_kernel<16><<<cg, 32 * kColWarps, 0, st>>>(P, ncell, cell0, Y, ldY, dO, lddo, row, cst, J, dTn);
  } else {
    jac_state_kernel<32><<<g, kPropThreads, smem, st>>>(P, ncell, cell0, T, p, Y, ldY, O, ldo, h0, dTn != nullptr,
                                                        row, cst);
    jac_columns_kernel<32><<<cg, 32 * kColWarps, 0, st>>>(P, ncell, cell0, Y, ldY, dO, lddo, row, cst, J, dTn);
  }
  return cudaGetLastError();
}

cudaError_t launch_eos_post(const EosParams& P, const RowMap& rows, const float* O, int64_t ldo,
                            const double* h0, double* T, const double* p, double* Y,
                            int64_t ldY, const int32_t* pre_status, int32_t* cell_status,
                            cudaStream_t st, const Source* src) {
  if (rows.nmax <= 0) return cudaSuccess;
  const Source s = src ? *src : Source{nullptr, 0, nullptr, 0.0, nullptr};
  if (P.n <= 16)
    return post_nm<16>(P, rows, O, ldo, h0, T, p, Y, ldY, pre_status, cell_status, st, s);
  return post_nm<32>(P, rows, O, ldo, h0, T, p, Y, ldY, pre_status, cell_status, st, s);
}

cudaError_t launch_props(const EosParams& P, int64_t n, const double* T, const double* p,
                         const double* Y, int64_t ldY, double* rho, double* h, double* cp,
                         double* Z, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (P.n <= 16) return props_nm<16>(P, n, T, p, Y, ldY, rho, h, cp, Z, st);
  return props_nm<32>(P, n, T, p, Y, ldY, rho, h, cp, Z, st);
}

cudaError_t launch_transport(const EosParams& P, int64_t n, const double* T, const double* p,
                             const double* Y, int64_t ldY, double* mu, double* lam, double* alpha,
                             cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (P.n <= 16) return transport_nm<16>(P, n, T, p, Y, ldY, mu, lam, alpha, st);
  return transport_nm<32>(P, n, T, p, Y, ldY, mu, lam, alpha, st);
}

// Cells the step's eos_pre launch covers in one pass of its resident blocks (SMs x blocks per
// SM x threads); 0 if the occupancy query fails.
int64_t eos_wave_cells(const EosParams& P, int xkind) {
  const size_t smem = eos_smem(P);
  auto wave = [&](auto kern) -> int64_t {
    int nb = 0, dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kThreads, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return (int64_t)sms * nb * kThreads;
  };
  if (P.n <= 16)
    return xkind == kXBF16 ? wave(eos_pre_kernel<16, __nv_bfloat16, kThreads>)
           : xkind == kXFP8 ? wave(eos_pre_kernel<16, __nv_fp8_e4m3, kThreads>) : wave(eos_pre_kernel<16, float, kThreads>);
  return xkind == kXBF16 ? wave(eos_pre_kernel<32, __nv_bfloat16, kThreads>)
         : xkind == kXFP8 ? wave(eos_pre_kernel<32, __nv_fp8_e4m3, kThreads>) : wave(eos_pre_kernel<32, float, kThreads>);
}

}  // namespace dfgb
