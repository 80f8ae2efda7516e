// tcgen05, TMA and mbarrier primitives (inline PTX) shared by the tensor-core kernels of mlp_tc.cu
// and mlp_split.cu, and the walk over a persistent kernel's work items.
#pragma once

#include "dfgb_internal.cuh"

namespace dfgb {
namespace {

constexpr int BM = 128;
constexpr int kRowBytes = 128;                 // K bytes per stage row (one swizzle span)
constexpr long long kWaitBudget = 2000000000LL;  // ~1 s of SM clocks per wait
constexpr int kSmemLimit = 232448;             // opt-in dynamic shared memory per block
constexpr uint32_t kSuspendNs = 200000;        // try_wait may park the thread this long

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity,
                                         uint32_t suspend = kSuspendNs) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(suspend)
      : "memory");
  return ok != 0;
}

// Bounded wait: true when the phase of the given parity completed; false after the clock
// budget or once another role of the CTA has given up (*abort set).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort,
                                          int* err, long long budget, uint32_t suspend) {
  if (mbar_try(bar, parity, suspend)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try(bar, parity, suspend)) return true;
    if (*abort) return false;
    if (clock64() - t0 > budget) {
      atomicOr(err, kErrTimeout);
      *abort = 1;
      return false;
    }
  }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 B
// apart (stride byte offset), leading byte offset unused for this layout, version 1.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor: FP32 accumulator, K-major A and B, M = 128 (256 for a CTA pair),
// N = BN (N / 8 in bits 17..22; BN = 0 leaves the field for a width chosen at run time).
template <bool FP8, int BN, int MROWS = BM>
__device__ constexpr uint32_t idesc() {
  return (1u << 4) | (FP8 ? 0u : ((1u << 7) | (1u << 10))) | ((uint32_t)(BN >> 3) << 17) |
         ((uint32_t)(MROWS >> 4) << 24);
}

// MN-major operands (the product's row or column index runs along memory): instruction-descriptor
// bits, and the descriptor of a 128-byte-swizzled tile made of boxes of 64 columns x 64 rows (k) of
// BF16, 128 bytes a row: 8-row groups 1024 B apart (stride byte offset), the next 64 columns one box
// (leading byte offset) further.
constexpr uint32_t kIdescMnA = 1u << 15, kIdescMnB = 1u << 16;
constexpr int kMnBox = 64 * 128;
__device__ __forceinline__ uint64_t desc_mn128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kMnBox >> 4) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

template <bool FP8>
__device__ __forceinline__ void mma_issue(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t id,
                                          uint32_t accum) {
  if (FP8) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accum)
        : "memory");
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accum)
        : "memory");
  }
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

// ---- CTA pairs (cta_group::2) ----
// Two CTAs of a cluster compute one 256-row tile: each holds its own 128 rows of A and half of
// the tile's BN rows of W in shared memory, the even CTA issues M = 256 MMAs that read both
// CTAs' operands and write each CTA's 128 accumulator rows into that CTA's tensor memory. Each
// SM then streams 128 + BN/2 operand rows per k-block for BN columns of MMA work instead of
// 128 + BN.

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Shared::cluster address of the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
}

// Arrival on a barrier of the peer CTA (release at cluster scope).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity,
                                                 uint32_t suspend = kSuspendNs) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(suspend)
      : "memory");
  return ok != 0;
}

// Bounded wait on a barrier that also receives arrivals from the peer CTA.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity,
                                                  volatile int* abort, int* err, long long budget,
                                                  uint32_t suspend) {
  if (mbar_try_cluster(bar, parity, suspend)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_cluster(bar, parity, suspend)) return true;
    if (*abort) return false;
    if (clock64() - t0 > budget) {
      atomicOr(err, kErrTimeout);
      *abort = 1;
      return false;
    }
  }
}

// TMA load into this CTA's shared memory whose completion is counted on a barrier of either
// CTA of the pair (bar_cluster: a shared::cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map,
                                                 uint32_t bar_cluster, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar_cluster)
      : "memory");
}

template <bool FP8>
__device__ __forceinline__ void mma_issue_pair(uint32_t dtmem, uint64_t a, uint64_t b,
                                               uint32_t id, uint32_t accum) {
  if (FP8) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accum)
        : "memory");
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accum)
        : "memory");
  }
}

// Arrives on the barrier at this offset in both CTAs of the pair once the MMAs issued so far
// have completed.
__device__ __forceinline__ void mma_commit_pair_both(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar), "h"((uint16_t)3)
      : "memory");
}

__device__ __forceinline__ void mma_commit_pair_local(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Starts loading 32 consecutive FP32 columns of this thread's TMEM lane into r; the values
// are valid only after tmem_wait(r).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

// Waits for this thread's outstanding TMEM loads; r is passed through so no use of it can be
// scheduled before the wait.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
        "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]),
        "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]),
        "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
        "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]),
        "+r"(r[31])
      :
      : "memory");
}

// Unit position in a staging row of RB bytes under the tensor map's swizzle: the 16-byte unit u
// of row r sits at u ^ swz(r), swz = (r >> 2) & 1 for 32-byte rows (32B swizzle), (r >> 1) & 3
// for 64-byte rows (64B swizzle), r & 7 for 128-byte rows (128B swizzle). Rows of eight
// consecutive lanes then cover all 32 banks.
template <int RB>
__device__ __forceinline__ int swz(int r) {
  return RB == 128 ? (r & 7) : (RB == 64 ? ((r >> 1) & 3) : ((r >> 2) & 1));
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"((uint64_t)map), "r"(x), "r"(y), "r"(src)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Waits until at most one bulk store group of this thread is still reading shared memory.
__device__ __forceinline__ void bulk_wait_read1() {
  asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}
// Waits until no bulk store group of this thread is still reading shared memory.
__device__ __forceinline__ void bulk_wait_read0() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// The grid stride of the work items in whole m units (q), n positions (r) and q mod tiles_n
// (rot). One copy per CTA, in shared memory: the epilogue warps have no registers to spare.
struct WalkStep {
  uint32_t q;
  int r, rot;
};

// Walks the work items t = first, first + step, ... of one CTA (or CTA pair). Item t lies in
// split t / (units_m tiles_n), m unit mu = (t mod units_m tiles_n) / tiles_n and n position
// r = t mod tiles_n; its n tile is r rotated by the m unit, (r + mu) mod tiles_n, so that the
// items one CTA visits a grid stride apart cycle through the n tiles (whose MMA widths differ
// when the last one is narrowed). The position advances by additions and compares: divisions
// per item cost the layers with short k loops a few per cent. Item counts fit in 32 bits (the
// launch checks).
struct ItemWalk {
  uint32_t mu;          // m unit within the split
  int split, r, rot;    // split, n position in the m unit, mu mod tiles_n
  __device__ __forceinline__ ItemWalk(uint32_t first, uint32_t units_m, int tiles_n) {
    if (units_m == 0) {
      mu = 0;
      split = 0x7FFFFFFF;   // no items
      r = rot = 0;
    } else {
      const uint32_t tiles_mn = units_m * (uint32_t)tiles_n;
      split = (int)(first / tiles_mn);
      const uint32_t rem = first - (uint32_t)split * tiles_mn;
      mu = rem / (uint32_t)tiles_n;
      r = (int)(rem - mu * (uint32_t)tiles_n);
      rot = (int)(mu % (uint32_t)tiles_n);
    }
  }
  __device__ __forceinline__ int nt(int tiles_n) const {
    const int x = r + rot;
    return x < tiles_n ? x : x - tiles_n;
  }
  __device__ __forceinline__ void next(const WalkStep& st, uint32_t units_m, int tiles_n) {
    mu += st.q;
    r += st.r;
    rot += st.rot;
    if (rot >= tiles_n) rot -= tiles_n;
    if (r >= tiles_n) {
      r -= tiles_n;
      ++mu;
      if (++rot == tiles_n) rot = 0;
    }
    if (mu >= units_m) {   // into a later split
      split += (int)(mu / units_m);
      mu %= units_m;
      rot = (int)(mu % (uint32_t)tiles_n);
    }
  }
};

}  // namespace
}  // namespace dfgb
