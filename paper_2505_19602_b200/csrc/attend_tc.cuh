// Tensor-core attention over the paged store for bf16, head_dim 128 (Sec. 3.3, Eq. 5):
// O = softmax(scale * Q K^T) V with online softmax.  A CTA's work is one of
//   a pair   : two 128-query tiles (A, B) of one slice; every key tile is streamed once for both;
//   a single : one 128-query tile.  A and B are then the same queries against the even and against the odd key tiles, and
//              the two partial results are combined at the end.  A single takes 0.55 of a pair's time, so it serves a map's
//              last odd tile, launches that do not fill the GPU with pairs, and a launch's last, partial wave (see
//              AttendTc::launch).  Where singles leave SMs idle as well, the CTAs of a cluster share a single's key tiles
//              and combine through distributed shared memory.
//
// Roles inside a CTA of 384 threads:
//   warp 0 (one thread) : TMA producer.  The query tiles once; then per 128-key tile the K and V rows into
//                         128B-swizzled shared memory: first the tiles of a not yet appended current map from the caller's
//                         tensors (those loads need neither the cache length nor the page table and go out while the
//                         length is still being read), then the history tiles page by page through the page table.
//   warp 1 (one thread) : tcgen05.mma issuer; owns the TMEM allocation (512 columns: two S/P buffers
//                         and two O accumulators).  The issue order is
//                         S_A(0), S_B(0), then per step j  PV_A(j), S_A(j+1), PV_B(j), S_B(j+1): while one
//                         tile's softmax runs, the tensor pipe works for the other tile, and a tile's next S
//                         product follows its PV product without a wait in between.
//   warps 4-7, 8-11     : softmax, one warpgroup per query tile (warps 4-7 tile A, warps 8-11 tile B), one
//                         thread per query row (TMEM lane), so that no row state is shared between threads and
//                         the two tiles' chains  S -> softmax -> PV  run concurrently, each hiding the other's
//                         hand-over latencies.  A thread sweeps its row of an S tile once, in four chunks of 32
//                         columns (tcgen05.ld), software-pipelined: p = exp2(s * c - m) of chunk cc + 1 against
//                         a lazy reference m (packed f32x2 arithmetic, in place) is issued before chunk cc is
//                         summed, checked and written as bf16 pairs over the first 64 columns of the row's S
//                         buffer (tcgen05.st; a chunk's P only covers columns already read), from where the PV
//                         product takes its A operand.  Only when a chunk's sum shows that an exponent left
//                         the lazy band (2^8) does the warp raise the reference: the chunk is recomputed, the
//                         P chunks already stored for this tile, the running sum and the O accumulator are
//                         scaled down, and the exponentials taken ahead for the next chunk are taken again.  Threads that own a row of the observation window also
//                         store that row's raw products (16-byte stores, key tile j in columns 128 j ..) for
//                         the compress that follows.  At the end every warp normalises its rows of the O tile and sends
//                         them out through its part of the query tile's shared memory; the two parts of a single are
//                         merged on the way, a cluster's parts by all warps afterwards.
//   warps 2-3           : append.  When the current map has not been copied into the store yet, its K/V
//                         tiles come from the caller's tensors, and the CTA whose turn it is writes each
//                         tile's rows from shared memory to the slice's pages (and their original
//                         positions), so the copy costs no extra read and stays off the critical path.
// What bounds it: a CTA's steps are two chains  S -> softmax -> P V  that take turns on the tensor pipe, 3 290 cycles per step
// of a pair (2 048 at the tensor peak; 3 480 while the MMA warp still formed its descriptors between the arrival of P and the
// issue).  Around the steps a CTA costs ~8 000 cycles: 3 400 to the first scores (4 440 before the queries and the first key
// tile were requested ahead of the length, with the tensor maps' descriptors prefetched), ~2 000 from the last product to the
// last row (the bulk stores and the wait for them took ~1 000 more), the launch of the next CTA 1 300.
// 128 slices x 4 096 queries: 1 052 -> 1 030 us per launch.
// Every mbarrier wait is bounded; a wait that gives up raises the sticky device status, sets a
// CTA-wide abort flag and all roles fall through to the common exit where TMEM is released.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <map>
#include <mutex>
#include <type_traits>
#include <string>

#include "common.cuh"

namespace scalekv {
namespace tc {

constexpr int kChunks = 4;                       // tcgen05.ld x32 loads per softmax thread (= query row) and S tile
// With two query tiles a PV product is issued in two parts: the steps over the keys of the first kEarlyChunks chunks
// as soon as their P is stored, under the sweep of the remaining chunks, and the rest when the tile's P is complete.
// What stands between the end of a sweep and the tile's next S tile is then 2 (4 - kEarlyChunks) + 8 MMAs, not 16.
constexpr int kEarlyChunks = 3;
static_assert(kEarlyChunks >= 1 && kEarlyChunks < kChunks, "both parts of a PV product need at least one chunk");
constexpr int kThreads = 128 + 2 * 128;          // warps: TMA, MMA, 2 x append, one softmax warpgroup per query tile
constexpr int kStages = 5;                       // one ring for the K and V tiles: K_0, V_0, K_1, V_1, ...
constexpr uint32_t kTileBytes = 128 * 128 * 2;   // one 128 x 128 bf16 operand tile
constexpr uint32_t kHalfBytes = kTileBytes / 2;  // 64 head-dim columns = one 128-byte swizzle span
constexpr uint32_t kOffQ = 0;                    // two query tiles (the dynamic shared memory must start 1024-byte aligned)
constexpr uint32_t kOffRing = kOffQ + 2 * kTileBytes;
constexpr uint32_t kOffBar = kOffRing + kStages * kTileBytes;
constexpr uint32_t kOffStat = kOffBar + 256;     // a shared single's rows: reference and sum of part A, of part B
constexpr uint32_t kSmemBytes = kOffStat + 2 * 128 * 8;
static_assert(kSmemBytes <= 232448, "more shared memory than a CTA can have");
// barrier slots (8 bytes each): one full/empty pair per ring stage, one S/P/PV barrier per S buffer or query tile
enum { bQFull = 0, bFull = 2, bEmpty = bFull + kStages, bSFull = bEmpty + kStages, bPFull = bSFull + 2, bPvDone = bPFull + 2,
       bFinal = bPvDone + 2, bPEarly = bFinal + 2, bPvEarly = bPEarly + 2, bCount = bPvEarly + 2 };
constexpr uint32_t kOffTmemSlot = 208;            // inside the barrier area, behind the barriers
static_assert(bCount * 8 <= kOffTmemSlot, "barriers overlap the TMEM slot");
static_assert(bCount <= 32, "one lane of the first warp initialises each barrier");
constexpr int kMaxSplit = 8;                      // CTAs that may share a single's keys (portable cluster size)
// where the CTAs of a cluster leave the parts of the rows that this one finishes (up to 128 + kMaxSplit - 1 rows of 512 bytes),
// and their references and sums
constexpr uint32_t kOffPartStat = kOffRing + (128 + kMaxSplit) * 512;
static_assert(kOffPartStat + (128 + kMaxSplit) * 8 <= kOffRing + kStages * kTileBytes, "the parts have to fit the ring");
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0, kColO = 256;       // S/P buffers at 0 and 128, O accumulators at 256 and 384
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false when the CTA is aborting or the time limit ran out (status raised).
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                                            unsigned long long limit_ns = kWaitLimitNs) {
  const unsigned long long t0 = globaltimer();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try(bar, parity)) return true;
    if (*abort_flag || *reinterpret_cast<volatile int *>(status) != 0) return false;
    if (globaltimer() - t0 > limit_ns) {
      *abort_flag = 1;
      atomicExch(status, kDevTimeout);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status) {
  if (mbar_try(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, abort_flag, status);
}
// For a CTA that gives up: waits for a copy of its own that is still under way, whatever the status, a second at most.
__device__ __noinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
  const unsigned long long t0 = globaltimer();
  while (!mbar_try(bar, parity) && globaltimer() - t0 < kWaitLimitNs / 2) {}
}
// Self-test of the bounded wait (scalekv_selftest_wait): one warp waits, with the given limit, on a barrier
// that nobody ever arrives at.  The wait must give up, raise the sticky status and return; a second warp that
// polls the CTA's abort flag (also bounded) shows that the other roles of a CTA see the give-up.
// out[0] = 1 when the wait returned false, out[1] = 1 when the second warp saw the abort flag.
__global__ void wait_probe_kernel(int *status, unsigned long long limit_ns, int *out) {
  __shared__ __align__(8) unsigned long long probe_bar;
  __shared__ int abort_word;
  const uint32_t bar = smem_u32(&probe_bar);
  if (threadIdx.x == 0) {
    abort_word = 0;
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  volatile int *abort_flag = &abort_word;
  if (threadIdx.x == 0) {
    const bool ok = mbar_try(bar, 0) || mbar_wait_slow(bar, 0, abort_flag, status, limit_ns);
    out[0] = ok ? 0 : 1;
  } else if (threadIdx.x == 32) {
    const unsigned long long t0 = globaltimer();
    int seen = 0;
    while (!seen && globaltimer() - t0 < 4 * limit_ns + 1000000ull) seen = *abort_flag;
    out[1] = seen;
  }
}
// Same, with a warp-uniform result (the callers go on to warp-collective tcgen05 instructions).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status));
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *tm, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
               "l"(tm), "r"(x), "r"(y), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *tm, int x, int y, int z, int w, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
// (orders nothing, and so does not wait for this thread's stores)
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// True in exactly one lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// The 64-bit shared-memory descriptors are passed as (low word, high word): the low word holds the
// start address field, so stepping through a tile is one 32-bit add per operand.
// Eight back-to-back MMAs of one 128 x 128 x 128 product, issued by the elected lane of a converged
// warp; the descriptors' start addresses advance by constant steps.  SS: both operands in shared
// memory (K-major tiles: steps of 32 B inside a 64-column half, then the next half).
__device__ __forceinline__ void tc_mma_ss_x8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred e, pf, pt;\n\t.reg .b64 da, db;\n\t.reg .b32 al, bl;\n\t"
      "elect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 pf, 0, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pf;\n\t"
      "add.u32 al, %1, 2;\n\tadd.u32 bl, %2, 2;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 4;\n\tadd.u32 bl, %2, 4;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 6;\n\tadd.u32 bl, %2, 6;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 1024;\n\tadd.u32 bl, %2, 1024;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 1026;\n\tadd.u32 bl, %2, 1026;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 1028;\n\tadd.u32 bl, %2, 1028;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 1030;\n\tadd.u32 bl, %2, 1030;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "}" ::"r"(d_tmem),
      "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc)
      : "memory");
}
// TS: A = P in TMEM (16 keys = 8 columns per step; a row's 128 bf16 values of P fill the first 64 columns of
// its S buffer), B = V in shared memory as the MN-major operand (16 keys = 2048 B per step).
__device__ __forceinline__ constexpr uint32_t p_col(int kk) { return (uint32_t)(kk * 8); }
// The first N of the eight steps (a_tmem and b_lo address the first of them).
template <int N>
__device__ __forceinline__ void tc_mma_ts_n(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                            uint32_t accumulate_first) {
  static_assert(N >= 1 && N <= 8, "one to eight steps");
  asm volatile(
      "{\n\t.reg .pred e, pf, pt, q;\n\t.reg .b64 db;\n\t.reg .b32 at, bl, nn;\n\t"
      "elect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 pf, %5, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\tmov.u32 nn, %13;\n\t"
      "mov.b64 db, {%2, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, pf;\n\t"
      "setp.gt.and.u32 q, nn, 1, e;\n\tadd.u32 at, %1, %6;\n\tadd.u32 bl, %2, 128;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "setp.gt.and.u32 q, nn, 2, e;\n\tadd.u32 at, %1, %7;\n\tadd.u32 bl, %2, 256;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "setp.gt.and.u32 q, nn, 3, e;\n\tadd.u32 at, %1, %8;\n\tadd.u32 bl, %2, 384;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "setp.gt.and.u32 q, nn, 4, e;\n\tadd.u32 at, %1, %9;\n\tadd.u32 bl, %2, 512;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "setp.gt.and.u32 q, nn, 5, e;\n\tadd.u32 at, %1, %10;\n\tadd.u32 bl, %2, 640;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "setp.gt.and.u32 q, nn, 6, e;\n\tadd.u32 at, %1, %11;\n\tadd.u32 bl, %2, 768;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "setp.gt.and.u32 q, nn, 7, e;\n\tadd.u32 at, %1, %12;\n\tadd.u32 bl, %2, 896;\n\tmov.b64 db, {bl, %3};\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "}" ::"r"(d_tmem),
      "r"(a_tmem), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate_first), "n"(p_col(1)), "n"(p_col(2)), "n"(p_col(3)), "n"(p_col(4)),
      "n"(p_col(5)), "n"(p_col(6)), "n"(p_col(7)), "n"(N)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float *v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const float *v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
      "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])),
      "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])), "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])),
      "r"(__float_as_uint(v[20])), "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])),
      "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])), "r"(__float_as_uint(v[27])),
      "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])), "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
      : "memory");
}
// 16 consecutive 32-bit columns (32 bf16 values of P) of this thread's TMEM lane
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t *r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t *v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]),
      "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// packed pairs of fp32 in one 64-bit register
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Shared-memory matrix descriptor, 128-byte swizzle, operand tiles whose 8-row groups are 1024 B
// apart.  K-major operands (Q, K): rows of 128 B, the leading offset is not used.  MN-major
// operand (V as [key][d]): 64 d-columns are contiguous, the next 64 start `lbo` bytes further.
// Low word: start address >> 4 (bits 0-13), leading byte offset >> 4 (bits 16-29).
// High word: stride byte offset >> 4 (bits 0-13), descriptor version (bit 14), swizzle mode (bits 29-31).
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo_bytes) {
  return ((saddr & 0x3FFFFu) >> 4) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
__host__ __device__ constexpr uint32_t desc_hi(uint32_t sbo_bytes) {
  return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14) | (2u << 29);
}
// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = 128, A K-major; B K-major or MN-major.
__host__ __device__ constexpr uint32_t instr_desc(bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
}

// Rare path of the softmax, taken by a whole warp when the sum of one of its rows' chunks shows that an
// exponent left the lazy band.  The chunk's 32 raw products are still intact in the row's S buffer (chunk cc
// sits in columns [32 cc, 32 cc + 32) of s_addr, the P chunks stored so far only cover columns below 16 cc) and
// are read again; `valid` of them are real keys.  Per lane the reference moves up to the chunk's maximum if
// that is larger (a lane that needs nothing gets the factor 1): the chunk's P is recomputed against the new
// reference and stored, and everything accumulated under the old one is multiplied by f = 2^(old - new): the
// running row sum, the P chunks p_first .. cc-1 stored for this tile that the tensor core has not been given yet
// (16 columns each), and - once the product that `pv_bar` stands for has landed: the previous PV product of the
// tile, or the early part of this one when its chunks have been handed over - the row's 128 columns of the O
// accumulator at o_addr.
// Everything goes in and out by value so that the caller's state stays in registers.
struct Raised { float m, l, sum; int o_landed, ok; };
__device__ __noinline__ Raised raise_reference(int valid, float c, float m, float l_run, uint32_t s_addr, int cc, int p_first,
                                               uint32_t o_addr, int with_o, int o_landed, uint32_t pv_bar, uint32_t pv_parity,
                                               volatile int *abort_flag, int *status) {
  float x[32];
  tc_ld32(s_addr + cc * 32, x);
  tc_wait_ld();
  float mt = -INFINITY;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (i < valid) mt = fmaxf(mt, x[i]);
  const float m_new = fmaxf(m, mt * c);
  const float f = ex2(m - m_new);
  float sum = 0.f;
  uint32_t pk[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float p0 = (2 * i < valid) ? ex2(fmaf(x[2 * i], c, -m_new)) : 0.f;
    const float p1 = (2 * i + 1 < valid) ? ex2(fmaf(x[2 * i + 1], c, -m_new)) : 0.f;
    sum += p0 + p1;
    pk[i] = pack_bf16(p0, p1);
  }
  tc_st16(s_addr + cc * 16, pk);
#pragma unroll 1
  for (int e = p_first; e < cc; ++e) {
    uint32_t r[16];
    tc_ld16(s_addr + e * 16, r);
    tc_wait_ld();
#pragma unroll
    for (int i = 0; i < 16; ++i)
      r[i] = pack_bf16(__uint_as_float(r[i] << 16) * f, __uint_as_float(r[i] & 0xffff0000u) * f);
    tc_st16(s_addr + e * 16, r);
  }
  if (with_o) {
    if (!o_landed) {
      if (!mbar_wait_warp(pv_bar, pv_parity, abort_flag, status)) return {m_new, l_run * f, sum, 0, 0};
      tc_fence_after();
      o_landed = 1;
    }
#pragma unroll 1
    for (int e = 0; e < 4; ++e) {
      float o[32];
      tc_ld32(o_addr + e * 32, o);
      tc_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) o[i] *= f;
      tc_st32(o_addr + e * 32, o);
    }
  }
  tc_wait_st();
  return {m_new, l_run * f, sum, o_landed, 1};
}

// Division of numbers below 2^21 (the plan sees to that) by a divisor below 2^21 the quick way (the remainder of 2^42 costs less than one quotient):
// a CTA finds its item with three of these, and its first loads wait for it.
constexpr long long kMaxItems = 1ll << 21;
struct Divisor {
  unsigned long long mul;
  int d;
  static Divisor of(int d) { return {(1ull << 42) / (unsigned)d + 1, d}; }
  __device__ __forceinline__ int div(int x) const { return (int)(((unsigned long long)(unsigned)x * mul) >> 42); }
};

struct Params {
  LayerView lv;
  TensorView O;
  float *lse;
  int n_k;
  int n_pair;          // items [0, n_pair) walk the slices pair by pair, the others tile by tile
  int cut_tile;        // tiles (of all slices) that the first n_pair items cover
  Divisor per_pair, per_tile, per_heads;   // items of a slice pair by pair, tiles of a slice, heads
  float scale_log2e;   // softmax scale * log2(e)
  int box_rows;        // rows per K/V TMA box = min(page_tokens, 128)
  int fused_append;    // 1: the current map's K/V rows are still in the caller's tensors; read them there
  int copy_in;         // 1: and copy them into the pages on the way
  int n_prev;          // original position of the current map's first token
  // observation window (Sec. 3.3): when win_logits is not null, the raw products <q, k> of the w window rows
  // against every cache entry are recorded in win_logits[slice][rank][column], column = 128 j + position in key tile j
  float *win_logits;
  float *win_lse;      // [slice][rank]: base-2 log-sum-exp of each window row's logits (its softmax normaliser)
  int ld_l;            // leading dimension of a logit row
  int w;
  int win_pos[kMaxWindow];   // ascending raster indices of the window rows inside the current map
};

// a / b for 0 <= a < 256 and 0 < b <= 128 (the true quotient of a + 1/2 is 1 / 256 or more from any integer, the approximate
// one a few units in the last place from the true one)
__device__ __forceinline__ int small_div(int a, int b) { return (int)__fdividef((float)a + 0.5f, (float)b); }
// rows that each CTA of a cluster finishes
__device__ __forceinline__ int cluster_share(int n_k, int first_row, int n_split) { return small_div(min(128, n_k - first_row) + n_split - 1, n_split); }
__device__ __forceinline__ uint32_t remote(uint32_t addr, int cta) {
  uint32_t ra;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(cta));
  return ra;
}

// The end of a softmax warp's work, behind its last sweep: 32 rows of O with references m and sums l are normalised and stored
// (have: there were keys for this tile and all have been swept; whole: nothing has been given up so far).  A function of its own so that the sweep's
// registers are not allocated around it.  window: this thread's row belongs to the observation window.
// A row that lacks a product, because some wait for it has run out, is left as it is: its accumulator and its query tile may still be in use.
// What a row needs besides its columns (log-sum-exp, addresses, the place of a window row) is worked out before the last product is
// waited for, which a row's log-sum-exp does not depend on, and the two parts of a shared single are read from TMEM at once.  us per launch of 16
// slices, a map in the pages, averages over sizes, worked out behind the wait and 32 columns at a time / so: 16-128 queries behind 21 entries 10.89 /
// 10.58, 520-1 024 behind 210 20.84 / 20.46; where a cluster shares the keys the code that runs once costs what it saves, 130-512 behind 209
// 16.05 / 16.07 (single sizes up to 3 % longer: 400 queries with their step 11.9 / 12.3), of 32 slices 16.68 / 16.57; 128 x 1 600: 206.1 / 204.7.
// The instance that records a window is scheduled anew with every change here: 32 columns at a time in clusters alone (15.83, 16.46) made its
// sweep 2-3 % slower at 4 096 queries and more, as did a pair's last tile shared by both warpgroups, the sums kept behind the wait 0.4 %, and
// a flag set in mbar_wait_slow for waits that end by the status 1 %.
__device__ __forceinline__ void finish_rows(const Params &prm, uint32_t base, uint32_t lane_addr, int slice, int first_row, int qt, bool pair,
                                         bool shared, bool have, bool whole, int n_split, float m, float l, bool window, volatile int *abort_flag,
                                         int *status) {
  const int n_k = prm.n_k;
  const int lane = threadIdx.x & 31, quarter = (threadIdx.x >> 5) & 3, row = quarter * 32 + lane;
  // Output rows leave through shared memory, so that a store instruction writes whole 64- or 128-byte pieces (a row written by its own
  // thread straight from the registers touches 32 lines per instruction) and neither another warp nor an asynchronous copy has
  // to be waited for.  16-byte pieces are permuted by the row's index against bank conflicts.
  const int b = prm.per_heads.div(slice), h = slice - b * prm.per_heads.d;
  const int r_own = first_row + (pair ? qt * 128 : 0) + row;             // this thread's row of its own tile
  const uint32_t stage0 = base + kOffQ + qt * kTileBytes + quarter * 8192;     // (the last product has read the query tile before it is used)
  char *obase = const_cast<char *>(prm.O.ptr) + ((long long)b * prm.O.sb + (long long)h * prm.O.sh) * 2;
  // a barrier that completes exactly once, after a tile's last PV product: the per-tile PV barrier will not do, a parity wait
  // cannot tell phases two apart and this warp may be that far behind it
  auto final_product = [&](int t) {
    const bool ok = mbar_wait_warp(base + kOffBar + 8 * (bFinal + t), 0, abort_flag, status);
    tc_fence_after();
    return ok;
  };
  auto window_rank = [&] {
    int rank = -1;
    if (window)
      for (int e = 0; e < prm.w; ++e)
        if (prm.win_pos[e] == r_own) rank = e;
    return rank;
  };
  auto row_sums = [&](float mr, float lr) {              // what is kept of a row besides its output
    const float y = mr + log2f(lr);
    if (prm.lse != nullptr && r_own < n_k) prm.lse[(size_t)slice * n_k + r_own] = y * 0.6931471805599453f;
    const int rank = window_rank();
    if (rank >= 0) prm.win_lse[(size_t)slice * prm.w + rank] = y;
  };
  const uint32_t stat = base + kOffStat + (uint32_t)row * 8;             // of this row in tile A; tile B's lie 1024 bytes further
  if (!shared) {
    if (have) row_sums(m, l);
    if (have && final_product(qt)) {
      // 32 columns of the warp's 32 rows at a time (128 of a row's 256 bytes there), eight 64-byte pieces a store instruction
      const float inv = 1.f / l;
      const uint32_t o_addr = lane_addr + kColO + qt * 128;
      const int sub = lane >> 2, piece = lane & 3, w0 = r_own - lane;
      char *out = obase + (long long)(w0 + sub) * prm.O.st * 2 + piece * 16;
      auto slot = [](int r, int i) { return (uint32_t)r * 256 + (uint32_t)(((i ^ ((r >> 1) & 3)) + 4 * (r & 1)) << 4); };
      float o[2][32];
      tc_ld32(o_addr, o[0]);
#pragma unroll
      for (int cc = 0; cc < kChunks; ++cc) {
        uint32_t pk[16];
        tc_wait_ld();
        if (cc + 1 < kChunks) tc_ld32(o_addr + (cc + 1) * 32, o[(cc + 1) & 1]);
#pragma unroll
        for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(o[cc & 1][2 * i] * inv, o[cc & 1][2 * i + 1] * inv);
        const uint32_t stage = stage0 + (cc & 1) * 128;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stage + slot(lane, i)), "r"(pk[4 * i]),
                       "r"(pk[4 * i + 1]), "r"(pk[4 * i + 2]), "r"(pk[4 * i + 3])
                       : "memory");
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = 8 * i + sub;
          uint4 val;
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(val.x), "=r"(val.y), "=r"(val.z), "=r"(val.w)
                       : "r"(stage + slot(r, piece)) : "memory");
          if (w0 + r < n_k) *reinterpret_cast<uint4 *>(out + i * prm.O.st * 16 + cc * 64) = val;
        }
      }
    }
  } else {
    // ---- the two parts of a shared single are merged, half of the columns by each warpgroup: the rows of both lie in the
    // same TMEM lanes, so all that is handed over are the references and sums.  Here and in finish_cluster every instruction
    // runs once or twice per launch, so the code is kept short and what a row needs alone is worked out before the rendezvous
    // (with the parts handed over in shared memory, one row at a time per warp in finish_cluster and pushes of single pieces, a
    // step of 16 slices x 144 / 256 / 400 / 576 queries took 13.7 / 14.3 / 16.9 / 19.1 us; now 10.7 / 11.3 / 14.4 / 18.4).
    if (!have) { m = -INFINITY; l = 0.f; }
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(stat + (uint32_t)qt * 1024), "f"(m), "f"(l) : "memory");
    // of a cluster the rows' owner: it gets this CTA's merged part, unnormalised, with its reference and sum
    const int own_rows = n_split > 1 ? cluster_share(n_k, first_row, n_split) : 128, owner = min(small_div(row, own_rows), n_split - 1);   // (rows beyond the map go nowhere)
    const int at = (int)blockIdx.z * own_rows + row - owner * own_rows;      // and the row's place there
    const uint32_t dst = n_split > 1 ? remote(base + kOffRing + (uint32_t)at * 512 + (uint32_t)qt * 256, owner) : 0;
    const int rank = n_split > 1 ? window_rank() : -1;
    if (!whole || (have && !final_product(qt))) {          // (no sum is negative)
      l = -1.f;
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(stat + (uint32_t)qt * 1024 + 4), "f"(l) : "memory");
    }
    if (n_split > 1) cluster_arrive_relaxed();             // this CTA's ring is free (this warp has never touched it)
    tc_fence_before();
    asm volatile("bar.sync 2, 256;" ::: "memory");         // both accumulators are complete, no product reads the query tile any more
    tc_fence_after();
    float o[64], other[64];
    const uint32_t o_addr = lane_addr + kColO + qt * 64;
#pragma unroll
    for (int cc = 0; cc < 2; ++cc) {
      tc_ld32(o_addr + qt * 128 + cc * 32, o + cc * 32);
      tc_ld32(o_addr + (qt ^ 1) * 128 + cc * 32, other + cc * 32);
    }
    float m2, l2;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(m2), "=f"(l2) : "r"(stat + (uint32_t)(qt ^ 1) * 1024) : "memory");
    whole = !(l < 0.f || l2 < 0.f);                        // (the same for the warp's rows)
    const float M = fmaxf(m, m2);
    float f1 = l > 0.f ? ex2(m - M) : 0.f, f2 = l2 > 0.f ? ex2(m2 - M) : 0.f;
    const float both = l * f1 + l2 * f2;
    if (n_split == 1) {
      const float inv = 1.f / both;
      f1 *= inv; f2 *= inv;
      if (qt == 0 && whole) row_sums(M, both);
    }
    const bool none1 = !__any_sync(0xffffffffu, l > 0.f), none2 = !__any_sync(0xffffffffu, l2 > 0.f);   // a part without keys left garbage
    const uint64_t ff1 = pack2(f1, f1), ff2 = pack2(f2, f2);
    tc_wait_ld();
    if (none1) {
#pragma unroll
      for (int i = 0; i < 64; ++i) o[i] = 0.f;
    }
    if (none2) {
#pragma unroll
      for (int i = 0; i < 64; ++i) other[i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
      unpack2(fma2(pack2(o[2 * i], o[2 * i + 1]), ff1, mul2(pack2(other[2 * i], other[2 * i + 1]), ff2)), o[2 * i], o[2 * i + 1]);
    if (n_split == 1) {
      if (!whole) return;
      // four 128-byte pieces a store instruction
      const uint32_t stage = stage0 + qt * 4096, mine = stage + lane * 128;
      const int w0 = first_row + quarter * 32 + (lane >> 3);
      char *out = obase + (long long)w0 * prm.O.st * 2 + qt * 128 + (lane & 7) * 16;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(mine + (uint32_t)((i ^ (lane & 7)) << 4)), "r"(pack_bf16(o[8 * i], o[8 * i + 1])),
                     "r"(pack_bf16(o[8 * i + 2], o[8 * i + 3])), "r"(pack_bf16(o[8 * i + 4], o[8 * i + 5])), "r"(pack_bf16(o[8 * i + 6], o[8 * i + 7]))
                     : "memory");
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        uint4 val;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(val.x), "=r"(val.y), "=r"(val.z), "=r"(val.w)
                     : "r"(stage + (uint32_t)r * 128 + (uint32_t)(((lane & 7) ^ (r & 7)) << 4)) : "memory");
        if (w0 + 4 * i < n_k) *reinterpret_cast<uint4 *>(out + i * prm.O.st * 8) = val;
      }
    } else {
      // the warpgroup's half of the row, 16-byte pieces permuted by its index
      const uint32_t mine = base + kOffQ + qt * kTileBytes + row * 256;
      if (whole) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(mine + (uint32_t)((i & 8) << 4) + (uint32_t)(((i & 7) ^ (row & 7)) << 4)), "f"(o[4 * i]),
                       "f"(o[4 * i + 1]), "f"(o[4 * i + 2]), "f"(o[4 * i + 3]) : "memory");
      }
      __syncwarp();
      // Off to the owners: 256 contiguous bytes (this warpgroup's half of a row) by 16 lanes at a time; stores of 16-byte
      // pieces of 32 rows travel between SMs piece by piece.
      cluster_wait();                                     // every CTA of the cluster is through with its ring
      if (qt == 0 && r_own < n_k)
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(remote(base + kOffPartStat + (uint32_t)at * 8, owner)), "f"(M), "f"(whole ? both : -1.f)
                     : "memory");
      if (!whole) return;
      const int half = lane >> 4, p16 = lane & 15;
#pragma unroll 8
      for (int e = 0; e < 16; ++e) {
        const int r = 2 * e + half;
        const uint32_t to = __shfl_sync(0xffffffffu, dst, r) + (uint32_t)p16 * 16;
        float4 x;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
                     : "r"(mine + (uint32_t)((r - lane) * 256) + (uint32_t)((p16 ^ (r & 7)) << 4)) : "memory");
        if (r_own - lane + r < n_k)
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w) : "memory");
      }
      __syncwarp();
      if (qt == 0)                                        // (for the row's owner to find after the cluster's barrier)
        asm volatile("st.shared.s32 [%0], %1;" ::"r"(mine), "r"(rank) : "memory");
    }
  }
}

// The end of a cluster's work: O = sum_e 2^(m_e - M) O_e / sum_e 2^(m_e - M) l_e with M the largest reference, for this CTA's
// share of the rows, from the parts that the CTAs of the cluster have left here.  A warp takes four rows at a time, a lane
// 16 columns of one.
__device__ __forceinline__ void finish_cluster(const Params &prm, uint32_t base, int slice, int q_first, int n_split) {
  const int n_k = prm.n_k;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = prm.per_heads.div(slice), h = slice - b * prm.per_heads.d;
  const int own_rows = cluster_share(n_k, q_first, n_split), r_lo = (int)blockIdx.z * own_rows, r_hi = min(r_lo + own_rows, min(128, n_k - q_first));
  char *obase = const_cast<char *>(prm.O.ptr) + ((long long)b * prm.O.sb + (long long)h * prm.O.sh) * 2;
  static_assert(kMaxSplit == 8, "eight lanes weigh the parts of a row");
  const int sub = lane >> 3, part = lane & 7;
#pragma unroll 1                                           // (code that runs once costs its fetching: no copies of it)
  for (int r0 = r_lo + warp * 4; r0 < r_hi; r0 += kThreads / 8) {
    const bool live = r0 + sub < r_hi;
    const int r = live ? r0 + sub : r0, at = r - r_lo;
    // lane e of a row weighs part e (a part without keys counts for nothing: it left zeros)
    float m = -INFINITY, sum = 0.f;
    if (part < n_split)
      asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(m), "=f"(sum) : "r"(base + kOffPartStat + (uint32_t)(part * own_rows + at) * 8));
    const bool whole = !(__ballot_sync(0xffffffffu, sum < 0.f) & (0xffu << (8 * sub)));       // no part has been given up
    float M = m;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float weight = sum > 0.f ? ex2(m - M) : 0.f;
    sum *= weight;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = 0.f;
    const uint32_t src = base + kOffRing + (uint32_t)at * 512 + (uint32_t)part * 16;
#pragma unroll 1
    for (int e = 0; e < n_split; ++e) {
      const float f = __shfl_sync(0xffffffffu, weight, sub * 8 + e);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float4 x;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
                     : "r"(src + (uint32_t)(e * own_rows) * 512 + i * 128));
        a[4 * i] = fmaf(x.x, f, a[4 * i]); a[4 * i + 1] = fmaf(x.y, f, a[4 * i + 1]);
        a[4 * i + 2] = fmaf(x.z, f, a[4 * i + 2]); a[4 * i + 3] = fmaf(x.w, f, a[4 * i + 3]);
      }
    }
    if (live && whole) {
      const float inv = 1.f / sum;
      const int qi = q_first + r;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<uint2 *>(obase + (long long)qi * prm.O.st * 2 + part * 8 + i * 64) =
            make_uint2(pack_bf16(a[4 * i] * inv, a[4 * i + 1] * inv), pack_bf16(a[4 * i + 2] * inv, a[4 * i + 3] * inv));
      if (part == 0) {
        const float y = M + log2f(sum);
        if (prm.lse != nullptr) prm.lse[(size_t)slice * n_k + qi] = y * 0.6931471805599453f;
        int rank;
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(rank) : "r"(base + kOffQ + (uint32_t)r * 256));
        if ((unsigned)rank < (unsigned)prm.w) prm.win_lse[(size_t)slice * prm.w + rank] = y;
      }
    }
  }
}

// kWindow: the launch records the observation window's logits; the instance without that code serves the launches
// that record nothing (its mere presence costs every warp's sweep 2-3 %).
template <bool kWindow>
__global__ void __launch_bounds__(kThreads, 1)
attend_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmKc,
                 const __grid_constant__ CUtensorMap tmVc, const __grid_constant__ Params prm) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  uint8_t *base_ptr = smem_raw;
  const uint32_t bars = base + kOffBar;
  volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + kOffBar + kOffTmemSlot);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + kOffBar + kOffTmemSlot + 4);
  auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const LayerView &lv = prm.lv;
  const int n_k = prm.n_k;
  // This CTA's queries: slice by slice, so that CTAs that run together share a slice's K and V in L2, first pair by pair
  // (a slice's last odd tile is a single), then, behind the first n_pair items, tile by tile.
  const int tiles = (n_k + 127) >> 7;                    // query tiles of a slice
  const int e = (int)blockIdx.x - prm.n_pair;
  const int at = e < 0 ? (int)blockIdx.x : prm.cut_tile + e;
  const int slice = e < 0 ? prm.per_pair.div(at) : prm.per_tile.div(at);
  const int q_tile = e < 0 ? 2 * (at - slice * prm.per_pair.d) : at - slice * prm.per_tile.d;
  const bool pair = e < 0 && q_tile + 1 < tiles;
  const int b = prm.per_heads.div(slice), h = slice - b * prm.per_heads.d;
  const int q_first = q_tile * 128;                      // first query row of tile A
  const int n_split = gridDim.z;                         // CTAs (of a cluster) that share this item's keys
  // What needs no global memory comes first: the lanes of warp 0 initialise one barrier each, warp 1 allocates the
  // TMEM, warp 2 fetches the tensor maps' descriptors.  When the launch allows it (programmatic stream serialisation) this part runs while the kernel before this
  // one in the stream is still finishing; `griddepcontrol.wait` then holds every thread until that kernel's writes
  // - cache lengths, page tables, pages, the status word - are visible.  (The grid behind this one comes up when every
  // CTA of this grid has issued its last products: see there.)
  if (warp == 0) {
    if (lane < bCount) {
      // arrivals per phase: a ring stage is released by the MMA warp's commit and the two append warps; P and early P
      // are announced by one lane of each of the four warps of a softmax warpgroup
      const bool four = (lane >= bPFull && lane < bPFull + 2) || (lane >= bPEarly && lane < bPEarly + 2);
      const bool three = lane >= bEmpty && lane < bEmpty + kStages;
      mbar_init(bar(lane), four ? 4u : (three ? 3u : 1u));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();                                        // lane 0 is about to use barriers that other lanes have initialised
  } else if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + kOffBar + kOffTmemSlot), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (warp == 2 && lane < 5) {
    const CUtensorMap *tm = lane == 0 ? &tmQ : (lane == 1 ? &tmKc : (lane == 2 ? &tmVc : (lane == 3 ? &tmK : &tmV)));
    asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool fused = prm.fused_append != 0;
  int *status = lv.status;
  // Set-up, one rendezvous for everything.  Warp 0 asks for the slice's length, sends the first loads on their way - the
  // queries and, unless the keys are split over a cluster, the first K tile of a current map in the caller's tensors -
  // and then decides for the whole CTA whether it runs at all (one thread, because the status word may change between two
  // threads' reads, and a CTA of which only a part left would go on with barriers and TMEM nobody set up): an earlier CTA
  // gave up - do not pile on; swizzled tiles need the alignment, and a slice must not outgrow its page table - report,
  // do not fault.  Everybody but warp 0 then waits on a named barrier for the barriers, the length, the decision and the
  // TMEM allocation; warp 0 needs nobody: it goes on to issue loads.
  volatile int *leave_slot = reinterpret_cast<volatile int *>(base_ptr + kOffBar + kOffTmemSlot + 8);
  volatile int *hist_slot = reinterpret_cast<volatile int *>(base_ptr + kOffBar + kOffTmemSlot + 12);
  volatile int *item_slot = hist_slot + 1;               // slice and first query row, for the end of the softmax warps' work
  int leave = 0, hist = 0;
  const int Tc = fused ? tiles : 0;                      // key tiles of a current map outside the pages
  const int early = n_split == 1 && Tc > 0 ? 1 : 0;       // ring tiles that are loaded right away
  // ring tile t (2 i is K, 2 i + 1 is V of the i-th key tile), which belongs to key tile c of the current map
  auto load_map_tile = [&](int t, int c) {               // one lane
    const int st = t % kStages;
    const CUtensorMap *tc = (t & 1) ? &tmVc : &tmKc;
    const uint32_t dst = base + kOffRing + st * kTileBytes;
    mbar_expect_tx(bar(bFull + st), kTileBytes);
    tma_load_4d(dst, tc, 0, c * 128, h, b, bar(bFull + st));
    tma_load_4d(dst + kHalfBytes, tc, 64, c * 128, h, b, bar(bFull + st));
  };
  if (warp == 0) {
    if (lane == 0) {
      const int len = *reinterpret_cast<volatile int *>(lv.hist_len + slice), st = *reinterpret_cast<volatile int *>(status);
      if (!(base & 1023u)) {
        const int nq = pair ? 2 : 1;
        for (int t = 0; t < nq; ++t) {                     // (tile A's first product need not wait for B's queries)
          mbar_expect_tx(bar(bQFull + t), kTileBytes);
          tma_load_4d(base + kOffQ + t * kTileBytes, &tmQ, 0, q_first + t * 128, h, b, bar(bQFull + t));
          tma_load_4d(base + kOffQ + t * kTileBytes + kHalfBytes, &tmQ, 64, q_first + t * 128, h, b, bar(bQFull + t));
          if (t == 0 && early > 0) load_map_tile(0, 0);
        }
      }
      hist = len;
      if (st != 0) leave = 1;
      else if ((base & 1023u) || hist + n_k > (lv.pages_per_slice << lv.page_shift)) { atomicExch(status, kDevCheck); leave = 1; }
      *abort_flag = 0;
      *leave_slot = leave;
      *hist_slot = hist;
      item_slot[0] = slice;
      item_slot[1] = q_first;
      // the length that the next scale finds unless a compress of this one evicts
      if (!leave && q_tile == 0 && blockIdx.z == 0) lv.next_len[slice] = hist + n_k;
    }
    leave = __shfl_sync(0xffffffffu, leave, 0);
    hist = __shfl_sync(0xffffffffu, hist, 0);
    __syncwarp();
    __threadfence_block();
    asm volatile("bar.arrive 1, %0;" ::"n"(kThreads) : "memory");
  } else {
    tc_fence_before();
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
    tc_fence_after();
    leave = *leave_slot;
    hist = *hist_slot;
  }
  // Key tiles: Tc of the current map when it still waits in the caller's tensors, then Th of the pages; each source ends in a
  // ragged tile.  This CTA streams the tiles lo .. lo + nt - 1.
  const int rows_h = fused ? hist : hist + n_k;          // entries in the pages
  const int Th = (rows_h + 127) >> 7;
  const int lo = (Tc + Th) * (int)blockIdx.z / n_split;
  const int nt = leave ? 0 : (Tc + Th) * ((int)blockIdx.z + 1) / n_split - lo;
  auto tile_valid = [&](int i) {   // number of real keys in tile i
    const int rest = i < Tc ? n_k - i * 128 : rows_h - (i - Tc) * 128;
    return rest < 128 ? rest : 128;
  };
  // A single's key tiles are shared by A and B - unless they are so few that the combination would cost more than it gives:
  // then A takes them all.  Two tiles are shared in small launches only (us per layer and step, 36 queries behind 21 entries,
  // A alone / shared: 16 slices 7.6 / 6.7, 32 slices 8.2 / 7.4, 64 slices 9.0 / 8.8, 96 slices 9.5 / 10.4, 128 slices 10.6 / 10.9).
  const bool shared = !pair && (n_split > 1 || nt > (gridDim.x <= 64 ? 1 : 2));
  // key tiles that the softmax of tile A / B sees
  auto n_steps = [&](int qt) { return shared ? (nt + 1 - qt) >> 1 : (pair || qt == 0 ? nt : 0); };
  const uint32_t tmem = warp == 0 ? 0u : *tmem_slot;

  if (warp < 4) {
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    // (the whole warp walks the loop so that addresses stay warp-uniform; one lane issues)
    const int R = prm.box_rows;
    const int last_page = rows_h > 0 ? (rows_h - 1) >> lv.page_shift : 0;
    const int *pt = lv.page_table + (size_t)slice * lv.pages_per_slice;
    bool ok = nt > 0;
    int t = early;
    for (; t < 2 * nt && ok; ++t) {
      const int st = t % kStages, i = lo + (t >> 1);
      ok = mbar_wait_warp(bar(bEmpty + st), ((t / kStages) & 1) ^ 1, abort_flag, status);
      if (!ok) break;
      if (i < Tc) {
        if (elect_one()) load_map_tile(t, i);
      } else if (elect_one()) {
        const CUtensorMap *tm = (t & 1) ? &tmV : &tmK;
        mbar_expect_tx(bar(bFull + st), kTileBytes);
        for (int r0 = 0; r0 < 128; r0 += R) {
          const int slot = (i - Tc) * 128 + r0;
          int lp = slot >> lv.page_shift;
          lp = lp > last_page ? last_page : lp;
          const int row = (__ldg(pt + lp) << lv.page_shift) + (slot & lv.page_mask);
          const uint32_t dst = base + kOffRing + st * kTileBytes + r0 * 128;
          tma_load_2d(dst, tm, 0, row, bar(bFull + st));
          tma_load_2d(dst + kHalfBytes, tm, 64, row, bar(bFull + st));
        }
      }
      __syncwarp();
    }
    if (!ok && !(base & 1023u)) {
      // this CTA gives up or has no keys: nothing may land in its shared memory once that is used for something else or gone
      mbar_drain(bar(bQFull), 0);
      if (pair) mbar_drain(bar(bQFull + 1), 0);
      for (int k = t > kStages ? t - kStages : 0; k < t; ++k) mbar_drain(bar(bFull + k % kStages), (k / kStages) & 1);
    }
    if (n_split > 1) cluster_arrive();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    // (the whole warp walks the loop and waits; one elected lane issues the MMAs and commits)
    constexpr uint32_t idesc_qk = instr_desc(false);
    constexpr uint32_t idesc_pv = instr_desc(true);
    constexpr uint32_t dhi = desc_hi(1024);
    const bool leader = elect_one();
    const uint32_t q_lo[2] = {desc_lo(base + kOffQ, 16), desc_lo(base + kOffQ + (pair ? kTileBytes : 0u), 16)};
    // ring tile of tile qt's K in step j (its V is the next one): a pair's tiles share it, a single's take turns
    auto ring_k = [&](int j, int qt) { return shared ? 4 * j + 2 * qt : 2 * j; };
    auto ring_full = [&](int t) { return mbar_wait_warp(bar(bFull + t % kStages), (t / kStages) & 1, abort_flag, status); };
    // A tile's chain is  sweep -> PV(j) -> S(j+1) -> sweep ..., so between the moment a tile's P is complete
    // and the issue of its next S product this warp does nothing but issue: the operands of both products
    // are waited for beforehand (they arrive long before P does), the two products go out back to back, and the
    // commits follow them.
    auto k_desc = [&](int kt) { return desc_lo(base + kOffRing + (kt % kStages) * kTileBytes, 16); };
    auto mma_s = [&](uint32_t kd, int qt) { tc_mma_ss_x8(tmem + kColS + qt * 128, q_lo[qt], kd, dhi, idesc_qk); };
    constexpr int kEarlySteps = 2 * kEarlyChunks;      // a chunk of 32 keys is two steps of 16
    auto mma_pv_early = [&](uint32_t vd, int qt, bool accumulate) {
      tc_mma_ts_n<kEarlySteps>(tmem + kColO + qt * 128, tmem + kColS + qt * 128, vd, dhi, idesc_pv, accumulate ? 1u : 0u);
    };
    auto mma_pv_rest = [&](uint32_t vd, int qt) {
      tc_mma_ts_n<8 - kEarlySteps>(tmem + kColO + qt * 128, tmem + kColS + qt * 128 + p_col(kEarlySteps), vd + 128 * kEarlySteps, dhi,
                                   idesc_pv, 1u);
    };
    const int steps[2] = {n_steps(0), n_steps(1)};
    bool ok = nt > 0;
    for (int qt = 0; qt < 2 && ok && steps[qt] > 0; ++qt) {
      const int kt = ring_k(0, qt);
      ok = mbar_wait_warp(bar(bQFull + (pair ? qt : 0)), 0, abort_flag, status) && ring_full(kt);
      if (!ok) break;
      tc_fence_after();
      mma_s(k_desc(kt), qt);
      if (leader) {
        tc_commit(bar(bSFull + qt));
        if (!pair || qt == 1) tc_commit(bar(bEmpty + kt % kStages));
      }
      __syncwarp();
    }
    for (int j = 0; j < steps[0] && ok; ++j) {
      for (int qt = 0; qt < 2 && ok; ++qt) {
        if (j >= steps[qt]) break;
        const bool more = j + 1 < steps[qt];
        const int vt = ring_k(j, qt) + 1, kt = ring_k(j + 1, qt);
        const uint32_t vd = desc_lo(base + kOffRing + (vt % kStages) * kTileBytes, kHalfBytes), kd = k_desc(kt);
        const uint32_t v_empty = bar(bEmpty + vt % kStages), k_empty = bar(bEmpty + kt % kStages);
        ok = ring_full(vt) && mbar_wait_warp(bar(bPEarly + qt), j & 1, abort_flag, status);
        if (!ok) break;
        tc_fence_after();
        mma_pv_early(vd, qt, j > 0);
        if (leader) tc_commit(bar(bPvEarly + qt));
        __syncwarp();
        ok = (!more || ring_full(kt)) && mbar_wait_warp(bar(bPFull + qt), j & 1, abort_flag, status);
        if (!ok) break;
        tc_fence_after();
        mma_pv_rest(vd, qt);
        if (more) mma_s(kd, qt);
        if (leader) {
          // after the last key tile the tile's one-shot barrier for the epilogue instead of an S barrier:
          // tile A normalises and stores its rows while tile B is still in its last sweep
          tc_commit(bar((more ? bSFull : bFinal) + qt));
          tc_commit(bar(bPvDone + qt));
          if (!pair || qt == 1) {
            tc_commit(v_empty);
            if (more) tc_commit(k_empty);
          }
        }
        __syncwarp();
      }
    }
    // Now the next grid of the stream may come up: its set-up runs under this grid's epilogues.  Not earlier: its CTAs
    // would sit and wait on every SM that this grid leaves free, and the compress of the layer before, on the other stream,
    // would find none (a graph of 32 layers with compresses, us per layer and step, trigger at the start -> here: 16 slices
    // x 576 / 784 / 1024 queries 36.8 -> 26.7, 54.1 -> 46.6, 77.7 -> 71.0, without any compress work 24.6, 46.8, 57.1).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (n_split > 1) cluster_arrive();
  } else {
    // ------------------------------------------------------------------ append (warps 2 and 3)
    // Every ring tile is waited for and released, so that the empty barrier's phases stay in step;
    // current-map tiles whose turn falls on this item are copied: rows [0, valid) of a tile go
    // to slots hist + 128 i + r of the slice, un-swizzled, 16 bytes per thread and step.
    // A tile that is copied holds its ring stage for a while, so no CTA gets two in a row: the items of a slice that is
    // walked pair by pair take turns.  In a slice that is walked tile by tile (or partly so) an item copies its own tiles.
    const bool turns = slice * prm.per_pair.d + prm.per_pair.d <= prm.n_pair;
    const int u = (warp - 2) * 32 + lane;
    const int chunk = u & 15, rsub = u >> 4;
    const uint32_t src_off = (uint32_t)(chunk >> 3) * kHalfBytes;
    bool ok = true;
    for (int t = 0; t < 2 * nt && ok; ++t) {
      const int st = t % kStages, i = lo + (t >> 1);
      ok = mbar_wait_warp(bar(bFull + st), (t / kStages) & 1, abort_flag, status);
      if (!ok) break;
      if (prm.copy_in && i < Tc &&
          (turns ? i - prm.per_pair.div(i) * prm.per_pair.d == q_tile >> 1 : i == q_tile || (pair && i == q_tile + 1))) {
        const int first = i * 128;
        const int nvalid = tile_valid(i);
        char *pool = (t & 1) ? lv.v_pool : lv.k_pool;
        const uint32_t tile = base + kOffRing + st * kTileBytes + src_off;
#pragma unroll 4
        for (int r = rsub; r < nvalid; r += 4) {
          uint4 val;
          const uint32_t addr = tile + r * 128 + (((chunk & 7) ^ (r & 7)) << 4);
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(val.x), "=r"(val.y), "=r"(val.z), "=r"(val.w) : "r"(addr));
          const size_t row = slot_row(lv, slice, hist + first + r);
          reinterpret_cast<uint4 *>(pool + row * 256)[chunk] = val;
          if ((t & 1) == 0 && chunk == 0) lv.pos_pool[row] = prm.n_prev + first + r;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(bEmpty + st));
    }
    if (n_split > 1) cluster_arrive();
  }
  } else {
    // ------------------------------------------------------------------ softmax + epilogue
    const int qt = (warp - 4) >> 2;              // the query tile this warpgroup serves
    const int quarter = warp & 3;                // the TMEM lane quarter this warp may access
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    const float c = prm.scale_log2e;
    const uint64_t c2 = pack2(c, c);
    const int my_first = q_first + (pair ? qt * 128 : 0);   // first query row of this warpgroup's tile
    float m = -INFINITY, l = 0.f;
    // where this thread's row of the observation window is recorded (nullptr: it owns none), and whether its warp owns any
    float *win_row = nullptr;
    bool wwarp = false;
    if (kWindow) {
      int rank = -1;
      for (int e = 0; e < prm.w; ++e)
        if (prm.win_pos[e] == my_first + row) rank = e;
      if (rank >= 0) win_row = prm.win_logits + ((size_t)slice * prm.w + rank) * prm.ld_l;
      wwarp = __any_sync(0xffffffffu, rank >= 0);
    }
    const uint32_t o_addr = lane_addr + kColO + qt * 128;
    bool ok = true;
    const int steps = n_steps(qt);
    const uint32_t s_addr = lane_addr + kColS + qt * 128;
    for (int j = 0; j < steps && ok; ++j) {
      const int i_tile = lo + (shared ? 2 * j + qt : j);
      const int valid = tile_valid(i_tile);      // real keys: < 128 only in a ragged tile
      // the tile's first column of the window row (taken here: the one thread that stores it is what its tile waits for)
      float *win_dst = kWindow ? win_row + (i_tile < Tc ? i_tile + Th : i_tile - Tc) * 128 : nullptr;
      ok = mbar_wait_warp(bar(bSFull + qt), j & 1, abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      int o_landed = 0;                          // the previous PV product of this tile has been waited for
      // The sweep is software-pipelined over the chunks: while chunk cc is summed, packed, checked and stored
      // ("back"), the exponentials of chunk cc + 1 ("front": x = s c - m and 2^x, in place in the chunk's registers)
      // are already issued, against the reference as it stands.  They are independent of chunk cc's check, so the
      // transcendental unit stays busy across the vote and the stores; in the rare case that the check raises the
      // reference, chunk cc + 1 is read again and redone.
      float v[2][32];
      auto log_window = [&](const float *x, int cc) {
        // The row's raw products go out as they are (the score kernel applies the softmax scale), 32
        // columns as eight 16-byte stores: every key tile owns 128 columns of a logit row, the history's tiles before
        // the current map's, so the current map starts at the next multiple of 128 behind the history and
        // every store is aligned.  Columns of a ragged tile beyond its keys hold finite values nobody reads.
        if (win_row != nullptr) {
          float4 *dst = reinterpret_cast<float4 *>(win_dst + cc * 32);
#pragma unroll
          for (int v4 = 0; v4 < 8; ++v4) dst[v4] = make_float4(x[4 * v4], x[4 * v4 + 1], x[4 * v4 + 2], x[4 * v4 + 3]);
        }
        __syncwarp();   // the tcgen05 instructions that follow want the warp converged
      };
      // (masked: a ragged tile, whose columns beyond the last key must not count)
      auto front = [&](float *x, int vc, auto masked) {      // vc: real keys in this chunk (>= 32: all)
        const uint64_t negm2 = pack2(-m, -m);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float a0, a1;
          unpack2(fma2(pack2(x[2 * i], x[2 * i + 1]), c2, negm2), a0, a1);
          if constexpr (decltype(masked)::value) {
            if (2 * i >= vc) a0 = -INFINITY;
            if (2 * i + 1 >= vc) a1 = -INFINITY;
          }
          x[2 * i] = ex2(a0);
          x[2 * i + 1] = ex2(a1);
        }
      };
      // 32 values of at most 2^8 sum to at most 2^13; a larger, infinite or NaN sum means that some x exceeded 8.
      auto back = [&](const float *pv, uint32_t *pk) -> float {
        uint64_t sum2a = pack2(0.f, 0.f), sum2b = sum2a;
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          sum2a = add2(sum2a, pack2(pv[2 * i], pv[2 * i + 1]));
          sum2b = add2(sum2b, pack2(pv[2 * i + 2], pv[2 * i + 3]));
          pk[i] = pack_bf16(pv[2 * i], pv[2 * i + 1]);
          pk[i + 1] = pack_bf16(pv[2 * i + 2], pv[2 * i + 3]);
        }
        float s0, s1, s2, s3;
        unpack2(sum2a, s0, s1);
        unpack2(sum2b, s2, s3);
        return (s0 + s1) + (s2 + s3);
      };
      auto sweep = [&](auto masked) {
      tc_ld32(s_addr, v[0]);
      tc_ld32(s_addr + 32, v[1]);
      tc_wait_ld();
      if (kWindow && wwarp) { log_window(v[0], 0); log_window(v[1], 1); }
      if (j == 0) {
        // no reference yet: the largest of the row's first 32 products serves; a later chunk that exceeds the band raises it
        // like any other.  Where all 32 are -inf (masked keys) it is the lowest number: differences from it are numbers.
        float mt = -INFINITY;
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float e0 = (i < valid) ? v[0][i] : -INFINITY;
          const float e1 = (i + 1 < valid) ? v[0][i + 1] : -INFINITY;
          mt = max3(mt, e0, e1);
        }
        m = fmaxf(mt * c, -FLT_MAX);
      }
      front(v[0], valid, masked);
#pragma unroll
      for (int cc = 0; cc < kChunks; ++cc) {
        uint32_t pk[16];
        const int vc = valid - cc * 32;
        // A ragged tile's chunks without keys: zeros, and no exponentials (the sweep is the larger part of a short CTA: small_image, maps of
        // up to 256 queries, 249 -> 235 us; one image of 13 scales 12 347 -> 12 195, its graph 11 634 -> 11 477.  Leaving their steps out of
        // the products as well needs a run-time number of them, which the MMA warp pays for in every tile: 3 to 4 % slower passes).
        auto empty = [&](int left) { return decltype(masked)::value && left <= 0; };
        if (empty(vc)) {
#pragma unroll
          for (int i = 0; i < 16; ++i) pk[i] = 0u;
          tc_st16(s_addr + cc * 16, pk);
        } else {
          if (cc + 1 < kChunks && !empty(vc - 32)) front(v[(cc + 1) & 1], vc - 32, masked);
          const float lt = back(v[cc & 1], pk);
          if (cc + 2 < kChunks) tc_ld32(s_addr + (cc + 2) * 32, v[cc & 1]);
          if (__any_sync(0xffffffffu, !(lt <= 8192.f))) {
            // Once the early chunks' P is with the tensor core, their product has to land before O is scaled, and only
            // the later chunks' P is still this thread's to scale.
            const bool late = cc >= kEarlyChunks;
            const Raised r = raise_reference(vc, c, m, l, s_addr, cc, late ? kEarlyChunks : 0, o_addr, (late || j > 0) ? 1 : 0,
                                             late ? (o_landed == 2) : (o_landed >= 1), bar((late ? bPvEarly : bPvDone) + qt),
                                             (late ? j : j - 1) & 1, abort_flag, status);
            ok = __all_sync(0xffffffffu, r.ok != 0);
            if (!ok) return;
            m = r.m; l = r.l + r.sum;
            if (r.o_landed) o_landed = late ? 2 : 1;
            if (cc + 1 < kChunks && !empty(vc - 32)) {
              // the next chunk's exponentials were taken against the old reference: once more, from its raw products
              tc_ld32(s_addr + (cc + 1) * 32, v[(cc + 1) & 1]);
              tc_wait_ld();
              front(v[(cc + 1) & 1], vc - 32, masked);
            }
          } else {
            tc_st16(s_addr + cc * 16, pk);
            l += lt;
          }
        }
        if (cc == kEarlyChunks - 1) {
          // P of the first chunks is complete: that part of the PV product may start under the rest of the sweep
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(bPEarly + qt));
        }
        if (cc + 2 < kChunks) tc_wait_ld();
      }
      // The window rows' products of the tile's second half are recorded here, not between the chunks (a branch
      // there costs every warp's schedule 2-3 %): columns 64-127 of the S buffer still hold them, P only covers
      // columns 0-63, and the buffer is not written again before this warp has arrived below.
      if (kWindow && wwarp && ok) {
        tc_ld32(s_addr + 64, v[0]);
        tc_ld32(s_addr + 96, v[1]);
        tc_wait_ld();
        log_window(v[0], 2);
        log_window(v[1], 3);
      }
      };
      if (valid < 128) sweep(std::true_type{}); else sweep(std::false_type{});
      if (!ok) break;
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(bPFull + qt));
    }
    finish_rows(prm, base, lane_addr, item_slot[0], item_slot[1], qt, pair, shared, ok && steps > 0, ok && !leave, n_split, m, l, kWindow && win_row != nullptr,
                abort_flag, status);
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(kTmemCols) : "memory");
  }
  if (n_split > 1) {
    if (warp < 4) cluster_wait();
    cluster_arrive();
    cluster_wait();
    if (!leave) finish_cluster(prm, base, item_slot[0], item_slot[1], n_split);
  }
}

}  // namespace tc

// Host side: tensor maps over the K and V pools (built once) and over Q (per call), launch.
struct AttendTc {
  using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  EncodeFn encode = nullptr;
  CUtensorMap tmK, tmV;
  bool on = false;
  int box_rows = 128;
  int n_sm = 148;
  int max_clusters[tc::kMaxSplit + 1] = {0};   // clusters of c CTAs that fit the device at once

  static const void *kernel(bool window) {
    return window ? (const void *)tc::attend_tc_kernel<true> : (const void *)tc::attend_tc_kernel<false>;
  }

  // How a launch is cut.  us per launch on a B200 (148 SMs; attends of a map in the pages, back to back from a graph) behind
  // 209 / 1 960 entries, one CTA for every pair or odd tile -> this rule:
  //   16 slices, 64 queries 7.9 / 21.2 -> 8.0 / 10.5, 144: 9.9 / 34.5 -> 8.9 / 13.6, 256: 12.2 / 36.7 -> 8.9 / 13.8, 400: 14.1 / 38.7 ->
  //   11.1 / 18.5, 576: 17.7 / 40.7 -> 13.4 / 27.5, 1 024: 23.9 / 48.8 -> 16.6 / 31.3;
  //   128 slices x 1 024 queries (512 pairs, 3.5 waves), the last 68 pairs as 136 singles: 104.2 / 221.6 -> 98.6 / 214.1.
  // n_pair: items that are walked pair by pair; items: all of them; split: CTAs that share an item's keys.
  struct Cut { int n_pair, items, split; };
  Cut cut(int tiles, int slices, int key_tiles) const {
    // What combining over a cluster costs, in steps (of two key tiles) of a single.  Behind 1 960 entries every split up to four
    // CTAs gains (16 slices x 256 queries, 1 / 2 / 3 / 4 CTAs: 23.9 / 16.5 / 13.7 / 13.3 us); behind 209 a split of two mostly
    // loses (unsplit / as here, 16 slices x 144, 256, 400 queries: 8.2 / 8.9, 9.3 / 8.9, 10.6 / 11.1; 32 slices x 144, 256: 8.4 /
    // 10.1, 9.5 / 10.1), so 0.9 is too little for the shortest launches.
    constexpr float kJoin = 0.9f;
    const int pairs = tiles / 2 * slices, odd = tiles % 2 * slices;
    auto steps = [&](int split) { const int per = (key_tiles + split - 1) / split; return (float)((per + 1) / 2); };
    if (2 * pairs + odd <= n_sm) {
      // every query tile finds an SM of its own: singles, their keys shared by as many CTAs as pay and fit
      const int items = 2 * pairs + odd;
      int split = 1;
      float best = steps(1);
      for (int c = 2; c <= tc::kMaxSplit && c <= key_tiles; ++c)
        if (items <= max_clusters[c] && steps(c) + kJoin < best) { best = steps(c) + kJoin; split = c; }
      return {0, items, split};
    }
    // Pairs.  They run in waves, more or less; where a last wave would leave more than half of the SMs idle its items are
    // worked on tile by tile, which needs twice as many SMs for 0.55 of the time.
    const int items = pairs + odd, last = items % n_sm;
    if (2 * last <= n_sm) {
      const int per = (tiles + 1) / 2, first = items - last;          // the tiles from item `first` on
      return {first, first + tiles * slices - (first / per * tiles + 2 * (first % per)), 1};
    }
    return {items, items, 1};
  }

  bool init(int dtype, int head_dim, void *k_pool, void *v_pool, long long n_pages, int page_tokens, std::string &err) {
    on = false;
    if (dtype != 0 || head_dim != 128) return true;   // f32 x 64 has a kernel of its own (attend_f32.cuh)
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn) {
      err = "cuTensorMapEncodeTiled not available";
      return false;
    }
    encode = reinterpret_cast<EncodeFn>(fn);
    box_rows = page_tokens < 128 ? page_tokens : 128;
    const cuuint64_t dims[2] = {128, (cuuint64_t)n_pages * (cuuint64_t)page_tokens};
    const cuuint64_t strides[1] = {256};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    for (int i = 0; i < 2; ++i) {
      CUresult r = encode(i == 0 ? &tmK : &tmV, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, i == 0 ? k_pool : v_pool, dims, strides, box,
                          estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) { err = "cuTensorMapEncodeTiled(pool) failed with code " + std::to_string((int)r); return false; }
    }
    for (bool window : {false, true})
      if (cudaFuncSetAttribute(kernel(window), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kSmemBytes) != cudaSuccess) {
        err = "cannot raise the dynamic shared memory limit";
        return false;
      }
    return on = read_device(err);
  }

  // What a launch has to know about the device.  The number of clusters of every size that run at once (a cluster has to fit
  // one GPC) takes the runtime about a millisecond to tell, so it is asked once per device.
  bool read_device(std::string &err) {
    struct Device { int n_sm = 0, clusters[tc::kMaxSplit + 1] = {0}; };
    static std::mutex lock;
    static std::map<int, Device> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { err = "no current device"; return false; }
    std::lock_guard<std::mutex> hold(lock);
    Device &d = known[dev];
    if (d.n_sm == 0) {
      int n = 0;
      if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { err = "cannot read the number of SMs"; return false; }
      for (int c = 2; c <= tc::kMaxSplit; ++c) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3(1, 1, c); cfg.blockDim = dim3(tc::kThreads); cfg.dynamicSmemBytes = tc::kSmemBytes;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = c;
        cfg.attrs = attr; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&d.clusters[c], kernel(true), &cfg) != cudaSuccess) { cudaGetLastError(); d.clusters[c] = 0; }
      }
      d.n_sm = n;
    }
    n_sm = d.n_sm;
    std::copy(d.clusters, d.clusters + tc::kMaxSplit + 1, max_clusters);
    return true;
  }
  bool enabled() const { return on; }

  // [B][H][n_k][128] bf16 view -> 4-D tensor map with boxes of 128 rows x 64 columns
  bool map_rows(CUtensorMap *tm, const TensorView &X, int n_k, int n_heads, int B, const char *what, std::string &err) {
    const cuuint64_t dims[4] = {128, (cuuint64_t)n_k, (cuuint64_t)n_heads, (cuuint64_t)B};
    const cuuint64_t strides[3] = {(cuuint64_t)X.st * 2, (cuuint64_t)X.sh * 2, (cuuint64_t)X.sb * 2};
    const cuuint32_t box[4] = {64, 128, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<char *>(X.ptr), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { err = std::string("cuTensorMapEncodeTiled(") + what + ") failed with code " + std::to_string((int)r); return false; }
    return true;
  }

  // Kc / Vc: the current map's K and V when they have not been copied into the store yet (the kernel
  // reads them there and copies them in), else nullptr.
  // hist: entries before the current map (an upper bound over the slices); only sizes the launch.
  // win_logits / win_pos / w: where to record the window rows' logits (nullptr: do not).
  bool launch(const LayerView &lv, const TensorView &Q, const TensorView &O, float *lse, int n_k, const TensorView *Kc,
              const TensorView *Vc, bool copy_in, int hist, int n_prev, float scale, float *win_logits, float *win_lse, int ld_l, const int *win_pos, int w,
              cudaStream_t stream, std::string &err) {
    CUtensorMap tmQ, tmKc, tmVc;
    const int B = lv.n_slices / lv.n_heads;
    if (!map_rows(&tmQ, Q, n_k, lv.n_heads, B, "Q", err)) return false;
    const bool fused = Kc != nullptr && Vc != nullptr;
    if (fused) {
      if (!map_rows(&tmKc, *Kc, n_k, lv.n_heads, B, "K", err) || !map_rows(&tmVc, *Vc, n_k, lv.n_heads, B, "V", err)) return false;
    } else {
      tmKc = tmQ;
      tmVc = tmQ;
    }
    tc::Params prm;
    prm.lv = lv; prm.O = O; prm.lse = lse; prm.n_k = n_k;
    prm.scale_log2e = scale * 1.4426950408889634f;
    prm.box_rows = box_rows;
    prm.fused_append = fused ? 1 : 0;
    prm.copy_in = (fused && copy_in) ? 1 : 0;
    prm.n_prev = n_prev;
    prm.win_logits = win_logits;
    prm.win_lse = win_lse;
    prm.ld_l = ld_l;
    prm.w = win_logits ? w : 0;
    for (int e = 0; e < kMaxWindow; ++e) prm.win_pos[e] = (win_logits && e < w) ? win_pos[e] : -1;
    const int tiles = (n_k + 127) / 128;
    const Cut how = cut(tiles, lv.n_slices, fused ? (hist + 127) / 128 + tiles : (hist + n_k + 127) / 128);
    const int per = (tiles + 1) / 2;
    prm.n_pair = how.n_pair;
    prm.cut_tile = how.n_pair / per * tiles + 2 * (how.n_pair % per);
    prm.per_pair = tc::Divisor::of(per); prm.per_tile = tc::Divisor::of(tiles); prm.per_heads = tc::Divisor::of(lv.n_heads);
    // programmatic stream serialisation: the kernel's set-up may overlap the end of the kernel before it in the stream
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(how.items, 1, how.split);
    cfg.blockDim = dim3(tc::kThreads);
    cfg.dynamicSmemBytes = tc::kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = (unsigned)how.split;
    cfg.attrs = attr;
    cfg.numAttrs = how.split > 1 ? 2 : 1;
    void *args[] = {&tmQ, &tmK, &tmV, &tmKc, &tmVc, &prm};
    const cudaError_t launched = cudaLaunchKernelExC(&cfg, kernel(win_logits != nullptr), args);
    if (launched != cudaSuccess) {
      err = "attend: kernel launch failed";
      return false;
    }
    return true;
  }
};

}  // namespace scalekv
