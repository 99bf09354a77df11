// sm_100a building blocks for the tensor-core kernels: mbarrier, TMA (cp.async.bulk.tensor),
// tcgen05 (TMEM alloc, MMA, commit, ld/st) as inline PTX, plus UMMA descriptor builders and the
// host-side tensor-map encoder.  Every device-side wait is bounded: on expiry it raises a
// CTA-wide abort flag and records a code in the caller's status word instead of spinning forever.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

namespace gqla {
namespace tc {

// ----------------------------------------------------------------------------- addresses
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(pred));
    return pred != 0;
}

// ----------------------------------------------------------------------------- issuing warps
// The warps that issue MMAs and TMA loads run converged: every lane goes through the same waits and address arithmetic, and what
// one thread issues (MMAs, commits, loads: the `on` argument) is predicated with elect_one.  These instructions take uniform
// registers; in a branch that only the elected lane enters every operand has to be moved there, and back-to-back MMAs of any
// shape then go out 60 cycles apart.  Converged (operands from shared memory, cycles per MMA): M = 128, N = 128 of a pair 35,
// M = 64, N = 32 28, M = 128, N = 32 44; from M = 128, N = 256 of a pair on the tensor core is the slower one either way (69).
// For the same reason trip counts and rows that come from memory go through warp_uniform, and waits through warp_all.
__device__ __forceinline__ bool warp_all(bool v) { return __all_sync(0xffffffffu, v); }
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// ----------------------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes, uint32_t on = 1) {
    asm volatile("{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %2, 0;\n\t@e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes), "r"(on)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking probe (try_wait may suspend the thread for a while before it answers; this never does).
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\tmbarrier.test_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Status codes written to the caller's status word when a bounded wait gives up.
constexpr int32_t kStatusTimeout = 7;  // == GQLA_ERR_TIMEOUT
constexpr uint32_t kWaitSpins = 1u << 22;

// CTA-wide abort protocol: `abort_flag` lives in shared memory.  Once set, every wait returns
// false immediately and every role loop drains to the common teardown (TMEM dealloc, exit).
struct Abort {
    volatile int32_t* flag;  // shared
    int32_t* status;         // global, may be null
    __device__ __forceinline__ bool raised() const { return *flag != 0; }
    __device__ __forceinline__ void raise(int32_t where) const {
        *flag = 1;
        if (status != nullptr) atomicCAS(status, 0, kStatusTimeout | (where << 8));
    }
};

// Index checks of a debug build (-DGQLA_DEBUG; the pool offers no compute-sanitizer): a violated check records
// kStatusDebug | (where << 8) in the status word and execution goes on -- nothing traps.  Compiled out otherwise.
constexpr int32_t kStatusDebug = 9;  // == GQLA_ERR_DEBUG_CHECK
#ifdef GQLA_DEBUG
#define GQLA_DEBUG_CHECK(cond, status_ptr, where)                                                     \
    do {                                                                                              \
        if (!(cond) && (status_ptr) != nullptr) atomicCAS((status_ptr), 0, kStatusDebug | ((where) << 8)); \
    } while (0)
#else
#define GQLA_DEBUG_CHECK(cond, status_ptr, where) \
    do {                                          \
    } while (0)
#endif

// Waits for phase `parity` of `bar`; false if aborted or timed out (and raises the abort).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, const Abort& ab, int32_t where) {
    for (uint32_t it = 0; it < kWaitSpins; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 63u && ab.raised()) return false;
    }
    ab.raise(where);
    return false;
}

// For barriers that have usually completed by the time they are looked at: a non-suspending probe first.
__device__ __forceinline__ bool mbar_wait_fast(uint64_t* bar, uint32_t parity, const Abort& ab, int32_t where) {
    if (mbar_test_wait(bar, parity)) return true;
    return mbar_wait(bar, parity, ab, where);
}

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ----------------------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// Asks for a 2D box to be brought into L2 (no shared-memory destination, no completion to wait for).
__device__ __forceinline__ void tma_prefetch_l2_2d(const CUtensorMap* m, int32_t x, int32_t y, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %3, 0;\n\t@e cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];\n\t}" ::"l"(
            reinterpret_cast<uint64_t>(m)),
        "r"(x), "r"(y), "r"(on)
        : "memory");
}
// 2D tiled load: coordinates (x = innermost, y).  x * elem_size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* m, int32_t x, int32_t y, uint64_t* bar, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(on)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* m, int32_t x, int32_t y, int32_t z,
                                            uint64_t* bar, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %6, 0;\n\t"
        "@e cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
        "[%2];\n\t}" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(on)
        : "memory");
}

// Small pages: the one box (a run of PG rows) that a sequence's end cuts.  What lies behind the end in its last page may be
// anything, NaN included, and a V row has to be zero there (zero weight times NaN is NaN), so the box is put together from
// boxes of eight rows and, for the eight that the end falls into, of one row; those behind the end start at `beyond`, the
// row count of the plane, and are filled with zeros.  A box of one row lands on a 128-byte boundary; the swizzle goes by the
// address, so it is where the whole box would have put it.  PG / 8 + 7 loads per column block, spread over the warp's
// lanes, once per sequence and row block: 88.6 us a step instead of 87.2 on 32 sequences of 300-8000 rows in pages of 64 rows
// (128 heads, absorb path).
template <int PG>
struct CutMaps {
    CUtensorMap rows8, row1;
};
template <>
struct CutMaps<0> {};
// Which run of a tile of `rows` rows the end cuts, -1 if none: `left` rows of the sequence remain at the tile's start.
template <int PG>
__device__ __forceinline__ int cut_run(int32_t left, int rows) {
    return left > 0 && left < rows && left % PG != 0 ? left / PG : -1;
}
// load(map, column block, row of the run, cache row); `row`: the run's first cache row, `valid` rows of it are the sequence's.
template <int PG, int BLOCKS, typename Load>
__device__ __forceinline__ void load_cut_run(const CutMaps<PG>& maps, int lane, int valid, int32_t row, int32_t beyond, Load load) {
    constexpr int N = PG / 8 + 8;  // boxes of a column block: eights, then the single rows of the eight that is cut
    const int mixed = valid % 8 != 0 ? valid / 8 : -1;
    for (int i = lane; i < BLOCKS * N; i += 32) {
        const int k = i % N;
        const int r = k < PG / 8 ? 8 * k : 8 * mixed + k - PG / 8;
        if (k < PG / 8 ? k == mixed : mixed < 0) continue;
        load(k < PG / 8 ? &maps.rows8 : &maps.row1, i / N, r, r < valid ? row + r : beyond);
    }
}

// Bulk store shared -> global (both 16-byte aligned, size a multiple of 16 bytes), tracked by bulk groups.
__device__ __forceinline__ void bulk_store(void* gdst, const void* ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_u32(ssrc)),
                 "r"(bytes)
                 : "memory");
}
// 2D tiled store shared -> global through a tensor map (x * elem_size a multiple of 16 bytes, y >= 0);
// rows and columns beyond the tensor's extent are clipped.  Tracked by bulk groups like bulk_store.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* m, const void* src, int32_t x, int32_t y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(smem_u32(src)), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until the bulk stores of this thread have finished READING shared memory.
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ----------------------------------------------------------------------------- TMEM
// Allocation is warp-collective (one full warp); the base address lands in shared memory.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// TMEM address: lane in bits [31:16], column in bits [15:0].
__device__ __forceinline__ uint32_t tmem_addr(uint32_t base, uint32_t lane, uint32_t col) {
    return base + (lane << 16) + col;
}

// Each thread of the warp reads N consecutive 32-bit columns of its own lane (lane = 32*(warp%4) + laneid).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,"
        "%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}
// 16 lanes x 8 columns spread over the 32 threads of the warp: thread t receives, of lanes t/4 and t/4 + 8 (counted
// from the address's lane), the columns 2 (t % 4) and 2 (t % 4) + 1 -- r[0], r[1] of the first lane, r[2], r[3] of the other.
__device__ __forceinline__ void tmem_ld_16x256b(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}
// Sixteen columns: r[4..7] are r[0..3] of the columns 8 further on.
__device__ __forceinline__ void tmem_ld_16x256b_x2(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r) {
    static_assert(N == 4 || N == 8 || N == 16 || N == 32, "unsupported width");
    if constexpr (N == 4) tmem_ld4(taddr, r);
    else if constexpr (N == 8) tmem_ld8(taddr, r);
    else if constexpr (N == 16) tmem_ld16(taddr, r);
    else tmem_ld32(taddr, r);
}
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t* r) {
    static_assert(N == 4 || N == 8 || N == 16 || N == 32, "unsupported width");
    if constexpr (N == 4) tmem_st4(taddr, r);
    else if constexpr (N == 8) tmem_st8(taddr, r);
    else if constexpr (N == 16) tmem_st16(taddr, r);
    else tmem_st32(taddr, r);
}
__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
// OR of a predicate over the `nthreads` threads that call it (named barrier 1).
// Warps that meet in named barriers leave a loop by such a vote on their own failed waits, not by the abort flag: a producer or
// issuer may raise that between the reads of two warps, of which one would then leave and one go on to the next barrier, which
// has no limit.
__device__ __forceinline__ bool bar_or(bool v, int nthreads) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(nthreads)
        : "memory");
    return r != 0;
}

// ----------------------------------------------------------------------------- UMMA descriptors
// Shared-memory matrix descriptor (64-bit):
//   [0,14)  start address >> 4        [16,30) leading-dimension byte offset >> 4
//   [32,46) stride-dimension byte offset >> 4     [46,48) descriptor version (1 on sm_100)
//   [49,52) base offset (0: tiles are 1024-byte aligned)      [61,64) swizzle mode (2 = 128-byte)
constexpr uint64_t kDescSw128 = (1ull << 46) | (2ull << 61);

// K-major operand tile written by TMA with 128-byte swizzle: rows of 64 bf16 (128 B); 8-row groups
// are 1024 B apart (SBO).  LBO is unused for swizzled K-major layouts (set to 1).
__device__ __forceinline__ uint64_t desc_kmajor_sw128(uint32_t smem_addr) {
    return kDescSw128 | (uint64_t)((smem_addr & 0x3FFFF) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32);
}
// MN-major operand from the same kind of tile ([k rows] x [64 mn elements = 128 B]): 8-k-row groups are
// 1024 B apart (SBO); consecutive 64-element MN blocks are `mn_block_bytes` apart (LBO).
__device__ __forceinline__ uint64_t desc_mnmajor_sw128(uint32_t smem_addr, uint32_t mn_block_bytes) {
    return kDescSw128 | (uint64_t)((smem_addr & 0x3FFFF) >> 4) | ((uint64_t)(mn_block_bytes >> 4) << 16) |
           ((uint64_t)(1024 >> 4) << 32);
}

// Instruction descriptor for kind::f16 with bf16 operands and fp32 accumulation:
//   [4,6) D format (1 = f32)  [7,10) A format (1 = bf16)  [10,13) B format (1 = bf16)
//   [15] A major (0 = K)  [16] B major (0 = K, 1 = MN)  [17,23) N >> 3  [24,29) M >> 4
__host__ __device__ constexpr uint32_t idesc_bf16(uint32_t M, uint32_t N, uint32_t a_mn_major, uint32_t b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn_major << 15) | (b_mn_major << 16) | ((N >> 3) << 17) |
           ((M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]; issued by ONE thread.
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(on)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]; A is K-major with one row per TMEM lane, two bf16 per 32-bit column.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(on)
        : "memory");
}
// Makes `bar` complete one arrival once every MMA issued so far by this thread has finished.
__device__ __forceinline__ void umma_commit(uint64_t* bar, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %1, 0;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)),
        "r"(on)
        : "memory");
}

// ----------------------------------------------------------------------------- CTA pairs (cta_group::2)
// Two CTAs of a cluster drive one MMA: each holds half of the M rows of A and D and supplies half of
// the N rows of B from its own shared memory (same offsets in both CTAs); the even-ranked CTA issues.
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of `local` (a shared::cta address of this CTA) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t mapa(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
// Arrival on a barrier of another CTA of the cluster.  Default (CTA-scope release) semantics on purpose:
// the cluster-scope release form costs a cluster-wide memory barrier (about 2000 cycles when measured in
// the softmax loop), and what the arrival publishes here -- shared-memory and tensor-memory contents of
// the arriving CTA, fenced beforehand -- is only ever read by that CTA's own tensor core.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t* dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish2() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// TMA load issued by either CTA of a pair into its OWN shared memory; the transaction bytes are
// credited to the mbarrier at cluster address `bar_cluster_addr` (normally the leader's).  No multicast.
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* m, int32_t x, int32_t y,
                                                 uint32_t bar_cluster_addr, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
        "%4}], [%2];\n\t}" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar_cluster_addr), "r"(x), "r"(y), "r"(on)
        : "memory");
}
// D[tmem] (+)= A[smem] * B[smem] across the CTA pair, issued by ONE thread of the leader.  The descriptors are
// given as (low word, high word): the high word of a shared-memory
// descriptor (SBO, version, swizzle) is a constant, so stepping through an operand is one 32-bit add.
// The issuing thread's instruction count per MMA matters: one MMA of the shapes used here is only 32-64
// cycles of tensor work.
constexpr uint32_t kDescHiSw128 = (uint32_t)((kDescSw128 | ((uint64_t)(1024 >> 4) << 32)) >> 32);
__device__ __forceinline__ uint32_t desc_lo(uint64_t desc) { return (uint32_t)desc; }
template <bool ACCUMULATE>
__device__ __forceinline__ void umma_ss2_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .b64 da, db;\n\t.reg .pred p, e;\n\t"
        "mov.b64 da, {%1, %4};\n\tmov.b64 db, {%2, %4};\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.ne.b32 e, %6, 0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(kDescHiSw128), "n"(ACCUMULATE ? 1 : 0), "r"(on)
        : "memory");
}
// The same for one CTA, with the two constant high words given and the accumulate flag a run-time value.
__device__ __forceinline__ void umma_ss_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                           uint32_t idesc, uint32_t accumulate, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .b64 da, db;\n\t.reg .pred p, e;\n\t"
        "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\tsetp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 e, %7, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(on)
        : "memory");
}
// Arrives (once every MMA issued so far has finished) on the barrier at the same offset in every CTA of `mask`.
__device__ __forceinline__ void umma_commit2(uint64_t* bar, uint16_t mask, uint32_t on = 1) {
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %2, 0;\n\t"
        "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}" ::"r"(
            smem_u32(bar)),
        "h"(mask), "r"(on)
        : "memory");
}

// ----------------------------------------------------------------------------- dependent launches
// Programmatic dependent launch: a kernel launched with launch_pdl may begin (its CTAs start and run their
// set-up: barrier init, TMEM allocation) while the previous kernel of the stream is still running, once
// every CTA of that kernel has executed pdl_launch_dependents or exited.  It must call pdl_wait before it
// touches global memory: the wait returns when the previous kernel has completed and its writes are
// visible.  Both instructions do nothing in a kernel launched the ordinary way.
//
// Every tensor-core kernel here signals its dependents before (or while) it allocates tensor memory, and
// tcgen05.alloc blocks until the columns are free.  That is only safe while two such CTAs can never share an
// SM: otherwise a dependent CTA could take the SM's tensor memory first and then sit in pdl_wait for a
// primary CTA that is blocked in its own allocation.  Shared memory rules it out -- each of these kernels
// asks for more than half of an SM's shared memory -- and every kernel states that with this check.
constexpr int kSmemPerSM = 233472;  // bytes of shared memory of one sm_100 SM
template <int kDynamicSmemBytes>
struct OneCtaPerSM {
    static_assert(2 * kDynamicSmemBytes > kSmemPerSM,
                  "two CTAs of a kernel that triggers its dependents before allocating tensor memory must not fit one SM");
    static constexpr bool value = true;
};
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

// ----------------------------------------------------------------------------- small math
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// x / y from x, y and the rounded reciprocal of y: the product, corrected once by its exact remainder (P. Markstein, Computation of
// elementary functions on the IBM RISC System/6000 processor, IBM J. Res. Dev. 34, 1990).  For where many x share one y: with a
// division per x a step took 14.0 us instead of 12.7 (one sequence of 3001 rows, GQA path), like this 12.4, uncorrected 12.6.
// The remainder of an infinite x is NaN, for which fminf gives a finite number: infinity stays what it is.
__device__ __forceinline__ float div_by(float x, float y, float recip) {
    const float q = x * recip;
    return fmaf(fminf(fmaf(-q, y, x), FLT_MAX), recip, q);
}
// A pair of fp32 values as N bf16 terms each, out[n * stride] the pair of terms n.  Three terms are the value itself: every
// term takes eight bits and the differences are exact, so nothing is left of the 24 bits (short of bf16's smallest number).
template <int N>
__device__ __forceinline__ void split_bf16(float x0, float x1, uint32_t* out, int stride) {
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const uint32_t t = pack_bf16(x0, x1);
        out[n * stride] = t;
        x0 -= __uint_as_float(t << 16);
        x1 -= __uint_as_float(t & 0xffff0000u);
    }
}

// ----------------------------------------------------------------------------- host: tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// bf16 tensor of `rank` dims (dims[0] innermost, contiguous); strides_bytes[i] is the byte stride of
// dim i+1.  128-byte swizzle, zero fill out of bounds.  Returns false on failure.
inline bool make_tmap_bf16(CUtensorMap* out, const void* base, int rank, const uint64_t* dims,
                           const uint64_t* strides_bytes, const uint32_t* box) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    cuuint64_t d[5], s[4];
    cuuint32_t b[5], e[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        b[i] = box[i];
        e[i] = 1;
        if (i + 1 < rank) s[i] = strides_bytes[i];
    }
    CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), d, s, b, e,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// One-byte elements (E4M3 codes); swizzle chosen by the caller (the 64-byte form for 64-byte rows).
inline bool make_tmap_u8(CUtensorMap* out, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                         const uint32_t* box, CUtensorMapSwizzle swizzle) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    cuuint64_t d[5], s[4];
    cuuint32_t b[5], e[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        b[i] = box[i];
        e[i] = 1;
        if (i + 1 < rank) s[i] = strides_bytes[i];
    }
    CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_UINT8, (cuuint32_t)rank, const_cast<void*>(base), d, s, b, e,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace gqla
