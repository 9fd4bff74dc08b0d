// cci_tc_common.cuh -- device helpers of the tensor-core kernels (tcgen05,
// mbarrier, cp.async, TMA) shared by cci_dense_tc.cu, cci_gemm_ws.cuh and cci_narrow.cu.
#pragma once

#include "cci_kernels.h"

namespace cci {
namespace tc {

constexpr long long kWaitLimit = 1ll << 31;  // clock cycles (about 1 s) per bounded wait

constexpr int kMaxStages = 9;
constexpr int kMaxHalo = 4;  // halo buffers of a 3x3 convolution tile ring

// barriers and TMEM slot of a tensor-core kernel (after its 1024-byte aligned
// stage buffers); up to kMaxStages pipeline stages
struct Smem {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t aux[kMaxStages];  // per-stage barrier of a second copy (fp32: raw activation tile landed)
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint64_t drain;
    uint64_t hfull[kMaxHalo];   // halo copies (3x3 convolutions): halo buffer landed
    uint64_t hempty[kMaxHalo];  // halo buffer free again (its chunk's MMAs completed)
    uint32_t tmem_base;
    int abort;
};


__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// one test of the phase with the given parity (kCluster: acquire at cluster
// scope, for phases that include arrivals released by the other CTA of a pair).
// A waiting thread is suspended in hardware until the phase completes (or the
// hint elapses) instead of spinning: the kernels hold a dozen warps that spend
// most of their time waiting, and spinning ones take issue slots from the warps
// issuing MMAs and copies on the same scheduler.
constexpr uint32_t kSuspendNs = 1000000;
template <bool kCluster>
__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity)
{
    uint32_t done;
    if constexpr (kCluster)
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity), "n"(kSuspendNs)
            : "memory");
    else
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity), "n"(kSuspendNs)
            : "memory");
    return done != 0;
}

// bounded wait for the phase with the given parity; false on timeout or abort.
// A phase already complete costs one test (no clock read).
template <bool kCluster = false>
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort, uint32_t *status)
{
    const uint32_t a = smem_u32(bar);
    if (mbar_try<kCluster>(a, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try<kCluster>(a, parity)) return true;
        if (*abort) return false;
        if (clock64() - t0 > kWaitLimit) {
            *abort = 1;
            report(status, CCI_ERR_TIMEOUT);
            return false;
        }
    }
}

// true in one lane of the (converged) warp, the same one at every call.  The
// tcgen05 and TMA instructions take their operands from uniform registers: behind
// this election the compiler knows that one thread runs them and forms the
// operands there, while behind a test of the lane number it moves every operand
// over with a per-lane sequence.  Measured on GB300 for a loop of wait, four
// 128 x 64 x 16 MMAs and a commit per stage: 361 cycles a stage behind lane == 0,
// 222 behind the election (192 are the tensor core's).  The few-column product
// issues behind it; the workspace GEMM still tests the lane number.
__device__ __forceinline__ bool elect_one()
{
    uint32_t e;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
    return e != 0;
}

// Programmatic dependent launch: wait until the grid before this one has completed
// and its writes are visible; let the grid after this one be scheduled (it waits
// the same way before it touches memory).
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void st_shared_v4_zero(uint32_t addr)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0) : "memory");
}

__device__ __forceinline__ void st_shared_b16(uint32_t addr, uint16_t v)
{
    asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}

// byte offset of (row, k) in a K-major tile of 128-byte rows with the 128-byte
// swizzle: 16-byte chunk j of row i sits at chunk position j ^ (i % 8)
__device__ __forceinline__ uint32_t sw128(int row, int k_elem)
{
    const int chunk = (k_elem >> 3) ^ (row & 7);
    return static_cast<uint32_t>(row * 128 + chunk * 16 + (k_elem & 7) * 2);
}

// tcgen05 shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row
// atoms of 1024 bytes (stride byte offset 1024), fixed field 0b001 at bit 46
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr & 0x3ffff) >> 4);       // start address
    d |= static_cast<uint64_t>(1) << 16;                       // leading byte offset (unused)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;               // stride byte offset
    d |= static_cast<uint64_t>(1) << 46;                       // fixed 0b001
    d |= static_cast<uint64_t>(2) << 61;                       // 128-byte swizzle
    return d;
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// store 32 consecutive 32-bit columns of this thread's TMEM lane (32x32b shape);
// follow with tcgen05.wait::st before the data is used
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

// ---- TMA (bulk tensor copies completing on an mbarrier) ----
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// 2-D tile load of the box at (x = inner element, y = row) into shared memory;
// x * element size must be a multiple of 16 bytes
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *tmap, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// 4-D tile load of the box at (c0 innermost, c1, c2, c3); c0 * element size must
// be a multiple of 16 bytes; the other coordinates may lie outside the tensor
// (those elements read as zero)
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void *tmap, int c0, int c1, int c2, int c3,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

// tile stores from shared memory (bulk-group completion); elements of the box
// outside the tensor are not written.  Coordinates must not be negative.
__device__ __forceinline__ void tma_store_2d(const void *tmap, uint32_t src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(src), "r"(c0), "r"(c1)
                 : "memory");
}

__device__ __forceinline__ void tma_store_4d(const void *tmap, uint32_t src, int c0, int c1, int c2, int c3)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// wait until at most N committed bulk groups still read their shared memory
template <int N>
__device__ __forceinline__ void bulk_wait_read()
{
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

// wait until every committed bulk group has completed
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// named barrier `id` over `n` threads (non-aligned form: the threads of a warp
// need not arrive converged)
__device__ __forceinline__ void named_sync(int id, int n)
{
    asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// named barrier `id` over `n` threads that returns the AND of every thread's v
__device__ __forceinline__ bool named_and(int id, int n, bool v)
{
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.red.and.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(v)), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void tma_prefetch_desc(const void *tmap)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}

}  // namespace tc
}  // namespace cci
