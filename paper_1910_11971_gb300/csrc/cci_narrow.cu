// cci_narrow.cu -- products of few columns (N <= 128, bf16): one launch that
// expands the packed weights and multiplies them, for serving and classifier heads.
//
// What bounds it: such a product reads each packed weight once and does little
// else, so its time is that of reading and expanding the packed weights, plus the
// latencies of one pass.  The workspace GEMM has one or two M tiles here: at most
// Cout / 64 CTAs, each walking the whole reduction behind a decompression launch
// that writes and re-reads the dense matrix.
//
// The split taken instead: D[co][n] with the output channels as the MMA's M.  A
// CTA owns 128 output channels and a part of the reduction; the CTAs of a tile
// form a cluster (1, 2, 4 or 8 parts: as many as the SMs hold at once, four
// stages each at least), so 4096 -> 4096 runs on 128 CTAs.  Four groups of four
// warps take the 64-deep stages in turn: a warp zeroes its 32 rows of the stage's
// 128-byte-swizzled A tile and scatters the kept weights into them (Alg. 2's
// index), eight weights per 16-byte load, loaded a stage ahead; one warp copies the
// activations' [n][64] tile by TMA; one warp issues the MMAs.  The scatter's work
// is that of the kept weights: the register expansion of the decompression, which
// tests every slot against every row, took 15.6 us instead of 7.2 at G = 32, K = 8
// (4096 -> 1024, 32 columns) and the same time at G = 8, K = 2.  The parts are
// summed through distributed shared memory: rank j takes every parts-th quad of
// columns, each part stores its sums of a quad straight from tensor memory into the
// owner's shared memory, and after one cluster barrier the owner adds them in
// rank order (the same sum whatever finishes first), adds bias, applies ReLU and
// writes rows of consecutive channels.
//
// The number of parts depends on Cout and R alone, never on N, so a product cut
// into chunks of columns gives the same bits as the whole.
//
// Where the rule lies (GB300, 348 shapes; device time per pass in a CUDA graph, in
// brackets the time of a call from the host, against decompression and GEMM, bf16
// G = 8, K = 2 unless said).  From 16 stages on 0.27 to 0.98 of their time, 0.55 in
// the mean: 16 x 4096 -> 4096 9.6 us (13.5) against 23.6 (24.8), 128 x 4096 -> 4096 12.7
// against 23.9, 16 x 4096 -> 1024 at G = 32, K = 8 6.2 against 23.2; also where the tiles
// fill the SMs and no reduction is split (more than 9728 channels): 16 x 4096 -> 32768
// 62.7 against 109.7, 128 x 4096 -> 9984 38.1 against 38.9.  Up to seven stages: 0.75 in
// the mean and at most 1.01 up to 16 columns; 0.98 and up to 1.26 from 64 on (64 x
// 448 -> 1000 7.4 against 5.9), as ten stages do (128 x 640 -> 512 7.8 against 6.7).
// Those stay here for the launch that a call saves, 13.6 us (64 x 448 -> 1000) against
// 20.2; in a captured graph they lose that up to 1.6 us.  Eight or nine stages, too few
// to split, stay with the GEMM: in this form 0.36 to 1.36 of its time over 76 shapes,
// slower from 64 columns on at up to 9728 channels (64 x 576 -> 512 8.6 against 6.3),
// 1.06 at most up to 16 columns (16 x 576 -> 4096 6.9 against 7.9).  More than 128
// columns would need smaller stages.
#include "cci_gemm_ws.cuh"

namespace cci {
namespace narrow {

constexpr int kM = 128;         // output channels of a tile
constexpr int kGroups = 4;      // expansion groups of four warps
constexpr int kWarps = 4 * kGroups + 2;
constexpr int kThreads = 32 * kWarps;
constexpr int kABytes = kM * 128;
constexpr int kMaxN = 128;      // columns
constexpr int kMinStages = 4;   // stages of a part, at least: one for each group
constexpr int kSplitStages = 10;  // stages of a reduction that is split, at least
constexpr int kWholeStages = 7;   // stages of a reduction that one part takes, at most
constexpr int kMaxParts = 8;    // portable cluster size

template <int NP>
struct Cfg {
    static constexpr int kStage = kABytes + NP * 128;
    // sums of this CTA's column quads: blocks of [128 channels][4 columns], one per part
    // and quad; quads are dealt to the parts in turn, so a round of them is kMaxParts
    static constexpr int kQuads = NP / 4 < kMaxParts ? kMaxParts : NP / 4;
    static constexpr int kSums = kQuads * kM * 16;
    static constexpr int kFit = (static_cast<int>(kMaxSmemPerBlock) - 2048 - kSums) / kStage;
    static constexpr int kStages = kFit < 8 ? kFit : 8;
    static constexpr int kTmem = NP < 32 ? 32 : NP;
    static constexpr size_t kSmem = 1024 + static_cast<size_t>(kStages) * kStage + kSums + 1024;
    static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(NP >> 3) << 17) |
                                       (static_cast<uint32_t>(kM >> 4) << 24);
    static_assert(kStages >= kGroups, "every group needs a stage");
    static_assert(kQuads % kMaxParts == 0, "whole rounds of quads");
    static_assert(kSmem <= kMaxSmemPerBlock, "stages over the per-block limit");
};

struct Smem {
    uint64_t full[8];   // the stage's weights are stored (one arrival per warp of its group)
    uint64_t xfull[8];  // the stage's activations have landed
    uint64_t empty[8];  // the stage's MMAs have completed
    uint64_t done;      // every MMA has completed
    uint32_t tmem_base;
    int abort;
};
static_assert(sizeof(Smem) <= 1024, "barriers");

// 16 bytes into the shared memory of a CTA of the cluster (shared::cluster address)
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

__device__ __forceinline__ float4 ld_shared_f4(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}

// Y[n][co] in the output type
__device__ __forceinline__ void store_y(const FwdParams &p, int n, int64_t co, float y)
{
    const int64_t off = static_cast<int64_t>(n) * p.Cout + co;
    if (p.out_bf16)
        reinterpret_cast<uint16_t *>(p.Y)[off] = static_cast<uint16_t>(ws::bf16x2_rn(__float_as_uint(y), 0u));
    else
        p.Y[off] = y;
}

constexpr int NB = 2;  // stages of a group whose weights are loaded ahead

// eight consecutive kept weights of a group and their indices (in: inside the layer)
struct Unit {
    uint4 v;
    uint2 i;
    bool in;
};

// true if an index set of the unit is not strictly increasing or has an index >= G
// (ws::pk::bad_sets on the unit's 8 / K sets)
template <int K>
__device__ __forceinline__ bool unit_bad(uint2 i, int G)
{
    const uint32_t w[2] = {i.x, i.y};
    uint32_t grows = 0x01000100u;
    if constexpr (K >= 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) grows &= ((w[q] >> 8) & 0x00ff00ffu) + 0x00ff00ffu - (w[q] & 0x00ff00ffu);
    }
    if constexpr (K >= 4)
        grows &= (ws::pk::prmt(w[0], w[1], 0x6622u) & 0x00ff00ffu) + 0x00ff00ffu -
                 (ws::pk::prmt(w[0], w[1], 0x5511u) & 0x00ff00ffu);
    if constexpr (K == 8) grows &= ((w[1] & 0xffu) + 0xffu - (w[0] >> 24)) | 0x01000000u;
    const uint32_t above = (0xffu & ~static_cast<uint32_t>(G - 1)) * 0x01010101u;
    return ((w[0] | w[1]) & above) != 0u || grows != 0x01000100u;
}

// Word order in which a lane scatters its unit (two weights per word): word x ^
// flip at step x.  The bank of a weight is 4 ((r / 8) ^ (row % 8)) + (r % 8) / 2:
// the lanes of a step should differ in (r % 8) / 2, and with K = 1 or 2 they hold
// the same one or two values of it unless some of them start at another word.
template <int K>
__device__ __forceinline__ int word_flip(int lane)
{
    return K == 1 ? (lane >> 3) & 3 : (K == 2 ? (lane >> 4) * 2 : 0);
}

// stores the unit's weights, of a group whose rows start at row0 of the warp's 32
// and from weight w0 of its 64 K in the stage on, into the zeroed rows at `rows`
// (128-byte rows, 128-byte swizzle)
template <int K>
__device__ __forceinline__ void scatter_unit(const Unit &u, uint32_t rows, int row0, int w0, int flip, int G)
{
    uint32_t w[4] = {u.v.x, u.v.y, u.v.z, u.v.w}, i[2] = {u.i.x, u.i.y};
    if constexpr (K <= 2) {
        const bool f2 = flip & 2;
        const uint32_t a = f2 ? w[2] : w[0], b = f2 ? w[3] : w[1], c = f2 ? w[0] : w[2], d = f2 ? w[1] : w[3];
        const uint32_t j0 = f2 ? i[1] : i[0], j1 = f2 ? i[0] : i[1];
        w[0] = a;
        w[1] = b;
        w[2] = c;
        w[3] = d;
        i[0] = j0;
        i[1] = j1;
    }
    if constexpr (K == 1) {
        const bool f1 = flip & 1;
        const uint32_t a = f1 ? w[1] : w[0], b = f1 ? w[0] : w[1], c = f1 ? w[3] : w[2], d = f1 ? w[2] : w[3];
        w[0] = a;
        w[1] = b;
        w[2] = c;
        w[3] = d;
#pragma unroll
        for (int h = 0; h < 2; ++h) i[h] = f1 ? ws::pk::prmt(i[h], 0u, 0x1032u) : i[h];
    }
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const uint32_t r = static_cast<uint32_t>((w0 + (x ^ (2 * flip))) / K);  // within the stage
        const uint32_t id = (i[x >> 2] >> (8 * (x & 3))) & static_cast<uint32_t>(G - 1);
        const uint32_t row = static_cast<uint32_t>(row0) + id;  // 0 .. 31
        const uint32_t at = rows + row * 128u + (((r >> 3) ^ (row & 7u)) << 4) + (r & 7u) * 2u;
        tc::st_shared_b16(at, static_cast<uint16_t>(x & 1 ? w[x >> 1] >> 16 : w[x >> 1]));
    }
}

// y + bias, ReLU (NaN gives 0)
__device__ __forceinline__ float finish(float y, const FwdParams &p, float bias)
{
    if (p.bias) y += bias;
    return p.relu ? fmaxf(y, 0.f) : y;
}

template <int K, int NP>
__global__ void __launch_bounds__(kThreads, 1)
    narrow_kernel(FwdParams p, const __grid_constant__ CUtensorMap tmX, int log_parts)
{
    using C = Cfg<NP>;
    constexpr int kStages = C::kStages;
    constexpr int kUG = 8 * K;  // units per group and stage
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t raw = tc::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t sums = base + kStages * C::kStage;
    Smem *S = reinterpret_cast<Smem *>(smem_raw + (sums - raw) + C::kSums);
    volatile int *abort = &S->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the cluster is a tile's parts (a power of two: no division before the first load)
    const int parts = 1 << log_parts;
    const int tile = static_cast<int>(blockIdx.x) >> log_parts, rank = static_cast<int>(blockIdx.x) & (parts - 1);
    const int nks = static_cast<int>((static_cast<uint32_t>(p.R) + 63u) >> 6);  // R < 2^31
    const int k0 = (rank * nks) >> log_parts;
    const int n_it = (((rank + 1) * nks) >> log_parts) - k0;

    // expansion warps: a warp builds the 32 rows (output channels) 32 (warp % 4) .. + 31
    // of its group's stages.  Its unit lane + 32 j of a stage: weights 8 ug .. + 7 of
    // the 64 K of group g_w + gl.  The first stages' weights are loaded here, while
    // the barriers and the tensor memory are set up.
    const int q = (warp >> 2) & (kGroups - 1);
    const int row_w = (warp & 3) * 32;
    const int lg = 31 - __clz(p.G);  // G is a power of two
    const int U = (8 * K + p.G - 1) >> lg;  // units per lane: 64 * 32 * K / G weights over 32 lanes of 8
    const int64_t g_w = (static_cast<int64_t>(tile) * kM + row_w) >> lg;  // the warp's first group
    const int64_t groups = p.Cout >> lg;
    const int hw = word_flip<K>(lane);
    Unit ring[NB][4];
    auto load = [&](Unit (&u)[4], int it) {
        const int r0 = (k0 + it) * 64;
        const int64_t left = (p.R - r0) * K;  // weights of a group from r0 on
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= U) break;
            const int e = lane + 32 * j, gl = e / kUG, ug = e % kUG;
            u[j].in = gl < (32 >> lg) && g_w + gl < groups && 8 * ug < left;
            if (u[j].in) {
                const int64_t off = ((g_w + gl) * p.R + r0) * K + 8 * ug;
                u[j].v = __ldg(reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(p.values) + off));
                u[j].i = __ldg(reinterpret_cast<const uint2 *>(p.idx + off));
            }
        }
    };
    tc::wait_prior_grid();  // a programmatic dependent of the kernel before it
    if (warp < 4 * kGroups) {
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (q + kGroups * b < n_it) load(ring[b], q + kGroups * b);
    }

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&S->full[s], 4);
            tc::mbar_init(&S->xfull[s], 1);
            tc::mbar_init(&S->empty[s], 1);
        }
        tc::mbar_init(&S->done, 1);
        S->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4 * kGroups + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc::smem_u32(&S->tmem_base)),
                     "r"(C::kTmem)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32 * 4 * kGroups) tc::tma_prefetch_desc(&tmX);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = S->tmem_base;
    // the next grid may be scheduled from here on: this block holds its tensor memory,
    // so a block of the next grid that takes some and then waits for this grid cannot
    // keep this one from its own
    tc::launch_next_grid();
    // the wait for this arrival, before the first store into another CTA, sees that
    // every CTA of the cluster runs
    if (parts > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    if (warp < 4 * kGroups) {
        // ---- expansion: group q builds the stages q, q + 4, ...
        bool bad = false, ok = true;
        int s = q;  // kGroups <= kStages
        uint32_t ph = 1u;  // a fresh barrier's preceding phase counts as complete
        for (int it = q; it < n_it && ok;) {
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                if (it >= n_it) break;
                ok = tc::mbar_wait(&S->empty[s], ph, abort, p.status);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                const uint32_t rows = base + s * C::kStage + static_cast<uint32_t>(row_w) * 128u;
#pragma unroll
                for (int z = 0; z < 8; ++z) tc::st_shared_v4_zero(rows + static_cast<uint32_t>(lane + 32 * z) * 16u);
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j >= U) break;
                    if (!ring[b][j].in) continue;
                    const int e = lane + 32 * j, gl = e / kUG, ug = e % kUG;
                    bad |= unit_bad<K>(ring[b][j].i, p.G);
                    scatter_unit<K>(ring[b][j], rows, gl << lg, 8 * ug, hw, p.G);
                }
                if (it + kGroups * NB < n_it) load(ring[b], it + kGroups * NB);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&S->full[s]);
                it += kGroups;
                s += kGroups;
                if (s >= kStages) {
                    s -= kStages;
                    ph ^= 1u;
                }
            }
        }
        if (bad) report(p.status, CCI_ERR_INDEX);
    } else if (warp == 4 * kGroups) {
        // ---- activations: the [NP][64] tile of each stage, rows past N filled with zero
        if (tc::elect_one()) {
            int s = 0, it = 0;
            uint32_t ph = 1u;
            for (; it < n_it; ++it) {
                if (!tc::mbar_wait(&S->empty[s], ph, abort, p.status)) break;
                tc::mbar_arrive_expect_tx(&S->xfull[s], NP * 128);
                tc::tma_load_2d(base + s * C::kStage + kABytes, &tmX, (k0 + it) * 64, 0, &S->xfull[s]);
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            // no copy is in flight when the block ends, also after an abort
            int no_abort = 0;
            for (int d = it > kStages ? it - kStages : 0; d < it; ++d)
                tc::mbar_wait(&S->xfull[d % kStages], (d / kStages) & 1, &no_abort, p.status);
        }
        __syncwarp();
    } else {
        if (tc::elect_one()) {
            int s = 0;
            uint32_t ph = 0u;
            const uint64_t desc0 = tc::sw128_desc(base);
            const uint32_t empty0 = tc::smem_u32(&S->empty[0]);
            for (int it = 0; it < n_it; ++it) {
                if (!tc::mbar_wait(&S->xfull[s], ph, abort, p.status)) break;
                if (!tc::mbar_wait(&S->full[s], ph, abort, p.status)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t ad = desc0 + static_cast<uint64_t>(s) * (C::kStage >> 4);
                ws::stage_f16<C::kIdesc>(tmem, ad, ad + (kABytes >> 4), it > 0 ? 1u : 0u, 1u, empty0 + 8u * s);
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            tc::mma_commit(&S->done);
        }
        __syncwarp();
    }

    // ---- the sums, one output channel per TMEM lane
    int no_abort = 0;
    const bool summed = tc::mbar_wait(&S->done, 0, &no_abort, p.status);
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (parts > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    const int m = (warp & 3) * 32 + lane;
    if (warp < 4 * kGroups && __all_sync(0xffffffffu, summed)) {
        const uint32_t lanes = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int64_t co = static_cast<int64_t>(tile) * kM + m;
        const float b = p.bias && co < p.Cout ? __ldg(p.bias + co) : 0.f;
        for (int c0 = (warp >> 2) * 32; c0 < NP; c0 += 32 * kGroups) {
            uint32_t v[32];
            tc::tmem_ld32(lanes + static_cast<uint32_t>(c0), v);
            if (parts == 1) {
                // a warp's 32 channels of a column are consecutive in Y
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int n = c0 + j;
                    if (n >= p.N || co >= p.Cout) continue;
                    store_y(p, n, co, finish(__uint_as_float(v[j]), p, b));
                }
            } else {
                // column quad c to CTA c mod parts, block c - c mod parts + this part of
                // [128 channels][4 columns]: 512 consecutive bytes a warp and store
                const uint32_t mask = static_cast<uint32_t>(parts - 1);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t c = static_cast<uint32_t>(c0 / 4 + j);
                    if (c0 + 4 * j < NP && c0 + 4 * j < p.N)
                        st_cluster_v4(ws::map_to_rank(sums + ((c & ~mask) + static_cast<uint32_t>(rank)) * (kM * 16u) +
                                                          static_cast<uint32_t>(m) * 16u, c & mask),
                                      v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (parts > 1) {
        ws::cluster_sync();  // every part's sums have landed; nothing is stored to another CTA after
        // one channel of one of this CTA's column quads per thread
        const int64_t co = static_cast<int64_t>(tile) * kM + (tid & 127);
        if (warp < 4 * kGroups && co < p.Cout) {
            const float b = p.bias ? __ldg(p.bias + co) : 0.f;
            for (int i = tid >> 7; 4 * (i * parts + rank) < p.N; i += kGroups) {
                const uint32_t at =
                    sums + static_cast<uint32_t>(i * parts) * (kM * 16u) + static_cast<uint32_t>(tid & 127) * 16u;
                float4 y = ld_shared_f4(at);
                for (int j = 1; j < parts; ++j) {
                    const float4 z = ld_shared_f4(at + static_cast<uint32_t>(j) * (kM * 16u));
                    y.x += z.x;
                    y.y += z.y;
                    y.z += z.z;
                    y.w += z.w;
                }
                const int n = 4 * (i * parts + rank);
                const float o[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (n + t < p.N) store_y(p, n + t, co, finish(o[t], p, b));
            }
        }
    }
    __syncthreads();
    if (warp == 4 * kGroups + 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmem) : "memory");
    }
}

// clusters of 1 << log_parts CTAs (one per SM; log_parts 1, 2 or 3) that a launch
// counts on running at once.  They stay inside a GPC, so larger ones leave SMs over:
// on 152 SMs 76, 35 and 15 (36 clusters of four were seen resident)
int64_t cluster_slots(int log_parts, int64_t sms)
{
    return log_parts == 1 ? sms / 2 : (log_parts == 2 ? sms * 15 / 64 : sms / 10);
}

template <int K, int NP>
cudaError_t launch(const FwdParams &p, cudaStream_t stream)
{
    using C = Cfg<NP>;
    CUtensorMap tmX{};
    const int64_t dims[2] = {p.Cin, p.N};
    const int box[2] = {64, NP};
    if (!ws::make_map(&tmX, p.X, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, dims, box)) return cudaErrorNotSupported;
    static SmemAttrCache attr_cache;
    const cudaError_t attr = smem_attr_once(narrow_kernel<K, NP>, static_cast<int>(C::kSmem), attr_cache);
    if (attr != cudaSuccess) return attr;
    const int64_t tiles = (p.Cout + kM - 1) / kM, nks = (p.R + 63) / 64;
    // parts of the reduction: doubled while the SMs hold them all and each keeps
    // kMinStages stages
    const int64_t sms = ws::sm_count();
    int log_parts = 0;
    while ((2 << log_parts) <= kMaxParts && tiles <= cluster_slots(log_parts + 1, sms) &&
           nks >= kSplitStages && nks >= (2 << log_parts) * kMinStages)
        ++log_parts;
    const int parts = 1 << log_parts;
    if (tiles * parts > 0x7fffffff) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(tiles * parts));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute la[2];
    la[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    la[0].val.programmaticStreamSerializationAllowed = 1;
    la[1].id = cudaLaunchAttributeClusterDimension;
    la[1].val.clusterDim.x = static_cast<unsigned>(parts);
    la[1].val.clusterDim.y = 1;
    la[1].val.clusterDim.z = 1;
    cfg.attrs = la;
    cfg.numAttrs = parts > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, narrow_kernel<K, NP>, p, tmX, log_parts);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int K>
cudaError_t launch_n(const FwdParams &p, cudaStream_t stream)
{
    // the MMA's N: the columns rounded up
    if (p.N <= 16) return launch<K, 16>(p, stream);
    if (p.N <= 32) return launch<K, 32>(p, stream);
    if (p.N <= 64) return launch<K, 64>(p, stream);
    return launch<K, 128>(p, stream);
}

}  // namespace narrow

bool narrow_ok(const FwdParams &p, int dtype, int64_t N)
{
    const bool gk = (p.G == 4 || p.G == 8 || p.G == 16 || p.G == 32) &&
                    (p.K == 1 || p.K == 2 || p.K == 4 || p.K == 8) && 2 * p.K <= p.G;
    auto at16 = [](const void *q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    const int64_t lim = int64_t(1) << 31, nks = (p.R + 63) / 64;
    return dtype == CCI_BF16 && !p.is_conv && N > 0 && N <= narrow::kMaxN && gk && p.Cin == p.R && p.R % 8 == 0 &&
           (nks <= narrow::kWholeStages || nks >= narrow::kSplitStages) && p.R < lim && p.Cout < lim && at16(p.X) &&
           at16(p.Y) && at16(p.values) && at16(p.idx);
}

cudaError_t launch_narrow(const FwdParams &p, cudaStream_t stream)
{
    switch (p.K) {
        case 1: return narrow::launch_n<1>(p, stream);
        case 2: return narrow::launch_n<2>(p, stream);
        case 4: return narrow::launch_n<4>(p, stream);
        default: return narrow::launch_n<8>(p, stream);
    }
}

}  // namespace cci
