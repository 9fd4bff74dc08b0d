// cci_gemm_ws_bf16.cu -- bf16 layers of the workspace family: the kernel
// configurations (activation source x N tile x CTAs per tile) and the choice
// among them.
#include "cci_gemm_ws.cuh"

namespace cci {

cudaError_t launch_gemm_ws_bf16(const FwdParams &p, cudaStream_t stream)
{
    using namespace ws;
    Plan pl;
    plan_layer(p, false, 64, &pl);
    const int asrc = pl.asrc;
    const int64_t m_tiles = m_tiles_of(p, asrc, pl.box);
    const int64_t nks = stages_of(p, asrc);
    // tiles of at most 4 stages: the output write dominates, two epilogue groups with
    // two staging buffers each, and the weights of a CTA's N tile resident (two chunks
    // of 256 channels or four of 128), when every CTA has one tile or the N tiles leave
    // less than a tenth of the SMs without whole rounds of them; longer ones keep the
    // shared memory for stages
    const int sbn = choose_bn(m_tiles, p.Cout, nks <= 2 ? 256 : 128, 1);
    const int64_t s_ct = (p.Cout + sbn - 1) / sbn, s_slots = resident_slots(s_ct);
    const bool short_k = nks <= 4 && (asrc == kA2d || asrc == kA4d) &&
                         (m_tiles * s_ct <= s_slots || 10 * s_slots >= 9 * sm_count());
    // short products of fewer than 64 reduction indices, and convolutions of fewer than
    // 64 channels, copy only those (stage_k_in; the kernels' q.kin is chosen alike)
    const int kin = short_k || asrc == kATap ? stage_k_in(p, false, asrc, false) : 64;
    if (kin < 64 && !build_a_maps(p, pl.box, asrc, false, kin, &pl.am)) return cudaErrorInvalidValue;
    // few tiles with a long reduction: split over clusters (3x3 layers of halo copies
    // from per-tap boxes)
    {
        const int src = asrc == kAHalo ? kA4d : asrc;
        const int64_t mt = call_m_tiles(p, m_tiles_of(p, src, pl.a4d)), stages = stages_of(p, src);
        const Split sp = src == kAGather ? choose_split(mt, p.Cout, stages, 800, 800)
                                         : choose_split(mt, p.Cout, stages, 220, 265);
        if (sp.log_parts > 0) {
            if (asrc == kAHalo) plan_layer(p, false, 64, &pl, -1);
#define CCI_WS_SPLIT(A, N)       \
    if (src == A && sp.bn == N) \
        return launch_cfg<false, A, N, 1, 1, false, false, true>(p, pl.box, pl.am, stream, sp.log_parts);
            CCI_WS_SPLIT(kA2d, 64)
            CCI_WS_SPLIT(kA2d, 128)
            CCI_WS_SPLIT(kA4d, 64)
            CCI_WS_SPLIT(kA4d, 128)
            CCI_WS_SPLIT(kATap, 64)
            CCI_WS_SPLIT(kATap, 128)
            CCI_WS_SPLIT(kAGather, 64)
            CCI_WS_SPLIT(kAGather, 128)
#undef CCI_WS_SPLIT
        }
    }
    // CTA pairs (256-row tiles, B split over the pair) halve each SM's B traffic,
    // which pays on long reductions with 256-wide N tiles; shorter or narrower
    // layers run faster on single CTAs (measured on the ResNet-50 stack)
    const bool pair = (asrc == kA2d || is_box(asrc)) && nks >= 16 && choose_bn(m_tiles, p.Cout, 256, 2) == 256;
    if (pair) {
        if (asrc == kA2d) return launch_cfg<false, kA2d, 256, 2>(p, pl.box, pl.am, stream);
        if (asrc == kATap) return launch_cfg<false, kATap, 256, 2>(p, pl.box, pl.am, stream);
        return launch_cfg<false, kA4d, 256, 2>(p, pl.box, pl.am, stream);
    }
    if (asrc == kAHalo) {
        // 3x3 convolutions from halo copies (tiles of nine stages per chunk at least)
        // CTA pairs (256-row tiles, each CTA copying its own halo and half of every
        // weight tile) for every layer but the 64 -> 64 ones: a pair's stage brings 8 KB
        // of weights per SM for 256 cycles of MMAs.  With the issue loops lean, 128-wide
        // tiles beat 256-wide ones (256 channels at 14 x 14, 128 images 27.5 -> 26.7 us)
        if (p.Cin >= 128 && p.Cout > 64 && m_tiles > 1)
            return launch_cfg<false, kAHalo, 128, 2>(p, pl.box, pl.am, stream);
        return launch_cfg<false, kAHalo, 64, 1>(p, pl.box, pl.am, stream);  // 64 channels out, or one M tile
    }
    if (short_k) {
#define CCI_WS_SHORT(A, N) \
    if (asrc == A && sbn == N) return launch_cfg<false, A, N, 1, 2>(p, pl.box, pl.am, stream);
        CCI_WS_SHORT(kA2d, 64)
        CCI_WS_SHORT(kA2d, 128)
        CCI_WS_SHORT(kA2d, 256)
        CCI_WS_SHORT(kA4d, 64)
        CCI_WS_SHORT(kA4d, 128)
        CCI_WS_SHORT(kA4d, 256)
#undef CCI_WS_SHORT
    }
    const int bn = choose_bn(m_tiles, p.Cout, 256, 1);
#define CCI_WS_CASE(A, N) \
    if (asrc == A && bn == N) return launch_cfg<false, A, N, 1>(p, pl.box, pl.am, stream);
    CCI_WS_CASE(kA2d, 64)
    CCI_WS_CASE(kA2d, 128)
    CCI_WS_CASE(kA2d, 256)
    CCI_WS_CASE(kA4d, 64)
    CCI_WS_CASE(kA4d, 128)
    CCI_WS_CASE(kA4d, 256)
    CCI_WS_CASE(kATap, 64)
    CCI_WS_CASE(kATap, 128)
    CCI_WS_CASE(kATap, 256)
    CCI_WS_CASE(kAGather, 64)
    CCI_WS_CASE(kAGather, 128)
    CCI_WS_CASE(kAGather, 256)
#undef CCI_WS_CASE
    return cudaErrorInvalidValue;
}

}  // namespace cci
