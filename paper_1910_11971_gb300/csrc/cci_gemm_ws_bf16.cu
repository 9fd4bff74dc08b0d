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
    // CTA pairs (256-row tiles, B split over the pair) halve each SM's B traffic.  With
    // 256-wide N tiles that pays on long reductions of more than one round of pairs:
    // a single round starts and ends faster on single CTAs (512 -> 512 at 7 x 7, 128
    // images 28.0 us paired, 26.5 single)
    const int64_t pairs = sm_count() / 2;
    auto pair_units = [&](int64_t mt, int bn) { return (mt + 1) / 2 * ((p.Cout + bn - 1) / bn); };
    const bool pair = (asrc == kA2d || is_box(asrc)) && nks >= 16 && choose_bn(m_tiles, p.Cout, 256, 2) == 256 &&
                      pair_units(m_tiles, 256) > pairs;
    if (pair) {
        if (asrc == kA2d) return launch_cfg<false, kA2d, 256, 2>(p, pl.box, pl.am, stream);
        if (asrc == kATap) return launch_cfg<false, kATap, 256, 2>(p, pl.box, pl.am, stream);
        return launch_cfg<false, kA4d, 256, 2>(p, pl.box, pl.am, stream);
    }
    if (asrc == kAHalo) {
        // 3x3 convolutions from halo copies: pairs with 128-wide N tiles (each CTA copying
        // its own halo and half of every weight tile, 8 KB a stage for 256 cycles of
        // MMAs) for every layer but those of 64 channels out.  Images narrower than the
        // tile leave rows of a halo tile unused; where pairs of per-tap boxes, which span
        // images, take fewer rounds, those (256 -> 256 at 14 x 14, 128 images 25.7 us in
        // four rounds of halos, 24.4 in three of boxes)
        if (p.Cin >= 128 && p.Cout > 64 && m_tiles > 1) {
            const int64_t m4 = m_tiles_of(p, kA4d, pl.a4d);
            if ((pair_units(m4, 128) + pairs - 1) / pairs < (pair_units(m_tiles, 128) + pairs - 1) / pairs) {
                plan_layer(p, false, 64, &pl, -1);
                return launch_cfg<false, kA4d, 128, 2>(p, pl.box, pl.am, stream);
            }
            return launch_cfg<false, kAHalo, 128, 2>(p, pl.box, pl.am, stream);
        }
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
    // per-tap boxes of long reductions, 128-wide N tiles, three rounds of pairs or more
    // (256 -> 256, stride 2 at 28 x 28, 128 images: 29.2 us single, 26.5 paired; at 32
    // images, one round, 12.0 and 12.7)
    if (asrc == kA4d && nks >= 16 && bn == 128 && pair_units(m_tiles, 128) > 2 * pairs)
        return launch_cfg<false, kA4d, 128, 2>(p, pl.box, pl.am, stream);
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
