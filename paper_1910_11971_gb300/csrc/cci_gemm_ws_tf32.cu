// cci_gemm_ws_tf32.cu -- fp32 layers of the workspace family (the split product:
// tf32 hi*hi plus bf16 cross terms): the kernel configurations and the choice
// among them.
#include "cci_gemm_ws.cuh"

namespace cci {

cudaError_t launch_gemm_ws_tf32(const FwdParams &p, cudaStream_t stream)
{
    using namespace ws;
    Plan pl;
    plan_layer(p, true, 32, &pl);
    const int asrc = pl.asrc;
    // few tiles with a long reduction: split over clusters
    const int64_t mt = call_m_tiles(p, m_tiles_of(p, asrc, pl.box)), stages = (p.R + 31) / 32;
    // (gathered fp32 stages of 128-wide tiles would be two: 64-wide ones only)
    const Split sp = asrc == kAGather ? choose_split(mt, p.Cout, stages, 1400, 1 << 20)
                                      : choose_split(mt, p.Cout, stages, 480, 560);
    if (sp.log_parts > 0) {
#define CCI_WS_SPLIT(A, N)        \
    if (asrc == A && sp.bn == N) \
        return launch_cfg<true, A, N, 1, 1, false, false, true>(p, pl.box, pl.am, stream, sp.log_parts);
        CCI_WS_SPLIT(kA2d, 64)
        CCI_WS_SPLIT(kA2d, 128)
        CCI_WS_SPLIT(kA4d, 64)
        CCI_WS_SPLIT(kA4d, 128)
        CCI_WS_SPLIT(kAGather, 64)
#undef CCI_WS_SPLIT
    }
    const int bn = choose_bn(m_tiles_of(p, asrc, pl.box), p.Cout, 128);
    // TMA-copied activations: clusters of two CTAs on adjacent M tiles share each
    // weight tile by multicast (half the weight copies per CTA)
#define CCI_WS_MC(A, N) \
    if (asrc == A && bn == N) return launch_cfg<true, A, N, 1, 1, false, true>(p, pl.box, pl.am, stream);
    CCI_WS_MC(kA2d, 64)
    CCI_WS_MC(kA2d, 128)
    CCI_WS_MC(kA4d, 64)
    CCI_WS_MC(kA4d, 128)
#undef CCI_WS_MC
#define CCI_WS_CASE(A, N) \
    if (asrc == A && bn == N) return launch_cfg<true, A, N, 1>(p, pl.box, pl.am, stream);
    CCI_WS_CASE(kAGather, 64)
    CCI_WS_CASE(kAGather, 128)
#undef CCI_WS_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_gemm_ws(const FwdParams &p, int dtype, cudaStream_t stream)
{
    return dtype == CCI_F32 ? launch_gemm_ws_tf32(p, stream) : launch_gemm_ws_bf16(p, stream);
}

}  // namespace cci
