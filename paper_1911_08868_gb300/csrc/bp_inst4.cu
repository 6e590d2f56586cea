// Instantiates the register-resident decoder kernel for one code length,
// 2^PCBP_LOGN (compiled once per n = 3..11).
#include "bp_kernel4.cuh"
#include "bp_launch.h"
#include "launch_smem.h"

#ifndef PCBP_LOGN
#error "PCBP_LOGN must be defined"
#endif

#define PCBP_CAT2(a, b) a##b
#define PCBP_CAT(a, b) PCBP_CAT2(a, b)

namespace pcbp {

namespace {
using Geo = G4<PCBP_LOGN>;
static_assert(PCBP_LOGN >= 7 || kShortCtas * Geo::tm_cols() <= 512, "no allocation waits for a CTA of its launch");

// pdl: programmatic dependent launch, the grid may start while the previous
// kernel of the stream still runs (for independent batches).
template <int FK, int WG, int PO = 0>
cudaError_t launch_variant(const WarpParams& P, const LaunchGeom& g, cudaStream_t st, bool pdl)
{
    constexpr auto kern = bp_decode_warp_kernel<PCBP_LOGN, FK, WG, PO>;
    const cudaError_t e = allow_dynamic_smem<kern>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(g.grid));
    cfg.blockDim = dim3(unsigned(g.slots * 32 * Geo::WPF));
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P);
}
}  // namespace

void PCBP_CAT(bp4_shape_, PCBP_LOGN)(int K, int slots, int* max_slots_out, size_t* smem_out)
{
    *max_slots_out = Geo::SLOTS;
    *smem_out = Geo::smem_bytes(K, slots);
}

cudaError_t PCBP_CAT(bp4_launch_, PCBP_LOGN)(const WarpParams& P, const LaunchGeom& g, int fkind, cudaStream_t st,
                                             bool pdl)
{
    const bool wg = (P.job.S.stop_kind & 2) != 0;
    if (fkind) {
        if (!warp_kernel_has(PCBP_LOGN, 1)) return cudaErrorInvalidValue;
        constexpr int FK = PCBP_LOGN <= 6 ? 1 : 0;
        return wg ? launch_variant<FK, 1>(P, g, st, pdl) : launch_variant<FK, 0>(P, g, st, pdl);
    }
    return wg ? launch_variant<0, 1>(P, g, st, pdl) : launch_variant<0, 0>(P, g, st, pdl);
}

// Scaled min-sum with the messages output (CRC stop or none; P.job.post set).
cudaError_t PCBP_CAT(bp4_launch_post_, PCBP_LOGN)(const WarpParams& P, const LaunchGeom& g, cudaStream_t st)
{
#if PCBP_LOGN >= 7
    if ((P.job.S.stop_kind & 2) || P.job.S.fkind) return cudaErrorInvalidValue;
    return launch_variant<0, 0, 1>(P, g, st, false);
#else
    return cudaErrorInvalidValue;
#endif
}

}  // namespace pcbp
