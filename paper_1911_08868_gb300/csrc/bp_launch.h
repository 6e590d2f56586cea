// Per-length launch entry points of the decoder kernels (one set per n):
// bp_* from bp_inst.cu (per-stage kernel, used for the trace entry), bp2_*
// from bp_inst2.cu (stage-grouped kernel), bp3_* from
// bp_inst3.cu (stage-grouped kernel with TMEM-resident group interiors,
// bp_decode with exact box-plus for n = 7..11), bp4_* from bp_inst4.cu
// (register-resident kernel, bp_decode otherwise).
#pragma once

#include <cuda_runtime.h>

#include "pcbp_internal.h"

namespace pcbp {

struct LaunchGeom {
    int grid;
    int slots;
    size_t smem;
};

#define PCBP_DECLARE_LEN(n)                                                                              \
    void bp_shape_##n(int* threads_per_slot_out, size_t* slot_bytes_out);                                \
    int bp_occupancy_##n(const LaunchGeom& g, bool trace, int fkind);                                    \
    cudaError_t bp_launch_##n(const BpParams& P, const LaunchGeom& g, bool trace, int fkind, cudaStream_t st); \
    void bp2_shape_##n(int* threads_per_slot_out, size_t* slot_bytes_out, int* max_slots_out);            \
    int bp2_occupancy_##n(const LaunchGeom& g, int fkind);                                                \
    cudaError_t bp2_launch_##n(const BpParams& P, const LaunchGeom& g, int fkind, cudaStream_t st, bool pdl);

PCBP_DECLARE_LEN(3)
PCBP_DECLARE_LEN(4)
PCBP_DECLARE_LEN(5)
PCBP_DECLARE_LEN(6)
PCBP_DECLARE_LEN(7)
PCBP_DECLARE_LEN(8)
PCBP_DECLARE_LEN(9)
PCBP_DECLARE_LEN(10)
PCBP_DECLARE_LEN(11)

#undef PCBP_DECLARE_LEN

#define PCBP_DECLARE_LEN3(n)                                                                  \
    void bp3_shape_##n(int* threads_per_slot_out, size_t* slot_bytes_out, int* max_slots_out); \
    void bp3_tables_##n(int N, int K, size_t* bytes);                                          \
    int bp3_occupancy_##n(const LaunchGeom& g, int fkind);                                     \
    cudaError_t bp3_launch_##n(const BpParams& P, const LaunchGeom& g, int fkind, cudaStream_t st, bool pdl); \
    cudaError_t bp3_launch_post_##n(const BpParams& P, const LaunchGeom& g, int fkind, cudaStream_t st);

PCBP_DECLARE_LEN3(7)
PCBP_DECLARE_LEN3(8)
PCBP_DECLARE_LEN3(9)
PCBP_DECLARE_LEN3(10)
PCBP_DECLARE_LEN3(11)

#undef PCBP_DECLARE_LEN3

// Lengths and f the register-resident kernel (bp4_*, bp_inst4.cu) is built for.  Scaled min-sum
// at every length: it takes 0.4 to 0.9 of the tensor-memory kernel's time per iteration (the table in
// bp_kernel4.cuh).  Exact box-plus below N = 128 only: its f is 8 times as long, and
// the unrolled iteration no longer fits the instruction cache (N = 256 with events 0.85 times the
// tensor-memory kernel's speed, N = 128 0.96).
constexpr bool warp_kernel_has(int n, int fkind) { return n >= 3 && n <= 11 && (fkind == 0 || n <= 6); }

struct WarpParams;

// CTAs of the register-resident kernel that an SM's tensor memory holds at once below N = 128.
constexpr int kShortCtas = 8;

#define PCBP_DECLARE_LEN4(n)                                                                       \
    void bp4_shape_##n(int K, int slots, int* max_slots_out, size_t* smem_out);                    \
    cudaError_t bp4_launch_##n(const WarpParams& P, const LaunchGeom& g, int fkind, cudaStream_t st, bool pdl); \
    cudaError_t bp4_launch_post_##n(const WarpParams& P, const LaunchGeom& g, cudaStream_t st);

PCBP_DECLARE_LEN4(3)
PCBP_DECLARE_LEN4(4)
PCBP_DECLARE_LEN4(5)
PCBP_DECLARE_LEN4(6)
PCBP_DECLARE_LEN4(7)
PCBP_DECLARE_LEN4(8)
PCBP_DECLARE_LEN4(9)
PCBP_DECLARE_LEN4(10)
PCBP_DECLARE_LEN4(11)

#undef PCBP_DECLARE_LEN4

}  // namespace pcbp
