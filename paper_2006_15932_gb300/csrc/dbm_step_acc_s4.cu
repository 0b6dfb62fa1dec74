// dbm_step_acc_s4.cu -- the fused step with the FP32 arithmetic options
// (FP64 thermo, stochastic rounding) instantiated for 4 species.
#include "dbm_step_impl.cuh"

namespace dbm {
template int launch_step_tma_t<4, tma_tile_x(4), tma_tile_y(4), 1, 1>(dbm_handle *, const CUtensorMap *, const CUtensorMap *, const void *, void *,
                                     cudaStream_t);
template int launch_step_tma_t<4, tma_tile_x(4), tma_tile_y(4), 1, 2>(dbm_handle *, const CUtensorMap *, const CUtensorMap *, const void *, void *,
                                     cudaStream_t);
template int launch_step_tma_t<4, tma_tile_x(4), tma_tile_y(4), 1, 3>(dbm_handle *, const CUtensorMap *, const CUtensorMap *, const void *, void *,
                                     cudaStream_t);
}  // namespace dbm
