// dbm_step_s8.cu -- fused step instantiated for 8 species.
#include "dbm_step_impl.cuh"

namespace dbm {
template int launch_step_t<8>(dbm_handle *, const void *, void *, cudaStream_t);
template int launch_step_staged_t<8, staged_tile_x(8), staged_tile_y(8), staged_cw(8)>(dbm_handle *, const CUtensorMap *, const CUtensorMap *,
                                                                const void *, void *, cudaStream_t);
}  // namespace dbm
