// dbm_step_s8.cu -- fused step instantiated for 8 species.
#include "dbm_step_impl.cuh"

namespace dbm {
template int launch_step_t<8>(dbm_handle *, const void *, void *, cudaStream_t);
template int launch_step_staged_t<8, PAIR_TX, PAIR_TY, 2>(dbm_handle *, const CUtensorMap *, const CUtensorMap *,
                                     const void *, void *, cudaStream_t);
template int launch_step_staged_t<8, STAGED_TX, STAGED_TY, 1>(dbm_handle *, const CUtensorMap *, const CUtensorMap *,
                                     const void *, void *, cudaStream_t);
}  // namespace dbm
