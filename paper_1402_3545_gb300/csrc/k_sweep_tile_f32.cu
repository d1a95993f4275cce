// k_sweep_tile_f32.cu -- the whole-column sweeps (sweep_tile.cuh) of one arithmetic policy.
#include "sweep_tile.cuh"

namespace tpmg {

template int launch_sweep_tile<PolF32, MODE_SMOOTH>(const Lv<PolF32>&, double, const PolF32::S*, const PolF32::S*, PolF32::S*, double*,
    const int*, cudaStream_t);
template int launch_sweep_tile<PolF32, MODE_LINESOLVE>(const Lv<PolF32>&, double, const PolF32::S*, const PolF32::S*, PolF32::S*, double*,
    const int*, cudaStream_t);
template int cg_tile_blocks<PolF32>(const Lv<PolF32>&);
template int launch_cg_tile<PolF32>(const Lv<PolF32>&, const Scalars*, PolF32::S*, const PolF32::S*, PolF32::S*, double*, cudaStream_t);

}  // namespace tpmg
