// k_sweep_tile_dw.cu -- the whole-column sweeps (sweep_tile.cuh) of one arithmetic policy.
#include "sweep_tile.cuh"

namespace tpmg {

template int launch_sweep_tile<PolDW, MODE_SMOOTH>(const Lv<PolDW>&, double, const PolDW::S*, const PolDW::S*, PolDW::S*, double*,
    const int*, cudaStream_t);
template int launch_sweep_tile<PolDW, MODE_LINESOLVE>(const Lv<PolDW>&, double, const PolDW::S*, const PolDW::S*, PolDW::S*, double*,
    const int*, cudaStream_t);
template int cg_tile_blocks<PolDW>(const Lv<PolDW>&);
template int launch_cg_tile<PolDW>(const Lv<PolDW>&, const Scalars*, PolDW::S*, const PolDW::S*, PolDW::S*, double*, cudaStream_t);

}  // namespace tpmg
