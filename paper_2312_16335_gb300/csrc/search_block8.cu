// Block-per-query search instantiations for LVQ-8 primaries (small batches).
#include "beam_block.cuh"

namespace lv {

int launch_search_block8(const BeamParams &p, int nc, size_t smem, cudaStream_t st) {
    switch (nc) {
        case 1: return launch_block_nc<1, 8>(p, smem, st);
        case 2: return launch_block_nc<2, 8>(p, smem, st);
        case 3: return launch_block_nc<3, 8>(p, smem, st);
        case 4: return launch_block_nc<4, 8>(p, smem, st);
        default: return fail(LV_ERR_ARG, "search: primary dimension too large for LVQ-8 (d <= 240)");
    }
}

}  // namespace lv
