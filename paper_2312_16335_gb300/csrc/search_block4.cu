// Block-per-query search instantiations for LVQ-4 primaries (small batches).
#include "beam_block.cuh"

namespace lv {

int launch_search_block4(const BeamParams &p, int nc, size_t smem, cudaStream_t st) {
    switch (nc) {
        case 1: return launch_block_nc<1, 4>(p, smem, st);
        case 2: return launch_block_nc<2, 4>(p, smem, st);
        case 3: return launch_block_nc<3, 4>(p, smem, st);
        default: return fail(LV_ERR_ARG, "search: primary dimension too large for LVQ-4 (d <= 352)");
    }
}

}  // namespace lv
