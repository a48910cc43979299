// TMA-staged step kernels for float population storage in a general geometry.
#include "step_tma.cuh"

namespace lbsc {

template <>
long long tma_step_general<float>(int op, int tile_y, int stages, bool tau_one, const CUtensorMap* map,
                                const StepArgs<float>* args, cudaStream_t stream)
{
    return tma_dispatch<float, true>(op, tile_y, stages, tau_one, map, args, stream);
}

}  // namespace lbsc
