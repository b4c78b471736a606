// inst_f32_d3q19.cu -- kernels and launchers of D3Q19 with the StoreF32 population format
#include "lbm_kernels.cuh"

namespace lbm {
const Dispatch& dispatch_f32_d3q19()
{
    static const Dispatch d = make_dispatch<19, StoreF32>();
    return d;
}
}  // namespace lbm
