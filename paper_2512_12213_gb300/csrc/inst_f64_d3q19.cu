// inst_f64_d3q19.cu -- kernels and launchers of D3Q19 with the StoreF64 population format
#include "lbm_kernels.cuh"

namespace lbm {
const Dispatch& dispatch_f64_d3q19()
{
    static const Dispatch d = make_dispatch<19, StoreF64>();
    return d;
}
}  // namespace lbm
