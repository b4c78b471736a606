// inst_bf16_d3q19.cu -- kernels and launchers of D3Q19 with the StoreBF16 population format
#include "lbm_kernels.cuh"

namespace lbm {
const Dispatch& dispatch_bf16_d3q19()
{
    static const Dispatch d = make_dispatch<19, StoreBF16>();
    return d;
}
}  // namespace lbm
