// inst_bf16_d2q9.cu -- kernels and launchers of D2Q9 with the StoreBF16 population format
#include "lbm_kernels.cuh"

namespace lbm {
const Dispatch& dispatch_bf16_d2q9()
{
    static const Dispatch d = make_dispatch<9, StoreBF16>();
    return d;
}
}  // namespace lbm
