// inst_f32_d2q9.cu -- kernels and launchers of D2Q9 with the StoreF32 population format
#include "lbm_kernels.cuh"

namespace lbm {
const Dispatch& dispatch_f32_d2q9()
{
    static const Dispatch d = make_dispatch<9, StoreF32>();
    return d;
}
}  // namespace lbm
