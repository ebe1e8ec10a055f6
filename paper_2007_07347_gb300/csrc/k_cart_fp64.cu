// k_cart_fp64.cu -- FP64 instance of cart_tile's kernel for the TMA staging (built with
// --fmad=false); with plain loads FP64 runs on k_cart64.cu.
#include "step_cart.cuh"

namespace sdugks {

cudaError_t prepare_cart_fp64() { return prepare_mode_p<P_FP64, 16, 16, CART_SPECIALISED_TMA>(); }

cudaError_t launch_cart_fp64_tma(const CartInst &m, const CartTma &tma, int par, cudaStream_t st)
{
    const dim3 grid((m.nx + 15) / 16, (m.ny + 15) / 16);
    return launch_step_kernel(m.early != 0, k_step_cart<P_FP64, 16, 16, CART_SPECIALISED_TMA>, grid, dim3(cart_threads<16, 16>()),
                              cart_step_smem<P_FP64, 16, 16, CART_SPECIALISED_TMA>(), st, m, par, tma.f[par], tma.W[par]);
}

}  // namespace sdugks
