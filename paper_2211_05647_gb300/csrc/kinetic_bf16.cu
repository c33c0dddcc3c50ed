// kinetic_bf16.cu -- BF16-storage instances of the plasma-row kernel (FP32
// arithmetic, stochastic rounding on store); see kinetic_impl.cuh.
#include "kinetic_impl.cuh"

namespace fp {

cudaError_t dispatch_kinetic_bf16(cudaStream_t st, const KinArgs<float> &a, int num_sms, int vpl, int l, int bps)
{
    return dispatch_kinetic<__nv_bfloat16, float>(st, a, num_sms, vpl, l, bps);
}

// rows of V = 16 .. 128 vectors, eight a lane, J summed as the (4, V / 4) shape sums it
cudaError_t dispatch_kinetic_bf16_wide(cudaStream_t st, const KinArgs<float> &a, int num_sms)
{
    switch (a.pitch / 8) {
    case 16: return run_kinetic<__nv_bfloat16, float, 8, 2, 4>(st, a, num_sms, 0);
    case 32: return run_kinetic<__nv_bfloat16, float, 8, 4, 4>(st, a, num_sms, 0);
    case 64: return run_kinetic<__nv_bfloat16, float, 8, 8, 4>(st, a, num_sms, 0);
    case 128: return run_kinetic<__nv_bfloat16, float, 8, 16, 4>(st, a, num_sms, 0);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fp
