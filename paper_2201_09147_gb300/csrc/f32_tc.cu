// FP32 path on the tensor cores (SDF_FP32 networks): half-precision head and
// remainder operands, FP32-level results (grad32_tc.cuh).
#include "grad32_tc.cuh"

namespace sdfnn {

template <int W>
static cudaError_t launch_grad32(const GradArgs& a, int num_sms, cudaStream_t s) {
    using C = G32<W, 2>;
    return launch_tc(grad32_tc_kernel<W>, C::THREADS, g32_layout<C>().total + 1024, C::TMEM_COLS, num_sms, s, &a);
}

cudaError_t launch_grad32_tc(const GradArgs& a, int num_sms, cudaStream_t s) {
    switch (a.net.width) {
    case 64:
        return launch_grad32<64>(a, num_sms, s);
    case 128:
        return launch_grad32<128>(a, num_sms, s);
    case 256:
        return launch_grad32<256>(a, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sdfnn
