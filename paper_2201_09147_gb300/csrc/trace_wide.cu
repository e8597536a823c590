// Launches of trace_wide_kernel (trace_wide.cuh).
#include "trace_wide.cuh"

namespace sdfnn {

template <int W, int OP, bool SPLIT, int TILES = 1>
static cudaError_t launch_wide(const LevelArgs& a, int num_sms, cudaStream_t s) {
    using C = WideCfg<W, OP, SPLIT, TILES>;
    return launch_tc(trace_wide_kernel<W, OP, SPLIT, TILES>, C::THREADS, wide_layout<C, W>(a.net.n_hidden).total + 1024,
                     C::TMEM_COLS, num_sms, s, &a);
}

// Widths 64 and 128 with head and remainder operands, width 256 without.
cudaError_t launch_trace_wide(const LevelArgs& a, int num_sms, cudaStream_t s) {
    const bool f16 = a.net.op_f16 != 0;
    switch (a.net.width) {
    case 64:
        return f16 ? launch_wide<64, kOpF16, true>(a, num_sms, s) : launch_wide<64, kOpBF16, true>(a, num_sms, s);
    case 128:
        return f16 ? launch_wide<128, kOpF16, true>(a, num_sms, s) : launch_wide<128, kOpBF16, true>(a, num_sms, s);
    case 256:
        if (a.n <= static_cast<int64_t>(num_sms) * 128) {
            if (a.net.op_fp8) return launch_wide<256, kOpE4M3, false>(a, num_sms, s);
            return f16 ? launch_wide<256, kOpF16, false>(a, num_sms, s)
                       : launch_wide<256, kOpBF16, false>(a, num_sms, s);
        }
        if (a.net.op_fp8) return launch_wide<256, kOpE4M3, false, 2>(a, num_sms, s);
        return f16 ? launch_wide<256, kOpF16, false, 2>(a, num_sms, s) : launch_wide<256, kOpBF16, false, 2>(a, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sdfnn
