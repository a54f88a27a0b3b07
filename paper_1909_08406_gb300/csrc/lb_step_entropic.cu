// The update with the exact entropic equilibrium (Eqs. (discreteentropiceq),
// (fivelagrangemultipliersystem)): k_step with a per-node Newton solve of the
// five Lagrange multipliers, FP32 arithmetic for FP32/FP16/BF16 storage.
// eq 3: with the entropic path length (entropic_path).  (The FP64 mode instantiates the same
// kernel in lb_step_f64.cu.)
#include "lb_kernels.cuh"

namespace gblb {

cudaError_t launch_step_entropic(int prec, int eq, const void* src, void* dst, const Dims& d, const LaunchConsts& c,
                                 double twobeta, int* err, cudaStream_t st) {
    auto run = [&](auto codec) {
        using C = decltype(codec);
        return launch_entries<kNode>(eq == 3 ? k_step<C, 3, true> : k_step<C, 2, true>, src, dst, d, st,
                                     step_consts<C, 2>(c), (float)twobeta, err, 0u);
    };
    switch (prec) {
        case kF32: return run(CodecF32{});
        case kF16: return run(CodecF16{});
        case kBF16: return run(CodecBF16{});
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gblb
