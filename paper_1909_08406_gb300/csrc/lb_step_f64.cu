// FP64 step kernel (parity mode).
#include "lb_kernels.cuh"

namespace gblb {

cudaError_t launch_step_f64(int eq, const void* src, void* dst, const Dims& d, const LaunchConsts& c,
                            double twobeta, int* err, cudaStream_t st) {
    switch (eq) {
        case 3: return launch_entries<kNode>(k_step<CodecF64, 3, true>, src, dst, d, st, step_consts<CodecF64, 2>(c), twobeta, err, 0u);
        case 2: return launch_entries<kNode>(k_step<CodecF64, 2, true>, src, dst, d, st, step_consts<CodecF64, 2>(c), twobeta, err, 0u);
        case 1: return launch_entries<kNode>(k_step<CodecF64, 1, true>, src, dst, d, st, c.sd, twobeta, err, 0u);
        default: return launch_entries<kNode>(k_step<CodecF64, 0, true>, src, dst, d, st, c.sd, twobeta, err, 0u);
    }
}

}  // namespace gblb
