// Conservation sums without any device allocation.
//
// lb_conserved needs a context, and a context allocates its buffers with
// cudaMalloc.  Some callers cannot allocate: code that runs under a memory
// budget owned by another allocator (a framework's caching allocator that
// holds all device memory), or latency-critical loops that must not pay
// cudaMalloc's implicit device synchronisation.  lb_conserved_noalloc serves
// them: the caller passes the populations and the output, both in its own
// device memory, and the only scratch -- one partial sum per
// block -- lives in the file-scope array below, which every GPU that loads
// this library holds until the process exits.
#include <mutex>

#include "gblb.h"
#include "lb_ctx.h"
#include "lb_kernels.cuh"

namespace gblb {

constexpr int kNoAllocMaxPlanes = 4096;  // 2 * nz must not exceed this: the entry point's limit, from when the
                                         // scratch held a sum per plane
constexpr int kNoAllocSlots = 152 * 3;   // blocks of the summing kernel at most

// Scratch shared by every call on a device: slot p holds the five FP64 sums of
// block p.  Each call writes every slot it reads back, so nothing carries over
// from an earlier call; calls that overlap on the GPU race on these slots.
static __device__ __align__(256) double g_noalloc_partials[kNoAllocSlots * 5];

// Blocks of the summing kernel, each with one slot of the scratch: one wave on 152 SMs.
template <class Codec>
constexpr int noalloc_blocks() {
    return 152 * sum_blocks_per_sm<Codec>();
}

// The blocks' sums in a fixed order, then the totals: mass = nodes + sum drho, momentum = sum j,
// energy = (3 theta0 nodes + sum dk) / 2.
__global__ void __launch_bounds__(kRedThreads) k_conserved_finish(const double* __restrict__ partials, int nblocks,
                                                                   double nodes, double theta0,
                                                                   double* __restrict__ out) {
    __shared__ double sh[5][kRedThreads];
    reduce_partials(partials, nblocks, sh);
    const int c = threadIdx.x;
    if (c >= 5) return;
    const double s = sh[c][0];
    out[c] = c == 0 ? nodes + s : c == 4 ? 0.5 * (3.0 * theta0 * nodes + s) : s;
}

template <class Codec>
static void launch_noalloc_sums(const void* populations, const Dims& d, const Consts<typename Codec::R>& K,
                                double theta0, double* partials, double* out, cudaStream_t st) {
    constexpr int nb = noalloc_blocks<Codec>();
    static_assert(nb <= kNoAllocSlots, "one scratch slot per block");
    const auto* f = static_cast<const typename Codec::raw_t*>(populations);
    if (sum_vector_ok<Codec>(populations, d))
        k_conserved<Codec, sum_width<Codec>()><<<nb, kRedThreads, 0, st>>>(f, d, K, partials, 0, d.nz);
    else
        k_conserved<Codec, 1><<<nb, kRedThreads, 0, st>>>(f, d, K, partials, 0, d.nz);
    k_conserved_finish<<<1, kRedThreads, 0, st>>>(partials, nb, (double)(2 * d.plane), theta0, out);
}

}  // namespace gblb

using namespace gblb;

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
double* g_partials_ptr[kMaxDevices] = {};
// Error message of the calling host thread's last failed call (errno-style, so that
// threads failing at the same time do not write one string concurrently).
thread_local std::string g_noalloc_msg;
}  // namespace

extern "C" {

lb_status lb_conserved_noalloc(const void* populations, lb_grid grid, lb_precision precision, double* out,
                               void* cuda_stream) {
    if (!populations || !out) {
        g_noalloc_msg = "lb_conserved_noalloc: null pointer";
        return LB_ERR_ARG;
    }
    if (grid.nx < 1 || grid.ny < 1 || grid.nz < 1 || grid.nx > (1 << 30) || grid.ny > (1 << 30)) {
        g_noalloc_msg = "lb_conserved_noalloc: grid extents must be >= 1";
        return LB_ERR_ARG;
    }
    if (2 * grid.nz > kNoAllocMaxPlanes) {
        g_noalloc_msg = "lb_conserved_noalloc: 2 * nz = " + std::to_string(2 * grid.nz) +
                        " planes exceeds the limit of " + std::to_string(kNoAllocMaxPlanes) + " planes";
        return LB_ERR_ARG;
    }
    if ((int)precision < LB_F64 || (int)precision > LB_F32_S16B) {
        g_noalloc_msg = "lb_conserved_noalloc: unknown precision";
        return LB_ERR_ARG;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        g_noalloc_msg = std::string("lb_conserved_noalloc: cudaGetDevice: ") + cudaGetErrorString(e);
        return LB_ERR_CUDA;
    }
    double* partials = nullptr;
    {
        // First call on a device, with that device current: look up the device address
        // of the scratch array (the host-side symbol is only a stand-in).
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_partials_ptr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_partials);
            if (e != cudaSuccess || !p) {
                g_noalloc_msg = std::string("lb_conserved_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e);
                return LB_ERR_CUDA;
            }
            g_partials_ptr[dev] = static_cast<double*>(p);
        }
        partials = g_partials_ptr[dev];
    }
    Dims d;
    d.nx = (int)grid.nx;
    d.ny = (int)grid.ny;
    d.nz = (int)grid.nz;
    d.plane = grid.nx * grid.ny * grid.nz;
    d.rows = 2 * grid.ny * grid.nz;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const LaunchConsts& lc = lattice_consts();
    switch ((int)precision) {
        case LB_F64: launch_noalloc_sums<CodecF64>(populations, d, lc.kd, lc.theta0, partials, out, st); break;
        case LB_F32: launch_noalloc_sums<CodecF32>(populations, d, lc.kf, lc.theta0, partials, out, st); break;
        case LB_F32_S16F: launch_noalloc_sums<CodecF16>(populations, d, lc.kf, lc.theta0, partials, out, st); break;
        default: launch_noalloc_sums<CodecBF16>(populations, d, lc.kf, lc.theta0, partials, out, st); break;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_noalloc_msg = std::string("lb_conserved_noalloc: launch: ") + cudaGetErrorString(e);
        return LB_ERR_CUDA;
    }
    return LB_OK;
}

const char* lb_conserved_noalloc_error(void) { return g_noalloc_msg.c_str(); }

}  // extern "C"
