// fp64 instantiations of the stream-collide kernels: storage and arithmetic
// in double.
#include "lbm_kernels.cuh"

namespace lbm {

cudaError_t launch_step_fp64(const KParams<double>& k, int N, const void* src, void* dst,
                             const DevBufs& b, cudaStream_t st) {
    return launch_step_t<double, double>(k, N, src, dst, b, st);
}

cudaError_t launch_init_fp64(const KParams<double>& k, int N, const double* rho0, void* dst,
                             const DevBufs& b, cudaStream_t st) {
    return launch_init_t<double, double>(k, N, rho0, dst, b, st);
}

cudaError_t allow_step_scratch_fp64(int set_id, int N) {
    switch (set_id) {
        case 0: return allow_scratch_n<SetD2V16>(N);
        case 1: return allow_scratch_n<SetD2V32>(N);
        case 2: return allow_scratch_n<SetD2V33>(N);
        case 3: return allow_scratch_n<SetD2V53>(N);
        case 4: return allow_scratch_n<SetD2V40>(N);
        case 5: return allow_scratch_n<SetD2V48>(N);
        default: return cudaSuccess;             // the generic kernel has no scratch
    }
}

}  // namespace lbm
