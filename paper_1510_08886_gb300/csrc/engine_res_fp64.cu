// Resident-chunk engine kernels, fp64 population storage and arithmetic.
// Compiled once per velocity set with LBM_RES_SET naming it, for that set's
// kernels, and once without, for the dispatch: the unrolled collisions of all
// sets (three wraps in x, two kinds of step, with and without a force) make one
// unit several times slower to compile than any other.
#include "engine_launch.cuh"

namespace lbm {

#define LBM_RES_UNIT(PREFIX, SET, N)                                                             \
    PREFIX template cudaError_t resident_one<SET, N, double>(const ResidentLaunch&, cudaStream_t); \
    PREFIX template int resident_attr_one<SET, N, double>(size_t);
#define LBM_RES_UNITS(PREFIX, SET) \
    LBM_RES_UNIT(PREFIX, SET, 2) LBM_RES_UNIT(PREFIX, SET, 3) LBM_RES_UNIT(PREFIX, SET, 4)

#ifdef LBM_RES_SET

LBM_RES_UNITS(, LBM_RES_SET)

#else

LBM_RES_UNITS(extern, SetD2V16)
LBM_RES_UNITS(extern, SetD2V32)
LBM_RES_UNITS(extern, SetD2V33)
LBM_RES_UNITS(extern, SetD2V53)
LBM_RES_UNITS(extern, SetD2V40)
LBM_RES_UNITS(extern, SetD2V48)

cudaError_t engine_resident_fp64(int set_id, int N, const ResidentLaunch& L, cudaStream_t st) {
    return engine_resident_t<double>(set_id, N, L, st);
}

int engine_resident_attr_fp64(int set_id, int N, size_t smem) {
    return engine_resident_attr_t<double>(set_id, N, smem);
}

#endif

}  // namespace lbm
