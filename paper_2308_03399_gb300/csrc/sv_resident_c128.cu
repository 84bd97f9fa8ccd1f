// complex128 instantiations of the resident run.
#include "sv_resident.cuh"

namespace sv {

const void* resident_kernel_c128(int threads) {
    return threads > 128 ? (const void*)k_resident<double, 256, false> : (const void*)k_resident<double, 128, false>;
}

}  // namespace sv
