// complex64 instantiations of the resident run without folded passes.
#include "sv_resident.cuh"

namespace sv {

const void* resident_kernel_c64(int threads) {
    return threads > 128 ? (const void*)k_resident<float, 512, false> : (const void*)k_resident<float, 128, false>;
}

}  // namespace sv
