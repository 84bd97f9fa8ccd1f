// Launcher of the resident runs and the complex64 instantiations for circuits
// with folded passes (the others are in sv_resident_c64.cu and
// sv_resident_c128.cu, so that they compile in parallel).
#include "sv_resident.cuh"

namespace sv {

const void* resident_kernel_c64(int threads);  // no folded passes
const void* resident_kernel_c128(int threads);

namespace {

template <class R> size_t res_smem(const ResDesc& p) {
    const size_t warps = resident_threads(sizeof(R) == 8, p.np) / 32, mb = p.mb;
    return ((size_t)1 << p.np) * sizeof(typename Cplx<R>::T) + 2 * mb * p.block_words * 4 + mb * p.max_stages * 16 +
           (p.folds ? mb * (16 * FOLD_SPARSE + 8 * FOLD_LD) * 16 : 0) + mb * p.br_bytes + MAX_PEND * 8 +
           warps * MAX_RED * 8 + RES_FINAL_BLOCKS * 8 + MAX_PEND * 4 + (((size_t)p.n_rows + 15) & ~(size_t)15);
}

const void* res_fn(int prec, int folds, int threads) {
    if (prec) return resident_kernel_c128(threads);
    if (!folds) return resident_kernel_c64(threads);
    return threads > 128 ? (const void*)k_resident<float, 512, true> : (const void*)k_resident<float, 128, true>;
}

// open addressing, at most half full; 0 marks a free slot
__global__ void k_history_count(const unsigned long long* hist, uint64_t n, unsigned long long* tab, uint64_t mask,
                                unsigned long long runs) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned long long h = hist[i] ? hist[i] : 1ull;
    for (uint64_t k = 0; k <= mask; ++k) {
        const unsigned long long old = atomicCAS(tab + HIST_COUNTS + ((h + k) & mask), 0ull, h);
        if (old == h) return;
        if (old == 0) {
            atomicAdd(tab, runs);
            atomicAdd(tab + 1, 1ull);
            return;
        }
    }
}

}  // namespace

cudaError_t launch_history_count(const unsigned long long* hist, uint64_t n, unsigned long long* tab,
                                 unsigned long long runs, cudaStream_t s) {
    const size_t slots = history_slots(n);
    cudaError_t e = cudaMemsetAsync(tab + 1, 0, 8 * (HIST_COUNTS - 1 + slots), s);
    if (e != cudaSuccess) return e;
    k_history_count<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(hist, n, tab, slots - 1, runs);
    return cudaGetLastError();
}

// Warps of a CTA and blocks prepared side by side: a warp per 32 groups of 16
// amplitudes while several CTAs fit an SM (their number, not the width of
// one, hides the latency chains), eight at 2^13 amplitudes, where shared
// memory leaves room for two CTAs, and sixteen at 2^14, for one.
int resident_threads(int prec, int np) {
    if (prec) return np >= 13 ? 256 : (np >= 11 ? 128 : (np == 10 ? 64 : 32));
    return np >= 14 ? 512 : (np >= 13 ? 256 : (np >= 11 ? 128 : (np == 10 ? 64 : 32)));
}
int resident_batch(int prec, int np) {
    const int warps = resident_threads(prec, np) / 32;
    return warps < 4 ? warps : (np >= 14 ? RES_MAX_BATCH : 4);
}

size_t resident_smem_bytes(int prec, const ResDesc& p) { return prec ? res_smem<double>(p) : res_smem<float>(p); }

cudaError_t init_resident() {
    cudaError_t e = cudaSuccess;
    for (int prec = 0; prec < 2; ++prec)
        for (int t : {128, 512})
            for (int folds = 0; folds < 2 && e == cudaSuccess; ++folds)
                e = cudaFuncSetAttribute(res_fn(prec, folds, t), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)RES_MAX_SMEM);
    return e;
}

cudaError_t launch_resident(const DevBatch& d, int prec, const ResDesc& p, int n_states, int n_sm, cudaStream_t s) {
    const int threads = resident_threads(prec, p.np);
    const size_t smem = resident_smem_bytes(prec, p);
    const void* f = res_fn(prec, p.folds, threads);
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int grid = n_states < per_sm * n_sm ? n_states : per_sm * n_sm;
    ResDesc r = p;
    r.n_states = n_states;
    void* args[] = {(void*)&d, (void*)&r};
    return cudaLaunchKernel(f, dim3(grid), dim3(threads), args, smem, s);
}

}  // namespace sv
