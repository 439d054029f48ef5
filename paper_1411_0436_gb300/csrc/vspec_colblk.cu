// vspec_colblk.cu — instances of the blocked kernel A (vspec_colblk.cuh).
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_colblk.cuh"

namespace {
template <int N2, int PT, int NPOL> const void *instance(size_t *smem) {
    *smem = vspec::ColBlk<N2, PT>::smem;
    return (const void *)vspec::fir_colblk_kernel<N2, PT, NPOL>;
}
template <int N2, int NPOL> const void *by_taps(int P, size_t *smem) {
    if constexpr (N2 == 512)
        if (P <= 1) return instance<N2, 1, NPOL>(smem);
    if constexpr (N2 < 512 || NPOL == 2)
        if (P > 8) return instance<N2, 16, NPOL>(smem);
    return instance<N2, 8, NPOL>(smem);
}
}  // namespace

// Kernel A for columns of N2 points and P taps, its dynamic shared memory in
// *smem; nullptr where there is none.
const void *vspec_pick_kernel_colblk(int N2, int npol, int P, size_t *smem) {
    // (2^20 single-pol with more than 8 taps: 8-byte tile rows of two frame sets
    // of 17 make a run's start too dear, 5 spectra 241 -> 262 us)
    if (N2 == 512) return npol == 2 ? by_taps<512, 2>(P, smem) : P <= 8 ? by_taps<512, 1>(P, smem) : nullptr;
    if (npol == 1 && N2 == 256) return by_taps<256, 1>(P, smem);
    if (npol == 1 && N2 == 128) return by_taps<128, 1>(P, smem);
    return nullptr;
}

// The kernels' bounds-check status word (debug builds), as vspec_ring_debug_flags.
cudaError_t vspec_colblk_debug_flags(unsigned *flags, bool clear) {
#ifdef VSPEC_DEBUG
    cudaError_t e = cudaMemcpyFromSymbol(flags, vspec::g_debug_flags, sizeof(unsigned));
    if (e != cudaSuccess || !clear) return e;
    const unsigned zero = 0;
    return cudaMemcpyToSymbol(vspec::g_debug_flags, &zero, sizeof(unsigned));
#else
    *flags = 0;
    (void)clear;
    return cudaSuccess;
#endif
}
