// vspec_rowbatch.cu — instances of the one-row kernel (vspec_rowbatch.cuh).
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_rowbatch.cuh"

namespace {
template <int N, int NPOL, int PT> const void *instance(size_t *smem) {
    *smem = vspec::RowBatch<N, NPOL, PT>::smem;
    return (const void *)vspec::row_batch_kernel<N, NPOL, PT>;
}
template <int N, int NPOL> const void *by_taps(int P, size_t *smem) {
    return P <= 1 ? instance<N, NPOL, 1>(smem) : P <= 8 ? instance<N, NPOL, 8>(smem) : instance<N, NPOL, 16>(smem);
}
template <int N> const void *by_pol(int npol, int P, size_t *smem) {
    return npol == 2 ? by_taps<N, 2>(P, smem) : by_taps<N, 1>(P, smem);
}
}  // namespace

// The kernel of a one-row transform of nchan channels with P taps, its dynamic
// shared memory in *smem; nullptr where there is none.
const void *vspec_pick_kernel_rowbatch(int nchan, int npol, int P, size_t *smem) {
    switch (nchan) {
        case 512: return by_pol<512>(npol, P, smem);
        case 1024: return by_pol<1024>(npol, P, smem);
        case 2048: return by_pol<2048>(npol, P, smem);
    }
    return nullptr;
}

const void *vspec_pick_fold_row(int npol) {
    return npol == 2 ? (const void *)vspec::fold_row_kernel<2> : (const void *)vspec::fold_row_kernel<1>;
}

// The kernels' bounds-check status word (debug builds), as vspec_ring_debug_flags.
cudaError_t vspec_rowbatch_debug_flags(unsigned *flags, bool clear) {
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
