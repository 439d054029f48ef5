// vspec_coldirgrp.cu — instances of the direct-FFT kernel A (vspec_coldirgrp.cuh).
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_coldirgrp.cuh"

namespace {
template <int N2> const void *instance(int npol, size_t *smem, int *groups) {
    using namespace vspec;
    *smem = ColDirGrp<N2>::smem;
    *groups = ColDirGrp<N2>::GROUPS;
    return npol == 2 ? (const void *)fir_coldirgrp_kernel<N2, 2> : (const void *)fir_coldirgrp_kernel<N2, 1>;
}
}  // namespace

// Kernel A for columns of N2 points (2 .. 256), its dynamic shared memory and
// groups per CTA; nullptr for other lengths.
const void *vspec_pick_kernel_coldirgrp(int N2, int npol, size_t *smem, int *groups) {
    switch (N2) {
        case 2: return instance<2>(npol, smem, groups);
        case 4: return instance<4>(npol, smem, groups);
        case 8: return instance<8>(npol, smem, groups);
        case 16: return instance<16>(npol, smem, groups);
        case 32: return instance<32>(npol, smem, groups);
        case 64: return instance<64>(npol, smem, groups);
        case 128: return instance<128>(npol, smem, groups);
        case 256: return instance<256>(npol, smem, groups);
    }
    return nullptr;
}

// The kernels' bounds-check status word (debug builds), as vspec_ring_debug_flags.
cudaError_t vspec_coldirgrp_debug_flags(unsigned *flags, bool clear) {
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
