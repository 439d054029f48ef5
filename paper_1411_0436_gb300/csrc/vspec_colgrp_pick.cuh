// vspec_colgrp_pick.cuh — instance table of kernel A for one window length
// (each window length is its own translation unit).
#pragma once
#include "vspec_colgrp.cuh"

namespace vspec {

// Kernel A for columns of N2 points and PT taps at most, its dynamic shared
// memory and groups per CTA. Four groups beat two (N2 = 64: 1199 against 1289
// us per 2048 spectra of 131072 channels), although a batch of 4 spectra unpacks
// 11 frames for 4 outputs and one of 8 spectra 15 for 8.
template <int N2, int PT> const void *colgrp_instance(size_t *smem, int *groups) {
    constexpr int GR = 4;
    *smem = ColGrp<N2, PT, GR>::smem;
    *groups = GR;
    return (const void *)fir_colgrp_kernel<N2, PT, GR, 2>;
}

// This translation unit's bounds-check status word (debug builds).
static inline cudaError_t colgrp_debug_flags(unsigned *flags, bool clear) {
#ifdef VSPEC_DEBUG
    cudaError_t e = cudaMemcpyFromSymbol(flags, g_debug_flags, sizeof(unsigned));
    if (e != cudaSuccess || !clear) return e;
    const unsigned zero = 0;
    return cudaMemcpyToSymbol(g_debug_flags, &zero, sizeof(unsigned));
#else
    *flags = 0;
    (void)clear;
    return cudaSuccess;
#endif
}

}  // namespace vspec
