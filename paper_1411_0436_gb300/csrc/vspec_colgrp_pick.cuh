// vspec_colgrp_pick.cuh — instance table of kernel A for one window length
// (each window length is its own translation unit).
#pragma once
#include "vspec_colgrp.cuh"

namespace vspec {

// Groups per CTA. Up to 8 taps four groups beat two (N2 = 64: 1199 against 1289
// us per 2048 spectra of 131072 channels), although a batch of 4 spectra unpacks
// 11 frames for 4 outputs and one of 8 spectra 15 for 8. With 16 taps the ring
// leaves room for two groups, or one beside the 128-point columns' padded tiles.
template <int N2, int PT> constexpr int colgrp_groups() {
    return PT <= 8 ? 4 : ColGrp<N2, PT, 2>::smem <= 232448 ? 2 : 1;
}

// Kernel A for columns of N2 points (2 .. 128) and PT taps at most, its dynamic
// shared memory and groups per CTA. (No plan asks for dual-pol 8-tap columns of
// at most 16 points, which pick_kernel_colreg gives to the register window, nor
// for single-pol 128-point columns, see colgrp_len: nullptr.)
template <int N2, int PT> const void *colgrp_instance(int npol, size_t *smem, int *groups) {
    constexpr int GR = colgrp_groups<N2, PT>();
    *smem = ColGrp<N2, PT, GR>::smem;
    *groups = GR;
    if constexpr (PT != 8 || N2 > 16)
        if (npol == 2) return (const void *)fir_colgrp_kernel<N2, PT, GR, 2>;
    if constexpr (N2 < 128)
        if (npol == 1) return (const void *)fir_colgrp_kernel<N2, PT, GR, 1>;
    return nullptr;
}
template <int PT> const void *pick_colgrp(int N2, int npol, size_t *smem, int *groups) {
    switch (N2) {
        case 2: return colgrp_instance<2, PT>(npol, smem, groups);
        case 4: return colgrp_instance<4, PT>(npol, smem, groups);
        case 8: return colgrp_instance<8, PT>(npol, smem, groups);
        case 16: return colgrp_instance<16, PT>(npol, smem, groups);
        case 32: return colgrp_instance<32, PT>(npol, smem, groups);
        case 64: return colgrp_instance<64, PT>(npol, smem, groups);
        case 128: return colgrp_instance<128, PT>(npol, smem, groups);
    }
    return nullptr;
}

// ... for interleaved sub-band tiles, dual-pol, of at most 8-point columns.
template <int PT> const void *pick_colgrp_bands(int N2) {
    switch (N2) {
        case 2: return (const void *)fir_colgrp_kernel<2, PT, colgrp_groups<2, PT>(), 2, true>;
        case 4: return (const void *)fir_colgrp_kernel<4, PT, colgrp_groups<4, PT>(), 2, true>;
        case 8: return (const void *)fir_colgrp_kernel<8, PT, colgrp_groups<8, PT>(), 2, true>;
    }
    return nullptr;
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
