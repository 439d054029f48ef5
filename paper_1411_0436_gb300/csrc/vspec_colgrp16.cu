// vspec_colgrp16.cu — instances of the grouped kernel A (vspec_colgrp.cuh), up to 16 taps.
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_colgrp_pick.cuh"

const void *vspec_pick_kernel_colgrp16(int N2, int npol, size_t *smem, int *groups) {
    return vspec::pick_colgrp<16>(N2, npol, smem, groups);
}
const void *vspec_pick_kernel_colgrp16_bands(int N2) { return vspec::pick_colgrp_bands<16>(N2); }
cudaError_t vspec_colgrp16_debug_flags(unsigned *flags, bool clear) { return vspec::colgrp_debug_flags(flags, clear); }
