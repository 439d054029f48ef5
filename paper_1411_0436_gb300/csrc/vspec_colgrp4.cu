// vspec_colgrp4.cu — instances of the grouped kernel A (vspec_colgrp.cuh), up to 4 taps.
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_colgrp_pick.cuh"

const void *vspec_pick_kernel_colgrp4(int N2, int npol, size_t *smem, int *groups) {
    return vspec::pick_colgrp<4>(N2, npol, smem, groups);
}
const void *vspec_pick_kernel_colgrp4_bands(int N2) { return vspec::pick_colgrp_bands<4>(N2); }
cudaError_t vspec_colgrp4_debug_flags(unsigned *flags, bool clear) { return vspec::colgrp_debug_flags(flags, clear); }
