// vspec_colgrp8.cu — instances of the grouped kernel A (vspec_colgrp.cuh), up to 8 taps.
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_colgrp_pick.cuh"

const void *vspec_pick_kernel_colgrp8(int N2, int npol, size_t *smem, int *groups) {
    return vspec::pick_colgrp<8>(N2, npol, smem, groups);
}
cudaError_t vspec_colgrp8_debug_flags(unsigned *flags, bool clear) { return vspec::colgrp_debug_flags(flags, clear); }
