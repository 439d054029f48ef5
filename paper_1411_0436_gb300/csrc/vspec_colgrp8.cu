// vspec_colgrp8.cu — instances of the grouped kernel A (vspec_colgrp.cuh), up to 8 taps.
#include <cuda_runtime.h>

#define VSPEC_NO_PLAN_TABLES
#include "vspec_colgrp_pick.cuh"

// Kernel A for columns of N2 = 32, 64 or 128 points, nullptr for other lengths.
const void *vspec_pick_kernel_colgrp8(int N2, size_t *smem, int *groups) {
    switch (N2) {
        case 32: return vspec::colgrp_instance<32, 8>(smem, groups);
        case 64: return vspec::colgrp_instance<64, 8>(smem, groups);
        case 128: return vspec::colgrp_instance<128, 8>(smem, groups);
    }
    return nullptr;
}
cudaError_t vspec_colgrp8_debug_flags(unsigned *flags, bool clear) { return vspec::colgrp_debug_flags(flags, clear); }
