// vspec_row4096.cuh — the 4096-point row kernel (kernel B) of dual-pol plans
// with uncompensated sums (2^19 channels with a pre-filter): the 2048-point
// kernel's scheme (vspec_row2048.cuh) with three radix-16 passes.
//
// One 512-thread CTA per SM, two groups of 256 threads that transform whole
// spectra on their own named barriers; rows of 64 KiB arrive as bulk copies into
// three buffers and are transformed in place, position a at a ^ ((a >> 4) & 7)
// from pass 1's stores on (free of bank conflicts in every pass: 8-lane phases
// are 8 consecutive positions, or 8 blocks of 16 in pass 3). The last pass gives
// a thread 16 consecutive channels, whose sums live in tensor memory: 64 columns
// for a run of kRow2048Run spectra and 64 for the finished runs, added over the
// groups in order once per segment.
//
// Pass-1 twiddles are in shared memory too: the row buffers leave L1 28 KB for
// the 30 KB of them, and the warps waited most on those loads (whole call, 128
// spectra: 763 us through L1, 740).
//
// Measured (GB300, 524288 channels, 128 spectra): 313 us against 382 us for four
// radix-8 passes of one CTA-wide group with register sums. Bound, like the
// 2048-point kernel, by the shared-memory data path.
#pragma once
#include "vspec_row2048.cuh"

namespace vspec {

struct Row4096 {
    static constexpr int GROUPS = 2, TG = 256, NBUF = 3, THREADS = TG * GROUPS, ROW = 4096;
    static constexpr uint32_t ROW_BYTES = ROW * 16;
    static constexpr uint32_t TMEM_COLS = 512;  // 4 warps of a lane quarter x (64 run + 64 total)
    static constexpr int TW1 = 15 * 256, TW2 = 15 * 16;  // float2 entries of the [q-1][j] tables
    // row buffers, pass-1 and pass-2 twiddles, barriers, the item last copied into each buffer, TMEM address, give-up flag
    static constexpr size_t smem = (size_t)NBUF * ROW_BYTES + (TW1 + TW2) * 8 + NBUF * 12 + 12;
    static_assert(smem <= 232448, "shared memory of one CTA");
};

__global__ void __launch_bounds__(Row4096::THREADS, 1) row4096_group_kernel(const __grid_constant__ RowParams p) {
    using G = Row4096;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    P2 *bufs = reinterpret_cast<P2 *>(smem_raw);                                           // [NBUF][4096]
    float2 *tw1s = reinterpret_cast<float2 *>(smem_raw + (size_t)G::NBUF * G::ROW_BYTES);  // [15][256]
    float2 *tw2s = tw1s + G::TW1;                                                          // [15][16]
    uint64_t *full = reinterpret_cast<uint64_t *>(tw2s + G::TW2);                          // [NBUF]
    volatile int *copied = reinterpret_cast<volatile int *>(full + G::NBUF);               // [NBUF]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(const_cast<int *>(copied) + G::NBUF);
    volatile int *gave_up = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int tid = threadIdx.x, g = tid / G::TG, ht = tid % G::TG, warp = tid >> 5;

    const Span sp = block_span(p.tiles, p.sc);
    const int n = (int)(sp.hi - sp.lo);  // items (row tile, spectrum) of this CTA
    // item i's row into buffer i mod NBUF (one thread at a time)
    auto issue = [&](int i) {
        const long long f = sp.lo + i;
        const int x = (int)(f / p.sc), s = (int)(f - (long long)x * p.sc);
        uint64_t *bar = full + i % G::NBUF;
        const uint32_t dst = tc::smem_addr(bufs + (size_t)(i % G::NBUF) * G::ROW);
        const float4 *src = reinterpret_cast<const float4 *>(p.Z) + (size_t)s * p.N + (size_t)x * G::ROW;
        if (!dbg_ok(s < p.sc && (long long)(x + 1) * G::ROW <= p.N, kDbgScratch | kDbgTile))
            src = reinterpret_cast<const float4 *>(p.Z);
        copied[i % G::NBUF] = i;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     :: "r"(tc::smem_addr(bar)), "r"(G::ROW_BYTES) : "memory");
#pragma unroll
        for (uint32_t h = 0; h < G::ROW_BYTES; h += G::ROW_BYTES / 2)
            asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         :: "r"(dst + h), "l"(reinterpret_cast<const unsigned char *>(src) + h), "r"(G::ROW_BYTES / 2),
                            "r"(tc::smem_addr(bar)) : "memory");
    };
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::smem_addr(tmem_slot)), "r"(G::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int e = tid; e < G::TW1 + G::TW2; e += G::THREADS) tw1s[e] = __ldg(p.twBt + e);
    if (tid == 0) {
        *gave_up = 0;
        for (int b = 0; b < G::NBUF; b++) tc::mbar_init(full + b, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        pdl_wait();  // kernel A's rows
        tc::fence_proxy_async();
        for (int i = 0; i < min(n, G::NBUF); i++) issue(i);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // this warp's lanes: rows 32 (warp mod 4) .. + 31 of tensor memory
    const uint32_t tm = *tmem_slot + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t tm_run = tm + 64 * (warp >> 2), tm_tot = tm_run + 256;

    auto bar = [&]() { asm volatile("bar.sync %0, 256;" :: "r"(1 + g) : "memory"); };
    const int j = ht & 15;
    const int sw1 = ht ^ ((ht >> 4) & 7);  // pass 1: position ht + 256 q at sw1 + 256 q
    const int base2 = (ht >> 4) * 256;     // pass 2: position base2 + 16 q + j at base2 + 16 q + (j ^ (q & 7))
    const float2 *tw1 = tw1s + ht;         // W_4096^(ht q) at tw1[256 (q - 1)]

    for (long long f = sp.lo; f < sp.hi;) {
        const int x = (int)(f / p.sc);  // row tile
        const long long base = (long long)x * p.sc;
        const long long fe = min(sp.hi, base + p.sc);
        const int i0 = (int)(f - sp.lo), i1 = (int)(fe - sp.lo);
        f = fe;
        int run = 0;          // spectra in the current run
        bool totals = false;  // finished runs are in tm_tot
        for (int i = i0 + ((g - i0) & (G::GROUPS - 1)); i < i1; i += G::GROUPS) {
            const int b = i % G::NBUF;
            P2 *row = bufs + (size_t)b * G::ROW;
            wait_row<G::NBUF>(p, full, copied, gave_up, i);
            __syncwarp();
            P2 v[16];
            // pass 1: block length 4096, butterfly j = ht over positions ht + 256 q
#pragma unroll
            for (int i = 0; i < 16; i++) v[bitrev4(i)] = row[ht + 256 * bitrev4(i)];
            Dft<16>::run(v);
#pragma unroll
            for (int q = 1; q < 16; q++) v[q] = cmul(v[q], tw1[256 * (q - 1)]);
            __syncwarp();  // the warp's lanes have read what they now overwrite
#pragma unroll
            for (int q = 0; q < 16; q++) row[sw1 + 256 * q] = v[q];
            bar();
            // pass 2: block length 256, unit ht / 16, butterfly j over positions j + 16 q
            P2 *r2 = row + base2;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int q = bitrev4(i);
                v[q] = r2[16 * q + (j ^ (q & 7))];
            }
            Dft<16>::run(v);
#pragma unroll
            for (int q = 1; q < 16; q++) v[q] = cmul(v[q], tw2s[16 * (q - 1) + j]);
#pragma unroll
            for (int q = 0; q < 16; q++) r2[16 * q + (j ^ (q & 7))] = v[q];
            bar();
            // pass 3: block length 16, channels 16 ht .. + 15: detection and sums.
            // The end of a run (and of the segment) adds the run to the totals.
            const bool last = run == kRow2048Run - 1 || i + G::GROUPS >= i1;
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");  // the previous spectrum's sums
            const P2 *r3 = row + 16 * ht;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int q = bitrev4(i);
                v[q] = r3[q ^ (ht & 7)];
            }
            tc::fence_proxy_async();  // this buffer's accesses before the next copy into it
            bar();
            if (ht == 0 && i + G::NBUF < n && !*gave_up) issue(i + G::NBUF);
            __syncwarp();
            Dft<16>::run(v);
#pragma unroll
            for (int k = 0; k < 4; k++) {  // four channels at a time: 16 columns
                uint32_t a[32];
                if (run) {
                    tmem_ld_wait<16>(tm_run + 16 * k, a);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; e++) a[e] = 0u;
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    float4 c = make_float4(__uint_as_float(a[4 * q]), __uint_as_float(a[4 * q + 1]),
                                           __uint_as_float(a[4 * q + 2]), __uint_as_float(a[4 * q + 3]));
                    acc_add<2>(c, v[4 * k + q]);
                    a[4 * q] = __float_as_uint(c.x);
                    a[4 * q + 1] = __float_as_uint(c.y);
                    a[4 * q + 2] = __float_as_uint(c.z);
                    a[4 * q + 3] = __float_as_uint(c.w);
                }
                if (last && totals) {
                    uint32_t t[32];
                    tmem_ld_wait<16>(tm_tot + 16 * k, t);
#pragma unroll
                    for (int e = 0; e < 16; e++)
                        a[e] = __float_as_uint(__uint_as_float(t[e]) + __uint_as_float(a[e]));
                }
                tmem_st_first16((last ? tm_tot : tm_run) + 16 * k, a);
            }
            if (last) totals = true;
            run = last ? 0 : run + 1;
        }
        // the groups' totals in group order: warp w takes columns 32 (w / 8) .. + 31 of
        // the sets of warps w mod 8 and w mod 8 + 8, channels 16 (tid mod 256) + 8 (w / 8) .. + 7
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float sum[32];
        bool any = false;
#pragma unroll
        for (int k = 0; k < G::GROUPS; k++) {
            if (i0 + ((k - i0) & (G::GROUPS - 1)) >= i1) continue;  // this group had no spectrum
            uint32_t t[32];
            tmem_ld_wait<32>(tm + 256 + 64 * (2 * k + ((warp >> 2) & 1)) + 32 * (warp >> 3), t);
#pragma unroll
            for (int e = 0; e < 32; e++) sum[e] = any ? sum[e] + __uint_as_float(t[e]) : __uint_as_float(t[e]);
            any = true;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();  // the sets are free for the next segment
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int slot = span_slot(p.tiles, p.sc, x);
        if (dbg_ok(slot < p.slots && (long long)(x + 1) * G::ROW <= p.N, kDbgSlot)) {
            float4 *part = reinterpret_cast<float4 *>(p.partial) + (size_t)slot * p.N + (size_t)x * G::ROW +
                           16 * (tid & 255) + 8 * (warp >> 3);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const float4 v = make_float4(sum[4 * q], sum[4 * q + 1], sum[4 * q + 2], sum[4 * q + 3]);
                // a reduction performed in L2: one writer per entry and launch
                if (p.store) part[q] = v;
                else atomicAdd(part + q, v);
            }
        }
    }
    pdl_trigger();
    if (*gave_up && tid == 0) drain_rows<G::NBUF>(full, copied, n);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(*tmem_slot), "r"(G::TMEM_COLS) : "memory");
}

}  // namespace vspec
