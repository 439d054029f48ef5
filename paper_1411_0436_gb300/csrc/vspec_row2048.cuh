// vspec_row2048.cuh — the 2048-point row kernel (kernel B) of dual-pol plans
// with uncompensated sums: row DFTs over n1, detection (§4: X^2, Y^2, Re XY*,
// Im XY*) and accumulation.
//
// One 512-thread CTA per SM, four groups of 128 threads. Each group
// transforms whole spectra by itself (three DIF passes, radix 16, 16, 8) and
// synchronises only on its own named barrier.
//
// What bounds it: per row point the passes move 80 bytes through shared
// memory and issue about 50 FMA-pipe instructions, each worth about half of
// the kernel's time when the phases (load, transform, store) of one CTA-wide
// barrier follow one another. Four groups that drift apart let one group's
// shared-memory phase run under another's arithmetic.
//  - Rows come in as one 32 KiB bulk copy each (cp.async.bulk, an mbarrier per
//    buffer), seven buffers deep, so three rows are in flight beyond the four
//    being transformed and no thread waits on a global load.
//  - A row is transformed in the buffer it landed in: position a lives at
//    a ^ ((a >> 3) & 7) from pass 1's stores on, which is free of bank
//    conflicts in every pass without padding. (Pass 1's loads, from the
//    landed linear order, and its stores touch the same eight elements of the
//    same eight lanes.)
//  - The per-channel sums live in tensor memory (one tcgen05.ld and .st of
//    32 columns per eight channels and spectrum), not in registers, so a
//    group of 128 threads can hold the 16 channels per thread of a whole row
//    beside a radix-16 butterfly. Per group: 64 columns for a run of
//    kRow2048Run spectra, 64 for the sums of the finished runs (the two-level
//    summation); the groups' sums are added in group order once per segment
//    and go to the CTA's partial-sum slot.
//  - Pass-1 twiddles are stored [q][j], one contiguous 8-byte load per lane;
//    they stay in the L1 left beside the buffers (15 KiB).
// Single-polarisation plans run it on pairs of spectra (RowMode): 65536 channels,
// 1024 spectra 201 -> 163 us against row2048_kernel.
// Measured (GB300, 131072 channels, 2048 spectra per launch): 0.86 ms against
// 1.06 ms for two 256-thread CTAs per SM with register sums, global loads and
// padded rows; 524288 channels direct 0.44 against 0.56 ms per 256 spectra. Of
// the SM cycles the FMA pipe is busy 61%, the shared-memory and L1 data path
// 78% (5 accesses of 16 bytes per point, to which the bulk copies add their
// writes): that path is the bound.
#pragma once
#include "vspec_kernels.cuh"
#include "vspec_kernels_tc.cuh"
#include "vspec_tc.cuh"
#include "vspec_tmem.cuh"

namespace vspec {

struct Row2048 {
    static constexpr int GROUPS = 4, NBUF = 7, THREADS = 128 * GROUPS;
    static constexpr uint32_t ROW_BYTES = 2048 * 16;
    static constexpr uint32_t TMEM_COLS = 512;  // GROUPS x (64 run + 64 total)
    static constexpr int TW1 = 15 * 128, TW2 = 15 * 8;  // float2 entries of the [q-1][j] tables
    // row buffers, pass-2 twiddles, barriers, the item last copied into each buffer, TMEM address, give-up flag
    static constexpr size_t smem = (size_t)NBUF * ROW_BYTES + TW2 * 8 + NBUF * 12 + 8;
    static_assert(smem <= 232448, "shared memory of one CTA");
};

// Order of a 16-point butterfly's loads: the inputs of its first additions
// (0 and 8, 4 and 12, ...) arrive next to each other.
__device__ __forceinline__ constexpr int bitrev4(int i) {
    return (i & 1) << 3 | (i & 2) << 1 | (i & 4) >> 1 | (i & 8) >> 3;
}

// Wait for the copy of item i into its buffer. The copy starts once the buffer's
// previous item is done, which may be another group's: until `copied` shows it,
// the barrier may be a phase behind, where the parity of the phase before it
// reads as complete. Both waits are bounded by p.wait_limit (vspec_set_wait_limit);
// one that gives up raises the plan's flag, and after it no row is copied any
// more and the others do not wait.
template <int NBUF>
__device__ __forceinline__ void wait_row(const RowParams &p, uint64_t *full, const volatile int *copied,
                                         volatile int *gave_up, int i) {
    const int b = i % NBUF;
    const uint32_t limit = *gave_up ? min(1u, p.wait_limit) : p.wait_limit;
    bool started = copied[b] == i;
    for (uint32_t it = 0; !started && it < limit; it++) started = copied[b] == i;
    if (!started || !tc::mbar_wait(full + b, (i / NBUF) & 1, limit)) {
        *gave_up = 1;
        if (p.wait_status) atomicExch(p.wait_status, 1);
    }
}
// After a wait that gave up: no copy of the CTA's n items may land once it has left.
template <int NBUF> __device__ __forceinline__ void drain_rows(uint64_t *full, const volatile int *copied, int n) {
    for (int b = 0; b < min(n, NBUF); b++) tc::mbar_wait(full + b, (copied[b] / NBUF) & 1);
}

// Scratch elements and sums: packed (X.re, Y.re, X.im, Y.im); split (X.re, X.im,
// Y.re, Y.im), the tensor-core column kernel's order; or pairs, packed elements
// whose halves are two spectra of a single polarisation (p.sc counts pairs):
// both powers go to the same float, 16 per thread; a run's sums in registers.
enum RowMode { kRowPacked = 0, kRowSplit = 1, kRowPairs = 2 };
template <int MODE>
__global__ void __launch_bounds__(Row2048::THREADS, 1) row2048_group_kernel(const __grid_constant__ RowParams p) {
    using G = Row2048;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    P2 *bufs = reinterpret_cast<P2 *>(smem_raw);                                  // [NBUF][2048]
    float2 *tw2s = reinterpret_cast<float2 *>(smem_raw + (size_t)G::NBUF * G::ROW_BYTES);  // [15][8]
    uint64_t *full = reinterpret_cast<uint64_t *>(tw2s + G::TW2);                 // [NBUF]
    volatile int *copied = reinterpret_cast<volatile int *>(full + G::NBUF);      // [NBUF]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(const_cast<int *>(copied) + G::NBUF);
    volatile int *gave_up = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int tid = threadIdx.x, g = tid >> 7, ht = tid & 127, warp = tid >> 5;

    const Span sp = block_span(p.tiles, p.sc);
    const int n = (int)(sp.hi - sp.lo);  // items (row tile, spectrum) of this CTA
    // item i's row into buffer i mod NBUF (one thread at a time)
    auto issue = [&](int i) {
        const long long f = sp.lo + i;
        const int x = (int)(f / p.sc), s = (int)(f - (long long)x * p.sc);
        uint64_t *bar = full + i % G::NBUF;
        const uint32_t dst = tc::smem_addr(bufs + (size_t)(i % G::NBUF) * 2048);
        const float4 *src = reinterpret_cast<const float4 *>(p.Z) + (size_t)s * p.N + (size_t)x * 2048;
        if (!dbg_ok(s < p.sc && (long long)(x + 1) * 2048 <= p.N, kDbgScratch | kDbgTile))
            src = reinterpret_cast<const float4 *>(p.Z);
        copied[i % G::NBUF] = i;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     :: "r"(tc::smem_addr(bar)), "r"(G::ROW_BYTES) : "memory");
        asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     :: "r"(dst), "l"(src), "r"(G::ROW_BYTES), "r"(tc::smem_addr(bar)) : "memory");
    };
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::smem_addr(tmem_slot)), "r"(G::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int e = tid; e < G::TW2; e += G::THREADS) tw2s[e] = __ldg(p.twBt + G::TW1 + e);
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
    const uint32_t tm_run = tm + 64 * g, tm_tot = tm + 256 + 64 * g;

    auto bar = [&]() { asm volatile("bar.sync %0, 128;" :: "r"(1 + g) : "memory"); };
    const int j = ht & 7;
    const int sw1 = ht ^ ((ht >> 3) & 7);       // pass 1: position ht + 128 q at sw1 + 128 q
    const int base2 = (ht >> 3) * 128;          // pass 2: position base2 + 8 q + j at base2 + 8 q + (j ^ (q & 7))
    const float2 *tw1 = p.twBt + ht;            // W_2048^(ht q) at tw1[128 (q - 1)]

    for (long long f = sp.lo; f < sp.hi;) {
        const int x = (int)(f / p.sc);  // row tile
        const long long base = (long long)x * p.sc;
        const long long fe = min(sp.hi, base + p.sc);
        const int i0 = (int)(f - sp.lo), i1 = (int)(fe - sp.lo);
        f = fe;
        int run = 0;           // spectra in the current run
        bool totals = false;   // finished runs are in tm_tot
        float rsum[16];        // pairs: the run's sums, channel 8 (ht + 128 k) + q at 8 k + q
        if constexpr (MODE == kRowPairs) {
#pragma unroll
            for (int e = 0; e < 16; e++) rsum[e] = 0.f;
        }
        for (int i = i0 + ((g - i0) & (G::GROUPS - 1)); i < i1; i += G::GROUPS) {
            const int b = i % G::NBUF;
            P2 *row = bufs + (size_t)b * 2048;
            wait_row<G::NBUF>(p, full, copied, gave_up, i);
            __syncwarp();
            // pass 1: block length 2048, butterfly j = ht over positions ht + 128 q
            {
                P2 v[16];
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const int q = bitrev4(i);
                    if constexpr (MODE == kRowSplit) {
                        const float4 e = reinterpret_cast<const float4 *>(row)[ht + 128 * q];
                        v[q] = make_p2(e.x, e.y, e.z, e.w);
                    } else {
                        v[q] = row[ht + 128 * q];
                    }
                }
                Dft<16>::run(v);
#pragma unroll
                for (int q = 1; q < 16; q++) v[q] = cmul(v[q], __ldg(tw1 + 128 * (q - 1)));
                __syncwarp();  // the warp's lanes have read what they now overwrite
#pragma unroll
                for (int q = 0; q < 16; q++) row[sw1 + 128 * q] = v[q];
            }
            bar();
            // pass 2: block length 128, unit ht / 8, butterfly j over positions j + 8 q
            {
                P2 v[16];
                P2 *r2 = row + base2;
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const int q = bitrev4(i);
                    v[q] = r2[8 * q + (j ^ (q & 7))];
                }
                Dft<16>::run(v);
#pragma unroll
                for (int q = 1; q < 16; q++) v[q] = cmul(v[q], tw2s[8 * (q - 1) + j]);
#pragma unroll
                for (int q = 0; q < 16; q++) r2[8 * q + (j ^ (q & 7))] = v[q];
            }
            bar();
            // pass 3: block length 8, blocks ht and ht + 128 (channels 8 t .. 8 t + 7): detection
            // and sums. The end of a run (and of the segment) adds the run to the totals.
            const bool last = run == kRow2048Run - 1 || i + G::GROUPS >= i1;
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");  // the previous spectrum's sums
#pragma unroll
            for (int k = 0; k < 2; k++) {
                P2 v[8];
                const P2 *r3 = row + 8 * (ht + 128 * k);
#pragma unroll
                for (int q = 0; q < 8; q++) v[q] = r3[q ^ j];
                if (k == 1) {
                    tc::fence_proxy_async();  // this buffer's accesses before the next copy into it
                    bar();
                    if (ht == 0 && i + G::NBUF < n && !*gave_up) issue(i + G::NBUF);
                    __syncwarp();
                }
                uint32_t a[32];
                if constexpr (MODE != kRowPairs) {
                    if (run) {
                        tmem_ld_wait<32>(tm_run + 32 * k, a);
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; e++) a[e] = 0u;
                    }
                }
                Dft<8>::run(v);
                if constexpr (MODE == kRowPairs) {
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        const float2 w = __ffma2_rn(v[q].re, v[q].re, __fmul2_rn(v[q].im, v[q].im));
                        rsum[8 * k + q] += w.x + w.y;
                    }
                    continue;
                }
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    float4 c = make_float4(__uint_as_float(a[4 * q]), __uint_as_float(a[4 * q + 1]),
                                           __uint_as_float(a[4 * q + 2]), __uint_as_float(a[4 * q + 3]));
                    acc_add<2>(c, v[q]);
                    a[4 * q] = __float_as_uint(c.x);
                    a[4 * q + 1] = __float_as_uint(c.y);
                    a[4 * q + 2] = __float_as_uint(c.z);
                    a[4 * q + 3] = __float_as_uint(c.w);
                }
                if (!last) {
                    tmem_st32(tm_run + 32 * k, a);
                } else {
                    if (totals) {
                        uint32_t t[32];
                        tmem_ld_wait<32>(tm_tot + 32 * k, t);
#pragma unroll
                        for (int e = 0; e < 32; e++)
                            a[e] = __float_as_uint(__uint_as_float(t[e]) + __uint_as_float(a[e]));
                    }
                    tmem_st32(tm_tot + 32 * k, a);
                }
            }
            if constexpr (MODE == kRowPairs) {
                if (last) {  // into columns 0 .. 15 of this thread's totals
                    uint32_t a[32];
                    if (totals) {
                        tmem_ld_wait<16>(tm_tot, a);
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; e++) a[e] = 0u;
                    }
#pragma unroll
                    for (int e = 0; e < 16; e++) {
                        a[e] = __float_as_uint(__uint_as_float(a[e]) + rsum[e]);
                        a[16 + e] = 0u;
                        rsum[e] = 0.f;
                    }
                    tmem_st32(tm_tot, a);
                }
            }
            if (last) totals = true;
            run = last ? 0 : run + 1;
        }
        // the groups' totals in group order: warp (g, w) takes columns 16 g ..
        // + 15 (pairs: 4 g .. + 3) of every set, channels 8 (ht + 128 (g / 2)) +
        // 4 (g mod 2) .. + 3
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float sum[16];
        bool any = false;
#pragma unroll
        for (int k = 0; k < G::GROUPS; k++) {
            if (i0 + ((k - i0) & (G::GROUPS - 1)) >= i1) continue;  // this group had no spectrum
            float t[16];
            // (pairs: the 16 channels' columns; the 4 of this warp are picked below)
            tmem_ld16_wait(tm + 256 + 64 * k + (MODE == kRowPairs ? 0 : 16 * g), t);
#pragma unroll
            for (int e = 0; e < 16; e++) sum[e] = any ? sum[e] + t[e] : t[e];
            any = true;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();  // the sets are free for the next segment
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int slot = span_slot(p.tiles, p.sc, x);
        if (dbg_ok(slot < p.slots && (long long)(x + 1) * 2048 <= p.N, kDbgSlot)) {
            using A = typename Elem<MODE == kRowPairs ? 1 : 2>::Acc;
            A *part = reinterpret_cast<A *>(p.partial) + (size_t)slot * p.N + (size_t)x * 2048 +
                           8 * (ht + 128 * (g >> 1)) + 4 * (g & 1);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                A v;
                if constexpr (MODE == kRowPairs)
                    v = g == 0 ? sum[q] : g == 1 ? sum[4 + q] : g == 2 ? sum[8 + q] : sum[12 + q];
                else
                    v = make_float4(sum[4 * q], sum[4 * q + 1], sum[4 * q + 2], sum[4 * q + 3]);
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

// Twiddles of a DIF pass in [q - 1][j] order: tw[(q - 1) m + j] = W_lb^(j q).
#ifndef VSPEC_NO_PLAN_TABLES
__global__ void gen_pass_tw_t_kernel(float2 *tw, Pass ps) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ps.m * (ps.r - 1)) return;
    tw[e] = root_of_unity((long long)(e % ps.m) * (e / ps.m + 1), ps.lb);
}
#endif

}  // namespace vspec
