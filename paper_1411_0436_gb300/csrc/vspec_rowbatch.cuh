// vspec_rowbatch.cuh — one-pass kernel of the one-row transforms (512, 1024 and
// 2048 channels): pre-filter, FFT, detection and accumulation in one CTA from
// the int8 input, with nothing in between leaving the SM.
//
// One 512-thread CTA per SM takes a run of consecutive spectra in batches of
// 8192 points (SPB spectra; 4096 points at 2048 channels dual-pol with more than
// 8 taps). Per batch:
//  - the pre-filter: each thread forms its points' outputs of the whole batch
//    from one walk over a ring of staged int8 frames, unpacking a sample once
//    for all the outputs it is a tap of (PT - 1 + SPB unpacks for SPB outputs);
//    the thread's coefficients stay in registers;
//  - three DIF passes through shared memory, radix R1, R2, 8 (the plan's row
//    pass list), element a at a ^ ((a >> 3) & 7), free of bank conflicts in
//    every pass;
//  - the last pass detects into per-thread sums in tensor memory (dual-pol: 32
//    columns, one load and one store per batch; single-pol: 8 registers): every
//    thread holds eight channels of one of 4096 / N sets of sums, two spectra
//    per batch. After kRunBatches batches the sets are added in order into the
//    CTA's partial-sum slot (two-level summation).
// The next batch's frames are copied over the ring's oldest while the passes
// run.
//
// Single-polarisation input uses the same paired arithmetic: a batch holds
// twice the spectra, and spectrum u of its first half and of its second half
// are the two halves of each pair. Both powers go to the same sum.
//
// What bounds it: about 104 bytes of shared-memory traffic and 113 FMA-pipe
// slots per point, phase after phase (four barriers per batch); on short
// calls its prologue (coefficients, PT - 1 leading frames) and latency.
// Measured (GB300, whole calls, us): 1024 channels dual-pol 8 taps 2048 spectra
// 66 -> 22.6, 4096 spectra 114 -> 35, direct 60 -> 29; single-pol 4096 spectra
// 72 -> 21; 2048 channels 4096 spectra 103 -> 64 (against the cluster kernel),
// direct 91 -> 47; dual-pol 16 taps 257 spectra 37 -> 20.5, 4096 179 -> 98; the others against the general row kernel, which unpacked
// every tap of every spectrum and kept its sums in shared memory.
#pragma once
#include "vspec_kernels.cuh"
#include "vspec_row2048.cuh"

namespace vspec {

template <int N_, int NPOL_, int PT_>
struct RowBatch {
    // (2048 channels, dual-pol, more than 8 taps: two spectra, the ring takes the room)
    static constexpr int N = N_, NPOL = NPOL_, PT = PT_, THREADS = 512,
                         SPB = N == 2048 && NPOL == 2 && PT > 8 ? 2 : 8192 / N;
    static constexpr int R1 = N == 512 ? 8 : 16, R2 = N == 2048 ? 16 : 8;  // then radix 8
    static constexpr int M1 = N / R1, KP = N / THREADS;   // first-pass stride; points per thread
    static constexpr int BS = NPOL == 2 ? SPB : 2 * SPB;  // spectra per batch
    static constexpr int RING = PT - 1 + BS;              // frames a batch spans
    static constexpr int W = 2 * NPOL;                    // bytes per sample
    static constexpr int UB = SPB < 8 ? SPB : 8;          // outputs formed together
    static constexpr int SETS = 4096 / N;                 // sets of sums
    static constexpr int TW1 = (R1 - 1) * M1, TW2 = (R2 - 1) * 8;  // twiddles, [q - 1][j]
    static constexpr int kRunBatches = kRow2048Run / 2;
    static constexpr size_t smem = (size_t)SPB * N * 16 + (size_t)RING * N * W + TW2 * 8 + 16;
    static_assert(R1 * R2 * 8 == N && KP >= 1, "pass list");
};

template <int N_, int NPOL_, int PT_>
__global__ void __launch_bounds__(512, 1) row_batch_kernel(const __grid_constant__ RowParams p) {
    using G = RowBatch<N_, NPOL_, PT_>;
    using A = typename Elem<NPOL_>::Acc;
    constexpr int N = G::N, NPOL = G::NPOL, PT = G::PT, SPB = G::SPB, RING = G::RING, W = G::W;
    static_assert(G::smem <= 232448, "shared memory of one CTA");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    P2 *data = reinterpret_cast<P2 *>(smem_raw);                        // [SPB][N]
    unsigned char *ring = smem_raw + (size_t)SPB * N * 16;              // [RING][N] samples
    float2 *tw2s = reinterpret_cast<float2 *>(ring + (size_t)RING * N * W);  // [R2 - 1][8]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tw2s + G::TW2);
    const int t = threadIdx.x, warp = t >> 5;
    const int D = PT - p.P;  // leading zero taps

    if constexpr (NPOL == 2) {
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         :: "r"(tc::smem_addr(tmem_slot)), "r"(128u) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    // p.tiles bands (see run_rows): an equal share of one band's spectra
    const int per = gridDim.x / p.tiles, rank = blockIdx.x % per;
    const int8_t *in = p.in + (long long)(blockIdx.x / per) * p.band_bytes;
    const int s_beg = (int)((long long)p.sc * rank / per), s_end = (int)((long long)p.sc * (rank + 1) / per);
    // Ring slot (fr - first) mod RING holds absolute frame fr, first the oldest
    // frame of the run's first spectrum (D leading taps have zero coefficients;
    // frames before the input are clamped).
    const long long first = p.s0 + s_beg - D;
    auto stage = [&](int rel, int cnt, int slot) {  // frames first + rel .. + cnt - 1 from ring slot `slot`
        constexpr int per = N * W / 16;             // 16-byte pieces of a frame
        for (int i = t; i < cnt * per; i += G::THREADS) {
            const int u = i / per, e = i % per;
            long long fr = first + rel + u;
            if (fr < 0) fr = 0;
            int sl = slot + u;
            if (sl >= RING) sl -= RING;
            const unsigned char *src = reinterpret_cast<const unsigned char *>(in) + (fr * N) * W + 16 * e;
            if (dbg_ok(fr < p.nframes, kDbgInput))
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             :: "r"(tc::smem_addr(ring + (size_t)sl * N * W + 16 * e)), "l"(src) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0, PT - 1 + min(G::BS, s_end - s_beg), 0);
    float cf[G::KP][PT];
#pragma unroll
    for (int k = 0; k < G::KP; k++)
#pragma unroll
        for (int h = 0; h < PT; h++) cf[k][h] = h >= D ? __ldg(p.coef + (size_t)(h - D) * N + t + 512 * k) : 0.f;
    for (int e = t; e < G::TW2; e += G::THREADS) tw2s[e] = __ldg(p.twBt + G::TW1 + e);
    if constexpr (NPOL == 2) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    uint32_t tm = 0;
    if constexpr (NPOL == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tm = *tmem_slot + ((uint32_t)((warp & 3) * 32) << 16) + 32 * (warp >> 2);
    }

    // last pass: block b8 of spectra set, set + SETS (channels 8 b8 .. + 7)
    const int b8 = t % (N / 8), set = t / (N / 8);
    float sum1[8];  // single-pol sums
#pragma unroll
    for (int q = 0; q < 8; q++) sum1[q] = 0.f;
    bool fresh = true;  // no sums in tensor memory yet
    bool store = p.store != 0;
    int batches = 0, r0 = 0;  // batches in the run; ring slot of the batch's oldest frame
    for (int s = s_beg; s < s_end; s += G::BS) {
        const int nb = min(G::BS, s_end - s);
        // single-pol: pair u holds spectra s + u and s + half + u
        const int half = NPOL == 2 ? 0 : (nb + 1) / 2;
        const int pairs = NPOL == 2 ? nb : half;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the batch's frames are visible; data is free
#pragma unroll
        for (int k = 0; k < G::KP; k++) {
            const int pt = t + 512 * k;
            float2 c2[PT];
#pragma unroll
            for (int h = 0; h < PT; h++) c2[h] = dup2(cf[k][h]);
#pragma unroll
            for (int ub = 0; ub < SPB; ub += G::UB) {
                if (ub >= pairs) break;
                P2 y[G::UB];
#pragma unroll
                for (int u = 0; u < G::UB; u++) y[u] = P2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int h = 0; h < PT - 1 + G::UB; h++) {
                    // (a short last batch reads older frames in the slots past its own; those outputs are not used)
                    int sl = r0 + ub + h;
                    if (sl >= RING) sl -= RING;
                    uint32_t w;
                    if constexpr (NPOL == 2) {
                        w = reinterpret_cast<const uint32_t *>(ring)[sl * N + pt];
                    } else {
                        int sy = r0 + ub + h + half;
                        if (sy >= RING) sy -= RING;
                        const unsigned short *r16 = reinterpret_cast<const unsigned short *>(ring);
                        w = (uint32_t)r16[sl * N + pt] | (uint32_t)r16[sy * N + pt] << 16;
                    }
                    const P2 v = unpack_p2(w ^ 0x80808080u);
#pragma unroll
                    for (int u = 0; u < G::UB; u++) {
                        if (h - u >= 0 && h - u < PT) {
                            y[u].re = __ffma2_rn(c2[h - u], v.re, y[u].re);
                            y[u].im = __ffma2_rn(c2[h - u], v.im, y[u].im);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < G::UB; u++) {
                    if (ub + u < pairs) {
                        // an odd single-pol batch: the last pair has no second spectrum
                        if (NPOL == 1 && half + ub + u >= nb) y[u].re.y = y[u].im.y = 0.f;
                        data[(ub + u) * N + (pt ^ ((pt >> 3) & 7))] = y[u];
                    }
                }
            }
        }
        __syncthreads();  // the batch's outputs are in data; its oldest frames are free
        if (s + G::BS < s_end) stage(s - s_beg + RING, min(G::BS, s_end - s - G::BS), r0);
        r0 += G::BS;
        if (r0 >= RING) r0 -= RING;
        // pass 1: block length N, butterfly j over a = j + M1 q
#pragma unroll
        for (int i = 0; i < 16 / G::R1; i++) {
            const int u = t + 512 * i, j = u % G::M1, sb = u / G::M1;
            if (sb < pairs) {
                P2 *d = data + sb * N + (j ^ ((j >> 3) & 7));
                P2 v[G::R1];
#pragma unroll
                for (int q = 0; q < G::R1; q++) v[q] = d[G::M1 * q];
                Dft<G::R1>::run(v);
                d[0] = v[0];
#pragma unroll
                for (int q = 1; q < G::R1; q++) d[G::M1 * q] = cmul(v[q], __ldg(p.twBt + G::M1 * (q - 1) + j));
            }
        }
        __syncthreads();
        // pass 2: block length 8 R2, block b, butterfly j over a = 8 R2 b + j + 8 q
#pragma unroll
        for (int i = 0; i < 16 / G::R2; i++) {
            const int u = t + 512 * i, j = u & 7, b = (u >> 3) % G::R1, sb = u / (8 * G::R1);
            if (sb < pairs) {
                P2 *d = data + sb * N + b * (8 * G::R2);
                P2 v[G::R2];
#pragma unroll
                for (int q = 0; q < G::R2; q++) v[q] = d[8 * q + (j ^ (q & 7))];
                Dft<G::R2>::run(v);
                d[j] = v[0];
#pragma unroll
                for (int q = 1; q < G::R2; q++) d[8 * q + (j ^ (q & 7))] = cmul(v[q], tw2s[8 * (q - 1) + j]);
            }
        }
        __syncthreads();
        // pass 3: block length 8, detection and sums
        if constexpr (NPOL == 2) {
            uint32_t a[32];
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");  // the previous batch's sums
            if (!fresh) {
                tmem_ld_wait<32>(tm, a);
            } else {
#pragma unroll
                for (int e = 0; e < 32; e++) a[e] = 0u;
            }
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const int sb = set + G::SETS * i;
                if (sb < pairs) {
                    const P2 *d = data + sb * N + 8 * b8;
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[q ^ (b8 & 7)];
                    Dft<8>::run(v);
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
                }
            }
            tmem_st32(tm, a);
            fresh = false;
        } else {
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const int sb = set + G::SETS * i;
                if (sb < pairs) {
                    const P2 *d = data + sb * N + 8 * b8;
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[q ^ (b8 & 7)];
                    Dft<8>::run(v);
#pragma unroll
                    for (int q = 0; q < 8; q++) {  // |X|^2 and |Y|^2, two spectra of the one polarisation
                        const float2 w2 = __ffma2_rn(v[q].re, v[q].re, __fmul2_rn(v[q].im, v[q].im));
                        sum1[q] += w2.x + w2.y;
                    }
                }
            }
        }
        // end of a run, or of the CTA's spectra: the sets of sums, in order, into the slot
        if (++batches == G::kRunBatches || s + G::BS >= s_end) {
            __syncthreads();  // the last pass has read data
            A *red = reinterpret_cast<A *>(data);  // [SETS][N], position 8 b + q at 8 b + (q ^ (b mod 8))
            if constexpr (NPOL == 2) {
                uint32_t a[32];
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tmem_ld_wait<32>(tm, a);
#pragma unroll
                for (int q = 0; q < 8; q++)
                    red[set * N + 8 * b8 + (q ^ (b8 & 7))] =
                        make_float4(__uint_as_float(a[4 * q]), __uint_as_float(a[4 * q + 1]),
                                    __uint_as_float(a[4 * q + 2]), __uint_as_float(a[4 * q + 3]));
                fresh = true;
            } else {
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    red[set * N + 8 * b8 + (q ^ (b8 & 7))] = sum1[q];
                    sum1[q] = 0.f;
                }
            }
            __syncthreads();
            if (dbg_ok((int)blockIdx.x < p.slots, kDbgSlot)) {
                A *part = reinterpret_cast<A *>(p.partial) + (size_t)blockIdx.x * N;
#pragma unroll
                for (int k = 0; k < G::KP; k++) {
                    const int pos = t + 512 * k, r = pos ^ ((pos >> 3) & 7);
                    A v = red[r];
                    for (int l = 1; l < G::SETS; l++) {
                        const A w = red[l * N + r];
                        if constexpr (NPOL == 2) v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
                        else v += w;
                    }
                    if (store) part[pos] = v;
                    else atomicAdd(part + pos, v);  // in L2; one writer per entry, in program order
                }
            }
            store = false;
            batches = 0;
            // (the next batch's first barrier orders these reads before data is written)
        }
    }
    pdl_trigger();
    if constexpr (NPOL == 2) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(*tmem_slot), "r"(128u) : "memory");
    }
}

// Fold of the one-row transforms' slots: position pos = M1 q1 + 8 q2 + q3 of
// every slot is channel q1 + R1 (q2 + R2 q3). A block is 8 positions x 64 slot
// lanes: lane y sums slots y, y + 64, ..., then eight threads of each position
// add eight lane sums in order, then one adds those eight. Band blockIdx.y has
// the slots blockIdx.y * slots .. (The general fold
// takes two launches over as many slots and 32-channel blocks that leave most
// SMs idle at these sizes.)
template <int NPOL>
__global__ void __launch_bounds__(512) fold_row_kernel(const void *partial, int slots, int N, int R1, int R2, void *out) {
    using A = typename Elem<NPOL>::Acc;
    __shared__ A lane_sum[64][8];
    const int tx = threadIdx.x, ty = threadIdx.y, pos = blockIdx.x * 8 + tx;
    const A *pp = reinterpret_cast<const A *>(partial) + (size_t)blockIdx.y * slots * N + pos;
    auto add = [](A &s, const A &v) {
        if constexpr (NPOL == 2) {
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        } else {
            s += v;
        }
    };
    A s;
    if constexpr (NPOL == 2) s = make_float4(0.f, 0.f, 0.f, 0.f);
    else s = 0.f;
    const int q3 = pos & 7, q2 = (pos >> 3) % R2, q1 = pos / (8 * R2);
    A *o = reinterpret_cast<A *>(out) + (size_t)blockIdx.y * N + q1 + R1 * (q2 + R2 * q3);
    A a = s;
    if (ty == 0) a = *o;
    pdl_wait();
    for (int g = ty; g < slots; g += 64) add(s, pp[(size_t)g * N]);
    lane_sum[ty][tx] = s;
    __syncthreads();
    if (ty < 8) {
        s = lane_sum[8 * ty][tx];
#pragma unroll
        for (int l = 1; l < 8; l++) add(s, lane_sum[8 * ty + l][tx]);
    }
    __syncthreads();
    if (ty < 8) lane_sum[ty][tx] = s;
    __syncthreads();
    if (ty) return;
#pragma unroll
    for (int l = 1; l < 8; l++) add(s, lane_sum[l][tx]);
    add(a, s);
    *o = a;
}

}  // namespace vspec
