// vspec_coldirgrp.cuh — kernel A of direct-FFT plans with 2048-point rows: column
// DFTs of N2 = 2 .. 256 points straight from the int8 input, four-step twiddle,
// stores to the chunk scratch.
//
// One 512-thread CTA per SM, four independent groups of 128 threads. Each group
// owns a tile of 2048 points (C = 2048 / N2 columns) and its own run of spectra,
// one spectrum at a time (16 points per thread), and synchronises only on its
// own named barrier: the groups drift apart, so that one group's loads, shared
// memory passes and stores run under another's arithmetic. Frames are copied
// DEPTH - 1 spectra ahead.
//
// Columns of at most 16 points are whole DFTs in registers from the staged
// bytes (natural order); longer ones take two DIF passes, radix 16 from the
// staged bytes into fp32 shared memory, then N2 / 16 (the plan's column pass
// list). A thread's 16 outputs sit at the same places for every spectrum of a
// run: their four-step twiddles (and the 16 window values, if there is a
// window) live in its lane of tensor memory.
//
// Single-polarisation plans (NPOL = 1) transform two spectra at once, pair s
// holding spectra s and s + half of the chunk (see vspec_colgrp.cuh).
//
// Measured (GB300, kernel A, against one 512-thread group per CTA with barriers
// between the passes): see pick_kernel_coldir.
#pragma once
#include "vspec_kernels.cuh"
#include "vspec_tc.cuh"
#include "vspec_tmem.cuh"

namespace vspec {

template <int N2_>
struct ColDirGrp {
    static constexpr int N2 = N2_, GROUPS = 4, TG = 128, PTS = 2048, C = PTS / N2;
    static constexpr bool kOnePass = N2 <= 16;
    static constexpr int R1 = kOnePass ? N2 : 16, R2 = N2 / R1, M1 = N2 / R1;
    static constexpr int DEPTH = 3;  // frames in shared memory per group
    static constexpr int TWC = kOnePass ? 0 : M1 * (R1 - 1);  // first-pass twiddles, [q - 1][j]
    static constexpr size_t group_bytes = (size_t)DEPTH * PTS * 4 + (kOnePass ? 0 : (size_t)PTS * 16);
    static constexpr size_t smem = GROUPS * group_bytes + TWC * 8 + 16;
    static_assert(N2 >= 2 && N2 <= 256 && smem <= 232448, "column shapes of this kernel");
};

template <int N2_, int NPOL>
__global__ void __launch_bounds__(512, 1) fir_coldirgrp_kernel(const __grid_constant__ ColParams p) {
    pdl_trigger();
    using G = ColDirGrp<N2_>;
    constexpr int N2 = G::N2, PTS = G::PTS, C = G::C, TG = G::TG, R1 = G::R1, R2 = G::R2, M1 = G::M1, DEPTH = G::DEPTH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, g = tid / TG, t = tid % TG, warp = tid >> 5;
    uint32_t *raw = reinterpret_cast<uint32_t *>(smem_raw + g * G::group_bytes);  // [DEPTH][PTS] words or 2 x halves
    P2 *data = reinterpret_cast<P2 *>(raw + DEPTH * PTS);                         // [PTS] (two passes)
    float2 *twc = reinterpret_cast<float2 *>(smem_raw + G::GROUPS * G::group_bytes);  // [R1 - 1][M1]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(twc + G::TWC);
    const size_t zs = p.zstride > 0 ? (size_t)p.zstride : (size_t)p.N;  // scratch spectrum stride

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::smem_addr(tmem_slot)), "r"(256u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if constexpr (!G::kOnePass)
        for (int e = tid; e < G::TWC; e += 512) twc[e] = __ldg(p.twA + p.pass[0].off + (e % M1) * (R1 - 1) + e / M1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = *tmem_slot + ((uint32_t)((warp & 3) * 32) << 16) + 64 * (warp >> 2);
    auto bar = [&]() { asm volatile("bar.sync %0, %1;" :: "r"(1 + g), "n"(TG) : "memory"); };

    // this group's share: as tile_split, with groups as the workers
    const int wk = blockIdx.x * G::GROUPS + g, nw = gridDim.x * G::GROUPS, TGR = p.G < 1 ? 1 : p.G;
    const long long T = (long long)(p.tiles / TGR) * p.sc;
    const int ng = nw / TGR, gi = wk / TGR;
    const long long lo = gi < ng ? T * gi / ng : 0, hi = gi < ng ? T * (gi + 1) / ng : 0;
    for (long long f = lo; f < hi;) {
        const long long base = f / p.sc * p.sc;  // first item of this super-tile
        int x = (int)(f / p.sc) * TGR + wk % TGR;
        const int s_beg = (int)(f - base);
        const int s_end = (int)(min(hi, base + p.sc) - base);
        f = base + s_end;
        int band = p.band;  // sub-band input (see ColParams)
        if (p.lsub) band = 0;
        else if (p.band < 0) {
            band = x % p.nsub;
            x /= p.nsub;
        }
        P2 *Zc = reinterpret_cast<P2 *>(p.Z) + (p.band < 0 && !p.lsub ? (size_t)band * p.N : 0);
        const int w0 = x * C;  // first column (or word) of the tile
        auto column = [&](int c) { return (w0 + c) >> p.lsub; };
        auto zcol = [&](int c) { return (p.lsub ? (size_t)((w0 + c) & (p.nsub - 1)) * p.N : 0) + column(c); };

        // frame of spectrum s into raw[buf] (16-byte copies; sub-band input not
        // interleaved in the tile: 4-byte copies of the band's samples)
        auto stage = [&](int s, int buf) {
            long long fr = p.s0 + s;
            if constexpr (NPOL == 1) {
                constexpr int per_row = C / 8;
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int e = (t + TG * i) % (PTS / 8), y = (t + TG * i) / (PTS / 8);
                    const long long fy = fr + y * p.half;
                    // (the second half's frame past the input is the spectrum that an odd chunk lacks)
                    if (fy >= p.nframes) {
                        if (!y) dbg_ok(false, kDbgInput);
                        continue;
                    }
                    const unsigned char *src = reinterpret_cast<const unsigned char *>(p.in) +
                                               (fy * p.N + (long long)p.N1 * (e / per_row) + w0 + e % per_row * 8) * 2;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                 :: "r"(tc::smem_addr(raw + buf * PTS + y * (PTS / 2) + 4 * e)), "l"(src) : "memory");
                }
            } else if (p.nsub > 1 && !p.lsub) {
                for (int e = t; e < PTS; e += TG) {
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(p.in) +
                                          (fr * p.N + w0 + (long long)p.N1 * (e / C) + e % C) * p.nsub + band;
                    if (dbg_ok(fr < p.nframes, kDbgInput))
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                                     :: "r"(tc::smem_addr(raw + buf * PTS + e)), "l"(src) : "memory");
                }
            } else {
                constexpr int per_row = C / 4;
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int e = t + TG * i;
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(p.in) +
                                          ((fr * p.N + (long long)p.N1 * (e / per_row)) << p.lsub) + w0 + e % per_row * 4;
                    if (dbg_ok(fr < p.nframes && e / per_row < p.N2 && column(e % per_row * 4 + 3) < p.N1, kDbgInput))
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                     :: "r"(tc::smem_addr(raw + buf * PTS + 4 * e)), "l"(src) : "memory");
                }
            }
        };
        bar();  // the previous run's frames are read
#pragma unroll
        for (int d = 0; d < DEPTH - 1; d++) {
            if (s_beg + d < s_end) stage(s_beg + d, d);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }

        // the run's four-step twiddles and window values, into this thread's lane
        {
            uint32_t v[32];
#pragma unroll
            for (int i = 0; i < 16; i++) {
                // output i: butterfly k = i / R of the last pass (radix R), row row0 + i mod R
                constexpr int R = G::kOnePass ? N2 : R2;
                const int e = t + TG * (i / R), c = e % C, row = (G::kOnePass ? 0 : e / C * R2) + i % R;
                if (!dbg_ok(row < p.N2 && column(c) < p.N1, kDbgTile)) continue;
                const float2 w = __ldg(p.twZ + (size_t)row * p.N1 + column(c));
                v[2 * i] = __float_as_uint(w.x);
                v[2 * i + 1] = __float_as_uint(w.y);
            }
            tmem_st32(tm, v);
            if (p.win) {
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    // input i: butterfly k = i / R1 of the first pass, row j + M1 (i mod R1)
                    const int e = t + TG * (i / R1), c = e % C, row = e / C + M1 * (i % R1);
                    v[i] = __float_as_uint(__ldg(p.coef + (size_t)row * p.N1 + column(c)));
                    v[16 + i] = 0u;
                }
                tmem_st32(tm + 32, v);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }

        for (int s = s_beg, buf = 0; s < s_end; s++, buf = buf + 1 == DEPTH ? 0 : buf + 1) {
            asm volatile("cp.async.wait_group %0;" :: "n"(DEPTH - 2) : "memory");
            bar();  // spectrum s's frame is visible; the buffer of s - 1 and data are free
            if (s + DEPTH - 1 < s_end) stage(s + DEPTH - 1, buf == 0 ? DEPTH - 1 : buf - 1);
            asm volatile("cp.async.commit_group;" ::: "memory");
            const uint32_t *rb = raw + buf * PTS;
            const bool no_y = NPOL == 1 && p.half + s >= p.nreal;  // an odd chunk's last pair
            uint32_t win[32];
            if (p.win) {
                tmem_ld_wait<16>(tm + 32, win);
            }
            auto sample = [&](int e, int i) {  // tile element e, input i of this thread
                uint32_t w;
                if constexpr (NPOL == 1) {
                    const unsigned short *r16 = reinterpret_cast<const unsigned short *>(rb);
                    w = (uint32_t)r16[e] | (no_y ? 0u : (uint32_t)r16[PTS + e] << 16);
                } else {
                    w = rb[e];
                }
                P2 v = unpack_p2(w ^ 0x80808080u);
                if (p.win) {
                    const float2 h = dup2(__uint_as_float(win[i]));
                    v = P2{__fmul2_rn(v.re, h), __fmul2_rn(v.im, h)};
                }
                return v;
            };
            P2 *zrow = Zc + (size_t)s * zs;
            uint32_t tw[32];
            auto twiddle = [&](int i) {
                return make_float2(__uint_as_float(tw[2 * i]), __uint_as_float(tw[2 * i + 1]));
            };
            if constexpr (G::kOnePass) {
#pragma unroll
                for (int k = 0; k < C / TG; k++) {
                    const int c = t + TG * k;
                    P2 v[N2];
#pragma unroll
                    for (int q = 0; q < N2; q++) v[q] = sample(q * C + c, k * N2 + q);
                    Dft<N2>::run(v);
                    if (k == 0) {  // (after the DFT, whose registers they would compete for)
                        tmem_ld_wait<32>(tm, tw);
                    }
                    P2 *z = zrow + zcol(c);
                    if (!dbg_ok(s < p.sc && column(c) < p.N1, kDbgScratch)) continue;
                    z[0] = v[0];
#pragma unroll
                    for (int q = 1; q < N2; q++) z[(size_t)q * p.N1] = cmul(v[q], twiddle(k * N2 + q));
                }
            } else {
                // first pass: butterfly j = t / C of column c = t mod C over rows j + M1 q
                {
                    P2 v[R1];
#pragma unroll
                    for (int q = 0; q < R1; q++) v[q] = sample(t + q * M1 * C, q);
                    Dft<R1>::run(v);
                    data[t] = v[0];
#pragma unroll
                    for (int q = 1; q < R1; q++) data[t + q * M1 * C] = cmul(v[q], twc[M1 * (q - 1) + t / C]);
                }
                bar();
                // second pass: block b of column c, rows b R2 + q, to the scratch
#pragma unroll
                for (int k = 0; k < C * R1 / TG; k++) {
                    const int e = t + TG * k, c = e % C, b = e / C;
                    P2 v[R2];
#pragma unroll
                    for (int q = 0; q < R2; q++) v[q] = data[(b * R2 + q) * C + c];
                    Dft<R2>::run(v);
                    if (k == 0) {
                        tmem_ld_wait<32>(tm, tw);
                    }
                    P2 *z = zrow + (size_t)(b * R2) * p.N1 + zcol(c);
                    if (!dbg_ok(s < p.sc && column(c) < p.N1, kDbgScratch)) continue;
#pragma unroll
                    for (int q = 0; q < R2; q++) z[(size_t)q * p.N1] = cmul(v[q], twiddle(k * R2 + q));
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(*tmem_slot), "r"(256u) : "memory");
}

}  // namespace vspec
