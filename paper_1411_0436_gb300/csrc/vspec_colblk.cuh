// vspec_colblk.cuh — kernel A of the longest transforms with 2048-point rows:
// columns of N2 = 512 points (2^20 channels; either polarisation count, direct
// or pre-filtered) and, single-pol pre-filtered, 128 and 256 (2^18, 2^19).
//
// A register window of fp32 frames does not fit beside such columns. The int8
// frames stay in shared memory instead (a ring of the PT - 1 + SPB that a batch
// of SPB spectra spans), and each thread forms its points' outputs from one
// walk over the ring: a frame's sample is unpacked once and added into every
// output it is a tap of (8 taps: 11 unpacks for 4 outputs, where reading the
// taps spectrum by spectrum takes 32, and 8 loads from L2). While the columns of
// a batch are transformed, the next frames are copied over the oldest.
//
// Tiles of 2048 points, four per thread. The column is three DIF passes (the
// plan's column pass list {8, N2 / 64, 8}) with four barriers per batch. Batches
// are four spectra, with more than 8 taps two (the ring takes the room). A tile
// row of 2048 / N2 samples is 8 to 32 input bytes: tile groups read a line's
// tiles together. The thread's coefficients and four-step twiddles are fixed
// for a run of spectra: they stay in registers, with more than 8 taps in its own
// lane of tensor memory (128 columns per warp of a lane quarter), from where
// they are read back per point and per batch (at 8 taps that is 2% slower).
//
// Shared memory element i of a spectrum lives, with tiles of 4 columns, at
// i ^ 4 when bit 5 of i is set: the last pass's 8-lane phases span two blocks 32
// elements apart, which would otherwise share banks; the other passes are
// contiguous over a warp either way.
//
// Single-polarisation plans run pairs of spectra, as in vspec_colgrp.cuh.
//
// It is bound, like the grouped kernels, by its phases' shared-memory and FMA
// time (8-byte tile rows: by the copies, one sector each). Kernel A, GB300, us:
// 2^20 dual-pol, 64 spectra: 8 taps 518 (gather kernel 1130), 16 taps 749 (gather
// 2840), direct 423 (general kernel 478); single-pol 8 taps, pairs: 2^18 256
// spectra 240 (general 230, whose rows are 4096 points and cost kernel B 280
// against 162), 2^19 128 spectra 276 (gather 716), 2^20 64 spectra 531 (712);
// 16 taps 2^18 351 (1045), 2^19 390 (1093).
#pragma once
#include "vspec_kernels.cuh"
#include "vspec_tc.cuh"
#include "vspec_tmem.cuh"

namespace vspec {

template <int N2_, int PT_>
struct ColBlk {
    static constexpr int N2 = N2_, PT = PT_, PTS = 2048, C = PTS / N2, THREADS = 512, KP = PTS / THREADS;
    static constexpr int SPB = PT > 8 ? 2 : 4, RING = PT + SPB - 1;
    static constexpr int M1 = N2 / 8, R2 = N2 / 64;          // first-pass stride, second radix
    static constexpr int TW1 = 7 * M1, TW2 = (R2 - 1) * 8;   // pass twiddles, [q - 1][j]
    static constexpr bool kTmem = PT > 8;                    // a run's constants in tensor memory
    static constexpr int TWZ = KP * 16;                      // tensor-memory column of the four-step twiddles
    // data [SPB][PTS] P2, frame ring [RING][PTS] u32, pass twiddles
    static constexpr size_t smem = (size_t)SPB * PTS * 16 + (size_t)RING * PTS * 4 + (TW1 + TW2) * 8 + 16;
    __device__ static constexpr int sw(int i) { return C == 4 ? i ^ ((i >> 3) & 4) : i; }
    static_assert(smem <= 232448, "shared memory of one CTA");
    static_assert(N2 >= 128 && N2 <= 512 && TWZ + 16 <= 128, "column shapes; a thread's tensor-memory columns");
};

template <int N2_, int PT_, int NPOL>
__global__ void __launch_bounds__(512, 1) fir_colblk_kernel(const __grid_constant__ ColParams p) {
    pdl_trigger();
    using G = ColBlk<N2_, PT_>;
    constexpr int PTS = G::PTS, C = G::C, PT = G::PT, SPB = G::SPB, RING = G::RING, R2 = G::R2, KP = G::KP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    P2 *data = reinterpret_cast<P2 *>(smem_raw);                      // [SPB][PTS]
    uint32_t *ring = reinterpret_cast<uint32_t *>(data + SPB * PTS);  // [RING][PTS] words, or [2][RING][PTS] halves
    float2 *tw1 = reinterpret_cast<float2 *>(ring + RING * PTS);      // [7][M1]
    float2 *tw2 = tw1 + G::TW1;                                       // [R2 - 1][8]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tw2 + G::TW2);
    const int t = threadIdx.x, warp = t >> 5, e = t & 255;
    const int D = PT - p.P;  // leading zero taps
    if (G::kTmem && warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::smem_addr(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = t; i < G::TW1; i += G::THREADS) tw1[i] = __ldg(p.twA + p.pass[0].off + (i % G::M1) * 7 + i / G::M1);
    for (int i = t; i < G::TW2; i += G::THREADS) tw2[i] = __ldg(p.twA + p.pass[1].off + (i % 8) * (R2 - 1) + i / 8);
    uint32_t tm = 0;
    if constexpr (G::kTmem) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tm = *tmem_slot + ((uint32_t)((warp & 3) * 32) << 16) + 128 * (warp >> 2);
    }

    const TileSplit sp = tile_split(p.tiles, p.sc, p.G);
    for (long long f = sp.lo; f < sp.hi;) {
        const long long base = f / p.sc * p.sc;  // first item of this super-tile
        const int x = (int)(f / p.sc) * sp.G + sp.r;
        const int s_beg = (int)(f - base);
        const int s_end = (int)(min(sp.hi, base + p.sc) - base);
        f = base + s_end;
        const int w0 = x * C;  // first column

        // Ring slot (fr - first) mod RING holds absolute frame fr, first the
        // oldest frame of the run's first spectrum (its D leading taps have zero
        // coefficients: their frames are not copied).
        const long long first = p.s0 + s_beg - D;
        auto stage = [&](int rel, int cnt, int slot, int halves) {  // frames first + rel .. + cnt - 1 from ring slot `slot`
            auto frame = [&](int u, long long *fr, int *sl) {
                *fr = first + rel + u;
                *sl = slot + u >= RING ? slot + u - RING : slot + u;
            };
            long long fr;
            int sl;
            if constexpr (NPOL == 1) {
                constexpr int CB = C * 2 < 16 ? C * 2 : 16, per = PTS * 2 / CB, per_row = C * 2 / CB;
                for (int i = t; i < halves * cnt * per; i += G::THREADS) {
                    const int y = i >= cnt * per, u = (i - y * cnt * per) / per, r = i % per;
                    frame(u, &fr, &sl);
                    if (y) fr += p.half;
                    const unsigned char *src = reinterpret_cast<const unsigned char *>(p.in) +
                                               (fr * p.N + (long long)p.N1 * (r / per_row) + w0) * 2 + r % per_row * CB;
                    unsigned char *dst = reinterpret_cast<unsigned char *>(ring) + (size_t)(y * RING + sl) * PTS * 2 + r * CB;
                    // (the second half's frames past the input belong to the spectrum an odd chunk lacks)
                    if (fr >= p.nframes) {
                        if (!y) dbg_ok(false, kDbgInput);
                        continue;
                    }
                    if constexpr (CB == 16)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(tc::smem_addr(dst)), "l"(src) : "memory");
                    else
                        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" :: "r"(tc::smem_addr(dst)), "l"(src), "n"(CB) : "memory");
                }
            } else {
                constexpr int per_row = C / 4;
                for (int i = t; i < cnt * (PTS / 4); i += G::THREADS) {
                    const int r = i % (PTS / 4);
                    frame(i / (PTS / 4), &fr, &sl);
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(p.in) + fr * p.N +
                                          (long long)p.N1 * (r / per_row) + w0 + r % per_row * 4;
                    if (dbg_ok(fr < p.nframes, kDbgInput))
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                     :: "r"(tc::smem_addr(ring + sl * PTS + 4 * r)), "l"(src) : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // (a run of an odd chunk's last pair alone has one spectrum per pair)
        stage(D, PT - 1 - D + min(SPB, s_end - s_beg), D, NPOL == 1 && p.half + s_beg >= p.nreal ? 1 : 2);

        // the run's constants: coefficient h of point k (tile element t + 512 k,
        // row n2 = that / C; in tensor memory at column 16 k + h); the twiddles of
        // the last pass's block e / C, outputs at rows 8 (e / C) + q
        auto coef = [&](int k, int h) {
            const int pt = t + 512 * k;
            return h < PT && h >= D ? __ldg(p.coef + (size_t)(h - D) * p.N + w0 + pt % C + (size_t)p.N1 * (pt / C)) : 0.f;
        };
        auto zw = [&](int q) { return __ldg(p.twZ + (size_t)(8 * (e / C) + q) * p.N1 + w0 + e % C); };
        float cr[G::kTmem ? 1 : KP][G::kTmem ? 1 : PT];
        float2 tz[8];
        if constexpr (G::kTmem) {
#pragma unroll
            for (int k = 0; k < KP; k += 2) {
                uint32_t v[32];
#pragma unroll
                for (int i = 0; i < 32; i++) v[i] = __float_as_uint(coef(k + i / 16, i % 16));
                tmem_st32(tm + 16 * k, v);
            }
            uint32_t v[32];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const float2 w = zw(q);
                v[2 * q] = __float_as_uint(w.x);
                v[2 * q + 1] = __float_as_uint(w.y);
                v[16 + 2 * q] = v[17 + 2 * q] = 0u;
            }
            tmem_st32(tm + G::TWZ, v);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        } else {
#pragma unroll
            for (int k = 0; k < KP; k++)
#pragma unroll
                for (int h = 0; h < PT; h++) cr[k][h] = coef(k, h);
#pragma unroll
            for (int q = 0; q < 8; q++) tz[q] = zw(q);
        }

        int r0 = 0;  // ring slot of the batch's oldest frame
        for (int s = s_beg; s < s_end; s += SPB) {
            const int nb = min(SPB, s_end - s);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();  // the batch's frames are visible; data is free
#pragma unroll
            for (int k = 0; k < KP; k++) {
                const int pt = t + 512 * k;
                float2 c2[PT];
                if constexpr (G::kTmem) {
                    uint32_t cf[32];
                    tmem_ld_wait<16>(tm + 16 * k, cf);
#pragma unroll
                    for (int h = 0; h < PT; h++) c2[h] = dup2(__uint_as_float(cf[h]));
                } else {
#pragma unroll
                    for (int h = 0; h < PT; h++) c2[h] = dup2(cr[k][h]);
                }
                P2 y[SPB];
#pragma unroll
                for (int h = 0; h < RING; h++) {
                    // (a short last batch reads older frames in the slots past its own; those outputs are not used)
                    const int sl = r0 + h >= RING ? r0 + h - RING : r0 + h;
                    uint32_t w;
                    if constexpr (NPOL == 1) {
                        const unsigned short *r16 = reinterpret_cast<const unsigned short *>(ring) + sl * PTS + pt;
                        w = (uint32_t)r16[0] | (uint32_t)r16[RING * PTS] << 16;
                    } else {
                        w = ring[sl * PTS + pt];
                    }
                    const P2 v = unpack_p2(w ^ 0x80808080u);
#pragma unroll
                    for (int u = 0; u < SPB; u++) {
                        if (h == u) {
                            y[u] = P2{__fmul2_rn(c2[0], v.re), __fmul2_rn(c2[0], v.im)};
                        } else if (h > u && h - u < PT) {
                            y[u].re = __ffma2_rn(c2[h - u], v.re, y[u].re);
                            y[u].im = __ffma2_rn(c2[h - u], v.im, y[u].im);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < SPB; u++) {
                    if (u < nb) {
                        if (NPOL == 1 && p.half + s + u >= p.nreal) y[u].re.y = y[u].im.y = 0.f;
                        data[u * PTS + G::sw(pt)] = y[u];
                    }
                }
            }
            __syncthreads();  // the batch's outputs are in data; the ring's oldest frames are free
            if (s + SPB < s_end) stage(s - s_beg + RING, min(SPB, s_end - s - SPB), r0, 2);
            r0 += SPB;
            if (r0 >= RING) r0 -= RING;
            // pass 1: block length N2, butterfly j = e / C over rows j + M1 q
#pragma unroll
            for (int h = 0; h < SPB / 2; h++) {
                const int sb = (t >> 8) + 2 * h;
                if (sb < nb) {
                    P2 *d = data + sb * PTS + G::sw(e);
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[256 * q];
                    Dft<8>::run(v);
                    d[0] = v[0];
#pragma unroll
                    for (int q = 1; q < 8; q++) d[256 * q] = cmul(v[q], tw1[G::M1 * (q - 1) + e / C]);
                }
            }
            __syncthreads();
            // pass 2: block length M1, block u / (8 C), butterfly j = (u / C) mod 8 over rows j + 8 q
#pragma unroll
            for (int h = 0; h < SPB * 4 / R2; h++) {
                const int u = (t + 512 * h) % (64 * C), sb = (t + 512 * h) / (64 * C), l = u % (8 * C);
                if (sb < nb) {
                    P2 *d = data + sb * PTS + u / (8 * C) * 256;
                    P2 v[R2];
#pragma unroll
                    for (int q = 0; q < R2; q++) v[q] = d[8 * C * q + (C == 4 ? l ^ (4 * (q & 1)) : l)];
                    Dft<R2>::run(v);
                    d[l] = v[0];
#pragma unroll
                    for (int q = 1; q < R2; q++)
                        d[8 * C * q + (C == 4 ? l ^ (4 * (q & 1)) : l)] = cmul(v[q], tw2[8 * (q - 1) + l / C]);
                }
            }
            if constexpr (G::kTmem) {
                uint32_t w[32];
                tmem_ld_wait<16>(tm + G::TWZ, w);
#pragma unroll
                for (int q = 0; q < 8; q++) tz[q] = make_float2(__uint_as_float(w[2 * q]), __uint_as_float(w[2 * q + 1]));
            }
            __syncthreads();
            // pass 3: block length 8, block b = e / C, rows 8 b + q, to the scratch
#pragma unroll
            for (int h = 0; h < SPB / 2; h++) {
                const int sb = (t >> 8) + 2 * h;
                if (sb < nb) {
                    const int b = e / C, c = e % C;
                    const P2 *d = data + sb * PTS + 8 * C * b + c;
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[C * (C == 4 ? q ^ (b & 1) : q)];
                    Dft<8>::run(v);
                    P2 *z = reinterpret_cast<P2 *>(p.Z) + (size_t)(s + sb) * p.N + (size_t)(8 * b) * p.N1 + w0 + c;
                    if (!dbg_ok(s + sb < p.sc && w0 + c < p.N1, kDbgScratch)) continue;
#pragma unroll
                    for (int q = 0; q < 8; q++) z[(size_t)q * p.N1] = cmul(v[q], tz[q]);
                }
            }
        }
        __syncthreads();  // the last batch's frames are read before the next run's copies
    }
    if constexpr (!G::kTmem) return;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(*tmem_slot), "r"(512u) : "memory");
}

}  // namespace vspec
