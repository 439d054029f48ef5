// vspec_colgrp.cuh — kernel A of the pre-filtered plans with 2048-point rows
// (4096 at 2^19): pre-filter, column DFTs of N2 = 2 .. 128 points, four-step
// twiddle, stores to the chunk scratch.
//
// One 512-thread CTA per SM, in GROUPS independent groups of TG threads. Each
// group owns a tile of 512 points (C = 512 / N2 columns) and its own run of
// spectra, and synchronises only on its own named barrier, so that the groups
// drift apart and one group's shared-memory phases run under another's
// arithmetic (measured figures: pick_kernel_colreg, build_plan). (One group of 512 threads with the frames in a register window
// issued fewer instructions but ran its phases one after another: FMA pipe 41%
// and LSU data path 53% of the cycles, each waiting for the other.)
//
// Per batch of SPB spectra (16 points per thread):
//  - the pre-filter: the int8 frames stay in a shared-memory ring of the
//    PT - 1 + SPB frames a batch spans; each thread forms a point's SPB outputs
//    from one walk over the ring, unpacking a sample once for all the outputs
//    it is a tap of. While the columns are transformed, the next frames are
//    copied over the oldest.
//  - the column DFTs: columns of at most 16 points are whole DFTs in registers
//    (one pass, natural order); longer ones take two DIF passes, radix 8 then
//    N2 / 8 (the plan's column pass list).
//  - every output times W_N^(n1 k2), stored to the scratch.
// A thread's coefficients and four-step twiddles are fixed for a run; they
// live in its own lane of tensor memory (at most 32 + 32 columns) and are read
// back with one tcgen05.ld per batch, instead of holding registers through the
// passes or taking shared-memory bandwidth.
//
// Single-polarisation plans (NPOL = 1) run the same paired arithmetic on two
// spectra at once: pair s of a chunk holds spectra s and s + half (the second
// half of the chunk), so a scratch element is (X, Y) of the same point in two
// spectra. An odd chunk's last pair has no second spectrum: its Y half is zero.
#pragma once
#include "vspec_kernels.cuh"
#include "vspec_tc.cuh"
#include "vspec_tmem.cuh"

namespace vspec {

template <int N2_, int PT_, int GROUPS_>
struct ColGrp {
    static constexpr int N2 = N2_, PT = PT_, GROUPS = GROUPS_, PTS = 512, C = PTS / N2;
    static constexpr bool kOnePass = N2 <= 16;
    static constexpr int R1 = kOnePass ? N2 : 8, R2 = N2 / R1, M1 = N2 / R1;
    static constexpr int TG = 512 / GROUPS, KP = PTS / TG;  // threads per group; points per thread
    static constexpr int SPB = 16 / GROUPS;                 // spectra per batch
    static constexpr int UB = SPB < 8 ? SPB : 8;            // outputs formed together
    static constexpr int RING = PT - 1 + SPB;               // frames a batch spans
    // Narrow tiles (C < 8 in the two-pass form): an 8-lane phase of the second
    // pass spans 8 / C blocks, C R2 elements apart; C pad elements after every
    // C R2 put them in different banks.
    static constexpr int PADG = !kOnePass && C < 8 ? C * R2 : 0, PADW = C;
    static constexpr int SS = PTS + (PADG ? PTS / PADG * PADW : 0);
    __device__ static constexpr int pad(int i) { return PADG ? i + i / PADG * PADW : i; }
    static constexpr int TWC = kOnePass ? 0 : M1 * (R1 - 1);  // first-pass twiddles, [q - 1][j]
    // distinct columns of a thread's outputs, and its four-step twiddles per column
    static constexpr int NC = C > TG ? C / TG : 1, NT = kOnePass ? N2 : R2;
    static constexpr int NCF = KP * PT;                      // coefficients of a thread
    static constexpr size_t group_bytes = (size_t)SPB * SS * 16 + (size_t)RING * PTS * 4;
    static constexpr size_t smem = GROUPS * group_bytes + TWC * 8 + 16;
    static_assert(NCF <= 32 && 2 * NC * NT <= 32, "a thread's tensor-memory columns");
};

template <int N2_, int PT_, int GROUPS_, int NPOL, bool BANDS = false>
__global__ void __launch_bounds__(512, 1) fir_colgrp_kernel(const __grid_constant__ ColParams p) {
    pdl_trigger();
    using G = ColGrp<N2_, PT_, GROUPS_>;
    constexpr int N2 = G::N2, PT = G::PT, PTS = G::PTS, C = G::C, TG = G::TG, KP = G::KP, SPB = G::SPB, RING = G::RING,
                  SS = G::SS, R1 = G::R1, R2 = G::R2, M1 = G::M1;
    static_assert(G::smem <= 232448, "shared memory of one CTA");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, g = tid / TG, t = tid % TG, warp = tid >> 5;
    P2 *data = reinterpret_cast<P2 *>(smem_raw + g * G::group_bytes);     // [SPB][SS]
    uint32_t *ring = reinterpret_cast<uint32_t *>(data + SPB * SS);       // [RING][PTS] words, or [2][RING][PTS] halves
    float2 *twc = reinterpret_cast<float2 *>(smem_raw + G::GROUPS * G::group_bytes);  // [R1 - 1][M1]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(twc + G::TWC);
    const int D = PT - p.P;  // leading zero taps
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
        // sub-band input (see ColParams): the tile's band, or (lsub) every band's
        // words side by side
        int band = p.band;
        if (p.lsub) band = 0;
        else if (p.band < 0) {
            band = x % p.nsub;
            x /= p.nsub;
        }
        P2 *Zc = reinterpret_cast<P2 *>(p.Z) + (p.band < 0 && !p.lsub ? (size_t)band * p.N : 0);
        const int w0 = x * C;  // first column (or word) of the tile
        auto column = [&](int c) { return (w0 + c) >> p.lsub; };
        auto zcol = [&](int c) { return (p.lsub ? (size_t)((w0 + c) & (p.nsub - 1)) * p.N : 0) + column(c); };
        // BANDS: interleaved tiles, columns transformed and stored in band order (BandOrder)
        static_assert(!BANDS || G::kOnePass, "whole columns");
        const BandOrder bo{p.nsub, p.lsub, p.lC - p.lsub};
        auto outcol = [&](int c) { return BANDS ? (w0 >> p.lsub) + bo.out_col(c) : column(c); };

        // Ring slot (fr - first) mod RING holds absolute frame fr, first the oldest
        // frame of the run's first spectrum. Its D leading taps have zero
        // coefficients: their frames are not copied (whatever bytes are in the slots
        // are finite samples).
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
                for (int i = t; i < halves * cnt * per; i += TG) {
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
            } else if (p.nsub > 1 && !p.lsub) {  // this band's samples, nsub words apart
                for (int i = t; i < cnt * PTS; i += TG) {
                    const int r = i % PTS;
                    frame(i / PTS, &fr, &sl);
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(p.in) +
                                          (fr * p.N + w0 + (long long)p.N1 * (r / C) + r % C) * p.nsub + band;
                    if (dbg_ok(fr < p.nframes, kDbgInput))
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                                     :: "r"(tc::smem_addr(ring + sl * PTS + r)), "l"(src) : "memory");
                }
            } else {
                constexpr int per_row = C / 4;
                for (int i = t; i < cnt * (PTS / 4); i += TG) {
                    const int r = i % (PTS / 4);
                    frame(i / (PTS / 4), &fr, &sl);
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(p.in) +
                                          ((fr * p.N + (long long)p.N1 * (r / per_row)) << p.lsub) + w0 + r % per_row * 4;
                    if (dbg_ok(fr < p.nframes, kDbgInput))
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                     :: "r"(tc::smem_addr(ring + sl * PTS + 4 * r)), "l"(src) : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // (the last run's readers of the ring are past its last barrier)
        // (a run of an odd chunk's last pair alone has one spectrum per pair)
        stage(D, PT - 1 - D + min(SPB, s_end - s_beg), D, NPOL == 1 && p.half + s_beg >= p.nreal ? 1 : 2);

        // the run's coefficients and four-step twiddles, into this thread's lane
        {
            uint32_t v[32];
#pragma unroll
            for (int i = 0; i < 32; i++) v[i] = 0u;
#pragma unroll
            for (int k = 0; k < KP; k++) {
                const int pt = t + TG * k;
                const float *h = p.coef + column(pt % C) + (size_t)p.N1 * (pt / C);
#pragma unroll
                for (int i = 0; i < PT; i++)
                    if (i >= D) v[k * PT + i] = __float_as_uint(__ldg(h + (size_t)(i - D) * p.N));
            }
            tmem_st32(tm, v);
#pragma unroll
            for (int i = 0; i < G::NC; i++) {
                const int e = t + TG * i, c = e % C, row0 = G::kOnePass ? 0 : (e / C) % R1 * R2;
#pragma unroll
                for (int q = 0; q < G::NT; q++) {
                    const float2 w = __ldg(p.twZ + (size_t)(row0 + q) * p.N1 + outcol(c));
                    v[2 * (i * G::NT + q)] = __float_as_uint(w.x);
                    v[2 * (i * G::NT + q) + 1] = __float_as_uint(w.y);
                }
            }
            tmem_st32(tm + 32, v);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
        int r0 = 0;  // ring slot of the batch's oldest frame
        for (int s = s_beg; s < s_end; s += SPB) {
            const int nb = min(SPB, s_end - s);
            uint32_t cf[32];
            tmem_ld_wait<(G::NCF + 7) / 8 * 8>(tm, cf);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            bar();  // the batch's frames are visible; data is free
#pragma unroll
            for (int k = 0; k < KP; k++) {
                const int pt = t + TG * k;
                float2 c2[PT];
#pragma unroll
                for (int h = 0; h < PT; h++) c2[h] = dup2(__uint_as_float(cf[k * PT + h]));
#pragma unroll
                for (int ub = 0; ub < SPB; ub += G::UB) {
                    if (ub >= nb) break;
                    P2 y[G::UB];
#pragma unroll
                    for (int h = 0; h < PT - 1 + G::UB; h++) {
                        // (a short last batch reads older frames in the slots past its own; those outputs are not used)
                        int sl = r0 + ub + h;
                        if (sl >= RING) sl -= RING;
                        uint32_t w;
                        if constexpr (NPOL == 1) {
                            const unsigned short *r16 = reinterpret_cast<const unsigned short *>(ring) + sl * PTS + pt;
                            w = (uint32_t)r16[0] | (uint32_t)r16[RING * PTS] << 16;
                        } else {
                            w = ring[sl * PTS + pt];
                        }
                        const P2 v = unpack_p2(w ^ 0x80808080u);
#pragma unroll
                        for (int u = 0; u < G::UB; u++) {
                            if (h == u) {
                                y[u] = P2{__fmul2_rn(c2[0], v.re), __fmul2_rn(c2[0], v.im)};
                            } else if (h > u && h - u < PT) {
                                y[u].re = __ffma2_rn(c2[h - u], v.re, y[u].re);
                                y[u].im = __ffma2_rn(c2[h - u], v.im, y[u].im);
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < G::UB; u++) {
                        if (ub + u < nb) {
                            if (NPOL == 1 && p.half + s + ub + u >= p.nreal) y[u].re.y = y[u].im.y = 0.f;
                            data[(ub + u) * SS + (BANDS ? pt / C * C + bo.of_word(pt % C) : G::pad(pt))] = y[u];
                        }
                    }
                }
            }
            bar();  // the batch's outputs are in data; its oldest frames are free
            if (s + SPB < s_end) stage(s - s_beg + RING, min(SPB, s_end - s - SPB), r0, 2);
            r0 += SPB;
            if (r0 >= RING) r0 -= RING;
            uint32_t tw[32];
            constexpr int NTW = 2 * G::NC * G::NT < 8 ? 8 : 2 * G::NC * G::NT;
            auto twiddle = [&](int i) {
                return make_float2(__uint_as_float(tw[2 * i]), __uint_as_float(tw[2 * i + 1]));
            };
            if constexpr (G::kOnePass) {
                tmem_ld_wait<NTW>(tm + 32, tw);
#pragma unroll
                for (int k = 0; k < SPB * C / TG; k++) {
                    const int e = t + TG * k, c = e % C, sb = e / C;
                    if (sb < nb) {
                        P2 v[N2];
                        const int rd = BANDS ? bo.of_out(c) : c;
#pragma unroll
                        for (int q = 0; q < N2; q++) v[q] = data[sb * SS + q * C + rd];
                        Dft<N2>::run(v);
                        P2 *z = Zc + (size_t)(s + sb) * zs + (BANDS ? (size_t)bo.out_band(c) * p.N + outcol(c) : zcol(c));
                        if (!dbg_ok(s + sb < p.sc && outcol(c) < p.N1, kDbgScratch)) continue;
                        z[0] = v[0];
#pragma unroll
                        for (int q = 1; q < N2; q++) z[(size_t)q * p.N1] = cmul(v[q], twiddle(k % G::NC * N2 + q));
                    }
                }
            } else {
                // first pass: butterfly j of column (sb, c) over rows j + M1 q
#pragma unroll
                for (int k = 0; k < SPB * C * M1 / TG; k++) {
                    const int e = t + TG * k, j = e / C % M1, sb = e / (C * M1);
                    if (sb < nb) {
                        P2 *d = data + sb * SS + e % (C * M1);
                        P2 v[R1];
#pragma unroll
                        for (int q = 0; q < R1; q++) v[q] = d[G::pad(q * M1 * C)];
                        Dft<R1>::run(v);
                        d[0] = v[0];
#pragma unroll
                        for (int q = 1; q < R1; q++) d[G::pad(q * M1 * C)] = cmul(v[q], twc[M1 * (q - 1) + j]);
                    }
                }
                tmem_ld_wait<NTW>(tm + 32, tw);
                bar();
                // second pass: block b of column (sb, c), rows b R2 + q, to the scratch
#pragma unroll
                for (int k = 0; k < SPB * C * R1 / TG; k++) {
                    const int e = t + TG * k, c = e % C, b = e / C % R1, sb = e / (C * R1);
                    if (sb < nb) {
                        const P2 *d = data + sb * SS + G::pad(b * R2 * C) + c;
                        P2 v[R2];
#pragma unroll
                        for (int q = 0; q < R2; q++) v[q] = d[q * C];
                        Dft<R2>::run(v);
                        P2 *z = Zc + (size_t)(s + sb) * zs + (size_t)(b * R2) * p.N1 + zcol(c);
                        if (!dbg_ok(s + sb < p.sc && column(c) < p.N1, kDbgScratch)) continue;
#pragma unroll
                        for (int q = 0; q < R2; q++) z[(size_t)q * p.N1] = cmul(v[q], twiddle(q));
                    }
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
