// vspec_colblk.cuh — kernel A for the longest pre-filtered transforms: dual-pol
// PFB of at most 8 taps with 512-point columns (2^20 channels).
//
// A register window of fp32 frames does not fit beside 512-point columns. The
// int8 frames stay in shared memory instead (a ring of the 11 that a batch of
// four spectra spans), and each thread forms its points' four outputs from one
// walk over the ring: a frame's sample is unpacked once and added into every
// output it is a tap of, 11 unpacks for 4 outputs where reading the taps
// spectrum by spectrum takes 32 (and 8 loads from L2). While the columns of a
// batch are transformed, the next four frames are copied over the four oldest.
//
// Tiles of C = 4 columns (2048 points, four per thread); the 512-point column
// is three radix-8 DIF passes (the plan's column pass list {8, 8, 8}), two
// butterflies per thread and pass, four barriers per 8192 outputs. A tile row
// is 16 input bytes: tile groups read a line's eight tiles together. The
// thread's coefficients (8 taps of 4 points) and its four-step twiddles stay
// in registers for the whole run of spectra.
//
// Shared memory element i of a spectrum lives at i ^ 4 when bit 5 of i is set:
// the last pass's 8-lane phases span two blocks 32 elements apart, which would
// otherwise share banks; the other passes are contiguous over a warp either
// way.
//
// Measured (GB300, 2^20 channels, 100 spectra, 8 taps): 0.78 ms against 1.77 ms
// for the gather kernel, the whole call 1.16 against 2.23 ms. It is bound, like
// the register-column kernel, by its phases' shared-memory and FMA time.
#pragma once
#include "vspec_kernels.cuh"

namespace vspec {

struct ColBlk {
    static constexpr int N2 = 512, C = 4, PTS = N2 * C, SPB = 4, PT = 8, RING = PT + SPB - 1, THREADS = 512;
    static constexpr int TW1 = 7 * 64, TW2 = 7 * 8;  // pass twiddles, [q - 1][j]
    // data [SPB][PTS] P2, frame ring [RING][PTS] u32, pass twiddles
    static constexpr size_t smem = (size_t)SPB * PTS * 16 + (size_t)RING * PTS * 4 + (TW1 + TW2) * 8;
    static_assert(smem <= 232448, "shared memory of one CTA");
};

__global__ void __launch_bounds__(ColBlk::THREADS, 1) fir_colblk_kernel(const __grid_constant__ ColParams p) {
    pdl_trigger();
    using G = ColBlk;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    P2 *data = reinterpret_cast<P2 *>(smem_raw);                         // [SPB][PTS]
    uint32_t *ring = reinterpret_cast<uint32_t *>(data + G::SPB * G::PTS);  // [RING][PTS]
    float2 *tw1 = reinterpret_cast<float2 *>(ring + G::RING * G::PTS);   // [7][64]
    float2 *tw2 = tw1 + G::TW1;                                          // [7][8]
    const int t = threadIdx.x, e = t & 255, c = t & 3;
    const int D = G::PT - p.P;  // leading zero taps
    for (int i = t; i < G::TW1; i += G::THREADS) tw1[i] = __ldg(p.twA + p.pass[0].off + (i % 64) * 7 + i / 64);
    for (int i = t; i < G::TW2; i += G::THREADS) tw2[i] = __ldg(p.twA + p.pass[1].off + (i % 8) * 7 + i / 8);

    const TileSplit sp = tile_split(p.tiles, p.sc, p.G);
    for (long long f = sp.lo; f < sp.hi;) {
        const long long base = f / p.sc * p.sc;  // first item of this super-tile
        const int x = (int)(f / p.sc) * sp.G + sp.r;
        const int s_beg = (int)(f - base);
        const int s_end = (int)(min(sp.hi, base + p.sc) - base);
        f = base + s_end;
        const int n1 = x * G::C + c;
        // point k of this thread: tile element t + 512 k, row n2 = t / 4 + 128 k
        float cf[4][G::PT];
#pragma unroll
        for (int k = 0; k < 4; k++)
#pragma unroll
            for (int h = 0; h < G::PT; h++)
                cf[k][h] = h >= D ? __ldg(p.coef + (size_t)(h - D) * p.N + n1 + (size_t)p.N1 * (t / 4 + 128 * k)) : 0.f;
        // last pass: block b = e / 4, outputs at rows 8 b + q
        float2 twz[8];
#pragma unroll
        for (int q = 0; q < 8; q++) twz[q] = __ldg(p.twZ + (size_t)(8 * (e >> 2) + q) * p.N1 + n1);

        // Ring slot (fr - first) mod RING holds absolute frame fr, first the
        // oldest frame of the run's first spectrum (D leading taps have zero
        // coefficients; frames before the input are clamped).
        const long long first = p.s0 + s_beg - D;
        auto stage = [&](int rel, int cnt, int slot) {  // frames first + rel .. + cnt - 1 from ring slot `slot`
            for (int i = t; i < cnt * (G::PTS / 4); i += G::THREADS) {
                const int u = i / (G::PTS / 4), n2 = i % (G::PTS / 4);
                long long fr = first + rel + u;
                if (fr < 0) fr = 0;
                int sl = slot + u;
                if (sl >= G::RING) sl -= G::RING;
                const uint32_t *src = reinterpret_cast<const uint32_t *>(p.in) + fr * p.N + x * G::C + (long long)p.N1 * n2;
                if (dbg_ok(fr < p.nframes, kDbgInput))
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                 :: "r"((uint32_t)__cvta_generic_to_shared(ring + sl * G::PTS + 4 * n2)), "l"(src) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // frames a batch of cnt spectra spans: PT - 1 + cnt
        stage(0, G::PT - 1 + min(G::SPB, s_end - s_beg), 0);
        int r0 = 0;  // ring slot of the batch's oldest frame
        for (int s = s_beg; s < s_end; s += G::SPB) {
            const int nb = min(G::SPB, s_end - s);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();  // the batch's frames are visible; data is free
#pragma unroll
            for (int k = 0; k < 4; k++) {
                float2 c2[G::PT];
#pragma unroll
                for (int h = 0; h < G::PT; h++) c2[h] = dup2(cf[k][h]);
                P2 y[G::SPB];
#pragma unroll
                for (int u = 0; u < G::SPB; u++) y[u] = P2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int h = 0; h < G::RING; h++) {
                    // (a short last batch reads slots of the previous frames past its own; their outputs are not stored)
                    const int sl = r0 + h >= G::RING ? r0 + h - G::RING : r0 + h;
                    const P2 v = unpack_p2(ring[sl * G::PTS + t + 512 * k] ^ 0x80808080u);
#pragma unroll
                    for (int u = 0; u < G::SPB; u++) {
                        if (h - u >= 0 && h - u < G::PT) {
                            y[u].re = __ffma2_rn(c2[h - u], v.re, y[u].re);
                            y[u].im = __ffma2_rn(c2[h - u], v.im, y[u].im);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < G::SPB; u++)
                    if (u < nb) data[u * G::PTS + ((t + 512 * k) ^ ((t >> 3) & 4))] = y[u];
            }
            __syncthreads();  // the batch's outputs are in data; the ring's four oldest frames are free
            if (s + G::SPB < s_end) stage(s - s_beg + G::RING, min(G::SPB, s_end - s - G::SPB), r0);
            r0 += G::SPB;
            if (r0 >= G::RING) r0 -= G::RING;
            // pass 1: block length 512, butterfly j = e / 4 over rows j + 64 q
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int sb = (t >> 8) + 2 * h;
                if (sb < nb) {
                    P2 *d = data + sb * G::PTS + (e ^ ((e >> 3) & 4));
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[256 * q];
                    Dft<8>::run(v);
                    d[0] = v[0];
#pragma unroll
                    for (int q = 1; q < 8; q++) d[256 * q] = cmul(v[q], tw1[64 * (q - 1) + (e >> 2)]);
                }
            }
            __syncthreads();
            // pass 2: block length 64, block e / 32, butterfly j = (e / 4) mod 8 over rows j + 8 q
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int sb = (t >> 8) + 2 * h;
                if (sb < nb) {
                    P2 *d = data + sb * G::PTS + (e >> 5) * 256;
                    const int l = e & 31;
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[32 * q + (l ^ (4 * (q & 1)))];
                    Dft<8>::run(v);
                    d[l] = v[0];
#pragma unroll
                    for (int q = 1; q < 8; q++) d[32 * q + (l ^ (4 * (q & 1)))] = cmul(v[q], tw2[8 * (q - 1) + (l >> 2)]);
                }
            }
            __syncthreads();
            // pass 3: block length 8, block b = e / 4, rows 8 b + q, to the scratch
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int sb = (t >> 8) + 2 * h;
                if (sb < nb) {
                    const int b = e >> 2;
                    const P2 *d = data + sb * G::PTS + 32 * b + c;
                    P2 v[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) v[q] = d[4 * (q ^ (b & 1))];
                    Dft<8>::run(v);
                    P2 *z = reinterpret_cast<P2 *>(p.Z) + (size_t)(s + sb) * p.N + (size_t)(8 * b) * p.N1 + n1;
                    if (!dbg_ok(s + sb < p.sc && n1 < p.N1, kDbgScratch)) continue;
#pragma unroll
                    for (int q = 0; q < 8; q++) z[(size_t)q * p.N1] = cmul(v[q], twz[q]);
                }
            }
        }
        __syncthreads();  // the last batch's frames are read before the next run's copies
    }
}

}  // namespace vspec
