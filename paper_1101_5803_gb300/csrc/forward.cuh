// Banded forward batch (FP32 contexts, one ray per pixel): model = B L s and
// Eq. chi2 for many sources at one lens (Section 3.2's refinement fitness).
//
// One CTA of FWD_THREADS threads per source at a time (persistent over the
// sources).  The source vector is staged in shared memory; the image is
// processed in bands of whole tile rows (two buffers: one band is filled
// while the previous one is convolved), each band's zero-padded L s values
// (its rows plus the K-1 halo rows) gathered straight into shared memory
// from a pixel-ordered map of the rays' cells and weights (k_fwd_rays), so
// L s never goes to global memory.  Each thread owns one 4x4 tile of the
// band and convolves it with the PSF taps (staged in shared memory, read as
// warp-uniform broadcasts), in a loop over two or three tap rows held in
// registers (each input row is loaded once for them; the loop body stays small
// enough for the instruction cache, which the fully unrolled 21x21 tile is
// not).  chi^2: FP32 per tile, FP64 across tiles.  A population of 1024 sources
// at 256 x 256 and K = 21: 1.89 -> 1.61 ms against one load per tap.
#pragma once

#include "fast.cuh"

namespace mirage {

constexpr int FWD_THREADS = 512;
constexpr int MAX_FTAP = 31 * 31;

struct FwdArgs {
    const Prob<float>* probs;
    CandScratch<float> cs;
    const float4* pixmap;  // [npix] {cell base (int bits) or -1, u, v, 0} in pixel order
    const int* flags;      // [n_flags] of k_fwd_rays' CTAs: 1 = has active pixels, 2 = invalid lens
    int n_flags;
    const float* S;   // [n_src][ns]
    int n_src;
    float* model;     // nullable [n_src][npix]
    double* chi2;     // [n_src]
    int* status;      // nullable [1]
    int band_tiles;   // tile rows per band
};

// shared memory: taps, source vector, then two bands of (band rows + K - 1) x Wp
__host__ inline size_t fwd_band_smem(const Prob<float>& P, int band_tiles) {
    return 16 + 2 * 33 * sizeof(double) + align_up<float>(sizeof(float) * P.K * P.kp, 16) +
           align_up<float>(sizeof(float) * P.ns, 16) +
           2 * sizeof(float) * (size_t)(band_tiles * TILE + P.K - 1) * P.Wp;
}

// The lens's rays in pixel order (one ray per pixel), sqrt(W) and the padded
// data: what the banded kernel reads.  `chunk` pixels per CTA, small enough to
// spread the FP64 trace over the device.  (A call on one 64 x 64 source: 282 us
// with one CTA tracing and sorting the rays by cell, as the solves need them, and
// this map read back from that; 91 us with the sort spread out; 55 us without.)
template <int UNUSED = 0>
__global__ void __launch_bounds__(RT_THREADS) k_fwd_rays(const Prob<float>* __restrict__ probs,
                                                         const double* __restrict__ lens, CandScratch<float> cs,
                                                         float4* __restrict__ pixmap, int* __restrict__ flags, int chunk) {
    const Prob<float>& P = probs[0];
    const LensT<double> L = make_lens<double>(lens);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.plen; i += gridDim.x * blockDim.x) {  // the zero frame
        const int yp = i / P.Wp, y = yp - P.hk, x = i - yp * P.Wp - P.xoff;
        if (L.bad || x < 0 || x >= P.nx || y < 0 || y >= P.ny) {
            cs.swp[i] = 0.f;
            cs.dpad[i] = 0.f;
        }
    }
    int active = 0;
    if (!L.bad) {
        const int j1 = min((int)(blockIdx.x + 1) * chunk, P.npix);
        for (int j = blockIdx.x * chunk + threadIdx.x; j < j1; j += blockDim.x) {
            const int y = j / P.nx, x = j - y * P.nx;
            int base;
            double u, v;
            const bool any = rt_ray(P, L, x, y, 0, base, u, v);
            pixmap[j] = make_float4(__int_as_float(base), (float)u, (float)v, 0.f);
            const float w = (any && P.mask[j]) ? 1.f / P.sigma[j] : 0.f;
            const int pp = (y + P.hk) * P.Wp + x + P.xoff;
            cs.swp[pp] = w;
            cs.dpad[pp] = P.d[j];
            active |= w != 0.f;
        }
    }
    active = __syncthreads_or(active);
    if (threadIdx.x == 0) flags[blockIdx.x] = L.bad ? 2 : (active != 0);
}

// RT rows of a 4x4 output tile: out[r][c] = sum_{a,b} t[a][b] in[r + a][c + b +
// SHF], NR tap rows at a time held in registers (t: shared, rows of KP taps, loaded four
// at a time).  What it runs into is shared-memory bandwidth: per warp and pair
// of tap rows, five window rows of 16-byte loads (140 cycles at K = 21) beside
// 168 cycles of FMAs an SM sub-partition; one load per tap (42 more cycles) put
// it over.  Three rows at a time share more of the window where the registers
// allow it.  (8 x 4 outputs a thread need half the window loads, but 128
// registers a thread spill or leave half the warps idle: 15.8k against 12.4k
// clocks at 128 x 128 and K = 11 on two SMs.)  Each output adds its terms in the
// order a, b.
template <int K, int NR, int RT>
__device__ __forceinline__ void conv4_rows(unsigned src_a, int Wp, unsigned tap_a, float (&acc)[RT][TILE]) {
    constexpr int SHF = xoff_of<float>((K - 1) / 2) - (K - 1) / 2, KP = (K + 3) & ~3;
    constexpr int NVW = (TILE + K - 1 + SHF + 3) / 4 * 4;
    float t[NR][KP];
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
        for (int v = 0; v < KP; v += 4) lds_vec(tap_a + (unsigned)((i * KP + v) * sizeof(float)), t[i] + v);
#pragma unroll
    for (int rr = 0; rr < RT + NR - 1; ++rr) {
        float in[NVW];
#pragma unroll
        for (int v = 0; v < NVW; v += 4) lds_vec(src_a + (unsigned)((rr * Wp + v) * sizeof(float)), in + v);
#pragma unroll
        for (int b = 0; b < K; ++b)
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const int r = rr - i;
                if (r >= 0 && r < RT) {
#pragma unroll
                    for (int c = 0; c < TILE; ++c) acc[r][c] = fmaf(t[i][b], in[SHF + b + c], acc[r][c]);
                }
            }
    }
}
template <int K, int RT = TILE>
__device__ __forceinline__ void conv4(const float* Pb, int Wp, const float* taps, float (&acc)[RT][TILE]) {
    constexpr int KP = (K + 3) & ~3, NR = K <= 13 ? 3 : 2, REST = K % NR;
    const unsigned src = smem_addr(Pb), tap = smem_addr(taps);
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < TILE; ++c) acc[r][c] = 0.f;
#pragma unroll 1
    for (int a = 0; a + NR <= K; a += NR) conv4_rows<K, NR, RT>(src + 4u * a * Wp, Wp, tap + 4u * a * KP, acc);
    if constexpr (REST > 0) conv4_rows<K, REST, RT>(src + 4u * (K - REST) * Wp, Wp, tap + 4u * (K - REST) * KP, acc);
}

template <int K>
__global__ void __launch_bounds__(FWD_THREADS, 1) k_forward_band(const __grid_constant__ FwdArgs FA) {
    constexpr int KP = (K + 3) & ~3;
    extern __shared__ __align__(16) unsigned char smem[];
    const Prob<float>& P = FA.probs[0];
    const CandScratch<float>& cs = FA.cs;
    const Geo<float> g = geo_of(P, 0);  // (the ray count is not used)
    double* red = reinterpret_cast<double*>(smem + 16);
    float* taps = reinterpret_cast<float*>(smem + 16 + 2 * 33 * sizeof(double));
    float* s_sh = taps + K * KP;
    float* band = s_sh + align_up<float>(g.ns, 4);
    const int tid = threadIdx.x, bs = blockDim.x;
    // taps of B: the flipped PSF, rows padded to KP
    for (int i = tid; i < K * KP; i += bs) {
        const int a = i / KP, b = i - a * KP;
        taps[i] = b < K ? P.psf[(K - 1 - a) * K + (K - 1 - b)] : 0.f;
    }
    const int BT = FA.band_tiles, BR = BT * TILE;
    const int tiles_y = g.ntiles / g.tiles_x;
    const int n_bands = (tiles_y + BT - 1) / BT;
    const int rows = BR + K - 1;  // band rows in the buffer
    const bool bad = FA.flags[0] == 2;
    if (blockIdx.x == 0 && FA.status) {
        int some = 0;
        for (int i = tid; i < FA.n_flags; i += bs) some |= FA.flags[i];
        some = __syncthreads_or(some);
        if (tid == 0) FA.status[0] = bad ? ST_BADPARAM : some ? 0 : ST_EMPTY;
    }
    int which = 0;
    for (int k = blockIdx.x; k < FA.n_src; k += gridDim.x) {
        __syncthreads();
        if (bad) {
            if (tid == 0) FA.chi2[k] = __longlong_as_double(0x7ff0000000000000LL);
            continue;
        }
        // stage the source (16-byte vectors when the row allows it)
        const float* src = FA.S + (long long)k * g.ns;
        if ((g.ns & 3) == 0 && ((reinterpret_cast<uintptr_t>(src) & 15) == 0)) {
            for (int i = tid; i < g.ns / 4; i += bs)
                reinterpret_cast<float4*>(s_sh)[i] = reinterpret_cast<const float4*>(src)[i];
        } else {
            for (int i = tid; i < g.ns; i += bs) s_sh[i] = src[i];
        }
        // band fill: L s of padded rows [b BR, b BR + rows) into dst, four
        // columns per step (row and column advanced without division)
        auto fill = [&](int b, float* dst) {
            const int y0 = b * BR - g.hk;  // image row of band row 0
            const int W4 = g.Wp >> 2, dr = bs / W4, dc = bs - dr * W4;
            int r = tid / W4, c4 = tid - (tid / W4) * W4;
            for (; r < rows;) {
                const int y = y0 + r;
                float4 val = make_float4(0.f, 0.f, 0.f, 0.f);
                if (y >= 0 && y < g.ny) {
                    float v4[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int x = c4 * 4 + q - g.xoff;
                        v4[q] = 0.f;
                        if (x >= 0 && x < g.nx) {
                            const float4 m = FA.pixmap[y * g.nx + x];
                            const int base = __float_as_int(m.x);
                            if (base >= 0) {
                                const float* s0 = s_sh + base;
                                v4[q] = (1.f - m.z) * ((1.f - m.y) * s0[0] + m.y * s0[1]) +
                                        m.z * ((1.f - m.y) * s0[g.sx] + m.y * s0[g.sx + 1]);
                            }
                        }
                    }
                    val = make_float4(v4[0], v4[1], v4[2], v4[3]);
                }
                reinterpret_cast<float4*>(dst)[r * W4 + c4] = val;
                r += dr;
                c4 += dc;
                if (c4 >= W4) {
                    c4 -= W4;
                    ++r;
                }
            }
        };
        // two band buffers: while band b is convolved, band b + 1 is filled;
        // odd warps fill first, even warps convolve first, so the fill's
        // global loads wait while the other half of the warps keep the FMA
        // pipe busy
        const int bandsz = rows * g.Wp;
        const bool fill_first = ((tid >> 5) & 1) != 0;
        __syncthreads();  // s staged
        fill(0, band);
        double chi = 0.0;
        for (int b = 0; b < n_bands; ++b) {
            __syncthreads();  // band b filled; band b - 1's convolution done
            float* cur = band + (b & 1) * bandsz;
            float* nxt = band + ((b + 1) & 1) * bandsz;
            if (fill_first && b + 1 < n_bands) fill(b + 1, nxt);
            // one 4x4 output tile per thread; the chi^2 operands are loaded
            // before the convolution so that their latency overlaps it
            const int ty_l = tid / g.tiles_x, tx = tid - ty_l * g.tiles_x;
            const int ty = b * BT + ty_l;
            if (ty_l < BT && ty < tiles_y) {
                V4<float> sw[TILE], dv[TILE];
#pragma unroll
                for (int rr = 0; rr < TILE; ++rr) {
                    const int pp = (ty * TILE + rr + g.hk) * g.Wp + tx * TILE + g.xoff;
                    sw[rr] = ld4(cs.swp + pp);
                    dv[rr] = ld4(cs.dpad + pp);
                }
                float acc[TILE][TILE];
                conv4<K>(cur + (ty_l * TILE) * g.Wp + tx * TILE, g.Wp, taps, acc);
                float ct = 0.f;  // the tile's 16 terms in FP32, then one FP64 add
#pragma unroll
                for (int rr = 0; rr < TILE; ++rr) {
                    const int y = ty * TILE + rr;
#pragma unroll
                    for (int cc = 0; cc < TILE; ++cc) {
                        const float res = sw[rr].v[cc] * (dv[rr].v[cc] - acc[rr][cc]);
                        ct = fmaf(res, res, ct);
                        const int x = tx * TILE + cc;
                        if (FA.model && y < g.ny && x < g.nx)
                            FA.model[(long long)k * g.nx * g.ny + y * g.nx + x] = acc[rr][cc];
                    }
                }
                chi += (double)ct;
            }
            if (!fill_first && b + 1 < n_bands) fill(b + 1, nxt);
        }
        const double cval = block_sum(chi, red, which);
        which ^= 1;
        if (tid == 0) FA.chi2[k] = cval;
    }
}

}  // namespace mirage
