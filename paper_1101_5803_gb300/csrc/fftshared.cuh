// FFT convolution of one image with the half spectrum in shared memory
// (single precision, M = 64 and 128; CTAs of 256 threads).
#pragma once

#include "fftconv.cuh"

namespace mirage {

// ---------------------------------------------------------------------------
// The same convolution in single precision for M = 64 and 128, with the half
// spectrum in shared memory and the transforms in registers.
//
// What bounds the batch form above at these sizes is not arithmetic (the 388
// transforms of B and B^T at M = 128 are 1.7 MFLOP, 14k clocks of one SM) but
// its passes: seven barriers of a few butterflies a thread for each of 12
// batches, and the spectra through L2.  Here a thread holds 16 points: a
// transform is two radix-4 passes, one exchange among its M / 16 threads (of
// one warp: no block barrier), and the other two passes, so that a convolution
// has two block barriers.  Every butterfly is that of fft_batch on the same
// operands, so the results are the same bits.  (64 x 64 image, 65 x 65 PSF, 16
// candidates x 8 lambdas: 327 -> 135 ms)
// ---------------------------------------------------------------------------
// a b with the first or the second product of the imaginary part inside the
// fused step.  Which of the two the compiler's contraction picks for cmul in
// fft_batch differs between its forward and inverse passes (found by comparing
// results); written out here, so that every transform gives the same bits.
__device__ __forceinline__ float2 fft_cmul_a(float2 a, float2 b) {
    return cx<float2>(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}
__device__ __forceinline__ float2 fft_cmul_b(float2 a, float2 b) {
    return cx<float2>(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ void fft_radix4(float2 a, float2 x1, float2 x2, float2 x3, float2 w1, bool inverse, float2& y0,
                                           float2& y1, float2& y2, float2& y3) {
    if (inverse) w1.y = -w1.y;
    const float2 w2 = fft_cmul_a(w1, w1), w3 = inverse ? fft_cmul_a(w2, w1) : fft_cmul_b(w2, w1);
    const float2 b = inverse ? fft_cmul_b(w1, x1) : fft_cmul_a(w1, x1), c = fft_cmul_a(w2, x2), d = fft_cmul_a(w3, x3);
    const float2 s0 = cx<float2>(a.x + c.x, a.y + c.y), s1 = cx<float2>(a.x - c.x, a.y - c.y);
    const float2 s2 = cx<float2>(b.x + d.x, b.y + d.y), s3 = cx<float2>(b.x - d.x, b.y - d.y);
    const float2 is3 = inverse ? cx<float2>(-s3.y, s3.x) : cx<float2>(s3.y, -s3.x);
    y0 = cx<float2>(s0.x + s2.x, s0.y + s2.y);
    y1 = cx<float2>(s1.x + is3.x, s1.y + is3.y);
    y2 = cx<float2>(s0.x - s2.x, s0.y - s2.y);
    y3 = cx<float2>(s1.x - is3.x, s1.y - is3.y);
}

// place of point i in a transform's exchange buffer (a gap after every 16
// points against bank conflicts)
__device__ __forceinline__ int fft_xi(int i) { return i + (i >> 4); }

// Transform of the points x[m] = data[t + TH m] (t = this thread of the
// transform's TH = M / 16) into x[m] = result[fft_out(t, m)].
template <int M>
__device__ __forceinline__ int fft_out(int t, int m) {
    if (M == 64) return t + 4 * (m >> 2) + 16 * (m & 3);
    return t + 8 * (m >> 3) + 16 * (m & 7);  // m & 7 = p + 4 (upper half)
}
template <int M>
__device__ __forceinline__ void fft_points(float2 (&x)[16], float2* buf, const float2* tw, int t, bool inverse) {
    float2 y[16];
#pragma unroll
    for (int i = 0; i < 4; ++i)  // span 1
        fft_radix4(x[i], x[i + 4], x[i + 8], x[i + 12], tw[1], inverse, y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
#pragma unroll
    for (int p = 0; p < 4; ++p)  // span 4: points 16 t + p + 4 q
        fft_radix4(y[p], y[4 + p], y[8 + p], y[12 + p], tw[7 + p], inverse, x[p], x[p + 4], x[p + 8], x[p + 12]);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) buf[fft_xi(16 * t + r)] = x[r];
    __syncwarp();
    if constexpr (M == 64) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {  // span 16
            const int j = t + 4 * h;
            fft_radix4(buf[fft_xi(j)], buf[fft_xi(j + 16)], buf[fft_xi(j + 32)], buf[fft_xi(j + 48)], tw[31 + j], inverse,
                       x[4 * h], x[4 * h + 1], x[4 * h + 2], x[4 * h + 3]);
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = t + 8 * h;
            float2 lo[4], hi[4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {  // span 16, points j + 16 u + 32 q
                float2(&o)[4] = u ? hi : lo;
                fft_radix4(buf[fft_xi(j + 16 * u)], buf[fft_xi(j + 16 * u + 32)], buf[fft_xi(j + 16 * u + 64)],
                           buf[fft_xi(j + 16 * u + 96)], tw[31 + j], inverse, o[0], o[1], o[2], o[3]);
            }
#pragma unroll
            for (int p = 0; p < 4; ++p) {  // span 64, radix 2
                float2 w = tw[63 + j + 16 * p];
                if (inverse) w.y = -w.y;
                const float2 a = lo[p], b = inverse ? fft_cmul_b(w, hi[p]) : fft_cmul_a(w, hi[p]);
                x[8 * h + p] = cx<float2>(a.x + b.x, a.y + b.y);
                x[8 * h + p + 4] = cx<float2>(a.x - b.x, a.y - b.y);
            }
        }
    }
}

// out = B x or B^T x: load(y, n) and store(y, n, v) as for fft_convolve
template <int M, class Load, class Store>
__device__ void fft_convolve_shared(const FftPlan<float>& f, Load load, int rows_in, Store store, int rows_out, int cols_out,
                                    bool corr) {
    constexpr int TH = M / 16, LD = M + 1, H1 = M / 2 + 1, half = M / 2;
    float2* F = f.b0;                                     // [H1][LD]
    const int grp = threadIdx.x / TH, t = threadIdx.x % TH, ng = blockDim.x / TH;
    float2* buf = F + H1 * LD + grp * (M + M / 16);
    const float2* tw = f.tw;
    const float2* S = f.S;
    float2 x[16];
    // rows, two at a time.  (All threads of a warp take every step of a loop:
    // the exchange synchronises the warp.)
    const int pairs_in = (rows_in + 1) >> 1, pairs_out = (rows_out + 1) >> 1;
    for (int p0 = 0; p0 < pairs_in; p0 += ng) {
        const int y = 2 * (p0 + grp);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int n = t + TH * m;
            x[m].x = y < rows_in ? load(y, n) : 0.f;
            x[m].y = y + 1 < rows_in ? load(y + 1, n) : 0.f;
        }
        fft_points<M>(x, buf, tw, t, false);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 16; ++m) buf[fft_xi(fft_out<M>(t, m))] = x[m];
        __syncwarp();
        if (y < rows_in)
            for (int k = t; k < H1; k += TH) {
                const float2 z = buf[fft_xi(k)], zm = buf[fft_xi((M - k) & (M - 1))];
                F[k * LD + y] = cx<float2>(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
                if (y + 1 < rows_in) F[k * LD + y + 1] = cx<float2>(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
            }
    }
    __syncthreads();
    // columns: transform, times S (or its conjugate), transform back
    for (int k0 = 0; k0 < H1; k0 += ng) {
        const int k = k0 + grp;
        const bool own = k < H1;
        float2 s[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) s[m] = own ? S[k * M + fft_out<M>(t, m)] : cx<float2>(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int n = t + TH * m;
            x[m] = own && n < rows_in ? F[k * LD + n] : cx<float2>(0.f, 0.f);
        }
        fft_points<M>(x, buf, tw, t, false);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            if (corr) s[m].y = -s[m].y;
            buf[fft_xi(fft_out<M>(t, m))] = fft_cmul_b(x[m], s[m]);
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 16; ++m) x[m] = buf[fft_xi(t + TH * m)];
        fft_points<M>(x, buf, tw, t, true);
        if (own)
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                const int n = fft_out<M>(t, m);
                if (n < rows_out) F[k * LD + n] = x[m];
            }
    }
    __syncthreads();
    // rows back
    for (int p0 = 0; p0 < pairs_out; p0 += ng) {
        const int y = 2 * (p0 + grp);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int k = t + TH * m, kk = k <= half ? k : M - k;
            float2 g1 = y < rows_out ? F[kk * LD + y] : cx<float2>(0.f, 0.f);
            float2 g2 = y + 1 < rows_out ? F[kk * LD + y + 1] : cx<float2>(0.f, 0.f);
            if (k > half) {
                g1.y = -g1.y;
                g2.y = -g2.y;
            }
            x[m] = cx<float2>(g1.x - g2.y, g1.y + g2.x);
        }
        fft_points<M>(x, buf, tw, t, true);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int n = fft_out<M>(t, m);
            if (n < cols_out && y < rows_out) {
                store(y, n, x[m].x);
                if (y + 1 < rows_out) store(y + 1, n, x[m].y);
            }
        }
    }
    __syncthreads();
}

// fft_rows_inverse hands thread tid its outputs in a fixed order; visit(y, n)
// in that order, for sums that have to be added in it
template <class Visit>
__device__ void fft_store_order(int M, Visit visit, int rows_out, int cols_out) {
    const int nb = fft_batch_count<float2>(M);
    for (int y0 = 0; y0 < rows_out; y0 += 2 * nb) {
        const int np = min(nb, (rows_out - y0 + 1) >> 1);
        for (int t = threadIdx.x; t < np * cols_out; t += blockDim.x) {
            const int p = t / cols_out, n = t - p * cols_out, y = y0 + 2 * p;
            visit(y, n);
            if (y + 1 < rows_out) visit(y + 1, n);
        }
    }
}

}  // namespace mirage
