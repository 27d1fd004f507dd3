// Surrogate network: a multilayer perceptron with SiLU hidden layers and a
// linear output layer, trained with mean-squared error and Adam.  Matrix
// products run on the BF16 tcgen05 tensor cores (FP32 accumulate in tensor
// memory);
// master weights, Adam moments, bias, activation and loss stay in FP32.
//
// It predicts, from the encoded lens vector, the standardised
// (log chi2, log10 lambda) of the L-curve corner, so that a genetic
// algorithm can screen its offspring and warm-start the exact solves.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mirage.h"
#include "tc05.cuh"

namespace {

thread_local std::string g_mlp_err;

int mlp_fail(int code, const std::string& msg) {
    g_mlp_err = msg;
    return code;
}

#define MCK(call)                                                                        \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess) return mlp_fail(MIRAGE_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// A layer's products on the fifth-generation tensor cores,
//   C[M x N] = sum_k A(m, k) B(k, n),
//   A(m, k) = A[m * sam + k * sak],  B(k, n) = B[k * sbk + n * sbn]  (BF16),
// with what follows them (bias, activation, loss gradient) applied to the
// accumulator before it leaves the CTA.
//
// What bounds the network is latency: a training step of the 7-256-256-256-2
// network on 256 rows is 0.2 GFLOP, and 27 launches of products, activations
// and sums took 194 us of it.  So a layer is one launch (its dW, db and dA
// together, which are independent), and a product one pass: a CTA of eight
// warps per 128 x BN tile loads up to TC_BK = 256 of K at once (every load in
// flight together), stages it as K-major core matrices (8 rows x 8 BF16),
// issues all its tcgen05.mma (K = 16 each, in order of k, so that an element
// is the same sum whatever the chunk) from one thread and waits once.  The
// core matrices lie TC_LBO bytes apart along K and TC_SBO along M and N, padded
// so that neither the row-wise stores nor the transposed ones (8 x 8 blocks
// turned in registers) meet in a bank.  Edges are zero-filled.  Should a
// completion wait run out (about a second), the tile is written as NaN.
constexpr int TC_BM = 128, TC_BK = 256, TC_T = 256;
constexpr int TC_LBO = 144, TC_SBO = TC_BK / 8 * TC_LBO + 16;

template <int BN>
constexpr int tc_smem_bytes() {
    return (TC_BM + BN) / 8 * TC_SBO + 16;
}
// byte offset of core-matrix row r (16 bytes: k-octet o)
__device__ __forceinline__ int tc_row(int r, int o) { return (r >> 3) * TC_SBO + o * TC_LBO + (r & 7) * 16; }

enum : int { EPI_PLAIN = 0, EPI_HIDDEN = 1, EPI_OUT = 2, EPI_BACK = 3 };

struct Gemm {
    const __nv_bfloat16* A = nullptr;
    long sam = 0, sak = 0;
    const float* Af = nullptr;  // FP32 rows of K in place of A
    const __nv_bfloat16* B = nullptr;
    long sbk = 0, sbn = 0;
    int M = 0, N = 0, K = 0, epi = EPI_PLAIN;
    float* C = nullptr;  // EPI_PLAIN: the product [M x N]
    // EPI_HIDDEN: z = product + bias into Z (nullable), silu(z) into H.
    // EPI_OUT: product + bias into Y; with T, 2 (y - T) / (M N) into D and H
    // (row r of the batch is row tidx[r] of T, or r).
    // EPI_BACK: product times silu'(Z) into D and H
    const float* bias = nullptr;
    float* Z = nullptr;
    __nv_bfloat16* H = nullptr;
    float* Y = nullptr;
    const float* T = nullptr;
    const int* tidx = nullptr;
    float* D = nullptr;
    int tm = 0, tiles = 0;  // tiles along M, in all
};
struct LayerArgs {
    Gemm g[2];
    // column sums of S [srows x scols] into sum (fixed order), 32 columns a CTA
    const float* S = nullptr;
    int srows = 0, scols = 0;
    float* sum = nullptr;
    long long* inc = nullptr;  // incremented by one
};

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_g(float z) {
    const float s = 1.f / (1.f + __expf(-z));
    return s * (1.f + z * (1.f - s));
}

// Launches of a chain are programmatic dependents of each other: a kernel lets
// the next one start (its CTAs become resident, allocate and wait) as soon as
// all its own run, and waits itself for the previous one's results before it
// reads or writes anything that they share
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// 8 x 8 transpose of BF16: v[i] holds row i (8 values); row j of the result
__device__ __forceinline__ uint4 tc_column(const uint4 (&v)[8], int j) {
    const unsigned sel = (j & 1) ? 0x7632u : 0x5410u;
    auto word = [&](const uint4& a) { return (j >> 1) == 0 ? a.x : (j >> 1) == 1 ? a.y : (j >> 1) == 2 ? a.z : a.w; };
    return make_uint4(__byte_perm(word(v[0]), word(v[1]), sel), __byte_perm(word(v[2]), word(v[3]), sel),
                      __byte_perm(word(v[4]), word(v[5]), sel), __byte_perm(word(v[6]), word(v[7]), sel));
}

// ROWS rows x kn (a multiple of 16, at most TC_BK) of an operand view into the
// core matrices at dst; zeros beyond K (rows beyond R only reach outputs that
// are not stored, and are left as they are)
template <int ROWS>
__device__ __forceinline__ void tc_stage(unsigned char* dst, const __nv_bfloat16* __restrict__ src, long s_row, long s_k,
                                         const float* __restrict__ srcf, int r0, int R, int k0, int K, int kn) {
    const bool al = ((uintptr_t)src & 15) == 0;
    const int tid = threadIdx.x, ko = kn >> 3;
    if (!srcf && s_k == 1 && (s_row & 7) == 0 && al && k0 + kn <= K) {
        // rows contiguous along k: copied straight to shared memory, eight lanes
        // taking 128 consecutive bytes of a row
        const int rows = min(ROWS, R - r0);
        const __nv_bfloat16* s0 = src + (long)r0 * s_row + k0;
#pragma unroll
        for (int i = 0; i < ROWS * (TC_BK / 8) / TC_T; ++i) {
            const int e = tid + TC_T * i, o = e % (TC_BK / 8), r = e / (TC_BK / 8);
            if (o < ko && r < rows)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(mirage::tc05::saddr(dst + tc_row(r, o))),
                             "l"(s0 + (long)r * s_row + 8 * o)
                             : "memory");
        }
        return;
    }
    if (!srcf && s_row == 1 && (s_k & 7) == 0 && al && (r0 + ROWS <= R || ((R - r0) & 7) == 0) && k0 + kn <= K) {
        // rows contiguous at one k: 8 x 8 blocks, turned in registers
        constexpr int MB = ROWS / 8, MQ = MB < 8 ? MB : 8;  // 8 row blocks x 4 k-octets a warp
#pragma unroll 1
        for (int e = tid; e < MB * ((ko + 3) & ~3); e += TC_T) {
            const int q = e / (4 * MQ), mb = e % MQ + MQ * (q % (MB / MQ)), kb = e / MQ % 4 + 4 * (q / (MB / MQ));
            if (kb >= ko || r0 + 8 * mb >= R) continue;
            uint4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = *reinterpret_cast<const uint4*>(src + (long)(k0 + 8 * kb + i) * s_k + r0 + 8 * mb);
#pragma unroll
            for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(dst + tc_row(8 * mb + j, kb)) = tc_column(v, j);
        }
        return;
    }
    // any other view, element by element
    const __nv_bfloat16 z = __float2bfloat16(0.f);
    const int rows = min(ROWS, R - r0);
    for (int e = tid; e < rows * kn; e += TC_T) {
        const int r = e / kn, k = e - r * kn, gr = r0 + r, gk = k0 + k;
        __nv_bfloat16 x = z;
        if (gk < K)
            x = srcf ? __float2bfloat16(srcf[(long)gr * K + gk]) : src[(long)gr * s_row + (long)gk * s_k];
        *reinterpret_cast<__nv_bfloat16*>(dst + tc_row(r, k >> 3) + (k & 7) * 2) = x;
    }
}

template <int BN>
__device__ void tc_tile(const Gemm& q, int tile, unsigned char* sm) {
    using namespace mirage::tc05;
    constexpr int TCOLS = BN < 32 ? 32 : BN;  // a power of two >= 32
    constexpr uint32_t ID = idesc(FMT_BF16, TC_BM, BN);
    unsigned char* sA = sm;
    unsigned char* sB = sA + TC_BM / 8 * TC_SBO;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sB + BN / 8 * TC_SBO);
    uint32_t* slot = reinterpret_cast<uint32_t*>(bar + 1);
    const int m0 = (tile % q.tm) * TC_BM, n0 = (tile / q.tm) * BN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    static_assert(TC_BM * (BN + 1) * 4 <= TC_BM / 8 * TC_SBO, "the accumulator tile fits where A was staged");
    if (warp == 0) tmem_alloc(slot, TCOLS);
    if (threadIdx.x == 32) bar_init(bar, 1);
    dep_wait();
    bool ok = true;
    uint32_t phase = 0, tmem = 0;
    for (int k0 = 0; k0 < q.K && ok; k0 += TC_BK) {
        const int kn = min(TC_BK, (q.K - k0 + 15) & ~15);
        tc_stage<TC_BM>(sA, q.A, q.sam, q.sak, q.Af, m0, q.M, k0, q.K, kn);
        tc_stage<BN>(sB, q.B, q.sbn, q.sbk, nullptr, n0, q.N, k0, q.K, kn);
        asm volatile("cp.async.wait_all;" ::: "memory");
        fence_async_smem();
        fence_before_sync();
        __syncthreads();
        fence_after_sync();
        tmem = *slot;
        if (threadIdx.x == 0) {
            for (int s = 0; s < kn / 16; ++s) {
                const uint64_t da = sdesc(saddr(sA) + s * 2 * TC_LBO, TC_LBO, TC_SBO);
                const uint64_t db = sdesc(saddr(sB) + s * 2 * TC_LBO, TC_LBO, TC_SBO);
                mma_bf16(tmem, da, db, ID, (k0 > 0 || s > 0) ? 1u : 0u);
            }
            commit(bar);
        }
        ok = __syncthreads_and(bar_wait(bar, phase)) != 0;  // one decision for the whole CTA
        phase ^= 1;
        fence_after_sync();
    }
    if (!ok) bar_wait(bar, phase ^ 1);  // (bounded) for the MMAs still in flight
    // accumulator to shared memory (warps w and w + 4 share tensor-memory lanes
    // 32 (w mod 4) .. and take the columns in turns of 16), then the epilogue
    // along rows: a thread's global accesses are its neighbours'
    constexpr int LD = BN + 1;
    float* tile_sm = reinterpret_cast<float*>(sm);
    __syncthreads();  // (the products have read the operands)
#pragma unroll 1
    for (int c0 = 16 * (warp >> 2); c0 < BN; c0 += 32) {
        float v[16];
        ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) tile_sm[((warp & 3) * 32 + lane) * LD + c0 + j] = v[j];
    }
    __syncthreads();
    const float nan = __int_as_float(0x7fc00000);
    const int rows = min(TC_BM, q.M - m0), cl = threadIdx.x % BN, rl = threadIdx.x / BN, col = n0 + cl;
    if (col < q.N) {
        const long i0 = (long)(m0 + rl) * q.N + col, step = (long)(TC_T / BN) * q.N;
        const float* ts = tile_sm + rl * LD + cl;
        // f(i, product) of this thread's elements, eight at a time
        auto each = [&](auto&& f) {
            constexpr int NR = TC_BM * BN / TC_T, U = NR < 8 ? NR : 8;
#pragma unroll 1
            for (int j0 = 0; j0 < NR; j0 += U)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = j0 + u;
                    if (rl + j * (TC_T / BN) < rows) f(i0 + j * step, ok ? ts[j * (TC_T / BN) * LD] : nan, m0 + rl + j * (TC_T / BN));
                }
        };
        const float bias = q.bias ? q.bias[col] : 0.f;
        if (q.epi == EPI_PLAIN) {
            float* C = q.C;
            each([&](long i, float p, int) { C[i] = p; });
        } else if (q.epi == EPI_HIDDEN) {
            float* Z = q.Z;
            __nv_bfloat16* H = q.H;
            each([&](long i, float p, int) {
                const float z = p + bias;
                if (Z) Z[i] = z;
                H[i] = __float2bfloat16(silu_f(z));
            });
        } else if (q.epi == EPI_OUT) {
            each([&](long i, float p, int r) {
                const float y = p + bias;
                q.Y[i] = y;
                if (q.T) {
                    const float d = y - q.T[(long)(q.tidx ? q.tidx[r] : r) * q.N + col];
                    const float g = 2.f * d / (float)((long)q.M * q.N);
                    q.D[i] = g;
                    q.H[i] = __float2bfloat16(g);
                }
            });
        } else {
            const float* __restrict__ Z = q.Z;
            float* __restrict__ D = q.D;
            __nv_bfloat16* __restrict__ H = q.H;
            each([&](long i, float p, int) {
                const float d = p * silu_g(Z[i]);
                D[i] = d;
                H[i] = __float2bfloat16(d);
            });
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        fence_after_sync();
        tmem_free(tmem, TCOLS);
    }
}

// sum[j] = sum_m S[m][j] for 32 columns, added in the order of m: the rows
// arrive in shared memory 256 at a time, one thread adds each column
__device__ void col_sums(const float* __restrict__ S, int rows, int cols, int j0, float* __restrict__ sum, float* sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    dep_wait();
    float s = 0.f;
    for (int m0 = 0; m0 < rows; m0 += 256) {
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int m = m0 + warp * 32 + i;
            v[i] = m < rows && j0 + lane < cols ? S[(long)m * cols + j0 + lane] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) sm[(warp * 32 + i) * 32 + lane] = v[i];
        __syncthreads();
        if (warp == 0) {
            const int n = min(256, rows - m0);
#pragma unroll 16
            for (int i = 0; i < n; ++i) s += sm[i * 32 + lane];
        }
        __syncthreads();
    }
    if (warp == 0 && j0 + lane < cols) sum[j0 + lane] = s;
}

template <int BN>
__global__ void __launch_bounds__(TC_T) k_layer(const __grid_constant__ LayerArgs a) {
    extern __shared__ __align__(128) unsigned char tc_sm[];
    dep_launch();
    int b = blockIdx.x;
    if (b == 0 && threadIdx.x == 0 && a.inc) {
        dep_wait();
        *a.inc += 1;
    }
    if (b < a.g[0].tiles) {
        tc_tile<BN>(a.g[0], b, tc_sm);
        return;
    }
    b -= a.g[0].tiles;
    if (b < a.g[1].tiles) {
        tc_tile<BN>(a.g[1], b, tc_sm);
        return;
    }
    col_sums(a.S, a.srows, a.scols, 32 * (b - a.g[1].tiles), a.sum, reinterpret_cast<float*>(tc_sm));
}

// x (FP32) -> BF16 activations
__global__ void k_to_bf16(const float* __restrict__ x, __nv_bfloat16* __restrict__ a, long n) {
    dep_launch();
    dep_wait();
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i < n) a[i] = __float2bfloat16(x[i]);
}

// dY = 2 (Y - T) / (n cols); loss partial sums.  With idx, row j of the
// batch targets row idx[j] of T.
__global__ void k_loss_grad(const float* __restrict__ Y, const float* __restrict__ T, const int* __restrict__ idx,
                            int cols, long total, float* __restrict__ dZ, __nv_bfloat16* __restrict__ dZh,
                            double* __restrict__ loss) {
    dep_launch();
    dep_wait();
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    double l = 0.0;
    if (i < total) {
        const long ti = idx ? (long)idx[i / cols] * cols + i % cols : i;
        const float d = Y[i] - T[ti];
        dZ[i] = 2.f * d / (float)total;
        dZh[i] = __float2bfloat16(dZ[i]);
        l = (double)d * (double)d;
    }
    if (loss) {
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(loss, l / (double)total);
    }
}

// Adam on every parameter; refresh the BF16 copy of the weights
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long n, float lr, float b1, float b2, float eps, float c1, float c2,
                       __nv_bfloat16* __restrict__ ph, const unsigned char* __restrict__ is_w) {
    dep_launch();
    dep_wait();
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    if (is_w[i]) ph[i] = __float2bfloat16(w);
}

// Minibatch rows of one training step: row slot j draws row
// h(seed, step, j) mod n with h the splitmix64 finaliser (a counter-based
// hash: the draw depends only on its three inputs)
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
struct Draw {
    int* idx;                // the rows' numbers ...
    __nv_bfloat16* a;        // ... and the rows (BF16)
    const float* x;
    int batch, n, cols;
    unsigned long long seed;
};
__device__ __forceinline__ void draw_rows(const Draw& d, long long step, long i) {
    if (i >= (long)d.batch * d.cols) return;
    const int j = (int)(i / d.cols), c = (int)(i - (long)j * d.cols);
    const unsigned long long key = d.seed * 0x9E3779B97F4A7C15ull + ((unsigned long long)step << 24) + (unsigned long long)j;
    const int row = (int)(mix64(key) % (unsigned long long)d.n);
    if (c == 0) d.idx[j] = row;
    d.a[i] = __float2bfloat16(d.x[(long)row * d.cols + c]);
}
// the rows of the first step of a training call
__global__ void k_draw(Draw d, const long long* __restrict__ dstep) {
    draw_rows(d, *dstep, blockIdx.x * (long)blockDim.x + threadIdx.x);
}

// The end of a step of the device-side training loop: Adam with the bias
// corrections of the device step counter (this step included), and, on the
// CTAs after the parameters' `nb`, the next step's rows
__global__ void k_adam_dev(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, long n, float lr, float b1, float b2, float eps,
                           const long long* __restrict__ dstep, __nv_bfloat16* __restrict__ ph,
                           const unsigned char* __restrict__ is_w, unsigned nb, Draw d) {
    dep_launch();
    dep_wait();
    if (blockIdx.x >= nb) {
        draw_rows(d, *dstep, (blockIdx.x - nb) * (long)blockDim.x + threadIdx.x);
        return;
    }
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float s = (float)*dstep;
    const float c1 = 1.f - powf(b1, s), c2 = 1.f - powf(b2, s);
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    if (is_w[i]) ph[i] = __float2bfloat16(w);
}

__global__ void k_params_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ ph, long n) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i < n) ph[i] = __float2bfloat16(p[i]);
}

struct Buf {
    void* p = nullptr;
    size_t n = 0;
    int ensure(size_t bytes) {
        if (bytes <= n) return MIRAGE_OK;
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            p = nullptr;
            cudaGetLastError();  // (reported here, not by a later launch's check)
            return mlp_fail(MIRAGE_ERR_NOMEM, "mlp: cudaMalloc failed");
        }
        n = bytes;
        return MIRAGE_OK;
    }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
};

inline unsigned blocks(long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

struct mirage_mlp {
    int device = 0;
    int L = 0;                 // weight layers
    std::vector<int> dims;     // L + 1
    std::vector<long> w_off, b_off;
    long n_params = 0;
    int step = 0;
    float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    Buf P, PH, M, V, G, ISW;   // params FP32, BF16 copy, Adam m, v, grads, weight mask
    Buf Z, A, DZ, DZH, LOSS;   // per-batch work (grown on demand; DZ and DZH twice: a layer's and the next one's)
    Buf IDX, DSTEP, Y;         // device-side training loop: minibatch rows, step counter, output
    cudaStream_t cap = nullptr;  // private stream on which the training step is captured
    long cap_rows = 0, cap_grad = 0;  // rows that A holds, and the gradients' buffers
    std::vector<long> z_off, a_off;  // per layer offsets into Z / A (elements)
};

namespace {

// dynamic shared memory of a layer launch: a product's tile or the column
// sums' rows
template <int BN>
constexpr int layer_smem() {
    return tc_smem_bytes<BN>() > 256 * 32 * 4 ? tc_smem_bytes<BN>() : 256 * 32 * 4;
}

// Work space for passes on n rows: activations alone for a prediction, and for a
// gradient the pre-activations and two layers' gradients as well.  A buffer that
// fails to grow is gone, so no batch fits until all are there, and the offsets
// change with the capacity.
int ensure_rows(mirage_mlp* m, int n) {
    if (n <= m->cap_rows) return MIRAGE_OK;
    std::vector<long> off(m->L + 1, 0);
    long at = 0;
    for (int l = 0; l <= m->L; ++l) {
        off[l] = at;
        at += ((long)n * m->dims[l] + 7) & ~7L;  // (16-byte rows stay aligned)
    }
    m->cap_rows = 0;
    if (const int r = m->A.ensure(sizeof(__nv_bfloat16) * at)) return r;
    m->a_off = off;
    m->cap_rows = n;
    return MIRAGE_OK;
}

// elements of one layer's gradient
long grad_rows(const mirage_mlp* m, long n) {
    return (n * *std::max_element(m->dims.begin(), m->dims.end()) + 7) & ~7L;
}

int ensure_grad(mirage_mlp* m, int n) {
    int r;
    if ((r = ensure_rows(m, n))) return r;
    if (n <= m->cap_grad) return MIRAGE_OK;
    std::vector<long> off(m->L + 1, 0);
    long zt = 0;
    for (int l = 1; l <= m->L; ++l) {
        off[l] = zt;
        zt += (long)n * m->dims[l];
    }
    m->cap_grad = 0;
    if ((r = m->Z.ensure(sizeof(float) * zt)) || (r = m->DZ.ensure(2 * sizeof(float) * grad_rows(m, n))) ||
        (r = m->DZH.ensure(2 * sizeof(__nv_bfloat16) * grad_rows(m, n))) || (r = m->LOSS.ensure(sizeof(double))))
        return r;
    m->z_off = off;
    m->cap_grad = n;
    return MIRAGE_OK;
}

// raises the layer kernels' shared-memory limit on the current device (once
// per network, outside any stream capture)
int gemm_setup() {
    MCK(cudaFuncSetAttribute(k_layer<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, layer_smem<16>()));
    MCK(cudaFuncSetAttribute(k_layer<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, layer_smem<32>()));
    return MIRAGE_OK;
}

// launch as a programmatic dependent of the stream's previous launch
template <class... P, class... Q>
cudaError_t launch_dep(void (*fn)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Q... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

// one launch of a layer's work, in N tiles of 16 columns for narrow products
// and 32 for the others (the 256-wide layers run in eight: more CTAs, each with
// a shorter epilogue)
template <int BN>
int launch_layer_bn(LayerArgs& a, cudaStream_t st) {
    unsigned grid = 0;
    for (Gemm& g : a.g) {
        g.tm = (g.M + TC_BM - 1) / TC_BM;
        g.tiles = g.M > 0 && g.N > 0 ? g.tm * ((g.N + BN - 1) / BN) : 0;
        grid += (unsigned)g.tiles;
    }
    if (a.S) grid += (unsigned)((a.scols + 31) / 32);
    if (!grid) return MIRAGE_OK;
    MCK(launch_dep(k_layer<BN>, grid, TC_T, layer_smem<BN>(), st, a));
    return MIRAGE_OK;
}
int launch_layer(LayerArgs& a, cudaStream_t st) {
    const int N = a.g[0].N;  // (the second product has the same width)
    if (N <= 16) return launch_layer_bn<16>(a, st);
    return launch_layer_bn<32>(a, st);
}

// The forward pass, one launch a layer: z_l (FP32, kept for a backward pass)
// and a_l (BF16) of the hidden layers, y of the last.  With idx, batch row j
// is row idx[j] of x; with tgt the last layer also leaves the loss gradient in
// DZ and DZH; inc is incremented (device step counter).
int forward_pass(mirage_mlp* m, const float* x, int n, float* y, cudaStream_t st, bool keep = false, const int* idx = nullptr,
                 const float* tgt = nullptr, long long* inc = nullptr) {
    int r;
    if ((r = keep ? ensure_grad(m, n) : ensure_rows(m, n))) return r;
    float* Z = (float*)m->Z.p;
    __nv_bfloat16* A = (__nv_bfloat16*)m->A.p;
    const float* P = (const float*)m->P.p;
    const __nv_bfloat16* PH = (const __nv_bfloat16*)m->PH.p;
    if (keep && !idx) {  // the backward pass reads the input as BF16 too (drawn rows already are)
        MCK(launch_dep(k_to_bf16, blocks((long)n * m->dims[0], 256), 256, 0, st, x, A, (long)n * m->dims[0]));
    }
    for (int l = 1; l <= m->L; ++l) {
        const int in = m->dims[l - 1], out = m->dims[l];
        LayerArgs a;
        Gemm& g = a.g[0];
        // Z_l = A_{l-1} W_l^T : A(m, k) = A[m in + k], B(k, j) = W[j in + k]
        if (l == 1 && !keep) g.Af = x;
        g.A = A + m->a_off[l - 1];
        g.sam = in;
        g.sak = 1;
        g.B = PH + m->w_off[l - 1];
        g.sbk = 1;
        g.sbn = in;
        g.M = n;
        g.N = out;
        g.K = in;
        g.bias = P + m->b_off[l - 1];
        if (l < m->L) {
            g.epi = EPI_HIDDEN;
            g.Z = keep ? Z + m->z_off[l] : nullptr;
            g.H = A + m->a_off[l];
        } else {
            g.epi = EPI_OUT;
            g.Y = y;
            g.T = tgt;
            g.tidx = idx;
            g.D = (float*)m->DZ.p;
            g.H = (__nv_bfloat16*)m->DZH.p;
        }
        if (l == 1) a.inc = inc;
        if ((r = launch_layer(a, st))) return r;
    }
    return MIRAGE_OK;
}

// gradients of the MSE into m->G (and the loss into m->LOSS if wanted)
int backward_pass(mirage_mlp* m, const float* x, const float* tgt, int n, float* yscratch, bool want_loss,
                  cudaStream_t st, const int* idx = nullptr, long long* inc = nullptr) {
    int r;
    if ((r = forward_pass(m, x, n, yscratch, st, true, idx, want_loss ? nullptr : tgt, inc))) return r;
    float* Z = (float*)m->Z.p;
    __nv_bfloat16* A = (__nv_bfloat16*)m->A.p;
    float* G = (float*)m->G.p;
    const __nv_bfloat16* PH = (const __nv_bfloat16*)m->PH.p;
    const int outL = m->dims[m->L];
    if (want_loss) {
        double* loss = (double*)m->LOSS.p;
        MCK(cudaMemsetAsync(loss, 0, sizeof(double), st));
        MCK(launch_dep(k_loss_grad, blocks((long)n * outL, 256), 256, 0, st, yscratch, tgt, idx, outL, (long)n * outL,
                       (float*)m->DZ.p, (__nv_bfloat16*)m->DZH.p, loss));
    }
    const long half = grad_rows(m, m->cap_grad);  // a layer's part of DZ and DZH
    for (int l = m->L, cur = 0; l >= 1; --l, cur ^= 1) {
        const int in = m->dims[l - 1], out = m->dims[l];
        float *dz = (float*)m->DZ.p + cur * half, *dzn = (float*)m->DZ.p + (cur ^ 1) * half;
        __nv_bfloat16 *dzh = (__nv_bfloat16*)m->DZH.p + cur * half, *dzhn = (__nv_bfloat16*)m->DZH.p + (cur ^ 1) * half;
        LayerArgs a;
        // dW_l = dZ^T A_{l-1}: [out x in];  A(mm, k) = dZ[k out + mm], B(k, j) = A_{l-1}[k in + j]
        Gemm& w = a.g[0];
        w.A = dzh;
        w.sam = 1;
        w.sak = out;
        w.B = A + m->a_off[l - 1];
        w.sbk = in;
        w.sbn = 1;
        w.C = G + m->w_off[l - 1];
        w.M = out;
        w.N = in;
        w.K = n;
        // db_l: column sums of dZ
        a.S = dz;
        a.srows = n;
        a.scols = out;
        a.sum = G + m->b_off[l - 1];
        if (l > 1) {
            // dA_{l-1} = dZ W_l: A(mm, k) = dZ[mm out + k], B(k, j) = W[k in + j]
            Gemm& d = a.g[1];
            d.A = dzh;
            d.sam = out;
            d.sak = 1;
            d.B = PH + m->w_off[l - 1];
            d.sbk = in;
            d.sbn = 1;
            d.M = n;
            d.N = in;
            d.K = out;
            d.epi = EPI_BACK;
            d.Z = Z + m->z_off[l - 1];
            d.D = dzn;
            d.H = dzhn;
        }
        if ((r = launch_layer(a, st))) return r;
    }
    return MIRAGE_OK;
}

// deterministic host RNG (splitmix64 + Box-Muller) for the initial weights
struct HostRng {
    unsigned long long s;
    unsigned long long next() {
        unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    }
    double uniform() { return ((next() >> 11) + 0.5) * (1.0 / 9007199254740992.0); }
    double normal() { return std::sqrt(-2.0 * std::log(uniform())) * std::cos(6.283185307179586 * uniform()); }
};

}  // namespace

extern "C" {

int mirage_mlp_create(mirage_mlp_t** out, int device, int n_layers, const int* dims, unsigned long long seed) {
    if (!out || n_layers < 1 || n_layers > 16 || !dims) return mlp_fail(MIRAGE_ERR_ARG, "mlp_create: bad arguments");
    *out = nullptr;
    for (int l = 0; l <= n_layers; ++l)
        if (dims[l] < 1 || dims[l] > 4096) return mlp_fail(MIRAGE_ERR_ARG, "mlp_create: layer width out of range");
    MCK(cudaSetDevice(device));
    if (const int rs = gemm_setup()) return rs;
    mirage_mlp* m = new mirage_mlp();
    m->device = device;
    m->L = n_layers;
    m->dims.assign(dims, dims + n_layers + 1);
    long off = 0;
    for (int l = 0; l < n_layers; ++l) {
        m->w_off.push_back(off);
        off += (long)dims[l + 1] * dims[l];
        m->b_off.push_back(off);
        off += dims[l + 1];
    }
    m->n_params = off;
    int r = 0;
    if ((r = m->P.ensure(sizeof(float) * off)) || (r = m->PH.ensure(sizeof(__nv_bfloat16) * off)) ||
        (r = m->M.ensure(sizeof(float) * off)) || (r = m->V.ensure(sizeof(float) * off)) ||
        (r = m->G.ensure(sizeof(float) * off)) || (r = m->ISW.ensure(off))) {
        delete m;
        return r;
    }
    // He-style initial weights (std sqrt(2 / fan_in)), zero biases
    std::vector<float> h(off, 0.f);
    std::vector<unsigned char> isw(off, 0);
    HostRng rng{seed};
    for (int l = 0; l < n_layers; ++l) {
        const double sd = std::sqrt(2.0 / dims[l]);
        for (long i = 0; i < (long)dims[l + 1] * dims[l]; ++i) {
            h[m->w_off[l] + i] = (float)(sd * rng.normal());
            isw[m->w_off[l] + i] = 1;
        }
    }
    if (cudaMemcpy(m->ISW.p, isw.data(), off, cudaMemcpyHostToDevice) != cudaSuccess) {
        delete m;
        return mlp_fail(MIRAGE_ERR_CUDA, "mlp_create: upload failed");
    }
    *out = m;
    return mirage_mlp_set_params(m, h.data(), off);
}

int mirage_mlp_destroy(mirage_mlp_t* m) {
    if (!m) return MIRAGE_OK;
    cudaSetDevice(m->device);
    Buf* bufs[] = {&m->P,  &m->PH,  &m->M,  &m->V,    &m->G,   &m->ISW,  &m->Z,
                   &m->A,  &m->DZ,  &m->DZH, &m->Y,   &m->LOSS, &m->IDX, &m->DSTEP};
    for (Buf* b : bufs) b->release();
    if (m->cap) cudaStreamDestroy(m->cap);
    delete m;
    return MIRAGE_OK;
}

long mirage_mlp_num_params(const mirage_mlp_t* m) { return m ? m->n_params : 0; }

int mirage_mlp_set_params(mirage_mlp_t* m, const float* host_params, long n) {
    if (!m || !host_params || n != m->n_params) return mlp_fail(MIRAGE_ERR_ARG, "mlp_set_params: size mismatch");
    MCK(cudaSetDevice(m->device));
    MCK(cudaMemcpy(m->P.p, host_params, sizeof(float) * n, cudaMemcpyHostToDevice));
    MCK(cudaMemset(m->M.p, 0, sizeof(float) * n));
    MCK(cudaMemset(m->V.p, 0, sizeof(float) * n));
    k_params_bf16<<<blocks(n, 256), 256>>>((const float*)m->P.p, (__nv_bfloat16*)m->PH.p, n);
    MCK(cudaGetLastError());
    MCK(cudaDeviceSynchronize());
    m->step = 0;
    return MIRAGE_OK;
}

int mirage_mlp_get_params(const mirage_mlp_t* m, float* host_params, long n) {
    if (!m || !host_params || n != m->n_params) return mlp_fail(MIRAGE_ERR_ARG, "mlp_get_params: size mismatch");
    MCK(cudaSetDevice(m->device));
    MCK(cudaMemcpy(host_params, m->P.p, sizeof(float) * n, cudaMemcpyDeviceToHost));
    return MIRAGE_OK;
}

int mirage_mlp_forward(mirage_mlp_t* m, const float* x, int n, float* y, void* stream) {
    if (!m || !x || !y || n < 0) return mlp_fail(MIRAGE_ERR_ARG, "mlp_forward: bad arguments");
    if (n == 0) return MIRAGE_OK;
    MCK(cudaSetDevice(m->device));
    return forward_pass(m, x, n, y, reinterpret_cast<cudaStream_t>(stream));
}

int mirage_mlp_grad(mirage_mlp_t* m, const float* x, const float* t, int n, float* grad, double* loss, float* y,
                    void* stream) {
    if (!m || !x || !t || !y || n < 1) return mlp_fail(MIRAGE_ERR_ARG, "mlp_grad: bad arguments");
    MCK(cudaSetDevice(m->device));
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int r = backward_pass(m, x, t, n, y, loss != nullptr, st);
    if (r) return r;
    if (grad) MCK(cudaMemcpyAsync(grad, m->G.p, sizeof(float) * m->n_params, cudaMemcpyDeviceToDevice, st));
    if (loss) MCK(cudaMemcpyAsync(loss, m->LOSS.p, sizeof(double), cudaMemcpyDeviceToDevice, st));
    return MIRAGE_OK;
}

int mirage_mlp_train_step(mirage_mlp_t* m, const float* x, const float* t, int n, float lr, double* loss, float* y,
                          void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int r = mirage_mlp_grad(m, x, t, n, nullptr, loss, y, stream);
    if (r) return r;
    m->step += 1;
    const float c1 = 1.f - std::pow(m->b1, (float)m->step), c2 = 1.f - std::pow(m->b2, (float)m->step);
    MCK(launch_dep(k_adam, blocks(m->n_params, 256), 256, 0, st, (float*)m->P.p, (const float*)m->G.p, (float*)m->M.p,
                   (float*)m->V.p, m->n_params, lr, m->b1, m->b2, m->eps, c1, c2, (__nv_bfloat16*)m->PH.p,
                   (const unsigned char*)m->ISW.p));
    return MIRAGE_OK;
}

int mirage_mlp_train(mirage_mlp_t* m, const float* x, const float* t, int n, int steps, int batch, float lr,
                     unsigned long long seed, void* stream) {
    if (!m || !x || !t || n < 1 || steps < 0 || batch < 1 || batch > (1 << 20))
        return mlp_fail(MIRAGE_ERR_ARG, "mlp_train: bad arguments");
    if (steps == 0) return MIRAGE_OK;
    MCK(cudaSetDevice(m->device));
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int r;
    // every buffer the step touches exists before the capture (no allocation inside it)
    if ((r = ensure_grad(m, batch)) || (r = m->IDX.ensure(sizeof(int) * (size_t)batch)) ||
        (r = m->DSTEP.ensure(sizeof(long long))) || (r = m->Y.ensure(sizeof(float) * (size_t)batch * m->dims[m->L])))
        return r;
    if (!m->cap) MCK(cudaStreamCreateWithFlags(&m->cap, cudaStreamNonBlocking));
    long long* dstep = (long long*)m->DSTEP.p;
    int* idx = (int*)m->IDX.p;
    float* y = (float*)m->Y.p;
    const long long s0 = m->step;
    MCK(cudaMemcpyAsync(dstep, &s0, sizeof(long long), cudaMemcpyHostToDevice, st));

    const Draw draw{idx, (__nv_bfloat16*)m->A.p, x, batch, n, m->dims[0], seed};
    const unsigned db = blocks((long)batch * m->dims[0], 256), nb = blocks(m->n_params, 256);
    k_draw<<<db, 256, 0, st>>>(draw, dstep);
    MCK(cudaGetLastError());

    // one training step: forward, MSE gradient, Adam, the next step's rows;
    // captured once
    cudaGraph_t graph = nullptr;
    MCK(cudaStreamBeginCapture(m->cap, cudaStreamCaptureModeThreadLocal));
    r = backward_pass(m, x, t, batch, y, false, m->cap, idx, dstep);
    if (!r && launch_dep(k_adam_dev, nb + db, 256, 0, m->cap, (float*)m->P.p, (const float*)m->G.p, (float*)m->M.p,
                         (float*)m->V.p, m->n_params, lr, m->b1, m->b2, m->eps, (const long long*)dstep,
                         (__nv_bfloat16*)m->PH.p, (const unsigned char*)m->ISW.p, nb, draw) != cudaSuccess)
        r = mlp_fail(MIRAGE_ERR_CUDA, "mlp_train: launch failed");
    const cudaError_t ec = cudaStreamEndCapture(m->cap, &graph);
    if (r) {
        if (graph) cudaGraphDestroy(graph);
        return r;
    }
    if (ec != cudaSuccess || !graph)
        return mlp_fail(MIRAGE_ERR_CUDA, std::string("mlp_train: capture failed: ") + cudaGetErrorString(ec));
    cudaGraphExec_t exec = nullptr;
    const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ei != cudaSuccess)
        return mlp_fail(MIRAGE_ERR_CUDA, std::string("mlp_train: instantiate failed: ") + cudaGetErrorString(ei));
    cudaError_t el = cudaSuccess;
    for (int k = 0; k < steps && el == cudaSuccess; ++k) el = cudaGraphLaunch(exec, st);
    cudaGraphExecDestroy(exec);
    if (el != cudaSuccess)
        return mlp_fail(MIRAGE_ERR_CUDA, std::string("mlp_train: graph launch failed: ") + cudaGetErrorString(el));
    m->step += steps;
    return MIRAGE_OK;
}

const char* mirage_mlp_last_error(void) { return g_mlp_err.c_str(); }

}  // extern "C"
