// C ABI of the lens-inversion inner loop: context, argument checks, scratch
// management, work-item planning, launches and CUDA-graph replay.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <initializer_list>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../../include/mirage.h"
#include "cluster.cuh"
#include "fast.cuh"
#include "forward.cuh"
#include "iterlc.cuh"
#include "kernels.cuh"
#include "table.h"

using namespace mirage;

namespace {

thread_local std::string g_last_error;

void set_error(const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_last_error = buf;
}

#define CK(call)                                                                        \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) {                                                        \
            set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, \
                      __LINE__);                                                        \
            return e_ == cudaErrorMemoryAllocation ? MIRAGE_ERR_NOMEM : MIRAGE_ERR_CUDA; \
        }                                                                               \
    } while (0)

const KernelTable& table() {
    static KernelTable t = [] {
        KernelTable k;
        std::memset(&k, 0, sizeof(k));
        fill_f32_k5(k);
        fill_f32_k7(k);
        fill_f32_k9(k);
        fill_f32_k11(k);
        fill_f32_k15(k);
        fill_f32_k21(k);
        fill_f32_gen(k);
        fill_f64(k);
        fill_fast(k);
        fill_fast1(k);
        fill_iter(k);
        fill_fwd_band(k);
        fill_cluster_a(k);
        fill_cluster_b(k);
        fill_cluster_c(k);
        fill_cluster_d(k);
        fill_cluster_e(k);
        return k;
    }();
    return t;
}

// grow-only device buffer owned by the context
struct DevBuf {
    void* p = nullptr;
    size_t n = 0;
    int ensure(size_t bytes) {
        if (bytes <= n) return MIRAGE_OK;
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
        size_t want = std::max<size_t>(bytes, 256);
        cudaError_t e = cudaMalloc(&p, want);
        if (e != cudaSuccess) {
            set_error("cudaMalloc(%zu) failed: %s", want, cudaGetErrorString(e));
            p = nullptr;
            return MIRAGE_ERR_NOMEM;
        }
        n = want;
        return MIRAGE_OK;
    }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
    template <typename U>
    U* as() const {
        return reinterpret_cast<U*>(p);
    }
};

struct GraphEntry {
    cudaGraphExec_t exec = nullptr;
    int launches = 0;
    DevBuf probs, meta;  // this graph's own copy of the launch metadata
};

}  // namespace

struct mirage_ctx {
    int device = 0;
    int precision = MIRAGE_FP32;
    int sm_count = 0;
    int max_smem = 0;
    int max_smem_sm = 0;
    int last_launches = 0;
    int last_kernels[MIRAGE_N_ITEM_KERNELS] = {};  // items of the last evaluation by kernel
    int reserved = 0;  // CTA slots the CGLS launches leave free (mirage_set_reserved_slots)
    // scratch
    DevBuf E, E64, Etmp, inv, cst, swp, dpad, nent, cstat, X, istat, slab, probs, cand_prob, items, counters;
    DevBuf stage;  // MIRAGE_MEM_HOST staging
    DevBuf fE, fE64, fEtmp, finv, fcst, fswp, fdpad, fnent, fcstat, fslab, fprob, fcand, fpix;
    DevBuf rt_cursor;  // per-cell cursors of the parallel ray placement
    DevBuf spec;       // PSF spectra of the FFT-convolution problems (FP64, then FP32)
    // pinned staging of the per-call uploads (problem descriptors, item
    // tables): the copies stay asynchronous; the event guards reuse
    void* pin = nullptr;
    size_t pin_n = 0;
    cudaEvent_t pin_ev = nullptr;
    bool pin_pending = false;
    std::map<std::string, GraphEntry> graphs;
    std::map<const void*, int> smem_set;  // kernel -> dynamic smem attribute set
    std::map<std::pair<const void*, std::pair<int, size_t>>, int> cl_active;  // resident clusters of (kernel, size, smem)
    cudaStream_t cap_stream = nullptr;   // graphs are captured here and launched on the caller's stream
    static constexpr int NSIDE = 32;
    cudaStream_t side[NSIDE] = {};  // concurrent kernel groups
    cudaEvent_t fork_ev = nullptr, join_ev[NSIDE] = {};
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};  // phase timing (opts.threads < 0)
    DevBuf clk;                                                  // per-phase SM clocks (opts.threads == -2)
    int timed = 0;
    std::vector<void*> scratch_seen;     // scratch pointers the cached graphs were captured with
};

// CTAs of a persistent CGLS launch: per_sm on every SM, less the slots the
// caller reserved for concurrent work on other streams (at least one)
static long long cgls_slots(const mirage_ctx* ctx, int per_sm) {
    return std::max<long long>(1, (long long)per_sm * ctx->sm_count - ctx->reserved);
}

// a PSF tap as the fast kernel's parameter: as is, or rounded to TF32
// (nearest, ties away from zero: the cvt.rna.tf32 rule) for the TF32
// precision variant
static float tap_value(float t, bool tf32) {
    if (!tf32) return t;
    unsigned u;
    std::memcpy(&u, &t, sizeof(u));
    if ((u & 0x7f800000u) != 0x7f800000u) u = (u + 0x1000u) & ~0x1fffu;
    float r;
    std::memcpy(&r, &u, sizeof(r));
    return r;
}

// relative CG iteration count of lambda index k of an n-point ascending
// grid: measured counts scale like lambda^-0.37, and the grids span about six
// decades log-spaced, so the count grows by 10^(2.2 / (n - 1)) per step
// towards small lambda
static double chain_weight(int n, int k) {
    return n > 1 ? std::pow(10.0, 2.2 * (double)(n - 1 - k) / (double)(n - 1)) : 1.0;
}

namespace {
void drop_graphs(mirage_ctx* ctx) {
    for (auto& kv : ctx->graphs) {
        if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
        kv.second.probs.release();
        kv.second.meta.release();
    }
    ctx->graphs.clear();
}
}  // namespace

namespace {

template <typename T>
constexpr int prec_of() {
    return sizeof(T) == 4 ? 0 : 1;
}

int check_geom(const mirage_geom_t& g) {
    if (g.nx < 1 || g.ny < 1 || g.nx > 4096 || g.ny > 4096) return MIRAGE_ERR_ARG;
    if (g.sx < 2 || g.sy < 2 || (long long)g.sx * g.sy > (1 << 20)) return MIRAGE_ERR_ARG;
    if (!(g.pix > 0) || !(g.sxmax > g.sxmin) || !(g.symax > g.symin)) return MIRAGE_ERR_ARG;
    if (g.kpsf < 1 || g.kpsf > MIRAGE_MAX_KPSF || (g.kpsf % 2) == 0) return MIRAGE_ERR_ARG;
    if (g.subpix < 1 || g.subpix > 8) return MIRAGE_ERR_ARG;
    if (g.reg < 0 || g.reg > 2) return MIRAGE_ERR_ARG;
    if (g.interp != MIRAGE_INTERP_BILINEAR && g.interp != MIRAGE_INTERP_NEAREST && g.interp != MIRAGE_INTERP_BICUBIC)
        return MIRAGE_ERR_ARG;
    if (!std::isfinite(g.cx) || !std::isfinite(g.cy)) return MIRAGE_ERR_ARG;
    return MIRAGE_OK;
}

template <typename T>
Prob<T> make_prob(const mirage_problem_t& mp, const void* d, const void* sigma, const void* mask, const void* psf) {
    const mirage_geom_t& g = mp.geom;
    Prob<T> P;
    std::memset(&P, 0, sizeof(P));
    P.nx = g.nx;
    P.ny = g.ny;
    P.npix = g.nx * g.ny;
    P.sx = g.sx;
    P.sy = g.sy;
    P.ns = g.sx * g.sy;
    P.reg = g.reg;
    P.interp = g.interp;
    P.nreg = g.reg == MIRAGE_REG_GRADIENT ? 2 * P.ns : P.ns;
    P.K = g.kpsf;
    P.hk = (g.kpsf - 1) / 2;
    P.kp = (g.kpsf + 3) & ~3;
    P.n_sub = g.subpix;
    P.Np = g.subpix * g.subpix;
    P.nrays = P.npix * P.Np;
    P.ncx = g.sx - 1;
    P.ncells = (g.sx - 1) * (g.sy - 1);
    P.tiles_x = (g.nx + TILE - 1) / TILE;
    P.tiles_y = (g.ny + TILE - 1) / TILE;
    P.ntiles = P.tiles_x * P.tiles_y;
    const int VW = 16 / (int)sizeof(T);
    P.xoff = (P.hk + VW - 1) / VW * VW;
    const int sh = P.xoff - P.hk;
    const int nvw = (TILE + g.kpsf - 1 + sh + VW - 1) / VW * VW;
    P.Wp = std::max((P.tiles_x - 1) * TILE + nvw, P.xoff + g.nx + P.hk);
    P.Wp = (P.Wp + VW - 1) / VW * VW;
    P.Hp = P.tiles_y * TILE + g.kpsf - 1;
    P.plen = P.Wp * P.Hp;
    P.pix = g.pix;
    P.cx = g.cx;
    P.cy = g.cy;
    P.sub0 = (0.5 / g.subpix - 0.5) * g.pix;
    P.subd = g.pix / g.subpix;
    P.hx = (g.sxmax - g.sxmin) / g.sx;
    P.hy = (g.symax - g.symin) / g.sy;
    P.c0x = g.sxmin + 0.5 * P.hx;
    P.c0y = g.symin + 0.5 * P.hy;
    P.invNp = (T)(1.0 / P.Np);
    P.d = reinterpret_cast<const T*>(d);
    P.sigma = reinterpret_cast<const T*>(sigma);
    P.mask = reinterpret_cast<const uint8_t*>(mask);
    P.psf = reinterpret_cast<const T*>(psf);
    return P;
}

int set_smem(mirage_ctx* ctx, const void* fn, size_t bytes) {
    auto it = ctx->smem_set.find(fn);
    if (it == ctx->smem_set.end()) {
        cudaFuncAttributes fa;
        CK(cudaFuncGetAttributes(&fa, fn));
        const int dyn_max = ctx->max_smem - (int)fa.sharedSizeBytes;
        CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max));
        CK(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
        it = ctx->smem_set.emplace(fn, dyn_max).first;
    }
    if ((long long)bytes > it->second) {
        set_error("work item needs %zu B of dynamic shared memory (limit %d)", bytes, it->second);
        return MIRAGE_ERR_UNSUPPORTED;
    }
    return MIRAGE_OK;
}

const void* pick_cgls(int prec, int place, int K) {
    const KernelTable& t = table();
    const void* f = K < MAX_K ? t.cgls[prec][place][K] : nullptr;  // wider PSFs: the runtime-K kernel
    return f ? f : t.cgls[prec][place][0];
}

// placement of the general kernel's work buffers for one problem
template <typename T>
int pick_place(const mirage_ctx* ctx, const Prob<T>& P, int want = 0) {
    if (P.fft_m) return PLACE_GLOBAL;  // the FFT path lives in the runtime-K global-memory kernel
    // a requested placement (mirage_opts_t.place: 1 SMEM, 2 MID, 3 GLOBAL,
    // 4 GLOBAL with two CTAs per SM) where it fits
    if (want == 1 && smem_bytes<T>(P, PLACE_SMEM) <= (size_t)ctx->max_smem) return PLACE_SMEM;
    if (want == 2 && sizeof(T) == 4 && smem_bytes<T>(P, PLACE_MID) <= (size_t)ctx->max_smem) return PLACE_MID;
    if (want == 3) return PLACE_GLOBAL;
    if (want == 4) {
        const KernelTable& t = table();
        if (sizeof(T) == 4 && (t.cgls[0][PLACE_GLOBAL2][P.K < MAX_K ? P.K : 0] || t.cgls[0][PLACE_GLOBAL2][0]) &&
            2 * (long long)smem_bytes<T>(P, PLACE_GLOBAL) <= ctx->max_smem_sm - 2048)
            return PLACE_GLOBAL2;
        return PLACE_GLOBAL;
    }
    if (want == 5 && sizeof(T) == 4) {
        const KernelTable& t = table();
        if ((t.cgls[0][PLACE_MID2][P.K < MAX_K ? P.K : 0] || t.cgls[0][PLACE_MID2][0]) &&
            2 * ((long long)smem_bytes<T>(P, PLACE_MID) + 1024) <= ctx->max_smem_sm)
            return PLACE_MID2;
    }
    if (smem_bytes<T>(P, PLACE_SMEM) <= (size_t)ctx->max_smem) return PLACE_SMEM;
    if (sizeof(T) == 4 && smem_bytes<T>(P, PLACE_MID) <= (size_t)ctx->max_smem) return PLACE_MID;
    // all in the slab: two CTAs per SM where that kernel is compiled for the
    // problem's PSF width (FP32; 1.47x faster at 256 x 256 with a 21 x 21 PSF,
    // where one 253-register CTA per SM could not hide the slab's latency)
    if (sizeof(T) == 4 && P.K < MAX_K && table().cgls[0][PLACE_GLOBAL2][P.K] &&
        2 * (long long)smem_bytes<T>(P, PLACE_GLOBAL) <= ctx->max_smem_sm - 2048)
        return PLACE_GLOBAL2;
    return PLACE_GLOBAL;
}

// FFT convolution of a problem's lambda-grid solves: forced by variant 5,
// never with variant 6 (direct convolution at any width), otherwise for PSFs
// of FFT_AUTO_K taps and wider.  The grid side is the
// smallest power of two >= max(nx, ny) + (K - 1) / 2 (at least 16, at most
// 1024); problems whose FFT buffers do not fit in shared memory keep the
// direct convolution.
constexpr int FFT_AUTO_K = 23;  // the first width without a compiled direct kernel; measured crossover 21..25

template <typename T>
void plan_fft(const mirage_ctx* ctx, Prob<T>& P, int variant) {
    P.fft_m = 0;
    P.fft_log = 0;
    if (variant == 6 || (variant != 5 && P.K < FFT_AUTO_K)) return;
    const int M = std::max(16, fft_size_for(std::max(P.nx, P.ny) + P.hk));
    if (M > 1024) return;
    Prob<T> Q = P;
    Q.fft_m = M;
    if (smem_bytes<T>(Q, PLACE_GLOBAL) > (size_t)ctx->max_smem) return;
    P.fft_m = M;
    while ((1 << P.fft_log) < M) ++P.fft_log;
}

const void* pick_fwd(int prec, int K) {
    const KernelTable& t = table();
    const void* f = K < MAX_K ? t.fwd[prec][K] : nullptr;
    return f ? f : t.fwd[prec][0];
}

// two-CTA-per-SM kernel when the problem qualifies (FP32 contexts only)
template <typename T>
const void* pick_fast(mirage_ctx* ctx, const Prob<T>& P, int mode, bool alone) {
    if (sizeof(T) != 4 || P.interp == MIRAGE_INTERP_BICUBIC) return nullptr;  // four-corner rays only
    const Prob<float>& Pf = *reinterpret_cast<const Prob<float>*>(&P);
    const size_t b = fast_smem_bytes(Pf);
    if (b == 0 || (long long)b > ctx->max_smem_sm / 2 - 1024 || Pf.K >= MAX_K) return nullptr;
    return table().fast[Pf.K][alone][mode];  // (alone: one CTA per SM)
}

// The cluster kernel's choice for one problem (C = 0: not eligible).
struct ClusterPlan {
    int C = 0, nt = 0;
    const void* fn = nullptr;
    size_t smem = 0;
    long long slab = 0;
};

// Clocks of one CG iteration of problem P: `lat` as one item alone sees it, `thr`
// the SM clocks that it takes up on a busy device, `busy` as an item sees it there
// (with another item's CTAs on its SMs where two fit).  Least-squares fits to the
// iterations of 147 systems (images 28 x 28 to 256 x 256, sources 12 x 12 to 128 x 128,
// K = 3 to 21, fields of 3.2 to 6.4 arcsec; one item alone, and 304 of them
// together), which they meet to 10% (general kernel, everything in shared memory),
// 15% (not everything) and 13% (cluster kernel).
struct IterCost {
    double lat, thr, busy;
};
// mapped part of the image: the source's area, magnified (measured: 0.6 to 0.95
// where the areas' ratio is 0.19 to 0.26, 0.27 at 0.06)
template <typename T>
double mapped_part(const Prob<T>& P) {
    const double area = P.hx * P.sx * P.hy * P.sy / (P.npix * P.pix * P.pix);
    return std::min(1.0, 0.07 + 3.2 * area);
}
// a source about as fine as the image has its L^T summed ray by ray
template <typename T>
bool gathers(const Prob<T>& P) {
    return 4 * P.ncells > P.plen;
}
template <typename T>
IterCost fast_cost(const Prob<T>& P) {
    const double c = 4.0 * P.K * P.K * P.npix / 130.0 + P.nrays;  // (27.5k each of two at 64 x 64, K = 9)
    return {2.0 * c, c, 2.0 * c};
}
template <typename T>
IterCost general_cost(const Prob<T>& P, int place) {
    if (P.fft_m) return {6.0 * P.fft_m * P.fft_m, 6.0 * P.fft_m * P.fft_m, 6.0 * P.fft_m * P.fft_m};
    // PSF widths without a kernel of their own loop over the taps at run time
    const bool unrolled = P.K < MAX_K && table().cgls[prec_of<T>()][place][P.K];
    const double k2 = P.K * P.K, per = (P.ntiles + NTHREADS - 1) / NTHREADS, pix = P.npix;
    const double rays = mapped_part(P) * P.nrays, fine = gathers(P) ? P.ns : 0.0;
    if (place == PLACE_SMEM || place == PLACE_SMEM2) {
        const double c = unrolled ? 7000.0 + 61.0 * k2 * per + 4.6 * pix + 0.2 * rays + 7.3 * fine
                                  : 9200.0 + k2 * (1.72 * P.ntiles + 81.0 * per) + 1.2 * pix + 3.5 * rays + 10.5 * fine;
        return {c, 1.05 * c, 1.05 * c};
    }
    if (layout_of(place) == PLACE_MID) {
        const double c = unrolled ? 78.0 * k2 * per + 4.2 * pix + 3.1 * rays + 780.0 * rays / P.ncells
                                  : 58000.0 + k2 * (0.93 * P.ntiles + 184.0 * per) + 3.4 * rays;
        return {c, 1.07 * c, 1.07 * c};
    }
    // (the slabs' traffic adds up: 2048 items at 256 x 256 and K = 21 took 1155k of SM
    // time an iteration with two CTAs an SM)
    const double c = (unrolled ? 123.0 : 430.0) * k2 * per + 5.9 * pix + 6.6 * rays;
    return {c, two_per_sm(place) ? 0.8 * c : c, two_per_sm(place) ? 1.6 * c : c};
}
inline IterCost cluster_cost(const Prob<float>& P, int C, int nt) {
    // a cell's rays are one thread's; of coarse sources, whole rows of cells are one
    // CTA's (13 x 14 cells on eight SMs: 164k clocks)
    const double f = mapped_part(P), rays = f * P.nrays, conv = f * P.K * P.K * P.npix, pix = P.npix;
    const double cell = rays / P.ncells, crowd = std::max(0.0, cell - 30.0), fine = gathers(P) ? P.ns : 0.0;
    const double lat = 18200.0 + 0.75 * rays + 700.0 * cell + 1000.0 * std::min(C, 4) * crowd +
                       (4000.0 + 2.6 * rays + 0.0185 * conv + 0.3 * pix + 20.4 * fine) / C;
    // SM time by CTA (two of 256 threads an SM, or one of 512) and cluster size: the
    // barriers' waits are partly the other CTA's, and no whole cluster fits on some SMs
    // (15 of eight on 152).  {1, rays, conv, pix, cell, crowd, fine}; the last two
    // of 512 threads from two image sizes
    static constexpr double w[2][4][7] = {{{11100, 2.38, 0.0144, 2.28, 461, 0, 11.4},
                                           {23400, 2.29, 0.0158, 1.05, 872, 2500, 11.7},
                                           {49400, 3.27, 0.0218, 1.54, 1730, 13100, 16.5},
                                           {86400, 5.87, 0.0203, 1.30, 3300, 33200, 23.1}},
                                          {{15600, 1.98, 0.0126, 2.58, 913, 1000, 0},
                                           {41400, 4.98, 0.0157, 1.15, 984, 2700, 0},
                                           {86000, 6.30, 0.0360, 1.00, 1730, 13100, 0},
                                           {90000, 14.9, 0.0218, 3.90, 3300, 33200, 0}}};
    const double* a = w[nt > NTHREADS][(C > 1) + (C > 2) + (C > 4)];
    const double thr = a[0] + a[1] * rays + a[2] * conv + a[3] * pix + a[4] * cell + a[5] * crowd + a[6] * fine;
    return {lat, thr, nt > NTHREADS ? lat : std::max(lat, 2.0 * thr / C)};
}

// dynamic shared memory of a cluster-kernel CTA: two CTAs of 256 threads share
// an SM, one of 512 has it alone
inline int cluster_smem_limit(const mirage_ctx* ctx, int nt) {
    return nt > NTHREADS ? ctx->max_smem - 1024 : std::min(ctx->max_smem, ctx->max_smem_sm / 2 - 1024);
}

template <typename T>
bool cluster_fits(const mirage_ctx* ctx, const Prob<T>& P, int C, ClusterPlan& out) {
    if constexpr (sizeof(T) == 4) {
        // one ray per pixel with four corners, a compiled PSF width
        if (P.Np != 1 || P.interp == MIRAGE_INTERP_BICUBIC || P.fft_m || P.K >= MAX_K || !table().cluster[P.K][0])
            return false;
        const ClusterCut u(P, C, cluster_smem_limit(ctx, ClusterCut(P, C, 0).nt));
        // halos reach the next band only; ring positions have 20 bits
        if (C > 1 && (u.bt * TILE < P.hk || P.tiles_y < C || P.sy < C)) return false;
        if (u.blen >= (1 << 20)) return false;
        const size_t b = u.bytes(P);
        if (b > (size_t)ctx->max_smem) return false;
        out.C = C;
        out.nt = u.nt;
        out.fn = table().cluster[P.K][u.nt > NTHREADS];
        out.smem = b;
        out.slab = (long long)cluster_slab_bytes(P);
        return true;
    }
    return false;
}

// clusters of `C` CTAs with `smem` bytes each that the device holds at once,
// less the caller's reserved slots
int cluster_slots(mirage_ctx* ctx, const void* fn, int C, int nt, size_t smem, int* out) {
    const auto key = std::make_pair(fn, std::make_pair(C, smem));
    auto it = ctx->cl_active.find(key);
    if (it == ctx->cl_active.end()) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(nt);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        CK(cudaOccupancyMaxActiveClusters(&n, fn, &cfg));
        it = ctx->cl_active.emplace(key, std::max(1, n)).first;
    }
    *out = std::max(1, it->second - (ctx->reserved + C - 1) / C);
    return MIRAGE_OK;
}

int launch_cluster(mirage_ctx* ctx, const void* fn, int clusters, int C, int nt, void** args, size_t smem,
                   cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)clusters * C);
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    CK(cudaLaunchKernelExC(&cfg, fn, args));
    ctx->last_launches++;
    return MIRAGE_OK;
}

// fast-kernel arguments (FP32 contexts only; never called for double)
template <typename T>
void set_fast_args(FastArgs& fa, const CglsArgs<T>& A) {
    if constexpr (sizeof(T) == 4) std::memcpy(&fa.A, &A, sizeof(A));
}

template <typename T>
void fill_scratch(CandScratch<T>& cs, mirage_ctx* ctx, bool fwd, long long sE, long long sInv, long long sCst,
                  long long sPad) {
    cs.E = (fwd ? ctx->fE : ctx->E).as<Entry<T>>();
    cs.E64 = sizeof(T) == 8 ? reinterpret_cast<Entry<double>*>(cs.E) : (fwd ? ctx->fE64 : ctx->E64).as<Entry<double>>();
    cs.Etmp = (fwd ? ctx->fEtmp : ctx->Etmp).as<Entry<double>>();
    cs.inv = (fwd ? ctx->finv : ctx->inv).as<int>();
    cs.cst = (fwd ? ctx->fcst : ctx->cst).as<int>();
    cs.swp = (fwd ? ctx->fswp : ctx->swp).as<T>();
    cs.dpad = (fwd ? ctx->fdpad : ctx->dpad).as<T>();
    cs.nent = (fwd ? ctx->fnent : ctx->nent).as<int>();
    cs.cstat = (fwd ? ctx->fcstat : ctx->cstat).as<int>();
    cs.sE = sE;
    cs.sInv = sInv;
    cs.sCst = sCst;
    cs.sPad = sPad;
}

int launch(mirage_ctx* ctx, const void* fn, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t st) {
    CK(cudaLaunchKernel(fn, grid, block, args, smem, st));
    ctx->last_launches++;
    return MIRAGE_OK;
}

// asynchronous upload of small host arrays through the context's pinned
// staging buffer (a pageable source would make the copy synchronise the
// stream); the host arrays may go away as soon as this returns
struct UploadPart {
    void* dst;
    const void* src;
    size_t bytes;
};
int upload(mirage_ctx* ctx, cudaStream_t st, std::initializer_list<UploadPart> parts) {
    size_t total = 0;
    for (const UploadPart& u : parts) total += (u.bytes + 15) / 16 * 16;
    if (ctx->pin_pending) {
        CK(cudaEventSynchronize(ctx->pin_ev));  // the previous call's copies have left the buffer
        ctx->pin_pending = false;
    }
    if (!ctx->pin_ev) CK(cudaEventCreateWithFlags(&ctx->pin_ev, cudaEventDisableTiming));
    if (total > ctx->pin_n) {
        if (ctx->pin) cudaFreeHost(ctx->pin);
        ctx->pin = nullptr;
        ctx->pin_n = 0;
        const size_t want = std::max<size_t>(total, 1 << 16);
        if (cudaHostAlloc(&ctx->pin, want, cudaHostAllocDefault) != cudaSuccess) {
            ctx->pin = nullptr;
            set_error("cudaHostAlloc(%zu) failed", want);
            return MIRAGE_ERR_NOMEM;
        }
        ctx->pin_n = want;
    }
    size_t off = 0;
    for (const UploadPart& u : parts) {
        if (!u.bytes) continue;
        char* h = static_cast<char*>(ctx->pin) + off;
        std::memcpy(h, u.src, u.bytes);
        CK(cudaMemcpyAsync(u.dst, h, u.bytes, cudaMemcpyHostToDevice, st));
        off += (u.bytes + 15) / 16 * 16;
    }
    CK(cudaEventRecord(ctx->pin_ev, st));
    ctx->pin_pending = true;
    return MIRAGE_OK;
}

// ray trace of candidates [cand0, cand0 + n_cand): many CTAs trace and one per
// candidate places the rays where their numbers fit in shared memory; larger
// images: one CTA per candidate, or, for fewer candidates than SMs, the split
// trace (many CTAs per candidate trace and count, one per candidate places)
template <typename T>
int launch_raytrace(mirage_ctx* ctx, const Prob<T>* dprobs, const int* dcand, const double* d_lens, int cand0,
                    int n_cand, const CandScratch<T>& cs, long long max_cells, long long max_npix, long long max_rays, cudaStream_t st);

#define TRY(x)                      \
    do {                            \
        int r_ = (x);               \
        if (r_ != MIRAGE_OK) return r_; \
    } while (0)

// staging of host arrays into one device block (MIRAGE_MEM_HOST)
struct Stager {
    std::vector<std::pair<size_t, std::pair<const void*, size_t>>> in;  // offset, (host ptr, bytes)
    std::vector<std::pair<size_t, std::pair<void*, size_t>>> out;
    size_t total = 0;
    size_t add_in(const void* h, size_t bytes) {
        const size_t o = total;
        total += (bytes + 255) / 256 * 256;
        if (h && bytes) in.push_back({o, {h, bytes}});
        return o;
    }
    size_t add_out(void* h, size_t bytes) {
        const size_t o = total;
        total += (bytes + 255) / 256 * 256;
        if (h && bytes) out.push_back({o, {h, bytes}});
        return o;
    }
};

template <typename T>
int launch_raytrace(mirage_ctx* ctx, const Prob<T>* dprobs, const int* dcand, const double* d_lens, int cand0,
                    int n_cand, const CandScratch<T>& cs, long long max_cells, long long max_npix, long long max_rays, cudaStream_t st) {
    constexpr int prec = prec_of<T>();
    const KernelTable& tb = table();
    const size_t cells_smem = (size_t)max_cells * 4;
    // Ray numbers in shared memory: two launches (one 64 x 64 candidate: 15 + 35 us;
    // a whole forward call on it 282 -> 91 us against the trace on one CTA).  The
    // CTAs of the trace take at least RT_MIN_PIX pixels, and there are no more of them
    // than the device holds at once (16 of 128 threads an SM).  Decided on the call's
    // largest problem: where its rays do not fit, all candidates take the forms below
    const size_t place_smem = sizeof(int) * (size_t)(max_cells + max_rays);
    if (place_smem <= (size_t)ctx->max_smem - 2048 && n_cand <= 65535) {
        constexpr long long RT_MIN_PIX = 32;
        long long chunk_l = std::max(RT_MIN_PIX, (max_npix * n_cand + 16 * ctx->sm_count - 1) / (16 * ctx->sm_count));
        int chunk = (int)std::min<long long>(chunk_l, RT_THREADS);
        const long long per = std::max<long long>(1, std::min((max_npix + chunk - 1) / chunk, (16LL * ctx->sm_count + n_cand - 1) / n_cand));
        int c0 = cand0;
        CandScratch<T> csv = cs;
        void* a1[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &chunk, &csv};
        TRY(launch(ctx, tb.rt_rays[prec], dim3((unsigned)per, n_cand), dim3(RT_THREADS), a1, 0, st));
        TRY(set_smem(ctx, tb.rt_cells[prec], place_smem));
        void* a2[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &csv};
        return launch(ctx, tb.rt_cells[prec], dim3(n_cand), dim3(RT_PLACE_THREADS), a2, place_smem, st);
    }
    if (n_cand < ctx->sm_count && max_npix >= 128 * 128) {
        const int chunk = 2 * NTHREADS;
        const int n_chunks = (int)((max_npix + chunk - 1) / chunk);
        CK(cudaMemsetAsync(cs.swp + (long long)cand0 * cs.sPad, 0, sizeof(T) * cs.sPad * n_cand, st));
        CK(cudaMemsetAsync(cs.dpad + (long long)cand0 * cs.sPad, 0, sizeof(T) * cs.sPad * n_cand, st));
        CK(cudaMemsetAsync(cs.cst + (long long)cand0 * cs.sCst, 0, sizeof(int) * cs.sCst * n_cand, st));
        CK(cudaMemsetAsync(cs.cstat + cand0, 0, sizeof(int) * n_cand, st));
        int c0 = cand0, ch = chunk;
        CandScratch<T> csv = cs;
        void* a1[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &ch, &csv};
        TRY(launch(ctx, tb.rt_trace[prec], dim3(n_chunks, n_cand), dim3(NTHREADS), a1, 0, st));
        TRY(set_smem(ctx, tb.rt_place[prec], cells_smem));
        void* a2[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &csv};
        TRY(launch(ctx, tb.rt_place[prec], dim3(n_cand), dim3(NTHREADS), a2, cells_smem, st));
        // one ray per pixel: parallel placement (the place kernel only scanned)
        TRY(ctx->rt_cursor.ensure(sizeof(int) * (size_t)cs.sCst * (cand0 + n_cand)));
        int* cur = ctx->rt_cursor.as<int>();
        long long cstr = cs.sCst;
        CK(cudaMemsetAsync(cur + (long long)cand0 * cstr, 0, sizeof(int) * cstr * n_cand, st));
        void* a3[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &ch, &csv, (void*)&cur, &cstr};
        TRY(launch(ctx, tb.rt_scatter[prec], dim3(n_chunks, n_cand), dim3(NTHREADS), a3, 0, st));
        void* a4[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &csv};
        return launch(ctx, tb.rt_sortcells[prec], dim3((unsigned)((max_cells + NTHREADS - 1) / NTHREADS), n_cand),
                      dim3(NTHREADS), a4, 0, st);
    }
    TRY(set_smem(ctx, tb.raytrace[prec], cells_smem));
    int c0 = cand0, nc = n_cand;
    CandScratch<T> csv = cs;
    void* args[] = {(void*)&dprobs, (void*)&dcand, (void*)&d_lens, &c0, &nc, &csv};
    return launch(ctx, tb.raytrace[prec], dim3(n_cand), dim3(NTHREADS), args, cells_smem, st);
}

// work item of the CGLS kernels: lambdas k_first..k_last of candidate c,
// solved in order by one CTA (see ChainPos)
inline int pack_chain(int c, int k_first, int k_last) { return (c * MAX_LAM + k_first) * MAX_LAM + k_last; }

template <typename T>
int eval_impl(mirage_ctx* ctx, const mirage_problem_t* probs, int n_probs, const double* lens, const int* prob_idx,
              int n_cand, const double* lambdas, const int* n_lam, int max_lam, const mirage_opts_t* opts,
              const void* warm_x, const int* lam_start, double* chi2, double* reg, int* iters, double* relres, int* item_status,
              int* corner, double* kappa, void* s_out, void* all_x, int* status, cudaStream_t st) {
    constexpr int prec = prec_of<T>();
    ctx->last_launches = 0;
    if (n_cand == 0) return MIRAGE_OK;
    if (!probs || n_probs < 1 || !lens || !prob_idx || !lambdas || !n_lam || !chi2 || !reg || !iters || !corner ||
        !status || max_lam < 1 || max_lam > MAX_LAM || n_cand < 0 || n_cand > INT_MAX / (MAX_LAM * MAX_LAM) - 1) {
        set_error("eval_batch: null pointer or size out of range");
        return MIRAGE_ERR_ARG;
    }
    const mirage_opts_t o = *opts;
    if (!(o.tol >= 0) || o.mode < 0 || o.mode > 1 || o.mem < 0 || o.mem > 1 || o.variant < 0 || o.variant > 7 ||
        !(o.inner_eta == 0.0 || (o.inner_eta >= 1e-4 && o.inner_eta <= 0.5)) || o.place < 0 || o.place > 5) {
        set_error("eval_batch: bad options");
        return MIRAGE_ERR_ARG;
    }
    for (int p = 0; p < n_probs; ++p) {
        if (check_geom(probs[p].geom) != MIRAGE_OK) {
            set_error("eval_batch: bad geometry of problem %d", p);
            return MIRAGE_ERR_ARG;
        }
        if (!probs[p].d || !probs[p].sigma || !probs[p].mask || !probs[p].psf) {
            set_error("eval_batch: null data pointer in problem %d", p);
            return MIRAGE_ERR_ARG;
        }
    }
    for (int c = 0; c < n_cand; ++c) {
        if (prob_idx[c] < 0 || prob_idx[c] >= n_probs || n_lam[c] < 1 || n_lam[c] > max_lam) {
            set_error("eval_batch: bad prob_idx / n_lam of candidate %d", c);
            return MIRAGE_ERR_ARG;
        }
    }
    const bool host = o.mem == MIRAGE_MEM_HOST;

    // sizes over the problems
    std::vector<Prob<T>> hp(n_probs);
    long long max_rays = 0, max_cells = 0, max_plen = 0, max_ns = 0, max_npix = 0;
    long long spec_stride = 0;
    for (int p = 0; p < n_probs; ++p) {
        hp[p] = make_prob<T>(probs[p], probs[p].d, probs[p].sigma, probs[p].mask, probs[p].psf);
        plan_fft<T>(ctx, hp[p], o.variant);
        if (hp[p].fft_m)
            spec_stride = std::max<long long>(spec_stride, (long long)((hp[p].fft_m >> 1) + 1) * hp[p].fft_m);
        max_npix = std::max<long long>(max_npix, hp[p].npix);
        max_rays = std::max<long long>(max_rays, hp[p].nrays);
        max_cells = std::max<long long>(max_cells, hp[p].ncells);
        max_plen = std::max<long long>(max_plen, hp[p].plen);
        max_ns = std::max<long long>(max_ns, hp[p].ns);
    }
    if ((long long)max_cells * 4 > ctx->max_smem - 2048) {
        set_error("source grid too large for the ray-trace kernel");
        return MIRAGE_ERR_UNSUPPORTED;
    }
    const long long sE = max_rays, sInv = max_rays, sCst = (max_cells + 1 + 3) / 4 * 4, sPad = (max_plen + 3) / 4 * 4;
    const long long nitems_all = (long long)n_cand * max_lam;

    // host staging: every array of the call goes through one device block
    const double* d_lens = lens;
    const double* d_lambdas = lambdas;
    const T* d_warm = reinterpret_cast<const T*>(warm_x);
    double *d_chi2 = chi2, *d_reg = reg, *d_relres = relres, *d_kappa = kappa;
    int *d_iters = iters, *d_istat = item_status, *d_corner = corner, *d_status = status;
    T *d_sout = reinterpret_cast<T*>(s_out), *d_allx = reinterpret_cast<T*>(all_x);
    if (host) {
        Stager sg;
        std::vector<size_t> po(4 * n_probs);
        for (int p = 0; p < n_probs; ++p) {
            const mirage_geom_t& g = probs[p].geom;
            const size_t np = (size_t)g.nx * g.ny;
            po[4 * p + 0] = sg.add_in(probs[p].d, np * sizeof(T));
            po[4 * p + 1] = sg.add_in(probs[p].sigma, np * sizeof(T));
            po[4 * p + 2] = sg.add_in(probs[p].mask, np);
            po[4 * p + 3] = sg.add_in(probs[p].psf, (size_t)g.kpsf * g.kpsf * sizeof(T));
        }
        const size_t o_lens = sg.add_in(lens, sizeof(double) * 7 * n_cand);
        const size_t o_lam = sg.add_in(lambdas, sizeof(double) * max_lam * n_cand);
        const size_t o_warm = sg.add_in(warm_x, warm_x ? sizeof(T) * nitems_all * max_ns : 0);
        const size_t o_chi2 = sg.add_out(chi2, sizeof(double) * nitems_all);
        const size_t o_reg = sg.add_out(reg, sizeof(double) * nitems_all);
        const size_t o_it = sg.add_out(iters, sizeof(int) * nitems_all);
        const size_t o_rr = sg.add_out(relres, relres ? sizeof(double) * nitems_all : 0);
        const size_t o_is = sg.add_out(item_status, item_status ? sizeof(int) * nitems_all : 0);
        const size_t o_cn = sg.add_out(corner, sizeof(int) * n_cand);
        const size_t o_kp = sg.add_out(kappa, kappa ? sizeof(double) * nitems_all : 0);
        const size_t o_so = sg.add_out(s_out, s_out ? sizeof(T) * n_cand * max_ns : 0);
        const size_t o_ax = sg.add_out(all_x, all_x ? sizeof(T) * nitems_all * max_ns : 0);
        const size_t o_st = sg.add_out(status, sizeof(int) * n_cand);
        TRY(ctx->stage.ensure(sg.total));
        char* base = ctx->stage.as<char>();
        for (auto& e : sg.in) CK(cudaMemcpyAsync(base + e.first, e.second.first, e.second.second, cudaMemcpyHostToDevice, st));
        for (int p = 0; p < n_probs; ++p)
            hp[p] = make_prob<T>(probs[p], base + po[4 * p], base + po[4 * p + 1], base + po[4 * p + 2],
                                 base + po[4 * p + 3]);
        d_lens = reinterpret_cast<const double*>(base + o_lens);
        d_lambdas = reinterpret_cast<const double*>(base + o_lam);
        d_warm = warm_x ? reinterpret_cast<const T*>(base + o_warm) : nullptr;
        d_chi2 = reinterpret_cast<double*>(base + o_chi2);
        d_reg = reinterpret_cast<double*>(base + o_reg);
        d_iters = reinterpret_cast<int*>(base + o_it);
        d_relres = relres ? reinterpret_cast<double*>(base + o_rr) : nullptr;
        d_istat = item_status ? reinterpret_cast<int*>(base + o_is) : nullptr;
        d_corner = reinterpret_cast<int*>(base + o_cn);
        d_kappa = kappa ? reinterpret_cast<double*>(base + o_kp) : nullptr;
        d_sout = s_out ? reinterpret_cast<T*>(base + o_so) : nullptr;
        d_allx = all_x ? reinterpret_cast<T*>(base + o_ax) : nullptr;
        d_status = reinterpret_cast<int*>(base + o_st);
        // run on device buffers, then copy back
        mirage_opts_t o2 = o;
        o2.mem = MIRAGE_MEM_DEVICE;
        o2.use_graph = 0;
        std::vector<mirage_problem_t> dp(probs, probs + n_probs);
        for (int p = 0; p < n_probs; ++p) {
            dp[p].d = base + po[4 * p];
            dp[p].sigma = base + po[4 * p + 1];
            dp[p].mask = reinterpret_cast<const uint8_t*>(base + po[4 * p + 2]);
            dp[p].psf = base + po[4 * p + 3];
        }
        TRY(eval_impl<T>(ctx, dp.data(), n_probs, d_lens, prob_idx, n_cand, d_lambdas, n_lam, max_lam, &o2, d_warm,
                         lam_start, d_chi2, d_reg, d_iters, d_relres, d_istat, d_corner, d_kappa, d_sout, d_allx, d_status,
                         st));
        const int nl = ctx->last_launches;
        for (auto& e : sg.out) CK(cudaMemcpyAsync(e.second.first, base + e.first, e.second.second, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        ctx->last_launches = nl;
        return MIRAGE_OK;
    }

    // ---- device path
    TRY(ctx->E.ensure(sizeof(Entry<T>) * n_cand * sE));
    if (sizeof(T) == 4) TRY(ctx->E64.ensure(sizeof(Entry<double>) * n_cand * sE));
    TRY(ctx->Etmp.ensure(sizeof(Entry<double>) * n_cand * sE));
    TRY(ctx->inv.ensure(sizeof(int) * n_cand * sInv));
    TRY(ctx->cst.ensure(sizeof(int) * n_cand * sCst));
    TRY(ctx->swp.ensure(sizeof(T) * n_cand * sPad));
    TRY(ctx->dpad.ensure(sizeof(T) * n_cand * sPad));
    TRY(ctx->nent.ensure(sizeof(int) * n_cand));
    TRY(ctx->cstat.ensure(sizeof(int) * n_cand));
    if (!d_allx) TRY(ctx->X.ensure(sizeof(T) * nitems_all * max_ns));
    if (!d_istat) TRY(ctx->istat.ensure(sizeof(int) * nitems_all));
    T* dX = d_allx ? d_allx : ctx->X.as<T>();
    int* dIst = d_istat ? d_istat : ctx->istat.as<int>();

    // per-candidate kernel class and work items
    std::vector<int> cls_of(n_probs);
    struct Group {
        const void* fn;
        bool fast = false;
        int cl = 0, nt = NTHREADS;  // cluster kernel: CTAs per item, threads a CTA
        int prob = -1;   // the single problem of the group, -2 if several
        int per_sm = 1;  // resident CTAs per SM
        long long slots = 0;  // CTAs (clusters) of the persistent launch
        double load = 0.0;     // estimated clocks of its items, one after another
        double longest = 0.0;  // estimated clocks of its longest item
        size_t smem = 0;
        long long slab = 0;
        std::vector<std::pair<double, int>> items;  // (sort key, packed)
    };
    std::map<std::pair<const void*, int>, Group> groups;
    std::vector<double> hlam;  // lambdas are device data: sort by index instead (ascending lambda = costlier)
    // kernel choice per problem: parameter taps need one PSF per launch
    std::vector<int> cands_of(n_probs, 0);
    for (int c = 0; c < n_cand; ++c) cands_of[prob_idx[c]]++;
    int n_used = 0;
    for (int p = 0; p < n_probs; ++p) n_used += cands_of[p] > 0;
    const int want = o.variant;
    long long n_items = 0;
    for (int c = 0; c < n_cand; ++c) n_items += n_lam[c];
    // no more items than SMs (or one candidate at a time): each CTA has an SM
    const bool alone = n_items <= ctx->sm_count || o.mode == MIRAGE_MODE_PLAIN;
    auto choose = [&](const Prob<T>& P, int& mode, bool& fast) -> const void* {
        fast = false;
        mode = 0;
        if (want == 4 || want == 6 || P.fft_m) return nullptr;
        int m = 1;                         // automatic: parameter taps (FFMA) when one PSF (measured
                                           // 7% faster than packed FFMA2 on the 64x64 workload)
        if (want == 1) m = 0;
        if (want == 2) m = 1;
        if (want == 3) m = 2;
        if (want == 7) m = 3;
        if (m > 0 && (n_used > 1 || P.K * P.K > MAX_PTAP)) m = 0;
        const void* f = pick_fast<T>(ctx, P, m, alone);
        if (!f && m == 1 && want == 0) {  // FFMA parameter taps are compiled for K = 9 only
            m = 2;
            f = pick_fast<T>(ctx, P, 2, alone);
        }
        if (!f && m > 0) {
            m = 0;
            f = pick_fast<T>(ctx, P, 0, alone);
        }
        if (f) {
            fast = true;
            mode = m;
        }
        return f;
    };
    // Kernel of the items that the two-CTA kernel does not take, unless a kernel
    // or a placement of the general kernel is asked for: the general kernel, or the
    // cluster kernel on 1, 2, 4 or 8 SMs.  All forms give the same bits.  (48 x 48 image
    // and source, K = 15: one item takes 23.7 us an iteration in the general kernel and
    // 13.8 on eight SMs; 304 such items 25 ms in the general kernel and 33 on
    // clusters of four)
    struct Form {
        IterCost it;
        ClusterPlan cp;  // C = 0: general or two-CTA kernel
    };
    // what a problem's items have in common
    struct ProbPlan {
        std::vector<Form> forms;  // [0]: without clusters; all by SM time an iteration, least first, in order
        std::vector<int> order;
        int quick = 0;            // the form with the shortest iteration
        double iters = 1.0;       // iterations of an item, relative to other problems'
        const void* fn = nullptr;  // the kernel without clusters, its shared memory, slab, CTAs per SM
        size_t smem = 0;
        long long slab = 0;
        int per_sm = 1, mode = 0;
        bool fast = false, big = false;
    };
    std::vector<ProbPlan> plan(n_probs);
    bool choice = false;  // some problem has several forms
    for (int p = 0; p < n_probs; ++p) {
        if (!cands_of[p]) continue;
        const Prob<T>& P = hp[p];
        ProbPlan& q = plan[p];
        int place = pick_place<T>(ctx, P, o.place);
        // FP64, everything in shared memory: two CTAs per SM (128 registers a
        // thread) where two fit and there are many items a slot.  At 32 x 32, 256
        // candidates x 10 lambdas took 159 ms with two and 191 with one, 64
        // candidates 55.5 and 48.9: with few items the longest one's time counts
        if (sizeof(T) == 8 && place == PLACE_SMEM && o.place == 0 && o.mode == MIRAGE_MODE_BATCHED &&
            n_items >= 8LL * ctx->sm_count && 2 * ((long long)smem_bytes<T>(P, PLACE_SMEM) + 1024) <= ctx->max_smem_sm)
            place = PLACE_SMEM2;
        q.big = place != PLACE_SMEM;
        q.fn = pick_cgls(prec, place, P.fft_m ? 0 : P.K);
        q.smem = smem_bytes<T>(P, layout_of(place));
        q.slab = (long long)slab_bytes<T>(P, layout_of(place));
        q.per_sm = two_per_sm(place) ? 2 : 1;
        if (const void* ff = choose(P, q.mode, q.fast)) {
            q.fn = ff;
            q.smem = fast_smem_bytes(*reinterpret_cast<const Prob<float>*>(&P));
            q.slab = (long long)fast_slab_bytes(*reinterpret_cast<const Prob<float>*>(&P));
            q.per_sm = 2;
        }
        q.forms.push_back(Form{q.fast ? fast_cost(P) : general_cost(P, place), ClusterPlan()});
        if constexpr (sizeof(T) == 4) {
            if (!q.fast && o.place == 0 && want != 4 && want != 5 && want != 6)
                for (int C = 1; C <= CL_MAX; C *= 2) {
                    Form x;
                    if (!cluster_fits<T>(ctx, P, C, x.cp)) continue;
                    x.it = cluster_cost(P, C, x.cp.nt);
                    q.forms.push_back(x);
                }
        }
        for (int i = 0; i < (int)q.forms.size(); ++i) {
            q.order.push_back(i);
            if (q.forms[i].it.lat < q.forms[q.quick].it.lat) q.quick = i;
        }
        std::stable_sort(q.order.begin(), q.order.end(), [&](int a, int b) { return q.forms[a].it.thr < q.forms[b].it.thr; });
        choice |= q.forms.size() > 1;
        // (25 to 36 at K = 3, 110 at 9, 170 at 15, 360 to 560 at 21, for PSFs of K / 6
        // pixels at one lambda; sources of 256 and 2304 pixels: 1 to 1.4)
        q.iters = P.K * std::pow((double)P.ns, 0.15);
    }
    // candidates of one problem and lambda count are alike: their items' forms and
    // groups are looked up once, and the weights of an n-point grid made once
    // (a map look-up and two powers an item took 90 us of a call of 256 x 16)
    struct Class {
        int p = 0, n = 0, count = 0;
        std::vector<const Form*> form;  // by lambda
        std::vector<Group*> group;
    };
    std::map<std::pair<int, int>, Class> classes;
    std::vector<Class*> class_of(n_cand);
    std::vector<std::vector<double>> weight(max_lam + 1);
    // iteration counts for estimates, by how they may fall from the smallest lambda
    // to the largest (see estimate)
    constexpr double FALL[2] = {0.8, 2.0};
    std::vector<std::vector<double>> fall[2];
    for (auto& f : fall) f.resize(max_lam + 1);
    for (int c = 0; c < n_cand; ++c) {
        Class*& cl = class_of[c];
        if (c > 0 && prob_idx[c] == prob_idx[c - 1] && n_lam[c] == n_lam[c - 1]) {
            cl = class_of[c - 1];
        } else {
            cl = &classes[{prob_idx[c], n_lam[c]}];
            cl->p = prob_idx[c];
            cl->n = n_lam[c];
        }
        cl->count++;
        const int n = n_lam[c];
        for (int k = (int)weight[n].size(); k < n; ++k) {
            weight[n].push_back(chain_weight(n, k));
            for (int j = 0; j < 2; ++j)
                fall[j][n].push_back(chain_weight(n, 0) * std::pow(10.0, -FALL[j] * k / std::max(1, n - 1)));
        }
    }
    // forms of some classes' items where an item may take `limit` clocks: the one of
    // least SM time that takes no longer, or else the quickest.  Without `each`, one
    // form for all items of a class (that of the smallest lambda's); limit < 0: no
    // clusters.  False once a larger limit changes nothing more
    typedef std::vector<Class*> Classes;
    const bool chains = lam_start && o.mode == MIRAGE_MODE_BATCHED;
    auto set_forms = [&](const Classes& some, double limit, bool each) {
        bool more = false;
        for (Class* cl : some) {
            const ProbPlan& q = plan[cl->p];
            cl->form.resize(cl->n);
            for (int k = 0; k < cl->n; ++k) {
                if (k > 0 && !each) {
                    cl->form[k] = cl->form[0];
                    continue;
                }
                const double w = q.iters * weight[cl->n][k];
                int f = limit < 0.0 ? 0 : q.quick;
                if (limit >= 0.0)
                    for (int i : q.order)
                        if (w * q.forms[i].it.lat <= limit) {
                            f = i;
                            break;
                        }
                more |= f != q.order[0];
                cl->form[k] = &q.forms[f];
            }
        }
        return more;
    };
    // Estimated clocks of the classes' items with these forms: the longest item (1.15
    // of the mean over candidates, up to 2 where problems differ, 2 in chains, which hold
    // several lambdas), or the work on all SMs, and
    // part of the other one, since the end of a call is never packed full.  How iteration
    // counts fall with lambda depends on the grid's values, which are device data: the
    // estimate is the geometric mean over counts that fall by 10^0.8 and by 10^2 from
    // the smallest lambda to the largest.  (Against the general kernel alone: 120 drawn
    // calls of 28 to 100 pixels a side and 1 to 128 candidates 1.40 times as fast in the
    // mean, the slowest 0.85; 14 calls of 12 to 400 unlike problems 1.3 to 4.1 times.)
    const double unlike = std::min(1.0, 0.125 * (n_used - 1));  // nine problems and more: 1
    double call_time = 0.0;                                     // (with the second)
    auto estimate = [&](const Classes& some, bool together) {
        double e = 0.0;
        bool cluster = false;
        for (const auto& ws : fall) {
            double sum = 0.0, alone = 0.0, busy = 0.0;
            for (const Class* cl : some) {
                const double it = plan[cl->p].iters;
                for (int k = 0; k < cl->n; ++k) {
                    const double w = it * ws[cl->n][k];
                    sum += (together ? cl->count : 1) * w * cl->form[k]->it.thr / ctx->sm_count;
                    alone = std::max(alone, w * cl->form[k]->it.lat);
                    busy = std::max(busy, w * cl->form[k]->it.busy);
                    cluster |= cl->form[k]->cp.C > 0 && !plan[cl->p].big;
                }
            }
            const double full = 0.5 * std::min(1.0, sum / busy);  // its part beside others
            const double longest = ((1.0 - full) * alone + full * busy) * (chains ? 2.0 : 1.15 + 0.85 * unlike);
            e += 0.5 * std::log(std::max(sum, longest) + 0.3 * std::min(sum, longest));
            call_time = std::max(sum, longest);
        }
        // clusters in place of the general kernel with everything in shared memory have to
        // be better by 1.1
        return e + (cluster ? 0.1 : 0.0);
    };
    auto search = [&](const Classes& some, bool together, bool mixed) {
        set_forms(some, -1.0, false);
        double best = estimate(some, together), limit = -1.0;
        const double first = call_time;
        bool each = false;
        for (int m = 0; m <= (int)mixed; ++m)
            for (double T_ = 0.0, more = 1.0; more; T_ = std::max(1.5 * T_, 0.1 * first)) {
                more = set_forms(some, T_, m == 1);
                // a plan that mixes the forms of one problem has to be better by 1.02 (forms
                // in turn hold each other up); with many unlike problems and few items a SM
                // it may be worse by 1.05
                const double e = estimate(some, together) + (n_items < 8LL * ctx->sm_count ? 0.02 - 0.07 * unlike : 0.02) * m;
                if (e < best) {
                    best = e;
                    limit = T_;
                    each = m == 1;
                }
            }
        set_forms(some, limit, each);
    };
    Classes all;
    for (auto& kv : classes) all.push_back(&kv.second);
    if (!choice) {
        set_forms(all, -1.0, false);
    } else if (o.mode == MIRAGE_MODE_PLAIN) {  // one candidate at a time
        for (Class* cl : all) search(Classes(1, cl), false, false);
    } else {
        search(all, true, !chains);  // (a chain's items share a kernel)
    }
    if (all.size() > 1 || choice) estimate(all, true);
    // groups: items of one kernel (and cluster size) share a launch
    std::fill(ctx->last_kernels, ctx->last_kernels + MIRAGE_N_ITEM_KERNELS, 0);
    for (auto& kv : classes) {
        Class& cl = kv.second;
        const ProbPlan& q = plan[cl.p];
        const std::vector<double>& w = weight[cl.n];
        cl.group.resize(cl.n);
        for (int k = 0; k < cl.n; ++k) {
            const Form& form = *cl.form[k];
            const ClusterPlan& cp = form.cp;
            const void* f = cp.C ? cp.fn : q.fn;
            if (!f) {
                set_error("no kernel for this PSF size");
                return MIRAGE_ERR_UNSUPPORTED;
            }
            Group*& gp = cl.group[k];
            if (k > 0 && cl.form[k] == cl.form[k - 1])
                gp = cl.group[k - 1];
            else
                gp = &groups[std::make_pair(f, cp.C ? 16 + cp.C : (int)q.big)];
            Group& g = *gp;
            g.fn = f;
            g.fast = q.fast;
            g.cl = cp.C;
            g.nt = cp.C ? cp.nt : NTHREADS;
            g.prob = (g.prob == -1 || g.prob == cl.p) ? cl.p : -2;
            g.per_sm = q.per_sm;
            g.smem = std::max(g.smem, cp.C ? cp.smem : q.smem);
            g.slab = std::max<long long>(g.slab, cp.C ? cp.slab : q.slab);
            g.load += cl.count * q.iters * w[k] * form.it.lat;
            g.longest = std::max(g.longest, q.iters * w[k] * form.it.lat);
            ctx->last_kernels[cp.C ? 3 + (cp.C > 1) + (cp.C > 2) + (cp.C > 4) : q.fast ? 0 : hp[cl.p].fft_m ? 2 : 1] += cl.count;
        }
    }
    // chained calls: each CTA slot's share of the estimated cost of the call
    double chain_budget = 0.0;
    if (lam_start) {
        double tw = 0.0;
        for (auto& kv : classes) {
            const Prob<T>& P = hp[kv.second.p];
            const double work = (double)P.plen * P.K * P.K + 8.0 * P.nrays;
            for (double wk : weight[kv.second.n]) tw += kv.second.count * work * wk;
        }
        chain_budget = tw / (double)cgls_slots(ctx, 2);
    }
    for (int c = 0; c < n_cand; ++c) {
        const Prob<T>& P = hp[prob_idx[c]];
        const std::vector<Group*>& group = class_of[c]->group;
        const double work = (double)P.plen * P.K * P.K + 8.0 * P.nrays;
        // lambda grids ascend: smaller k = smaller lambda = more CG iterations
        auto cost_of = [&](int k) { return work * (double)(n_lam[c] - k + 4); };
        if (lam_start) {
            // chains from the predicted corner: down to the smallest lambda,
            // and up from the next one.  A chain is cut into segments (each
            // further segment starts cold) whose estimated cost stays within
            // one CTA slot's share of the whole call, so that no work unit
            // outlasts the persistent queue's balance.  Costs follow the
            // iteration counts of log-spaced grids, which grow geometrically
            // towards small lambda
            const int ks = std::min(std::max(lam_start[c], 0), n_lam[c] - 1);
            const std::vector<double>& w = weight[n_lam[c]];
            auto wk = [&](int k) { return work * w[k]; };
            auto push_run = [&](int ka, int kb, double cd) {
                group[0]->items.push_back({-cd, pack_chain(c, ka, kb)});
            };
            int ka = ks;
            double cd = 0.0;
            for (int k = ks; k >= 0; --k) {
                if (k < ka && cd + wk(k) > chain_budget) {
                    push_run(ka, k + 1, cd);
                    ka = k;
                    cd = 0.0;
                }
                cd += wk(k);
            }
            push_run(ka, 0, cd);
            if (ks + 1 < n_lam[c]) {
                ka = ks + 1;
                cd = 0.0;
                for (int k = ks + 1; k < n_lam[c]; ++k) {
                    if (k > ka && cd + wk(k) > chain_budget) {
                        push_run(ka, k - 1, cd);
                        ka = k;
                        cd = 0.0;
                    }
                    cd += wk(k);
                }
                push_run(ka, n_lam[c] - 1, cd);
            }
        } else {
            for (int k = 0; k < n_lam[c]; ++k) group[k]->items.push_back({-cost_of(k), pack_chain(c, k, k)});
        }
    }
    std::vector<int> all_items;
    std::vector<size_t> g_off;
    std::vector<Group*> glist;
    for (auto& kv : groups) glist.push_back(&kv.second);
    // the others fill in behind the first group's tail: where the groups share the device
    // (see the launches), first the group with the longest item, otherwise the one
    // with the most work
    bool shared = n_items < 4LL * ctx->sm_count;
    for (Group* g : glist) shared |= g->cl > 0;
    std::stable_sort(glist.begin(), glist.end(), [&](const Group* a, const Group* b) {
        return shared ? a->longest > b->longest : a->load > b->load;
    });
    for (Group* gp : glist) {
        Group& g = *gp;
        std::stable_sort(g.items.begin(), g.items.end(),
                         [](const std::pair<double, int>& a, const std::pair<double, int>& b) { return a.first < b.first; });
        g_off.push_back(all_items.size());
        for (auto& it : g.items) all_items.push_back(it.second);
    }
    // plain mode: one candidate per launch sequence, items grouped per candidate
    std::vector<int> plain_items;
    std::vector<int> plain_off(n_cand + 1, 0);
    if (o.mode == MIRAGE_MODE_PLAIN) {
        for (int c = 0; c < n_cand; ++c) {
            plain_off[c] = (int)plain_items.size();
            for (int k = n_lam[c] - 1 + 0; k >= 0; --k) plain_items.push_back(pack_chain(c, k, k));
        }
        plain_off[n_cand] = (int)plain_items.size();
    }
    const std::vector<int>& items_v = o.mode == MIRAGE_MODE_PLAIN ? plain_items : all_items;

    const size_t n_counters = std::max<size_t>(glist.size(), (size_t)n_cand) + 1;
    // device metadata block: cand_prob[n_cand] | n_lam[n_cand] | items[...]
    std::vector<int> meta;
    meta.reserve(2 * n_cand + items_v.size());
    meta.insert(meta.end(), prob_idx, prob_idx + n_cand);
    meta.insert(meta.end(), n_lam, n_lam + n_cand);
    meta.insert(meta.end(), items_v.begin(), items_v.end());
    TRY(ctx->counters.ensure(sizeof(int) * n_counters));
    // taps of the fast kernels' launch groups (kernel parameters)
    std::vector<std::vector<float>> gtaps(glist.size());
    for (size_t gi = 0; gi < glist.size(); ++gi) {
        Group* g = glist[gi];
        if (!g->fast || g->prob < 0) continue;
        const Prob<T>& P = hp[g->prob];
        const int K = P.K;
        std::vector<T> psf((size_t)K * K);
        CK(cudaMemcpy(psf.data(), P.psf, sizeof(T) * K * K, cudaMemcpyDefault));
        std::vector<float>& tp = gtaps[gi];
        tp.assign(2 * MAX_PTAP, 0.f);
        for (int a = 0; a < K; ++a)
            for (int b = 0; b < K; ++b) {
                tp[a * K + b] = tap_value((float)psf[(K - 1 - a) * K + (K - 1 - b)], o.variant == 7);
                tp[MAX_PTAP + a * K + b] = tap_value((float)psf[a * K + b], o.variant == 7);
            }
    }
    // per-CTA global slab (bytes): FP64 refinement buffers, plus all work
    // buffers for items that do not fit in shared memory
    long long slab_stride = 0;
    std::vector<long long> g_slab_off(glist.size(), 0);  // first slab slot of each group
    long long slab_slots = 0;
    for (size_t gi = 0; gi < glist.size(); ++gi) {
        Group* g = glist[gi];
        slab_stride = std::max(slab_stride, (g->slab + 255) / 256 * 256);
        // groups run concurrently: each owns its own CTA slots of the slab
        g_slab_off[gi] = slab_slots;
        g->slots = cgls_slots(ctx, g->per_sm);
        if (g->cl) {
            int n = 0;
            TRY(set_smem(ctx, g->fn, g->smem));
            TRY(cluster_slots(ctx, g->fn, g->cl, g->nt, g->smem, &n));
            g->slots = n;
        }
        slab_slots += std::min<long long>(g->slots, (long long)g->items.size());
    }
    if (o.mode == MIRAGE_MODE_PLAIN) slab_slots = std::max<long long>(slab_slots, max_lam);
    TRY(ctx->slab.ensure((size_t)slab_stride * std::max<long long>(slab_slots, 1)));
    if (spec_stride) TRY(ctx->spec.ensure((sizeof(double2) + sizeof(float2)) * (size_t)spec_stride * n_probs));

    // graph key: everything that shapes the launch sequence
    std::string key;
    const bool graph = o.use_graph && o.mode == MIRAGE_MODE_BATCHED;
    if (graph) {
        // a grown scratch buffer invalidates every captured graph
        std::vector<void*> now = {ctx->E.p, ctx->E64.p, ctx->Etmp.p, ctx->inv.p, ctx->cst.p, ctx->swp.p, ctx->dpad.p,
                                  ctx->nent.p, ctx->cstat.p, ctx->X.p, ctx->istat.p, ctx->slab.p, ctx->counters.p,
                                  ctx->spec.p};
        if (now != ctx->scratch_seen) {
            drop_graphs(ctx);
            ctx->scratch_seen = now;
        }
        auto addb = [&](const void* p, size_t n) { key.append(reinterpret_cast<const char*>(p), n); };
        addb(&n_cand, sizeof(n_cand));
        addb(&max_lam, sizeof(max_lam));
        addb(hp.data(), sizeof(Prob<T>) * hp.size());
        addb(meta.data(), sizeof(int) * meta.size());
        const void* ptrs[] = {d_lens, d_lambdas, d_warm, d_chi2, d_reg, d_relres, d_kappa, d_iters, d_istat,
                              d_corner, d_status, d_sout, d_allx, st};
        addb(ptrs, sizeof(ptrs));
        addb(&o.tol, sizeof(o.tol));
        addb(&o.maxit, sizeof(o.maxit));
        addb(&o.replace_every, sizeof(o.replace_every));
        addb(&o.variant, sizeof(o.variant));
        addb(&o.inner_eta, sizeof(o.inner_eta));
        addb(&o.place, sizeof(o.place));
        for (auto& tp : gtaps)
            if (!tp.empty()) addb(tp.data(), sizeof(float) * tp.size());
        auto it = ctx->graphs.find(key);
        if (it != ctx->graphs.end()) {
            CK(cudaGraphLaunch(it->second.exec, st));
            ctx->last_launches = it->second.launches;
            return MIRAGE_OK;
        }
        if (!ctx->cap_stream) CK(cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
    }
    GraphEntry ge;
    DevBuf& probs_buf = graph ? ge.probs : ctx->probs;
    DevBuf& meta_buf = graph ? ge.meta : ctx->items;
    TRY(probs_buf.ensure(sizeof(Prob<T>) * n_probs));
    TRY(meta_buf.ensure(sizeof(int) * meta.size()));

    // uploads (before any capture)
    TRY(upload(ctx, st, {{probs_buf.p, hp.data(), sizeof(Prob<T>) * n_probs},
                         {meta_buf.p, meta.data(), sizeof(int) * meta.size()}}));

    CandScratch<T> cs;
    fill_scratch<T>(cs, ctx, false, sE, sInv, sCst, sPad);
    const Prob<T>* dprobs = probs_buf.as<Prob<T>>();
    const int* dcand = meta_buf.as<int>();
    const int* dnlam = dcand + n_cand;
    const int* ditems = dcand + 2 * n_cand;
    int* dcnt = ctx->counters.as<int>();
    const KernelTable& tb = table();

    for (Group* g : glist) TRY(set_smem(ctx, g->fn, g->smem));
    if (spec_stride) TRY(set_smem(ctx, tb.psf_spectra[prec], fft_smem_bytes(1024, false)));
    TRY(set_smem(ctx, tb.raytrace[prec], (size_t)max_cells * 4));
    if (4 * (max_cells + max_rays) <= ctx->max_smem - 2048) TRY(set_smem(ctx, tb.rt_cells[prec], sizeof(int) * (size_t)(max_cells + max_rays)));
    TRY(set_smem(ctx, tb.rt_place[prec], (size_t)max_cells * 4));

    CglsArgs<T> A;
    std::memset(&A, 0, sizeof(A));
    A.probs = dprobs;
    A.cand_prob = dcand;
    A.lens = d_lens;
    A.lambdas = d_lambdas;
    A.tol = o.tol;
    A.eta = o.inner_eta > 0.0 ? o.inner_eta : 0.01;
    A.maxit = o.maxit;
    A.replace_every = o.replace_every;
    A.max_lam = max_lam;
    A.max_ns = (int)max_ns;
    A.warm_x = d_warm;
    A.cs = cs;
    A.slab = ctx->slab.p;
    A.slab_stride = slab_stride;
    A.X = dX;
    A.chi2 = d_chi2;
    A.reg = d_reg;
    A.iters = d_iters;
    A.relres = d_relres;
    A.istat = dIst;
    A.phase_clk = nullptr;
    double2* d_spec64 = nullptr;
    float2* d_spec32 = nullptr;
    if (spec_stride) {
        d_spec64 = ctx->spec.as<double2>();
        if (sizeof(T) == 4) d_spec32 = reinterpret_cast<float2*>(d_spec64 + spec_stride * n_probs);
        A.spec64 = d_spec64;
        A.spec32 = d_spec32;
        A.spec_stride = spec_stride;
    }
    if (!graph && o.threads == -2) {
        TRY(ctx->clk.ensure(FAST_NPH * sizeof(unsigned long long)));
        CK(cudaMemsetAsync(ctx->clk.p, 0, FAST_NPH * sizeof(unsigned long long), st));
        A.phase_clk = ctx->clk.as<unsigned long long>();
    }

    const cudaStream_t launch_st = st;
    if (graph) {
        st = ctx->cap_stream;
        CK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    }
    int rc = MIRAGE_OK;
    if (spec_stride) {  // PSF spectra of the FFT problems (once per call)
        void* sa[] = {(void*)&dprobs, (void*)&d_spec64, (void*)&d_spec32, (void*)&spec_stride};
        rc = launch(ctx, tb.psf_spectra[prec], dim3(n_probs), dim3(NTHREADS), sa, fft_smem_bytes(1024, false), st);
    }
    do {
        if (rc) break;
        const bool timing = !graph && o.threads < 0;
        ctx->timed = 0;
        if (timing && !ctx->ev[0])
            for (int e = 0; e < 4; ++e) cudaEventCreate(&ctx->ev[e]);
        if (o.mode == MIRAGE_MODE_BATCHED) {
            if (timing) cudaEventRecord(ctx->ev[0], st);
            // 1) ray trace every candidate
            rc = launch_raytrace<T>(ctx, dprobs, dcand, d_lens, 0, n_cand, cs, max_cells, max_npix, max_rays, st);
            if (rc) break;
            // 2) CGLS items, one persistent launch per kernel class
            if (cudaMemsetAsync(dcnt, 0, sizeof(int) * n_counters, st) != cudaSuccess) {
                set_error("cudaMemsetAsync failed");
                rc = MIRAGE_ERR_CUDA;
                break;
            }
            if (timing) cudaEventRecord(ctx->ev[1], st);
            // kernel groups (different kernels or placements) run on side
            // streams so that one group's tail overlaps the next group
            const bool fork = glist.size() > 1;
            const int n_side = (int)std::min<size_t>(ctx->NSIDE, 2 * glist.size());
            if (fork) {
                if (!ctx->fork_ev) {
                    if (cudaEventCreateWithFlags(&ctx->fork_ev, cudaEventDisableTiming) != cudaSuccess) {
                        set_error("cudaEventCreate failed");
                        rc = MIRAGE_ERR_CUDA;
                        break;
                    }
                    for (int i = 0; i < ctx->NSIDE; ++i) {
                        cudaStreamCreateWithFlags(&ctx->side[i], cudaStreamNonBlocking);
                        cudaEventCreateWithFlags(&ctx->join_ev[i], cudaEventDisableTiming);
                    }
                }
                cudaEventRecord(ctx->fork_ev, st);
                for (int i = 0; i < n_side; ++i) cudaStreamWaitEvent(ctx->side[i], ctx->fork_ev, 0);
            }
            // Groups share the device from the start where there are clusters or few items
            // a SM, each with the CTAs that finish its items in the call's estimated time
            // (and half as many more: iteration counts are estimates), and each launches
            // the rest of the CTAs that it could use behind them: those start as other
            // groups end.  (One group after the other, each on all SMs, leaves the last
            // group's longest item alone on the device: the uneven batch of 48 candidates
            // then ran at 0.97 of the speed of the general kernels alone, side by side at
            // 1.40; two PSF widths at 64 x 64, 32 candidates x 12 lambdas, 13.1 and 10.2 ms.)
            // Many items fill in behind each other anyway, and shares cost more than they
            // give: four PSF widths, 192 candidates, 27.2 ms one after the other, 28.5 to
            // 31 side by side
            const bool split = fork && shared;
            for (int part = 0; part < (split ? 2 : 1) && !rc; ++part)
                for (size_t gi = 0; gi < glist.size() && !rc; ++gi) {
                    Group* g = glist[gi];
                    const cudaStream_t gs = fork ? ctx->side[(2 * gi + part) % ctx->NSIDE] : st;
                    const long long full = std::min<long long>(g->slots, (long long)g->items.size());
                    const long long first =
                        split ? std::min(full, std::max<long long>(1, (long long)std::ceil(1.5 * g->load / call_time))) : full;
                    const int grid = (int)(part == 0 ? first : full - first);
                    if (!grid) continue;
                    A.slab = ctx->slab.as<unsigned char>() + (g_slab_off[gi] + (part ? first : 0)) * slab_stride;
                    A.items = ditems + g_off[gi];
                    A.n_items = (int)g->items.size();
                    A.counter = dcnt + gi;
                    if (g->cl) {
                        A.max_smem = cluster_smem_limit(ctx, g->nt);
                        void* args[] = {&A};
                        rc = launch_cluster(ctx, g->fn, grid, g->cl, g->nt, args, g->smem, gs);
                    } else if (g->fast) {
                        FastArgs fa;
                        std::memset(&fa, 0, sizeof(fa));
                        set_fast_args<T>(fa, A);
                        if (!gtaps[gi].empty()) std::memcpy(fa.ptap, gtaps[gi].data(), sizeof(fa.ptap));
                        void* args[] = {&fa};
                        rc = launch(ctx, g->fn, dim3(grid), dim3(NTHREADS), args, g->smem, gs);
                    } else {
                        void* args[] = {&A};
                        rc = launch(ctx, g->fn, dim3(grid), dim3(NTHREADS), args, g->smem, gs);
                    }
                }
            if (fork) {
                for (int i = 0; i < n_side; ++i) {
                    cudaEventRecord(ctx->join_ev[i], ctx->side[i]);
                    cudaStreamWaitEvent(st, ctx->join_ev[i], 0);
                }
            }
            if (rc) break;
            if (timing) cudaEventRecord(ctx->ev[2], st);
            // 3) L-curve corner, status, s_out
            {
                int nc = n_cand, ml = max_lam, mns = (int)max_ns, c0 = 0;
                const int* ist = dIst;
                const int* cst = cs.cstat;
                const T* Xc = dX;
                void* args[] = {&c0, &nc, &ml, &mns, (void*)&dnlam, (void*)&dcand, (void*)&dprobs, (void*)&d_chi2,
                                (void*)&d_reg, (void*)&ist, (void*)&cst, (void*)&Xc, &d_corner, &d_kappa, &d_sout,
                                &d_status};
                rc = launch(ctx, tb.finalize[prec], dim3(n_cand), dim3(128), args, 0, st);
            }
            if (timing) {
                cudaEventRecord(ctx->ev[3], st);
                ctx->timed = 1;
            }
        } else {
            // plain: per candidate, ray trace (1 CTA), its lambdas (1 CTA each), finalize
            if (cudaMemsetAsync(dcnt, 0, sizeof(int) * n_counters, st) != cudaSuccess) {
                set_error("cudaMemsetAsync failed");
                rc = MIRAGE_ERR_CUDA;
                break;
            }
            for (int c = 0; c < n_cand && !rc; ++c) {
                const Prob<T>& P = hp[prob_idx[c]];
                const ProbPlan& q = plan[prob_idx[c]];
                const ClusterPlan& cp = class_of[c]->form[0]->cp;
                const void* fn = cp.C ? cp.fn : q.fn;
                const size_t item_smem = cp.C ? cp.smem : q.smem;
                TRY(set_smem(ctx, fn, item_smem));
                int cand0 = c, nc = 1;
                rc = launch_raytrace<T>(ctx, dprobs, dcand, d_lens, c, 1, cs, max_cells, max_npix, max_rays, st);
                if (rc) break;
                A.items = ditems + plain_off[c];
                A.n_items = plain_off[c + 1] - plain_off[c];
                A.counter = dcnt + c;
                if (cp.C) {
                    A.max_smem = cluster_smem_limit(ctx, cp.nt);
                    void* a2[] = {&A};
                    rc = launch_cluster(ctx, fn, A.n_items, cp.C, cp.nt, a2, item_smem, st);
                } else if (q.fast) {
                    FastArgs fa;
                    std::memset(&fa, 0, sizeof(fa));
                    set_fast_args<T>(fa, A);
                    if (q.mode > 0) {
                        std::vector<T> psf((size_t)P.K * P.K);
                        CK(cudaMemcpy(psf.data(), P.psf, sizeof(T) * P.K * P.K, cudaMemcpyDefault));
                        for (int a = 0; a < P.K; ++a)
                            for (int b = 0; b < P.K; ++b) {
                                fa.ptap[0][a * P.K + b] =
                                    tap_value((float)psf[(P.K - 1 - a) * P.K + (P.K - 1 - b)], q.mode == 3);
                                fa.ptap[1][a * P.K + b] = tap_value((float)psf[a * P.K + b], q.mode == 3);
                            }
                    }
                    void* a2[] = {&fa};
                    rc = launch(ctx, fn, dim3(A.n_items), dim3(NTHREADS), a2, item_smem, st);
                } else {
                    void* a2[] = {&A};
                    rc = launch(ctx, fn, dim3(A.n_items), dim3(NTHREADS), a2, item_smem, st);
                }
                if (rc) break;
                int ml = max_lam, mns = (int)max_ns;
                const int* ist = dIst;
                const int* cst = cs.cstat;
                const T* Xc = dX;
                void* a3[] = {&cand0, &nc, &ml, &mns, (void*)&dnlam, (void*)&dcand, (void*)&dprobs, (void*)&d_chi2,
                              (void*)&d_reg, (void*)&ist, (void*)&cst, (void*)&Xc, &d_corner, &d_kappa, &d_sout,
                              &d_status};
                rc = launch(ctx, tb.finalize[prec], dim3(1), dim3(128), a3, 0, st);
            }
        }
    } while (0);

    if (graph) {
        cudaGraph_t gr = nullptr;
        cudaError_t e = cudaStreamEndCapture(st, &gr);
        if (rc != MIRAGE_OK) {
            if (gr) cudaGraphDestroy(gr);
            ge.probs.release();
            ge.meta.release();
            return rc;
        }
        if (e != cudaSuccess) {
            set_error("cudaStreamEndCapture failed: %s", cudaGetErrorString(e));
            if (gr) cudaGraphDestroy(gr);
            return MIRAGE_ERR_CUDA;
        }
        e = cudaGraphInstantiate(&ge.exec, gr, 0);
        cudaGraphDestroy(gr);
        if (e != cudaSuccess) {
            set_error("cudaGraphInstantiate failed: %s", cudaGetErrorString(e));
            ge.probs.release();
            ge.meta.release();
            return MIRAGE_ERR_CUDA;
        }
        ge.launches = ctx->last_launches;
        GraphEntry& slot = ctx->graphs[key];
        slot = ge;
        ge.probs.p = nullptr;  // ownership moved to the cache entry
        ge.meta.p = nullptr;
        CK(cudaGraphLaunch(slot.exec, launch_st));
    }
    return rc;
}

template <typename T>
int forward_impl(mirage_ctx* ctx, const mirage_problem_t* prob, const double* lens, const void* s, int n_src,
                 void* model, double* chi2, int* status, cudaStream_t st) {
    constexpr int prec = prec_of<T>();
    ctx->last_launches = 0;
    if (!prob || !lens || !s || !chi2 || n_src < 0) {
        set_error("forward: null pointer");
        return MIRAGE_ERR_ARG;
    }
    if (check_geom(prob->geom) != MIRAGE_OK || !prob->d || !prob->sigma || !prob->mask || !prob->psf) {
        set_error("forward: bad problem");
        return MIRAGE_ERR_ARG;
    }
    if (n_src == 0) return MIRAGE_OK;
    Prob<T> P = make_prob<T>(*prob, prob->d, prob->sigma, prob->mask, prob->psf);
    if ((long long)P.ncells * 4 > ctx->max_smem - 2048) {
        set_error("source grid too large for the ray-trace kernel");
        return MIRAGE_ERR_UNSUPPORTED;
    }
    const long long sE = P.nrays, sInv = P.nrays, sCst = (P.ncells + 1 + 3) / 4 * 4, sPad = (P.plen + 3) / 4 * 4;
    TRY(ctx->fE.ensure(sizeof(Entry<T>) * sE));
    if (sizeof(T) == 4) TRY(ctx->fE64.ensure(sizeof(Entry<double>) * sE));
    TRY(ctx->fEtmp.ensure(sizeof(Entry<double>) * sE));
    TRY(ctx->finv.ensure(sizeof(int) * sInv));
    TRY(ctx->fcst.ensure(sizeof(int) * sCst));
    TRY(ctx->fswp.ensure(sizeof(T) * sPad));
    TRY(ctx->fdpad.ensure(sizeof(T) * sPad));
    TRY(ctx->fnent.ensure(sizeof(int)));
    TRY(ctx->fcstat.ensure(sizeof(int)));
    TRY(ctx->fprob.ensure(sizeof(Prob<T>) + sizeof(int)));
    const int grid = std::min(n_src, 2 * ctx->sm_count);
    const long long stride = (P.plen + 63) / 64 * 64;
    TRY(ctx->fslab.ensure(sizeof(T) * stride * grid));
    std::vector<char> up(sizeof(Prob<T>) + sizeof(int), 0);
    std::memcpy(up.data(), &P, sizeof(P));
    TRY(upload(ctx, st, {{ctx->fprob.p, up.data(), up.size()}}));
    const Prob<T>* dprob = ctx->fprob.as<Prob<T>>();
    const int* dcand = reinterpret_cast<const int*>(ctx->fprob.as<char>() + sizeof(Prob<T>));
    CandScratch<T> cs;
    fill_scratch<T>(cs, ctx, true, sE, sInv, sCst, sPad);
    const KernelTable& tb = table();
    if constexpr (sizeof(T) == 4) {
        // banded kernel: taps as kernel parameters, L s gathered into shared memory
        const void* fb = (P.Np == 1 && P.interp != MIRAGE_INTERP_BICUBIC && P.K < MAX_K && P.K * P.K <= MAX_FTAP)
                             ? tb.fwdb[P.K]
                             : nullptr;
        if (fb && P.tiles_x <= FWD_THREADS) {
            const int bt = std::min(FWD_THREADS / P.tiles_x, P.tiles_y);
            const size_t smb = fwd_band_smem(P, bt);
            if ((long long)smb <= ctx->max_smem) {
                // the rays in pixel order are all that this kernel reads: no
                // placement by cells
                const int chunk = (int)std::min<long long>(RT_THREADS, std::max(32LL, (P.npix + 8LL * ctx->sm_count - 1) / (8LL * ctx->sm_count)));
                const int n_rays_cta = (P.npix + chunk - 1) / chunk;
                const size_t pix_bytes = (sizeof(float4) * (size_t)P.npix + 15) / 16 * 16;
                TRY(ctx->fpix.ensure(pix_bytes + sizeof(int) * (size_t)n_rays_cta));
                float4* pm = ctx->fpix.as<float4>();
                int* flags = reinterpret_cast<int*>(ctx->fpix.as<char>() + pix_bytes);
                {
                    CandScratch<float> csv = cs;
                    const Prob<float>* dp0 = dprob;
                    int ch = chunk;
                    void* ap[] = {(void*)&dp0, (void*)&lens, &csv, (void*)&pm, (void*)&flags, &ch};
                    TRY(launch(ctx, tb.fwd_rays, dim3(n_rays_cta), dim3(RT_THREADS), ap, 0, st));
                }
                std::vector<unsigned char> fab(sizeof(FwdArgs), 0);
                FwdArgs* fa = reinterpret_cast<FwdArgs*>(fab.data());
                fa->probs = dprob;
                fa->cs = cs;
                fa->pixmap = pm;
                fa->flags = flags;
                fa->n_flags = n_rays_cta;
                fa->S = reinterpret_cast<const float*>(s);
                fa->n_src = n_src;
                fa->model = reinterpret_cast<float*>(model);
                fa->chi2 = chi2;
                fa->status = status;
                fa->band_tiles = bt;
                TRY(set_smem(ctx, fb, smb));
                void* a3[] = {fa};
                TRY(launch(ctx, fb, dim3(std::min(n_src, ctx->sm_count)), dim3(FWD_THREADS), a3, smb, st));
                return MIRAGE_OK;
            }
        }
    }
    TRY(launch_raytrace<T>(ctx, dprob, dcand, lens, 0, 1, cs, P.ncells, (long long)P.npix, (long long)P.nrays, st));
    const void* fn = pick_fwd(prec, P.K);
    const size_t smem = align_up<T>(sizeof(T) * P.K * P.kp, 16) + 2 * 33 * sizeof(double) + 16;
    TRY(set_smem(ctx, fn, smem));
    const T* S = reinterpret_cast<const T*>(s);
    T* M = reinterpret_cast<T*>(model);
    T* slab = ctx->fslab.as<T>();
    long long sstr = stride;
    void* a2[] = {(void*)&dprob, &cs, (void*)&S, &n_src, &M, &chi2, &slab, &sstr, &status};
    TRY(launch(ctx, fn, dim3(grid), dim3(NTHREADS), a2, smem, st));
    return MIRAGE_OK;
}

// fixed-iteration CGLS with the iteration L-curve (mirage_eval_iter)
template <typename T>
int iter_impl(mirage_ctx* ctx, const mirage_problem_t* probs, int n_probs, const double* lens, const int* prob_idx,
              int n_cand, int n_iter, const void* bhat, long long bhat_stride, double* chi2, double* reg,
              double* dof, int* corner, double* kappa, void* s_out, int* status, cudaStream_t st) {
    constexpr int prec = prec_of<T>();
    ctx->last_launches = 0;
    if (n_cand == 0) return MIRAGE_OK;
    if (!probs || n_probs < 1 || !lens || !prob_idx || !chi2 || !reg || !corner || !status || n_cand < 0 ||
        n_iter < 1 || n_iter > MAX_LAM - 1 || (bhat && bhat_stride < 1)) {
        set_error("eval_iter: null pointer or size out of range (1 <= n_iter <= %d)", MAX_LAM - 1);
        return MIRAGE_ERR_ARG;
    }
    std::vector<Prob<T>> hp(n_probs);
    long long max_rays = 0, max_cells = 0, max_plen = 0, max_ns = 0, max_npix = 0;
    size_t smem = 0, slab = 0;
    int k_all = -1;
    for (int p = 0; p < n_probs; ++p) {
        if (check_geom(probs[p].geom) != MIRAGE_OK || !probs[p].d || !probs[p].sigma || !probs[p].mask ||
            !probs[p].psf) {
            set_error("eval_iter: bad problem %d", p);
            return MIRAGE_ERR_ARG;
        }
        hp[p] = make_prob<T>(probs[p], probs[p].d, probs[p].sigma, probs[p].mask, probs[p].psf);
        if (bhat && (long long)probs[p].geom.nx * probs[p].geom.ny > bhat_stride) {
            set_error("eval_iter: bhat_stride below the pixel count of problem %d", p);
            return MIRAGE_ERR_ARG;
        }
        max_rays = std::max<long long>(max_rays, hp[p].nrays);
        max_cells = std::max<long long>(max_cells, hp[p].ncells);
        max_plen = std::max<long long>(max_plen, hp[p].plen);
        max_ns = std::max<long long>(max_ns, hp[p].ns);
        max_npix = std::max<long long>(max_npix, hp[p].npix);
        smem = std::max(smem, iter_smem_bytes<T>(hp[p].K, hp[p].kp));
        slab = std::max(slab, iter_slab_bytes<T>(hp[p], n_iter));
        k_all = (k_all == -1 || k_all == hp[p].K) ? hp[p].K : 0;
    }
    for (int c = 0; c < n_cand; ++c)
        if (prob_idx[c] < 0 || prob_idx[c] >= n_probs) {
            set_error("eval_iter: bad prob_idx of candidate %d", c);
            return MIRAGE_ERR_ARG;
        }
    if (max_cells * 4 > ctx->max_smem - 2048) {
        set_error("source grid too large for the ray-trace kernel");
        return MIRAGE_ERR_UNSUPPORTED;
    }
    const long long sE = max_rays, sInv = max_rays, sCst = (max_cells + 1 + 3) / 4 * 4, sPad = (max_plen + 3) / 4 * 4;
    TRY(ctx->E.ensure(sizeof(Entry<T>) * n_cand * sE));
    if (sizeof(T) == 4) TRY(ctx->E64.ensure(sizeof(Entry<double>) * n_cand * sE));
    TRY(ctx->Etmp.ensure(sizeof(Entry<double>) * n_cand * sE));
    TRY(ctx->inv.ensure(sizeof(int) * n_cand * sInv));
    TRY(ctx->cst.ensure(sizeof(int) * n_cand * sCst));
    TRY(ctx->swp.ensure(sizeof(T) * n_cand * sPad));
    TRY(ctx->dpad.ensure(sizeof(T) * n_cand * sPad));
    TRY(ctx->nent.ensure(sizeof(int) * n_cand));
    TRY(ctx->cstat.ensure(sizeof(int) * n_cand));
    TRY(ctx->probs.ensure(sizeof(Prob<T>) * n_probs));
    TRY(ctx->cand_prob.ensure(sizeof(int) * n_cand));
    TRY(ctx->counters.ensure(sizeof(int)));
    const int grid = std::min(n_cand, 2 * ctx->sm_count);
    TRY(ctx->slab.ensure(slab * grid));
    TRY(upload(ctx, st, {{ctx->probs.p, hp.data(), sizeof(Prob<T>) * n_probs},
                         {ctx->cand_prob.p, prob_idx, sizeof(int) * n_cand}}));
    CK(cudaMemsetAsync(ctx->counters.p, 0, sizeof(int), st));
    CandScratch<T> cs;
    fill_scratch<T>(cs, ctx, false, sE, sInv, sCst, sPad);
    const Prob<T>* dprobs = ctx->probs.as<Prob<T>>();
    const int* dcand = ctx->cand_prob.as<int>();
    const KernelTable& tb = table();
    TRY(launch_raytrace<T>(ctx, dprobs, dcand, lens, 0, n_cand, cs, max_cells, max_npix, max_rays, st));
    const void* fn = (k_all > 0 && k_all < MAX_K && tb.iter[prec][k_all]) ? tb.iter[prec][k_all] : tb.iter[prec][0];
    TRY(set_smem(ctx, fn, smem));
    IterArgs<T> A;
    std::memset(&A, 0, sizeof(A));
    A.probs = dprobs;
    A.cand_prob = dcand;
    A.cs = cs;
    A.n_cand = n_cand;
    A.n_iter = n_iter;
    A.max_ns = (int)max_ns;
    A.bhat = reinterpret_cast<const T*>(bhat);
    A.bhat_stride = bhat_stride;
    A.counter = ctx->counters.as<int>();
    A.slab = ctx->slab.p;
    A.slab_stride = (long long)slab;
    A.chi2 = chi2;
    A.reg = reg;
    A.dof = dof;
    A.kappa = kappa;
    A.corner = corner;
    A.s_out = reinterpret_cast<T*>(s_out);
    A.status = status;
    void* a2[] = {&A};
    TRY(launch(ctx, fn, dim3(grid), dim3(NTHREADS), a2, smem, st));
    return MIRAGE_OK;
}

}  // namespace

extern "C" {

int mirage_create(mirage_ctx_t** out, int device, int precision) {
    if (!out) return MIRAGE_ERR_ARG;
    *out = nullptr;
    if (precision != MIRAGE_FP32 && precision != MIRAGE_FP64) {
        set_error("precision must be MIRAGE_FP32 or MIRAGE_FP64");
        return MIRAGE_ERR_ARG;
    }
    CK(cudaSetDevice(device));
    mirage_ctx* c = new mirage_ctx();
    c->device = device;
    c->precision = precision;
    cudaError_t e1 = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device);
    cudaError_t e2 = cudaDeviceGetAttribute(&c->max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    cudaError_t e3 = cudaDeviceGetAttribute(&c->max_smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
    if (e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess) {
        set_error("cudaDeviceGetAttribute failed");
        delete c;
        return MIRAGE_ERR_CUDA;
    }
    (void)table();
    *out = c;
    return MIRAGE_OK;
}

int mirage_destroy(mirage_ctx_t* ctx) {
    if (!ctx) return MIRAGE_OK;
    cudaSetDevice(ctx->device);
    drop_graphs(ctx);
    if (ctx->cap_stream) cudaStreamDestroy(ctx->cap_stream);
    for (int i = 0; i < ctx->NSIDE; ++i) {
        if (ctx->side[i]) cudaStreamDestroy(ctx->side[i]);
        if (ctx->join_ev[i]) cudaEventDestroy(ctx->join_ev[i]);
    }
    if (ctx->fork_ev) cudaEventDestroy(ctx->fork_ev);
    for (int e = 0; e < 4; ++e)
        if (ctx->ev[e]) cudaEventDestroy(ctx->ev[e]);
    DevBuf* bufs[] = {&ctx->E, &ctx->E64, &ctx->Etmp, &ctx->inv, &ctx->cst, &ctx->swp, &ctx->dpad, &ctx->nent, &ctx->cstat,
                      &ctx->X, &ctx->istat, &ctx->slab, &ctx->probs, &ctx->cand_prob, &ctx->items, &ctx->counters,
                      &ctx->stage, &ctx->fE, &ctx->fE64, &ctx->fEtmp, &ctx->finv, &ctx->fcst, &ctx->fswp, &ctx->fdpad,
                      &ctx->fnent, &ctx->fcstat, &ctx->fslab, &ctx->fprob, &ctx->fcand, &ctx->fpix, &ctx->rt_cursor, &ctx->clk,
                      &ctx->spec};
    for (DevBuf* b : bufs) b->release();
    if (ctx->pin_pending) cudaEventSynchronize(ctx->pin_ev);
    if (ctx->pin) cudaFreeHost(ctx->pin);
    if (ctx->pin_ev) cudaEventDestroy(ctx->pin_ev);
    delete ctx;
    return MIRAGE_OK;
}

int mirage_eval_batch(mirage_ctx_t* ctx, const mirage_problem_t* probs, int n_probs, const double* lens,
                      const int* prob_idx, int n_cand, const double* lambdas, const int* n_lam, int max_lam,
                      const mirage_opts_t* opts, const void* warm_x, const int* lam_start, double* chi2,
                      double* reg, int* iters, double* relres, int* item_status, int* corner, double* kappa,
                      void* s_out, void* all_x, int* status, void* stream) {
    if (!ctx || !opts) return MIRAGE_ERR_ARG;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return MIRAGE_ERR_CUDA;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (ctx->precision == MIRAGE_FP32)
        return eval_impl<float>(ctx, probs, n_probs, lens, prob_idx, n_cand, lambdas, n_lam, max_lam, opts, warm_x,
                                lam_start, chi2, reg, iters, relres, item_status, corner, kappa, s_out, all_x, status, st);
    return eval_impl<double>(ctx, probs, n_probs, lens, prob_idx, n_cand, lambdas, n_lam, max_lam, opts, warm_x,
                             lam_start, chi2, reg, iters, relres, item_status, corner, kappa, s_out, all_x, status, st);
}

int mirage_lcurve(const double* chi2, const double* reg, const int* n_lam, int n_cand, int max_lam, int* corner,
                  double* kappa, int* flags, void* stream) {
    if (n_cand == 0) return MIRAGE_OK;
    if (!chi2 || !reg || !n_lam || !corner || n_cand < 0 || max_lam < 1 || max_lam > MAX_LAM) {
        set_error("lcurve: bad argument");
        return MIRAGE_ERR_ARG;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    k_lcurve<0><<<(n_cand + 127) / 128, 128, 0, st>>>(chi2, reg, n_lam, n_cand, max_lam, corner, kappa, flags);
    CK(cudaGetLastError());
    return MIRAGE_OK;
}

int mirage_forward(mirage_ctx_t* ctx, const mirage_problem_t* prob, const double* lens, const void* s, int n_src,
                   void* model, double* chi2, int* status, void* stream) {
    if (!ctx) return MIRAGE_ERR_ARG;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return MIRAGE_ERR_CUDA;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (ctx->precision == MIRAGE_FP32) return forward_impl<float>(ctx, prob, lens, s, n_src, model, chi2, status, st);
    return forward_impl<double>(ctx, prob, lens, s, n_src, model, chi2, status, st);
}

int mirage_eval_iter(mirage_ctx_t* ctx, const mirage_problem_t* probs, int n_probs, const double* lens,
                     const int* prob_idx, int n_cand, int n_iter, const void* bhat, long long bhat_stride,
                     double* chi2, double* reg, double* dof, int* corner, double* kappa, void* s_out, int* status,
                     void* stream) {
    if (!ctx) return MIRAGE_ERR_ARG;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return MIRAGE_ERR_CUDA;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (ctx->precision == MIRAGE_FP32)
        return iter_impl<float>(ctx, probs, n_probs, lens, prob_idx, n_cand, n_iter, bhat, bhat_stride, chi2, reg,
                                dof, corner, kappa, s_out, status, st);
    return iter_impl<double>(ctx, probs, n_probs, lens, prob_idx, n_cand, n_iter, bhat, bhat_stride, chi2, reg, dof,
                             corner, kappa, s_out, status, st);
}

int mirage_set_reserved_slots(mirage_ctx_t* ctx, int slots) {
    if (!ctx || slots < 0) {
        set_error("set_reserved_slots: bad arguments");
        return MIRAGE_ERR_ARG;
    }
    if (slots != ctx->reserved) drop_graphs(ctx);  // captured launches carry the old grid
    ctx->reserved = slots;
    return MIRAGE_OK;
}

int mirage_last_launch_count(const mirage_ctx_t* ctx) { return ctx ? ctx->last_launches : 0; }

int mirage_last_item_kernels(const mirage_ctx_t* ctx, int* out) {
    if (!ctx || !out) return MIRAGE_ERR_ARG;
    std::copy(ctx->last_kernels, ctx->last_kernels + MIRAGE_N_ITEM_KERNELS, out);
    return MIRAGE_OK;
}

static_assert(MAX_LAM == MIRAGE_MAX_LAM, "lambda grid limit of the header and the kernels");

int mirage_last_phase_clocks(mirage_ctx_t* ctx, unsigned long long* clk) {
    static_assert(FAST_NPH == MIRAGE_N_PHASE_CLOCKS, "phase clock count of the header and the kernel");
    if (!ctx || !clk || !ctx->clk.p) return MIRAGE_ERR_ARG;
    CK(cudaMemcpy(clk, ctx->clk.p, FAST_NPH * sizeof(unsigned long long), cudaMemcpyDeviceToHost));
    return MIRAGE_OK;
}

int mirage_last_phase_ms(mirage_ctx_t* ctx, double* ms) {
    if (!ctx || !ms) return MIRAGE_ERR_ARG;
    if (!ctx->timed) {
        set_error("no timed batched call on this context");
        return MIRAGE_ERR_ARG;
    }
    for (int i = 0; i < 3; ++i) {
        float t = 0.f;
        CK(cudaEventSynchronize(ctx->ev[i + 1]));
        CK(cudaEventElapsedTime(&t, ctx->ev[i], ctx->ev[i + 1]));
        ms[i] = t;
    }
    return MIRAGE_OK;
}

const char* mirage_last_error(void) { return g_last_error.c_str(); }

}  // extern "C"

// Internal accessors shared with the allocation-free entry point (noalloc.cu).
namespace mirage {
const KernelTable& kernel_table() { return table(); }
int geometry_ok(const mirage_geom_t& g) { return check_geom(g); }
template <typename T>
Prob<T> problem_layout(const mirage_problem_t& p) {
    return make_prob<T>(p, p.d, p.sigma, p.mask, p.psf);
}
template Prob<float> problem_layout<float>(const mirage_problem_t&);
template Prob<double> problem_layout<double>(const mirage_problem_t&);
}  // namespace mirage
