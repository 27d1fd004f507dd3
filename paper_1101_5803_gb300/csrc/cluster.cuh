// General CGLS item kernel on a thread-block cluster (FP32 contexts, one
// ray per pixel, four-corner interpolation): the systems that the two-CTA
// kernel of fast.cuh cannot take.
//
// What bounds it: per CG iteration 4 K^2 N_pix FP32 operations of B and B^T
// (at 256 x 256 and K = 21, 0.24 ms on one SM), and how long the longest
// item of a call is.  k_cgls keeps one item on one SM and these images in an
// L2-resident slab, so its convolutions wait for L2 and a call ends with one
// SM at work.  Here C CTAs (1, 2, 4 or 8 SMs) share one item:
//   * only tiles that hold a mapped pixel are convolved: L p is zero and sqrt(W)
//     too elsewhere, so B L p is weighted away there and u is not read (60% of
//     the tiles of the 256 x 256 system are left, 27% of the uneven batch's);
//   * the image's rows with such tiles are cut into C bands of whole tile rows;
//     each CTA keeps its band of L p and of W B L p, with the K - 1 halo rows,
//     in its own shared memory.  A value in a neighbour's halo is also stored
//     there, through distributed shared memory, when it is made;
//   * the source rows are cut into C runs of about equal ray counts.  A CTA
//     interpolates the rays of its own cells (L p, stored to the bands that
//     hold the pixels), sums L^T over its own cells and one more cell row, so
//     that its source pixels need no other CTA's cells, and keeps p and H p of
//     its rows and two rows around them in shared memory;
//   * every sum over the image or the source is added up as k_cgls adds it:
//     its 256 threads own the tiles and source pixels t = v + 256 k, so the
//     terms are stored and virtual thread v's terms are added in that order,
//     the last warps of each CTA taking one warp of virtual threads each.  An
//     item's results are thus bit for bit those of k_cgls, for any C.
// Measured, clocks of an iteration in k_cgls and here on eight SMs: 1555k and
// 159k at 256 x 256 and K = 21, 172k and 57k at 128 x 128 and K = 15, 51k and 35k
// at 48 x 48 (image and source) and K = 15.
#pragma once

#include <type_traits>

#include "forward.cuh"

namespace mirage {

constexpr int CL_MAX = 8;      // largest (portable) cluster
constexpr int CL_STAGE = 2048;  // rays of L^T staged at a time at least (as many as shared memory holds)

__device__ __forceinline__ unsigned cl_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// the address in CTA `rank`'s shared memory of this CTA's shared address a
__device__ __forceinline__ unsigned cl_map(unsigned a, unsigned rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_st(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_st(unsigned a, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_st(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_st4(unsigned a, const float* v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
}
__device__ __forceinline__ float cl_ld(unsigned a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cl_ld4(unsigned a, float* v) {
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(a)
                 : "memory");
}
// barrier of all threads of the cluster; what any of them wrote before it
// (shared or global) is seen by all after it
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void cl_copy16(unsigned dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cl_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// How one problem is cut over C CTAs of NT threads (host and device)
struct ClusterCut {
    int C, nt;
    int bt;       // tile rows per band
    int blen;     // floats of one band buffer (bt tile rows + K - 1 rows)
    int cap;      // source rows per CTA at most
    int blen2;    // floats allocated for the band of W B L p, which stages the rays of L^T too (stage of them)
    int stage;
    int zlen;     // floats of the scratch shared by sqrt(W) B L p and the cell sums
    // max_smem: dynamic shared memory that a CTA may take
    __host__ __device__ ClusterCut(const Prob<float>& P, int c, int max_smem) {
        C = c;
        bt = (P.tiles_y + C - 1) / C;
        nt = bt * P.tiles_x > NTHREADS ? 2 * NTHREADS : NTHREADS;
        blen = (bt * TILE + P.K - 1) * P.Wp;
        cap = C == 1 ? P.sy : (5 * P.sy + 4 * C - 1) / (4 * C) + 1;
        const int q = bt * TILE * P.tiles_x * TILE;
        zlen = q > 4 * (cap + 1) * P.sx ? q : 4 * (cap + 1) * P.sx;
        if (zlen < (cap + 4) * P.sx) zlen = (cap + 4) * P.sx;
        blen2 = blen > 4 * CL_STAGE ? blen : 4 * CL_STAGE;
        // a CTA's share of the rays and some more, where there is room for it
        const int want = 4 * (P.nrays / C + P.nrays / (4 * C));
        const long long room = ((long long)max_smem - (long long)bytes(P)) / (long long)sizeof(float) - 4;
        if (want > blen2 && room > 0) blen2 += want - blen2 < (int)room ? want - blen2 : (int)room;
        blen2 &= ~3;
        stage = blen2 / 4;
    }
    __host__ __device__ size_t bytes(const Prob<float>& P) const;
};

struct ClusterCtl {
    int item, more, brk, stop, best_it, it, total_it;
    float a, b;
    double gam, g0, best;
    int row[CL_MAX + 1];       // source-row boundaries of the CTAs
    float ws[2][8];            // FP32 warp sums of the virtual threads
    double wd[2][8];           // FP64 warp sums
    ChainPos ch;
    double rhsn, prev_rel, target;
};

// Constants of the current item, written by thread 0 and read from shared
// memory where they are used: held in registers they spill, and the shared
// memory leaves too little L1 for the spilled lines of 512 threads (measured:
// each phase paid an L2 round trip or two, 95k against 71k clocks an
// iteration of the 128 x 128 system).  Shared arrays are byte offsets.
struct ClusterItem {
    Geo<float> g;
    unsigned PA, PB, Z, p, h, gv, mi, mb, tl;
    int row0, ty0, ty1, tyA, tyB, hop, R, nx4, tiles, act, bt, blen, hn, stage;
    int i0, i1, pr0, pr1, hr0, hr1, e0, e1, cell0, cell1, r0, r1;
    float lamT;
    int cstat, gather;
    double lam;
    double *Pa, *Pb, *Pc, *Rs, *x64, *xb, *sv, *h64;
    float *gvg, *zg, *xg, *hg;
    int4* rec;
    const float *swp, *dpad, *psf;
    const Entry<float>* E;
    const Entry<double>* E64;
    const int* cst;
};
constexpr size_t CL_TAPS = (sizeof(ClusterCtl) + 15) / 16 * 16 + (sizeof(ClusterItem) + 15) / 16 * 16;

__host__ __device__ inline size_t ClusterCut::bytes(const Prob<float>& P) const {
    const ClusterCut& u = *this;
    size_t o = CL_TAPS;
    o += align_up<float>(sizeof(float) * 2 * P.K * P.kp, 16);                     // taps
    o += align_up<float>(sizeof(float) * u.blen, 16);                             // band of L p, then u
    o += align_up<float>(sizeof(float) * u.blen2, 16);                            // band of W B L p, then staged rays
    o += align_up<float>(sizeof(float) * u.zlen, 16);                             // sqrt(W) B L p / cell sums / z
    o += align_up<float>(sizeof(float) * (u.cap + 4) * P.sx, 16);                 // p
    o += align_up<float>(sizeof(float) * (P.nreg / P.ns) * (u.cap + 2) * P.sx, 16);  // H p
    o += 2 * align_up<float>(sizeof(float) * u.cap * P.sx, 16);                   // g, M^-1
    o += 2 * align_up<float>(sizeof(unsigned short) * u.bt * P.tiles_x, 16);      // mapped-pixel bits of the tiles, tile list
    return o;
}
// global work space of one cluster
__host__ __device__ inline size_t cluster_slab_bytes(const Prob<float>& P) {
    const size_t pl = align_up<float>(P.plen, 4), pn = align_up<float>(P.ns, 4), pr = align_up<float>(P.nreg, 4);
    return align_up<float>(sizeof(double) * (4 * pl + 3 * pn + pr) + sizeof(float) * (3 * pn + pr) +
                               sizeof(int4) * (size_t)P.nrays, 256);
}

__device__ inline void cluster_item_fill(ClusterItem& I, const Prob<float>& P, const CglsArgs<float>& A, int c, int k,
                                         int C, int rank, int cid) {
    const CandScratch<float>& cs = A.cs;
    I.g = geo_of(P, cs.nent[c]);
    const ClusterCut u(P, C, A.max_smem);
    unsigned o = (unsigned)(CL_TAPS + align_up<float>(sizeof(float) * 2 * P.K * P.kp, 16));
    auto carve = [&](size_t bytes) { const unsigned q = o; o += (unsigned)align_up<float>(bytes, 16); return q; };
    I.PA = carve(sizeof(float) * u.blen);
    I.PB = carve(sizeof(float) * u.blen2);
    I.Z = carve(sizeof(float) * u.zlen);
    I.p = carve(sizeof(float) * (u.cap + 4) * P.sx);
    I.h = carve(sizeof(float) * (P.nreg / P.ns) * (u.cap + 2) * P.sx);
    I.gv = carve(sizeof(float) * u.cap * P.sx);
    I.mi = carve(sizeof(float) * u.cap * P.sx);
    I.mb = carve(sizeof(unsigned short) * u.bt * P.tiles_x);
    I.tl = carve(sizeof(unsigned short) * u.bt * P.tiles_x);
    I.stage = u.stage;
    I.blen = u.blen;
    I.hn = (u.cap + 2) * P.sx;
    const size_t pl = align_up<float>(P.plen, 4), pn = align_up<float>(P.ns, 4), pr = align_up<float>(P.nreg, 4);
    double* d = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(A.slab) + (long long)cid * A.slab_stride);
    I.Pa = d; d += pl;
    I.Pb = d; d += pl;
    I.Pc = d; d += pl;
    I.Rs = d; d += pl;
    I.x64 = d; d += pn;
    I.xb = d; d += pn;
    I.sv = d; d += pn;
    I.h64 = d; d += pr;
    float* f = reinterpret_cast<float*>(d);
    I.gvg = f; f += pn;
    I.zg = f; f += pn;
    I.xg = f; f += pn;
    I.hg = f; f += pr;
    I.rec = reinterpret_cast<int4*>(f);
    I.swp = cs.swp + (long long)c * cs.sPad;
    I.dpad = cs.dpad + (long long)c * cs.sPad;
    I.psf = P.psf;
    I.E = cs.E + (long long)c * cs.sE;
    I.E64 = cs.E64 + (long long)c * cs.sE;
    I.cst = cs.cst + (long long)c * cs.sCst;
    I.cstat = cs.cstat[c];
    I.lam = A.lambdas[(long long)c * A.max_lam + k];
    I.lamT = (float)I.lam;
    I.nx4 = P.tiles_x * TILE;
    I.gather = 4 * P.ncells > P.plen;  // the form of L^T that k_cgls takes
    I.tyA = P.tiles_y;  // (the mapped tile rows follow)
    I.tyB = 0;
}
// ... and, once the mapped tile rows [tyA, tyB) are known and the source rows cut
__device__ inline void cluster_item_rows(ClusterItem& I, const int* row, int C, int rank) {
    // bands of equal height; a halo reaches the next band only
    I.bt = max((I.tyB - I.tyA + C - 1) / C, C > 1 ? (I.g.hk + TILE - 1) / TILE : 1);
    I.ty0 = min(I.tyA + rank * I.bt, I.tyB);
    I.ty1 = min(I.ty0 + I.bt, I.tyB);
    I.row0 = I.ty0 * TILE;
    I.R = I.bt * TILE;
    I.hop = I.R * I.g.Wp;  // from a band to the next
    I.tiles = (I.ty1 - I.ty0) * I.g.tiles_x;
    const int b0 = row[rank], b1 = row[rank + 1], sx = I.g.sx, sy = I.g.sy, ncx = I.g.ncx;
    I.i0 = b0 * sx;
    I.i1 = b1 * sx;
    I.pr0 = max(b0 - 2, 0);
    I.pr1 = min(b1 + 2, sy);
    I.hr0 = max(b0 - 1, 0);
    I.hr1 = min(b1 + 1, sy);
    I.e0 = I.cst[min(b0, sy - 1) * ncx];  // rays of the own cells
    I.e1 = I.cst[min(b1, sy - 1) * ncx];
    I.cell0 = I.hr0 * ncx;                // cells of L^T: the own ones and the row before
    I.cell1 = b1 > b0 ? min(b1, sy - 1) * ncx : I.cell0;
    I.r0 = I.cst[I.cell0];                // ... and their rays
    I.r1 = I.cst[I.cell1];
}

// The refinement's double-float convolution (conv64_df_gen) over this CTA's
// band: the FP64 input's band and halo split into hi and lo in the two band
// buffers, which hold zeros again on return.  mode 0: the image residual
// into Rs, sqrt(W) times it into Pb; mode 1: the convolution into Pc.
template <int K, int NT>
__device__ __noinline__ void cl_conv64(const ClusterItem& I, const double* src, float* hi, float* lo, const float* taps,
                                       const unsigned short* tiles, int mode) {
    const Geo<float>& g = I.g;
    const int blen = I.blen, Wp = g.Wp, tiles_x = g.tiles_x, g0 = I.row0 * Wp;  // padded position of local position 0
    {
        const int n = min(blen, g.plen - g0);
        for (int i = threadIdx.x; i < blen; i += NT) {
            const double v = i < n ? __ldcg(src + g0 + i) : 0.0;
            df_split(v, hi[i], lo[i]);
        }
    }
    __syncthreads();
    const unsigned short* list = tiles;
    const int act = I.act, units = act * TILE;  // four pixels of one row each
    for (int u = threadIdx.x; u < units; u += NT) {
        const int r = u / act, t = list[u - r * act], ty = t / tiles_x, y = ty * TILE + r, tx = t - ty * tiles_x;
        const int base = y * Wp + tx * TILE + g.sh;
        float s[TILE], c[TILE];
#pragma unroll
        for (int q = 0; q < TILE; ++q) s[q] = c[q] = 0.f;
#pragma unroll 1
        for (int a = 0; a < K; ++a) {
            const float* hrow = hi + base + a * Wp;
            const float* lrow = lo + base + a * Wp;
            const float* trow = taps + a * ((K + 3) & ~3);
            float xh[K + TILE - 1], xl[K + TILE - 1];
#pragma unroll
            for (int j = 0; j < K + TILE - 1; ++j) {
                xh[j] = hrow[j];
                xl[j] = lrow[j];
            }
#pragma unroll
            for (int b = 0; b < K; ++b) {
                const float tt = trow[b];
#pragma unroll
                for (int q = 0; q < TILE; ++q) df_madd(s[q], c[q], tt, xh[b + q], xl[b + q]);
            }
        }
        const int p0 = g0 + (y + g.hk) * Wp + tx * TILE + g.xoff;
#pragma unroll
        for (int q = 0; q < TILE; ++q) {
            const int pp = p0 + q;
            const double v = (double)s[q] + (double)c[q];
            if (mode == 0) {
                const double sw = (double)I.swp[pp];
                const double res = sw * ((double)I.dpad[pp] - v);
                I.Rs[pp] = res;
                I.Pb[pp] = sw * res;
            } else {
                I.Pc[pp] = v;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < blen; i += NT) {
        hi[i] = 0.f;
        lo[i] = 0.f;
    }
}

template <int K, int NT>
__global__ void __launch_bounds__(NT, 2 * NTHREADS / NT) k_cgls_cluster(CglsArgs<float> A) {
    constexpr int HK = (K - 1) / 2, KP = (K + 3) & ~3, VT = NTHREADS, NVW = VT / 32;  // VT virtual threads in NVW warps
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned C = cl_size(), rank = cl_rank();
    ClusterCtl* ctl = reinterpret_cast<ClusterCtl*>(smem);
    ClusterItem& I = *reinterpret_cast<ClusterItem*>(smem + (sizeof(ClusterCtl) + 15) / 16 * 16);
    const Geo<float>& g = I.g;
    float* taps = reinterpret_cast<float*>(smem + CL_TAPS);
    auto sh = [&](unsigned o) { return reinterpret_cast<float*>(smem + o); };
    // tiles by rows where there are fewer tiles than threads: a whole tile, two
    // rows or one row a thread (a warp alone on its scheduler takes as long for
    // 92 tiles as for 512)
    auto by_rows = [&](int act, auto&& f) {
        if (2 * act > NT)
            f(std::integral_constant<int, 4>());
        else if (4 * act > NT)
            f(std::integral_constant<int, 2>());
        else
            f(std::integral_constant<int, 1>());
    };
    auto clear_stage = [&]() {  // the staged rays of L^T
        float* PB = sh(I.PB);
        const int n = min(I.blen, 4 * min(I.stage, I.r1 - I.r0));
        for (int i = tid; i < n; i += NT) PB[i] = 0.f;
    };
    auto tile_list = [&]() { return reinterpret_cast<const unsigned short*>(smem + I.tl); };
    ChainPos& ch = ctl->ch;  // (thread 0 of each CTA moves it)
    int fslot = 0, dslot = 0;  // halves of the warp-sum slots, alternated

    // ---- sums in the order of k_cgls.  Virtual warp w is taken by CTA w mod
    // C (by one of its last warps); its sum goes to every CTA, and after a
    // cl_sync every CTA adds the eight warp sums as k_cgls does
    auto tile_at = [&](int t, int& ty, int& tx) {
        const int w = g.tiles_x;
        ty = t / w;
        tx = t - ty * w;
    };
    // FP64 (block_sum): chain(v) is virtual thread v's sum
    auto dsum_start = [&](auto&& chain) {
        dslot ^= 1;
        for (int w = (int)rank + (NT / 32 - 1 - warp) * (int)C; w < NVW; w += (NT / 32) * (int)C) {
            const double s = warp_sum(chain(32 * w + lane));
            if (lane < (int)C) cl_st(cl_map(smem_addr(&ctl->wd[dslot][w]), lane), s);
        }
    };
    auto dsum_end = [&]() {
        const double* r = ctl->wd[dslot];
        return ((r[0] + r[4]) + (r[2] + r[6])) + ((r[1] + r[5]) + (r[3] + r[7]));
    };
    // (terms are loaded eight at a time, so that the loads' latencies overlap)
    auto squares = [&](const double* a, int n) {
        return [=](int v) {
            double s = 0.0;
            for (int i = v; i < n; i += 8 * VT) {
                double t[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) t[j] = i + j * VT < n ? __ldcg(a + i + j * VT) : 0.0;
#pragma unroll
                for (int j = 0; j < 8; ++j) s += t[j] * t[j];
            }
            return s;
        };
    };
    // FP32 (block_sum_to0, by one thread of each CTA)
    auto fsum_start = [&](auto&& chain) {
        fslot ^= 1;
        for (int w = (int)rank + (NT / 32 - 1 - warp) * (int)C; w < NVW; w += (NT / 32) * (int)C) {
            float s = chain(32 * w + lane);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane < (int)C) cl_st(cl_map(smem_addr(&ctl->ws[fslot][w]), lane), s);
        }
    };
    auto fsum_end = [&]() {
        double t = 0.0;
        for (int i = 0; i < NVW; ++i) t += (double)ctl->ws[fslot][i];
        return t;
    };
    auto grad_chain = [&](int v) {
        const float *ga = I.gvg, *za = I.zg;
        const int n = g.ns;
        float s = 0.f;
        for (int i = v; i < n; i += 8 * VT) {
            float a[8], b[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                a[j] = i + j * VT < n ? __ldcg(ga + i + j * VT) : 0.f;
                b[j] = i + j * VT < n ? __ldcg(za + i + j * VT) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) s = fmaf(a[j], b[j], s);
        }
        return s;
    };

    if (tid == 0) ch = ChainPos();
    while (true) {
        cl_sync();
        if (tid == 0) ctl->more = ch.next();
        __syncthreads();
        if (!ctl->more) {
            if (rank == 0 && tid == 0) {
                const int it = atomicAdd(A.counter, 1);
                for (unsigned r = 0; r < C; ++r) cl_st(cl_map(smem_addr(&ctl->item), r), it);
            }
            cl_sync();
            if (ctl->item >= A.n_items) break;
            if (tid == 0) ch.start(A.items[ctl->item]);
        }
        if (tid == 0)
            cluster_item_fill(I, A.probs[A.cand_prob[ch.c]], A, ch.c, ch.k, (int)C, (int)rank, (int)(blockIdx.x / C));
        __syncthreads();
        auto item_at = [&]() { return (long long)ch.c * A.max_lam + ch.k; };
        if (I.cstat & (ST_BADPARAM | ST_EMPTY)) {
            if (rank == 0) {
                const long long ok = item_at();
                float* X = A.X + ok * A.max_ns;
                for (int i = tid; i < g.ns; i += NT) X[i] = 0.f;
                if (tid == 0) {
                    A.chi2[ok] = (I.cstat & ST_BADPARAM) ? __longlong_as_double(0x7ff0000000000000LL) : 0.0;
                    A.reg[ok] = 0.0;
                    A.iters[ok] = 0;
                    if (A.relres) A.relres[ok] = 0.0;
                    if (A.istat) A.istat[ok] = I.cstat;
                }
            }
            __syncthreads();
            if (tid == 0) ch.prev_ok = false;
            continue;
        }

        // ---- cut of the source rows: the smallest row whose rays start at or
        // after the CTA's share, within the rows that a CTA has room for
        if (tid < (int)C) {
            const int want = (int)(((long long)tid * g.nent) / (int)C);
            int lo = 0, hi = g.sy - 1;
            while (lo < hi) {
                const int m = (lo + hi) >> 1;
                if (I.cst[m * g.ncx] >= want)
                    hi = m;
                else
                    lo = m + 1;
            }
            ctl->row[tid] = tid == 0 ? 0 : lo;
        }
        {  // first and last tile row with a mapped pixel
            int lo = I.g.plen, hi = 0;
            const Entry<float>* E = I.E;
            const int n = g.nent;
#pragma unroll 8
            for (int e = tid; e < n; e += NT) {
                const int pp = E[e].ppos;
                lo = min(lo, pp);
                hi = max(hi, pp);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0) {
                atomicMin(&I.tyA, (lo / g.Wp - HK) / TILE);
                atomicMax(&I.tyB, (hi / g.Wp - HK) / TILE + 1);
            }
        }
        __syncthreads();
        if (tid == 0) {
            const int cap = ClusterCut(A.probs[A.cand_prob[ch.c]], (int)C, A.max_smem).cap;
            ctl->row[C] = g.sy;
            for (int j = 1; j < (int)C; ++j)
                ctl->row[j] = max(min(ctl->row[j], ctl->row[j - 1] + cap), max(ctl->row[j - 1], g.sy - ((int)C - j) * cap));
            cluster_item_rows(I, ctl->row, (int)C, (int)rank);
        }
        __syncthreads();
        for (int i = tid; i < 2 * K * KP; i += NT) {
            const int h = i / (K * KP), m = i - h * K * KP, a = m / KP, b = m - a * KP;
            // [0] flipped PSF (B), [1] PSF (B^T); rows padded to KP
            taps[i] = b >= K ? 0.f : h == 0 ? I.psf[(K - 1 - a) * K + (K - 1 - b)] : I.psf[a * K + b];
        }
        {
            float *PA = sh(I.PA), *PB = sh(I.PB);
            const int g0 = I.row0 * g.Wp, n = g.plen - g0;
            for (int i = tid; i < I.blen; i += NT) {
                PA[i] = 0.f;
                PB[i] = i < n ? I.swp[g0 + i] : 0.f;  // sqrt(W) of the band and its halo, for the preconditioner
            }
            // the FP64 images outside the tiles that are convolved: zeros in L x, and zero
            // times the data in the weighted residuals, which is a NaN, as it is in k_cgls,
            // at an unusable pixel whose value is not finite
            const int part = (g.plen + (int)C - 1) / (int)C, i1 = min((int)(rank + 1) * part, g.plen);
            for (int i = rank * part + tid; i < i1; i += NT) {
                const double z = 0.0 * (double)I.dpad[i];
                I.Pa[i] = 0.0;
                I.Pb[i] = z;
                I.Rs[i] = z;
            }
        }
        cl_sync();  // (a slice may lie in another CTA's band)
        // ---- omega = diag(B^T W B) of the own band into Pa (see lwl_diag_at)
        for (int t = tid; t < (I.ty1 - I.ty0) * TILE * I.nx4; t += NT) {
            const int y = t / I.nx4, x = t - y * I.nx4, Wp = g.Wp;
            const float* srow = sh(I.PB) + y * Wp + x + g.sh;
            float om = 0.f;
#pragma unroll 1
            for (int a = 0; a < K; ++a)
#pragma unroll
                for (int b = 0; b < K; ++b) {
                    const float f = taps[K * KP + a * KP + b], s = srow[a * Wp + b];
                    om = fmaf(f * f, s * s, om);
                }
            const int pp = (I.row0 + y + HK) * Wp + x + g.xoff;
            I.Pa[pp] = (double)om;
            const double s = (double)I.swp[pp];
            I.Pb[pp] = s * s * (double)I.dpad[pp];  // W d, for ||rhs||
        }
        // ---- the own rays, with the owner of their pixel and its place there
        for (int e = I.e0 + tid; e < I.e1; e += NT) {
            const Entry<float> en = I.E[e];
            const int R = I.R, y = en.ppos / g.Wp - HK - I.tyA * TILE, o = y / R, yl = y - o * R;
            int4 q;
            q.x = (en.ppos - I.tyA * TILE * g.Wp - o * I.hop) | (o << 20) | (o > 0 && yl < HK ? 1 << 24 : 0) |
                  (o + 1 < (int)C && yl >= R - HK ? 1 << 25 : 0);
            q.y = en.base;
            q.z = __float_as_int(en.u);
            q.w = __float_as_int(en.v);
            I.rec[e] = q;
        }
        cl_sync();
        for (int i = I.i0 + tid; i < I.i1; i += NT) {
            const int ib = i / g.sx, ia = i - ib * g.sx;
            sh(I.mi)[i - I.i0] = 1.f / (lwl_diag_at<float>(g, I.E, I.cst, I.Pa, ia, ib) + I.lamT * hth_diag_at<float>(g, ia, ib));
        }
        for (int i = tid; i < I.blen; i += NT) sh(I.PB)[i] = 0.f;
        for (int e = I.e0 + tid; e < I.e1; e += NT) {  // L applied to ones marks the mapped pixels
            const int m = I.rec[e].x;
            cl_st(cl_map(smem_addr(smem) + I.PA + 4u * (m & 0xfffff), (m >> 20) & 15), 1.f);
        }
        cl_sync();
        for (int t = tid; t < I.tiles; t += NT) {
            int ty, tx;
            tile_at(t, ty, tx);
            unsigned m = 0;
            for (int q = 0; q < 16; ++q)
                if (sh(I.PA)[(ty * TILE + (q >> 2) + HK) * g.Wp + tx * TILE + (q & 3) + g.xoff] != 0.f) m |= 1u << q;
            reinterpret_cast<unsigned short*>(smem + I.mb)[t] = (unsigned short)m;
        }
        __syncthreads();
        if (warp == 0) {  // the tiles to convolve, then the others
            const unsigned short* mb = reinterpret_cast<const unsigned short*>(smem + I.mb);
            unsigned short* list = reinterpret_cast<unsigned short*>(smem + I.tl);
            int na = 0, nz = 0;
            for (int t0 = 0; t0 < I.tiles; t0 += 32) {
                const int t = t0 + lane;
                const bool in = t < I.tiles, a = in && mb[t] != 0;
                const unsigned am = __ballot_sync(0xffffffffu, a), zm = __ballot_sync(0xffffffffu, in && !a), below = (1u << lane) - 1u;
                if (a) list[na + __popc(am & below)] = (unsigned short)t;
                if (in && !a) list[I.tiles - 1 - nz - __popc(zm & below)] = (unsigned short)t;
                na += __popc(am);
                nz += __popc(zm);
            }
            if (lane == 0) I.act = na;
        }
        for (int t = tid; t < (I.ty1 - I.ty0) * TILE * I.nx4; t += NT) {  // Pa back to zero
            const int y = t / I.nx4, x = t - y * I.nx4;
            I.Pa[(I.row0 + y + HK) * g.Wp + x + g.xoff] = 0.0;
        }
        if (ch.warm && ch.prev_ok) {
            // x64 still holds the previous lambda's solution
        } else if (A.warm_x) {
            const float* x0 = A.warm_x + item_at() * A.max_ns;
            for (int i = I.i0 + tid; i < I.i1; i += NT) I.x64[i] = (double)x0[i];
        } else {
            for (int i = I.i0 + tid; i < I.i1; i += NT) I.x64[i] = 0.0;
        }
        __syncthreads();

        // this thread's first ray of L^T, where one stage holds them all (see there)
        auto run_at = [](int t, int n) { return (int)((long long)t * n / NT); };
        int run0 = run_at(tid, I.r1 - I.r0);
        if (run0 > 0)  // (with fewer rays than threads several shares start at 0)
            while (run0 < I.r1 - I.r0 && I.rec[I.r0 + run0].y == I.rec[I.r0 + run0 - 1].y) ++run0;

        // ---- ||rhs|| = ||L^T B^T W d|| in FP64
        cl_conv64<K, NT>(I, I.Pb, sh(I.PA), sh(I.PB), taps + K * KP, tile_list(), 1);
        cl_sync();
        for (int i = I.i0 + tid; i < I.i1; i += NT) {
            const int ib = i / g.sx, ia = i - ib * g.sx;
            I.sv[i] = apply_LT_at<float, double, double, false>(g, I.E64, I.cst, I.Pc, ia, ib);
        }
        cl_sync();
        dsum_start(squares(I.sv, g.ns));
        cl_sync();
        if (tid == 0) ctl->rhsn = sqrt(dsum_end());

        int status = 0, total_it = 0, slow = 0;
        constexpr int MAX_OUTER = 16;
        bool reverted = false;
        for (int outer = 0;; ++outer) {
            // ---- FP64 residual of x64 (residual64)
            {
                const Entry<double>* E64 = I.E64;
                const double* x64 = I.x64;
                double* Pa = I.Pa;
                const int sx = g.sx, e1 = I.e1;
                for (int e = I.e0 + tid; e < e1; e += NT) {
                    const Entry<double> en = E64[e];
                    const double u = en.u, vv = en.v;
                    const double* s0 = x64 + en.base;
                    const double s00 = __ldcg(s0), s10 = __ldcg(s0 + 1), s01 = __ldcg(s0 + sx), s11 = __ldcg(s0 + sx + 1);
                    Pa[en.ppos] = (1.0 - vv) * ((1.0 - u) * s00 + u * s10) + vv * ((1.0 - u) * s01 + u * s11);
                }
            }
            for (int i = I.i0 + tid; i < I.i1; i += NT) {
                I.h64[i] = apply_H_row<float, double>(g, I.x64, i);
                if (g.nreg > g.ns) I.h64[g.ns + i] = apply_H_row<float, double>(g, I.x64, g.ns + i);
            }
            cl_sync();
            cl_conv64<K, NT>(I, I.Pa, sh(I.PA), sh(I.PB), taps, tile_list(), 0);
            cl_sync();
            dsum_start([&](int v) {
                const int nt = g.ntiles, Wp = g.Wp;
                double s = 0.0;
                for (int t = v; t < nt; t += VT) {
                    int ty, tx;
                    tile_at(t, ty, tx);
                    const double* q = I.Rs + (ty * TILE + HK) * Wp + tx * TILE + g.xoff;
                    double r[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) r[j] = __ldcg(q + (j >> 2) * Wp + (j & 3));
#pragma unroll
                    for (int j = 0; j < 16; ++j) s += r[j] * r[j];
                }
                return s;
            });
            cl_conv64<K, NT>(I, I.Pb, sh(I.PA), sh(I.PB), taps + K * KP, tile_list(), 1);
            cl_sync();
            if (rank == 0 && tid == 0) A.chi2[item_at()] = dsum_end();
            for (int i = I.i0 + tid; i < I.i1; i += NT) {
                const int ib = i / g.sx, ia = i - ib * g.sx;
                const double v = fma(-I.lam, apply_HT_at<float, double>(g, I.h64, i, ia, ib),
                                     apply_LT_at<float, double, double, false>(g, I.E64, I.cst, I.Pc, ia, ib));
                sh(I.gv)[i - I.i0] = (float)v;
                I.sv[i] = v;
            }
            dsum_start(squares(I.h64, g.nreg));
            cl_sync();
            if (rank == 0 && tid == 0) A.reg[item_at()] = dsum_end();
            dsum_start(squares(I.sv, g.ns));
            cl_sync();
            const double rel64 = ctl->rhsn > 0 ? sqrt(dsum_end()) / ctl->rhsn : 0.0, prev_rel = outer > 0 ? ctl->prev_rel : 1e300;
            if (A.relres && rank == 0 && tid == 0) A.relres[item_at()] = rel64;
            if (reverted) {  // the best iterate, evaluated again
                status |= ST_STAG;
                break;
            }
            if (outer > 0 && !(rel64 <= prev_rel)) {  // back to the best iterate (see k_cgls)
                for (int i = I.i0 + tid; i < I.i1; i += NT) I.x64[i] = I.xb[i];
                cl_sync();
                reverted = true;
                continue;
            }
            if (!isfinite(rel64)) {
                status |= ST_BREAK;
                break;
            }
            if (!(rel64 > A.tol)) break;
            const int maxit = A.maxit > 0 ? A.maxit : 25 * g.ns;
            if (total_it >= maxit || outer >= MAX_OUTER) {
                status |= ST_MAXIT;
                break;
            }
            slow = (outer > 0 && rel64 > 0.9 * prev_rel) ? slow + 1 : 0;
            if (slow >= 2) {
                status |= ST_STAG;
                break;
            }
            // ---- inner solve of A d = r by Jacobi-preconditioned CG from d = 0
            for (int i = I.i0 + tid; i < I.i1; i += NT) {
                I.xb[i] = I.x64[i];
                I.xg[i] = 0.f;
                const float gv = sh(I.gv)[i - I.i0];
                I.gvg[i] = gv;
                I.zg[i] = sh(I.mi)[i - I.i0] * gv;
            }
            cl_sync();
            for (int j = I.pr0 * g.sx + tid; j < I.pr1 * g.sx; j += NT) sh(I.p)[j - I.pr0 * g.sx] = __ldcg(I.zg + j);
            fsum_start(grad_chain);
            cl_sync();
            if (tid == 0) {
                ctl->prev_rel = rel64;
                ctl->target = fmax(A.eta, fmin(MAX_TARGET, FINAL_MARGIN * A.tol / rel64));
                const double gam = fsum_end();
                ctl->gam = gam;
                ctl->g0 = gam;
                ctl->best = 1.0;
                ctl->best_it = 0;
                ctl->it = 0;
                ctl->total_it = total_it;
                ctl->brk = !isfinite(gam);
                ctl->stop = ctl->brk || !(gam > 0.0) || total_it >= maxit;
            }
            __syncthreads();
            while (!ctl->stop) {
                // L p of the own rays, to the bands that hold their pixels
                {
                    float *PA = sh(I.PA), *p = sh(I.p) - I.pr0 * g.sx;
                    const unsigned PAs = smem_addr(PA);
                    const int4* rec = I.rec;
                    const int sx = g.sx, e1 = I.e1, hop = I.hop;
                    for (int e = I.e0 + tid; e < e1; e += 8 * NT) {
                        int4 q[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) q[j] = rec[min(e + j * NT, e1 - 1)];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float u = __int_as_float(q[j].z), v = __int_as_float(q[j].w);
                            const float* s0 = p + q[j].y;
                            const float val = (1.f - v) * ((1.f - u) * s0[0] + u * s0[1]) + v * ((1.f - u) * s0[sx] + u * s0[sx + 1]);
                            if (e + j * NT < e1) {
                                const int m = q[j].x;
                                const unsigned a = PAs + 4u * (m & 0xfffff), o = (m >> 20) & 15;
                                if (o == rank)
                                    PA[m & 0xfffff] = val;
                                else
                                    cl_st(cl_map(a, o), val);
                                if (m & (1 << 24)) cl_st(cl_map(a + 4u * hop, o - 1), val);
                                if (m & (1 << 25)) cl_st(cl_map(a - 4u * hop, o + 1), val);
                            }
                        }
                    }
                }
                // H p of the own rows and the rows next to them
                {
                    const float* pv = sh(I.p) - I.pr0 * g.sx;  // indexed by source pixel
                    float* h = sh(I.h) - I.hr0 * g.sx;
                    const int j1 = I.hr1 * g.sx, i0 = I.i0, i1 = I.i1;
                    for (int i = I.hr0 * g.sx + tid; i < j1; i += NT) {
                        const bool mine = i >= i0 && i < i1;
                        const float v = apply_H_row<float, float>(g, pv, i);
                        h[i] = v;
                        if (mine) I.hg[i] = v;
                        if (g.nreg > g.ns) {
                            const float v2 = apply_H_row<float, float>(g, pv, g.ns + i);
                            h[I.hn + i] = v2;
                            if (mine) I.hg[g.ns + i] = v2;
                        }
                    }
                }
                cl_sync();  // bands of L p complete
                // sqrt(W) B L p into Z, W B L p into the band and its neighbours' halos
                {
                    const int act = I.act, Wp = g.Wp, nx4 = I.nx4, xoff = g.xoff;
                    const unsigned short* list = tile_list();
                    for (int i = I.tiles - 1 - tid; i >= act; i -= NT) {  // the others' zeros for delta's sum
                        int ty, tx;
                        tile_at(list[i], ty, tx);
                        float* zt = sh(I.Z) + ty * TILE * nx4 + tx * TILE;
#pragma unroll
                        for (int r = 0; r < TILE; ++r) st4(zt + r * nx4, V4<float>{{0.f, 0.f, 0.f, 0.f}});
                    }
                    const int R = I.R, hop = I.hop;
                    by_rows(act, [&](auto rt) {
                        constexpr int RT = decltype(rt)::value;
                        for (int i = tid; i < act * (TILE / RT); i += NT) {
                            const int part = i / act;
                            int ty, tx;
                            tile_at(list[i - part * act], ty, tx);
                            const int y0 = ty * TILE + part * RT;
                            float* zt = sh(I.Z) + y0 * nx4 + tx * TILE;
                            // sqrt(W) of the rows arrives in its place of Z while they are convolved
                            const float* sg = I.swp + (I.row0 + y0 + HK) * Wp + tx * TILE + xoff;
#pragma unroll
                            for (int r = 0; r < RT; ++r) cl_copy16(smem_addr(zt + r * nx4), sg + r * Wp);
                            float acc[RT][TILE];
                            conv4<K, RT>(sh(I.PA) + y0 * Wp + tx * TILE, Wp, taps, acc);
                            cl_copy_wait();
                            float* PB = sh(I.PB);
#pragma unroll
                            for (int r = 0; r < RT; ++r) {
                                const int y = y0 + r, lp = (y + HK) * Wp + tx * TILE + xoff;
                                const V4<float> sw = ld4(zt + r * nx4);
                                V4<float> o, w;
#pragma unroll
                                for (int cc = 0; cc < 4; ++cc) {
                                    o.v[cc] = sw.v[cc] * acc[r][cc];
                                    w.v[cc] = sw.v[cc] * o.v[cc];
                                }
                                st4(zt + r * nx4, o);
                                st4(PB + lp, w);
                                if (rank > 0 && y < HK) cl_st4(cl_map(smem_addr(PB + lp + hop), rank - 1), w.v);
                                if (rank + 1 < C && y >= R - HK) cl_st4(cl_map(smem_addr(PB + lp) - 4u * hop, rank + 1), w.v);
                            }
                        }
                    });
                }
                cl_sync();  // bands of W B L p and all of Z complete
                // delta = p^T A p = ||sqrt(W) B L p||^2 + lam ||H p||^2
                fsum_start([&](int v) {
                    const float* hg = I.hg;
                    const int nr = g.nreg, nt = g.ntiles, nx4 = I.nx4, bt = I.bt;
                    const unsigned Zs = smem_addr(smem) + I.Z;
                    float dh = 0.f, cq = 0.f, q[2][16];
                    // (tiles outside the bands are zeros)
                    const int tA = I.tyA * g.tiles_x, tB = min(I.tyB * g.tiles_x, nt), tyA = I.tyA;
                    const int t0 = v + (tA > v ? (tA - v + VT - 1) / VT * VT : 0);
                    auto load_tiles = [&](int t) {
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            int ty, tx;
                            tile_at(min(t + j * VT, tB - 1), ty, tx);
                            const int o = (ty - tyA) / bt;
                            const unsigned a = cl_map(Zs + 4u * ((ty - tyA - o * bt) * TILE * nx4 + tx * TILE), o);
#pragma unroll
                            for (int r = 0; r < TILE; ++r) cl_ld4(a + 4u * r * nx4, q[j] + 4 * r);
                        }
                    };
                    load_tiles(t0);
                    for (int i = v; i < nr; i += 16 * VT) {
                        float h[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) h[j] = i + j * VT < nr ? __ldcg(hg + i + j * VT) : 0.f;
#pragma unroll
                        for (int j = 0; j < 16; ++j) dh = fmaf(h[j], h[j], dh);
                    }
                    for (int t = t0; t < tB; t += 2 * VT) {
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            if (t + j * VT < tB) {
#pragma unroll
                                for (int m = 0; m < 16; ++m) cq = fmaf(q[j][m], q[j][m], cq);
                            }
                        if (t + 2 * VT < tB) load_tiles(t + 2 * VT);
                    }
                    return fmaf(I.lamT, dh, cq);
                });
                // u = B^T W B L p of the own band, at mapped pixels (the others stay zero)
                {
                    const int act = I.act, Wp = g.Wp;
                    const unsigned short* list = tile_list();
                    by_rows(act, [&](auto rt) {
                        constexpr int RT = decltype(rt)::value;
                        for (int i = tid; i < act * (TILE / RT); i += NT) {
                            const int part = i / act, t = list[i - part * act];
                            int ty, tx;
                            tile_at(t, ty, tx);
                            const int y0 = ty * TILE + part * RT;
                            float acc[RT][TILE];
                            conv4<K, RT>(sh(I.PB) + y0 * Wp + tx * TILE, Wp, taps + K * KP, acc);
                            float* PA = sh(I.PA) + (y0 + HK) * Wp + tx * TILE + g.xoff;
                            const unsigned m = reinterpret_cast<unsigned short*>(smem + I.mb)[t] >> (4 * part * RT);
#pragma unroll
                            for (int r = 0; r < RT; ++r)
#pragma unroll
                                for (int cc = 0; cc < 4; ++cc)
                                    if (m & (1u << (r * 4 + cc))) PA[r * Wp + cc] = acc[r][cc];
                        }
                    });
                }
                cl_sync();  // u complete, delta's warp sums here, Z read
                if (tid == 0) {
                    const double delta = fsum_end();
                    if (!(delta > 0.0) || !isfinite(delta)) {
                        ctl->brk = 1;
                        ctl->stop = 1;
                    } else {
                        ctl->a = (float)(ctl->gam / delta);
                    }
                }
                // L^T u: the four corner sums of each cell's rays, in ray order.  The
                // rays' u, weights and cells are staged in the band of W B L p (loads
                // coalesced, eight in flight a thread); then every thread walks an
                // equal run of whole cells (a cell belongs to the run that its first
                // ray falls in), so that the lanes of a warp stay about equally busy:
                // one cell a lane had a warp wait for its fullest cell (measured:
                // 12k against 5k clocks at 128 x 128 on two SMs).
                // Where the cell sums would not fit an image (a source about as fine as
                // the image), k_cgls sums each source pixel's rays directly, and so does
                // this: then the rays are only staged, with the starts of their cells
                {
                    float4* S = reinterpret_cast<float4*>(sh(I.PB));
                    const float* PA = sh(I.PA);
                    const unsigned PAs = smem_addr(PA);
                    const int4* rec = I.rec;
                    float4* Zc = reinterpret_cast<float4*>(sh(I.Z)) - I.hr0 * g.sx;  // indexed by the cell's base
                    const int n4 = I.i1 - I.hr0 * g.sx;
                    const int r1 = I.r1, stage = I.stage;
                    const bool gather = I.gather;
                    if (gather) {
                        int* cz = reinterpret_cast<int*>(sh(I.Z));
                        for (int i = I.cell0 + tid; i <= I.cell1; i += NT) cz[i - I.cell0] = I.cst[i] - I.r0;
                    } else {
                        for (int i = tid; i < n4; i += NT) Zc[I.hr0 * g.sx + i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    for (int s0 = I.r0; s0 < r1; s0 += stage) {
                        if (gather && r1 - I.r0 > stage) break;  // (read where they are)
                        const int n = min(stage, r1 - s0);
                        for (int e = tid; e < n; e += 8 * NT) {
                            int4 q[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) q[j] = rec[s0 + min(e + j * NT, n - 1)];
                            float U[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const unsigned o = (q[j].x >> 20) & 15;
                                U[j] = o == rank ? PA[q[j].x & 0xfffff] : cl_ld(cl_map(PAs + 4u * (q[j].x & 0xfffff), o));
                            }
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                if (e + j * NT < n)
                                    S[e + j * NT] = make_float4(U[j], __int_as_float(q[j].z), __int_as_float(q[j].w), __int_as_float(q[j].y));
                        }
                        if (gather) break;
                        __syncthreads();
                        // this thread's run [k0, k1): from the first cell start at or after its
                        // share's start to the next thread's.  A cell that the stage cuts
                        // goes on from its stored sums (by thread 0 of the next pass)
                        int k0 = run0;
                        const int k1 = run_at(tid + 1, n);
                        if (n < r1 - I.r0) {
                            k0 = run_at(tid, n);
                            if (k0 > 0)
                                while (k0 < n && __float_as_int(S[k0].w) == __float_as_int(S[k0 - 1].w)) ++k0;
                        }
                        if (k1 > k0) {
                            int key = __float_as_int(S[k0].w);
                            float4 c = Zc[key];
                            bool go = true;
                            for (int m = k0; go; m += 4) {  // four rays' loads together
                                float4 r[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) r[j] = S[min(m + j, n - 1)];
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    if (go) {
                                        const int kn = __float_as_int(r[j].w);
                                        if (m + j >= n || kn != key) {  // a cell is complete (or the stage's end reached)
                                            Zc[key] = c;
                                            go = m + j < k1;
                                            c = make_float4(0.f, 0.f, 0.f, 0.f);
                                            key = kn;
                                        }
                                        const float uU = r[j].y * r[j].x, u0 = r[j].x - uU;  // u U, (1-u) U
                                        c.x = fmaf(1.f - r[j].z, u0, c.x);
                                        c.y = fmaf(1.f - r[j].z, uU, c.y);
                                        c.z = fmaf(r[j].z, u0, c.z);
                                        c.w = fmaf(r[j].z, uU, c.w);
                                    }
                            }
                        }
                        if (s0 + stage < r1) __syncthreads();  // the stage is free again
                    }
                }
                __syncthreads();
                if (ctl->brk) break;
                // ... then per source pixel the corners it receives, and the CG updates
                {
                    const float a = ctl->a, lamT = I.lamT, invNp = g.invNp;
                    const int sx = g.sx, sy = g.sy, i0 = I.i0, i1 = I.i1;
                    const float* cp = sh(I.Z) - 4 * I.hr0 * sx;
                    const bool gather = I.gather, staged = I.r1 - I.r0 <= I.stage;
                    auto ray_at = [&](int k) {  // ray r0 + k: U, u, v
                        if (staged) return reinterpret_cast<const float4*>(sh(I.PB))[k];
                        const int4 q = I.rec[I.r0 + k];
                        const unsigned o = (q.x >> 20) & 15;
                        const float U = cl_ld(cl_map(smem_addr(smem) + I.PA + 4u * (q.x & 0xfffff), o));
                        return make_float4(U, __int_as_float(q.z), __int_as_float(q.w), 0.f);
                    };
                    const float* hx = sh(I.h) - I.hr0 * sx;
                    float *gv_sh = sh(I.gv) - i0, *mi = sh(I.mi) - i0;
                    for (int i = i0 + tid; i < i1; i += NT) {
                        const int ib = i / sx, ia = i - ib * sx;
                        float acc = 0.f;
                        if (gather) {
#pragma unroll
                            for (int d = 0; d < 4; ++d) {
                                const int iy0 = ib - (d >> 1), ix0 = ia - (d & 1);
                                if (iy0 < 0 || iy0 > sy - 2 || ix0 < 0 || ix0 > sx - 2) continue;
                                const int* cz = reinterpret_cast<const int*>(sh(I.Z)) + (iy0 * (sx - 1) + ix0 - I.cell0);
                                const int k1 = cz[1];
                                for (int k = cz[0]; k < k1; k += 4) {  // four rays' loads together
                                    float4 r[4];
#pragma unroll
                                    for (int j = 0; j < 4; ++j) r[j] = ray_at(min(k + j, k1 - 1));
#pragma unroll
                                    for (int j = 0; j < 4; ++j)
                                        if (k + j < k1)
                                            acc = fmaf((d & 1 ? r[j].y : 1.f - r[j].y) * (d & 2 ? r[j].z : 1.f - r[j].z), r[j].x, acc);
                                }
                            }
                        } else {
                            if (ib <= sy - 2 && ia <= sx - 2) acc += cp[4 * i + 0];
                            if (ib <= sy - 2 && ia >= 1) acc += cp[4 * (i - 1) + 1];
                            if (ib >= 1 && ia <= sx - 2) acc += cp[4 * (i - sx) + 2];
                            if (ib >= 1 && ia >= 1) acc += cp[4 * (i - sx - 1) + 3];
                        }
                        float ht;
                        if (g.reg == 1) {
                            const float* hy = hx + I.hn;
                            ht = -hx[i] - hy[i];
                            if (ia > 0) ht += hx[i - 1];
                            if (ib > 0) ht += hy[i - sx];
                        } else {
                            ht = apply_HT_at<float, float>(g, hx, i, ia, ib);
                        }
                        const float ap = gather ? fmaf(lamT, ht, acc) : acc * invNp + lamT * ht;  // (invNp = 1)
                        const float gv = fmaf(-a, ap, gv_sh[i]);
                        gv_sh[i] = gv;
                        I.gvg[i] = gv;
                        I.zg[i] = mi[i] * gv;
                    }
                    if (!gather) clear_stage();
                }
                cl_sync();  // g and z complete
                if (I.gather) clear_stage();
                fsum_start(grad_chain);
                {
                    const float a = ctl->a;
                    const float* pv = sh(I.p) - I.pr0 * g.sx;
                    float *xg = I.xg, *z_sh = sh(I.Z);  // (Z is free again)
                    const float* zg = I.zg;
                    const int i1 = I.i1, j0 = I.pr0 * g.sx, j1 = I.pr1 * g.sx;
                    for (int j = j0 + tid; j < j1; j += NT) z_sh[j - j0] = __ldcg(zg + j);  // for the p update
                    for (int i = I.i0 + tid; i < i1; i += NT) xg[i] = fmaf(a, pv[i], xg[i]);
                }
                cl_sync();  // gamma's warp sums here
                if (tid == 0) {
                    const double gnew = fsum_end();
                    ctl->b = (float)(gnew / ctl->gam);
                    ctl->gam = gnew;
                }
                if (tid == 32) {  // (beside beta's division)
                    const double gnew = fsum_end();
                    const int it = ++ctl->it;
                    ++ctl->total_it;
                    // The decisions of k_cgls, with rel = sqrt(gnew / g0): in FP64 only
                    // where a single-precision ratio (good to 1e-6) leaves them open
                    const float ratio = __fdividef((float)gnew, (float)ctl->g0);
                    const float tt = (float)ctl->target, hb = 0.5f * (float)ctl->best;
                    const bool clear = (float)gnew > 1e-30f && (float)ctl->g0 > 1e-30f && ratio < 1e30f &&
                                       ratio > 1.0001f * (tt * tt) && ratio > 1.0001f * (hb * hb);
                    if (clear && ctl->total_it < (A.maxit > 0 ? A.maxit : 25 * g.ns) &&
                        it - ctl->best_it <= max(4000, 2 * g.ns)) {
                        // above the target and no halving of the residual: go on
                    } else {
                        const double rel = sqrt(gnew / ctl->g0);
                        if (!isfinite(gnew)) {
                            ctl->brk = 1;
                            ctl->stop = 1;
                        } else if (!(rel > ctl->target) || ctl->total_it >= (A.maxit > 0 ? A.maxit : 25 * g.ns)) {
                            ctl->stop = 1;
                        } else if (rel < 0.5 * ctl->best) {
                            ctl->best = rel;
                            ctl->best_it = it;
                        } else if (it - ctl->best_it > max(4000, 2 * g.ns)) {
                            ctl->stop = 1;
                        }
                    }
                }
                __syncthreads();
                // p of the own rows and of the rows around them
                {
                    const float bt = ctl->b;
                    float *p = sh(I.p), *z_sh = sh(I.Z);
                    const int n = (I.pr1 - I.pr0) * g.sx;
                    for (int j = tid; j < n; j += NT) p[j] = fmaf(bt, p[j], z_sh[j]);
                }
                __syncthreads();
            }
            total_it = ctl->total_it;
            if (ctl->brk) {
                status |= ST_BREAK;
                break;
            }
            for (int i = I.i0 + tid; i < I.i1; i += NT) I.x64[i] += (double)I.xg[i];
            cl_sync();
        }
        {
            const long long ok = item_at();
            float* X = A.X + ok * A.max_ns;
            for (int i = I.i0 + tid; i < I.i1; i += NT) X[i] = (float)I.x64[i];
            if (rank == 0 && tid == 0) {
                A.iters[ok] = total_it;
                if (A.istat) A.istat[ok] = status | I.cstat;
            }
        }
        __syncthreads();
        if (tid == 0) ch.prev_ok = !(status & ST_BREAK);
    }
}

}  // namespace mirage
