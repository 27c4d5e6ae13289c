// The single-slice projector bodies shared by the single-state kernels, the
// persistent batched phases and the dependency-driven batched epoch: the
// forward band-chunk body (forward_tile_body) and the tiled back projection
// with its update epilogue (back_tile_body).
//
// COH: the images and ratios the body reads may have been written earlier in
// the same kernel launch (the dependency-driven epoch), so they are read with
// plain loads instead of the read-only data path.  WIDE (forward): the block
// is wider than kBlock threads; the threads past kBlock take part in the
// barriers only.
#pragma once

#include "epilogue.cuh"

namespace petvr {

namespace {

constexpr int kTile = 16;           // single slice: a block owns a kTile x kTile tile (kTile^2 == kBlock)
constexpr int kChunk = 16;          // views per shared-memory pass
constexpr int kTileBlockMax = 1024; // threads of a tile block: kTile * kTile / run per view of a chunk
// Threads of a persistent back block: one 256-thread block per tile, whose
// threads loop over the runs of subsets with more than 8 views (run 8) or 4
// views (run 4).  Measured on the 64-reconstruction batch (most members need
// 512 threads for one run per thread): 118k pairs/s at 256 threads (five
// blocks per SM), 111k at 288-320, 102k at 512 (two blocks per SM).
constexpr int kPersistentBackMax = 256;
constexpr int kPersistentBackRegs = 48;  // five 256-thread blocks per SM

// The bands [kb, ke) of one ray from this thread, every fourth one from kb on:
// sum of share times pixel, in units of the ray length per band.
//
// A band costs ~16 instructions: its lower end from the batch's base by one
// FMA, the floor by a directed-rounding add (kRound), the share by one
// saturating multiply, then two loads and three FMAs.  256^2, ncu: a full ratio
// pass 23.2 us and 14.4M warp instructions (33.2 us and 22.0M with floorf, the
// comparison of both band ends and contiguous bands per lane), a subset pass
// 6.9 us (7.9).
template <bool COH>
__device__ __forceinline__ float walk_bands(const FwdArgs &a, const ViewParams &vp, float uf, int ui, float hm,
                                            int n_minor, int kb, int ke) {
    const int s_major = vp.col ? 1 : a.nx;
    const int s_minor = vp.col ? a.nx : 1;
    const float *img1 = a.img + s_minor;
    // the band's lower end is at its far boundary when the line moves down
    const float k_end = (vp.du < 0.0f ? 1.0f : 0.0f) - hm;
    float acc = 0.0f;
    // kBatch bands at a time: all their offsets and shares first, then the
    // loads, then the FMAs in band order, so that the loads of a batch are in
    // flight together.
    constexpr int kBatch = 4;
    for (int k = kb; k < ke; k += 4 * kBatch) {
        // the batch's base position: the integer part of kc du goes into the
        // pixel index, so that what is left stays small and exact
        const float kc = (float)k + k_end;
        const float tp = fmaf(kc, vp.du, kRound);
        const float base = uf + fmaf(kc, vp.du_lo, fmaf(kc, vp.du, kRound - tp));
        const unsigned iu = (unsigned)ui + __float_as_uint(tp) - 2u * kRoundBits;
        int m0[kBatch];
        float c0[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const float lo = fmaf(4.0f * (float)b, vp.du, base);
            const float t = __fadd_rd(lo, kRound);
            m0[b] = (int)(__float_as_uint(t) + iu);
            c0[b] = band_share(t - (kRound - 1.0f), lo, vp.inv_adu);
        }
        // a piece outside the image (or of a band past ke) is not loaded and
        // adds 0; the upper pixel is loaded only where the line reaches it.
        // lo is monotone in b, so when both pixels of the first and last band
        // are inside the image every band's are: no checks then.
        float x0[kBatch], x1[kBatch];
        const int off = k * s_major;
        if (k + 4 * (kBatch - 1) < ke && (unsigned)m0[0] < (unsigned)(n_minor - 1) &&
            (unsigned)m0[kBatch - 1] < (unsigned)(n_minor - 1)) {
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int o = m0[b] * s_minor + (off + 4 * b * s_major);
                x0[b] = ld_data<COH>(a.img + o);
                x1[b] = c0[b] < 1.0f ? ld_data<COH>(img1 + o) : 0.0f;
            }
        } else {
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int o = m0[b] * s_minor + (off + 4 * b * s_major);
                const bool live = k + 4 * b < ke;
                x0[b] = live && (unsigned)m0[b] < (unsigned)n_minor ? ld_data<COH>(a.img + o) : 0.0f;
                x1[b] = live && c0[b] < 1.0f && (unsigned)(m0[b] + 1) < (unsigned)n_minor ? ld_data<COH>(img1 + o)
                                                                                         : 0.0f;
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            acc = fmaf(c0[b], x0[b], acc);
            acc = fmaf(1.0f - c0[b], x1[b], acc);
        }
    }
    return acc * vp.L;
}

// The same for the consecutive bands [kb, ke), with the weights of
// band_split() in its own rounding (states with a BF16 table, see kRefRounding).
template <bool COH>
__device__ __forceinline__ float walk_bands_ref(const FwdArgs &a, const ViewParams &vp, float uf, int ui, float hm,
                                                int n_minor, int kb, int ke) {
    const int s_major = vp.col ? 1 : a.nx;
    const int s_minor = vp.col ? a.nx : 1;
    const float *img1 = a.img + s_minor;
    float acc = 0.0f;
    float kc = (float)kb - hm;
    float va = band_point(vp, uf, kc);
    constexpr int kBatch = 4;
    for (int k = kb; k < ke; k += kBatch) {
        int m0[kBatch];
        float c0[kBatch], c1[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            kc += 1.0f;
            const float vb = band_point(vp, uf, kc);
            const float t = band_split_ref(vp, va, vb, c0[b], c1[b]);
            m0[b] = (int)(__float_as_uint(t) - kRoundBits) + ui;
            va = vb;
        }
        float x0[kBatch], x1[kBatch];
        const int off = k * s_major;
        if (k + kBatch <= ke && (unsigned)m0[0] < (unsigned)(n_minor - 1) &&
            (unsigned)m0[kBatch - 1] < (unsigned)(n_minor - 1)) {
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int o = m0[b] * s_minor + (off + b * s_major);
                x0[b] = ld_data<COH>(a.img + o);
                x1[b] = c1[b] != 0.0f ? ld_data<COH>(img1 + o) : 0.0f;
            }
        } else {
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int o = m0[b] * s_minor + (off + b * s_major);
                const bool live = k + b < ke;
                x0[b] = live && (unsigned)m0[b] < (unsigned)n_minor ? ld_data<COH>(a.img + o) : 0.0f;
                x1[b] = live && c1[b] > 0.0f && (unsigned)(m0[b] + 1) < (unsigned)n_minor ? ld_data<COH>(img1 + o)
                                                                                         : 0.0f;
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            acc = fmaf(c0[b], x0[b], acc);
            acc = fmaf(c1[b], x1[b], acc);
        }
    }
    return acc;
}

// Single-slice forward: a block takes RAYS adjacent rays of the view range
// and splits each ray's bands over CHUNKS threads (RAYS * CHUNKS = kBlock): a
// warp is 8 adjacent rays times 4 band lanes, and the CHUNKS / 4 warps of a ray
// group take contiguous ranges of bands.  Inside a warp's range the 4 lanes
// take every fourth band, so that one load touches 8 neighbouring pixels of 4
// rows on a row-driven view and 4 neighbouring columns of the ~10 rows the 8
// rays cross on a column-driven one (with contiguous chunks per lane those
// were 32 different rows).  REF: consecutive bands per lane (kRefRounding).
//
// Chunk sums are reduced by xor-shuffles (within the warp) and then over
// warps through shared memory, always in the same order, so the result is
// deterministic.
template <int CHUNKS, int MODE, bool LL, bool REF = false, bool COH = false, bool WIDE = false>
__device__ __forceinline__ void forward_tile_body(const FwdArgs &a, const int bx) {
    constexpr int RAYS = kBlock / CHUNKS;        // rays per block
    constexpr int WPG = CHUNKS / 4;              // warps per group of 8 rays
    const RayRange rr = ray_range(a);
    const int n_rays = (rr.v_end - rr.v_begin) * a.nb;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int r8 = lane & 7;
    const int c4 = lane >> 3;                    // band lane
    const int ray_local = 8 * (warp / WPG) + r8;
    const int ray = bx * RAYS + ray_local;     // 32-bit: a plan has fewer than 2^31 rays

    // the ray's geometry: plan constants only, so it may overlap the end of
    // the kernel before this one
    ViewParams vp{};
    float uf = 0.0f;
    int kb = 0, ke = 0, n_minor = 0, ui = 0;
    float hm = 0.0f;
    // WIDE: a block wider than kBlock; its threads past kBlock take no ray
    if (ray < n_rays && (!WIDE || threadIdx.x < kBlock)) {
        const int q = div_by_bins(ray, a.nb_mul, a.nb_shift);
        const int j = ray - q * a.nb;
        const int v = __ldg(a.order + rr.v_begin + q);
        vp = a.views[v];
        const float2 u = __ldg(a.uc + (long long)v * a.nb + j);
        const int n_major = vp.col ? a.nx : a.ny;
        n_minor = vp.col ? a.ny : a.nx;
        hm = 0.5f * (float)n_major;
        ui = (int)u.x + (n_minor >> 1);
        uf = u.y;
        int k_lo, k_hi;
        band_range(vp, u.x + u.y, n_major, n_minor, k_lo, k_hi);
        // the ranges are aligned to the same bands for every ray of the view,
        // so neighbouring lanes read the same image rows
        if (REF) {
            const int per = (n_major + CHUNKS - 1) / CHUNKS;
            const int chunk = 4 * (warp % WPG) + c4;
            kb = max(k_lo, chunk * per);
            ke = min(k_hi, (chunk + 1) * per);
        } else {
            const int per = ((n_major + WPG - 1) / WPG + 3) & ~3;
            const int wk = (warp % WPG) * per;
            kb = max(k_lo & ~3, wk) + c4;
            ke = min(k_hi, wk + per);
        }
    }
    pdl_wait();
    pdl_trigger();
    // counts and background of the ray this thread finishes below: issued now
    // (they may come from the kernel before, hence after the wait) so that
    // their latency hides behind the band walk
    const int ray_f = bx * RAYS + (int)threadIdx.x;
    const bool fin = threadIdx.x < RAYS && ray_f < n_rays;
    const long long gi = rr.off + ray_f;
    float g_f = 0.0f, w_f = a.w_scalar;
    if (fin) {
        if (MODE == FWD_RATIO || LL) g_f = __ldg(a.g + gi);
        if (a.w) w_f = __ldg(a.w + gi);
    }
    float acc = 0.0f;
    if (kb < ke)
        acc = REF ? walk_bands_ref<COH>(a, vp, uf, ui, hm, n_minor, kb, ke)
                  : walk_bands<COH>(a, vp, uf, ui, hm, n_minor, kb, ke);
    // the 4 chunks of each ray in this warp, then the warps of its group
    acc += __shfl_xor_sync(0xffffffffu, acc, 8);
    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
    __shared__ float red[kBlock / 32][8];
    if (lane < 8 && (!WIDE || warp < kBlock / 32)) red[warp][lane] = acc;
    __syncthreads();

    double ll = 0.0;
    if (threadIdx.x < RAYS) {
        const int g = threadIdx.x >> 3;
        float sum = 0.0f;
#pragma unroll
        for (int w = 0; w < WPG; ++w) sum += red[g * WPG + w][threadIdx.x & 7];
        if (fin) {
            const float yhat = sum + w_f;
            if (MODE == FWD_YHAT) a.out[ray_f] = yhat;
            if (MODE == FWD_RATIO || LL) {
                const float g = g_f;
                if (MODE == FWD_RATIO) a.out[ray_f] = (yhat != 0.0f) ? g / yhat : 0.0f;
                if (LL) {
                    if (yhat > 0.0f) {
                        ll = (g > 0.0f ? (double)g * (double)logf(yhat) : 0.0) - (double)yhat;
                    } else if (g > 0.0f) {
                        // g log(yhat) with yhat <= 0 and g > 0: the objective is -inf there
                        // (latched as well when the caller gave a status word)
                        ll = -(double)INFINITY;
                        if (a.status) atomicExch(a.status, (int)PET_ERR_NUMERIC);
                    } else {
                        ll = -(double)yhat;
                    }
                }
            }
        }
    }
    if (LL) {
        __shared__ double dred[kBlock / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);
        if (lane == 0 && (!WIDE || warp < kBlock / 32)) dred[warp] = ll;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < kBlock / 32; ++i) s += dred[i];
            a.ll_partials[bx] = s;
        }
    }
}

// One item of a batched forward, with the member's band-chunk count and rounding.
template <int MODE, bool LL, bool COH = false, bool WIDE = false>
__device__ __forceinline__ void forward_item(const FwdArgs &a, int shape, int bx) {
    if constexpr (MODE == FWD_RATIO && !LL) {
        if (a.ref) {
            if (shape == 8)
                forward_tile_body<8, MODE, LL, kRefRounding, COH, WIDE>(a, bx);
            else if (shape == 16)
                forward_tile_body<16, MODE, LL, kRefRounding, COH, WIDE>(a, bx);
            else
                forward_tile_body<32, MODE, LL, kRefRounding, COH, WIDE>(a, bx);
            return;
        }
    }
    if (shape == 8)
        forward_tile_body<8, MODE, LL, false, COH, WIDE>(a, bx);
    else if (shape == 16)
        forward_tile_body<16, MODE, LL, false, COH, WIDE>(a, bx);
    else
        forward_tile_body<32, MODE, LL, false, COH, WIDE>(a, bx);
}

// Single-slice path: a block owns a kTile x kTile pixel tile.  For each view,
// the tile's bands are cut into runs of kRun pixels along the view's minor
// axis; one thread walks the rays that can cross a run in band order and
// adds each ray's two band pieces into per-view partial sums in shared
// memory (every (view, pixel) slot has exactly one writer, so no atomics).
// Then each thread sums its pixel's partials over the views in a fixed order
// and applies the update.  Each ray-band split is evaluated once per run
// instead of once per pixel it touches.  Views are processed in chunks of
// kChunk to bound shared memory.
template <int EPI, typename TQ, int kRun, bool GENPOT, bool COH = false>
__device__ __forceinline__ void back_tile_body(const BackArgs &a, const int t, const int bx) {
    extern __shared__ unsigned char smem_raw[];
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    float *s_part = reinterpret_cast<float *>(smem_raw);                       // [kChunk][kTile*kTile]
    ViewParams *s_views = reinterpret_cast<ViewParams *>(s_part + kChunk * kTile * kTile);   // [kChunk]
    int *s_vid = reinterpret_cast<int *>(s_views + kChunk);
    const int r_view0 = a.t_dev ? vb : a.r_view0;
    const int nthr = blockDim.x;                  // >= kTile * kTile; one run per thread when nv <= nthr / 32

    const int tiles_x = (a.nx + kTile - 1) / kTile;
    const int x0 = (bx % tiles_x) * kTile;
    const int y0 = (bx / tiles_x) * kTile;
    constexpr int kRunsPerBand = kTile / kRun;
    constexpr int kRunsPerView = kTile * kRunsPerBand;

    float acc = 0.0f;
    for (int q0 = 0; q0 < nv; q0 += kChunk) {
        const int nq = min(kChunk, nv - q0);
        for (int q = threadIdx.x; q < nq; q += nthr) {
            const int v = __ldg(a.order + vb + q0 + q);
            s_vid[q] = v;
            s_views[q] = a.views[v];
        }
        for (int e = threadIdx.x; e < nq * kTile * kTile; e += nthr) s_part[e] = 0.0f;
        __syncthreads();
        if (q0 == 0) {
            // the staging above read plan constants only; the ratios and the
            // images below come from earlier kernels
            pdl_wait();
            pdl_trigger();
        }
        for (int run = threadIdx.x; run < nq * kRunsPerView; run += nthr) {
            const int ql = run / kRunsPerView;
            const int rem = run - ql * kRunsPerView;
            const int band = rem / kRunsPerBand;          // band offset inside the tile
            const int seg = rem - band * kRunsPerBand;
            const ViewParams vp = s_views[ql];
            const int v = s_vid[ql];
            const int k = (vp.col ? x0 : y0) + band;      // major index
            const int mstart = (vp.col ? y0 : x0) + seg * kRun;
            const int n_major = vp.col ? a.nx : a.ny;
            const int n_minor = vp.col ? a.ny : a.nx;
            const int mlen = min(kRun, n_minor - mstart);
            if (k >= n_major || mlen <= 0) continue;
            const int m0rel = mstart - (n_minor >> 1);
            const float kc = (float)k - 0.5f * (float)n_major;
            int jlo, jhi;
            candidate_bins(vp, kc, (float)m0rel, (float)(m0rel + mlen), a.nb, jlo, jhi);
            // local pixel index of minor offset c inside the run: row-driven runs
            // go along x, column-driven runs along y
            const int lbase = vp.col ? (seg * kRun) * kTile + band : band * kTile + seg * kRun;
            const int lstep = vp.col ? kTile : 1;
            float *pp = s_part + ql * kTile * kTile + lbase;
            const float2 *ucv = a.uc + v * a.nb;
            const float *rv = a.r + (vb + q0 + ql - r_view0) * a.nb;
            for (int j = jlo; j <= jhi; ++j) {
                const float2 u = __ldg(ucv + j);
                float fl, w0, w1;
                band_split(vp, band_point(vp, u.y, kc), band_point(vp, u.y, kc + 1.0f), fl, w0, w1);
                const int c = (int)fl + (int)u.x - m0rel;
                const float r = ld_data<COH>(rv + j);
                if ((unsigned)c < (unsigned)mlen) pp[c * lstep] += w0 * r;
                if (w1 > 0.0f && (unsigned)(c + 1) < (unsigned)mlen) pp[(c + 1) * lstep] += w1 * r;
            }
        }
        __syncthreads();
        if (threadIdx.x < kTile * kTile)
            for (int ql = 0; ql < nq; ++ql) acc += s_part[ql * kTile * kTile + threadIdx.x];
        __syncthreads();
    }
    pdl_wait();   // returns at once after the wait above; covers an empty subset
    if (threadIdx.x < kTile * kTile) {
        const int ix = x0 + (threadIdx.x % kTile);
        const int iy = y0 + (threadIdx.x / kTile);
        if (ix < a.nx && iy < a.ny) {
            const int n = iy * a.nx + ix;
            apply_epilogue<EPI, TQ, GENPOT, COH>(a, t, n, n, ix, iy, 0, acc);
        }
    }
}

}  // namespace

}  // namespace petvr
