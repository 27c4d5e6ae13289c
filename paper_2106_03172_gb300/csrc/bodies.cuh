// The single-slice projector bodies shared by the single-state kernels, the
// persistent batched phases and the dependency-driven batched epoch: the
// forward band-chunk body (forward_tile_body) and the tiled back projection
// with its update epilogue (back_tile_body).
//
// COH: the images and ratios the body reads may have been written earlier in
// the same kernel launch (the dependency-driven epoch), so they are read with
// plain loads instead of the read-only data path.
#pragma once

#include <type_traits>

#include "epilogue.cuh"

namespace petvr {

namespace {

constexpr int kTile = 16;           // single slice: a block owns a kTile x kTile pixel tile

constexpr int kSubsetBatch = 4;

// The bands [kb, ke) of one ray from this thread, every fourth one from kb on:
// sum of share times pixel, in units of the ray length per band.
//
// A band costs ~16 instructions: its lower end from the batch's base by one
// FMA, the floor by a directed-rounding add (kRound), the share by one
// saturating multiply, then two loads and three FMAs.  256^2, ncu: a full ratio
// pass 23.2 us and 14.4M warp instructions (33.2 us and 22.0M with floorf, the
// comparison of both band ends and contiguous bands per lane), a subset pass
// 6.9 us (7.9).
template <bool COH, int kBatch>
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
template <int CHUNKS, int MODE, bool LL, bool REF = false, bool COH = false>
__device__ __forceinline__ void forward_tile_body(const FwdArgs &a, const int bx) {
    const int tid = threadIdx.x;
    constexpr int RAYS = kBlock / CHUNKS;        // rays per block
    constexpr int WPG = CHUNKS / 4;              // warps per group of 8 rays
    const RayRange rr = ray_range(a);
    const int n_rays = (rr.v_end - rr.v_begin) * a.nb;
    const int warp = tid >> 5;
    const int lane = tid & 31;
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
    if (ray < n_rays) {
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
    const int ray_f = bx * RAYS + tid;
    const bool fin = tid < RAYS && ray_f < n_rays;
    const long long gi = rr.off + ray_f;
    float g_f = 0.0f, w_f = a.w_scalar;
    if (fin) {
        if (MODE == FWD_RATIO || LL) g_f = __ldg(a.g + gi);
        if (a.w) w_f = __ldg(a.w + gi);
    }
    float acc = 0.0f;
    if (kb < ke)
        acc = REF ? walk_bands_ref<COH>(a, vp, uf, ui, hm, n_minor, kb, ke)
                  : walk_bands<COH, CHUNKS >= 32 ? kSubsetBatch : 4>(a, vp, uf, ui, hm, n_minor, kb, ke);
    // the 4 chunks of each ray in this warp, then the warps of its group
    acc += __shfl_xor_sync(0xffffffffu, acc, 8);
    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
    __shared__ float red[kBlock / 32][8];
    if (lane < 8) red[warp][lane] = acc;
    __syncthreads();

    double ll = 0.0;
    if (tid < RAYS) {
        const int g = tid >> 3;
        float sum = 0.0f;
#pragma unroll
        for (int w = 0; w < WPG; ++w) sum += red[g * WPG + w][tid & 7];
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
    // every ray of the block is finished in its first warp (RAYS <= 32): the FP64
    // sums, slow on GB300 (2 lanes per SM and clock), stay there
    if (LL && warp == 0) {
#pragma unroll
        for (int o = RAYS / 2; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);
        if (lane == 0) a.ll_partials[bx] = ll;
    }
}

// One item of a batched forward, with the member's band-chunk count and rounding.
template <int MODE, bool LL, bool COH = false>
__device__ __forceinline__ void forward_item(const FwdArgs &a, int shape, int bx) {
    if constexpr (MODE == FWD_RATIO && !LL) {
        if (a.ref) {
            if (shape == 8)
                forward_tile_body<8, MODE, LL, kRefRounding, COH>(a, bx);
            else if (shape == 16)
                forward_tile_body<16, MODE, LL, kRefRounding, COH>(a, bx);
            else
                forward_tile_body<32, MODE, LL, kRefRounding, COH>(a, bx);
            return;
        }
    }
    if (shape == 8)
        forward_tile_body<8, MODE, LL, false, COH>(a, bx);
    else if (shape == 16)
        forward_tile_body<16, MODE, LL, false, COH>(a, bx);
    else
        forward_tile_body<32, MODE, LL, false, COH>(a, bx);
}

// ---- back projection ------------------------------------------------------------

// Single-slice path: a block owns a kTile x kTile pixel tile, a thread PX pixels
// (a column of PX neighbours along y; the block has kTile^2 / PX threads).  For
// each view of the subset two tables are staged in shared memory: the bins
// whose rays can meet the tile (offset, and ratio times ray length), and per
// band of the tile the displacement of a ray over the bands from the image
// centre.  A pixel then takes its candidate bins and adds share times ratio in
// registers, views and bins in increasing order, so the result is
// deterministic (and the same for any PX) and needs no atomics.
constexpr int kStageViews = 32;        // views per pass
constexpr int kStageBins = 1024;       // staged bins per pass
constexpr int kViewGroups = 4;         // groups of threads on launches over all views
constexpr int kUnrolledCand = 3;       // candidate counts with an unrolled view loop

// Per-view constants of a tile.  A ray's offset from pixel m at its band's
// lower end is x = u_j + P - m, with P = kc du its displacement over the kc
// bands from the image centre; the ray meets the pixel for -|du| < x < 1, so
// the candidates are the bins of that range, u_j = (j - (nb - 1) / 2) K + off.
// They are found from approximate positions, with a margin far above their
// rounding; a candidate that misses the pixel gets share 0.
struct alignas(16) TileView {
    float inv_adu, invK;
    unsigned base;    // staged entry of bin 0, less kRoundBits (see kRound)
    int flags;        // bit 0: column-driven; above it: the number of candidate bins
    float du, du_lo;
    float k0;         // centred major coordinate of the tile's first band's lower end
    float cst;        // first candidate: floor((m - P) invK + cst)
    float L;          // ray length per band
    int j0, v;        // first staged bin; view
    int pad;
};

struct TileShared {
    float4 bins[kStageBins];                // [view][bw]: offset (integer, fraction), ratio times L
    float4 bands[kStageViews * kTile];      // [view][band]: P (integer, fraction), cst - P invK
    TileView views[kStageViews];
};

// The candidates of a thread's PX pixels are taken together: the next pixel
// along y shifts x by `step`.
template <int PX>
__device__ __forceinline__ void tile_view(const BackArgs &a, const ViewParams &vp, int v, int x0, int y0, int q,
                                          TileView &tv) {
    const int n_minor = vp.col ? a.ny : a.nx;
    const int n_major = vp.col ? a.nx : a.ny;
    const float adu = fabsf(vp.du);
    const float step = (float)(PX - 1) * (vp.col ? -1.0f : vp.du);
    const float eps = 1e-3f + 4e-7f * (float)(a.nb + a.nx + a.ny);
    const float first = vp.invK > 0.0f ? -adu : 1.0f;
    const float off = (n_minor & 1) ? 0.5f : 0.0f;
    tv.inv_adu = vp.inv_adu;
    tv.invK = vp.invK;
    tv.du = vp.du;
    tv.du_lo = vp.du_lo;
    tv.k0 = (float)(vp.col ? x0 : y0) - 0.5f * (float)n_major + (vp.du < 0.0f ? 1.0f : 0.0f);
    tv.cst = fmaf(first - off, vp.invK, 0.5f * (float)(a.nb - 1)) + fminf(0.0f, -step * vp.invK) + (1.0f - eps);
    const int nc = (int)floorf(fmaf(1.0f + adu + fabsf(step), fabsf(vp.invK), 2.0f * eps)) + 1;
    tv.flags = (vp.col ? 1 : 0) | (nc << 1);
    tv.L = vp.L;
    tv.v = v;
    // smallest first candidate over the tile's corners, less one for rounding
    const float m0 = (float)((vp.col ? y0 : x0) - (n_minor >> 1));
    const float ma = fminf(m0 * vp.invK, (m0 + (float)(kTile - 1)) * vp.invK);
    const float slope = -vp.du * vp.invK;
    const float pa = slope * tv.k0, pb = slope * (tv.k0 + (float)(kTile - 1));
    tv.j0 = (int)floorf(ma + fminf(pa, pb) + tv.cst) - 1;
    tv.base = (unsigned)(q * a.bw - tv.j0) - kRoundBits;
}

// A ray's offset as staged.  On an axis-aligned view only the pixel a ray lies
// in matters, so its fraction is moved well inside that pixel.
__device__ __forceinline__ float2 staged_offset(float2 u, float du) {
    if (du == 0.0f) u.y = u.y < 0.0f ? -0.5f : 0.25f;
    return u;
}

// Share of a ray's band in the pixel it meets at offset x: the part of the
// band with -|du| < x < 1, as band_share() and its complement.
__device__ __forceinline__ float pixel_share(float x, float inv_adu) {
    return __saturatef(fmaf(-x, inv_adu, inv_adu)) - __saturatef(-x * inv_adu);
}

// Staged bins of a pass: warp w takes the 32-bin pieces w, w + NT / 32, ... of
// the views, two pieces' loads in flight at a time.  `load(view, bin, entry,
// live)` starts one entry's load and returns what stores it.
template <int NT, class Load>
__device__ __forceinline__ void stage_bins(int nq, int bw, Load &&load) {
    const int per_view = (bw + 31) >> 5;
    const int n = nq * per_view;
    const int lane = threadIdx.x & 31;
    for (int c = threadIdx.x >> 5; c < n; c += 2 * (NT / 32)) {
        const int d = c + NT / 32;
        const int qc = per_view == 1 ? c : c / per_view, qd = per_view == 1 ? d : d / per_view;
        const int ic = (c - qc * per_view) * 32 + lane, id = (d - qd * per_view) * 32 + lane;
        const bool more = d < n;
        auto first = load(qc, ic, qc * bw + ic, ic < bw);
        auto second = load(more ? qd : qc, id, qd * bw + id, more && id < bw);
        first();
        second();
    }
}

// Bound by instruction issue on the all-subset launches (two pixels a thread
// share the candidates, three for a pair where bins are as wide as pixels,
// against two each) and by the launch's dependent round trips on subset
// launches (one pixel a thread, for twice the warps).  x is formed from integer
// and fractional parts separately (exact integers, fractions below 2), so its
// error does not grow with the image.  Against runs of 8 pixels a thread that
// walked their rays with sums in shared memory (back_run_body): 256^2 anchor of
// 21 subsets 40.1 -> 31.0 us (ncu), an update (both projections, in a graph)
// 8.8 -> 6.7 us, 512^2 with 60 views a subset 90 -> 61 us.
//
// GROUPS > 1: group g of the block's threads takes the views g, g + GROUPS, ...
// of a pass, and the groups' sums are added in order (launches over all views,
// whose few tiles would otherwise walk every view one after another).
template <int EPI, typename TQ, bool GENPOT, int PX, bool COH = false, int GROUPS = 1>
__device__ __forceinline__ void back_tile_body(const BackArgs &a, const int t, const int bx) {
    constexpr int NT = kTile * kTile / PX;
    extern __shared__ unsigned char smem_raw[];
    const int tid = GROUPS > 1 ? threadIdx.x % NT : threadIdx.x;
    const int group = GROUPS > 1 ? threadIdx.x / NT : 0;
    TileShared &sh = *reinterpret_cast<TileShared *>(smem_raw);
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    const int r_view0 = a.t_dev ? vb : a.r_view0;
    const int tiles_x = (a.nx + kTile - 1) / kTile;
    const int x0 = (bx % tiles_x) * kTile;
    const int y0 = (bx / tiles_x) * kTile;
    const int tx = tid % kTile, ty = tid / kTile * PX;
    const bool staged = a.bw <= kStageBins;   // else (bins far finer than pixels) bins are read in place
    const int per_pass = staged ? min(kStageViews, kStageBins / a.bw) : kStageViews;
    const float mx = (float)(x0 + tx - (a.nx >> 1)), my = (float)(y0 + ty - (a.ny >> 1));

    float acc[PX] = {};
    for (int q0 = 0; q0 < nv; q0 += per_pass) {
        const int nq = min(per_pass, nv - q0);
        if (q0 > 0) __syncthreads();             // the pass before is done with shared memory
        if (threadIdx.x < nq) {
            const int v = __ldg(a.order + vb + q0 + threadIdx.x);
            tile_view<PX>(a, a.views[v], v, x0, y0, threadIdx.x, sh.views[threadIdx.x]);
        }
        __syncthreads();
        // plan constants before the wait for the kernel ahead, ratios after it
        for (int i = threadIdx.x; i < nq * kTile; i += NT * GROUPS) {
            const TileView &tv = sh.views[i / kTile];
            const float kc = tv.k0 + (float)(i % kTile);
            const float tp = fmaf(kc, tv.du, kRound);
            const float pi = tp - kRound;
            const float pf = fmaf(kc, tv.du_lo, fmaf(kc, tv.du, -pi));
            sh.bands[i] = make_float4(pi, pf, fmaf(-(pi + pf), tv.invK, tv.cst), 0.0f);
        }
        if (staged)
            stage_bins<NT * GROUPS>(nq, a.bw, [&](int q, int i, int e, bool live) {
                const int j = sh.views[q].j0 + i;
                float2 u = make_float2(0.0f, 0.0f);
                if (live && (unsigned)j < (unsigned)a.nb)
                    u = __ldg(a.uc + sh.views[q].v * a.nb + j);
                return [=, &sh](void) {
                    if (live) *reinterpret_cast<float2 *>(sh.bins + e) = staged_offset(u, sh.views[q].du);
                };
            });
        if (q0 == 0) {
            pdl_wait();
            pdl_trigger();
        }
        if (staged)
            stage_bins<NT * GROUPS>(nq, a.bw, [&](int q, int i, int e, bool live) {
                const int j = sh.views[q].j0 + i;
                float r = 0.0f;
                if (live && (unsigned)j < (unsigned)a.nb)
                    r = ld_data<COH>(a.r + (vb + q0 + q - r_view0) * a.nb + j);
                return [=, &sh](void) {
                    if (live) sh.bins[e].z = r * sh.views[q].L;
                };
            });
        __syncthreads();
        // NC > 0: that many candidates of every view (the plan's most; the ones
        // a view does not have miss the pixel), without branches, so that the
        // views of an unrolled group overlap
        auto gather = [&](auto nc) {
            constexpr int NC = decltype(nc)::value;
#pragma unroll (NC == 2 ? 2 / PX : 1)
            for (int q = group; q < nq; q += GROUPS) {
                const float4 vc = *reinterpret_cast<const float4 *>(&sh.views[q]);     // inv_adu, invK, base, flags
                const int flags = __float_as_int(vc.w);
                const bool col = flags & 1;
                const float m = col ? my : mx;
                const float4 *bands = sh.bands + q * kTile + (col ? tx : ty);
                float b[PX], pf[PX];
                float e = 0.0f;
#pragma unroll
                for (int p = 0; p < PX; ++p) {
                    const float4 bd = bands[col ? 0 : p];
                    if (p == 0) e = fmaf(m, vc.y, bd.z);
                    b[p] = m + (col ? (float)p : 0.0f) - bd.x;
                    pf[p] = bd.y;
                }
                auto add = [&](float ui, float uf, float r) {
#pragma unroll
                    for (int p = 0; p < PX; ++p) {
                        const float w = pixel_share((ui - b[p]) + (uf + pf[p]), vc.x);
                        if (w > 0.0f) acc[p] = fmaf(w, r, acc[p]);
                    }
                };
                if (NC > 0 || staged) {
                    const float4 *ent = sh.bins + (__float_as_uint(__fadd_rd(e, kRound)) + __float_as_uint(vc.z));
                    float4 en[NC > 0 ? NC : 1];
#pragma unroll
                    for (int c = 0; c < NC; ++c) en[c] = ent[c];
#pragma unroll
                    for (int c = 0; c < NC; ++c) add(en[c].x, en[c].y, en[c].z);
                    if (NC == 0)
#pragma unroll 1
                        for (int c = 0; c < flags >> 1; ++c) add(ent[c].x, ent[c].y, ent[c].z);
                } else {
                    const int j0 = (int)floorf(e);
#pragma unroll 1
                    for (int j = max(j0, 0); j < min(j0 + (flags >> 1), a.nb); ++j) {
                        const float2 u = staged_offset(__ldg(a.uc + sh.views[q].v * a.nb + j), sh.views[q].du);
                        add(u.x, u.y, ld_data<COH>(a.r + (vb + q0 + q - r_view0) * a.nb + j) * sh.views[q].L);
                    }
                }
            }
        };
        const int most = PX == 1 ? a.cand1 : a.cand2;
        if (!staged || most > kUnrolledCand)
            gather(std::integral_constant<int, 0>());
        else if (most == 2)
            gather(std::integral_constant<int, 2>());
        else
            gather(std::integral_constant<int, 3>());
    }
    pdl_wait();   // returns at once after the wait above; covers an empty subset
    if constexpr (GROUPS > 1) {
        float *sums = reinterpret_cast<float *>(smem_raw);      // [GROUPS][PX][NT]
        __syncthreads();
        if (group > 0)
#pragma unroll
            for (int p = 0; p < PX; ++p) sums[(group * PX + p) * NT + tid] = acc[p];
        __syncthreads();
        if (group > 0) return;
#pragma unroll
        for (int g = 1; g < GROUPS; ++g)
#pragma unroll
            for (int p = 0; p < PX; ++p) acc[p] += sums[(g * PX + p) * NT + tid];
    }
    const int ix = x0 + tx;
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        const int iy = y0 + ty + p;
        if (ix < a.nx && iy < a.ny) {
            const int n = iy * a.nx + ix;
            apply_epilogue<EPI, TQ, GENPOT, COH>(a, t, n, n, ix, iy, 0, acc[p]);
        }
    }
}

// The reference rounding (kRefRounding): for each view, the tile's bands are cut
// into runs of kRun pixels along the view's minor axis; one thread walks the
// rays that can cross a run in order and adds each ray's two band pieces into
// per-view partial sums in shared memory (every (view, pixel) slot has exactly
// one writer, so no atomics).  Then each thread sums its pixels' partials over
// the views in a fixed order and applies the update.  A gather per pixel in
// this rounding takes 1.3 times the instructions (it evaluates both ends of
// every candidate's band twice).
constexpr int kRun = 8;
constexpr int kRunBlock = 256;         // threads of a looping block (at least the tile's pixels)
constexpr int kRunThreadsMax = 512;
constexpr int kRunViews = 16;          // views per shared-memory pass

struct RunShared {
    float part[kRunViews][kTile * kTile];
    ViewParams views[kRunViews];
    int vid[kRunViews];
};

template <int EPI, typename TQ, bool GENPOT, bool COH = false>
__device__ __forceinline__ void back_run_body(const BackArgs &a, const int t, const int bx) {
    extern __shared__ unsigned char smem_raw[];
    RunShared &sh = *reinterpret_cast<RunShared *>(smem_raw);
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    const int r_view0 = a.t_dev ? vb : a.r_view0;
    const int nthr = blockDim.x;                  // >= kTile * kTile

    const int tiles_x = (a.nx + kTile - 1) / kTile;
    const int x0 = (bx % tiles_x) * kTile;
    const int y0 = (bx / tiles_x) * kTile;
    constexpr int kRunsPerBand = kTile / kRun;
    constexpr int kRunsPerView = kTile * kRunsPerBand;

    float acc = 0.0f;
    for (int q0 = 0; q0 < nv; q0 += kRunViews) {
        const int nq = min(kRunViews, nv - q0);
        for (int q = threadIdx.x; q < nq; q += nthr) {
            const int v = __ldg(a.order + vb + q0 + q);
            sh.vid[q] = v;
            sh.views[q] = a.views[v];
        }
        for (int e = threadIdx.x; e < nq * kTile * kTile; e += nthr) sh.part[0][e] = 0.0f;
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
            const ViewParams vp = sh.views[ql];
            const int v = sh.vid[ql];
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
            float *pp = sh.part[ql] + lbase;
            const float2 *ucv = a.uc + v * a.nb;
            const float *rv = a.r + (vb + q0 + ql - r_view0) * a.nb;
            for (int j = jlo; j <= jhi; ++j) {
                const float2 u = __ldg(ucv + j);
                float w0, w1;
                const float tl = band_split_ref(vp, band_point(vp, u.y, kc), band_point(vp, u.y, kc + 1.0f), w0, w1);
                const int c = (int)(__float_as_uint(tl) - kRoundBits) + (int)u.x - m0rel;
                const float r = ld_data<COH>(rv + j);
                if ((unsigned)c < (unsigned)mlen) pp[c * lstep] += w0 * r;
                if (w1 > 0.0f && (unsigned)(c + 1) < (unsigned)mlen) pp[(c + 1) * lstep] += w1 * r;
            }
        }
        __syncthreads();
        if (threadIdx.x < kTile * kTile)
            for (int ql = 0; ql < nq; ++ql) acc += sh.part[ql][threadIdx.x];
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

inline size_t run_smem_bytes() { return sizeof(RunShared); }
inline size_t tile_smem_bytes() { return sizeof(TileShared); }

// Member update of one tile: the member's algorithm selects the epilogue (the
// single-state launch's template argument).
template <bool GENPOT, int PX, bool COH = false>
__device__ __forceinline__ void member_update_tile(int algo, const BackArgs &b, int t, int tile) {
    switch (algo) {
        case PET_ALGO_OSEM: back_tile_body<EPI_OSEM, float, GENPOT, PX, COH>(b, t, tile); break;
        case PET_ALGO_SVREM: back_tile_body<EPI_SVREM, float, GENPOT, PX, COH>(b, t, tile); break;
        case PET_ALGO_SAGA: back_tile_body<EPI_SAGA, float, GENPOT, PX, COH>(b, t, tile); break;
        case PET_ALGO_SGA: back_tile_body<EPI_SGA, float, GENPOT, PX, COH>(b, t, tile); break;
        case PET_ALGO_SEM: back_tile_body<EPI_SEM, float, GENPOT, PX, COH>(b, t, tile); break;
        case PET_ALGO_SAGAEM: back_tile_body<EPI_SAGAEM, float, GENPOT, PX, COH>(b, t, tile); break;
        default: back_tile_body<EPI_SVRG, float, GENPOT, PX, COH>(b, t, tile); break;
    }
}

}  // namespace

}  // namespace petvr
