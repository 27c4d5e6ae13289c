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

constexpr int kTile = 16;           // single slice: a block owns a kTile x kTile tile, a thread one pixel
static_assert(kTile * kTile == kBlock, "one pixel of the tile per thread");

// The consecutive bands [kb, ke) of one ray: sum of weight times pixel.
//
// A band costs ~22 instructions: its far end by two FMAs, the floor by a
// directed-rounding add (kRound), the weights (band_weights), then two loads
// and two FMAs.
template <bool COH>
__device__ __forceinline__ float walk_bands(const FwdArgs &a, const ViewParams &vp, float uf, int ui, float hm,
                                            int n_minor, int kb, int ke) {
    const int s_major = vp.col ? 1 : a.nx;
    const int s_minor = vp.col ? a.nx : 1;
    const float *img1 = a.img + s_minor;
    float acc = 0.0f;
    float kc = (float)kb - hm;
    float va = band_point(vp, uf, kc);
    // kBatch bands at a time: all their offsets and weights first, then the
    // loads, then the FMAs in band order, so that the loads of a batch are in
    // flight together.
    constexpr int kBatch = 4;
    for (int k = kb; k < ke; k += kBatch) {
        int m0[kBatch];
        float c0[kBatch], c1[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            kc += 1.0f;
            const float vb = band_point(vp, uf, kc);
            const float t = band_weights(vp.L, vp.Lm, fminf(va, vb), fmaxf(va, vb), c0[b], c1[b]);
            m0[b] = (int)(__float_as_uint(t) - kRoundBits) + ui;
            va = vb;
        }
        // a piece outside the image (or of a band past ke) is not loaded and
        // adds 0; the upper pixel is loaded only where the line reaches it.
        // The lower end is monotone in the band, so when both pixels of the
        // first and last band are inside the image every band's are: no checks.
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
// and splits each ray's bands into CHUNKS contiguous chunks (RAYS * CHUNKS =
// kBlock).  Inside a warp, lane = 8 * chunk + ray: the 32 lanes are 8
// adjacent rays times 4 chunks, so one warp load touches 4 image rows with
// 8 neighbouring pixels each.  Chunk sums are reduced by xor-shuffles
// (within the warp) and then over warps through shared memory, always in the
// same order, so the result is deterministic.
template <int CHUNKS, int MODE, bool LL, bool COH = false>
__device__ __forceinline__ void forward_tile_body(const FwdArgs &a, const int bx) {
    const int tid = threadIdx.x;
    constexpr int RAYS = kBlock / CHUNKS;        // rays per block
    constexpr int WPG = CHUNKS / 4;              // warps per group of 8 rays
    const RayRange rr = ray_range(a);
    const int n_rays = (rr.v_end - rr.v_begin) * a.nb;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int r8 = lane & 7;
    const int chunk = 4 * (warp % WPG) + (lane >> 3);
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
        // chunks are aligned to the same bands for every ray of the view, so
        // neighbouring lanes read the same image rows
        const int per = (n_major + CHUNKS - 1) / CHUNKS;
        kb = max(k_lo, chunk * per);
        ke = min(k_hi, (chunk + 1) * per);
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
    float acc = kb < ke ? walk_bands<COH>(a, vp, uf, ui, hm, n_minor, kb, ke) : 0.0f;
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

// One item of a batched forward, with the member's band-chunk count.
template <int MODE, bool LL, bool COH = false>
__device__ __forceinline__ void forward_item(const FwdArgs &a, int shape, int bx) {
    if (shape == 8)
        forward_tile_body<8, MODE, LL, COH>(a, bx);
    else if (shape == 16)
        forward_tile_body<16, MODE, LL, COH>(a, bx);
    else
        forward_tile_body<32, MODE, LL, COH>(a, bx);
}

// ---- back projection ------------------------------------------------------------

// Single-slice path: a block owns a kTile x kTile pixel tile, a thread one pixel.
// For each view of the subset two tables are staged in shared memory: the bins
// whose rays can meet the tile (offset and ratio), and per band of the tile the
// position of its lower end.  A pixel takes its candidate bins and adds weight
// times ratio in registers, a sum per view over its bins in increasing order,
// then over the views, so the result is deterministic and needs no atomics.
constexpr int kStageViews = 32;        // views per pass
constexpr int kStageBins = 1024;       // staged bins per pass
constexpr int kUnrolledCand = 3;       // largest candidate count with a loop of its own

// Per-view constants of a tile.  A ray's offset from pixel m at its band's
// lower end is x = u_j + P - m, with P = kc du its displacement over the kc
// bands from the image centre; the ray meets the pixel for -|du| < x < 1, so
// the candidates are the bins of that range, u_j = (j - (nb - 1) / 2) K + off.
// They are found from approximate positions, with a margin far above their
// rounding; a candidate that misses the pixel adds nothing.
struct alignas(16) TileView {
    float du, du_lo;
    float step;       // from a band's lower end to its upper end: +1 or -1
    float k0;         // centred major coordinate of the lower end of the tile's first band
    float L, Lm;
    unsigned base;    // staged entry of bin 0, less kRoundBits (see kRound)
    int flags;        // bit 0: column-driven; above it: the number of candidate bins
    float invK;
    float cst;        // first candidate: floor((m - P) invK + cst)
    int j0, v;        // first staged bin; view
};

struct TileShared {
    float4 bins[kStageBins];                // [view][bw]: offset (integer, fraction), ratio
    float4 bands[kStageViews * kTile];      // [view][band]: kc of the lower end, cst - P invK, invK, kc of the upper end
    TileView views[kStageViews];
};

__device__ __forceinline__ void tile_view(const BackArgs &a, const ViewParams &vp, int v, int x0, int y0, int q,
                                          TileView &tv) {
    const int n_minor = vp.col ? a.ny : a.nx;
    const int n_major = vp.col ? a.nx : a.ny;
    const float adu = fabsf(vp.du);
    const float eps = 1e-3f + 4e-7f * (float)(a.nb + a.nx + a.ny);
    const float first = vp.invK > 0.0f ? -adu : 1.0f;
    const float off = (n_minor & 1) ? 0.5f : 0.0f;
    tv.du = vp.du;
    tv.du_lo = vp.du_lo;
    tv.step = vp.du < 0.0f ? -1.0f : 1.0f;
    tv.L = vp.L;
    tv.Lm = vp.Lm;
    tv.invK = vp.invK;
    tv.k0 = (float)(vp.col ? x0 : y0) - 0.5f * (float)n_major + (vp.du < 0.0f ? 1.0f : 0.0f);
    tv.cst = fmaf(first - off, vp.invK, 0.5f * (float)(a.nb - 1)) + (1.0f - eps);
    const int nc = (int)floorf(fmaf(1.0f + adu, fabsf(vp.invK), 2.0f * eps)) + 1;
    tv.flags = (vp.col ? 1 : 0) | (nc << 1);
    tv.v = v;
    // smallest first candidate over the tile's corners, less one for rounding
    const float m0 = (float)((vp.col ? y0 : x0) - (n_minor >> 1));
    const float ma = fminf(m0 * vp.invK, (m0 + (float)(kTile - 1)) * vp.invK);
    const float slope = -vp.du * vp.invK;
    const float pa = slope * tv.k0, pb = slope * (tv.k0 + (float)(kTile - 1));
    tv.j0 = (int)floorf(ma + fminf(pa, pb) + tv.cst) - 1;
    tv.base = (unsigned)(q * a.bw - tv.j0) - kRoundBits;
}

// Staged bins of a pass: warp w of the NT threads takes the 32-bin pieces w, w +
// NT / 32, ... of the views, two pieces' loads in flight at a time.  `load(view,
// bin, entry, live)` starts one entry's load and returns what stores it.
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

// Bound by the launch's dependent round trips on subset launches: the bins
// arrive in one, and the views' chains overlap.  The weights are band_weights()
// of the positions the forward computes, bit for bit (the ends come in order,
// so the floor, the share and the test of the upper end are all there is to a
// candidate).  Against runs (back_run_body) as the updates had them before: a
// 256^2 SAGA epoch of 21 updates 190 -> 162 us, a 201x147 SVRG run 474 -> 381, a 512^2
// reconstruction 3924 -> 3160; update_by_runs has the points where runs win.
template <int EPI, typename TQ, bool GENPOT, bool COH = false>
__device__ __forceinline__ void back_tile_body(const BackArgs &a, const int t, const int bx) {
    constexpr int NT = kTile * kTile;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileShared &sh = *reinterpret_cast<TileShared *>(smem_raw);
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    const int r_view0 = a.t_dev ? vb : a.r_view0;
    const int tiles_x = (a.nx + kTile - 1) / kTile;
    const int x0 = (bx % tiles_x) * kTile;
    const int y0 = (bx / tiles_x) * kTile;
    const int tx = threadIdx.x % kTile, ty = threadIdx.x / kTile;
    const bool staged = a.bw <= kStageBins;      // else (bins far finer than pixels) bins are read in place
    const int per_pass = staged ? min(kStageViews, kStageBins / a.bw) : kStageViews;
    const float mx = (float)(x0 + tx - (a.nx >> 1)), my = (float)(y0 + ty - (a.ny >> 1));

    float acc = 0.0f;
    for (int q0 = 0; q0 < nv; q0 += per_pass) {
        const int nq = min(per_pass, nv - q0);
        if (q0 > 0) __syncthreads();             // the pass before is done with shared memory
        if (threadIdx.x < nq) {
            const int v = __ldg(a.order + vb + q0 + threadIdx.x);
            tile_view(a, a.views[v], v, x0, y0, threadIdx.x, sh.views[threadIdx.x]);
        }
        __syncthreads();
        // plan constants before the wait for the kernel ahead, ratios after it
        for (int i = threadIdx.x; i < nq * kTile; i += NT) {
            const TileView &tv = sh.views[i / kTile];
            const float kc = tv.k0 + (float)(i % kTile);
            sh.bands[i] = make_float4(kc, fmaf(-(kc * tv.du), tv.invK, tv.cst), tv.invK, kc + tv.step);
        }
        if (staged)
            stage_bins<NT>(nq, a.bw, [&](int q, int i, int e, bool live) {
                const int j = sh.views[q].j0 + i;
                float2 u = make_float2(0.0f, 0.0f);
                if (live && (unsigned)j < (unsigned)a.nb) u = __ldg(a.uc + sh.views[q].v * a.nb + j);
                return [=, &sh](void) {
                    if (live) *reinterpret_cast<float2 *>(sh.bins + e) = u;
                };
            });
        if (q0 == 0) {
            pdl_wait();
            pdl_trigger();
        }
        if (staged)
            stage_bins<NT>(nq, a.bw, [&](int q, int i, int e, bool live) {
                const int j = sh.views[q].j0 + i;
                float r = 0.0f;
                if (live && (unsigned)j < (unsigned)a.nb)
                    r = ld_data<COH>(a.r + (vb + q0 + q - r_view0) * a.nb + j);
                return [=, &sh](void) {
                    if (live) sh.bins[e].z = r;
                };
            });
        __syncthreads();
        // NC > 0: that many candidates of every view (the plan's most; the ones
        // a view does not have miss the pixel), without branches, so that the
        // views of an unrolled group overlap
        auto gather = [&](auto nc) {
            constexpr int NC = decltype(nc)::value;
#pragma unroll (NC == 2 ? 2 : 1)
            for (int q = 0; q < nq; ++q) {
                const float2 vc = *reinterpret_cast<const float2 *>(&sh.views[q].du);       // du, du_lo
                const float4 vd = *reinterpret_cast<const float4 *>(&sh.views[q].L);        // L, Lm, base, flags
                const int flags = __float_as_int(vd.w);
                const bool col = flags & 1;
                const float m = col ? my : mx;
                const float4 bd = sh.bands[q * kTile + (col ? tx : ty)];
                const float e = fmaf(m, bd.z, bd.y);
                float part = 0.0f;
                auto add = [&](float ui, float uf, float r) {
                    const float lo = fmaf(bd.x, vc.x, fmaf(bd.x, vc.y, uf));        // band_point()
                    const float fl1 = __fadd_rd(lo, kRound) - (kRound - 1.0f);
                    float w0 = fminf((fl1 - lo) * vd.y, vd.x);                      // band_weights()
                    if (fmaf(bd.w, vc.x, fmaf(bd.w, vc.y, uf)) <= fl1) w0 = vd.x;
                    const float w1 = vd.x - w0;
                    const float c = fl1 + (ui - m);        // 1: the ray's lower pixel is this one, 0: its upper one
                    if (c == 1.0f) part = fmaf(w0, r, part);
                    if (c == 0.0f && w1 > 0.0f) part = fmaf(w1, r, part);
                };
                if (NC > 0) {
                    const float4 *ent = sh.bins + (__float_as_uint(__fadd_rd(e, kRound)) + __float_as_uint(vd.z));
                    float4 en[NC > 0 ? NC : 1];
#pragma unroll
                    for (int k = 0; k < NC; ++k) en[k] = ent[k];
#pragma unroll
                    for (int k = 0; k < NC; ++k) add(en[k].x, en[k].y, en[k].z);
                } else {
                    const int j0 = (int)floorf(e);
                    const float4 *ent = sh.bins + (q * a.bw - sh.views[q].j0);
#pragma unroll 1
                    for (int j = max(j0, 0); j < min(j0 + (flags >> 1), a.nb); ++j) {
                        if (staged) {
                            add(ent[j].x, ent[j].y, ent[j].z);
                        } else {
                            const float2 u = __ldg(a.uc + sh.views[q].v * a.nb + j);
                            add(u.x, u.y, ld_data<COH>(a.r + (vb + q0 + q - r_view0) * a.nb + j));
                        }
                    }
                }
                acc += part;
            }
        };
        if (staged && a.cand == 2)
            gather(std::integral_constant<int, 2>());
        else if (staged && a.cand == 3)
            gather(std::integral_constant<int, 3>());
        else
            gather(std::integral_constant<int, 0>());
    }
    pdl_wait();   // returns at once after the wait above; covers an empty subset
    const int ix = x0 + tx, iy = y0 + ty;
    if (ix < a.nx && iy < a.ny) {
        const int n = iy * a.nx + ix;
        apply_epilogue<EPI, TQ, GENPOT, COH>(a, t, n, n, ix, iy, 0, acc);
    }
}

// All-subset launches (anchors, table fills), plain back projections, and the updates
// and batch members that are faster this way (update_by_runs, batch_runs): for each
// view, the tile's bands are cut into runs of kRun pixels along the view's minor
// axis; one thread walks the rays that can cross a run in order and adds each
// ray's two band pieces into per-view partial sums in shared memory (every
// (view, pixel) slot has exactly one writer, so no atomics).  Then each thread
// sums its pixel's partials over the views in order.  The same weights and
// order of sums as back_tile_body, bit for bit, in fewer instructions (a band
// is evaluated once for the run, not for every pixel it can touch) but a longer
// chain: 256^2, 21 subsets 40 us and 29.7M warp instructions, staged bins 43 us
// and 35.3M (ncu).
constexpr int kRun = 8;

// Views per shared-memory pass of an NT-thread block (0: as many threads as the
// launch has): a run per thread at 512 threads and more, two per thread at 256.
template <int NT>
constexpr int kRunViews = NT > 512 ? NT / 32 : 16;

template <int VIEWS>
struct RunShared {
    float part[VIEWS][kTile * kTile];
    ViewParams views[VIEWS];
    int vid[VIEWS];
};

template <int EPI, typename TQ, bool GENPOT, int NT, bool COH = false>
__device__ __forceinline__ void back_run_body(const BackArgs &a, const int t, const int bx) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kViews = kRunViews<NT>;
    RunShared<kViews> &sh = *reinterpret_cast<RunShared<kViews> *>(smem_raw);
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    const int r_view0 = a.t_dev ? vb : a.r_view0;
    const int nthr = NT ? NT : blockDim.x;        // >= kTile * kTile

    const int tiles_x = (a.nx + kTile - 1) / kTile;
    const int x0 = (bx % tiles_x) * kTile;
    const int y0 = (bx / tiles_x) * kTile;
    constexpr int kRunsPerBand = kTile / kRun;
    constexpr int kRunsPerView = kTile * kRunsPerBand;

    float acc = 0.0f;
    for (int q0 = 0; q0 < nv; q0 += kViews) {
        const int nq = min(kViews, nv - q0);
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
                const float e0 = band_point(vp, u.y, kc), e1 = band_point(vp, u.y, kc + 1.0f);
                float w0, w1;
                const float tl = band_weights(vp.L, vp.Lm, fminf(e0, e1), fmaxf(e0, e1), w0, w1);
                const int c = (int)(__float_as_uint(tl) - kRoundBits) + (int)u.x - m0rel;
                const float r = ld_data<COH>(rv + j);
                if ((unsigned)c < (unsigned)mlen) pp[c * lstep] += w0 * r;
                if (w1 > 0.0f && (unsigned)(c + 1) < (unsigned)mlen) pp[(c + 1) * lstep] += w1 * r;
            }
        }
        __syncthreads();
        if (NT == kTile * kTile || threadIdx.x < kTile * kTile)
            for (int ql = 0; ql < nq; ++ql) acc += sh.part[ql][threadIdx.x];
        __syncthreads();
    }
    pdl_wait();   // returns at once after the wait above; covers an empty subset
    const int ix = x0 + (threadIdx.x % kTile);
    const int iy = y0 + (threadIdx.x / kTile);
    if ((NT == kTile * kTile || threadIdx.x < kTile * kTile) && ix < a.nx && iy < a.ny) {
        const int n = iy * a.nx + ix;
        apply_epilogue<EPI, TQ, GENPOT, COH>(a, t, n, n, ix, iy, 0, acc);
    }
}

template <int NT>
constexpr size_t run_smem_bytes() {
    return sizeof(RunShared<kRunViews<NT>>);
}
inline size_t tile_smem_bytes() { return sizeof(TileShared); }

// One tile of a batch member (256 threads), by runs (RUNS: a kernel that has them)
// or staged bins, the same bits.
template <int EPI, typename TQ, bool GENPOT, bool RUNS, bool COH>
__device__ __forceinline__ void member_tile(bool runs, const BackArgs &b, int t, int tile) {
    if (RUNS && runs)
        back_run_body<EPI, TQ, GENPOT, kBlock, COH>(b, t, tile);
    else
        back_tile_body<EPI, TQ, GENPOT, COH>(b, t, tile);
}

// Member update of one tile: the member's algorithm and table type select
// the epilogue (the single-state launch's template arguments).
template <bool GENPOT, bool RUNS, bool COH = false>
__device__ __forceinline__ void member_update_tile(int algo, int table_dtype, bool runs, const BackArgs &b, int t,
                                                   int tile) {
    switch (algo) {
        case PET_ALGO_OSEM: member_tile<EPI_OSEM, float, GENPOT, RUNS, COH>(runs, b, t, tile); break;
        case PET_ALGO_SVREM: member_tile<EPI_SVREM, float, GENPOT, RUNS, COH>(runs, b, t, tile); break;
        case PET_ALGO_SAGA:
            if (table_dtype == PET_TABLE_BF16)
                member_tile<EPI_SAGA, __nv_bfloat16, GENPOT, RUNS, COH>(runs, b, t, tile);
            else
                member_tile<EPI_SAGA, float, GENPOT, RUNS, COH>(runs, b, t, tile);
            break;
        case PET_ALGO_SGA: member_tile<EPI_SGA, float, GENPOT, RUNS, COH>(runs, b, t, tile); break;
        case PET_ALGO_SEM: member_tile<EPI_SEM, float, GENPOT, RUNS, COH>(runs, b, t, tile); break;
        case PET_ALGO_SAGAEM: member_tile<EPI_SAGAEM, float, GENPOT, RUNS, COH>(runs, b, t, tile); break;
        default: member_tile<EPI_SVRG, float, GENPOT, RUNS, COH>(runs, b, t, tile); break;
    }
}

}  // namespace

}  // namespace petvr
