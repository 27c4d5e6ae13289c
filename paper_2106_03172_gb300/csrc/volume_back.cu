// Back projections for volumes (K2 + K3): slice stacks (nz independent
// slices sharing one 2-D geometry) and multi-ring scanners (fully 3-D lines
// of response through a voxel volume), each ending in the same per-pixel
// update as the single-slice kernels (epilogue.cuh).  The multi-ring weights
// come from the expressions the forward projector uses (piece_fraction /
// piece_zeta / layer_fraction), so A^T is the exact transpose of A.
#include <algorithm>
#include <cmath>

#include "epilogue.cuh"

namespace petvr {

namespace {

// Slice-stack path: the geometry is shared by every slice.  A warp takes 4
// consecutive pixels and a window of 8 ZW consecutive slices; its lanes are
// 4 pixel groups x 8 z-lanes, and z-lane l carries slices l, l + 8, ... of the
// window, so each ratio load reads 8 consecutive floats of a bin's slice
// column ([view][bin][z]: coalesced).  The groups walk the subset's views in
// the same order (their candidate bins differ by about one, so the warp stays
// converged).  In each view, z-lane l of a group evaluates the band piece of
// candidate bin jlo + l of its pixel and the group's lanes take the weight by
// a shuffle; views and candidates are added in order (deterministic).  Each
// lane then applies the update to its own slices.
template <int EPI, typename TQ, bool GENPOT, int ZW>
__global__ void __launch_bounds__(kBlock) back_slim_kernel(const BackArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ViewParams *s_views = reinterpret_cast<ViewParams *>(smem_raw);
    const int t = a.t_dev ? __ldg(a.t_dev) : a.t0 + (int)blockIdx.y;
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    int *s_vid = reinterpret_cast<int *>(s_views + nv);
    stage_views(a, vb, nv, s_views, s_vid);
    __syncthreads();
    const int r_view0 = a.t_dev ? vb : a.r_view0;

    // 32-bit index arithmetic: images and sinograms are below 2^31 elements (checked at plan time)
    const int n_win = (a.nz + 8 * ZW - 1) / (8 * ZW);
    const int lane = threadIdx.x & 31;
    const int zl = lane & 7;                              // z-lane
    const int pg = lane >> 3;                             // pixel group
    const unsigned gmask = 0xffu << (8 * pg);             // the group's 8 z-lanes
    const int wid = blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5);
    const int quad = wid / n_win;
    const int win = wid - quad * n_win;
    const int n = kStackPixels * quad + pg;               // pixel
    const bool live = n < a.nx * a.ny;
    const int ix = n % a.nx;
    const int iy = n / a.nx;
    const int z0 = win * 8 * ZW + zl;                     // this lane's first slice
    const int n_zi = live ? min(ZW, max(0, (a.nz - z0 + 7) / 8)) : 0;

    float acc[ZW];
#pragma unroll
    for (int i = 0; i < ZW; ++i) acc[i] = 0.0f;
    if (live) {
        for (int q = 0; q < nv; ++q) {
            const ViewParams vp = s_views[q];
            const int v = s_vid[q];
            const int k = vp.col ? ix : iy;              // major index
            const int minor = vp.col ? iy : ix;
            const int n_major = vp.col ? a.nx : a.ny;
            const int n_minor = vp.col ? a.ny : a.nx;
            const int mrel = minor - (n_minor >> 1);
            const float kc = (float)k - 0.5f * (float)n_major;
            int jlo, jhi;
            candidate_bins(vp, kc, (float)mrel, (float)mrel + 1.0f, a.nb, jlo, jhi);
            const float2 *ucv = a.uc + v * a.nb;
            const float *rv = a.r + (vb + q - r_view0) * a.nb * a.nz + z0;
            for (int jb = jlo; jb <= jhi; jb += 8) {     // the same trip count for the group's 8 lanes
                const int j = jb + zl;
                float w = 0.0f;
                if (j <= jhi) {
                    const float2 u = __ldg(ucv + j);
                    float fl, w0, w1;
                    band_split(vp, band_point(vp, u.y, kc), band_point(vp, u.y, kc + 1.0f), fl, w0, w1);
                    const int c0 = (int)fl + (int)u.x;
                    w = (c0 == mrel) ? w0 : ((c0 + 1 == mrel) ? w1 : 0.0f);
                }
                const int nc = min(8, jhi - jb + 1);
                for (int b = 0; b < nc; ++b) {
                    const float wb = __shfl_sync(gmask, w, b, 8);
                    if (wb == 0.0f) continue;
                    const float *rj = rv + (jb + b) * a.nz;
#pragma unroll
                    for (int i = 0; i < ZW; ++i)
                        if (i < n_zi) acc[i] = fmaf(wb, __ldg(rj + 8 * i), acc[i]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < ZW; ++i)
        if (i < n_zi) {
            const int z = z0 + 8 * i;
            apply_epilogue<EPI, TQ, GENPOT>(a, t, (long long)n * a.nz + z, n, ix, iy, z, acc[i]);
        }
}

// Slice-stack path: the geometry is shared by every slice.  A warp takes one
// pixel and a window of 32 W consecutive slices, lane l the slices l, l + 32,
// ... of the window, so a load instruction reads 32 consecutive floats of one
// bin's slice column ([view][bin][z]).  The lanes share the candidate bins of
// the subset's views among them (a.cands per view), evaluate each one's band
// piece once for all slices, and leave the nonzero weights, in view and bin
// order, in shared memory; the warp then walks that list in order
// (deterministic), and each lane applies the update to its own slices.  Bound
// by instruction issue.  47 slices of 128^2 (ncu), against 4 pixels x 8 z-lanes
// (back_slim_kernel's layout): anchor of 14 subsets 291 -> 230 us, an update
// 38 -> 30 us.
constexpr int kStackPieces = 96;     // list entries per warp (a round adds up to 32)

template <int EPI, typename TQ, bool GENPOT, int W>
__global__ void __launch_bounds__(kBlock, 5) back_stack_kernel(const BackArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float2 s_piece[kBlock / 32][kStackPieces];   // ratio offset, weight
    ViewParams *s_views = reinterpret_cast<ViewParams *>(smem_raw);
    const int t = a.t_dev ? __ldg(a.t_dev) : a.t0 + (int)blockIdx.y;
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    int *s_vid = reinterpret_cast<int *>(s_views + nv);
    stage_views(a, vb, nv, s_views, s_vid);
    __syncthreads();
    const int r_view0 = a.t_dev ? vb : a.r_view0;

    // 32-bit index arithmetic: images and sinograms are below 2^31 elements (checked at plan time)
    const int n_win = (a.nz + 32 * W - 1) / (32 * W);
    const int lane = threadIdx.x & 31;
    float2 *piece = s_piece[threadIdx.x >> 5];
    const int wid = blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5);
    const int n = n_win == 1 ? wid : wid / n_win;         // pixel
    const int win = n_win == 1 ? 0 : wid - n * n_win;
    if (n >= a.nx * a.ny) return;                         // the whole warp
    const int ix = n % a.nx;
    const int iy = n / a.nx;
    const int z0 = win * 32 * W + lane;                   // this lane's first slice

    float acc[W] = {};
    // a lane past the last slice reads that slice again and drops the sum
    const float *r[W];
#pragma unroll
    for (int i = 0; i < W; ++i) r[i] = a.r + min(z0 + 32 * i, a.nz - 1);
    // views per round; a view with more than 32 candidates takes cand_rounds rounds
    const int per_round = 32 / a.cands;
    const int rounds = (nv + per_round - 1) / per_round * a.cand_rounds;
    const int lq = lane / a.cands, lc = lane - lq * a.cands;
    int np = 0;
    for (int round = 0; round < rounds; ++round) {
        const int part = a.cand_rounds == 1 ? 0 : round % a.cand_rounds;
        const int q = (a.cand_rounds == 1 ? round : round / a.cand_rounds) * per_round + lq;
        float w = 0.0f;
        int off = 0;
        if (lq < per_round && q < nv) {
            const ViewParams vp = s_views[q];
            const int k = vp.col ? ix : iy;              // major index
            const int minor = vp.col ? iy : ix;
            const int n_major = vp.col ? a.nx : a.ny;
            const int n_minor = vp.col ? a.ny : a.nx;
            const int mrel = minor - (n_minor >> 1);
            const float kc = (float)k - 0.5f * (float)n_major;
            int jlo, jhi;
            candidate_bins(vp, kc, (float)mrel, (float)mrel + 1.0f, a.nb, jlo, jhi);
            const int j = jlo + lc + 32 * part;
            if (j <= jhi) {
                const float2 u = __ldg(a.uc + s_vid[q] * a.nb + j);
                float w0, w1;
                const float e0 = band_point(vp, u.y, kc), e1 = band_point(vp, u.y, kc + 1.0f);
                const float t = band_weights(vp.L, vp.Lm, fminf(e0, e1), fmaxf(e0, e1), w0, w1);
                const int c0 = (int)(__float_as_uint(t) - kRoundBits) + (int)u.x;
                w = (c0 == mrel) ? w0 : ((c0 + 1 == mrel) ? w1 : 0.0f);
                off = ((vb + q - r_view0) * a.nb + j) * a.nz;
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, w != 0.0f);
        if (w != 0.0f) piece[np + __popc(mask & ((1u << lane) - 1))] = make_float2(__int_as_float(off), w);
        np += __popc(mask);
        if (np <= kStackPieces - 32 && round + 1 < rounds) continue;     // room for another round
        __syncwarp();
        add_pieces<W>(piece, np, r, acc);
        __syncwarp();
        np = 0;
    }
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const int z = z0 + 32 * i;
        if (z < a.nz)
            apply_epilogue<EPI, TQ, GENPOT>(a, t, (long long)n * a.nz + z, n, ix, iy, z, acc[i]);
    }
}

// Multi-ring path: kLanes lanes per voxel share the subset's views (lane l
// takes views l, l+4, ...).  For each candidate bin the band piece of the
// voxel's pixel is found as in the slice-stack path; each ring pair then adds
// the part of that piece inside the voxel's layer (piece_fraction /
// piece_zeta / layer_fraction, the forward projector's own expressions).
template <int EPI, typename TQ, bool GENPOT>
__global__ void __launch_bounds__(kBlock) ring_back_kernel(const BackArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ViewParams *s_views = reinterpret_cast<ViewParams *>(smem_raw);
    const int t = a.t_dev ? __ldg(a.t_dev) : a.t0 + (int)blockIdx.y;
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    int *s_vid = reinterpret_cast<int *>(s_views + nv);
    stage_views(a, vb, nv, s_views, s_vid);
    __syncthreads();
    const int r_view0 = a.t_dev ? vb : a.r_view0;

    // 32-bit index arithmetic: images and sinograms are below 2^31 elements (checked at plan time)
    const int L = a.nz, P = a.pairs;
    const int plane = a.nx * a.ny * L;
    const long long gid = (long long)blockIdx.x * kBlock + threadIdx.x;
    const long long i = gid / kLanes;                    // voxel
    const int lane = (int)(gid % kLanes);
    const bool live = i < plane;
    const int iv = (int)i;
    const int iz = iv % L;
    const int n = iv / L;
    const int ix = n % a.nx;
    const int iy = n / a.nx;

    float acc = 0.0f;
    if (live) {
        for (int q = lane; q < nv; q += kLanes) {
            const ViewParams vp = s_views[q];
            const int v = s_vid[q];
            const int k = vp.col ? ix : iy;              // major index
            const int minor = vp.col ? iy : ix;
            const int n_major = vp.col ? a.nx : a.ny;
            const int n_minor = vp.col ? a.ny : a.nx;
            const int mrel = minor - (n_minor >> 1);
            const float kc = (float)k - 0.5f * (float)n_major;
            int jlo, jhi;
            candidate_bins(vp, kc, (float)mrel, (float)mrel + 1.0f, a.nb, jlo, jhi);
            const float2 *ucv = a.uc + v * a.nb;
            const float4 *lzv = a.lz + v * a.nb * P;
            const float *rv = a.r + (vb + q - r_view0) * a.nb * P;
            for (int j = jlo; j <= jhi; ++j) {
                const float2 u = __ldg(ucv + j);
                float fl, w0, w1;
                band_split(vp, band_point(vp, u.y, kc), band_point(vp, u.y, kc + 1.0f), fl, w0, w1);
                const int c0 = (int)fl + (int)u.x;
                const int side = (c0 == mrel) ? 0 : ((c0 + 1 == mrel && w1 > 0.0f) ? 1 : -1);
                if (side < 0) continue;
                const float w = side ? w1 : w0;
                float f_lo, f_hi;
                piece_fraction(vp, w0, w1, side == 1, f_lo, f_hi);
                for (int pr = 0; pr < P; ++pr) {
                    const float4 lz = __ldg(lzv + j * P + pr);
                    const float fr = layer_fraction(piece_zeta(lz, kc, f_lo), piece_zeta(lz, kc, f_hi), iz);
                    if (fr > 0.0f) acc = fmaf((w * lz.z) * fr, __ldg(rv + j * P + pr), acc);
                }
            }
        }
    }
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (!live || lane != 0) return;
    apply_epilogue<EPI, TQ, GENPOT>(a, t, i, n, ix, iy, iz, acc);
}

// Multi-ring path for volumes of at most LMAX layers: a block owns kColumns
// pixel columns (a warp 32 neighbours along x) and kViewLanes groups of its
// warps share the subset's views, so that a warp's columns walk one view's bins
// together.  Every candidate bin's band piece is found once per column and each
// ring pair's share is added to the layers its axial range crosses (piece_layers;
// per-layer sums in registers).  The groups' sums meet in shared memory and are
// added pairwise, and every thread updates voxels of the block's columns.
//
// Bound by instruction issue and, on subset launches, by the launch's latency.
// Against four lanes per column on a view each (diverging) and a loop over the
// layers with a division each: an SVREM epoch of the 2-ring 128^2 x 3 volume
// 879 -> 687 us.
constexpr int kColumns = 64;
constexpr int kViewLanes = kBlock / kColumns;

template <int EPI, typename TQ, bool GENPOT, int LMAX>
__global__ void __launch_bounds__(kBlock) ring_back_column_kernel(const BackArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float s_sum[kViewLanes][LMAX][kColumns];
    ViewParams *s_views = reinterpret_cast<ViewParams *>(smem_raw);
    const int t = a.t_dev ? __ldg(a.t_dev) : a.t0 + (int)blockIdx.y;
    const int vb = __ldg(a.sub_off + t);
    const int nv = __ldg(a.sub_off + t + 1) - vb;
    int *s_vid = reinterpret_cast<int *>(s_views + nv);
    stage_views(a, vb, nv, s_views, s_vid);
    __syncthreads();
    const int r_view0 = a.t_dev ? vb : a.r_view0;

    // 32-bit index arithmetic: images and sinograms are below 2^31 elements (checked at plan time)
    const int L = a.nz, P = a.pairs;
    const int npix = a.nx * a.ny;
    const int col = threadIdx.x % kColumns, group = threadIdx.x / kColumns;
    const int n = blockIdx.x * kColumns + col;           // pixel
    const int iy = n / a.nx;
    const int ix = n - iy * a.nx;

    float acc[LMAX];
#pragma unroll
    for (int iz = 0; iz < LMAX; ++iz) acc[iz] = 0.0f;
    if (n < npix) {
        for (int q = group; q < nv; q += kViewLanes) {
            const ViewParams vp = s_views[q];
            const int v = s_vid[q];
            const int k = vp.col ? ix : iy;              // major index
            const int minor = vp.col ? iy : ix;
            const int n_major = vp.col ? a.nx : a.ny;
            const int n_minor = vp.col ? a.ny : a.nx;
            const int mrel = minor - (n_minor >> 1);
            const float kc = (float)k - 0.5f * (float)n_major;
            int jlo, jhi;
            candidate_bins(vp, kc, (float)mrel, (float)mrel + 1.0f, a.nb, jlo, jhi);
            const float2 *ucv = a.uc + v * a.nb;
            const float4 *lzv = a.lz + v * a.nb * P;
            const float *rv = a.r + (vb + q - r_view0) * a.nb * P;
            for (int j = jlo; j <= jhi; ++j) {
                const float2 u = __ldg(ucv + j);
                const float e0 = band_point(vp, u.y, kc), e1 = band_point(vp, u.y, kc + 1.0f);
                float w0, w1;
                const float tl = band_weights(vp.L, vp.Lm, fminf(e0, e1), fmaxf(e0, e1), w0, w1);
                const int c0 = (int)(__float_as_uint(tl) - kRoundBits) + (int)u.x;
                const int side = (c0 == mrel) ? 0 : ((c0 + 1 == mrel && w1 > 0.0f) ? 1 : -1);
                if (side < 0) continue;
                const float w = side ? w1 : w0;
                float f_lo, f_hi;
                piece_fraction(vp, w0, w1, side == 1, f_lo, f_hi);
                for (int pr = 0; pr < P; ++pr) {
                    const float4 lz = __ldg(lzv + j * P + pr);
                    const float wr = __ldg(rv + j * P + pr);
                    const float wl = w * lz.z;
                    piece_layers(piece_zeta(lz, kc, f_lo), piece_zeta(lz, kc, f_hi), L, [&](int layer, float fr) {
#pragma unroll
                        for (int iz = 0; iz < LMAX; ++iz)
                            if (iz == layer) acc[iz] = fmaf(wl * fr, wr, acc[iz]);
                    });
                }
            }
        }
    }
#pragma unroll
    for (int iz = 0; iz < LMAX; ++iz) s_sum[group][iz][col] = acc[iz];
    __syncthreads();
    // voxel e of the block's columns, in image order
    for (int e = threadIdx.x; e < kColumns * L; e += kBlock) {
        const int c = e / L, iz = e - c * L;
        const int m = blockIdx.x * kColumns + c;
        if (m >= npix) break;
        static_assert(kViewLanes == 4, "the order of the sum");
        const float val = (s_sum[0][iz][c] + s_sum[2][iz][c]) + (s_sum[1][iz][c] + s_sum[3][iz][c]);
        const int my = m / a.nx, mx = m - my * a.nx;
        apply_epilogue<EPI, TQ, GENPOT>(a, t, m * L + iz, m, mx, my, iz, val);
    }
}

// Back-projection launches of one epilogue / table type / potential.
struct VolumeBack {
    const BackArgs &a;
    int ny_grid;
    cudaStream_t s;
    int max_views;

    // Launch with the views of the largest subset staged in shared memory.  Beside
    // the kernels' own at most kOwnShared bytes, 48 KB hold 787 views of them.
    template <auto kKernel>
    pet_status launch(dim3 grid) const {
        constexpr size_t kPerView = sizeof(ViewParams) + sizeof(int), kOwnShared = 8 << 10;
        const size_t smem = (size_t)max_views * kPerView;
        if (smem + kOwnShared > (48 << 10)) {
            const cudaError_t e = allow_shared_memory<kKernel>(kMaxViews * kPerView);
            if (e != cudaSuccess)
                return set_error(PET_ERR_CUDA, std::string("volume back projection: ") + cudaGetErrorString(e));
        }
        kKernel<<<grid, kBlock, smem, s>>>(a);
        return check_launch("volume back projection");
    }

    template <int EPI, typename TQ, bool GENPOT>
    pet_status run() const {
        if (a.axial && a.nz <= 8) {                     // multi-ring, layers in registers
            const dim3 grid((unsigned)((a.nx * a.ny + kColumns - 1) / kColumns), (unsigned)ny_grid);
            return a.nz <= 4 ? launch<ring_back_column_kernel<EPI, TQ, GENPOT, 4>>(grid)
                             : launch<ring_back_column_kernel<EPI, TQ, GENPOT, 8>>(grid);
        }
        if (a.axial) {                                  // multi-ring, one voxel per lane group
            const long long threads = (long long)a.nx * a.ny * a.nz * kLanes;
            const dim3 grid((unsigned)((threads + kBlock - 1) / kBlock), (unsigned)ny_grid);
            return launch<ring_back_kernel<EPI, TQ, GENPOT>>(grid);
        }
        const int w = stack_lane_slices(a.nz);
        const long long pixels = (long long)a.nx * a.ny;
        // one warp per kStackPixels pixels, or per pixel and slice window
        const long long warps = w == 0 ? (pixels + kStackPixels - 1) / kStackPixels : pixels * stack_windows(a.nz);
        const dim3 grid((unsigned)((warps + kBlock / 32 - 1) / (kBlock / 32)), (unsigned)ny_grid);
        switch (w) {
            case 0: return launch<back_slim_kernel<EPI, TQ, GENPOT, kSlimSlices / 8>>(grid);
            case 1: return launch<back_stack_kernel<EPI, TQ, GENPOT, 1>>(grid);
            default: return launch<back_stack_kernel<EPI, TQ, GENPOT, 2>>(grid);
        }
    }
};

}  // namespace

// candidate_bins() gives the bins whose positions lie in a range of (1 + |du| +
// 2 kCandEps) |cos| <= sqrt(2) + 2 kCandEps pixels, over bin spacings; the rest
// is margin for the positions' rounding.
void stack_candidates(double pixel_mm, double bin_mm, int nb, int nx, int ny, int &cands, int &rounds) {
    const double ratio = pixel_mm / bin_mm;
    const double most = (1.41422 + 2.0 * kCandEps) * ratio + 1e-2 + 2e-6 * ((double)nb + nx + ny);
    const int n = most < nb ? (int)std::floor(most) + 1 : nb;
    cands = std::min(n, 32);
    rounds = (n + 31) / 32;
}

pet_status launch_back_volume(const BackArgs &a, int epi, int table_dtype, int n_subsets_grid, cudaStream_t s,
                              int max_views) {
    return with_epilogue(epi, table_dtype, a.pot, VolumeBack{a, n_subsets_grid, s, max_views});
}

}  // namespace petvr
