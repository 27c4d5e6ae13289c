// Back projection as a pixel-driven gather (K2), fused with the per-pixel
// update of each method (K3).
//
// b_n = sum_{m in S_t} a_mn r_m as a gather per pixel (no atomics, so the
// result is deterministic).  Single slices use tiles that stage the bins they
// need of every view (back_tile_kernel, here) or walk runs of 8 pixels
// (back_run_kernel), with the same bits; slice stacks and multi-ring volumes
// have their own kernels in volume_back.cu (a lane per slice of a pixel; each
// band piece split over the layers its axial range crosses).  In each view only
// the bins whose ray can cross the pixel's major band at the pixel are
// candidates (usually 2-3), found from the bin spacing K, and each candidate's
// weight comes from band_point() / band_weights(), the functions the forward
// kernels use, so A^T here is the exact transpose of A there.
//
// The epilogue then applies the method's update with b_n still in a
// register (the penalty's neighbours, 4 in a plane and 2 more along z in a
// volume, are read from f^k, §3):
//   OSEM   f' = root(a = f b, S = sens_t, beta / N_s)                (§2.2, §3)
//   SVREM  s' = (1-alpha) s + alpha (N_s f b - N_s f_anc B_t + s_anc),
//          f' = root(a = s', S = sens, beta)                        (§2.3, §3)
//   SAGA   q = b - sens_t - (beta/N_s) grad R(f);
//          f' = max(0, f + alpha d (q - q_t + qbar)); qbar += (q - q_t)/N_s;
//          q_t = q                                                  (§4)
//   SVRG   f' = max(0, f + alpha d (b - B_t - (beta/N_s) grad R(f) + q~))
//          (the anchor's penalty terms cancel against those inside q~) (§4)
//   ANCHOR B_t = b for every subset t at once (grid.y = t)
//   SAGA_INIT table_t = b - sens_t - (beta/N_s) grad R(f) for every t.
#include <algorithm>

#include "bodies.cuh"

namespace petvr {

namespace {

constexpr int kBackMinBlocks = 4;

template <int EPI, typename TQ, bool GENPOT>
__global__ void __launch_bounds__(kBlock, kBackMinBlocks) back_tile_kernel(const BackArgs a) {
    const int t = a.t_dev ? __ldg(a.t_dev) : a.t0 + (int)blockIdx.y;
    back_tile_body<EPI, TQ, GENPOT>(a, t, blockIdx.x);
}

// Runs: at 48 registers two 512-thread blocks fit an SM, or five of 256.
constexpr int kRunRegs = 48;

template <int EPI, typename TQ, bool GENPOT, int NT>
__global__ void __maxnreg__(kRunRegs) back_run_kernel(const BackArgs a) {
    const int t = a.t_dev ? __ldg(a.t_dev) : a.t0 + (int)blockIdx.y;
    back_run_body<EPI, TQ, GENPOT, NT>(a, t, blockIdx.x);
}

// All-subset launches and plain back projections without that bound: the compiler
// takes 40 registers for table fills (six blocks of 256 threads an SM; 48 for
// anchors) and for 512 threads (three an SM), and 57 for 1024 (one).
template <int EPI, typename TQ, bool GENPOT, int NT>
__global__ void __launch_bounds__(NT) back_run_all_kernel(const BackArgs a) {
    back_run_body<EPI, TQ, GENPOT, NT>(a, a.t0 + (int)blockIdx.y, blockIdx.x);
}

// Persistent batched back projection + update: a resident grid whose blocks
// claim work items until the list is exhausted.  An item is one tile of a
// member's update (WK_BACK_UPDATE) or one (subset, tile) of a member's anchor
// back projection (WK_BACK_ANCHOR), by runs or staged bins, with the bits of the
// member's own launches.
// Thread 0 claims the item and writes its arguments to shared memory; the
// segment table is staged in shared memory once per block.
// GENPOT: the members of this launch use an edge-preserving potential.
// RUNS: some member's bins are wide enough for runs (batch_runs); a kernel without
// them is 1 to 3% faster for the others.
template <bool GENPOT, bool RUNS>
__global__ void __launch_bounds__(kBlock, kBackMinBlocks)
    persistent_back_kernel(const BatchMember *ms, const WorkSeg *segs, int n_segs, int n_items, int iter,
                           int in_is_img, int *claim) {
    __shared__ WorkSeg s_segs[kSegSmem];
    __shared__ BackArgs s_b;
    __shared__ int s_item, s_t, s_tile, s_kind, s_algo, s_tq, s_runs;
    for (int i = threadIdx.x; i < n_segs && i < kSegSmem; i += blockDim.x) s_segs[i] = segs[i];
    const WorkSeg *tab = n_segs <= kSegSmem ? s_segs : segs;
    // the segment table and member descriptors were copied in before the
    // kernel ahead of this one; the claim counter was zeroed by a kernel, so
    // wait for the kernel ahead before the first claim
    pdl_wait();
    pdl_trigger();
    // the first item of each block is its own index; later ones are claimed
    // (the counter counts claims beyond the grid's first items)
    for (int round = 0;; ++round) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const int g = round == 0 ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(claim, 1);
            s_item = g;
            if (g < n_items) {
                const WorkSeg sg = tab[find_segment(tab, n_segs, g)];
                const BatchMember &m = ms[sg.member];
                BackArgs b{};
                b.views = m.views;
                b.uc = m.uc;
                b.order = m.order;
                b.sub_off = m.sub_off;
                b.nx = m.nx;
                b.ny = m.ny;
                b.nz = 1;
                b.nb = m.nb;
                b.ns = m.ns;
                b.bw = m.bw;
                b.cand = m.cand;
                const int local = g - sg.first;
                if (sg.kind == WK_BACK_ANCHOR) {
                    const int t = local / sg.tiles;
                    b.r = m.ratio_full;
                    b.r_view0 = 0;
                    b.out = const_cast<float *>(m.B);
                    s_t = t;
                    s_tile = local - t * sg.tiles;
                } else {
                    b.t_dev = m.seq + iter;
                    b.r = m.ratio;
                    b.f = in_is_img ? m.img : m.alt;
                    b.f_out = in_is_img ? m.alt : m.img;
                    b.sens_t = m.sens_t;
                    b.sens = m.sens;
                    b.beta = m.beta;
                    b.pot = m.pot;
                    b.delta = m.delta;
                    b.alpha = m.alpha;
                    b.alpha_dev = m.alphas ? m.alphas + iter : nullptr;
                    b.s_hat = m.s_hat;
                    b.f_anc = m.f_anc;
                    b.s_anc = m.s_anc;
                    b.B = m.B;
                    b.d = m.d;
                    b.table = m.table;
                    b.qbar = m.qbar;
                    b.qtil = m.qtil;
                    s_t = __ldg(m.seq + iter);
                    s_tile = local;
                }
                s_b = b;
                s_kind = sg.kind;
                s_algo = m.algo;
                s_tq = m.table_dtype;
                s_runs = m.runs;
            }
        }
        __syncthreads();
        if (s_item >= n_items) break;
        const int t = s_t, tile = s_tile;
        if (s_kind == WK_BACK_ANCHOR)
            member_tile<EPI_ANCHOR, float, false, RUNS, false>(s_runs, s_b, t, tile);
        else
            member_update_tile<GENPOT, RUNS>(s_algo, s_tq, s_runs, s_b, t, tile);
    }
}

// Dynamic shared memory (at least `base` bytes) that a subset launch of `blocks`
// blocks asks for to bound how many of them an SM holds.  A dependent launch's
// blocks are placed while the kernel ahead still runs, and pile up on the SMs
// that have room, up to the register limit of four, while others stay empty:
// the fullest SM sets the time.  Bounded to one above the even share; a tighter
// bound was faster alone and slower with several streams.  256^2: a SAGA epoch
// 160 us (no bound: 176), the four-method step on four streams 2055 us (1994);
// at an even share of three and more the register limit does.
// The kernel's allowance is the amount of the tightest bound, whatever this launch asks for.
template <auto kKernel>
size_t residency_smem(int blocks, size_t base) {
    const int cap = (blocks + sm_count() - 1) / sm_count() + 1;      // 2 and more
    if (cap > 3) return base;
    constexpr size_t kPerSm = 227 << 10;                             // shared memory of an SM
    const size_t need = kPerSm / (size_t)(cap + 1);
    return need > base && allow_shared_memory<kKernel>(kPerSm / 3) == cudaSuccess ? need : base;
}

// Whether an update from `views` views over `tiles` tiles takes runs instead of
// staged bins (the same bits).  A thread of the staged bins reads two or three
// candidates a view in an unrolled loop, however wide the bins, and more of them in
// a loop of its own; a run evaluates each band it meets once, in a longer chain, and
// 16 views at a time.  us per SAGA update in a graph, staged bins (runs):
// - up to two tiles an SM: 512 threads.  More than three candidates: 64^2 at 4 bins a
//   pixel x 5 views 7.3 (8.0), x 6 8.4 (7.9), x 16 17.2 (11.0); 128^2 at 2.2 x 9 9.3
//   (9.7), x 14 12.4 (10.2).  Three: 48^2 at 1.54 bins a pixel x 10 6.2 (5.6), 256^2
//   x 14 12.3 (11.1), x 20 17.3 (15.7); at 2, 128^2 x 20 10.9 (13.0).  Two: a bin a
//   pixel 128^2 x 14 6.7 (7.0), x 60 16.8 (18.8); two tiles an SM, 256^2 x 9 8.1
//   (9.2), x 12 9.1 (9.5), x 14 10.0 (8.8), x 20 11.5 (11.9), x 32 17.3 (15.7), x 60
//   25.8 (25.7; beside other streams the staged bins are 3% faster); wider bins, of
//   which a run meets fewer: 201x199 at 0.6 x 14 8.2 (6.8).
// - up to four: a thread a run.  300^2 at 2.2 x 12 20.2 (16.1), at 4 x 16 38.2 (39.4);
//   350^2 at 1 x 6 8.8 (10.1).
// - beyond: 256 threads.  Few views 512^2 x 4 14.0 (12.0), x 2 10.0 (10.6); wider bins
//   800x700 at 0.6 x 8 31.4 (24.4); four or five candidates 400^2 at 2.2 x 8 21.2
//   (18.2); more, 400^2 at 12 x 8 57.5 (64.7).
// 1444 points against runs everywhere with a thread each: 0.88 of the time on
// average (staged bins everywhere 0.93, and a quarter of the points slower).
bool update_by_runs(const BackArgs &a, int tiles, int views) {
    const int sms = sm_count();
    const bool wide_bins = a.fineness < 0.9f;
    if (tiles > 4 * sms)
        return a.cand <= 2 ? wide_bins || (views > 2 && views <= 6) : a.cand == 4 || a.cand == 5;
    constexpr int kPass = kRunViews<512>, kNever = kMaxViews;
    const int passes = (views + kPass - 1) / kPass;
    if (tiles > 2 * sms) return a.cand > 3 && a.fineness < 3.0f && views > 8 * passes;
    int most = kNever;                                      // views up to which staged bins are faster
    const bool few = tiles <= sms / 8;
    if (a.cand > 3)
        most = (few ? 5 : 8) * passes;
    else if (a.cand == 3 && a.fineness < 1.8f)
        most = tiles > sms ? 12 : (few ? 9 : 12) * passes;
    else if (a.cand == 3)
        most = few ? 15 * passes : kNever;
    else if (wide_bins)
        most = (tiles > sms ? 8 : 10) * passes;
    else if (tiles > sms)
        most = passes <= 2 ? 12 * passes : kNever;
    return views > most;
}

// Single-slice back-projection launch of one epilogue / table type / potential.
struct TileBack {
    const BackArgs &a;
    int ny_grid;
    cudaStream_t s;
    int max_views;

    template <auto kKernel, int NT>
    pet_status run_launch(dim3 grid, int threads = NT) const {
        launch_dependent(kKernel, grid, dim3((unsigned)threads), run_smem_bytes<NT>(), s, a);
        return check_launch("back_run_kernel");
    }

    // Plain back projections (no update behind them): runs, one per thread and pass.
    // The blocks of a launch are placed while the kernel ahead still runs, so an SM
    // that can take three piles them up where two each would do.  Forward + back in
    // a graph, bins = pixels:
    // - up to two blocks an SM: 512 threads at 48 registers, 128^2 x 64 views
    //   18.5 us (40 registers, so three an SM: 24.2), 256^2 x 90 36.3 (44.7);
    // - one block an SM and several passes: 1024 threads, 128^2 x 90 16.4 (21.5);
    //   with 256^2's 256 tiles 38.7 (36.3);
    // - more blocks: 512 threads, three an SM, 300^2 x 30 18.0 (two: 20.7);
    // - many blocks, few views: 256 threads (a run each), 512^2 x 6 13.9 (15.2);
    //   300^2's 361 tiles 8.1 (7.4).
    pet_status run_plain(dim3 grid) const {
        const int blocks = (int)(grid.x * grid.y), sms = sm_count();
        if (blocks <= sms && max_views > 64) return run_launch<back_run_all_kernel<EPI_PLAIN, float, false, 1024>, 1024>(grid);
        if (blocks <= 2 * sms) return run_launch<back_run_kernel<EPI_PLAIN, float, false, 512>, 512>(grid);
        if (blocks > 3 * sms && max_views <= 8)
            return run_launch<back_run_kernel<EPI_PLAIN, float, false, kBlock>, kBlock>(grid);
        return run_launch<back_run_all_kernel<EPI_PLAIN, float, false, 512>, 512>(grid);
    }

    template <int EPI, typename TQ, bool GENPOT>
    pet_status run() const {
        const int tiles = ((a.nx + kTile - 1) / kTile) * ((a.ny + kTile - 1) / kTile);
        const dim3 grid((unsigned)tiles, (unsigned)ny_grid);
        if constexpr (EPI == EPI_PLAIN) {
            return run_plain(grid);
        } else if constexpr (EPI == EPI_ANCHOR || EPI == EPI_SAGA_INIT || EPI == EPI_SAGAEM_INIT) {
            // A table fill takes five blocks an SM (48 registers) unless six spare a
            // round of blocks or there are many rounds: 64^2 x 6 subsets 18.9 us (six:
            // 20.6), 201^2 x 7 53.3 (54.8); 256^2 x 3 80.3 (76.1), x 21 80.2 (78.6).
            if constexpr (EPI == EPI_SAGA_INIT) {
                const int blocks = tiles * ny_grid, sms = sm_count();
                const int rounds5 = (blocks + 5 * sms - 1) / (5 * sms), rounds6 = (blocks + 6 * sms - 1) / (6 * sms);
                if (rounds5 == rounds6 && blocks <= 8 * sms)
                    return run_launch<back_run_kernel<EPI, TQ, GENPOT, kBlock>, kBlock>(grid);
            }
            return run_launch<back_run_all_kernel<EPI, TQ, GENPOT, kBlock>, kBlock>(grid);
        } else {
            if (update_by_runs(a, tiles, max_views)) {
                const int sms = sm_count();
                if (tiles <= 2 * sms) return run_launch<back_run_kernel<EPI, TQ, GENPOT, 512>, 512>(grid);
                return run_launch<back_run_kernel<EPI, TQ, GENPOT, 0>, 0>(
                    grid, tiles > 4 * sms ? kBlock : std::max(kBlock, 32 * std::min(max_views, kRunViews<0>)));
            }
            constexpr auto k = back_tile_kernel<EPI, TQ, GENPOT>;
            const size_t smem = tile_smem_bytes();
            launch_dependent(k, grid, dim3(kBlock), a.t_dev ? residency_smem<k>(tiles, smem) : smem, s, a);
            return check_launch("back_tile_kernel");
        }
    }
};

}  // namespace

// Bins a tile stages per view.  Over the tile's kTile x kTile pixels the first
// candidate moves by at most (kTile - 1) (|cos| + |sin|) <= sqrt(2) (kTile - 1)
// pixel / bin, and a pixel has at most (1 + |du|) |cos| <= sqrt(2) pixel / bin + 1
// of them; the unrolled loops always read two or three, and the rest is margin
// for rounding (see tile_view).  Bin numbers of 2^20 and more are beyond what the
// candidates' float positions resolve: such plans read their bins in place
// (a value above kStageBins).
void tile_bins(double pixel_mm, double bin_mm, int nb, int nx, int ny, int &bw, int &cand) {
    const double ratio = pixel_mm / bin_mm;
    const double eps = 1e-3 + 4e-7 * ((double)nb + nx + ny);
    bw = kStageBins + 1;
    cand = kUnrolledCand + 1;
    if (nb >= (1 << 20) || ratio > (double)kStageBins) return;
    cand = std::max(2, (int)std::floor(1.41422 * ratio + 2.0 * eps) + 1);
    bw = std::min(kStageBins + 1, (int)std::ceil((kTile - 1) * 1.41422 * ratio) + cand + 4);
}

// Members of a batch fill the grid and are bound by issue: those whose bins are wider
// than a pixel, of which a run meets fewer, take runs.  Epoch of 5 updates from 8
// views each, 64 SAGA members of 64^2 to 200^2, us with staged bins (runs): 0.6 bins a
// pixel 457 (405), 0.77 483 (447), 1.0 524 (503); 24 members of 64^2 to 256^2 with 5
// to 60 views at 1.0, 12 updates 1630 (1758).  In one dependency-driven launch: 0.6
// 532 (498), 0.77 581 (559), 1.0 647 (642), and 2106 (2209).
bool batch_runs(const pet_plan *pl) { return pl->fineness < 0.9f; }

pet_status launch_persistent_back(const BatchMember *d_members, const WorkSeg *d_segs, int n_segs, int n_items,
                                  int iter, int in_is_img, int *claim, bool general_potential, bool runs,
                                  cudaStream_t s) {
    if (n_items <= 0) return PET_OK;
    void (*k)(const BatchMember *, const WorkSeg *, int, int, int, int, int *) =
        runs ? (general_potential ? persistent_back_kernel<true, true> : persistent_back_kernel<false, true>)
             : (general_potential ? persistent_back_kernel<true, false> : persistent_back_kernel<false, false>);
    const size_t smem = tile_smem_bytes();
    static int resident[4] = {};   // blocks per SM of each kernel
    int &per_sm = resident[(general_potential ? 1 : 0) + (runs ? 2 : 0)];
    if (per_sm == 0 &&
        (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)k, kBlock, smem) != cudaSuccess ||
         per_sm < 1))
        per_sm = 1;
    const int grid = std::min(n_items, per_sm * sm_count());
    ProfileScope prof(1, s);
    launch_dependent(k, dim3((unsigned)grid), dim3(kBlock), smem, s, d_members, d_segs, n_segs, n_items,
                     iter, in_is_img, claim);
    return check_launch("persistent_back_kernel");
}

pet_status launch_back(const BackArgs &a, int epi, int table_dtype, int n_subsets_grid,
                       cudaStream_t s, int max_views) {
    ProfileScope prof(n_subsets_grid > 1 ? 2 : 1, s);
    if (a.axial || a.nz > 1) return launch_back_volume(a, epi, table_dtype, n_subsets_grid, s, max_views);
    return with_epilogue(epi, table_dtype, a.pot, TileBack{a, n_subsets_grid, s, max_views});
}

}  // namespace petvr
