// project_pts.cu -- tilings and launch of the FP32 point-owner projection
// kernel (project_pts.cuh): shared-memory size and dispatch over the compiled
// (dims, free columns, fixed-column multipliers) variants.
#include <algorithm>

#include "project_pts.cuh"

namespace priest {

namespace {

using pts::kSmemCap;
using pts::kSmemHalf;
// Samples one warp takes per item of the persistent launch: enough to bury
// the staging of the item's tables, few enough for an even end.
constexpr int kSamplesPerWarp = 4;

}  // namespace

namespace {

pts::PtsLayout layout_of(const Shape &sh, int G, int warps, int C)
{
    return pts::pts_layout(G, sh.dims, sh.nf, sh.nv, sh.n_p, sh.n_obs, sh.n_static, warps, C > 1 ? warps / C : 0);
}

}  // namespace

size_t pts_smem_bytes(const Shape &sh, int G, int warps, int C)
{
    return layout_of(sh, G, warps, C).total * sizeof(float);
}

// Degree 10 with the "at rest" end (5 free coefficients per axis), 2-D or
// 3-D; or 2-D with the end position only (7 free coefficients: the paper's
// four boundary rows per axis).
bool pts_supported(const Shape &sh)
{
    return sh.nv == 11 && ((sh.nf == 5 && (sh.dims == 2 || sh.dims == 3)) || (sh.nf == 7 && sh.dims == 2));
}

// One CTA whose first `warps` warps take 32 / G samples each (fewer warps when
// their lists do not fit).  The results depend on G alone: a sample's sums stay
// within its lanes.
Tiling pts_tiling(const Shape &sh, int G, int warps)
{
    Tiling t;
    t.kind = 1;
    t.R = G;
    t.C = 1;
    int w = std::max(1, std::min(warps, pts::kMaxWarps));
    while (w > 1 && pts_smem_bytes(sh, G, w, 1) > kSmemCap) --w;
    t.ws = w;
    t.S = w * (32 / G);
    t.threads = 32 * pts::kMaxWarps;
    t.smem = pts_smem_bytes(sh, G, w, 1);
    t.smem_fix = layout_of(sh, G, w, 1).total_fix * sizeof(float);
    if (!pts_supported(sh) || t.smem > kSmemCap) t.smem = 0;
    return t;
}

// Warps that project one sample together (0: one warp).  Teams shorten an
// iteration's chain and repeat its state steps in every warp, so they pay while
// warps are few.  Four warps up to two samples per SM (one CTA; 110 samples, K =
// 50: 2-D replan 125 against 147 us for one warp each, 3-D ellipsoids 141 against
// 225, two samples per SM 152 against 234; clutter without active velocity rows
// even).  Two warps up to eight samples per SM for 3-D and for seven columns, whose
// rows are long (600 samples: 230 against 253 us and 146 against 163); 2-D with
// five columns is even or 5 % slower with them (clutter 92 against 87 us, replan
// 159 against 161), so one warp projects it.
int pts_team_size(const Shape &sh, int samples_per_sm)
{
    if (samples_per_sm <= 2) return 4;
    return samples_per_sm <= 8 && (sh.dims == 3 || sh.nf == 7) ? 2 : 0;
}

// One CTA of `teams` teams of C warps, a sample each; smem 0: does not fit.
Tiling pts_team_tiling(const Shape &sh, int teams, int C)
{
    Tiling t;
    t.kind = 1;
    t.R = 32;
    t.C = C;
    t.ws = teams * C;
    t.S = teams;
    t.threads = 32 * pts::kMaxWarps;
    t.smem = pts_smem_bytes(sh, 32, t.ws, t.C);
    t.smem_fix = layout_of(sh, 32, t.ws, t.C).total_fix * sizeof(float);
    if (!pts_supported(sh) || t.ws > pts::kMaxWarps || t.smem > kSmemCap) t.smem = 0;
    return t;
}

// Lanes per sample: 16 leave the fixed work of an iteration (node test,
// butterfly, state-lane steps) to two samples at once; 32 halve the rows per
// lane, which counts when an SM holds few samples, and reach every n_p.  (3-D and
// seven columns keep more per lane than 128 registers hold for two samples.)
int pts_group(const Shape &sh, int samples_per_sm)
{
    return (sh.dims == 2 && sh.nf == 5 && samples_per_sm > 16 && sh.n_p <= 16 * pts::kMaxStrides) ? 16 : 32;
}

// A served request shares its launches with whatever else is there, so its lanes
// per sample, on which its sums depend, are its own shape's.  The busy server's: bursts
// of 8 / 32 / 64 uneven requests take 2.1 / 5.8 / 9.1 ms with 16 lanes, 2.3 / 6.4 / 10.5
// with 32, 2.5 / 6.3 / 9.4 when requests below 512 samples have 32 (two launches a
// step, each with its tail).  The price is a request alone: 0.44 / 0.55 ms (64 samples, 50
// / 300 obstacles) against 0.40 / 0.45 with 32 lanes; arrivals at 500 / 2,000 a second see
// a median of 0.71 / 1.47 ms against 0.61 / 1.33 (p99 1.84 / 3.65 against 1.68 / 3.49).
int pts_serve_group(const Shape &sh) { return pts_group(sh, 1 << 20); }

// Item of the persistent launch: as many warps as leave room for two CTAs per
// SM, but at least four.  A launch with few samples per SM spreads them over two
// CTAs of each SM; one with many takes kSamplesPerWarp rounds per item.
Tiling pts_batch_tiling(const Shape &sh, int G, int samples_per_sm)
{
    const int per = 32 / G;
    int w = pts::kMaxWarps;
    while (w > 4 && pts_smem_bytes(sh, G, w, 1) > kSmemHalf) --w;
    Tiling t = pts_tiling(sh, G, w);
    const int half = std::max(1, (samples_per_sm + 1) / 2), round = per * t.ws;
    const int rounds = std::max(1, std::min(kSamplesPerWarp, half / (3 * round)));
    t.S = std::max(1, std::min(half < round ? half : rounds * round, sh.N));
    t.ws = std::min(t.ws, (t.S + per - 1) / per);
    t.threads = 32 * pts::kMaxWarps;
    return t;
}

namespace {

int sm_count()
{
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    return n_sm;
}

template <int G, int DIMS, int NF, bool WL, int TEAM>
cudaError_t launch_pts_one(const ProjParams<float> &p, const Tiling &t, cudaStream_t st)
{
    static size_t granted = 0;  // per instantiation
    const int grid = (p.N + t.S - 1) / t.S;
    // (teams of four: one CTA per SM by their registers)
    const size_t smem = WL ? pts::pts_smem_with_fix(t.smem, t.smem_fix, TEAM < 4 && grid > sm_count()) : t.smem;
    cudaError_t e = reserve_smem(pts::pts_kernel<G, DIMS, NF, WL, TEAM>, smem, granted);
    if (e != cudaSuccess) return e;
    return launch_pdl(pts::pts_kernel<G, DIMS, NF, WL, TEAM>, dim3(grid), dim3(t.threads), smem, st, p);
}

template <int DIMS, int NF>
cudaError_t launch_pts_wl(const ProjParams<float> &p, const Tiling &t, cudaStream_t st)
{
    if constexpr (DIMS == 2 && NF == 5)
        if (t.R == 16)
            return p.want_lambda ? launch_pts_one<16, DIMS, NF, true, 1>(p, t, st)
                                 : launch_pts_one<16, DIMS, NF, false, 1>(p, t, st);
    if (t.R != 32) return cudaErrorInvalidValue;
    if (t.C == 4)
        return p.want_lambda ? launch_pts_one<32, DIMS, NF, true, 4>(p, t, st)
                             : launch_pts_one<32, DIMS, NF, false, 4>(p, t, st);
    if (t.C == 2)
        return p.want_lambda ? launch_pts_one<32, DIMS, NF, true, 2>(p, t, st)
                             : launch_pts_one<32, DIMS, NF, false, 2>(p, t, st);
    return p.want_lambda ? launch_pts_one<32, DIMS, NF, true, 1>(p, t, st)
                         : launch_pts_one<32, DIMS, NF, false, 1>(p, t, st);
}

template <int G, int DIMS, int NF, bool WL>
cudaError_t launch_pts_batch_one(const ProjParams<float> *params, const int2 *items, int n_items, int *counter,
                                 size_t smem, int grid, cudaStream_t st)
{
    static size_t granted = 0;
    auto kern = pts::pts_batch_kernel<G, DIMS, NF, WL>;
    cudaError_t e = reserve_smem(kern, smem, granted);
    if (e != cudaSuccess) return e;
    constexpr int threads = 32 * pts::kMaxWarps;
    if (grid <= 0) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        grid = std::max(1, per_sm) * sm_count();
    }
    kern<<<std::min(grid, n_items), threads, smem, st>>>(params, items, n_items, counter);
    return cudaGetLastError();
}

template <int DIMS, int NF>
cudaError_t launch_pts_batch_wl(const ProjParams<float> *params, const int2 *items, int n_items, int *counter, int G,
                                int want_lambda, size_t smem, int grid, cudaStream_t st)
{
    auto launch = [&](auto one) { return one(params, items, n_items, counter, smem, grid, st); };
    if constexpr (DIMS == 2 && NF == 5)
        if (G == 16)
            return want_lambda ? launch(launch_pts_batch_one<16, DIMS, NF, true>)
                               : launch(launch_pts_batch_one<16, DIMS, NF, false>);
    if (G != 32) return cudaErrorInvalidValue;
    return want_lambda ? launch(launch_pts_batch_one<32, DIMS, NF, true>)
                       : launch(launch_pts_batch_one<32, DIMS, NF, false>);
}

}  // namespace

size_t pts_batch_smem(size_t smem, size_t smem_fix, int n_items)
{
    return pts::pts_smem_with_fix(smem, smem_fix, n_items > sm_count());
}

// Persistent point-owner launch over (problem, first sample) items, G lanes per sample.
cudaError_t launch_project_pts_batch(const ProjParams<float> *params, const int2 *items, int n_items, int *counter,
                                     int dims, int nf, int G, int want_lambda, size_t smem, int grid, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    if (dims == 2 && nf == 5)
        return launch_pts_batch_wl<2, 5>(params, items, n_items, counter, G, want_lambda, smem, grid, st);
    if (dims == 2 && nf == 7)
        return launch_pts_batch_wl<2, 7>(params, items, n_items, counter, G, want_lambda, smem, grid, st);
    if (dims == 3 && nf == 5)
        return launch_pts_batch_wl<3, 5>(params, items, n_items, counter, G, want_lambda, smem, grid, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_project_pts(const ProjParams<float> &p, const Tiling &t, cudaStream_t st)
{
    if (p.N <= 0) return cudaSuccess;
    if (p.nv != 11 || (t.R != 16 && t.R != 32) || t.ws < 1 || t.ws > pts::kMaxWarps || t.S < 1 ||
        (t.C != 1 && t.C != 2 && t.C != 4) ||
        t.S > (t.C > 1 ? t.ws / t.C : t.ws * (32 / t.R)) || t.threads != 32 * pts::kMaxWarps || p.n_p > t.R * pts::kMaxStrides)
        return cudaErrorInvalidValue;
    if (p.dims == 2 && p.nf == 5) return launch_pts_wl<2, 5>(p, t, st);
    if (p.dims == 2 && p.nf == 7) return launch_pts_wl<2, 7>(p, t, st);
    if (p.dims == 3 && p.nf == 5) return launch_pts_wl<3, 5>(p, t, st);
    return cudaErrorInvalidValue;  // not a compiled variant
}

}  // namespace priest
