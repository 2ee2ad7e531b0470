// project.cu -- tile selection and dispatch of the fused projection kernel
// (project_kernel.cuh): a cost model for the default tiling and the list of
// compiled (points per item, CTA size) variants the autotuner times.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>
#include <vector>

#include "project_kernel.cuh"

namespace priest {

namespace {

struct Variant {
    int dims, R, threads;
};

template <typename Real>
const std::vector<Variant> &variants()
{
    static const std::vector<Variant> f32 = {{2, 4, 512}, {2, 5, 512}, {2, 8, 512}, {2, 5, 1024},
                                             {3, 4, 512}, {3, 5, 256}, {3, 5, 512}};
    static const std::vector<Variant> f64 = {{2, 4, 256}, {3, 4, 256}};
    return sizeof(Real) == 8 ? f64 : f32;
}

constexpr size_t kSmemCap = 227 * 1024;


}  // namespace

template <typename Real>
size_t project_smem_bytes(const Shape &sh, int S, int C)
{
    size_t total = detail::smem_layout(sh.dims, sh.nv, sh.nf, sh.n_p, sh.n_obs, S, C, sh.use_bounds).total;
    if (sizeof(Real) == 4) total = detail::pair_layout(sh.dims, sh.n_obs, sh.n_static, C, total).total;
    return total * sizeof(Real);
}

// Lane groups of one sample's obstacle loop: R points per item, spaced by the
// group count (FP32); blocks of 32 lanes x R points (FP64).
template <typename Real>
int lane_groups(int n_p, int R)
{
    if (sizeof(Real) == 4) return (n_p + R - 1) / R;
    return ((n_p + 32 * R - 1) / (32 * R)) * 32;
}

// Samples per CTA for a given group size: enough that the grid covers the SMs
// once, at most one group per ws warps of the CTA, and at most 15 groups when
// groups use named barriers (ids 1..15).
int samples_per_cta(int n_samples, int n_sm, int threads, int ws)
{
    int S = std::max(1, (n_samples + n_sm - 1) / n_sm);
    S = std::min(S, threads / (32 * ws));
    if (ws > 1) S = std::min(S, 15);
    return std::max(1, S);
}

// PRIEST_PROJECT_KERNEL=chunked in the environment keeps the FP32 projection
// on the chunked kernel (comparisons).
bool pts_allowed()
{
    static const bool allowed = [] {
        const char *v = getenv("PRIEST_PROJECT_KERNEL");
        return !(v && std::string(v) == "chunked");
    }();
    return allowed;
}

// Where the chunked kernel projects a shape that the point-owner kernel covers: in
// 2-D, among many obstacles that mostly move (no grid), most pairs are active, and the
// chunked kernel's sums per time stamp are cheaper than the pairs' own.  How many are
// active follows from the share of the obstacles' box that their discs fill (crowd)
// and, at the same share, from how near the straight line's mean speed is to the
// bound: a sample with no speed to spare cannot leave the obstacles it is in.
// Point-owner / chunked, us a pass (K = 50 to 92; 110, 1,000 and 2,000 samples):
//   mean speed above the bound, share 0.19:  143 / 129, 210 / 187, 247 / 341
//                               share 0.27:  164 / 136, 239 / 195, 271 / 364
//                               share 0.43:  221 / 165, 341 / 280, 386 / 605
//                               share 0.69:  270 / 154, 420 / 272, 472 / 606
//   0.55 of the bound,          share 0.69:  210 / 209, 261 / 425, 286 / 959
//                               share 1.34:  257 / 258, 440 / 652, 664 / 1622
//                               share 2.66:  524 / 357, 803 / 1051, 5645 / 2819
//   seven columns, above,       share 0.32:  177 / 241, 271 / 331, 405 / 719
//                               share 0.55:  273 / 262, 394 / 374, 600 / 872
//   share 0.42, by the mean speed over the bound, 110 and 400 samples: 1.0 189 / 166 and
//   292 / 212, 0.89 177 / 167 and 279 / 213, 0.8 167 / 167 and 264 / 213, 0.67 145 / 165 and
//   219 / 213 (share 0.27: 0.89 147 / 146 and 230 / 187, 0.67 130 / 146 and 175 / 192)
// (circles on a corridor and, at 0.55 of the bound, crossing traffic; chunked times before
// the tiling's last 2 to 10 %).  With at most three samples per SM the chunked kernel spreads
// each over a third of an SM or more, and from a share of 1.2 on it is the faster one whatever
// the speed: 0.55 of the bound, half of the acceleration bound, K = 60, 110 and 400 samples:
//   share 1.3, discs that stay in a 5 x 3 m box:    16 184 / 157 and 254 / 194, 33 261 / 169 and
//                                       337 / 222, 130 462 / 243 and 661 / 346
//              that cross it:           16 235 / 157 and 356 / 194, 33 340 / 167 and 454 / 218
//              that leave it or a 14 x 20 m box: 24 to 120 discs, 0.98 to 2.4 times the chunked time
//   share 0.7:  those that stay or cross 0.95 to 3.2 times, those that leave 0.74 to 1.6 times
//   seven columns, share 1.1: 329 / 290 and 436 / 340, 0.69: 277 / 284 and 331 / 336
// With more samples, what is faster at shares of 1.2 to 2 depends on how long the discs stay
// on the way, which the share of their first box does not tell (1,000 samples, share 1.3: 0.73 to
// 2.7 times, 1.9: 1.04 and more).  3-D: the point-owner kernel is faster at every share (33 to
// 200 spheres: 127 to 386 against 186 to 1,021).  The route depends on the obstacles' values, so
// it takes the model's tiling: trial launches would stall a replanner in the middle of its run,
// or break its capture.
bool pts_crowded(const Shape &sh, int samples_per_sm)
{
    if (!pts_allowed() || !pts_supported(sh) || sh.dims != 2 || sh.n_static >= kGridMinStatic || sh.n_obs < 12) return false;
    double d2 = 0.0;
    for (int ax = 0; ax < sh.dims; ++ax) d2 += (sh.bf[ax][0] - sh.b0[ax][0]) * (sh.bf[ax][0] - sh.b0[ax][0]);
    const bool hurried = std::sqrt(d2) > 0.85 * sh.vmax * sh.horizon;
    if (!hurried) return sh.crowd >= (samples_per_sm > 3 ? 2.0 : 1.2);
    return sh.crowd >= (sh.nf == 5 && samples_per_sm <= 8 ? 0.25 : 1.0);
}

// Default tiling: the point-owner kernel for the shapes it covers; otherwise the
// largest compiled variant, the largest warp group that
// fits the CTA, and the obstacle chunk count that gives each group's threads
// about one item each, within the shared-memory cap.
template <typename Real>
Tiling choose_tiling(const Shape &sh, int n_samples, int n_sm)
{
    const int m = std::max(1, (n_samples + n_sm - 1) / n_sm);  // an SM's share of the samples
    const bool crowded = sizeof(Real) == 4 && pts_crowded(sh, m);
    Tiling own;
    own.smem = 0;
    if (sizeof(Real) == 4 && pts_supported(sh) && pts_allowed()) {
        // the share in as few CTAs of equal size as hold it; few samples per SM: a team of warps
        // for each (pts_team_size)
        if (const int C = pts_team_size(sh, m)) {
            const int fit = 8 / C, n = (m + fit - 1) / fit;
            own = pts_team_tiling(sh, (m + n - 1) / n, C);
            if (size_t(n) * (own.smem + 1024) > size_t(228) * 1024) own.smem = 0;
        }
        if (own.smem == 0) {
            const int G = pts_group(sh, m), w = (m * G + 31) / 32, ctas = (w + 7) / 8;
            own = pts_tiling(sh, G, (w + ctas - 1) / ctas);
        }
        if (own.smem > 0 && !crowded) return own;
    }
    Tiling t;
    t.R = sizeof(Real) == 8 ? 4 : 5;
    t.threads = sizeof(Real) == 8 ? 256 : 512;
    const int S0 = m;
    t.ws = 1;
    while (t.ws < 8 && S0 * 32 * (2 * t.ws) <= t.threads && S0 <= 15) t.ws *= 2;
    int S = samples_per_cta(n_samples, n_sm, t.threads, t.ws);
    while (S > 1 && project_smem_bytes<Real>(sh, S, 1) > kSmemCap) S = std::max(1, S * 3 / 4);
    auto chunks = [&](int R) { return std::max(1, (32 * t.ws) / lane_groups<Real>(sh.n_p, R)); };
    // crowded: four points an item, unless five fill the lanes better (33 circles, K = 50: 110 samples of
    // 80 stamps 141 against 174 us with five, 1,200 of 150 stamps 315 against 288)
    if (crowded && 5 * lane_groups<Real>(sh.n_p, 5) * chunks(5) <= 6 * lane_groups<Real>(sh.n_p, 4) * chunks(4)) t.R = 4;
    int C = std::min(chunks(t.R), std::max(1, std::min(16, sh.n_obs)));
    while (C > 1 && project_smem_bytes<Real>(sh, S, C) > kSmemCap) --C;
    if (crowded) {
        // no more chunks than their obstacle pairs need, each costs its partial sums (20 circles,
        // 300 samples 163 -> 152 us)
        auto pairs = [](int n, int c) { return (n + 2 * c - 1) / (2 * c); };
        const int n_mov = sh.n_obs - sh.n_static;
        while (C > 1 && pairs(sh.n_static, C - 1) == pairs(sh.n_static, C) && pairs(n_mov, C - 1) == pairs(n_mov, C)) --C;
    }
    t.S = S;
    t.C = C;
    t.smem = project_smem_bytes<Real>(sh, S, C);
    // (the chunked kernel stages whole tables: it holds fewer obstacles and time stamps)
    return t.smem > kSmemCap && own.smem > 0 ? own : t;
}

// Candidates for the autotuner: every compiled variant for the dimension,
// every warp-group size that fits, and the chunk counts that keep each
// group's pair loop within two rounds of items, within the shared-memory cap.
template <typename Real>
std::vector<Tiling> tiling_candidates(const Shape &sh, int n_samples, int n_sm)
{
    std::vector<Tiling> out;
    for (const Variant &v : variants<Real>()) {
        if (v.dims != sh.dims) continue;
        for (int ws = 1; ws <= 8 && 32 * ws <= v.threads; ws *= 2) {
            int S = samples_per_cta(n_samples, n_sm, v.threads, ws);
            while (S > 1 && project_smem_bytes<Real>(sh, S, 1) > kSmemCap) S = std::max(1, S * 3 / 4);
            const int ng = lane_groups<Real>(sh.n_p, v.R);
            const int cmax = std::max(1, std::min(16, sh.n_obs));
            for (int C = 1; C <= cmax; ++C) {
                const size_t smem = project_smem_bytes<Real>(sh, S, C);
                if (smem > kSmemCap) break;
                const int rounds = (ng * C + 32 * ws - 1) / (32 * ws);
                if (rounds > 2) break;
                Tiling t;
                t.S = S;
                t.C = C;
                t.R = v.R;
                t.threads = v.threads;
                t.ws = ws;
                t.smem = smem;
                out.push_back(t);
            }
        }
    }
    return out;
}

template <typename Real>
Tiling batch_tiling(const Shape &sh, bool chunked)
{
    if (sizeof(Real) == 4 && pts_supported(sh) && pts_allowed() && !chunked) {
        const Tiling p = pts_batch_tiling(sh, pts_group(sh, 1 << 20), 1 << 20);
        if (p.smem > 0) return p;
    }
    Tiling t;
    t.R = sizeof(Real) == 8 ? 4 : 5;
    t.threads = sizeof(Real) == 8 ? 256 : 512;
    t.ws = (sh.dims == 2 && sizeof(Real) == 4) ? 2 : 1;
    t.S = std::max(1, std::min(sh.N, t.threads / (32 * t.ws)));
    if (t.ws > 1) t.S = std::min(t.S, 15);
    const int ng = lane_groups<Real>(sh.n_p, t.R);
    t.C = std::max(1, std::min(std::min(16, std::max(1, sh.n_obs)), (32 * t.ws) / ng));
    while (t.S > 1 && project_smem_bytes<Real>(sh, t.S, t.C) > kSmemCap) t.S = std::max(1, t.S / 2);
    t.smem = project_smem_bytes<Real>(sh, t.S, t.C);
    if (t.smem > kSmemCap) t.smem = 0;
    return t;
}

// Candidates of the batched launch's autotuner: warp-group sizes and chunk
// counts for the batched variant's CTA, within the shared-memory cap.
template <typename Real>
std::vector<Tiling> batch_candidates(const Shape &sh)
{
    std::vector<Tiling> out;
    const int threads = sizeof(Real) == 8 ? 256 : 512;
    for (int ws = 1; ws <= 4; ws *= 2) {
        Tiling t;
        t.R = sizeof(Real) == 8 ? 4 : 5;
        t.threads = threads;
        t.ws = ws;
        t.S = std::max(1, std::min(sh.N, threads / (32 * ws)));
        if (ws > 1) t.S = std::min(t.S, 15);
        for (int C = 1; C <= std::min(4, std::max(1, sh.n_obs)); C *= 2) {
            t.C = C;
            int S = t.S;
            while (S > 1 && project_smem_bytes<Real>(sh, S, C) > kSmemCap) S = std::max(1, S / 2);
            Tiling u = t;
            u.S = S;
            u.smem = project_smem_bytes<Real>(sh, S, C);
            if (u.smem <= kSmemCap) out.push_back(u);
        }
    }
    return out;
}

template <typename Real>
cudaError_t launch_project(const ProjParams<Real> &p, const Tiling &t, cudaStream_t st)
{
    if (p.N <= 0) return cudaSuccess;
    if constexpr (sizeof(Real) == 8) {
        if (p.dims == 2) return launch_variant<Real, 2, 4, 256>(p, t, st);
        return launch_variant<Real, 3, 4, 256>(p, t, st);
    } else {
        if (t.kind == 1) return launch_project_pts(p, t, st);
        if (t.S * 32 * t.ws > t.threads) return cudaErrorInvalidValue;
        if (p.dims == 2) {
            if (t.R == 4 && t.threads == 512) return launch_variant<Real, 2, 4, 512>(p, t, st);
            if (t.R == 5 && t.threads == 512) return launch_variant<Real, 2, 5, 512>(p, t, st);
            if (t.R == 8 && t.threads == 512) return launch_variant<Real, 2, 8, 512>(p, t, st);
            if (t.R == 5 && t.threads == 1024) return launch_variant<Real, 2, 5, 1024>(p, t, st);
            return cudaErrorInvalidValue;  // not a compiled variant
        }
        if (t.R == 4 && t.threads == 512) return launch_variant<Real, 3, 4, 512>(p, t, st);
        if (t.R == 5 && t.threads == 256) return launch_variant<Real, 3, 5, 256>(p, t, st);
        if (t.R == 5 && t.threads == 512) return launch_variant<Real, 3, 5, 512>(p, t, st);
        return cudaErrorInvalidValue;
    }
}

// Batched launches use one variant per precision and dimension: 2-D
// (R = 5, 512 threads), 3-D (R = 5, 512 threads), FP64 (R = 4, 256 threads).
template <typename Real>
cudaError_t launch_project_batch(const ProjParams<Real> *params_dev, const int2 *items_dev, int n_items,
                                 int *counter_dev, int dims, [[maybe_unused]] int R, int nf, int nv, int want_lambda,
                                 size_t smem, int grid, cudaStream_t st, int kind)
{
    if (n_items <= 0) return cudaSuccess;
    if constexpr (sizeof(Real) == 4) {
        if (kind == 1)
            return launch_project_pts_batch(params_dev, items_dev, n_items, counter_dev, dims, nf, R, want_lambda,
                                            smem, grid, st);
    }
    if constexpr (sizeof(Real) == 8) {
        if (dims == 2)
            return launch_variant_batch<Real, 2, 4, 256>(params_dev, items_dev, n_items, counter_dev, nf, nv,
                                                         want_lambda, smem, grid, st);
        return launch_variant_batch<Real, 3, 4, 256>(params_dev, items_dev, n_items, counter_dev, nf, nv,
                                                     want_lambda, smem, grid, st);
    } else {
        if (dims == 2)
            return launch_variant_batch<Real, 2, 5, 512>(params_dev, items_dev, n_items, counter_dev, nf, nv,
                                                         want_lambda, smem, grid, st);
        return launch_variant_batch<Real, 3, 5, 512>(params_dev, items_dev, n_items, counter_dev, nf, nv,
                                                     want_lambda, smem, grid, st);
    }
}

template cudaError_t launch_project_batch<float>(const ProjParams<float> *, const int2 *, int, int *, int, int, int,
                                                 int, int, size_t, int, cudaStream_t, int);
template cudaError_t launch_project_batch<double>(const ProjParams<double> *, const int2 *, int, int *, int, int,
                                                  int, int, int, size_t, int, cudaStream_t, int);
template size_t project_smem_bytes<float>(const Shape &, int, int);
template size_t project_smem_bytes<double>(const Shape &, int, int);
template Tiling choose_tiling<float>(const Shape &, int, int);
template Tiling choose_tiling<double>(const Shape &, int, int);
template std::vector<Tiling> tiling_candidates<float>(const Shape &, int, int);
template std::vector<Tiling> tiling_candidates<double>(const Shape &, int, int);
template Tiling batch_tiling<float>(const Shape &, bool);
template Tiling batch_tiling<double>(const Shape &, bool);
template std::vector<Tiling> batch_candidates<float>(const Shape &);
template std::vector<Tiling> batch_candidates<double>(const Shape &);
template cudaError_t launch_project<float>(const ProjParams<float> &, const Tiling &, cudaStream_t);
template cudaError_t launch_project<double>(const ProjParams<double> &, const Tiling &, cudaStream_t);

}  // namespace priest
