// pts_layout.cuh -- sizes and shared-memory layout of the FP32 point-owner
// projection (project_pts.cuh), for the host and the kernel.
#pragma once

#include "priest_internal.cuh"

namespace priest {
namespace pts {

constexpr int kMaxWarps = 8;    // warps of one CTA
constexpr int kMaxStrides = 16; // strides of G time stamps
constexpr int kPairs = 256;     // obstacle pairs a sample may list (a multiple of 32)
constexpr int kShortLived = 6;  // iterations of a list that lasted too short
constexpr int kRetry = 16;      // iterations without a list before the next try
constexpr int kMaxTeam = 4;     // most warps of one sample's team
// A team's exchange floats: two buffers of {sums of g [3][32], the test's answer}, {r^2, c_1}
// [kMaxTeam][2] doubles, the fixed columns' sums [kMaxTeam][32]
constexpr int kXchFlag = 3 * 32, kXchBuf = kXchFlag + 8, kXchEnd = 2 * kXchBuf, kXchFix = kXchEnd + 4 * kMaxTeam,
              kXch = kXchFix + kMaxTeam * 32;

// Shared-memory layout (float units, every block 32-byte aligned); np is n_p
// rounded up to 2 G and the row blocks are arrays of 16 bytes over the stamps, so
// the lanes of a group read neighbouring banks.
//   header [24]               ints: the offsets and sizes below (Hdr); floats: the origin, the extent, 1 / T
//   rows  [chunks][np][4]     per time stamp, positions: nf free columns of P, then the
//                             fixed-coefficient part of each axis
//   vrows [2][pchunks][np / 2][4]  the same of Pd and Pdd, stamps 2 u and 2 u + 1
//                             interleaved: {v0(2u), v0(2u + 1), v1(2u), v1(2u + 1)}
//   tv    [np]                time stamps
//   node  [32 / G][nfn][32][4]  node rows {P, Pdd} of two columns a time (nfn = (nf + 1) / 2)
//   obs   [n_obs][4]          2-D {1/a, -o_x/a, -o_y/a, a}, 3-D {1/a, -o_x/a, -o_y/a, -o_z/b}
//   obq   [n_obs][4]          3-D {kUnit/b, a, b, max(1/a, 1/b)}
//   mov   [n_moving][4]       {-v_x/a, -v_y/a[, -v_z/b]}
//   grid  [gl.smem]           the static-obstacle grid of the tables
//   per warp, for each of its 32 / G samples:
//     c [nf][4 | 8]           coefficients, each twice: {x, x, y, y[, z, z, -, -]}
//     stage [4 G][4]          active pairs on their way to a lane: {r (dims), t}
//     list [kPairs][4]        kUnit {1/a, -o_x(t)/a, -o_y(t)/a} and 2-D a, 3-D -kUnit o_z(t)/b
//     tj [kPairs]             (ints) time stamp | obstacle << 16
//     moved [nf][dims][2]     coefficients since the rebuild of the {pair, rate} lists
//   xch   [teams][kXch]       what a team's warps tell one another
//   fix   [3][fchunks][np][4] fixed columns (multipliers on request, when it fits)
constexpr int kRows = 24;  // offset of the rows
constexpr int kOrigin = 16, kExtent = 19, kRate = 20;  // of the header's floats (kRate: 1 / horizon)
__host__ __device__ constexpr int coef_floats(int dims, int nf) { return nf * (dims == 2 ? 4 : 8); }
__host__ __device__ constexpr int moved_at(int G, int dims, int nf)
{
    return coef_floats(dims, nf) + 16 * G + 5 * kPairs + (nf & 1) * 4;
}
__host__ __device__ constexpr int sample_floats(int G, int dims, int nf)
{
    return (moved_at(G, dims, nf) + 2 * nf * dims + 7) & ~7;
}
struct PtsLayout {
    int np, nch, pch, nfch;
    size_t rows, vrows, node, tv, obs, obq, mov, grid, gsz, warp0, wsz, xch, fix, total, total_fix;
};

__host__ __device__ inline PtsLayout pts_layout(int G, int dims, int nf, int nv, int n_p, int n_obs, int n_static,
                                                int warps, int teams)
{
    PtsLayout L;
    L.np = (n_p + 2 * G - 1) & ~(2 * G - 1);
    L.nch = (nf + dims + 3) / 4;
    L.pch = (nf + dims + 1) / 2;
    L.nfch = (nv - nf + 3) / 4;
    size_t o = 0;
    auto take = [&o](size_t n) {
        const size_t at = o;
        o = align8(o + n);
        return at;
    };
    take(kRows);
    L.rows = take(size_t(L.nch) * L.np * 4);
    L.vrows = take(size_t(2) * L.pch * L.np * 2);
    L.node = take(size_t(32 / G) * ((nf + 1) / 2) * 128);
    L.tv = take(size_t(L.np));
    L.obs = take(size_t(n_obs) * 4);
    L.obq = take(dims == 3 ? size_t(n_obs) * 4 : 0);
    L.mov = take(size_t(n_obs - n_static) * 4);
    L.gsz = n_static >= kGridMinStatic ? grid_layout(n_static).smem : 0;
    L.grid = take(L.gsz);
    L.warp0 = o;
    L.wsz = size_t(32 / G) * sample_floats(G, dims, nf);
    o += L.wsz * warps;
    L.xch = o;
    o += size_t(kXch) * teams;
    L.total = o;
    L.fix = o;
    L.total_fix = o + size_t(3) * L.nfch * L.np * 4;
    return L;
}

// Shared memory of a CTA alone on its SM, and of each of two that share one (228 KB
// less 1 KB and the static part of each).
constexpr size_t kSmemCap = 227 * 1024;
constexpr size_t kSmemHalf = 112 * 1024;

// Dynamic shared memory of a launch that returns multipliers: `with_fix` bytes, which
// hold the fixed columns' rows of every problem, or `smem` without them.  The rows
// are read by every active row of every iteration (from global memory when they are
// not here), and never cost an SM its second CTA (`two`: the launch has CTAs for it).
inline size_t pts_smem_with_fix(size_t smem, size_t with_fix, bool two)
{
    if (with_fix > kSmemCap || (two && smem <= kSmemHalf && with_fix > kSmemHalf)) return smem;
    return with_fix;
}

}  // namespace pts
}  // namespace priest
