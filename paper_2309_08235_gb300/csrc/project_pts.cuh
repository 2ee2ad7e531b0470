// project_pts.cuh -- FP32 fused projection with point-owning lanes (Sec. III-A;
// Appendix eqs. lagrange, comp_alpha .. comp_zeta, lag, affine_trans /
// matrix_vec / comp_zeta), the hot path of the FP32 solver.
//
// G = 32 or 16 lanes project one sample through all K iterations; lane l of the
// group owns the time stamps t = l, l + G, ... .  A residual row is zero wherever
// its constraint is inactive, and few are active at a time (on the measured
// scenes a handful of the n_p n_o obstacle pairs of a sample, and the velocity /
// acceleration rows of none to all of its time stamps), so an iteration
// evaluates only the rows that can be active:
//   * obstacle pairs: the pairs (t, j) within a_j + delta at the last rebuild,
//     sorted by (t, j), with the obstacle's scaled offset terms at time t, spread
//     evenly over the lanes (the owners of t meet uneven numbers of obstacles);
//   * velocity rows: all of them, or none while the bound cannot be reached;
//   * acceleration and workspace rows: one bit per block of time stamps in which
//     some norm (coordinate) was within a margin of its bound.
// Position and acceleration are polynomials of degree 10 and 8 in time, and a
// polynomial of degree n is bounded on its interval by 1 / cos(n pi / 2m) times
// its maximum over m Chebyshev nodes (Ehlich and Zeller 1964).  The lanes
// evaluate the displacement of 32 nodes since the last rebuild, from the
// coefficients' differences (which keep their digits wherever the frame's origin
// lies); while the bound stays below the margins, every pair and row left out is
// inactive.  (The start's velocity is fixed, so the change of velocity is bounded by
// that of the acceleration times the time.)  The margins also pay for the rounding of
// the rows, which grows with the coefficients (row_rounding): far from the origin the
// lists shrink what may move before a rebuild, and where rounding alone eats the
// margin every pair is screened.  So nothing is approximated: the sums are bitwise
// those of evaluating every pair.  The m-th active pair in (t, j) order is added
// by lane m mod G, whatever was listed beside it, and velocity, acceleration and
// workspace rows by the owner of t, in a fixed order.
//
// An iteration is then: the free coefficients from shared memory; the node
// test; the listed pairs, each row . c + base and its residual, the active ones
// through shared memory to the lane that adds row^T residual to its share of g;
// the other listed rows; a transposing butterfly that leaves each of the
// dims * nf sums of g in a "state lane"; the multiplier and shared-inverse
// steps in those lanes (W u by shuffles); the new coefficients back to shared
// memory.  The chain of one iteration is what bounds it (a warp waits on its own
// results: 1,600 cycles an iteration with one sample per scheduler, and at 16
// warps per SM 51 % of the issue slots), so the code is straight-line where it
// can be: loops run to warp-uniform trip counts over branch-free bodies (lists
// are padded with a pair that is never active), the first trip runs beside the
// node test, and velocity / acceleration rows go two time stamps to an f32x2 FMA.
// No CTA barrier: a CTA's warps share only the problem's tables.  With few samples
// per SM a team of warps shares the chain (project_samples).
//
// Before, threads owned two time stamps of a sample, evaluated all their rows in
// every iteration and met at a CTA barrier; per pass, before -> now: 2-D clutter
// (N = 1000, n_p = 100, 100 obstacles, K = 100) 195 -> 123 us, 64 uneven 2-D
// problems (K = 60) 4,534 -> 1,585 us, 3-D ellipsoids (N = 2000, n_p = 150, 200
// obstacles, K = 100) 826 -> 492 us, a replan of 110 samples (K = 50) 123 -> 101.
// Slower than before: samples that keep velocity rows or many pairs active (an iteration
// of 1,700 cycles, plus 300 a block of rows, 320 a trip of 32 pairs, 5,000 and more a
// rebuild): 27 circles on a diagonal, 574 samples, K = 75, 220 us against 179; 9 moving
// circles, 36 samples, K = 92, 220 against 200; 16 circles, 1,520 samples, 170 against 148.
//
// The multipliers of the fixed columns (returned only on request) follow from
// the linearity of eq. lag: lambda_B^K = lambda_B^0 - rho sum_k P_B^T r^k, so
// each lane sums its P_B^T r over the iterations and the group reduces once.
#pragma once

#include <cfloat>
#include <type_traits>

#include "project_kernel.cuh"
#include "pts_layout.cuh"

namespace priest {
namespace pts {

using detail::ffma2;
using detail::fmul2;

constexpr unsigned kAll = 0xffffffffu;
// 1 / cos(n pi / 64), rounded up: bound of a degree-n polynomial by 32 nodes
constexpr float kNodeBoundPos = 1.1340f;  // n = 10
constexpr float kNodeBoundAcc = 1.0825f;  // n = 8
// Velocity / acceleration margin where the bound is close, as a share of the
// acceleration bound.
constexpr float kAccMargin = 0.15f;

// The butterfly's value of a lane of the group: V values over G lanes, halved
// at each exchange (the lower half of the lanes keeps the first (n + 1) / 2
// values); -1 where the lane ends up with padding.
__host__ __device__ constexpr int val_of(int G, int V, int lane)
{
    int v = 0, n = V, real = V;
    for (int off = G / 2; off >= 1; off >>= 1) {
        if (n == 1) break;
        const int m = (n + 1) / 2;
        if (lane & off) {
            v += m;
            real -= m;
        } else {
            real = real < m ? real : m;
        }
        n = m;
    }
    return (real >= 1 && n == 1) ? v : -1;
}

// The first lane that ends up with value v.
__host__ __device__ constexpr int lane_of(int G, int V, int v)
{
    int l = G - 1;
    for (int i = G - 1; i >= 0; --i) l = val_of(G, V, i) == v ? i : l;
    return l;
}
template <int G, int V, int I>
struct LaneOf {
    static constexpr int value = lane_of(G, V, I);
};

// Sums h[] over the group; the lane's value val_of(G, V, lane) is returned.  A
// halving exchange costs half the shuffles of the one before (12 for ten
// values over 32 lanes, 50 for a plain butterfly of each).
template <int N, int OFF>
__device__ __forceinline__ float reduce_step(float *h, int lane)
{
    if constexpr (N == 1) {
        h[0] += __shfl_xor_sync(kAll, h[0], OFF);
    } else {
        constexpr int M = (N + 1) / 2;
        const bool hi = (lane & OFF) != 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const float up = i + M < N ? h[i + M] : 0.f;
            const float send = hi ? h[i] : up, keep = hi ? up : h[i];
            h[i] = keep + __shfl_xor_sync(kAll, send, OFF);
        }
    }
    if constexpr (OFF > 1)
        return reduce_step<(N + 1) / 2, OFF / 2>(h, lane);
    else
        return h[0];
}

// The CTA's dynamic shared memory in floats; every access below is an offset
// into it, so addresses stay 32-bit and the tables' offsets are read where used.
__device__ __forceinline__ float *smem()
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<float *>(smem_raw);
}
enum Hdr {  // kGrid, kFix: 0 = none
    kVrows, kNode, kTv, kObs, kObq, kMov, kGrid, kFix, kNp, kStamps, kStatic, kObstacles, kNext, kXchAt
};
__device__ __forceinline__ int hdr(int i) { return reinterpret_cast<const int *>(smem())[i]; }
__device__ __forceinline__ float4 ld4s(int off) { return *reinterpret_cast<const float4 *>(smem() + off); }

// Free columns of the position row at time stamp t and its fixed part.
template <int DIMS, int NF>
__device__ __forceinline__ void load_row(int np, int t, float (&row)[NF], float (&x)[DIMS])
{
    constexpr int NCH = (NF + DIMS + 3) / 4;
    float v[4 * NCH];
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
        const float4 w = ld4s(kRows + (i * np + t) * 4);
        v[4 * i] = w.x;
        v[4 * i + 1] = w.y;
        v[4 * i + 2] = w.z;
        v[4 * i + 3] = w.w;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) row[f] = v[f];
#pragma unroll
    for (int ax = 0; ax < DIMS; ++ax) x[ax] = v[NF + ax];
}

// x = base + row . c
template <int DIMS, int NF>
__device__ __forceinline__ void eval_row(int np, int t, const float (&c)[NF][DIMS], float (&row)[NF], float (&x)[DIMS])
{
    load_row<DIMS, NF>(np, t, row, x);
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) x[ax] = fmaf(row[f], c[f][ax], x[ax]);
}

// Velocity (q = 0) or acceleration (q = 1) at stamps 2 u and 2 u + 1, one f32x2
// FMA per term.
template <int DIMS, int NF>
__device__ __forceinline__ void eval_pair(int vrows, int np, int q, int u, const float2 (&c)[NF][DIMS], float2 (&row)[NF],
                                          float2 (&x)[DIMS])
{
    constexpr int PCH = (NF + DIMS + 1) / 2;
    float2 v[2 * PCH];
#pragma unroll
    for (int i = 0; i < PCH; ++i) {
        const float4 w = ld4s(vrows + ((q * PCH + i) * (np / 2) + u) * 4);
        v[2 * i] = make_float2(w.x, w.y);
        v[2 * i + 1] = make_float2(w.z, w.w);
    }
#pragma unroll
    for (int ax = 0; ax < DIMS; ++ax) x[ax] = v[NF + ax];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        row[f] = v[f];
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) x[ax] = ffma2(row[f], c[f][ax], x[ax]);
    }
}

template <int DIMS>
__device__ __forceinline__ float2 norm2(const float2 (&x)[DIMS])
{
    const float2 s = ffma2(x[1], x[1], fmul2(x[0], x[0]));
    return DIMS == 3 ? ffma2(x[DIMS - 1], x[DIMS - 1], s) : s;
}

// The pairs' scaled offsets are carried in units of 2^-60, so that the square of any
// normal offset is normal (next to an obstacle's centre it would not be) and the
// kernel's roots need no care for denormals; powers of two change no other bit.  (With
// that care, rsqrtf, 64 problems took 1,648 us a pass instead of 1,567.)
constexpr float kUnit = 0x1p60f, kPerUnit = 0x1p-60f;
constexpr float kTouch = 0x1p120f;  // the square at the obstacle's boundary: active below it

// 1 / sqrt(q), q normal or infinite: rsqrtf without its care for denormals, the same
// value otherwise.
__device__ __forceinline__ float rsqrt_normal(float q)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(q));
    return y;
}

// Scaled offset terms of obstacle j at time t: {1/a, -o_x/a, -o_y/a, a (2-D) or
// -o_z/b}; moving obstacles (j >= ns) follow the static ones.
template <int DIMS>
__device__ __forceinline__ float4 pair_terms(int j, float t, int ns)
{
    float4 o = ld4s(hdr(kObs) + 4 * j);
    if (j >= ns) {
        const float4 v = ld4s(hdr(kMov) + 4 * (j - ns));
        o.y = fmaf(t, v.x, o.y);
        o.z = fmaf(t, v.y, o.z);
        if (DIMS == 3) o.w = fmaf(t, v.z, o.w);
    }
    return o;
}

// Scaled offset of the position x from an obstacle and its square.
template <int DIMS>
__device__ __forceinline__ float scaled_offset(const float (&x)[DIMS], const float4 &o, float ib, float (&d)[DIMS])
{
    d[0] = fmaf(x[0], o.x, o.y);
    d[1] = fmaf(x[1], o.x, o.z);
    if constexpr (DIMS == 2) {
        return fmaf(d[0], d[0], d[1] * d[1]);
    } else {
        d[DIMS - 1] = fmaf(x[DIMS - 1], ib, o.w);
        return fmaf(d[0], d[0], fmaf(d[1], d[1], d[DIMS - 1] * d[DIMS - 1]));
    }
}

// Whether a point within delta of the position x may touch the obstacle with
// the offset terms o (3-D: b its {1/b, a, b, max(1/a, 1/b)}).
template <int DIMS>
__device__ __forceinline__ bool near_pair(const float (&x)[DIMS], const float4 &o, const float4 &b, float delta)
{
    float d[DIMS];
    const float q = scaled_offset<DIMS>(x, o, b.x, d), lim = fmaf(delta, DIMS == 3 ? b.w : o.x, 1.f);
    return q < lim * lim;
}

// What the screening of a sample's positions keeps in registers.
template <int DIMS>
struct Screen {
    int ns, no, obs, obq, nx, ny, start, ent;  // nx = 0: no grid
    float x0, y0, ih, delta;

    __device__ __forceinline__ explicit Screen(float margin)
    {
        ns = hdr(kStatic);
        no = hdr(kObstacles);
        obs = hdr(kObs);
        obq = hdr(kObq);
        delta = margin;
        const int go = hdr(kGrid);
        const float *g = smem() + go;
        nx = go ? __float_as_int(g[4]) : 0;
        ny = go ? __float_as_int(g[5]) : 0;
        x0 = g[0];
        y0 = g[1];
        ih = g[2];
        start = 2 * (go + 8);
        ent = 2 * (go + int(grid_layout(ns).ent));
    }
    __device__ __forceinline__ static int u16(int i) { return reinterpret_cast<const unsigned short *>(smem())[i]; }
    __device__ __forceinline__ float4 semi(int j) const
    {
        if constexpr (DIMS == 2) return make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 b = ld4s(obq + 4 * j);
        return make_float4(b.x * kPerUnit, b.y, b.z, b.w);
    }

    // Calls hit(j, terms), in increasing j, for every static obstacle that a point
    // within delta of the position x may touch: those of the grid's cell when
    // there is a grid (four at a time, their loads in flight together), all of
    // them otherwise.
    template <typename Hit>
    __device__ __forceinline__ void fixed(const float (&x)[DIMS], bool valid, Hit hit) const
    {
        int e0 = 0, e1 = valid ? ns : 0;
        if (nx > 0) {
            const float fx = (x[0] - x0) * ih, fy = (x[1] - y0) * ih;
            const bool in = valid && fx >= 0.f && fx < float(nx) && fy >= 0.f && fy < float(ny);
            const int cell = in ? min(int(fy), ny - 1) * nx + min(int(fx), nx - 1) : 0;
            e0 = u16(start + cell);
            e1 = in ? u16(start + cell + 1) : e0;
        }
#pragma unroll 1
        for (int e = e0; e < e1; e += 4) {
            int j[4];
            float4 o[4];
            bool near[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int ei = min(e + i, e1 - 1);
                j[i] = nx > 0 ? u16(ent + ei) : ei;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                o[i] = ld4s(obs + 4 * j[i]);
                near[i] = e + i < e1 && near_pair<DIMS>(x, o[i], semi(j[i]), delta);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (near[i]) hit(j[i], o[i]);
        }
    }

    // The same for the moving obstacles at time t: those that can come near the
    // box of the group's positions in its time span [t0, t1] (one lane tests one
    // obstacle).  All lanes of the warp call it together.
    template <int G, typename Hit>
    __device__ __forceinline__ void moving(const float (&x)[DIMS], bool valid, float t, float t0, float t1, Hit hit) const
    {
        if (no == ns) return;
        float lo[DIMS], hi[DIMS];
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) {
            lo[ax] = valid ? x[ax] : FLT_MAX;
            hi[ax] = valid ? x[ax] : -FLT_MAX;
        }
#pragma unroll
        for (int off = G / 2; off >= 1; off >>= 1)
#pragma unroll
            for (int ax = 0; ax < DIMS; ++ax) {
                lo[ax] = fminf(lo[ax], __shfl_xor_sync(kAll, lo[ax], off));
                hi[ax] = fmaxf(hi[ax], __shfl_xor_sync(kAll, hi[ax], off));
            }
        const int gl = threadIdx.x & (G - 1);
#pragma unroll 1
        for (int j0 = ns; j0 < no; j0 += G) {
            bool may = false;
            const int j = j0 + gl;
            if (j < no) {
                // the scaled offset's range over the box and the span misses [-lim, lim] on some
                // axis (lim with room for rounding; a NaN position is near nothing)
                const float4 o0 = pair_terms<DIMS>(j, t0, ns), o1 = pair_terms<DIMS>(j, t1, ns), b = semi(j);
                const float lim = 1.01f * fmaf(delta, DIMS == 3 ? b.w : o0.x, 1.f);
                may = true;
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) {
                    const float i = ax == 2 ? b.x : o0.x;
                    const float a0 = ax == 0 ? o0.y : ax == 1 ? o0.z : o0.w, a1 = ax == 0 ? o1.y : ax == 1 ? o1.z : o1.w;
                    may = may && fmaf(hi[ax], i, fmaxf(a0, a1)) > -lim && fmaf(lo[ax], i, fminf(a0, a1)) < lim;
                }
            }
            unsigned m = __ballot_sync(kAll, may);
            if (G == 16) m = (m | (m >> 16)) & 0xffffu;  // either sample's
#pragma unroll 1
            while (m) {  // four at a time, their loads in flight together
                int jm[4];
                float4 o[4];
                bool near[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    near[i] = valid && m != 0u;
                    jm[i] = m ? j0 + __ffs(m) - 1 : j0;
                    m &= m - 1u;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    o[i] = pair_terms<DIMS>(jm[i], t, ns);
                    near[i] = near_pair<DIMS>(x, o[i], semi(jm[i]), delta) && near[i];
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (near[i]) hit(jm[i], o[i]);
            }
        }
    }
};

// The terms o of a pair in the lists' unit.
template <int DIMS>
__device__ __forceinline__ float4 listed_terms(const float4 &o)
{
    return make_float4(kUnit * o.x, kUnit * o.y, kUnit * o.z, DIMS == 3 ? kUnit * o.w : o.w);
}

// Residual of an active pair (d its scaled offset in the lists' unit, q = |d|^2 < kTouch):
// r = Delta (1 - 1 / |scaled offset|); at the centre the target is o + (a, 0) (2-D) /
// o + (0, 0, b) (3-D).
template <int DIMS>
__device__ __forceinline__ void pair_residual(const float (&d)[DIMS], float q, float a, float b, float (&r)[DIMS])
{
    const float w = kPerUnit - rsqrt_normal(fmaxf(q, FLT_MIN));
#pragma unroll
    for (int ax = 0; ax < DIMS; ++ax) r[ax] = ((DIMS == 3 && ax == 2 ? b : a) * w) * d[ax];
    constexpr int up = DIMS == 3 ? DIMS - 1 : 0;
    r[up] = q > 0.f ? r[up] : -(DIMS == 3 ? b : a);
}

// Its squared norm (final pass; out of line, away from the registers of the iteration).
template <int DIMS>
__device__ __noinline__ float pair_square(const float (&d)[DIMS], float q, float a, float b)
{
    if (!(q > 0.f)) return DIMS == 3 ? b * b : a * a;
    const float w = fmaf(-kUnit, rsqrt_normal(q), 1.f), u = kPerUnit * kPerUnit;
    // (next to the centre, |Delta|^2 / |scaled offset|^2: the square would be denormal)
    const bool tiny = q < FLT_MIN * kTouch;
    float d2 = a * a * (tiny ? 1.f : q * u);
    if constexpr (DIMS == 3) {
        const float s = tiny ? rsqrt_normal(q) : kPerUnit, x = s * d[0], y = s * d[1], z = s * d[DIMS - 1];
        d2 = fmaf(b * b * z, z, a * a * fmaf(x, x, y * y));
    }
    return tiny ? d2 : w * w * d2;
}

// Free columns {of the Bernstein basis, of its second derivative} at one of 32
// Chebyshev nodes of [0, T] (degree 10; only bounds use them).
template <int NF>
__device__ __forceinline__ void node_rows(int node, float horizon, float2 (&row)[NF + 1])
{
    const float tau = 0.5f - 0.5f * cospif(float(2 * node + 1) * (1.f / 64.f)), u = 1.f - tau;
    const float c10[11] = {1.f, 10.f, 45.f, 120.f, 210.f, 252.f, 210.f, 120.f, 45.f, 10.f, 1.f};
    const float c8[9] = {1.f, 8.f, 28.f, 56.f, 70.f, 56.f, 28.f, 8.f, 1.f};
    float tp[11], up[11], b8[9];
    tp[0] = up[0] = 1.f;
#pragma unroll
    for (int i = 1; i <= 10; ++i) {
        tp[i] = tp[i - 1] * tau;
        up[i] = up[i - 1] * u;
    }
#pragma unroll
    for (int j = 0; j <= 8; ++j) b8[j] = c8[j] * tp[j] * up[8 - j];
    const float sc = 90.f / (horizon * horizon);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int j = kFree0 + f;
        row[f].x = c10[j] * tp[j] * up[10 - j];
        row[f].y = sc * (b8[j - 2] - (j - 1 <= 8 ? 2.f * b8[j - 1 <= 8 ? j - 1 : 0] : 0.f) + (j <= 8 ? b8[j <= 8 ? j : 0] : 0.f));
    }
    row[NF] = make_float2(0.f, 0.f);
}

// A 4-byte asynchronous copy into shared memory; zero when !in (src is not read).
__device__ __forceinline__ void copy4(float *dst, const float *src, bool in)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// Starts the copies of the problem's tables into shared memory (all threads of
// the CTA; each waits for its own, then a barrier).
template <int G, int DIMS, int NF, bool WL>
__device__ void stage_tables(const ProjParams<float> &p, float *sm, const PtsLayout &L, bool with_fix)
{
    const int tid = threadIdx.x, T = blockDim.x, np_ = p.n_p;
    const int fbs = fb_stride(NF), nfp = nf_padded(NF);
    // asynchronous 4-byte copies (zeros beyond the last time stamp): every load is in flight at once
    auto put = [&](size_t at, int q, int t, int e) {  // e-th value of the row of kind q at stamp t
        const bool in = t < np_ && e < NF + DIMS;
        const float *src = !in ? p.tab
                               : e < NF ? p.tab + p.lay.fb + size_t(t) * fbs + q * nfp + e
                                        : p.tab + p.lay.base + (q * DIMS + (e - NF)) * np_ + t;
        copy4(sm + at, src, in);
    };
    constexpr int RW = 4 * ((NF + DIMS + 3) / 4), VW = 4 * ((NF + DIMS + 1) / 2);
    for (int t = tid; t < L.np; t += T)
#pragma unroll
        for (int e = 0; e < RW; ++e) put(L.rows + (size_t(e / 4) * L.np + t) * 4 + e % 4, 0, t, e);
    // (the halves of the CTA take a kind each)
    const int hp = L.np / 2, q = tid >= T / 2 ? 1 : 0;
    for (int u = tid - q * (T / 2); u < hp; u += T / 2)
#pragma unroll
        for (int z = 0; z < VW; ++z)
            put(L.vrows + (size_t(q * (VW / 4) + z / 4) * hp + u) * 4 + z % 4, 1 + q, 2 * u + (z & 1),
                2 * (z / 4) + ((z >> 1) & 1));
    for (int t = tid; t < L.np; t += T) copy4(sm + L.tv + t, p.tab + (t < np_ ? p.lay.tval + t : 0), t < np_);
    constexpr int ST = DIMS == 2 ? 12 : 16;
    for (int j = tid; j < p.n_obs; j += T) {
        // 2-D {-2 o_x, -2 o_y, thr, a | 1/a, -o_x/a, -o_y/a, 0 | -v_x/a, -v_y/a, 0, 0};
        // 3-D {-2 o_x, -2 o_y, -2 kappa o_z, thr | kappa, a, b, 0 | 1/a, -o_x/a, -o_y/a, -o_z/b |
        //      1/b, -v_x/a, -v_y/a, -v_z/b}
        const float *o = p.tab + p.lay.obs + size_t(j) * ST;
        float *d = sm + L.obs + 4 * size_t(j);
        for (int i = 0; i < 4; ++i) copy4(d + i, o + (DIMS == 3 ? 8 + i : i < 3 ? 4 + i : 3), true);
        if (DIMS == 3) {
            float *q = sm + L.obq + 4 * size_t(j);
            copy4(q + 1, o + 5, true);
            copy4(q + 2, o + 6, true);
            q[0] = kUnit * o[12];
            q[3] = fmaxf(o[8], o[12]);
        }
        if (j >= p.n_static)
            for (int i = 0; i < DIMS; ++i) copy4(sm + L.mov + 4 * size_t(j - p.n_static) + i, o + (DIMS == 3 ? 13 : 8) + i, true);
    }
    for (int i = tid; i < int(L.gsz); i += T) copy4(sm + L.grid + i, p.tab + p.lay.grid + i, true);
    if constexpr (WL) {
        if (with_fix)
            for (int i = tid; i < 3 * L.np; i += T) {
                const int f = i / L.np, t = i - f * L.np;
                for (int e = 0; e < 4 * L.nfch; ++e) {
                    const int col = e < kFree0 ? e : e + NF;
                    const bool in = t < np_ && col < p.nv;
                    copy4(sm + L.fix + (size_t(f * L.nfch + e / 4) * L.np + t) * 4 + e % 4,
                          p.tab + (in ? p.lay.basis + (size_t(f) * np_ + t) * p.nv + col : 0), in);
                }
            }
    }
}

// du += W u over the free columns of the lane's axis, the u of column F from
// its state lane.
template <int G, int DIMS, int NF, int F>
__device__ __forceinline__ void gather_u(float u, int src0, const float (&wrow)[NF], float &du)
{
    if constexpr (F < NF) {
        constexpr int V = DIMS * NF;
        float uf;
        if constexpr (DIMS == 2) {
            // the first exchange splits the axes, so an axis fills one half of the group
            static_assert(LaneOf<G, V, NF + F>::value == LaneOf<G, V, F>::value + G / 2, "axes in halves");
            uf = __shfl_sync(kAll, u, LaneOf<G, V, F>::value, G / 2);
        } else {
            static_assert(LaneOf<G, V, NF + F>::value - LaneOf<G, V, F>::value == LaneOf<G, V, NF>::value, "evenly spaced");
            uf = __shfl_sync(kAll, u, LaneOf<G, V, F>::value + src0);
        }
        du = fmaf(wrow[F], uf, du);
        gather_u<G, DIMS, NF, F + 1>(u, src0, wrow, du);
    }
}

// One sample's warp-level view: group lane, coefficient block, staging, list.
template <int G, int DIMS, int NF>
struct Group {
    int gl, pc;  // lane of the group; offset of the coefficient block
    __device__ __forceinline__ float4 *stage() const
    {
        return reinterpret_cast<float4 *>(smem() + pc + coef_floats(DIMS, NF) + (NF & 1) * 4);
    }
    __device__ __forceinline__ float4 *list() const { return stage() + 4 * G; }
    __device__ __forceinline__ int *tj() const { return reinterpret_cast<int *>(list() + kPairs); }
    __device__ __forceinline__ int moved() const { return pc + moved_at(G, DIMS, NF); }
};

// The sample's coefficients, each in both halves of a register pair.
template <int DIMS, int NF>
__device__ __forceinline__ void load_coefs(int pc, float2 (&c)[NF][DIMS])
{
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const float4 v = ld4s(pc + f * (DIMS == 2 ? 4 : 8));
        c[f][0] = make_float2(v.x, v.y);
        c[f][1] = make_float2(v.z, v.w);
        if constexpr (DIMS == 3) c[f][DIMS - 1] = *reinterpret_cast<const float2 *>(smem() + pc + f * 8 + 4);
    }
}

template <int DIMS, int NF>
__device__ __forceinline__ void load_coefs(int pc, float (&c)[NF][DIMS])
{
    float2 d[NF][DIMS];
    load_coefs<DIMS, NF>(pc, d);
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) c[f][ax] = d[f][ax].x;
}

// What rounding can make of the difference between two evaluations of a sample's
// rows (positions, velocities, accelerations; the larger of a warp's two samples).
// A row is a chain of NF FMAs that starts at its fixed part, and each rounds by at
// most u = 2^-24 of its partial sum: the result less the terms to come, so at most
// |result| + (sum of their |columns|) max |c|.  The columns' part, summed over the
// chain and the largest over the horizon, is kappa: 2.13, 9.54 / T, 81.4 / T^2 with
// five free columns, 4.25, 60 / T, 1530 / T^2 with seven.  A position is a mean of the
// coefficients (Bernstein), so at most the largest one's distance from the origin.
struct Rounding {
    float pos, vel, acc;
};
template <int G, int DIMS, int NF>
__device__ __forceinline__ Rounding row_rounding(const float2 (&c)[NF][DIMS], float vmax, float amax)
{
    static_assert(NF == 5 || NF == 7, "kappa");
    float most = 0.f, sum = 0.f, extent = smem()[kExtent];
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) {
            most = fmaxf(most, fabsf(c[f][ax].x));
            sum += fabsf(c[f][ax].x);
            extent = fmaxf(extent, fabsf(c[f][ax].x - smem()[kOrigin + ax]));
        }
    if (!(sum <= FLT_MAX)) most = INFINITY;  // a NaN, which the maxima drop, has no margin
    if (G == 16) {
        most = fmaxf(most, __shfl_xor_sync(kAll, most, 16));
        extent = fmaxf(extent, __shfl_xor_sync(kAll, extent, 16));
    }
    const float w = most * smem()[kRate], w2 = w * smem()[kRate];
    constexpr float two = 2.f * (DIMS == 2 ? 1.4143f : 1.7321f) * 5.9605e-8f;  // evaluations, axes
    Rounding r;
    r.pos = two * fmaf(NF == 5 ? 2.2f : 4.3f, most, (NF + 1) * extent);
    r.vel = two * fmaf(NF == 5 ? 9.6f : 60.f, w, (NF + 1) * vmax);
    r.acc = two * fmaf(NF == 5 ? 82.f : 1530.f, w2, (NF + 1) * amax);
    return r;
}

// The scaled offset of the pair with the listed terms o (3-D: obstacle j), its square
// and the semi-axes.
template <int DIMS>
__device__ __forceinline__ float listed_offset(const float (&x)[DIMS], const float4 &o, int j, float (&d)[DIMS], float &a,
                                               float &b)
{
    float ib = 0.f;
    a = o.w;
    b = 0.f;
    if constexpr (DIMS == 3) {
        const float4 v = ld4s(hdr(kObq) + 4 * j);
        ib = v.x;
        a = v.y;
        b = v.z;
    }
    return scaled_offset<DIMS>(x, o, ib, d);
}

// Exclusive prefix sum of n over the group and (total) its sum.
template <int G>
__device__ __forceinline__ int group_scan(int n, int gl, int &total)
{
    int inc = n;
#pragma unroll
    for (int off = 1; off < G; off <<= 1) {
        const int o = __shfl_up_sync(kAll, inc, off, G);
        if (gl >= off) inc += o;
    }
    total = __shfl_sync(kAll, inc, G - 1, G);
    return inc - n;
}

// Barrier of a team's warps.
template <int TEAM>
__device__ __forceinline__ void team_sync(int team)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(32 * TEAM) : "memory");
}

// Lists the pairs of every time stamp (sorted by (t, j)), padded to a multiple
// of G; returns the trips of the longest list of the warp, -1 when a sample has
// more than kPairs.  The strides of G time stamps one after another; in a team
// one to a warp at a time (role and totals, 2 TEAM ints of shared memory: where
// a warp's stride begins in the list follows from the others' totals; `list` is
// the group that holds it).
template <int TEAM, int G, int DIMS, int NF>
__device__ __forceinline__ int build_list(Group<G, DIMS, NF> gr, Group<G, DIMS, NF> list, float delta, int role, int team,
                                          int *totals)
{
    float c[NF][DIMS];
    load_coefs<DIMS, NF>(gr.pc, c);
    const int np = hdr(kNp), n_p = hdr(kStamps), tvo = hdr(kTv);
    const Screen<DIMS> sc(delta);
    float4 *lst = list.list();
    int *tj = list.tj();
    int base = 0;
#pragma unroll 1
    for (int q0 = 0, turn = 0; q0 < n_p; q0 += TEAM * G, turn ^= 1) {
        const int r0 = q0 + role * G, t = r0 + gr.gl, tc = TEAM > 1 ? min(t, np - 1) : t;
        const bool valid = t < n_p;
        float row[NF], x[DIMS];
        eval_row<DIMS, NF>(np, tc, c, row, x);
        const float tt = smem()[tvo + tc], ta = smem()[tvo + min(r0, n_p - 1)], tb = smem()[tvo + min(r0 + G, n_p) - 1];
        auto screen = [&](auto hit) {
            sc.fixed(x, valid, hit);
            sc.template moving<G>(x, valid, tt, ta, tb, hit);
        };
        // the first five hits of a lane are kept, a second screening serves longer ones
        int n = 0;
        unsigned long long kept = 0ull;
        screen([&](int j, const float4 &) {
            if (n < 5) kept |= static_cast<unsigned long long>(j) << (12 * n);
            ++n;
        });
        int total;
        int at = base + group_scan<G>(n, gr.gl, total);
        if constexpr (TEAM > 1) {
            // (the next round writes the other half: a warp is there only past the barrier that
            // follows every read of this one)
            if (gr.gl == 0) totals[TEAM * turn + role] = total;
            team_sync<TEAM>(team);
            total = 0;
#pragma unroll
            for (int i = 0; i < TEAM; ++i) {
                const int v = totals[TEAM * turn + i];
                if (i < role) at += v;
                total += v;
            }
        }
        base += total;
        auto write = [&](int j, const float4 &o) {
            if (at < kPairs) {
                lst[at] = listed_terms<DIMS>(o);
                tj[at] = t | (j << 16);
            }
            ++at;
        };
        if (__any_sync(kAll, n > 5)) {
            screen(write);
        } else {
#pragma unroll 1
            for (int i = 0; i < n; ++i) {
                const int j = int(kept & 4095u);
                kept >>= 12;
                write(j, pair_terms<DIMS>(j, tt, sc.ns));
            }
        }
    }
    const int most = __reduce_max_sync(kAll, base);
    const int trips = most > kPairs ? -1 : max(1, (most + G - 1) / G);
    // padding: a pair that is never active
    if (TEAM == 1 || role == 0)
        for (int e = base + gr.gl; e < trips * G; e += G) {
            lst[e] = make_float4(0.f, 4.f * kUnit, 0.f, 0.f);
            tj[e] = 0;
        }
    if constexpr (TEAM > 1)
        team_sync<TEAM>(team);
    else
        __syncwarp();
    return trips;
}

// Every pair screened now, in the list's order (more pairs than a list holds,
// or lists off): add(t, r) at the lane that the pair's number among the active
// ones gives, r.x the squared residual instead when SQUARE.  Used out of line, away
// from the registers of the iteration.
template <bool SQUARE, int G, int DIMS, int NF, typename Add>
__device__ __forceinline__ void dense_pairs(const Group<G, DIMS, NF> &gr, float delta, Add add)
{
    float c[NF][DIMS];
    load_coefs<DIMS, NF>(gr.pc, c);
    const int np = hdr(kNp), n_p = hdr(kStamps), tvo = hdr(kTv);
    const Screen<DIMS> sc(delta);
    float4 *buf = gr.list();  // active pairs of one stride, kPairs at a time
    int base = 0;             // active pairs so far
#pragma unroll 1
    for (int r0 = 0; r0 < n_p; r0 += G) {
        const int t = r0 + gr.gl;
        float row[NF], x[DIMS];
        eval_row<DIMS, NF>(np, t, c, row, x);
        const float tt = smem()[tvo + t], ta = smem()[tvo + r0], tb = smem()[tvo + min(r0 + G, n_p) - 1];
        auto each = [&](auto use) {
            auto hit = [&](int j, const float4 &o) {
                float d[DIMS], a, b;
                const float q = listed_offset<DIMS>(x, listed_terms<DIMS>(o), j, d, a, b);
                if (q < kTouch) use(d, q, a, b);
            };
            sc.fixed(x, t < n_p, hit);
            sc.template moving<G>(x, t < n_p, tt, ta, tb, hit);
        };
        int n = 0, total;
        each([&](const float (&)[DIMS], float, float, float) { ++n; });
        const int first = group_scan<G>(n, gr.gl, total);
        const int most = __reduce_max_sync(kAll, total);
#pragma unroll 1
        for (int w0 = 0; w0 < most; w0 += kPairs) {
            int at = first - w0;
            each([&](const float (&d)[DIMS], float q, float a, float b) {
                if (at >= 0 && at < kPairs) {
                    if constexpr (SQUARE) {
                        buf[at].x = pair_square<DIMS>(d, q, a, b);
                    } else {
                        float r[DIMS];
                        pair_residual<DIMS>(d, q, a, b, r);
                        buf[at] = make_float4(r[0], r[1], DIMS == 3 ? r[DIMS - 1] : 0.f, __int_as_float(t));
                    }
                }
                ++at;
            });
            __syncwarp();
            const int end = min(total - w0, kPairs);
            for (int i = (gr.gl - base - w0) & (G - 1); i < end; i += G) {
                const float4 v = buf[i];
                add(__float_as_int(v.w), v);
            }
            __syncwarp();
        }
        base += total;
    }
}

// g += sum of row^T r over the sample's active pairs; gfix (may be null): the
// fixed columns' sums, fix: the fixed columns of P in global memory.
template <int G, int DIMS, int NF>
__device__ __noinline__ void dense_sums(Group<G, DIMS, NF> gr, float delta, float (*g)[DIMS], float (*gfix)[DIMS],
                                        const float *fix, int nv)
{
    const int np = hdr(kNp);
    dense_pairs<false, G, DIMS, NF>(gr, delta, [&](int t, const float4 &v) {
        float row[NF], x[DIMS];
        load_row<DIMS, NF>(np, t, row, x);
        const float r[3] = {v.x, v.y, v.z};
        for (int ax = 0; ax < DIMS; ++ax) {
            for (int f = 0; f < NF; ++f) g[f][ax] = fmaf(row[f], r[ax], g[f][ax]);
            if (gfix)
                for (int f = 0; f < 11 - NF; ++f)
                    gfix[f][ax] = fmaf(fix[size_t(t) * nv + (f < kFree0 ? f : f + NF)], r[ax], gfix[f][ax]);
        }
    });
}

// The lane's sum of the squared residuals of the sample's active pairs.
template <int G, int DIMS, int NF>
__device__ __noinline__ double dense_squares(Group<G, DIMS, NF> gr, float delta)
{
    double r2 = 0.0;
    dense_pairs<true, G, DIMS, NF>(gr, delta, [&](int, const float4 &v) { r2 += double(v.x); });
    return r2;
}

// Which velocity / acceleration rows can become active before the acceleration
// has changed by sqrt(tau2) at some node: blocks of two time stamps per lane,
// velocity in the low half word (all or none), acceleration in the high one.
struct RateRows {
    float tau2;
    unsigned bits;
};
template <int G, int DIMS, int NF>
__device__ __forceinline__ RateRows rate_rows(Group<G, DIMS, NF> gr, float vmax, float amax)
{
    float2 c[NF][DIMS];
    load_coefs<DIMS, NF>(gr.pc, c);
    const int np = hdr(kNp), vrows = hdr(kVrows);
    float v2 = 0.f, a2 = 0.f;  // largest squares (a NaN counts as large)
    auto top = [](float m, float x) { return x <= m ? m : x; };
#pragma unroll 1
    for (int u = gr.gl; u < np / 2; u += G) {
        float2 row[NF], v[DIMS], a[DIMS];
        eval_pair<DIMS, NF>(vrows, np, 0, u, c, row, v);
        eval_pair<DIMS, NF>(vrows, np, 1, u, c, row, a);
        const float2 nv2 = norm2<DIMS>(v), na2 = norm2<DIMS>(a);
        v2 = top(top(v2, nv2.x), nv2.y);
        a2 = top(top(a2, na2.x), na2.y);
    }
    v2 = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(v2)));
    a2 = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(a2)));
    // the velocity changes by at most `reach` times what the acceleration does (NF = 5: it is
    // fixed at both ends)
    const float reach = (NF == 5 ? 0.5f : 1.f) * smem()[hdr(kTv) + hdr(kStamps) - 1];
    const Rounding rd = row_rounding<G, DIMS, NF>(c, vmax, amax);
    const float slv = 0.95f * (vmax - sqrtf(v2)) - rd.vel, sla = 0.95f * (amax - sqrtf(a2)) - rd.acc;
    const unsigned all = (1u << (np / (2 * G))) - 1u;
    float da = fminf(sla, slv / reach);
    unsigned vel = 0u, acc = 0u;
    if (!(da > 0.05f * amax)) {
        da = fmaxf(sla, kAccMargin * amax);
        if (!(slv > reach * da)) vel = all;
    }
    if (!(sla >= da)) {
        // blocks with an acceleration within the margin (a NaN counts as within)
        const float la = fmaxf(0.f, amax - 1.05f * da - rd.acc), la2 = la * la;
#pragma unroll 1
        for (int u = gr.gl, i = 0; u < np / 2; u += G, ++i) {
            float2 row[NF], a[DIMS];
            eval_pair<DIMS, NF>(vrows, np, 1, u, c, row, a);
            const float2 na2 = norm2<DIMS>(a);
            if (!(na2.x <= la2 && na2.y <= la2)) acc |= 1u << i;
        }
        acc = __reduce_or_sync(kAll, acc);
        // nearly all blocks: all of them, which needs no test where the velocity is on too
        if (4 * __popc(acc) >= 3 * __popc(all)) acc = all;
    }
    RateRows rr;
    rr.bits = vel | (acc << 16);
    rr.tau2 = vel == all && acc == all ? INFINITY : (da / kNodeBoundAcc) * (da / kNodeBoundAcc);
    return rr;
}

// Strides of time stamps with a position within delta of the workspace's walls
// or beyond them.
template <int DIMS>
__device__ __forceinline__ void wall(const ProjParams<float> &p, int ax, float &lo, float &hi)
{
    const float o = p.tab[p.lay.origin + ax];
    lo = p.smin[ax] - o;
    hi = p.smax[ax] - o;
}
template <int G, int DIMS, int NF>
__device__ __noinline__ unsigned wall_rows(Group<G, DIMS, NF> gr, const ProjParams<float> &p, float delta)
{
    float c[NF][DIMS];
    load_coefs<DIMS, NF>(gr.pc, c);
    const int np = hdr(kNp), n_p = hdr(kStamps);
    unsigned bits = 0u;
#pragma unroll 1
    for (int t = gr.gl, i = 0; t < n_p; t += G, ++i) {
        float row[NF], x[DIMS];
        eval_row<DIMS, NF>(np, t, c, row, x);
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) {
            float lo, hi;
            wall<DIMS>(p, ax, lo, hi);
            if (x[ax] > hi - delta || x[ax] < lo + delta) bits |= 1u << i;
        }
    }
    return __reduce_or_sync(kAll, bits);
}

// a1 / a2: the sample's free coefficient and multiplier in each state lane, and
// its row of W: all that a warp reads from global memory before the first
// iteration, so that the reads of a CTA's first samples run beside the staging
// of the tables.
template <int NF>
struct Start {
    float c, lam, wrow[NF];
};
template <int G, int DIMS, int NF>
__device__ __forceinline__ Start<NF> sample_start(const ProjParams<float> &p, int s_first, int s_end)
{
    constexpr int V = DIMS * NF;
    const int lane = threadIdx.x & 31, gl = lane & (G - 1), nv = p.nv, D = DIMS * nv;
    const int s = min(s_first + lane / G, s_end - 1), val = val_of(G, V, gl);
    const bool stv = val >= 0;
    const int sax = stv ? val / NF : 0, sf = stv ? val - sax * NF : 0, sd = sax * nv + kFree0 + sf;
    const size_t row0 = size_t(s) * D;
    double x64;
    if (p.mode == 0) {
        x64 = stv ? p.xi_in[row0 + sd] : 0.0;
    } else {
        // mu + L z: every coefficient's sum split over PARTS lanes (FP64 issues slowly here)
        constexpr int PARTS = G / V;
        const size_t seg = p.seg_len > 0 ? size_t(s / p.seg_len) : 0;  // D-PRIEST distribution
        const int v = gl % V, part = gl / V, d = (v / NF) * nv + kFree0 + v % NF;
        double acc = 0.0;
        x64 = stv ? p.mu[seg * D + sd] : 0.0;
        if (part < PARTS) {
            const double *Lrow = p.Lc + (seg * D + d) * D, *zi = p.z + row0;
            for (int q = part; q <= d; q += PARTS) acc = fma(Lrow[q], zi[q], acc);
        }
#pragma unroll
        for (int k = 0; k < PARTS; ++k) x64 += __shfl_sync(kAll, acc, (stv ? val : 0) + k * V, G);
    }
    Start<NF> st;
    st.c = stv ? float(x64) : 0.f;
    st.lam = stv && p.lam_in ? float(p.lam_in[row0 + sd]) : 0.f;
#pragma unroll
    for (int f = 0; f < NF; ++f) st.wrow[f] = stv ? p.tab[p.lay.W + sf * NF + f] : 0.f;
    return st;
}

// The projection of samples s_first and (G = 16) s_first + 1 by the calling
// warp; samples from s_end on repeat the last one and write nothing.  pw: the
// warp's shared block.
//
// TEAM > 1 warps project the one sample s_first, for launches that leave an SM few
// samples, where one warp's chain of an iteration is all that is waited for.
// Role 0 keeps and adds the obstacle and workspace rows; of four warps, roles 1
// and 2 add the velocity and acceleration rows of alternate blocks of time stamps
// and role 3 makes the node test beside them; of two, role 1 does both.  The
// partial sums of g and the test's answer meet in shared memory (one barrier an
// iteration); when the lists no longer hold, the sums are dropped, the lists
// rebuilt (a stride of time stamps to a warp) and the iteration done again, once:
// lists just built hold, and are not tested, so an iteration takes at most two
// passes whatever the test's arithmetic makes of its inputs.  Every warp repeats the
// multiplier and shared-inverse steps.
template <int G, int DIMS, int NF, bool WL, int TEAM>
__device__ __forceinline__ void project_samples(const ProjParams<float> &p, int pw, int s_first, int s_end, int role,
                                                int team, const Start<NF> &start)
{
    static_assert(TEAM == 1 || (G == 32 && (TEAM == 2 || TEAM == 4)), "a team's warps hold one sample");
    const bool pos = TEAM == 1 || role == 0, rate = TEAM == 1 || role == 1 || (TEAM == 4 && role == 2);
    const bool tester = TEAM > 1 && role == TEAM - 1;
    const unsigned rate_mask = TEAM == 4 ? (role == 1 ? 0xaaaa5555u : role == 2 ? 0x5555aaaau : 0u) : rate ? ~0u : 0u;
    constexpr int V = DIMS * NF, NB = 11 - NF, NN = 32 / G;
    constexpr int CS = coef_floats(DIMS, NF) / NF;  // floats per column in the coefficient block
    const int lane = threadIdx.x & 31, gl = lane & (G - 1), nv = p.nv, D = DIMS * nv;
    Group<G, DIMS, NF> gr;
    gr.gl = gl;
    gr.pc = pw + (lane / G) * sample_floats(G, DIMS, NF);
    const int pc = gr.pc;
    const bool live = s_first + lane / G < s_end;
    const int s = min(s_first + lane / G, s_end - 1);
    const int np = hdr(kNp), n_p = hdr(kStamps), vrows = hdr(kVrows);

    // ---- the sample's state lanes
    const int val = val_of(G, V, gl);
    const bool stv = val >= 0;
    const int sax = stv ? val / NF : 0, sf = stv ? val - sax * NF : 0;
    const int sd = sax * nv + kFree0 + sf;
    const int src0 = (lane & ~(G - 1)) + (DIMS == 3 ? sax * LaneOf<G, V, NF>::value : 0);
    const size_t row0 = size_t(s) * D;
    float stC = start.c, stLam = start.lam;
    const float stXi = stC;
    float wrow[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) wrow[f] = start.wrow[f];
    float2 *stp = reinterpret_cast<float2 *>(smem() + pc + sf * CS + 2 * sax);  // this lane's coefficient
    float2 *stm = reinterpret_cast<float2 *>(smem() + gr.moved()) + sf * DIMS + sax;
    float refP = stC, refA = stC;  // the coefficient at the last rebuild of the pair and rate lists
    __syncwarp();
    if (stv) *stp = make_float2(stC, stC);
    if (stv) *stm = make_float2(0.f, 0.f);
    gr.list()[gl] = make_float4(0.f, 4.f * kUnit, 0.f, 0.f);  // (evaluated once before the first rebuild)
    gr.tj()[gl] = 0;
    __syncwarp();

    const float rho = p.rho, vmax = p.vmax, amax = p.amax;
    const int K = p.K;
    const bool bounds = p.use_bounds != 0, lists = p.list_on != 0;
    // the obstacles' margin; without obstacles any positive length serves the other rows (finite:
    // margins are halved until they are below a share of it)
    const float delta = fminf(p.list_delta > 0.f ? p.list_delta : 0.01f * vmax * smem()[hdr(kTv) + n_p - 1], FLT_MAX);
    const int nblk = np / (2 * G);  // blocks of two time stamps per lane (at most 8)
    auto load_node = [&](int i, float2 (&node)[NF + 1]) {
#pragma unroll
        for (int f = 0; f < (NF + 1) / 2; ++f) {
            const float4 v = ld4s(hdr(kNode) + ((i * ((NF + 1) / 2) + f) * 32 + lane) * 4);
            node[2 * f] = make_float2(v.x, v.y);
            if (2 * f + 1 <= NF) node[2 * f + 1] = make_float2(v.z, v.w);
        }
    };
    // a negative threshold makes the first iteration build
    float tauP2 = lists ? -1.f : INFINITY, tauA2 = tauP2;
    int trips = lists ? 1 : -1;  // of the pair list (the longest of the warp); -1: screen every time stamp
    // warp-uniform: blocks of the velocity (low half) and acceleration rows, strides of the workspace's
    unsigned rates = lists ? 0u : (((1u << nblk) - 1u) * 65537u) & rate_mask;
    unsigned mbx = bounds && !lists && pos ? (2u << ((n_p - 1) / G)) - 1u : 0u;
    constexpr int NFCH = (NB + 3) / 4;
    const int fix = WL ? hdr(kFix) : 0;
    float gfix[WL ? NB : 1][DIMS];
#pragma unroll
    for (int f = 0; f < (WL ? NB : 1); ++f)
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) gfix[f][ax] = 0.f;
    auto add_fix = [&](const float (&r)[DIMS], int q, int t) {
        if constexpr (WL) {
#pragma unroll
            for (int i = 0; i < NFCH; ++i) {
                float4 w;
                if (fix) {
                    w = ld4s(fix + ((q * NFCH + i) * np + t) * 4);
                } else {
                    const float *b = p.tab + p.lay.basis + (size_t(q) * n_p + min(t, n_p - 1)) * nv;
                    auto at = [&](int f) { return f < NB ? b[f < kFree0 ? f : f + NF] : 0.f; };
                    w = make_float4(at(4 * i), at(4 * i + 1), at(4 * i + 2), at(4 * i + 3));
                }
                const float v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (4 * i + u < NB)
#pragma unroll
                        for (int ax = 0; ax < DIMS; ++ax) gfix[4 * i + u][ax] = fmaf(v[u], r[ax], gfix[4 * i + u][ax]);
            }
        }
    };

    float c[NF][DIMS];
    // which lists the nodes' displacement since the last rebuild no longer proves: bit 0 the
    // positions', bit 1 the rates'
    auto outdated = [&]() {
        float e_p = 0.f, e_a = 0.f;  // its square
        float2 m[NF][DIMS];
#pragma unroll
        for (int f = 0; f < NF * DIMS; f += 2) {
            const int at = gr.moved() + 2 * f;
            if (f + 1 < NF * DIMS) {
                const float4 v = ld4s(at);
                m[f / DIMS][f % DIMS] = make_float2(v.x, v.y);
                m[(f + 1) / DIMS][(f + 1) % DIMS] = make_float2(v.z, v.w);
            } else {
                m[f / DIMS][f % DIMS] = *reinterpret_cast<const float2 *>(smem() + at);
            }
        }
#pragma unroll
        for (int i = 0; i < NN; ++i) {
            float2 e[DIMS], node[NF + 1];
            load_node(i, node);
#pragma unroll
            for (int ax = 0; ax < DIMS; ++ax) e[ax] = fmul2(node[0], m[0][ax]);
#pragma unroll
            for (int f = 1; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) e[ax] = ffma2(node[f], m[f][ax], e[ax]);
            const float2 n = norm2<DIMS>(e);
            // (a NaN or an overflow is beyond every finite threshold)
            e_p = fmaxf(e_p, fminf(n.x, FLT_MAX));
            e_a = fmaxf(e_a, fminf(n.y, FLT_MAX));
        }
        if (!__any_sync(kAll, e_p > tauP2 || e_a > tauA2)) return 0;
        return (__any_sync(kAll, e_p > tauP2) ? 1 : 0) | (__any_sync(kAll, e_a > tauA2) ? 2 : 0);
    };
    // the warp's part of the rebuild, for every sample it holds.  Lists that lasted only a few
    // iterations are rebuilt with twice the margin, those of too many pairs with half of it,
    // which it then keeps to (never beyond the margin that the grid's cells were filled for, in
    // its header); rounding may take two fifths of a margin.  (A margin doubled again after it
    // overflowed built two or three lists a rebuild: 14 moving circles, 574 samples, K = 75,
    // 341 us a pass against 266; 45, 400 samples, K = 60, 625 against 379.)
    float reach = delta;
    float widest =
        fminf(hdr(kGrid) && __float_as_int(smem()[hdr(kGrid) + 4]) > 0 ? smem()[hdr(kGrid) + 7] : 8.f * delta, FLT_MAX);
    int built = -kShortLived;
    auto rebuild = [&](int need, int k) {
        const bool need_p = need & 1, need_a = need & 2;
        if (need_p) {
            float rounding;
            {
                float2 cc[NF][DIMS];
                load_coefs<DIMS, NF>(pc, cc);
                rounding = row_rounding<G, DIMS, NF>(cc, vmax, amax).pos;
            }
            if (k - built < kShortLived) reach = fminf(2.f * reach, widest);
            reach = fmaxf(reach, fminf(4.f * rounding, widest));
            built = k;
            refP = stC;
            if (pos || TEAM > 1) {
                Group<G, DIMS, NF> held = gr;  // role 0's block holds the list
                held.pc -= role * sample_floats(G, DIMS, NF);
                trips = -1;
                while (rounding <= 0.4f * reach) {
                    trips = build_list<TEAM>(gr, held, reach, role, team,
                                             reinterpret_cast<int *>(smem() + hdr(kXchAt) + team * kXch + kXchEnd));
                    if (trips >= 0 || reach < 0.3f * delta) break;
                    reach *= 0.5f;
                    widest = fmaxf(reach, 0.25f * delta);
                }
                if (trips < 0) reach = delta;
                // (no list: nothing is tested, so every stride's workspace rows too)
                if (bounds && pos) mbx = trips >= 0 ? wall_rows<G, DIMS, NF>(gr, p, reach) : (2u << ((n_p - 1) / G)) - 1u;
            }
            // largest displacement between rebuilds: 7/8 of the margin (the rest covers the rounding
            // of the tests) less that of the rows; without a list every pair is screened, and a list
            // tried again kRetry iterations on
            const float far = fmaf(0.875f / kNodeBoundPos, reach, -rounding);
            tauP2 = trips >= 0 ? far * far : INFINITY;
        }
        if (need_a) refA = stC;
        if (need_a && (rate || tester)) {
            const RateRows rr = rate_rows<G, DIMS, NF>(gr, vmax, amax);
            rates = rr.bits & rate_mask;
            tauA2 = rr.tau2;
        }
    };
    bool fresh = false;  // the lists were built for this iteration's coefficients (the same in all of a team)
    if (TEAM > 1 && lists) {
        rebuild(3, 0);
        fresh = true;
    }
    for (int k = 0, turn = 0;; ++k, ++turn) {
        load_coefs<DIMS, NF>(pc, c);
        if (trips < 0 && lists && k - built >= kRetry) tauP2 = -1.f;
        // the pair that trip e of the list gives this lane: its residual and whether it is active
        auto trip = [&](int e, float (&r)[DIMS], int &t) {
            const float4 o = gr.list()[e * G + gl];
            const int w = gr.tj()[e * G + gl];
            t = w & 0xffff;
            float row[NF], x[DIMS], d[DIMS], a, b;
            eval_row<DIMS, NF>(np, t, c, row, x);
            const float q = listed_offset<DIMS>(x, o, w >> 16, d, a, b);
            pair_residual<DIMS>(d, q, a, b, r);
            return q < kTouch;
        };
        float r0[DIMS];
        int t0, need = 0;
        bool in0;
        float gfix0[TEAM > 1 && WL ? NB : 1][DIMS];  // gfix at the start of the iteration
        const bool last = TEAM > 1 && k == K;        // only the test is left
        if constexpr (TEAM > 1) {
            if (pos) {
                in0 = trip(0, r0, t0);
            }
            if (tester && !fresh) need = outdated();
            if constexpr (WL)
#pragma unroll
                for (int f = 0; f < NB; ++f)
#pragma unroll
                    for (int ax = 0; ax < DIMS; ++ax) gfix0[f][ax] = gfix[f][ax];
        } else {
            // ---- the first trip's chain runs beside the node test's
            for (bool tested = false;; tested = true) {
                in0 = trip(0, r0, t0);
                if (tested) break;
                need = outdated();
                if (need == 0) break;
                rebuild(need, k);
            }
            if (k == K) break;
        }

        // ---- the lane's share of g = F^T (F xi_bar - e): the listed pairs first, the m-th active
        //      one at lane m mod G
        float g[NF][DIMS];
        bool act = false;
        auto add = [&](const float (&row)[NF], const float (&r)[DIMS]) {
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) g[f][ax] = fmaf(row[f], r[ax], g[f][ax]);
        };
        if (!pos || last) {
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) g[f][ax] = 0.f;
        } else if (trips >= 0) {
            int n = 0;  // active so far
            auto put = [&](bool in, const float (&r)[DIMS], int t) {
                unsigned m = __ballot_sync(kAll, in);
                if (G == 16) m = (m >> (lane & 16)) & 0xffffu;
                if (in)
                    gr.stage()[(n + __popc(m & ((1u << gl) - 1u))) & (4 * G - 1)] =
                        make_float4(r[0], r[1], DIMS == 3 ? r[DIMS - 1] : 0.f, __int_as_float(t));
                n += __popc(m);
            };
            auto get = [&](int m) {  // the lane's m-th active pair, zero when there is none
                const bool have = m < n;
                const float4 v = gr.stage()[m & (4 * G - 1)];
                const int t = have ? __float_as_int(v.w) : 0;
                float row[NF], x[DIMS], r[DIMS];
                r[0] = have ? v.x : 0.f;
                r[1] = have ? v.y : 0.f;
                if constexpr (DIMS == 3) r[DIMS - 1] = have ? v.z : 0.f;
                load_row<DIMS, NF>(np, t, row, x);
                add(row, r);
                add_fix(r, 0, t);
                act = act || have;
            };
            put(in0, r0, t0);
            int done = 0;  // of them taken (a multiple of G, the same over the group)
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) g[f][ax] = 0.f;
            // the stage holds 4 G pairs: the oldest G are taken before they could be overwritten,
            // the others at the end
            bool last = false;
#pragma unroll 1
            for (int e = 1;; ++e) {
                if (e < trips) {
                    float r[DIMS];
                    int t;
                    const bool in = trip(e, r, t);
                    put(in, r, t);
                    if (e < 3 || !__any_sync(kAll, n - done > 3 * G)) continue;
                } else {
                    last = true;
                }
                __syncwarp();
                const bool now = last || n - done > 3 * G;
                get(now ? done + gl : 0x7fffffff);
                done += now ? G : 0;
                __syncwarp();
                if (last && !__any_sync(kAll, n > done)) break;
            }
        } else {
            float gg[NF][DIMS], gf[WL ? NB : 1][DIMS];
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) gg[f][ax] = 0.f;
#pragma unroll
            for (int f = 0; f < (WL ? NB : 1); ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) gf[f][ax] = gfix[f][ax];
            dense_sums<G, DIMS, NF>(gr, 0.f, gg, WL ? gf : nullptr, p.tab + p.lay.basis, nv);
            act = true;
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) g[f][ax] = gg[f][ax];
#pragma unroll
            for (int f = 0; f < (WL ? NB : 1); ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) gfix[f][ax] = gf[f][ax];
        }
        // velocity (q = 0) and acceleration (q = 1) rows, two time stamps per lane at a time
#pragma unroll 1
        for (unsigned m = last ? 0u : rates; m; m &= m - 1) {
            const int bit = __ffs(m) - 1, q = bit >> 4, u = (bit & 15) * G + gl;
            const float lim = q ? amax : vmax;
            float2 row[NF], v[DIMS], cc[NF][DIMS];
            load_coefs<DIMS, NF>(pc, cc);
            eval_pair<DIMS, NF>(vrows, np, q, u, cc, row, v);
            const float2 n2 = norm2<DIMS>(v);
            // (a NaN counts as active, so it is not lost)
            const bool i0 = !(n2.x <= lim * lim), i1 = !(n2.y <= lim * lim);
            if (__any_sync(kAll, i0 || i1)) {
                const float w0 = i0 ? fmaf(-lim, rsqrtf(n2.x), 1.f) : 0.f;
                const float w1 = i1 ? fmaf(-lim, rsqrtf(n2.y), 1.f) : 0.f;
                float ra[NF], rb[NF], a0[DIMS], a1[DIMS];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    ra[f] = row[f].x;
                    rb[f] = row[f].y;
                }
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) {
                    a0[ax] = w0 * v[ax].x;
                    a1[ax] = w1 * v[ax].y;
                }
                add(ra, a0);
                add_fix(a0, 1 + q, 2 * u);
                add(rb, a1);
                add_fix(a1, 1 + q, 2 * u + 1);
                act = act || i0 || i1;
            }
        }
        if (bounds) {
#pragma unroll 1
            for (unsigned m = last ? 0u : mbx; m; m &= m - 1) {
                const int t = gl + G * (__ffs(m) - 1);
                float row[NF], x[DIMS], r[DIMS];
                eval_row<DIMS, NF>(np, t, c, row, x);
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) {
                    float lo, hi;
                    wall<DIMS>(p, ax, lo, hi);
                    r[ax] = t < n_p ? fmaxf(0.f, x[ax] - hi) - fmaxf(0.f, lo - x[ax]) : 0.f;
                    act = act || r[ax] != 0.f;
                }
                add(row, r);
                add_fix(r, 0, t);
            }
        }
        // ---- g over the group, into the state lanes (zero when no row is active)
        float gs = 0.f;
        if (__any_sync(kAll, act)) {
            float h[V];
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) h[ax * NF + f] = g[f][ax];
            gs = reduce_step<V, G / 2>(h, lane);
        }
        if constexpr (TEAM > 1) {
            // (two buffers: a warp writes one again only after the others have read it, past the
            // next iteration's barrier)
            float *x = smem() + hdr(kXchAt) + team * kXch + (turn & 1) * kXchBuf;
            if (role < 3) x[role * 32 + lane] = gs;
            if (tester && lane == 0) x[kXchFlag] = __int_as_float(need);
            team_sync<TEAM>(team);
            need = __float_as_int(x[kXchFlag]);
            if (need != 0) {
                rebuild(need, k);
                if constexpr (WL)
#pragma unroll
                    for (int f = 0; f < NB; ++f)
#pragma unroll
                        for (int ax = 0; ax < DIMS; ++ax) gfix[f][ax] = gfix0[f][ax];
            }
            if (last) break;
            fresh = need != 0;
            if (fresh) {
                --k;
                continue;
            }
            gs = x[lane] + x[32 + lane];
            if (TEAM == 4) gs += x[64 + lane];
        }
        // ---- multiplier step (eq. lag) and shared-inverse step:
        //      lambda^{k+1} = lambda^k - rho g, u = xi + lambda^{k+1} - rho g - c, c += W u
        stLam = fmaf(-rho, gs, stLam);
        const float u = fmaf(-rho, gs, stXi + stLam) - stC;
        float du = 0.f;
        gather_u<G, DIMS, NF, 0>(u, src0, wrow, du);
        stC += du;
        if (stv) {
            *stp = make_float2(stC, stC);
            *stm = make_float2(stC - refP, stC - refA);
        }
        __syncwarp();
    }

    // ---- a9: r = sqrt(sum of squared residual rows), c_1
    double r2 = 0.0, c1 = 0.0;
    float2 cc[NF][DIMS];
    load_coefs<DIMS, NF>(pc, cc);
#pragma unroll 1
    for (int u = TEAM > 1 ? gl + (role - 1) * G : gl; 2 * u < n_p && (TEAM == 1 || !pos); u += TEAM == 4 ? 3 * G : G) {
        float2 vrow[NF], vv[DIMS], av[DIMS];
        eval_pair<DIMS, NF>(vrows, np, 0, u, cc, vrow, vv);
        eval_pair<DIMS, NF>(vrows, np, 1, u, cc, vrow, av);
        const float2 v22 = norm2<DIMS>(vv), a22 = norm2<DIMS>(av);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int t = 2 * u + half;
            if (t >= n_p) break;
            float row[NF], x[DIMS], v[DIMS], a[DIMS];
            if (bounds || p.cost.kind == 1) eval_row<DIMS, NF>(np, t, c, row, x);
#pragma unroll
            for (int ax = 0; ax < DIMS; ++ax) {
                v[ax] = half ? vv[ax].y : vv[ax].x;
                a[ax] = half ? av[ax].y : av[ax].x;
            }
            const float v2 = half ? v22.y : v22.x, a2 = half ? a22.y : a22.x;
            const float fv = (v2 > vmax * vmax) ? 1.f - vmax * rsqrtf(v2) : 0.f;
            const float fa = (a2 > amax * amax) ? 1.f - amax * rsqrtf(a2) : 0.f;
            float rq = v2 * fv * fv + a2 * fa * fa;
            if (bounds) {
#pragma unroll
                for (int ax = 0; ax < DIMS; ++ax) {
                    float lo, hi;
                    wall<DIMS>(p, ax, lo, hi);
                    hi = fmaxf(0.f, x[ax] - hi);
                    lo = fmaxf(0.f, lo - x[ax]);
                    rq = fmaf(hi, hi, fmaf(lo, lo, rq));
                }
            }
            r2 += double(rq);
            c1 += double(point_cost<float, DIMS>(p.cost, x, v, a, a2));
        }
    }
    if (!pos) {
        // the pairs are role 0's
    } else if (trips >= 0) {
        // squares to the lanes as above, so that the sum does not depend on the list
        int n = 0, done = gl;
#pragma unroll 1
        for (int e = 0; e < trips; ++e) {
            const float4 o = gr.list()[e * G + gl];
            const int w = gr.tj()[e * G + gl];
            float row[NF], x[DIMS], d[DIMS], a, b;
            eval_row<DIMS, NF>(np, w & 0xffff, c, row, x);
            const float q = listed_offset<DIMS>(x, o, w >> 16, d, a, b);
            const bool in = q < kTouch;
            unsigned m = __ballot_sync(kAll, in);
            if (G == 16) m = (m >> (lane & 16)) & 0xffffu;
            if (in) gr.stage()[(n + __popc(m & ((1u << gl) - 1u))) & (4 * G - 1)].x = pair_square<DIMS>(d, q, a, b);
            n += __popc(m);
            __syncwarp();
            if (done < n) {  // at most one per trip
                r2 += double(gr.stage()[done & (4 * G - 1)].x);
                done += G;
            }
            __syncwarp();
        }
    } else {
        r2 += dense_squares<G, DIMS, NF>(gr, 0.f);
    }
    {
        // the lower half of the group ends with r2, the upper half with c_1
        const bool hi = (gl & (G / 2)) != 0;
        double v = (hi ? c1 : r2) + __shfl_xor_sync(kAll, hi ? r2 : c1, G / 2);
#pragma unroll
        for (int off = G / 4; off >= 1; off >>= 1) v += __shfl_xor_sync(kAll, v, off);
        if constexpr (TEAM > 1) {
            float *x = smem() + hdr(kXchAt) + team * kXch;
            double *xd = reinterpret_cast<double *>(x + kXchEnd);
            if (gl == 0) xd[2 * role] = v;
            if (gl == G / 2) xd[2 * role + 1] = v;
            if constexpr (WL) {
                constexpr int VB = NB * DIMS;
                float gb[VB];
#pragma unroll
                for (int i = 0; i < VB; ++i) gb[i] = gfix[i % NB][i / NB];
                const float gsum = reduce_step<VB, G / 2>(gb, lane);
                const int vb = val_of(G, VB, gl);
                if (vb >= 0) x[kXchFix + 32 * role + vb] = gsum;
            }
            team_sync<TEAM>(team);
            if (role != 0) return;
            const int at = gl == 0 ? 0 : 1;
            v = xd[at] + xd[2 + at];
            if (TEAM == 4) v += xd[4 + at] + xd[6 + at];
        }
        if (live && gl == 0) p.r_out[s] = sqrt(v);
        if (live && gl == G / 2) p.c1_out[s] = v;
    }
    // ---- xi_bar (boundary coefficients from the closed form) and multipliers
    if (live)
        for (int d = gl; d < D; d += G) {
            const int ax = d / nv, col = d - ax * nv, f = col - kFree0;
            p.xi_bar[row0 + d] = (f >= 0 && f < NF) ? double(smem()[pc + f * CS + 2 * ax]) : p.cB[ax * kMaxNv + col];
        }
    if (p.lam_out) {
        // (with 32 lanes each value sits in two neighbouring ones)
        if (live && stv && (G == 16 || (gl & 1) == 0)) p.lam_out[row0 + sd] = double(stLam);
        if constexpr (WL) {
            constexpr int VB = NB * DIMS;
            auto put = [&](int i, float gsum) {
                const int ax = i / NB, f = i - ax * NB;
                const size_t gi = row0 + ax * nv + (f < kFree0 ? f : f + NF);
                const float l0 = p.lam_in ? float(p.lam_in[gi]) : 0.f;
                if (live) p.lam_out[gi] = double(fmaf(-rho, gsum, l0));
            };
            float gb[VB];
#pragma unroll
            for (int i = 0; i < VB; ++i) gb[i] = gfix[i % NB][i / NB];
            if constexpr (TEAM > 1) {
                const float *x = smem() + hdr(kXchAt) + team * kXch + kXchFix;
                if (gl < VB) put(gl, TEAM == 4 ? (x[gl] + x[32 + gl]) + x[64 + gl] : x[gl] + x[32 + gl]);
            } else if constexpr (VB <= G) {
                const float gsum = reduce_step<VB, G / 2>(gb, lane);
                const int vb = val_of(G, VB, gl);
                if (vb >= 0) put(vb, gsum);
            } else {
#pragma unroll
                for (int i = 0; i < VB; ++i) {
#pragma unroll
                    for (int off = G / 2; off >= 1; off >>= 1) gb[i] += __shfl_xor_sync(kAll, gb[i], off);
                    if (gl == i % G) put(i, gb[i]);
                }
            }
        }
    }
}

// Samples s0 .. s0 + count - 1 of one problem by the CTA's first `warps`
// warps (all threads call it; the shared block is free again after the call).
template <int G, int DIMS, int NF, bool WL, int TEAM>
__device__ void pts_body(const ProjParams<float> &p, int s0, int count, int warps)
{
    float *sm = smem();
    const PtsLayout L = pts_layout(G, DIMS, NF, p.nv, p.n_p, p.n_obs, p.n_static, warps, TEAM > 1 ? warps / TEAM : 0);
    bool with_fix = false;
    if constexpr (WL) {
        unsigned dyn;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
        with_fix = L.total_fix * sizeof(float) <= dyn;
    }
    if (threadIdx.x == 0) {
        int *h = reinterpret_cast<int *>(sm);
        h[kVrows] = int(L.vrows);
        h[kNode] = int(L.node);
        h[kTv] = int(L.tv);
        h[kObs] = int(L.obs);
        h[kObq] = int(L.obq);
        h[kMov] = int(L.mov);
        h[kGrid] = L.gsz && p.list_grid ? int(L.grid) : 0;
        h[kFix] = with_fix ? int(L.fix) : 0;
        h[kNp] = L.np;
        h[kStamps] = p.n_p;
        h[kStatic] = p.n_static;
        h[kObstacles] = p.n_obs;
        h[kNext] = (32 / G) * warps;
        h[kXchAt] = int(L.xch);
    }
    if (threadIdx.x < 32) {
        // node i of lane l: l mod G + i G
        const float horizon = p.tab[p.lay.tval + p.n_p - 1];
#pragma unroll
        for (int i = 0; i < 32 / G; ++i) {
            float2 r[NF + 1];
            node_rows<NF>((threadIdx.x & (G - 1)) + i * G, horizon, r);
#pragma unroll
            for (int f = 0; f < (NF + 1) / 2; ++f)
                reinterpret_cast<float4 *>(sm + L.node)[(i * ((NF + 1) / 2) + f) * 32 + threadIdx.x] =
                    make_float4(r[2 * f].x, r[2 * f].y, r[2 * f + 1].x, r[2 * f + 1].y);
        }
    }
    stage_tables<G, DIMS, NF, WL>(p, sm, L, with_fix);
    if (threadIdx.x >= 32 * (kMaxWarps - 1)) {
        // the origin, the fixed coefficients' largest distance from it, 1 / T (the last warp: the
        // first ones have samples to start; read beside the staging)
        const int lane = threadIdx.x & 31;
        float e = 0.f;
        for (int d = lane; d < DIMS * p.nv; d += 32) {
            const int ax = d / p.nv, col = d - ax * p.nv;
            if (col < kFree0 || col >= kFree0 + NF)
                e = fmaxf(e, float(fabs(p.cB[ax * kMaxNv + col] - double(p.tab[p.lay.origin + ax]))));
        }
        e = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(e)));
        if (lane == 0) sm[kExtent] = e;
        if (lane == 0) sm[kRate] = 1.f / p.tab[p.lay.tval + p.n_p - 1];
        if (lane < DIMS) sm[kOrigin + lane] = p.tab[p.lay.origin + lane];
    }
    const int warp = threadIdx.x >> 5, team = warp / TEAM, first = TEAM > 1 ? team : (32 / G) * warp;
    const bool works = warp < warps && first < count;
    Start<NF> start;
    if (works) start = sample_start<G, DIMS, NF>(p, s0 + first, s0 + count);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (!works) return;
    if constexpr (TEAM > 1) {
        // (count is at most the number of teams)
        project_samples<G, DIMS, NF, WL, TEAM>(p, int(L.warp0 + warp * L.wsz), s0 + team, s0 + count,
                                               warp - TEAM * team, team, start);
    } else {
        // a warp's first samples by its number, then whichever are next
        constexpr int NN = 32 / G;  // samples per warp
        const int pw = int(L.warp0 + warp * L.wsz);
        int i = first;
        for (;;) {
            project_samples<G, DIMS, NF, WL, 1>(p, pw, s0 + i, s0 + count, 0, 0, start);
            if (NN * warps >= count) break;
            if ((threadIdx.x & 31) == 0) i = atomicAdd(reinterpret_cast<int *>(sm) + kNext, NN);
            i = __shfl_sync(kAll, i, 0);
            if (i >= count) break;
            start = sample_start<G, DIMS, NF>(p, s0 + i, s0 + count);
        }
    }
}

// One CTA per p.S samples; its first p.WS warps take them, all stage the tables.
// (Teams of four leave an SM one CTA, so their warps may keep 255 registers.)
template <int G, int DIMS, int NF, bool WL, int TEAM>
__global__ void __launch_bounds__(32 * kMaxWarps, TEAM == 4 ? 1 : 2) pts_kernel(const ProjParams<float> p)
{
    pdl_trigger();
    pdl_wait();
    const int s0 = blockIdx.x * p.S;
    pts_body<G, DIMS, NF, WL, TEAM>(p, s0, min(p.S, p.N - s0), p.WS);
}

// Persistent form over many problems: CTAs take (problem, first sample)
// items (p.S samples by p.WS warps) through an atomic counter until none is
// left; the item's parameters are staged in shared memory.  *next must be zero
// at launch.
template <int G, int DIMS, int NF, bool WL>
__global__ void __launch_bounds__(32 * kMaxWarps, 2)
    pts_batch_kernel(const ProjParams<float> *params, const int2 *items, int n_items, int *next)
{
    __shared__ int s_item;
    __shared__ ProjParams<float> s_p;  // the item's parameters, read from shared memory where used
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(next, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= n_items) break;
        const int2 w = items[it];
        if (threadIdx.x == 0) s_p = params[w.x];
        __syncthreads();
        pts_body<G, DIMS, NF, WL, 1>(s_p, w.y, min(s_p.S, s_p.N - w.y), s_p.WS);
        __syncthreads();
    }
}

}  // namespace pts
}  // namespace priest
