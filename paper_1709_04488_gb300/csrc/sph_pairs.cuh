// Pair kernels of the grad-h SPH neighbour loop (templates; the translation
// units sph_pairs.cu and sph_pairs_m6.cu instantiate them for the M4 and M6
// kernels).
//
// Work unit: one warp per leaf cell (the paper's OpenMP unit of work is an
// active leaf cell, Sec. 5.2.1, and neighbours are gathered per leaf, not per
// particle, Sec. 4.2).  LPP lanes serve each particle of the leaf; the warp
// walks the tree over the leaves once per leaf, stages candidate particles in
// shared memory (positions relative to the query leaf: leaf reference points
// differenced in FP64, then cast), and each lane keeps its own list of
// in-range candidates so that the arithmetic runs without divergence.
//
// FP64 problems (SPH_PREC_FP64): this GPU runs FP64 at 1/64 of the FP32 rate,
// so the walk, the staging and the tests of the candidates run in FP32, in a
// frame of the domain's size (Frame), with the rounding of the staged
// coordinates to spare (stage_err), and only the pairs that pass take FP64:
// their distance from the FP64 positions, the exact membership, the sums.  The
// FP64 pipe is 74 % busy in k_forces and 70 % in k_density (36864 particles of
// the Sod tube, two lanes per particle: 947 -> 660 us and 626 -> 510 us;
// smaller problems 1.7-4 times faster).
//
//  k_density   Eqs. SPHRHO, HRHO, OMEGA: Newton-Raphson on
//              F(h) = rho(h) - m (eta/h)^3 over the cached list of (r^2, m_j)
//              with the same bracketing fallback as the oracle; the list is
//              rebuilt if h outgrows it.  Particles whose list overflows, or
//              that need too many rebuilds, go to k_density_fallback, which
//              re-walks the tree in every iteration.
//  k_forces    Eqs. GRADHMOMEQN, GRADHENEQN, MON97ARTVISC, MON97ENERGYDISS
//              and the signal speed of Eq. SPH_DT.  Every pair term is formed
//              from an exactly antisymmetric pair vector with order-independent
//              FP32 operations, so that F_ij = -F_ji bit for bit; m_i a_i is
//              accumulated with
//              error-free (TwoSum) compensated FP32 sums combined in FP64,
//              which keeps sum_i m_i a_i near FP64 round-off.
#pragma once
#include "sph_internal.cuh"
#include "sph_leaf.cuh"
#include "sph_tuned.h"

#include <type_traits>

namespace sph {

namespace {

constexpr unsigned FULL = 0xffffffffu;
// class index of a lanes-per-particle count; 32 (block-step tasks, one
// particle per warp) shares 8's slot: a tick launches only its tasks' class
__host__ __device__ constexpr int lpp_log2(int l) { return l == 1 ? 0 : l == 2 ? 1 : l == 4 ? 2 : 3; }
constexpr double kListMargin = 1.03;  // list radius = R_K h * margin (R_K: support in units of h)

constexpr int kMaxRebuild = 6;

template <typename T>
__device__ __forceinline__ T tinf();
template <>
__device__ __forceinline__ float tinf<float>() { return INFINITY; }
template <>
__device__ __forceinline__ double tinf<double>() { return INFINITY; }

// a < b for a >= 0 (or -1) and b > 0: in FP64 on the bit patterns, which keeps
// the comparison off the FP64 pipe
__device__ __forceinline__ bool lt_pos(float a, float b) { return a < b; }
__device__ __forceinline__ bool lt_pos(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }

// Two FP32 values in one 64-bit register and the packed operations on them
// (each half rounded as the scalar operation rounds it).
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float a, float b)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(F2 x, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// a - b, rounded once: fma(b, -1, a)
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return fma2(b, pack2(-1.f, -1.f), a); }

// Smoothing kernels of Sec. 2, W(r, h) = sigma f(q) / h^3 with q = r / h and
// support q < R: fdf(q) gives f and f', df(q) f' alone.
template <int K>
struct Kern;

// M4 cubic spline: sigma = 1/pi, R = 2.
template <>
struct Kern<SPH_KERNEL_M4> {
    static constexpr double R = 2.0;
    static constexpr double sigma = 1.0 / kPi;
    template <typename T>
    static __device__ __forceinline__ void fdf(T q, T &f, T &df)
    {
        T t = lt_pos(q, T(2)) ? T(2) - q : T(0);
        T t2 = t * t;
        T f2 = T(0.25) * t2 * t, df2 = T(-0.75) * t2;
        T q2 = q * q;
        T f1 = T(1) + q2 * (T(0.75) * q - T(1.5));
        T df1 = q * (T(2.25) * q - T(3));
        bool in = lt_pos(q, T(1));
        f = in ? f1 : f2;
        df = in ? df1 : df2;
    }
    template <typename T>
    static __device__ __forceinline__ T df(T q);  // rounding fixed operation by operation (force pass)
};

// M6 quintic spline: f = (3-q)^5 - 6 (2-q)^5 + 15 (1-q)^5 (each term while
// its bracket is positive), sigma = 1/(120 pi), R = 3.  Inside q < 1 the
// three terms are summed as their expanded polynomial 66 - 60 q^2 + 30 q^4
// - 10 q^5 (f' = -120 q + 120 q^3 - 50 q^4), which avoids the cancellation
// of f' -> 0 at q -> 0; beyond q = 1 the brackets are used directly.
template <>
struct Kern<SPH_KERNEL_M6> {
    static constexpr double R = 3.0;
    static constexpr double sigma = 1.0 / (120.0 * kPi);
    template <typename T>
    static __device__ __forceinline__ void fdf(T q, T &f, T &df)
    {
        T a = lt_pos(q, T(3)) ? T(3) - q : T(0);
        T c = lt_pos(q, T(2)) ? T(2) - q : T(0);
        T a4 = (a * a) * (a * a), c4 = (c * c) * (c * c);
        T f2 = a4 * a - T(6) * (c4 * c), df2 = T(30) * c4 - T(5) * a4;
        T q2 = q * q;
        T f1 = T(66) + q2 * (T(-60) + q2 * (T(30) - T(10) * q));
        T df1 = q * (T(-120) + q2 * (T(120) - T(50) * q));
        bool in = lt_pos(q, T(1));
        f = in ? f1 : f2;
        df = in ? df1 : df2;
    }
    template <typename T>
    static __device__ __forceinline__ T df(T q);  // rounding fixed operation by operation (force pass)
};

// f, f' and sigma of the kernel a problem selects (warp-uniform; for the
// slow path, which serves particles of any problem)
template <typename T>
__device__ __forceinline__ void kern_fdf(int k, T q, T &f, T &df)
{
    if (k == SPH_KERNEL_M6) Kern<SPH_KERNEL_M6>::fdf(q, f, df);
    else Kern<SPH_KERNEL_M4>::fdf(q, f, df);
}
__device__ __forceinline__ double kern_sigma(int k)
{
    return k == SPH_KERNEL_M6 ? Kern<SPH_KERNEL_M6>::sigma : Kern<SPH_KERNEL_M4>::sigma;
}

// Softened gravity of the M4 kernel (Eqs. GRAVFORCEKERNEL, GRADHZETA): the
// enclosed mass fraction M(q) = 4 int_0^q f s^2 ds of a unit-mass kernel
// (phi' = M / r^2) and the potential shape psi (phi = psi(q)/h, psi' = M/q^2,
// -1/q from q = 2 on).  zeta needs psi + M/q (= -h^2 dphi/dh), which vanishes
// from q = 2 on and is psi(0) = -7/5 at q = 0.
template <typename T>
__device__ __forceinline__ T grav_mass(T q)
{
    const T q3 = q * q * q;
    if (q >= T(2)) return T(1);
    if (q < T(1)) return T(4) * q3 * (T(1.0 / 3.0) + q * q * (T(-0.3) + T(0.125) * q));
    return T(4) * (q3 * (T(2.0 / 3.0) + q * (T(-0.75) + q * (T(0.3) - q * T(1.0 / 24.0)))) - T(1.0 / 60.0));
}
template <typename T>
__device__ __forceinline__ T grav_psi_plus_mq(T q)
{
    if (q >= T(2)) return T(0);
    const T q2 = q * q;
    T psi;
    if (q < T(1)) psi = q2 * (T(2.0 / 3.0) + q2 * (T(-0.3) + T(0.1) * q)) - T(1.4);
    else psi = q2 * (T(4.0 / 3.0) + q * (T(-1) + q * (T(0.3) - q * T(1.0 / 30.0)))) + T(1.0 / 15.0) / q - T(1.6);
    return psi + (q > T(0) ? grav_mass(q) / q : T(0));
}

template <typename T>
__device__ __forceinline__ T rsqrt_t(T x);
template <>
__device__ __forceinline__ float rsqrt_t<float>(float x) { return rsqrtf(x); }
template <>
__device__ __forceinline__ double rsqrt_t<double>(double x) { return rsqrt(x); }

template <typename T>
__device__ __forceinline__ T mul_rn(T a, T b);
template <>
__device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <>
__device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <typename T>
__device__ __forceinline__ T add_rn(T a, T b);
template <>
__device__ __forceinline__ float add_rn<float>(float a, float b) { return __fadd_rn(a, b); }
template <>
__device__ __forceinline__ double add_rn<double>(double a, double b) { return __dadd_rn(a, b); }
template <typename T>
__device__ __forceinline__ T sub_rn(T a, T b);
template <>
__device__ __forceinline__ float sub_rn<float>(float a, float b) { return __fsub_rn(a, b); }
template <>
__device__ __forceinline__ double sub_rn<double>(double a, double b) { return __dsub_rn(a, b); }
template <typename T>
__device__ __forceinline__ T fma_rn(T a, T b, T c);
template <>
__device__ __forceinline__ float fma_rn<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <>
__device__ __forceinline__ double fma_rn<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
// (The force pass evaluates a pair's terms at several inlined call sites;
// spelling every operation that feeds m_i a_i with these intrinsics keeps the
// compiler from contracting them differently at different sites, so both
// particles of a pair get the same bits.)

template <typename T>
__device__ __forceinline__ T Kern<SPH_KERNEL_M4>::df(T q)
{
    const T t = lt_pos(q, T(2)) ? sub_rn(T(2), q) : T(0);
    const T df2 = mul_rn(mul_rn(T(-0.75), t), t);
    const T df1 = mul_rn(q, fma_rn(T(2.25), q, T(-3)));
    return lt_pos(q, T(1)) ? df1 : df2;
}

template <typename T>
__device__ __forceinline__ T Kern<SPH_KERNEL_M6>::df(T q)
{
    const T a = lt_pos(q, T(3)) ? sub_rn(T(3), q) : T(0);
    const T c = lt_pos(q, T(2)) ? sub_rn(T(2), q) : T(0);
    const T a2 = mul_rn(a, a), c2 = mul_rn(c, c);
    const T df2 = fma_rn(T(30), mul_rn(c2, c2), mul_rn(T(-5), mul_rn(a2, a2)));
    const T df1 = mul_rn(q, fma_rn(mul_rn(q, q), fma_rn(T(-50), q, T(120)), T(-120)));
    return lt_pos(q, T(1)) ? df1 : df2;
}

// 2/(rho_i + rho_j): a deterministic function of the commutative sum, so
// both sides of a pair get the same bits (fast reciprocal in FP32)
__device__ __forceinline__ float fast_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double fast_div(double a, double b) { return a / b; }

// a length in the unit of the FP32 copies (FP64 problems: the walk's frame)
__device__ __forceinline__ float frame_len(float v, double) { return v; }
__device__ __forceinline__ float frame_len(double v, double unit) { return (float)(v * unit); }
__device__ __forceinline__ float frame_len_ru(float v, double) { return v; }
__device__ __forceinline__ float frame_len_ru(double v, double unit) { return __double2float_ru(v * unit); }

// sorted particle index carried in the w slot of a staged vector: bit
// pattern in FP32 staging (only ever copied), exact value in FP64 staging
__device__ __forceinline__ float bits_as_t(int v, float) { return __int_as_float(v); }
__device__ __forceinline__ double bits_as_t(int v, double) { return (double)v; }
__device__ __forceinline__ int t_as_bits(float v) { return __float_as_int(v); }
__device__ __forceinline__ int t_as_bits(double v) { return (int)v; }

// The query box of a walk, in the warp's scratch (read back at each node
// test as broadcast vectors).  The leaves that pass decide the slots of the
// staged candidates, hence (at several lanes per particle) the order of the
// sums, so their test has one definition (leaf_within, leaf_overlap).  It
// takes about 15 operations per axis; node_gap takes 7 and agrees with it to
// within s, 1e-5 of the problem's coordinates and the reach (five times the
// definition's own slack), so that only boxes within s of the boundary, well
// under one test in ten, are decided by the definition, and the nodes above
// the leaves, which only have to pass what holds such a leaf, never are.
// (With the definition at the leaves and a one-sided test above: cloud 8e6
// 62.3 ms for two evaluations, M6 lattice of 37^3 3.84 ms for five; with
// this 57.9 and 3.47 ms.)
struct QueryBox {
    float4 ax[3];  // per axis: lo + hi, hi - lo, 2 L (infinity if isolated)
    // squared distances (of doubled coordinates) below which a box is within
    // R for sure and above which it is not; s doubled; R^2 of the definition
    float in2, out2, s2, R2;
};
// cmax: bound of the problem's and its boxes' |coordinates|
__device__ __forceinline__ void set_query(QueryBox &qb, const float4 &lo, const float4 &hi, float R, const PhysParams &ph,
                                          float cmax)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < 3) {
        const float l = lane == 0 ? lo.x : lane == 1 ? lo.y : lo.z, h = lane == 0 ? hi.x : lane == 1 ? hi.y : hi.z;
        qb.ax[lane] = make_float4(l + h, h - l, ph.periodic ? 2.f * ph.box_len_f[lane] : INFINITY, 0.f);
    } else if (lane == 3) {
        const float s = 1e-5f * (cmax + R) + 1e-29f;
        const float in = 2.f * (R - 2.f * s), out = 2.f * (R + 2.f * s);
        qb.in2 = in > 0.f ? in * in : -1.f;
        qb.out2 = out * out;
        qb.s2 = 2.f * s;
        qb.R2 = R * R * 1.00001f;
    }
    __syncwarp();
}

// bound of the problem's |coordinates| (F64: in the walk's frame)
template <bool F64>
__device__ __forceinline__ float coord_bound(const PhysParams &ph, const ProbDyn &d)
{
    return F64 ? frame_of(ph, d).max : ph.periodic ? ph.coord_max : d.coord_max;
}

// twice the gap between the query box and [blo, bhi] along one axis (minimum
// image if periodic), negative where they overlap
__device__ __forceinline__ float node_gap(const float4 &qa, float blo, float bhi)
{
    const float d = qa.x - (blo + bhi);
    return fminf(fabsf(d), fabsf(qa.z - fabsf(d))) - (qa.y + (bhi - blo));
}
__device__ __forceinline__ float node_dist2(const QueryBox &qb, const float4 &blo, const float4 &bhi, float u = 1.f)
{
    const float gx = fmaxf(node_gap(qb.ax[0], blo.x, bhi.x), 0.f) * u;
    const float gy = fmaxf(node_gap(qb.ax[1], blo.y, bhi.y), 0.f) * u;
    const float gz = fmaxf(node_gap(qb.ax[2], blo.z, bhi.z), 0.f) * u;
    return gx * gx + gy * gy + gz * gz;
}
__device__ __forceinline__ float node_sep(const QueryBox &qb, const float4 &blo, const float4 &bhi)
{
    return fmaxf(node_gap(qb.ax[0], blo.x, bhi.x),
                 fmaxf(node_gap(qb.ax[1], blo.y, bhi.y), node_gap(qb.ax[2], blo.z, bhi.z)));
}

// The definition, along one axis: the centres' distance and the reach of the
// two boxes, grown for the FP32 rounding of the box coordinates; overlap in
// every image where the reach spans half the box.
__device__ __forceinline__ bool axis_dist(const float4 &qa, float blo, float bhi, int periodic, float L, float &d,
                                          float &reach)
{
    const float ca = 0.5f * qa.x, ha = 0.5f * qa.y;
    const float cb = 0.5f * (blo + bhi), hb = 0.5f * (bhi - blo);
    reach = ha + hb;
    reach += 2e-6f * (fabsf(ca) + fabsf(cb) + reach) + 1e-30f;
    d = fabsf(ca - cb);
    if (periodic) {
        if (reach >= 0.5f * L) return true;
        if (d > L) d -= L;
        d = fminf(d, L - d);
    }
    return false;
}
__device__ __forceinline__ float axis_gap(const float4 &qa, float blo, float bhi, int periodic, float L)
{
    float d, reach;
    return axis_dist(qa, blo, bhi, periodic, L, d, reach) ? 0.f : fmaxf(d - reach, 0.f);
}
__device__ __forceinline__ bool axis_overlap(const float4 &qa, float blo, float bhi, int periodic, float L)
{
    float d, reach;
    return axis_dist(qa, blo, bhi, periodic, L, d, reach) || d <= reach;
}
// Do two boxes come within (Euclidean) distance R of each other?  Tighter
// than growing one box by R along each axis: the grown box's corners, where
// no point is within R, are left out.
__device__ __forceinline__ bool leaf_within(const QueryBox &qb, const float4 &blo, const float4 &bhi, const PhysParams &ph)
{
    const float gx = axis_gap(qb.ax[0], blo.x, bhi.x, ph.periodic, ph.box_len_f[0]);
    const float gy = axis_gap(qb.ax[1], blo.y, bhi.y, ph.periodic, ph.box_len_f[1]);
    const float gz = axis_gap(qb.ax[2], blo.z, bhi.z, ph.periodic, ph.box_len_f[2]);
    return gx * gx + gy * gy + gz * gz <= qb.R2;
}
__device__ __forceinline__ bool leaf_overlap(const QueryBox &qb, const float4 &blo, const float4 &bhi, const PhysParams &ph)
{
    return axis_overlap(qb.ax[0], blo.x, bhi.x, ph.periodic, ph.box_len_f[0]) &&
           axis_overlap(qb.ax[1], blo.y, bhi.y, ph.periodic, ph.box_len_f[1]) &&
           axis_overlap(qb.ax[2], blo.z, bhi.z, ph.periodic, ph.box_len_f[2]);
}

// Tests of one node per lane, called by the whole warp: the position box
// within R (up_within: nodes above the leaves), the smoothing-sphere box
// overlapping the query.  u: a power of two, where the query's R and cmax
// were given in units of 1 / u (gaps multiplied by it before they are squared).
__device__ __forceinline__ bool up_within(const QueryBox &qb, const NodeBox &nb, float u = 1.f)
{
    return node_dist2(qb, nb.plo, nb.phi, u) <= qb.out2;
}
__device__ __forceinline__ bool up_overlap(const QueryBox &qb, const NodeBox &nb, float u = 1.f)
{
    return node_sep(qb, nb.slo, nb.shi) * u <= qb.s2;
}
__device__ __forceinline__ bool box_within(const QueryBox &qb, const NodeBox &nb, const PhysParams &ph)
{
    const float g2 = node_dist2(qb, nb.plo, nb.phi);
    bool ok = g2 <= qb.in2;
    const bool edge = !ok && g2 <= qb.out2;
    if (__any_sync(FULL, edge) && edge) ok = leaf_within(qb, nb.plo, nb.phi, ph);
    return ok;
}
__device__ __forceinline__ bool box_overlap(const QueryBox &qb, const NodeBox &nb, const PhysParams &ph)
{
    const float g = node_sep(qb, nb.slo, nb.shi);
    bool ok = g <= -qb.s2;
    const bool edge = !ok && g <= qb.s2;
    if (__any_sync(FULL, edge) && edge) ok = leaf_overlap(qb, nb.slo, nb.shi, ph);
    return ok;
}

// Warp-cooperative depth-first walk of one problem's tree, one step at a time:
// next() returns the next level-1 node (up to 32 sibling leaves, in order) that
// lies under nodes whose boxes pass up(box), or -1.  The caller tests its
// leaves, one per lane, and stages the ones that pass in one round of memory
// accesses.  (A step function, so that the caller's staging has one call site:
// each inlined one is a copy, and the instruction cache was the second
// largest stall of the wrap-list force launch.)  The nodes still to open of
// each level are kept in the lanes (lane l: level l's), not in an array a
// run-time level indexes.
struct Walk {
    unsigned m, sm;
    int base, sb, lvl, top;
    __device__ __forceinline__ void start(const ProbDyn &d)
    {
        top = lvl = d.top_level + 1;  // (one node above the top level holds it; top level 0: the leaves' only node)
        m = 1u;
        sm = 0u;
        base = sb = 0;
    }
    template <class Up>
    __device__ __forceinline__ int next(const BatchView &b, const ProbDyn &d, Up &&up)
    {
        const int lane = threadIdx.x & 31;
        for (;;) {
            while (m == 0u) {
                if (lvl == top) return -1;
                ++lvl;
                m = __shfl_sync(FULL, sm, lvl);
                base = __shfl_sync(FULL, sb, lvl);
            }
            const int node = base + __ffs(m) - 1;
            m &= m - 1u;
            if (lvl == 1) return node;
            const int ch = node * kBranch + lane;
            bool ok = false;
            if (ch < d.node_cnt[lvl - 1]) ok = up(b.nodes[lvl - 1][d.node_off[lvl - 1] + ch]);
            const unsigned cm = __ballot_sync(FULL, ok);
            if (cm == 0u) continue;
            if (lane == lvl) {
                sm = m;
                sb = base;
            }
            --lvl;
            m = cm;
            base = node * kBranch;
        }
    }
};
// lanes of a level-1 node that hold a leaf
__device__ __forceinline__ unsigned leaf_lanes(int cnt0, int node)
{
    const int n = cnt0 - node * kBranch;
    return n >= 32 ? FULL : (1u << n) - 1u;
}

template <typename T>
__device__ __forceinline__ int warp_incl_scan(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int w = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += w;
    }
    return v;
}

// Per-warp scratch for staging one group of up to 32 candidate leaves.
template <typename T>
struct StageScratch {
    // per candidate leaf, in order: its shift (FP64 difference of reference
    // points, cast) and (w) its first sorted index less its first element
    typename Vec4<T>::type leaf[32];
    T L[3], Li[3];             // box lengths and their inverses (periodic wraps)
    T C[3];                    // centre of the query leaf's box (in its frame)
    QueryBox qb;               // the walk's query
    float ihl[3];              // 2 / box length
    float thr[3];              // candidate extents (packed units) from which a leaf pair is ambiguous
};

// Periodic minimum images.  A pair vector is formed as (o_i - o_j) - D from
// the particles' offsets o from their leaves' reference points (at most E_A,
// E_B in magnitude) and the minimum-image shift D of the two reference
// points, so it is the minimum image of every pair within R unless
// E_A + E_B + R >= L/2 ("ambiguous" leaf pairs: few particles per box length,
// or leaves that span much of a thin box).  The particles of an ambiguous
// candidate leaf are moved, as they are staged, to their image nearest to
// the centre of the query leaf's box; the staged vectors are then minimum
// images unless W_A/2 + R >= L/2 (W_A the query box's width), in which case
// each pair vector is wrapped as well.  The force pass wraps the pair
// vectors of ambiguous leaf pairs it evaluates, r - L rint(r / L), which is
// odd in r: the vectors of i-j and j-i stay exact negatives.  The box
// lengths sit in the warp's scratch.  All of this runs in the launches that
// serve the wrap list: the common launches test each candidate leaf as they
// walk (per axis, from the extents the leaf pass packs into the leaves'
// boxes) and at the first ambiguous pair put the query leaf, with nothing
// written yet, on that list.
__device__ __forceinline__ float half_box(const PhysParams &ph)
{
    return 0.5f * fminf(ph.box_len_f[0], fminf(ph.box_len_f[1], ph.box_len_f[2])) * 0.99999f;
}

template <typename T>
__device__ __forceinline__ T box_L(const PhysParams &ph, int a);
template <>
__device__ __forceinline__ float box_L<float>(const PhysParams &ph, int a) { return ph.box_len_f[a]; }
template <>
__device__ __forceinline__ double box_L<double>(const PhysParams &ph, int a) { return ph.box_len[a]; }
template <typename T>
__device__ __forceinline__ T box_Li(const PhysParams &ph, int a);
template <>
__device__ __forceinline__ float box_Li<float>(const PhysParams &ph, int a) { return ph.box_inv_f[a]; }
template <>
__device__ __forceinline__ double box_Li<double>(const PhysParams &ph, int a) { return ph.box_inv[a]; }

// lanes 0..2 copy the box lengths (times the power of two u, as lo and hi
// are) and the query box's centre into the warp's scratch
template <typename T, typename V>
__device__ __forceinline__ void load_box(StageScratch<T> &sc, const PhysParams &ph, const V &lo, const V &hi, T u = T(1))
{
    const int lane = threadIdx.x & 31;
    if (lane < 3) {
        sc.L[lane] = box_L<T>(ph, lane) * u;
        sc.Li[lane] = box_Li<T>(ph, lane) * (T(1) / u);
        sc.C[lane] = T(0.5) * (lane == 0 ? lo.x + hi.x : lane == 1 ? lo.y + hi.y : lo.z + hi.z);
        sc.ihl[lane] = 2.f * ph.box_inv_f[lane];
    }
    __syncwarp();
}

// A leaf pair (A, B) is ambiguous for pairs within R when on some axis
// E_A + E_B + R >= L/2, from the leaves' packed offset extents (slo.w, in
// units of L/2046).  set_thr (lanes 0..2) stores, for query leaf A and reach
// R, the extent of B from which that holds; ambiguous(E_B) tests it.
template <typename T>
__device__ __forceinline__ void set_thr(StageScratch<T> &sc, float ea, float R)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < 3)
        sc.thr[lane] = 1023.f * (0.99999f - R * sc.ihl[lane]) - (float)((__float_as_uint(ea) >> (10 * lane)) & 1023u);
    __syncwarp();
}
template <typename T>
__device__ __forceinline__ bool ambiguous(float eb, const StageScratch<T> &sc)
{
    const unsigned b = __float_as_uint(eb);
    return (float)(b & 1023u) >= sc.thr[0] || (float)((b >> 10) & 1023u) >= sc.thr[1] ||
           (float)((b >> 20) & 1023u) >= sc.thr[2];
}

// bits of `m` (lanes of a group), renumbered by the order of the lanes set in
// `mask`
__device__ __forceinline__ unsigned by_order(unsigned m, unsigned mask)
{
    if (m == 0u) return 0u;
    const int lane = threadIdx.x & 31;
    return __reduce_or_sync(FULL, (m >> lane) & 1u ? 1u << __popc(mask & ((1u << lane) - 1u)) : 0u);
}

// largest h (plo.w) and largest leaf offset extent (slo.w) of a problem,
// carried up to its top nodes
__device__ __forceinline__ void problem_top_max(const BatchView &b, const ProbDyn &dy, float &hmax, float &extmax)
{
    const int lane = threadIdx.x & 31, top = dy.top_level;
    float h = 0.f, e = 0.f;
    if (lane < dy.node_cnt[top]) {
        const NodeBox &nb = b.nodes[top][dy.node_off[top] + lane];
        h = nb.plo.w;
        e = nb.slo.w;
    }
    hmax = warp_max(h);
    extmax = warp_max(e);
}

// half of the query box's largest width
template <typename V>
__device__ __forceinline__ float half_width(const V &lo, const V &hi)
{
    return 0.5f * (float)fmax(hi.x - lo.x, fmax(hi.y - lo.y, hi.z - lo.z)) * 1.00001f;
}

// minimum image of a pair vector
template <typename T>
__device__ __forceinline__ void wrap3s(const StageScratch<T> &sc, T &x, T &y, T &z)
{
    x = fma_rn(-sc.L[0], rint(mul_rn(x, sc.Li[0])), x);
    y = fma_rn(-sc.L[1], rint(mul_rn(y, sc.Li[1])), y);
    z = fma_rn(-sc.L[2], rint(mul_rn(z, sc.Li[2])), z);
}

// move staged point q to its periodic image nearest to c (unchanged when q
// is already that image)
template <typename T, typename V>
__device__ __forceinline__ void wrap_near(const StageScratch<T> &sc, V &q, T cx, T cy, T cz)
{
    q.x = fma_rn(-sc.L[0], rint(mul_rn(sub_rn(q.x, cx), sc.Li[0])), q.x);
    q.y = fma_rn(-sc.L[1], rint(mul_rn(sub_rn(q.y, cy), sc.Li[1])), q.y);
    q.z = fma_rn(-sc.L[2], rint(mul_rn(sub_rn(q.z, cz), sc.Li[2])), q.z);
}

// Squared distance from point q to the box [lo, hi] (zero inside).
template <typename T, typename V>
__device__ __forceinline__ T box_dist2(const V &q, const V &lo, const V &hi)
{
    T dx = fmax(fmax(lo.x - q.x, q.x - hi.x), T(0));
    T dy = fmax(fmax(lo.y - q.y, q.y - hi.y), T(0));
    T dz = fmax(fmax(lo.z - q.z, q.z - hi.z), T(0));
    return dx * dx + dy * dy + dz * dz;
}

// min_image, decided on the bit pattern of |d|: the comparisons would run on
// the FP64 pipe, 1/64 of the FP32 rate
__device__ __forceinline__ double min_image_bits(double d, double L, int periodic)
{
    if (periodic) {
        const long long ad = __double_as_longlong(d) & 0x7fffffffffffffffll;
        if (ad > __double_as_longlong(0.5 * L)) d += __longlong_as_double(__double_as_longlong(L) | (~__double_as_longlong(d) & (1ll << 63)));
    }
    return d;
}
// shift of candidate leaf B's reference point from the query leaf A's: FP64
// difference, minimum image, cast (SCALED: in units of 1 / unit)
template <typename T, bool SCALED>
__device__ __forceinline__ T leaf_shift(double cb, double ca, double L, int periodic, double unit)
{
    const double d = min_image_bits(cb - ca, L, periodic);
    return SCALED ? (T)(d * unit) : (T)d;
}

// Stage the particles of the leaves first + k (bit k of mask) that keep()
// accepts, compacted into slots [nbuf, ...) of the warp's candidate buffer of
// capacity CH; flush() runs first whenever fewer than 32 slots are free.
// The particles are read 32 at a time, one per lane, through load(j) (j the
// sorted index) and moved into the query leaf A's frame by the leaf shift
// before keep(q, o) sees them (o: which candidate leaf of the group, in
// order; keep may move q to another periodic image).  group(has, B, stB, o,
// D) runs on every lane once per call (lane k: candidate leaf first + k if
// has); store(slot, q, o, idx) writes a kept particle (idx: its index within
// its leaf).  The leaf of element e follows from the leaves' first elements
// that fall into the chunk, one bit each, gathered by one warp reduction
// (a binary search over the first elements took five dependent shared-memory
// reads per chunk).
template <typename T, int CH, bool SCALED = false, class Group, class Load, class Keep, class Store, class Flush>
__device__ __forceinline__ void stage_group(const BatchView &b, int A, unsigned mask, int first, const PhysParams &ph,
                                            double unit, int &nbuf, StageScratch<T> &sc, Group &&group, Load &&load,
                                            Keep &&keep, Store &&store, Flush &&flush)
{
    using V = typename Vec4<T>::type;
    const int lane = threadIdx.x & 31;
    const bool has = (mask >> lane) & 1u;
    const unsigned below = (1u << lane) - 1u;
    const int ord = __popc(mask & below);
    int stB = 0, nB = 0;
    V D{};
    if (has) {
        const int B = first + lane;
        stB = b.leaf_start[B];
        nB = b.leaf_start[B + 1] - stB;
        const double *cb = b.leaf_c + 3LL * B, *ca = b.leaf_c + 3LL * A;
        D.x = leaf_shift<T, SCALED>(cb[0], ca[0], ph.box_len[0], ph.periodic, unit);
        D.y = leaf_shift<T, SCALED>(cb[1], ca[1], ph.box_len[1], ph.periodic, unit);
        D.z = leaf_shift<T, SCALED>(cb[2], ca[2], ph.box_len[2], ph.periodic, unit);
    }
    group(has, first + lane, stB, ord, D);
    const int incl = warp_incl_scan<T>(nB);
    const int tot = __shfl_sync(FULL, incl, 31);
    // first element of this lane's leaf (beyond every chunk without one)
    const int fe = has ? incl - nB : 0x40000000;
    __syncwarp();  // earlier readers of the scratch are done
    if (has) {
        D.w = bits_as_t(stB - fe, T(0));
        sc.leaf[ord] = D;
    }
    __syncwarp();
    // element e0 + lane of the chunk at e0: which leaf, its index there, its
    // staged vector; `started` leaves begin before the chunk, the last of
    // them `into` elements before it
    int started = 0, into = 0;
    V qn{}, sn{};
    int on = 0, idxn = 0;
    auto fetch = [&](int e0) {
        const unsigned x = (unsigned)(fe - e0);
        const unsigned M = __reduce_or_sync(FULL, x < 32u ? 1u << x : 0u);
        const unsigned le = M & (below | (1u << lane));
        if (e0 + lane < tot) {
            on = started + __popc(le) - 1;
            idxn = le ? lane - (31 - __clz(le)) : lane + into;
            sn = sc.leaf[on];
            qn = load(e0 + lane + t_as_bits(sn.w));
        }
        started += __popc(M);
        into = M ? __clz(M) + 1 : into + 32;
    };
    // the particles are loaded one chunk of 32 ahead: a chunk's load (an L2
    // round trip) overlaps the filtering, storing and flushing of the chunk
    // before it (flush() leaves the scratch and the loaded arrays alone)
    fetch(0);
    for (int e0 = 0; e0 < tot; e0 += 32) {
        V q = qn;
        q.x += sn.x;
        q.y += sn.y;
        q.z += sn.z;
        const int o = on, idx = idxn;
        if (e0 + 32 < tot) fetch(e0 + 32);
        if (nbuf > CH - 32) flush();
        const bool ok = e0 + lane < tot && keep(q, o);
        const unsigned bal = __ballot_sync(FULL, ok);
        if (ok) store(nbuf + __popc(bal & below), q, o, idx);
        nbuf += __popc(bal);
    }
}

// The staged coordinates of FP64 problems and of the neighbour lists are
// rounded copies; a pair is decided by them only outside a band around the
// radius.  Roundings of a staged particle q (of a leaf with shift D; moved to
// the image q') against a query particle p, in units of 2^-24, per axis: the
// offset q - D, the shift, their sum, the image (box length, product, sum),
// p, the difference and its own image come to at most 2 |D| + 3 |q| + 7 |q'|
// + 6 |p|, so three axes move the distance by less than 0.8 stage_err, and
// a reach grown by 2 stage_err misses no pair.  It scales with separations,
// leaf widths and reaches, not with the domain (1e-6 of the domain, as large as
// h where that is 1e-6 of it, let every staged particle of a clump pass to
// FP64).
template <typename V>
__device__ __forceinline__ float abs3(const V &v) { return fmaxf(fabsf(v.x), fmaxf(fabsf(v.y), fabsf(v.z))); }
__device__ __forceinline__ float box_abs(const float4 &lo, const float4 &hi) { return fmaxf(abs3(lo), abs3(hi)); }
// D, q, q' as above, pmax: largest |coordinate| of the query particles
__device__ __forceinline__ float stage_err(float D, float q, float q1, float pmax) { return 1e-6f * (D + q + q1 + pmax); }
// squares below this may have underflowed (lengths below 1e-18 of the domain)
constexpr float kTinySq = 1e-36f;

// Box of the query leaf's particles in its own frame (offsets from the
// reference point), over the lanes with on set.
template <typename V, typename T>
__device__ __forceinline__ void frame_box(const V &x, bool on, V &lo, V &hi)
{
    lo.x = warp_min(on ? x.x : tinf<T>());
    lo.y = warp_min(on ? x.y : tinf<T>());
    lo.z = warp_min(on ? x.z : tinf<T>());
    hi.x = warp_max(on ? x.x : -tinf<T>());
    hi.y = warp_max(on ? x.y : -tinf<T>());
    hi.z = warp_max(on ? x.z : -tinf<T>());
}

// sum over the LPP lanes that serve one particle
template <int LPP, typename T>
__device__ __forceinline__ T group_sum(T v)
{
#pragma unroll
    for (int o = 1; o < LPP; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}
template <int LPP, typename T>
__device__ __forceinline__ T group_max(T v)
{
#pragma unroll
    for (int o = 1; o < LPP; o <<= 1) {
        T w = __shfl_xor_sync(FULL, v, o);
        v = w > v ? w : v;
    }
    return v;
}
template <int LPP>
__device__ __forceinline__ bool group_any(bool v)
{
    int x = v ? 1 : 0;
#pragma unroll
    for (int o = 1; o < LPP; o <<= 1) x |= __shfl_xor_sync(FULL, x, o);
    return x != 0;
}

// One Newton-Raphson update of the h-rho solve with the oracle's bracketing
// (Eqs. SPHRHO, HRHO).  Returns true when |h_new - h| < tol h; h then stays
// (it is within the tolerance of the root, and the caller's sums at h stay
// valid), else h becomes h_new.
template <typename T>
__device__ __forceinline__ bool nr_update(T &h, T &lo, T &hi, T rho, T drho, T m, T eta3, T tol)
{
    T hinv = T(1) / h;
    T hinv3 = hinv * hinv * hinv;
    T F = rho - m * eta3 * hinv3;
    T dF = drho + T(3) * m * eta3 * hinv3 * hinv;
    if (F < T(0)) lo = h;
    else hi = h;
    T hn = dF > T(0) ? h - F / dF : T(-1);
    bool bad = !(hn >= lo) || !(hn <= hi) || !(hn >= T(0.5) * h) || !(hn <= T(2) * h) || !(dF > T(0));
    if (bad) hn = (hi == tinf<T>()) ? T(2) * h : T(0.5) * (lo + hi);
    const bool conv = fabs(hn - h) < tol * h;
    if (!conv) h = hn;
    return conv;
}

// The items of a pair kernel's warp: one by position first, the first warp of
// every block before the second ones, so that a launch of fewer items than
// warps spreads over all SMs (tickets alone went to the warps of the blocks
// that started first, four to an SM, and left the other SMs idle); tickets
// after that.
__device__ __forceinline__ int first_item() { return (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x); }
__device__ __forceinline__ int next_item(int *ticket)
{
    int t = 0;
    if ((threadIdx.x & 31) == 0) t = atomicAdd(ticket, 1);
    return (int)(gridDim.x * (blockDim.x >> 5)) + __shfl_sync(FULL, t, 0);
}

// The FP32 kernels' candidate buffer: NA arrays (the negated coordinates and
// what else a test needs) of CH candidates, slot k in the section of the lanes
// with k % LPP == sub, at place k / LPP.  A lane reads its section four
// candidates at a time and tests them two at a time in packed operations:
// about 8 instructions a candidate in place of 11, where every one of them
// issues for the whole warp's union of neighbourhoods (density pass: cloud 1e6
// 1.62 -> 1.42 ms, Sedov 64^3 237 -> 209 us, Sod 36864 63.9 -> 59.7 us).  Sections are padded by
// four, for the sentinels behind the last candidate and to set their banks
// apart.
template <int CH, int LPP, int NA>
struct CandBuf {
    static constexpr int NARR = NA, SEC = (CH / LPP + 3) / 4 * 4 + 4;
    static constexpr size_t bytes = sizeof(float) * NA * SEC * LPP;
    float v[NA][SEC * LPP];
    static __device__ __forceinline__ int place(int slot) { return slot % LPP * SEC + slot / LPP; }
    // candidates of lane section `sub` among n
    static __device__ __forceinline__ int mine(int n, int sub) { return (n - sub + LPP - 1) / LPP; }
    // far points behind the last candidates, so that the tests take whole fours
    __device__ __forceinline__ void pad(int n)
    {
        // (the square of their distance overflows to infinity; four, as a lane
        // may go to the end of the longest section, one candidate beyond its own)
        for (int t = threadIdx.x & 31; t < 4 * LPP; t += 32) v[0][t % LPP * SEC + mine(n, t % LPP) + t / LPP] = -3e38f;
    }
};
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

template <typename T, int LPP, bool UM, int K>
struct DCfg {
    using V = typename Vec4<T>::type;
    // list entries per lane: room for ~2x the mean neighbour count per
    // particle within the list radius (M4 at eta = 1.2: ~63; M6 at eta = 1.0:
    // ~123, served by 2 or more lanes per particle)
    static constexpr bool D64 = sizeof(T) == 8;
    // (FP64, two or four lanes, deals its entries to the lanes by rank; room for
    // a first h 1.26 and 1.36 times too large in a uniform M4 problem)
    static constexpr int LCAP = K == SPH_KERNEL_M6 ? (LPP <= 2 ? 96 : LPP == 4 ? 64 : 32)
                                                     : LPP == 1 ? SPH_DENS_LCAP1 : LPP == 2 ? 64 : LPP == 4 ? 40 : 24;
    static constexpr int CH = SPH_DENS_CH;
    static constexpr int WPB = D64 ? 2 : 4;
    static constexpr int MINB = D64 ? 4 : K == SPH_KERNEL_M6 ? SPH_MINB_M6 : LPP == 1 ? SPH_DENS_MINB1 : SPH_DENS_MINB;  // blocks per SM the registers allow
    // FP64: rows of pairs waiting for their FP64 distance, candidates per room check
    static constexpr int LC = 32, SB = 32;
    static constexpr size_t wait = D64 ? (size_t)LC * 32 * sizeof(int) + CH * sizeof(int) : 0;
    static constexpr int LW = UM ? 1 : 2;  // list words per entry: r^2 (and m_j unless masses are equal)
    static constexpr size_t scratch = (sizeof(StageScratch<float>) + 31) & ~(size_t)31;
    // (a row beyond the capacity takes the entries that no longer fit)
    static constexpr size_t lists = (size_t)(LCAP + 1) * 32 * LW * sizeof(T);
    // (more lanes: too few candidates each for the fours to pay; M6: 96 registers, spills)
    static constexpr bool PACK = !D64 && K == SPH_KERNEL_M4 && LPP <= 2;
    using Cand = CandBuf<CH, LPP, UM ? 3 : 4>;      // (PACK: -x, -y, -z, m)
    static constexpr size_t cands = PACK ? (Cand::bytes + 31) & ~(size_t)31 : CH * sizeof(float4);
    static constexpr size_t per_warp = cands + lists + scratch + wait;
    static constexpr size_t smem = WPB * per_warp;
};

// Block-step tasks (k0 >= 0): the lane group pp serves the (k0 + pp)-th
// particle of the leaf whose step ends now; returns its position in the
// leaf and whether there is one.  k0 < 0: the whole leaf, position pp.
template <typename T>
__device__ __forceinline__ bool task_member(const BatchView &b, int st, int nA, int k0, int pp, int &pos)
{
    const int lane = threadIdx.x & 31;
    if (k0 < 0) {
        pos = pp;
        return pp < nA;
    }
    const unsigned dm = __ballot_sync(FULL, lane < nA && ((const T *)b.slev)[st + (lane < nA ? lane : 0)] > T(0));
    const int ord = k0 + pp;
    const bool on = ord < __popc(dm);
    pos = on ? (int)__fns(dm, 0u, ord + 1) : 0;
    return on;
}

// A task's position box (its particles only) in absolute float coordinates,
// from their offsets x (staged, leaf frame) as the leaf build forms the
// leaf's: each offset widened for its one rounding, plus the leaf's
// reference point rounded down (up).  w of plo: hmax.
__device__ __forceinline__ float task_widen_dn(float v) { return __fsub_rd(v, fabsf(v) * 2.4e-7f); }
__device__ __forceinline__ float task_widen_up(float v) { return __fadd_ru(v, fabsf(v) * 2.4e-7f); }

template <typename V>
__device__ __forceinline__ void task_box(const BatchView &b, int leaf, const V &x, bool on, float hmax, NodeBox &box)
{
    const float o[3] = {(float)x.x, (float)x.y, (float)x.z};
    float lo[3], hi[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = warp_min(on ? task_widen_dn(o[a]) : INFINITY);
        hi[a] = warp_max(on ? task_widen_up(o[a]) : -INFINITY);
    }
    const float *cf = b.leaf_cf + 6LL * leaf;  // reference point rounded down (0..2) and up (3..5)
    box.plo = make_float4(__fadd_rd(cf[0], lo[0]), __fadd_rd(cf[1], lo[1]), __fadd_rd(cf[2], lo[2]), hmax);
    box.phi = make_float4(__fadd_ru(cf[3], hi[0]), __fadd_ru(cf[4], hi[1]), __fadd_ru(cf[5], hi[2]), box.phi.w);
}

// Outputs of the density solve for sorted particle s (one lane per particle).
template <typename T>
__device__ __forceinline__ void density_epilogue(const BatchView &b, const ProbStatic &ps, long long s,
                                                 typename Vec4<T>::type pi, T h, T S0, T S1, int use_pred,
                                                 T sigma, double unit, T Z = T(0))
{
    using V = typename Vec4<T>::type;
    const PhysParams &ph = ps.ph;
    long long g = b.perm[s];
    long long i = g - ps.base;
    double u = use_pred ? b.up[g] : ps.u[i];
    double v[3] = {use_pred ? b.vpx[g] : ps.vx[i], use_pred ? b.vpy[g] : ps.vy[i],
                   use_pred ? b.vpz[g] : ps.vz[i]};
    T hinv, rho, omega, P, c;
    // block time-steps: a particle whose step does not end now keeps the h,
    // rho, Omega, P and c of its last solve (restaged here for the force pass)
    const bool keep = b.block_on && ((const T *)b.slev)[s] < T(0);
    if (keep) {
        h = (T)ps.h[i];
        hinv = T(1) / h;
        rho = (T)ps.rho[i];
        omega = (T)ps.omega[i];
        P = (T)ps.P[i];
        c = (T)ps.c[i];
    } else {
        hinv = T(1) / h;
        T hinv3 = hinv * hinv * hinv;
        rho = sigma * S0 * hinv3;
        T drho = -sigma * hinv3 * hinv * (T(3) * S0 + S1);
        omega = T(1) + h / (T(3) * rho) * drho;
        if (ph.eos == SPH_EOS_ISOTHERMAL) {
            c = (T)ph.cs_iso;
            P = c * c * rho;
        } else {
            P = (T)(ph.gamma - 1.0) * rho * (T)u;
            c = sqrt((T)ph.gamma * P / rho);
        }
    }
    T A = P / (omega * rho * rho);
    b.sh[s] = (double)h;
    b.hf[s] = frame_len_ru(h, unit);
    b.srho[s] = (double)rho;
    b.somega[s] = (double)omega;
    b.sP[s] = (double)P;
    b.sc[s] = (double)c;
    if (!keep) {
        ps.h[i] = (double)h;
        ps.rho[i] = (double)rho;
        ps.omega[i] = (double)omega;
        ps.P[i] = (double)P;
        ps.c[i] = (double)c;
    }
    V q;
    q.x = pi.x;
    q.y = pi.y;
    q.z = pi.z;
    q.w = hinv;
    ((V *)b.ph)[s] = q;
    q.x = (T)v[0];
    q.y = (T)v[1];
    q.z = (T)v[2];
    q.w = c;
    ((V *)b.vc)[s] = q;
    q.x = A;
    q.y = rho;
    q.z = pi.w;
    q.w = (T)u;
    ((V *)b.th)[s] = q;
    if (ph.av_switch)  // viscosity switch (Morris & Monaghan's alpha is kicked and predicted like u)
        ((T *)b.sal)[s] = (T)(use_pred && ph.av_switch == SPH_AV_MORRIS_MONAGHAN ? b.ap[g] : ps.alpha[i]);
    if (ph.av_switch == SPH_AV_CULLEN_DEHNEN) ((T *)b.scd)[s] = (T)ps.dalpha[i];  // the previous div v
    // gravity: zeta = dh/drho sum_j m_j dphi/dh = Z / (3 rho h) (Z = sum_j m_j (psi + M/q)),
    // kept as the weight G zeta / (2 Omega) of the force pass's zeta term
    if (ph.gravity) {
        if (keep) {
            ((T *)b.szg)[s] = (T)b.bzeta[g];
        } else {
            const T wz = (T)(0.5 * ph.G) * Z / (T(3) * rho * h * omega);
            ((T *)b.szg)[s] = wz;
            if (b.bzeta) b.bzeta[g] = (double)wz;  // block-step contexts keep it for the ticks that do not solve
        }
    }
    if (!(isfinite((double)rho) && isfinite((double)omega) && isfinite((double)P)))
        atomicOr(&ps.diag->status, ST_NONFINITE);
}

// FP64 density: Newton-Raphson on the FP64 lists in FP32 arithmetic, as far
// as FP32 resolves h, so that the FP64 iteration that follows (same stopping
// rule, FP64 sums) starts within ~1e-7 of the root and needs two passes over
// the list where the previous step's h needs four; h stays as it is where
// it is that close already, or where the FP32 steps leave [0.8, 1.25] of it.
template <int LPP, bool UM, int K, typename T>
__device__ __forceinline__ void presolve_f32(const T *lr, const T *lm, int cnt, bool on, T mi, T mu_all, T eta3, T hs, T &h)
{
    using KF = Kern<K>;
    const int lane = threadIdx.x & 31;
    // the zero is that of S0 - g: one rounding for the constants
    const float g = (float)(mi * eta3 / T(KF::sigma)), mu = (float)mu_all;
    const float h0 = (float)h, hlim = fminf(1.25f * h0, (float)hs * 0.9999f);
    float x = h0, xi_last = 1.f, d_last = 0.f;
    bool go = on, moved = false;
    for (int it = 0; it < 6 && __any_sync(FULL, go); ++it) {
        float S0 = 0.f, S1 = 0.f;
        const float xi = 1.f / x;
        if (go)
            for (int e = 0; e < cnt; ++e) {
                const float q = (float)lr[e * 32 + lane] * xi;
                const float mj = UM ? mu : (float)lm[e * 32 + lane];
                float f, df;
                KF::fdf(q, f, df);
                S0 += mj * f;
                S1 += mj * q * df;
            }
        S0 = group_sum<LPP>(S0);
        S1 = group_sum<LPP>(S1);
        if (go) {
            const float F = S0 - g;
            const float dF = xi * (3.f * (g - S0) - S1);
            const float d = F / dF, xn = dF > 0.f ? x - d : -1.f;
            const float step = fabsf(xn - x);
            if (!(xn >= 0.8f * h0) || !(xn <= hlim)) {
                go = moved = false;
            } else if (it == 0 && step < 1e-5f * x) {
                go = false;
            } else {
                go = step >= 1e-6f * x;
                x = xn;
                xi_last = xi;
                d_last = d;
                moved = true;
            }
        }
    }
    // the last step from the 1/h that the sums used, unrounded: what is left
    // is the sums' rounding (rounding 1/h, h and three constants to FP32 left
    // 1e-14 in h after one FP64 pass, twice that of a longer FP64 iteration)
    if (moved) h = T(1) / (T)xi_last - (T)d_last;
}

// One query leaf of the density pass.  WRAP: pair vectors are wrapped to
// the minimum image where they may miss it (see the wrap helpers).  Returns
// false, having written nothing, when the plain variant meets an ambiguous
// leaf pair.
template <typename T, int LPP, bool UM, int K, bool WRAP>
__device__ __forceinline__ bool density_leaf(const BatchView &b, int leaf, int k0, unsigned char *mine, int use_pred)
{
    using C = DCfg<T, LPP, UM, K>;
    using KF = Kern<K>;
    constexpr float KR_f = (float)KF::R;        // support radius in units of h
    constexpr float KR_cap = KR_f * 1.0001f;    // walk radius -> largest h it covers
    const T sigma = T(KF::sigma);
    using V = typename C::V;
    const int lane = threadIdx.x & 31;
    constexpr bool D64 = C::D64;
    constexpr bool PACK = C::PACK;
    float4 *cand = reinterpret_cast<float4 *>(mine);                     // (not PACK)
    typename C::Cand &cb = *reinterpret_cast<typename C::Cand *>(mine);  // (PACK)
    T *lr = reinterpret_cast<T *>(mine + C::cands);  // r_ij^2 per entry (FP64: r_ij)
    T *lm = lr + (C::LCAP + 1) * 32;  // used only when masses differ
    StageScratch<float> &sc = *reinterpret_cast<StageScratch<float> *>(mine + C::cands + C::lists);
    // FP64: the staged candidates' sorted indices, and the pairs that wait
    int *code = reinterpret_cast<int *>(mine + C::cands + C::lists + C::scratch), *lst = code + C::CH;
    const int pp = lane / LPP, sub = lane % LPP;
    const V *pm = (const V *)b.pm;
    const int p = b.leaf_pid[leaf];
    const ProbStatic &ps = b.prob[p];
    const T mu_all = (T)ps.m_uniform;
    const int st = b.leaf_start[leaf], nA = b.leaf_start[leaf + 1] - st;
    const ProbDyn &dy = b.dyn[p];
    const PhysParams &ph = ps.ph;
    NodeBox boxA = b.nodes[0][leaf];
    int pos;
    const bool active = task_member<T>(b, st, nA, k0, pp, pos);
    const long long s = st + (active ? pos : 0);
    const V pi = pm[s];
    const float4 pf = b.pmf[s];  // (FP32: pi)
    const T mi = pi.w;
    // FP64: the walk's frame and the particle's position
    const double unit = D64 ? frame_of(ph, dy).unit : 1.0;
    const double X[3] = {D64 ? b.sx[s] : 0.0, D64 ? b.sy[s] : 0.0, D64 ? b.sz[s] : 0.0};
    // a block-step task walks from the box of its own particles (the others
    // of the leaf keep their last solve, restaged by k_block_restage)
    if (k0 >= 0) task_box(b, leaf, pf, active, boxA.plo.w, boxA);
    float4 flo, fhi;
    frame_box<float4, float>(pf, active, flo, fhi);
    // (FP64) this lane's largest stage_err since the buffer was last emptied
    const float pmax = D64 ? box_abs(flo, fhi) : 0.f;
    float emax = 0.f;
    const float halfL = ph.periodic ? half_box(ph) : INFINITY;
    const T eta3 = (T)(ph.eta * ph.eta * ph.eta);
    const T tol = (T)ph.h_tol;
    const int maxit = ph.h_max_iter;
    const double Lmin = ph.periodic ? fmin(ph.box_len[0], fmin(ph.box_len[1], ph.box_len[2])) : INFINITY;
    const T hbox = (T)(Lmin / (2.0 * KF::R));  // support beyond half the box: SPH_EBOX
    T h = active ? (T)b.sh[s] : T(1);
    // the leaf pass predicted this particle's sphere from the same start
    const float hpred = active ? __fmul_ru(kHPredict, __double2float_ru(D64 ? b.sh[s] * unit : b.sh[s])) : 0.f;
    if (active && !(h > T(0))) {
        double ext = ph.periodic ? fmax(ph.box_len[0], fmax(ph.box_len[1], ph.box_len[2])) : 1.0 / dy.dom_inv;
        h = (T)(ph.eta * cbrt(ext * ext * ext / (double)(ps.n > 0 ? ps.n : 1)));
    }
    if (ph.periodic) load_box(sc, ph, flo, fhi);
    bool to_wrap = false;  // (plain variant) met an ambiguous leaf pair: the wrapping variant takes the leaf
    T lo = T(0), hi = tinf<T>();
    int it = 0;
    bool conv = !active, fail = false, need = false, noconv = false;
    bool kept = false;  // converged by tolerance: the sums at the returned h are kS0, kS1
    T kS0 = T(0), kS1 = T(0);
    int knn = 0;
    int cnt = 0;
    long long pairs = 0, tested = 0;
    // bal: in-range candidates are dealt to the particle's LPP lanes by
    // their rank among the group's hits instead of by slot, so that the
    // lists fill evenly; taken after a slot-dealt list overflowed
    bool bal = false;
    // candidate-leaf groups of the last walk (lane k holds group k) and
    // the walk radius they cover, kept for the force pass unless the
    // recent records outgrew their h (then the force pass walks)
    const bool record = k0 < 0 && ps.diag->reuse_hold == 0;
    int ng = 0, g_first = 0;
    unsigned g_mask = 0u;
    float Rq_last = 0.f;
    for (int attempt = 0;; ++attempt) {
        const T hs = h * (T)kListMargin;
        const float hsf = frame_len(hs, unit);
        float Rq = warp_max((active && !fail) ? __fmul_ru(KR_f, hsf) : 0.f) * 1.0001f;
        const T R2 = (T(KF::R) * hs) * (T(KF::R) * hs);
        Rq_last = Rq;
        if (!D64 && ph.periodic) set_thr(sc, boxA.slo.w, Rq);
        const bool wrap2 = (WRAP || D64) && half_width(flo, fhi) + Rq >= halfL;  // staged vectors may still need a wrap
        ng = 0;
        cnt = 0;
        int gcnt = 0, at = lane;  // at: where this lane's next entry goes
        int g0 = 0;  // (FP64) waiting entries start at this rank, so that the dealing goes on where it stopped
        const float Rs = KR_f * hsf;
        const float R2t = active && !fail ? (float)R2 : -1.f;  // (FP64: see flush)
        bool ovf = false;
        int nbuf = 0;
        // FP64: the waiting pairs' distances, from the FP64 positions
        auto drain = [&]() {
            __syncwarp();
            const int n = gcnt > sub ? (gcnt - sub - 1) / LPP + 1 : 0;
            for (int e = sub < g0 ? 1 : 0; e < n; ++e) {
                const int j = lst[e * 32 + lane];
                const T dx = (T)min_image_bits(X[0] - b.sx[j], ph.box_len[0], ph.periodic);
                const T dyy = (T)min_image_bits(X[1] - b.sy[j], ph.box_len[1], ph.periodic);
                const T dz = (T)min_image_bits(X[2] - b.sz[j], ph.box_len[2], ph.periodic);
                const T r2 = dx * dx + dyy * dyy + dz * dz;
                if (lt_pos(r2, R2)) {
                    if (cnt < C::LCAP) {
                        lr[cnt * 32 + lane] = sqrt(r2);
                        if (!UM) lm[cnt * 32 + lane] = (T)b.sm[j];
                        ++cnt;
                    } else {
                        ovf = true;
                    }
                }
            }
            g0 = gcnt = gcnt % LPP;
            __syncwarp();
        };
        auto flush = [&]() {
            __syncwarp();  // staged candidates visible to every lane
            if constexpr (D64) {
                // tested in FP32 with the coordinates' error to spare; the hits
                // are dealt to the particle's lanes by rank
                const unsigned below = (1u << sub) - 1u;
                const float Rt = Rs * 1.00001f + 2.f * warp_max(emax);
                const float R2t = active && !fail ? Rt * Rt + kTinySq : -1.f;
                emax = 0.f;
                for (int kb = 0; kb < nbuf; kb += C::SB) {
                    if (__any_sync(FULL, gcnt > C::LC * LPP - C::SB)) drain();
                    const int ke = min(kb + C::SB, nbuf);
#pragma unroll 4
                    for (int kk = kb; kk < ke; kk += LPP) {
                        const int k = kk + sub;
                        bool hit = false;
                        if (k < ke) {
                            const float4 c = cand[k];
                            float dx = pf.x - c.x, dyy = pf.y - c.y, dz = pf.z - c.z;
                            if (wrap2) wrap3s<float>(sc, dx, dyy, dz);
                            hit = dx * dx + dyy * dyy + dz * dz < R2t;
                        }
                        const unsigned gm = (__ballot_sync(FULL, hit) >> (pp * LPP)) & ((1u << LPP) - 1u);
                        if (hit) {
                            const int e = gcnt + __popc(gm & below);
                            lst[(e / LPP) * 32 + pp * LPP + e % LPP] = code[k];
                        }
                        gcnt += __popc(gm);
                    }
                }
            } else if (LPP == 1 || !bal) {
                // (an entry beyond the capacity goes to the spare row: no
                // branch on the append path)
                const int nk = C::Cand::mine(nbuf, sub), at0 = sub * C::Cand::SEC;
                auto append = [&](float r2, float mj) {
                    const int o = min(at, C::LCAP * 32 + lane);
                    if (r2 < R2t) {
                        lr[o] = r2;  // (its root where the lists are read: off the append path)
                        if (!UM) lm[o] = mj;
                        at += 32;
                    }
                };
                auto mass = [&](int k) { return UM ? 0.f : cb.v[C::Cand::NARR - 1][at0 + k]; };
                // (r^2 in the same order of operations on every path of a launch; the
                // launches differ in it only to keep the bits they have had)
                auto dist2 = [](float dx, float dyy, float dz) {
                    return WRAP ? fma_rn(dz, dz, fma_rn(dyy, dyy, mul_rn(dx, dx)))
                                : fma_rn(dz, dz, fma_rn(dx, dx, mul_rn(dyy, dyy)));
                };
                if constexpr (!PACK) {
#pragma unroll 4
                    for (int k = sub; k < nbuf; k += LPP) {
                        const float4 c = cand[k];
                        float dx = pf.x - c.x, dyy = pf.y - c.y, dz = pf.z - c.z;
                        if (wrap2) wrap3s<float>(sc, dx, dyy, dz);
                        append(dist2(dx, dyy, dz), c.w);
                    }
                } else if (wrap2) {
                    for (int k = 0; k < nk; ++k) {
                        float dx = pf.x + cb.v[0][at0 + k], dyy = pf.y + cb.v[1][at0 + k], dz = pf.z + cb.v[2][at0 + k];
                        wrap3s<float>(sc, dx, dyy, dz);
                        append(dist2(dx, dyy, dz), mass(k));
                    }
                } else {
                    cb.pad(nbuf);
                    __syncwarp();
                    const F2 px = pack2(pf.x, pf.x), py = pack2(pf.y, pf.y), pz = pack2(pf.z, pf.z);
                    for (int k = 0; k < nk; k += 4) {
                        const float4 x = ld4(cb.v[0] + at0 + k), y = ld4(cb.v[1] + at0 + k), z = ld4(cb.v[2] + at0 + k);
#pragma unroll
                        for (int h2 = 0; h2 < 2; ++h2) {
                            const F2 dx = px + (h2 ? pack2(x.z, x.w) : pack2(x.x, x.y));
                            const F2 dyy = py + (h2 ? pack2(y.z, y.w) : pack2(y.x, y.y));
                            const F2 dz = pz + (h2 ? pack2(z.z, z.w) : pack2(z.x, z.y));
                            float ra, rb;
                            unpack2(fma2(dz, dz, WRAP ? fma2(dyy, dyy, dx * dx) : fma2(dx, dx, dyy * dyy)), ra, rb);
                            append(ra, mass(k + 2 * h2));
                            append(rb, mass(k + 2 * h2 + 1));
                        }
                    }
                }
            } else {
                const unsigned below = (1u << sub) - 1u;
                for (int k0 = 0; k0 < nbuf; k0 += LPP) {
                    const int k = k0 + sub;
                    bool hit = false;
                    T r = T(0), mj = T(0);  // (r: r_ij^2)
                    if (k < nbuf) {
                        float4 q;
                        if constexpr (PACK) {
                            const int c = C::Cand::place(k);
                            q = make_float4(-cb.v[0][c], -cb.v[1][c], -cb.v[2][c], UM ? 0.f : cb.v[C::Cand::NARR - 1][c]);
                        } else {
                            q = cand[k];
                        }
                        float dx = pf.x - q.x, dyy = pf.y - q.y, dz = pf.z - q.z;
                        if (wrap2) wrap3s<float>(sc, dx, dyy, dz);
                        const float r2 = dx * dx + dyy * dyy + dz * dz;
                        hit = r2 < R2t;
                        r = r2;
                        mj = q.w;
                    }
                    const unsigned gm = (__ballot_sync(FULL, hit) >> (pp * LPP)) & (LPP == 32 ? FULL : (1u << (LPP & 31)) - 1u);
                    if (hit) {
                        const int e = gcnt + __popc(gm & below);
                        if (e < C::LCAP * LPP) {
                            const int o = (e / LPP) * 32 + pp * LPP + e % LPP;
                            lr[o] = r;
                            if (!UM) lm[o] = mj;
                        } else {
                            ovf = true;
                        }
                    }
                    gcnt += __popc(gm);
                }
            }
            tested += (nbuf - sub + LPP - 1) / LPP;
            __syncwarp();
            nbuf = 0;
        };
        const float Rq2 = Rq * Rq;
        set_query(sc.qb, boxA.plo, boxA.phi, Rq, ph, coord_bound<D64>(ph, dy));
        // visit leaves within Rq (gather) or whose predicted smoothing
        // spheres reach this leaf (what the force pass will need); stage
        // only the former
        bool near = false;  // this lane's last tested node is within Rq
        Walk wk;
        wk.start(dy);
        for (;;) {
            const int node = wk.next(b, dy, [&](const NodeBox &nb) {
                return up_within(sc.qb, nb) || (record && up_overlap(sc.qb, nb));
            });
            if (node < 0) break;
            const int first = dy.node_off[0] + node * kBranch;
            const bool in = (leaf_lanes(dy.node_cnt[0], node) >> lane) & 1u;
            const NodeBox &nb = b.nodes[0][first + (in ? lane : 0)];
            near = box_within(sc.qb, nb, ph);
            const unsigned mask = __ballot_sync(FULL, (record ? box_overlap(sc.qb, nb, ph) || near : near) && in);
            if (mask == 0u) continue;
            if (lane == ng) {
                g_first = first;
                g_mask = mask;
            }
            ++ng;
            // the leaf-level tests just made: stage the leaves within Rq
            const unsigned gm = __ballot_sync(FULL, near && ((mask >> lane) & 1u));
            if (gm == 0u) continue;
            // candidate leaves that form an ambiguous pair with A (periodic)
            // (FP64 takes its pairs' minimum images from the positions: every
            // staged candidate moves to its image nearest the query box)
            const unsigned am =
                !D64 && ph.periodic ? __ballot_sync(FULL, ((gm >> lane) & 1u) && ambiguous(b.nodes[0][first + lane].slo.w, sc))
                                    : 0u;
            if (!WRAP && am) to_wrap = true;
            if (!WRAP && to_wrap) break;
            const unsigned amo = WRAP ? by_order(am, gm) : 0u;
            stage_group<float, C::CH, D64>(
                b, leaf, gm, first, ph, unit, nbuf, sc, [](bool, int, int, int, const float4 &) {},
                [&](int j) {
                    float4 q = b.pmf[j];
                    if (D64) q.w = __int_as_float(j);
                    return q;
                },
                [&](float4 &q, int o) {
                    const float aq = D64 ? abs3(q) : 0.f;
                    if (D64 ? ph.periodic != 0 : WRAP && ((amo >> o) & 1u))
                        wrap_near<float>(sc, q, sc.C[0], sc.C[1], sc.C[2]);
                    const float d2 = box_dist2<float>(q, flo, fhi);
                    if constexpr (D64) {
                        const float e = stage_err(abs3(sc.leaf[o]), aq, abs3(q), pmax), Rt = Rq + 2.f * e;
                        if (!(d2 < Rt * Rt + kTinySq)) return false;
                        emax = fmaxf(emax, e);
                        return true;
                    }
                    return d2 < Rq2;
                },
                [&](int slot, const float4 &q, int, int) {
                    if constexpr (!PACK) {
                        cand[slot] = q;
                        if (D64) code[slot] = __float_as_int(q.w);
                    } else {
                        const int c = C::Cand::place(slot);
                        cb.v[0][c] = -q.x;
                        cb.v[1][c] = -q.y;
                        cb.v[2][c] = -q.z;
                        if (!UM) cb.v[C::Cand::NARR - 1][c] = q.w;
                    }
                },
                flush);
        }
        flush();
        if (D64) drain();
        if (!WRAP && to_wrap) break;
        if (D64) {
        } else if (LPP == 1 || !bal) {
            cnt = at >> 5;
            ovf = cnt > C::LCAP;
            cnt = min(cnt, C::LCAP);
        }
        if (!D64 && LPP > 1 && bal) {
            const int mine_n = gcnt > sub ? (gcnt - sub - 1) / LPP + 1 : 0;
            cnt = mine_n < C::LCAP ? mine_n : C::LCAP;
        }
        if (!D64 && LPP > 1 && !bal && __any_sync(FULL, ovf)) {
            bal = true;  // same radius again, dealt by rank
            --attempt;
            continue;
        }
        if (group_any<LPP>(ovf) && active && !fail) fail = true;
        if constexpr (D64)
            if (attempt == 0 && maxit >= 16 && tol < T(1e-9)) presolve_f32<LPP, UM, K>(lr, lm, cnt, active && !fail, mi, mu_all, eta3, hs, h);
        // Newton-Raphson on the cached lists
        for (;;) {
            bool go = active && !conv && !fail && !need;
            if (!__any_sync(FULL, go)) break;
            T S0 = T(0), S1 = T(0);
            int nn = 0;
            if (go) {
                const T hinv = T(1) / h;
                for (int e = 0; e < cnt; ++e) {
                    T q = (D64 ? lr[e * 32 + lane] : sqrt(lr[e * 32 + lane])) * hinv;
                    T mj = UM ? mu_all : lm[e * 32 + lane];
                    T f, df;
                    KF::fdf(q, f, df);
                    S0 += mj * f;
                    S1 += mj * q * df;
                    nn += lt_pos(q, T(KF::R));
                }
            }
            S0 = group_sum<LPP>(S0);
            S1 = group_sum<LPP>(S1);
            nn = group_sum<LPP>(nn);
            if (go) {
                ++it;
                if (sub == 0) pairs += nn;
                T hinv = T(1) / h;
                T hinv3 = hinv * hinv * hinv;
                T rho = sigma * S0 * hinv3;
                T drho = -sigma * hinv3 * hinv * (T(3) * S0 + S1);
                bool c = nr_update(h, lo, hi, rho, drho, mi, eta3, tol);
                if (c) {
                    kept = true;
                    kS0 = S0;
                    kS1 = S1;
                    knn = nn;
                }
                if (h > hbox) {
                    atomicOr(&ps.diag->status, ST_BOX);
                    c = true;
                    kept = false;
                }
                if (!c && it >= maxit) {
                    noconv = true;
                    c = true;
                }
                conv = c;
                if (h > hs) need = true;
            }
        }
        if (!__any_sync(FULL, need)) break;
        if (attempt + 1 >= kMaxRebuild) {
            if (need) fail = true;
            break;
        }
        need = false;
    }
    if (!WRAP && to_wrap) return false;  // nothing written yet
    // record the last walk's groups for the force pass (lane 0 reserves
    // pool space); not recorded: the force pass walks for this leaf (a
    // block-step task records nothing: its force pass always walks)
    if (k0 < 0) {
        int base = 0;
        if (lane == 0) {
            base = record && ng <= kMaxLeafGroups ? atomicAdd(&b.counters[kPoolCounter], ng) : -1;
            const bool fits = base >= 0 && (long long)base + ng <= b.group_cap;
            b.leaf_gofs[leaf] = fits ? base : 0;
            b.leaf_ngroups[leaf] = fits ? ng : -1;
            b.leaf_hcap[leaf] = Rq_last / KR_cap;
            base = fits ? base : -1;
        }
        base = __shfl_sync(FULL, base, 0);
        if (base >= 0 && lane < ng) b.group_pool[base + lane] = make_int2(g_first, (int)g_mask);
    }
    // final evaluation at the returned h, unless the sums there are kept
    T S0 = kS0, S1 = kS1;
    int nn = knn;
    const bool fin = active && !fail;
    const bool redo = fin && !kept;
    if (__any_sync(FULL, redo)) {
        T R0 = T(0), R1 = T(0);
        int rn = 0;
        if (redo) {
            const T hinv = T(1) / h;
            for (int e = 0; e < cnt; ++e) {
                T q = (D64 ? lr[e * 32 + lane] : sqrt(lr[e * 32 + lane])) * hinv;
                T mj = UM ? mu_all : lm[e * 32 + lane];
                T f, df;
                KF::fdf(q, f, df);
                R0 += mj * f;
                R1 += mj * q * df;
                rn += lt_pos(q, T(KF::R));
            }
        }
        R0 = group_sum<LPP>(R0);
        R1 = group_sum<LPP>(R1);
        rn = group_sum<LPP>(rn);
        if (redo) {
            S0 = R0;
            S1 = R1;
            nn = rn;
            if (sub == 0) pairs += rn;
        }
    }
    T Z = T(0);  // gravity (wrap-list launch): sum_j m_j (psi + M/q) at the final h
    if (WRAP && ph.gravity) {
        if (fin) {
            const T hinv = T(1) / h;
            for (int e = 0; e < cnt; ++e)
                Z += (UM ? mu_all : lm[e * 32 + lane]) * grav_psi_plus_mq((D64 ? lr[e * 32 + lane] : sqrt(lr[e * 32 + lane])) * hinv);
        }
        Z = group_sum<LPP>(Z);
    }
    if (fin && sub == 0) {
        density_epilogue<T>(b, ps, s, pi, h, S0, S1, use_pred, sigma, unit, Z);
        if (noconv && !(b.block_on && ((const T *)b.slev)[s] < T(0))) {  // (a kept solve is not this one)
            atomicOr(&ps.diag->status, ST_NOCONV);
            atomicAdd(&ps.diag->unconverged, 1);
        }
        // the recorded candidate groups cover this particle's pairs only
        // if its final h stays within the walk radius and its prediction
        const float hf = frame_len_ru(h, unit);
        if (hf > hpred || hf > Rq_last / KR_cap) atomicOr(&b.dyn[p].lists_stale, 1);
    }
    if (active && fail && sub == 0) {
        int k = atomicAdd(&b.counters[kSlowCounter], 1);
        b.fallback_list[k] = (int)s;
        b.sh[s] = (double)h;  // best guess so far
        b.hf[s] = hpred;      // for the slow path's coverage check
    }
    // statistics (one atomic per warp per quantity)
    long long tp = warp_sum(pairs), tt = warp_sum(tested);
    int itn = (fin && sub == 0) ? it : 0;
    long long its = warp_sum((long long)itn);
    int itmax = warp_max(itn);
    int nmin = warp_min((fin && sub == 0) ? nn : 0x7fffffff);
    int nmax = warp_max((fin && sub == 0) ? nn : 0);
    long long nsum = warp_sum((long long)((fin && sub == 0) ? nn : 0));
    if (lane == 0) {
        ProbDiag *dg = ps.diag;
        atomicAdd((unsigned long long *)&dg->density_pairs, (unsigned long long)tp);
        atomicAdd((unsigned long long *)&dg->candidates, (unsigned long long)tt);
        atomicAdd((unsigned long long *)&dg->nr_iter, (unsigned long long)its);
        atomicAdd((unsigned long long *)&dg->ngb_sum, (unsigned long long)nsum);
        atomicMax(&dg->nr_max, itmax);
        if (nmax > 0) {
            atomicMin(&dg->ngb_min, nmin);
            atomicMax(&dg->ngb_max, nmax);
        }
    }
    return true;
}

// WRAP: the launch that serves the wrap list (leaves whose pair vectors may
// miss the minimum image); the other launch puts them there.
template <typename T, int LPP, bool UM, int K, bool WRAP>
__global__ void __launch_bounds__(DCfg<T, LPP, UM, K>::WPB * 32, DCfg<T, LPP, UM, K>::MINB) k_density(BatchView b, int use_pred)
{
    chain_entry();
    using C = DCfg<T, LPP, UM, K>;
    extern __shared__ __align__(32) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char *mine = smem + wib * C::per_warp;
    // block-step ticks: the wrap-list launch serves the tick's tasks (leaf <<
    // 5 | first due ordinal) directly; the common launch does not run
    const bool tasks = WRAP && b.block_on && b.block_tasks;
    const int nleaf = tasks ? b.counters[kBlockTasks] : WRAP ? b.counters[kDensWrapList] : b.counters[0];
    const int cls = lpp_log2(LPP) + (UM ? 4 : 0) + 8 * K;
    for (int item = first_item();; item = next_item(&b.counters[(WRAP ? kDensityWrapCounter : kDensityCounter) + cls])) {
        if (item >= nleaf) break;
        const int what = !WRAP ? item : tasks ? b.btask[item] : b.wrap_list[item];
        const int leaf = tasks ? what >> 5 : what, k0 = tasks ? what & 31 : -1;
        const ProbStatic &ps = b.prob[b.leaf_pid[leaf]];
        if ((tasks ? b.block_lanes : ps.lpp) != LPP || (ps.uniform_m != 0) != UM || ps.ph.kernel != K) continue;
        if (!WRAP && ps.ph.gravity) {  // gravity's zeta runs in the wrap-list launch only
            if (lane == 0) b.wrap_list[atomicAdd(&b.counters[kDensWrapList], 1)] = leaf;
            continue;
        }
        if (!density_leaf<T, LPP, UM, K, WRAP>(b, leaf, k0, mine, use_pred) && lane == 0) {
            b.wrap_list[atomicAdd(&b.counters[kDensWrapList], 1)] = leaf;
            atomicAdd(&ps.diag->wrap_leaves, 1);
        }
    }
}

// Slow path: one warp per particle for the particles whose per-lane lists in
// k_density overflowed or outgrew their radius.  The warp stages the leaf's
// candidate leaves in groups, as k_density does, gathers the particle's
// neighbours (within R_K h x 1.1) into a list spread over its 32 lanes (up to
// kFbPerLane each) and iterates on it, walking the tree again only when h
// outgrows the list; if even that list overflows, every iteration walks the
// tree and sums the staged candidates directly.
constexpr int kFbPerLane = 24;
constexpr int kFbCH = 128;
constexpr double kFbMargin = 1.1;

template <typename T>
struct FbCfg {
    using V = typename Vec4<T>::type;
    static constexpr int WPB = 4;
    static constexpr size_t scratch = (sizeof(StageScratch<T>) + 31) & ~(size_t)31;
    static constexpr size_t per_warp = kFbCH * sizeof(V) + (size_t)2 * kFbPerLane * 32 * sizeof(T) + scratch;
    static constexpr size_t smem = WPB * per_warp;
};

template <typename T>
__global__ void __launch_bounds__(FbCfg<T>::WPB * 32) k_density_fallback(BatchView b, int use_pred)
{
    chain_entry();
    using C = FbCfg<T>;
    using V = typename C::V;
    extern __shared__ __align__(32) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char *mine = smem + wib * C::per_warp;
    V *cand = reinterpret_cast<V *>(mine);
    T *fr = reinterpret_cast<T *>(mine + kFbCH * sizeof(V));
    T *fm = fr + kFbPerLane * 32;
    StageScratch<T> &sc = *reinterpret_cast<StageScratch<T> *>(fm + kFbPerLane * 32);
    const int nf = b.counters[kSlowCounter];
    const V *pm = (const V *)b.pm;
    int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int k = w; k < nf; k += nw) {
        const long long s = b.fallback_list[k];
        const int leaf = (int)b.flag[s] - 1;
        const int p = b.leaf_pid[leaf];
        const ProbStatic &ps = b.prob[p];
        const ProbDyn &dy = b.dyn[p];
        const PhysParams &ph = ps.ph;
        const NodeBox boxA = b.nodes[0][leaf];
        constexpr bool D64 = sizeof(T) == 8;  // (the walk in its frame, the staged positions as they are)
        const double unit = D64 ? frame_of(ph, dy).unit : 1.0;
        const V pi = pm[s];
        const T eta3 = (T)(ph.eta * ph.eta * ph.eta);
        const T tol = (T)ph.h_tol;
        double Lmin = ph.periodic ? fmin(ph.box_len[0], fmin(ph.box_len[1], ph.box_len[2])) : INFINITY;
        const int kk = ph.kernel;
        const T KR = (T)ph.kr, sigma = (T)kern_sigma(kk);
        const bool per = ph.periodic != 0;  // (every staged candidate moves to its image nearest s)
        if (per) load_box(sc, ph, pi, pi);
        T h = (T)b.sh[s];
        T lo = T(0), hi = tinf<T>();
        int it = 0;
        bool conv = false, noconv = false;
        long long pairs = 0;
        T S0, S1;
        int nn;
        // every particle within the support R_K hh of particle s, staged in
        // groups of leaves; fn(r2, m_j) sees one candidate per lane
        auto visit_all = [&](T hh, auto &&fn) {
            const float Rq = __fmul_ru(ph.kr_f, frame_len(hh, unit)) * 1.0001f;
            const T Rt = D64 ? KR * hh * T(1.0001) : (T)Rq, Rq2 = Rt * Rt;
            set_query(sc.qb, boxA.plo, boxA.phi, Rq, ph, coord_bound<D64>(ph, dy));
            int nbuf = 0;
            auto flush = [&]() {
                __syncwarp();
                for (int e = lane; e < nbuf; e += 32) {
                    const V c = cand[e];
                    T dx = pi.x - c.x, dyy = pi.y - c.y, dz = pi.z - c.z;
                    fn(dx * dx + dyy * dyy + dz * dz, c.w);
                }
                __syncwarp();
                nbuf = 0;
            };
            Walk wk;
            wk.start(dy);
            for (;;) {
                const int node = wk.next(b, dy, [&](const NodeBox &nb) { return up_within(sc.qb, nb); });
                if (node < 0) break;
                const int first = dy.node_off[0] + node * kBranch;
                const bool in = (leaf_lanes(dy.node_cnt[0], node) >> lane) & 1u;
                const unsigned mask = __ballot_sync(FULL, box_within(sc.qb, b.nodes[0][first + (in ? lane : 0)], ph) && in);
                if (mask)
                    stage_group<T, kFbCH>(
                        b, leaf, mask, first, ph, unit, nbuf, sc, [](bool, int, int, int, const V &) {},
                        [&](int j) { return pm[j]; },
                        [&](V &q, int) {
                            if (per) wrap_near<T>(sc, q, pi.x, pi.y, pi.z);  // then pi - q is the minimum image
                            return box_dist2<T>(q, pi, pi) < Rq2;
                        },
                        [&](int slot, const V &q, int, int) { cand[slot] = q; }, flush);
            }
            flush();
        };
        bool direct = false;
        T hs = T(0);
        int cnt = 0;
        auto build = [&]() {
            hs = h * (T)kFbMargin;
            const T R2 = (KR * hs) * (KR * hs);
            cnt = 0;
            bool ovf = false;
            visit_all(hs, [&](T r2, T mj) {
                if (r2 < R2) {
                    if (cnt < kFbPerLane) {
                        fr[cnt * 32 + lane] = sqrt(r2);
                        fm[cnt * 32 + lane] = mj;
                        ++cnt;
                    } else {
                        ovf = true;
                    }
                }
            });
            direct = __any_sync(FULL, ovf);
            __syncwarp();
        };
        T Z = T(0);  // gravity: sum_j m_j (psi + M/q)
        auto sums = [&](T hh) {
            S0 = T(0);
            S1 = T(0);
            Z = T(0);
            nn = 0;
            const T hinv = T(1) / hh;
            if (!direct) {
                for (int e = 0; e < cnt; ++e) {
                    T f, df, qq = fr[e * 32 + lane] * hinv;
                    kern_fdf(kk, qq, f, df);
                    T mj = fm[e * 32 + lane];
                    S0 += mj * f;
                    S1 += mj * qq * df;
                    if (ph.gravity) Z += mj * grav_psi_plus_mq(qq);
                    nn += qq < KR;
                }
            } else {
                const T R2 = (KR * hh) * (KR * hh);
                visit_all(hh, [&](T r2, T mj) {
                    if (r2 < R2) {
                        T f, df, qq = sqrt(r2) * hinv;
                        kern_fdf(kk, qq, f, df);
                        S0 += mj * f;
                        S1 += mj * qq * df;
                        if (ph.gravity) Z += mj * grav_psi_plus_mq(qq);
                        ++nn;
                    }
                });
            }
            S0 = warp_sum(S0);
            S1 = warp_sum(S1);
            Z = warp_sum(Z);
            nn = warp_sum(nn);
        };
        build();
        while (!conv) {
            if (!direct && h > hs) build();
            sums(h);
            ++it;
            pairs += nn;
            T hinv = T(1) / h;
            T hinv3 = hinv * hinv * hinv;
            T rho = sigma * S0 * hinv3;
            T drho = -sigma * hinv3 * hinv * (T(3) * S0 + S1);
            bool c = nr_update(h, lo, hi, rho, drho, pi.w, eta3, tol);
            if ((double)h > Lmin / (2.0 * ph.kr)) {
                if (lane == 0) atomicOr(&ps.diag->status, ST_BOX);
                c = true;
            }
            if (!c && it >= ph.h_max_iter) {
                noconv = true;
                c = true;
            }
            conv = c;
        }
        if (!direct && h > hs) build();
        sums(h);
        pairs += nn;
        if (lane == 0) {
            const float hf = frame_len_ru(h, unit);
            if (hf > b.hf[s] || hf > b.leaf_hcap[leaf]) atomicOr(&b.dyn[p].lists_stale, 1);
            density_epilogue<T>(b, ps, s, pi, h, S0, S1, use_pred, sigma, unit, Z);
            if (noconv) {
                atomicOr(&ps.diag->status, ST_NOCONV);
                atomicAdd(&ps.diag->unconverged, 1);
            }
            ProbDiag *dg = ps.diag;
            atomicAdd((unsigned long long *)&dg->density_pairs, (unsigned long long)pairs);
            atomicAdd((unsigned long long *)&dg->nr_iter, (unsigned long long)it);
            atomicAdd((unsigned long long *)&dg->fallback, 1ull);
            atomicAdd((unsigned long long *)&dg->ngb_sum, (unsigned long long)nn);
            atomicMax(&dg->nr_max, it);
            atomicMin(&dg->ngb_min, nn);
            atomicMax(&dg->ngb_max, nn);
        }
    }
}

// ---------------------------------------------------------------------------
// forces
// ---------------------------------------------------------------------------
// Force walk: the staged candidates (CH per chunk) are tested against the
// lane's particle and each pair found is appended to the lane's list as a
// 16-bit code (slot of its leaf in the warp's table of candidate leaves << 5 |
// index within that leaf); the lists are evaluated, reading the partner's
// data from global memory, when one of them or the table fills and at the end,
// so that every lane evaluates about the same number of pairs.
template <typename T, int LPP, int K>
struct FCfg {
    using V = typename Vec4<T>::type;
    static constexpr int CH = SPH_FORCE_CH;
    static constexpr bool D64 = sizeof(T) == 8;
    // list entries per lane, and candidates tested per list-room check: at
    // one lane per particle a lane holds all of its particle's ~60 pairs
    static constexpr int LC = LPP == 1 ? SPH_FORCE_LC1 : SPH_FORCE_LC;
    static constexpr int SB = LPP == 1 ? SPH_FORCE_SB1 : SPH_FORCE_SB;
    static constexpr int TAB = D64 ? 0 : SPH_FORCE_TAB;  // candidate leaves per table fill (<= 2048)
    static constexpr int WPB = D64 ? 2 : 4;
    static constexpr int MINB = D64 ? 4 : K == SPH_KERNEL_M6 ? SPH_MINB_M6 : LPP == 1 ? SPH_FORCE_MINB1 : SPH_FORCE_MINB;  // blocks per SM the registers allow
    using Code = std::conditional_t<D64, int, unsigned short>;  // (FP64: the sorted index itself)
    static constexpr size_t scratch = (sizeof(StageScratch<float>) + 31) & ~(size_t)31;
    // (two lanes per particle: Sod 36864 71.7 -> 67.6 us; at one, where five
    // blocks leave 96 registers, the packed form was 10 % slower)
    static constexpr bool PACK = !D64 && K == SPH_KERNEL_M4 && LPP == 2;
    using Cand = CandBuf<CH, LPP, 4>;  // (PACK: -x, -y, -z, 1/h)
    static constexpr int NCODE = PACK ? Cand::SEC * LPP : CH;  // (codes are placed as the candidates)
    static constexpr size_t cands = PACK ? (Cand::bytes + 31) & ~(size_t)31 : CH * sizeof(float4);
    static constexpr size_t codes = ((size_t)(NCODE + LC * 32) * sizeof(Code) + 31) & ~(size_t)31;
    static_assert(TAB <= 2048 && LC >= 2 * SB / LPP, "force list layout");
    static_assert(!PACK || SB / LPP % 4 == 0, "the tests take whole fours between room checks");
    static constexpr size_t per_warp = cands + TAB * sizeof(float4) + scratch + codes;
    static constexpr size_t smem = WPB * per_warp;
};

// Compensated sum with an error-free transformation per addition (Knuth's
// branch-free TwoSum): s + c carries the exact running sum to O(n eps^2),
// whatever the signs and magnitudes of the terms.
template <typename T>
struct TwoSumAcc {
    T s, c;
    __device__ __forceinline__ void add(T x)
    {
        T t = add_rn(s, x);
        T xp = t - s;
        T sp = t - xp;
        T e = (s - sp) + (x - xp);
        c = c + e;
        s = t;
    }
};

// two TwoSumAcc at once (packed FP32)
struct TwoSumAcc2 {
    F2 s, c;
    __device__ __forceinline__ void add(F2 x)
    {
        const F2 t = s + x, xp = t - s, sp = t - xp;
        c = c + ((s - sp) + (x - xp));
        s = t;
    }
};

template <typename T>
struct ForceSum {
    TwoSumAcc<T> x{T(0), T(0)}, y{T(0), T(0)}, z{T(0), T(0)};
    __device__ __forceinline__ void add(T w, T rx, T ry, T rz)
    {
        x.add(mul_rn(w, rx));
        y.add(mul_rn(w, ry));
        z.add(mul_rn(w, rz));
    }
    __device__ __forceinline__ void get(double &fx, double &fy, double &fz) const
    {
        fx = (double)x.s + (double)x.c;
        fy = (double)y.s + (double)y.c;
        fz = (double)z.s + (double)z.c;
    }
};
template <>
struct ForceSum<float> {
    TwoSumAcc2 xy;
    TwoSumAcc<float> z{0.f, 0.f};
    __device__ __forceinline__ ForceSum() : xy{pack2(0.f, 0.f), pack2(0.f, 0.f)} {}
    __device__ __forceinline__ void add(float w, float rx, float ry, float rz)
    {
        xy.add(pack2(w, w) * pack2(rx, ry));
        z.add(mul_rn(w, rz));
    }
    __device__ __forceinline__ void get(double &fx, double &fy, double &fz) const
    {
        float s[2], c[2];
        unpack2(xy.s, s[0], s[1]);
        unpack2(xy.c, c[0], c[1]);
        fx = (double)s[0] + (double)c[0];
        fy = (double)s[1] + (double)c[1];
        fz = (double)z.s + (double)z.c;
    }
};

// conductivity signal speed (Sec. 2.1.1): Wadsley |v_ij . r_hat| (gm1 = 0)
// or Price sqrt(|P_i - P_j| / rho_bar), P = gm1 rho u from the staged
// (A, rho, m, u) vectors
template <typename T, typename V>
__device__ __forceinline__ T ac_speed(T vdr, const V &ti, const V &tj, T gm1, T rhob_inv)
{
    if (gm1 > T(0)) return sqrt(gm1 * fabs(ti.y * ti.w - tj.y * tj.w) * rhob_inv);
    return fabs(vdr);
}

template <typename V>
__device__ __forceinline__ V ld_ro(const V *p);
template <>
__device__ __forceinline__ float4 ld_ro<float4>(const float4 *p) { return __ldg(p); }
template <>
__device__ __forceinline__ dbl4 ld_ro<dbl4>(const dbl4 *p)
{
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p));
    const double2 c = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    dbl4 v;
    v.x = a.x;
    v.y = a.y;
    v.z = c.x;
    v.w = c.y;
    return v;
}

// One query leaf of the force pass.  Rall: the reach of the problem's pairs,
// R_K x its largest h (periodic problems); WRAP: the leaf is on the wrap
// list and its pair vectors are wrapped where they may miss the minimum
// image.  Returns false (writing nothing) when the plain launch meets an
// ambiguous leaf pair.
template <typename T, int LPP, int K, bool WRAP, bool CD>
__device__ __forceinline__ bool force_leaf(const BatchView &b, int leaf, int k0, unsigned char *mine, float Rall)
{
    using C = FCfg<T, LPP, K>;
    using KF = Kern<K>;
    constexpr float KR_f = (float)KF::R;
    using V = typename C::V;
    const int lane = threadIdx.x & 31;
    constexpr bool D64 = C::D64;
    constexpr bool PACK = C::PACK;
    float4 *cand = reinterpret_cast<float4 *>(mine);  // staged (offset + leaf shift, 1/h; FP64: R_K h)
    typename C::Cand &cb = *reinterpret_cast<typename C::Cand *>(mine);   // (PACK)
    float4 *table = reinterpret_cast<float4 *>(mine + C::cands);  // per candidate leaf: (leaf shift, first sorted index)
    StageScratch<float> &sc = *reinterpret_cast<StageScratch<float> *>(table + C::TAB);
    using Code = typename C::Code;
    Code *code = reinterpret_cast<Code *>(mine + C::cands + C::TAB * sizeof(float4) + C::scratch);
    Code *lst = code + C::NCODE;
    const int pp = lane / LPP, sub = lane % LPP;
    const V *gph = (const V *)b.ph, *gvc = (const V *)b.vc, *gth = (const V *)b.th;
    const int p = b.leaf_pid[leaf];
    const ProbStatic &ps = b.prob[p];
    const int st = b.leaf_start[leaf], nA = b.leaf_start[leaf + 1] - st;
    const ProbDyn &dy = b.dyn[p];
    const PhysParams &ph = ps.ph;
    NodeBox boxA = b.nodes[0][leaf];
    int pos;
    const bool active = task_member<T>(b, st, nA, k0, pp, pos);
    const int s = st + (active ? pos : 0);
    const V xi = gph[s], vi = gvc[s], ti = gth[s];
    // the walk's copy of the particle, its membership data (FP64: R_K h) and its position
    float4 xf;
    if constexpr (D64) {
        xf = b.pmf[s];
        xf.w = __fmul_ru(KR_f, b.hf[s]);
    } else {
        xf = xi;
    }
    const double unit = D64 ? frame_of(ph, dy).unit : 1.0;
    const double X[3] = {D64 ? b.sx[s] : 0.0, D64 ? b.sy[s] : 0.0, D64 ? b.sz[s] : 0.0};
    // a block-step task walks from the box of its own particles, whose
    // largest h sets the gather reach
    if (k0 >= 0) task_box(b, leaf, xf, active, warp_max(active ? b.hf[s] : 0.f), boxA);
    const T alpha = (T)ph.alpha_av, beta = (T)ph.beta_av, aac = (T)ph.alpha_ac;
    // Price conductivity: v'_sig = sqrt(|P_i - P_j| / rho_bar) with P = (gamma - 1) rho u
    // (adiabatic); 0 selects Wadsley's |v_ij . r_hat|
    const T gm1_price = WRAP && ph.ac_signal == SPH_AC_PRICE ? (T)(ph.gamma - 1.0) : T(0);
    const bool adi = ph.eos == SPH_EOS_ADIABATIC;
    const T sigma = T(KF::sigma);
    const T hi2 = mul_rn(xi.w, xi.w), hi4 = mul_rn(hi2, hi2);
    // viscosity switch (served by the wrap-list launch): alpha_ij = (alpha_i + alpha_j)/2,
    // beta_ij = beta/alpha_max alpha_ij
    const bool sw = WRAP && ph.av_switch != 0;
    const T* __restrict__ sal = (const T *)b.sal;
    const T alpha_i = sw ? sal[s] : alpha, bratio = (T)ph.beta_ratio;
    T dvs = T(0);  // sum_j m_j v_ij . grad_i W(h_i) (switch: div v)
    // Cullen & Dehnen (its own launch, so that the other options keep their
    // registers): the gradient sums G_ab = sum_j m_j v_ij,a grad_i,b W(h_i)
    // and the signed density sum_j sign(D_j) m_j W(r_ij, h_i)
    constexpr bool cdw = CD;
    const T* __restrict__ scd = (const T *)b.scd;
    T cg[9] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
    T cr = T(0);
    // gravity (wrap-list launch): the zeta term of Eq. SPHSELFGRAV has the pressure
    // term's form, with P/(Omega rho^2) + G zeta/(2 Omega) per particle
    const bool grav = WRAP && ph.gravity != 0;
    const T* __restrict__ szg = (const T *)b.szg;
    const T Ai_g = grav ? add_rn(ti.x, szg[s]) : ti.x;
    // block time-steps (wrap-list launch): only the particles whose step ends
    // now (staged level + 1 > 0) take forces; they record the largest level
    // among their neighbours and lift inactive neighbours more than
    // block_gap levels below them (Saitoh & Makino's limiter)
    const bool blk = WRAP && b.block_on;
    const T* __restrict__ slev = (const T *)b.slev;
    const T li1 = blk ? slev[s] : T(0);
    const bool due = blk ? (active && li1 > T(0)) : active;
    if (blk && !__any_sync(FULL, due)) return true;  // no particle of this leaf ends its step now
    const T lgap = (T)ph.block_gap;
    T mlev = T(0);
    // the sums of m_i a_i; x and y together in packed FP32 (additions only, so
    // the same bits)
    ForceSum<T> acc;
    T du = T(0), vs = T(-1);
    int pairs = 0, tested = 0;
    const float R = __fmul_ru(KR_f, boxA.plo.w) * 1.0001f;
    const float RA2 = R * R;
    float4 flo, fhi;
    frame_box<float4, float>(xf, active, flo, fhi);
    // (FP64) this lane's largest stage_err since the buffer was last emptied
    const float pmax = D64 ? box_abs(flo, fhi) : 0.f;
    float emax = 0.f;
    const float halfL = ph.periodic ? half_box(ph) : INFINITY;
    if (ph.periodic) {
        load_box(sc, ph, flo, fhi);
        if (!D64) set_thr(sc, boxA.slo.w, Rall);
    }
    const bool wrap2 = (WRAP || D64) && half_width(flo, fhi) + Rall >= halfL;  // staged vectors may still need a wrap
    bool to_wrap = false;  // (plain variant) met an ambiguous leaf pair: the wrapping variant takes the leaf
    int nbuf = 0, cnt = 0, ntab = 0, tA = -1, gcnt = 0;  // gcnt (FP64): hits dealt to the particle's lanes
    unsigned am = 0u;
    // table entry of a candidate leaf: its shift and first sorted index,
    // stored as ~index for an ambiguous leaf pair (whose pair vectors the
    // evaluation wraps)
    auto fetch = [&](int e, T &rx, T &ry, T &rz, T &hinv_j, V &a1, V &a2, int &j) {
        if constexpr (D64) {
            // the minimum image of the FP64 positions' difference: odd, so
            // particle j forms exactly -r_ij
            j = lst[e * 32 + lane];
            rx = min_image_bits(X[0] - b.sx[j], ph.box_len[0], ph.periodic);
            ry = min_image_bits(X[1] - b.sy[j], ph.box_len[1], ph.periodic);
            rz = min_image_bits(X[2] - b.sz[j], ph.box_len[2], ph.periodic);
            hinv_j = gph[j].w;
        } else {
            const unsigned cd = lst[e * 32 + lane];
            const float4 tb = table[cd >> 5];
            const int tv = __float_as_int(tb.w);
            j = (WRAP && tv < 0 ? ~tv : tv) + (int)(cd & 31u);
            const V a0 = ld_ro(gph + j);
            // r_ij = (o_i - o_j) - D_AB: IEEE subtraction is sign-symmetric and
            // D_BA = -D_AB exactly, so particle j forms exactly -r_ij
            rx = sub_rn(sub_rn(xi.x, a0.x), tb.x);
            ry = sub_rn(sub_rn(xi.y, a0.y), tb.y);
            rz = sub_rn(sub_rn(xi.z, a0.z), tb.z);
            if (WRAP && tv < 0) wrap3s<float>(sc, rx, ry, rz);
            hinv_j = a0.w;
        }
        a1 = ld_ro(gvc + j);
        a2 = ld_ro(gth + j);
    };
    auto eval_lists = [&]() {
        __syncwarp();
        if (D64) cnt = gcnt > sub ? (gcnt - sub - 1) / LPP + 1 : 0;
        for (int e = 0; e < cnt; ++e) {
            V a1, a2;
            T rx, ry, rz, hinv_j;
            int j;
            fetch(e, rx, ry, rz, hinv_j, a1, a2, j);
            // every operation below up to m_i a_i with fixed rounding (odd
            // in r where it must be: particle j forms exactly the negatives)
            const T r2 = fma_rn(rz, rz, fma_rn(ry, ry, mul_rn(rx, rx)));
            if constexpr (D64) {  // tested in FP32 with room to spare until here
                const T hm = lt_pos(xi.w, hinv_j) ? xi.w : hinv_j;
                if (!lt_pos(r2 * hm * hm, T(KF::R * KF::R))) continue;
                ++pairs;
            }
            const T rinv = rsqrt_t(r2);
            const T r = mul_rn(r2, rinv);
            const T qi = mul_rn(r, xi.w), qj = mul_rn(r, hinv_j);
            const T hj2 = mul_rn(hinv_j, hinv_j);
            const T gi = mul_rn(mul_rn(sigma, KF::df(qi)), hi4);
            const T gj = mul_rn(mul_rn(sigma, KF::df(qj)), mul_rn(hj2, hj2));
            const T pterm = add_rn(mul_rn(Ai_g, gi), mul_rn(grav ? add_rn(a2.x, szg[j]) : a2.x, gj));
            const T vx = sub_rn(vi.x, a1.x), vy = sub_rn(vi.y, a1.y), vz = sub_rn(vi.z, a1.z);
            const T vdr = mul_rn(fma_rn(vz, rz, fma_rn(vy, ry, mul_rn(vx, rx))), rinv);
            const T mu = vdr < T(0) ? vdr : T(0);
            const T rhob_inv = fast_div(T(2), add_rn(ti.y, a2.y));
            const T gbar = mul_rn(T(0.5), add_rn(gi, gj));
            T al = alpha, be = beta;
            if (sw) {
                al = mul_rn(T(0.5), add_rn(alpha_i, sal[j]));
                be = mul_rn(bratio, al);
            }
            dvs += a2.z * vdr * gi;  // (div v: the switch's source, and the next step's h prediction)
            if (cdw) {
                const T mg = a2.z * gi * rinv;
                cg[0] += mg * vx * rx;
                cg[1] += mg * vx * ry;
                cg[2] += mg * vx * rz;
                cg[3] += mg * vy * rx;
                cg[4] += mg * vy * ry;
                cg[5] += mg * vy * rz;
                cg[6] += mg * vz * rx;
                cg[7] += mg * vz * ry;
                cg[8] += mg * vz * rz;
                if (qi < T(KF::R)) {
                    T f, df;
                    KF::fdf(qi, f, df);
                    cr += (scd[j] < T(0) ? -a2.z : a2.z) * f;
                }
            }
            const T vsig = fma_rn(-be, mu, add_rn(vi.w, a1.w));
            const T visc = mul_rn(mul_rn(mul_rn(al, vsig), mu), rhob_inv);
            const T S = fma_rn(visc, gbar, -pterm);
            const T wgt = mul_rn(mul_rn(mul_rn(ti.z, a2.z), S), rinv);
            acc.add(wgt, rx, ry, rz);
            if (adi)
                du += a2.z * (ti.x * vdr * gi +
                              rhob_inv * gbar * (T(-0.5) * al * vsig * mu * mu + aac * ac_speed(vdr, ti, a2, gm1_price, rhob_inv) * (ti.w - a2.w)));
            vs = lt_pos(vs, vsig) ? vsig : vs;
            if (blk) {
                const T lj = slev[j], aj = fabs(lj);
                mlev = aj > mlev ? aj : mlev;
                if (due && lj < T(0) && aj < li1 - lgap) atomicMax(&b.breq[b.perm[j]], (int)(li1 - lgap) - 1);
            }
        }
        if (!D64) pairs += cnt;
        cnt = gcnt = 0;
        __syncwarp();  // table and lists free for reuse
    };
    // membership: r_ij < R_K max(h_i, h_j), decided on the staged
    // (offset + shift) difference; where its rounding differs from the
    // pair vector's the pair sits at q = R_K, where f' and the force vanish
    auto test = [&]() {
        __syncwarp();  // staged candidates visible to every lane
        const int self = tA >= 0 ? ((tA << 5) | pos) : -1;
        const float e2 = D64 ? 2.f * warp_max(emax) : 0.f;
        emax = 0.f;
        if constexpr (PACK) {
            if (!wrap2) {
                cb.pad(nbuf);
                __syncwarp();
                const F2 px = pack2(xf.x, xf.x), py = pack2(xf.y, xf.y), pz = pack2(xf.z, xf.z);
                const int nk = C::Cand::mine(nbuf, 0), at0 = sub * C::Cand::SEC;
                for (int kb = 0; kb < nk; kb += C::SB / LPP) {
                    if (__any_sync(FULL, cnt > C::LC - C::SB / LPP)) eval_lists();
                    const int ke = min(kb + C::SB / LPP, nk);
                    for (int k = kb; k < ke; k += 4) {
                        const float4 x = ld4(cb.v[0] + at0 + k), y = ld4(cb.v[1] + at0 + k), z = ld4(cb.v[2] + at0 + k),
                                     w = ld4(cb.v[3] + at0 + k);
                        const uint2 c4 = *reinterpret_cast<const uint2 *>(code + at0 + k);
#pragma unroll
                        for (int h2 = 0; h2 < 2; ++h2) {
                            const F2 rx = px + (h2 ? pack2(x.z, x.w) : pack2(x.x, x.y));
                            const F2 ry = py + (h2 ? pack2(y.z, y.w) : pack2(y.x, y.y));
                            const F2 rz = pz + (h2 ? pack2(z.z, z.w) : pack2(z.x, z.y));
                            const float wa = h2 ? w.z : w.x, wb = h2 ? w.w : w.y;
                            const F2 hm = pack2(xf.w < wa ? xf.w : wa, xf.w < wb ? xf.w : wb);
                            float ta, tb;
                            unpack2((fma2(rz, rz, fma2(rx, rx, ry * ry)) * hm) * hm, ta, tb);
                            const unsigned cc = h2 ? c4.y : c4.x;
                            const int ca = (int)(cc & 0xffffu), cd = (int)(cc >> 16);
                            if (active && ca != self && ta < (float)(KF::R * KF::R)) lst[cnt++ * 32 + lane] = (Code)ca;
                            if (active && cd != self && tb < (float)(KF::R * KF::R)) lst[cnt++ * 32 + lane] = (Code)cd;
                        }
                    }
                }
                tested += (nbuf - sub + LPP - 1) / LPP;
                __syncwarp();
                nbuf = 0;
                return;
            }
        }
        for (int k0 = 0; k0 < nbuf; k0 += C::SB) {
            const int ke = k0 + C::SB < nbuf ? k0 + C::SB : nbuf;
            if constexpr (D64) {
                // FP32, with the coordinates' error to spare; the hits are dealt
                // to the particle's lanes by rank
                if (__any_sync(FULL, gcnt > C::LC * LPP - C::SB)) eval_lists();
                const unsigned below = (1u << sub) - 1u;
#pragma unroll 4
                for (int kk = k0; kk < ke; kk += LPP) {
                    const int k = kk + sub;
                    bool hit = false;
                    int j = 0;
                    if (k < ke) {
                        const float4 c = cand[k];
                        float rx = xf.x - c.x, ry = xf.y - c.y, rz = xf.z - c.z;
                        if (wrap2) wrap3s<float>(sc, rx, ry, rz);
                        const float Rm = fmaxf(xf.w, c.w) * 1.00001f + e2;
                        j = code[k];
                        hit = active && j != s && rx * rx + ry * ry + rz * rz < Rm * Rm + kTinySq;
                    }
                    const unsigned gm = (__ballot_sync(FULL, hit) >> (pp * LPP)) & ((1u << LPP) - 1u);
                    if (hit) {
                        const int e = gcnt + __popc(gm & below);
                        lst[(e / LPP) * 32 + pp * LPP + e % LPP] = j;
                    }
                    gcnt += __popc(gm);
                }
                continue;
            }
            if (__any_sync(FULL, cnt > C::LC - C::SB / LPP)) eval_lists();
#pragma unroll 4
            for (int k = k0 + sub; k < ke; k += LPP) {
                float4 c;
                int cd;
                if constexpr (PACK) {
                    const int at = C::Cand::place(k);
                    c = make_float4(-cb.v[0][at], -cb.v[1][at], -cb.v[2][at], cb.v[3][at]);
                    cd = code[at];
                } else {
                    c = cand[k];
                    cd = code[k];
                }
                float rx = xf.x - c.x, ry = xf.y - c.y, rz = xf.z - c.z;
                if (wrap2) wrap3s<float>(sc, rx, ry, rz);
                const float r2 = rx * rx + ry * ry + rz * rz;
                const float hm = xf.w < c.w ? xf.w : c.w;
                if (active && cd != self && r2 * hm * hm < (float)(KF::R * KF::R))
                    lst[cnt++ * 32 + lane] = (Code)cd;
            }
        }
        tested += (nbuf - sub + LPP - 1) / LPP;
        __syncwarp();
        nbuf = 0;
    };
    set_query(sc.qb, boxA.plo, boxA.phi, R, ph, coord_bound<D64>(ph, dy));
    auto node_test = [&](const NodeBox &nb) {
        const bool near = box_within(sc.qb, nb, ph);
        return box_overlap(sc.qb, nb, ph) || near;
    };
    auto visit = [&](unsigned mask, int first) {
            int jq = 0;  // (FP64) the staged particle's sorted index
            if (!D64 && ntab + __popc(mask) > C::TAB) {
                test();
                eval_lists();
                ntab = 0;
                tA = -1;
            }
            // candidate leaves that form an ambiguous pair with A (periodic)
            // (FP64: see the density pass)
            am = !D64 && ph.periodic ? __ballot_sync(FULL, ((mask >> lane) & 1u) && ambiguous(b.nodes[0][first + lane].slo.w, sc))
                                     : 0u;
            if (!WRAP && am) to_wrap = true;
            if (!WRAP && to_wrap) return;
            const unsigned amo = WRAP ? by_order(am, mask) : 0u;
            stage_group<float, C::CH, D64>(
                b, leaf, mask, first, ph, unit, nbuf, sc,
                [&](bool has, int B, int stB, int ord, const float4 &D) {
                    if (D64) return;
                    if (has) {
                        float4 t = D;
                        t.w = __int_as_float((am >> lane) & 1u ? ~stB : stB);
                        table[ntab + ord] = t;
                    }
                    const unsigned ka = (unsigned)(leaf - first);  // the query leaf itself in this group
                    if (ka < 32u && ((mask >> ka) & 1u)) tA = ntab + __popc(mask & ((1u << ka) - 1u));
                },
                [&](int j) {
                    if constexpr (D64) {
                        float4 q = b.pmf[j];
                        q.w = __int_as_float(j);
                        return q;
                    } else {
                        return gph[j];
                    }
                },
                [&](float4 &q, int o) {
                    const float aq = D64 ? abs3(q) : 0.f;
                    if (D64 ? ph.periodic != 0 : WRAP && ((amo >> o) & 1u))
                        wrap_near<float>(sc, q, sc.C[0], sc.C[1], sc.C[2]);
                    const float d2 = box_dist2<float>(q, flo, fhi);
                    if constexpr (D64) {
                        jq = __float_as_int(q.w);
                        q.w = __fmul_ru(KR_f, b.hf[jq]);
                        const float e = stage_err(abs3(sc.leaf[o]), aq, abs3(q), pmax), Rj = fmaxf(R, q.w) * 1.0001f + 2.f * e;
                        if (!(d2 < Rj * Rj + kTinySq)) return false;
                        emax = fmaxf(emax, e);
                        return true;
                    }
                    return d2 < RA2 || d2 * q.w * q.w < (float)(KF::R * KF::R * 1.0001);
                },
                [&](int slot, const float4 &q, int o, int idx) {
                    const Code cd = (Code)(D64 ? jq : (((ntab + o) << 5) | idx));
                    if constexpr (PACK) {
                        const int at = C::Cand::place(slot);
                        cb.v[0][at] = -q.x;
                        cb.v[1][at] = -q.y;
                        cb.v[2][at] = -q.z;
                        cb.v[3][at] = q.w;
                        code[at] = cd;
                    } else {
                        cand[slot] = q;
                        code[slot] = cd;
                    }
                },
                test);
            ntab += __popc(mask);
    };
    // the candidate groups the density walk recorded cover every pair
    // unless some final h outgrew them (then walk the tree again).  One lane
    // per particle: a loop of its own for either way, so that the walk's state
    // takes no registers beside the recorded groups' (in one loop k_forces
    // was 11 % slower at 1e6 particles); else one loop, so that the staging and
    // the evaluation are there once, with lane g holding group g (at most 32
    // are recorded)
    const int ngl = k0 < 0 && !dy.lists_stale ? b.leaf_ngroups[leaf] : -1;
    auto offer = [&](int first, unsigned in) {
        const bool mine_in = (in >> lane) & 1u;
        const bool ok = node_test(b.nodes[0][first + (mine_in ? lane : __ffs(in) - 1)]);
        const unsigned fm = __ballot_sync(FULL, ok && mine_in);
        if (fm) visit(fm, first);
    };
    auto next_node = [&](Walk &wk) {
        return wk.next(b, dy, [&](const NodeBox &nb) { return up_within(sc.qb, nb) || up_overlap(sc.qb, nb); });
    };
    if constexpr ((LPP == 1 && !WRAP) || CD) {
        if (ngl >= 0) {
            const int2 *rec = b.group_pool + b.leaf_gofs[leaf];
            for (int g = 0; g < ngl && !to_wrap; ++g) offer(rec[g].x, (unsigned)rec[g].y);
        } else {
            Walk wk;
            wk.start(dy);
            for (int node; !to_wrap && (node = next_node(wk)) >= 0;)
                offer(dy.node_off[0] + node * kBranch, leaf_lanes(dy.node_cnt[0], node));
        }
    } else {
        int2 rec = make_int2(0, 0);
        if (lane < ngl) rec = b.group_pool[b.leaf_gofs[leaf] + lane];
        Walk wk;
        wk.start(dy);
        for (int g = 0; !to_wrap; ++g) {
            int first;
            unsigned in;
            if (ngl >= 0) {
                if (g >= ngl) break;
                first = __shfl_sync(FULL, rec.x, g);
                in = (unsigned)__shfl_sync(FULL, rec.y, g);
            } else {
                const int node = next_node(wk);
                if (node < 0) break;
                first = dy.node_off[0] + node * kBranch;
                in = leaf_lanes(dy.node_cnt[0], node);
            }
            offer(first, in);
        }
    }
    test();
    eval_lists();
    if (!WRAP && to_wrap) return false;
    // combine the lanes of each particle; FP64 for the compensated sums
    double Fx, Fy, Fz;
    acc.get(Fx, Fy, Fz);
    Fx = group_sum<LPP>(Fx);
    Fy = group_sum<LPP>(Fy);
    Fz = group_sum<LPP>(Fz);
    du = group_sum<LPP>(du);
    vs = group_max<LPP>(vs);
    dvs = group_sum<LPP>(dvs);
    if (cdw) {
#pragma unroll
        for (int k = 0; k < 9; ++k) cg[k] = group_sum<LPP>(cg[k]);
        cr = group_sum<LPP>(cr);
    }
    if (blk) mlev = group_max<LPP>(mlev);
    // a = F / m in FP64 (m a stays F to FP64 round-off), one reciprocal
    // per particle (none for equal masses); the CFL step C h / v_sig of
    // Eq. SPH_DT in the pair precision (FP32: the FP64 pipe is much
    // narrower than the FP32 one on this part)
    T dti = tinf<T>();
    if (due && sub == 0) {
        long long g = b.perm[s];
        long long i = g - ps.base;
        if (blk) b.bnml[g] = (int)mlev - 1;
        const double minv = ps.uniform_m ? ps.inv_m_uniform : 1.0 / ps.m[i];
        double a[3] = {Fx * minv, Fy * minv, Fz * minv};
        const T vsig_t = vs < T(0) ? T(2) * vi.w : vs;
        ps.ax[i] = a[0];
        ps.ay[i] = a[1];
        ps.az[i] = a[2];
        ps.du[i] = adi ? (double)du : 0.0;
        ps.vsig[i] = (double)vsig_t;
        // div v = -(1/(Omega rho)) sum_j m_j v_ij . grad_i W(h_i): the next
        // step starts its h iteration from h exp(div v dt / 3) (continuity,
        // with h ~ rho^-1/3)
        b.divv[g] = (float)(-(double)dvs / (b.somega[s] * b.srho[s]));
        if (sw && !cdw) {  // Morris & Monaghan: decay towards alpha_min, growth where compressed
            const double divv = -(double)dvs / (b.somega[s] * b.srho[s]);
            const double ai = (double)alpha_i;
            ps.dalpha[i] = -(ai - ph.alpha_min) * ph.av_decay * (double)vi.w / b.sh[s] +
                           (divv < 0.0 ? -divv * (ph.alpha_av - ai) : 0.0);
        }
        if (cdw) {  // Cullen & Dehnen: velocity gradient, shear, signed density, limiter
            const double rho_i = b.srho[s], f = -1.0 / (b.somega[s] * rho_i);
            double V[9];
            for (int k = 0; k < 9; ++k) V[k] = f * (double)cg[k];
            const double dv = V[0] + V[4] + V[8];
            double ss = 0.0;
            for (int p2 = 0; p2 < 3; ++p2)
                for (int q2 = 0; q2 < 3; ++q2) {
                    const double sab = 0.5 * (V[3 * p2 + q2] + V[3 * q2 + p2]) - (p2 == q2 ? dv / 3.0 : 0.0);
                    ss += sab * sab;
                }
            const double hinv_i = (double)xi.w, w0 = Kern<K>::sigma * hinv_i * hinv_i * hinv_i;
            T f0, df0;
            KF::fdf(T(0), f0, df0);
            const double self = (ps.dalpha[i] < 0.0 ? -1.0 : 1.0) * (double)ti.z * (double)f0;
            const double R = ((double)cr + self) * w0 / rho_i;
            const double om = 1.0 - R, qq = 2.0 * om * om * om * om * dv;
            b.cdold[g] = ps.dalpha[i];
            b.cdxi[g] = (qq * qq + ss) > 0.0 ? qq * qq / (qq * qq + ss) : 0.0;
            ps.dalpha[i] = dv;
        }
        dti = (T)ph.c_cfl * (T)b.sh[s] / vsig_t;
        if (!(isfinite(a[0]) && isfinite(a[1]) && isfinite(a[2]) && isfinite(du)))
            atomicOr(&ps.diag->status, ST_NONFINITE);
    }
    const T dmin = warp_min(dti);
    long long tp = warp_sum((long long)pairs), tt = warp_sum((long long)tested);
    if (lane == 0) {
        if (dmin < INFINITY)
            atomicMin(&ps.diag->dt_min_bits, (unsigned long long)__double_as_longlong((double)dmin));
        atomicAdd((unsigned long long *)&ps.diag->force_pairs, (unsigned long long)tp);
        atomicAdd((unsigned long long *)&ps.diag->candidates, (unsigned long long)tt);
    }
    return true;
}

// WRAP: the launch that serves the wrap list (leaves whose pair vectors may
// miss the minimum image); the other launch puts them there.
template <typename T, int LPP, int K, bool WRAP, bool CD>
__global__ void __launch_bounds__(FCfg<T, LPP, K>::WPB * 32, FCfg<T, LPP, K>::MINB) k_forces(BatchView b)
{
    chain_entry();
    using C = FCfg<T, LPP, K>;
    extern __shared__ __align__(32) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char *mine = smem + wib * C::per_warp;
    // block-step ticks: the wrap-list launch serves the tick's tasks (leaf
    // << 5 | first due ordinal) directly; the common launch does not run
    const bool tasks = WRAP && b.block_on && b.block_tasks;
    const int nleaf = tasks ? b.counters[kBlockTasks] : WRAP ? b.counters[kForceWrapList] : b.counters[0];
    const int cls = lpp_log2(LPP) + 4 * K;
    int last_p = -1;
    float Rall = 0.f;  // periodic: pairs reach R_K x the problem's largest h
    for (int item = first_item();;
         item = next_item(&b.counters[(CD ? kForceCdCounter : WRAP ? kForceWrapCounter : kForceCounter) + cls])) {
        if (item >= nleaf) break;
        const int what = !WRAP ? item : tasks ? b.btask[item] : b.wrap_list[item];
        const int leaf = tasks ? what >> 5 : what, k0 = tasks ? what & 31 : -1;
        const int p = b.leaf_pid[leaf];
        const ProbStatic &ps = b.prob[p];
        if ((tasks ? b.block_lanes : ps.lpp) != LPP || ps.ph.kernel != K) continue;  // served by another launch
        if (WRAP && (ps.ph.av_switch == SPH_AV_CULLEN_DEHNEN) != CD) continue;  // (the switch's own launch)
        if (!WRAP && (ps.ph.av_switch || ps.ph.ac_signal || ps.ph.gravity || b.block_on)) {
            // the viscosity switch, Price's conductivity and gravity's zeta term run in the
            // wrap-list launch only, which keeps the common path's registers for the default scheme
            if (lane == 0) b.wrap_list[atomicAdd(&b.counters[kForceWrapList], 1)] = leaf;
            continue;
        }
        if (ps.ph.periodic && p != last_p) {  // (consecutive leaves mostly share a problem)
            float extmax;
            problem_top_max(b, b.dyn[p], Rall, extmax);
            Rall = __fmul_ru((float)Kern<K>::R, Rall) * 1.0001f;
            last_p = p;
        }
        if (!force_leaf<T, LPP, K, WRAP, CD>(b, leaf, k0, mine, Rall) && lane == 0) {
            b.wrap_list[atomicAdd(&b.counters[kForceWrapList], 1)] = leaf;
            atomicAdd(&ps.diag->wrap_leaves, 1);
        }
    }
}

template <typename KernFn>
void set_smem(KernFn k, size_t bytes)
{
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T, int LPP, bool UM, int K, bool WRAP>
cudaError_t run_density(const BatchView &b, int use_pred, cudaStream_t st)
{
    using C = DCfg<T, LPP, UM, K>;
    static int per_sm = 0;
    if (!per_sm) {
        set_smem(k_density<T, LPP, UM, K, WRAP>, C::smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_density<T, LPP, UM, K, WRAP>, C::WPB * 32, C::smem);
        if (per_sm < 1) per_sm = 1;
    }
    // the wrap-list launch serves few leaves (mostly none) unless a problem
    // has gravity or the launch is a block-step tick's
    launch_chain(SPH_DEP(b), k_density<T, LPP, UM, K, WRAP>, dev_info().sm_count * (WRAP && !b.any_gravity && !(b.block_on && b.block_tasks) ? 1 : per_sm), C::WPB * 32, C::smem, st, b, use_pred);
    return cudaGetLastError();
}

template <typename T>
void run_density_fallback(const BatchView &b, int use_pred, cudaStream_t st)
{
    using C = FbCfg<T>;
    static bool init = false;
    if (!init) {
        set_smem(k_density_fallback<T>, C::smem);
        init = true;
    }
    launch_chain(SPH_DEP(b), k_density_fallback<T>, dev_info().sm_count * 4, C::WPB * 32, C::smem, st, b, use_pred);
}

// Block-step ticks, after the leaves: each leaf with particles whose step
// ends now gives one task per 32 / block_lanes of them (in sorted order), so
// that a task's block_lanes lanes per particle and its box (of those
// particles only) keep the pair kernels' latency short when few particles of
// a leaf are due; the leaf's other particles keep the h, rho, Omega, P and c
// of their last solve and are restaged (with their drifted offsets and
// predicted v, u) for the force pass.  One warp per leaf (<= 32 particles),
// lane = position in the leaf.
template <typename T>
__device__ __forceinline__ void block_tasks_one(const BatchView &b, int leaf, int n, long long s, bool due, int use_pred)
{
    using V = typename Vec4<T>::type;
    const int lane = threadIdx.x & 31;
    const int d = __popc(__ballot_sync(FULL, due));
    const int size = 32 / b.block_lanes, nt = (d + size - 1) / size;
    int base = 0;
    if (lane == 0 && nt > 0) base = atomicAdd(&b.counters[kBlockTasks], nt);
    base = __shfl_sync(FULL, base, 0);
    if (lane < nt) b.btask[base + lane] = (leaf << 5) | (lane * size);
    const double unit = sizeof(T) == 8 ? frame_of(b.prob[0].ph, b.dyn[0]).unit : 1.0;
    if (lane < n && !due) density_epilogue<T>(b, b.prob[0], s, ((const V *)b.pm)[s], T(1), T(0), T(0), use_pred, T(0), unit);
}

// the tasks of a tick that built its leaves
template <typename T>
__global__ void __launch_bounds__(256) k_block_tasks(BatchView b, int use_pred)
{
    chain_entry();
    const int lane = threadIdx.x & 31;
    const int nleaf = b.counters[0];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int leaf = w; leaf < nleaf; leaf += nw) {
        const int st = b.leaf_start[leaf], n = b.leaf_start[leaf + 1] - st;
        const long long s = st + (lane < n ? lane : 0);
        const bool due = lane < n && ((const T *)b.slev)[s] > T(0);
        block_tasks_one<T>(b, leaf, n, s, due, use_pred);
    }
}

// A tick that keeps the order and the leaves (tree reuse, Sec. 4.2), one
// warp per leaf: the drift of its particles, their gather into sorted order
// and the staging of their levels, the leaf's offsets and boxes and the tree
// above it (as the leaf pass does for kept leaves), then its tasks and the
// restaging of its particles that keep their solve: one pass instead of four.
template <typename T, typename T4>
__global__ void __launch_bounds__(256) k_block_leaf_tick(BatchView b, int use_pred)
{
    chain_entry();
    const int lane = threadIdx.x & 31;
    const int nleaf = b.counters[0];
    if (blockIdx.x == 0)
        for (int p = threadIdx.x; p < b.nprob; p += blockDim.x) b.dyn[p].lists_stale = 0;
    const long long k0 = b.scratch64[4], k1 = b.scratch64[5];
    const double tau = __longlong_as_double(b.scratch64[7]);
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int leaf = w; leaf < nleaf; leaf += nw) {
        const int st = b.leaf_start[leaf], n = b.leaf_start[leaf + 1] - st;
        const long long s = st + (lane < n ? lane : 0);
        bool due = false;
        if (lane < n) {
            const ProbStatic &ps = b.prob[0];
            const long long g = b.perm[s], i = g - ps.base;
            const double m = ps.m[i], h = ps.h[i];  // (read with the drift's inputs, not after its stores)
            const int lv = b.blev[g];
            double x[3];
            due = drift_one(b, g, k0, k1, tau, x);
            b.sx[s] = x[0];
            b.sy[s] = x[1];
            b.sz[s] = x[2];
            b.sm[s] = m;
            b.sh[s] = h;
            const T v = (T)(lv + 1);
            ((T *)b.slev)[s] = due ? v : -v;
        }
        const unsigned dm = __ballot_sync(FULL, due);
        if (lane == 0 && dm) atomicAdd((unsigned long long *)&b.scratch64[3], (unsigned long long)__popc(dm));
        __syncwarp();  // the leaf's gathered particles visible to the whole warp
        leaf_props_one<T4, true>(b, leaf);
        __syncwarp();
        block_tasks_one<T>(b, leaf, n, s, due, use_pred);
    }
}

template <typename T, int LPP, int K, bool WRAP, bool CD = false>
cudaError_t run_forces(const BatchView &b, cudaStream_t st)
{
    using C = FCfg<T, LPP, K>;
    static bool init = false;
    if (!init) {
        set_smem(k_forces<T, LPP, K, WRAP, CD>, C::smem);
        init = true;
    }
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_forces<T, LPP, K, WRAP, CD>, C::WPB * 32, C::smem);
    if (per_sm < 1) per_sm = 1;
    // the wrap list is short unless a problem uses the viscosity switch or Price's conductivity
    int grid = dev_info().sm_count * (WRAP && !b.any_general ? 1 : per_sm);
    launch_chain(SPH_DEP(b), k_forces<T, LPP, K, WRAP, CD>, grid, C::WPB * 32, C::smem, st, b);
    cudaError_t e = cudaGetLastError();
    // the Cullen & Dehnen problems' leaves on the wrap list: their own launch
    // (never with block steps, the only users of whole-warp particles)
    if constexpr (WRAP && !CD && LPP != 32)
        if (e == cudaSuccess && b.any_cd) e = run_forces<T, LPP, K, true, true>(b, st);
    return e;
}

// The density launches of kernel K: one per class (lanes per particle, equal
// masses) present in the batch; class bit lanes_index + 4 u + 8 K.  FP64
// runs 2 or 4 lanes per particle, M6 at least 2 (the host never selects
// fewer).  WRAP: the launches that serve the wrap list.
template <int K, bool WRAP>
cudaError_t density_classes(const BatchView &b, int precision, int use_pred, cudaStream_t st)
{
    for (int cls = 0; cls < 8; ++cls) {
        if (!(b.dens_mask & (1 << (cls + 8 * K)))) continue;
        const int k = cls & 3;
        const bool um = cls >= 4;
        cudaError_t e;
        if (precision == SPH_PREC_FP64) {
            if (k == 2) e = um ? run_density<double, 4, true, K, WRAP>(b, use_pred, st) : run_density<double, 4, false, K, WRAP>(b, use_pred, st);
            else e = um ? run_density<double, 2, true, K, WRAP>(b, use_pred, st) : run_density<double, 2, false, K, WRAP>(b, use_pred, st);
        } else {
            switch (k) {
            case 0:
                if constexpr (K == SPH_KERNEL_M4) {
                    e = um ? run_density<float, 1, true, K, WRAP>(b, use_pred, st) : run_density<float, 1, false, K, WRAP>(b, use_pred, st);
                    break;
                }
                [[fallthrough]];  // (M6 never runs one lane per particle)
            case 1: e = um ? run_density<float, 2, true, K, WRAP>(b, use_pred, st) : run_density<float, 2, false, K, WRAP>(b, use_pred, st); break;
            case 2: e = um ? run_density<float, 4, true, K, WRAP>(b, use_pred, st) : run_density<float, 4, false, K, WRAP>(b, use_pred, st); break;
            default:
                // block-step tasks of one particle with a whole warp (M4, FP32)
                if constexpr (K == SPH_KERNEL_M4 && WRAP) {
                    if (b.block_on && b.block_tasks && b.block_lanes == 32) {
                        e = um ? run_density<float, 32, true, K, WRAP>(b, use_pred, st) : run_density<float, 32, false, K, WRAP>(b, use_pred, st);
                        break;
                    }
                }
                e = um ? run_density<float, 8, true, K, WRAP>(b, use_pred, st) : run_density<float, 8, false, K, WRAP>(b, use_pred, st);
                break;
            }
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The force launches of kernel K, one per lanes-per-particle class present
// (class bit lanes_index + 4 K).
template <int K, bool WRAP>
cudaError_t force_classes(const BatchView &b, int precision, cudaStream_t st)
{
    for (int k = 0; k < 4; ++k) {
        if (!(b.lpp_mask & (1 << (k + 4 * K)))) continue;
        cudaError_t e;
        if (precision == SPH_PREC_FP64) {
            if (k == 2) e = run_forces<double, 4, K, WRAP>(b, st);
            else e = run_forces<double, 2, K, WRAP>(b, st);
        } else {
            switch (k) {
            case 0:
                if constexpr (K == SPH_KERNEL_M4) {
                    e = run_forces<float, 1, K, WRAP>(b, st);
                    break;
                }
                [[fallthrough]];
            case 1: e = run_forces<float, 2, K, WRAP>(b, st); break;
            case 2: e = run_forces<float, 4, K, WRAP>(b, st); break;
            default:
                if constexpr (K == SPH_KERNEL_M4 && WRAP) {
                    if (b.block_on && b.block_tasks && b.block_lanes == 32) {
                        e = run_forces<float, 32, K, WRAP>(b, st);
                        break;
                    }
                }
                e = run_forces<float, 8, K, WRAP>(b, st);
                break;
            }
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

// the launches of one kernel (M4, M6) and kind (common, wrap list), each
// instantiated in a translation unit of its own so that they compile in
// parallel
cudaError_t density_launches_m4(const BatchView &b, int precision, int use_pred, cudaStream_t st);
cudaError_t density_launches_m6(const BatchView &b, int precision, int use_pred, cudaStream_t st);
cudaError_t density_launches_m4_wrap(const BatchView &b, int precision, int use_pred, cudaStream_t st);
cudaError_t density_launches_m6_wrap(const BatchView &b, int precision, int use_pred, cudaStream_t st);
cudaError_t force_launches_m4(const BatchView &b, int precision, cudaStream_t st);
cudaError_t force_launches_m6(const BatchView &b, int precision, cudaStream_t st);
cudaError_t force_launches_m4_wrap(const BatchView &b, int precision, cudaStream_t st);
cudaError_t force_launches_m6_wrap(const BatchView &b, int precision, cudaStream_t st);

}  // namespace sph
