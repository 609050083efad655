// rlb_step_f32.cuh -- the fused step of the FP32-storage form.
//
// One thread updates two x-adjacent cells (x0, x0 + 1) of one (y, z) row.
// Populations are stored, streamed and relaxed in FP32.  The moment sums
// T^00 and T^0a are accumulated error-free as double-float pairs (TwoSum),
// and E^2 - |M|^2, the quantity whose cancellation grows like gamma^2 in the
// Landau-frame recovery, is formed in double-float before one rounding; the
// rest of the recovery (a well-conditioned function of E^2 - |M|^2, E, M and
// N^0), tau and the equilibrium coefficients are FP32.  No FP64 instruction
// is issued.  The previous level's recovery is the same arithmetic on its
// stored float sums.  The REC64 variant (rlb_options.recovery_fp64) runs
// both recoveries in FP64 from the exact double values of the sums instead;
// it exists to measure what FP64 buys over the double-float form.
//
// Conservation: the float equilibrium coefficients carry fixed roundings of
// irrational constants (weights, 4/xi0, 13/9, ...) that would bias their
// lattice moments identically at every step.  The previous level is kept as
// the raw moment sums of time t - dt (sum f, sum c_a f, sum h), so the
// moments 2 f^eq(t) - f^eq(t - dt) must have are known exactly; after the
// coefficients are formed, their closed-form lattice sums are compared with
// those targets and the rest coefficient (T^00, N^0) and the axis
// first-order coefficient (T^0a) absorb the difference, so only unbiased
// per-cell roundings remain.
#pragma once

#include <utility>

#include "rlb_bulk.cuh"
#include "rlb_classes.cuh"
#include "rlb_device.cuh"
#include "rlb_internal.h"
#include "rlb_pair.cuh"

namespace rlb {

namespace f32 {

// xi0^2 split into float hi + lo where a double-float value is needed
template <int LAT>
struct Xi0Sq {
    static constexpr float hi = float(Lat<LAT>::xi0sq);
    static constexpr float lo = float(Lat<LAT>::xi0sq - double(float(Lat<LAT>::xi0sq)));
};

template <int... Is, typename F>
__device__ __forceinline__ void for_pops(std::integer_sequence<int, Is...>, F &&fn)
{
    (fn(std::integral_constant<int, Is>{}), ...);
}
#define RLB_F32_POPS std::make_integer_sequence<int, 19>{}

// the population classes of the symmetry reductions (rlb_classes.cuh)
using rlb::has_vy;
using rlb::has_vz;
using rlb::mult;
using rlb::rep;

// Storage of a grid in FP32 form: rows are padded to an even length nxe =
// nx + nx % 2, and cell (x, y, z) has the storage index i = x + nxe (y + ny z).
// Blocks of kBlk consecutive storage cells hold their 38 populations (f, then
// h) one after the other: population k of cell i is at float
//   (i / kBlk) kBlk 38 + k kBlk + i % kBlk,
// so that every population of a cell sits at a compile-time distance from its
// first one and a thread needs one address per stencil position for all 38
// (with one plane per population each load cost two more instructions for its
// address, 14 % of the step's instructions).  A pair of cells (even i) never
// straddles a block; 32 cells are one 128-byte line per population.  The
// previous level has 5 values per cell in blocks of its own.
constexpr int kBlk = 32;
constexpr int kPops = 38;
__host__ __device__ __forceinline__ size_t blk_at(long long i) { return size_t(i >> 5) * (kBlk * kPops) + size_t(i & 31); }
__host__ __device__ __forceinline__ size_t blk_prev_at(long long i) { return size_t(i >> 5) * (kBlk * 5) + size_t(i & 31); }

// Fix-ups of the x stencil v[0..5] = x0-2 .. x0+3 of a pair at a row's ends:
// clamped (open) or ghost (inlet) values, and the ends of rows of odd length,
// whose last pair (ODD1: x0 = nx - 1) holds one pad cell and whose last but
// one (ODD3: x0 = nx - 3) ends two cells before it.  Periodic rows of even
// length need none (the pair's address wraps); those of odd length take one
// extra value (EX) where the wrapped cells are not an aligned pair.
enum {
    XF_LO_CLAMP = 1, XF_LO_GHOST = 2, XF_HI_CLAMP = 4, XF_HI_GHOST = 8, XF_HI_ODD1 = 16, XF_HI_ODD3 = 32,
    XF_HI_ODD1G = 64, XF_HI_ODD3G = 128, XF_LO_EX = 256, XF_HI_EX = 512, XF_HI_WRAP1 = 1024, XF_HI_SELF = 2048
};

__device__ __forceinline__ int map1(int c, int n, int lo, int hi)
{
    if (c >= 0 && c < n) return c;
    const int bc = c < 0 ? lo : hi;
    if (bc == BC_PERIODIC) {
        int m = c % n;
        return m < 0 ? m + n : m;
    }
    return c < 0 ? 0 : n - 1;
}

// Where the stencil values of one population come from.  get(slot): the pairs
// at x0-2, x0, x0+2 (slots 0, 1, 2); nb<A, D>(slot): the pair at distance D
// along axis A, the k-th one that population needs there (slot 3 A + k).
// values loaded into registers
struct Sten {
    f2 v[9];
    float ex;
};
struct RegSrc {
    const Sten &s;
    __device__ __forceinline__ f2 get(int slot) const { return s.v[slot]; }
    template <int A, int D>
    __device__ __forceinline__ f2 nb(int slot) const { return s.v[slot]; }
    __device__ __forceinline__ float extra() const { return s.ex; }
};
// TileSrc (rlb_bulk.cuh): the block's bulk-copied tiles

// x0-2 .. x0+3 of one population: three aligned pairs, patched at a row's ends
template <bool ODDP, typename Src>
__device__ __forceinline__ void xstencil(const Src &src, unsigned xfix, float ghost, float (&v)[6])
{
    const f2 a = src.get(0), b = src.get(1), c = src.get(2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y; v[4] = c.x; v[5] = c.y;
    if (xfix) {
        if (xfix & XF_LO_CLAMP) { v[0] = v[2]; v[1] = v[2]; }
        if (xfix & XF_LO_GHOST) { v[0] = ghost; v[1] = ghost; }
        if (xfix & XF_HI_CLAMP) { v[4] = v[3]; v[5] = v[3]; }
        if (xfix & XF_HI_GHOST) { v[4] = ghost; v[5] = ghost; }
        if (xfix & XF_HI_ODD1) { v[3] = v[2]; v[4] = v[2]; v[5] = v[2]; }
        if (xfix & XF_HI_ODD3) v[5] = v[4];
        if (xfix & XF_HI_ODD1G) { v[3] = ghost; v[4] = ghost; v[5] = ghost; }
        if (xfix & XF_HI_ODD3G) v[5] = ghost;
        if constexpr (ODDP) {
            if (xfix & XF_LO_EX) { v[0] = v[1]; v[1] = src.extra(); }
            if (xfix & XF_HI_EX) v[5] = src.extra();
            if (xfix & XF_HI_WRAP1) { v[3] = v[4]; v[4] = v[5]; }
            if (xfix & XF_HI_SELF) v[5] = v[2];
        }
    }
}

// Divisions and the logarithm of the per-cell scalar work (recovery, tau,
// kappa, 1/gamma): the fast intrinsics (a few ulp, operands far from the
// range limits of __fdividef) unless RLB_F32_IEEE_DIV is defined.  The
// conserved sums do not depend on them: the equilibrium's lattice sums are
// set to exact targets afterwards (weigh2).
__device__ __forceinline__ float fdiv(float a, float b)
{
#ifdef RLB_F32_IEEE_DIV
    return a / b;
#else
    return __fdividef(a, b);
#endif
}
__device__ __forceinline__ float flog(float a)
{
#ifdef RLB_F32_IEEE_DIV
    return logf(a);
#else
    return __logf(a);
#endif
}

struct Mac2 {
    f2 P, ux, uy, uz, n;
};

// equilibrium coefficients of a pair, weights and diagonal factors folded in
struct W2 {
    f2 r0, a0, ab[3], ad[3], d0, db[3], dd[3], dk[3];
};

// K0, Kb, Kd, Ko of the f equilibrium (see rlb_device.cuh) for a pair
template <int LAT>
__device__ __forceinline__ void coef_f2(const Mac2 &m, f2 &K0, f2 (&Kb)[3], f2 (&Kd)[3], f2 (&Ko)[3])
{
    const f2 u2 = fma2(m.ux, m.ux, fma2(m.uy, m.uy, m.uz * m.uz));
    const f2 g = f2{sqrtf(1.0f + u2.x), sqrtf(1.0f + u2.y)};
    const f2 A = m.P * bc(Lat<LAT>::f_inv_sigma2);
    K0 = A * fma2(bc(-16.0f / 15.0f), u2, bc(1.0f));
    const f2 b = A * bc(float(Lat<LAT>::four_over_xi0)) * g;
    Kb[0] = b * m.ux; Kb[1] = b * m.uy; Kb[2] = b * m.uz;
    const f2 d = A * bc(Lat<LAT>::f_a3f);
    Kd[0] = d * m.ux * m.ux; Kd[1] = d * m.uy * m.uy; Kd[2] = d * m.uz * m.uz;
    const f2 o = A * bc(Lat<LAT>::f_a2f);
    Ko[0] = o * m.ux * m.uy; Ko[1] = o * m.ux * m.uz; Ko[2] = o * m.uy * m.uz;
}

template <int LAT>
__device__ __forceinline__ void coef_h2(const Mac2 &m, f2 &K0, f2 (&Kb)[3], f2 (&Kd)[3], f2 (&Ko)[3])
{
    const f2 u2p = fma2(m.ux, m.ux, fma2(m.uy, m.uy, m.uz * m.uz));
    const f2 g = f2{sqrtf(1.0f + u2p.x), sqrtf(1.0f + u2p.y)};
    const f2 ig = f2{fdiv(1.0f, g.x), fdiv(1.0f, g.y)};
    const f2 ux = m.ux * ig, uy = m.uy * ig, uz = m.uz * ig;
    const f2 B = m.n * g;
    const f2 uu = fma2(ux, ux, fma2(uy, uy, uz * uz));
    K0 = B * fma2(bc(-1.5f), uu, bc(float(Lat<LAT>::c0ct)));
    const f2 b3 = B * bc(3.0f);
    Kb[0] = b3 * ux; Kb[1] = b3 * uy; Kb[2] = b3 * uz;
    const f2 b45 = B * bc(4.5f);
    Kd[0] = b45 * ux * ux; Kd[1] = b45 * uy * uy; Kd[2] = b45 * uz * uz;
    const f2 b9 = B * bc(9.0f);
    Ko[0] = b9 * ux * uy; Ko[1] = b9 * ux * uz; Ko[2] = b9 * uy * uz;
}

// weights folded in (Eqs. 43-45 or 59-60) and the lattice sums set to the
// exact targets: T0 = sum_i G_i, Ta = sum_i c_ia G_i (only for f).  The rest
// weight w0 enters only through the target (sum_i w_i = 1).
template <int DM>
__device__ __forceinline__ W2 weigh2(f2 K0, const f2 (&Kb)[3], const f2 (&Kd)[3], const f2 (&Ko)[3],
                                     float w0, float w1, float w2, f2 T0, const f2 *Ta)
{
    (void)w0;
    W2 e;
    e.a0 = bc(w1) * K0;
    e.d0 = bc(w2) * K0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        e.ab[j] = bc(w1) * Kb[j];
        e.ad[j] = bc(w1) * Kd[j];
        e.db[j] = bc(float(DM) * w2) * Kb[j];
        e.dd[j] = bc(float(DM * DM) * w2) * Kd[j];
        e.dk[j] = bc(float(DM * DM) * w2) * Ko[j];
    }
    // sum_i G_i = r0 + 6 a0 + 12 d0 + 2 sum ad + 8 sum dd: the rest coefficient
    // is the remainder that makes this equal T0, with the other terms summed
    // error-free (their roundings are correlated, all being K0 times fixed
    // weights, and a float sum of them is biased); one final rounding
    df2 R{bc(0.0f), bc(0.0f)};
    {
        const f2 p6 = bc(6.0f) * e.a0, p12 = bc(12.0f) * e.d0;
        acc(R, p6);
        acc(R, fma2(bc(6.0f), e.a0, -p6));
        acc(R, p12);
        acc(R, fma2(bc(12.0f), e.d0, -p12));
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        acc(R, e.ad[j] + e.ad[j]);
        acc(R, bc(8.0f) * e.dd[j]);
    }
    {
        f2 s, er;
        two_sum(T0, -R.hi, s, er);
        e.r0 = s + (er - R.lo);
    }
    if (Ta) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // sum_i c_ia G_i = 2 ab_a + 8 DM db_a (8 DM db and the halving are exact)
            e.ab[j] = bc(0.5f) * (Ta[j] - bc(float(8 * DM)) * e.db[j]);
        }
    }
    return e;
}

template <int I>
__device__ __forceinline__ f2 eq2(const W2 &e)
{
    constexpr int cx = cdir<I, 0>(), cy = cdir<I, 1>(), cz = cdir<I, 2>();
    constexpr int sh = shell<I>();
    if constexpr (sh == 0) {
        return e.r0;
    } else if constexpr (sh == 1) {
        constexpr int a = cx != 0 ? 0 : (cy != 0 ? 1 : 2);
        constexpr int s = cx + cy + cz;
        const f2 base = e.a0 + e.ad[a];
        return s > 0 ? base + e.ab[a] : base - e.ab[a];
    } else {
        constexpr int a = cx != 0 ? 0 : 1;
        constexpr int b = cz != 0 ? 2 : 1;
        constexpr int ca = a == 0 ? cx : cy, cb = b == 2 ? cz : cy;
        constexpr int ko = (a == 0 && b == 1) ? 0 : ((a == 0 && b == 2) ? 1 : 2);
        f2 v = e.d0 + (e.dd[a] + e.dd[b]);
        v = ca > 0 ? v + e.db[a] : v - e.db[a];
        v = cb > 0 ? v + e.db[b] : v - e.db[b];
        v = ca * cb > 0 ? v + e.dk[ko] : v - e.dk[ko];
        return v;
    }
}

// The coefficients as the update takes them from this thread's shared-memory
// slots (slot k at q[k * stride]): the rest value, then per axis the even part
// a0 + ad and the odd part ab, then per plane (xy, xz, yz) the even part
// d0 + (dd_a + dd_b), the odd parts db per axis and dk per plane.  They are
// read where a population needs them and hold no registers between.
constexpr int kEqSlots = 16;
__device__ __forceinline__ void park_eq(const W2 &e, f2 *q, int stride)
{
    q[0] = e.r0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        q[(1 + j) * stride] = e.a0 + e.ad[j];
        q[(4 + j) * stride] = e.ab[j];
        q[(10 + j) * stride] = e.db[j];
        q[(13 + j) * stride] = e.dk[j];
    }
    q[7 * stride] = e.d0 + (e.dd[0] + e.dd[1]);
    q[8 * stride] = e.d0 + (e.dd[0] + e.dd[2]);
    q[9 * stride] = e.d0 + (e.dd[1] + e.dd[2]);
}
// the same values in an array of registers (slot k at q[k]): the bulk-staged
// kernel, whose shared memory holds tiles instead.  zero: -0, which the compiler
// does not know, so that the products ab, db and dk round once here, as they do
// on their way to shared memory, and are not fused into the sums that use them.
__device__ __forceinline__ void hold_eq(const W2 &e, f2 (&q)[kEqSlots], f2 zero)
{
    park_eq(e, q, 1);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        q[4 + j] = q[4 + j] + zero;
        q[10 + j] = q[10 + j] + zero;
        q[13 + j] = q[13 + j] + zero;
    }
}
template <int I>
__device__ __forceinline__ f2 eq_parked(const f2 *q, int stride)
{
    constexpr int cx = cdir<I, 0>(), cy = cdir<I, 1>(), cz = cdir<I, 2>();
    constexpr int sh = shell<I>();
    if constexpr (sh == 0) {
        return q[0];
    } else if constexpr (sh == 1) {
        constexpr int a = cx != 0 ? 0 : (cy != 0 ? 1 : 2);
        const f2 base = q[(1 + a) * stride], b = q[(4 + a) * stride];
        return cx + cy + cz > 0 ? base + b : base - b;
    } else {
        constexpr int a = cx != 0 ? 0 : 1;
        constexpr int b = cz != 0 ? 2 : 1;
        constexpr int ca = a == 0 ? cx : cy, cb = b == 2 ? cz : cy;
        constexpr int ko = (a == 0 && b == 1) ? 0 : ((a == 0 && b == 2) ? 1 : 2);
        f2 v = q[(7 + ko) * stride];
        const f2 da = q[(10 + a) * stride], db = q[(10 + b) * stride], dk = q[(13 + ko) * stride];
        v = ca > 0 ? v + da : v - da;
        v = cb > 0 ? v + db : v - db;
        return ca * cb > 0 ? v + dk : v - dk;
    }
}

// Landau-frame recovery of a pair from the raw sums S = sum f, V_a = sum c_a f
// (double-float) and Sh = sum h: E = xi0^2 S, M = xi0 V,
// E^2 - |M|^2 = xi0^2 (xi0^2 S^2 - |V|^2) formed in double-float,
// P = (E^2 - |M|^2) / (E + sqrt(E^2 + 3 (E^2 - |M|^2))), gamma^2 = (E + P)/(4 P),
// u' = M / (4 P gamma), n = N^0 / gamma
// (FAST = false: IEEE division, for the macroscopic output)
template <int LAT, bool FAST = true>
__device__ __forceinline__ Mac2 recover2(const df2 &S, const df2 &Vx, const df2 &Vy, const df2 &Vz,
                                         f2 Sh, bool &ok0, bool &ok1)
{
    constexpr float kXi0 = float(Lat<LAT>::xi0), kXi0Sq = float(Lat<LAT>::xi0sq);
    auto dv = [](float a, float b) {
        if constexpr (FAST) return fdiv(a, b);
        else return a / b;
    };
    const df2 V2 = dadd(dadd(sq(Vx), sq(Vy)), sq(Vz));
    const df2 Dr = dadd(dscale(sq(S), Xi0Sq<LAT>::hi, Xi0Sq<LAT>::lo), dneg(V2));
    const f2 D = bc(kXi0Sq) * (Dr.hi + Dr.lo);
    const f2 E = bc(kXi0Sq) * (S.hi + S.lo);
    const f2 root2 = fma2(E, E, bc(3.0f) * D);
    const f2 den = E + f2{sqrtf(root2.x), sqrtf(root2.y)};
    Mac2 m;
    m.P = f2{dv(D.x, den.x), dv(D.y, den.y)};
    const f2 fourP = bc(4.0f) * m.P;
    const f2 g2 = f2{dv(E.x + m.P.x, fourP.x), dv(E.y + m.P.y, fourP.y)};
    const f2 g = f2{sqrtf(g2.x), sqrtf(g2.y)};
    const f2 s = f2{dv(kXi0, fourP.x * g.x), dv(kXi0, fourP.y * g.y)};
    m.ux = (Vx.hi + Vx.lo) * s;
    m.uy = (Vy.hi + Vy.lo) * s;
    m.uz = (Vz.hi + Vz.lo) * s;
    m.n = f2{dv(kXi0 * Sh.x, g.x), dv(kXi0 * Sh.y, g.y)};
    ok0 = E.x > 0.0f && D.x > 0.0f && isfinite(m.n.x) && isfinite(s.x);
    ok1 = E.y > 0.0f && D.y > 0.0f && isfinite(m.n.y) && isfinite(s.y);
    return m;
}

// The same recovery in FP64 (REC64 step variant): the double-float sums are
// converted to double exactly (hi + lo), the Landau-frame recovery runs in
// double arithmetic (rlb_device.cuh: recover, IEEE division and square root)
// and its results are rounded once to float for the equilibrium coefficients.
template <int LAT>
__device__ __forceinline__ Mac2 recover2_64(const df2 &S, const df2 &Vx, const df2 &Vy, const df2 &Vz,
                                            const df2 &Hs, bool &ok0, bool &ok1)
{
    constexpr double xi0 = Lat<LAT>::xi0, xi0sq = Lat<LAT>::xi0sq;
    auto dd = [](float hi, float lo) { return double(hi) + double(lo); };
    Macro a, b;
    ok0 = recover(xi0sq * dd(S.hi.x, S.lo.x), xi0 * dd(Vx.hi.x, Vx.lo.x), xi0 * dd(Vy.hi.x, Vy.lo.x),
                  xi0 * dd(Vz.hi.x, Vz.lo.x), xi0 * dd(Hs.hi.x, Hs.lo.x), a);
    ok1 = recover(xi0sq * dd(S.hi.y, S.lo.y), xi0 * dd(Vx.hi.y, Vx.lo.y), xi0 * dd(Vy.hi.y, Vy.lo.y),
                  xi0 * dd(Vz.hi.y, Vz.lo.y), xi0 * dd(Hs.hi.y, Hs.lo.y), b);
    Mac2 m;
    m.P = f2{float(a.P), float(b.P)};
    m.ux = f2{float(a.ux), float(b.ux)};
    m.uy = f2{float(a.uy), float(b.uy)};
    m.uz = f2{float(a.uz), float(b.uz)};
    m.n = f2{float(a.n), float(b.n)};
    return m;
}

// a float sum as a double-float with zero low part
__device__ __forceinline__ df2 as_df2(f2 v) { return df2{v, bc(0.0f)}; }

// tau from eta/s (Eq. 41 with the entropy of Sec. III), float
template <int LAT>
__device__ __forceinline__ float tau1(float P, float n, float eta_over_s)
{
    const float T = fdiv(P, n);
    const float lam = fdiv(n * float(kPi2Over16), T * T * T);
    const float sfac = fmaxf(4.0f - flog(lam), float(kSMin));
    return 0.5f + fdiv(Lat<LAT>::f_nu2 * eta_over_s * sfac, 4.0f * T);
}

// streaming increment of population I along axis A for the pair (+ bulk lap)
template <bool IS_F, int I, int A, int LAT, typename Src>
__device__ __forceinline__ void axis2(const Src &src, const float (&xv)[6], f2 C, float k1, float k2, float hl,
                                      f2 &inc, f2 &lap)
{
    constexpr int sb = 3 * A;   // first staging slot of axis A (A = 1, 2)
    constexpr int c = cdir<I, A, LAT>();
    constexpr bool need_lap = IS_F && I != 0;
    const float k = (c == 1 || c == -1) ? k1 : k2;
    if constexpr (A == 0) {
        if constexpr (c > 0) {
            const float dm3 = xv[1] - xv[0], dm1 = xv[2] - xv[1], dp1 = xv[3] - xv[2], dp3 = xv[4] - xv[3];
            const float mA = mm(dp1, dm1), mB = mm(dm1, dm3), mC = mm(dp3, dp1);
            const f2 D = fma2(bc(hl), mk(mA, mC) - mk(mB, mA), mk(dm1, dp1));
            inc = fma2(bc(-k), D, inc);
            if constexpr (need_lap) lap = lap + (mk(dp1, dp3) - mk(dm1, dp1));
        } else if constexpr (c < 0) {
            const float dm1 = xv[2] - xv[1], dp1 = xv[3] - xv[2], dp3 = xv[4] - xv[3], dp5 = xv[5] - xv[4];
            const float m1 = mm(dm1, dp1), m2 = mm(dp1, dp3), m3 = mm(dp3, dp5);
            const f2 D = fma2(bc(-hl), mk(m2, m3) - mk(m1, m2), mk(dp1, dp3));
            inc = fma2(bc(k), D, inc);
            if constexpr (need_lap) lap = lap + (mk(dp1, dp3) - mk(dm1, dp1));
        } else if constexpr (need_lap) {
            const float dm1 = xv[2] - xv[1], dp1 = xv[3] - xv[2], dp3 = xv[4] - xv[3];
            lap = lap + (mk(dp1, dp3) - mk(dm1, dp1));
        }
    } else {
        if constexpr (c > 0) {
            const f2 Aq = src.template nb<A, -2>(sb);
            const f2 B = src.template nb<A, -1>(sb + 1);
            const f2 Dq = src.template nb<A, 1>(sb + 2);
            const f2 d0 = B - Aq, d1 = C - B, d2 = Dq - C;
            const f2 Dv = fma2(bc(hl), mm(d2, d1) - mm(d1, d0), d1);
            inc = fma2(bc(-k), Dv, inc);
            if constexpr (need_lap) lap = lap + (d2 - d1);
        } else if constexpr (c < 0) {
            const f2 B = src.template nb<A, -1>(sb);
            const f2 Dq = src.template nb<A, 1>(sb + 1);
            const f2 Eq = src.template nb<A, 2>(sb + 2);
            const f2 e0 = C - B, e1 = Dq - C, e2 = Eq - Dq;
            const f2 Dv = fma2(bc(-hl), mm(e1, e2) - mm(e0, e1), e1);
            inc = fma2(bc(k), Dv, inc);
            if constexpr (need_lap) lap = lap + (e1 - e0);
        } else if constexpr (need_lap) {
            const f2 B = src.template nb<A, -1>(sb);
            const f2 Dq = src.template nb<A, 1>(sb + 1);
            lap = lap + ((Dq - C) - (C - B));
        }
    }
}

// f (or h) + streaming (+ bulk) of population I for the pair: the explicit part of Eq. 57
template <int DIM, bool IS_F, int I, int LAT, bool ODDP, typename Src>
__device__ __forceinline__ f2 streamed2(const Src &src, unsigned xfix, float ghost, float k1, float k2, float hl,
                                        float kb)
{
    constexpr bool xneed = cdir<I, 0, LAT>() != 0 || (IS_F && I != 0);
    float xv[6];
    f2 C;
    if constexpr (xneed) {
        xstencil<ODDP>(src, xfix, ghost, xv);
        C = mk(xv[2], xv[3]);
    } else {
        C = src.get(1);
    }
    f2 inc = bc(0.0f), lap = bc(0.0f);
    if constexpr (xneed) axis2<IS_F, I, 0, LAT>(src, xv, C, k1, k2, hl, inc, lap);
    if constexpr (DIM > 1) axis2<IS_F, I, 1, LAT>(src, xv, C, k1, k2, hl, inc, lap);
    if constexpr (DIM > 2) axis2<IS_F, I, 2, LAT>(src, xv, C, k1, k2, hl, inc, lap);
    if constexpr (IS_F && I != 0) inc = fma2(bc(kb), lap, inc);
    return C + inc;
}

// ---------------------------------------------------------------------------
// Sources and destinations of one pair's update (the IO of update_pair).  An
// item is one class of f (J < NP) or of h (J - NP):
//   begin()          start the loads of the first items' stencils
//   own<J>()         the pair's own populations
//   pre<S, J>()      the explicit part (streamed2) of item J, the S-th taken
//   put<J>(v)        the new populations
//   prev<K>(), put_prev<K>(v)   the previous level's K-th value
// ---------------------------------------------------------------------------
template <int NP, int J>
struct Item {
    static constexpr bool IS_F = J < NP;
    static constexpr int I = rep<NP>(IS_F ? J : J - NP);
    static constexpr int K = IS_F ? I : 19 + I;   // population of the block
};

// The order in which update_pair takes the items: f then h; in Euler mode f
// and h of each class in turn
template <bool EULER, int NP>
constexpr int item_at(int s)
{
    return EULER ? (s % 2 ? NP + s / 2 : s / 2) : s;
}

// Grids: stencils straight from global memory into registers, kAhead items
// before their use.  Staging them through shared memory by cp.async (two items
// ahead) took 74 % of the L1 data path's wavefronts: every value went through
// it three times.  Distance measured on the 512 x 256 x 256 and 2048 x 1024
// shock-clouds, ms a step at 1 / 2 / 3 / 4 items: 4.29 / 3.78 / 3.55 / 3.97
// and 0.199 / 0.190 / 0.177 / 0.183 (3-D: 92 bytes a thread spilled at 3, none
// at 2); an L2 prefetch of the
// rows ahead on top measured slower (3.59 to 3.76 ms, 0.180 to 0.205 ms).
template <int DIM, bool EULER, int NP, int LAT, bool ODDP>
struct BlockIO {
    const StepParams &p;
    const char *c, *l, *r;        // population 0 of the pairs at x0, x0-2, x0+2 (mapped)
    const char *y[4], *z[4];      // of the rows at y-2, y-1, y+1, y+2 and the planes at z-2 .. z+2 (mapped)
    const char *e;                // ODDP: of the extra value (XF_LO_EX, XF_HI_EX)
    char *o;                      // of the pair in the buffer written
    float *pv;                    // previous level of the pair
    unsigned xfix;
    float kb;
    static constexpr int kAhead = EULER ? 2 : (DIM == 1 ? 4 : 3);
    Sten st[kAhead + 1];

    static constexpr int NI = 2 * NP;

    template <int K>
    static __device__ __forceinline__ f2 ld(const char *q)
    {
        f2 v;
        asm volatile("ld.global.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "l"(q), "n"(K * kBlk * 4));
        return v;
    }
    template <int J>
    __device__ __forceinline__ void load(Sten &s) const
    {
        using T = Item<NP, J>;
        constexpr bool need_lap = T::IS_F && T::I != 0;
        constexpr int cx = cdir<T::I, 0, LAT>(), cy = cdir<T::I, 1, LAT>(), cz = cdir<T::I, 2, LAT>();
        if constexpr (cx != 0 || need_lap) {
            s.v[0] = ld<T::K>(l);
            s.v[2] = ld<T::K>(r);
            if constexpr (ODDP) {
                s.ex = 0.0f;
                if (xfix & (XF_LO_EX | XF_HI_EX))
                    asm volatile("ld.global.f32 %0, [%1+%2];" : "=f"(s.ex) : "l"(e), "n"(T::K * kBlk * 4));
            }
        }
        s.v[1] = ld<T::K>(c);
        auto axis = [&](auto ac, const char *const (&q)[4]) {
            constexpr int A = decltype(ac)::value;
            constexpr int cc = A == 1 ? cy : cz;
            if constexpr (cc > 0) {
                s.v[3 * A] = ld<T::K>(q[0]);
                s.v[3 * A + 1] = ld<T::K>(q[1]);
                s.v[3 * A + 2] = ld<T::K>(q[2]);
            } else if constexpr (cc < 0) {
                s.v[3 * A] = ld<T::K>(q[1]);
                s.v[3 * A + 1] = ld<T::K>(q[2]);
                s.v[3 * A + 2] = ld<T::K>(q[3]);
            } else if constexpr (need_lap) {
                s.v[3 * A] = ld<T::K>(q[1]);
                s.v[3 * A + 1] = ld<T::K>(q[2]);
            }
        };
        if constexpr (DIM > 1) axis(std::integral_constant<int, 1>{}, y);
        if constexpr (DIM > 2) axis(std::integral_constant<int, 2>{}, z);
    }
    __device__ __forceinline__ void begin()
    {
        for_pops(std::make_integer_sequence<int, kAhead>{}, [&](auto sc) {
            constexpr int S = decltype(sc)::value;
            load<item_at<EULER, NP>(S)>(st[S]);
        });
    }
    template <int J>
    __device__ __forceinline__ f2 own() const
    {
        return ld<Item<NP, J>::K>(c);
    }
    template <int S, int J>
    __device__ __forceinline__ f2 pre()
    {
        using T = Item<NP, J>;
        if constexpr (S + kAhead < NI) load<item_at<EULER, NP>(S + kAhead)>(st[(S + kAhead) % (kAhead + 1)]);
        const RegSrc src{st[S % (kAhead + 1)]};
        return streamed2<DIM, T::IS_F, T::I, LAT, ODDP>(src, xfix, T::IS_F ? p.f_ghost_f[T::I] : p.f_ghost_h[T::I],
                                                        p.f_k1, p.f_k2, p.f_half_lim, kb);
    }
    template <int J>
    __device__ __forceinline__ void put(f2 v) const
    {
        *reinterpret_cast<float2 *>(o + Item<NP, J>::K * kBlk * 4) = make_float2(v.x, v.y);
    }
    template <int K>
    __device__ __forceinline__ f2 prev() const
    {
        const float2 v = *reinterpret_cast<const float2 *>(pv + K * kBlk);
        return f2{v.x, v.y};
    }
    template <int K>
    __device__ __forceinline__ void put_prev(f2 v) const
    {
        *reinterpret_cast<float2 *>(pv + K * kBlk) = make_float2(v.x, v.y);
    }
};

// Planes of stride ps (the bulk-staged grids): the own pair and the previous
// level
struct PlaneIO {
    static constexpr int NP = 19;
    const StepParams &p;
    const float *f, *h;
    float *fo, *ho, *pv;
    long long ps;
    int idx0;
    unsigned xfix;
    float kb;
    template <int J>
    __device__ __forceinline__ f2 own() const
    {
        const float *q = (Item<NP, J>::IS_F ? f : h) + Item<NP, J>::I * ps + idx0;
        const float2 v = __ldg(reinterpret_cast<const float2 *>(q));
        return f2{v.x, v.y};
    }
    template <int J>
    __device__ __forceinline__ void put(f2 v) const
    {
        float *q = (Item<NP, J>::IS_F ? fo : ho) + Item<NP, J>::I * ps + idx0;
        *reinterpret_cast<float2 *>(q) = make_float2(v.x, v.y);
    }
    template <int K>
    __device__ __forceinline__ f2 prev() const
    {
        const float2 v = *reinterpret_cast<const float2 *>(pv + K * ps + idx0);
        return f2{v.x, v.y};
    }
    template <int K>
    __device__ __forceinline__ void put_prev(f2 v) const
    {
        *reinterpret_cast<float2 *>(pv + K * ps + idx0) = make_float2(v.x, v.y);
    }
};

// 3-D grids staged by bulk copies (rlb_bulk.cuh)
template <int LAT>
struct BulkIO : PlaneIO {
    Bulk *bk;
    static constexpr int NI = 38;
    __device__ __forceinline__ void begin() {}
    template <int S, int J>
    __device__ __forceinline__ f2 pre()
    {
        using T = Item<NP, J>;
        constexpr int b = J % kBulkBufs;
        constexpr unsigned par = unsigned(J / kBulkBufs) & 1u;
        if (!bk->failed && !mbar_wait(&bk->full[b], par)) {
            bk->failed = true;
            atomicOr(p.status, unsigned(ST_TIMEOUT));
        }
        bk->failed = __any_sync(0xffffffffu, bk->failed);   // warp-uniform: the issue below is warp-wide
        const TileSrc src{bk->ctr + b * kTileFloats, bk->zpl + b * kTileFloats};
        const f2 r = streamed2<3, T::IS_F, T::I, LAT, false>(src, xfix, T::IS_F ? p.f_ghost_f[T::I] : p.f_ghost_h[T::I],
                                                             p.f_k1, p.f_k2, p.f_half_lim, kb);
        // this warp is done with buffer b: it counts itself out, and the
        // warp that counts the last of the 8 refills the buffer with item
        // J + kBulkBufs (release fence before the count, acquire after
        // it, then the generic-to-async proxy fence before the copies
        // overwrite what the other warps read)
        if constexpr (J + kBulkBufs < NI) {
            __syncwarp();
            int last = 0;
            if (bk->lane == 0) {
                asm volatile("fence.acq_rel.cta;" ::: "memory");
                last = (atomicAdd(&bk->done[b], 1) & 7) == 7;
                if (last) asm volatile("fence.acq_rel.cta;" ::: "memory");
            }
            if (__shfl_sync(0xffffffffu, last, 0) && !bk->failed) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                bulk_issue<NP, J + kBulkBufs, LAT>(*bk, p, f, h);
            }
        }
        return r;
    }
};

// The update of one pair of cells (Eq. 57 for f and h), shared by the grid
// kernels and the batched tube kernel.  io: where its values come from and go
// to (above); has1: the pair's second cell is inside the grid; eos = eta/s of
// the cell's grid or tube.
//
// park (viscous step): this thread's slots in shared memory, slot k at
// park[k * pstride]: the h-equilibrium coefficients wait there while the f
// populations are updated (kParkH slots), and with EQ_PARKED the coefficients in
// use too (kEqSlots more), which leaves their registers to the stencils in
// flight.  Grids of 2 and 3 dimensions take EQ_PARKED (3-D: 3.58 ms a step with
// three items in flight; with the f coefficients in registers one item fits,
// 4.15 ms); in one dimension an item is three pairs and registers suffice
// (EQ_FOLD).  EQ_HELD: the bulk-staged kernel (hold_eq).
//
// NP = 7 or 14: the 1-D or 2-D symmetry reduction (see rep and mult); only
// the class representatives are read and written, and the previous level's
// zero sums (sum c_z f; 1-D also sum c_y f) are left alone.
enum { EQ_FOLD, EQ_PARKED, EQ_HELD };
template <bool EULER, int EQ, int NP, int LAT, bool REC64, typename IO>
__device__ __forceinline__ void update_pair(const StepParams &p, IO &io, bool has1, float eos, f2 *park = nullptr,
                                            int pstride = 0)
{
    static_assert(NP == 19 || !EULER, "the symmetry reductions are viscous");
    static_assert(!REC64 || (!EULER && NP == 19), "the FP64 recovery is a variant of the viscous 19-population step");
    io.begin();
    const f2 zero = bc(__uint_as_float(0x80000000u | (unsigned(p.nx) >> 31)));   // see hold_eq

    if constexpr (!EULER) {
        // raw sums of the local populations: S = sum f, V_a = sum c_a f
        // (double-float), Sh = sum h
        df2 S{bc(0.0f), bc(0.0f)}, Vx = S, Vy = S, Vz = S, Hs = S;
        for_pops(std::make_integer_sequence<int, NP>{}, [&](auto kc) {
            constexpr int k = decltype(kc)::value;
            constexpr int I = rep<NP>(k), m = mult<NP>(k);
            const f2 v = io.template own<k>();
            // m c_i v with m and c_i powers of two: exact
            auto scaled = [&](auto wc) {
                constexpr int w = decltype(wc)::value;
                return w == 1 ? v : (w == -1 ? -v : bc(float(w)) * v);
            };
            acc(S, scaled(std::integral_constant<int, m>{}));
            constexpr int cx = cdir<I, 0, LAT>(), cy = cdir<I, 1, LAT>(), cz = cdir<I, 2, LAT>();
            if constexpr (cx != 0) acc(Vx, scaled(std::integral_constant<int, cx * m>{}));
            // under a reduction sum c_y f (1-D) and sum c_z f are zero
            if constexpr (has_vy<NP>() && cy != 0) acc(Vy, scaled(std::integral_constant<int, cy * m>{}));
            if constexpr (has_vz<NP>() && cz != 0) acc(Vz, scaled(std::integral_constant<int, cz * m>{}));
            const f2 hv = io.template own<NP + k>();
            acc(Hs, m == 1 ? hv : bc(float(m)) * hv);
        });
        const f2 Sh = Hs.hi + Hs.lo;
        bool ok0, ok1;
        Mac2 mt;
        if constexpr (REC64) mt = recover2_64<LAT>(S, Vx, Vy, Vz, Hs, ok0, ok1);
        else mt = recover2<LAT>(S, Vx, Vy, Vz, Sh, ok0, ok1);
        if (!ok0 || (has1 && !ok1)) atomicOr(p.status, unsigned(ST_NONPHYSICAL));

        f2 kap;
        {
            float t0, t1;
            if (p.f_tau_override > 0.0f) {
                t0 = t1 = p.f_tau_override;
            } else {
                t0 = tau1<LAT>(mt.P.x, mt.n.x, eos);
                t1 = tau1<LAT>(mt.P.y, mt.n.y, eos);
            }
            const float kw = p.f_kw;
            const float w0 = fdiv(kw, t0), w1 = fdiv(kw, t1);
            kap = f2{fdiv(w0, 1.0f + w0), fdiv(w1, 1.0f + w1)};
        }

        // the previous level holds the raw moment sums of time t - dt, so the
        // targets of 2 f^eq(t) - f^eq(t - dt) are exact: T = 2 S(t) - S(t - dt)
        const f2 Sp = io.template prev<0>();
        const f2 Vpx = io.template prev<1>();
        const f2 Vpy = has_vy<NP>() ? io.template prev<2>() : bc(0.0f);
        const f2 Vpz = has_vz<NP>() ? io.template prev<3>() : bc(0.0f);
        const f2 Shp = io.template prev<4>();
        // the previous level's recovery: the same arithmetic as this level's,
        // from its stored float sums.  Its validity is not checked again: the
        // same sums passed the check as the current level one step earlier
        // (or in rlb_init), and the flags' registers cost spills here.
        Mac2 mp;
        {
            bool okp0, okp1;
            if constexpr (REC64)
                mp = recover2_64<LAT>(as_df2(Sp), as_df2(Vpx), as_df2(Vpy), as_df2(Vpz), as_df2(Shp), okp0, okp1);
            else
                mp = recover2<LAT>(as_df2(Sp), as_df2(Vpx), as_df2(Vpy), as_df2(Vpz), Shp, okp0, okp1);
            (void)okp0;
            (void)okp1;
        }
        const f2 T0 = fma2(bc(2.0f), S.hi + S.lo, -Sp);
        f2 Ta[3];
        Ta[0] = fma2(bc(2.0f), Vx.hi + Vx.lo, -Vpx);
        Ta[1] = fma2(bc(2.0f), Vy.hi + Vy.lo, -Vpy);
        Ta[2] = fma2(bc(2.0f), Vz.hi + Vz.lo, -Vpz);

        // h coefficients of 2 h^eq(t) - h^eq(t - dt) (Eq. 58) and their N^0
        // target, formed now so that mt and mp die before the f loop
        f2 H0, Hb[3], Hd[3], Ho[3];
        {
            f2 L0, Lb[3], Ld[3], Lo[3];
            coef_h2<LAT>(mt, H0, Hb, Hd, Ho);
            coef_h2<LAT>(mp, L0, Lb, Ld, Lo);
            H0 = fma2(bc(2.0f), H0, -L0);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                Hb[j] = fma2(bc(2.0f), Hb[j], -Lb[j]);
                Hd[j] = fma2(bc(2.0f), Hd[j], -Ld[j]);
                Ho[j] = fma2(bc(2.0f), Ho[j], -Lo[j]);
            }
        }
        f2 T0h = fma2(bc(2.0f), Sh, -Shp);
        {
            f2 K0, Kb[3], Kd[3], Ko[3], L0, Lb[3], Ld[3], Lo[3];
            coef_f2<LAT>(mt, K0, Kb, Kd, Ko);
            coef_f2<LAT>(mp, L0, Lb, Ld, Lo);
            K0 = fma2(bc(2.0f), K0, -L0);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                Kb[j] = fma2(bc(2.0f), Kb[j], -Lb[j]);
                Kd[j] = fma2(bc(2.0f), Kd[j], -Ld[j]);
                Ko[j] = fma2(bc(2.0f), Ko[j], -Lo[j]);
            }
            const W2 ef = weigh2<Lat<LAT>::dmag>(K0, Kb, Kd, Ko, float(Lat<LAT>::w0), float(Lat<LAT>::w1), float(Lat<LAT>::w2), T0, Ta);
            // the raw sums of this level become the next step's previous level
            io.template put_prev<0>(S.hi + S.lo);
            io.template put_prev<1>(Vx.hi + Vx.lo);
            if constexpr (has_vy<NP>()) io.template put_prev<2>(Vy.hi + Vy.lo);
            if constexpr (has_vz<NP>()) io.template put_prev<3>(Vz.hi + Vz.lo);
            io.template put_prev<4>(Sh);
            f2 *hp = park + (EQ == EQ_PARKED ? kEqSlots * pstride : 0);
            hp[0] = H0;
            hp[10 * pstride] = T0h;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                hp[(1 + j) * pstride] = Hb[j];
                hp[(4 + j) * pstride] = Hd[j];
                hp[(7 + j) * pstride] = Ho[j];
            }
            f2 held[kEqSlots];
            if constexpr (EQ == EQ_PARKED) park_eq(ef, park, pstride);
            if constexpr (EQ == EQ_HELD) hold_eq(ef, held, zero);
            for_pops(std::make_integer_sequence<int, NP>{}, [&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const f2 pre = io.template pre<k, k>();
                f2 q;
                if constexpr (EQ == EQ_PARKED) q = eq_parked<rep<NP>(k)>(park, pstride);
                else if constexpr (EQ == EQ_HELD) q = eq_parked<rep<NP>(k)>(held, 1);
                else q = eq2<rep<NP>(k)>(ef);
                io.template put<k>(fma2(kap, q - pre, pre));
            });
        }
        {
            const f2 *hp = park + (EQ == EQ_PARKED ? kEqSlots * pstride : 0);
            H0 = hp[0];
            T0h = hp[10 * pstride];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                Hb[j] = hp[(1 + j) * pstride];
                Hd[j] = hp[(4 + j) * pstride];
                Ho[j] = hp[(7 + j) * pstride];
            }
            const W2 eh = weigh2<Lat<LAT>::dmag>(H0, Hb, Hd, Ho, float(Lat<LAT>::wh0), float(Lat<LAT>::wh1), float(Lat<LAT>::wh2), T0h, nullptr);
            f2 held[kEqSlots];
            if constexpr (EQ == EQ_PARKED) park_eq(eh, park, pstride);
            if constexpr (EQ == EQ_HELD) hold_eq(eh, held, zero);
            for_pops(std::make_integer_sequence<int, NP>{}, [&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const f2 pre = io.template pre<NP + k, NP + k>();
                f2 q;
                if constexpr (EQ == EQ_PARKED) q = eq_parked<rep<NP>(k)>(park, pstride);
                else if constexpr (EQ == EQ_HELD) q = eq_parked<rep<NP>(k)>(held, 1);
                else q = eq2<rep<NP>(k)>(eh);
                io.template put<NP + k>(fma2(kap, q - pre, pre));
            });
        }
    } else {
        // Euler mode (Sec. III): f, h <- equilibria of the streamed state
        df2 S{bc(0.0f), bc(0.0f)}, Vx = S, Vy = S, Vz = S, Hs = S;
        for_pops(RLB_F32_POPS, [&](auto ic) {
            constexpr int I = decltype(ic)::value;
            const f2 v = io.template pre<2 * I, I>();
            acc(S, v);
            constexpr int cx = cdir<I, 0, LAT>(), cy = cdir<I, 1, LAT>(), cz = cdir<I, 2, LAT>();
            if constexpr (cx != 0) acc(Vx, cx > 0 ? (cx == 1 ? v : v + v) : (cx == -1 ? -v : -(v + v)));
            if constexpr (cy != 0) acc(Vy, cy > 0 ? (cy == 1 ? v : v + v) : (cy == -1 ? -v : -(v + v)));
            if constexpr (cz != 0) acc(Vz, cz > 0 ? (cz == 1 ? v : v + v) : (cz == -1 ? -v : -(v + v)));
            acc(Hs, io.template pre<2 * I + 1, 19 + I>());
        });
        const f2 Sh = Hs.hi + Hs.lo;
        bool ok0, ok1;
        const Mac2 mt = recover2<LAT>(S, Vx, Vy, Vz, Sh, ok0, ok1);
        if (!ok0 || (has1 && !ok1)) atomicOr(p.status, unsigned(ST_NONPHYSICAL));
        const f2 Ta[3] = {Vx.hi + Vx.lo, Vy.hi + Vy.lo, Vz.hi + Vz.lo};
        f2 K0, Kb[3], Kd[3], Ko[3];
        coef_f2<LAT>(mt, K0, Kb, Kd, Ko);
        const W2 ef = weigh2<Lat<LAT>::dmag>(K0, Kb, Kd, Ko, float(Lat<LAT>::w0), float(Lat<LAT>::w1), float(Lat<LAT>::w2), S.hi + S.lo, Ta);
        coef_h2<LAT>(mt, K0, Kb, Kd, Ko);
        const W2 eh = weigh2<Lat<LAT>::dmag>(K0, Kb, Kd, Ko, float(Lat<LAT>::wh0), float(Lat<LAT>::wh1), float(Lat<LAT>::wh2), Sh, nullptr);
        for_pops(RLB_F32_POPS, [&](auto ic) {
            constexpr int I = decltype(ic)::value;
            io.template put<I>(eq2<I>(ef));
            io.template put<19 + I>(eq2<I>(eh));
        });
        io.template put_prev<0>(S.hi + S.lo);
        io.template put_prev<1>(Ta[0]);
        io.template put_prev<2>(Ta[1]);
        io.template put_prev<3>(Ta[2]);
        io.template put_prev<4>(Sh);
    }
}

// The tile (bx, by, bz) of this block when blocks are taken in slabs of
// slab_by block rows, z-planes in order within a slab (blocks start in the
// order of their linear index): the planes the z-stencils of the resident
// blocks read stay in L2 until the blocks of the neighbouring planes have
// read them, instead of a whole z-plane of the grid per step in z.
// slab_by = 0 or >= the block rows: the plain x, y, z order.
__device__ __forceinline__ void slab_order(int slab_by, unsigned &bx, unsigned &by, unsigned &bz)
{
    const unsigned nbx = gridDim.x, nby = gridDim.y, nbz = gridDim.z, sb = unsigned(slab_by);
    if (sb == 0u || sb >= nby) return;
    const unsigned L = blockIdx.x + nbx * (blockIdx.y + nby * blockIdx.z);
    const unsigned s = L / (nbx * sb * nbz);
    const unsigned rows = min(sb, nby - s * sb);
    const unsigned r = L - s * (nbx * sb * nbz);
    bz = r / (nbx * rows);
    const unsigned q = r - bz * (nbx * rows);
    by = s * sb + q / nbx;
    bx = q - (q / nbx) * nbx;
}

#ifndef RLB_F32_MINB
#define RLB_F32_MINB 2
#endif
#ifndef RLB_F32_BY
#define RLB_F32_BY 8
#endif

// threads per block of the 1-D form: one size for all lengths.  us a step with 32 /
// 64 / 128, all populations (1-D reduction): 200 cells 5.28 / 5.22 / 5.36 (3.12 /
// 3.17 / 3.21), 800 6.12 / 5.83 / 5.20 (3.61 / 3.46 / 3.22), 2000 6.35 / 6.23 /
// 5.74, 8192 6.41 / 6.68 / 6.64 (3.72 / 4.12 / 4.07), 20000 6.89 / 6.55 / 6.44,
// 200000 16.15 / 16.02 / 15.93; where 128 is not the best it loses 3 % (9 %)
constexpr int kTubeThreads = 128;
constexpr int kParkH = 11;   // f2 slots per thread in shared memory of the parked h coefficients
// dynamic shared memory of one block of nthr threads
constexpr size_t park_bytes(int nthr, int dim) { return sizeof(f2) * size_t(nthr) * (kParkH + (dim > 1 ? kEqSlots : 0)); }

// NP = 14: the 2-D symmetry reduction (DIM = 2, viscous step).  ODDP: nx odd
// with a periodic x face.  LIN: blocks of one row of 32 BY threads take
// consecutive cell pairs t of the storage order (rows of nxe / 2 pairs), for
// grids whose nx does not fill the tiles; otherwise blocks of 32 x BY threads
// take tiles of 64 x BY cells in one z-plane (the 1-D form: one row of tiles)
template <int DIM, bool EULER, bool ODDP, int LAT, int NP = 19, bool LIN = false, bool REC64 = false>
__global__ void __launch_bounds__(32 * RLB_F32_BY, RLB_F32_MINB)
    step_f32_kernel(const StepParams p, const float *__restrict__ f, float *__restrict__ fo, float *__restrict__ prev)
{
    extern __shared__ f2 s_park[];
    const int nxe = p.nx + (p.nx & 1);
    int x0, y, z;
    if constexpr (LIN) {
        const unsigned ppr = unsigned(nxe) >> 1;
        const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
        const unsigned row = t / ppr;
        x0 = 2 * int(t - row * ppr);
        y = int(row % unsigned(p.ny));
        z = int(row / unsigned(p.ny));
        if (z >= p.nz) return;
    } else {
        unsigned bx = blockIdx.x, by = blockIdx.y, bz = blockIdx.z;
        if constexpr (DIM == 3) slab_order(p.slab_by, bx, by, bz);
        x0 = 2 * (bx * blockDim.x + threadIdx.x);
        y = by * blockDim.y + threadIdx.y;
        z = bz;
        if (x0 >= p.nx || y >= p.ny) return;
    }
    const int i0 = x0 + nxe * (y + p.ny * z);
    const bool has1 = x0 + 1 < p.nx;
    const char *base = reinterpret_cast<const char *>(f);
    auto at = [&](int i) { return base + sizeof(float) * blk_at(i); };

    BlockIO<DIM, EULER, NP, LAT, ODDP> io{p};
    io.c = at(i0);
    io.o = reinterpret_cast<char *>(fo) + (io.c - base);
    io.pv = prev + blk_prev_at(i0);
    io.kb = p.f_kbulk;
    // a row of one cell: the periodic neighbour is the cell itself (clamped)
    const int lo = p.nx == 1 && p.bc_lo[0] == BC_PERIODIC ? int(BC_OUTFLOW) : p.bc_lo[0];
    const int hi = p.nx == 1 && p.bc_hi[0] == BC_PERIODIC ? int(BC_OUTFLOW) : p.bc_hi[0];
    int ol = -2, orr = 2;
    unsigned xfix = 0u;
    if (x0 == 0) {   // x0-2, x0-1 are outside
        ol = 0;
        if (lo != BC_PERIODIC) xfix |= lo == BC_OUTFLOW ? XF_LO_CLAMP : XF_LO_GHOST;
        else if (ODDP) { ol = p.nx - 3; xfix |= XF_LO_EX; }
        else ol = p.nx - 2;
    }
    if (x0 + 2 >= p.nx) {   // x0+2, x0+3 are outside (and x0+1 at the end of an odd row)
        orr = 0;
        if (hi == BC_PERIODIC) {
            orr = -x0;
            if (ODDP && !has1) xfix |= XF_HI_WRAP1;
        } else if (has1) {
            xfix |= hi == BC_OUTFLOW ? XF_HI_CLAMP : XF_HI_GHOST;
        } else {
            xfix |= hi == BC_OUTFLOW ? XF_HI_ODD1 : XF_HI_ODD1G;
        }
    } else if (x0 + 3 == p.nx) {   // x0+3 is outside
        if (hi != BC_PERIODIC) xfix |= hi == BC_OUTFLOW ? XF_HI_ODD3 : XF_HI_ODD3G;
        else xfix |= x0 == 0 ? XF_HI_SELF : XF_HI_EX;
    }
    io.l = at(i0 + ol);
    io.r = at(i0 + orr);
    if constexpr (ODDP) io.e = at(i0 + ((xfix & XF_LO_EX) ? p.nx - 1 : ((xfix & XF_HI_EX) ? -x0 : 0)));
    io.xfix = xfix;
    {
        const int ds[4] = {-2, -1, 1, 2};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (DIM > 1) io.y[k] = at(i0 + (map1(y + ds[k], p.ny, p.bc_lo[1], p.bc_hi[1]) - y) * nxe);
            if constexpr (DIM > 2) io.z[k] = at(i0 + (map1(z + ds[k], p.nz, p.bc_lo[2], p.bc_hi[2]) - z) * nxe * p.ny);
        }
    }
    grid_wait();
    // threads per block as the launcher sets them (rlb_step_f32_launch.cuh), a
    // compile-time constant so that the shared-memory slots of this thread
    // sit at fixed offsets from one base address
    constexpr int nthr = (DIM == 1 && !LIN) ? kTubeThreads : 32 * RLB_F32_BY;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    update_pair<EULER, (DIM > 1) ? EQ_PARKED : EQ_FOLD, NP, LAT, REC64>(p, io, has1, p.f_eta_over_s, s_park + tid, nthr);
}

}  // namespace f32
}  // namespace rlb
