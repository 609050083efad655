// rlb_kernels.cuh -- kernels of the fused RLB time step.
//
// One thread updates one cell: it reads the 19 + 19 local populations,
// forms the moments and the Landau-frame macroscopic state of time t,
// evaluates the extrapolated equilibria 2 f^eq(t) - f^eq(t - dt) from the
// current and the stored previous macroscopic state, streams every
// population with the minmod flux difference of its own neighbours
// (plus the bulk Laplacian for f), applies the implicit update of Eq. 57
// and writes the populations of t + dt and the macroscopic state of t.
#pragma once

#include <utility>

#include "rlb_classes.cuh"
#include "rlb_device.cuh"
#include "rlb_internal.h"

namespace rlb {

template <int... Is, typename F>
__device__ __forceinline__ void for_pops(std::integer_sequence<int, Is...>, F &&fn)
{
    (fn(std::integral_constant<int, Is>{}), ...);
}
#define RLB_POPS std::make_integer_sequence<int, 19>{}

// plain loads, after grid_wait (not the read-only path: see there)
template <typename T>
__device__ __forceinline__ T ldg(const T *p)
{
    static_assert(sizeof(T) == 8, "the FP64 form");
    T v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

// value of a neighbour (slot k of the axis map) or the inlet ghost value
template <typename T>
__device__ __forceinline__ T nbr(const T *q, int idx, const AxisNbr &a, int k, T ghost)
{
    return ((a.ghost >> k) & 1u) ? ghost : ldg(q + idx + a.off[k]);
}

// f + streaming (+ bulk) of a population: the explicit part of Eq. 57.  v[a]:
// its values at -1, +1 and, upwind, -2 or +2 along axis a; way: the
// population's steps along the axes and whether it carries the bulk term
// (way_of).  Along each axis it moves on, the sum receives minus dt (c0/ct)
// times the conservative minmod flux difference h^a(x) - h^a(x - e_a) (Eqs.
// 47-53).  The bulk term's central second difference sum_A [q(x + e_A) -
// 2 q(x) + q(x - e_A)] is taken as s - 2 DIM q(x) in one fused operation
// (exact coefficients, so that its sum over a periodic grid carries no
// systematic rounding).
constexpr int kWayBulk = 512;
constexpr int way_of(int cx, int cy, int cz, bool bulk)
{
    return (cx + 2) | (cy + 2) << 3 | (cz + 2) << 6 | (bulk ? kWayBulk : 0);
}
struct Sten64 {
    double v[3][3];
};
template <int DIM>
__device__ __forceinline__ double streamed(const Sten64 &q, double qc, double k1, double k2, double hl, double kbulk,
                                           int way)
{
    double acc = qc, s = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int c = ((way >> 3 * a) & 7) - 2;
        const double (&v)[3] = q.v[a];
        if (c > 0) {
            const double d0 = v[0] - v[2], d1 = qc - v[0], d2 = v[1] - qc;
            const double D = fma(hl, minmod(d2, d1) - minmod(d1, d0), d1);
            acc = fma(-(c == 1 ? k1 : k2), D, acc);
        } else if (c < 0) {
            const double e0 = qc - v[0], e1 = v[1] - qc, e2 = v[2] - v[1];
            const double D = fma(-hl, minmod(e1, e2) - minmod(e0, e1), e1);
            acc = fma(c == -1 ? k1 : k2, D, acc);
        }
        if (way & kWayBulk) {
            if (a == 0) s = v[1] + v[0];
            else s += v[1] + v[0];
        }
    }
    if (way & kWayBulk) acc = fma(kbulk, fma(double(-2 * DIM), qc, s), acc);
    return acc;
}
template <int DIM>
__device__ __noinline__ double streamed_called(const Sten64 q, double qc, double k1, double k2, double hl, double kbulk,
                                               int way)
{
    return streamed<DIM>(q, qc, k1, k2, hl, kbulk, way);
}

// ---------------------------------------------------------------------------
// The same explicit part with the differences, the limiter and the Laplacian
// in 64-bit fixed point.  GB300 issues FP64 operations at 1/64 of the float
// rate and the integer pipes are idle beside them, so the 19 FP64 operations
// of a diagonal population's stencil (12 of an axis one) are replaced by
// integer ones and 4 FP64 operations (two conversions, two fused
// multiply-adds); the step needs 378 fewer of its 1208 FP64 operations a cell.
//
// The stencil's values are written as integers in units of 2^(E - 1081), E
// the largest biased exponent among them, i.e. with their 53 bits shifted up
// by at most kFxGap: every value whose exponent lies within kFxGap of E is
// represented exactly, so differences, limited slopes and second differences
// are exact (in FP64 each rounds).  Headroom: values < 2^59, differences <
// 2^60, 2 D per axis < 2^62, two axes and the Laplacian (< 6 2^60) < 2^63.
// Stencils with a wider spread of exponents, zeros, subnormal or non-finite
// values take the FP64 form above: inlined at every population (FX_INLINE), or
// one function that they all call (FX_CALL).  Inlined it makes the code of a
// step about twice as long, and a kernel with a warp or two per scheduler waits
// for instructions: the four-warp kernel (step_split_kernel) takes 22 us a step
// on 64 x 64 cells inlined, 18.2 called, and in 3-D 151 registers, with which a
// fourth block does not fit on an SM (32 x 32 x 18 cells 64 us), or 126 (34 us);
// tiles with a block or less an SM 58.4 us on 16 x 16 x 8 cells, 50.6 called.
// With four warps per scheduler the call costs more than it saves (1024 x 512
// cells 690 us inlined, 756 called), but not in Euler mode, whose streaming is
// all in one loop (64 x 64 cells 34.7 and 27.4, 256 x 128 x 128 5080 and 4310).
// FX_NONE: the FP64 form alone, for 1-D tubes in Euler mode with one warp per
// scheduler, which gain nothing from the fixed point (800 cells 23.5 us called,
// 20.7 so).
// ---------------------------------------------------------------------------
enum { FX_INLINE, FX_CALL, FX_NONE };
constexpr int kFxGap = 6;

__device__ __forceinline__ long long to_fx(double x, int e0)   // e0 = E - kFxGap
{
    const int hi = __double2hiint(x);
    const unsigned mh = (unsigned(hi) & 0xfffffu) | 0x100000u;
    const unsigned long long m = (static_cast<unsigned long long>(mh) << 32) | unsigned(__double2loint(x));
    const int sh = ((hi >> 20) & 0x7ff) - e0;
    const long long v = static_cast<long long>(m << sh);
    const long long sg = hi >> 31;
    return (v ^ sg) - sg;
}
// minmod(a, b) of Eq. 53: a clamped between 0 and b
__device__ __forceinline__ long long fx_minmod(long long a, long long lo, long long hi)
{
    const long long m = a < hi ? a : hi;
    return m > lo ? m : lo;
}
// k 2^(E - 1081) for a positive normal k (exponent arithmetic on its bits)
__device__ __forceinline__ double fx_scaled(double k, int e)
{
    return __hiloint2double(__double2hiint(k) + ((e - 1081) << 20), __double2loint(k));
}

// gap: kFxGap, or -1 when a prefactor is too small for fx_scaled (the FP64 form
// is taken); lim: -1 for the minmod limiter, 0 for none
template <int DIM, bool IS_F, int I, int LAT, int FORM>
__device__ __forceinline__ double streamed_fx(const double *q, int idx, const AxisNbr (&am)[3], double qc, double ghost,
                                              double k1, double k2, double hl, double kbulk, int gap, long long lim)
{
    constexpr bool need_lap = IS_F && I != 0;
    constexpr int c[3] = {cdir<I, 0, LAT>(), DIM > 1 ? cdir<I, 1, LAT>() : 0, DIM > 2 ? cdir<I, 2, LAT>() : 0};
    constexpr bool moves = c[0] != 0 || c[1] != 0 || c[2] != 0;
    if constexpr (!moves && !need_lap) {
        return qc;
    } else {
        Sten64 st = {};
        double (&v)[3][3] = st.v;
        auto load = [&](auto &&take) {
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                if (c[a] != 0 || need_lap) {
                    v[a][0] = take(nbr(q, idx, am[a], 1, ghost));
                    v[a][1] = take(nbr(q, idx, am[a], 2, ghost));
                }
                if (c[a] > 0) v[a][2] = take(nbr(q, idx, am[a], 0, ghost));
                if (c[a] < 0) v[a][2] = take(nbr(q, idx, am[a], 3, ghost));
            }
        };
        constexpr int way = way_of(c[0], c[1], c[2], need_lap);
        auto same = [](double x) { return x; };
        if constexpr (FORM == FX_NONE) {
            load(same);
            return streamed<DIM>(st, qc, k1, k2, hl, kbulk, way);
        }
        unsigned hx = unsigned(__double2hiint(qc)) & 0x7fffffffu, hn = hx;
        load([&](double x) {
            const unsigned h = unsigned(__double2hiint(x)) & 0x7fffffffu;
            hx = max(hx, h);
            hn = min(hn, h);
            return x;
        });
        const int E = int(hx >> 20), En = int(hn >> 20);
        if (E - En > gap || E >= 0x7ff || En < 512) {
            if constexpr (FORM == FX_CALL) {
                return streamed_called<DIM>(st, qc, k1, k2, hl, kbulk, way);
            } else {
                load(same);   // again, rather than held for a branch that is seldom taken
                return streamed<DIM>(st, qc, k1, k2, hl, kbulk, way);
            }
        }
        const int e0 = E - kFxGap;
        const long long fc = to_fx(qc, e0);
        long long T = 0, L = 0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            if (c[a] == 0 && !need_lap) continue;
            const long long m1 = to_fx(v[a][0], e0), p1 = to_fx(v[a][1], e0);
            const long long dm = fc - m1, dp = p1 - fc;   // across x - 1/2 and x + 1/2
            if (c[a] > 0) {
                const long long dd = m1 - to_fx(v[a][2], e0);
                const long long lo = dm < 0 ? dm : 0, hi = dm < 0 ? 0 : dm;
                T -= 2 * dm + (lim & (fx_minmod(dp, lo, hi) - fx_minmod(dd, lo, hi)));
            } else if (c[a] < 0) {
                const long long dd = to_fx(v[a][2], e0) - p1;
                const long long lo = dp < 0 ? dp : 0, hi = dp < 0 ? 0 : dp;
                T += 2 * dp - (lim & (fx_minmod(dd, lo, hi) - fx_minmod(dm, lo, hi)));
            }
            if (need_lap) L += dp - dm;
        }
        double acc = qc;
        if constexpr (moves) {
            constexpr int cm = c[0] != 0 ? c[0] : (c[1] != 0 ? c[1] : c[2]);
            acc = fma(fx_scaled(0.5 * (cm == 1 || cm == -1 ? k1 : k2), E), double(T), acc);
        }
        if constexpr (need_lap) {
            if (kbulk != 0.0) acc = fma(fx_scaled(kbulk, E), double(L), acc);
        }
        return acc;
    }
}

// The moment sums are taken in four parts: the rest and axis populations, and
// the diagonals of the xy, xz and yz planes.  Mirror images stay together and
// in the order +, -, so that a component that vanishes by symmetry sums to
// exactly zero (a part cut across such pairs left 1e-16, which grows over
// thousands of steps).  step_split_kernel gives each part to a warp; the two
// kernels agree bit for bit.
constexpr int part_of(int i) { return i < 7 ? 0 : 1 + (i - 7) / 4; }
// class K is the first of its part that moves along axis A (A = 3: the first)
template <int NP, int A, int K>
constexpr bool first_of_part()
{
    bool first = true;
    [&]<int... J>(std::integer_sequence<int, J...>) {
        ((first = first && !(J < K && part_of(rep<NP>(J)) == part_of(rep<NP>(K)) &&
                             (A == 3 || (A == 0 ? kDir[rep<NP>(J)].x : (A == 1 ? kDir[rep<NP>(J)].y : kDir[rep<NP>(J)].z)) != 0))), ...);
    }(std::make_integer_sequence<int, NP>{});
    return first;
}
template <bool FIRST>
__device__ __forceinline__ void add_to(double &s, double c, double v)
{
    if constexpr (FIRST) s = c * v;
    else s += c * v;
}

template <typename T>
__device__ __forceinline__ void flag(const StepParams &p, unsigned bits)
{
    atomicOr(p.status, bits);
}

// LIN: blocks of one row of threads take consecutive cells of the x-fastest
// order (grids whose nx, ny do not fill the tiles); otherwise blocks of
// 32 x 4 threads take tiles of 32 x 4 cells in one z-plane (the 1-D form:
// one row of tiles)
// NP = 7 or 14: the 1-D or 2-D symmetry reduction (rlb_classes.cuh); only
// the class representatives' planes are read and written
//
// Bound by the FP64 pipe (631 operations a cell, 1208 before the fixed-point
// streaming and the shared sums) together with the latency of its chains, so
// warps count: at 128 registers (four blocks of 128 per SM; the own
// populations are loaded again rather than held) the 256 x 128 x 128 cloud
// takes 6.3 ms a step, with two, three and five blocks 8.6, 6.8 and 6.6 (9.9
// before, at 255 registers).  At 128 it spills 76 to 140 bytes a thread in 3-D, up
// to 52 in 2-D.
#ifndef RLB_F64_MINB
#define RLB_F64_MINB 4
#endif
template <typename T, int DIM, bool EULER, int LAT, bool LIN = false, int NP = 19, int FORM = EULER ? FX_CALL : FX_INLINE>
__global__ void __launch_bounds__(128, RLB_F64_MINB) step_kernel(const StepParams p, const T *__restrict__ f,
                                                   const T *__restrict__ h, T *__restrict__ fo,
                                                   T *__restrict__ ho, T *__restrict__ prev)
{
    int x, y, z;
    if constexpr (LIN) {
        const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
        const unsigned row = t / unsigned(p.nx);
        x = int(t - row * unsigned(p.nx));
        y = int(row % unsigned(p.ny));
        z = int(row / unsigned(p.ny));
        if (z >= p.nz) return;
    } else {
        x = blockIdx.x * blockDim.x + threadIdx.x;
        y = blockIdx.y * blockDim.y + threadIdx.y;
        z = blockIdx.z;
        if (x >= p.nx || y >= p.ny) return;
    }
    const int idx = x + p.nx * (y + p.ny * z);
    const long long ps = p.ps;

    AxisNbr am[3];
    am[0] = axis_map(x, p.nx, 1, p.bc_lo[0], p.bc_hi[0]);
    if (DIM > 1) am[1] = axis_map(y, p.ny, p.nx, p.bc_lo[1], p.bc_hi[1]);
    if (DIM > 2) am[2] = axis_map(z, p.nz, p.nx * p.ny, p.bc_lo[2], p.bc_hi[2]);

    const T k1 = T(p.k1), k2 = T(p.k2), hl = T(p.half_lim), kbulk = T(p.kbulk);
    // (stencils in fixed point have exponents of at least 512)
    const int gap = k1 > 1e-60 && (kbulk == 0.0 || kbulk > 1e-60) ? kFxGap : -1;
    const long long lim = hl != 0.0 ? -1LL : 0LL;
    grid_wait();

    static_assert(NP == 19 || (NP == 7 && DIM == 1 && !EULER) || (NP == 14 && DIM == 2 && !EULER),
                  "the symmetry reductions are 1-D or 2-D and viscous");
    if constexpr (!EULER) {
        // moments of f(t), h(t) at the cell (Eq. 36 with p_i^0 = xi0); class k
        // counts mult(k) equal populations (powers of two: exact scaling)
        // (parts: part_of)
        double sf[4] = {0.0, 0.0, 0.0, 0.0}, sh[4] = {0.0, 0.0, 0.0, 0.0}, mx[4] = {0.0, 0.0, 0.0, 0.0},
               my[4] = {0.0, 0.0, 0.0, 0.0}, mz[4] = {0.0, 0.0, 0.0, 0.0};
        for_pops(std::make_integer_sequence<int, NP>{}, [&](auto kc) {
            constexpr int k = decltype(kc)::value;
            constexpr int I = rep<NP>(k), m = mult<NP>(k), w = part_of(I);
            const double fv = ldg(f + I * ps + idx), hv = ldg(h + I * ps + idx);
            constexpr int cx = cdir<I, 0, LAT>(), cy = cdir<I, 1, LAT>(), cz = cdir<I, 2, LAT>();
            add_to<first_of_part<NP, 3, k>()>(sf[w], double(m), fv);
            add_to<first_of_part<NP, 3, k>()>(sh[w], double(m), hv);
            if constexpr (cx != 0) add_to<first_of_part<NP, 0, k>()>(mx[w], double(cx * m), fv);
            if constexpr (has_vy<NP>() && cy != 0) add_to<first_of_part<NP, 1, k>()>(my[w], double(cy * m), fv);
            if constexpr (has_vz<NP>() && cz != 0) add_to<first_of_part<NP, 2, k>()>(mz[w], double(cz * m), fv);
        });
        auto sum4 = [](const double (&s)[4]) { return (s[0] + s[1]) + (s[2] + s[3]); };
        MacroG mt;
        const bool ok = recover_g(Lat<LAT>::xi0sq * sum4(sf), Lat<LAT>::xi0 * sum4(mx), Lat<LAT>::xi0 * sum4(my),
                                  Lat<LAT>::xi0 * sum4(mz), Lat<LAT>::xi0 * sum4(sh), mt);
        if (!ok) flag<T>(p, ST_NONPHYSICAL);
        const double tau = p.tau_override > 0.0 ? p.tau_override : tau_of<LAT>(mt.P, mt.n, p.eta_over_s);
        // f(t+dt) = pre + kappa (G - pre), kappa = omega / (1 + omega) with
        // omega = kw / tau: Eq. 57 solved for f(t+dt), in the form whose
        // rounding does not scale the conserved sums
        const T kap = T(p.kw / (tau + p.kw));

        MacroG mp;
        mp.P = double(prev[0 * ps + idx]);
        mp.ux = double(prev[1 * ps + idx]);
        mp.uy = double(prev[2 * ps + idx]);
        mp.uz = double(prev[3 * ps + idx]);
        mp.n = double(prev[4 * ps + idx]);
        gamma_of(mp);
        Coef<double> a, b;
        coef_h_g<LAT>(mt, a);
        coef_h_g<LAT>(mp, b);
        const Coef<double> ch = extrapolate(a, b);
        // the h coefficients wait in shared memory during the f loop
        __shared__ double parked[10][128];
        const int tid = threadIdx.x + blockDim.x * threadIdx.y;
        parked[0][tid] = ch.K0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            parked[1 + j][tid] = ch.Kb[j];
            parked[4 + j][tid] = ch.Kd[j];
            parked[7 + j][tid] = ch.Ko[j];
        }
        coef_f_g<LAT>(mt, a);
        coef_f_g<LAT>(mp, b);
        prev[0 * ps + idx] = T(mt.P);
        prev[1 * ps + idx] = T(mt.ux);
        prev[2 * ps + idx] = T(mt.uy);
        prev[3 * ps + idx] = T(mt.uz);
        prev[4 * ps + idx] = T(mt.n);
        {
            const EqP kf = fold<Lat<LAT>::dmag>(extrapolate(a, b), Lat<LAT>::w0, Lat<LAT>::w1, Lat<LAT>::w2);
            for_pops(std::make_integer_sequence<int, NP>{}, [&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr int I = rep<NP>(k);
                const T pre = streamed_fx<DIM, true, I, LAT, FORM>(f + I * ps, idx, am, ldg(f + I * ps + idx),
                                                                   T(p.ghost_f[I]), k1, k2, hl, kbulk, gap, lim);
                fo[I * ps + idx] = fma(kap, eq_pop<I>(kf) - pre, pre);
            });
        }
        {
            Coef<double> c;
            c.K0 = parked[0][tid];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                c.Kb[j] = parked[1 + j][tid];
                c.Kd[j] = parked[4 + j][tid];
                c.Ko[j] = parked[7 + j][tid];
            }
            const EqP kh = fold<Lat<LAT>::dmag>(c, Lat<LAT>::wh0, Lat<LAT>::wh1, Lat<LAT>::wh2);
            for_pops(std::make_integer_sequence<int, NP>{}, [&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr int I = rep<NP>(k);
                const T pre = streamed_fx<DIM, false, I, LAT, FORM>(h + I * ps, idx, am, ldg(h + I * ps + idx),
                                                                    T(p.ghost_h[I]), k1, k2, hl, kbulk, gap, lim);
                ho[I * ps + idx] = fma(kap, eq_pop<I>(kh) - pre, pre);
            });
        }
    } else {
        // Euler mode (Sec. III): f, h <- equilibria of the streamed state
        double sf = 0.0, sh = 0.0, mx = 0.0, my = 0.0, mz = 0.0;
        for_pops(RLB_POPS, [&](auto ic) {
            constexpr int I = decltype(ic)::value;
            const T qc = ldg(f + I * ps + idx);
            const double fv = streamed_fx<DIM, true, I, LAT, FORM>(f + I * ps, idx, am, qc, T(p.ghost_f[I]), k1, k2, hl,
                                                                   kbulk, gap, lim);
            sf += fv;
            if constexpr (cdir<I, 0, LAT>() != 0) mx += double(cdir<I, 0, LAT>()) * fv;
            if constexpr (cdir<I, 1, LAT>() != 0) my += double(cdir<I, 1, LAT>()) * fv;
            if constexpr (cdir<I, 2, LAT>() != 0) mz += double(cdir<I, 2, LAT>()) * fv;
            const T qh = ldg(h + I * ps + idx);
            sh += streamed_fx<DIM, false, I, LAT, FORM>(h + I * ps, idx, am, qh, T(p.ghost_h[I]), k1, k2, hl, kbulk, gap,
                                                        lim);
        });
        Macro mt;
        const bool ok = recover(Lat<LAT>::xi0sq * sf, Lat<LAT>::xi0 * mx, Lat<LAT>::xi0 * my, Lat<LAT>::xi0 * mz, Lat<LAT>::xi0 * sh, mt);
        if (!ok) flag<T>(p, ST_NONPHYSICAL);
        Coef<double> a;
        coef_f<LAT>(mt, a);
        const EqW<T> kf = weigh_f<T, LAT>(a);
        coef_h<LAT>(mt, a);
        const EqW<T> kh = weigh_h<T, LAT>(a);
        for_pops(RLB_POPS, [&](auto ic) {
            constexpr int I = decltype(ic)::value;
            fo[I * ps + idx] = eq_pop<I>(kf);
            ho[I * ps + idx] = eq_pop<I>(kh);
        });
        prev[0 * ps + idx] = T(mt.P);
        prev[1 * ps + idx] = T(mt.ux);
        prev[2 * ps + idx] = T(mt.uy);
        prev[3 * ps + idx] = T(mt.uz);
        prev[4 * ps + idx] = T(mt.n);
    }
}

// ---------------------------------------------------------------------------
// Small grids (viscous step).  One warp issues FP64 instructions at its
// scheduler's share of the pipe, one per 64 clocks, so on a grid with fewer
// warps of cells than schedulers a step takes the time of one warp's FP64
// instructions whatever the number of SMs (31 us a step on an 800-cell tube;
// 13 us here).
// Here the four warps of a block, one per scheduler, share 32 cells: each
// takes the f and h of one part (part_of), and between the moments and the
// relaxation warp 3 recovers the macroscopic state while the others form the
// explicit parts of their populations, then warps 0 and 1 the equilibria of f
// and h and warp 2 tau.
// ---------------------------------------------------------------------------
template <typename F>
__device__ __forceinline__ void by_warp(int w, F &&fn)
{
    if (w == 0) fn(std::integral_constant<int, 0>{});
    else if (w == 1) fn(std::integral_constant<int, 1>{});
    else if (w == 2) fn(std::integral_constant<int, 2>{});
    else fn(std::integral_constant<int, 3>{});
}

// how many items before J are in its part
template <int NP>
constexpr int item_rank(int J)
{
    int reps[NP] = {}, n = 0;
    [&]<int... K>(std::integer_sequence<int, K...>) { ((reps[K] = rep<NP>(K)), ...); }(std::make_integer_sequence<int, NP>{});
    for (int i = 0; i < J; ++i) n += part_of(reps[i < NP ? i : i - NP]) == part_of(reps[J < NP ? J : J - NP]);
    return n;
}

struct FoldedSums {   // EqP of 32 cells in shared memory
    double v[19][32];
    __device__ __forceinline__ void put(const EqP &e, int l)
    {
        v[0][l] = e.r0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            v[1 + j][l] = e.ax[j];
            v[4 + j][l] = e.ab[j];
            v[7 + j][l] = e.p[j];
            v[10 + j][l] = e.m[j];
            v[13 + j][l] = e.s[j];
            v[16 + j][l] = e.t[j];
        }
    }
    template <int I>
    __device__ __forceinline__ double pop(int l) const
    {
        constexpr int cx = cdir<I, 0>(), cy = cdir<I, 1>(), cz = cdir<I, 2>();
        if constexpr (shell<I>() == 0) {
            return v[0][l];
        } else if constexpr (shell<I>() == 1) {
            constexpr int a = cx != 0 ? 0 : (cy != 0 ? 1 : 2);
            return cx + cy + cz > 0 ? v[1 + a][l] + v[4 + a][l] : v[1 + a][l] - v[4 + a][l];
        } else {
            constexpr int ca = cx != 0 ? cx : cy, cb = cz != 0 ? cz : cy;
            constexpr int j = cz == 0 ? 0 : (cx != 0 ? 1 : 2);
            if constexpr (ca > 0) return cb > 0 ? v[7 + j][l] + v[13 + j][l] : v[10 + j][l] + v[16 + j][l];
            else return cb > 0 ? v[10 + j][l] - v[16 + j][l] : v[7 + j][l] - v[13 + j][l];
        }
    }
};

template <int DIM, int LAT, int NP>
__global__ void __launch_bounds__(128) step_split_kernel(const StepParams p, const double *__restrict__ f,
                                                         const double *__restrict__ h, double *__restrict__ fo,
                                                         double *__restrict__ ho, double *__restrict__ prev)
{
    __shared__ double part[4][5][32], mac[7][32], s_kap[32];
    __shared__ FoldedSums kf, kh;
    const int l = threadIdx.x, w = threadIdx.y;
    const long long cells = (long long)p.nx * p.ny * p.nz, cell = 32LL * blockIdx.x + l;
    const bool in = cell < cells;   // lanes past the last cell repeat it and write nothing
    const int idx = int(in ? cell : cells - 1);
    const int row = idx / p.nx, x = idx - row * p.nx, z = row / p.ny, y = row - z * p.ny;
    const long long ps = p.ps;
    AxisNbr am[3];
    am[0] = axis_map(x, p.nx, 1, p.bc_lo[0], p.bc_hi[0]);
    if (DIM > 1) am[1] = axis_map(y, p.ny, p.nx, p.bc_lo[1], p.bc_hi[1]);
    if (DIM > 2) am[2] = axis_map(z, p.nz, p.nx * p.ny, p.bc_lo[2], p.bc_hi[2]);
    const double k1 = p.k1, k2 = p.k2, hl = p.half_lim, kbulk = p.kbulk;
    const int gap = k1 > 1e-60 && (kbulk == 0.0 || kbulk > 1e-60) ? kFxGap : -1;
    const long long lim = hl != 0.0 ? -1LL : 0LL;
    grid_wait();

    constexpr int NI = 2 * NP, NJ = 14;   // the largest part: 7 populations of each kind
    // fn(J, j) for the items J (f class J, else h class J - NP) of this warp,
    // j counting them
    auto items = [&](auto &&fn) {
        by_warp(w, [&](auto wc) {
            for_pops(std::make_integer_sequence<int, NI>{}, [&](auto Jc) {
                constexpr int J = decltype(Jc)::value, W = decltype(wc)::value;
                if constexpr (part_of(rep<NP>(J < NP ? J : J - NP)) == W)
                    fn(Jc, std::integral_constant<int, item_rank<NP>(J)>{});
            });
        });
    };
    double own[NJ];
    {
        double sf = 0.0, sh = 0.0, mx = 0.0, my = 0.0, mz = 0.0;
        items([&](auto Jc, auto jc) {
            constexpr int J = decltype(Jc)::value, k = J < NP ? J : J - NP, I = rep<NP>(k), m = mult<NP>(k);
            const double v = ldg((J < NP ? f : h) + I * ps + idx);
            own[decltype(jc)::value] = v;
            if constexpr (J < NP) {
                sf += double(m) * v;
                if constexpr (cdir<I, 0, LAT>() != 0) mx += double(cdir<I, 0, LAT>() * m) * v;
                if constexpr (has_vy<NP>() && cdir<I, 1, LAT>() != 0) my += double(cdir<I, 1, LAT>() * m) * v;
                if constexpr (has_vz<NP>() && cdir<I, 2, LAT>() != 0) mz += double(cdir<I, 2, LAT>() * m) * v;
            } else {
                sh += double(m) * v;
            }
        });
        part[w][0][l] = sf;
        part[w][1][l] = mx;
        part[w][2][l] = my;
        part[w][3][l] = mz;
        part[w][4][l] = sh;
    }
    Coef<double> b;   // the previous level's: of f in warp 0, of h in warp 1
    if (w < 2) {
        MacroG mp;
        mp.P = prev[0 * ps + idx];
        mp.ux = prev[1 * ps + idx];
        mp.uy = prev[2 * ps + idx];
        mp.uz = prev[3 * ps + idx];
        mp.n = prev[4 * ps + idx];
        gamma_of(mp);
        if (w == 0) coef_f_g<LAT>(mp, b);
        else coef_h_g<LAT>(mp, b);
    }
    __syncthreads();

    double pre[NJ];
    auto explicit_parts = [&]() {
        items([&](auto Jc, auto jc) {
            constexpr int J = decltype(Jc)::value, j = decltype(jc)::value, I = rep<NP>(J < NP ? J : J - NP);
            pre[j] = streamed_fx<DIM, (J < NP), I, LAT, FX_CALL>((J < NP ? f : h) + I * ps, idx, am, own[j],
                                                        J < NP ? p.ghost_f[I] : p.ghost_h[I], k1, k2, hl, kbulk, gap, lim);
        });
    };
    if (w == 3) {
        double s[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) s[k] = (part[0][k][l] + part[1][k][l]) + (part[2][k][l] + part[3][k][l]);
        MacroG m;
        const bool ok = recover_g(Lat<LAT>::xi0sq * s[0], Lat<LAT>::xi0 * s[1], Lat<LAT>::xi0 * s[2],
                                  Lat<LAT>::xi0 * s[3], Lat<LAT>::xi0 * s[4], m);
        if (!ok && in) flag<double>(p, ST_NONPHYSICAL);
        const double v[7] = {m.P, m.ux, m.uy, m.uz, m.n, m.g, m.ig};
#pragma unroll
        for (int k = 0; k < 7; ++k) mac[k][l] = v[k];
        if (in) {
#pragma unroll
            for (int k = 0; k < 5; ++k) prev[k * ps + idx] = v[k];
        }
    } else {
        explicit_parts();
    }
    __syncthreads();
    if (w == 3) {
        explicit_parts();
    } else if (w == 2) {
        const double tau = p.tau_override > 0.0 ? p.tau_override : tau_of<LAT>(mac[0][l], mac[4][l], p.eta_over_s);
        s_kap[l] = p.kw / (tau + p.kw);
    } else {
        MacroG m;
        m.P = mac[0][l];
        m.ux = mac[1][l];
        m.uy = mac[2][l];
        m.uz = mac[3][l];
        m.n = mac[4][l];
        m.g = mac[5][l];
        m.ig = mac[6][l];
        Coef<double> a;
        if (w == 0) {
            coef_f_g<LAT>(m, a);
            kf.put(fold<Lat<LAT>::dmag>(extrapolate(a, b), Lat<LAT>::w0, Lat<LAT>::w1, Lat<LAT>::w2), l);
        } else {
            coef_h_g<LAT>(m, a);
            kh.put(fold<Lat<LAT>::dmag>(extrapolate(a, b), Lat<LAT>::wh0, Lat<LAT>::wh1, Lat<LAT>::wh2), l);
        }
    }
    __syncthreads();
    if (!in) return;
    const double kap = s_kap[l];
    items([&](auto Jc, auto jc) {
        constexpr int J = decltype(Jc)::value, j = decltype(jc)::value, I = rep<NP>(J < NP ? J : J - NP);
        const double g = J < NP ? kf.template pop<I>(l) : kh.template pop<I>(l);
        (J < NP ? fo : ho)[I * ps + idx] = fma(kap, g - pre[j], pre[j]);
    });
}

}  // namespace rlb
