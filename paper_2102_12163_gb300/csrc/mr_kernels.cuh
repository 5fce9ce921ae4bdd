// mr_kernels.cuh -- sm_103a kernels of the multiresolution-adaptive lattice
// Boltzmann step (Bellotti, Gouarin, Graille, Massot, arXiv 2102.12163).
//
// A thread block owns one instance at a time and runs every phase of the step
// on it, with block barriers between phases; blocks pull instances from an
// atomic work queue sorted largest first (persistent launch).  Inside a step:
//
//   adapt (Section 4.1)
//     A1  projection up the current tree (Def. Projection operator): one
//         conservative update of the internal cells, in the last step's S5
//     A2  details of the pairs of the tree, threshold T, Harten flags (Sections
//         3.2, 3.4, 4.2) -> KEEP / REF bitmasks
//     A3  enlargement H: same-level dilation and children of REF pairs
//     A4  grading G, sweeping fine to coarse over the words of the tree (Def.
//         Graded tree)
//     A5  list compaction (internal cells, leaves, pairs to transfer, ghost
//         pairs): word operations, popcount and prefix scan
//     A6  data transfer: prediction of the new pairs, coarse to fine
//   step (Sections 4.3, 4.5)
//     S1  leaves collision (eq. LeavesCollision)
//     S2  projection of the collided values up the new tree
//     S3  ghost prediction coarse to fine (reconstruction operator, Section 3.3)
//     S4  boundary reconstruction on the first / last finest cell of every
//         leaf from the per-level-gap tables -> interface array Phi
//     S5  compact stream (eq. AdaptiveStreamPhase) + mass audit (FP64 totals)
//
// The cell arrays are dense per level (every cell of every level has a slot),
// the tree is a bit array over the cells, and every per-cell phase walks a
// compacted list so its work is proportional to the tree.  A block spends most
// of a step on the dependent instructions of its busiest warp (it issues in a
// quarter of the cycles, its loads hit L1): fewer instructions on that path are
// what shortens a step.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "mr_common.h"

namespace mrg {

constexpr double C1 = -0.125;  // prediction coefficient c_1 for gamma = 1 (Section 3.1)
constexpr unsigned FULL = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------
// arithmetic: the FP64 path uses explicitly rounded operations (never fused)
// in the collision, so that it follows the same rounding sequence as a plain
// IEEE evaluation of the formulas; the FP32 path lets the compiler fuse.
template <typename T>
struct Ar;
template <>
struct Ar<double> {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
};
template <>
struct Ar<float> {
    static __device__ __forceinline__ float add(float a, float b) { return a + b; }
    static __device__ __forceinline__ float sub(float a, float b) { return a - b; }
    static __device__ __forceinline__ float mul(float a, float b) { return a * b; }
};

template <typename T>
struct V2;
template <>
struct V2<double> {
    using type = double2;
};
template <>
struct V2<float> {
    using type = float2;
};

// ---------------------------------------------------------------------------
// cells and bitmasks in heap numbering
//
// Cell k of level l is h = 2^l + k: its level is 31 - clz(h), its parent h / 2,
// its children 2h and 2h + 1, its neighbours h +- 1 (wrapped or clamped inside
// [2^l, 2^(l+1))).  A set of cells is one bit array over h, word h / 32, so word
// w >= 1 holds 32 cells of level 5 + log2(w), word 0 the levels 0..4, the words
// of a level follow one another, and the children of word w's cells are words
// 2w and 2w + 1: the same numbering again, on words.
//
// The tree is the set I of its internal cells (a pair of siblings is in the
// tree exactly when its parent is internal), with the cells above Jmin marked
// too, so that cell h is in the tree exactly when I holds h / 2.  That is half
// the words of a set of cells, and siblings need no closing.

__device__ __forceinline__ int level_of(uint32_t h) { return 31 - __clz(h); }
__device__ __forceinline__ uint32_t level_first(uint32_t h) { return 0x80000000u >> __clz(h); }
__device__ __forceinline__ bool bit_of(const uint32_t *a, uint32_t h) { return (a[h >> 5] >> (h & 31u)) & 1u; }
// the cell a places to the right of h on its level, whose first cell is lo
// (bc 0 periodic: wrapped, 1 copy: the boundary cell)
__device__ __forceinline__ uint32_t neighbour(uint32_t h, int a, uint32_t lo, int bc) {
    if (bc == 0) return lo | ((h + (uint32_t)a) & (lo - 1u));
    const int x = (int)h + a;
    return (uint32_t)min(max(x, (int)lo), (int)(2u * lo - 1u));
}

// bits 0, 2, ..., 30 of x -> bits 0..15
__device__ __forceinline__ uint32_t compact_even(uint32_t x) {
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return __byte_perm(x, 0u, 0x4420);
}
// 16 parent bits -> 32 child bits (both children of every parent)
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
    x = __byte_perm(x, 0u, 0x4140);
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x | (x << 1);
}
// the 32 cells of word w whose parents are in p: p's word w / 2 spread
__device__ __forceinline__ uint32_t children_word(const uint32_t *p, uint32_t w) { return spread16(p[w >> 1] >> (16u * (w & 1u))); }

// word 0 of a bit array (levels 2, 3, 4 at bits 4..7, 8..15, 16..31) dilated by
// one cell on each of its levels
__device__ __forceinline__ uint32_t dilate_word0(uint32_t x, int bc) {
    // the shifts, without what crosses from one level into the next
    uint32_t d = x | ((x << 1) & ~0x00010116u) | ((x >> 1) & ~0x8000808Bu);
    if (bc == 0)
        d |= ((x & 0x10u) << 3) | ((x & 0x80u) >> 3) | ((x & 0x100u) << 7) | ((x & 0x8000u) >> 7) | ((x & 0x10000u) << 15) |
             ((x & 0x80000000u) >> 15);
    return d;
}
// the words beside word w >= 1 on its level (get(j): word j); 0 beyond a copy boundary
template <class Get>
__device__ __forceinline__ void words_beside(Get get, uint32_t w, int bc, uint32_t &xl, uint32_t &xr) {
    const uint32_t lo = level_first(w);
    if (bc == 0) {
        xl = get(lo | ((w - 1u) & (lo - 1u)));
        xr = get(lo | ((w + 1u) & (lo - 1u)));
    } else {
        xl = w == lo ? 0u : get(w - 1u);
        xr = w + 1u == 2u * lo ? 0u : get(w + 1u);
    }
}
// x dilated by r <= 3 cells, given the words on its left and right
__device__ __forceinline__ uint32_t dilate_edges(uint32_t x, uint32_t xl, uint32_t xr, int r) {
    uint32_t d = x;
    for (int s = 1; s <= r; ++s) d |= __funnelshift_l(xl, x, s) | __funnelshift_r(x, xr, s);
    return d;
}
// word w of the bit array a dilated by r cells on its level
__device__ __forceinline__ uint32_t dilate_word(const uint32_t *a, uint32_t w, int r, int bc) {
    uint32_t x = a[w];
    if (w == 0u) {
        for (int s = 0; s < r; ++s) x = dilate_word0(x, bc);
        return x;
    }
    uint32_t xl, xr;
    words_beside([&](uint32_t j) { return a[j]; }, w, bc, xl, xr);
    return dilate_edges(x, xl, xr, r);
}
// Grading, one word: the 16 parents of word x's cells that must be internal,
// those of every cell within r of a marked one
__device__ __forceinline__ uint32_t graded_parents(uint32_t x, uint32_t xl, uint32_t xr, int r) {
    const uint32_t d = dilate_edges(x, xl, xr, r);
    return compact_even(d | (d >> 1));
}

// ---------------------------------------------------------------------------
// shared memory: per-team state and per-block tables

// eps_l = 2^{l - Jmax} eps (Prop. ErrorControl) and the Harten level
// 2^{mu_bar + 1} eps_l, with their roundings to float
struct Thresholds {
    double eps_l[MAXLEV + 1], big_l[MAXLEV + 1];
    float eps_f[MAXLEV + 1], big_f[MAXLEV + 1];
    __device__ __forceinline__ void set(const InstDesc &d, int l) {
        // the powers of two as factors (exact; 2^{l - Jmax}, |l - Jmax| <= 24)
        const double el = d.eps * __longlong_as_double((long long)(1023 + l - d.Jmax) << 52);
        // 2^{mu_bar + 1} eps_l in factors that are numbers, for any mu_bar
        // >= 0 (mr_run_static takes all): one factor up to 999; 2101 doublings are
        // infinity for every positive eps_l
        double bl = el;
#pragma unroll 1
        for (int k = min(d.mu_bar, 2100) + 1; k > 0; k -= 1000) bl *= __longlong_as_double((long long)(1023 + min(k, 1000)) << 52);
        eps_l[l] = el;
        big_l[l] = bl;
        eps_f[l] = (float)el;
        big_f[l] = (float)bl;
    }
};

template <typename T>
struct TeamSmem {
    InstDesc d;
    int cw_seg[MAXLEV + 2];  // candidate words of level l >= 5: entries [cw_seg[l], cw_seg[l+1]) of their list
    int seg[NSEG][MAXLEV + 2];
    Thresholds th;
    double dx_l[MAXLEV + 1];  // cell size per level
    double mass[3];
    double audit[3];  // per field
    unsigned long long updates, steps, passes;
    int cur, nleaf, status, near_ties, ncw;
    uint32_t deplev[2];  // levels holding transfer (0) / ghost (1) pairs that wait on the same list
#ifdef MRG_PHASE_TIMERS
    long long tlast;
    unsigned long long ptime[NPHASE];
#endif
};

// block-team scratch: scan partials of the warps, and the audit's partial sums
// (FP64: one a thread up to 256 threads; FP32: a float-float pair a thread up to 128)
template <typename T, int NT>
struct BlockScratch {
    static constexpr int NPART = sizeof(T) == 4 || NT < 256 ? 128 : 256;
    uint32_t scan_w[2][2][32];
    double red[3][NPART];
};

template <typename T, int NT>
struct BlockSmem {
    Tables<T> tab;
    BlockScratch<T, NT> scratch;
    TeamSmem<T> team;
    int idx;
};

// ---------------------------------------------------------------------------
// scheme: vectorial D1Q2^n (Section 2.1, equilibria of Sections 5.1 and 5.3)

// 2^-n exactly, built from its exponent field (0 <= n <= 126): no conversion
// instruction, which for a double would occupy GB300's scarce FP64 units
template <typename T>
__device__ __forceinline__ T pow2m(int n) {
    if constexpr (sizeof(T) == 8)
        return __longlong_as_double((long long)(1023 - n) << 52);
    else
        return __int_as_float((127 - n) << 23);
}

// x * 2^k (|k| <= 1022), bit for bit the correctly rounded product, in integer
// arithmetic where the exponent field allows (zero, or a normal operand and
// result) and with the multiply otherwise: GB300's FP64 units are scarce,
// integer units are not.
__device__ __forceinline__ double scale2(double x, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FFull);
    if ((b << 1) == 0ull) return x;
    if (e > 0 && e < 0x7FF && e + k > 0 && e + k < 0x7FF)
        return __longlong_as_double((long long)(b + ((unsigned long long)(long long)k << 52)));
    return x * __longlong_as_double((long long)(1023 + k) << 52);
}
__device__ __forceinline__ float scale2(float x, int k) { return x * ldexpf(1.0f, k); }

// x / 2, bit for bit the product x * 0.5, on the integer units where the
// exponent field allows (a normal operand and result, four instructions; or
// zero) and with the multiply otherwise
__device__ __forceinline__ double half_f64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if ((hi & 0x7FF00000u) - 0x00200000u < 0x7FD00000u) return __hiloint2double((int)(hi - 0x00100000u), __double2loint(x));
    if (((hi << 1) | (unsigned)__double2loint(x)) == 0u) return x;
    return __dmul_rn(x, 0.5);
}
template <typename T>
__device__ __forceinline__ T half_of(T x) {
    if constexpr (sizeof(T) == 8)
        return half_f64(x);
    else
        return T(0.5) * x;
}

// the scheme constants in the path's precision: FP64, or the float copies the
// host rounds once (no double-to-float conversion per cell in the FP32 path)
template <typename T>
__device__ __forceinline__ T lam_of(const InstDesc &d) {
    if constexpr (sizeof(T) == 8) return d.lam; else return d.lam_f;
}
template <typename T>
__device__ __forceinline__ T eqp_of(const InstDesc &d) {
    if constexpr (sizeof(T) == 8) return d.eqp; else return d.eqp_f;
}
template <typename T>
__device__ __forceinline__ T s_of(const InstDesc &d, int i) {
    if constexpr (sizeof(T) == 8) return d.s[i]; else return d.s_f[i];
}
template <typename T>
__device__ __forceinline__ T minv_of(const InstDesc &d, int h, int i) {
    if constexpr (sizeof(T) == 8) return d.minv[h][i]; else return d.minv_f[h][i];
}
// 1 - s[i] and the equilibria's constant factors: in FP64 rounded once on the
// host (GB300's FP64 pipe is the scarce one), in FP32 computed in place (the
// loads cost the FP32 kernel registers, the operations cost it nothing)
template <typename T>
__device__ __forceinline__ T oms_of(const InstDesc &d, int i) {
    if constexpr (sizeof(T) == 8) return d.oms[i]; else return 1.0f - d.s_f[i];
}
template <typename T>
__device__ __forceinline__ void eq_consts(const InstDesc &d, T &a, T &b, T &c, T &g2) {
    if constexpr (sizeof(T) == 8) {
        a = d.eu_a; b = d.eu_b; c = d.eu_c; g2 = d.sw_g2;
    } else {
        const float gg = d.eqp_f;
        a = 1.5f - 0.5f * gg;
        b = gg - 1.0f;
        c = 0.5f * (1.0f - gg);
        g2 = 0.5f * gg;
    }
}

// Quotients in FP64 from a reciprocal (P. Markstein, IBM J. Res. Dev. 34(1),
// 1990): with r = RN(1 / y), q0 = RN(x r) is within one ulp of x / y, the
// residual x - q0 y is exact in one FMA, and q0 + residual r rounded once is the
// correctly rounded quotient, bit for bit the division, as long as the quotient
// and the residual's last bit are normal numbers.  Other operands and non-finite
// values take the division; a zero numerator (a state at rest has many) stays on
// the short path.
// |x| from 2^-959 to 2^961, or zero: x over a number within 2^+-18 of 1
__device__ __forceinline__ bool mid_range(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    return ((hi >> 20) & 0x7FFu) - 64u < 1920u || ((hi << 1) | (unsigned)__double2loint(x)) == 0u;
}
// |x| from 2^-480 to 2^480, or zero: x over another such number
__device__ __forceinline__ bool half_range(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    return ((hi >> 20) & 0x7FFu) - 543u < 960u || ((hi << 1) | (unsigned)__double2loint(x)) == 0u;
}
// exponents within 300 of 1's (or zero): cubes and quotients of such numbers
// neither overflow nor underflow
__device__ __forceinline__ bool cube_range(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    return ((hi >> 20) & 0x7FFu) - 723u < 600u || ((hi << 1) | (unsigned)__double2loint(x)) == 0u;
}
__device__ __forceinline__ double markstein(double x, double y, double r) {
    const double q0 = __dmul_rn(x, r);
    return __fma_rn(__fma_rn(-q0, y, x), r, q0);
}
// x / y.  The hardware's division sequence leaves its short path for a zero
// numerator, which a fluid at rest has in every cell: FP64 goes by the
// reciprocal, FP32 answers a zero itself.
template <typename T>
__device__ __forceinline__ T quotient(T x, T y) {
    if constexpr (sizeof(T) == 8) {
        if (y != 0.0 && half_range(y) && half_range(x)) return markstein(x, y, __drcp_rn(y));
        return __ddiv_rn(x, y);
    } else {
        if (x == 0.0f && y != 0.0f && fabsf(y) < __int_as_float(0x7F800000)) return x * y;  // the zero of the quotient's sign
        return x / y;
    }
}
// x / (2 lambda), half of what the collision adds to and takes from a moment,
// for a lambda that is no power of two (halving is exact, so its halves are the
// halves of the rounded quotient by lambda)
template <typename T>
__device__ __forceinline__ T div_2lam(T x, const InstDesc &d) {
    if constexpr (sizeof(T) == 8) {
        if (!mid_range(x)) return half_f64(__ddiv_rn(x, d.lam));
        return markstein(x, d.lam2, d.rlam2);
    } else {
        return 0.5f * __fdiv_rn(x, d.lam_f);  // FP32 divisions are cheap; the register budget is not
    }
}

// equilibria of the relaxed moments; the constant factors (0.5 g, 1.5 - 0.5
// gamma_gas, gamma_gas - 1, 0.5 (1 - gamma_gas)) come rounded from the host,
// the same values the expressions would give per cell
// EXACT: each quotient of the formulas rounded by itself (the initial datum,
// which equals a plain IEEE evaluation bit for bit); else FP64 Euler takes the
// velocity u = rho u / rho once and multiplies by it: as many roundings on the
// way to each flux (one ulp for the quadratic ones, two for the cubic), 14 FP64
// instructions instead of 28 for the four quotients' part of the collision.
template <typename T, int NF, bool EXACT = false>
__device__ __forceinline__ void equilibria(const InstDesc &d, T eqp, const T *mc, T *meq) {
    using A = Ar<T>;
    T ca, cb, cc, g2;
    eq_consts<T>(d, ca, cb, cc, g2);
    if constexpr (NF == 1) {
        if (d.eq == 0)
            meq[0] = A::mul(eqp, mc[0]);  // advection: c m0
        else
            meq[0] = half_of<T>(A::mul(mc[0], mc[0]));  // Burgers: m0^2 / 2
    } else if constexpr (NF == 2) {
        // shallow water (h, hu): hu, hu^2 / h + g h^2 / 2
        meq[0] = mc[1];
        meq[1] = A::add(quotient<T>(A::mul(mc[1], mc[1]), mc[0]), A::mul(g2, A::mul(mc[0], mc[0])));
    } else {
        // Euler (rho, rho u, E), Section 5.3
        T gg = eqp;
        T u2 = A::mul(mc[1], mc[1]);
        meq[0] = mc[1];
        if constexpr (sizeof(T) == 8) {
            if constexpr (EXACT) {
                // the two quotients by rho from one reciprocal
                const double em = A::mul(mc[2], mc[1]), u3 = A::mul(u2, mc[1]);
                if (mc[0] != 0.0 && half_range(mc[0]) && half_range(u2) && half_range(em)) {
                    const double r = __drcp_rn(mc[0]);
                    meq[1] = A::add(A::mul(ca, markstein(u2, mc[0], r)), A::mul(cb, mc[2]));
                    meq[2] = A::add(A::mul(gg, markstein(em, mc[0], r)), A::mul(cc, quotient<T>(u3, A::mul(mc[0], mc[0]))));
                    return;
                }
            } else if (mc[0] != 0.0 && cube_range(mc[0]) && cube_range(mc[1]) && cube_range(mc[2])) {
                const double u = markstein(mc[1], mc[0], __drcp_rn(mc[0])), mu = A::mul(mc[1], u);
                meq[1] = A::add(A::mul(ca, mu), A::mul(cb, mc[2]));
                meq[2] = A::add(A::mul(gg, A::mul(mc[2], u)), A::mul(cc, A::mul(mu, u)));
                return;
            }
        }
        meq[1] = A::add(A::mul(ca, quotient<T>(u2, mc[0])), A::mul(cb, mc[2]));
        meq[2] = A::add(A::mul(gg, quotient<T>(A::mul(mc[2], mc[1]), mc[0])),
                        A::mul(cc, quotient<T>(A::mul(u2, mc[1]), A::mul(mc[0], mc[0]))));
    }
}

// half of m* / lambda, an exact power-of-two scaling when lambda = 2^k (the same
// value as the division)
template <typename T>
__device__ __forceinline__ T half_over_lam(T x, const InstDesc &d) {
    return d.lam_log2 != NOT_POW2 ? scale2(x, -d.lam_log2 - 1) : div_2lam<T>(x, d);
}
// relaxed moment (1 - s) m + s m_eq of field i, m = lambda (f+ - f-); full
// relaxation is m_eq itself (0 m + 1 m_eq), five FP64 operations fewer
template <typename T>
__device__ __forceinline__ T relaxed(const InstDesc &d, int i, T fp, T fm, T meq) {
    using A = Ar<T>;
    const T s = s_of<T>(d, i);
    if constexpr (sizeof(T) == 8)
        if (s == 1.0) return meq;
    return A::add(A::mul(oms_of<T>(d, i), A::mul(lam_of<T>(d), A::sub(fp, fm))), A::mul(s, meq));
}

// leaves collision on the q populations of one cell: m = M f, relax, f* = M^-1 m*
template <typename T, int NF>
__device__ __forceinline__ void collide(const InstDesc &d, T *f) {
    using A = Ar<T>;
    T mc[NF], meq[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i) mc[i] = A::add(f[2 * i], f[2 * i + 1]);
    equilibria<T, NF>(d, eqp_of<T>(d), mc, meq);
#pragma unroll
    for (int i = 0; i < NF; ++i) {
        // f+- = (mc +- m* / lambda) / 2, the halves taken first (exact)
        const T g = half_over_lam<T>(relaxed<T>(d, i, f[2 * i], f[2 * i + 1], meq[i]), d), m = half_of<T>(mc[i]);
        f[2 * i] = A::add(m, g);
        f[2 * i + 1] = A::sub(m, g);
    }
}

// populations at equilibrium of the conserved moments (initial datum), in FP64
template <int NF>
__device__ __forceinline__ void equilibrium_populations(const InstDesc &d, const double *mc, double *f) {
    using A = Ar<double>;
    double meq[NF];
    equilibria<double, NF, true>(d, d.eqp, mc, meq);
#pragma unroll
    for (int i = 0; i < NF; ++i) {
        const double g = half_over_lam<double>(meq[i], d), m = half_f64(mc[i]);
        f[2 * i] = A::add(m, g);
        f[2 * i + 1] = A::sub(m, g);
    }
}

// ---- shallow water on one velocity set (Section 5.2): D1Q3 (Q = 3), D1Q5 (Q = 5)
// velocities v^h = lambda w^h, w = (0, 1, -1, 2, -2); moments m^i = sum_h (v^h)^i f^h
__device__ __forceinline__ int dq_w(int h) { return h == 0 ? 0 : (h & 1) ? (h + 1) / 2 : -(h / 2); }

// moments of the velocity set through the even and odd parts of its two velocity
// pairs: m^i = lambda^i (p1 + 2^i p2), p the sums (i even) or differences (i odd)
template <typename T, int Q>
__device__ __forceinline__ void dq_moments(T lam, const T *f, T *m) {
    const T s1 = f[1] + f[2], d1 = f[1] - f[2];
    if constexpr (Q == 3) {
        m[0] = f[0] + s1;
        m[1] = lam * d1;
        m[2] = (lam * lam) * s1;
    } else {
        const T s2 = f[3] + f[4], d2 = f[3] - f[4], l2 = lam * lam;
        m[0] = f[0] + (s1 + s2);
        m[1] = lam * (d1 + T(2) * d2);
        m[2] = l2 * (s1 + T(4) * s2);
        m[3] = (l2 * lam) * (d1 + T(8) * d2);
        m[4] = (l2 * l2) * (s1 + T(16) * s2);
    }
}
// f + M^{-1} dm for dm with zero conserved rows.  M^{-1} carries the same mirror
// symmetry: the populations +-w get the even moments' part alike and the odd
// moment's part with opposite signs.
template <typename T, int Q>
__device__ __forceinline__ void dq_add(const InstDesc &d, const T *dm, T *f) {
    if constexpr (Q == 3) {
        f[0] = f[0] + minv_of<T>(d, 0, 2) * dm[2];
        const T a = minv_of<T>(d, 1, 2) * dm[2];
        f[1] = f[1] + a;
        f[2] = f[2] + a;
    } else {
        f[0] = f[0] + (minv_of<T>(d, 0, 2) * dm[2] + minv_of<T>(d, 0, 4) * dm[4]);
#pragma unroll
        for (int h = 1; h < 5; h += 2) {
            const T a = minv_of<T>(d, h, 2) * dm[2] + minv_of<T>(d, h, 4) * dm[4], b = minv_of<T>(d, h, 3) * dm[3];
            f[h] = f[h] + (a + b);
            f[h + 1] = f[h + 1] + (a - b);
        }
    }
}
// collision: the relaxed moments i >= 2 move to (1 - s^i) m^i + s^i m^{i,eq}, with
// m^{2,eq} = (hu)^2 / h + g h^2 / 2, m^{3,eq} = lambda^2 hu, m^{4,eq} = lambda^2
// m^{2,eq}; f* = f + M^{-1} (m* - m) (the conserved rows of m* - m are zero)
template <typename T, int Q>
__device__ __forceinline__ void dq_collide(const InstDesc &d, T *f) {
    const T lam = lam_of<T>(d);
    T m[Q], meq[Q], dm[Q];
    dq_moments<T, Q>(lam, f, m);
    T ca, cb, cc, g2;
    eq_consts<T>(d, ca, cb, cc, g2);
    meq[2] = quotient<T>(m[1] * m[1], m[0]) + g2 * (m[0] * m[0]);
    if constexpr (Q == 5) {
        meq[3] = (lam * lam) * m[1];
        meq[4] = (lam * lam) * meq[2];
    }
#pragma unroll
    for (int i = 2; i < Q; ++i) dm[i] = s_of<T>(d, i - 2) * (meq[i] - m[i]);
    dq_add<T, Q>(d, dm, f);
}

// populations at equilibrium of (h, hu), in FP64: f = M^{-1} (h, hu, m^{2,eq}, ...)
template <int Q>
__device__ __forceinline__ void dq_equilibrium_populations(const InstDesc &d, const double *mc, double *f) {
    double m[5];
    m[0] = mc[0];
    m[1] = mc[1];
    m[2] = quotient<double>(mc[1] * mc[1], mc[0]) + (0.5 * d.eqp) * (mc[0] * mc[0]);
    if constexpr (Q == 5) {
        m[3] = (d.lam * d.lam) * mc[1];
        m[4] = (d.lam * d.lam) * m[2];
    }
#pragma unroll
    for (int h = 0; h < Q; ++h) {
        double acc = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) acc = acc + d.minv[h][i] * m[i];
        f[h] = acc;
    }
}

// NaN or infinity, from the exponent field (integer units)
__device__ __forceinline__ bool nonfinite(double x) { return (__double2hiint(x) & 0x7FF00000) == 0x7FF00000; }
__device__ __forceinline__ bool nonfinite(float x) { return (__float_as_uint(x) & 0x7F800000u) == 0x7F800000u; }

// ---------------------------------------------------------------------------
// FP64 threshold decisions on bit patterns.  Non-negative doubles order as
// their bit patterns, so max |d| over the populations and its comparisons with
// eps_l and the Harten level run on the integer units instead of GB300's
// scarce FP64 pipe, with the same outcome as the floating-point max and >=
// (a NaN detail is skipped, as fmax skips it).
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
    return b > 0x7FF0000000000000ull ? 0ull : b;
}
// keep / refine decisions of a pair with max |detail| bits Db, and whether it
// lies within 1e-12 relative of eps_l or of the Harten level: an integer
// pre-filter (1e-12 relative is at most 9008 units in the last place) and the
// exact test behind it
__device__ __forceinline__ void decide_bits(unsigned long long Db, double el, double bl, bool hasref, bool &keepit,
                                            bool &refit, bool &tie) {
    const unsigned long long eb = (unsigned long long)__double_as_longlong(el),
                             bb = (unsigned long long)__double_as_longlong(bl);
    keepit = Db >= eb;
    refit = hasref && Db >= bb;
    const long long de = (long long)(Db - eb), db = (long long)(Db - bb);
    tie = false;
    if ((de < 16384 && de > -16384) || (hasref && db < 16384 && db > -16384)) {
        const double D = __longlong_as_double((long long)Db);
        tie = fabs(D - el) <= 1e-12 * el || (hasref && fabs(D - bl) <= 1e-12 * bl);
    }
}

// ---------------------------------------------------------------------------
// prediction stencils and the threshold decision of one pair

// sum_a c_a (f_{p+a} - f_{p-a}) of population h with the stencil of half-width
// g (coefficients c, in increasing a), given the gamma = 1 sum first (used as it
// is when g = 1); V: cell x at V + x q, lo: first cell of p's level
template <typename T, int q>
__device__ __forceinline__ T wide_sum(const T *V, uint32_t p, uint32_t lo, int bc, int g, const T *c, int h, T first) {
    if (g == 1) return first;
    auto at = [&](int a) { return V[neighbour(p, a, lo, bc) * (uint32_t)q + (uint32_t)h]; };
    T sum = c[0] * (at(1) - at(-1));
#pragma unroll 1
    for (int a = 2; a <= g; ++a) sum = sum + c[a - 1] * (at(a) - at(-a));
    return sum;
}

// Keep / refine decision of the children of p (Sections 3.2, 3.4, 4.2), and
// whether it lies within 1e-12 relative of a threshold.  FP64: the detail in
// double.  FP32: the detail in float with a rigorous bound on its rounding
// error; only when a threshold lies within that bound is the detail recomputed
// in FP64 from the stored values, so every decision equals the one the exact
// detail of the stored state gives.
template <typename T, int q, bool WIDE>
__device__ __forceinline__ void pair_decision(const T *V, uint32_t p, int Jmax, int bc, int g, const Tables<T> &tab,
                                              const Thresholds &th, bool &keepit, bool &refit, bool &tie) {
    const uint32_t lo = level_first(p);
    const int l = level_of(p) + 1;
    const bool hasref = l < Jmax;
    tie = false;
    const T *vk = V + 2u * p * (uint32_t)q, *vp = V + p * (uint32_t)q, *vl = V + neighbour(p, -1, lo, bc) * (uint32_t)q,
            *vr = V + neighbour(p, 1, lo, bc) * (uint32_t)q;
    const T *c = tab.pc[g];
    if constexpr (sizeof(T) == 8) {
        unsigned long long Db = 0ull;
#pragma unroll
        for (int h = 0; h < q; ++h) {
            double sum = C1 * (vr[h] - vl[h]);
            if constexpr (WIDE) sum = wide_sum<T, q>(V, p, lo, bc, g, c, h, sum);
            const unsigned long long b = abs_bits(vk[h] - (vp[h] + sum));
            Db = b > Db ? b : Db;
        }
        decide_bits(Db, th.eps_l[l], th.big_l[l], hasref, keepit, refit, tie);
    } else {
        float D = 0.0f, B = 0.0f;
#pragma unroll
        for (int h = 0; h < q; ++h) {
            const float xk = vk[h], xp = vp[h], xl = vl[h], xr = vr[h];
            float sum = float(C1) * (xr - xl), mag = fabsf(xl) + fabsf(xr);
            if constexpr (WIDE) {
                sum = wide_sum<T, q>(V, p, lo, bc, g, c, h, sum);
#pragma unroll 1
                for (int a = 2; a <= g; ++a)
                    mag += fabsf(V[neighbour(p, a, lo, bc) * (uint32_t)q + h]) + fabsf(V[neighbour(p, -a, lo, bc) * (uint32_t)q + h]);
            }
            D = fmaxf(D, fabsf(xk - (xp + sum)));
            B = fmaxf(B, fabsf(xk) + fabsf(xp) + mag);
        }
        // the rounding of the detail: for gamma = 1 4 times the bound of its
        // evaluation; (6 gamma + 2) u times the sum of |inputs| else (3 gamma + 1
        // roundings, each at most u times that sum, with a factor 2 margin)
        B *= WIDE && g > 1 ? (float)(6 * g + 2) * 0x1p-24f : 0x1p-21f;
        const float el = th.eps_f[l], bl = th.big_f[l];
        // the band also covers the rounding of the thresholds to float
        const bool amb = fabsf(D - el) <= B + el * 0x1p-22f || (hasref && fabsf(D - bl) <= B + bl * 0x1p-22f);
        if (amb) {
            double Dd = 0.0;
#pragma unroll 1
            for (int h = 0; h < q; ++h) {
                double sum = (WIDE ? (double)c[0] : C1) * ((double)vr[h] - (double)vl[h]);
                if constexpr (WIDE)
                    for (int a = 2; a <= g; ++a)
                        sum = sum + (double)c[a - 1] * ((double)V[neighbour(p, a, lo, bc) * (uint32_t)q + h] -
                                                        (double)V[neighbour(p, -a, lo, bc) * (uint32_t)q + h]);
                Dd = fmax(Dd, fabs((double)vk[h] - ((double)vp[h] + sum)));
            }
            const double e64 = th.eps_l[l], b64 = th.big_l[l];
            keepit = Dd >= e64;
            refit = hasref && Dd >= b64;
            tie = fabs(Dd - e64) <= 1e-12 * e64 || (hasref && fabs(Dd - b64) <= 1e-12 * b64);
        } else {
            keepit = D >= el;
            refit = hasref && D >= bl;
        }
    }
}

// ---------------------------------------------------------------------------
// the instance worker; the TS threads of the block form the team

constexpr int QMAX = 6;  // populations of the largest scheme (vectorial D1Q2^3)

// WIDE: prediction stencils gamma = 2, 3 (the gamma = 1 code is a separate instantiation)
// SPM: word passes over every word (0) or over candidate words (1, the
// large-instance variant K_LARGE alone: code that a kernel carries costs it
// even where it does not run)
template <typename T, int NF, int TS, bool WIDE, int SPM>
struct Worker {
    // NF = 1, 2, 3: vectorial D1Q2^NF; NF = 4: D1Q3, NF = 5: D1Q5 shallow water
    static constexpr bool DQ = NF >= 4;
    static constexpr int nf = DQ ? 2 : NF;                     // conserved moments
    static constexpr int q = DQ ? (NF == 4 ? 3 : 5) : 2 * NF;  // populations
    static_assert(TS >= 64 && TS % 64 == 0, "team width");
    TeamSmem<T> &sm;
    const Tables<T> &tab;
    BlockScratch<T, TS> &bx;
    const InstDesc &d;
    T *V;         // cell h at V + h q
    const WideTables<T> *wide;
    uint32_t *M;  // bit arrays (shared memory when they fit, else global)
    const int tid;
    const int bc, Jmin, Jmax;

    __device__ Worker(TeamSmem<T> &s, const Tables<T> &tb, BlockScratch<T, TS> &x, int rank, uint32_t *masks, const void *wd)
        : sm(s), tab(tb), bx(x), d(s.d), tid(rank), bc(s.d.bc), Jmin(s.d.Jmin), Jmax(s.d.Jmax) {
        V = (T *)d.V - (1LL << d.Jmin) * q;
        M = masks;
        wide = (const WideTables<T> *)wd;
    }

    // leaves collision of the q populations of one cell
    __device__ __forceinline__ void collide_cell(T *f) const {
        if constexpr (DQ)
            dq_collide<T, q>(d, f);
        else
            collide<T, NF>(d, f);
    }

    // team barrier; every one ends a pass whose results the next pass reads.
    // The variants that run large single instances count them (the chain of
    // dependent passes of a step, the floor of its latency) by the team's last
    // thread after the barrier; the batch variants do not: the count cost them
    // 7 % (measured), most of their passes being short.
    __device__ __forceinline__ void sync() const {
        __syncthreads();
        if constexpr (SPM != 0)
            if (tid == TS - 1) ++sm.passes;
    }

    // profiling build: cycles since the previous tick charged to phase p (after a team barrier)
    __device__ __forceinline__ void tick(int p) {
#ifdef MRG_PHASE_TIMERS
        sync();
        if (tid == 0) {
            long long t = clock64();
            if (p < NPHASE) sm.ptime[p] += (unsigned long long)(t - sm.tlast);
            sm.tlast = t;
        }
#else
        (void)p;
#endif
    }

    __device__ __forceinline__ uint32_t *mask(int m) const { return M + m * d.Wtot; }
    // candidate-word list of the step (word indices, sorted)
    __device__ __forceinline__ uint32_t *cwl() const { return M + NMASK * d.Wtot; }
    // occupancy array of tree buffer b (M_I0 or M_I1): bit w is set when word w of that tree is not empty
    __device__ __forceinline__ uint32_t *occ(int b) const { return M + (long long)(NMASK + 1) * d.Wtot + b * d.OW; }
    __device__ __forceinline__ uint32_t *list(int L) const { return d.lists + d.list_off[L]; }
    // first word of the word passes (it holds the cells of level Jmin - 1) and
    // their number; i-th word of a pass: a candidate word, or the words in turn
    __device__ __forceinline__ uint32_t first_word() const { return (1u << (Jmin - 1)) >> 5; }
    __device__ __forceinline__ int nwords() const {
        if constexpr (SPM != 0) return sm.ncw;
        return d.Wtot - (int)first_word();
    }
    __device__ __forceinline__ uint32_t word_at(int i) const {
        if constexpr (SPM != 0) return cwl()[i];
        return first_word() + (uint32_t)i;
    }
    // index of the segment end of a whole list (levels below 5 share one segment)
    __device__ __forceinline__ int top() const { return Jmax > 5 ? Jmax : 5; }
    // the cells above Jmin among the bits of word w
    __device__ __forceinline__ uint32_t above(uint32_t w) const {
        if (w == 0u) return Jmin >= 5 ? 0xFFFFFFFEu : (1u << (1 << Jmin)) - 2u;
        return Jmin > 5 && w < (1u << (Jmin - 5)) ? FULL : 0u;
    }
    __device__ __forceinline__ T *cell(uint32_t h) const { return V + h * (uint32_t)q; }
    // Interface values at interface x of the finest lattice (0 .. N).  D1Q2^n in
    // FP32 keeps them in heap order, the interfaces between two cells of one parent
    // level by level (x = 0 and N in the two places left): those of neighbouring
    // leaves lie side by side, where in the order of x each had a line of L1 to
    // itself (batch of 4096 at 256 threads 116 -> 109 us a step, 163 -> 153 over
    // 1024 steps).  FP64 waits on its units, not on L1: the same order gave the
    // batch 0.5 % and cost a lone instance 2.6 % in index arithmetic.  D1Q3 / D1Q5
    // keep finest cells, in the order of x.
    __device__ __forceinline__ T *phi(uint32_t x) const {
        if constexpr (!DQ && sizeof(T) == 4) {
            const uint32_t N = 1u << Jmax;
            x = x == N ? 0u : (N + x) >> __ffs((int)x);
        }
        return (T *)d.Phi + x * (uint32_t)q;
    }
    __device__ __forceinline__ uint32_t nb(uint32_t h, int a, uint32_t lo) const { return neighbour(h, a, lo, bc); }

    // the q populations of cell h in registers; two a load where the cells are
    // aligned for it (even q: a cell starts at a multiple of two values)
    __device__ __forceinline__ void load_cell(uint32_t h, T *f) const { load_pops(cell(h), f); }
    __device__ __forceinline__ void load_pops(const T *p, T *f) const {
        if constexpr (q % 2 == 0) {
#pragma unroll
            for (int j = 0; j < q / 2; ++j) {
                const auto v = reinterpret_cast<const typename V2<T>::type *>(p)[j];
                f[2 * j] = v.x;
                f[2 * j + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < q; ++j) f[j] = p[j];
        }
    }
    __device__ __forceinline__ void store_cell(uint32_t h, const T *f) const {
        T *p = cell(h);
        if constexpr (q % 2 == 0) {
#pragma unroll
            for (int j = 0; j < q / 2; ++j) {
                typename V2<T>::type v;
                v.x = f[2 * j];
                v.y = f[2 * j + 1];
                reinterpret_cast<typename V2<T>::type *>(p)[j] = v;
            }
        } else {
#pragma unroll
            for (int j = 0; j < q; ++j) p[j] = f[j];
        }
    }

    // float-float accumulation (hi + lo, error-free transformation TwoSum of
    // Knuth): the FP32 path keeps its mass audit off the FP64 pipe
    static __device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
        s = a + b;
        const float bb = s - a;
        e = (a - (s - bb)) + (b - bb);
    }
    static __device__ __forceinline__ void ff_add(float &hi, float &lo, float xh, float xl) {
        float s, e;
        two_sum(hi, xh, s, e);
        hi = s;
        lo = lo + (xl + e);
    }
    // Partial sums of the team, field by field, in shared memory (one barrier),
    // and the sum of field j of them by one warp: the warps TS / 32 - 1 - j fold one
    // field each, valid in their lane 0, while the others go on.  GB300's FP64
    // units take a warp-wide instruction whole whatever its active lanes, so
    // additions are kept off most warps: a thread's own sum is a partial up to
    // 256 threads (shuffle rounds fold wider blocks to 256), and one warp adds
    // eight a lane and shuffles.  Warps without a leaf (the first n threads have
    // one) only write their zeros.  A fixed order: deterministic.
    __device__ __forceinline__ void team_partials(double (&x)[3], int n) {
        constexpr int G = TS / NPART;  // lanes per partial sum: 1, 2, 4, or 8 (FP32 at 1024 threads)
        if ((tid & ~31) < n)
#pragma unroll
            for (int j = 0; j < nf; ++j)
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) x[j] += __shfl_down_sync(FULL, x[j], o);
        if ((tid & (G - 1)) == 0)
#pragma unroll
            for (int j = 0; j < nf; ++j) bx.red[j][tid / G] = x[j];
        sync();
    }
    static constexpr int NPART = BlockScratch<T, TS>::NPART;
    __device__ __forceinline__ double team_fold(int j) const {
        const int lane = tid & 31;
        double v = bx.red[j][lane];
#pragma unroll
        for (int k = 32; k < NPART; k += 32) v += bx.red[j][lane + k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
        return v;
    }
    // the same in float-float, a pair in a double's room
    __device__ __forceinline__ void team_partials_ff(float (&hi)[3], float (&lo)[3], int n) {
        constexpr int G = TS / NPART;
        if ((tid & ~31) < n)
#pragma unroll
            for (int j = 0; j < nf; ++j)
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) {
                    const float h2 = __shfl_down_sync(FULL, hi[j], o), l2 = __shfl_down_sync(FULL, lo[j], o);
                    ff_add(hi[j], lo[j], h2, l2);
                }
        if ((tid & (G - 1)) == 0)
#pragma unroll
            for (int j = 0; j < nf; ++j) reinterpret_cast<float2 *>(bx.red[j])[tid / G] = make_float2(hi[j], lo[j]);
        sync();
    }
    __device__ __forceinline__ double team_fold_ff(int j) const {
        const float2 *red = reinterpret_cast<const float2 *>(bx.red[j]);
        const int lane = tid & 31;
        float2 v = red[lane];
#pragma unroll
        for (int k = 32; k < NPART; k += 32) {
            const float2 y = red[lane + k];
            ff_add(v.x, v.y, y.x, y.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_down_sync(FULL, v.x, o), l2 = __shfl_down_sync(FULL, v.y, o);
            ff_add(v.x, v.y, h2, l2);
        }
        return (double)v.x + (double)v.y;
    }
    // field that this thread's warp folds, or -1
    __device__ __forceinline__ int fold_field() const {
        const int j = TS / 32 - 1 - (tid >> 5);
        return j < nf ? j : -1;
    }

    // ---- S1: leaves collision (eq. LeavesCollision) ---------------------------
    __device__ void collide_all() {
        const uint32_t *lst = list(L_LEAF);
        const int n = sm.nleaf;
#pragma unroll 1
        for (int i = tid; i < n; i += TS) {
            const uint32_t h = lst[i];
            T f[q];
            load_cell(h, f);
            collide_cell(f);
            store_cell(h, f);
        }
    }

    // equilibria of the relaxed moments at one cell (populations g)
    __device__ __forceinline__ void relaxed_equilibria(const T *g, T *meq) const {
        if constexpr (DQ) {
            const T lam = lam_of<T>(d);
            T h = T(0), hu = T(0);
#pragma unroll
            for (int c = 0; c < q; ++c) {
                h = h + g[c];
                hu = hu + ((T)dq_w(c) * lam) * g[c];
            }
            T ca, cb, cc, g2;
            eq_consts<T>(d, ca, cb, cc, g2);
            meq[0] = quotient<T>(hu * hu, h) + g2 * (h * h);
            if constexpr (q == 5) {
                meq[1] = (lam * lam) * hu;
                meq[2] = (lam * lam) * meq[0];
            }
        } else {
            using A = Ar<T>;
            T mc[NF];
#pragma unroll
            for (int i = 0; i < NF; ++i) mc[i] = A::add(g[2 * i], g[2 * i + 1]);
            equilibria<T, NF>(d, eqp_of<T>(d), mc, meq);
        }
    }

    // the populations of every finest cell by the reconstruction operator
    // (Definition V): the internal cells hold projections; every cell outside the
    // tree is predicted, level by level
    __device__ void fill_finest() {
        const uint32_t *I = mask(sm.cur);
#pragma unroll 1
        for (int l = Jmin; l < Jmax; ++l) {
            const uint32_t lo = 1u << l;
#pragma unroll 1
            for (uint32_t p = lo + tid; p < 2u * lo; p += TS)
                if (!bit_of(I, p)) predict_pair(p, lo);
            sync();
        }
    }

    // S1 with the reconstructed collision (Section 4.5, eq. reconstructedCollision):
    // the pre-collision populations are reconstructed on every finest cell; a
    // thread (a small leaf) or a warp (a large one) averages the equilibria of the
    // relaxed moments over the leaf's 2^dj finest cells (into the interface array,
    // free until S4); then every leaf relaxes towards those averages.  A barrier has
    // to lie between a step and this: the end of a step's audit still reads the
    // interface array (an adaptation has many; without one a launch holds one step).
    __device__ __noinline__ void collide_reconstructed() {
        fill_finest();
        constexpr int NR = DQ ? q - 2 : nf;  // relaxed moments
        constexpr int NWARP = TS / 32;
        const int lane = tid & 31, warp = tid >> 5;
        const uint32_t *leaves = list(L_LEAF);
        T *Phi = (T *)d.Phi;
        const long long stride = d.N + 1;
        const int nl = sm.nleaf;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            // a leaf of up to four finest cells (most leaves): one thread
            const uint32_t hl = leaves[i];
            const int dj = Jmax - level_of(hl);
            if (dj > 2) continue;
            T acc[3] = {T(0), T(0), T(0)};
#pragma unroll 1
            for (uint32_t c = hl << dj; c < (hl + 1u) << dj; ++c) {
                T g[q], meq[3];
                load_cell(c, g);
                relaxed_equilibria(g, meq);
#pragma unroll
                for (int r = 0; r < NR; ++r) acc[r] = acc[r] + meq[r];
            }
#pragma unroll
            for (int r = 0; r < NR; ++r) Phi[r * stride + i] = acc[r] * pow2m<T>(dj);
        }
#pragma unroll 1
        for (int i = warp; i < nl; i += NWARP) {
            const uint32_t hl = leaves[i];
            const int dj = Jmax - level_of(hl);
            if (dj <= 2) break;  // the leaves are sorted, coarse first
            const uint32_t first = hl << dj, end = first + (1u << dj);
            T acc[3] = {T(0), T(0), T(0)};
#pragma unroll 1
            for (uint32_t c = first + lane; c < end; c += 32) {
                T g[q], meq[3];
                load_cell(c, g);
                relaxed_equilibria(g, meq);
#pragma unroll
                for (int r = 0; r < NR; ++r) acc[r] = acc[r] + meq[r];
            }
#pragma unroll
            for (int r = 0; r < NR; ++r)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[r] = acc[r] + __shfl_xor_sync(FULL, acc[r], o);
            if (lane == 0)
#pragma unroll
                for (int r = 0; r < NR; ++r) Phi[r * stride + i] = acc[r] * pow2m<T>(dj);
        }
        sync();
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t hc = leaves[i];
            T f[q], mavg[3];
            load_cell(hc, f);
#pragma unroll
            for (int r = 0; r < NR; ++r) mavg[r] = Phi[r * stride + i];
            if constexpr (DQ) {
                T m[q], dm[q];
                dq_moments<T, q>(lam_of<T>(d), f, m);
#pragma unroll
                for (int r = 2; r < q; ++r) dm[r] = s_of<T>(d, r - 2) * (mavg[r - 2] - m[r]);
                dq_add<T, q>(d, dm, f);
            } else {
                using A = Ar<T>;
#pragma unroll
                for (int j = 0; j < NF; ++j) {
                    const T m = half_of<T>(A::add(f[2 * j], f[2 * j + 1]));
                    const T g = half_over_lam<T>(relaxed<T>(d, j, f[2 * j], f[2 * j + 1], mavg[j]), d);
                    f[2 * j] = A::add(m, g);
                    f[2 * j + 1] = A::sub(m, g);
                }
            }
            store_cell(hc, f);
        }
        sync();
    }

    // ---- S2: projection sweep, fine to coarse (Def. Projection operator) -------
    // part j of cell h's populations (PP of them): the mean of its two children's
    static constexpr int PP = sizeof(T) == 4 && q % 2 == 0 ? 2 : 1, NPARTS = q / PP;
    __device__ __forceinline__ void project_part(uint32_t h, int j) const {
        T *p = V + (h * (uint32_t)q + (uint32_t)(PP * j));
        const T *c = V + (2u * h * (uint32_t)q + (uint32_t)(PP * j));
        if constexpr (PP == 2) {
            const auto x = *reinterpret_cast<const typename V2<T>::type *>(c), y = *reinterpret_cast<const typename V2<T>::type *>(c + q);
            typename V2<T>::type m;
            m.x = half_of<T>(x.x + y.x);
            m.y = half_of<T>(x.y + y.y);
            *reinterpret_cast<typename V2<T>::type *>(p) = m;
        } else {
            *p = half_of<T>(c[0] + c[q]);
        }
    }
    // One level per barrier; the levels of at most 32 cells by one warp, without
    // block barriers.  Ends with a barrier.  A thread takes one population of a
    // cell: a level holds some ten cells, and an FP64 instruction costs its warp's
    // quarter of the SM 64 cycles whatever its active lanes, so q cells x
    // populations side by side take one addition's time where a loop over the
    // populations took q.  (FP32 is short of instructions, not of FP64 units: two
    // populations a thread.)  The next level's cell is fetched before the barrier.
    __device__ void upsweep() {
        const uint32_t *li = list(L_INT);
        const int ls = Jmin > 6 ? Jmin : 6;
        constexpr int cpb = TS / NPARTS;  // cells of a block pass
        const int c = tid / NPARTS, j = tid - c * NPARTS;
        int l = Jmax - 1;
        if (l >= ls) {
            int b = sm.seg[L_INT][l], e = sm.seg[L_INT][l + 1];
            uint32_t h = c < cpb && b + c < e ? li[b + c] : 0u;
#pragma unroll 1
            for (;;) {
                const int eb = b;
                if (h) project_part(h, j);
#pragma unroll 1
                for (int i = b + c + cpb; c < cpb && i < e; i += cpb) project_part(li[i], j);
                const bool some = b < e;
                --l;
                if (l >= ls) {
                    e = eb;
                    b = sm.seg[L_INT][l];
                    h = c < cpb && b + c < e ? li[b + c] : 0u;
                }
                if (some) sync();
                if (l < ls) break;
            }
        }
        if (Jmin < 6) {
            if (tid < 32) {
                const uint32_t *I = mask(sm.cur);
#pragma unroll 1
                for (l = Jmax - 1 < 5 ? Jmax - 1 : 5; l >= Jmin; --l) {
#pragma unroll 1
                    for (int i = tid; i < (NPARTS << l); i += 32) {
                        const uint32_t k = (uint32_t)i / (uint32_t)NPARTS, h = (1u << l) + k;
                        if (bit_of(I, h)) project_part(h, i - (int)k * NPARTS);
                    }
                    __syncwarp();
                }
            }
            sync();
        }
    }

    // A1 by conservation.  The stream (S5) moves every leaf by sigma 2^-dj times
    // the difference of what crosses its two edges, one value per interface
    // shared by the two cells it separates (for |w| = 2 the sum of the two cells
    // upwind of it), so the size-weighted mean of the leaves under an internal
    // cell moves by the same expression at the cell's own two edges (the inner
    // interfaces cancel), and the internal cells hold the projection of f* (S2;
    // ghosts lie outside the tree).  One update of every internal cell, all
    // levels in one pass, therefore equals the level-by-level projection of the
    // streamed leaves up to rounding, and replaces its Jmax - Jmin dependent
    // passes.  It runs in the stream's own pass: it reads only Phi, which S4
    // completed, and the internal cells, which the leaves' stream does not touch.
    // With it the internal cells hold the projection of the leaves between any
    // two calls: the initial state projects them, the stream moves them, and a
    // cell that becomes internal is the projection of the pair predicted from it.
    __device__ __forceinline__ void project_by_flux_pass() {
        const uint32_t *li = list(L_INT);
        const int e = sm.seg[L_INT][top()];
#pragma unroll 1
        for (int i = tid; i < e; i += TS) {
            const uint32_t h = li[i];
            T f[q];
            if constexpr (DQ)
                stream_cell_dq(h, f);
            else
                stream_cell(h, f);
            store_cell(h, f);
        }
    }
    // the D1Q2^n stream of cell h (leaf or internal): f + w (Phi[first] - Phi[next])
    __device__ __forceinline__ void stream_cell(uint32_t h, T *f) const {
        const int dj = Jmax - level_of(h);
        const uint32_t first = (h << dj) & ((1u << Jmax) - 1u);
        uint32_t next = first + (1u << dj);
        if (bc == 0) next &= (1u << Jmax) - 1u;
        const T w = pow2m<T>(dj);
        load_cell(h, f);
        T x[q], y[q];
        load_pops(phi(first), x);
        load_pops(phi(next), y);
#pragma unroll
        for (int j = 0; j < q; ++j) f[j] = f[j] + ((j & 1) ? -w : w) * (x[j] - y[j]);
    }

    // ---- A2: details of the pairs of the tree, threshold T, Harten flags ----
    // KEEP / REF bits go to the pair's parent p (both children of a kept pair
    // are kept)
    __device__ void details() {
        const uint32_t *lst = list(L_INT);
        const int e = sm.seg[L_INT][top()];
        uint32_t *keep = mask(M_KEEP), *ref = mask(M_REF);
#pragma unroll 1
        for (int i = tid; i < e; i += TS) {
            const uint32_t p = lst[i];
            bool keepit, refit, tie;
            pair_decision<T, q, WIDE>(V, p, Jmax, bc, WIDE ? d.gamma : 1, tab, sm.th, keepit, refit, tie);
            if (tie) atomicAdd(&sm.near_ties, 1);
            if (keepit) {
                const uint32_t bit = 1u << (p & 31u);
                atomicOr(&keep[p >> 5], bit);
                if (refit) atomicOr(&ref[p >> 5], bit);
            }
        }
    }
    // ---- candidate words of the step -----------------------------------------
    // (gamma = 1.)  A cell that becomes internal is within one cell of a kept
    // one, a child of a refined one, or an ancestor that grading requires, and
    // those lie within three cells of an internal cell of the old tree on their
    // level, or of a child of one; ghost parents lie one cell further.  All of
    // them are in the words next to (+-1 word) a word that holds an old internal
    // cell or a child word of one.  Those words, and the first 32 words, are
    // the step's candidates.  The word passes (enlargement, grading, list
    // compaction, clearing) visit them only; every other word of every bit array
    // stays zero.  The list is built from the occupancy array of the old tree,
    // a heap of words, by a block scan.
    __device__ __forceinline__ uint32_t cand_bits(const uint32_t *oc, uint32_t j) const {
        if (j == 0u) return FULL;
        auto near = [&](uint32_t i) { return oc[i] | children_word(oc, i); };
        uint32_t xl, xr;
        words_beside(near, j, bc, xl, xr);
        return dilate_edges(near(j), xl, xr, 1);
    }
    __device__ void build_cw() {
        constexpr int NW = TS / 32;
        const int lane = tid & 31, warp = tid >> 5;
        const uint32_t *oc = occ(sm.cur);
        uint32_t *cw = cwl();
        const int OW = d.OW;
        int run = 0;
        if (tid >= 5 && tid < 10) sm.cw_seg[tid] = 1 << (tid - 5);  // words 0..31 are all candidates
#pragma unroll 1
        for (int r = 0, base = 0; base < OW; ++r, base += TS) {
            const uint32_t j = base + tid;
            uint32_t c = j < (uint32_t)OW ? cand_bits(oc, j) : 0u;
            const uint32_t cnt = __popc(c);
            uint32_t x = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL, x, o);
                if (lane >= o) x += y;
            }
            uint32_t *sw = bx.scan_w[r & 1][0];  // alternate buffers: one barrier per round
            if (lane == 31) sw[warp] = x;
            sync();
            const uint32_t v = lane < NW ? sw[lane] : 0u;
            const uint32_t before = __reduce_add_sync(FULL, lane < warp ? v : 0u);
            const uint32_t tot = __reduce_add_sync(FULL, v);
            uint32_t off = run + before + x - cnt;
            // the words of level l >= 10 start with occupancy word 2^(l - 10)
            if (j > 0u && j < (uint32_t)OW && (j & (j - 1u)) == 0u) sm.cw_seg[10 + level_of(j)] = off;
#pragma unroll 1
            while (c) {
                const int b = __ffs(c) - 1;
                c &= c - 1u;
                cw[off++] = 32u * j + (uint32_t)b;
            }
            run += tot;
        }
        if (tid == 0) {
            sm.cw_seg[Jmax] = run;
            sm.ncw = run;
        }
        sync();
    }

    // ---- A3: H(T) per word: kept pairs dilated by sigma (one pair for sigma = 1
    // and 2), children of refined pairs
    __device__ void enlarge(uint32_t *In) {
        const uint32_t *keep = mask(M_KEEP), *ref = mask(M_REF);
        const int n = nwords();
#pragma unroll 1
        for (int i = tid; i < n; i += TS) {
            const uint32_t w = word_at(i);
            In[w] = dilate_word(keep, w, 1, bc) | children_word(ref, w) | above(w);
        }
    }

    // ---- A4: grading (Def. Graded tree), fine to coarse -----------------------
    // An internal cell p of level l needs the cells p + delta, |delta| <= gamma,
    // in the tree: their parents must be internal.  The levels of more than 32
    // words take one block pass each; the others go to one warp: lane i holds
    // word i of the current level in a register, the words beside it and the
    // folded halves arrive by shuffles, and no block barrier separates them.
    __device__ void grade(uint32_t *In) {
        const int g = WIDE ? d.gamma : 1;
        const int lwarp = Jmax - 1 < 10 ? Jmax - 1 : 10;
#pragma unroll 1
        for (int l = Jmax - 1; l > lwarp && l > Jmin; --l) {
            // words of level l - 1 from level l
            int b = 1 << (l - 6), e = 2 * b;
            if constexpr (SPM != 0) {
                b = sm.cw_seg[l - 1];
                e = sm.cw_seg[l];
            }
#pragma unroll 1
            for (int i = b + tid; i < e; i += TS) {
                const uint32_t w = SPM != 0 ? cwl()[i] : (uint32_t)i;
                const uint32_t x0 = In[2u * w], x1 = In[2u * w + 1u];
                const uint32_t lo = level_first(w);
                const bool first = w == lo, last = w + 1u == 2u * lo;
                uint32_t xl, xr;
                if (bc == 0) {
                    xl = In[first ? 4u * lo - 1u : 2u * w - 1u];
                    xr = In[last ? 2u * lo : 2u * w + 2u];
                } else {
                    xl = first ? 0u : In[2u * w - 1u];
                    xr = last ? 0u : In[2u * w + 2u];
                }
                In[w] |= graded_parents(x0, xl, x1, g) | (graded_parents(x1, x0, xr, g) << 16);
            }
            sync();
        }
        if (tid < 32) {
            const int lane = tid;
            int l = lwarp;
            uint32_t x0 = 0u;  // the level's 32 cells when l = 5
            if (l >= 5) {
                const uint32_t W = 1u << (l - 5);
                uint32_t x = lane < (int)W ? In[W + lane] : 0u;
#pragma unroll 1
                for (; l > 5 && l > Jmin; --l) {
                    const int n = 1 << (l - 5);
                    const uint32_t up = lane < n / 2 ? In[n / 2 + lane] : 0u;
                    uint32_t xl = __shfl_sync(FULL, x, (lane - 1) & (n - 1)), xr = __shfl_sync(FULL, x, (lane + 1) & (n - 1));
                    if (bc != 0) {
                        if (lane == 0) xl = 0u;
                        if (lane == n - 1) xr = 0u;
                    }
                    const uint32_t z = graded_parents(x, xl, xr, g);
                    const uint32_t z0 = __shfl_sync(FULL, z, (2 * lane) & 31), z1 = __shfl_sync(FULL, z, (2 * lane + 1) & 31);
                    x = up | z0 | (z1 << 16);
                    if (lane < n / 2) In[n / 2 + lane] = x;
                }
                x0 = x;
            }
            // level 5 (one word) and the levels of word 0, by lane 0
            if (lane == 0 && Jmin < 5) {
                uint32_t y = In[0];
                if (l == 5) {
                    const uint32_t e = bc == 0 ? x0 : 0u;
                    y |= graded_parents(x0, e, e, g) << 16;
                    l = 4;
                }
#pragma unroll 1
                for (; l > Jmin; --l) {
                    uint32_t z = y;
                    for (int s = 0; s < g; ++s) z = dilate_word0(z, bc);
                    z &= (2u << (2 * (1 << l) - 1)) - (1u << (1 << l));  // the cells of level l
                    z = (z | (z >> 1)) & 0x55555555u;                    // bit 2p: parent p
                    y |= compact_even(z);
                }
                In[0] = y;
            }
        }
        sync();
    }

    // ---- A5: list compaction -------------------------------------------------
    // With the tree graded every list is a word operation: internal cells I,
    // leaves (children of I outside I), pairs new to the tree I \ I_old, whose
    // values the transfer predicts (an internal cell among them is its
    // children's projection at once), and ghost pairs.  The reconstruction
    // window of a leaf reaches 2 gamma cells, gamma pairs, and so does the
    // closure of the ghosts under prediction stencils: a ghost within 2 gamma
    // cells of a tree cell has its parent within gamma of a tree cell and its
    // stencil within 2 gamma of it; and beyond an internal cell's gamma
    // neighbours (in the tree) the next cells are within reach of a leaf.  The
    // ghost pairs are therefore the gamma-dilation of I without I, at every
    // level but the finest.  (A sweep with its own marks per level, from fine to
    // coarse, gave the same sets; the marks were a third of the step's bit work.)
    //
    // Rounds of TS units; a unit is a word or, when there are fewer words than
    // threads, a part of one, so that the threads share the entries of dense
    // words.  A block scan of the units' counts, two counts per 32-bit value,
    // places the entries (the lists stay sorted).  KEEP and REF, read for the
    // last time by A3, are cleared on the way.
    __device__ void build_lists(const uint32_t *In, const uint32_t *Io, uint32_t *occn) {
        constexpr int NW = TS / 32;
        const int lane = tid & 31, warp = tid >> 5;
        const int g = WIDE ? d.gamma : 1;
        const int nw = nwords();
        uint32_t *keep = mask(M_KEEP), *ref = mask(M_REF);
        int s = 0;
        while (s < 3 && (nw << (s + 1)) <= TS) ++s;
        const int nu = nw << s, width = 32 >> s;
        const uint32_t wend = d.Wtot;
        uint32_t run[NLIST] = {0u, 0u, 0u, 0u};
        if (tid == 0) sm.deplev[0] = sm.deplev[1] = 0u;  // new lists: gathered again by predict_fill
#pragma unroll 1
        for (int r = 0, base = 0; base < nu; ++r, base += TS) {
            const int u = base + tid;
            uint32_t m[3] = {0u, 0u, 0u}, lf0 = 0u, lf1 = 0u, w = 0u, xp = 0u;
            const bool whole = u < nu && (u & ((1 << s) - 1)) == 0;  // the first unit of its word
            if (u < nu) {
                w = word_at(u >> s);
                const uint32_t x = In[w], pm = (FULL >> (32 - width)) << ((u & ((1 << s) - 1)) * width);
                xp = x & pm;
                if (2u * w < wend || w == 0u) m[L_GH] = dilate_word(In, w, g, bc) & ~x & pm;
                if (w == 0u) m[L_GH] &= (1u << (Jmax - 1 < 5 ? 1 << (Jmax - 1) : 31)) * (Jmax - 1 < 5 ? 1u : 2u) - 1u;
                if (whole) {
                    keep[w] = 0u;
                    ref[w] = 0u;
                    if constexpr (SPM != 0)
                        if (x) atomicOr(&occn[w >> 5], 1u << (w & 31u));
                }
            }
            // most words of a fine level are empty: a warp without entries skips the scan
            const bool some = __any_sync(FULL, (xp | m[L_GH]) != 0u);
            // per round at most 1024 x 32 internal cells and new pairs (16 bits
            // each), 1024 x 64 leaves (17 bits), 1024 x 28 ghost pairs (15 bits)
            uint32_t x01 = 0u, x23 = 0u, c01 = 0u, c23 = 0u;
            if (some) {
                if (xp) {
                    const uint32_t c0 = 2u * w < wend ? In[2u * w] : 0u, c1 = 2u * w + 1u < wend ? In[2u * w + 1u] : 0u;
                    m[L_INT] = xp & ~above(w);
                    m[L_PRED] = xp & ~Io[w];
                    lf0 = spread16(xp) & ~c0;
                    lf1 = spread16(xp >> 16) & ~c1;
                }
                x01 = c01 = (uint32_t)__popc(m[0]) | ((uint32_t)__popc(m[1]) << 16);
                x23 = c23 = (uint32_t)(__popc(lf0) + __popc(lf1)) | ((uint32_t)__popc(m[2]) << 17);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y01 = __shfl_up_sync(FULL, x01, o), y23 = __shfl_up_sync(FULL, x23, o);
                    if (lane >= o) {
                        x01 += y01;
                        x23 += y23;
                    }
                }
            }
            uint32_t(*sw)[32] = bx.scan_w[r & 1];  // alternate buffers: one barrier per round
            if (lane == 31) {
                sw[0][warp] = x01;
                sw[1][warp] = x23;
            }
            sync();
            const uint32_t v01 = lane < NW ? sw[0][lane] : 0u, v23 = lane < NW ? sw[1][lane] : 0u;
            const uint32_t t01 = __reduce_add_sync(FULL, v01), t23 = __reduce_add_sync(FULL, v23);
            // the first word of a level; a candidate list may leave whole levels out
            const bool starts = whole && w > 0u && (SPM != 0 || (w & (w - 1u)) == 0u);
            if (some || __any_sync(FULL, starts)) {
                x01 += __reduce_add_sync(FULL, lane < warp ? v01 : 0u) - c01;
                x23 += __reduce_add_sync(FULL, lane < warp ? v23 : 0u) - c23;
                const uint32_t at[3] = {run[0] + (x01 & 0xFFFFu), run[1] + (x01 >> 16), run[2] + (x23 >> 17)};
                if (starts) {
                    const int l = 5 + level_of(w);
                    int k = l;
                    if constexpr (SPM != 0) {
                        const uint32_t before = word_at((u >> s) - 1);  // a list starts with words 0, 1, ...
                        k = before == 0u ? 5 : 6 + level_of(before);
                    }
                    for (; k <= l; ++k)
#pragma unroll
                        for (int L = 0; L < NSEG; ++L) sm.seg[L][k] = at[L];
                }
                const uint32_t h0 = 32u * w;
#pragma unroll
                for (int L = 0; L < NSEG; ++L) {
                    uint32_t *dst = list(L) + at[L];
                    uint32_t x = m[L];
#pragma unroll 1
                    while (x) {
                        *dst++ = h0 + (uint32_t)__ffs(x) - 1u;
                        x &= x - 1u;
                    }
                }
                uint32_t *dst = list(L_LEAF) + run[3] + (x23 & 0x1FFFFu);
#pragma unroll 1
                while (lf0) {
                    *dst++ = 2u * h0 + (uint32_t)__ffs(lf0) - 1u;
                    lf0 &= lf0 - 1u;
                }
#pragma unroll 1
                while (lf1) {
                    *dst++ = 2u * h0 + 31u + (uint32_t)__ffs(lf1);
                    lf1 &= lf1 - 1u;
                }
            }
            run[0] += t01 & 0xFFFFu;
            run[1] += t01 >> 16;
            run[2] += t23 >> 17;
            run[3] += t23 & 0x1FFFFu;
        }
        if (tid == 0) {
            // the end of the finest level (and of the levels that no candidate word reached)
            int k = top();
            if constexpr (SPM != 0) k = 6 + level_of(word_at(nw - 1));
            for (; k <= top(); ++k)
#pragma unroll
                for (int L = 0; L < NSEG; ++L) sm.seg[L][k] = run[L];
            sm.nleaf = run[3];
        }
        sync();
    }

    // ---- A6 / S3: prediction of listed pairs ----------------------------------
    // the children of p from p's level, whose first cell is lo (Section 3.1)
    __device__ __forceinline__ void predict_pair(uint32_t p, uint32_t lo) const {
        T a[2 * q];
        const T *vp = cell(p), *vl = cell(nb(p, -1, lo)), *vr = cell(nb(p, 1, lo));
#pragma unroll
        for (int h = 0; h < q; ++h) {
            T t = T(C1) * (vr[h] - vl[h]);  // exact: c_1 is a power of two
            if constexpr (WIDE) t = wide_sum<T, q>(V, p, lo, bc, d.gamma, tab.pc[d.gamma], h, t);
            a[h] = vp[h] + t;
            a[q + h] = vp[h] - t;
        }
        store_cell(2u * p, a);
        store_cell(2u * p + 1u, a + q);
    }
    // whether the stencil of the pair's prediction holds a cell outside the tree I
    __device__ __forceinline__ bool stencil_outside(const uint32_t *I, uint32_t p, uint32_t lo) const {
        const int g = WIDE ? d.gamma : 1;
        bool all = true;
        for (int a = -g; a <= g; ++a) all = all && bit_of(I, nb(p, a, lo) >> 1);
        return !all;
    }
    // A listed pair whose stencil lies in the tree I (the old tree for the
    // transfer, the current one for the ghosts) reads only tree values, so those
    // pairs go in one pass over all levels; the others, whose stencils hold
    // pairs of the same list, follow level by level, coarse to fine, on the
    // levels that have any.
    __device__ void predict_fill(int L, const uint32_t *I) {
        const uint32_t *lst = list(L);
        uint32_t *dep = &sm.deplev[L == L_GH ? 1 : 0];
        const int n = sm.seg[L][top()];
#pragma unroll 1
        for (int i = tid; i < n; i += TS) {
            const uint32_t p = lst[i], lo = level_first(p);
            if (stencil_outside(I, p, lo))
                atomicOr(dep, lo);
            else
                predict_pair(p, lo);
        }
        sync();
        uint32_t lv = *dep;
#pragma unroll 1
        while (lv) {
            const int l = __ffs(lv) - 1;
            lv &= lv - 1u;
            const int b = l >= 5 ? sm.seg[L][l] : 0, e = sm.seg[L][l >= 5 ? l + 1 : 5];
#pragma unroll 1
            for (int i = b + tid; i < e; i += TS) {
                const uint32_t p = lst[i], lo = 1u << l;
                if (level_of(p) == l && stencil_outside(I, p, lo)) predict_pair(p, lo);
            }
            sync();
        }
    }

    // ---- mesh adaptation ----------------------------------------------------
    __device__ void adapt() {
        uint32_t *Io = mask(sm.cur), *In = mask(sm.cur ^ 1);
        tick(NPHASE);
        if constexpr (SPM != 0) {
            build_cw();
            uint32_t *on = occ(sm.cur ^ 1);  // the occupancy array the list compaction will fill
#pragma unroll 1
            for (int j = tid; j < d.OW; j += TS) on[j] = 0u;
        }
        tick(T_CANDIDATES);
        if (!(sm.status & ST_DETAILS)) details();  // else the initial state came with its decisions
        sync();
        tick(T_DETAILS);
        enlarge(In);
        sync();
        tick(T_ENLARGE);
        grade(In);
        tick(T_GRADE);
        build_lists(In, Io, SPM != 0 ? occ(sm.cur ^ 1) : nullptr);
        tick(T_LISTS);
        predict_fill(L_PRED, Io);
        if constexpr (SPM != 0) {
            // the old tree's buffer holds the next step's new tree: clear it (its
            // cells lie in candidate words); without candidate words the
            // enlargement writes every word
            const uint32_t *cw = cwl();
            const int ncw = sm.ncw;
#pragma unroll 1
            for (int i = tid; i < ncw; i += TS) Io[cw[i]] = 0u;
        }
        tick(T_TRANSFER);
        if (tid == 0) {
            sm.cur ^= 1;
            sm.updates += (unsigned long long)sm.nleaf;
            if (sm.status & ST_DETAILS) {
                sm.near_ties += d.st->first_ties;
                sm.status &= ~(int)ST_DETAILS;
            }
        }
        sync();
    }

    // ---- one step of the adaptive scheme on the current mesh -----------------
    __device__ void lbm_step() {
        tick(NPHASE);
        if (sm.status & ST_DETAILS) {
            // the step moves the state that the initial decisions belong to
            clear_masks();
            sync();
            if (tid == 0) sm.status &= ~(int)ST_DETAILS;
        }
        if constexpr (WIDE) {
            if (d.collision)
                collide_reconstructed();  // S1, eq. reconstructedCollision
            else
                collide_all();
        } else {
            collide_all();  // S1
        }
        sync();
        tick(T_COLLIDE);
        upsweep();  // S2
        tick(T_UPSWEEP_S);
        predict_fill(L_GH, mask(sm.cur));  // S3
        tick(T_GHOSTS);
        if constexpr (DQ)
            reconstruct_dq();  // S4 (gamma = 1)
        else if (WIDE && d.gamma > 1) {
            if constexpr (WIDE) {
                if (d.gamma == 2)
                    reconstruct_wide<2>();
                else
                    reconstruct_wide<3>();
            }
        } else
            reconstruct_edges();
        sync();
        tick(T_RECON);
        if constexpr (DQ)
            stream_dq();  // S5
        else
            stream_and_audit();
        tick(T_STREAM);
    }

    // sum of four products; FP32: compensated (Kahan) accumulation
    static __device__ __forceinline__ T dot4(const T *w, T x0, T x1, T x2, T x3) {
        if constexpr (sizeof(T) == 8) {
            return fma(w[3], x3, fma(w[2], x2, fma(w[1], x1, w[0] * x0)));
        } else {
            T p[4] = {w[0] * x0, w[1] * x1, w[2] * x2, w[3] * x3};
            T s = T(0), comp = T(0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                T y = p[j] - comp;
                T t = s + y;
                comp = (t - s) - y;
                s = t;
            }
            return s;
        }
    }

    // weights next to a finer neighbour.  FP64: t4, on the two children of the
    // neighbour, the leaf and its other neighbour (the leaf's predicted children
    // and the projection of the refined neighbour folded into the weights: four
    // FP64 operations instead of eight).  FP32: t1, on the neighbour's children and
    // the leaf's own predicted ones (the operations are cheap there).
    // sec 1: those of the second cell from the edge.
    __device__ __forceinline__ const T *finer_weights(int dj, int sec = 0) const {
        if constexpr (sizeof(T) == 8) return sec ? tab.t42[dj] : tab.t4[dj];
        return sec ? tab.t12[dj] : tab.t1[dj];
    }
    // S4: first / last finest-cell values of every leaf -> Phi, from the
    // per-level-gap tables.  One sum of four products for both stencils, so that
    // a warp whose leaves mix them evaluates it once: next to a finer neighbour
    // the finer weights, else the cells of the leaf's level with the weights cf;
    // the mirrored sum for the last value.
    __device__ void reconstruct_edges() {
        const uint32_t *I = mask(sm.cur);
        const uint32_t *leaves = list(L_LEAF);
        const int nl = sm.nleaf;
        const uint32_t N = 1u << Jmax;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t h = leaves[i], lo = level_first(h);
            const int dj = Jmax - level_of(h);
            const uint32_t hl = nb(h, -1, lo), hr = nb(h, 1, lo);
            const bool at_left = bc == 1 && h == lo, at_right = bc == 1 && h + 1u == 2u * lo;
            const uint32_t first = (h << dj) & (N - 1u);
            uint32_t next = first + (1u << dj);
            if (bc == 0) next &= N - 1u;
            T *pf = phi(first), *pn = phi(next);
            if (dj == 0) {
                const T *v = cell(h);
#pragma unroll
                for (int j = 0; j < NF; ++j) {
                    const T vp = v[2 * j], vm = v[2 * j + 1];
                    pn[2 * j] = vp;
                    pf[2 * j + 1] = vm;
                    if (at_left) pf[2 * j] = vp;
                    if (at_right) pn[2 * j + 1] = vm;
                }
                continue;
            }
            const bool fin_l = !at_left && bit_of(I, hl), fin_r = !at_right && bit_of(I, hr);
            // where the two outer values of each sum come from
            const T *l0 = fin_l ? cell(2u * hl) : cell(nb(h, -2, lo)), *l1 = fin_l ? cell(2u * hl + 1u) : cell(hl);
            const T *r0 = fin_r ? cell(2u * hr) : cell(hr), *r1 = fin_r ? cell(2u * hr + 1u) : cell(nb(h, 2, lo));
            const T *vm1 = cell(hl), *v0 = cell(h), *vp1 = cell(hr);
            const T *wl = fin_l ? finer_weights(dj) : tab.cf[dj], *wr = fin_r ? finer_weights(dj) : tab.cf[dj], *bf = tab.bf[dj];
            const T wm[4] = {wr[3], wr[2], wr[1], wr[0]};
#pragma unroll
            for (int j = 0; j < NF; ++j) {
                {  // velocity +lambda: the last value (and the first at the left boundary)
                    const int c = 2 * j;
                    const T a = vm1[c], b = v0[c], e = vp1[c];
                    T x0 = a, x1 = b;
                    if (sizeof(T) == 4 && fin_r) {
                        const T tt = T(C1) * (e - a);
                        x0 = b + tt;
                        x1 = b - tt;
                    }
                    pn[c] = at_right ? bf[0] * b + bf[1] * a : dot4(wm, x0, x1, r0[c], r1[c]);
                    if (at_left) pf[c] = bf[0] * b + bf[1] * e;
                }
                {  // velocity -lambda: the first value (and the last at the right boundary)
                    const int c = 2 * j + 1;
                    const T a = vm1[c], b = v0[c], e = vp1[c];
                    T x2 = b, x3 = e;
                    if (sizeof(T) == 4 && fin_l) {
                        const T tt = T(C1) * (e - a);
                        x2 = b + tt;
                        x3 = b - tt;
                    }
                    pf[c] = at_left ? bf[0] * b + bf[1] * e : dot4(wl, l0[c], l1[c], x2, x3);
                    if (at_right) pn[c] = bf[0] * b + bf[1] * a;
                }
            }
        }
    }

    // First (LAST = false) or last finest value of population c of the leaf h,
    // by the reconstruction operator of Section 3.3 (Definition V): the window
    // h - 2G .. h + 2G (tree and ghost values) is predicted level by level down
    // to Jmax around the leaf's first (last) finest cell, and wherever a finer
    // level holds a cell of the tree (the children of refined neighbours) its
    // value is used instead.  Out-of-domain cells take the value of the nearest
    // domain cell (copy boundary) or wrap (periodic), as in the prediction.
    template <int G, bool LAST>
    __device__ __noinline__ T edge_walk(const uint32_t *I, const T *cf, int c, uint32_t h) const {
        constexpr int W = 4 * G + 1, C = 2 * G, E = LAST ? 1 : 0;
        T w[W], nw[W];
        uint32_t lo = level_first(h);
#pragma unroll
        for (int t = 0; t < W; ++t) w[t] = cell(nb(h, t - C, lo))[c];
#pragma unroll 1
        for (int m = level_of(h); m < Jmax; ++m) {
            h = 2u * h + E;
            lo *= 2u;
            T vlo = T(0), vhi = T(0);  // values of the first and last cells of the level (copy boundary)
#pragma unroll
            for (int t = 0; t < W; ++t) {
                // window position t is cell h + t - C; its parent is window position pp of the level above
                const int pp = C + ((E + t - C) >> 1);
                const bool odd = ((E + t - C) & 1) != 0;
                const uint32_t x = h + (uint32_t)(t - C);
                const bool inside = bc == 0 || (x >= lo && x < 2u * lo);
                const uint32_t xc = lo | (x & (lo - 1u));
                T v;
                if (inside && bit_of(I, xc >> 1)) {
                    v = cell(xc)[c];
                } else {
                    T sum = cf[0] * (w[pp + 1] - w[pp - 1]);
#pragma unroll
                    for (int a = 2; a <= G; ++a) sum = sum + cf[a - 1] * (w[pp + a] - w[pp - a]);
                    v = odd ? w[pp] - sum : w[pp] + sum;
                }
                nw[t] = v;
                if (x == lo) vlo = v;
                if (x == 2u * lo - 1u) vhi = v;
            }
            if (bc != 0) {
#pragma unroll
                for (int t = 0; t < W; ++t) {
                    const uint32_t x = h + (uint32_t)(t - C);
                    if (x < lo) nw[t] = vlo;
                    if (x >= 2u * lo) nw[t] = vhi;
                }
            }
#pragma unroll
            for (int t = 0; t < W; ++t) w[t] = nw[t];
        }
        return w[C];
    }

    // S4 with the stencil of half-width G = 2 or 3: the first / last finest value
    // of a leaf from its level's window (h - 2G .. h + 2G) and the tables.  Where
    // a cell p of the window within G of the leaf is refined, the tree's children
    // of p stand in the window one level down in the place of the predicted ones;
    // the two differ by the pair's detail, with opposite signs, and the weights of
    // that window carry the difference.  Further down the window holds no tree
    // cell: a cell two levels below the leaf's needs, graded, the cells within G
    // of its parent in the tree, and the leaf's children are not.  So a value
    // costs 4G products and 2G + 3 operations a refined cell, where the
    // level-by-level walk (edge_walk) predicted the whole window at each of the
    // Jmax - l levels: 178K of a step's 238K cycles on a gamma = 3 batch (FP64).
    // The walk is left for a leaf within 2G cells of both copy boundaries.
    // The weights of a window sum to one, so they go to the differences from the
    // leaf's value, which is added last: a constant state comes back as it is, and
    // the weights' rounding and the sum's count for the differences alone.  Random
    // windows in FP32, rms error in units of 2^-24 at gaps 1 / 2 / 8, gamma = 3:
    // 0.46 / 0.48 / 0.55, the walk 0.46 / 0.72 / 1.44, the weights on the values
    // themselves 0.93 / 1.05 / 1.39.  The subtractions cost 3 to 5 % of a gamma = 3
    // step in FP64 (batch of 300: 87.3 -> 89.9 us), 1 to 3 % with gamma = 2 and up to
    // 3 % in FP32; a chain of products a side of the window gained nothing.
    // Gap 1 is the predicted child by the exact coefficients (by the tables: 95 us).
    template <int G>
    __device__ __noinline__ void reconstruct_wide() {
        constexpr int C = 2 * G, W = 4 * G + 1;
        const uint32_t *I = mask(sm.cur);
        const uint32_t *leaves = list(L_LEAF);
        const int nl = sm.nleaf;
        const T *cf = tab.pc[G];
        const T *wt = G == 2 ? &wide->w2[0][0][0] : &wide->w3[0][0][0];
        const uint32_t N = 1u << Jmax;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t h = leaves[i], lo = level_first(h);
            const int dj = Jmax - level_of(h);
            const bool at_left = bc == 1 && h == lo, at_right = bc == 1 && h + 1u == 2u * lo;
            const uint32_t first = (h << dj) & (N - 1u);
            uint32_t next = first + (1u << dj);
            if (bc == 0) next &= N - 1u;
            const int kl = bc == 0 ? C : min((int)(h - lo), C), kr = bc == 0 ? C : min((int)(2u * lo - 1u - h), C);
            unsigned refined = 0u;  // cells within G that are internal
            if (dj > 0)
#pragma unroll
                for (int o = -G; o <= G; ++o)
                    // beyond a copy boundary stands the boundary cell, whose children are predicted there like its own
                    if (o != 0 && (o > 0 ? o <= kr : -o <= kl) && bit_of(I, nb(h, o, lo))) refined |= 1u << (o + G);
#pragma unroll 1
            for (int e = 0; e < q + (at_left ? NF : 0) + (at_right ? NF : 0); ++e) {
                // population and end: +lambda its last value, -lambda its first; at a boundary the other end too
                int c = e;
                bool last = (c & 1) == 0;
                if (e >= q) {
                    const bool l = at_left && e < q + NF;
                    c = 2 * (e - q - (at_left && !l ? NF : 0)) + (l ? 0 : 1);
                    last = !l;
                }
                T *out = phi(last ? next : first) + c;
                const T *vc = V + c;
                auto at = [&](uint32_t x) { return vc[x * (uint32_t)q]; };
                const T xc = at(h);
                if (dj == 0) {
                    *out = xc;
                    continue;
                }
                const int sg = last ? -1 : 1, k = last ? kr : kl, r = last ? kl : kr;  // distances, mirrored for the last value
                // sum_a c_a (x_{p+a} - x_{p-a}), mirrored for the last value
                auto slope = [&](uint32_t p) {
                    T s = cf[0] * (at(nb(p, sg, lo)) - at(nb(p, -sg, lo)));
#pragma unroll
                    for (int a = 2; a <= G; ++a) s = s + cf[a - 1] * (at(nb(p, sg * a, lo)) - at(nb(p, -sg * a, lo)));
                    return s;
                };
                if (dj == 1) {  // the predicted child itself
                    *out = xc + slope(h);
                    continue;
                }
                if (kl < C && kr < C) {
                    *out = last ? edge_walk<G, true>(I, cf, c, h) : edge_walk<G, false>(I, cf, c, h);
                    continue;
                }
                const int code = k < C ? 1 + k : r < C ? 1 + C + r : 0;
                const T *w = wt + (code * (MAXDJ + 1) + dj) * W;
                T sum = T(0);
#pragma unroll
                for (int t = 0; t < W; ++t)
                    if (t != C) sum = sum + w[t] * (at(nb(h, sg * (t - C), lo)) - xc);
                if (refined) {
                    const int k1 = 2 * k, r1 = 2 * r + 1;  // of the child at that end
                    const int code1 = code == 0 ? 0 : k < C ? (k1 < C ? 1 + k1 : 0) : (r1 < C ? 1 + C + r1 : 0);
                    const T *w1 = wt + (code1 * (MAXDJ + 1) + dj - 1) * W + C;
                    unsigned m = refined;
#pragma unroll 1
                    while (m) {
                        const int po = __ffs(m) - 1 - G, o = sg * po;
                        m &= m - 1u;
                        const uint32_t p = nb(h, po, lo);
                        const T detail = at(last ? 2u * p + 1u : 2u * p) - (at(p) + slope(p));
                        sum = sum + (w1[2 * o] - (o < G ? w1[2 * o + 1] : T(0))) * detail;
                    }
                }
                sum = sum + xc;
                *out = sum;
            }
        }
    }

    // S4 for the D1Q3 / D1Q5 schemes: every leaf writes the reconstructed
    // finest values it holds within |w^h| cells of its edges, by finest
    // position: a +v population needs the cells left of each interface (the
    // last |w| cells of a leaf), a -v population the cells right of it (the
    // first |w|); at a copy boundary also the cell next to the boundary, which
    // the clamped out-of-domain cells copy.  Second cells from an edge use the
    // second-cell tables.
    __device__ __noinline__ void reconstruct_dq() {
        const uint32_t *I = mask(sm.cur);
        const uint32_t *leaves = list(L_LEAF);
        const int nl = sm.nleaf;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t hc = leaves[i], lo = level_first(hc);
            const int dj = Jmax - level_of(hc);
            const uint32_t first = (hc << dj) & ((1u << Jmax) - 1u), last = first + (1u << dj) - 1u;
            const bool at_left = bc == 1 && hc == lo, at_right = bc == 1 && hc + 1u == 2u * lo;
            const uint32_t hl = nb(hc, -1, lo), hr = nb(hc, 1, lo);
            const bool fin_l = dj > 0 && !at_left && bit_of(I, hl), fin_r = dj > 0 && !at_right && bit_of(I, hr);
            const T *v0p = cell(hc), *vm1p = cell(hl), *vp1p = cell(hr), *vm2p = cell(nb(hc, -2, lo)), *vp2p = cell(nb(hc, 2, lo));
            const T *clp = cell(2u * hl), *crp = cell(2u * hr);
#pragma unroll 1
            for (int h = 1; h < q; ++h) {
                const int w = dq_w(h), a = w < 0 ? -w : w;
                if (dj == 0) {
                    phi(first)[h] = v0p[h];
                    continue;
                }
                const T vm1 = vm1p[h], v0 = v0p[h], vp1 = vp1p[h];
                // cell `sec` (0: first / last, 1: second from that edge) next to the left or right
                // edge: one sum of four products for both stencils (as in reconstruct_edges)
                auto from_left = [&](int sec) -> T {
                    const T *bf = sec ? tab.bf2[dj] : tab.bf[dj], *cf = sec ? tab.cf2[dj] : tab.cf[dj];
                    if (at_left) return bf[0] * v0 + bf[1] * vp1;
                    T x0, x1, x2, x3;
                    if (fin_l) {
                        x0 = clp[h];
                        x1 = clp[q + h];
                        x2 = v0;
                        x3 = vp1;
                        if constexpr (sizeof(T) == 4) {
                            const T tt = T(C1) * (vp1 - vm1);
                            x2 = v0 + tt;
                            x3 = v0 - tt;
                        }
                    } else {
                        x0 = vm2p[h];
                        x1 = vm1;
                        x2 = v0;
                        x3 = vp1;
                    }
                    return dot4(fin_l ? finer_weights(dj, sec) : cf, x0, x1, x2, x3);
                };
                auto from_right = [&](int sec) -> T {
                    const T *bf = sec ? tab.bf2[dj] : tab.bf[dj], *cf = sec ? tab.cf2[dj] : tab.cf[dj];
                    if (at_right) return bf[0] * v0 + bf[1] * vm1;
                    T x0, x1, x2, x3;
                    if (fin_r) {
                        x0 = vm1;
                        x1 = v0;
                        if constexpr (sizeof(T) == 4) {
                            const T tt = T(C1) * (vp1 - vm1);
                            x0 = v0 + tt;
                            x1 = v0 - tt;
                        }
                        x2 = crp[h];
                        x3 = crp[q + h];
                    } else {
                        x0 = vm1;
                        x1 = v0;
                        x2 = vp1;
                        x3 = vp2p[h];
                    }
                    const T *wt = fin_r ? finer_weights(dj, sec) : cf;
                    const T wm[4] = {wt[3], wt[2], wt[1], wt[0]};
                    return dot4(wm, x0, x1, x2, x3);
                };
                if (w > 0) {
                    phi(last)[h] = from_right(0);
                    if (a == 2) phi(last - 1u)[h] = from_right(1);
                    if (at_left) phi(first)[h] = from_left(0);
                } else {
                    phi(first)[h] = from_left(0);
                    if (a == 2) phi(first + 1u)[h] = from_left(1);
                    if (at_right) phi(last)[h] = from_right(0);
                }
            }
        }
    }

    // the D1Q3 / D1Q5 stream of cell h (eq. AdaptiveStreamPhase with |w| <= 2):
    // f + sigma 2^-dj sum_{delta=1}^{|w|} (V[first + eta] - V[next + eta]),
    // eta = -delta (sigma > 0) or delta - 1 (sigma < 0), V the finest values of
    // reconstruct_dq (wrapped, or clamped at a copy boundary)
    __device__ __forceinline__ uint32_t finest_at(int i) const {
        const int N = 1 << Jmax;
        return (uint32_t)(bc == 0 ? (i & (N - 1)) : min(max(i, 0), N - 1));
    }
    __device__ __forceinline__ void stream_cell_dq(uint32_t hc, T *f) const {
        const int dj = Jmax - level_of(hc);
        const int first = (int)((hc << dj) & ((1u << Jmax) - 1u)), next = first + (1 << dj);
        const T wgt = pow2m<T>(dj);
        load_cell(hc, f);
#pragma unroll
        for (int h = 1; h < q; ++h) {
            const int w = dq_w(h), a = w < 0 ? -w : w;
            auto across = [&](int dl) {
                const int eta = w > 0 ? -dl : dl - 1;
                return phi(finest_at(first + eta))[h] - phi(finest_at(next + eta))[h];
            };
            T acc = across(1);
            if (a == 2) acc = acc + across(2);
            f[h] = f[h] + (w > 0 ? wgt : -wgt) * acc;
        }
    }

    // S5 for the D1Q3 / D1Q5 schemes, with the audit of (h, hu)
    __device__ __noinline__ void stream_dq() {
        const uint32_t *leaves = list(L_LEAF);
        double macc[3] = {0.0, 0.0, 0.0};
        float fhi[3] = {0.0f, 0.0f, 0.0f}, flo[3] = {0.0f, 0.0f, 0.0f};
        bool bad = false;
        const int nl = sm.nleaf;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t hc = leaves[i];
            T fn[q];
            stream_cell_dq(hc, fn);
            store_cell(hc, fn);
#pragma unroll
            for (int h = 0; h < q; ++h) bad |= nonfinite(fn[h]);
            audit_cell(hc, fn, macc, fhi, flo);
        }
        if (bad) atomicOr(&sm.status, (int)ST_NONFINITE);
        project_by_flux_pass();  // A1 of the next adaptation, same pass
        finish_audit(macc, fhi, flo, nl);
    }

    // the audit's partial sums of one leaf: dx_l m_j in FP64, or, in the FP32
    // path, 2^-l m_j summed exactly per leaf into float-float partials
    // (relative error near 2^-44) and scaled by b - a at the end
    __device__ __forceinline__ void audit_cell(uint32_t h, const T *f, double (&macc)[3], float (&fhi)[3], float (&flo)[3]) const {
        const int l = level_of(h);
        if constexpr (sizeof(T) == 8) {
            const double dx = sm.dx_l[l];
            if constexpr (DQ) {
                double m0 = f[0] + (f[1] + f[2]), m1 = f[1] - f[2];
                if constexpr (q == 5) {
                    m0 += f[3] + f[4];
                    m1 += 2.0 * (f[3] - f[4]);
                }
                macc[0] += dx * m0;
                macc[1] += dx * m1;  // times lambda at the end
            } else {
#pragma unroll
                for (int j = 0; j < nf; ++j) macc[j] += dx * ((double)f[2 * j] + (double)f[2 * j + 1]);
            }
        } else {
            const float sc = pow2m<float>(l);
            if constexpr (DQ) {
                float a0 = 0.0f, e0 = 0.0f, a1 = 0.0f, e1 = 0.0f;
#pragma unroll
                for (int c = 0; c < q; ++c) {
                    ff_add(a0, e0, (float)f[c], 0.0f);
                    ff_add(a1, e1, (float)(dq_w(c)) * (float)f[c], 0.0f);
                }
                ff_add(fhi[0], flo[0], a0 * sc, e0 * sc);
                ff_add(fhi[1], flo[1], a1 * sc, e1 * sc);
            } else {
#pragma unroll
                for (int j = 0; j < nf; ++j) {
                    float sj, ej;
                    two_sum((float)f[2 * j], (float)f[2 * j + 1], sj, ej);
                    ff_add(fhi[j], flo[j], sj * sc, ej * sc);
                }
            }
        }
    }
    // End of a step: the totals of the conserved moments over the n leaves, and
    // the residual of their change against what crossed a copy boundary, one
    // field to a warp.  One barrier, after which the stream's results are there;
    // nothing before the next step's end reads what the folding warps write but
    // by the thread that wrote it (or after further barriers).
    __device__ __forceinline__ void finish_audit(double (&macc)[3], float (&fhi)[3], float (&flo)[3], int n) {
        if constexpr (sizeof(T) == 8)
            team_partials(macc, n);
        else
            team_partials_ff(fhi, flo, n);
        const int j = fold_field();
        if (j < 0) return;
        double total;
        if constexpr (sizeof(T) == 8)
            total = team_fold(j);
        else
            total = team_fold_ff(j);
        if ((tid & 31) != 0) return;
        if constexpr (sizeof(T) == 4) total *= d.b - d.a;
        double flux = 0.0;
        if constexpr (DQ) {
            // copy boundary: what leaves through x = a and x = b, sum over the
            // populations of sigma 2^-Jmax-weighted telescoped stream terms
            if (j == 1) total *= d.lam;
            if (bc == 1) {
                const double dxJ = sm.dx_l[Jmax];
                for (int h = 1; h < q; ++h) {
                    const int w = dq_w(h), a = w < 0 ? -w : w;
                    double t = 0.0;
                    for (int dl = 1; dl <= a; ++dl) {
                        const int eta = w > 0 ? -dl : dl - 1;
                        t += (double)phi(finest_at(eta))[h] - (double)phi(finest_at((1 << Jmax) + eta))[h];
                    }
                    t *= (w > 0 ? dxJ : -dxJ);
                    flux += j == 0 ? t : (w * d.lam) * t;
                }
            }
        } else if (bc == 1) {
            const T *p0 = phi(0u), *pN = phi(1u << Jmax);
            flux = sm.dx_l[Jmax] * (((double)p0[2 * j] - (double)pN[2 * j]) - ((double)p0[2 * j + 1] - (double)pN[2 * j + 1]));
        }
        sm.audit[j] = fmax(sm.audit[j], fabs(total - sm.mass[j] - flux));
        sm.mass[j] = total;
        if (j == 0) sm.steps += 1ULL;
    }

    // S5: f^{n+1} = f* + sigma 2^-dj (Phi[first] - Phi[next]); mass audit
    // (totals sum dx_l (f+ + f-) over the leaves)
    __device__ void stream_and_audit() {
        const uint32_t *leaves = list(L_LEAF);
        double macc[3] = {0.0, 0.0, 0.0};
        float fhi[3] = {0.0f, 0.0f, 0.0f}, flo[3] = {0.0f, 0.0f, 0.0f};
        bool bad = false;
        const int nl = sm.nleaf;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t h = leaves[i];
            T fn[q];
            stream_cell(h, fn);
            store_cell(h, fn);
#pragma unroll
            for (int j = 0; j < q; ++j) bad |= nonfinite(fn[j]);
            audit_cell(h, fn, macc, fhi, flo);
        }
        if (bad) atomicOr(&sm.status, (int)ST_NONFINITE);
        project_by_flux_pass();  // A1 of the next adaptation, same pass
        finish_audit(macc, fhi, flo, nl);
    }

    // ---- initial state -------------------------------------------------------
    // KEEP and REF, and the tree buffer beside the current one
    __device__ __forceinline__ void clear_masks() {
#pragma unroll 1
        for (int w = tid; w < d.Wtot; w += TS) {
            mask(sm.cur ^ 1)[w] = 0u;
            mask(M_KEEP)[w] = 0u;
            mask(M_REF)[w] = 0u;
        }
    }

    // arbitrary graded tree (one byte per cell) and values
    __device__ __noinline__ void init_state(const unsigned char *Rb, const double *vals) {
        if (tid == 0) sm.cur = M_I0;
        sync();
        clear_masks();
        uint32_t *I = mask(M_I0);
        const uint32_t off = 1u << Jmin;
#pragma unroll 1
        for (int w = tid; w < d.Wtot; w += TS) {
            uint32_t x = above(w);
            for (uint32_t b = 0; b < 32u; ++b) {
                const uint32_t h = 32u * w + b;  // internal: its first child is in the tree
                if (h >= off && h < (1u << Jmax) && Rb[2u * h - off]) x |= 1u << b;
            }
            I[w] = x;
        }
        // population-major input to the cell-major layout
#pragma unroll 1
        for (long long c = tid; c < (long long)q * d.S; c += TS) {
            const long long hh = c / d.S, k = c - hh * d.S;
            cell((uint32_t)(k + off))[hh] = (T)vals[c];
        }
        finish_init();
    }

    __device__ __noinline__ void finish_init() {
        if constexpr (SPM != 0) {
            // every word is a candidate of this first listing
            uint32_t *cw = cwl();
#pragma unroll 1
            for (int w = tid; w < d.Wtot; w += TS) cw[w] = (uint32_t)w;
#pragma unroll 1
            for (int j = tid; j < d.OW; j += TS) {
                occ(M_I0)[j] = 0u;
                occ(M_I1)[j] = 0u;
            }
            if (tid == 0) sm.ncw = d.Wtot;
        }
        sync();
        uint32_t *I = mask(M_I0);
        build_lists(I, I, SPM != 0 ? occ(M_I0) : nullptr);  // the tree is its own old tree
        upsweep();
        // FP64 totals of the initial leaves
        const uint32_t *leaves = list(L_LEAF);
        double macc[3] = {0.0, 0.0, 0.0};
        const int nl = sm.nleaf;
#pragma unroll 1
        for (int i = tid; i < nl; i += TS) {
            const uint32_t h = leaves[i];
            const T *f = cell(h);
            const double dx = sm.dx_l[level_of(h)];
            if constexpr (DQ) {
                double m0 = 0.0, m1 = 0.0;
                for (int c = 0; c < q; ++c) {
                    m0 += (double)f[c];
                    m1 += (dq_w(c) * d.lam) * (double)f[c];
                }
                macc[0] += dx * m0;
                macc[1] += dx * m1;
            } else {
                for (int j = 0; j < nf; ++j) macc[j] += dx * ((double)f[2 * j] + (double)f[2 * j + 1]);
            }
        }
        team_partials(macc, nl);
        if (const int j = fold_field(); j >= 0) {
            const double total = team_fold(j);
            if ((tid & 31) == 0) {
                sm.mass[j] = total;
                sm.audit[j] = 0.0;
            }
        }
        if (tid == 0) {
            sm.status = 0;
            sm.near_ties = 0;
            sm.updates = 0ULL;
        }
        if (tid == TS - 32) sm.steps = 0ULL;  // the thread that counts them
        if (tid == TS - 1) sm.passes = 0ULL;  // the thread that counts the barriers
        sync();
    }
};

// ---------------------------------------------------------------------------
// instance state in and out of shared memory (TS threads of the team)

template <typename T, int TS>
__device__ void load_instance(TeamSmem<T> &sm, const InstDesc &dg, int tid) {
    // the descriptor and the list segments, word by word
    for (int i = tid; i < (int)(sizeof(InstDesc) / 4); i += TS) ((uint32_t *)&sm.d)[i] = ((const uint32_t *)&dg)[i];
    const InstState &st = *dg.st;
    if (tid == 0) {
        sm.cur = st.cur;
        sm.nleaf = st.nleaf;
        sm.status = st.status;
        sm.near_ties = st.near_ties;
        sm.deplev[0] = st.deplev[0];
        sm.deplev[1] = st.deplev[1];
        sm.updates = st.updates;
        sm.steps = st.steps;
        sm.passes = st.passes;
        for (int j = 0; j < 3; ++j) {
            sm.mass[j] = st.mass[j];
            sm.audit[j] = st.audit;
        }
#ifdef MRG_PHASE_TIMERS
        for (int p = 0; p < NPHASE; ++p) sm.ptime[p] = st.ptime[p];
        sm.tlast = clock64();
#endif
    }
    for (int l = tid; l <= MAXLEV; l += TS) {
        sm.th.set(dg, l);
        sm.dx_l[l] = (dg.b - dg.a) * pow2m<double>(l);
    }
    for (int i = tid; i < NSEG * (MAXLEV + 2); i += TS) (&sm.seg[0][0])[i] = (&st.seg[0][0])[i];
    __syncthreads();
}

template <typename T, int TS>
__device__ void store_instance(TeamSmem<T> &sm, int tid) {
    // the barrier count of the last pass is written after that pass's barrier
    __syncthreads();
    InstState &st = *sm.d.st;
    if (tid == 0) {
        st.cur = sm.cur;
        st.nleaf = sm.nleaf;
        st.status = sm.status;
        st.near_ties = sm.near_ties;
        st.deplev[0] = sm.deplev[0];
        st.deplev[1] = sm.deplev[1];
        st.updates = sm.updates;
        st.steps = sm.steps;
        st.passes = sm.passes;
        st.audit = fmax(sm.audit[0], fmax(sm.audit[1], sm.audit[2]));
        for (int j = 0; j < 3; ++j) st.mass[j] = sm.mass[j];
#ifdef MRG_PHASE_TIMERS
        for (int p = 0; p < NPHASE; ++p) st.ptime[p] = sm.ptime[p];
#endif
    }
    for (int i = tid; i < NSEG * (MAXLEV + 2); i += TS) (&st.seg[0][0])[i] = (&sm.seg[0][0])[i];
    __syncthreads();
}

// one instance for the launch's steps
template <typename T, int NF, int TS, bool WIDE, int SPM>
__device__ __forceinline__ void run_instance(TeamSmem<T> &sm, const Tables<T> &tab, BlockScratch<T, TS> &bx, const LaunchArgs &a, int tid,
                             uint32_t *masks) {
    Worker<T, NF, TS, WIDE, SPM> w(sm, tab, bx, tid, masks, a.wide);
    if (a.phases & PH_INIT_STATE) w.init_state((const unsigned char *)a.aux0, (const double *)a.aux1);
#pragma unroll 1
    for (int n = 0; n < a.nsteps; ++n) {
        if (a.phases & PH_ADAPT) w.adapt();
        if (a.phases & PH_STEP) w.lbm_step();
    }
}

// The bit arrays live in shared memory (smask, room for `cap` words) when the
// instance fits: the current tree is copied in at the start and back at the
// end; KEEP and REF are clear between two adaptations (but for the decisions
// that come with an initial state, ST_DETAILS), and every adaptation writes the
// other tree buffer.
template <typename T, int TS, bool WIDE, bool SCALAR, int SPM>
__device__ void run_team(TeamSmem<T> &sm, const Tables<T> &tab, BlockScratch<T, TS> &bx, const LaunchArgs &a,
                         const InstDesc &dg, int tid, uint32_t *smask, int cap) {
    load_instance<T, TS>(sm, dg, tid);
    const int W = sm.d.Wtot, OW = sm.d.OW;
    const long long region = smem_region_words(W, OW);
    const bool local = smask != nullptr && region <= cap;
    uint32_t *masks = local ? smask : sm.d.masks;
    const long long oo = (long long)(NMASK + 1) * W + (long long)sm.cur * OW;  // occupancy of the current tree
    if constexpr (SPM != 0) {
        // the other tree buffer starts empty: a step writes its new tree there in candidate words only
        uint32_t *other = masks + (long long)(sm.cur ^ 1) * W;
        for (int g = tid; g < W; g += TS) other[g] = 0u;
    }
    if (local) {
        const uint32_t *gi = sm.d.masks + (long long)sm.cur * W;
        uint32_t *li = smask + sm.cur * W;
        uint32_t *gk = sm.d.masks + (long long)M_KEEP * W, *gr = sm.d.masks + (long long)M_REF * W;
        const bool first = (sm.status & ST_DETAILS) != 0;  // the initial state's decisions, taken once
        for (int g = tid; g < W; g += TS) {
            li[g] = gi[g];
            smask[M_KEEP * W + g] = first ? gk[g] : 0u;
            smask[M_REF * W + g] = first ? gr[g] : 0u;
            if (first) gk[g] = gr[g] = 0u;
        }
        if constexpr (SPM != 0)
            for (int g = tid; g < OW; g += TS) smask[oo + g] = sm.d.masks[oo + g];
    }
    __syncthreads();
    if constexpr (SCALAR) {
        run_instance<T, 1, TS, WIDE, SPM>(sm, tab, bx, a, tid, masks);
    } else {
        // scheme variant: D1Q2^nf, or D1Q3 / D1Q5 shallow water (equilibria 4, 5)
        const int var = sm.d.eq == 4 ? 4 : sm.d.eq == 5 ? 5 : sm.d.nf;
        switch (var) {
        case 1: run_instance<T, 1, TS, WIDE, SPM>(sm, tab, bx, a, tid, masks); break;
        case 2: run_instance<T, 2, TS, WIDE, SPM>(sm, tab, bx, a, tid, masks); break;
        case 4: run_instance<T, 4, TS, WIDE, SPM>(sm, tab, bx, a, tid, masks); break;
        case 5: run_instance<T, 5, TS, WIDE, SPM>(sm, tab, bx, a, tid, masks); break;
        default: run_instance<T, 3, TS, WIDE, SPM>(sm, tab, bx, a, tid, masks); break;
        }
    }
    if (local) {
        uint32_t *gi = sm.d.masks + (long long)sm.cur * W;
        const uint32_t *li = smask + sm.cur * W;
        for (int g = tid; g < W; g += TS) gi[g] = li[g];
        if (a.phases & PH_INIT_STATE)  // clear there too, for a launch that keeps them there
            for (int g = tid; g < W; g += TS) {
                sm.d.masks[(long long)M_KEEP * W + g] = 0u;
                sm.d.masks[(long long)M_REF * W + g] = 0u;
            }
        const long long oc = (long long)(NMASK + 1) * W + (long long)sm.cur * OW;
        if constexpr (SPM != 0)
            for (int g = tid; g < OW; g += TS) sm.d.masks[oc + g] = smask[oc + g];
    }
    store_instance<T, TS>(sm, tid);
}

// Persistent kernel: each block takes instances from the queue (largest first)
// and advances one at a time with all its threads.  KIND selects the code the
// kernel holds: K_FAST every scheme with gamma = 1 and the leaves collision;
// K_LARGE the same schemes with the word passes over candidate words, for
// instances of at least CW_MIN_WORDS words per bitmask; K_GENERAL and K_RECOLL
// wide prediction stencils (gamma = 2, 3) and the reconstructed collision, at
// any size with the word passes over every word; K_SCALAR the gamma = 1 code
// of the scalar D1Q2 scheme alone, whose smaller register footprint lets more
// blocks share an SM (a larger MINB).
template <typename T, int NT, int MINB, int KIND>
__global__ void __launch_bounds__(NT, MINB) mr_persistent(LaunchArgs a) {
    constexpr bool WIDE = KIND == K_GENERAL || KIND == K_RECOLL;
    constexpr int SPM = KIND == K_LARGE ? 1 : 0;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BlockSmem<T, NT> &bs = *reinterpret_cast<BlockSmem<T, NT> *>(smem_raw);
    uint32_t *smask = a.smem_mask_words > 0
                          ? reinterpret_cast<uint32_t *>(smem_raw + ((sizeof(BlockSmem<T, NT>) + 15) / 16) * 16)
                          : nullptr;
    {
        const uint32_t *src = (const uint32_t *)a.tables;
        uint32_t *dst = (uint32_t *)&bs.tab;
        for (int i = threadIdx.x; i < (int)(sizeof(Tables<T>) / 4); i += NT) dst[i] = src[i];
    }
    for (;;) {
        if (threadIdx.x == 0) bs.idx = atomicAdd(a.queue, 1);
        __syncthreads();
        const int idx = bs.idx;
        __syncthreads();
        if (idx >= a.n) {
            // every block takes one number past the instances; the last leaves the
            // queue at zero for the next launch
            if (threadIdx.x == 0 && idx == a.n + (int)gridDim.x - 1) *a.queue = 0;
            return;
        }
        run_team<T, NT, WIDE, KIND == K_SCALAR, SPM>(bs.team, bs.tab, bs.scratch, a, a.descs[a.order[idx]], threadIdx.x, smask,
                                                a.smem_mask_words);
    }
}

}  // namespace mrg

// One translation unit per (precision, block size) instantiation keeps the
// build parallel; mr_dispatch.cu routes a launch to the right one.  MINB,
// MINB_S, MINB_G and MINB_R are the resident blocks per SM the fast, scalar,
// general and reconstructed-collision kernels are compiled for: the scalar
// code fits in fewer registers, the wide-stencil code runs faster with more
// registers and fewer resident blocks.
#define MRG_INSTANTIATE(T, NT, MINB, MINB_S, MINB_G, MINB_R, TAG)                                  \
    static size_t mrg_dyn_##TAG(int mask_words) {                                                 \
        size_t base = (sizeof(mrg::BlockSmem<T, NT>) + 15) / 16 * 16;                              \
        return base + (size_t)mask_words * sizeof(uint32_t);                                       \
    }                                                                                             \
    template <int M, int K>                                                                       \
    static int mrg_allow_##TAG() {                                                                \
        return (int)cudaFuncSetAttribute(mrg::mr_persistent<T, NT, M, K>,                         \
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024); \
    }                                                                                             \
    /* the attribute belongs to the current device: raised once per device ordinal */             \
    static int mrg_attr_##TAG() {                                                                 \
        static std::atomic<int> done[64];                                                         \
        int dev = 0;                                                                              \
        if (cudaGetDevice(&dev) != cudaSuccess) return (int)cudaErrorInvalidDevice;                \
        if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_acquire)) return 0;          \
        int rc = mrg_allow_##TAG<MINB, mrg::K_FAST>() | mrg_allow_##TAG<MINB_G, mrg::K_GENERAL>() | \
                 mrg_allow_##TAG<MINB_S, mrg::K_SCALAR>() | mrg_allow_##TAG<MINB_R, mrg::K_RECOLL>() | \
                 mrg_allow_##TAG<MINB, mrg::K_LARGE>();                                           \
        if (!rc && dev >= 0 && dev < 64) done[dev].store(1, std::memory_order_release);            \
        return rc;                                                                                \
    }                                                                                             \
    template <int M, int K>                                                                       \
    static int mrg_occ1_##TAG(size_t dyn, int *nb) {                                              \
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, mrg::mr_persistent<T, NT, M, K>, NT, dyn); \
    }                                                                                             \
    template <int M, int K>                                                                       \
    static int mrg_go_##TAG(int grid, const mrg::LaunchArgs &a, size_t dyn, cudaStream_t s, int prio) { \
        cudaLaunchConfig_t cfg = {};                                                              \
        cfg.gridDim = dim3((unsigned)grid);                                                       \
        cfg.blockDim = dim3(NT);                                                                  \
        cfg.dynamicSmemBytes = dyn;                                                               \
        cfg.stream = s;                                                                           \
        cudaLaunchAttribute at[1];                                                                \
        at[0].id = cudaLaunchAttributePriority;                                                   \
        at[0].val.priority = prio;                                                                \
        cfg.attrs = at;                                                                           \
        cfg.numAttrs = 1;                                                                         \
        return (int)cudaLaunchKernelEx(&cfg, mrg::mr_persistent<T, NT, M, K>, a);                 \
    }                                                                                             \
    int mrg_launch_##TAG(int grid, const mrg::LaunchArgs &a, cudaStream_t s, int prio) {           \
        int rc = mrg_attr_##TAG();                                                                \
        if (rc) return rc;                                                                        \
        const size_t dyn = mrg_dyn_##TAG(a.smem_mask_words);                                       \
        switch (a.kind) {                                                                         \
        case mrg::K_FAST: return mrg_go_##TAG<MINB, mrg::K_FAST>(grid, a, dyn, s, prio);           \
        case mrg::K_GENERAL: return mrg_go_##TAG<MINB_G, mrg::K_GENERAL>(grid, a, dyn, s, prio);   \
        case mrg::K_SCALAR: return mrg_go_##TAG<MINB_S, mrg::K_SCALAR>(grid, a, dyn, s, prio);     \
        case mrg::K_RECOLL: return mrg_go_##TAG<MINB_R, mrg::K_RECOLL>(grid, a, dyn, s, prio);     \
        case mrg::K_LARGE: return mrg_go_##TAG<MINB, mrg::K_LARGE>(grid, a, dyn, s, prio);         \
        }                                                                                         \
        return (int)cudaErrorInvalidValue;                                                        \
    }                                                                                             \
    int mrg_occ_##TAG(int kind, int mask_words, int *nb) {                                        \
        int rc = mrg_attr_##TAG();                                                                \
        if (rc) return rc;                                                                        \
        const size_t dyn = mrg_dyn_##TAG(mask_words);                                              \
        switch (kind) {                                                                           \
        case mrg::K_FAST: return mrg_occ1_##TAG<MINB, mrg::K_FAST>(dyn, nb);                       \
        case mrg::K_GENERAL: return mrg_occ1_##TAG<MINB_G, mrg::K_GENERAL>(dyn, nb);               \
        case mrg::K_SCALAR: return mrg_occ1_##TAG<MINB_S, mrg::K_SCALAR>(dyn, nb);                 \
        case mrg::K_RECOLL: return mrg_occ1_##TAG<MINB_R, mrg::K_RECOLL>(dyn, nb);                   \
        case mrg::K_LARGE: return mrg_occ1_##TAG<MINB, mrg::K_LARGE>(dyn, nb);                     \
        }                                                                                         \
        return (int)cudaErrorInvalidValue;                                                        \
    }                                                                                             \
    int mrg_minb_##TAG(int kind) {                                                                \
        return kind == mrg::K_SCALAR ? MINB_S : kind == mrg::K_GENERAL ? MINB_G                     \
             : kind == mrg::K_RECOLL ? MINB_R : MINB;                                             \
    }                                                                                             \
    size_t mrg_smem_##TAG(int mask_words) { return mrg_dyn_##TAG(mask_words); }
