// Plain FP64 evaluation of the per-cell arithmetic of one P-LBM step (Sec. II): every
// quantity is formed term by term in the order the equations write it, with one rounding
// per product and per sum (the FP64 kernels are compiled with -fmad=false), so that two
// correct FP64 evaluations of the step round identically.
//
//  - Eq. Density / Momentum: rho = sum_i f_i, rho u = sum_i f_i c_i + F/2, sums over the
//    velocities in the order of Eq. VelocitySet (D2Q9); D3Q19, which the paper does not
//    give, uses the storage order (rest, the six axis links, the twelve edge links).
//  - Eq. Interaction_Potential: psi = sqrt(2 (p_EOS - rho/3) / G).
//  - M1_a = sum_i w_i psi(x + c_i) c_ia / c_s^2, M2_ab = sum_i w_i psi(x + c_i)
//    (c_ia c_ib - c_s^2 d_ab) / c_s^4 (Sec. II), with 1/c_s^2 = 3 and 1/c_s^4 = 9 exact.
//  - Eq. Shan_Chen_Force and Eq. interactionForce (eps term read as in Eq.
//    New_Pressure_Tensor: -G/12 (2 kappa - 2 - 3 eps)).
//  - Eq. Single_Phase_EDF, Eq. Guo_Forcing_Scheme, Eq. LBE (BGK), and its moment-space
//    form f* = f - M^-1 S M (f - f^eq) + M^-1 (I - S/2) M Ft (MRT; bases of Lallemand & Luo
//    2000 for D2Q9 and d'Humieres et al. 2002 for D3Q19, every row of M evaluated, the
//    conserved rows relaxed with 1/tau like the stress rows).
// Zero terms (a zero velocity component or basis coefficient) are skipped: adding an exact
// zero to a sum that starts at +0 changes no bit.
//
// What bounds these kernels is the FP64 pipe (2 operations per clock and SM), so every operation that
// cannot change a bit is left out:
//  - a sum starts with its first term, not with 0 + term;
//  - a product that differs in sign only from one at hand (opposite velocities, signs of the basis and
//    of c) is that one, subtracted;
//  - a product with a power of two is exact, so product and sum are one fused multiply-add;
//  - a division by a number used often (tau, G, 3, the density span of tau(rho)) multiplies by its
//    reciprocal, held as a pair of doubles, and corrects the quotient by its exact remainder: four
//    operations for the correctly rounded quotient (Markstein 1990; quotient below).
// Microseconds a step: 96^3 D3Q19 MRT 2640 -> 2300, 301 x 203 D2Q9 BGK with tau(rho) 69 -> 59; the same
// bits.
#pragma once
#include "plb_device.cuh"

namespace plb {
namespace plain {

constexpr double CS2 = 1.0 / 3.0;   // c_s^2 (Eq. VelocitySet); 1/c_s^2 = 3, 1/c_s^4 = 9

// Storage slot of the n-th velocity in the summation order.
template <class L> struct Order;
template <> struct Order<D2Q9> {
    // Eq. VelocitySet: rest, (1,0), (0,1), (-1,0), (0,-1), (1,1), (-1,1), (-1,-1), (1,-1)
    __host__ __device__ static constexpr int slot(int n) {
        constexpr int t[9] = {0, 1, 3, 2, 4, 5, 8, 6, 7};
        return t[n];
    }
};
template <> struct Order<D3Q19> {
    __host__ __device__ static constexpr int slot(int n) { return n; }
};

template <class L> __host__ __device__ constexpr int cc(int n, int a) {
    return a == 0 ? L::cx(Order<L>::slot(n)) : (a == 1 ? L::cy(Order<L>::slot(n)) : L::cz(Order<L>::slot(n)));
}

// Shan-Chen weights omega(|c|^2) of Eq. Shan_Chen_Force (D3Q19: 3 w_i).
template <class L> __host__ __device__ constexpr double omega_sc(int n) {
    const int c2 = cc<L>(n, 0) * cc<L>(n, 0) + cc<L>(n, 1) * cc<L>(n, 1) + cc<L>(n, 2) * cc<L>(n, 2);
    if (c2 == 0) return 0.0;
    if (L::Q == 9) return c2 == 1 ? 1.0 / 3.0 : 1.0 / 12.0;
    return c2 == 1 ? 1.0 / 6.0 : 1.0 / 12.0;
}

// c_a c_b - c_s^2 d_ab.
template <class L> __host__ __device__ constexpr double cc2(int n, int a, int b) {
    return (double)(cc<L>(n, a) * cc<L>(n, b)) - (a == b ? CS2 : 0.0);
}

// Rows of the orthogonal moment bases, all Q of them, at velocity n of the summation order.
template <class L> __host__ __device__ constexpr double basis(int k, int n) {
    const double x = cc<L>(n, 0), y = cc<L>(n, 1), z = cc<L>(n, 2), c2 = x * x + y * y + z * z;
    if (L::Q == 9) {
        // rho, e, eps, jx, qx, jy, qy, pxx, pxy
        return k == 0 ? 1.0
             : k == 1 ? -4.0 + 3.0 * c2
             : k == 2 ? 4.0 - 10.5 * c2 + 4.5 * c2 * c2
             : k == 3 ? x
             : k == 4 ? (-5.0 + 3.0 * c2) * x
             : k == 5 ? y
             : k == 6 ? (-5.0 + 3.0 * c2) * y
             : k == 7 ? x * x - y * y
                      : x * y;
    }
    // rho, e, eps, jx, qx, jy, qy, jz, qz, 3pxx, 3pixx, pww, piww, pxy, pyz, pxz, mx, my, mz
    return k == 0 ? 1.0
         : k == 1 ? 19.0 * c2 - 30.0
         : k == 2 ? (21.0 * c2 * c2 - 53.0 * c2 + 24.0) / 2.0
         : k == 3 ? x
         : k == 4 ? (5.0 * c2 - 9.0) * x
         : k == 5 ? y
         : k == 6 ? (5.0 * c2 - 9.0) * y
         : k == 7 ? z
         : k == 8 ? (5.0 * c2 - 9.0) * z
         : k == 9 ? 3.0 * x * x - c2
         : k == 10 ? (3.0 * c2 - 5.0) * (3.0 * x * x - c2)
         : k == 11 ? y * y - z * z
         : k == 12 ? (3.0 * c2 - 5.0) * (y * y - z * z)
         : k == 13 ? x * y
         : k == 14 ? y * z
         : k == 15 ? x * z
         : k == 16 ? (y * y - z * z) * x
         : k == 17 ? (z * z - x * x) * y
                   : (x * x - y * y) * z;
}

template <class L> __host__ __device__ constexpr double basis_norm2(int k) {
    double s = 0.0;
    for (int n = 0; n < L::Q; ++n) s += basis<L>(k, n) * basis<L>(k, n);
    return s;
}

// Whether velocity n is the first with a non-zero entry in row k.
template <class L> __host__ __device__ constexpr bool first_entry(int k, int n) {
    for (int m = 0; m < n; ++m)
        if (basis<L>(k, m) != 0.0) return false;
    return true;
}

// Relaxation rate of row k: 0 = 1/tau (conserved and stress rows), else the Phys::s_rate kind.
template <class L> __host__ __device__ constexpr int rate_kind(int k) {
    if (L::Q == 9) return k == 1 ? 1 : k == 2 ? 2 : (k == 4 || k == 6) ? 3 : 0;
    return k == 1 ? 1 : k == 2 ? 2 : (k == 4 || k == 6 || k == 8) ? 3 : (k == 10 || k == 12) ? 4
         : (k >= 16) ? 5 : 0;
}

// Pressure of the EOS times p_scale: Peng & Robinson (1976) or Eq. EOS, as written.
__host__ __device__ inline double pressure(const PlainPhys &q, int eos_kind, double rho) {
    double pr;
    if (eos_kind == 0) {
        const double br = q.b * rho;
        pr = rho * q.R * q.T / (1.0 - br) - q.a_alpha * rho * rho / (1.0 + 2.0 * br - br * br);
    } else {
        const double sr = sqrt(rho);
        pr = q.P * (2.0 * rho * rho * rho + q.rv_2rl * rho * rho - q.sv3 * rho * rho * sr + q.sv2rl * rho * sr +
                    q.svrlrl * sr);
    }
    return q.p_scale * pr;
}

// The argument 2 (p - rho/3) / G of the square root of Eq. Interaction_Potential.
__host__ __device__ inline double psi_arg(const PlainPhys &q, int eos_kind, double rho) {
    return 2.0 * (pressure(q, eos_kind, rho) - rho / 3.0) / q.G;
}

// a / b, rounded to nearest.  rh + rl is 1 / b (rh the double nearest to it, rl the rest), so
// q = RN(a rh + RN(a rl)) misses a / b by less than half an ulp and 2^-50 ulp: it is one of the two doubles
// around a / b, its remainder a - q b is a double, and RN(q + remainder rh) is the nearest one
// (Markstein 1990, theorem on the final step).  For a outside 2^-900 .. 2^900 or b outside 2^-100 ..
// 2^100, where a remainder could be subnormal or a product overflow, the division itself.  (The tests
// are on the exponents, off the FP64 pipe.)
__device__ __forceinline__ double quotient(double a, double b, const Recip &r) {
    const unsigned hi = (unsigned)__double2hiint(a), er = ((unsigned)__double2hiint(r.h) >> 20) & 0x7ffu;
    const bool zero = (hi << 1 | (unsigned)__double2loint(a)) == 0u;
    if (((hi >> 20 & 0x7ffu) - 123u >= 1800u && !zero) || er - 923u >= 200u) return a / b;
    const double q = __fma_rn(a, r.h, __dmul_rn(a, r.l));
    const double v = __fma_rn(__fma_rn(-b, q, a), r.h, q);
    // (a zero dividend: the sums above can lose the sign of the quotient)
    return zero ? __hiloint2double((int)((hi ^ (unsigned)__double2hiint(b)) & 0x80000000u), 0) : v;
}

// 1 / b as a pair of doubles.
__host__ __device__ inline Recip reciprocal(double b) {
    Recip r;
    r.h = 1.0 / b;
    r.l = fma(-b, r.h, 1.0) * r.h;
    return r;
}

// rho of Eq. Density.
template <class L> __device__ __forceinline__ double density(const double *f) {
    double r = f[Order<L>::slot(0)];
    Unroll<1, L::Q>::run([&](auto nc) { r = r + f[Order<L>::slot(decltype(nc)::value)]; });
    return r;
}

// psi of Eq. Interaction_Potential; raises the device flags on a domain error.
__device__ __forceinline__ double psi(const KParams &p, double rho) {
    if (!(rho > 0.0) || !(rho < INFINITY)) {
        atomicOr(p.flags, FLAG_NONFINITE);
        return 0.0;
    }
    // psi_arg, its divisions by 3 and by G through their reciprocals
    constexpr double third = 1.0 / 3.0;
    const Recip r3 = {third, 0x1.5555555555555p-56};
    const double arg = quotient(2.0 * (pressure(p.pl, p.eos_kind, rho) - quotient(rho, 3.0, r3)), p.pl.G, p.pl.inv_G);
    if (!(arg >= 0.0)) {
        atomicOr(p.flags, FLAG_PSI_DOMAIN);
        return 0.0;
    }
    return sqrt(arg);
}

// Whether velocity n is the first of the summation order with a non-zero c_a (c_a c_b).
template <class L> __host__ __device__ constexpr bool first_of(int n, int a, int b) {
    for (int m = 0; m < n; ++m)
        if (cc<L>(m, a) * cc<L>(m, b) != 0) return false;
    return true;
}

// sum = sum +- term; the first term of a sum starts it.
template <bool FIRST, bool PLUS> __device__ __forceinline__ void add_term(double &sum, double term) {
    if (FIRST) sum = PLUS ? term : -term;
    else sum = PLUS ? sum + term : sum - term;
}

// Total force density at a cell (Eqs. Shan_Chen_Force, interactionForce, plus the body
// force) from a psi field of row pitch sy and plane pitch sz; pc points at the cell's psi.
template <class L, class Pol>
__device__ __forceinline__ void force(const KParams &p, const double *__restrict__ pc, int sy, int sz, double F[3]) {
    constexpr int D = L::D;
    const PlainPhys &q = p.pl;
    double M1[3], sc[3], M2[3][3];
    Unroll<0, L::Q>::run([&](auto nc) {
        constexpr int n = decltype(nc)::value;
        const double pn = Pol::ro(pc + (cc<L>(n, 0) + cc<L>(n, 1) * sy + cc<L>(n, 2) * sz));
        const double wp = L::w(Order<L>::slot(n)) * pn;
        const double w3 = wp * 3.0, w9 = wp * 9.0, os = omega_sc<L>(n) * pn;
        const double full = wp * (1.0 - CS2) * 9.0, part = wp * (0.0 - CS2) * 9.0;   // a = b, c_a != 0 or = 0
        Unroll<0, D>::run([&](auto ac) {
            constexpr int a = decltype(ac)::value, ca = cc<L>(n, a);
            if constexpr (ca != 0) {
                add_term<first_of<L>(n, a, a), (ca > 0)>(M1[a], w3);
                add_term<first_of<L>(n, a, a), (ca > 0)>(sc[a], os);
            }
            add_term<n == 0, true>(M2[a][a], ca != 0 ? full : part);
            Unroll<a + 1, D>::run([&](auto bc) {
                constexpr int b = decltype(bc)::value, cab = ca * cc<L>(n, b);
                if constexpr (cab != 0) add_term<first_of<L>(n, a, b), (cab > 0)>(M2[a][b], w9);
            });
        });
    });
    const double psi0 = Pol::ro(pc);
    double trM2 = M2[0][0];
#pragma unroll
    for (int b = 1; b < D; ++b) trM2 = trM2 + M2[b][b];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a >= D) {
            F[a] = 0.0;
            continue;
        }
        const double Fsc = -q.G * psi0 * sc[a];
        double M1M2 = M1[0] * M2[0][a];
#pragma unroll
        for (int b = 1; b < D; ++b) M1M2 = M1M2 + M1[b] * (a <= b ? M2[a][b] : M2[b][a]);
        const double Fint = Fsc - q.K1 * M1M2 + q.K2 * M1[a] * trM2;
        F[a] = Fint + q.fext[a];
    }
}

// Component a of the velocity of storage slot i.
template <class L> __host__ __device__ constexpr int cs(int i, int a) {
    return a == 0 ? L::cx(i) : (a == 1 ? L::cy(i) : L::cz(i));
}

// The products (c_a c_b - c_s^2 d_ab) x_a y_b that the quadratic terms sum: a = b with c_a != 0 (full)
// and c_a = 0 (part), and a != b up to sign (off).
template <class L> struct Products {
    double full[3], part[3], off[3][3];
    __device__ __forceinline__ Products(const double *x, const double *y) {
#pragma unroll
        for (int a = 0; a < L::D; ++a) {
            full[a] = (1.0 - CS2) * x[a] * y[a];
            part[a] = (0.0 - CS2) * x[a] * y[a];
#pragma unroll
            for (int b = 0; b < L::D; ++b)
                if (a != b) off[a][b] = x[a] * y[b];
        }
    }
    // their sum for the velocity of storage slot I (the same for -c)
    template <int I> __device__ __forceinline__ double sum() const {
        double s;
        Unroll<0, L::D>::run([&](auto ac) {
            constexpr int a = decltype(ac)::value;
            Unroll<0, L::D>::run([&](auto bc) {
                constexpr int b = decltype(bc)::value, cab = cs<L>(I, a) * cs<L>(I, b);
                if constexpr (a == b) add_term<a == 0, true>(s, cab != 0 ? full[a] : part[a]);
                else if constexpr (cab != 0) add_term<false, (cab > 0)>(s, off[a][b]);
            });
        });
        return s;
    }
};

// c . x for the velocity of storage slot I.
template <class L, int I> __device__ __forceinline__ double along(const double *x) {
    double s = 0.0;
    Unroll<0, L::D>::run([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        constexpr bool one = (a == 0 || cs<L>(I, 0) == 0) && (a <= 1 || cs<L>(I, 1) == 0);
        if constexpr (cs<L>(I, a) != 0) add_term<one, (cs<L>(I, a) > 0)>(s, x[a]);
    });
    return s;
}

// f^eq of Eq. Single_Phase_EDF into storage slots; opposite velocities (slots i, i + 1) share their terms.
template <class L> __device__ __forceinline__ void equilibrium(double rho, const double u[3], double *fe) {
    const Products<L> uu(u, u);
    fe[0] = L::w(0) * rho * (1.0 + uu.template sum<0>() * 4.5);
    Unroll<0, (L::Q - 1) / 2>::run([&](auto rc) {
        constexpr int i = 2 * decltype(rc)::value + 1;
        const double cu = along<L, i>(u) * 3.0, quad = uu.template sum<i>() * 4.5, wr = L::w(i) * rho;
        fe[i] = wr * (1.0 + cu + quad);
        fe[i + 1] = wr * (1.0 - cu + quad);
    });
}

// The bracket of Eq. Guo_Forcing_Scheme (without 1 - 1/(2 tau)) into storage slots.
template <class L> __device__ __forceinline__ void guo(const double F[3], const double u[3], double *Ft) {
    const Products<L> Fu(F, u);
    Ft[0] = L::w(0) * (Fu.template sum<0>() * 9.0);
    Unroll<0, (L::Q - 1) / 2>::run([&](auto rc) {
        constexpr int i = 2 * decltype(rc)::value + 1;
        const double cF = along<L, i>(F) * 3.0, quad = Fu.template sum<i>() * 9.0;
        Ft[i] = L::w(i) * (cF + quad);
        Ft[i + 1] = L::w(i) * (quad - cF);
    });
}

// Whether |v| is a power of two (basis entries: 1, 2, 4, 8 among others).
__host__ __device__ constexpr bool is_pow2(double v) {
    v = v < 0 ? -v : v;
    return v == 1.0 || v == 2.0 || v == 4.0 || v == 8.0;
}

// sum + m x for a basis entry m, rounded after the product and after the sum.
template <bool FIRST> __device__ __forceinline__ double project(double m, double x, double sum) {
    if (FIRST) return m * x;
    return is_pow2(m) ? __fma_rn(m, x, sum) : sum + m * x;
}

// In place: pre-collision populations f (storage slots) -> post-collision populations.
template <class L, int MRT> __device__ __forceinline__ void collide(const KParams &p, double *f, const double F[3]) {
    constexpr int Q = L::Q, D = L::D;
    const PlainPhys &q = p.pl;
    const double rho = density<L>(f);
    double u[3] = {0.0, 0.0, 0.0};
    Unroll<0, D>::run([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        double m;
        Unroll<0, Q>::run([&](auto nc) {
            constexpr int n = decltype(nc)::value;
            if constexpr (cc<L>(n, a) != 0) add_term<first_of<L>(n, a, a), (cc<L>(n, a) > 0)>(m, f[Order<L>::slot(n)]);
        });
        u[a] = (m + F[a] / 2.0) / rho;
    });
    double tau = q.tau_l;
    Recip itau = q.inv_tau;
    if (p.var_tau) {
        double wgt = quotient(rho - q.tau_rho_v, q.d_rho, q.inv_d_rho);
        if (wgt < 0.0) wgt = 0.0;
        if (wgt > 1.0) wgt = 1.0;
        tau = q.tau_v + wgt * q.d_tau;
        itau = reciprocal(tau);
    }
    double fneq[Q], Ft[Q];
    equilibrium<L>(rho, u, fneq);
    guo<L>(F, u, Ft);
#pragma unroll
    for (int i = 0; i < Q; ++i) fneq[i] = f[i] - fneq[i];
    if constexpr (!MRT) {
        const double kg = 1.0 - 0.5 * itau.h;                    // 1 / (2 tau) is half of 1 / tau
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = f[i] - quotient(fneq[i], tau, itau) + kg * Ft[i];
    } else {
        // row by row: moments of f - f^eq and of the bracket, and their part of M^-1
        double corr[Q];
        Unroll<0, Q>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            double mneq = 0.0, mf = 0.0;
            Unroll<0, Q>::run([&](auto nc) {
                constexpr int n = decltype(nc)::value;
                constexpr double m = basis<L>(k, n);
                if constexpr (m != 0.0) {
                    constexpr bool one = first_entry<L>(k, n);
                    mneq = project<one>(m, fneq[Order<L>::slot(n)], mneq);
                    mf = project<one>(m, Ft[Order<L>::slot(n)], mf);
                }
            });
            constexpr int kind = rate_kind<L>(k);
            const double s = kind == 0 ? itau.h : q.s_rate[kind];
            const double half = kind == 0 ? 1.0 - itau.h / 2.0 : q.s_half[kind];
            const double dm = s * mneq;
            const double mF = half * mf;
            const double dmf = mF - dm;
            Unroll<0, Q>::run([&](auto nc) {
                constexpr int n = decltype(nc)::value;
                constexpr double mi = basis<L>(k, n) / basis_norm2<L>(k);
                if constexpr (mi != 0.0) add_term<k == 0, (mi > 0.0)>(corr[n], (mi > 0.0 ? mi : -mi) * dmf);
            });
        });
        Unroll<0, Q>::run([&](auto nc) {
            constexpr int n = decltype(nc)::value;
            f[Order<L>::slot(n)] = f[Order<L>::slot(n)] + corr[n];
        });
    }
}

}  // namespace plain
}  // namespace plb
