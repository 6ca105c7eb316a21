// Stillinger-Weber terms of one edge and one shell, in plain FP64 or in dual numbers v + eps d
// (a value with its derivative along one direction).  Shared by the FP64 force kernels and by the
// adjoint's dual-number kernel.
//
// FP64 runs at 2 lanes a cycle and SM here, so these kernels cost what they issue in FP64: every
// fused multiply-add is written out (fma_), divisions are replaced by one reciprocal square root
// and one reciprocal an edge, the derivatives of r and of the unit vector are taken in closed
// form, and the triplets of an atom go through the moments of its shell (O(m), not O(m^2)).
// Real parts are the same operations in both number types, whatever the compiler's contraction
// mode, so a dual run repeats the plain run's values bit for bit.
#pragma once
#include <cuda_runtime.h>

#include "nefe.h"

namespace nefe {

struct Dd {
    double v, d;
};
__host__ __device__ __forceinline__ Dd mk(double v, double d) { Dd r; r.v = v; r.d = d; return r; }
__host__ __device__ __forceinline__ double val(double a) { return a; }
__host__ __device__ __forceinline__ double val(Dd a) { return a.v; }
__host__ __device__ __forceinline__ double dua(double) { return 0.0; }
__host__ __device__ __forceinline__ double dua(Dd a) { return a.d; }
template <typename A> struct is_dual { static constexpr bool value = false; };
template <> struct is_dual<Dd> { static constexpr bool value = true; };
template <typename A, typename B> struct sum_type { using t = Dd; };
template <> struct sum_type<double, double> { using t = double; };
template <typename A, typename B, typename C>
using sum3 = typename sum_type<typename sum_type<A, B>::t, C>::t;

__device__ __forceinline__ Dd operator+(Dd a, Dd b) { return mk(__dadd_rn(a.v, b.v), __dadd_rn(a.d, b.d)); }
__device__ __forceinline__ Dd operator-(Dd a) { return mk(-a.v, -a.d); }
__device__ __forceinline__ Dd operator-(Dd a, Dd b) { return mk(__dsub_rn(a.v, b.v), __dsub_rn(a.d, b.d)); }

// a b and a b + c, each real part one rounded operation.
template <typename A, typename B>
__device__ __forceinline__ typename sum_type<A, B>::t mul_(A a, B b) {
    if constexpr (!is_dual<A>::value && !is_dual<B>::value) return __dmul_rn(a, b);
    else if constexpr (!is_dual<A>::value) return mk(__dmul_rn(a, b.v), __dmul_rn(a, b.d));
    else if constexpr (!is_dual<B>::value) return mk(__dmul_rn(a.v, b), __dmul_rn(a.d, b));
    else return mk(__dmul_rn(a.v, b.v), __fma_rn(a.v, b.d, __dmul_rn(a.d, b.v)));
}
template <typename A, typename B, typename C>
__device__ __forceinline__ sum3<A, B, C> fma_(A a, B b, C c) {
    if constexpr (!is_dual<A>::value && !is_dual<B>::value && !is_dual<C>::value) {
        return __fma_rn(a, b, c);
    } else {
        const double v = __fma_rn(val(a), val(b), val(c));
        double d;
        if constexpr (is_dual<C>::value) {
            d = dua(c);
            if constexpr (is_dual<B>::value) d = __fma_rn(val(a), dua(b), d);
            if constexpr (is_dual<A>::value) d = __fma_rn(dua(a), val(b), d);
        } else {
            if constexpr (is_dual<B>::value) {
                d = __dmul_rn(val(a), dua(b));
                if constexpr (is_dual<A>::value) d = __fma_rn(dua(a), val(b), d);
            } else {
                d = __dmul_rn(dua(a), val(b));
            }
        }
        return mk(v, d);
    }
}

// SW parameters; TP = Dd: the differentiable ones carry the parameter direction.
template <typename TP>
struct SWp {
    double eps, sig, inv_sig, c0, rc2;
    TP A, B, p, q, a, lam, gam;
    int int_pq;         // p == 4 and q == 0: s^-p and s^-q by multiplications
    int want_log;       // ln s is needed (general exponents, or a direction in p or q)
};

template <typename T>
struct EdgeT {
    T ux, uy, uz;       // unit vector
    T ir, id, g;        // 1/r, 1/(r/sigma - a), exp(gamma id)
    T phi, dphi;        // pair term, dphi/dr
    double r;           // length (real part)
    T pg[5];            // d phi / d(A, B, p, q, a) (GRAD)
};

// Edge terms for the vector d (w: its derivative, T = Dd).  False (and every term 0) at or beyond
// the cutoff, within 1e-12 sigma.
template <typename T, typename TP, bool GRAD>
__device__ __forceinline__ bool sw_edge_terms(const SWp<TP>& P, const double (&d)[3], const double (&w)[3], EdgeT<T>& e) {
    const double r2 = __fma_rn(d[2], d[2], __fma_rn(d[1], d[1], __dmul_rn(d[0], d[0])));
    const double ir = rsqrt(r2);
    const double r = __dmul_rn(r2, ir);
    e.r = r;
    const double den = __fma_rn(r, P.inv_sig, -val(P.a));
    const bool in = r2 < P.rc2 && !(den >= -1e-12);   // (coincident atoms give NaN and stay in)
    const double id = 1.0 / (in ? den : -1.0);
    const double u[3] = {in ? __dmul_rn(d[0], ir) : 0.0, in ? __dmul_rn(d[1], ir) : 0.0, in ? __dmul_rn(d[2], ir) : 0.0};
    const double e1v = in ? exp(id) : 0.0, gv = in ? exp(__dmul_rn(val(P.gam), id)) : 0.0;
    T e1, is, rp, rq, ls;
    const double isv = __dmul_rn(ir, P.sig);
    double rpv, rqv, lsv = 0.0;
    if (P.want_log || GRAD) lsv = -log(isv);
    if (P.int_pq) {
        const double is2 = __dmul_rn(isv, isv);
        rpv = __dmul_rn(is2, is2);
        rqv = 1.0;
    } else {
        rpv = exp(-__dmul_rn(val(P.p), lsv));
        rqv = exp(-__dmul_rn(val(P.q), lsv));
    }
    if constexpr (is_dual<T>::value) {
        const double rd = __fma_rn(u[2], w[2], __fma_rn(u[1], w[1], __dmul_rn(u[0], w[0])));   // r'
        e.ux = mk(u[0], __dmul_rn(__fma_rn(-u[0], rd, w[0]), ir));
        e.uy = mk(u[1], __dmul_rn(__fma_rn(-u[1], rd, w[1]), ir));
        e.uz = mk(u[2], __dmul_rn(__fma_rn(-u[2], rd, w[2]), ir));
        const double sl = __dmul_rn(rd, ir);                     // s'/s = (ln s)'
        e.ir = mk(ir, -__dmul_rn(ir, sl));
        double dend = __dmul_rn(rd, P.inv_sig);
        if constexpr (is_dual<TP>::value) dend = __dsub_rn(dend, dua(P.a));
        const double idd = -__dmul_rn(__dmul_rn(id, id), dend);
        e.id = mk(id, idd);
        e1 = mk(e1v, __dmul_rn(e1v, idd));
        double gl = __dmul_rn(val(P.gam), idd);
        if constexpr (is_dual<TP>::value) gl = __fma_rn(dua(P.gam), id, gl);
        e.g = mk(gv, __dmul_rn(gv, gl));
        is = mk(isv, -__dmul_rn(isv, sl));
        ls = mk(lsv, sl);
        double pl = -__dmul_rn(val(P.p), sl), ql = -__dmul_rn(val(P.q), sl);
        if constexpr (is_dual<TP>::value) {
            pl = __fma_rn(-dua(P.p), lsv, pl);
            ql = __fma_rn(-dua(P.q), lsv, ql);
        }
        rp = mk(rpv, __dmul_rn(rpv, pl));
        rq = mk(rqv, __dmul_rn(rqv, ql));
    } else {
        e.ux = u[0]; e.uy = u[1]; e.uz = u[2];
        e.ir = ir; e.id = id; e.g = gv;
        e1 = e1v; is = isv; ls = lsv; rp = rpv; rq = rqv;
    }
    // phi = eps A (B s^-p - s^-q) e1
    const T Ee = mul_(P.eps, e1);
    const T ea = mul_(P.A, Ee);
    const T Brp = mul_(P.B, rp);
    const T br = Brp - rq;
    const T id2 = mul_(e.id, e.id);
    e.phi = mul_(ea, br);
    const T k = fma_(P.q, rq, -mul_(P.p, Brp));
    e.dphi = mul_(fma_(mul_(ea, k), is, -mul_(e.phi, id2)), P.inv_sig);
    if constexpr (GRAD) {
        e.pg[0] = mul_(Ee, br);
        e.pg[1] = mul_(ea, rp);
        e.pg[2] = -mul_(mul_(ea, Brp), ls);
        e.pg[3] = mul_(mul_(ea, rq), ls);
        e.pg[4] = mul_(e.phi, id2);
    }
    return in;
}

// Moments of a shell: G = sum g, m1 = sum g u, M = sum g u u^T.
template <typename T>
struct MomT {
    T G, x, y, z, xx, yy, zz, xy, xz, yz;
};
template <typename T>
__device__ __forceinline__ void mom_add(MomT<T>& M, T ux, T uy, T uz, T g) {
    const T gx = mul_(g, ux), gy = mul_(g, uy), gz = mul_(g, uz);
    M.G = M.G + g; M.x = M.x + gx; M.y = M.y + gy; M.z = M.z + gz;
    M.xx = fma_(gx, ux, M.xx); M.yy = fma_(gy, uy, M.yy); M.zz = fma_(gz, uz, M.zz);
    M.xy = fma_(gx, uy, M.xy); M.xz = fma_(gx, uz, M.xz); M.yz = fma_(gy, uz, M.yz);
}

// Force that an atom's terms exert on the leg atom of edge a: the triplets (i; a, b) over every
// partner b != a, and half of the pair force (the other half comes from the same edge seen from
// its far end).  The atom itself receives minus the sum of these.  With c_b = u_a.u_b, the sums
// over b are the moments' less the b = a term (c = 1):
//   S1 = sum g_b (c_b - c0) u_b = M u - c0 m1 - g (1 - c0) u,
//   S2 = sum g_b (c_b - c0) c_b = u.M u - c0 u.m1 - g (1 - c0),
//   S3 = sum g_b (c_b - c0)^2   = u.M u - 2 c0 u.m1 + c0^2 G - g (1 - c0)^2,
// and the leg force is (k1 S2 - k2 S3 - dphi/2) u - k1 S1 with k1 = 2 eps lambda g / r and
// k2 = eps lambda dg/dr = -eps lambda g gamma id^2 / sigma.  s3 returns S3.
template <typename T, typename TP>
__device__ __forceinline__ void sw_leg(const SWp<TP>& P, const MomT<T>& M, T ux, T uy, T uz, T ir, T id, T g, T dphi,
                                       T& lx, T& ly, T& lz, T& s3) {
    const double c0 = P.c0, mc0 = -c0, c1 = 1.0 - c0;
    const T Mux = fma_(M.xx, ux, fma_(M.xy, uy, mul_(M.xz, uz)));
    const T Muy = fma_(M.xy, ux, fma_(M.yy, uy, mul_(M.yz, uz)));
    const T Muz = fma_(M.xz, ux, fma_(M.yz, uy, mul_(M.zz, uz)));
    const T q = fma_(ux, Mux, fma_(uy, Muy, mul_(uz, Muz)));
    const T pm = fma_(ux, M.x, fma_(uy, M.y, mul_(uz, M.z)));
    const T self = mul_(c1, g);
    const T t = fma_(mc0, pm, q);                               // u.M u - c0 u.m1
    const T s2 = t - self;
    s3 = fma_(mc0, fma_(mc0, M.G, pm), t) - mul_(c1, self);
    const T eg = mul_(mul_(P.eps, P.lam), g);
    const T k1 = mul_(mul_(2.0, eg), ir);
    const T mk2 = mul_(mul_(mul_(eg, P.gam), mul_(id, id)), P.inv_sig);   // -k2
    const T cc = fma_(k1, s2, fma_(mk2, s3, mul_(-0.5, dphi)));
    lx = fma_(cc, ux, -mul_(k1, fma_(mc0, M.x, fma_(-self, ux, Mux))));
    ly = fma_(cc, uy, -mul_(k1, fma_(mc0, M.y, fma_(-self, uy, Muy))));
    lz = fma_(cc, uz, -mul_(k1, fma_(mc0, M.z, fma_(-self, uz, Muz))));
}

inline SWp<double> sw_params_real(const nefe_sw_params& p) {
    SWp<double> c;
    c.eps = p.eps; c.sig = p.sigma; c.inv_sig = 1.0 / p.sigma; c.c0 = p.cos0;
    const double rc = p.a * p.sigma;
    c.rc2 = rc * rc;
    c.A = p.A; c.B = p.B; c.p = p.p; c.q = p.q; c.a = p.a; c.lam = p.lambda3; c.gam = p.gamma;
    c.int_pq = (p.p == 4.0 && p.q == 0.0) ? 1 : 0;
    c.want_log = c.int_pq ? 0 : 1;
    return c;
}
inline SWp<Dd> sw_params_dual(const nefe_sw_params& p, const double* d) {
    const SWp<double> r = sw_params_real(p);
    SWp<Dd> c;
    c.eps = r.eps; c.sig = r.sig; c.inv_sig = r.inv_sig; c.c0 = r.c0; c.rc2 = r.rc2; c.int_pq = r.int_pq;
    c.A = mk(r.A, d[0]); c.B = mk(r.B, d[1]); c.p = mk(r.p, d[2]); c.q = mk(r.q, d[3]);
    c.a = mk(r.a, d[4]); c.lam = mk(r.lam, d[5]); c.gam = mk(r.gam, d[6]);
    c.want_log = (r.want_log || d[2] != 0.0 || d[3] != 0.0) ? 1 : 0;
    return c;
}

// ------------------------------------------------------------------------------------
// Fractional positions x/L as 32-bit fixed point: the difference of two wraps to the nearest
// image by itself, with a resolution of L 2^-32.  x (1/L) is added to 1.5 2^20, whose unit in the
// last place is 2^-32: the sum's low word is the fraction.  Beyond 2^19 boxes (or not finite) the
// remainder is taken first.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ int wrap_sub(int a, int b) { return (int)((unsigned)a - (unsigned)b); }
__device__ __forceinline__ int wrap_add(int a, int b) { return (int)((unsigned)a + (unsigned)b); }
__device__ __forceinline__ int frac32(double x, double inv_L) {
    const double magic = 1572864.0;              // 1.5 2^20
    double s = __fma_rn(x, inv_L, magic);
    if ((__double_as_longlong(s) >> 52) != (__double_as_longlong(magic) >> 52)) {
        const double t = __dmul_rn(x, inv_L);
        s = __dadd_rn(t - floor(t), magic);
    }
    return (int)(unsigned)(unsigned long long)__double_as_longlong(s);
}
// The same with kFracLow more bits (the fraction times 2^42, by the unit of 1.5 2^10), modulo 2^42.
constexpr int kFracLow = 10;
__device__ __forceinline__ long long frac42(double x, double inv_L) {
    const double magic = 1536.0;                 // 1.5 2^10
    double s = __fma_rn(x, inv_L, magic);
    if ((__double_as_longlong(s) >> 52) != (__double_as_longlong(magic) >> 52)) {
        const double t = __dmul_rn(x, inv_L);
        s = __dadd_rn(t - floor(t), magic);
    }
    return __double_as_longlong(s) & ((1LL << (32 + kFracLow)) - 1);
}

}  // namespace nefe
