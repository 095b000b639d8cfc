// cell_ops.cuh -- per-cell device arithmetic shared by the single-domain
// kernels and the batched-ensemble kernel: closures (Eq. 2-4, Eq. A6), grid
// neighbours and the two stencil forms of the Picard operator.
#pragma once

#include <math.h>

#include "f64m.cuh"
#include "ix64.cuh"
#include "rf_internal.cuh"

namespace rf {

// van Genuchten / Mualem closures (Eq. 2-4), evaluated in double-float
// arithmetic (ff.cuh) with FP64 only at the input and the outputs.
// With u = -alpha h, L = log u, x = u^n = exp(n L), l1 = log(1 + x):
//   Se = (1 + x)^-m = exp(-m l1)                               (Eq. 2)
//   u^(n-1) = x / u (since m n = n - 1), so (x/(1+x))^m = (x/u) Se = ys
//   Se^(1/m) = 1/(1+x) = w, so 1 - Se^(1/m) = x/(1+x) and
//   K = Ks Se^(1/2) (1 - ys)^2                                   (Eq. 4)
//     with 1 - ys = -expm1(m log(1 - w)) when ys > 1/2 (dry soil, where
//     1 - ys would cancel)
//   C = (theta_s-theta_r) alpha n m u^(n-1) (1+x)^-(m+1)
//     = (theta_s-theta_r) alpha n m ys w                         (Eq. 3)
// (h < 0 only; closure() below handles h >= 0 and the other models.)
__device__ __forceinline__ void closure_vg_df(const DevSoil &s, double Ks, double h, const FFTables *__restrict__ tab,
                                              double &th, double &K, double &C)
{
    const double dth = s.theta_s - s.theta_r;
    const double ud = -s.alpha * h;
    if (ud < 1e-30) {                     // (-alpha h)^n underflows: the wet limit
        th = s.theta_s;
        K = Ks;
        C = 0.0;
        return;
    }
    const ff u = ff_from_d(ud);
    const ff L = ff_log(u, tab);
    const ff nL = ff_mul(ff_make(s.n_hi, s.n_lo), L);
    if (nL.hi > 80.0f) {                  // x > e^80: Se = x^-m, K and C vanish at double range
        th = s.theta_r + dth * ff_to_d(ff_exp(ff_neg(ff_mul(ff_make(s.m_hi, s.m_lo), nL)), tab));
        K = 0.0;
        C = 0.0;
        return;
    }
    const ff x = ff_exp(nL, tab);
    const ff onepx = ff_add_f(x, 1.0f);
    const ff l1 = ff_log(onepx, tab);
    const ff mm = ff_make(s.m_hi, s.m_lo);
    const ff se = ff_exp(ff_neg(ff_mul(mm, l1)), tab);
    const ff w = ff_div(ff_make(1.0f, 0.0f), onepx);
    const ff ys = ff_mul(ff_div(x, u), se);
    ff omy;
    if (ys.hi <= 0.5f) {
        omy = ff_add_f(ff_neg(ys), 1.0f);
    } else {
        const ff lg = (w.hi < 0.0078125f) ? ff_log1p_small(ff_neg(w)) : ff_log(ff_add_f(ff_neg(w), 1.0f), tab);
        const ff z = ff_mul(mm, lg);
        omy = (z.hi > -0.0078125f) ? ff_neg(ff_expm1_small(z)) : ff_add_f(ff_neg(ff_exp(z, tab)), 1.0f);
    }
    th = s.theta_r + dth * ff_to_d(se);
    K = Ks * ff_to_d(ff_mul(ff_sqrt(se), ff_mul(omy, omy)));
    C = s.cfac * ff_to_d(ff_mul(ys, w));
}

// The same van Genuchten / Mualem closures (h < 0) in FP64, for the states
// outside the fixed-point form's range (fx64.cuh), with the
// table-driven exp / log of f64m.cuh: with u = -alpha h, L = log u (as a
// double-double), x = exp(n L), l1 = log1p(x) (double-double):
//   Se = exp(-m l1), w = 1/(1+x), ys = (x/(1+x))^m = (x/u) Se,
//   K = Ks sqrt(Se) (1 - ys)^2 with 1 - ys = -expm1(m log1p(-w)) when
//   ys > 1/2, C = (theta_s-theta_r) alpha n m ys w;
// sqrt(Se) = exp(-m l1 / 2) and Se its square (f64_exp_sqr), 1/u and w
// from the one reciprocal 1/(u (1 + x)), since each divide, square root
// and exponential costs GB300's narrow FP64 pipe a dozen instructions.
// n L and m l1 are formed with their rounding errors (two-product), so x and
// Se keep a few units in the last place however large |L| or l1 are.
// Beyond x = e^700 (a suction far outside any soil state) theta = theta_r +
// dtheta x^-m and K = C = 0; below u = 1e-30 (h within 1e-30/alpha of 0) ys
// is taken as exp(m (n L - l1)), the quotient x/u being out of range.
__device__ __forceinline__ void closure_vg_fp64(const DevSoil &s, double Ks, double h,
                                                const FFTables *__restrict__ tab, double &th, double &K, double &C)
{
    const double dth = s.theta_s - s.theta_r;
    const double u = -s.alpha * h;
    double Lh, Ll;
    f64_log_dd(u, tab, Lh, Ll);
    const double nh = s.n * Lh;
    const double nl = fma(s.n, Lh, -nh) + s.n * Ll;
    if (nh > 700.0) {
        th = s.theta_r + dth * f64_exp_nc(fmax(-s.m * nh, -700.0), tab);
        K = 0.0;
        C = 0.0;
        return;
    }
    // x = u^n; below e^-700 it is 0 to double precision beside 1 (Se = 1)
    const double x = nh >= -700.0 ? f64_exp_dd(nh, nl, tab) : 0.0;
    const double onepx = 1.0 + x;
    // one reciprocal serves w = 1/(1 + x) and 1/u (separate ones where the
    // product would overflow)
    const double uo = u * onepx;
    double w, iu;
    if (uo < 1e300) {
        const double q = rcp64(uo);
        w = q * u;
        iu = q * onepx;
    } else {
        w = rcp64(onepx);
        iu = rcp64(u);
    }
    double l1h, l1l;
    if (x >= 0.0078125) f64_log1p_big_dd(x, onepx, w, tab, l1h, l1l);
    else f64_log1p_dd(x, tab, l1h, l1l);
    // Se^(1/2) = exp(-m l1 / 2), with Se = (Se^(1/2))^2 from the same
    // exponential (K needs the root, theta and C need Se)
    const double hm = 0.5 * s.m;
    const double sh = -hm * l1h;                   // in [-350, 0]
    double s2, se;
    f64_exp_sqr(sh, fma(-hm, l1h, -sh) - hm * l1l, tab, s2, se);
    const double ys = u >= 1e-30 ? (x * iu) * se : f64_exp(s.m * ((nh - l1h) + (nl - l1l)), tab);
    double omy;
    if (ys <= 0.5) {
        omy = 1.0 - ys;
    } else {
        // 1 - ys = -expm1(m log(1 - w)), log(1 - w) = log(x/(1+x)) = n L - l1:
        // l1 inherits the rounding of x (about 1e-16 absolute), so the
        // difference of the two double-doubles serves only while |n L - l1| >
        // log(3/2), i.e. x < 2; beyond, log1p(-w)
        const double lw = x < 2.0 ? (nh - l1h) + (nl - l1l) : f64_log1p(-w, tab);
        omy = -f64_expm1_neg(s.m * lw, tab);
    }
    th = s.theta_r + dth * se;
    K = Ks * s2 * (omy * omy);
    C = s.cfac * (ys * w);
}

// Brooks and Corey's closures (the alternative Sec. 1 names), FP64: air-entry
// head h_b = -1/alpha, pore-size index lambda = n; Se = (h_b / h)^lambda below
// h_b and 1 above; theta = theta_r + (theta_s - theta_r) Se, C = dtheta/dh =
// -lambda (theta_s - theta_r) Se / h, K = Ks Se^((2 + 3 lambda)/lambda).
__device__ __forceinline__ void closure_bc(const DevSoil &s, double Ks, double h, double &th, double &K, double &C)
{
    const double hb = -1.0 / s.alpha, lam = s.n;
    if (h >= hb) {
        th = s.theta_s;
        K = Ks;
        C = 0.0;
        return;
    }
    const double ls = lam * log(hb / h);          // log Se
    const double se = exp(ls);
    const double dth = s.theta_s - s.theta_r;
    th = s.theta_r + dth * se;
    C = -lam * dth * se / h;
    K = Ks * exp(ls * (2.0 + 3.0 * lam) / lam);
}

// Closures of one cell at head h < 0 outside the fixed-point range or of
// another model or arithmetic.  fp64 selects FP64 van Genuchten arithmetic
// instead of double-float.  Gardner (Eq. A6, a test model): K = Ks e^(alpha
// h), theta = theta_r + (theta_s-theta_r) e^(alpha h), in FP64.
__device__ __forceinline__ void closure_general(const DevSoil &s, double Ks, double h, const FFTables *__restrict__ tab,
                                                bool fp64, double &th, double &K, double &C)
{
    if (s.model == M_GARDNER) {
        const double dth = s.theta_s - s.theta_r;
        const double e = exp(s.alpha * h);
        K = Ks * e;
        th = s.theta_r + dth * e;
        C = dth * s.alpha * e;
        return;
    }
    if (s.model == M_BROOKS_COREY) {
        closure_bc(s, Ks, h, th, K, C);
        return;
    }
    if (fp64) closure_vg_fp64(s, Ks, h, tab, th, K, C);
    else closure_vg_df(s, Ks, h, tab, th, K, C);
}

// The same out of line, for the cells that the fixed-point form leaves over:
// two functions (4.2 M cells in range: 145 us; 154 with one and a switch).
struct Closure3 {
    double th, K, C;
};
static __device__ __noinline__ Closure3 closure_rest(const DevSoil *s, double Ks, double h, const FFTables *tab)
{
    Closure3 r;
    closure_general(*s, Ks, h, tab, true, r.th, r.K, r.C);
    return r;
}
static __device__ __noinline__ Closure3 closure_rest_df(const DevSoil *s, double Ks, double h, const FFTables *tab)
{
    Closure3 r;
    closure_general(*s, Ks, h, tab, false, r.th, r.K, r.C);
    return r;
}

// Closures of one cell at head h: theta*, K, C.  For h >= 0 (tie included)
// theta* = theta_s + S h, K = Ks, C = S, which makes d(theta*)/dh equal to
// Eq. 3 on both branches.  Unless arith is ARITH_DF, van Genuchten cells run in
// 64-bit fixed point (fx64.cuh; tables fx, global or a shared copy) wherever
// the state is in its range; the others in FP64, or with ARITH_FX_DF in
// double-float arithmetic (4.2 M cells all out of range: 975 and 213 us).
__device__ __forceinline__ void closure(const DevSoil &s, double Ks, double h, const FFTables *__restrict__ tab,
                                        const FxTables *__restrict__ fx, int arith, double &th, double &K, double &C)
{
    const unsigned long long hb = (unsigned long long)__double_as_longlong(h);
    if (hb <= 0x7ff0000000000000ULL || hb == 0x8000000000000000ULL) {   // h >= 0
        th = s.theta_s + s.S * h;
        K = Ks;
        C = s.S;
        return;
    }
    uint64_t se, kr, cr;
    if (arith != ARITH_DF && fx_closure_vg(s.fx, hb & 0x7fffffffffffffffULL, fx, se, kr, cr)) {
        th = fma(s.dth, __longlong_as_double((long long)se), s.theta_r);
        K = Ks * __longlong_as_double((long long)kr);
        C = s.cfac * __longlong_as_double((long long)cr);
        return;
    }
    const Closure3 r = arith == ARITH_FP64 ? closure_rest(&s, Ks, h, tab) : closure_rest_df(&s, Ks, h, tab);
    th = r.th;
    K = r.K;
    C = r.C;
}

// The same in double-float arithmetic throughout, inline: for the closure
// kernels' instance of that choice (4.2 M cells: 233 us, out of line 246).
__device__ __forceinline__ void closure_df(const DevSoil &s, double Ks, double h, const FFTables *__restrict__ tab,
                                           double &th, double &K, double &C)
{
    if (h >= 0.0) {
        th = s.theta_s + s.S * h;
        K = Ks;
        C = s.S;
        return;
    }
    closure_general(s, Ks, h, tab, false, th, K, C);
}

// K at a Dirichlet face's head.  Out of line: the face loops are unrolled and
// few cells carry such a face.
static __device__ __noinline__ double closure_face(const DevSoil *s, double Ks, double h, const FFTables *tab,
                                                   int arith)
{
    double th, K, C;
    closure(*s, Ks, h, tab, &tab->fx, arith, th, K, C);
    return K;
}

// Neighbour across face f of cell p = (i,j,k); false when outside the grid.
__device__ __forceinline__ bool neighbour(const Grid &g, long long p, int i, int j, int k, int f, long long &q)
{
    switch (f) {
    case F_XMIN: q = p - 1; return i > 0;
    case F_XMAX: q = p + 1; return i < g.nx - 1;
    case F_YMIN: q = p - g.nx; return j > 0;
    case F_YMAX: q = p + g.nx; return j < g.ny - 1;
    case F_ZMIN: q = p - g.sxy; return k > 0;
    default:     q = p + g.sxy; return k < g.nz - 1;
    }
}

// FP64 stencil with stored coefficients; get(q) supplies the vector value.
template <class Get>
__device__ __forceinline__ double apply64(const Grid &g, long long p, const double *__restrict__ Tx,
                                          const double *__restrict__ Ty, const double *__restrict__ Tz,
                                          const double *__restrict__ diag, Get get)
{
    int i, j, k;
    cell_ijk(g, p, i, j, k);
    double acc = diag[p] * get(p);
    if (i > 0) acc -= Tx[p - 1] * get(p - 1);
    if (i < g.nx - 1) acc -= Tx[p] * get(p + 1);
    if (j > 0) acc -= Ty[p - g.nx] * get(p - g.nx);
    if (j < g.ny - 1) acc -= Ty[p] * get(p + g.nx);
    if (k > 0) acc -= Tz[p - g.sxy] * get(p - g.sxy);
    if (k < g.nz - 1) acc -= Tz[p] * get(p + g.sxy);
    return acc;
}

// Terms of boundary face f of cell p: diagonal (diag, cb) and right side.
__device__ __forceinline__ void boundary_face(const Grid &g, const DevSoil *__restrict__ soils,
                                              const uint8_t *__restrict__ zone, const double *__restrict__ Ks,
                                              const StepParams &sp, long long p, int f, double hnP, double KP,
                                              double &diag, double &cb, double &rhs)
{
    const double gs = g.gf[f];
    int type = sp.bc_type[f];
    double hD = 0.0;
    if (type == BC_SEEPAGE) {
        if (hnP >= 0.0) { type = BC_DIRICHLET; hD = 0.0; }
        else type = BC_ZERO_FLUX;
    } else if (type == BC_DIRICHLET) {
        hD = sp.bc_val[f];
    }
    if (type == BC_DIRICHLET) {
        const double KD = closure_face(&soils[zone[p]], Ks[p], hD, g.tab, g.arith);
        const double T = KD * g.wb[f];
        diag += T;
        cb += T;
        rhs += T * hD + gs * KD * g.A[f];
    } else if (type == BC_FLUX) {
        rhs += sp.bc_val[f] * g.A[f];
    } else if (type == BC_FREE_DRAINAGE) {
        rhs += gs * KP * g.A[f];       // unit gradient: gravity outflow K(h^k) A (gs = -1 at a z-up bottom)
    }
}

// The positive arithmetic of the assembly on the integer pipes (ix64.cuh),
// with FP64 for operands outside the range in which products of the integer
// form stay normal numbers.
constexpr long long K_CLOSED = (long long)0xbff0000000000000ULL;   // bits of K = -1 (inactive, outside)

// T = Kbar A/d of the face between cells with the bits a, b of K (0 when
// either is closed); hw its A/(2 d), ihw the same unpacked.
__device__ __forceinline__ double face_coef(const Grid &g, long long a, long long b, double hw, const IxNum &ihw)
{
    if ((a | b) < 0) return 0.0;
    if (g.ix_ok && (unsigned)(a >> 52) - 400u < 1200u && (unsigned)(b >> 52) - 400u < 1200u)
        return __longlong_as_double((long long)ix_pack(ix_add_mul(ix_unpack(a), ix_unpack(b), ihw)));
    const double x = __longlong_as_double(a), y = __longlong_as_double(b);
    double s = x + y;
    if (g.harmonic) s = s > 0.0 ? 4.0 * x * y / s : 0.0;
    return s * hw;
}

// c = V_dt (theta^k - theta^n) / (h^k - h^n), dth and dh the differences.
__device__ __forceinline__ double chord_c(double dth, double dh, double V_dt)
{
    const double f = ix_div(V_dt, __longlong_as_double(__double_as_longlong(dh) & 0x7fffffffffffffffLL));
    return __longlong_as_double(__double_as_longlong(dth) ^
                                (__double_as_longlong(dh) & (long long)0x8000000000000000ULL)) * f;
}

// Diagonal of a cell: c plus its six face coefficients.  In FP64 the six adds
// were a quarter of the assembly's instructions on the FP64 pipe.
__device__ __forceinline__ double diag_sum(double c, const double (&T)[6])
{
    const uint64_t b[7] = {(uint64_t)__double_as_longlong(c),    (uint64_t)__double_as_longlong(T[0]),
                           (uint64_t)__double_as_longlong(T[1]), (uint64_t)__double_as_longlong(T[2]),
                           (uint64_t)__double_as_longlong(T[3]), (uint64_t)__double_as_longlong(T[4]),
                           (uint64_t)__double_as_longlong(T[5])};
    uint64_t s;
    if (ix_sum7(b, s)) return __longlong_as_double((long long)s);
    return c + (((T[0] + T[1]) + (T[2] + T[3])) + (T[4] + T[5]));
}

// Storage part of a cell: c = V C^k / dt and its share s0 of the right side.
// form: storage_form(sp), held by the caller.
enum { STORE_CHORD = 0, STORE_MODIFIED = 1, STORE_BDF2 = 2 };
__device__ __forceinline__ int storage_form(const StepParams &sp)
{
    return sp.bdf2 ? STORE_BDF2 : sp.modified ? STORE_MODIFIED : STORE_CHORD;
}
__device__ __forceinline__ void storage_terms(int form, const StepParams &sp, double V_dt, double eps, double hkP,
                                              double hnP, double thk, double thn, double can,
                                              const double *__restrict__ thp, long long p, double &c, double &s0)
{
    if (form == STORE_BDF2) {
        // variable-step BDF2 (the multistep alternative Sec. 2.2 names) in the
        // mixed form V/dt [a0 theta^{n+1} - a1 theta^n + a2 theta^{n-1}],
        // theta^{n+1} linearised about h^k as in the modified Picard form
        c = V_dt * (sp.a0 * can);
        s0 = V_dt * (sp.a0 * can * hkP - (sp.a0 * thk - sp.a1 * thn + sp.a2 * thp[p]));
    } else if (form == STORE_MODIFIED) {
        // modified Picard (Sec. 2.2, mass-conservative variant): theta*(h^{k+1})
        // ~ theta*(h^k) + C(h^k) (h^{k+1} - h^k), so the storage term is
        // c (h^{k+1} - h^k) + V (theta*(h^k) - theta*(h^n)) / dt
        c = V_dt * can;
        s0 = c * hkP - V_dt * (thk - thn);
    } else {
        // classical Picard with the chord slope of theta* between h^n and h^k;
        // |dh| > eps compared on the IEEE bit patterns (both non-negative)
        const double dh = hkP - hnP;
        const bool chord = (__double_as_longlong(dh) & 0x7fffffffffffffffLL) > __double_as_longlong(eps);
        c = chord ? chord_c(thk - thn, dh, V_dt) : V_dt * can;
        s0 = c * hnP;
    }
}

// One cell of the Picard system (Sec. 2.2; see k_assemble):
//   c = V C^k / dt (chord slope of theta*, or C(h^k) when |h^k - h^n| <= eps),
//   interior faces T_f = Kbar_f A_f/d_f with Kbar_f = (K_P + K_N)/2 (or the
//   harmonic mean 2 K_P K_N / (K_P + K_N)) and explicit gravity T_f gd_f,
//   gd_f the elevation gradient along the face's outward normal times d_f
//   (+d top, -d bottom, 0 lateral on a z-up grid),
//   boundary terms of the face classes flagged in fl.
// With RESID, sT = sum over interior faces of T_f h^k_N (for b - A h^k).
// thp: theta*(h^{n-1}), read only by the BDF2 storage.
struct CellSystem {
    double c, rhs, diag, cb, sT, KP;
    double s0;        // storage part of rhs
    double Tup[3];
};

template <bool RESID>
__device__ __forceinline__ void assemble_cell(const Grid &g, const DevSoil *__restrict__ soils,
                                              const uint8_t *__restrict__ zone, const double *__restrict__ Ks,
                                              uint8_t fl, const StepParams &sp, long long p, int i, int j, int k,
                                              const double *__restrict__ hk, const double *__restrict__ hn,
                                              const double *__restrict__ thk, const double *__restrict__ thn,
                                              const double *__restrict__ K, const double *__restrict__ Can,
                                              const double *__restrict__ thp, double eps, double V_dt,
                                              CellSystem &out)
{
    const double hkP = hk[p], hnP = hn[p], KP = K[p];
    const long long kb = __double_as_longlong(KP);
    double c, s0;
    storage_terms(storage_form(sp), sp, V_dt, eps, hkP, hnP, thk[p], thn[p], Can[p], thp, p, c, s0);
    double T[6], sT = 0.0;
#pragma unroll
    for (int f = 0; f < 6; f++) {
        long long q;
        const bool in = neighbour(g, p, i, j, k, f, q);
        const long long kn = in ? __double_as_longlong(K[q]) : K_CLOSED;
        T[f] = face_coef(g, kb, kn, g.hw[f], ix_unpack((uint64_t)__double_as_longlong(g.hw[f])));
        if (RESID) {
            const double hN = kn >= 0 ? hk[q] : 0.0;
            sT = f == 0 ? T[f] * hN : fma(T[f], hN, sT);
        }
    }
    double diag = diag_sum(c, T);
    double rhs = fma(T[5], g.gd[F_ZMAX], fma(T[4], g.gd[F_ZMIN], s0));   // explicit gravity
    if (g.tilted) {
        rhs = fma(T[0], g.gd[F_XMIN], fma(T[1], g.gd[F_XMAX], rhs));
        rhs = fma(T[2], g.gd[F_YMIN], fma(T[3], g.gd[F_YMAX], rhs));
    }
    double cb = c;
    if (fl & 0x3f) {
        for (int f = 0; f < 6; f++)
            if (fl & (1u << f)) boundary_face(g, soils, zone, Ks, sp, p, f, hnP, KP, diag, cb, rhs);
    }
    out.c = c;
    out.s0 = s0;
    out.rhs = rhs;
    out.diag = diag;
    out.cb = cb;
    out.sT = sT;
    out.KP = KP;
    out.Tup[0] = T[1];
    out.Tup[1] = T[3];
    out.Tup[2] = T[5];
}

// Boundary inflow (fin >= 0) and outflow (fout >= 0) of one cell's boundary
// faces in the linear system solved for x (the water balance of Sec. 2.2's
// chord-slope scheme): Dirichlet T_D (h_D - x) + gf K(h_D) A, imposed flux,
// free drainage gf K(h^k) A, seepage as Dirichlet 0 while h^n >= 0.
__device__ __forceinline__ void boundary_fluxes(const Grid &g, const DevSoil &s, double Ksp, uint8_t fl,
                                                const StepParams &sp, double xp, double hnP, double Kold,
                                                double &fin, double &fout)
{
    fin = 0.0;
    fout = 0.0;
#pragma unroll
    for (int f = 0; f < 6; f++) {
        if (!(fl & (1u << f))) continue;
        const double gs = g.gf[f];
        int type = sp.bc_type[f];
        double hD = 0.0, flux = 0.0;
        if (type == BC_SEEPAGE) {
            if (hnP >= 0.0) { type = BC_DIRICHLET; hD = 0.0; }
            else type = BC_ZERO_FLUX;
        } else if (type == BC_DIRICHLET) {
            hD = sp.bc_val[f];
        }
        if (type == BC_DIRICHLET) {
            const double KD = closure_face(&s, Ksp, hD, g.tab, g.arith);
            const double T = KD * g.wb[f];
            flux = T * hD + gs * KD * g.A[f] - T * xp;
        } else if (type == BC_FLUX) {
            flux = sp.bc_val[f] * g.A[f];
        } else if (type == BC_FREE_DRAINAGE) {
            flux = gs * Kold * g.A[f];
        }
        if (flux > 0.0) fin += flux;
        else fout -= flux;
    }
}

}  // namespace rf
