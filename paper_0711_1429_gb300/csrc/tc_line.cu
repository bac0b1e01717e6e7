// Line phase: for every Fourier pair (m, alpha) the radial rows of Eq. 6 (v)
// and Eq. 7 (eta), the banded radial solves, the Runge-Kutta memory and the
// reconstruction of u, w from continuity; plus the mean flow (m = alpha = 0).
//
// The 32 threads of a warp hold 32 consecutive azimuthal indices at one axial
// slot, so every radial point is one coalesced 512-byte access per field.
//
// Notation (Appendix): D f = f', D_* f = f' + f/r, k^2 = alpha^2 + m^2/r^2,
// c = 1/k^2, c1..c3 its r-derivatives, nu = 2/Re.  On row j a chain operator
// applied to (coefficient x field) is the row stencil (d0, l1, l2, l4 for
// I, D, D D_*, D D_* D D_*) applied to the pointwise product; D D g is
// written D D_* g - D(g/r).
//
// Runge-Kutta (3 substeps, explicit third order + Crank-Nicolson): substep k
// solves (M - beta_k dt L) x^k = H_k + gamma_k dt E(x^(k-1)) with the stored
//   H_k = (M + alpha_k dt L) x^(k-1) + zeta_k dt E(x^(k-2)),
// and prepares H_(k+1) = RHS_k + zeta_(k+1) dt E(x^(k-1)) + (beta_k +
// alpha_(k+1)) dt L x^k, using M x^k = RHS_k + beta_k dt L x^k.
#include "tc_internal.h"
#include "tc_dfloat.h"
#include <type_traits>

__device__ __forceinline__ dfloat fma(dfloat a, dfloat b, dfloat c) { return a * b + c; }

namespace {

struct Coef { double k2, c, c1, c2, c3; };

// k^2, c = 1/k^2 = r^2/g and its r-derivatives, g = alpha^2 r^2 + m^2:
// c1 = 2 r m^2/g^2, c2 = 2 m^2 (m^2 - 3 alpha^2 r^2)/g^3,
// c3 = -24 m^2 alpha^2 r (m^2 - alpha^2 r^2)/g^4.
__device__ __forceinline__ Coef coef_at(double r, double rinv, double m, double al) {
    const double m2 = m * m, a2 = al * al, r2 = r * r;
    Coef o;
    o.k2 = a2 + m2 * rinv * rinv;
    const double g = a2 * r2 + m2;
    const double gi = 1.0 / g;
    const double gi2 = gi * gi;
    o.c = r2 * gi;
    o.c1 = 2.0 * r * m2 * gi2;
    o.c2 = 2.0 * m2 * (m2 - 3.0 * a2 * r2) * gi2 * gi;
    o.c3 = -24.0 * m2 * a2 * r * (m2 - a2 * r2) * gi2 * gi2;
    return o;
}

__device__ __forceinline__ double2 cz() { return make_double2(0.0, 0.0); }
// a + s * b
__device__ __forceinline__ double2 caxpy(double2 a, double s, double2 b) { return make_double2(fma(s, b.x, a.x), fma(s, b.y, a.y)); }
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
// finiteness from the exponent bits (integer pipe, no float64 compare)
__device__ __forceinline__ bool dfinite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

__device__ __forceinline__ double2 ld_prod(const double2* p, size_t o) { return p[o]; }
__device__ __forceinline__ double2 ld_prod(const float2* p, size_t o) { float2 f = p[o]; return make_double2(d_bits(f.x), d_bits(f.y)); }

// generic complex helpers for float2 / double2
template <typename CT> __device__ __forceinline__ CT tz() { CT r; r.x = 0; r.y = 0; return r; }
template <typename CT> __device__ __forceinline__ CT tadd(CT a, CT b) { CT r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
template <typename CT> __device__ __forceinline__ CT tsub(CT a, CT b) { CT r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
template <typename CT, typename T> __device__ __forceinline__ CT taxpy(CT a, T s, CT b) { CT r; r.x = fma(s, b.x, a.x); r.y = fma(s, b.y, a.y); return r; }
template <typename CT, typename T> __device__ __forceinline__ CT tscale(T s, CT a) { CT r; r.x = s * a.x; r.y = s * a.y; return r; }
__device__ __forceinline__ double2 to_d2(double2 a) { return a; }
// float32 <-> float64 through the integer conversions of tc_dfloat.h (the
// float64 pipe is the mixed line phase's bottleneck); the double-float form
// converts with float64 instructions, which measured faster there (fewer
// registers in a kernel that is already at its register budget)
__device__ __forceinline__ double2 to_d2(float2 a) { return make_double2(d_bits(a.x), d_bits(a.y)); }
__device__ __forceinline__ double2 to_d2(dcomplex a) { return make_double2((double)a.x, (double)a.y); }
// the same exact widening by bit operations and one float64 add (d_of), for
// the mixed form's continuity term
__device__ __forceinline__ double2 to_d2_bits(dcomplex a) { return make_double2(d_of(a.x), d_of(a.y)); }
template <typename CT> __device__ __forceinline__ CT from_d2(double2 a);
template <> __device__ __forceinline__ double2 from_d2<double2>(double2 a) { return a; }
template <> __device__ __forceinline__ float2 from_d2<float2>(double2 a) { return make_float2(f_bits(a.x), f_bits(a.y)); }
template <> __device__ __forceinline__ dcomplex from_d2<dcomplex>(double2 a) { dcomplex r; r.x = dfloat(a.x); r.y = dfloat(a.y); return r; }
__device__ __forceinline__ dcomplex dc_bits(double2 a) { dcomplex r; r.x = df_bits(a.x); r.y = df_bits(a.y); return r; }
__device__ __forceinline__ dcomplex dc_fma(const dcomplex& a, dfloat s, const dcomplex& b) {
    dcomplex r;
    r.x = df_fma(a.x, s, b.x);
    r.y = df_fma(a.y, s, b.y);
    return r;
}
__device__ __forceinline__ dcomplex dc_scale(dfloat s, const dcomplex& a) {
    dcomplex r;
    r.x = s * a.x;
    r.y = s * a.y;
    return r;
}
__device__ __forceinline__ dcomplex dc_i(const dcomplex& a) {   // i a
    dcomplex r;
    r.x = -a.y;
    r.y = a.x;
    return r;
}
__device__ __forceinline__ dcomplex dc_of(float2 a) { dcomplex r; r.x = dfloat(a.x, 0.0f); r.y = dfloat(a.y, 0.0f); return r; }
__device__ __forceinline__ double2 ld_prod(const dcomplex* p, size_t o) { return to_d2(p[o]); }
__device__ __forceinline__ dfloat as_df(float2 v) { return dfloat(v.x, v.y); }

// element types of the three forms: 0 float64, 1 mixed (float32 explicit
// rows), 2 double-float explicit rows
template <int MODE> struct LineTypes;
template <> struct LineTypes<0> { typedef double T; typedef double2 CT; };
template <> struct LineTypes<1> { typedef float T; typedef float2 CT; };
template <> struct LineTypes<2> { typedef dfloat T; typedef dcomplex CT; };

// Pair index -> (n slot, j); returns false for pairs that are not evolved:
// the axial Nyquist slot, (0,0) (mean flow) and (0, n<0) (conjugates).
__device__ __forceinline__ bool pair_info(const TcDev& d, int pair, double& m, double& al, long long& partner) {
    const int s = pair / d.Nh, j = pair - s * d.Nh;
    if (s == d.Nz / 2) return false;
    if (j == 0 && (s == 0 || s > d.Nz / 2)) return false;
    const int n = s < d.Nz / 2 ? s : s - d.Nz;
    m = j * d.m0;
    al = n * d.alpha0;
    partner = (j == 0) ? (long long)(d.Nz - s) * d.Nh : -1;
    return true;
}

#define TAB(base, k, row, comp) (base)[((size_t)((k) * d.Nr + (row)) * 5 + (comp)) * d.npairs + pair]

// Reduced band row on the unknowns 1..Nr-2: entries on columns j-2..j+2.
struct Row5 { double a, b, dd, c, e; };

}  // namespace

// ---------------------------------------------------------------------------
// Band of the v rows (interior j = 2..Nr-3), entry s multiplies v_{j-2+s}:
//   mass      M = d0 - l2 c + l1 c1
//   implicit  L = nu [2 l2 - l4 c + l1 (c2/r + c3 - c1/r^2 - 2 m^2 c/r^3)
//                     - 2 l2 c1/r - d0 k^2]
// (Eq. 6 with D_1 read as D and D[(1/r) DD(1/k^2) v] read as D[(c2/r) v]).
__device__ void v_band(const TcDev& d, int j, double m, double al, double* M5, double* L5) {
    for (int s = 0; s < 5; ++s) {
        const int i = j - 2 + s;
        const double r = d.r[i], ri = d.rinv[i];
        const Coef q = coef_at(r, ri, m, al);
        const double w0 = d.d0[j * 5 + s], w1 = d.l1[j * 5 + s], w2 = d.l2[j * 5 + s], w4 = d.l4[j * 5 + s];
        M5[s] = w0 - w2 * q.c + w1 * q.c1;
        L5[s] = d.nu * (2.0 * w2 - w4 * q.c
                        + w1 * (q.c2 * ri + q.c3 - q.c1 * ri * ri - 2.0 * m * m * q.c * ri * ri * ri)
                        - 2.0 * w2 * q.c1 * ri - w0 * q.k2);
    }
}

// eta rows j = 1..Nr-2: mass d0, implicit nu (l2 - d0 k^2), from start[j].
__device__ void eta_band(const TcDev& d, int j, double m, double al, double* L5) {
    const int st = d.start[j];
    for (int s = 0; s < 5; ++s) {
        const int i = st + s;
        const double ri = d.rinv[i];
        const double k2 = al * al + m * m * ri * ri;
        L5[s] = d.nu * (d.l2[j * 5 + s] - d.d0[j * 5 + s] * k2);
    }
}

// Pentadiagonal LU without pivoting of the reduced system on unknowns
// 1..Nr-2, rows produced by `row(i)`; stores per row (m2, m1, 1/diag, c', e)
// and returns false on a vanishing pivot.
template <typename RowFn>
__device__ bool band_lu(const TcDev& d, double* tab, int k, int pair, RowFn row) {
    double p2d = 1, p2c = 0, p2e = 0, p1d = 1, p1c = 0, p1e = 0;
    bool ok = true;
    for (int i = 1; i <= d.Nr - 2; ++i) {
        Row5 R = row(i);
        const double scale = fabs(R.a) + fabs(R.b) + fabs(R.dd) + fabs(R.c) + fabs(R.e);
        const double m2 = (i >= 3) ? R.a / p2d : 0.0;
        double b = R.b - m2 * p2c;
        double dd = R.dd - m2 * p2e;
        const double m1 = (i >= 2) ? b / p1d : 0.0;
        dd = dd - m1 * p1c;
        const double cc = R.c - m1 * p1e;
        if (!(fabs(dd) > 1e-13 * scale)) ok = false;
        TAB(tab, k, i, 0) = m2;
        TAB(tab, k, i, 1) = m1;
        TAB(tab, k, i, 2) = 1.0 / dd;
        TAB(tab, k, i, 3) = cc;
        TAB(tab, k, i, 4) = R.e;
        p2d = p1d; p2c = p1c; p2e = p1e;
        p1d = dd; p1c = cc; p1e = R.e;
    }
    return ok;
}

// k^2 = alpha^2 + m^2/r^2 of the implicit eta band
__device__ __forceinline__ double k2_at(double m, double al, double ri) {
    return __fma_rn(__dmul_rn(m, m), __dmul_rn(ri, ri), __dmul_rn(al, al));
}

// Per-pair tables: LU factors of (M - beta_k dt L) for v and eta, k = 0..2,
// with the boundary rows folded in, and the implicit band L of the v rows.
__global__ void __launch_bounds__(128) k_setup(TcDev d) {
    const int pair = blockIdx.x * blockDim.x + threadIdx.x;
    if (pair >= d.npairs) return;
    double m, al;
    long long partner;
    if (!pair_info(d, pair, m, al, partner)) return;
    const int N = d.Nr;
    const double* e0 = d.dwall;       // D at r_0 on points 0..4
    const double* e1 = d.dwall + 5;   // D at r_{N-1} on points N-5..N-1
    bool ok = true;
    for (int i = 0; i < N; ++i) {
        const Coef q = coef_at(d.r[i], d.rinv[i], m, al);
        d.tab_c[(size_t)i * d.npairs + pair] = q.c;
        if (d.tab_c1) d.tab_c1[(size_t)i * d.npairs + pair] = q.c1;
        if (d.tab_cx) {
            const dfloat a(q.c), b(q.c1);
            d.tab_cx[(size_t)i * d.npairs + pair] = make_float2(a.hi, a.lo);
            d.tab_c1x[(size_t)i * d.npairs + pair] = make_float2(b.hi, b.lo);
        }
    }
    // implicit band of the v rows (substep independent)
    for (int j = 2; j <= N - 3; ++j) {
        double M5[5], L5[5];
        v_band(d, j, m, al, M5, L5);
        for (int s = 0; s < 5; ++s) TAB(d.tab_lv, 0, j, s) = L5[s];
    }
    // and of the eta rows, over nu
    for (int j = 1; j <= N - 2; ++j)
        for (int s = 0; s < 5; ++s)
            TAB(d.tab_le, 0, j, s) = fma(-d.d0[j * 5 + s], k2_at(m, al, d.rinv[d.start[j] + s]), d.l2[j * 5 + s]);
    for (int k = 0; k < 3; ++k) {
        const double bdt = d.rk_beta[k] * d.dt;
        // ---- v system ----
        auto vrow_full = [&](int j, double* A) {
            double M5[5], L5[5];
            v_band(d, j, m, al, M5, L5);
            for (int s = 0; s < 5; ++s) A[s] = M5[s] - bdt * L5[s];
        };
        double A2[5], A3[5];
        vrow_full(2, A2);
        vrow_full(N - 3, A3);
        // row 1 (Dv(r_0) = 0 on v_1..v_4) minus f * row 2 eliminates v_4
        const double fv = e0[4] / A2[4];
        const Row5 v1r = {0.0, 0.0, e0[1] - fv * A2[1], e0[2] - fv * A2[2], e0[3] - fv * A2[3]};
        // row N-2 (Dv(r_{N-1}) = 0 on v_{N-5}..v_{N-2}) minus g * row N-3
        const double gv = e1[0] / A3[0];
        const Row5 vNr = {e1[1] - gv * A3[1], e1[2] - gv * A3[2], e1[3] - gv * A3[3], 0.0, 0.0};
        ok &= band_lu(d, d.tab_luv, k, pair, [&](int i) -> Row5 {
            if (i == 1) return v1r;
            if (i == N - 2) return vNr;
            double A[5];
            vrow_full(i, A);
            Row5 R = {A[0], A[1], A[2], A[3], A[4]};
            if (i == 2) R.a = 0.0;          // column 0: v_0 = 0
            if (i == N - 3) R.e = 0.0;      // column N-1: v_{N-1} = 0
            return R;
        });
        TAB(d.tab_luv, k, 0, 0) = fv;
        TAB(d.tab_luv, k, N - 1, 0) = gv;
        // ---- eta system ----
        auto erow_full = [&](int j, double* A) {
            double L5[5];
            eta_band(d, j, m, al, L5);
            for (int s = 0; s < 5; ++s) A[s] = d.d0[j * 5 + s] - bdt * L5[s];
        };
        double B1[5], B2[5], B3[5], BN[5];
        erow_full(1, B1);          // start 0: columns 0..4
        erow_full(2, B2);
        erow_full(N - 3, B3);
        erow_full(N - 2, BN);      // start N-5
        const double fe = B1[4] / B2[4];
        const Row5 e1r = {0.0, 0.0, B1[1] - fe * B2[1], B1[2] - fe * B2[2], B1[3] - fe * B2[3]};
        const double ge = BN[0] / B3[0];
        const Row5 eNr = {BN[1] - ge * B3[1], BN[2] - ge * B3[2], BN[3] - ge * B3[3], 0.0, 0.0};
        ok &= band_lu(d, d.tab_lue, k, pair, [&](int i) -> Row5 {
            if (i == 1) return e1r;
            if (i == N - 2) return eNr;
            double A[5];
            erow_full(i, A);
            Row5 R = {A[0], A[1], A[2], A[3], A[4]};
            if (i == 2) R.a = 0.0;
            if (i == N - 3) R.e = 0.0;
            return R;
        });
        TAB(d.tab_lue, k, 0, 0) = fe;
        TAB(d.tab_lue, k, N - 1, 0) = ge;
    }
    if (!ok) atomicOr(d.flag + 1, 1);
}

// ---------------------------------------------------------------------------
// The line phase of one substep, for the pairs of the azimuthal columns
// ja .. ja + jw - 1 in every axial slot (all pairs when ja = 0, jw = Ntheta/2):
// two kernels.
//
// k_explicit, one warp per 32 pairs and chunk of radial rows: the explicit rows E
// (Eq. 6 rows 2..Nr-3, Eq. 7 rows 1..Nr-2), the right sides
// RHS = H_k + gamma_k dt E (v: scratch, eta: in place, which no explicit row
// reads) and H = RHS + zeta_(k+1) dt E.
// k_solve, two warps per 16 pairs (k_solve_shared, eight, for few pairs): one warp runs the recurrences of v (the
// banded solve and later the compact Dv solve), another those of eta; what is not
// serial in r -- the right sides l1 . v of the Dv solve, H += (beta_k + alpha_(k+1))
// dt L x, and u, w from continuity -- all warps share by radial rows.
//
// What bounds it: the float64 pipe, 64 cycles for a warp's operation on its quarter
// of an SM, however few lanes it has.  One thread that walked a pair's whole line
// kept a small case on the few quarters its warps filled (256 pairs: eight) and
// put every operation of a row behind the one before; only the recurrences, an
// eighth of the operations, are serial in r.  Per substep, line phase of the
// float64 form before and now: 33x16x16 333 -> 45 us, 64x32x64 684 -> 82,
// 129x128x128 1118 -> 536, 129x512x170 2897 -> 2400, 257x512x512 15.5 -> 13.5 ms; of
// the mixed form: 129x128x128 923 -> 350 us, 257x512x512 7.9 (the best of that kernel's
// launch shapes) -> 8.0 ms.
//
// Explicit rows: sums over the 5 stencil points of d0 . A + l1 . B (+ l2 . C for
// v), where A, B, C are pointwise "inner" functions of the products and of u, v, w
// at that point.  With the five products a = uu - vv, uv, uw, vw, b = ww - vv:
//   v:   A = -i alpha uv - i m/r vw + b/r                 - 2 i nu m w/r^2
//        B = i alpha c1 uv - i m (2c/r^2 - c1/r) vw + c alpha^2 a
//            + 2 c alpha m/r uw + c m^2/r^2 b             - 2 i nu m c1 w/r^2
//        C = -i alpha c uv - i m c/r vw                   + 2 i nu m c w/r^2
//            - 3 nu c1 (i alpha u + i m/r w)              [continuity term]
//   eta: A = m alpha a/r - 2 i m uv/r^2 + (m^2/r^2 - alpha^2) uw - alpha m b/r
//            + 2 i alpha vw/r + 4 i nu m u/r^3 + 2 nu m alpha v/r^2
//        B = -i m uv/r + i alpha vw + 2 i nu m u/r^2
// (the terms of Eqs. 6-7 regrouped per stencil; the vv parts cancel because
// c k^2 = 1).  In the mixed form everything except the continuity term is
// formed in float32 from the float32 products, and the continuity term in
// double-float arithmetic; in the double-float form all explicit rows are
// formed in double-float arithmetic (float32 pipe) from the double-float
// products; the right sides, the solves, the RK memory and the
// reconstruction are float64 in every form.
//
// Inner functions as listed above (float32 of the mixed form), C without the
// continuity term.  Which product of a sum of two is fused is written out, so that
// the rounding does not depend on what the compiler makes of the surrounding loop.
__device__ __forceinline__ float sum2(float p, float x, float q, float y) { return fmaf(p, x, __fmul_rn(q, y)); }
__device__ __forceinline__ float2 ifma(float s, float2 x, float2 acc) { return make_float2(fmaf(-s, x.y, acc.x), fmaf(s, x.x, acc.y)); }
__device__ __forceinline__ void inner_terms(const float2& pa, const float2& uv, const float2& uw, const float2& vw, const float2& pb,
                                            const float2& U, const float2& V, const float2& W, float ri, float c, float c1,
                                            float mt, float at, float nut, float2& a, float2& b, float2& cc, float2& ae,
                                            float2& be) {
    const float ri2 = ri * ri, mr = mt * ri;
    // v rows
    a = make_float2(sum2(at, uv.y, mr, vw.y), sum2(-mr, vw.x, -at, uv.x));
    a = taxpy(a, ri, pb);
    a = ifma(-2.0f * nut * mt * ri2, W, a);
    const float q1 = at * c1, q2 = -mt * sum2(2.0f * c, ri2, -c1, ri);
    b = make_float2(sum2(-q2, vw.y, -q1, uv.y), sum2(q1, uv.x, q2, vw.x));
    b = taxpy(b, c * at * at, pa);
    b = taxpy(b, c * 2.0f * at * mt * ri, uw);
    b = taxpy(b, c * mt * mt * ri2, pb);
    b = ifma(-2.0f * nut * mt * c1 * ri2, W, b);
    const float q3 = -at * c, q4 = -mt * c * ri;
    cc = make_float2(sum2(-q4, vw.y, -q3, uv.y), sum2(q3, uv.x, q4, vw.x));
    cc = ifma(2.0f * nut * mt * c * ri2, W, cc);
    // eta rows
    const float q5 = mt * at * ri, q6 = -2.0f * mt * ri2;
    ae = make_float2(sum2(q5, pa.x, -q6, uv.y), sum2(q5, pa.y, q6, uv.x));
    ae = taxpy(ae, sum2(mt * mt, ri2, -at, at), uw);
    ae = taxpy(ae, -at * mt * ri, pb);
    ae = ifma(2.0f * at * ri, vw, ae);
    ae = ifma(4.0f * nut * mt * ri2 * ri, U, ae);
    ae = taxpy(ae, 2.0f * nut * mt * at * ri2, V);
    be = make_float2(sum2(-at, vw.y, mr, uv.y), sum2(at, vw.x, -mr, uv.x));
    be = ifma(2.0f * nut * mt * ri2, U, be);
}
// The same with the continuity term, for the float64 and double-float forms, in
// which the arithmetic is what costs: shared sums are formed once (57 float64
// operations a point instead of 88, coefficients included).
//   Q = alpha uv + m/r vw,  S = 2 nu m/r^2 w,  T = Q - S
//   A = -i (Q + S) + b/r,   C = -i (c T + 3 nu c1 (alpha u + m/r w))
//   B = i (c1 T - 2 c m/r^2 vw) + c (alpha^2 a + 2 alpha m/r uw + m^2/r^2 b)
//   N = m/r uv - alpha vw - 2 nu m/r^2 u,  B_eta = -i N
//   A_eta = m alpha/r (a - b) + (m^2/r^2 - alpha^2) uw + 2 nu m alpha/r^2 v + (2/r) B_eta
// The last term of A_eta is left to the stencil of B_eta: l1e = l1 + 2 d0/r.
template <typename T> struct IsPair { static constexpr bool value = false; };
template <> struct IsPair<dfloat> { static constexpr bool value = true; };
template <typename T, typename CT>
__device__ __forceinline__ void inner_terms_shared(const CT& pa, const CT& uv, const CT& uw, const CT& vw, const CT& pb,
                                                   const CT& U, const CT& V, const CT& W, T ri, T c, T c1, T mt, T at,
                                                   T at2, T nu2, T nu3, CT& a, CT& b, CT& cc, CT& ae, CT& be) {
    const T mr = mt * ri, mr2 = mr * ri, mra = mr * at, n2 = nu2 * mr2;      // nu2 = 2 nu, nu3 = 3 nu
    const CT Q = taxpy(tscale(mr, vw), at, uv);
    CT Tm, Tp;                                  // Q - S, Q + S
    if constexpr (sizeof(T) == sizeof(double) && !IsPair<T>::value) { Tm = taxpy(Q, -n2, W); Tp = taxpy(Q, n2, W); }
    else { const CT S = tscale(n2, W); Tm = tsub(Q, S); Tp = tadd(Q, S); }
    a.x = fma(ri, pb.x, Tp.y);
    a.y = fma(ri, pb.y, -Tp.x);
    const CT ph = taxpy(tscale(mr, W), at, U);
    const CT Z = taxpy(tscale(c, Tm), nu3 * c1, ph);
    cc.x = Z.y;
    cc.y = -Z.x;
    const CT Y = taxpy(tscale(c1, Tm), (T)-2 * c * mr2, vw);
    const CT R = taxpy(taxpy(tscale(at2, pa), (T)2 * mra, uw), mr * mr, pb);
    b.x = fma(c, R.x, -Y.y);
    b.y = fma(c, R.y, Y.x);
    const CT N = taxpy(taxpy(tscale(mr, uv), -at, vw), -n2, U);
    be.x = N.y;
    be.y = -N.x;
    ae = taxpy(taxpy(tscale(mra, tsub(pa, pb)), fma(mr, mr, -at2), uw), n2 * at, V);
}

// The radial solves and sums have real coefficients, so the real and the imaginary
// part of a pair are two lanes of a warp: a warp instruction of the float64 pipe
// takes 64 cycles of its quarter of the SM however many of its lanes are in use, and
// each lane then has half the operations and registers.  Component c of a field at
// row i is base[2 i P], base = (double*)field + 2 pair + c.
struct RowTables { const double *d0, *l1, *dsol, *rinv; };   // the case's own, or copies in shared memory

// Implicit part of the next RK memory on row jr (SMR91 low storage):
// H_(k+1) += (beta_k + alpha_(k+1)) dt L x^(k+1), with L the band of row jr from the
// per-pair table, applied to the window x of x^(k+1) on the row's five stencil
// points.  k_solve calls it after its solves; the deferred form (k_rk_memory), after
// a k_solve that left it out, has the same operations on the same operands, so both
// give the same bits.
__device__ __forceinline__ void rk_memory_row(const TcDev& d, const double* __restrict__ tab, double* H, int pair, int jr,
                                              const double* x, double hdt) {
    double acc = 0.0;
    for (int s = 0; s < 5; ++s) acc = fma(TAB(tab, 0, jr, s), x[s], acc);
    H[2 * (size_t)jr * d.npairs] = fma(hdt, acc, H[2 * (size_t)jr * d.npairs]);
}
// The rows centred on i0 <= i < i1 (v: 2 .. Nr - 3; the one-sided eta rows 1 and
// Nr - 2 with their neighbours).
__device__ __forceinline__ void rk_memory_rows(const TcDev& d, int k, int pair, int comp, int i0, int i1) {
    const int N = d.Nr, kn = (k + 1) % 3;
    const size_t P2 = 2 * (size_t)d.npairs;
    const double hdt = (d.rk_beta[k] + d.rk_alpha[kn]) * d.dt, hdtnu = hdt * d.nu;
    const size_t o = 2 * (size_t)pair + comp;
    const double *v = reinterpret_cast<const double*>(d.v) + o, *e = reinterpret_cast<const double*>(d.eta) + o;
    double *Hv = reinterpret_cast<double*>(d.Hv) + o, *He = reinterpret_cast<double*>(d.He) + o;
    i0 = i0 < 2 ? 2 : i0;
    i1 = i1 > N - 2 ? N - 2 : i1;
    if (i0 >= i1) return;
    double xv[5], xe[5];
    for (int s = 0; s < 4; ++s) { xv[s + 1] = v[(i0 - 2 + s) * P2]; xe[s + 1] = e[(i0 - 2 + s) * P2]; }
    for (int i = i0; i < i1; ++i) {
        for (int s = 0; s < 4; ++s) { xv[s] = xv[s + 1]; xe[s] = xe[s + 1]; }
        xv[4] = v[(i + 2) * P2];
        xe[4] = e[(i + 2) * P2];
        rk_memory_row(d, d.tab_lv, Hv, pair, i, xv, hdt);
        rk_memory_row(d, d.tab_le, He, pair, i, xe, hdtnu);
        if (i == 2) rk_memory_row(d, d.tab_le, He, pair, 1, xe, hdtnu);
        if (i == N - 3) rk_memory_row(d, d.tab_le, He, pair, N - 2, xe, hdtnu);
    }
}

// thread idx -> pair among the columns ja .. ja + jw - 1 of every axial slot;
// false for a thread without a pair to evolve
__device__ __forceinline__ bool line_pair(const TcDev& d, int ja, int jw, int idx, int& pair, double& m, double& al,
                                          long long& partner) {
    if (idx >= d.Nz * jw) return false;
    pair = (idx / jw) * d.Nh + ja + idx % jw;
    partner = -1;
    return pair_info(d, pair, m, al, partner);
}
// Right sides of v between the two kernels: the last third of zbuf, free from
// the theta rows to the next z inverse, in zbuf's own layout, so that a column
// group's share is its own columns' (the float32 planes of the mixed form fill
// the first half of the buffer).
__device__ __forceinline__ double2* rhs_scratch(const TcDev& d, int pair) {
    return reinterpret_cast<double2*>(d.zbuf) + 2 * (size_t)d.Nr * d.Mzx * d.Nh + pair;
}

// The rows' inputs on their way through shared memory: in the mixed and the
// double-float form the arithmetic of a row (float32 pipe) is shorter than its loads
// take, and the registers of the stencils leave no room for a row's 34 to 44 words
// ahead of time.  Every thread copies its own words (cp.async) RING - 1 rows ahead,
// so that no barrier is needed.  (Line phase of the mixed form, 257x512x512: 8.28 ->
// 8.14 ms; of the double-float form, 129x512x170: 1.84 -> 1.78.)  The
// float64 form is bound by the float64 pipe and loads into registers.
constexpr int EXPLICIT_WARPS = 4;
template <int MODE> struct RowRing {
    typedef typename LineTypes<MODE>::CT CT;
    static constexpr int RING = MODE > 0 ? 3 : 0, NT = 32 * EXPLICIT_WARPS;
    static constexpr int FIELDS = 5 * sizeof(CT) * NT, H = FIELDS + 48 * NT, COEF = H + 32 * NT, BYTES = COEF + 16 * NT;
    unsigned char* base;
    __device__ CT& prod(int q) const { return *reinterpret_cast<CT*>(base + (q * NT + threadIdx.x) * sizeof(CT)); }
    __device__ double2& field(int q) const { return *reinterpret_cast<double2*>(base + FIELDS + (q * NT + threadIdx.x) * 16); }
    __device__ double2& memory(int q) const { return *reinterpret_cast<double2*>(base + H + (q * NT + threadIdx.x) * 16); }
    __device__ float2& coef(int q) const { return *reinterpret_cast<float2*>(base + COEF + (q * NT + threadIdx.x) * 8); }
};
template <int BYTES> __device__ __forceinline__ void copy_async(void* to, const void* from) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(to);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(from) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(a), "l"(from) : "memory");
}

// Rows centred on c0 <= j < c1 of 2 .. Nr - 3; the one-sided eta rows 1 and
// Nr - 2 go with their neighbours 2 and Nr - 3, whose points they use.
template <int MODE>
__device__ __forceinline__ void explicit_rows(const TcDev& d, int k, int ja, int jw, int idx, int c0, int c1) {
    constexpr bool MIXED = (MODE == 1);
    typedef typename LineTypes<MODE>::T T;
    typedef typename LineTypes<MODE>::CT CT;
    int pair;
    double m, al;
    long long partner;
    if (!line_pair(d, ja, jw, idx, pair, m, al, partner)) return;
    const int N = d.Nr;
    const size_t P = d.npairs, SP = (size_t)d.Mzx * d.Nh;
    const CT* __restrict__ prod = reinterpret_cast<const CT*>(d.prod);
    const double2* __restrict__ fu = d.u;
    const double2* __restrict__ fv = d.v;
    const double2* __restrict__ fw = d.w;
    double2* rhsv = rhs_scratch(d, pair);
    const size_t PS = (size_t)N * P;            // product stride
    const int kn = (k + 1) % 3;
    const double gdt = d.rk_gamma[k] * d.dt;
    const double zdt = d.rk_zeta[kn] * d.dt;
    const double nu = d.nu;
    const T mt = (T)m, at = (T)al, nut = (T)nu;
    const T at2 = at * at, nu2 = (T)2 * nut, nu3 = (T)3 * nut;
    // double-float constants of the mixed form's continuity term
    const dfloat mD(m), alD(al), m3nu(-3.0 * nu);
    const dfloat* l2x = reinterpret_cast<const dfloat*>(d.l2x);
    const dfloat* rinvx = reinterpret_cast<const dfloat*>(d.rinvx);
    const T *w0s, *w1s, *w2s, *w1e;
    if constexpr (MODE == 1) { w0s = d.d0f; w1s = d.l1f; w2s = d.l2f; w1e = d.l1f; }
    else if constexpr (MODE == 2) {
        w0s = reinterpret_cast<const dfloat*>(d.d0x);
        w1s = reinterpret_cast<const dfloat*>(d.l1x);
        w2s = reinterpret_cast<const dfloat*>(d.l2x);
        w1e = reinterpret_cast<const dfloat*>(d.l1ex);
    } else { w0s = d.d0; w1s = d.l1; w2s = d.l2; w1e = d.l1e; }

    CT Av[5], Bv[5], Cv[5], Ae[5], Be[5];
    dcomplex Cp[5];                             // continuity inner function (mixed form)
    for (int s = 0; s < 5; ++s) Av[s] = Bv[s] = Cv[s] = Ae[s] = Be[s] = tz<CT>();
    auto erow = [&](int j, double2 H) {         // explicit eta row j, its right side and H
        CT acc = tz<CT>();
        for (int s = 0; s < 5; ++s) {
            acc = taxpy(acc, w0s[j * 5 + s], Ae[s]);
            acc = taxpy(acc, w1e[j * 5 + s], Be[s]);
        }
        const double2 E = to_d2(acc);
        const size_t o = (size_t)j * P + pair;
        const double2 r = caxpy(H, gdt, E);
        d.He[o] = caxpy(r, zdt, E);
        d.eta[o] = r;
    };
    auto vrow = [&](int j, double2 H) {
        CT acc = tz<CT>();
        for (int s = 0; s < 5; ++s) {
            acc = taxpy(acc, w0s[j * 5 + s], Av[s]);
            acc = taxpy(acc, w1s[j * 5 + s], Bv[s]);
            acc = taxpy(acc, w2s[j * 5 + s], Cv[s]);
        }
        double2 E;
        if constexpr (MIXED) {
            // float32 rows plus the continuity term -3 nu l2 . (c' phi) in
            // double-float, then widened to float64
            dcomplex cc;
            for (int s = 0; s < 5; ++s) cc = dc_fma(cc, l2x[j * 5 + s], Cp[s]);
            E = to_d2_bits(dc_fma(dc_of(acc), m3nu, cc));
        } else {
            E = to_d2(acc);
        }
        const size_t o = (size_t)j * P + pair;
        const double2 r = caxpy(H, gdt, E);
        d.Hv[o] = caxpy(r, zdt, E);
        rhsv[(size_t)j * SP] = r;
    };
    typedef RowRing<MODE> Ring;
    extern __shared__ double sm[];
    int rd = 0, wr = 0;
    auto fetch = [&](int i) {
        if constexpr (Ring::RING > 0) {
            if (i < c1 + 2) {
                const Ring g{reinterpret_cast<unsigned char*>(sm) + wr * Ring::BYTES};
                wr = wr + 1 == Ring::RING ? 0 : wr + 1;
                const size_t o = (size_t)i * P + pair;
#pragma unroll
                for (int q = 0; q < 5; ++q) copy_async<sizeof(CT)>(&g.prod(q), prod + o + q * PS);
                copy_async<16>(&g.field(0), fu + o);
                copy_async<16>(&g.field(1), fv + o);
                copy_async<16>(&g.field(2), fw + o);
                copy_async<8>(&g.coef(0), d.tab_cx + o);
                copy_async<8>(&g.coef(1), d.tab_c1x + o);
                if (i >= c0 + 2) {
                    copy_async<16>(&g.memory(0), d.Hv + o - 2 * P);
                    copy_async<16>(&g.memory(1), d.He + o - 2 * P);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    };
    if constexpr (Ring::RING > 0)
        for (int q = 0; q < Ring::RING - 1; ++q) fetch(c0 - 2 + q);
    for (int i = c0 - 2; i < c1 + 2; ++i) {
        Ring g{reinterpret_cast<unsigned char*>(sm) + rd * Ring::BYTES};
        if constexpr (Ring::RING > 0) {
            fetch(i + Ring::RING - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(Ring::RING > 0 ? Ring::RING - 1 : 0) : "memory");
            rd = rd + 1 == Ring::RING ? 0 : rd + 1;
        }
        for (int s = 0; s < 4; ++s) {
            Av[s] = Av[s + 1]; Bv[s] = Bv[s + 1]; Cv[s] = Cv[s + 1]; Cp[s] = Cp[s + 1];
            Ae[s] = Ae[s + 1]; Be[s] = Be[s + 1];
        }
        const size_t o = (size_t)i * P + pair;
        CT pa, uv, uw, vw, pb;
        double2 Ud, Vd, Wd, Hv, He;
        const int j = i - 2;
        if constexpr (Ring::RING > 0) {
            pa = g.prod(0); uv = g.prod(1); uw = g.prod(2); vw = g.prod(3); pb = g.prod(4);
            Ud = g.field(0); Vd = g.field(1); Wd = g.field(2);
            Hv = g.memory(0); He = g.memory(1);
        } else {
            pa = prod[o]; uv = prod[o + PS]; uw = prod[o + 2 * PS]; vw = prod[o + 3 * PS]; pb = prod[o + 4 * PS];
            Ud = fu[o]; Vd = fv[o]; Wd = fw[o];
        }
        const CT U = from_d2<CT>(Ud), V = from_d2<CT>(Vd), W = from_d2<CT>(Wd);
        if constexpr (MODE == 1) {
            const float2 cx = g.coef(0), c1x = g.coef(1);
            inner_terms(pa, uv, uw, vw, pb, U, V, W, d.rinvf[i], cx.x, c1x.x, mt, at, nut, Av[4], Bv[4], Cv[4], Ae[4], Be[4]);
            // phi = i alpha u + (i m/r) w, times c', in double-float
            const dcomplex phi = dc_i(dc_fma(dc_scale(alD, dc_bits(Ud)), mD * rinvx[i], dc_bits(Wd)));
            Cp[4] = dc_scale(as_df(c1x), phi);
        } else {
            T ri, c, c1f;
            if constexpr (MODE == 2) { ri = as_df(d.rinvx[i]); c = as_df(g.coef(0)); c1f = as_df(g.coef(1)); }
            else { ri = d.rinv[i]; c = d.tab_c[o]; c1f = d.tab_c1[o]; }
            inner_terms_shared(pa, uv, uw, vw, pb, U, V, W, ri, c, c1f, mt, at, at2, nu2, nu3, Av[4], Bv[4], Cv[4], Ae[4],
                               Be[4]);
        }
        if (j < c0) continue;
        if constexpr (Ring::RING == 0) { Hv = d.Hv[o - 2 * P]; He = d.He[o - 2 * P]; }
        vrow(j, Hv);
        erow(j, He);
        if (j == 2) erow(1, d.He[P + pair]);
        if (j == N - 3) erow(N - 2, d.He[(size_t)(N - 2) * P + pair]);
    }
}

// Recurrences over n rows whose loads do not depend on them: the loads of four
// rows stay ahead of the four rows being computed.  (A ring of eight rows, each
// loaded as its registers come free, was slower, 13.2 -> 14.1 ms of the line phase at
// 257x512x512: more loads in flight than a warp has scoreboards to tell apart, so that
// waiting for a row waits for later ones.)
template <typename D, int B = 4, typename Load, typename Step>
__device__ __forceinline__ void rows_ahead(int n, Load load, Step step) {
    D cur[B], nxt[B];
#pragma unroll
    for (int q = 0; q < B; ++q)
        if (q < n) load(q, cur[q]);
    for (int b = 0; b < n; b += B) {
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (b + B + q < n) load(b + B + q, nxt[q]);
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (b + q < n) step(b + q, cur[q]);
#pragma unroll
        for (int q = 0; q < B; ++q) cur[q] = nxt[q];
    }
}
struct FwdRow { double r, m2, m1; };
struct BackRow { double y, inv, c, e; };
struct OneRow { double z; };
struct MeanRow { double y, a, b, inv; };

// The banded solve of one component of one field (right sides of rows 1 .. Nr - 2
// from rhs(j)), y and then x in f (rows P2 apart), the conjugate with sign `cj` in
// g unless null.  Returns false if a value is not finite.
template <typename Rhs>
__device__ __forceinline__ bool band_solve(const TcDev& d, const double* __restrict__ lu, int k, int pair, double* f, double* g,
                                           double cj, Rhs rhs) {
    const int N = d.Nr;
    const size_t P2 = 2 * (size_t)d.npairs;
    double y1 = 0.0, y2 = 0.0;                  // y_(j-1), y_(j-2)
    rows_ahead<FwdRow>(
        N - 2,
        [&](int q, FwdRow& w) {
            const int j = q + 1;
            w.r = rhs(j);
            w.m2 = TAB(lu, k, j, 0);
            w.m1 = TAB(lu, k, j, 1);
        },
        [&](int q, const FwdRow& w) {
            const double y = fma(-w.m1, y1, fma(-w.m2, y2, w.r));
            f[(size_t)(q + 1) * P2] = y;
            y2 = y1; y1 = y;
        });
    bool ok = true;
    double x1 = 0.0, x2 = 0.0;                  // x_(i+1), x_(i+2)
    rows_ahead<BackRow>(
        N - 2,
        [&](int q, BackRow& w) {
            const int i = N - 2 - q;
            w.y = f[(size_t)i * P2];
            w.inv = TAB(lu, k, i, 2);
            w.c = TAB(lu, k, i, 3);
            w.e = TAB(lu, k, i, 4);
        },
        [&](int q, const BackRow& w) {
            const int i = N - 2 - q;
            const double x = w.inv * fma(-w.e, x2, fma(-w.c, x1, w.y));
            ok = ok && dfinite(x);
            f[(size_t)i * P2] = x;
            if (g) g[(size_t)i * P2] = cj * x;
            x2 = x1; x1 = x;
        });
    f[0] = 0.0;
    f[(size_t)(N - 1) * P2] = 0.0;
    if (g) { g[0] = 0.0; g[(size_t)(N - 1) * P2] = 0.0; }
    return ok;
}

// l1 . v on the rows i0 <= i < i1 of 1 .. Nr - 2 (one-sided on the first and the
// last: Dv itself), into S: the right sides of the Dv solve.
__device__ __forceinline__ void derivative_rows(const TcDev& d, const RowTables& t, const double* v, double* S, int i0, int i1) {
    const int N = d.Nr;
    const size_t P2 = 2 * (size_t)d.npairs, S2 = 2 * (size_t)d.Mzx * d.Nh;
    i0 = i0 < 2 ? 2 : i0;
    i1 = i1 > N - 2 ? N - 2 : i1;
    if (i0 >= i1) return;
    double x[5];
    for (int s = 0; s < 4; ++s) x[s + 1] = v[(i0 - 2 + s) * P2];
    auto row = [&](int j) {
        double acc = 0.0;
        for (int s = 0; s < 5; ++s) acc = fma(t.l1[j * 5 + s], x[s], acc);
        S[(size_t)j * S2] = acc;
    };
    for (int i = i0; i < i1; ++i) {
        for (int s = 0; s < 4; ++s) x[s] = x[s + 1];
        x[4] = v[(i + 2) * P2];
        row(i);
        if (i == 2) row(1);
        if (i == N - 3) row(N - 2);
    }
}
// Dv in S: 0 on the walls; explicit one-sided rows 1 and Nr - 2 (there already);
// compact rows d0 . Dv = l1 . v on rows 2 .. Nr - 3, solved with the reversed
// factorisation dsol, whose elimination runs from the outer wall in.
__device__ __forceinline__ void derivative_solve(const TcDev& d, const RowTables& t, double* S) {
    const int N = d.Nr;
    const size_t S2 = 2 * (size_t)d.Mzx * d.Nh;
    const double D1 = S[S2], DN = S[(size_t)(N - 2) * S2];
    double z1 = 0.0, z2 = 0.0;
    rows_ahead<OneRow>(
        N - 4, [&](int q, OneRow& w) { w.z = S[(size_t)(N - 3 - q) * S2]; },
        [&](int q, const OneRow& w) {
            const int j = N - 3 - q;
            const double* w0 = t.d0 + j * 5;
            double r = w.z;
            if (j == N - 3) r = fma(-w0[3], DN, r);
            if (j == N - 4) r = fma(-w0[4], DN, r);
            if (j == 2) r = fma(-w0[1], D1, r);
            if (j == 3) r = fma(-w0[0], D1, r);
            const double* c = t.dsol + j * 5;
            const double z = fma(-c[1], z1, fma(-c[0], z2, r));
            S[(size_t)j * S2] = z;
            z2 = z1; z1 = z;
        });
    double p1 = 0.0, p2 = 0.0;
    rows_ahead<OneRow>(
        N - 4, [&](int q, OneRow& w) { w.z = S[(size_t)(q + 2) * S2]; },
        [&](int q, const OneRow& w) {
            const double* c = t.dsol + (q + 2) * 5;
            const double Dv = c[2] * fma(-c[4], p2, fma(-c[3], p1, w.z));
            S[(size_t)(q + 2) * S2] = Dv;
            p2 = p1; p1 = Dv;
        });
    S[0] = 0.0;
    S[(size_t)(N - 1) * S2] = 0.0;
}
// u = (i alpha D_*v - (i m/r) eta)/k^2,   w = ((i m/r) D_*v + i alpha eta)/k^2 on the
// rows i0 <= i < i1: the factor i takes each lane's value to the other component.
__device__ __forceinline__ void velocity_rows(const TcDev& d, const RowTables& t, int pair, int comp, double m, double al,
                                              long long partner, const double* S, int i0, int i1) {
    const size_t P = d.npairs, P2 = 2 * P, S2 = 2 * (size_t)d.Mzx * d.Nh;
    const size_t o = 2 * (size_t)pair + comp, x = 2 * (size_t)pair + 1 - comp;
    const double *v = reinterpret_cast<const double*>(d.v) + o, *e = reinterpret_cast<const double*>(d.eta) + o;
    double *u = reinterpret_cast<double*>(d.u), *w = reinterpret_cast<double*>(d.w);
    for (int i = i0; i < i1; ++i) {
        const double ri = t.rinv[i], c = d.tab_c[(size_t)i * P + pair];
        const double Dsv = fma(ri, v[(size_t)i * P2], S[(size_t)i * S2]), E = e[(size_t)i * P2];
        const double ca = c * al, cm = c * m * ri;
        const double su = fma(ca, Dsv, -cm * E), sw = fma(cm, Dsv, ca * E);
        u[x + (size_t)i * P2] = comp ? -su : su;
        w[x + (size_t)i * P2] = comp ? -sw : sw;
        if (partner >= 0) {
            u[2 * (size_t)partner + 1 - comp + (size_t)i * P2] = -su;
            w[2 * (size_t)partner + 1 - comp + (size_t)i * P2] = -sw;
        }
    }
}

template <bool NOH>
__device__ __forceinline__ void solve_body(const TcDev& d, int k, int ja, int jw, int block) {
    const int warp = threadIdx.x >> 5, comp = threadIdx.x & 1;
    int pair = 0;
    double m = 0.0, al = 0.0;
    long long partner = -1;
    const bool act = line_pair(d, ja, jw, block * 16 + ((threadIdx.x & 31) >> 1), pair, m, al, partner);
    const int N = d.Nr;
    const RowTables t{d.d0, d.l1, d.dsol, d.rinv};
    const size_t o = 2 * (size_t)pair + comp, P2 = 2 * (size_t)d.npairs, S2 = 2 * (size_t)d.Mzx * d.Nh;
    double* S = reinterpret_cast<double*>(rhs_scratch(d, pair)) + comp;
    double* const v = reinterpret_cast<double*>(d.v) + o;
    if (act) {
        const double cj = comp ? -1.0 : 1.0;
        bool ok;
        if (warp == 0) {
            const double fv = TAB(d.tab_luv, k, 0, 0), gv = TAB(d.tab_luv, k, N - 1, 0);
            ok = band_solve(d, d.tab_luv, k, pair, v, partner >= 0 ? reinterpret_cast<double*>(d.v) + 2 * partner + comp : nullptr, cj,
                            [&](int j) { return j == 1 ? -fv * S[2 * S2] : j == N - 2 ? -gv * S[(size_t)(N - 3) * S2] : S[(size_t)j * S2]; });
        } else {
            double* const e = reinterpret_cast<double*>(d.eta) + o;
            const double fe = TAB(d.tab_lue, k, 0, 0), ge = TAB(d.tab_lue, k, N - 1, 0);
            // the folded right sides, before y overwrites the rows they use
            const double e1 = fma(-fe, e[2 * P2], e[P2]), eN = fma(-ge, e[(size_t)(N - 3) * P2], e[(size_t)(N - 2) * P2]);
            ok = band_solve(d, d.tab_lue, k, pair, e, partner >= 0 ? reinterpret_cast<double*>(d.eta) + 2 * partner + comp : nullptr, cj,
                            [&](int j) { return j == 1 ? e1 : j == N - 2 ? eN : e[(size_t)j * P2]; });
        }
        if (!ok) atomicOr(d.flag, 1);
    }
    const int i0 = warp * N / 2, i1 = (warp + 1) * N / 2;      // the warp's share of the radial rows
    __syncthreads();
    if (act) derivative_rows(d, t, v, S, i0, i1);
    __syncthreads();
    if (act && warp == 0) derivative_solve(d, t, S);
    __syncthreads();
    if (act) {
        if (!NOH) rk_memory_rows(d, k, pair, comp, i0, i1);
        velocity_rows(d, t, pair, comp, m, al, partner, S, i0, i1);
    }
}

// The same for few pairs: eight warps, of which the recurrences still have one each, so
// that what counts is the time of one row of them.  The factors come through a ring in
// shared memory (cp.async, 16 rows deep: the latency of a load is several rows), and
// what one sweep leaves for the next (y, x, the right sides and z of the Dv solve)
// stays in shared memory.  Same operations, same bits.  Line phase of
// 129x128x128 623 -> 536 us, mixed form 437 -> 350.
constexpr int SOLVE_WARPS = 8, RING_ROWS = 16;
struct DvRow { double z, a, b, c; };
struct RkRow { double tv[5], te[5], Hv, He, e; };
struct VelRow { double c, e; };
// n rows of three words each per lane, p[w] + row stride[w], four rows at a time.  A
// lone warp issues an instruction every few cycles, so the sources are pointers that
// advance, not indexed tables.
struct Ring3 { const double* p[3]; long long stride[3]; };
template <typename Step> __device__ __forceinline__ void ring_rows(double* ring, int n, Ring3 s, Step step) {
    constexpr int B = 4, NB = RING_ROWS / B;
    double* const mine = ring + (threadIdx.x & 31);
    int left = n;
    auto issue = [&](int slot) {
        double* o = mine + slot * (B * 96);
#pragma unroll
        for (int q = 0; q < B; ++q) {
            if (q < left)
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    copy_async<8>(o + (q * 3 + w) * 32, s.p[w]);
                    s.p[w] += s.stride[w];
                }
        }
        left -= B;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int b = 0; b < NB - 1; ++b) issue(b);
    for (int b = 0; b < n; b += B) {
        issue((b / B + NB - 1) % NB);
        asm volatile("cp.async.wait_group %0;" ::"n"(NB - 1) : "memory");
        const double* o = mine + (b / B % NB) * (B * 96);
        double w[B][3];
#pragma unroll
        for (int q = 0; q < B; ++q)
#pragma unroll
            for (int t = 0; t < 3; ++t) w[q][t] = o[(q * 3 + t) * 32];
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (b + q < n) step(b + q, w[q]);
    }
}
// band_solve on the ring: right sides at r + j S2 but r1 and rN for rows 1 and Nr - 2; y
// and then x in Y, x in f as well
__device__ __forceinline__ bool band_solve_shared(const TcDev& d, const double* __restrict__ lu, int k, int pair, double* ring, double* Y,
                                                  double* f, double* g, double cj, const double* r, size_t S2, double r1, double rN) {
    const int N = d.Nr;
    const long long P = d.npairs, P2 = 2 * P;
    double y1 = 0.0, y2 = 0.0;
    double* Yq = Y + 32;
    const double* l = &TAB(lu, k, 1, 0);
    ring_rows(ring, N - 2, Ring3{{r + S2, l, l + P}, {(long long)S2, 5 * P, 5 * P}}, [&](int q, const double* w) {
        const double b = q == 0 ? r1 : q == N - 3 ? rN : w[0];
        const double y = fma(-w[2], y1, fma(-w[1], y2, b));
        *Yq = y;
        Yq += 32;
        y2 = y1; y1 = y;
    });
    unsigned top = 0;                           // largest exponent field
    double x1 = 0.0, x2 = 0.0;
    f += (N - 2) * P2;
    if (g) g += (N - 2) * P2;
    l = &TAB(lu, k, N - 2, 2);
    ring_rows(ring, N - 2, Ring3{{l, l + P, l + 2 * P}, {-5 * P, -5 * P, -5 * P}}, [&](int q, const double* w) {
        Yq -= 32;
        const double x = w[0] * fma(-w[2], x2, fma(-w[1], x1, *Yq));
        const unsigned ex = (unsigned)__double2hiint(x) & 0x7ff00000u;
        top = ex > top ? ex : top;
        *Yq = x;
        *f = x;
        f -= P2;
        if (g) { *g = cj * x; g -= P2; }
        x2 = x1; x1 = x;
    });
    Y[0] = Y[(N - 1) * 32] = 0.0;
    f[0] = f[(N - 1) * P2] = 0.0;
    if (g) g[0] = g[(N - 1) * P2] = 0.0;
    return top != 0x7ff00000u;
}
template <bool NOH>
__device__ __forceinline__ void solve_shared_body(const TcDev& d, int k, int ja, int jw, int block) {
    extern __shared__ double sm[];
    const int N = d.Nr, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, comp = threadIdx.x & 1;
    double *const d0 = sm, *const l1 = d0 + 5 * N, *const dsol = l1 + 5 * N, *const rinv = dsol + 5 * N;
    double *const V = rinv + N + lane, *const D = V + 32 * N;               // D: y of eta before
    double* const ring = rinv + N + 64 * N + warp * RING_ROWS * 96;         // of warps 0 and 1
    for (int i = threadIdx.x; i < 5 * N; i += 32 * SOLVE_WARPS) { d0[i] = d.d0[i]; l1[i] = d.l1[i]; dsol[i] = d.dsol[i]; }
    for (int i = threadIdx.x; i < N; i += 32 * SOLVE_WARPS) rinv[i] = d.rinv[i];
    int pair = 0;
    double m = 0.0, al = 0.0;
    long long partner = -1;
    const bool act = line_pair(d, ja, jw, block * 16 + (lane >> 1), pair, m, al, partner);
    const size_t P = d.npairs, P2 = 2 * P, S2 = 2 * (size_t)d.Mzx * d.Nh, o = 2 * (size_t)pair + comp;
    const double* S = reinterpret_cast<const double*>(rhs_scratch(d, pair)) + comp;
    double *const v = reinterpret_cast<double*>(d.v) + o, *const e = reinterpret_cast<double*>(d.eta) + o;
    if (act && warp < 2) {
        const double cj = comp ? -1.0 : 1.0;
        bool ok;
        if (warp == 0) {
            const double r1 = -TAB(d.tab_luv, k, 0, 0) * S[2 * S2], rN = -TAB(d.tab_luv, k, N - 1, 0) * S[(size_t)(N - 3) * S2];
            ok = band_solve_shared(d, d.tab_luv, k, pair, ring, V, v, partner >= 0 ? reinterpret_cast<double*>(d.v) + 2 * partner + comp : nullptr,
                                   cj, S, S2, r1, rN);
        } else {
            const double fe = TAB(d.tab_lue, k, 0, 0), ge = TAB(d.tab_lue, k, N - 1, 0);
            const double e1 = fma(-fe, e[2 * P2], e[P2]), eN = fma(-ge, e[(size_t)(N - 3) * P2], e[(size_t)(N - 2) * P2]);
            ok = band_solve_shared(d, d.tab_lue, k, pair, ring, D, e, partner >= 0 ? reinterpret_cast<double*>(d.eta) + 2 * partner + comp : nullptr,
                                   cj, e, P2, e1, eN);
        }
        if (!ok) atomicOr(d.flag, 1);
    }
    __syncthreads();
    // l1 . v
    for (int j = 1 + warp; j < N - 1; j += SOLVE_WARPS) {
        const int st = j == 1 ? 0 : j == N - 2 ? N - 5 : j - 2;
        double acc = 0.0;
        for (int s = 0; s < 5; ++s) acc = fma(l1[j * 5 + s], V[(st + s) * 32], acc);
        D[j * 32] = acc;
    }
    __syncthreads();
    // the Dv recurrences, the RK memory beside them
    if (warp == 0) {
        const double D1 = D[32], DN = D[(N - 2) * 32];
        double *Dq = D + (N - 3) * 32, *q = dsol + (N - 3) * 5;
        D[(N - 3) * 32] = fma(-d0[(N - 3) * 5 + 3], DN, D[(N - 3) * 32]);
        D[(N - 4) * 32] = fma(-d0[(N - 4) * 5 + 4], DN, D[(N - 4) * 32]);
        D[64] = fma(-d0[11], D1, D[64]);
        D[96] = fma(-d0[15], D1, D[96]);
        double z1 = 0.0, z2 = 0.0;
        rows_ahead<DvRow>(
            N - 4,
            [&](int, DvRow& w) {
                w.z = *Dq; w.a = q[0]; w.b = q[1];
                Dq -= 32; q -= 5;
            },
            [&](int r, const DvRow& w) {
                const double z = fma(-w.b, z1, fma(-w.a, z2, w.z));
                D[(N - 3 - r) * 32] = z;
                z2 = z1; z1 = z;
            });
        double p1 = 0.0, p2 = 0.0;
        Dq = D + 64;
        q = dsol + 10;
        rows_ahead<DvRow>(
            N - 4,
            [&](int, DvRow& w) {
                w.z = *Dq; w.a = q[2]; w.b = q[3]; w.c = q[4];
                Dq += 32; q += 5;
            },
            [&](int r, const DvRow& w) {
                const double x = w.a * fma(-w.c, p2, fma(-w.b, p1, w.z));
                D[(2 + r) * 32] = x;
                p2 = p1; p1 = x;
            });
        D[0] = D[(N - 1) * 32] = 0.0;
    } else if (act && !NOH) {
        const int n = SOLVE_WARPS - 1, i0 = 2 + (warp - 1) * (N - 4) / n, i1 = 2 + warp * (N - 4) / n;
        const double hdt = (d.rk_beta[k] + d.rk_alpha[(k + 1) % 3]) * d.dt, hdtnu = hdt * d.nu;
        double *Hv = reinterpret_cast<double*>(d.Hv) + o, *He = reinterpret_cast<double*>(d.He) + o;
        double xe[5];
        if (i0 < i1)
            for (int s = 0; s < 4; ++s) xe[s + 1] = e[(i0 - 2 + s) * P2];
        rows_ahead<RkRow, 1>(
            i1 - i0,
            [&](int q, RkRow& w) {
                const int i = i0 + q;
#pragma unroll
                for (int s = 0; s < 5; ++s) { w.tv[s] = TAB(d.tab_lv, 0, i, s); w.te[s] = TAB(d.tab_le, 0, i, s); }
                w.Hv = Hv[(size_t)i * P2];
                w.He = He[(size_t)i * P2];
                w.e = e[(size_t)(i + 2) * P2];
            },
            [&](int q, const RkRow& w) {
                const int i = i0 + q;
                for (int s = 0; s < 4; ++s) xe[s] = xe[s + 1];
                xe[4] = w.e;
                double av = 0.0, ae = 0.0;
#pragma unroll
                for (int s = 0; s < 5; ++s) { av = fma(w.tv[s], V[(i - 2 + s) * 32], av); ae = fma(w.te[s], xe[s], ae); }
                Hv[(size_t)i * P2] = fma(hdt, av, w.Hv);
                He[(size_t)i * P2] = fma(hdtnu, ae, w.He);
                if (i == 2) rk_memory_row(d, d.tab_le, He, pair, 1, xe, hdtnu);
                if (i == N - 3) rk_memory_row(d, d.tab_le, He, pair, N - 2, xe, hdtnu);
            });
    }
    __syncthreads();
    if (!act) return;
    // u and w: as in velocity_rows
    const size_t x = 2 * (size_t)pair + 1 - comp;
    double *u = reinterpret_cast<double*>(d.u), *w = reinterpret_cast<double*>(d.w);
    const int n = (N - warp + SOLVE_WARPS - 1) / SOLVE_WARPS;
    rows_ahead<VelRow, 2>(
        n,
        [&](int q, VelRow& r) {
            const size_t i = warp + q * SOLVE_WARPS;
            r.c = d.tab_c[i * P + pair];
            r.e = e[i * P2];
        },
        [&](int q, const VelRow& r) {
            const size_t i = warp + q * SOLVE_WARPS;
            const double ri = rinv[i];
            const double Dsv = fma(ri, V[i * 32], D[i * 32]);
            const double ca = r.c * al, cm = r.c * m * ri;
            const double su = fma(ca, Dsv, -cm * r.e), sw = fma(cm, Dsv, ca * r.e);
            u[x + i * P2] = comp ? -su : su;
            w[x + i * P2] = comp ? -sw : sw;
            if (partner >= 0) {
                u[2 * (size_t)partner + 1 - comp + i * P2] = -su;
                w[2 * (size_t)partner + 1 - comp + i * P2] = -sw;
            }
        });
}
static size_t solve_smem(int Nr) { return (80 * (size_t)Nr + 2 * RING_ROWS * 96) * sizeof(double); }
// Which of the two: up to WIDE_GROUPS blocks of 16 pairs.  Line phase with
// two and with eight warps: 512 blocks (129x128x128) 623 and 536 us, 2720 (129x512x170)
// 2.39 and 2.47 ms, 8192 (257x512x512) 13.4 and 19.2 ms.
constexpr long long WIDE_GROUPS = 8 * 152;
static bool solve_wide(long long groups, int Nr) { return groups < WIDE_GROUPS && solve_smem(Nr) <= 200 * 1024; }

// The implicit part of the next RK memory (rk_memory_row) for the pairs of
// the columns ja .. ja + jw - 1, after a k_solve of substep k launched with NOH.  It
// needs only the results of that kernel, so it can run beside the next substep's
// plane phase.
// Grid-stride over the pairs: launched beside the theta rows it runs in few
// blocks (four per SM), so that it takes mostly what the rows leave free.
// What bounds it there is the float64 pipe, so a thread walks a pair's whole line with
// both components, and the eta band, formed with the table's own operations (where the
// pipe has more time to spare than the memory), serves both: 32 operations a point
// against 40 with a lane per component, 2.31 -> 2.06 ms alone at 257x512x512.  Step of
// the mixed form there: 38.9 -> 37.25 ms (solves with the RK memory in them: 39.0; with
// the band read here: 38.8); of 129x512x170: 7.66 -> 7.45 (7.73).
__global__ void __launch_bounds__(128) k_rk_memory(const __grid_constant__ TcDev d, int k, int ja, int jw) {
    const int N = d.Nr, kn = (k + 1) % 3, n = d.Nz * jw;
    const size_t P = d.npairs;
    const double hdt = (d.rk_beta[k] + d.rk_alpha[kn]) * d.dt, hdtnu = hdt * d.nu;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
        int pair;
        double m, al;
        long long partner;
        if (!line_pair(d, ja, jw, idx, pair, m, al, partner)) continue;
        const double2 *v = d.v + pair, *e = d.eta + pair;
        double2 xv[5], xe[5];
        double k2[5];
        for (int s = 0; s < 4; ++s) { xv[s + 1] = v[s * P]; xe[s + 1] = e[s * P]; k2[s + 1] = k2_at(m, al, d.rinv[s]); }
        auto eta_row = [&](int j) {
            double2 acc = cz();
            for (int s = 0; s < 5; ++s) acc = caxpy(acc, fma(-d.d0[j * 5 + s], k2[s], d.l2[j * 5 + s]), xe[s]);
            double2* H = d.He + (size_t)j * P + pair;
            *H = caxpy(*H, hdtnu, acc);
        };
        for (int i = 2; i < N - 2; ++i) {
            for (int s = 0; s < 4; ++s) { xv[s] = xv[s + 1]; xe[s] = xe[s + 1]; k2[s] = k2[s + 1]; }
            xv[4] = v[(i + 2) * P];
            xe[4] = e[(i + 2) * P];
            k2[4] = k2_at(m, al, d.rinv[i + 2]);
            double2 acc = cz();
            for (int s = 0; s < 5; ++s) acc = caxpy(acc, TAB(d.tab_lv, 0, i, s), xv[s]);
            double2* H = d.Hv + (size_t)i * P + pair;
            *H = caxpy(*H, hdt, acc);
            eta_row(i);
            if (i == 2) eta_row(1);
            if (i == N - 3) eta_row(N - 2);
        }
    }
}

// ---------------------------------------------------------------------------
// Initial RK memory H_1 = (M + alpha_1 dt L) x for v and eta, and u, w, as k_solve
// after its solves: the rows i0 <= i < i1 of H_1, both components by one thread, since
// the bands cost more than the sums with them.  The one-sided eta rows 1 and Nr - 2 go
// with their neighbours.
__device__ __forceinline__ void init_rows(const TcDev& d, int pair, double m, double al, int i0, int i1) {
    const int N = d.Nr;
    const size_t P = d.npairs;
    const double adt = d.rk_alpha[0] * d.dt;
    const double2 *v = d.v + pair, *e = d.eta + pair;
    double2 *Hv = d.Hv + pair, *He = d.He + pair;
    if (i0 == 0) Hv[0] = Hv[P] = He[0] = cz();
    if (i1 == N) Hv[(size_t)(N - 2) * P] = Hv[(size_t)(N - 1) * P] = He[(size_t)(N - 1) * P] = cz();
    i0 = i0 < 2 ? 2 : i0;
    i1 = i1 > N - 2 ? N - 2 : i1;
    if (i0 >= i1) return;
    double c[5], c1[5], k2[5];                  // 1/k^2, its derivative and k^2 at the row's points
    double2 xv[5], xe[5];
    auto point = [&](int i) {
        for (int s = 0; s < 4; ++s) { c[s] = c[s + 1]; c1[s] = c1[s + 1]; k2[s] = k2[s + 1]; xv[s] = xv[s + 1]; xe[s] = xe[s + 1]; }
        const size_t o = (size_t)i * P;
        const double ri = d.rinv[i];
        c[4] = d.tab_c[o + pair];
        c1[4] = d.tab_c1 ? d.tab_c1[o + pair] : coef_at(d.r[i], ri, m, al).c1;
        k2[4] = al * al + m * m * ri * ri;
        xv[4] = v[o];
        xe[4] = e[o];
    };
    auto eta_row = [&](int j) {
        double2 h = cz();
        for (int s = 0; s < 5; ++s) {
            const double L5 = d.nu * (d.l2[j * 5 + s] - d.d0[j * 5 + s] * k2[s]);
            h = caxpy(h, d.d0[j * 5 + s] + adt * L5, xe[s]);
        }
        He[(size_t)j * P] = h;
    };
    for (int i = i0 - 2; i < i0 + 2; ++i) point(i);
    for (int j = i0; j < i1; ++j) {
        point(j + 2);
        double2 h = cz();
        for (int s = 0; s < 5; ++s) {           // mass band M = d0 - l2 c + l1 c'
            const double M5 = d.d0[j * 5 + s] - d.l2[j * 5 + s] * c[s] + d.l1[j * 5 + s] * c1[s];
            h = caxpy(h, M5 + adt * TAB(d.tab_lv, 0, j, s), xv[s]);
        }
        Hv[(size_t)j * P] = h;
        eta_row(j);
        if (j == 2) eta_row(1);
        if (j == N - 3) eta_row(N - 2);
    }
}
// One warp solves for Dv, the others take the rows of H_1.  Bound by the float64 pipe
// (94 operations a pair and row).  257x512x512: 6.16 ms with four warps (two: 6.37; a
// lane per component of a row, which formed the bands twice and, in the double-float
// form, c' five times a row: 9.1 and in that form 15.4, now 6.94); 129x512x170: 1.63 ->
// 1.06 and 2.62 -> 1.20; 129x128x128, eight warps: 0.36 -> 0.27 and 0.59 -> 0.31.
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS, WARPS > 4 ? 2 : 4) k_init(const __grid_constant__ TcDev d) {
    const int warp = threadIdx.x >> 5, comp = threadIdx.x & 1;
    int pair = 0;
    double m = 0.0, al = 0.0;
    long long partner = -1;
    const bool act = line_pair(d, 0, d.Nh, blockIdx.x * 16 + ((threadIdx.x & 31) >> 1), pair, m, al, partner);
    const RowTables t{d.d0, d.l1, d.dsol, d.rinv};
    double* S = reinterpret_cast<double*>(rhs_scratch(d, pair)) + comp;
    const int N = d.Nr;
    if (act) derivative_rows(d, t, reinterpret_cast<const double*>(d.v) + 2 * (size_t)pair + comp, S, warp * N / WARPS, (warp + 1) * N / WARPS);
    __syncthreads();
    if (act) {
        if (warp == 0) derivative_solve(d, t, S);
        else {                              // the pair's two lanes take half of the rows each
            const int w = 2 * (warp - 1) + comp;
            init_rows(d, pair, m, al, w * N / (2 * WARPS - 2), (w + 1) * N / (2 * WARPS - 2));
        }
    }
    __syncthreads();
    if (act) velocity_rows(d, t, pair, comp, m, al, partner, S, warp * N / WARPS, (warp + 1) * N / WARPS);
}

// ---------------------------------------------------------------------------
// Mean flow (m = alpha = 0), zero mean pressure gradient (Sec. 4):
//   dW/dt = nu D D_* W - D(vw) - 2 vw/r,   dU/dt = nu (D D_* U + U/r^2) - D(uv) - uv/r,
// rows 1..Nr-2 with Dirichlet values W(R_i) = 1, W(R_o) = Re_o/Re_i, U = 0.
// One block: the right sides in parallel, then one thread each for U and W runs
// the banded solve with the factors of mean_lu (the system is the same in every
// step), from shared memory: the recurrences are the latency of a few thousand
// dependent operations, so nothing else is left in them.
__device__ __forceinline__ void mean_L(const TcDev& d, int j, int s, double& lu, double& lw) {
    const double w0 = d.d0[j * 5 + s], w2 = d.l2[j * 5 + s], ri = d.rinv[d.start[j] + s];
    lu = d.nu * (w2 + w0 * ri * ri);
    lw = d.nu * w2;
}
// H_1 = (M + alpha_1 dt L) x, and u(0,0) = U, w(0,0) = W
__global__ void __launch_bounds__(256) k_mean_init(TcDev d) {
    const int N = d.Nr;
    const double adt = d.rk_alpha[0] * d.dt;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        double hu = 0.0, hw = 0.0;
        if (j >= 1 && j <= N - 2) {
            const int st = d.start[j];
            for (int s = 0; s < 5; ++s) {
                double lu, lw;
                mean_L(d, j, s, lu, lw);
                hu += (d.d0[j * 5 + s] + adt * lu) * d.U[st + s];
                hw += (d.d0[j * 5 + s] + adt * lw) * d.W[st + s];
            }
        }
        d.HU[j] = hu;
        d.HW[j] = hw;
        d.u[(size_t)j * d.npairs] = make_double2(d.U[j], 0.0);
        d.w[(size_t)j * d.npairs] = make_double2(d.W[j], 0.0);
    }
}
template <typename PT>
__device__ __forceinline__ void mean_body(const TcDev& d, int k) {
    extern __shared__ double sm[];
    const int N = d.Nr;
    double* lu = sm;                   // [2][N][5] factors of this substep
    double* rhs = lu + 2 * N * 5;      // [2][N]
    double* x = rhs + 2 * N;           // [2][N]
    const PT* prod = reinterpret_cast<const PT*>(d.prod);
    const size_t PS = (size_t)N * d.npairs;
    const int kn = (k + 1) % 3;
    const double bdt = d.rk_beta[k] * d.dt;
    const double gdt = d.rk_gamma[k] * d.dt, zdt = d.rk_zeta[kn] * d.dt;
    for (int i = threadIdx.x; i < 10 * N; i += blockDim.x) {
        const int p = i / (5 * N);
        lu[i] = d.mean_lu[(size_t)(p * 3 + k) * N * 5 + (i - p * 5 * N)];
    }
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        if (j < 1 || j > N - 2) continue;
        const int st = d.start[j];
        double eu = 0.0, ew = 0.0;
        for (int s = 0; s < 5; ++s) {
            const int i = st + s;
            const double w0 = d.d0[j * 5 + s], w1 = d.l1[j * 5 + s], ri = d.rinv[i];
            const double uv = ld_prod(prod, (size_t)i * d.npairs + PS).x;
            const double vw = ld_prod(prod, (size_t)i * d.npairs + 3 * PS).x;
            eu += -w1 * uv - w0 * uv * ri;
            ew += -w1 * vw - 2.0 * w0 * vw * ri;
        }
        double ru = d.HU[j] + gdt * eu, rw = d.HW[j] + gdt * ew;
        d.HU[j] = ru + zdt * eu;
        d.HW[j] = rw + zdt * ew;
        // the Dirichlet values W(r_0) = 1, W(r_(N-1)) = W_outer to the right side (U: 0)
        double a, b;
        if (st == 0) { mean_L(d, j, 0, a, b); rw -= d.d0[j * 5] - bdt * b; }
        if (st + 4 == N - 1) { mean_L(d, j, 4, a, b); rw -= (d.d0[j * 5 + 4] - bdt * b) * d.W_outer; }
        rhs[j] = ru;
        rhs[N + j] = rw;
    }
    __syncthreads();
    if (threadIdx.x % 32 == 0 && threadIdx.x / 32 < 2) {
        const int p = threadIdx.x / 32;
        const double* q = lu + p * N * 5;
        double* rp = rhs + p * N;
        double* xp = x + p * N;
        rp[1] -= q[0] * rp[2];                          // fold the one-sided rows
        rp[N - 2] -= q[(N - 1) * 5] * rp[N - 3];
        double y1 = 0, y2 = 0;
        rows_ahead<MeanRow>(
            N - 2, [&](int r, MeanRow& w) { w.y = rp[r + 1]; w.a = q[(r + 1) * 5]; w.b = q[(r + 1) * 5 + 1]; },
            [&](int r, const MeanRow& w) {
                const double y = fma(-w.b, y1, fma(-w.a, y2, w.y));
                xp[r + 1] = y;
                y2 = y1; y1 = y;
            });
        double x1 = 0, x2 = 0;
        rows_ahead<MeanRow>(
            N - 2,
            [&](int r, MeanRow& w) {
                const int i = N - 2 - r;
                w.y = xp[i]; w.a = q[i * 5 + 4]; w.b = q[i * 5 + 3]; w.inv = q[i * 5 + 2];
            },
            [&](int r, const MeanRow& w) {
                const double x = w.inv * fma(-w.a, x2, fma(-w.b, x1, w.y));
                xp[N - 2 - r] = x;
                x2 = x1; x1 = x;
            });
        xp[0] = p == 0 ? 0.0 : 1.0;
        xp[N - 1] = p == 0 ? 0.0 : d.W_outer;
    }
    __syncthreads();
    // H_(k+1) += (beta_k + alpha_(k+1)) dt L x, write the profiles
    const double hdt = (d.rk_beta[k] + d.rk_alpha[kn]) * d.dt;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        if (j >= 1 && j <= N - 2) {
            const int st = d.start[j];
            double su = 0.0, sw = 0.0;
            for (int s = 0; s < 5; ++s) {
                double a, b;
                mean_L(d, j, s, a, b);
                su += a * x[st + s];
                sw += b * x[N + st + s];
            }
            d.HU[j] += hdt * su;
            d.HW[j] += hdt * sw;
        }
        d.U[j] = x[j];
        d.W[j] = x[N + j];
        d.u[(size_t)j * d.npairs] = make_double2(x[j], 0.0);
        d.w[(size_t)j * d.npairs] = make_double2(x[N + j], 0.0);
    }
}
template <typename PT>
__global__ void __launch_bounds__(256) k_mean(TcDev d, int k) { mean_body<PT>(d, k); }
__device__ __forceinline__ void mean_any(const TcDev& d, int k) {
    if (d.prec == 1) mean_body<float2>(d, k);
    else if (d.prec == 2) mean_body<dcomplex>(d, k);
    else mean_body<double2>(d, k);
}

// The solves of 16 pairs a block; with `mean`, the last block advances the mean flow.
template <bool NOH>
__global__ void __launch_bounds__(64, 12) k_solve(const __grid_constant__ TcDev d, int k, int ja, int jw) {
    solve_body<NOH>(d, k, ja, jw, blockIdx.x);
}
template <bool NOH>
__global__ void __launch_bounds__(32 * SOLVE_WARPS, 2) k_solve_shared(const __grid_constant__ TcDev d, int k, int ja, int jw, bool mean) {
    if (mean && blockIdx.x == gridDim.x - 1) mean_any(d, k);
    else solve_shared_body<NOH>(d, k, ja, jw, blockIdx.x);
}
// Many cases of one form in one launch: bmap[block] = (case, 16 pairs of the case;
// -1: the case's mean flow)
__global__ void __launch_bounds__(64, 12) k_solve_b(const TcDev* __restrict__ ds, const int2* __restrict__ bmap, int k) {
    const int2 m = bmap[blockIdx.x];
    solve_body<false>(ds[m.x], k, 0, ds[m.x].Nh, m.y);
}
__global__ void __launch_bounds__(32 * SOLVE_WARPS, 2)
k_solve_shared_b(const TcDev* __restrict__ ds, const int2* __restrict__ bmap, int k) {
    const int2 m = bmap[blockIdx.x];
    const TcDev& d = ds[m.x];
    if (m.y < 0) mean_any(d, k);
    else solve_shared_body<false>(d, k, 0, d.Nh, m.y);
}

// The explicit rows, four warps a block: warp w of the launch takes chunk w % nch
// (Lc rows each) of the 32 pairs w / nch, so that the warps of a block mostly share
// the points at their chunks' ends.  With `mean`, the last block advances the mean
// flow, which needs the products only.  Three blocks per SM; the mixed form, with
// fewer registers, four (five steps of 129x128x128: 7.27 -> 7.01 ms).
template <int MODE>
__device__ __forceinline__ void explicit_body(const TcDev& d, int k, int ja, int jw, int Lc, int block) {
    const int nch = (d.Nr - 4 + Lc - 1) / Lc;
    const int w = block * EXPLICIT_WARPS + (threadIdx.x >> 5);
    const int pg = w / nch, c0 = 2 + (w - pg * nch) * Lc, c1 = min(c0 + Lc, d.Nr - 2);
    explicit_rows<MODE>(d, k, ja, jw, pg * 32 + (threadIdx.x & 31), c0, c1);
}
template <int MODE>
__global__ void __launch_bounds__(32 * EXPLICIT_WARPS, MODE == 1 ? 4 : 3)
k_explicit(const __grid_constant__ TcDev d, int k, int ja, int jw, int Lc, int mean) {
    if (mean && blockIdx.x == gridDim.x - 1) mean_body<typename LineTypes<MODE>::CT>(d, k);
    else explicit_body<MODE>(d, k, ja, jw, Lc, blockIdx.x);
}
// The same rows for few pairs (float64 form): a warp that forms the inner functions of
// all the points of its rows by itself repeats those of its neighbours, and at one or
// four rows a warp (64x32x64) that is half of its time.  Here a block takes 16 pairs,
// a lane per component, and 8 R rows; its warps share the inner functions of the
// 8 R + 4 points through shared memory.  Same operations per component as
// inner_terms_shared, same bits.  Line phase of
// 33x16x16 53 -> 47 us.
constexpr int WIDE_WARPS = 8;
struct PointRow { double p[5], u, v, w, c, c1; };
struct HRow { double v, e; };
__global__ void __launch_bounds__(32 * WIDE_WARPS, 2)
k_explicit_wide(const __grid_constant__ TcDev d, int k, int ja, int jw, int R) {
    extern __shared__ double sm[];
    const int N = d.Nr, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, comp = lane & 1;
    const int nch = (N - 4 + WIDE_WARPS * R - 1) / (WIDE_WARPS * R), grp = blockIdx.x / nch;
    const int c0 = 2 + (blockIdx.x - grp * nch) * WIDE_WARPS * R;
    const int c1 = c0 + WIDE_WARPS * R < N - 2 ? c0 + WIDE_WARPS * R : N - 2, np = c1 - c0 + 4;
    int pair = 0;
    double m = 0.0, al = 0.0;
    long long partner = -1;
    const bool act = line_pair(d, ja, jw, grp * 16 + (lane >> 1), pair, m, al, partner);
    const size_t P = d.npairs, P2 = 2 * P, PS2 = (size_t)N * P2, o0 = 2 * (size_t)pair + comp;
    const double* __restrict__ prod = reinterpret_cast<const double*>(d.prod) + o0;
    const double* __restrict__ fu = reinterpret_cast<const double*>(d.u) + o0;
    const double* __restrict__ fv = reinterpret_cast<const double*>(d.v) + o0;
    const double* __restrict__ fw = reinterpret_cast<const double*>(d.w) + o0;
    const double mt = m, at = al, at2 = at * at, nu2 = 2.0 * d.nu, nu3 = 3.0 * d.nu;
    // i z of a value whose components lie in the two lanes: the other's, negated in the real lane
    auto times_i = [&](double z) {
        const double o = __shfl_xor_sync(0xffffffffu, z, 1);
        return comp ? o : -o;
    };
    rows_ahead<PointRow, 2>(
        (np - warp + WIDE_WARPS - 1) / WIDE_WARPS,
        [&](int q, PointRow& x) {
            const size_t i = c0 - 2 + warp + q * WIDE_WARPS;
#pragma unroll
            for (int t = 0; t < 5; ++t) x.p[t] = prod[i * P2 + t * PS2];
            x.u = fu[i * P2]; x.v = fv[i * P2]; x.w = fw[i * P2];
            x.c = d.tab_c[i * P + pair];
            x.c1 = d.tab_c1[i * P + pair];
        },
        [&](int q, const PointRow& x) {
            const int s = warp + q * WIDE_WARPS;
            const double ri = d.rinv[c0 - 2 + s], c = x.c, c1f = x.c1;
            const double pa = x.p[0], uv = x.p[1], uw = x.p[2], vw = x.p[3], pb = x.p[4];
            const double mr = mt * ri, mr2 = mr * ri, mra = mr * at, n2 = nu2 * mr2;
            const double Q = fma(at, uv, mr * vw);
            const double Tm = fma(-n2, x.w, Q), Tp = fma(n2, x.w, Q);
            const double ph = fma(at, x.u, mr * x.w);
            const double Z = fma(nu3 * c1f, ph, c * Tm);
            const double Y = fma(-2.0 * c * mr2, vw, c1f * Tm);
            const double Rr = fma(mr * mr, pb, fma(2.0 * mra, uw, at2 * pa));
            const double Nn = fma(-n2, x.u, fma(-at, vw, mr * uv));
            double* o = sm + s * 160 + lane;
            o[0] = fma(ri, pb, -times_i(Tp));
            o[32] = fma(c, Rr, times_i(Y));
            o[64] = -times_i(Z);
            o[96] = fma(n2 * at, x.v, fma(fma(mr, mr, -at2), uw, mra * (pa - pb)));
            o[128] = -times_i(Nn);
        });
    double *Hv = reinterpret_cast<double*>(d.Hv) + o0, *He = reinterpret_cast<double*>(d.He) + o0;
    double *eta = reinterpret_cast<double*>(d.eta) + o0, *rhsv = reinterpret_cast<double*>(rhs_scratch(d, pair)) + comp;
    const size_t S2 = 2 * (size_t)d.Mzx * d.Nh;
    const double gdt = d.rk_gamma[k] * d.dt, zdt = d.rk_zeta[(k + 1) % 3] * d.dt;
    __syncthreads();
    if (!act) return;
    auto erow = [&](int j, int s, double H) {   // eta row j on the points s ..
        double E = 0.0;
#pragma unroll
        for (int t = 0; t < 5; ++t) {
            const double* x = sm + (s + t) * 160 + lane;
            E = fma(d.d0[j * 5 + t], x[96], E);
            E = fma(d.l1e[j * 5 + t], x[128], E);
        }
        const double r = fma(gdt, E, H);
        He[(size_t)j * P2] = fma(zdt, E, r);
        eta[(size_t)j * P2] = r;
    };
    rows_ahead<HRow, 2>(
        (c1 - c0 - warp + WIDE_WARPS - 1) / WIDE_WARPS,
        [&](int q, HRow& h) {
            const size_t j = c0 + warp + q * WIDE_WARPS;
            h.v = Hv[j * P2];
            h.e = He[j * P2];
        },
        [&](int q, const HRow& h) {
            const int s = warp + q * WIDE_WARPS, j = c0 + s;
            double E = 0.0;
#pragma unroll
            for (int t = 0; t < 5; ++t) {
                const double* x = sm + (s + t) * 160 + lane;
                E = fma(d.d0[j * 5 + t], x[0], E);
                E = fma(d.l1[j * 5 + t], x[32], E);
                E = fma(d.l2[j * 5 + t], x[64], E);
            }
            const double r = fma(gdt, E, h.v);
            Hv[(size_t)j * P2] = fma(zdt, E, r);
            rhsv[(size_t)j * S2] = r;
            erow(j, s, h.e);
            if (j == 2) erow(1, s, He[P2]);
            if (j == N - 3) erow(N - 2, s, He[(size_t)(N - 2) * P2]);
        });
}
// Many cases of one form in one launch: emap[block] = (case, block within the
// case; -1: the case's mean flow)
template <int MODE>
__global__ void __launch_bounds__(32 * EXPLICIT_WARPS, MODE == 1 ? 4 : 3)
k_explicit_b(const TcDev* __restrict__ ds, const int2* __restrict__ emap, int k, int Lc) {
    const int2 m = emap[blockIdx.x];
    const TcDev& d = ds[m.x];
    if (m.y < 0) mean_body<typename LineTypes<MODE>::CT>(d, k);
    else explicit_body<MODE>(d, k, 0, d.Nh, Lc, m.y);
}

// ---------------------------------------------------------------------------
// Diagnostics: kinetic energy and strain-rate density, every Fourier slot (the (0,0)
// slot holds the mean flow U, W), 16 slots a block, a lane per component as in
// k_solve.  (One thread per slot was the latency of six recurrences and an energy kernel
// that read u, v, w again: a restart of 129x128x128 with its statistics, k_init with a
// thread per pair included, 1662 -> 670 us, and 585 with the rows of k_init as they are.)
//
// First radial derivative of u, v and w, the operator of the energy budget: explicit
// one-sided 5-point D on the walls (dwall) and on rows 1, Nr-2 (l1 rows with d0 = 1),
// compact rows d0 . Df = l1 . f on 2..Nr-3 solved with the reversed factorisation
// dsol.  All warps share the right sides by rows, one warp per field runs its
// recurrences, then all share the densities: 2 S:S with the cylindrical strain
// components
//   S_rr = Dv, S_tt = (i m/r) w + v/r, S_zz = i alpha u,
//   S_rt = (Dw - w/r + (i m/r) v)/2, S_rz = (i alpha v + Du)/2,
//   S_tz = ((i m/r) u + i alpha w)/2,
// and |u|^2 + |v|^2 + |w|^2, times the Parseval weight (1 for m = 0, 2 otherwise), into
// dens[0] and dens[1], [r][slot].
constexpr int DIAG_WARPS = 4;
__global__ void __launch_bounds__(32 * DIAG_WARPS)
k_strain(const __grid_constant__ TcDev d, double* __restrict__ D, double* __restrict__ dens) {
    const int warp = threadIdx.x >> 5, comp = threadIdx.x & 1;
    const int pair = blockIdx.x * 16 + ((threadIdx.x & 31) >> 1);
    const bool act = pair < d.npairs;
    const int N = d.Nr;
    const size_t P = d.npairs, P2 = 2 * P, o = act ? 2 * (size_t)pair + comp : comp;
    const double* f[3] = {reinterpret_cast<const double*>(d.u), reinterpret_cast<const double*>(d.v), reinterpret_cast<const double*>(d.w)};
    const int i0 = warp * N / DIAG_WARPS, i1 = (warp + 1) * N / DIAG_WARPS;
    if (act) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double* F = f[q] + o;
            double* R = D + q * N * P2 + o;
            for (int j = i0; j < i1; ++j) {
                const int st = j < 2 ? 0 : j > N - 3 ? N - 5 : j - 2;
                const double* w = j == 0 ? d.dwall : j == N - 1 ? d.dwall + 5 : d.l1 + j * 5;
                double acc = 0.0;
                for (int s = 0; s < 5; ++s) acc = fma(w[s], F[(size_t)(st + s) * P2], acc);
                R[(size_t)j * P2] = acc;
            }
        }
    }
    __syncthreads();
    if (act && warp < 3) {
        double* R = D + warp * N * P2 + o;
        const double D0 = R[0], D1 = R[P2], DM = R[(size_t)(N - 2) * P2], DN = R[(size_t)(N - 1) * P2];
        double z1 = 0.0, z2 = 0.0;
        rows_ahead<OneRow>(
            N - 4, [&](int q, OneRow& w) { w.z = R[(size_t)(N - 3 - q) * P2]; },
            [&](int q, const OneRow& w) {
                const int j = N - 3 - q;
                const double* w0 = d.d0 + j * 5;
                double r = w.z;
                if (j == 2) r = fma(-w0[1], D1, fma(-w0[0], D0, r));
                if (j == 3) r = fma(-w0[0], D1, r);
                if (j == N - 4) r = fma(-w0[4], DM, r);
                if (j == N - 3) r = fma(-w0[4], DN, fma(-w0[3], DM, r));
                const double* c = d.dsol + j * 5;
                const double z = fma(-c[1], z1, fma(-c[0], z2, r));
                R[(size_t)j * P2] = z;
                z2 = z1; z1 = z;
            });
        double p1 = 0.0, p2 = 0.0;
        rows_ahead<OneRow>(
            N - 4, [&](int q, OneRow& w) { w.z = R[(size_t)(q + 2) * P2]; },
            [&](int q, const OneRow& w) {
                const double* c = d.dsol + (q + 2) * 5;
                const double x = c[2] * fma(-c[4], p2, fma(-c[3], p1, w.z));
                R[(size_t)(q + 2) * P2] = x;
                p2 = p1; p1 = x;
            });
    }
    __syncthreads();
    const int sl = act ? pair / d.Nh : 0, j = act ? pair - sl * d.Nh : 0;
    const int n = sl < d.Nz / 2 ? sl : (sl == d.Nz / 2 ? 0 : sl - d.Nz);
    const double m = j * d.m0, al = n * d.alpha0;
    const double wgt = j == 0 ? 1.0 : 2.0, sg = comp ? 1.0 : -1.0;      // i a: other component times sg
    const double *Du = D + o, *Dv = D + N * P2 + o, *Dw = D + 2 * N * P2 + o;
    const size_t x = o + 1 - 2 * comp;
    for (int i = i0; i < i1; ++i) {
        const size_t row = (size_t)i * P2;
        const double ri = d.rinv[i], imr = sg * m * ri, ial = sg * al;
        const double U = f[0][o + row], V = f[1][o + row], W = f[2][o + row];
        const double Ux = f[0][x + row], Vx = f[1][x + row], Wx = f[2][x + row];
        const double srr = Dv[row], stt = fma(imr, Wx, ri * V), szz = ial * Ux;
        const double srt = fma(imr, Vx, fma(-ri, W, Dw[row])), srz = fma(ial, Vx, Du[row]), stz = fma(imr, Ux, ial * Wx);
        double a = wgt * fma(2.0, fma(srr, srr, fma(stt, stt, szz * szz)), fma(srt, srt, fma(srz, srz, stz * stz)));
        double b = wgt * fma(U, U, fma(V, V, W * W));
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        b += __shfl_xor_sync(0xffffffffu, b, 1);
        if (act) dens[(size_t)comp * N * P + (size_t)i * P + pair] = comp ? b : a;
    }
}

// dprof[r], eprof[r] = sums over the slots of dens[0][r], dens[1][r] (fixed order:
// reproducible)
__global__ void __launch_bounds__(256) k_slot_sum(TcDev d, const double* __restrict__ dens) {
    const int r = blockIdx.x;
    const double* x = dens + ((size_t)blockIdx.y * d.Nr + r) * d.npairs;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < d.npairs; i += 4 * blockDim.x)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + q * (int)blockDim.x < d.npairs) a[q] += x[i + q * blockDim.x];
    __shared__ double red[256];
    red[threadIdx.x] = (a[0] + a[1]) + (a[2] + a[3]);
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) (blockIdx.y ? d.eprof : d.dprof)[r] = red[0];
}

void tc_launch_diagnostics(const TcDev& d, cudaStream_t s) {
    double* D = reinterpret_cast<double*>(d.pbuf);      // 3 Nr npairs complex, of TC_NPROD Nr Mzx Nh
    double* dens = reinterpret_cast<double*>(d.zbuf);
    k_strain<<<(d.npairs + 15) / 16, 32 * DIAG_WARPS, 0, s>>>(d, D, dens);
    k_slot_sum<<<dim3(d.Nr, 2), 256, 0, s>>>(d, dens);
}

// ---------------------------------------------------------------------------
// After a field is set: zero the (0,0) slot and the axial Nyquist slot, and
// make the m = 0 column Hermitian (slot Nz - n = conj(slot n)), so that the
// field is real.  One thread per (r, element) of the j = 0 column and of the
// Nyquist slot.
__global__ void __launch_bounds__(256) k_realify(TcDev d, double2* f) {
    const int r = blockIdx.y;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int Nz = d.Nz, Nh = d.Nh;
    if (r >= d.Nr || idx >= Nz + Nh) return;
    double2* pl = f + (size_t)r * d.npairs;
    if (idx < Nz) {
        const int s = idx;                               // slot of the j = 0 column
        if (s == 0) pl[0] = cz();
        else if (s > Nz / 2) pl[(size_t)s * Nh] = cconj(pl[(size_t)(Nz - s) * Nh]);
    } else {
        pl[(size_t)(Nz / 2) * Nh + (idx - Nz)] = cz();   // Nyquist slot, every j
    }
}

void tc_launch_realify(const TcDev& d, double2* field, cudaStream_t s) {
    k_realify<<<dim3((d.Nz + d.Nh + 255) / 256, d.Nr), 256, 0, s>>>(d, field);
}

void tc_launch_setup_tables(const TcDev& d, cudaStream_t s) {
    k_setup<<<(d.npairs + 127) / 128, 128, 0, s>>>(d);
}

static size_t mean_smem(int Nr) { return (size_t)14 * Nr * sizeof(double); }
// Radial rows per warp of k_explicit.  A chunk of L rows forms the inner functions at
// L + 4 points (57 float64 operations each) and 65 operations a row; a quarter of an
// SM runs one warp's operation in 64 cycles, so a launch takes as many times that
// work as each of the 608 quarters has warps.  The rule takes the shortest; line_block
// 128 is the rule, the other accepted values pin a length (tc_set_tiles).
// shared memory of k_explicit: the rows on their way in, or the mean flow's block (Nr > 0)
static size_t explicit_smem(int prec, int Nr) {
    const size_t ring = prec == 1 ? (size_t)RowRing<1>::RING * RowRing<1>::BYTES : prec == 2 ? (size_t)RowRing<2>::RING * RowRing<2>::BYTES : 0;
    const size_t mean = Nr > 0 ? mean_smem(Nr) : 0;
    return ring > mean ? ring : mean;
}
static int explicit_rule(int Nr, long long groups, long long& best) {
    const int nc = Nr - 4;
    int rows = 64;
    best = 0;
    for (int L : {64, 48, 32, 24, 16, 12, 8, 6, 4, 3, 2, 1}) {
        const long long warps = groups * ((nc + L - 1) / L), per = (warps + 607) / 608;
        const int l = L < nc ? L : nc;
        const long long cost = (per > 4 ? (warps * 16 + 607) / 608 : per * 16) * (57 * (l + 4) + 65 * l);
        if (best == 0 || cost < best) { best = cost; rows = L; }
    }
    return rows;
}
static int explicit_rows_per_warp(int line_block, int Nr, long long groups) {
    switch (line_block) {
        case 64: return 8;
        case 256: return 64;
        case 1003: return 16;
        case 1004: return 32;
        case 2007: return 4;
        case 3001: return 128;
        default: break;
    }
    long long cost;
    return explicit_rule(Nr, groups, cost);
}
// Rows per warp of k_explicit_wide, 0 where k_explicit takes less time by the same
// count (33 + 29 operations a point and row here) or the launch is not the float64
// form's own choice.
static int explicit_wide_rows(int prec, int line_block, int Nr, long long groups) {
    if (prec != 0 || line_block != 128 || !solve_wide(2 * groups, Nr)) return 0;
    long long best;
    explicit_rule(Nr, groups, best);
    int rows = 0;
    for (int R : {1, 2, 3, 4, 6, 8}) {
        const int n = 8 * R < Nr - 4 ? 8 * R : Nr - 4;
        const long long blocks = 2 * groups * ((Nr - 4 + 8 * R - 1) / (8 * R)), per = 2 * ((blocks + 151) / 152);
        const long long cost = (per > 4 ? (blocks * 32 + 151) / 152 : per * 16) * (33 * ((n + 4 + 7) / 8) + 29 * ((n + 7) / 8));
        if (cost < best) { best = cost; rows = R; }
    }
    return rows;
}
void tc_launch_line_chunk(const TcDev& d, int k, cudaStream_t s, int ja, int jw, bool mean, bool deferred) {
    const int groups = (d.Nz * jw + 31) / 32, half = (d.Nz * jw + 15) / 16;
    const int Lc = explicit_rows_per_warp(d.line_block, d.Nr, groups);
    const long long warps = (long long)groups * ((d.Nr - 4 + Lc - 1) / Lc);
    const bool noh = deferred && d.prec != 0, wide = solve_wide(half, d.Nr);
    // the mean flow goes with the longer launch: the solves where they are latency
    const bool early = mean && !wide;
    const int grid = (int)((warps + EXPLICIT_WARPS - 1) / EXPLICIT_WARPS) + (early ? 1 : 0);
    const size_t sm = explicit_smem(d.prec, early ? d.Nr : 0);
    const int R = explicit_wide_rows(d.prec, d.line_block, d.Nr, groups);
    if (R > 0)
        k_explicit_wide<<<half * ((d.Nr - 4 + 8 * R - 1) / (8 * R)), 32 * WIDE_WARPS, (8 * R + 4) * 160 * sizeof(double), s>>>(d, k, ja, jw, R);
    else if (d.prec == 1) k_explicit<1><<<grid, 32 * EXPLICIT_WARPS, sm, s>>>(d, k, ja, jw, Lc, early);
    else if (d.prec == 2) k_explicit<2><<<grid, 32 * EXPLICIT_WARPS, sm, s>>>(d, k, ja, jw, Lc, early);
    else k_explicit<0><<<grid, 32 * EXPLICIT_WARPS, sm, s>>>(d, k, ja, jw, Lc, early);
    if (wide) {
        const size_t sw = solve_smem(d.Nr);     // more than the mean flow's block takes
        if (noh) k_solve_shared<true><<<half + (mean ? 1 : 0), 32 * SOLVE_WARPS, sw, s>>>(d, k, ja, jw, mean);
        else k_solve_shared<false><<<half + (mean ? 1 : 0), 32 * SOLVE_WARPS, sw, s>>>(d, k, ja, jw, mean);
    } else {
        if (noh) k_solve<true><<<half, 64, 0, s>>>(d, k, ja, jw);
        else k_solve<false><<<half, 64, 0, s>>>(d, k, ja, jw);
    }
}
void tc_launch_line_phase(const TcDev& d, int k, cudaStream_t s, bool mean) { tc_launch_line_chunk(d, k, s, 0, d.Nh, mean, false); }

void tc_launch_rk_memory(const TcDev& d, int k, cudaStream_t s, int ja, int jw, bool background) {
    int blocks = (d.Nz * jw + 127) / 128;
    if (background) {
        static int sms = 0;
        if (!sms) {
            int dev = 0;
            cudaGetDevice(&dev);
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
        }
        blocks = blocks < 4 * sms ? blocks : 4 * sms;
    }
    k_rk_memory<<<blocks, 128, 0, s>>>(d, k, ja, jw);
}

const void* tc_rk_memory_kernel() { return (const void*)k_rk_memory; }

void tc_launch_mean_phase(const TcDev& d, int k, cudaStream_t s) {
    if (d.prec == 1) k_mean<float2><<<1, 256, mean_smem(d.Nr), s>>>(d, k);
    else if (d.prec == 2) k_mean<dcomplex><<<1, 256, mean_smem(d.Nr), s>>>(d, k);
    else k_mean<double2><<<1, 256, mean_smem(d.Nr), s>>>(d, k);
}

// The launches over many cases: which of the two takes the mean flows (the solves
// where they are wide), and the blocks of one case in each.
static long long half_groups(const TcDev& d) { return (d.npairs + 15) / 16; }
void tc_line_batch_plan(const TcDev* ds, int ncases, int& Lc, bool& wide) {
    long long half = 0, groups = 0;
    int maxNr = 0;
    for (int i = 0; i < ncases; ++i) {
        half += half_groups(ds[i]);
        groups += (ds[i].npairs + 31) / 32;
        maxNr = ds[i].Nr > maxNr ? ds[i].Nr : maxNr;
    }
    Lc = explicit_rows_per_warp(128, maxNr, groups);
    wide = solve_wide(half, maxNr);
}
int tc_line_batch_explicit_blocks(const TcDev& d, int Lc) {
    const long long warps = (long long)((d.npairs + 31) / 32) * ((d.Nr - 4 + Lc - 1) / Lc);
    return (int)((warps + EXPLICIT_WARPS - 1) / EXPLICIT_WARPS);
}
int tc_line_batch_solve_blocks(const TcDev& d) { return (int)half_groups(d); }
void tc_launch_explicit_batch(int prec, const TcDev* ds, const int2* emap, int nblocks, int maxNr, int Lc, bool mean, int k,
                              cudaStream_t s) {
    const size_t sm = explicit_smem(prec, mean ? maxNr : 0);
    if (prec == 1) k_explicit_b<1><<<nblocks, 32 * EXPLICIT_WARPS, sm, s>>>(ds, emap, k, Lc);
    else if (prec == 2) k_explicit_b<2><<<nblocks, 32 * EXPLICIT_WARPS, sm, s>>>(ds, emap, k, Lc);
    else k_explicit_b<0><<<nblocks, 32 * EXPLICIT_WARPS, sm, s>>>(ds, emap, k, Lc);
}
void tc_launch_solve_batch(const TcDev* ds, const int2* bmap, int nblocks, int maxNr, bool wide, int k, cudaStream_t s) {
    if (wide) k_solve_shared_b<<<nblocks, 32 * SOLVE_WARPS, solve_smem(maxNr), s>>>(ds, bmap, k);
    else k_solve_b<<<nblocks, 64, 0, s>>>(ds, bmap, k);
}

cudaError_t tc_set_line_kernel_attributes() {
    const int lim = 200 * 1024;
    for (const void* f : {(const void*)k_mean<double2>, (const void*)k_mean<dcomplex>, (const void*)k_mean<float2>,
                          (const void*)k_explicit<0>, (const void*)k_explicit<1>, (const void*)k_explicit<2>,
                          (const void*)k_explicit_b<0>, (const void*)k_explicit_b<1>, (const void*)k_explicit_b<2>,
                          (const void*)k_explicit_wide, (const void*)k_solve_shared<true>, (const void*)k_solve_shared<false>,
                          (const void*)k_solve_shared_b}) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void tc_launch_init_state(const TcDev& d, cudaStream_t s) {
    const int half = (d.npairs + 15) / 16;
    if (half < WIDE_GROUPS) k_init<8><<<half, 256, 0, s>>>(d);
    else k_init<4><<<half, 32 * 4, 0, s>>>(d);
    k_mean_init<<<1, 256, 0, s>>>(d);
}
