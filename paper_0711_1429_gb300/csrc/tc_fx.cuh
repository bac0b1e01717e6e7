// 64-bit fixed-point complex transforms: the arithmetic of the float64 and
// double-float plane phase (kernels in tc_fx_kernels.cuh).
//
// Why: per cycle and SM GB300 does 2 float64 operations, but 60 64-bit integer
// additions and 32 products of 32-bit integers to 64 bits (measured with
// dependent chains of each).  A 64 x 64-bit product kept to its upper half is
// three of those products, so a transform in 64-bit fixed point takes about a
// tenth of the float64 pipe's time.  One block scale per transform replaces
// the exponents: all values of a column share the power of two that its data
// allow, with 62 bits below it.  Additions are then exact and a product is
// rounded at 2^-62 of the scale, so the error relative to the norm of the
// column -- the only kind of accuracy a float64 transform has either, since
// every output is a sum over all inputs -- is below the float64 transform's
// (length 768, relative to the norm, before the result is rounded to float64:
// 3e-17 to 1e-16, where a float64 transform has 1.3e-16 to 2.2e-16).
//
// Scale: the inputs of a column are bounded by their largest component and
// by the sum of their magnitudes (fx_scale); no intermediate value of any
// pass exceeds the bound min(points summed x largest, sum), reduced by the
// factor 1/4 that every twiddled pass applies.  Everything is integer
// arithmetic on those bounds, so the result does not depend on the launch
// shape or on the order of the threads.
//
// The functions compile for the host too (the CPU tests run the same code).
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

typedef long long fx_t;
struct alignas(16) fxc { fx_t x, y; };
// A twiddle as fixed point with 62 fraction bits, each component in two signed
// halves: value = (h 2^32 + l) / 2^62.
struct alignas(16) fxw { int rh, rl, ih, il; };

FX_HD fxc fx_add(fxc a, fxc b) { fxc r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
FX_HD fxc fx_sub(fxc a, fxc b) { fxc r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
// a + S i b
template <int S> FX_HD fxc fx_addi(fxc a, fxc b) {
    fxc r;
    if (S < 0) { r.x = a.x + b.y; r.y = a.y - b.x; } else { r.x = a.x - b.y; r.y = a.y + b.x; }
    return r;
}
// signed halves of a: a = h 2^32 + l
FX_HD int fx_lo(fx_t a) { return (int)a; }
FX_HD int fx_hi(fx_t a) { return (int)(a >> 32) + (int)((unsigned)(int)a >> 31); }
// a b + c in one instruction (written out: the compiler otherwise splits the
// 64-bit addition from the product)
FX_HD fx_t fx_wide(int a, int b, fx_t c) {
#if defined(__CUDA_ARCH__)
    fx_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (fx_t)a * b + c;
#endif
}
// Upper half of a product whose cross terms sum to m: the product of the low
// halves is at most a quarter of the last bit and is left out.
FX_HD fx_t fx_up(fx_t m) { return (fx_t)(int)(m >> 32); }
// Half a unit of that upper half: the cross terms of a twiddle are summed from
// it, so that they are rounded and a product of zero stays zero.  It is read
// from constant memory because a literal would cost two extra additions in
// place of the multiply-add's own.
#if defined(__CUDACC__)
static __constant__ fx_t fx_half_unit = 0x80000000LL;
#endif
FX_HD fx_t fx_rnd() {
#if defined(__CUDA_ARCH__)
    return fx_half_unit;
#else
    return 0x80000000LL;
#endif
}

// a b / 2^64
FX_HD fx_t fx_mulhi(fx_t a, fx_t b) {
    const int ah = fx_hi(a), al = fx_lo(a), bh = fx_hi(b), bl = fx_lo(b);
    return fx_wide(ah, bh, 0) + fx_up(fx_wide(al, bh, fx_wide(ah, bl, 0)));
}
// s + a k / 2^64 for a constant k = (kh 2^32 + kl)
FX_HD fx_t fx_mulk(fx_t s, fx_t a, int kh, int kl) {
    const int h = fx_hi(a), l = fx_lo(a);
    return fx_wide(h, kh, s) + fx_up(fx_wide(l, kh, fx_wide(h, kl, 0)));
}
// s + (a k + b j) / 2^64
FX_HD fx_t fx_mulk2(fx_t s, fx_t a, int kh, int kl, fx_t b, int jh, int jl) {
    const int ah = fx_hi(a), al = fx_lo(a), bh = fx_hi(b), bl = fx_lo(b);
    return fx_wide(bh, jh, fx_wide(ah, kh, s)) + fx_up(fx_wide(bl, jh, fx_wide(bh, jl, fx_wide(al, kh, fx_wide(ah, kl, 0)))));
}
// a w / 4 (S < 0) or a conj(w) / 4 (S > 0); w is a forward twiddle.  Four products
// a component, not three as in (x + y) c - y (c + d): that form saves a fifth of
// the multiply-adds and no instructions, and it does not keep the values equal
// that a constant signal has to keep (w = 1 then rounds as the untwiddled value).
template <int S> FX_HD fxc fx_tw(fxc a, fxw w) {
    const int xh = fx_hi(a.x), xl = fx_lo(a.x), yh = fx_hi(a.y), yl = fx_lo(a.y);
    const int nh = -w.ih, nl = -w.il;
    const int ph = S < 0 ? nh : w.ih, pl = S < 0 ? nl : w.il;      // times y in the real part
    const int qh = S < 0 ? w.ih : nh, ql = S < 0 ? w.il : nl;      // times x in the imaginary part
    const fx_t h = fx_rnd();
    fxc r;
    r.x = fx_wide(yh, ph, fx_wide(xh, w.rh, 0)) + fx_up(fx_wide(yl, ph, fx_wide(yh, pl, fx_wide(xl, w.rh, fx_wide(xh, w.rl, h)))));
    r.y = fx_wide(yh, w.rh, fx_wide(xh, qh, 0)) + fx_up(fx_wide(xl, qh, fx_wide(xh, ql, fx_wide(yl, w.rh, fx_wide(yh, w.rl, h)))));
    return r;
}
// constants as round(k 2^64), |k| < 1/2, and their signed halves
constexpr fx_t FX_S60 = -2471395088767036514LL;   // sin(2 pi/3) - 1 = sqrt(3)/2 - 1
constexpr fx_t FX_C45 = -5402926248376769404LL;   // cos(pi/4) - 1 = sqrt(2)/2 - 1
constexpr fx_t FX_C22 = -1404174782535421627LL;   // cos(pi/8) - 1 = sqrt(2 + sqrt(2))/2 - 1
constexpr fx_t FX_S22 = 7059263338087549767LL;   // sin(pi/8) = sqrt(2 - sqrt(2))/2
FX_HD constexpr int fx_clo(fx_t c) { return (int)c; }
FX_HD constexpr int fx_chi(fx_t c) { return (int)((c - (int)c) >> 32); }

// ---- R-point transforms X_k = sum_r v_r exp(S 2 pi i r k/R), in place -------------
template <int S> FX_HD void fx_dft4(fxc& v0, fxc& v1, fxc& v2, fxc& v3) {
    const fxc a0 = fx_add(v0, v2), a1 = fx_sub(v0, v2), a2 = fx_add(v1, v3), a3 = fx_sub(v1, v3);
    v0 = fx_add(a0, a2); v1 = fx_addi<S>(a1, a3); v2 = fx_sub(a0, a2); v3 = fx_addi<-S>(a1, a3);
}
template <int S> FX_HD void fx_dft3(fxc& v0, fxc& v1, fxc& v2) {
    constexpr int kh = fx_chi(FX_S60), kl = fx_clo(FX_S60);
    const fxc sm = fx_add(v1, v2), df = fx_sub(v1, v2);
    fxc t, h;
    t.x = v0.x - (sm.x >> 1); t.y = v0.y - (sm.y >> 1);
    h.x = fx_mulk(df.x, df.x, kh, kl); h.y = fx_mulk(df.y, df.y, kh, kl);      // sin(2 pi/3) df
    v0 = fx_add(v0, sm);
    v1 = fx_addi<S>(t, h);
    v2 = fx_addi<-S>(t, h);
}
template <int S> FX_HD void fx_dft8(fxc* v) {
    constexpr int kh = fx_chi(FX_C45), kl = fx_clo(FX_C45);
    fx_dft4<S>(v[0], v[2], v[4], v[6]);          // E_k in v[0], v[2], v[4], v[6]
    fx_dft4<S>(v[1], v[3], v[5], v[7]);          // O_k in v[1], v[3], v[5], v[7]
    const fxc p = fx_addi<S>(v[3], v[3]);        // (1 + S i) O_1
    const fxc q = fx_addi<-S>(v[7], v[7]);       // (1 - S i) O_3 = -sqrt(2) w^3 O_3
    fxc o1, o3;
    o1.x = fx_mulk(p.x, p.x, kh, kl); o1.y = fx_mulk(p.y, p.y, kh, kl);
    o3.x = fx_mulk(q.x, q.x, kh, kl); o3.y = fx_mulk(q.y, q.y, kh, kl);
    const fxc e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o2 = v[5];
    v[0] = fx_add(e0, o0); v[4] = fx_sub(e0, o0);
    v[1] = fx_add(e1, o1); v[5] = fx_sub(e1, o1);
    v[2] = fx_addi<S>(e2, o2); v[6] = fx_addi<-S>(e2, o2);
    v[3] = fx_sub(e3, o3); v[7] = fx_add(e3, o3);
}
// a times exp(S i pi/8), exp(S i pi/4), exp(S i 3 pi/8)
template <int S> FX_HD fxc fx_rot1(fxc a) {
    constexpr int ch = fx_chi(FX_C22), cl = fx_clo(FX_C22), sh = fx_chi(FX_S22), sl = fx_clo(FX_S22);
    fxc r;
    r.x = fx_mulk2(a.x, a.x, ch, cl, a.y, S > 0 ? -sh : sh, S > 0 ? -sl : sl);
    r.y = fx_mulk2(a.y, a.y, ch, cl, a.x, S > 0 ? sh : -sh, S > 0 ? sl : -sl);
    return r;
}
template <int S> FX_HD fxc fx_rot2(fxc a) {
    constexpr int kh = fx_chi(FX_C45), kl = fx_clo(FX_C45);
    const fxc p = fx_addi<S>(a, a);
    fxc r;
    r.x = fx_mulk(p.x, p.x, kh, kl); r.y = fx_mulk(p.y, p.y, kh, kl);
    return r;
}
template <int S> FX_HD fxc fx_rot3(fxc a) {
    constexpr int ch = fx_chi(FX_C22), cl = fx_clo(FX_C22), sh = fx_chi(FX_S22), sl = fx_clo(FX_S22);
    fxc r;
    r.x = fx_mulk2(S > 0 ? -a.y : a.y, a.x, sh, sl, a.y, S > 0 ? -ch : ch, S > 0 ? -cl : cl);
    r.y = fx_mulk2(S > 0 ? a.x : -a.x, a.y, sh, sl, a.x, S > 0 ? ch : -ch, S > 0 ? cl : -cl);
    return r;
}
template <int S> FX_HD void fx_dft16(fxc* v) {
#pragma unroll
    for (int j = 0; j < 4; ++j) fx_dft4<S>(v[j], v[j + 4], v[j + 8], v[j + 12]);
    // element j + 4 k holds Y_j[k]: multiply by exp(S 2 pi i j k/16)
    fxc z; z.x = 0; z.y = 0;
    v[5] = fx_rot1<S>(v[5]);
    v[9] = fx_rot2<S>(v[9]);
    v[13] = fx_rot3<S>(v[13]);
    v[6] = fx_rot2<S>(v[6]);
    v[10] = fx_addi<S>(z, v[10]);
    v[14] = fx_rot2<S>(fx_addi<S>(z, v[14]));                 // 3 pi/4
    v[7] = fx_rot3<S>(v[7]);
    v[11] = fx_rot2<S>(fx_addi<S>(z, v[11]));
    v[15] = fx_rot1<S>(fx_sub(z, v[15]));                     // 9 pi/8
    fxc x[16];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        fxc a = v[4 * k], b = v[4 * k + 1], c = v[4 * k + 2], d = v[4 * k + 3];
        fx_dft4<S>(a, b, c, d);
        x[k] = a; x[k + 4] = b; x[k + 8] = c; x[k + 12] = d;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = x[k];
}
// Radices 6 = 2 x 3 and 12 = 3 x 4 by the prime-factor map: no inner twiddles.
// The inverse (S > 0) runs the 3-point transforms first, where the zero
// middle third of a padded spectrum drops one input of each; the forward runs
// them last, where the unread middle third drops one output of each.
template <int S> FX_HD void fx_dft6(fxc* v) {
    fxc a[2][3];
    if (S > 0) {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            a[p][0] = v[(3 * p) % 6]; a[p][1] = v[(3 * p + 2) % 6]; a[p][2] = v[(3 * p + 4) % 6];
            fx_dft3<S>(a[p][0], a[p][1], a[p][2]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            v[(4 * k) % 6] = fx_add(a[0][k], a[1][k]);
            v[(3 + 4 * k) % 6] = fx_sub(a[0][k], a[1][k]);
        }
    } else {
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const fxc p = v[(2 * n) % 6], q = v[(3 + 2 * n) % 6];
            a[0][n] = fx_add(p, q); a[1][n] = fx_sub(p, q);
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            fx_dft3<S>(a[p][0], a[p][1], a[p][2]);
#pragma unroll
            for (int k = 0; k < 3; ++k) v[(3 * p + 4 * k) % 6] = a[p][k];
        }
    }
}
template <int S> FX_HD void fx_dft12(fxc* v) {
    fxc a[3][4];
    if (S > 0) {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            a[0][n] = v[(3 * n) % 12]; a[1][n] = v[(4 + 3 * n) % 12]; a[2][n] = v[(8 + 3 * n) % 12];
            fx_dft3<S>(a[0][n], a[1][n], a[2][n]);
        }
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            fx_dft4<S>(a[p][0], a[p][1], a[p][2], a[p][3]);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[(4 * p + 9 * k) % 12] = a[p][k];
        }
    } else {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
#pragma unroll
            for (int n = 0; n < 4; ++n) a[p][n] = v[(4 * p + 3 * n) % 12];
            fx_dft4<S>(a[p][0], a[p][1], a[p][2], a[p][3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            fx_dft3<S>(a[0][k], a[1][k], a[2][k]);
#pragma unroll
            for (int p = 0; p < 3; ++p) v[(4 * p + 9 * k) % 12] = a[p][k];
        }
    }
}
template <int R, int S> FX_HD void fx_dft(fxc* v) {
    static_assert(R == 3 || R == 4 || R == 6 || R == 8 || R == 12 || R == 16, "radix");
    if constexpr (R == 3) fx_dft3<S>(v[0], v[1], v[2]);
    else if constexpr (R == 4) fx_dft4<S>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 6) fx_dft6<S>(v);
    else if constexpr (R == 8) fx_dft8<S>(v);
    else if constexpr (R == 12) fx_dft12<S>(v);
    else fx_dft16<S>(v);
}

// ---- plans ---------------------------------------------------------------------
// Two or three levels of radices R0, R1, R2.  Level L transforms the elements
// st(L) apart (st(0) = M/R0, st(1) = M/(R0 R1), last level 1) inside blocks of
// st(L) R, in place.  The inverse runs the levels upwards (decimation in
// frequency: natural order in, twiddles after the butterfly), the forward
// downwards (decimation in time: twiddles first, natural order out), so the
// values between the two are in digit-reversed order, which nothing that
// happens there minds, and a pass never moves a value: one barrier a pass.
// T threads a column (one butterfly per thread and pass); for the theta rows
// the row pairs G of a block and the threads W (a multiple of 32, >= G T) of
// each of its three roles.
template <int M> struct FxPlan;
#define FX_PLAN(M_, A, B, C, T_, G_, W_)                                          \
    template <> struct FxPlan<M_> {                                               \
        static constexpr int R0 = A, R1 = B, R2 = C, NP = C > 1 ? 3 : 2, T = T_, G = G_, W = W_; \
        static_assert(A * B * C == M_ && G_ * T_ <= W_ && W_ % 32 == 0, "plan");  \
        static_assert(T_ * A >= M_ && T_ * B >= M_ && (C == 1 || T_ * C >= M_), "threads"); \
    };
FX_PLAN(12, 3, 4, 1, 4, 8, 32)
FX_PLAN(18, 3, 6, 1, 6, 5, 32)
FX_PLAN(24, 6, 4, 1, 6, 5, 32)
FX_PLAN(32, 4, 8, 1, 8, 4, 32)
FX_PLAN(36, 6, 6, 1, 6, 5, 32)
FX_PLAN(48, 6, 8, 1, 8, 4, 32)
FX_PLAN(64, 8, 8, 1, 8, 4, 32)
FX_PLAN(72, 12, 6, 1, 12, 5, 64)
FX_PLAN(96, 12, 8, 1, 12, 5, 64)
FX_PLAN(128, 16, 8, 1, 16, 4, 64)
FX_PLAN(144, 6, 4, 6, 36, 4, 160)
FX_PLAN(192, 6, 4, 8, 48, 2, 96)
FX_PLAN(216, 6, 6, 6, 36, 4, 160)
FX_PLAN(256, 8, 4, 8, 64, 1, 64)
FX_PLAN(288, 6, 6, 8, 48, 2, 96)
FX_PLAN(384, 6, 8, 8, 64, 1, 64)
FX_PLAN(432, 12, 6, 6, 72, 1, 96)
FX_PLAN(512, 8, 8, 8, 64, 1, 64)
FX_PLAN(576, 12, 6, 8, 96, 1, 96)
FX_PLAN(768, 12, 8, 8, 96, 1, 96)
FX_PLAN(864, 12, 12, 6, 144, 1, 160)
FX_PLAN(1024, 16, 8, 8, 128, 1, 128)
FX_PLAN(1152, 12, 12, 8, 144, 1, 160)
FX_PLAN(1536, 16, 12, 8, 192, 1, 192)
#define FX_LENGTHS_A(X) X(12) X(24) X(48) X(128) X(192) X(768)
#define FX_LENGTHS_B(X) X(18) X(32) X(72) X(144) X(384) X(1024)
#define FX_LENGTHS_C(X) X(36) X(96) X(216) X(432) X(512) X(1536)
#define FX_LENGTHS_D(X) X(64) X(256) X(288) X(576) X(864) X(1152)
#define FX_LENGTHS(X) FX_LENGTHS_A(X) FX_LENGTHS_B(X) FX_LENGTHS_C(X) FX_LENGTHS_D(X)

// smallest planned length >= m (0: none)
inline int fx_length(int m) {
    int best = 0;
#define FX_PICK(M) if (M >= m && (best == 0 || M < best)) best = M;
    FX_LENGTHS(FX_PICK)
#undef FX_PICK
    return best;
}

template <int M, int L> FX_HD constexpr int fx_radix() {
    return L == 0 ? FxPlan<M>::R0 : L == 1 ? FxPlan<M>::R1 : FxPlan<M>::R2;
}
template <int M, int L> FX_HD constexpr int fx_stride() {
    return L == 0 ? M / FxPlan<M>::R0 : L == 1 ? M / (FxPlan<M>::R0 * FxPlan<M>::R1) : 1;
}
// element r of butterfly t of level L, and its place in shared memory: one
// element of padding after eight keeps the last level's stride off one
// another's banks
template <int M, int L> FX_HD constexpr int fx_pos(int t, int r) {
    constexpr int R = fx_radix<M, L>(), st = fx_stride<M, L>();
    return L == 0 ? t + r * st : (t / st) * (st * R) + t % st + r * st;
}
FX_HD constexpr int fx_pad(int i) { return i + (i >> 3); }
template <int M, int L> FX_HD int fx_at(int t, int r) {
    constexpr int R = fx_radix<M, L>(), st = fx_stride<M, L>();
    if constexpr (st % 8 == 0) return fx_pad(fx_pos<M, L>(t, 0)) + r * (st + st / 8);
    else if constexpr (st == 1 && R == 8) return 9 * t + r;
    else return fx_pad(fx_pos<M, L>(t, r));
}
// natural index of the value at position p of the digit-reversed order
template <int M> FX_HD constexpr int fx_index(int p) {
    constexpr int s0 = fx_stride<M, 0>(), s1 = fx_stride<M, 1>();
    return p / s0 + FxPlan<M>::R0 * (p % s0 / s1 + FxPlan<M>::R1 * (p % s1));
}
// Twiddle table of one length: entry [r - 1][tt] of level 0, then of level 1,
// stands for exp(-2 pi i r tt/(st R)), tt < st; then the R0 entries [r][tt] of
// level 0 times a scale factor, which the axial forward transform uses.
template <int M, int L> FX_HD constexpr int fx_tw_off() {
    return L == 0 ? 0 : fx_stride<M, 0>() * (fx_radix<M, 0>() - 1);
}
template <int M> FX_HD constexpr int fx_tw_scaled() {
    return fx_tw_off<M, 1>() + (FxPlan<M>::NP == 3 ? fx_stride<M, 1>() * (fx_radix<M, 1>() - 1) : 0);
}
template <int M> FX_HD constexpr int fx_tw_count() { return fx_tw_scaled<M>() + M; }
// Level L of the inverse (S > 0: transform, then twiddles) or the forward
// (S < 0: twiddles, then transform) for butterfly t.  Where there are twiddles
// every value is divided by 4, rounded; zero stays zero.
template <int M, int S, int L, bool SCALED = false> FX_HD void fx_butterfly(fxc* v, int t, const fxw* tw) {
    constexpr int R = fx_radix<M, L>(), st = fx_stride<M, L>();
    if constexpr (S > 0) fx_dft<R, S>(v);
    if constexpr (L + 1 < FxPlan<M>::NP) {
        const fxw* w = tw + (SCALED ? fx_tw_scaled<M>() : fx_tw_off<M, L>()) + (L == 0 ? t : t % st);
        if constexpr (!SCALED) {
            v[0].x = (v[0].x + 2) >> 2;
            v[0].y = (v[0].y + 2) >> 2;
        }
#pragma unroll
        for (int r = SCALED ? 0 : 1; r < R; ++r) v[r] = fx_tw<S>(v[r], w[(SCALED ? r : r - 1) * st]);
    }
    if constexpr (S < 0) fx_dft<R, S>(v);
}

// ---- scales --------------------------------------------------------------------
FX_HD constexpr int fx_clog2(int n) { int k = 0; while ((1 << k) < n) ++k; return k; }
FX_HD int fx_bitlen(unsigned x) {
#if defined(__CUDA_ARCH__)
    return 32 - __clz((int)x);
#else
    int n = 0;
    while (x) { ++n; x >>= 1; }
    return n;
#endif
}
// |x| in units of 2^(emax - 1023 - 18), rounded up (hi: upper word of a float64
// without its sign, emax: the largest exponent field of the column)
FX_HD unsigned fx_mag(unsigned hi, unsigned emax) {
    const unsigned sh = emax - (hi >> 20);
    return ((((hi & 0xfffffu) | 0x100000u) >> 2) >> (sh > 31 ? 31 : sh)) + 1u;
}
// Headroom of the passes: `one` bounds the log2 of one value, `sum` that of
// the sum of all magnitudes; returns the log2 bound of every intermediate value
// (the transform of a pass sums without scaling, each twiddle divides by 4).
template <int M, int S> FX_HD int fx_headroom(int one, int sum) {
    typedef FxPlan<M> P;
    constexpr int RA = S > 0 ? P::R0 : (P::NP == 3 ? P::R2 : P::R1);
    int b = one > sum ? sum : one;
    int p = one + fx_clog2(RA) < sum ? one + fx_clog2(RA) : sum;
    b = p > b ? p : b;
    if constexpr (P::NP == 3) {
        p = (one + fx_clog2(RA * P::R1) < sum ? one + fx_clog2(RA * P::R1) : sum) - 2;
        b = p > b ? p : b;
    }
    p = (one + fx_clog2(M) < sum ? one + fx_clog2(M) : sum) - 2 * (P::NP - 1);
    return p > b ? p : b;
}
#define FX_NONFINITE 0x7ff00000u
// Scale of a column from its largest upper word and its sum of fx_mag: the
// exponent field EB of a power of two above every intermediate value, so that
// the fixed-point value of x is x 2^(62 - (EB - 1023)).  `extra`: log2 of the
// complex values formed from `extra` components.
template <int M, int S> FX_HD int fx_scale(unsigned umax, unsigned usum, int extra) {
    const int emax = (int)(umax >> 20);
    return fx_headroom<M, S>(emax + 1 + extra, emax + fx_bitlen(usum) - 18);
}
#define FX_ZERO 4000   // a scale that makes every value zero

// float64 (as its two words) -> fixed point with scale EB; subnormal numbers have exponent
// 1 and no hidden bit: the upper word less e - 1 in the exponent field has the hidden bit
// where there is one.  (Two instructions a value; a branch to another conversion for the
// columns that need it cost the axial inverse 16 registers.)
FX_HD fx_t fx_from(unsigned hi, unsigned lo, int EB) {
    const int ex = (int)((hi >> 20) & 0x7ffu), e = ex < 1 ? 1 : ex;
    int rs = EB - e;
    rs = rs > 63 ? 63 : rs;
    const unsigned mh = (hi & 0x7fffffffu) - ((unsigned)(e - 1) << 20);
    const unsigned long long m = ((((unsigned long long)mh << 32) | lo) << 10) >> rs;
    const fx_t s = (fx_t)((int)hi >> 31);
    return ((fx_t)m ^ s) - s;
}
FX_HD int fx_clz(unsigned long long a) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)a);
#else
    return __builtin_clzll(a);
#endif
}
// fixed point -> bits of the float64 F 2^(eb - 1023), rounded to nearest over the
// whole range: subnormal below the normal numbers, infinite beyond the largest (the
// carry of a rounding at the top of either ends there by itself).  Where fx_normal(eb)
// every |F| <= 2^62 but zero is a normal number, and RANGE = false leaves the ends of
// the range out (same bits): they cost 5% of the axial forward transform.
FX_HD bool fx_normal(int eb) { return (unsigned)(eb - 1) < 1984u; }
template <bool RANGE = true> FX_HD unsigned long long fx_bits(fx_t F, int eb) {
    const fx_t s = F >> 63;
    const unsigned long long a = (unsigned long long)((F ^ s) - s);
    if (a == 0) return 0;
    const int lz = fx_clz(a);
    const unsigned long long m = a << lz;
    const int e = eb + 63 - lz;
    unsigned long long b;
    if (!RANGE || (unsigned)(e - 1) < 2046u) b = ((unsigned long long)(unsigned)(e - 1) << 52) + (m >> 11) + ((m >> 10) & 1);
    else if (e > 0) b = 0x7ff0000000000000ull;
    else b = e < -51 ? (unsigned long long)(e == -52) : (m >> (12 - e)) + ((m >> (11 - e)) & 1);
    return b | ((unsigned long long)s & 0x8000000000000000ull);
}
// x 2^s, s of either sign
FX_HD fx_t fx_shift(fx_t x, int s) { return s >= 0 ? (fx_t)((unsigned long long)x << s) : x >> (s < -63 ? 63 : -s); }
// EB of the value that pass NP - 1 leaves: each twiddled pass divides by 4
template <int M> FX_HD constexpr int fx_gain() { return 2 * (FxPlan<M>::NP - 1); }

#include <cmath>
#include <vector>
// Host: the twiddle table of a planned length M (empty for another length);
// scale: the factor of its scaled part.
inline std::vector<fxw> fx_table(int M, long double scale) {
    int R[3] = {0, 0, 0}, np = 0;
#define FX_RADICES(L) if (M == L) { R[0] = FxPlan<L>::R0; R[1] = FxPlan<L>::R1; R[2] = FxPlan<L>::R2; np = FxPlan<L>::NP; }
    FX_LENGTHS(FX_RADICES)
#undef FX_RADICES
    if (!np) return {};
    std::vector<fxw> t;
    auto half = [](long double c, int& h, int& l) {
        fx_t v = (fx_t)llroundl(c * 4611686018427387904.0L);       // 2^62
        if ((int)v == (int)0x80000000) ++v;                        // the low half can be negated
        l = (int)v;
        h = (int)((v - l) >> 32);
    };
    auto put = [&](int n, int st, int r0, int r1, long double f) {     // roots of unity of order n
        for (int r = r0; r < r1; ++r)
            for (int tt = 0; tt < st; ++tt) {
                const long double a = -6.283185307179586476925286766559005768L * (long double)(r * tt) / (long double)n;
                fxw w;
                half(f * cosl(a), w.rh, w.rl);
                half(f * sinl(a), w.ih, w.il);
                t.push_back(w);
            }
    };
    put(M, M / R[0], 1, R[0], 1.0L);
    if (np == 3) put(M / R[0], M / (R[0] * R[1]), 1, R[1], 1.0L);
    put(M, M / R[0], 0, R[0], scale);
    return t;
}
