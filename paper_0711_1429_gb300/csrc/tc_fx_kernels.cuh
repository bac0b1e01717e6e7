// Plane phase of the float64 and double-float forms in 64-bit fixed point
// (arithmetic, plans and scales in tc_fx.cuh).  The three kernels are those of
// tc_fft_impl.cuh with another arithmetic; the planes between them stay in
// fixed point, with the exponents of a column (axial inverse) or of a row
// (theta rows) beside them.  Instantiated per transform length by tc_fx_a.cu ..
// tc_fx_d.cu.
//
// A transform takes two or three passes of radix 3 to 16 held in registers,
// one butterfly per thread and pass, in place in one padded shared-memory
// column per transform, with one barrier between two passes.  The first pass
// takes its values from global memory, the last one leaves them in registers.
// The rows of zbuf and pbuf are the axial points in digit-reversed order: the
// theta rows treat every row alike.  The largest value and the sum of
// magnitudes of a column, both reduced as integers, give its scale.
//
// What bounds them: 32-bit integer issue (about 120 instructions a point of a
// 768-point transform, half of them in the twiddles), at 40 to 60% of the issue
// rate between barriers and loads, where the float64 transforms they replace kept
// the float64 pipe 92% busy.  Per substep of 257x512x512 in the float64 form: axial
// inverse 6.25 -> 1.61 ms, theta rows 30.96 -> 7.83, axial forward 10.60 -> 2.93; of
// 129x512x170 (axial length 255, now 256): 1.99 -> 0.27, 5.18 -> 1.32, 4.29 -> 0.57;
// in the double-float form there 1.04 -> 0.27, 2.15 -> 1.32, 1.63 -> 0.65.
#pragma once
#include "tc_fx.cuh"
#include "tc_internal.h"
#include "tc_dfloat.h"
#include <type_traits>

__device__ __forceinline__ unsigned fx_hiabs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ fx_t fx_of(double x, int EB) {
    return fx_from((unsigned)__double2hiint(x), (unsigned)__double2loint(x), EB);
}
template <bool RANGE> __device__ __forceinline__ double fx_to(fx_t F, int eb) { return __longlong_as_double((long long)fx_bits<RANGE>(F, eb)); }
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }
__device__ __forceinline__ unsigned umax2(unsigned a, unsigned b) { return a > b ? a : b; }
// barrier of one role's threads (barriers 1 .. 3; 0 is the block's)
__device__ __forceinline__ void role_sync(int role, int n) { asm volatile("bar.sync %0, %1;" ::"r"(role + 1), "r"(n) : "memory"); }

// Threads and columns of one block of the axial kernels: the z tile of the
// handle, or as many columns as keep a block within 384 threads (the registers
// of a 12-point butterfly leave room for two such blocks on an SM).
template <int M> FX_HD constexpr int fx_z_columns() {
    int c = 8;
    while (c > 1 && c * FxPlan<M>::T > 384) c /= 2;
    return c;
}
template <int M> FX_HD constexpr int fx_z_threads(int ct) { return (ct * FxPlan<M>::T + 31) / 32 * 32; }

// resident blocks asked for: what 80 registers a thread allow
template <int M> FX_HD constexpr int fx_z_blocks() { return 65536 / (fx_z_threads<M>(fx_z_columns<M>()) * 80); }

// reduction of one word per thread over the threads of a column (lanes with
// the same low bits of the thread index), into cell[c]
template <bool ADD> __device__ __forceinline__ void fx_column_reduce(unsigned v, unsigned* cell, int ct, int c) {
    for (int o = 16; o >= ct; o >>= 1) {
        const unsigned w = __shfl_xor_sync(0xffffffffu, v, o);
        v = ADD ? v + w : umax2(v, w);
    }
    if ((threadIdx.x & 31) < (unsigned)ct) {
        if (ADD) atomicAdd(cell + c, v);
        else atomicMax(cell + c, v);
    }
}

// the values of butterfly t of level L of a column (elements 1 << lct apart)
template <int M, int L> __device__ __forceinline__ void fx_put(const fxc* v, fxc* col, int t, int lct) {
#pragma unroll
    for (int r = 0; r < fx_radix<M, L>(); ++r) col[fx_at<M, L>(t, r) << lct] = v[r];
}
template <int M, int L> __device__ __forceinline__ void fx_get(fxc* v, const fxc* col, int t, int lct) {
#pragma unroll
    for (int r = 0; r < fx_radix<M, L>(); ++r) v[r] = col[fx_at<M, L>(t, r) << lct];
}
// a level in the middle of a transform, in place
template <int M, int S> __device__ __forceinline__ void fx_middle(fxc* col, int t, int lct, const fxw* tw) {
    if (t < M / fx_radix<M, 1>()) {
        fxc w[fx_radix<M, 1>()];
        fx_get<M, 1>(w, col, t, lct);
        fx_butterfly<M, S, 1>(w, t, tw);
        fx_put<M, 1>(w, col, t, lct);
    }
}

// legs of the first pass that lie wholly in the zero band of a padded
// spectrum, and outputs of the last pass wholly in the band never read
template <int M, int R> FX_HD constexpr bool fx_dead_leg(int r) {
    return r * (M / R) * 3 >= M && ((r + 1) * (M / R) - 1) * 3 <= 2 * M;
}

// Exponents beside the planes: the value of F is F 2^(e - 1023).
#define FX_NONE (-(1 << 20))    // below every exponent: no value at all
#define FX_BAD (1 << 20)        // above every exponent: one with a NaN or an infinity
__device__ __forceinline__ unsigned fx_abs_hi(fx_t F) {      // |F| < (this) 2^32
    const int h = (int)(F >> 32);
    return (unsigned)(h ^ (h >> 31)) + 1u;
}

// ---- axial inverse: u, v, w (spectral) -> zbuf[f][r][q][j], zexp[f][r][j] ----------
// A column is written with its largest component in [2^61, 2^62).
template <int M>
__global__ void __launch_bounds__(fx_z_threads<M>(fx_z_columns<M>()), fx_z_blocks<M>())
kx_zinv(const __grid_constant__ TcDev d1, const TcDev* __restrict__ ds, const int2* __restrict__ ymap, int col0, int lct) {
    constexpr int R = fx_radix<M, 0>(), NP = FxPlan<M>::NP, RL = fx_radix<M, NP - 1>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned cmx[8], csm[8], omx[8];
    const int2 ym = ds ? ymap[blockIdx.y] : make_int2(0, blockIdx.y);
    const TcDev& d = ds ? ds[ym.x] : d1;
    const int rp = ym.y, f = blockIdx.z, ct = 1 << lct;
    const int Nz = d.Nz, Nh = d.Nh, Nr = d.Nr;
    const int c = threadIdx.x & (ct - 1), t = threadIdx.x >> lct;
    const int j = col0 + blockIdx.x * ct + c;
    const double2* src = (f == 0 ? d.u : f == 1 ? d.v : d.w) + (size_t)rp * Nz * Nh + j;
    fxc* col = reinterpret_cast<fxc*>(smem_raw) + c;
    if (threadIdx.x < 8) { cmx[threadIdx.x] = 0; csm[threadIdx.x] = 0; omx[threadIdx.x] = 0; }
    double2 x[R];
    const bool on = t < M / R;
    unsigned mx = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        x[r] = make_double2(0.0, 0.0);
        if (!fx_dead_leg<M, R>(r)) {
            const int p = t + r * (M / R);
            const int s = p < Nz / 2 ? p : (p > M - Nz / 2 ? Nz - (M - p) : -1);
            if (on && s >= 0) x[r] = src[(size_t)s * Nh];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (!fx_dead_leg<M, R>(r)) mx = umax2(mx, umax2(fx_hiabs(x[r].x), fx_hiabs(x[r].y)));
    fx_column_reduce<false>(mx, cmx, ct, c);
    __syncthreads();
    const unsigned um = cmx[c];
    unsigned sm = 0;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (!fx_dead_leg<M, R>(r)) sm += fx_mag(fx_hiabs(x[r].x), um >> 20) + fx_mag(fx_hiabs(x[r].y), um >> 20);
    fx_column_reduce<true>(on ? sm : 0u, csm, ct, c);
    __syncthreads();
    const int EB = fx_scale<M, 1>(um, csm[c], 1);
    if (on) {
        fxc v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r].x = v[r].y = 0;
            if (!fx_dead_leg<M, R>(r)) { v[r].x = fx_of(x[r].x, EB); v[r].y = fx_of(x[r].y, EB); }
        }
        fx_butterfly<M, 1, 0>(v, t, d.twx_z);
        fx_put<M, 0>(v, col, t, lct);
    }
    __syncthreads();
    if constexpr (NP == 3) {
        fx_middle<M, 1>(col, t, lct, d.twx_z);
        __syncthreads();
    }
    const bool last = t < M / RL;
    fxc v[RL];
    unsigned om = 0;
    if (last) {
        fx_get<M, NP - 1>(v, col, t, lct);
        fx_butterfly<M, 1, NP - 1>(v, t, d.twx_z);
#pragma unroll
        for (int r = 0; r < RL; ++r) om = umax2(om, umax2(fx_abs_hi(v[r].x), fx_abs_hi(v[r].y)));
    }
    fx_column_reduce<false>(om, omx, ct, c);
    __syncthreads();
    if (!last) return;
    const int up = 30 - fx_bitlen(omx[c]);          // |F| < 2^62 after the shift by up >= -1
    fxc* out = reinterpret_cast<fxc*>(d.zbuf) + ((size_t)f * Nr + rp) * M * Nh + j;
#pragma unroll
    for (int r = 0; r < RL; ++r) {
        fxc o;
        o.x = up >= 0 ? v[r].x << (up & 31) : v[r].x >> 1;
        o.y = up >= 0 ? v[r].y << (up & 31) : v[r].y >> 1;
        out[(size_t)fx_pos<M, NP - 1>(t, r) * Nh] = o;
    }
    if (t == 0)
        d.zexp[((size_t)f * Nr + rp) * Nh + j] = um >= FX_NONFINITE ? FX_BAD : EB - 62 + fx_gain<M>() - up;
}

// ---- axial forward: pbuf, pexp -> spectral products, scaled by 1/(Mt Mz) -----------
template <int M, bool DF>
__global__ void __launch_bounds__(fx_z_threads<M>(fx_z_columns<M>()), fx_z_blocks<M>())
kx_zfwd(const __grid_constant__ TcDev d1, const TcDev* __restrict__ ds, const int2* __restrict__ ymap, int col0, int lct) {
    constexpr int NP = FxPlan<M>::NP, R = fx_radix<M, NP - 1>(), RL = fx_radix<M, 0>();
    typedef typename std::conditional<DF, dcomplex, double2>::type PO;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned cmx[8], csm[8];
    const int2 ym = ds ? ymap[blockIdx.y] : make_int2(0, blockIdx.y);
    const TcDev& d = ds ? ds[ym.x] : d1;
    const int rp = ym.y, pr = blockIdx.z, ct = 1 << lct;
    const int Nz = d.Nz, Nh = d.Nh, Nr = d.Nr;
    const int c = threadIdx.x & (ct - 1), t = threadIdx.x >> lct;
    const int j = col0 + blockIdx.x * ct + c;
    const fxc* src = reinterpret_cast<const fxc*>(d.pbuf) + ((size_t)pr * Nr + rp) * M * Nh + j;
    const int* ex = d.pexp + ((size_t)(pr >> 1) * Nr + rp) * M;     // products 0, 1 | 2, 3 | 4 share exponents
    fxc* col = reinterpret_cast<fxc*>(smem_raw) + c;
    if (threadIdx.x < 8) { cmx[threadIdx.x] = 0; csm[threadIdx.x] = 0; }
    fxc v[R];
    int e[R];
    const bool on = t < M / R;
    // largest value as the exponent of its leading bit, offset to be unsigned
    // (0: nothing but zeros)
    constexpr int OFF = 1 << 22;
    unsigned mx = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        v[r].x = v[r].y = 0;
        e[r] = FX_NONE;
        if (on) {
            const int q = fx_pos<M, NP - 1>(t, r);
            e[r] = ex[q];
            v[r] = src[(size_t)q * Nh];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (e[r] == FX_NONE) v[r].x = v[r].y = 0;
        else
            mx = umax2(mx, (unsigned)(OFF + e[r] + fx_bitlen(fx_abs_hi(v[r].x) | fx_abs_hi(v[r].y))));
    fx_column_reduce<false>(mx, cmx, ct, c);
    __syncthreads();
    const int top = (int)cmx[c] - OFF;           // every component is < 2^(top + 32 - 1023)
    const bool bad = top >= FX_BAD;
    unsigned sm = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // |value| in units of 2^(top + 32 - 1023 - 19), rounded up
        const int sh = top - e[r] - 19;
        const unsigned a = fx_abs_hi(v[r].x), b = fx_abs_hi(v[r].y);
        sm += sh >= 0 ? (a >> (sh > 31 ? 31 : sh)) + (b >> (sh > 31 ? 31 : sh)) + 2u : (a + b) << (-sh & 31);
    }
    fx_column_reduce<true>(on && !bad ? sm : 0u, csm, ct, c);
    __syncthreads();
    const int EB = fx_headroom<M, -1>(top + 32 + 1, top + 32 - 19 + fx_bitlen(csm[c]));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int s = 62 + e[r] - EB;
        v[r].x = fx_shift(v[r].x, s); v[r].y = fx_shift(v[r].y, s);
    }
    if (on) {
        fx_butterfly<M, -1, NP - 1>(v, t, d.twx_z);
        fx_put<M, NP - 1>(v, col, t, lct);
    }
    __syncthreads();
    if constexpr (NP == 3) {
        fx_middle<M, -1>(col, t, lct, d.twx_z);
        __syncthreads();
    }
    if (t >= M / RL) return;
    fxc z[RL];
    fx_get<M, 0>(z, col, t, lct);
    fx_butterfly<M, -1, 0, true>(z, t, d.twx_z);
    const int eb = EB - 62 + fx_gain<M>() + d.kexp;
    PO* out = reinterpret_cast<PO*>(d.prod) + ((size_t)pr * Nr + rp) * Nz * Nh + j;
    auto put = [&](int s, double2 o) {
        if constexpr (DF) {
            dcomplex e;
            e.x = df_bits(o.x); e.y = df_bits(o.y);
            out[(size_t)s * Nh] = e;
        } else out[(size_t)s * Nh] = o;
    };
    auto store = [&](auto range) {          // with the ends of the float64 range and the mark, or without
#pragma unroll
        for (int r = 0; r < RL; ++r) {
            if (fx_dead_leg<M, RL>(r)) continue;
            const int q = fx_pos<M, 0>(t, r);
            const int s = q < Nz / 2 ? q : (q > M - Nz / 2 ? Nz - (M - q) : -1);
            if (s < 0) continue;
            double2 o = make_double2(fx_to<range.value>(z[r].x, eb), fx_to<range.value>(z[r].y, eb));
            if (range.value && bad) o.x = o.y = fx_nan();
            put(s, o);
        }
    };
    if (fx_normal(eb) && !bad) store(std::false_type());
    else store(std::true_type());
    if (t == 0) put(Nz / 2, make_double2(0.0, 0.0));       // axial Nyquist slot
}

// ---- theta rows: two rows q0 = 2 qp, q1 = q0 + 1 at a time ----------------------
// As in k_rows2 every transform has the full length: three inverse columns,
// u + i v of q0, u + i v of q1 and w(q0) + i w(q1), then five forward ones,
// (uu - vv) + i uv and uw + i vw of each row and (ww - vv)(q0) + i (ww - vv)(q1).
// Each inverse column has its own W threads (roles 0, 1, 2).  The products are
// formed by the threads that hold u and v at a point; w comes from role 2's
// column and ww - vv goes back into it, uw + i vw into a fourth and fifth
// column.  Roles 0 and 1 then transform their two columns one after the other.
// The scale of the inverse transforms comes from the columns' exponents (the
// same for every row of the plane).  A row pair's products are normalised by
// the largest physical u, v and w and by their mean squares, which bound the
// forward transform's values (sum |u w| <= sqrt(sum u^2 sum w^2)).
template <int M> FX_HD constexpr int fx_rows_smem() { return 5 * FxPlan<M>::G * (M + M / 8) * (int)sizeof(fxc); }
// resident blocks asked for: what 72 registers a thread allow
#ifndef FX_ROWS_REGS
#define FX_ROWS_REGS 72
#endif
template <int M> FX_HD constexpr int fx_rows_blocks() {
    constexpr int b = 65536 / (3 * FxPlan<M>::W * FX_ROWS_REGS), s = 225 * 1024 / (fx_rows_smem<M>() + 2048);
    return b < 1 || s < 1 ? 1 : (b < s ? b : s);
}

template <int M>
__global__ void __launch_bounds__(3 * FxPlan<M>::W, fx_rows_blocks<M>())
kx_rows(const __grid_constant__ TcDev d1, const TcDev* __restrict__ ds, const int2* __restrict__ ymap) {
    typedef FxPlan<M> P;
    constexpr int NP = P::NP, T = P::T, G = P::G, W = P::W;
    constexpr int R = fx_radix<M, 0>(), RL = fx_radix<M, NP - 1>(), MP = M + M / 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int emax[2];                      // largest column exponent of u, v and of w
    __shared__ unsigned esum[2];                 // sum of the columns' sizes relative to it
    __shared__ unsigned omx[3][G], osq[3][G];
    const int2 ym = ds ? ymap[blockIdx.y] : make_int2(0, blockIdx.y);
    const TcDev& d = ds ? ds[ym.x] : d1;
    const int rp = ym.y, Nr = d.Nr, Mz = d.Mzx, Nh = d.Nh;
    const fxw* tw = d.twx_t;
    const int role = threadIdx.x / W, in = threadIdx.x - role * W;
    const bool on = in < G * T;                  // not a spare thread of the role
    const int g = on ? in / T : 0, t = on ? in - g * T : 0;
    const int q0 = 2 * (blockIdx.x * G + g);
    const bool have0 = on && q0 < Mz, have1 = on && q0 + 1 < Mz;
    fxc* const bufs = reinterpret_cast<fxc*>(smem_raw);
    fxc* const col = bufs + (role * G + g) * MP;
    fxc* const colw = bufs + (2 * G + g) * MP;
    fxc* const col2 = bufs + ((role < 2 ? 3 + role : 2) * G + g) * MP;
    if (threadIdx.x < 2) { emax[threadIdx.x] = FX_NONE; esum[threadIdx.x] = 0; }
    if (threadIdx.x < 3 * G) { (&omx[0][0])[threadIdx.x] = 0; (&osq[0][0])[threadIdx.x] = 0; }
    // ---- scale of the inverse transforms: every |u|, |v| of a row is at most the
    // sum over the columns of twice their largest modulus (< 2^62.5 units) ----
    const size_t es = (size_t)Nr * Nh;
    const int* zx = d.zexp + (size_t)rp * Nh;
    const int* ze = zx + role * es;              // role k looks through field k
    const int wk = role == 2;
    __syncthreads();
    {
        int a = FX_NONE;
        for (int j = in; j < Nh; j += W) a = max(a, ze[j]);
        a = __reduce_max_sync(0xffffffffu, a);
        if ((threadIdx.x & 31) == 0) atomicMax(&emax[wk], a);
    }
    __syncthreads();
    const int em0 = emax[0], em1 = emax[1];
    const bool bad = em0 >= FX_BAD || em1 >= FX_BAD;
    {
        const int em = wk ? em1 : em0;
        unsigned a = 0;
        for (int j = in; j < Nh; j += W) {
            const int sh = em - ze[j];
            a += sh > 18 ? 1u : (1u << 18) >> sh;
        }
        a = __reduce_add_sync(0xffffffffu, a);
        if ((threadIdx.x & 31) == 0) atomicAdd(&esum[wk], a);
    }
    __syncthreads();
    // one value X + i Y: modulus < 2 sqrt(2) 2^62 units of 2^(em - 1023); the sum
    // over both halves of the spectrum: 2 sqrt(2) 2^62 per column.  (w(q0) + i w(q1):
    // every column counts for both rows.)
    const int EBuv = fx_headroom<M, 1>(em0 + 64, em0 + 62 + 2 + fx_bitlen(esum[0]) - 18);
    const int EBw = fx_headroom<M, 1>(em1 + 64, em1 + 62 + 3 + fx_bitlen(esum[1]) - 18);
    const int EB = role == 2 ? EBw : EBuv;
    // ---- first inverse pass: the spectra X + i Y of two real signals ----
    const size_t fs = (size_t)Nr * Mz * Nh;
    {
        const fxc* zb = reinterpret_cast<const fxc*>(d.zbuf) + (size_t)rp * Mz * Nh;
        const bool haveX = role == 1 ? have1 : have0, haveY = role == 0 ? have0 : have1;
        const fxc* X = zb + (role == 2 ? 2 * fs : 0) + (size_t)(haveX ? q0 + (role == 1) : 0) * Nh;
        const fxc* Y = zb + (role == 2 ? 2 * fs : fs) + (size_t)(haveY ? q0 + (role != 0) : 0) * Nh;
        const int* xe = zx + (role == 2 ? 2 * es : 0);
        const int* ye = zx + (role == 2 ? 2 * es : es);
        if (on && t < M / R) {
            fxc v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r].x = v[r].y = 0;
                if (!fx_dead_leg<M, R>(r)) {
                    const int p = t + r * (M / R);
                    const bool neg = p >= Nh;                // the conjugate half
                    const int j = !neg ? p : (p > M - Nh ? M - p : -1);
                    if (j >= 0) {
                        fxc x, y;
                        x.x = x.y = y.x = y.y = 0;
                        int sx = 63, sy = 63;
                        if (haveX) { x = X[j]; sx = EB - 62 - xe[j]; }
                        if (haveY) { y = Y[j]; sy = EB - 62 - ye[j]; }
                        sx = sx > 63 ? 63 : sx;              // >= 2: the scale lies above every column
                        sy = sy > 63 ? 63 : sy;
                        const fx_t hx = 1LL << (sx - 1), hy = 1LL << (sy - 1);
                        x.x = (x.x + hx) >> sx; x.y = (x.y + hx) >> sx;
                        y.x = (y.x + hy) >> sy; y.y = (y.y + hy) >> sy;
                        // p < Nh: X + i Y; p > M - Nh: conj X + i conj Y; the imaginary
                        // parts at j = 0 are not part of a real signal
                        if (p == 0) { x.y = 0; y.y = 0; }
                        v[r].x = neg ? x.x + y.y : x.x - y.y;
                        v[r].y = neg ? y.x - x.y : y.x + x.y;
                    }
                }
            }
            fx_butterfly<M, 1, 0>(v, t, tw);
            fx_put<M, 0>(v, col, t, 0);
        }
    }
    role_sync(role, W);
    if constexpr (NP == 3) {
        if (on) fx_middle<M, 1>(col, t, 0, tw);
        role_sync(role, W);
    }
    // ---- last inverse pass; largest value and mean square of the signals ----
    // (integers, so the order of the threads does not matter; whole warps of a row
    // pair use one atomic)
    auto reduce = [&](unsigned v, unsigned* cell, bool add, bool mine) {
        if constexpr (T % 32 == 0) {
            v = add ? __reduce_add_sync(0xffffffffu, v) : __reduce_max_sync(0xffffffffu, v);
            if ((threadIdx.x & 31) != 0) return;
        } else if (!mine) return;
        if (add) atomicAdd(cell, v);
        else atomicMax(cell, v);
    };
    constexpr int SH = 17;
    const bool last = on && t < M / RL;
    fxc v[RL];
#pragma unroll
    for (int r = 0; r < RL; ++r) v[r].x = v[r].y = 0;
    if (last) {
        fx_get<M, NP - 1>(v, col, t, 0);
        fx_butterfly<M, 1, NP - 1>(v, t, tw);
        if (role == 2) fx_put<M, NP - 1>(v, col, t, 0);
    }
    {
        unsigned om = 0, sq = 0;
#pragma unroll
        for (int r = 0; r < RL; ++r) {
            const unsigned ua = fx_abs_hi(v[r].x), ub = fx_abs_hi(v[r].y);
            om = umax2(om, umax2(ua, ub));
            const unsigned qa = (ua >> SH) + 1u, qb = (ub >> SH) + 1u;
            sq += qa * qa + qb * qb;
        }
        reduce(last ? om : 0u, &omx[role][g], false, last);
        reduce(last ? (sq >> 6) + 1u : 0u, &osq[role][g], true, last);
    }
    __syncthreads();
    // ---- normalisation: |u|, |v| < 2^62 jointly in both rows, |w| < 2^62 ----
    const int suv = 30 - fx_bitlen(umax2(omx[0][g], omx[1][g])), sw = 30 - fx_bitlen(omx[2][g]);
    const int Euv = EBuv - suv, Ew = EBw - sw;
    // log2 of the sums of squares after normalisation, in units of products / 2^64
    const int luv = fx_bitlen(umax2(osq[0][g], osq[1][g])) + 6 + 2 * SH + 2 * suv;
    const int lw = fx_bitlen(osq[2][g]) + 6 + 2 * SH + 2 * sw;
    int hs = fx_headroom<M, -1>(61, (luv > lw ? luv : lw) + 2) - 62;
    hs = hs < 0 ? 0 : hs > 62 ? 62 : hs;
    const int Em = Euv > Ew ? Euv : Ew;
    // ---- products: own column = (uu - vv, uv), col2 = (uw, vw), role 2's = ww - vv ----
    if (role < 2 && last) {
        const int dW = 2 * (Em - Ew) > 63 ? 63 : 2 * (Em - Ew), dV = 2 * (Em - Euv) > 63 ? 63 : 2 * (Em - Euv);
#pragma unroll
        for (int r = 0; r < RL; ++r) {
            const int at = fx_at<M, NP - 1>(t, r);
            fx_t* cell = &colw[at].x + role;
            const fx_t u = fx_shift(v[r].x, suv), w_ = fx_shift(v[r].y, suv), w = fx_shift(*cell, sw);
            const fx_t us = u >> hs, vs = w_ >> hs, ws = w >> hs;
            const fx_t vv = fx_mulhi(vs, w_);
            fxc b;
            b.x = fx_mulhi(us, u) - vv;
            b.y = fx_mulhi(us, w_);
            col[at] = b;
            b.x = fx_mulhi(us, w);
            b.y = fx_mulhi(vs, w);
            col2[at] = b;
            *cell = (fx_mulhi(ws, w) >> dW) - (vv >> dV);
        }
    }
    // exponents of the results: a product of values with exponents a, b (E - 62 +
    // gain each, / 2^64, shifted by hs), the forward gain and the unpacking's 1/2
    const int base = 2 * (fx_gain<M>() - 62) - 1023 + 64 + hs + fx_gain<M>() - 1;
    auto exponent = [&](int e) { return bad ? FX_BAD : e; };
    __syncthreads();
    // ---- forward transforms, two real signals each: role 2 one, the others two ----
    fxc* const pb = reinterpret_cast<fxc*>(d.pbuf) + (size_t)rp * Mz * Nh;
    int* const pe = d.pexp + (size_t)rp * Mz;
    const size_t pes = (size_t)Nr * Mz;
    for (int k = 0; k < (role == 2 ? 1 : 2); ++k) {
        fxc* const c = k ? col2 : col;
        if (last) {
            fxc z[RL];
            fx_get<M, NP - 1>(z, c, t, 0);
            fx_butterfly<M, -1, NP - 1>(z, t, tw);
            fx_put<M, NP - 1>(z, c, t, 0);
        }
        role_sync(role, W);
        if constexpr (NP == 3) {
            if (on) fx_middle<M, -1>(c, t, 0, tw);
            role_sync(role, W);
        }
        if (on && t < M / R) {
            fxc z[R];
            fx_get<M, 0>(z, c, t, 0);
            fx_butterfly<M, -1, 0>(z, t, tw);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (!fx_dead_leg<M, R>(r)) c[fx_at<M, 0>(t, r)] = z[r];
        }
        role_sync(role, W);
        // two products of one row (roles 0, 1), or one of both (role 2)
        const bool w1 = role == 1 ? have1 : have0, w2 = role == 0 ? have0 : have1;
        fxc* o1 = pb + (role == 2 ? 4 * fs : (size_t)(2 * k) * fs) + (size_t)(q0 + (role == 1)) * Nh;
        fxc* o2 = role == 2 ? o1 + Nh : o1 + fs;
        if (on) {
            for (int j = t; j < Nh; j += T) {
                const fxc a = c[fx_pad(j)], b = c[fx_pad(j == 0 ? 0 : M - j)];
                fxc o;
                o.x = a.x + b.x; o.y = a.y - b.y;
                if (w1) o1[j] = o;
                o.x = a.y + b.y; o.y = b.x - a.x;
                if (w2) o2[j] = o;
            }
        }
        if (t == 0) {
            if (role == 2) {
                const int e = exponent(base + 2 * Em);
                if (have0) pe[2 * pes + q0] = e;
                if (have1) pe[2 * pes + q0 + 1] = e;
            } else if (w1) {
                pe[k * pes + q0 + role] = exponent(base + Euv + (k ? Ew : Euv));
            }
        }
    }
}

// ---- physical output of one field: theta rows of zbuf's first field ---------------
// Two rows (axial points) per complex transform, X(q0) + i X(q1), each block G such
// pairs of one radial plane.  The rows come in the axial transform's digit-reversed
// order and leave in natural order, as float64; zr: that transform's radices and
// strides (R0, R1, st0, st1).  Scale: twice the sum of the moduli of the pair's own
// values bounds every intermediate one; the sum of the columns' largest values (as in
// kx_rows) would leave two bits of the result unused.
template <int M>
__global__ void __launch_bounds__(FxPlan<M>::W)
kx_phys(const __grid_constant__ TcDev d, int4 zr) {
    typedef FxPlan<M> P;
    constexpr int NP = P::NP, T = P::T, G = P::G, W = P::W;
    constexpr int R = fx_radix<M, 0>(), RL = fx_radix<M, NP - 1>(), MP = M + M / 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int emax;
    __shared__ unsigned rsum[G];
    const int rp = blockIdx.y, Mz = d.Mz, Nh = d.Nh, in = threadIdx.x;
    const fxw* tw = d.twx_t;
    const bool on = in < G * T;
    const int g = on ? in / T : 0, t = on ? in - g * T : 0;
    const int q0 = 2 * (blockIdx.x * G + g);
    const bool have0 = on && q0 < Mz, have1 = on && q0 + 1 < Mz;
    fxc* const col = reinterpret_cast<fxc*>(smem_raw) + g * MP;
    if (in == 0) emax = FX_NONE;
    if (in < G) rsum[in] = 0;
    const int* zx = d.zexp + (size_t)rp * Nh;
    __syncthreads();
    {
        int a = FX_NONE;
        for (int j = in; j < Nh; j += W) a = max(a, zx[j]);
        a = __reduce_max_sync(0xffffffffu, a);
        if ((in & 31) == 0) atomicMax(&emax, a);
    }
    __syncthreads();
    const int em = emax;
    const fxc* zb = reinterpret_cast<const fxc*>(d.zbuf) + (size_t)rp * Mz * Nh;
    if (on) {
        auto modulus = [](fxc x) {                  // upper words: max + min/2 is above the modulus
            const unsigned a = fx_abs_hi(x.x), b = fx_abs_hi(x.y);
            return a > b ? a + (b >> 1) : b + (a >> 1);
        };
        unsigned a = 0;
        for (int j = t; j < Nh; j += T) {
            const int sh = 12 + em - zx[j];
            unsigned m = 2;
            if (have0) m += modulus(zb[(size_t)q0 * Nh + j]);
            if (have1) m += modulus(zb[(size_t)(q0 + 1) * Nh + j]);
            a += (sh > 31 ? 0 : m >> sh) + 1;
        }
        atomicAdd(&rsum[g], a);
    }
    __syncthreads();
    int EB = fx_headroom<M, 1>(em + 64, em + 45 + fx_bitlen(rsum[g]));
    if (EB < em + 63) EB = em + 63;
    if (on && t < M / R) {
        fxc v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r].x = v[r].y = 0;
            if (!fx_dead_leg<M, R>(r)) {
                const int p = t + r * (M / R);
                const bool neg = p >= Nh;
                const int j = !neg ? p : (p > M - Nh ? M - p : -1);
                if (j >= 0) {
                    fxc x, y;
                    x.x = x.y = y.x = y.y = 0;
                    if (have0) x = zb[(size_t)q0 * Nh + j];
                    if (have1) y = zb[(size_t)(q0 + 1) * Nh + j];
                    int s = EB - 62 - zx[j];
                    s = s > 63 ? 63 : s;
                    const fx_t h = 1LL << (s - 1);
                    x.x = (x.x + h) >> s; x.y = (x.y + h) >> s;
                    y.x = (y.x + h) >> s; y.y = (y.y + h) >> s;
                    if (p == 0) { x.y = 0; y.y = 0; }
                    v[r].x = neg ? x.x + y.y : x.x - y.y;
                    v[r].y = neg ? y.x - x.y : y.x + x.y;
                }
            }
        }
        fx_butterfly<M, 1, 0>(v, t, tw);
        fx_put<M, 0>(v, col, t, 0);
    }
    __syncthreads();
    if constexpr (NP == 3) {
        if (on) fx_middle<M, 1>(col, t, 0, tw);
        __syncthreads();
    }
    fxc v[RL];
    const bool last = on && t < M / RL;
    if (last) {
        fx_get<M, NP - 1>(v, col, t, 0);
        fx_butterfly<M, 1, NP - 1>(v, t, tw);
    }
    __syncthreads();
    if (last) {
#pragma unroll
        for (int r = 0; r < RL; ++r) col[fx_pad(fx_index<M>(fx_pos<M, NP - 1>(t, r)))] = v[r];
    }
    __syncthreads();
    if (!on) return;
    const int eb = EB - 62 + fx_gain<M>();
    const bool bad = em >= FX_BAD;
    auto row = [&](int q) {
        return d.phys + ((size_t)rp * Mz + q / zr.z + zr.x * (q % zr.z / zr.w + zr.y * (q % zr.w))) * M;
    };
    double* o0 = row(have0 ? q0 : 0);
    double* o1 = row(have1 ? q0 + 1 : 0);
    auto store = [&](auto range) {          // as in kx_zfwd
        for (int p = t; p < M; p += T) {
            const fxc a = col[fx_pad(p)];
            if (have0) o0[p] = range.value && bad ? fx_nan() : fx_to<range.value>(a.x, eb);
            if (have1) o1[p] = range.value && bad ? fx_nan() : fx_to<range.value>(a.y, eb);
        }
    };
    if (fx_normal(eb) && !bad) store(std::false_type());
    else store(std::true_type());
}

// ---- host launchers ----------------------------------------------------------
// which: 0 axial inverse, 1 theta rows, 2 axial forward, for the azimuthal
// columns col0 .. col0 + ncols - 1 of one case (ds == nullptr) or of every plane
// in ymap (nplanes rows).
template <int M> static void fx_launch_z(const TcDev& d, const TcDev* ds, const int2* ymap, int nplanes, int which,
                                         cudaStream_t s, int col0, int ncols) {
    int lct = 0;
    while ((2 << lct) <= d.ztile && (2 << lct) <= fx_z_columns<M>()) ++lct;      // ztile is 1, 2, 4 or 8
    const int ct = 1 << lct, nth = fx_z_threads<M>(ct), sm = ct * (M + M / 8) * (int)sizeof(fxc);
    if (which == 0 || which == 3)           // 3: one field (d.u), for the physical output
        kx_zinv<M><<<dim3(ncols / ct, nplanes, which == 0 ? 3 : 1), nth, sm, s>>>(d, ds, ymap, col0, lct);
    else if (d.prec == 2) kx_zfwd<M, true><<<dim3(ncols / ct, nplanes, TC_NPROD), nth, sm, s>>>(d, ds, ymap, col0, lct);
    else kx_zfwd<M, false><<<dim3(ncols / ct, nplanes, TC_NPROD), nth, sm, s>>>(d, ds, ymap, col0, lct);
}
template <int M> static void fx_launch_rows(const TcDev& d, const TcDev* ds, const int2* ymap, int nplanes, cudaStream_t s) {
    const int pairs = (d.Mzx + 1) / 2;
    kx_rows<M><<<dim3((pairs + FxPlan<M>::G - 1) / FxPlan<M>::G, nplanes), 3 * FxPlan<M>::W, fx_rows_smem<M>(), s>>>(d, ds, ymap);
}
template <int M> static void fx_launch_phys(const TcDev& d, int4 zr, cudaStream_t s) {
    const int pairs = (d.Mz + 1) / 2;
    kx_phys<M><<<dim3((pairs + FxPlan<M>::G - 1) / FxPlan<M>::G, d.Nr), FxPlan<M>::W, fx_rows_smem<M>() / 5, s>>>(d, zr);
}
template <int M> static int4 fx_order() { return make_int4(FxPlan<M>::R0, FxPlan<M>::R1, fx_stride<M, 0>(), fx_stride<M, 1>()); }
// shared-memory opt-in of the kernels of length M that the axial or the theta
// transforms use, or (phys) those of the physical output in either direction
template <int M> static void fx_attributes(bool rows, bool z, bool phys, cudaError_t& e) {
    auto set = [&](const void* f, int bytes) {
        const cudaError_t r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (r != cudaSuccess) e = r;
    };
    const int zb = fx_z_columns<M>() * (M + M / 8) * (int)sizeof(fxc);
    if (z || phys) set((const void*)kx_zinv<M>, zb);
    if (z) { set((const void*)kx_zfwd<M, false>, zb); set((const void*)kx_zfwd<M, true>, zb); }
    if (rows) set((const void*)kx_rows<M>, fx_rows_smem<M>());
    if (rows || phys) set((const void*)kx_phys<M>, fx_rows_smem<M>() / 5);
}
#define FX_CASE_Z(M) case M: fx_launch_z<M>(d, ds, ymap, nplanes, which, s, col0, ncols); return true;
#define FX_CASE_ROWS(M) case M: fx_launch_rows<M>(d, ds, ymap, nplanes, s); return true;
#define FX_CASE_PHYS(M) case M: fx_launch_phys<M>(d, zr, s); return true;
#define FX_CASE_ORDER(M) case M: zr = fx_order<M>(); return true;
#define FX_CASE_ATTR(M) if (Mtx == M || Mzx == M) fx_attributes<M>(Mtx == M, Mzx == M, false, e);
#define FX_CASE_PHYS_ATTR(M) fx_attributes<M>(false, false, true, e);
// The launchers of one group of lengths: false for a length of another group.
#define FX_INSTANTIATE(TAG, LIST)                                                                                        \
    bool tc_fx_z_##TAG(const TcDev& d, const TcDev* ds, const int2* ymap, int nplanes, int which, cudaStream_t s,        \
                       int col0, int ncols) {                                                                           \
        switch (d.Mzx) { LIST(FX_CASE_Z) default: return false; }                                                       \
    }                                                                                                                   \
    bool tc_fx_rows_##TAG(const TcDev& d, const TcDev* ds, const int2* ymap, int nplanes, cudaStream_t s) {              \
        switch (d.Mtx) { LIST(FX_CASE_ROWS) default: return false; }                                                    \
    }                                                                                                                   \
    bool tc_fx_phys_##TAG(const TcDev& d, int4 zr, cudaStream_t s) { switch (d.Mt) { LIST(FX_CASE_PHYS) default: return false; } } \
    bool tc_fx_order_##TAG(int M, int4& zr) { switch (M) { LIST(FX_CASE_ORDER) default: return false; } }                \
    bool tc_fx_attributes_##TAG(int Mtx, int Mzx, cudaError_t& e) { LIST(FX_CASE_ATTR) return e == cudaSuccess; }        \
    void tc_fx_phys_attributes_##TAG(cudaError_t& e) { LIST(FX_CASE_PHYS_ATTR) }
