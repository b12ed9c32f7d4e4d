// complex128 DFT stages in 64-bit fixed point.
//
// GB300 issues 2 FP64 operations per clock and SM, but 128 32-bit integer additions and 64 32 x 32 -> 64-bit
// multiply-adds (measured: add.f64 1.7, fma.f64 2.0, a 64-bit integer addition 42, mad.wide 64 lanes per clock
// and SM), so a DFT in FP64 arithmetic is bound by that unit alone: about 6 clocks per element and radix-8
// stage with its twiddle, where HBM delivers an element per 1.4 clocks.  Here a group of values that one
// sub-DFT mixes is brought to a common exponent E (that of its largest component), held as signed 64-bit
// integers through all its stages, and rounded back to FP64 once at the end.
//
// Scale: a component x becomes x 2^(K - (E - 1023)), |x| < 2^(E - 1022), with K = 59 - rho for a first stage of
// 2^rho points, so that after that stage every modulus is below 2^60.5 (2^(K + 1.5) grown by 2^rho); before each
// later stage of 2^rho points the values are scaled down by 2^rho (rounding), which restores the same bound.
// Roundings are about a unit at 2^K = 2^56 or more of the largest input, against 2^53 for FP64: the error is below
// FP64's.  Twiddles are Q62 (+1 is 1 - 2^-62); a product keeps the high 64 bits, the low x low partial product
// being left out (its mean is added as a constant).
//
// The way back to FP64 is the conversion instruction (2 per clock and SM, on the otherwise idle FP64 unit) and an
// integer addition to the exponent; done in integer instructions it took 44 of a complex value's 271 in a two-stage
// pass and the integer pipe was the bound.
//
// A group with a component that is infinite, NaN, or too small or large to be scaled (fx_plain) is left to the
// FP64 path of the caller.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_device.cuh"

namespace fftu {

template <> struct real_of<longlong2> { using type = long long; };

// Lowest biased exponent a group is scaled with: results stay normal down to 2^-(128 - 63 + 40) of it.
constexpr int kFxMinExp = 128;
constexpr int kFxMaxExp = 1984;

__device__ __forceinline__ double2 fx_bits(longlong2 v) {
    return mk<double2>(__longlong_as_double(v.x), __longlong_as_double(v.y));
}
// Magnitude key of a value: the larger of its components' high words without sign.
__device__ __forceinline__ int fx_key(double2 v) {
    const int a = __double2hiint(v.x) & 0x7fffffff, b = __double2hiint(v.y) & 0x7fffffff;
    return a > b ? a : b;
}
// The largest key of a group of values: false when the group needs the FP64 path.  A zero key can hide
// denormals in the low words (lo_or: their OR); exact zeros are served.
__device__ __forceinline__ bool fx_plain(int key, unsigned lo_or) {
    const int e = key >> 20;
    return (e >= kFxMinExp && e <= kFxMaxExp) || (key == 0 && lo_or == 0);
}
// Biased exponent the group is scaled with.
__device__ __forceinline__ int fx_exp(int key) {
    const int e = key >> 20;
    return e > kFxMinExp ? e : kFxMinExp;
}

constexpr int kFxTop = 59;  // K + rho of the first stage

// x 2^(K - (E - 1023)), truncated toward zero (unbiased for data of both signs); |x| < 2^(E - 1022).
// K in [52, 62).
template <int K> __device__ __forceinline__ long long fx_in(double x, int E) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const unsigned h = __funnelshift_l(lo, mh, K - 52), l = lo << (K - 52);
    const int d = E - ((hi >> 20) & 0x7ff);  // >= 0; zeros and denormals: d >= kFxMinExp, shifted out
    const int d2 = d > 32 ? d - 32 : 0;
    unsigned l2 = __funnelshift_rc(l, h, d);  // shifts clamp at 32
    l2 = __funnelshift_rc(l2, 0u, d2);
    const unsigned h2 = __funnelshift_rc(h, 0u, d);
    const long long s = (long long)(hi >> 31);
    const long long m = (long long)(((unsigned long long)h2 << 32) | l2);
    return (m ^ s) - s;
}

// The double nearest to v 2^e (normal results); v = 0 gives +0.
__device__ __forceinline__ double fx_out(long long v, int e) {
    const double y = __ll2double_rn(v);
    const int hi = __double2hiint(y);
    return __hiloint2double(hi == 0 ? 0 : hi + (e << 20), __double2loint(y));
}
// Exponent of the results of a DFT of 2^lg points whose inputs were scaled with E.
__device__ __forceinline__ int fx_out_exp(int E, int lg) { return E - 1023 - kFxTop + lg; }

// Twiddle in Q62, each part as hi 2^31 + lo with 0 <= lo < 2^31: (re hi, re lo, im hi, im lo).
__device__ __forceinline__ int2 fx_q62(double w) {
    long long q = __double2ll_rn(w * 4611686018427387904.0);
    if (q > 4611686018427387903ll) q = 4611686018427387903ll;
    return make_int2((int)(q >> 31), (int)(q & 0x7fffffff));
}

// a w (forward) or a conj(w) (inverse); |a| < 2^60.5, so that both cross products fit one accumulator.
template <int DIR> __device__ __forceinline__ longlong2 fx_cmul(longlong2 a, int4 w) {
    const int rh = (int)(a.x >> 31), rl = (int)(a.x & 0x7fffffff);
    const int ih = (int)(a.y >> 31), il = (int)(a.y & 0x7fffffff);
    constexpr long long half = 1ll << 30;
    longlong2 r;
    // re = ar wr - ai wi (forward), ar wr + ai wi (inverse)
    const int sih = DIR < 0 ? -ih : ih, sil = DIR < 0 ? -il : il;
    long long A = (long long)rh * w.x + (long long)sih * w.z;
    long long M = (long long)rh * w.y + (long long)sih * w.w + (long long)rl * w.x + (long long)sil * w.z + half +
                  (DIR < 0 ? 0 : half);
    r.x = A + (M >> 31);
    // im = ai wr + ar wi (forward), ai wr - ar wi (inverse)
    const int srh = DIR < 0 ? rh : -rh, srl = DIR < 0 ? rl : -rl;
    A = (long long)ih * w.x + (long long)srh * w.z;
    M = (long long)ih * w.y + (long long)srh * w.w + (long long)il * w.x + (long long)srl * w.z + half +
        (DIR < 0 ? half : 0);
    r.y = A + (M >> 31);
    return r;
}
// The twiddle w 2^-sh.
__device__ __forceinline__ int4 fx_scale_tw(int4 w, int sh) {
    if (sh == 0) return w;
    const long long half = 1ll << (sh - 1);
    const long long re = (((long long)w.x << 31) + w.y + half) >> sh, im = (((long long)w.z << 31) + w.w + half) >> sh;
    return make_int4((int)(re >> 31), (int)(re & 0x7fffffff), (int)(im >> 31), (int)(im & 0x7fffffff));
}
// a c for a constant c > 0 in Q62.
template <long long C> __device__ __forceinline__ long long fx_mulc(long long a) {
    constexpr int ch = (int)(C >> 31), cl = (int)(C & 0x7fffffff);
    const int h = (int)(a >> 31), l = (int)(a & 0x7fffffff);
    const long long M = (long long)h * cl + (long long)l * ch + (1ll << 30);
    return (long long)h * ch + (M >> 31);
}
constexpr long long kFxH = 3260954456333195553ll;   // sqrt(1/2) 2^62
constexpr long long kFxC1 = 4260642322793532497ll;  // cos(pi/8) 2^62
constexpr long long kFxS1 = 1764815834521887442ll;  // sin(pi/8) 2^62

// x (1 + DIR i) / sqrt 2
template <int DIR> __device__ __forceinline__ longlong2 fx_w8(longlong2 a) {
    return mk<longlong2>(fx_mulc<kFxH>(a.x - DIR * a.y), fx_mulc<kFxH>(a.y + DIR * a.x));
}
// x (-1 + DIR i) / sqrt 2
template <int DIR> __device__ __forceinline__ longlong2 fx_w8_3(longlong2 a) {
    return mk<longlong2>(fx_mulc<kFxH>(-a.x - DIR * a.y), fx_mulc<kFxH>(DIR * a.x - a.y));
}

template <int DIR> __device__ __forceinline__ void fx_dft8(longlong2 *v) {
    longlong2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    longlong2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    bfly4<DIR>(e0, e1, e2, e3);
    bfly4<DIR>(o0, o1, o2, o3);
    o1 = fx_w8<DIR>(o1);
    o2 = mul_w4<DIR>(o2);
    o3 = fx_w8_3<DIR>(o3);
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1);
    v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2);
    v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3);
    v[7] = csub(e3, o3);
}

// x (C + DIR S i) for constants in Q62 of either sign
template <int DIR, long long C, long long S> __device__ __forceinline__ longlong2 fx_mulw(longlong2 a) {
    constexpr long long c = C < 0 ? -C : C, s = S < 0 ? -S : S;
    const long long xr = fx_mulc<c>(a.x), yr = fx_mulc<c>(a.y), xi = fx_mulc<s>(a.x), yi = fx_mulc<s>(a.y);
    const long long cr = C < 0 ? -xr : xr, cj = C < 0 ? -yr : yr;
    constexpr int g = (S < 0 ? -1 : 1) * DIR;
    return mk<longlong2>(cr - g * yi, cj + g * xi);
}

template <int DIR> __device__ __forceinline__ void fx_dft16(longlong2 *v) {
#pragma unroll
    for (int q = 0; q < 4; ++q) bfly4<DIR>(v[q], v[q + 4], v[q + 8], v[q + 12]);
    v[1 + 4 * 1] = fx_mulw<DIR, kFxC1, kFxS1>(v[1 + 4 * 1]);
    v[1 + 4 * 2] = fx_w8<DIR>(v[1 + 4 * 2]);
    v[1 + 4 * 3] = fx_mulw<DIR, kFxS1, kFxC1>(v[1 + 4 * 3]);
    v[2 + 4 * 1] = fx_w8<DIR>(v[2 + 4 * 1]);
    v[2 + 4 * 2] = mul_w4<DIR>(v[2 + 4 * 2]);
    v[2 + 4 * 3] = fx_w8_3<DIR>(v[2 + 4 * 3]);
    v[3 + 4 * 1] = fx_mulw<DIR, kFxS1, kFxC1>(v[3 + 4 * 1]);
    v[3 + 4 * 2] = fx_w8_3<DIR>(v[3 + 4 * 2]);
    v[3 + 4 * 3] = fx_mulw<DIR, -kFxC1, -kFxS1>(v[3 + 4 * 3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) bfly4<DIR>(v[0 + 4 * k], v[1 + 4 * k], v[2 + 4 * k], v[3 + 4 * k]);
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int t = k + 1; t < 4; ++t) {
            longlong2 tmp = v[t + 4 * k];
            v[t + 4 * k] = v[k + 4 * t];
            v[k + 4 * t] = tmp;
        }
}

template <int R, int DIR> __device__ __forceinline__ void fx_dft(longlong2 *v) {
    if constexpr (R == 2) {
        dft2<DIR>(v);
    } else if constexpr (R == 4) {
        dft4<DIR>(v);
    } else if constexpr (R == 8) {
        fx_dft8<DIR>(v);
    } else if constexpr (R == 16) {
        fx_dft16<DIR>(v);
    }
}

// a 2^-sh (rounding).
__device__ __forceinline__ longlong2 fx_scale_down(longlong2 a, int sh) {
    const long long half = (1ll << sh) >> 1;
    return mk<longlong2>((a.x + half) >> sh, (a.y + half) >> sh);
}

template <int R> __host__ __device__ constexpr int lg_of() { return R == 2 ? 1 : R == 4 ? 2 : R == 8 ? 3 : R == 16 ? 4 : R == 32 ? 5 : 0; }

}  // namespace fftu
