// complex128 DFT stages in 64-bit fixed point.
//
// GB300 issues 2 FP64 operations per clock and SM, but 128 32-bit integer additions and 64 32 x 32 -> 64-bit
// multiply-adds (measured: add.f64 1.7, fma.f64 2.0, a 64-bit integer addition 42, mad.wide 64 lanes per clock
// and SM), so a DFT in FP64 arithmetic is bound by that unit alone: about 6 clocks per element and radix-8
// stage with its twiddle, where HBM delivers an element per 1.4 clocks.  Here a group of values that one
// sub-DFT mixes is brought to a common exponent E (that of its largest component), held as signed 64-bit
// integers through all its stages, and rounded back to FP64 once at the end.
//
// Scale: a component x becomes x 2^(K - (E - 1023)), |x| < 2^(E - 1022), with K = 60 - rho for a first stage of
// 2^rho points, so that after that stage every modulus is below 2^61.5 (2^(K + 1.5) grown by 2^rho); a stage that no other follows
// has K = 59 - rho.  Later stages scale down to stay below 2^61.5 where a product with a halved twiddle follows (2^60.5: with a whole
// one) and below 2^62.5 where none does.  Where shifts that suffice for any data are few in all (kFxFixed bits), they ride in the
// twiddle tables.
// Longer groups are shifted only as far as their data ask for it (block floating point): a stage finds the largest component that
// it leaves in each group (fx_size), and the next one shifts by what its own results need (fx_shift).  A fiber of the first stage
// whose values are all small in its group is held finer up to its store (fx_fine).
// Shifts for any data lose the low bits of groups that a few values dominate (an impulse, a spectral line, a point source over a
// background), whose later stages hardly grow.  Relative L2 error of 4096 points in four stages, ten seeds, with FP64 butterflies,
// with a shift by every stage's rho, and as here:
//   one nonzero value                   1.5e-16   1.9e-14   1.1e-16
//   1 over a background of 1e-3         2.3e-16   1.1e-14   2.6e-16
//   1 over a background of 1e-2         2.3e-16   9.9e-15   2.4e-16
//   plane wave                          1.6e-16   3.1e-16   7.6e-17
//   normal                              2.5e-16   4.1e-16   7.9e-17
//   uniform                             2.4e-16   1.5e-16   7.8e-17
// (4 to 2048 points: at most 1.04 times FP64's on any of these.)
//
// Twiddles are Q62 (+1 is 1 - 2^-62); a product keeps the high 64 bits, the low x low partial product
// being left out (its mean is added as a constant).
//
// The way back to FP64 is the conversion instruction (2 per clock and SM, on the otherwise idle FP64 unit) and an
// integer addition to the exponent; done in integer instructions it took 44 of a complex value's 271 in a two-stage
// pass and the integer pipe was the bound.
//
// A group whose largest component is below 2^-895 or above 2^962 is multiplied by a power of two before its conversion, and its
// results by the inverse.  One with an infinity or NaN is left to the FP64 path of the caller.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_device.cuh"

namespace fftu {

template <> struct real_of<longlong2> { using type = long long; };

// Lowest and highest biased exponent of a group that is scaled as it is: its results stay normal down to
// 2^-(128 - 63 + 40) of it.  Others: multiplied by 2^kFxBoost or 2^-kFxBoost first.
constexpr int kFxMinExp = 128;
constexpr int kFxMaxExp = 1984;
constexpr int kFxBoost = 960;
// Most bits that shifts for any data may take: 256 points.  Its relative error for one nonzero value is that of FP64 butterflies,
// 9.4e-17; with 5 bits (512 points) 1.5 times theirs.
constexpr int kFxFixed = 4;

__device__ __forceinline__ double2 fx_bits(longlong2 v) {
    return mk<double2>(__longlong_as_double(v.x), __longlong_as_double(v.y));
}
// Magnitude key of R values: the largest of their components' high words without sign; 0 only where all of them are zeros.
template <int R> __device__ __forceinline__ int fx_keys(const double2 *v) {
    int key = 0;
#pragma unroll
    for (int r = 0; r < R; ++r)
        key = __vimax3_s32(key, __double2hiint(v[r].x) & 0x7fffffff, __double2hiint(v[r].y) & 0x7fffffff);
    if (key == 0) {  // denormals whose high words are zero
        unsigned lo = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) lo |= (unsigned)__double2loint(v[r].x) | (unsigned)__double2loint(v[r].y);
        key = lo != 0;
    }
    return key;
}
__device__ __forceinline__ bool fx_finite(int key) { return key < 0x7ff00000; }
// Whether values up to this key are scaled as they are.
__device__ __forceinline__ bool fx_plain(int key) {
    const int e = key >> 20;
    return key == 0 || (e >= kFxMinExp && e <= kFxMaxExp);
}
// The power of two that a group of this key is multiplied by before its conversion (denormals then are ordinary values).
__device__ __forceinline__ int fx_boost(int key) { return fx_plain(key) ? 0 : (key >> 20) < kFxMinExp ? kFxBoost : -kFxBoost; }
template <int R> __device__ __forceinline__ void fx_times(double2 *v, int up) {  // v 2^up
    const double f = __hiloint2double((1023 + up) << 20, 0);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = mk<double2>(v[r].x * f, v[r].y * f);
}
// The key of such a group after the multiplication: the exponent and which it was (bits 31 and 0).
__device__ __forceinline__ int fx_far_key(int key, int boost) {
    return (int)(0x80000000u | (unsigned)(max(key >> 20, 1) + boost) << 20 | (boost > 0 ? 1u : 0u));
}
__device__ __forceinline__ bool fx_far(int key) { return key < 0; }
__device__ __forceinline__ int fx_far_boost(int key) { return key & 1 ? kFxBoost : -kFxBoost; }
// Biased exponent the group is scaled with.
__device__ __forceinline__ int fx_exp(int key) { return max((key >> 20) & 0x7ff, kFxMinExp); }

// Whether a fiber of the first stage whose own values have this key holds them at 2^kFxFine times its group's scale, up to its store:
// all of them are that much smaller than the largest of the group (a point source elsewhere), which would cost them their low bits.
constexpr int kFxFine = 3;
__device__ __forceinline__ bool fx_fine(int own, int group) { return (own >> 20) + kFxFine <= fx_exp(group) && !fx_far(group); }

constexpr int kFxTop = 60;  // K + rho of a first stage that others follow

// x 2^(K - (E - 1023)), truncated toward zero (unbiased for data of both signs); |x| < 2^(E - 1022).
// K in [52, 62).
template <int K> __device__ __forceinline__ long long fx_in(double x, int E) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const int d = E - ((hi >> 20) & 0x7ff);  // >= 0; denormals of groups not boosted: d >= kFxMinExp, shifted out
    const long long m = (long long)(((((unsigned long long)mh << 32) | lo) << (K - 52)) >> min(d, 63));
    return hi < 0 ? -m : m;
}

// The double nearest to v 2^e (normal results); v = 0 gives +0.
__device__ __forceinline__ double fx_out(long long v, int e) {
    const double y = __ll2double_rn(v);
    const int hi = __double2hiint(y);
    return __hiloint2double(hi == 0 ? 0 : hi + (e << 20), __double2loint(y));
}
// Exponent of the results of a first stage of 2^rho points with K = kFxTop - rho, shifted by `shift` in all.
__device__ __forceinline__ int fx_out_exp(int E, int rho, int shift) { return E - 1023 - kFxTop + rho + shift; }

// Twiddle in Q62, each part as hi 2^31 + lo with 0 <= lo < 2^31: (re hi, re lo, im hi, im lo).
__device__ __forceinline__ int2 fx_q62(double w) {
    long long q = __double2ll_rn(w * 4611686018427387904.0);
    if (q > 4611686018427387903ll) q = 4611686018427387903ll;
    return make_int2((int)(q >> 31), (int)(q & 0x7fffffff));
}

// a w (forward) or a conj(w) (inverse); |a| < 2^60.5, or |a| < 2^61.5 and w halved, so that both cross products fit one
// accumulator.  A product of 0 is 0.
template <int DIR> __device__ __forceinline__ longlong2 fx_cmul(longlong2 a, int4 w) {
    const int rh = (int)(a.x >> 31), rl = (int)(a.x & 0x7fffffff);
    const int ih = (int)(a.y >> 31), il = (int)(a.y & 0x7fffffff);
    constexpr long long half = 1ll << 30;
    longlong2 r;
    // re = ar wr - ai wi (forward), ar wr + ai wi (inverse)
    const int sih = DIR < 0 ? -ih : ih, sil = DIR < 0 ? -il : il;
    long long A = (long long)rh * w.x + (long long)sih * w.z;
    long long M = (long long)rh * w.y + (long long)sih * w.w + (long long)rl * w.x + (long long)sil * w.z + half +
                  (DIR < 0 ? 0 : half - 1);
    r.x = A + (M >> 31);
    // im = ai wr + ar wi (forward), ai wr - ar wi (inverse)
    const int srh = DIR < 0 ? rh : -rh, srl = DIR < 0 ? rl : -rl;
    A = (long long)ih * w.x + (long long)srh * w.z;
    M = (long long)ih * w.y + (long long)srh * w.w + (long long)il * w.x + (long long)srl * w.z + half +
        (DIR < 0 ? half - 1 : 0);
    r.y = A + (M >> 31);
    return r;
}
// The twiddle w 2^-sh.
__device__ __forceinline__ int4 fx_scale_tw(int4 w, int sh) {
    const long long half = (1ll << sh) >> 1;
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

// A bound of R stored values: every component is at most 2^32 (x + 1) in size.
template <int R> __device__ __forceinline__ int fx_size(const longlong2 *v) {
    int hi = 0, lo = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int a = (int)(v[r].x >> 32), b = (int)(v[r].y >> 32);
        hi = __vimax3_s32(hi, a, b);
        lo = __vimin3_s32(lo, a, b);
    }
    return max(hi, ~lo);
}
// The shift of a stage of 2^rho points on a group of that size, so that its results stay below 2^60.5 (room 4), 2^61.5 (3) or
// 2^62.5 (2): components below 2^b, b = 64 - clz, moduli below 2^(b + 1/2 + rho) after the stage.
constexpr int kFxRoomProduct = 4, kFxRoomHalved = 3, kFxRoomNone = 2;
__device__ __forceinline__ int fx_shift(int size, int rho, int room) { return max(0, rho + room - __clz(size)); }
// Raise a group's entry to at least `value`; warp: all lanes raise the same one (32 atomics on one word take turns).
__device__ __forceinline__ void fx_raise(int *entry, int value, int warp) {
    if (warp) {
        value = __reduce_max_sync(~0u, value);
        if ((threadIdx.x & 31) != 0) return;
    }
    atomicMax(entry, value);
}
// a 2^-sh (rounding).
__device__ __forceinline__ longlong2 fx_scale_down(longlong2 a, int sh) {
    const long long half = (1ll << sh) >> 1;
    return mk<longlong2>((a.x + half) >> sh, (a.y + half) >> sh);
}
__device__ __forceinline__ long long fx_shr(long long a, int sh) {  // sh < 32
    const unsigned lo = __funnelshift_r((unsigned)a, (unsigned)(a >> 32), sh);
    return (long long)(((unsigned long long)(unsigned)((int)(a >> 32) >> sh) << 32) | lo);
}
// The values of a stage times 2^-sh, rounded down; fx_mend after the DFT adds what that takes away on average, (1 - 2^-sh) / 2 of
// a unit from each value and so R times it from output 0 (one addition per DFT in place of one per value).
template <int R> __device__ __forceinline__ void fx_floor(longlong2 *v, int sh) {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = mk<longlong2>(fx_shr(v[r].x, sh), fx_shr(v[r].y, sh));
}
template <int R> __device__ __forceinline__ void fx_mend(longlong2 *v, int sh) {
    const int c = ((R << sh) - R) >> (sh + 1);
    v[0].x += c;
    v[0].y += c;
}

template <int R> __host__ __device__ constexpr int lg_of() { return R == 2 ? 1 : R == 4 ? 2 : R == 8 ? 3 : R == 16 ? 4 : R == 32 ? 5 : 0; }

}  // namespace fftu
