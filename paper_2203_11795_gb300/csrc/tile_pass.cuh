// Tile passes: one or more adjacent axes in one HBM round trip, all their positions in a tile.
//
// Two forms.  Phase A (Superstep 0 and the Put of Algorithm 2.3, Sec. 2.2): on each axis F_{n_l/p_l} on every residue
// class s, the twiddle w_{n_l}^{k s}, and the position s n_l/p_l + k.  Whole axes: where the library chooses the grid,
// fftu_exec needs only the transform and not the data between the supersteps.  Superstep 0, the Put and Superstep 2
// act on each axis by itself (tensor products, Sec. 2.2), so an axis whose length fits a tile runs all three inside
// shared memory, as the radix split (Sec. 2.1.1, eq. radix) of one F_{n_l}: phase A and phase B of that axis cost one
// pass instead of two.
//
// The array is viewed as [outer][G][inner] with G the product of the pass' axes.  A tile holds all G positions for
// V = 2^lg_v adjacent inner positions (inner > 1) or V adjacent outer positions (inner = 1, contiguous memory).
// Tile index e: [g][v] or [v][g], g row-major over the axes, so tile order is memory order.  Each axis is split
// into digits of at most 5 bits, highest first; a stage transforms one digit in place:
// A pass of one stage stores from the registers it loaded into (phase A: after a barrier).
//   x[j + T r] (j in [T]: the axis' lower digits) -> F_R over r -> k in the digit's place, times w_{R T}^{k j}.
// In phase A the digits split m (i = s + p m) and s, the lowest bits of the axis, stays in place until the store.
// The first stage loads its fibers from HBM into registers and the last one stores them to HBM, with the digits
// of each axis in reverse (k = k_1 + R_1 k_2 + ...); between stages the tile is in shared memory, one barrier per
// stage (a stage writes the slots it read).  Every load of a tile precedes its stores, so a pass may be in place.
//
// Shared slot of e: e ^ ((e >> swz[0]) & m) ^ ((e >> swz[1]) & m), m = 15 (8-byte elements) or 7 (16-byte): linear over
// XOR, so the slots of a fiber are the first one's XOR stage constants; the planner picks the shifts that leave
// the stages' accesses without bank conflicts.
//
// Arithmetic: FP32 (complex64); for complex128 fixed point (fixed64.cuh) with one exponent per sub-DFT, and a tile with
// an infinity or NaN is run again in FP64 from its input.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "fft_device.cuh"
#include "fftu_internal.h"
#include "fixed64.cuh"

namespace fftu {

// ARITH of a tile pass; kTpF32w: complex64 with radix-32 stages (a kernel of its own, with twice the registers)
constexpr int kTpF32 = 0, kTpFixed = 1, kTpF64 = 2, kTpF32w = 3;
// OPT bits: the pointwise product in the last store; twiddles straight from the root tables instead of the stages' shared
// tables; a pass of one stage; passes that follow one another in one launch (loads from L2); complex128 stages that shift
// their inputs, by their groups' sizes or as any data need (a kernel of its own: the others would lose 2%).
constexpr int kTpMul = 1, kTpGlobalTw = 2, kTpSingle = 4, kTpChain = 8, kTpShifts = 16;
template <int ARITH> struct tp_type;
template <> struct tp_type<kTpF32> { using elem = float2; using work = float2; using tw = float2; };
template <> struct tp_type<kTpF32w> : tp_type<kTpF32> {};
template <> struct tp_type<kTpFixed> { using elem = double2; using work = longlong2; using tw = int4; };
template <> struct tp_type<kTpF64> { using elem = double2; using work = double2; using tw = double2; };

template <int ARITH, typename P> __device__ __forceinline__ int tp_slot(const P &a, int e) {
    constexpr int m = sizeof(typename tp_type<ARITH>::elem) == 8 ? 15 : 7;
    return e ^ ((e >> a.swz[0]) & m) ^ ((e >> a.swz[1]) & m);
}
// Not unrolled: the fields (kernel parameters) would otherwise be kept in registers across a CTA's tiles.
__device__ __forceinline__ unsigned tp_fields(const BitField *f, int n, unsigned x) {
    unsigned o = 0;
#pragma unroll 1
    for (int i = 0; i < n; ++i) o |= ((x >> f[i].sh) & f[i].mask) << f[i].dst;
    return o;
}

template <int ARITH, int DIR>
__device__ __forceinline__ typename tp_type<ARITH>::work tp_twiddle(typename tp_type<ARITH>::work x,
                                                                    typename tp_type<ARITH>::tw w) {
    if constexpr (ARITH == kTpFixed) return fx_cmul<DIR>(x, w);
    else return cmul(x, dirw<DIR>(w));
}
template <int ARITH, int DIR, int R> __device__ __forceinline__ void tp_dft(typename tp_type<ARITH>::work *v) {
    if constexpr (ARITH == kTpFixed) fx_dft<R, DIR>(v);
    else dft_small<R, DIR>(v);
}

// Load of an input element.  In a launch whose passes follow one another other SMs wrote it during the kernel: from L2.
template <int OPT, typename E> __device__ __forceinline__ E tp_load(const E *p) {
    if constexpr ((OPT & kTpChain) != 0) return __ldcg(p);
    else return *p;
}
// Shared slots of the values of the fiber whose value 0 is at `slot`.  A launch of one pass has the XOR constants of all
// values in the constant bank, an operand of the XOR.  A batch has its descriptors in shared memory: there a value's slot
// is the slot of the value without its lowest bit, XOR that bit's constant (5 loads a stage instead of 32 or 64).
template <typename STAGE, int R> struct TpSlots {
    const STAGE &s;
    int slot, at[std::is_same_v<STAGE, TileStage> ? 1 : R];
    __device__ __forceinline__ TpSlots(const STAGE &s_, int slot_) : s(s_), slot(slot_) {
        if constexpr (!std::is_same_v<STAGE, TileStage>) {
            asm volatile("" : "+r"(slot));  // computed again for a stage's stores rather than kept in registers
            at[0] = slot;
        }
    }
    __device__ __forceinline__ int operator()(int r) {  // r ascending, known at compile time
        if constexpr (std::is_same_v<STAGE, TileStage>) {
            return slot ^ s.rx[r];
        } else {
            const int low = r & -r;
            if (r) at[r] = at[r ^ low] ^ s.rb[low == 1 ? 0 : low == 2 ? 1 : low == 4 ? 2 : low == 8 ? 3 : 4];
            return at[r];
        }
    }
};
// The column of stage s's twiddle table for the fiber at tile index e0.
__device__ __forceinline__ int tp_column(const TileStageCore &s, int e0) {
    const int low = (e0 >> s.lo) & ((1 << (s.tw_kind == 1 ? s.lg_q : s.lg_p)) - 1);
    if (s.tw_kind == 1) return low;
    const int up = (e0 >> (s.pos + s.lg_r)) & ((1 << (s.lg_q - s.lg_p)) - 1);
    return low | (up << s.lg_p);
}
// Exponent of w_n for output digit r in column q.
__device__ __forceinline__ unsigned tp_exponent(const TileStageCore &s, unsigned r, unsigned q) {
    if (s.tw_kind == 1) return (r * q) << s.lg_step;
    const unsigned kp = tp_fields(s.k, s.nk, q >> s.lg_p);
    return (kp + (r << s.lg_step)) * (q & ((1u << s.lg_p) - 1));
}
// The twiddles of a stage on its fiber.
template <int ARITH, int DIR, int OPT, int R>
__device__ __forceinline__ void tp_twiddles(const TileStageCore &s, int e0, typename tp_type<ARITH>::work *v,
                                            const typename tp_type<ARITH>::tw *tabs) {
    const int q = tp_column(s, e0);
    if constexpr (ARITH == kTpF64) {
        const double2 *tw = static_cast<const double2 *>(s.tw64);
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = cmul(v[r], dirw<DIR>(tw[tp_exponent(s, r, q)]));
    } else if constexpr ((OPT & kTpGlobalTw) != 0) {
        const typename tp_type<ARITH>::tw *tw = static_cast<const typename tp_type<ARITH>::tw *>(s.tw);
        if (s.tw_kind == 2) v[0] = tp_twiddle<ARITH, DIR>(v[0], __ldg(tw + tp_exponent(s, 0, q)));
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = tp_twiddle<ARITH, DIR>(v[r], __ldg(tw + tp_exponent(s, r, q)));
    } else {
        const typename tp_type<ARITH>::tw *t = tabs + s.tab + q;
        if (s.tw_kind == 2) v[0] = tp_twiddle<ARITH, DIR>(v[0], t[0]);
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = tp_twiddle<ARITH, DIR>(v[r], t[r << s.lg_q]);
    }
}

// One stage of radix R.  FIRST: from src; LAST: to dst (both: a pass of one digit).  Returns false (kTpFixed, FIRST)
// when the tile needs FP64 arithmetic.  emax (kTpFixed): per group the largest key, then the sizes (fx_size)
// that some stages leave for the next one.
template <int ARITH, int DIR, int OPT, int R, bool FIRST, bool LAST, typename P>
__device__ __forceinline__ bool tp_stage(const P &a, int si, typename tp_type<ARITH>::work *sm,
                                         const typename tp_type<ARITH>::tw *tabs, int *emax,
                                         const typename tp_type<ARITH>::elem *src,
                                         typename tp_type<ARITH>::elem *dst) {
    using T = tp_type<ARITH>;
    using W = typename T::work;
    constexpr int RHO = lg_of<R>();
    constexpr bool kShifts = ARITH == kTpFixed && (OPT & kTpShifts) != 0;
    int phi0 = threadIdx.x;
    asm volatile("" : "+r"(si), "+r"(phi0));  // per tile: nothing derived from them is kept in registers across tiles
    const auto &s = a.st[si];
    const int fibers = 1 << (a.lg_tile - RHO);
    // kTpFixed, FIRST: one fiber per thread at most (blockDim >= fibers), every thread at the barrier
    constexpr bool kOnce = ARITH == kTpFixed && FIRST;
#pragma unroll 1
    for (int phi = phi0; kOnce || phi < fibers; phi += blockDim.x) {
        int e0;
        if constexpr (LAST && !FIRST) e0 = (int)tp_fields(a.last, a.nlast, (unsigned)phi);
        else e0 = ((phi >> s.pos) << (s.pos + RHO)) | (phi & ((1 << s.pos) - 1));
        W v[R];
        int slot = 0;
        if constexpr (!(FIRST && LAST)) slot = tp_slot<ARITH>(a, e0);
        int key = 0;
        [[maybe_unused]] int *em = nullptr;   // kTpFixed: the group's entries
        [[maybe_unused]] bool fine = false;  // a fiber of small values in its group (fx_fine)
        if constexpr (FIRST) {
            const unsigned off = a.lg_inner < 0 ? (unsigned)e0
                                                : (((unsigned)e0 >> a.lg_v) << a.lg_inner) | (e0 & ((1 << a.lg_v) - 1));
            const typename T::elem *p = src + off;
            if constexpr (ARITH == kTpFixed) {
                double2 x[R];
                if (phi < fibers) {
#pragma unroll
                    for (int r = 0; r < R; ++r) x[r] = tp_load<OPT>(p + ((size_t)r << a.in_bit));
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) x[r] = mk<double2>(0.0, 0.0);
                }
                key = fx_keys<R>(x);
                em = emax + tp_fields(a.group, a.ngroup, (unsigned)e0);
                if (phi < fibers) fx_raise(em, key, s.warp);
                if (__syncthreads_or(!fx_plain(key))) {  // rare: a fiber, though perhaps no group, is out of range
                    const int group = phi < fibers ? *em : 0, up = fx_boost(group);
                    if (__syncthreads_or(!fx_finite(group))) return false;
                    if (up) {
                        fx_times<R>(x, up);
                        *em = key = fx_far_key(group, up);
                    }
                    __syncthreads();
                }
                if (phi >= fibers) break;
                const int own = key;
                key = *em;
                if constexpr (!LAST) fine = fx_fine(own, key);
                const int E = fx_exp(key) - (fine ? kFxFine : 0);
#pragma unroll
                for (int r = 0; r < R; ++r)
                    v[r] = mk<longlong2>(fx_in<kFxTop - LAST - RHO>(x[r].x, E), fx_in<kFxTop - LAST - RHO>(x[r].y, E));
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = tp_load<OPT>(p + ((size_t)r << a.in_bit));
            }
        } else {
            TpSlots<std::remove_const_t<std::remove_reference_t<decltype(s)>>, R> at(s, slot);
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = sm[at(r)];
        }
        [[maybe_unused]] int sh = 0, shift = FIRST ? 1 : a.shifts.fixed;  // kTpFixed: of all stages (a first stage alone: one less in K)
        if constexpr (ARITH == kTpFixed && !FIRST) {
            if constexpr (LAST || kShifts) em = emax + tp_fields(a.group, a.ngroup, (unsigned)e0);
            if constexpr (LAST) key = *em;
            if constexpr (LAST && kShifts) {
#pragma unroll 1
                for (int i = 1; i <= a.shifts.sizes; ++i)
                    shift += fx_shift(em[i << a.lg_groups], a.shifts.lg[i], a.shifts.room[i]);
            }
            if constexpr (kShifts) {
                sh = s.pre;
                if (s.size_in) sh = fx_shift(em[s.size_in << a.lg_groups], RHO, s.tw_kind ? kFxRoomHalved : kFxRoomNone);
                if (s.pre || s.size_in) fx_floor<R>(v, sh);
            }
        }
        tp_dft<ARITH, DIR, R>(v);
        if constexpr (kShifts && !FIRST) {
            if (s.pre || s.size_in) fx_mend<R>(v, sh);
        }
        if constexpr (LAST) {
            if (s.tw_kind) tp_twiddles<ARITH, DIR, OPT, R>(s, e0, v, tabs);  // phase A: w_n^{k s} of the last axis
            typename T::elem *q;
            if constexpr (FIRST) {
                if (a.once) __syncthreads();  // every thread has one fiber: all loads of the tile are done
            }
            q = dst + tp_fields(a.out, a.nout, (unsigned)phi);
            [[maybe_unused]] const int x0 = fx_out_exp(fx_exp(key), a.st[0].lg_r, shift) + a.lg_scale;
            [[maybe_unused]] const auto f = (typename real_of<W>::type)a.scale;
            [[maybe_unused]] const bool far = ARITH == kTpFixed && fx_far(key);
            // kTpMul: the pointwise factor at the same natural index
            [[maybe_unused]] const typename T::elem *m =
                (OPT & kTpMul) ? static_cast<const typename T::elem *>(a.mul) + (q - static_cast<typename T::elem *>(a.dst)) : nullptr;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                typename T::elem y;
                if constexpr (ARITH == kTpFixed) y = mk<double2>(fx_out(v[r].x, x0), fx_out(v[r].y, x0));
                else y = a.lg_scale != 0 ? cscale(v[r], f) : v[r];
                if constexpr ((OPT & kTpMul) != 0) {
                    if (!far) y = cmul(y, m[(size_t)r << a.out_bit]);
                }
                q[(size_t)r << a.out_bit] = y;
            }
            if constexpr (ARITH == kTpFixed) {
                if (far) {  // rare: the stored values are read again, which leaves the loop above as it is without
#pragma unroll 1
                    for (int r = 0; r < R; ++r) {
                        double2 *y = q + ((size_t)r << a.out_bit);
                        fx_times<1>(y, -fx_far_boost(key));
                        if constexpr ((OPT & kTpMul) != 0) *y = cmul(*y, m[(size_t)r << a.out_bit]);
                    }
                }
            }
        } else {
            if constexpr (ARITH == kTpFixed) {  // the stage's shift for any data, where its table does not bring it
                if ((OPT & kTpGlobalTw) != 0 && s.tw_kind) {
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = fx_scale_down(v[r], s.sh);
                } else if (s.tw_kind == 1) {
                    v[0] = fx_scale_down(v[0], s.sh);
                }
            }
            if (s.tw_kind) tp_twiddles<ARITH, DIR, OPT, R>(s, e0, v, tabs);
            if constexpr (ARITH == kTpFixed && FIRST) {
                if (fine) {
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = fx_scale_down(v[r], kFxFine);
                }
            }
            if constexpr (kShifts) {
                if (s.size_out) fx_raise(em + (s.size_out << a.lg_groups), fx_size<R>(v), s.warp);
            }
            TpSlots<std::remove_const_t<std::remove_reference_t<decltype(s)>>, R> at(s, slot);
#pragma unroll
            for (int r = 0; r < R; ++r) sm[at(r)] = v[r];
        }
        if constexpr (kOnce) break;
    }
    return true;
}

template <int ARITH, int DIR, int OPT, bool FIRST, bool LAST, typename P>
__device__ __forceinline__ bool tp_stage_any(const P &a, int si, typename tp_type<ARITH>::work *sm,
                                             const typename tp_type<ARITH>::tw *tabs, int *emax,
                                             const typename tp_type<ARITH>::elem *src,
                                             typename tp_type<ARITH>::elem *dst) {
    switch (a.st[si].lg_r) {
        case 1: return tp_stage<ARITH, DIR, OPT, 2, FIRST, LAST>(a, si, sm, tabs, emax, src, dst);
        case 2: return tp_stage<ARITH, DIR, OPT, 4, FIRST, LAST>(a, si, sm, tabs, emax, src, dst);
        case 3: return tp_stage<ARITH, DIR, OPT, 8, FIRST, LAST>(a, si, sm, tabs, emax, src, dst);
        case 4:
            if constexpr (ARITH == kTpF32 || ARITH == kTpF32w)
                return tp_stage<ARITH, DIR, OPT, 16, FIRST, LAST>(a, si, sm, tabs, emax, src, dst);
            break;
        default:
            if constexpr (ARITH == kTpF32w)
                return tp_stage<ARITH, DIR, OPT, 32, FIRST, LAST>(a, si, sm, tabs, emax, src, dst);
            break;
    }
    return true;
}

// Twiddle tables of the stages (F32 / Fixed).
template <int ARITH, typename P>
__device__ __forceinline__ void tp_tables(const P &a, typename tp_type<ARITH>::tw *tabs) {
    using TW = typename tp_type<ARITH>::tw;
    for (int si = 0; si < a.nst; ++si) {
        const auto &s = a.st[si];
        if (s.tw_kind == 0) continue;
        const TW *tw = static_cast<const TW *>(s.tw);
        const int n = 1 << (s.lg_r + s.lg_q);
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            TW w = tw[tp_exponent(s, (unsigned)i >> s.lg_q, (unsigned)i & ((1u << s.lg_q) - 1))];
            if constexpr (ARITH == kTpFixed) {
                w = fx_scale_tw(w, s.sh);
            }
            tabs[s.tab + i] = w;
        }
    }
}

template <int ARITH, int DIR, int OPT, typename P>
__device__ __forceinline__ bool tp_run(const P &a, typename tp_type<ARITH>::work *sm,
                                       const typename tp_type<ARITH>::tw *tabs, int *emax,
                                       const typename tp_type<ARITH>::elem *src, typename tp_type<ARITH>::elem *dst) {
    if constexpr ((OPT & kTpSingle) != 0) return tp_stage_any<ARITH, DIR, OPT, true, true>(a, 0, sm, tabs, emax, src, dst);
    if (!tp_stage_any<ARITH, DIR, OPT, true, false>(a, 0, sm, tabs, emax, src, dst)) return false;
    __syncthreads();
    for (int si = 1; si + 1 < a.nst; ++si) {
        tp_stage_any<ARITH, DIR, OPT, false, false>(a, si, sm, tabs, emax, src, dst);
        __syncthreads();
    }
    tp_stage_any<ARITH, DIR, OPT, false, true>(a, a.nst - 1, sm, tabs, emax, src, dst);
    return true;
}

template <int DIR, int OPT, typename P>
__device__ __noinline__ void tp_run_fp64(const P &a, double2 *sm, const double2 *src, double2 *dst) {
    tp_run<kTpF64, DIR, OPT>(a, sm, nullptr, nullptr, src, dst);
}

// complex128: entries of the exponent groups (tp_stage).
template <typename P> __host__ __device__ __forceinline__ int tp_entries(const P &a) {
    return (1 + a.shifts.sizes) << a.lg_groups;
}

// Element offset of tile t.
template <typename P> __device__ __forceinline__ int64_t tp_base(const P &a, int64_t t) {
    if (a.lg_inner < 0) return t << a.lg_tile;
    const int lg_c = a.lg_inner - a.lg_v;  // tiles along the inner positions
    return ((t >> lg_c) << (a.lg_g + a.lg_inner)) + ((t & (((int64_t)1 << lg_c) - 1)) << a.lg_v);
}

}  // namespace fftu
