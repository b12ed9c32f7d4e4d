// Tile passes (tile_pass.cuh): kernel, launch, and the planner that splits a pass into stages.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <utility>

#include "fft_device.cuh"
#include "fftu_internal.h"
#include "tile_pass.cuh"

namespace fftu {
namespace {

// Grid: prepare_t.  The twiddle tables are built once per CTA.  64 registers (1024 threads per SM, in CTAs of 256 for the usual
// tiles), 128 with radix-32 stages.
template <int ARITH, int DIR, int OPT>
__global__ void __launch_bounds__(ARITH == kTpF32w ? 512 : 1024) tile_pass_kernel(const __grid_constant__ TilePass a) {
    using T = tp_type<ARITH>;
    using E = typename T::elem;
    extern __shared__ __align__(128) unsigned char tp_raw[];
    auto *sm = reinterpret_cast<typename T::work *>(tp_raw);
    auto *tabs = reinterpret_cast<typename T::tw *>(tp_raw + a.tab_off);
    int *emax = reinterpret_cast<int *>(tp_raw + a.emax_off);
    // The next kernel of the stream may start once every CTA of this one has; it waits below for all of this kernel's
    // writes, as this one does for its predecessor's (small arrays are bound by launch and table latency).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tp_tables<ARITH>(a, tabs);  // plan data, not written by earlier kernels
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // a.chunk tiles in a row, or (0) every gridDim.x-th tile
    const int64_t step = a.chunk ? 1 : gridDim.x, first = a.chunk ? blockIdx.x * (int64_t)a.chunk : blockIdx.x;
    const int64_t end = a.chunk && first + a.chunk < a.tiles ? first + a.chunk : a.tiles;
    for (int64_t t = first; t < end; t += step) {
        __syncthreads();  // tables ready; the previous tile's last stage done with its slots and exponents
        if constexpr (ARITH == kTpFixed) {
            for (int i = threadIdx.x; i < tp_entries(a); i += blockDim.x) emax[i] = 0;
            __syncthreads();
        }
        const int64_t base = tp_base(a, t);
        const E *src = static_cast<const E *>(a.src) + base;
        E *dst = static_cast<E *>(a.dst) + base;
        if (!tp_run<ARITH, DIR, OPT>(a, sm, tabs, emax, src, dst)) {
            if constexpr (ARITH == kTpFixed) tp_run_fp64<DIR, OPT>(a, reinterpret_cast<double2 *>(sm), src, dst);
        }
    }
}

int ilog2(int64_t v) {
    int r = 0;
    while ((int64_t(1) << r) < v) ++r;
    return r;
}

// Digits of an axis of 2^bits points, highest first: at most 2^top points each, the larger ones first.
int split_digits(int bits, int top, int *dig) {
    const int k = (bits + top - 1) / top;
    if (top == 3 && bits == 4) {  // complex128: a thread holds 8 values of the first stage
        dig[0] = 3;
        dig[1] = 1;
        return 2;
    }
    for (int i = 0; i < k; ++i) dig[i] = bits / k + (i < bits % k ? 1 : 0);
    return k;
}

// Rank over GF(2) of n vectors of m bits.
int gf2_rank(int *v, int n) {
    int rank = 0;
    for (int b = 1; b < 16; b <<= 1) {
        int p = -1;
        for (int i = rank; i < n; ++i)
            if (v[i] & b) {
                p = i;
                break;
            }
        if (p < 0) continue;
        const int t = v[p];
        v[p] = v[rank];
        v[rank] = t;
        for (int i = 0; i < n; ++i)
            if (i != rank && (v[i] & b)) v[i] ^= v[rank];
        ++rank;
    }
    return rank;
}

template <int ARITH, int DIR>
cudaError_t launch_t(const TilePass &a, cudaStream_t st) {
    // programmatic launch: the CTAs may start, and build their tables, while the kernel before this one finishes
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.grid);
    cfg.blockDim = dim3((unsigned)a.threads);
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if constexpr (ARITH == kTpFixed) {
        if (a.shifts.any)
            return a.mul ? cudaLaunchKernelEx(&cfg, tile_pass_kernel<ARITH, DIR, kTpMul | kTpShifts>, a)
                         : cudaLaunchKernelEx(&cfg, tile_pass_kernel<ARITH, DIR, kTpShifts>, a);
    }
    switch ((a.mul ? kTpMul : 0) | (a.nst == 1 ? kTpSingle : 0)) {
        case 0: return cudaLaunchKernelEx(&cfg, tile_pass_kernel<ARITH, DIR, 0>, a);
        case kTpMul: return cudaLaunchKernelEx(&cfg, tile_pass_kernel<ARITH, DIR, kTpMul>, a);
        case kTpSingle: return cudaLaunchKernelEx(&cfg, tile_pass_kernel<ARITH, DIR, kTpSingle>, a);
        default: return cudaLaunchKernelEx(&cfg, tile_pass_kernel<ARITH, DIR, kTpMul | kTpSingle>, a);
    }
}

template <int ARITH, int DIR, int OPT>
cudaError_t prepare_opt(const TilePass &a, int *per_sm) {
    cudaError_t e = cudaFuncSetAttribute(tile_pass_kernel<ARITH, DIR, OPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMaxDynSmem);
    if (e != cudaSuccess || !per_sm) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, tile_pass_kernel<ARITH, DIR, OPT>, a.threads, a.smem);
}

template <int ARITH, int DIR>
cudaError_t prepare_t(TilePass &a) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = a.nst == 1 ? prepare_opt<ARITH, DIR, kTpMul | kTpSingle>(a, nullptr)
                               : prepare_opt<ARITH, DIR, kTpMul>(a, nullptr);
    if (e == cudaSuccess)
        e = a.nst == 1 ? prepare_opt<ARITH, DIR, kTpSingle>(a, &per_sm) : prepare_opt<ARITH, DIR, 0>(a, &per_sm);
    if constexpr (ARITH == kTpFixed) {
        if (e == cudaSuccess && a.shifts.any) {
            e = prepare_opt<ARITH, DIR, kTpMul | kTpShifts>(a, nullptr);
            if (e == cudaSuccess) e = prepare_opt<ARITH, DIR, kTpShifts>(a, &per_sm);
        }
    }
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
    // The twiddle tables are built once per CTA.  Where they are a small part of a tile, a CTA per tile: the SMs take the
    // tiles in order as they come free, so that the last wave is short and neighbouring tiles stay close in time.
    // Persistent against a CTA per tile: complex128 64^4 599 and 534 us, 128^3 94 and 81, 256 x 16 x 16 x 256 696 and 631
    // (tables of up to a seventh of the tile), 2048^2 202 and 206; complex64 32^5 335 and 322 (a 64th), 256^3 134.5 and
    // 135.8 (a 16th), 1024 x 4096 37 and 41, 256 x 256 x 128 on 8^3 89 and 95.  With larger tables, a few tiles in a row per
    // CTA, for as many as keep that proportion, in complex128 and on long complex64 axes: 512 x 512 x 64 complex128
    // persistent 620 and 595, 64 x 1024 x 1024 complex64 638 and 597; not on shorter complex64 axes (512 x 64 x 512 146 and
    // 151), for fewer than four waves of them (32 x 1024 x 1024 286 and 293) or one of complex128 (2048^2 202 and 201).
    const size_t tables = a.emax_off - a.tab_off, tile = (size_t)(ARITH == kTpFixed ? 16 : 8) << a.lg_tile;
    const int64_t resident = a.resident = sms * per_sm;
    const int64_t c = std::max<int64_t>(1, (tables * (ARITH == kTpFixed ? 7 : 32) + tile - 1) / tile);
    const bool rows = ARITH == kTpFixed || (ARITH == kTpF32w && a.lg_g >= 10);
    a.chunk = c == 1 || (rows && (ARITH == kTpFixed ? 1 : 4) * c * resident <= a.tiles) ? (int)c : 0;
    a.grid = a.chunk ? (int)((a.tiles + c - 1) / c) : (int)std::min(a.tiles, resident);
    return e;
}

}  // namespace

bool make_tile_pass(int d, const int64_t *n, const int64_t *p, int l0, int l1, int is_double, int wide, int lg_v,
                    const void *const *tw, const void *const *tw64, TilePass &a) {
    std::memset(&a, 0, sizeof(a));
    int64_t outer = 1, inner = 1, G = 1;
    for (int l = 0; l < l0; ++l) outer *= n[l];
    for (int l = l0; l <= l1; ++l) G *= n[l];
    for (int l = l1 + 1; l < d; ++l) inner *= n[l];
    if (outer * G * inner > ((int64_t)1 << 31)) return false;  // 32-bit element offsets within a tile
    const bool contiguous = inner == 1;
    a.lg_g = ilog2(G);
    a.lg_v = lg_v;
    a.lg_inner = contiguous ? -1 : ilog2(inner);
    a.lg_tile = a.lg_g + lg_v;
    if (a.lg_tile > 14) return false;
    a.tiles = (contiguous ? outer : outer * inner) >> lg_v;
    const int top = is_double ? 3 : wide ? 5 : 4;
    a.wide = wide;
    // stage order: the slowest axis' first digit, the other axes' digits, the slowest axis' remaining digits: the
    // first and last stage then run across rows, with lanes along memory.  A contiguous group whose slowest axis
    // has one digit gets it split, so that the last stage is not the contiguous axis' only digit.
    struct Dig {
        int axis, bits, pos;
    } dg[kTpStages];
    int order[kTpStages], nd = 0, no = 0;
    int lo_of[FFTU_MAX_DIMS], lg_p[FFTU_MAX_DIMS], first_of[FFTU_MAX_DIMS], count_of[FFTU_MAX_DIMS];
    int lo = contiguous ? 0 : lg_v;
    for (int l = l1; l >= l0; --l) {
        lg_p[l] = p ? ilog2(p[l]) : 0;
        const int bits = ilog2(n[l]) - lg_p[l];
        int dig[8];
        int k = split_digits(bits, top, dig);
        if (l == l0 && l1 > l0 && contiguous && k == 1 && bits >= 2) {
            dig[1] = bits / 2;
            dig[0] = bits - dig[1];
            k = 2;
        }
        // one digit in phase A: the Put moves s, so loads and stores need a barrier between them.  A strided axis takes
        // one fiber per thread and a barrier in its only stage; contiguous lines two stages (lanes along memory).
        if (p && l0 == l1 && k == 1 && lg_p[l] > 0 && contiguous) {
            if (bits < 2) return false;
            dig[1] = bits / 2;
            dig[0] = bits - dig[1];
            k = 2;
        }
        lo_of[l] = lo;
        first_of[l] = nd;
        count_of[l] = k;
        a.lg_dft += bits;
        int q = lo + lg_p[l] + bits;
        for (int i = 0; i < k; ++i) {
            if (nd >= kTpStages) return false;
            q -= dig[i];
            dg[nd++] = {l, dig[i], q};
        }
        lo += lg_p[l] + bits;
    }
    if (count_of[l0] > 0) order[no++] = first_of[l0];
    for (int l = l1; l > l0; --l)
        for (int i = 0; i < count_of[l]; ++i) order[no++] = first_of[l] + i;
    for (int i = 1; i < count_of[l0]; ++i) order[no++] = first_of[l0] + i;
    if (no == 0) return false;
    if (no == 1 && p && l1 > l0) return false;  // (axes of length 2 beside it: left to the strided pass)
    a.once = no == 1 && p && lg_p[l0] > 0;
    a.nst = no;
    // output position of every tile bit (element-offset bits, relative to the tile's base): an axis' first (highest)
    // digit holds the lowest bits of k; the class s goes above k
    int out_bit[32], k_bit[kTpStages];
    for (int b = 0; b < a.lg_tile; ++b) out_bit[b] = b;
    for (int l = l1; l >= l0; --l) {
        int k_at = 0;
        for (int i = 0; i < count_of[l]; ++i) {
            const Dig &g = dg[first_of[l] + i];
            k_bit[first_of[l] + i] = k_at;
            for (int b = 0; b < g.bits; ++b) out_bit[g.pos + b] = lo_of[l] + k_at + b;
            k_at += g.bits;
        }
        for (int b = 0; b < lg_p[l]; ++b) out_bit[lo_of[l] + b] = lo_of[l] + k_at + b;
    }
    if (!contiguous)
        for (int b = 0; b < a.lg_tile; ++b)
            if (out_bit[b] >= lg_v) out_bit[b] += a.lg_inner - lg_v;
    const Dig &df = dg[order[0]], &dl = dg[order[no - 1]];
    a.in_bit = contiguous ? df.pos : df.pos - lg_v + a.lg_inner;
    a.out_bit = out_bit[dl.pos];
    // the last stage's lanes follow the output: its tile bits in order of their output position
    int tb[32], nt = 0;
    for (int b = 0; b < a.lg_tile; ++b)
        if (b < dl.pos || b >= dl.pos + dl.bits) tb[nt++] = b;
    for (int i = 1; i < nt && no > 1; ++i)  // (a single stage keeps the order of its loads)
        for (int k = i; k > 0 && out_bit[tb[k - 1]] > out_bit[tb[k]]; --k) std::swap(tb[k - 1], tb[k]);
    for (int i = 0; i < nt;) {
        int j = i + 1;
        while (j < nt && tb[j] == tb[j - 1] + 1) ++j;
        if (a.nlast >= kTpFields) return false;
        a.last[a.nlast++] = {i, (1 << (j - i)) - 1, tb[i]};
        i = j;
    }
    for (int i = 0; i < nt;) {
        int j = i + 1;
        while (j < nt && out_bit[tb[j]] == out_bit[tb[j - 1]] + 1) ++j;
        if (a.nout >= kTpFields) return false;
        a.out[a.nout++] = {i, (1 << (j - i)) - 1, out_bit[tb[i]]};
        i = j;
    }
    // exponent groups: the tile bits no digit covers
    for (int b = 0; b < a.lg_tile;) {
        bool digit = false;
        for (int i = 0; i < nd; ++i)
            if (b >= dg[i].pos && b < dg[i].pos + dg[i].bits) digit = true;
        if (digit) {
            ++b;
            continue;
        }
        BitField *f = a.ngroup ? &a.group[a.ngroup - 1] : nullptr;
        if (f && f->sh + ilog2(f->mask + 1) == b) {
            f->mask = f->mask * 2 + 1;
        } else {
            if (a.ngroup >= kTpFields) return false;
            a.group[a.ngroup++] = {b, 1, a.lg_groups};
        }
        ++a.lg_groups;
        ++b;
    }
    // swizzle: the shifts that leave the lanes of one wavefront (16 of 8 bytes, 8 of 16) in distinct slots
    const int lw = is_double ? 3 : 4, m = (1 << lw) - 1;
    int best = 1 << 30;
    const int least = no > 2 ? 2 * no - 2 : no;  // every stage without conflicts
    for (int s1 = 1; s1 <= 13 && best > least; ++s1)
        for (int s2 = s1; s2 <= 13 && best > least; ++s2) {
            auto slot = [&](int e) { return (e ^ (e >> s1) ^ (s2 == s1 ? 0 : e >> s2)) & m; };
            int cost = 0;
            for (int si = 0; si < no; ++si) {
                const Dig &g = dg[order[si]];
                int v[4], k = 0;
                if (si == no - 1) {
                    for (int i = 0; i < lw && i < nt; ++i) v[k++] = slot(1 << tb[i]);
                } else {
                    for (int b = 0; b < a.lg_tile && k < lw; ++b)
                        if (b < g.pos || b >= g.pos + g.bits) v[k++] = slot(1 << b);
                }
                cost += (1 << (k - gf2_rank(v, k))) * (si == 0 || si == no - 1 ? 1 : 2);
            }
            if (cost < best) {
                best = cost;
                a.swz[0] = s1;
                a.swz[1] = s2 == s1 ? 30 : s2;
            }
        }
    auto slot = [&](int e) { return e ^ ((e >> a.swz[0]) & m) ^ ((e >> a.swz[1]) & m); };
    int tab = 0;
    for (int si = 0; si < no; ++si) {
        const int id = order[si];
        const Dig &g = dg[id];
        const int l = g.axis, first = first_of[l], at = id - first;
        TileStage &s = a.st[si];
        s.lg_r = g.bits;
        s.pos = g.pos;
        s.tw = tw[l];
        s.tw64 = tw64[l];
        for (int b = 0; b < g.bits; ++b) s.rb[b] = slot(1 << (g.pos + b));
        for (int r = 0; r < 1 << g.bits; ++r) s.rx[r] = slot(r << g.pos);
        const int lo_m = lo_of[l] + lg_p[l];  // lowest bit of m
        if (at + 1 < count_of[l]) {  // w_{R T}^{r j} = w_n^{r j n / (R T)}
            s.tw_kind = 1;
            s.lo = lo_m;
            s.lg_q = g.pos - lo_m;
            s.lg_step = ilog2(n[l]) - g.bits - s.lg_q;
        } else if (lg_p[l] > 0) {  // w_n^{k s}, k = k_prev + r 2^k_bit
            s.tw_kind = 2;
            s.lo = lo_of[l];
            s.lg_p = lg_p[l];
            s.lg_q = ilog2(n[l]) - g.bits;
            s.lg_step = k_bit[id];
            for (int i = 0; i < at; ++i) {
                if (s.nk >= 2) return false;
                const Dig &h = dg[first + i];
                s.k[s.nk++] = {h.pos - (g.pos + g.bits), (1 << h.bits) - 1, k_bit[first + i]};
            }
        }
        s.tab = tab;
        if (s.tw_kind) tab += 1 << (g.bits + s.lg_q);
    }
    if (is_double) {
        // The shift before each later stage (fixed64.cuh): what any data need, from 2^61.5 after the first stage, to stay within
        // the stages' limits; the largest ones by the groups' sizes, until the others take kFxFixed bits at most.  A product
        // halves in any case.
        int need[kTpStages], least[kTpStages], total = 0;
        bool sized[kTpStages] = {};
        for (;;) {
            int bound = 61, most = 0;  // and a half
            total = no > 1 && a.st[no - 1].tw_kind ? 1 : 0;
            for (int si = 1; si < no; ++si) {
                const int limit = a.st[si].tw_kind ? 61 : 62, grown = bound + a.st[si].lg_r;
                least[si] = a.st[si - 1].tw_kind ? 1 : 0;
                need[si] = sized[si] ? least[si] : std::max(least[si], grown - limit);
                bound = std::min(grown - need[si], limit);
                total += need[si];
                if (need[si] > least[si] && (!most || need[si] - least[si] > need[most] - least[most])) most = si;
            }
            if (total <= kFxFixed || !most) break;
            sized[most] = true;
        }
        if (no > 1 && a.st[no - 1].tw_kind) a.st[no - 1].sh = 1;
        for (int si = 1; si < no; ++si)
            if (sized[si]) {
                a.st[si].size_in = a.st[si - 1].size_out = (int8_t)++a.shifts.sizes;
                a.shifts.lg[a.shifts.sizes] = a.st[si].lg_r;
                a.shifts.room[a.shifts.sizes] = a.st[si].tw_kind ? kFxRoomHalved : kFxRoomNone;
            }
        for (int si = 1; si < no; ++si) {
            if (a.st[si - 1].tw_kind) a.st[si - 1].sh = need[si];
            else a.st[si].pre = (int8_t)need[si];
            if (a.st[si].pre || a.st[si].size_in) a.shifts.any = 1;
        }
        a.shifts.fixed = total;
        for (int si = 0; si < no; ++si) {
            const TileStage &s = a.st[si];
            bool one = a.lg_tile - s.lg_r >= 5;
            for (int b = 0; b < 5; ++b) {
                const int e = b < s.pos ? b : b + s.lg_r;
                for (int i = 0; i < a.ngroup; ++i)
                    if (e >= a.group[i].sh && e < a.group[i].sh + ilog2(a.group[i].mask + 1)) one = false;
            }
            a.st[si].warp = one;
        }
    }
    const size_t es = is_double ? 16 : 8;
    a.tab_off = no > 1 ? es << a.lg_tile : 0;
    a.emax_off = a.tab_off + tab * es;
    a.smem = a.emax_off + (is_double ? sizeof(int) * tp_entries(a) : 0);
    // complex128: one fiber of the first stage per thread (its exponent covers all of them); complex64: 16 values
    a.threads = is_double ? 1 << (a.lg_tile - a.st[0].lg_r) : a.lg_tile > 9 + wide ? 1 << (a.lg_tile - 4 - wide) : 32;
    if (a.once) a.threads = 1 << (a.lg_tile - a.st[0].lg_r);
    if (a.threads > (wide ? 512 : 1024) || a.smem > (size_t)kMaxDynSmem) return false;
    a.scale = 1.0;
    return true;
}

cudaError_t prepare_tile_pass(TilePass &a, int is_double, int dir) {
    if (is_double) return dir < 0 ? prepare_t<kTpFixed, -1>(a) : prepare_t<kTpFixed, 1>(a);
    if (a.wide) return dir < 0 ? prepare_t<kTpF32w, -1>(a) : prepare_t<kTpF32w, 1>(a);
    return dir < 0 ? prepare_t<kTpF32, -1>(a) : prepare_t<kTpF32, 1>(a);
}

cudaError_t launch_tile_pass(const TilePass &a, int is_double, int dir, cudaStream_t st) {
    if (is_double) return dir < 0 ? launch_t<kTpFixed, -1>(a, st) : launch_t<kTpFixed, 1>(a, st);
    if (a.wide) return dir < 0 ? launch_t<kTpF32w, -1>(a, st) : launch_t<kTpF32w, 1>(a, st);
    return dir < 0 ? launch_t<kTpF32, -1>(a, st) : launch_t<kTpF32, 1>(a, st);
}

}  // namespace fftu
