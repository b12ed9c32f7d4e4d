// Register-resident form of the generic fused phase B: the tile's axes are grouped from the last
// one down into groups of at most 16 values (two adjacent axes where p_l p_{l-1} <= 16); each group is one
// stage in which a thread holds one fiber (all values of the group's axes for fixed other tile indices):
// the first stage loads its fibers from HBM, the last one stores them, the others go through shared memory.
// complex128 fibers are transformed in fixed point (fixed64.cuh), each with its own exponent.
#pragma once

#include "fft_device.cuh"
#include "fftu_internal.h"
#include "generic_tiles.cuh"

namespace fftu {

struct PBGroups {
    int n;
    int off[FFTU_MAX_DIMS], lo[FFTU_MAX_DIMS], hi[FFTU_MAX_DIMS];
    int64_t lst_lo[FFTU_MAX_DIMS], lst_hi[FFTU_MAX_DIMS];
};

// lg_scale: the result is multiplied by 2^lg_scale in the last stage (1/N is a power of two), then by mul[] at
// the same index (MUL).
template <typename C, int DIR, bool MUL, int LO, int HI>
__device__ __forceinline__ void pb_stage(const PhaseBFused &b, const PBGroups &g, int gi, int64_t base, C *sm,
                                         C *__restrict__ data, bool first, bool last, int lg_scale) {
    constexpr int PG = LO * HI;
    constexpr int LG = lg_of<PG>();
    const int off = g.off[gi];
    const int fibers = (b.P * b.Mt) >> LG;
    const int64_t slo = g.lst_lo[gi], shi = g.lst_hi[gi];
    for (int phi = threadIdx.x; phi < fibers; phi += blockDim.x) {
        const int e0 = ((phi >> off) << (off + LG)) | (phi & ((1 << off) - 1));
        C v[PG];
        int64_t go = 0;
        if (first || last) go = base + phaseb_offset(b, e0);
        if (first) {
#pragma unroll
            for (int j = 0; j < PG; ++j) v[j] = data[go + (j % LO) * slo + (j / LO) * shi];
        } else {
#pragma unroll
            for (int j = 0; j < PG; ++j) v[j] = sm[e0 + (j << off)];
        }
        fiber_dft<DIR, LO, HI>(v, last ? lg_scale : 0);
        if (last) {
#pragma unroll
            for (int j = 0; j < PG; ++j) {
                C x = v[j];
                if (sizeof(C) == 8 && lg_scale != 0) x = cscale(x, (typename real_of<C>::type)b.scale);
                if constexpr (MUL) x = cmul(x, static_cast<const C *>(b.mul)[go + (j % LO) * slo + (j / LO) * shi]);
                data[go + (j % LO) * slo + (j / LO) * shi] = x;
            }
        } else {
#pragma unroll
            for (int j = 0; j < PG; ++j) sm[e0 + (j << off)] = v[j];
        }
    }
}

}  // namespace fftu
