// kc_nearest.cuh -- the nearest of a set of centers for every point of a packed
// array (the skip kernel's assignment, EIM's cells).
#pragma once

#include "kc_internal.cuh"

namespace kc {
namespace {

constexpr int NEAREST_NT = 256, NEAREST_C = 16;
constexpr int NEAREST_DCH = 256;   // coordinates staged at a time

// Canonical minimum over centers [0, count) of every point (bits into mind) and
// the center that gives it (asg, lowest on ties); at(c, j) is coordinate j of
// center c.  A warp takes a block, its lanes four points each; centers go
// sixteen at a time (64 running sums, kept in registers over the chunks of
// coordinates), staged in cs ([up to NEAREST_DCH][NEAREST_C]: 16 KB, so that no
// d needs an opt-in to more shared memory).
template <int DC, typename At>
__device__ __forceinline__ void nearest_centers(const float *__restrict__ pk, int64_t n, int d_, int count, float *cs,
                                                At at, uint32_t *__restrict__ mind, uint16_t *__restrict__ asg) {
    static_assert(DC <= NEAREST_DCH, "specialisations stage all coordinates at once");
    const int d = DC > 0 ? DC : d_;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nb = nblocks(n);
    for (int64_t g = blockIdx.x; g * (NEAREST_NT / 32) < nb; g += gridDim.x) {
        const int64_t b = g * (NEAREST_NT / 32) + warp;
        uint32_t m[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
        uint32_t a[4] = {0u, 0u, 0u, 0u};
        for (int c0 = 0; c0 < count; c0 += NEAREST_C) {
            float acc[NEAREST_C][4];
            for (int j0 = 0; j0 < d; j0 += NEAREST_DCH) {
                const int jn = DC > 0 ? DC : (d - j0 < NEAREST_DCH ? d - j0 : NEAREST_DCH);
                __syncthreads();
                for (int e = threadIdx.x; e < NEAREST_C * jn; e += NEAREST_NT) {
                    const int c = c0 + e % NEAREST_C, j = j0 + e / NEAREST_C;
                    cs[e] = c < count ? at(c, j) : 0.f;
                }
                __syncthreads();
                if (b >= nb) continue;
                if (j0 == 0) {
#pragma unroll
                    for (int c = 0; c < NEAREST_C; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.f;
                }
                const float4 *src = reinterpret_cast<const float4 *>(pk + (b * d + j0) * BLK) + lane;
#pragma unroll 4
                for (int j = 0; j < jn; ++j) {
                    const float4 v = __ldg(src + j * (BLK / 4));
#pragma unroll
                    for (int c = 0; c < NEAREST_C; ++c) {
                        const float cc = cs[j * NEAREST_C + c];
                        acc[c][0] = sq_step(acc[c][0], v.x, cc);
                        acc[c][1] = sq_step(acc[c][1], v.y, cc);
                        acc[c][2] = sq_step(acc[c][2], v.z, cc);
                        acc[c][3] = sq_step(acc[c][3], v.w, cc);
                    }
                }
            }
            if (b >= nb) continue;
#pragma unroll
            for (int c = 0; c < NEAREST_C; ++c)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t s = __float_as_uint(acc[c][q]);
                    if (c0 + c < count && s < m[q]) {
                        m[q] = s;
                        a[q] = (uint32_t)(c0 + c);
                    }
                }
        }
        if (b < nb) {   // rows past n are written too (padding, never read as points)
            reinterpret_cast<uint4 *>(mind + b * BLK)[lane] = make_uint4(m[0], m[1], m[2], m[3]);
            reinterpret_cast<uint2 *>(asg + b * BLK)[lane] = make_uint2(a[0] | (a[1] << 16), a[2] | (a[3] << 16));
        }
    }
}

// Dynamic shared memory and grid of a kernel around it.
inline size_t nearest_smem(int d) { return (size_t)NEAREST_C * (d < NEAREST_DCH ? d : NEAREST_DCH) * sizeof(float); }
inline int nearest_grid(int64_t n, int sms) {
    const int64_t groups = (nblocks(n) + NEAREST_NT / 32 - 1) / (NEAREST_NT / 32);
    return (int)(groups < (int64_t)sms * 8 ? groups : (int64_t)sms * 8);
}

}  // namespace
}  // namespace kc
