// kc_gon.cuh -- device helpers shared by the persistent Gonzalez kernels
// (kc_gon.cu, kc_gonskip.cu): block sweeps, the exchange slots and the
// assignment of blocks to CTAs and warps.
#pragma once

#include <type_traits>

#include "kc_internal.cuh"

namespace kc {
namespace {

constexpr int GROUP_NT = 1024;   // group mode: one CTA per SM
constexpr int QUEUE_NT = 256;    // queue mode: several CTAs per SM
constexpr int JOIN_BUDGETS = 16; // wait for a group's CTAs to leave their earlier instances, in spin-wait budgets

template <typename T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<int32_t> { using type = int4; };

__device__ __forceinline__ uint64_t ld_relaxed_u64(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(uint64_t *p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// UNR: coordinates in flight in the generic loop (DC <= 0).  BATCH, its form: the
// loads written out ahead of the terms, with one more batch for the remainder
// (1) or a load at a time (2); groups of UNR, then by fours (0); a plain unrolled
// loop (3).  In the 1024-thread kernels the compiler mixed loads and terms of
// the plain loop differently from build to build (us a step: 800k x 256 on 98
// CTAs 147 or 160, written out 129; 1.5M x 24 30.5 or 32, 27.8; 4M x 40 111, 98;
// int32 2M x 64 87 to 100, 88), and the loop written out beats the full unrolling
// of d = 64 too (1.5M x 64 70.2 / 65.2, 8M x 64 309 / 297).  The remainder as a
// batch made the claimed-block instantiation a third slower (5M x 37 128 -> 173,
// one by one 116), and below twelve coordinates on up to 64 CTAs the plain loop
// is the better one (80k x 9 3.0 / 2.8).  In the 256-thread kernels the groups are
// (MRG on 2M x 64 18.2 ms, written out 22.2).
template <typename T, int DC, int UNR, int BATCH>
__device__ __forceinline__ void dist4(const T *__restrict__ blk, int d, const T *cs, int lane,
                                      typename AccOf<T>::type acc[4]) {
    using V4 = typename Vec4<T>::type;
    using A = typename AccOf<T>::type;
    const V4 *src = reinterpret_cast<const V4 *>(blk) + lane;
    A a0 = A(0), a1 = A(0), a2 = A(0), a3 = A(0);
    if constexpr (DC > 0) {
#pragma unroll
        for (int j = 0; j < DC; ++j) {
            const V4 v = __ldg(src + j * (BLK / 4));
            const T c = cs[j];
            a0 = sq_step(a0, v.x, c);
            a1 = sq_step(a1, v.y, c);
            a2 = sq_step(a2, v.z, c);
            a3 = sq_step(a3, v.w, c);
        }
    } else if constexpr (BATCH == 1 || BATCH == 2) {
        int j = 0;
#pragma unroll 1
        for (; j + UNR <= d; j += UNR) {
            V4 v[UNR];
#pragma unroll
            for (int t = 0; t < UNR; ++t) v[t] = __ldg(src + (j + t) * (BLK / 4));
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const T c = cs[j + t];
                a0 = sq_step(a0, v[t].x, c);
                a1 = sq_step(a1, v[t].y, c);
                a2 = sq_step(a2, v[t].z, c);
                a3 = sq_step(a3, v[t].w, c);
            }
        }
        if constexpr (BATCH == 2) {
#pragma unroll 1
            for (; j < d; ++j) {
                const V4 v = __ldg(src + j * (BLK / 4));
                const T c = cs[j];
                a0 = sq_step(a0, v.x, c);
                a1 = sq_step(a1, v.y, c);
                a2 = sq_step(a2, v.z, c);
                a3 = sq_step(a3, v.w, c);
            }
        } else if (j < d) {
            V4 v[UNR - 1];
#pragma unroll
            for (int t = 0; t < UNR - 1; ++t)
                if (j + t < d) v[t] = __ldg(src + (j + t) * (BLK / 4));
#pragma unroll
            for (int t = 0; t < UNR - 1; ++t)
                if (j + t < d) {
                    const T c = cs[j + t];
                    a0 = sq_step(a0, v[t].x, c);
                    a1 = sq_step(a1, v[t].y, c);
                    a2 = sq_step(a2, v[t].z, c);
                    a3 = sq_step(a3, v[t].w, c);
                }
        }
    } else if constexpr (BATCH == 3) {
#pragma unroll UNR
        for (int j = 0; j < d; ++j) {
            const V4 v = __ldg(src + j * (BLK / 4));
            const T c = cs[j];
            a0 = sq_step(a0, v.x, c);
            a1 = sq_step(a1, v.y, c);
            a2 = sq_step(a2, v.z, c);
            a3 = sq_step(a3, v.w, c);
        }
    } else {
        // whole groups of UNR coordinates, then by fours: a loop unrolled by eight
        // loads what is left one at a time (MRG on 10M x 4, m = 64: 5.4 ms, so 3.7,
        // by fours alone 4.1; 3M x 30 14.3, 13.3, 15.1)
        int j = 0;
#pragma unroll 1
        for (; j + UNR <= d; j += UNR) {
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const V4 v = __ldg(src + (j + t) * (BLK / 4));
                const T c = cs[j + t];
                a0 = sq_step(a0, v.x, c);
                a1 = sq_step(a1, v.y, c);
                a2 = sq_step(a2, v.z, c);
                a3 = sq_step(a3, v.w, c);
            }
        }
#pragma unroll 4
        for (; j < d; ++j) {
            const V4 v = __ldg(src + j * (BLK / 4));
            const T c = cs[j];
            a0 = sq_step(a0, v.x, c);
            a1 = sq_step(a1, v.y, c);
            a2 = sq_step(a2, v.z, c);
            a3 = sq_step(a3, v.w, c);
        }
    }
    acc[0] = a0;
    acc[1] = a1;
    acc[2] = a2;
    acc[3] = a3;
}

// The blocks of CTA r (of G, W warps each) over [b0, b1] are
// b(i) = b0 + r W + i % W + (i / W) G W for i = 0, 1, ... (increasing in i).
// Within a step the CTA's warps take i from a counter in shared memory (ctr;
// the next index is claimed while the current block is processed), so a warp
// whose loads came back sooner takes more blocks and the CTA's share is done
// when its blocks are, not when its slowest warp's fixed list is.  A block's
// minima stay with the CTA, which orders every step's accesses with its
// barriers.  ctr null: the fixed assignment i = warp + j W.
__device__ __forceinline__ int64_t cta_block(int64_t b0, int r, int G, int W, int i) {
    return b0 + (int64_t)r * W + (i % W) + (int64_t)(i / W) * G * W;
}
__device__ __forceinline__ int claim_block(int *ctr, int lane) {
    int v = 0;
    if (lane == 0) v = atomicAdd(ctr, 1);
    return __shfl_sync(0xFFFFFFFFu, v, 0);
}

// First block of the group's shared tail: with a tail counter, the CTAs own
// the blocks below it (7/8 of the range, whole rounds of G W blocks) and any
// warp of the group claims the rest, two blocks at a time, from a per-step
// counter in global memory, so the group's step ends when its blocks are done
// rather than when the CTA that got the least bandwidth is.  Blocks of the
// tail change CTA from step to step: their minima are read past L1 and every
// step's writes are fenced before the step's slot is published (gon_solve).
__device__ __forceinline__ int64_t tail_start(int64_t b0, int64_t b1, int G, int W, bool tail) {
    if (!tail) return b1 + 1;
    const int64_t GW = (int64_t)G * W;
    const int64_t rounds = (b1 - b0 + 1) * 7 / 8 / GW;
    return rounds >= 2 ? b0 + rounds * GW : b1 + 1;
}

// Warp 0: wait for slots [FIRST, G) of this step and return their maximum (with
// FIRST > 0 v0 takes part too).  The status word and the cycle budget are looked
// at every 32nd round only: a status load in each round made the round twice
// as long (1M x 10, resident: 4.2 -> 3.6 us a step with the 32-bit warp
// reductions of warp_max_u64).
template <int FIRST = 0>
__device__ __forceinline__ uint64_t poll_slots(const uint64_t *slots, int G, long long timeout, DevStatus *st, int step,
                                               bool *abort_out, uint64_t v0 = 0) {
    const int lane = threadIdx.x & 31;
    uint64_t g = FIRST ? v0 : 0;
    bool ab = false;
    for (int s0 = 0; s0 < G && !ab; s0 += 128) {
        uint64_t v[4];
        unsigned pend = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (s0 + q * 32 + lane < G && s0 + q * 32 + lane >= FIRST) pend |= 1u << q;
        const long long t0 = clock64();
        int n = 0;
        while (pend) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (pend >> q & 1u) v[q] = ld_relaxed_u64(slots + s0 + q * 32 + lane);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if ((pend >> q & 1u) && v[q] != 0) {
                    g = umax64(g, v[q]);
                    pend &= ~(1u << q);
                }
            if (pend && (++n & 31) == 0 && (clock64() - t0 > timeout || ld_volatile_i32(&st->code) != 0)) {
                set_status(st, KC_ERR_TIMEOUT, 3, step);
                ab = true;
                break;
            }
        }
    }
    *abort_out = __any_sync(0xFFFFFFFFu, ab);
    return warp_max_u64(g);
}

// Exchanges of large groups go through the group's first CTA (the leader): it
// alone polls the slots, and publishes the step's key and the new center's
// coordinates as 64-bit words that carry the step's tag, which the others
// poll; below LEADER_MIN CTAs every CTA polls the slots and loads the
// coordinates itself.
// The words (bc, zeroed before the launch, tags ascending) are reused every
// step: the leader writes them after every slot of the step is set, and a CTA
// sets its slot after it has read the words of the step before.
// 152 CTAs that poll one row of slots slow each other's publishing down (an
// exchange alone: 7000 cycles, 2800 through a leader; 16 CTAs: 1640 against
// 2600).  GON at k = 100 on 1M points, us a step, all polling against leader:
// d = 2 3.88 / 3.59, d = 3 4.14 / 3.66.
constexpr int LEADER_MIN = 40;

// Warp 0 of the others: words [0, W) of the leader; word w to put(w, bits).
template <typename Put>
__device__ __forceinline__ bool follow_leader(const uint64_t *bc, uint32_t tag, int W, long long timeout, DevStatus *st,
                                              int step, Put put) {
    bool ab = false;
    for (int w = threadIdx.x & 31; w < W; w += 32) {
        uint64_t x = ld_relaxed_u64(bc + w);
        const long long t0 = clock64();
        for (int n = 1; (uint32_t)(x >> 32) != tag; ++n) {
            x = ld_relaxed_u64(bc + w);
            if ((n & 31) == 0 && (clock64() - t0 > timeout || ld_volatile_i32(&st->code) != 0)) {
                set_status(st, KC_ERR_TIMEOUT, 3, step);
                ab = true;
                break;
            }
        }
        if (ab) break;
        put(w, (uint32_t)x);
    }
    return __any_sync(0xFFFFFFFFu, ab);
}

__device__ __forceinline__ int64_t out_index(const GonInst &I, int64_t local) {
    return I.map ? I.map[local] : I.base + local;
}

template <typename T>
__device__ bool instance_ok(const GonInst &I, DevStatus *st) {
    if constexpr (std::is_same<T, int32_t>::value) {
        if (!int_range_ok(I.range2, I.d)) {
            set_status(st, KC_ERR_RANGE, 2, 0);
            return false;
        }
    }
    return true;
}

// Last instance of insts[0, m) whose CTA group starts at or before this CTA.
__device__ __forceinline__ const GonInst *find_group(const GonInst *insts, int m) {
    int lo = 0, hi = m - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (insts[mid].cta0 <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    return insts + lo;
}

// The CTA's copy of its instance in shared memory, a word per thread (a
// thread that copies the whole struct holds it in registers and spills).
// Ends with a barrier.
__device__ __forceinline__ void copy_instance(GonInst &I, const GonInst *src) {
    static_assert(sizeof(GonInst) % 4 == 0 && sizeof(GonInst) / 4 <= 256, "one word per thread");
    constexpr int W = sizeof(GonInst) / 4;
    if (threadIdx.x < W) reinterpret_cast<uint32_t *>(&I)[threadIdx.x] = reinterpret_cast<const uint32_t *>(src)[threadIdx.x];
    __syncthreads();
    if (threadIdx.x == 0 && I.it1 == 0) I.it1 = I.k;
    __syncthreads();
}

}  // namespace
}  // namespace kc
