// kc_gonskip.cu -- Gonzalez steps that leave out the distances a triangle
// inequality proves irrelevant (single large float instances).
//
// GON (Section 3.1) evaluates every point against every new center c.  Let a
// be an earlier center, rho a bound on the distances of a group of points to
// a, and M the largest of their running minima.  If d(a, c) >= rho + sqrt(M),
// then d(x, c) >= d(a, c) - d(x, a) >= sqrt(M) for every point x of the group:
// no minimum can fall and the group need not be read (the test of Elkan,
// "Using the triangle inequality to accelerate k-means", ICML 2003, for groups
// of points and the farthest-first order).  On clustered points, once every
// cluster holds a center, a step touches the points of one cluster only.
//
// The streaming kernels (kc_gon.cu) stay the better ones while nearly every
// group is touched, and on points without structure for good.  So a solve
// starts on those, in segments of 16, 16, 32, ... steps:
//   probe    after each segment, on a sample of the points: would the rest of
//            the steps be faster here?  If so a device word gets the step
//            number, and the remaining streaming segments return at once;
//   assign   every point's minimum over the centers so far and the center
//            that gives it;
//   skip     the remaining steps, one persistent cooperative launch.
// 8M x 64, 100 Gaussian clusters, k = 1024 (GB300): 314 -> 41.3 ms per solve
// (32 streaming steps 9.8 ms, probes 0.04, assignment 1.2, 992 skip steps and
// their regroupings 29; 11.9 us a step once the clusters are covered, the
// 20 MB of one cluster's points per step being 2.9 us of it at the HBM rate);
// with the bf16 sweep before the change-over 181 -> 34.4 ms.
#include <algorithm>
#include <cstdlib>

#include "kc_gon.cuh"
#include "kc_nearest.cuh"

namespace kc {

namespace {

constexpr int SKIP_NT = 512;            // 128 registers a thread: a unit's 64 loads in flight per warp
constexpr int SKIP_W = SKIP_NT / 32;    // warps of a CTA
constexpr int UNIT = 32;                // points of a unit (one per lane)
constexpr int SKIP_BINS = 2048;         // most bins of a regrouping (two per center)
constexpr int SKIP_TILE = UNIT * 33;    // words of a warp's transpose tile

// ------------------------------------------------------------------ probe
// Would the skip kernel pay from here on?  One sampled point per warp, its
// lanes over the first it0 centers: its nearest center a and distance m.  The
// last CTA then bins the sample as the regrouping would (by a, near or far)
// and counts the points in bins that the newest center c (the winner of step
// it0 - 1) touches: d(a, c) < 2 sqrt(largest m of the bin).  With that share
// of the points touched a step takes fixed_us + share unit_us, the change-over
// (assignment, two regroupings) `once`.  What becomes of the share:
//  - where a fifth of the points or more are near (m at most a quarter of the
//    largest), the centers so far cover that part of the clusters, a new one
//    touches the other points only, and covering them takes about it0 (1 / near
//    - 1) more steps, over which the share falls to the few points of a cluster
//    (where nearly all are, outliers are being taken, and the others are still
//    to show what they are: a tenth);
//  - elsewhere (no clusters, or each has its center) it stays about what it is.
// *route is set to it0 when the steps left would take a tenth less time that
// way and the next ones no longer than a sweep (at the last probe they may, if
// all together take a seventh less); there is no way back.  Taking the share to
// fall on any points (its square) cost 10M x 8 uniform, k = 500, 61 ms against
// 30, and one cluster of 10M x 10, k = 1024, 153 against 72.
constexpr int PROBE_NT = 256, PROBE_CTAS = 128, PROBE_S = PROBE_CTAS * PROBE_NT / 32;
constexpr int PROBE_MAX = 256;         // most centers at a probe

__device__ __forceinline__ float row_dist_any(const float *__restrict__ x, const float *__restrict__ c, int d) {
    float acc = 0.f;
    int j = 0;
#pragma unroll 1
    for (; j + 16 <= d; j += 16) {
        float u[16], v[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            u[t] = __ldg(x + j + t);
            v[t] = __ldg(c + j + t);
        }
#pragma unroll
        for (int t = 0; t < 16; ++t) acc = sq_step(acc, u[t], v[t]);
    }
#pragma unroll 4
    for (; j < d; ++j) acc = sq_step(acc, __ldg(x + j), __ldg(c + j));
    return acc;
}

__global__ void __launch_bounds__(PROBE_NT) gon_probe_kernel(const float *__restrict__ rm,
                                                             const int64_t *__restrict__ rmap, int64_t n, int d,
                                                             const int64_t *__restrict__ centers, const uint64_t *key,
                                                             int it0, float sweep_us, float unit_us, float fixed_us,
                                                             float once_us, int left, bool last_probe, int *route,
                                                             unsigned *done, uint2 *sample, const DevStatus *st) {
    if (ld_volatile_i32(&st->code) != 0 || ld_volatile_i32(route) != 0) return;
    const uint64_t K = *key;
    if (key_val(K) == 0) return;   // the solve has stopped early
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * (PROBE_NT / 32) + (threadIdx.x >> 5);
    const int64_t x = (int64_t)w * (n / PROBE_S > 0 ? n / PROBE_S : 1);
    // with an rmap, rm holds the rows of the global indices, as centers does
    if (x < n) {   // uniform over the warp
        const float *px = rm + (rmap ? rmap[x] : x) * d;
        uint64_t best = ~0ull;   // (distance bits, center), smallest
        for (int i = lane; i < it0; i += 32) {
            const uint64_t k = ((uint64_t)__float_as_uint(row_dist_any(px, rm + centers[i] * d, d)) << 32) | (uint32_t)i;
            best = k < best ? k : best;
        }
        best = ~warp_max_u64(~best);
        if (lane == 0) __stcg(sample + w, make_uint2((uint32_t)(best >> 32), (uint32_t)best));
    } else if (lane == 0) {
        __stcg(sample + w, make_uint2(0u, 0xFFFFFFFFu));
    }
    __shared__ int last;
    __shared__ unsigned rmax[2 * PROBE_MAX];   // largest m of each bin (float bits)
    __shared__ float dc[PROBE_MAX];            // d(a, c)
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int64_t cw = key_idx(K);
    const float *cn = rm + (rmap ? rmap[cw] : cw) * d;
    const uint32_t far = __float_as_uint(0.25f * __uint_as_float(key_val(K)));
    for (int i = threadIdx.x; i < it0; i += PROBE_NT) {
        dc[i] = sqrtf(row_dist_any(rm + centers[i] * d, cn, d));
        rmax[2 * i] = rmax[2 * i + 1] = 0u;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < PROBE_S; q += PROBE_NT) {
        const uint2 s = __ldcg(sample + q);
        if (s.y < (uint32_t)it0) atomicMax(&rmax[2 * s.y + (s.x > far)], s.x);
    }
    __syncthreads();
    int touched = 0, total = 0, near = 0;
    for (int q = threadIdx.x; q < PROBE_S; q += PROBE_NT) {
        const uint2 s = __ldcg(sample + q);
        if (s.y >= (uint32_t)it0) continue;
        ++total;
        near += s.x <= far;
        touched += dc[s.y] < 2.f * sqrtf(__uint_as_float(rmax[2 * s.y + (s.x > far)]));
    }
    __shared__ int sum[3];
    if (threadIdx.x < 3) sum[threadIdx.x] = 0;
    __syncthreads();
    atomicAdd(&sum[0], touched);
    atomicAdd(&sum[1], total);
    atomicAdd(&sum[2], near);
    __syncthreads();
    if (threadIdx.x == 0) {
        *done = 0u;   // ready for the next probe
        const float share = (float)sum[0] / (float)max(sum[1], 1), nearf = (float)sum[2] / (float)max(sum[1], 1);
        float later = share;   // mean over the steps left
        if (nearf >= 0.2f) {
            const float cover = (float)it0 * (1.f / nearf - 1.f), l = (float)left;
            later *= fmaxf(l < cover ? 1.f - 0.5f * l / cover : 0.5f * cover / l, 0.1f);
            if (nearf > 0.9f) later = fmaxf(later, 0.1f);
        }
        const float save = (float)left * (sweep_us - later * unit_us - fixed_us) - once_us;
        const bool soon = share * unit_us + fixed_us <= 1.1f * sweep_us;   // from the next step on
        if ((soon || last_probe) && save > (soon ? 0.1f : 0.15f) * (float)left * sweep_us) *route = it0;
    }
}

// ----------------------------------------------------------------- assign
// Minimum over the first *route centers of every point of the packed array
// (into mind) and the position of the center that gives it (asg).
template <int DC>
__global__ void __launch_bounds__(NEAREST_NT, 2) gon_assign_kernel(GonInst I, uint16_t *asg, const int *route,
                                                                   const DevStatus *st) {
    extern __shared__ __align__(16) float as_cen[];
    const int it0 = ld_volatile_i32(route);
    if (it0 == 0 || ld_volatile_i32(&st->code) != 0) return;
    nearest_centers<DC>((const float *)I.pk, I.n, I.d, it0, as_cen,
                        [&](int c, int j) { return I.cenT[(int64_t)j * I.kcap + c]; }, I.mind, asg);
}

// The first *route centers' coordinates, transposed ([d][kcap]).
__global__ void gon_center_rows_kernel(GonInst I, const int *route, const DevStatus *st) {
    const int it0 = ld_volatile_i32(route);
    if (it0 == 0 || ld_volatile_i32(&st->code) != 0) return;
    const int64_t total = (int64_t)it0 * I.d;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / I.d), j = (int)(e - (int64_t)i * I.d);
        I.cenT[(int64_t)j * I.kcap + i] = I.rm[I.centers[i] * I.d + j];
    }
}

// ------------------------------------------------------------------- skip
//
// The points are first regrouped: a counting sort by (nearest center, near or
// far from it) puts points of one Voronoi cell into units of 32 (a unit never
// spans two cells: every bin starts at a multiple of 32, the gaps hold no
// point), and the coordinates are packed again in that order.  Unit u keeps,
// in the shared memory of the CTA that owns its block, its center a_u, rho_u
// >= the distance of any of its points to a_u, and the largest key of its
// running minima.  A new center c can lower a minimum of the unit only if
//   d(c, a_u) < rho_u + sqrt(largest minimum of the unit),
// so a step evaluates d(c, a) for the centers of the regrouping, tests every
// unit (a few instructions each) and streams the coordinates of the units
// that remain; all others cost nothing but their cached key.
// Bounds: D the exact distance, s(x, c) >= (1 - g) D(x, c)^2, so s(x, c) >= m
// follows from D(x, c) >= sqrt(m) (1 + 2 g); D(x, a_u) <= sqrt(s(x, a_u)) (1 +
// 2 g) = its contribution to rho_u; D(c, a_u) >= h = sqrt(t) (1 - 2 g - 2^-18)
// with t the float value of |c - a_u|^2 (summed in any order); every step is
// rounded to the safe side, and the 2^-18 covers products that underflow (t
// below 2^-100 gives h = 0).
//
// The regrouping is done at the first step and again when the step count has
// doubled and the units touched since make it worthwhile; its phases are
// separated by the group's own barrier (slot rows behind the k exchange rows).
constexpr int SKIP_ROUNDS = 6;   // regrouping decisions

// Positions of the regrouped arrays, at most: a unit per bin is begun for nothing.
__host__ __device__ inline int64_t skip_extent(int64_t n) { return nblocks(n + (int64_t)(UNIT - 1) * SKIP_BINS) * BLK; }

struct ShSkip {
    uint64_t red[32];
    uint64_t key;
    int abort;
    int ntouch;
    unsigned long long touched;   // units evaluated since the last regrouping
    int scan[32];
};

__device__ __forceinline__ float bound_up(float m, float g2) {   // sqrt(m) (1 + 2 g), rounded up
    return __fmul_ru(__fsqrt_ru(m), __fadd_ru(1.f, g2));
}

// Warp 0 of every CTA: publish v in the slot row and wait for all G (a few
// times a solve, so every CTA polls); the sum or the largest of the slots.
// The caller has barriers on both sides.
template <bool SUM>
__device__ uint64_t skip_round(uint64_t *row, int r, int G, uint64_t v, const GonArgs &a, int step, bool *ab) {
    __threadfence();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) st_relaxed_u64(row + r, v);
    uint64_t out = poll_slots(row, G, a.timeout_cycles, a.st, step, ab);
    __threadfence();
    if (SUM) {   // every slot is set: read them once more
        out = 0;
        for (int q = threadIdx.x & 31; q < G; q += 32) out += ld_relaxed_u64(row + q) - 1;
#pragma unroll
        for (int o = 16; o; o >>= 1) out += __shfl_xor_sync(0xFFFFFFFFu, out, o);
    }
    return out;
}

struct SkipMem {   // shared memory of a CTA
    float *cs;                 // [d] the newest center
    float *h;                  // [SKIP_BINS / 2] lower bounds on its distances to the regrouping's centers
    unsigned long long *key;   // [units] cached keys
    float *rho;                // [units]
    uint32_t *list;            // [units] touched units
    uint16_t *rep;             // [units]
    unsigned *bins;            // scratch: [2 SKIP_BINS] counts, offsets; then the transpose tiles
    float *tile;               // [SKIP_W][SKIP_TILE]; between regroupings the centers, [d][ncen]
    float *part;               // [SKIP_NT]
};

// Do the regrouping's centers fit where the tiles are?
__device__ __forceinline__ bool rep_shared(int ncen, int d) { return ncen * d <= SKIP_W * SKIP_TILE; }

// One point's row number in rm.
__device__ __forceinline__ int64_t row_of(const GonSkip &K, uint32_t x) { return K.rmap ? K.rmap[x] : (int64_t)x; }

// Counting sort of the positions by bin and repacking of the CTA's blocks.
// from / to: the state (perm, mind, asg) before and after; from.perm null: the
// identity over n points.  Returns the number of positions (0: gave up).
struct SkipState {
    uint32_t *perm, *mind;
    uint16_t *asg;
};
constexpr uint32_t NO_POINT = 0xFFFFFFFFu;

template <int DC>
__device__ __noinline__ int64_t skip_regroup(const GonArgs &a, const GonInst &I, const GonSkip &SK, ShSkip &sh, const SkipMem &M, int r,
                                             int ncen, uint32_t far, int64_t npos, const SkipState &from,
                                             const SkipState &to, uint64_t *rows) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = DC > 0 ? DC : I.d, G = I.G, nbin = 2 * ncen;
    const float g2 = a.skip.g2;
    unsigned *cnt = M.bins, *off = M.bins + SKIP_BINS;
    for (int b = tid; b < nbin; b += SKIP_NT) cnt[b] = 0;
    __syncthreads();
    const int64_t p0 = npos * r / G, p1 = npos * (r + 1) / G, extent = skip_extent(I.n);
    auto bin_of = [&](int64_t i) { return 2 * (int)__ldcg(from.asg + i) + (__ldcg(from.mind + i) > far ? 1 : 0); };
#pragma unroll 4
    for (int64_t i = p0 + tid; i < p1; i += SKIP_NT)
        if (!from.perm || __ldcg(from.perm + i) != NO_POINT) {
            const int b = bin_of(i);
            if (KC_IN_RANGE(a.st, b, nbin, KC_AT_SKIP_BIN)) atomicAdd(&cnt[b], 1u);
        }
    __syncthreads();
    for (int b = tid; b < nbin; b += SKIP_NT) __stcg(SK.hist + (int64_t)r * SKIP_BINS + b, cnt[b]);
    __syncthreads();
    if (warp == 0) {
        bool ab = false;
        skip_round<false>(rows, r, G, 1, a, ncen, &ab);
        if (lane == 0) sh.abort = ab;
    }
    __syncthreads();
    if (sh.abort) return 0;
    // totals over the CTAs and the part of the CTAs before this one
    for (int b = tid; b < SKIP_BINS; b += SKIP_NT) {
        unsigned tot = 0, mine = 0;
        if (b < nbin) {
#pragma unroll 8
            for (int q = 0; q < G; ++q) {
                const unsigned v = __ldcg(SK.hist + (int64_t)q * SKIP_BINS + b);
                if (q < r) mine += v;
                tot += v;
            }
        }
        cnt[b] = tot;
        off[b] = mine;
    }
    __syncthreads();
    // exclusive scan of the padded totals: BPT bins per thread
    constexpr int BPT = SKIP_BINS / SKIP_NT;
    unsigned tot[BPT], uni[BPT], inc = 0;
#pragma unroll
    for (int q = 0; q < BPT; ++q) {
        tot[q] = cnt[BPT * tid + q];
        uni[q] = (tot[q] + UNIT - 1) / UNIT;
        inc += uni[q];
    }
    const unsigned mine = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) sh.scan[warp] = (int)inc;
    __syncthreads();
    if (warp == 0) {
        unsigned v = lane < SKIP_W ? (unsigned)sh.scan[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned w = __shfl_up_sync(0xFFFFFFFFu, v, o);
            if (lane >= o) v += w;
        }
        sh.scan[lane] = (int)v;
    }
    __syncthreads();
    const unsigned units = (unsigned)sh.scan[31];
    unsigned first = inc - mine + (warp ? (unsigned)sh.scan[warp - 1] : 0u);
    // cnt: first unit of each bin; off: next position of this CTA's points
#pragma unroll
    for (int q = 0; q < BPT; ++q) {
        off[BPT * tid + q] += first * UNIT;
        cnt[BPT * tid + q] = first;
        if (r == 0)   // the gap behind the bin's points
            for (unsigned p = first * UNIT + tot[q]; p < (first + uni[q]) * UNIT; ++p) __stcg(to.perm + p, NO_POINT);
        first += uni[q];
    }
    // positions of the last block past the last unit
    if (r == 0 && tid == 0)
        for (unsigned p = units * UNIT; p % BLK != 0; ++p) __stcg(to.perm + p, NO_POINT);
    __syncthreads();
#pragma unroll 4
    for (int64_t i = p0 + tid; i < p1; i += SKIP_NT) {
        const uint32_t x = from.perm ? __ldcg(from.perm + i) : (uint32_t)i;
        if (x == NO_POINT) continue;
        const unsigned p = atomicAdd(&off[bin_of(i)], 1u);
        if (!KC_IN_RANGE(a.st, p, extent, KC_AT_SKIP_BIN)) continue;
        __stcg(to.perm + p, x);
        __stcg(to.mind + p, __ldcg(from.mind + i));
        __stcg(to.asg + p, __ldcg(from.asg + i));
    }
    __syncthreads();
    if (warp == 0) {
        bool ab = false;
        skip_round<false>(rows + G, r, G, 1, a, ncen, &ab);
        if (lane == 0) sh.abort = ab;
    }
    __syncthreads();
    if (sh.abort) return 0;
    const int64_t out = ((int64_t)units * UNIT + BLK - 1) / BLK * BLK;
    const int64_t nb = out / BLK;
    // the CTA's units: their centers (before the tiles overwrite the bins) ...
    const int nu = (int)((nb - r + G - 1) / G) * (BLK / UNIT);
    if (!KC_IN_RANGE(a.st, nu, a.skip.units + 1, KC_AT_SKIP_UNIT) || !KC_IN_RANGE(a.st, out, extent + 1, KC_AT_SKIP_BIN)) return 0;
    for (int u = tid; u < nu; u += SKIP_NT) {
        const unsigned gu = (unsigned)((int64_t)(u / (BLK / UNIT)) * G + r) * (BLK / UNIT) + u % (BLK / UNIT);
        int lo = 0, hi = nbin - 1;   // the last bin that starts at or before the unit
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cnt[mid] <= gu) lo = mid;
            else hi = mid - 1;
        }
        M.rep[u] = (uint16_t)(lo / 2);
    }
    __syncthreads();
    // ... and their coordinates, transposed 32 points x 32 coordinates at a time
    float *tile = M.tile + warp * SKIP_TILE;
    float *pk = (float *)I.pk;
    const float *__restrict__ rm = I.rm;
    for (int u = warp; u < nu; u += SKIP_W) {
        const int64_t b = (int64_t)(u / (BLK / UNIT)) * G + r;
        const int64_t p = b * BLK + (u % (BLK / UNIT)) * UNIT + lane;
        uint32_t x = __ldcg(to.perm + p);
        if (x != NO_POINT && !KC_IN_RANGE(a.st, x, I.n, KC_AT_SKIP_ROW)) x = NO_POINT;
        const uint32_t m = x != NO_POINT ? __ldcg(to.mind + p) : 0u;
        const int64_t row = x != NO_POINT ? row_of(SK, x) : -1;
        const uint64_t key = warp_max_u64(x != NO_POINT ? make_key(m, x) : 0);
        if (lane == 0) {
            M.key[u] = key;
            M.rho[u] = bound_up(__uint_as_float(key_val(key)), g2);
        }
        for (int j0 = 0; j0 < d; j0 += 32) {
            float v[UNIT];   // all 32 rows' loads in flight
#pragma unroll
            for (int q = 0; q < UNIT; ++q) {
                const int64_t rq = __shfl_sync(0xFFFFFFFFu, row, q);
                v[q] = rq >= 0 && j0 + lane < d ? __ldg(rm + rq * d + j0 + lane) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < UNIT; ++q) tile[q * 33 + lane] = v[q];
            __syncwarp();
            float *dst = pk + (b * d + j0) * BLK + (u % (BLK / UNIT)) * UNIT + lane;
#pragma unroll 8
            for (int j = 0; j < 32; ++j)
                if (j0 + j < d) __stcg(dst + j * BLK, tile[lane * 33 + j]);
            __syncwarp();
        }
    }
    __syncthreads();
    // the centers' coordinates for skip_bounds: in shared memory where the
    // tiles were, or (too many) in global memory, written by the first CTA
    // ([d][ncen] both; read by the others behind the caller's barrier)
    if (rep_shared(ncen, d)) {
        for (int e = tid; e < ncen * d; e += SKIP_NT) {
            const int i = e / d, j = e - i * d;
            M.tile[j * ncen + i] = __ldg(rm + __ldcg(I.centers + i) * d + j);
        }
    } else if (r == 0) {
        for (int e = tid; e < ncen * d; e += SKIP_NT) {
            const int i = e / d, j = e - i * d;
            __stcg(I.cenT + (int64_t)j * ncen + i, __ldg(rm + __ldcg(I.centers + i) * d + j));
        }
    }
    __syncthreads();
    return out;
}

// h[i]: a lower bound on the distance of the newest center (cs) to center i;
// 2^s threads share a center's coordinates (no order to keep here).
__device__ __forceinline__ void skip_bounds(const GonInst &I, const SkipMem &M, int d, int ncen, float f) {
    const bool shared = rep_shared(ncen, d);
    int s = 0;
    while (s < 4 && (ncen << (s + 1)) <= SKIP_NT && (4 << s) <= d) ++s;
    const int per = 1 << s, sub = threadIdx.x >> (31 - __clz(SKIP_NT) - s);
    // thread = sub * (SKIP_NT / per) + center: a warp's lanes read neighbouring centers
    const int width = SKIP_NT >> s;
    float *part = M.part;   // [SKIP_NT]
    for (int i0 = 0; i0 < ncen; i0 += width) {
        const int i = i0 + (threadIdx.x & (width - 1));
        float acc = 0.f;
        if (i < ncen) {
            if (shared) {
#pragma unroll 4
                for (int j = sub; j < d; j += per) acc = sq_step(acc, M.tile[j * ncen + i], M.cs[j]);
            } else {
#pragma unroll 8
                for (int j = sub; j < d; j += per) acc = sq_step(acc, __ldcg(I.cenT + (int64_t)j * ncen + i), M.cs[j]);
            }
        }
        part[threadIdx.x] = acc;
        __syncthreads();
        if (threadIdx.x < width && i < ncen) {
            for (int o = 1; o < per; ++o) acc = __fadd_rn(acc, part[o * width + threadIdx.x]);
            M.h[i] = acc >= 0x1p-100f && acc <= 3.0e38f ? __fmul_rd(__fsqrt_rd(acc), f) : 0.f;
        }
        __syncthreads();
    }
}

// The touched units (list[0, n)): distances, minima, assignments, keys.  A
// warp takes a unit, a lane one point, up to 64 coordinate loads in flight.
template <int DC>
__device__ __forceinline__ void skip_units(const GonArgs &a, const GonInst &I, const SkipMem &M, const SkipState &S, int n,
                                           int r, int it) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int d = DC > 0 ? DC : I.d, G = I.G;
    const float *pk = (const float *)I.pk;
    for (int e = warp; e < n; e += SKIP_W) {
        const int u = (int)M.list[e];
        if (!KC_IN_RANGE(a.st, u, a.skip.units, KC_AT_SKIP_UNIT)) continue;
        const int64_t b = (int64_t)(u / (BLK / UNIT)) * G + r;
        const int q = (u % (BLK / UNIT)) * UNIT + lane;
        const int64_t p = b * BLK + q;
        const float *src = pk + b * d * BLK + q;
        const uint32_t x = __ldcg(S.perm + p), o = __ldcg(S.mind + p);
        float acc = 0.f;
        int j = 0;
#pragma unroll 1
        for (; j + 64 <= d; j += 64) {
            float v[64];
#pragma unroll
            for (int t = 0; t < 64; ++t) v[t] = __ldcg(src + (j + t) * BLK);
#pragma unroll
            for (int t = 0; t < 64; ++t) acc = sq_step(acc, v[t], M.cs[j + t]);
        }
        if (DC % 64 != 0 || DC == 0) {
#pragma unroll 1
            for (; j + 16 <= d; j += 16) {
                float v[16];
#pragma unroll
                for (int t = 0; t < 16; ++t) v[t] = __ldcg(src + (j + t) * BLK);
#pragma unroll
                for (int t = 0; t < 16; ++t) acc = sq_step(acc, v[t], M.cs[j + t]);
            }
            float v[16];
#pragma unroll
            for (int t = 0; t < 16; ++t) v[t] = j + t < d ? __ldcg(src + (j + t) * BLK) : 0.f;
#pragma unroll
            for (int t = 0; t < 16; ++t)
                if (j + t < d) acc = sq_step(acc, v[t], M.cs[j + t]);
        }
        const uint32_t s = __float_as_uint(acc);
        if (x != NO_POINT && s < o) {
            __stcg(S.mind + p, s);
            __stcg(S.asg + p, (uint16_t)it);
        }
        const uint64_t key = warp_max_u64(x != NO_POINT ? make_key(min(s, o), x) : 0);
        if (lane == 0) M.key[u] = key;
    }
}

template <int DC>
__global__ void __launch_bounds__(SKIP_NT, 1) gon_skip_kernel(GonArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ GonInst I;
    __shared__ GonSkip SK;
    __shared__ ShSkip sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) SK = a.skip;
    copy_instance(I, &a.single);
    const int it0 = ld_volatile_i32(a.route);
    if (it0 == 0 || ld_volatile_i32(&a.st->code) != 0) return;
    const int r = (int)blockIdx.x, G = I.G, k = I.k;
    const int d = DC > 0 ? DC : I.d;
    const float g2 = a.skip.g2;
    SkipMem M;
    M.key = reinterpret_cast<unsigned long long *>(smem_raw);
    M.rho = reinterpret_cast<float *>(M.key + a.skip.units);
    M.list = reinterpret_cast<uint32_t *>(M.rho + a.skip.units);
    M.cs = reinterpret_cast<float *>(M.list + a.skip.units);
    M.h = M.cs + ((d + 3) & ~3);
    M.bins = reinterpret_cast<unsigned *>(M.h + SKIP_BINS / 2);
    M.tile = reinterpret_cast<float *>(M.bins);
    M.part = M.tile + SKIP_W * SKIP_TILE;
    M.rep = reinterpret_cast<uint16_t *>(M.part + SKIP_NT);
    uint64_t K = *I.final_key;   // the streaming steps' last winner: center it0
    __syncthreads();             // every thread has read it before it is overwritten at the end

    if (warp == 0) {
        const int64_t c = key_idx(K);
        const bool ok = KC_IN_RANGE(a.st, c, I.n, KC_AT_CENTER_LOAD) && KC_IN_RANGE(a.st, it0, I.kcap, KC_AT_CENTER_COPY);
        if (ok) {
            for (int j = lane; j < d; j += 32) M.cs[j] = I.rm[row_of(SK, (uint32_t)c) * d + j];
            if (r == 0 && lane == 0) I.centers[it0] = out_index(I, c);
        }
        if (lane == 0) {
            sh.abort = !ok;
            sh.ntouch = 0;
            sh.touched = 0;
        }
    }
    __syncthreads();
    if (sh.abort) return;
    // the state in point order, then the two regrouped ones in turn
    SkipState S[2] = {{nullptr, I.mind, SK.asg[0]}, {SK.perm[0], SK.mind[0], SK.asg[1]}};
    // slot rows of the regroupings: behind the exchange rows of the k steps
    uint64_t *xrow = I.slots + (int64_t)k * slot_stride(G) * (I.lp_kind ? 2 : 1);
    uint64_t *const xrow0 = xrow;
    int cur = 0, ncen = 0, nu = 0, it;
    int64_t npos = I.n;
    int next = it0, rounds = 0;   // step of the next regrouping decision
    for (it = it0; it < k; ++it) {
        if (it == next) {
            bool go = rounds == 0;
            // this decision's rows: the touched units' sum, two of a regrouping, the centers
            if (!KC_IN_RANGE(a.st, (xrow - xrow0) / G + 3, 4 * SKIP_ROUNDS, KC_AT_SLOT)) break;
            if (!go) {
                // regroup again when the units touched since the last one are
                // more than a few percent and enough steps remain
                if (warp == 0) {
                    bool ab = false;
                    const uint64_t t = skip_round<true>(xrow, r, G, sh.touched + 1, a, it, &ab);
                    if (lane == 0) {
                        sh.key = t;
                        sh.abort = ab;
                    }
                }
                __syncthreads();
                if (sh.abort) break;
                const double share = (double)sh.key * UNIT / ((double)npos * (it - ncen));
                go = share > 0.03 && share * (k - it) > 6.0;   // its cost: a few whole sweeps
                __syncthreads();
                xrow += G;
            }
            if (go) {
                const uint32_t far = __float_as_uint(0.25f * __uint_as_float(key_val(K)));
                const int64_t np = skip_regroup<DC>(a, I, SK, sh, M, r, it, far, npos, S[cur], S[cur ^ 1], xrow);
                if (np == 0) break;
                xrow += 2 * G;
                npos = np;
                if (rounds == 0) S[0] = {SK.perm[1], SK.mind[1], SK.asg[0]};
                cur ^= 1;
                ncen = it;
                nu = (int)((npos / BLK - r + G - 1) / G) * (BLK / UNIT);
                if (tid == 0) sh.touched = 0;
                __syncthreads();
                if (!rep_shared(ncen, d)) {   // the first CTA's copy of the centers
                    if (warp == 0) {
                        bool ab = false;
                        skip_round<false>(xrow, r, G, 1, a, it, &ab);
                        if (lane == 0) sh.abort = ab;
                    }
                    __syncthreads();
                    if (sh.abort) break;
                    xrow += G;
                }
            }
            ++rounds;
            next = 2 * it <= SKIP_BINS / 2 && rounds < SKIP_ROUNDS ? 2 * it : k;
        }
        skip_bounds(I, M, d, ncen, a.skip.f);
        for (int u0 = 0; u0 < nu; u0 += SKIP_NT) {
            const int u = u0 + tid;
            bool touch = false;
            if (u < nu) {
                const float m = __uint_as_float(key_val(M.key[u]));
                touch = m > 0.f && __fsub_rd(M.h[M.rep[u]], M.rho[u]) < bound_up(m, g2);
            }
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, touch);
            int at = 0;
            if (lane == 0 && bal) at = atomicAdd(&sh.ntouch, __popc(bal));
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            at += __popc(bal & ((1u << lane) - 1u));
            if (touch && KC_IN_RANGE(a.st, at, a.skip.units, KC_AT_SKIP_UNIT)) M.list[at] = (uint32_t)u;
        }
        __syncthreads();
        const int nt = sh.ntouch;
        skip_units<DC>(a, I, M, S[cur], nt, r, it);
        __syncthreads();
        uint64_t best = 0;
        for (int u = tid; u < nu; u += SKIP_NT) best = umax64(best, M.key[u]);
        best = warp_max_u64(best);
        if (lane == 0) sh.red[warp] = best;
        if (tid == 0) {
            sh.ntouch = 0;
            sh.touched += nt;
        }
        __syncthreads();
        if (warp == 0) {
            uint64_t v = lane < SKIP_W ? sh.red[lane] : 0;
            v = warp_max_u64(v);
            uint64_t g = v;
            bool ab = false;
            const bool more = it + 1 < k;
            // the CTA's candidate may be the next center: have its row on the way
            if (more && v != 0) {
                const float *row = I.rm + row_of(SK, key_idx(v)) * d;
                for (int j = lane * 8; j < d; j += 256) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + j));
            }
            const bool lead = G > LEADER_MIN;
            const uint32_t tag = (I.lp_kind ? 2u : 1u) * ((uint32_t)it + 1);   // above the streaming steps' tags
            if (G > 1) {
                uint64_t *row = I.slots + (int64_t)it * slot_stride(G);
                const bool held = a.withhold == it + 1 && r == G - 1;
                if (lane == 0 && !held && !(lead && r == 0)) st_relaxed_u64(row + r, v ? v : 1);
                if (!lead || r == 0) {
                    g = lead ? poll_slots<1>(row, G, a.timeout_cycles, a.st, it, &ab, v)
                             : poll_slots(row, G, a.timeout_cycles, a.st, it, &ab);
                } else {
                    uint32_t kw = 0;
                    ab = follow_leader(I.bc, tag, more ? d + 2 : 2, a.timeout_cycles, a.st, it, [&](int w, uint32_t b) {
                        if (w < 2) kw = b;
                        else M.cs[w - 2] = __uint_as_float(b);
                    });
                    g = ((uint64_t)__shfl_sync(0xFFFFFFFFu, kw, 0) << 32) | __shfl_sync(0xFFFFFFFFu, kw, 1);
                }
            }
            if (!ab && more && (!lead || r == 0)) {
                const int64_t c = key_idx(g);
                if (key_val(g) == 0 || KC_IN_RANGE(a.st, c, I.n, KC_AT_CENTER_LOAD)) {
                    const float *src = key_val(g) != 0 ? I.rm + row_of(SK, (uint32_t)c) * d : nullptr;
                    for (int j = lane; j < d; j += 32) {
                        const float x = src ? __ldg(src + j) : 0.f;
                        M.cs[j] = x;
                        if (lead) st_relaxed_u64(I.bc + 2 + j, ((uint64_t)tag << 32) | __float_as_uint(x));
                    }
                } else {
                    ab = true;
                }
            }
            if (lead && r == 0 && !ab && lane < 2)
                st_relaxed_u64(I.bc + lane, ((uint64_t)tag << 32) | (lane == 0 ? g >> 32 : g & 0xFFFFFFFFu));
            if (!ab && more && key_val(g) != 0 && r == 0 && lane == 0) I.centers[it + 1] = out_index(I, key_idx(g));
            if (lane == 0) {
                sh.key = g;
                sh.abort = ab;
            }
        }
        __syncthreads();
        if (sh.abort) break;
        K = sh.key;
        if (key_val(K) == 0) {   // every point is at distance 0: stop early
            ++it;
            break;
        }
    }
    if (sh.abort) return;

    // the minima in point order, for the radius recheck (I.mind is no longer read)
    for (int u = warp; u < nu; u += SKIP_W) {
        const int64_t p = ((int64_t)(u / (BLK / UNIT)) * G + r) * BLK + (u % (BLK / UNIT)) * UNIT + lane;
        const uint32_t x = __ldcg(S[cur].perm + p);
        if (x != NO_POINT && KC_IN_RANGE(a.st, x, I.n, KC_AT_SKIP_ROW)) I.mind[x] = __ldcg(S[cur].mind + p);
    }
    if (r == 0 && tid == 0) {
        *I.k_out = it;
        *I.final_key = K;
    }
}

void *pick_skip(int d) {
    switch (d) {
        case 16: return (void *)gon_skip_kernel<16>;
        case 32: return (void *)gon_skip_kernel<32>;
        case 64: return (void *)gon_skip_kernel<64>;
        default: return (void *)gon_skip_kernel<0>;
    }
}

// Most units of one CTA, and the shared memory for them.
int skip_units_max(int64_t n, int G) {
    const int64_t nb = skip_positions(n) / BLK;
    return (int)((nb + G - 1) / G) * (BLK / UNIT);
}
size_t skip_smem(int d, int units) {
    return (size_t)units * 18 + ((size_t)((d + 3) & ~3) + SKIP_BINS / 2 + (size_t)SKIP_W * SKIP_TILE + SKIP_NT) * 4;
}

}  // namespace

int64_t skip_positions(int64_t n) { return skip_extent(n); }
int64_t skip_route_words() { return 8 + 2 * PROBE_S; }
int64_t skip_hist_words(int G) { return (int64_t)G * SKIP_BINS; }
int64_t skip_slot_rows() { return 4 * SKIP_ROUNDS; }

int gon_skip_segments(int dtype, int d, int64_t n, int k, int grid, int *ends, int cap) {
    const char *env = getenv("KC_GON_SKIP");
    if (env && atoi(env) == 0) return 0;
    if (dtype != KC_F32 || k > 32768 || d > 4096) return 0;
    // Below d = 8 a point is little more than its state (10M x 3, k = 250: 8.8
    // ms streaming, 12.2 here; 8M x 2, k = 400: 8.1 and 8.1), and a solve of a
    // few ms has little to win beside its probes.
    if (!env && (d < 8 || (double)n * d * k < 1e10)) return 0;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (skip_smem(d, skip_units_max(n, grid)) + sizeof(ShSkip) + sizeof(GonInst) + 1024 > (size_t)optin) return 0;
    // a probe costs about 30 us with the launch behind it: after 16, 32, 64, ...
    // steps of a solve of 15 ms or more, after 16, 64 and 256 of a shorter one
    const int grow = (double)n * (4.0 * d + 4.0) * k >= 1e11 ? 2 : 4;
    int m = 0;
    for (int e = 16; m < cap && e <= PROBE_MAX && 4 * e <= 3 * k; e *= grow) ends[m++] = e;
    return m;
}

bool gon_skip_possible(int dtype, int d, int64_t n, int k, int grid) {
    int ends[8];
    return gon_skip_segments(dtype, d, n, k, grid, ends, 8) > 0;
}

cudaError_t launch_gon_probe(const GonArgs &a, int it0, bool last, unsigned *words, cudaStream_t s) {
    const GonInst &I = a.single;
    // microseconds: a whole sweep at the HBM rate, or the one of L2 where the
    // points stay there (half the bytes in mixed precision), the assignment at
    // the FP32 rate and two regroupings
    const double n = (double)I.n, bytes = n * (I.d * (I.lp_kind ? 2.0 : 4.0) + 4.0);
    const float sweep = (float)(bytes / (bytes < 100e6 ? 14e6 : 6.9e6));
    // all units touched: perm and assignment too, and less even than a sweep
    // (8M x 64: a quarter of the units in 90 us); or a warp's waits, about 2 us
    // for a unit's first batch of loads and 1 for each further one (a tenth of the
    // units of 10M x 10, one batch, in 26 us, of 4M x 32, two, in 12)
    const int batches = I.d / 64 + (I.d % 64 + 15) / 16;
    const float unit = (float)std::max(1.25 * n * (I.d * 4.0 + 12.0) / 6.9e6,
                                       n / UNIT / (SKIP_W * (double)I.G) * (1.0 + batches));
    const float once = (float)(n * I.d * it0 / 1.2e7 + 2.0 * n * (8.0 * I.d + 100.0) / 4e6 + 60.0);
    const char *env = getenv("KC_GON_SKIP");   // testing: 1 = change over at the first probe
    const bool force = env && atoi(env) > 0;
    // beyond a streaming step's exchange, with the tests of all units (10M x 10, a tenth
    // of the units touched: 36 us a step, 26 of them the units, 3.5 the exchange)
    const float fixed = (float)(3.0 + n / 2e6);
    gon_probe_kernel<<<PROBE_CTAS, PROBE_NT, 0, s>>>(I.rm, a.skip.rmap, I.n, I.d, I.centers, I.final_key, it0,
                                                     force ? 1e9f : sweep, unit, fixed, once, I.k - it0, last, a.route,
                                                     words, reinterpret_cast<uint2 *>(words + 4), a.st);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_gon_skip(GonArgs &a, int last, cudaStream_t s) {
    const GonInst &I = a.single;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    gon_center_rows_kernel<<<(int)std::min<int64_t>(sms, ((int64_t)last * I.d + 255) / 256), 256, 0, s>>>(I, a.route, a.st);
    const size_t smem_a = nearest_smem(I.d);
    const int ga = nearest_grid(I.n, sms);
    if (I.d == 64) gon_assign_kernel<64><<<ga, NEAREST_NT, smem_a, s>>>(I, a.skip.asg[0], a.route, a.st);
    else gon_assign_kernel<0><<<ga, NEAREST_NT, smem_a, s>>>(I, a.skip.asg[0], a.route, a.st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    void *fn = pick_skip(I.d);
    a.skip.units = skip_units_max(I.n, a.grid);
    // FP64 is slow here: taken once, not by every thread
    a.skip.g2 = (float)(2.0 * f32_gamma(I.d)) + 0x1p-22f;
    a.skip.f = (float)(1.0 - 2.0 * f32_gamma(I.d) - 0x1p-18);
    const size_t smem = skip_smem(I.d, a.skip.units);
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    note_launches(3);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.grid);
    cfg.blockDim = dim3(SKIP_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {&a};
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace kc
