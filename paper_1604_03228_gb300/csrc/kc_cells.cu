// kc_cells.cu -- EIM's prune by Voronoi cells (Algorithm 2; float points).
//
// A round of EIM removes from R every x with d(x, S) <= thr, the block of
// |R| x |S| distances Section 5.2 finds dominant.  Here the points are first
// assigned to the nearest of P pivots (rows of S), once per call.  With rho_p
// a bound on the distances of the points of R in cell p to pivot p, and
// sigma_q the same for S and cell q, the pairs of the two cells cannot lie
// within thr of each other when
//   d(p, q) - rho_p - sigma_q > sqrt(thr),
// so each round sorts R and S by cell and compares cell p of R only with the
// cells of S that this leaves (near lists).  Everything else is decided as
// before, by the same tests on the same canonical distances; R and S are sets,
// so their order does not matter.
// Bounds (f32_gamma(d) = g; see kc_gonskip.cu): D(x, p) <= sqrt(s) (1 + 2 g),
// D(p, q) >= sqrt(t) (1 - 2 g - 2^-18), s(x, c) > thr follows from D(x, c) >
// sqrt(thr) (1 + 2 g); all rounded to the safe side.
#include <algorithm>

#include "kc_internal.cuh"
#include "kc_nearest.cuh"

namespace kc {

namespace {

constexpr uint32_t NO_POINT = 0xFFFFFFFFu;

// ----------------------------------------------------------------- assign
// Nearest pivot of every point of the packed array and its canonical distance
// (three CTAs per SM for d = 2; with two EIM on 1M x 2 takes 1.76 ms, not 1.73).
template <int DC>
__global__ void __launch_bounds__(NEAREST_NT, DC == 2 ? 3 : 2) cells_assign_kernel(const float *__restrict__ pk, int64_t n, int d,
                                                                     const float *__restrict__ piv, int P,
                                                                     uint16_t *__restrict__ cell,
                                                                     uint32_t *__restrict__ dist) {
    extern __shared__ __align__(16) float as_c[];
    const int dd = DC > 0 ? DC : d;
    nearest_centers<DC>(pk, n, d, P, as_c, [=](int c, int j) { return __ldg(piv + (int64_t)c * dd + j); }, dist, cell);
}

// The same for a few thousand rows (d < 16): a CTA takes 32 of them, a lane one,
// and its warps share the pivots, so that it takes the time of P / 8 pivots
// (the kernel above walks all P in each warp: 8853 x 12, P = 553, 70 us of 1.5
// ms of an EIM call).
constexpr int SAMPLE_NT = 256, SAMPLE_D = 16;
__global__ void __launch_bounds__(SAMPLE_NT) cells_sample_kernel(const float *__restrict__ rows, int64_t n, int d,
                                                                 const float *__restrict__ piv, int P,
                                                                 uint16_t *__restrict__ cell, uint32_t *__restrict__ dist) {
    __shared__ unsigned long long best[SAMPLE_NT / 32][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    float x[SAMPLE_D];
#pragma unroll
    for (int j = 0; j < SAMPLE_D; ++j) x[j] = i < n && j < d ? rows[i * d + j] : 0.f;
    unsigned long long b = ~0ull;   // (distance bits, pivot), smallest
    for (int p = warp; p < P; p += SAMPLE_NT / 32) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < SAMPLE_D; ++j) acc = sq_step(acc, x[j], j < d ? __ldg(piv + (int64_t)p * d + j) : 0.f);
        const unsigned long long k = ((unsigned long long)__float_as_uint(acc) << 32) | (unsigned)p;
        b = k < b ? k : b;
    }
    best[warp][lane] = b;
    __syncthreads();
    if (warp == 0 && i < n) {
        for (int w = 1; w < SAMPLE_NT / 32; ++w) b = best[w][lane] < b ? best[w][lane] : b;
        cell[i] = (uint16_t)b;
        dist[i] = (uint32_t)(b >> 32);
    }
}

// ------------------------------------------------------------------- sort
// Counting sort of a list of points by cell.  Counts and the largest distance
// of each cell, then (one CTA) the cells' starts, padded to `unit`, then the
// scatter: a CTA reserves a range of each cell for its chunk of the list.
constexpr int SORT_NT = 512, SORT_CHUNK = 8192;

__global__ void __launch_bounds__(SORT_NT) cells_count_kernel(const uint32_t *__restrict__ list, int64_t cnt, int P,
                                                              const uint16_t *__restrict__ cell,
                                                              const uint32_t *__restrict__ dist, unsigned *count,
                                                              unsigned *rad, DevStatus *st) {
    extern __shared__ unsigned sc[];   // [P] counts, [P] radii
    unsigned *sr = sc + P;
    for (int i = threadIdx.x; i < 2 * P; i += SORT_NT) sc[i] = 0;
    __syncthreads();
    for (int64_t c0 = (int64_t)blockIdx.x * SORT_CHUNK; c0 < cnt; c0 += (int64_t)gridDim.x * SORT_CHUNK) {
        const int64_t c1 = c0 + SORT_CHUNK < cnt ? c0 + SORT_CHUNK : cnt;
#pragma unroll 4
        for (int64_t i = c0 + threadIdx.x; i < c1; i += SORT_NT) {
            const uint32_t x = list ? list[i] : (uint32_t)i;
            const int p = cell[x];
            if (!KC_IN_RANGE(st, p, P, KC_AT_CELL)) continue;
            const uint32_t v = dist[x];
            atomicAdd(&sc[p], 1u);
            if (v > sr[p]) atomicMax(&sr[p], v);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P; i += SORT_NT) {
        if (sc[i]) atomicAdd(&count[i], sc[i]);
        if (sr[i]) atomicMax(&rad[i], sr[i]);
    }
}

// start[0..P] (padded), cursor = start; one CTA, P <= 1024.
__global__ void __launch_bounds__(1024) cells_starts_kernel(const unsigned *__restrict__ count, int P, int unit,
                                                            unsigned *__restrict__ start, unsigned *__restrict__ cursor) {
    __shared__ unsigned ws[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned mine = t < P ? (count[t] + unit - 1) / unit * unit : 0u;
    unsigned inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) ws[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        unsigned v = ws[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned w = __shfl_up_sync(0xFFFFFFFFu, v, o);
            if (lane >= o) v += w;
        }
        ws[lane] = v;
    }
    __syncthreads();
    const unsigned first = inc - mine + (warp ? ws[warp - 1] : 0u);
    if (t < P) start[t] = cursor[t] = first;
    if (t == 0) start[P] = ws[31];
}

__global__ void __launch_bounds__(SORT_NT) cells_scatter_kernel(const uint32_t *__restrict__ list, int64_t cnt, int P,
                                                                const uint16_t *__restrict__ cell, unsigned *cursor,
                                                                uint32_t *__restrict__ out, int64_t extent,
                                                                DevStatus *st) {
    extern __shared__ unsigned sc[];   // [P]
    for (int64_t c0 = (int64_t)blockIdx.x * SORT_CHUNK; c0 < cnt; c0 += (int64_t)gridDim.x * SORT_CHUNK) {
        const int64_t c1 = c0 + SORT_CHUNK < cnt ? c0 + SORT_CHUNK : cnt;
        for (int i = threadIdx.x; i < P; i += SORT_NT) sc[i] = 0;
        __syncthreads();
#pragma unroll 4
        for (int64_t i = c0 + threadIdx.x; i < c1; i += SORT_NT) atomicAdd(&sc[cell[list[i]]], 1u);
        __syncthreads();
        for (int i = threadIdx.x; i < P; i += SORT_NT)
            if (sc[i]) sc[i] = atomicAdd(&cursor[i], sc[i]);
        __syncthreads();
#pragma unroll 4
        for (int64_t i = c0 + threadIdx.x; i < c1; i += SORT_NT) {
            const uint32_t x = list[i];
            const unsigned p = atomicAdd(&sc[cell[x]], 1u);
            if (KC_IN_RANGE(st, p, extent, KC_AT_CELL_POS)) out[p] = x;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------- near
// Cell p of R against every cell q of S: q joins p's list unless its points
// are provably farther than thr.  One CTA per p; the cell itself comes first
// when it holds points of S (most removals are found there).
constexpr int NEAR_NT = 256;
__global__ void __launch_bounds__(NEAR_NT) cells_near_kernel(const float *__restrict__ piv, int P, int d,
                                                             const unsigned *__restrict__ rcount,
                                                             const unsigned *__restrict__ rrad,
                                                             const unsigned *__restrict__ scount,
                                                             const unsigned *__restrict__ srad,
                                                             const uint32_t *thr_p, float g2, float f,
                                                             uint16_t *__restrict__ near, int *__restrict__ nnear,
                                                             DevStatus *st) {
    extern __shared__ float np[];   // [d] pivot p
    __shared__ int cnt;
    const int p = blockIdx.x;
    for (int j = threadIdx.x; j < d; j += NEAR_NT) np[j] = piv[(int64_t)p * d + j];
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    const bool any = rcount[p] != 0;
    if (threadIdx.x == 0 && any && scount[p] != 0) {
        near[(int64_t)p * P] = (uint16_t)p;
        cnt = 1;
    }
    __syncthreads();
    auto up = [&](unsigned m) { return __fmul_ru(__fsqrt_ru(__uint_as_float(m)), __fadd_ru(1.f, g2)); };
    const float need = __fadd_ru(up(*thr_p), up(rrad[p]));
    for (int q = threadIdx.x; q < P && any; q += NEAR_NT) {
        if (q == p || scount[q] == 0) continue;
        float t = 0.f;
#pragma unroll 8
        for (int j = 0; j < d; ++j) t = sq_step(t, np[j], __ldg(piv + (int64_t)q * d + j));
        const float h = t >= 0x1p-100f && t <= 3.0e38f ? __fmul_rd(__fsqrt_rd(t), f) : 0.f;
        if (h > __fadd_ru(need, up(srad[q]))) continue;
        const int at = atomicAdd(&cnt, 1);
        if (KC_IN_RANGE(st, at, P, KC_AT_CELL)) near[(int64_t)p * P + at] = (uint16_t)q;
    }
    __syncthreads();
    if (threadIdx.x == 0) nnear[p] = cnt;
}

// Pairs that the near lists leave: the sum over the cells p of R's points of p
// times S's points of the cells near p.  One CTA per p.
constexpr int PAIRS_NT = 128;
__global__ void __launch_bounds__(PAIRS_NT) cells_pairs_kernel(const uint16_t *__restrict__ near,
                                                               const int *__restrict__ nnear, int P,
                                                               const unsigned *__restrict__ rcount,
                                                               const unsigned *__restrict__ scount,
                                                               unsigned long long *pairs) {
    const int p = blockIdx.x, m = nnear[p];
    unsigned sum = 0;
    for (int e = threadIdx.x; e < m; e += PAIRS_NT) sum += scount[near[(int64_t)p * P + e]];
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(pairs, (unsigned long long)sum * rcount[p]);
}

// The near lists as center tiles of `tile` positions of sorted S (whose cells
// start at multiples of it): tiles[p][0 .. ntile[p]).
__global__ void __launch_bounds__(256) cells_tiles_kernel(const uint16_t *__restrict__ near, const int *__restrict__ nnear,
                                                          int P, const unsigned *__restrict__ sstart, int tile, int cap,
                                                          int *__restrict__ tiles, int *__restrict__ ntile, DevStatus *st) {
    __shared__ int cnt;
    const int p = blockIdx.x, m = nnear[p];
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    for (int e = 0; e < m; ++e) {
        const int q = near[(int64_t)p * P + e];
        const int t0 = (int)(sstart[q] / tile), t1 = (int)(sstart[q + 1] / tile);
        const int at = cnt;
        __syncthreads();
        for (int t = t0 + threadIdx.x; t < t1; t += 256)
            if (KC_IN_RANGE(st, at + t - t0, cap, KC_AT_TILE)) tiles[(int64_t)p * cap + at + t - t0] = t;
        if (threadIdx.x == 0) cnt = at + t1 - t0;
        __syncthreads();
    }
    if (threadIdx.x == 0) ntile[p] = cnt;
}

// ------------------------------------------------------------------ prune
// The CUDA-core prune by cells: a CTA takes CP_NT points of one cell of sorted
// R, and walks the near cells of S (rows sorted, contiguous) in shared-memory
// tiles that several small cells share; a thread stops at its first center
// within thr, the CTA when all of its points are decided.
constexpr int CP_NT = 128, CP_TILE_BYTES = 16 * 1024;
template <int DR>
__global__ void __launch_bounds__(CP_NT) cells_prune_kernel(const float *__restrict__ src, int d,
                                                            const uint32_t *__restrict__ R,
                                                            const unsigned *__restrict__ rstart, int P,
                                                            const uint8_t *__restrict__ inS,
                                                            const float *__restrict__ Ss,
                                                            const unsigned *__restrict__ sstart,
                                                            const uint16_t *__restrict__ near,
                                                            const int *__restrict__ nnear, const uint32_t *thr_p,
                                                            uint32_t *__restrict__ Rn, unsigned long long *rnn, int64_t n,
                                                            int64_t sn, int64_t rn, DevStatus *st) {
    __shared__ __align__(16) float cs[CP_TILE_BYTES / 4];
    constexpr int TILE = CP_TILE_BYTES / (DR * 4);
    const uint32_t thr = *thr_p;
    const int64_t total = rstart[P];
    const int lane = threadIdx.x & 31;
    for (int64_t r0 = (int64_t)blockIdx.x * CP_NT; r0 < total; r0 += (int64_t)gridDim.x * CP_NT) {
        int lo = 0, hi = P - 1;   // the last cell that starts at or before r0
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (rstart[mid] <= r0) lo = mid;
            else hi = mid - 1;
        }
        const int p = lo;
        const uint32_t x = R[r0 + threadIdx.x];
        // d(x, S) = 0 for sampled points
        bool removed = x == NO_POINT || !KC_IN_RANGE(st, x, n, KC_AT_EIM_INDEX) || inS[x];
        float xc[DR];
#pragma unroll
        for (int j = 0; j < DR; ++j) xc[j] = (!removed && j < d) ? src[(int64_t)x * d + j] : 0.f;
        const int m = nnear[p];
        int e = 0, off = 0;   // near cell and position within it
        while (e < m) {
            if (__syncthreads_and(removed)) break;
            int fill = 0;
            while (e < m && fill < TILE) {
                const int q = near[(int64_t)p * P + e];
                const int64_t s0 = (int64_t)sstart[q] + off;
                const int len = (int)(sstart[q + 1] - s0);
                const int take = len < TILE - fill ? len : TILE - fill;
                for (int i = threadIdx.x; i < take * DR; i += CP_NT) {
                    const int c = i / DR, j = i - c * DR;
                    cs[(fill + c) * DR + j] = j < d && KC_IN_RANGE(st, s0 + c, sn, KC_AT_CELL_POS) ? Ss[(s0 + c) * d + j] : 0.f;
                }
                fill += take;
                if (take == len) {
                    ++e;
                    off = 0;
                } else {
                    off += take;
                }
            }
            __syncthreads();
            if (!removed) {
                for (int c = 0; c < fill; ++c) {
                    float acc = 0.f;
#pragma unroll
                    for (int j = 0; j < DR; ++j) acc = sq_step(acc, xc[j], cs[c * DR + j]);
                    if (__float_as_uint(acc) <= thr) {
                        removed = true;
                        break;
                    }
                }
            }
        }
        // survivors, one counter update per warp
        const unsigned keep = __ballot_sync(0xFFFFFFFFu, !removed);
        unsigned long long at = 0;
        if (lane == 0 && keep) at = atomicAdd(rnn, (unsigned long long)__popc(keep));
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
        at += __popc(keep & ((1u << lane) - 1u));
        if (!removed && KC_IN_RANGE(st, at, rn, KC_AT_CELL_POS)) Rn[at] = x;
        __syncthreads();
    }
}

// Pivot rows: the rows of the centers a Gonzalez run on `rows` selected (the
// first one again past *k_out).
__global__ void pivot_rows_kernel(const float *__restrict__ rows, int64_t n, int d, const int64_t *__restrict__ centers,
                                  const int32_t *k_out, int P, float *__restrict__ piv) {
    const int kc = (int)dev_count(k_out, P);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)P * d; e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / d);
        const int64_t c = i < kc ? centers[i] : 0;
        piv[e] = rows[(c >= 0 && c < n ? c : 0) * d + (e - (int64_t)i * d)];
    }
}

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

}  // namespace

cudaError_t launch_pivot_rows(const float *rows, int64_t n, int d, const int64_t *centers, const int32_t *k_out, int P,
                              float *piv, cudaStream_t s) {
    pivot_rows_kernel<<<std::max(1, std::min((int)(((int64_t)P * d + 255) / 256), sm_count() * 4)), 256, 0, s>>>(
        rows, n, d, centers, k_out, P, piv);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cells_assign(const float *pk, int64_t n, int d, const CellBufs &C, cudaStream_t s) {
    const size_t smem = nearest_smem(d);
    const int g = nearest_grid(n, sm_count());
    if (d == 64) cells_assign_kernel<64><<<g, NEAREST_NT, smem, s>>>(pk, n, d, C.piv, C.P, C.cell, C.dist);
    else if (d == 2) cells_assign_kernel<2><<<g, NEAREST_NT, smem, s>>>(pk, n, d, C.piv, C.P, C.cell, C.dist);
    else cells_assign_kernel<0><<<g, NEAREST_NT, smem, s>>>(pk, n, d, C.piv, C.P, C.cell, C.dist);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cells_sort(const uint32_t *list, int64_t cnt, int unit, const CellBufs &C, CellSort &O, DevStatus *st,
                              cudaStream_t s) {
    cudaMemsetAsync(O.count, 0, 2 * (size_t)C.P * sizeof(unsigned), s);   // counts and radii
    cudaMemsetAsync(O.idx, 0xFF, (size_t)(cnt + (int64_t)C.P * (unit - 1)) * sizeof(uint32_t), s);
    const int g = (int)std::min<int64_t>((cnt + SORT_CHUNK - 1) / SORT_CHUNK, (int64_t)sm_count() * 4);
    const size_t sm = (size_t)C.P * sizeof(unsigned);
    cells_count_kernel<<<g, SORT_NT, 2 * sm, s>>>(list, cnt, C.P, C.cell, C.dist, O.count, O.count + C.P, st);
    cells_starts_kernel<<<1, 1024, 0, s>>>(O.count, C.P, unit, O.start, O.cursor);
    cells_scatter_kernel<<<g, SORT_NT, sm, s>>>(list, cnt, C.P, C.cell, O.cursor, O.idx, cnt + (int64_t)C.P * (unit - 1), st);
    note_launches(3);
    return cudaGetLastError();
}

cudaError_t launch_cells_near(int d, const CellBufs &C, const CellSort &R, const CellSort &S, const uint32_t *thr,
                              DevStatus *st, cudaStream_t s) {
    const double g = f32_gamma(d);   // on the host: FP64 is slow on the device
    cells_near_kernel<<<C.P, NEAR_NT, (size_t)d * sizeof(float), s>>>(
        C.piv, C.P, d, R.count, R.count + C.P, S.count, S.count + C.P, thr, (float)(2.0 * g) + 0x1p-22f,
        (float)(1.0 - 2.0 * g - 0x1p-18), C.near, C.nnear, st);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cells_sample(const float *rows, int64_t cnt, int d, const CellBufs &C, CellSort &O, DevStatus *st,
                                cudaStream_t s) {
    cells_sample_kernel<<<(int)((cnt + 31) / 32), SAMPLE_NT, 0, s>>>(rows, cnt, d, C.piv, C.P, C.cell, C.dist);
    cudaMemsetAsync(O.count, 0, 2 * (size_t)C.P * sizeof(unsigned), s);
    const int g = (int)std::min<int64_t>((cnt + SORT_CHUNK - 1) / SORT_CHUNK, (int64_t)sm_count() * 4);
    cells_count_kernel<<<g, SORT_NT, 2 * (size_t)C.P * sizeof(unsigned), s>>>(nullptr, cnt, C.P, C.cell, C.dist, O.count,
                                                                              O.count + C.P, st);
    note_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_cells_pairs(const CellBufs &C, const CellSort &R, const CellSort &S, unsigned long long *pairs,
                               cudaStream_t s) {
    cudaMemsetAsync(pairs, 0, sizeof(unsigned long long), s);
    cells_pairs_kernel<<<C.P, PAIRS_NT, 0, s>>>(C.near, C.nnear, C.P, R.count, S.count, pairs);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cells_tiles(const CellBufs &C, const CellSort &S, int tile, int cap, int *tiles, int *ntile,
                               DevStatus *st, cudaStream_t s) {
    cells_tiles_kernel<<<C.P, 256, 0, s>>>(C.near, C.nnear, C.P, S.start, tile, cap, tiles, ntile, st);
    note_launches(1);
    return cudaGetLastError();
}

int cells_prune_unit() { return CP_NT; }

cudaError_t launch_cells_prune(const float *src, int d, int64_t rn, const uint8_t *inS, const float *Ss,
                               const CellBufs &C, const CellSort &R, const CellSort &S, const uint32_t *thr, uint32_t *Rn,
                               unsigned long long *rnn, int64_t n, int64_t sn, DevStatus *st, cudaStream_t s) {
    const int64_t ctas = (rn + (int64_t)C.P * (CP_NT - 1)) / CP_NT;
    const int g = (int)std::min<int64_t>(ctas, (int64_t)sm_count() * 64);
    auto run = [&](auto kern) {
        kern<<<g, CP_NT, 0, s>>>(src, d, R.idx, R.start, C.P, inS, Ss, S.start, C.near, C.nnear, thr, Rn, rnn, n, sn, rn,
                                 st);
    };
    if (d <= 2) run(cells_prune_kernel<2>);
    else if (d <= 4) run(cells_prune_kernel<4>);
    else if (d <= 8) run(cells_prune_kernel<8>);
    else run(cells_prune_kernel<16>);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace kc
