// Blocked Floyd-Warshall in the (min, +) semiring, for the component tables APSP(C)
// (Algorithm 1, per-component APSP) and for the boundary graph (Algorithm 1, APSP of BG).
//
// The paper computes APSP(C) with the GPU algorithm of its reference [ipdps-apsp] and
// the boundary-graph rows with Dijkstra's algorithm; both are exact all-pairs distance
// computations, and here both are the three-phase blocked Floyd-Warshall of
// Venkataraman, Sahni and Mukhopadhyaya (J. Exp. Algorithmics 8, 2003).  For pivot block r:
//   phase 1: close the diagonal tile (r, r) with plain Floyd-Warshall, in shared memory;
//   phase 2: row tiles (r, J) <- D*(r, r) (x) D(r, J)   [(x) = min-plus product]
//   phase 3: tiles (I, J), I, J != r <- min(D(I, J), D(I, r) (x) D(r, J)).
// Every matrix here is symmetric (undirected graphs; a + b = b + a and min is
// order-free, so float sums keep the symmetry exactly), so phase 2 writes each row tile
// also transposed into the column tile (J, r), and phase 3 reads the column panel
// D(I, r) as the transpose of the row tile D(r, I).  Both panels of phase 3 are then
// row-major rows of the pivot block, staged into shared memory with cp.async.
//
// Arithmetic: int32 (add, min) or float32 (add, three-input min over two k steps).
#include <cuda_runtime.h>

#include <string.h>

#include <algorithm>

#include <type_traits>
#include <vector>

#include "common.cuh"
#include "fw_tile.cuh"
#include "order.h"

namespace spq {

namespace {

// ---------------- phase 1: closure of the diagonal tile ----------------
template <typename T>
__global__ void __launch_bounds__(NTH) k_phase1(T* __restrict__ base, const MatDesc* __restrict__ descs,
                                                int32_t nmat, int32_t r, const int32_t* __restrict__ sel) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T(*S)[T_] = reinterpret_cast<T(*)[T_]>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int32_t mi = blockIdx.y; mi < nmat; mi += gridDim.y) {
        const MatDesc d = descs[sel ? sel[mi] : mi];
        const int64_t n = d.n;
        const int32_t R = (int32_t)((n + T_ - 1) / T_);
        if (r >= R) continue;
        T* M = base + d.off;
        const int64_t o = (int64_t)r * T_;
        for (int idx = tid; idx < T_ * T_ / 4; idx += NTH) {
            int i = idx >> 5, c4 = idx & 31;
            int64_t gr = o + i, gc = o + c4 * 4;
            int4 v = (gr < n && gc < n) ? *reinterpret_cast<const int4*>(M + gr * n + gc) : inf4<T>();
            *reinterpret_cast<int4*>(&S[i][c4 * 4]) = v;
        }
        __syncthreads();
        T acc[8][8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = S[own(ty, i)][own(tx, j)];
        const int K = (int)((n - o) < T_ ? (n - o) : T_);
        int k = 0;
        if constexpr (std::is_same<T, float>::value) {
            // two pivot steps per barrier: row k + 1 after step k is formed on the fly,
            // min(D(k+1, x), D(k+1, k) + D(k, x)), and both steps fold into one
            // three-input min; the owners then publish rows k + 2 and k + 3
            for (; k + 1 < K; k += 2) {
                float a0[8], b0[8], a1[8], b1[8];
                const float4 p0 = *reinterpret_cast<const float4*>(&S[k][ty * 4]);
                const float4 p1 = *reinterpret_cast<const float4*>(&S[k][64 + ty * 4]);
                const float4 q0 = *reinterpret_cast<const float4*>(&S[k][tx * 4]);
                const float4 q1 = *reinterpret_cast<const float4*>(&S[k][64 + tx * 4]);
                const float4 u0 = *reinterpret_cast<const float4*>(&S[k + 1][ty * 4]);
                const float4 u1 = *reinterpret_cast<const float4*>(&S[k + 1][64 + ty * 4]);
                const float4 v0 = *reinterpret_cast<const float4*>(&S[k + 1][tx * 4]);
                const float4 v1 = *reinterpret_cast<const float4*>(&S[k + 1][64 + tx * 4]);
                const float skk = S[k][k + 1];
                const float pa[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
                const float qa[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
                const float ua[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
                const float va[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    a0[i] = pa[i];
                    b0[i] = qa[i];
                    a1[i] = fminf(ua[i], skk + pa[i]);
                    b1[i] = fminf(va[i], skk + qa[i]);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = fmin3(acc[i][j], a0[i] + b0[j], a1[i] + b1[j]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = own(ty, i);
                    if (row == k + 2 || row == k + 3) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) S[row][own(tx, j)] = acc[i][j];
                    }
                }
                __syncthreads();
            }
        }
#pragma unroll 1
        for (; k < K; ++k) {
            // row k of S is current: by symmetry it is also column k
            T a[8], b[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                a[i] = S[k][own(ty, i)];
                b[i] = S[k][own(tx, i)];
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = MP<T>::upd1(acc[i][j], a[i], b[j]);
            const int kn = k + 1;
            if (kn < K) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (own(ty, i) == kn) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) S[kn][own(tx, j)] = acc[i][j];
                    }
            }
            __syncthreads();
        }
        store_c<T>(acc, M, n, o, o, tx, ty);
        __syncthreads();
    }
}

// ---------------- phase 2: pivot row tiles (and their transposes) ----------------
template <typename T>
__global__ void __launch_bounds__(NTH, SPQ_FW_MIN_CTAS) k_phase2(T* __restrict__ base, const MatDesc* __restrict__ descs,
                                                   int32_t nmat, int32_t r, uint32_t* __restrict__ row_finite,
                                                   int32_t flag_stride, const int32_t* __restrict__ sel,
                                                   int32_t trail = 0, uint32_t* __restrict__ kmask = nullptr,
                                                   int32_t kstride = 0) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T>& sm = *reinterpret_cast<PanelSmem<T>*>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int32_t mi = blockIdx.y; mi < nmat; mi += gridDim.y) {
        const MatDesc d = descs[sel ? sel[mi] : mi];
        const int64_t n = d.n;
        const int32_t R = (int32_t)((n + T_ - 1) / T_);
        // (elimination form: the row tiles right of the pivot only)
        const int32_t J = trail ? r + 1 + (int32_t)blockIdx.x : (int32_t)blockIdx.x + ((int32_t)blockIdx.x >= r ? 1 : 0);
        if (r >= R || J >= R) continue;
        T* M = base + d.off;
        const int64_t o = (int64_t)r * T_, cj = (int64_t)J * T_;
        T acc[8][8];
        load_c<T>(acc, M, n, o, cj, tx, ty);
        // An all-infinite row tile stays all-infinite (D*(r,r) (x) inf = inf), and so
        // does its transpose: nothing to compute or store.
        bool fin = false;
        const T inf = Inf<T>::value();
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) fin |= acc[i][j] < inf;
        if (!__syncthreads_or(fin)) continue;
        if (kmask) {  // (as in k_phase2_cand: chunk skipping, then the row mask for phase 3)
            __shared__ uint32_t rm[4];
            tile_row_mask<T>(acc, rm, tid, tx, ty);
            uint32_t cm = 0u;
#pragma unroll
            for (int c = 0; c < NCHUNK; ++c) cm |= rm[c] ? (1u << c) : 0u;
            minplus_panels_masked<T>(acc, M, n, o, o, cj, sm, tid, tx, ty, cm);
            tile_row_mask<T>(acc, rm, tid, tx, ty);
            if (tid < 4) kmask[(int64_t)mi * kstride + (int64_t)J * 4 + tid] = rm[tid];
        } else {
            minplus_panels<T>(acc, M, n, o, o, cj, sm, tid, tx, ty);
        }
        store_c<T>(acc, M, n, o, cj, tx, ty);
        store_c_transposed<T>(acc, M, n, o, cj, tx, ty);
        if (row_finite && tid == 0) row_finite[(int64_t)mi * flag_stride + J] = 1u;
    }
}

// Ordered list of the marked tiles J in [lo, hi) of one flag row: out[0] = count,
// out[1..] = J ascending.  Whole block; ends with a barrier.
__device__ void compact_row(const uint32_t* __restrict__ f, int32_t lo, int32_t hi, uint32_t* __restrict__ out) {
    __shared__ uint32_t cnt;
    __shared__ uint32_t wsum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    for (int32_t base = lo; base < hi; base += blockDim.x) {
        const int32_t J = base + threadIdx.x;
        const bool take = J < hi && __ldcg(f + J) != 0u;
        const unsigned ballot = __ballot_sync(0xffffffffu, take);
        if (lane == 0) wsum[warp] = __popc(ballot);
        __syncthreads();
        uint32_t off = cnt;
        for (int w = 0; w < warp; ++w) off += wsum[w];
        if (take) out[1 + off + __popc(ballot & ((1u << lane) - 1u))] = (uint32_t)J;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t tot = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += wsum[w];
            cnt += tot;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = cnt;
    __syncthreads();
}

// Upper-triangle task t (0 <= t < c(c+1)/2) -> pair (x, y), 0 <= x <= y < c, row-major.
// (float estimate of the row, then exact integer correction; c < 2^16 tiles.)
__device__ __forceinline__ void tri_pair(int64_t t, int64_t c, int64_t& x, int64_t& y) {
    const int32_t ti = (int32_t)t, ci = (int32_t)c;
    const float b = 2.0f * (float)ci + 1.0f;
    int32_t xx = (int32_t)((b - sqrtf(fmaxf(b * b - 8.0f * (float)ti, 0.0f))) * 0.5f);
    xx = xx < 0 ? 0 : (xx > ci - 1 ? ci - 1 : xx);
    while (xx > 0 && xx * ci - xx * (xx - 1) / 2 > ti) --xx;
    while (xx + 1 < ci && (xx + 1) * ci - (xx + 1) * xx / 2 <= ti) ++xx;
    x = xx;
    y = xx + (ti - (xx * ci - xx * (xx - 1) / 2));
}

// Phase-3 update of tile (I, J), I <= J, and, by symmetry, of (J, I) = (I, J)^T.
template <typename T>
__device__ __forceinline__ void phase3_tile(T* __restrict__ M, int64_t n, int64_t o, int64_t I, int64_t J,
                                            PanelSmem<T>& sm, int tid, int tx, int ty) {
    const int64_t ci = I * T_, cj = J * T_;
    T acc[8][8];
    load_c<T>(acc, M, n, ci, cj, tx, ty);
    minplus_panels<T>(acc, M, n, o, ci, cj, sm, tid, tx, ty);
    store_c<T>(acc, M, n, ci, cj, tx, ty);
    if (I != J) store_c_transposed<T>(acc, M, n, ci, cj, tx, ty);
}

// ---------------- phase 3 over the matrices active in round r ----------------
// sel[0..nsel) = matrices with more than r + 1 tile rows; p3off[0..nsel] = exclusive
// prefix of their task counts Rm(Rm + 1)/2 (Rm = tiles per side minus the pivot).
template <typename T>
__global__ void __launch_bounds__(NTH, SPQ_FW_MIN_CTAS) k_phase3_sel(T* __restrict__ base,
                                                                     const MatDesc* __restrict__ descs,
                                                                     const int32_t* __restrict__ sel, int32_t nsel,
                                                                     const int64_t* __restrict__ p3off, int32_t r) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T>& sm = *reinterpret_cast<PanelSmem<T>*>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t total = p3off[nsel];
    for (int64_t t = blockIdx.x; t < total; t += gridDim.x) {
        int32_t lo = 0, hi = nsel;
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if (p3off[mid] <= t) lo = mid; else hi = mid;
        }
        const MatDesc d = descs[sel[lo]];
        const int64_t Rm = (d.n + T_ - 1) / T_ - 1;
        int64_t I, J;
        tri_pair(t - p3off[lo], Rm, I, J);
        I += (I >= r);
        J += (J >= r);
        phase3_tile<T>(base + d.off, d.n, (int64_t)r * T_, I, J, sm, tid, tx, ty);
    }
}

// ---------------- phase 3, single large matrix: persistent over a tile list ----------------
// list[0] = count c, list[1..c] = ascending tile indices J != r whose row tile (r, J)
// holds a finite entry; every (I, J) in list x list is updated, the pairs I < J once
// for both triangles.  Tiles outside list x list keep their values: their pivot panel
// is entirely infinite, so min(D, inf + x) = D.
template <typename T>
__global__ void __launch_bounds__(NTH, SPQ_FW_MIN_CTAS) k_phase3_list(T* __restrict__ M, int64_t n, int32_t r,
                                                                      const uint32_t* __restrict__ list) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T>& sm = *reinterpret_cast<PanelSmem<T>*>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t c = list[0];
    for (int64_t t = blockIdx.x; t < c * (c + 1) / 2; t += gridDim.x) {
        int64_t x, y;
        tri_pair(t, c, x, y);
        phase3_tile<T>(M, n, (int64_t)r * T_, list[1 + x], list[1 + y], sm, tid, tx, ty);
    }
}

// Build the tile list of round r from the flags phase 2 set (and clear the flags).
// Also accumulates the number of phase-3 tiles into tiles[0] and of phase-2 tiles with a
// finite entry (the ones phase 2 computed) into tiles[1].
__global__ void k_compact(uint32_t* __restrict__ flags, int32_t R, int32_t r, uint32_t* __restrict__ list,
                          unsigned long long* __restrict__ tiles) {
    __shared__ uint32_t cnt;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    for (int32_t base = 0; base < R; base += blockDim.x) {
        int32_t J = base + threadIdx.x;
        bool take = J < R && J != r && flags[J] != 0u;
        unsigned ballot = __ballot_sync(0xffffffffu, take);
        // ordered compaction: warp prefix, then warps in order
        __shared__ uint32_t wsum[32];
        int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (lane == 0) wsum[warp] = __popc(ballot);
        __syncthreads();
        uint32_t off = cnt;
        for (int w = 0; w < warp; ++w) off += wsum[w];
        if (take) list[1 + off + __popc(ballot & ((1u << lane) - 1u))] = (uint32_t)J;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t tot = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += wsum[w];
            cnt += tot;
        }
        __syncthreads();
    }
    for (int32_t J = threadIdx.x; J < R; J += blockDim.x) flags[J] = 0u;
    if (threadIdx.x == 0) {
        list[0] = cnt;
        tiles[0] += (unsigned long long)cnt * (cnt + 1) / 2;  // phase-3 tiles of this round
        tiles[1] += (unsigned long long)cnt;                  // phase-2 tiles computed (finite)
    }
}

// ---------------- many matrices with infinite-panel skipping ----------------
// Per matrix mi (one CTA each): compact the flags of round r into the list at
// lists[mi * lstride] (count, then tile indices) and write the matrix's phase-3 task
// count c(c+1)/2 into offs[mi] (offs is scanned to task offsets afterwards).
__global__ void k_compact_many(uint32_t* __restrict__ flags, int32_t fstride, const MatDesc* __restrict__ descs,
                               int32_t nmat, int32_t r, uint32_t* __restrict__ lists, int32_t lstride,
                               uint32_t* __restrict__ offs, unsigned long long* __restrict__ tiles) {
    __shared__ uint32_t cnt;
    __shared__ uint32_t wsum[32];
    const int32_t mi = blockIdx.x;
    if (mi >= nmat) return;
    const int32_t R = (descs[mi].n + T_ - 1) / T_;
    uint32_t* f = flags + (int64_t)mi * fstride;
    uint32_t* list = lists + (int64_t)mi * lstride;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int32_t base = 0; base < R && r < R; base += blockDim.x) {
        const int32_t J = base + threadIdx.x;
        const bool take = J < R && J != r && f[J] != 0u;
        const unsigned ballot = __ballot_sync(0xffffffffu, take);
        if (lane == 0) wsum[warp] = __popc(ballot);
        __syncthreads();
        uint32_t off = cnt;
        for (int w = 0; w < warp; ++w) off += wsum[w];
        if (take) list[1 + off + __popc(ballot & ((1u << lane) - 1u))] = (uint32_t)J;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t tot = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += wsum[w];
            cnt += tot;
        }
        __syncthreads();
    }
    for (int32_t J = threadIdx.x; J < R; J += blockDim.x) f[J] = 0u;
    if (threadIdx.x == 0) {
        const uint32_t c = r < R ? cnt : 0u;
        list[0] = c;
        offs[mi] = c * (c + 1) / 2;
        atomicAdd(&tiles[0], (unsigned long long)c * (c + 1) / 2);
        atomicAdd(&tiles[1], (unsigned long long)c);
    }
}

// Phase 3 over the task lists of every matrix: offs[0..nmat] holds the exclusive task
// offsets (offs[nmat] = total); task t belongs to the matrix whose range holds it.
template <typename T>
__global__ void __launch_bounds__(NTH, SPQ_FW_MIN_CTAS) k_phase3_many(T* __restrict__ base,
                                                                      const MatDesc* __restrict__ descs, int32_t nmat,
                                                                      int32_t r, const uint32_t* __restrict__ lists,
                                                                      int32_t lstride,
                                                                      const uint32_t* __restrict__ offs,
                                                                      const uint32_t* __restrict__ kmask = nullptr,
                                                                      int32_t kstride = 0) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T>& sm = *reinterpret_cast<PanelSmem<T>*>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t total = offs[nmat];
    const int64_t o = (int64_t)r * T_;
    for (int64_t t = blockIdx.x; t < total; t += gridDim.x) {
        int32_t lo = 0, hi = nmat;  // largest mi with offs[mi] <= t
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if ((int64_t)offs[mid] <= t) lo = mid; else hi = mid;
        }
        const MatDesc d = descs[lo];
        const uint32_t* list = lists + (int64_t)lo * lstride;
        int64_t x, y;
        tri_pair(t - (int64_t)offs[lo], (int64_t)list[0], x, y);
        const int64_t I = list[1 + x], J = list[1 + y];
        if (!kmask) {
            phase3_tile<T>(base + d.off, d.n, o, I, J, sm, tid, tx, ty);
            continue;
        }
        // only the chunks of pivot rows finite in both row tiles (masks set by k_phase2)
        const uint32_t* km = kmask + (int64_t)lo * kstride;
        uint32_t cm = 0u;
#pragma unroll
        for (int q = 0; q < NCHUNK; ++q) cm |= (km[I * 4 + q] & km[J * 4 + q]) ? (1u << q) : 0u;
        T* M = base + d.off;
        const int64_t ci = I * T_, cj = J * T_;
        T acc[8][8];
        load_c<T>(acc, M, d.n, ci, cj, tx, ty);
        minplus_panels_masked<T>(acc, M, d.n, o, ci, cj, sm, tid, tx, ty, cm);
        store_c<T>(acc, M, d.n, ci, cj, tx, ty);
        if (I != J) store_c_transposed<T>(acc, M, d.n, ci, cj, tx, ty);
    }
}

// ---------------- elimination form (forward rounds) ----------------
// A step holds one round of every run of rounds that is active in it, of one matrix or of
// many (ents[o ..], one per blockIdx.y): runs do not depend on one another and touch
// disjoint tiles except those with both indices >= shared_from, which they update with
// atomicMin.  Three launches a step: phase 1, phase 2 over the candidates of the round's row
// with the compaction in each run's last CTA, phase 3 over its list.  (One stream per run
// took three launches a round of every run: on 2^20 vertices 3,000 launches and as many
// hardware queues as runs, on 2^16 vertices 18.0 of 30 ms serialised device time in rounds of
// a few tiles.)  What bounds a step of few tiles is the time of one tile on one CTA, so
// tiles are split into column strips where a step's tiles would leave CTAs idle.
template <typename T>
struct ElimEnt {
    T* M;
    int64_t N;
    uint32_t* rowflags;  // R x R marks (see ElimScratch)
    uint32_t* scratch;   // of the run
    int32_t r, R, shared_from, first;  // the round; first: the first of its run
};

// A run's scratch.  list / cand: count, then ascending tile indices J > r: the finite row
// tiles of round r (phase 3 updates list x list), the marked tiles of row r (phase 2's
// candidates).  kmask: 4 words per tile J, the finite rows of row tile (r, J) after phase 2
// (phase 3 multiplies only the 32-row chunks finite in both panels); kacc: the same while
// phase 2's CTAs collect it, zero otherwise.
// Marks: 1 a tile that may hold a finite entry, 2 one marked in this round, whose cells are
// not initialised yet (phase 3 starts it from infinity; 1 from the next compaction on).
struct ElimScratch {
    uint32_t *list, *cand, *counter, *kmask, *kacc;
    unsigned long long* tiles;  // phase-3 tiles, finite phase-2 tiles
    __device__ ElimScratch(uint32_t* p, int32_t R)
        : list(p),
          cand(p + R + 2),
          counter(p + 2 * R + 8),
          kmask(p + ((2 * R + 13) & ~3)),  // (16-byte words; the run's scratch is 16-byte aligned)
          kacc(kmask + 4 * R),
          tiles(reinterpret_cast<unsigned long long*>(p + 2 * R + 4)) {}
    static int64_t words(int32_t R) { return 10 * (int64_t)R + 13; }
};

// Phase 1: closure of the diagonal tile, 1,024 threads, each owning a 4 x 4 block (rows
// 4ty.., columns 4tx..); two pivot steps per barrier as in k_phase1, the sums two at a time
// by packed adds.  blockIdx.x = 1: the candidates of a run's first round, meanwhile.
template <typename T>
__global__ void __launch_bounds__(1024, 1) k_elim_phase1(const ElimEnt<T>* __restrict__ ents) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ElimEnt<T> en = ents[blockIdx.y];
    if (blockIdx.x == 1) {
        if (en.first)
            compact_row(en.rowflags + (int64_t)en.r * en.R, en.r + 1, en.R, ElimScratch(en.scratch, en.R).cand);
        return;
    }
    T* __restrict__ M = en.M;
    const int64_t n = en.N;
    T(*S)[T_] = reinterpret_cast<T(*)[T_]>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int64_t o = (int64_t)en.r * T_;
    for (int idx = tid; idx < T_ * T_ / 4; idx += 1024) {
        const int i = idx >> 5, c4 = idx & 31;
        const int64_t gr = o + i, gc = o + c4 * 4;
        int4 v = (gr < n && gc < n) ? *reinterpret_cast<const int4*>(M + gr * n + gc) : inf4<T>();
        *reinterpret_cast<int4*>(&S[i][c4 * 4]) = v;
    }
    __syncthreads();
    auto row4 = [&](int k, int at, T (&v)[4]) {
        const int4 x = *reinterpret_cast<const int4*>(&S[k][at]);
        const int y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = *reinterpret_cast<const T*>(&y[i]);
    };
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) row4(4 * ty + i, 4 * tx, acc[i]);
    const int K = (int)((n - o) < T_ ? (n - o) : T_);
    int k = 0;
    // rows k and k + 1 are current (by symmetry also columns k and k + 1); row k + 1
    // after step k is min(D(k+1, x), D(k+1, k) + D(k, x)), formed on the fly
    for (; k + 1 < K; k += 2) {
        T a0[4], b0[4], a1[4], b1[4];
        row4(k, 4 * ty, a0);
        row4(k, 4 * tx, b0);
        row4(k + 1, 4 * ty, a1);
        row4(k + 1, 4 * tx, b1);
        const T skk = S[k][k + 1];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            a1[i] = MP<T>::upd1(a1[i], skk, a0[i]);
            b1[i] = MP<T>::upd1(b1[i], skk, b0[i]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (std::is_same<T, float>::value) {
                const float2 x0 = make_float2(a0[i], a0[i]), x1 = make_float2(a1[i], a1[i]);
#pragma unroll
                for (int j = 0; j < 4; j += 2) {
                    const float2 s0 = __fadd2_rn(x0, make_float2(b0[j], b0[j + 1]));
                    const float2 s1 = __fadd2_rn(x1, make_float2(b1[j], b1[j + 1]));
                    acc[i][j] = fmin3(acc[i][j], s0.x, s1.x);
                    acc[i][j + 1] = fmin3(acc[i][j + 1], s0.y, s1.y);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = MP<T>::upd2(acc[i][j], a0[i], b0[j], a1[i], b1[j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = 4 * ty + i;
            if (row == k + 2 || row == k + 3)
                *reinterpret_cast<int4*>(&S[row][4 * tx]) = as_int4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        }
        __syncthreads();
    }
    for (; k < K; ++k) {
        T a[4], b[4];
        row4(k, 4 * ty, a);
        row4(k, 4 * tx, b);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = MP<T>::upd1(acc[i][j], a[i], b[j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (4 * ty + i == k + 1)
                *reinterpret_cast<int4*>(&S[k + 1][4 * tx]) = as_int4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t gr = o + 4 * ty + i, gc = o + 4 * tx;
        if (gr < n && gc < n)
            *reinterpret_cast<int4*>(M + gr * n + gc) = as_int4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
}

// A step's tiles are split into strips when fewer than this many would be at work: one per SM
// of a GB300 (a strip takes a quarter of a tile's time, so up to there the split shortens the step).
constexpr int64_t kStripTiles = 152;

// Phase 2: the candidate row tiles (r, J) <- D*(r, r) (x) D(r, J) and their transposes.  A
// candidate that is all infinite stays so and is unmarked.  The last CTA of the run to finish
// (counted; the counter is left at 0) does the compaction.
template <typename T>
__global__ void __launch_bounds__(NTH, SPQ_FW_MIN_CTAS) k_elim_phase2(const ElimEnt<T>* __restrict__ ents,
                                                                      int32_t skip_inf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T>& sm = *reinterpret_cast<PanelSmem<T>*>(smem_raw);
    __shared__ uint32_t rm[4];
    const ElimEnt<T> en = ents[blockIdx.y];
    const ElimScratch sc(en.scratch, en.R);
    T* __restrict__ M = en.M;
    const int64_t n = en.N;
    const int32_t r = en.r, R = en.R;
    const int tid = threadIdx.x;
    const int64_t o = (int64_t)r * T_;
    const uint32_t c = sc.cand[0];
    // the B panel is the tile's own rows: the chunks of rows that are all infinite are
    // skipped; then the updated tile's finite rows are recorded for phase 3
    if ((int64_t)c * gridDim.y <= kStripTiles) {
        const int sx = tid & 7, sy = tid >> 3;
        for (uint32_t ci = blockIdx.x; ci < c * kStrips; ci += gridDim.x) {
            const int32_t J = (int32_t)sc.cand[1 + ci / kStrips];
            const int64_t cs = (int64_t)J * T_ + (ci % kStrips) * SW;
            T acc[4][4];
            load_strip<T>(acc, M, n, o, cs, sx, sy);
            strip_row_mask<T>(acc, rm, tid, sy);
            uint32_t cm = 0u;
#pragma unroll
            for (int q = 0; q < NCHUNK; ++q) cm |= rm[q] ? (1u << q) : 0u;
            if (cm == 0u) continue;
            minplus_strip_masked<T>(acc, M, n, o, o, cs, sm, tid, sx, sy, cm);
            strip_row_mask<T>(acc, rm, tid, sy);
            if (tid < 4 && rm[tid]) atomicOr(&sc.kacc[(int64_t)J * 4 + tid], rm[tid]);
            store_strip<T>(acc, M, n, o, cs, sx, sy);
            store_strip_transposed<T>(acc, M, n, o, cs, sx, sy);
        }
    } else {
        const int tx = tid & 15, ty = tid >> 4;
        for (uint32_t ci = blockIdx.x; ci < c; ci += gridDim.x) {
            const int32_t J = (int32_t)sc.cand[1 + ci];
            const int64_t cj = (int64_t)J * T_;
            T acc[8][8];
            load_c<T>(acc, M, n, o, cj, tx, ty);
            tile_row_mask<T>(acc, rm, tid, tx, ty);
            uint32_t cm = 0u;
#pragma unroll
            for (int q = 0; q < NCHUNK; ++q) cm |= rm[q] ? (1u << q) : 0u;
            if (cm == 0u) continue;
            minplus_panels_masked<T>(acc, M, n, o, o, cj, sm, tid, tx, ty, cm);
            tile_row_mask<T>(acc, rm, tid, tx, ty);
            if (tid < 4) sc.kacc[(int64_t)J * 4 + tid] = rm[tid];
            store_c<T>(acc, M, n, o, cj, tx, ty);
            store_c_transposed<T>(acc, M, n, o, cj, tx, ty);
        }
    }
    __shared__ uint32_t last;
    __threadfence();  // (this CTA's tiles and masks, before its ticket)
    __syncthreads();
    if (tid == 0) last = atomicAdd(sc.counter, 1u) == gridDim.x - 1u ? 1u : 0u;
    __syncthreads();
    if (!last) return;
    __threadfence();  // (every other CTA's writes, after their tickets)
    // the previous round's new tiles are initialised now
    const uint32_t pc = sc.list[0];
    for (uint32_t t = tid; t < pc * pc; t += blockDim.x) {
        const uint32_t x = t / pc, y = t % pc;
        if (y > x) {
            uint32_t* f = en.rowflags + (int64_t)sc.list[1 + x] * R + sc.list[1 + y];
            if (__ldcg(f) == 2u) *f = 1u;
        }
    }
    __syncthreads();  // (a tile of row r marked there may be unmarked here)
    for (uint32_t ci = tid; ci < c; ci += blockDim.x) {
        const int64_t J = sc.cand[1 + ci];
        uint4* ka = reinterpret_cast<uint4*>(sc.kacc + J * 4);
        uint4* km = reinterpret_cast<uint4*>(sc.kmask + J * 4);
        const uint4 m = __ldcg(ka);
        *km = m;
        *ka = make_uint4(0u, 0u, 0u, 0u);
        if (!(m.x | m.y | m.z | m.w)) en.rowflags[(int64_t)r * R + J] = 0u;
    }
    __syncthreads();
    if (!skip_inf)  // (no skipping: every tile of the row takes part)
        for (int32_t J = r + 1 + tid; J < R; J += blockDim.x) en.rowflags[(int64_t)r * R + J] = 0xffffffffu;
    __syncthreads();
    compact_row(en.rowflags + (int64_t)r * R, r + 1, R, sc.list);
    const uint32_t lc = sc.list[0];
    for (uint32_t t = tid; t < lc * lc; t += blockDim.x) {
        const uint32_t x = t / lc, y = t % lc;
        if (y > x) {
            uint32_t* f = en.rowflags + (int64_t)sc.list[1 + x] * R + sc.list[1 + y];
            if (__ldcg(f) == 0u) *f = 2u;
        }
    }
    if (tid == 0) {
        sc.tiles[0] += (unsigned long long)lc * (lc + 1) / 2;
        sc.tiles[1] += (unsigned long long)lc;
        *sc.counter = 0u;
    }
    __syncthreads();
    if (r + 1 < R) compact_row(en.rowflags + (int64_t)(r + 1) * R, r + 2, R, sc.cand);
}

// Phase 3: tiles (I, J), I <= J of the run's list, <- min(D(I, J), D(r, I)^T (x) D(r, J)).
template <typename T>
__global__ void __launch_bounds__(NTH, SPQ_FW_MIN_CTAS) k_elim_phase3(const ElimEnt<T>* __restrict__ ents,
                                                                      int32_t skip_inf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PanelSmem<T>& sm = *reinterpret_cast<PanelSmem<T>*>(smem_raw);
    const ElimEnt<T> en = ents[blockIdx.y];
    const ElimScratch sc(en.scratch, en.R);
    T* __restrict__ M = en.M;
    const int64_t n = en.N;
    const int tid = threadIdx.x;
    const int64_t c = sc.list[0], tiles = c * (c + 1) / 2;
    const int64_t o = (int64_t)en.r * T_;
    const bool strips = tiles * gridDim.y <= kStripTiles;
    for (int64_t t = blockIdx.x; t < (strips ? tiles * kStrips : tiles); t += gridDim.x) {
        int64_t x, y;
        tri_pair(strips ? t / kStrips : t, c, x, y);
        const int64_t I = sc.list[1 + x], J = sc.list[1 + y];
        uint32_t cm = (1u << NCHUNK) - 1u;
        if (skip_inf) {  // only the chunks of pivot rows finite in both panels
            cm = 0u;
#pragma unroll
            for (int q = 0; q < NCHUNK; ++q) cm |= (sc.kmask[I * 4 + q] & sc.kmask[J * 4 + q]) ? (1u << q) : 0u;
        }
        const bool fresh = I < J && en.rowflags[I * en.R + J] == 2u;
        const bool shared = !fresh && I >= en.shared_from;
        const int64_t ci = I * T_, cj = J * T_;
        if (strips) {
            const int sx = tid & 7, sy = tid >> 3;
            const int64_t cs = cj + (t % kStrips) * SW;
            T acc[4][4];
            if (fresh) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = Inf<T>::value();
            } else {
                load_strip<T>(acc, M, n, ci, cs, sx, sy);
            }
            minplus_strip_masked<T>(acc, M, n, o, ci, cs, sm, tid, sx, sy, cm);
            if (shared) {
                store_strip_min<T>(acc, M, n, ci, cs, sx, sy, false);
                if (I != J) store_strip_min<T>(acc, M, n, ci, cs, sx, sy, true);
            } else {
                store_strip<T>(acc, M, n, ci, cs, sx, sy);
                if (I != J) store_strip_transposed<T>(acc, M, n, ci, cs, sx, sy);
            }
        } else {
            const int tx = tid & 15, ty = tid >> 4;
            T acc[8][8];
            if (fresh) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = Inf<T>::value();
            } else {
                load_c<T>(acc, M, n, ci, cj, tx, ty);
            }
            minplus_panels_masked<T>(acc, M, n, o, ci, cj, sm, tid, tx, ty, cm);
            if (shared) {
                store_c_min<T>(acc, M, n, ci, cj, tx, ty);
                if (I != J) store_c_transposed_min<T>(acc, M, n, ci, cj, tx, ty);
            } else {
                store_c<T>(acc, M, n, ci, cj, tx, ty);
                if (I != J) store_c_transposed<T>(acc, M, n, ci, cj, tx, ty);
            }
        }
    }
}

// Sum of the runs' tile counters (run i's at base + off[i]).
__global__ void k_elim_tiles(const uint32_t* __restrict__ base, const int64_t* __restrict__ off, int32_t nrun,
                             unsigned long long* __restrict__ out) {
    unsigned long long a = 0, b = 0;
    for (int32_t i = threadIdx.x; i < nrun; i += blockDim.x) {
        const unsigned long long* t = reinterpret_cast<const unsigned long long*>(base + off[i]);
        a += t[0];
        b += t[1];
    }
    atomicAdd(&out[0], a);
    atomicAdd(&out[1], b);
}

int g_sms = 0;
int sms() {
    if (g_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

template <typename T>
cudaError_t set_smem_attrs() {
    static bool done = false;
    if (done) return cudaSuccess;
    cudaError_t e;
    e = cudaFuncSetAttribute(k_phase1<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, T_ * T_ * (int)sizeof(T));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_elim_phase1<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, T_ * T_ * (int)sizeof(T));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_phase2<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PanelSmem<T>));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_phase3_list<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PanelSmem<T>));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_elim_phase2<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PanelSmem<T>));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_elim_phase3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PanelSmem<T>));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_phase3_many<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PanelSmem<T>));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_phase3_sel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PanelSmem<T>));
    if (e != cudaSuccess) return e;
    done = true;
    return cudaSuccess;
}

}  // namespace

// The forward rounds of every matrix (see common.cuh).
template <typename T>
cudaError_t elim_forward(const std::vector<ElimMat<T>>& mats, bool skip_inf, double* updates, FwProfile* prof,
                         cudaStream_t st, ElimPlan* keep) {
    if (updates) *updates = 0.0;
    cudaError_t e = set_smem_attrs<T>();
    if (e != cudaSuccess || mats.empty()) {
        if (keep) keep->ready = true;
        return e;
    }
    const size_t psm = sizeof(PanelSmem<T>);
    const bool replay = keep && keep->ready;
    ElimPlan local;
    ElimPlan& p = replay ? *keep : local;
    if (!replay) {
        // the runs of every matrix, each from the step after the last of its dependencies'
        struct Run {
            int32_t mat, lo, hi, shared_from, start;
            int64_t scratch;
        };
        std::vector<Run> runs;
        int64_t words = 0;
        int32_t nstep = 0;
        double diag = 0.0;
        for (size_t m = 0; m < mats.size(); ++m) {
            const int32_t R = (int32_t)((mats[m].N + T_ - 1) / T_);
            diag += R;
            std::vector<ElimTask> one(1);
            one[0].hi = one[0].shared_from = R;
            const std::vector<ElimTask>& tasks = mats[m].tasks && !mats[m].tasks->empty() ? *mats[m].tasks : one;
            const size_t base = runs.size();
            for (const ElimTask& tk : tasks) {
                int32_t start = 0;
                for (int32_t d : tk.deps) start = std::max(start, runs[base + d].start + runs[base + d].hi - runs[base + d].lo);
                runs.push_back(Run{(int32_t)m, tk.lo, tk.hi, tk.shared_from, start, words});
                words += round_up(ElimScratch::words(R), 4);
                nstep = std::max(nstep, start + tk.hi - tk.lo);
            }
        }
        std::vector<std::vector<ElimEnt<T>>> steps(nstep);
        const size_t o_off = ((size_t)words * 4 + 15) & ~(size_t)15, o_out = o_off + runs.size() * 8;
        size_t total = 0;
        for (const Run& ru : runs) total += (size_t)std::max(ru.hi - ru.lo, 0);
        const size_t o_ent = (o_out + 16 + 15) & ~(size_t)15;
        if ((e = scratch_alloc((void**)&p.mem, o_ent + total * sizeof(ElimEnt<T>), st)) != cudaSuccess) return e;
        std::vector<int64_t> off;
        for (const Run& ru : runs) {
            const ElimMat<T>& m = mats[ru.mat];
            const int32_t R = (int32_t)((m.N + T_ - 1) / T_);
            off.push_back(ru.scratch + 2 * R + 4);
            for (int32_t r = ru.lo; r < ru.hi; ++r)
                steps[ru.start + r - ru.lo].push_back(ElimEnt<T>{m.M, m.N, m.rowflags,
                                                                 reinterpret_cast<uint32_t*>(p.mem) + ru.scratch, r, R,
                                                                 ru.shared_from, r == ru.lo ? 1 : 0});
        }
        std::vector<ElimEnt<T>> ents;
        ents.reserve(total);
        for (const auto& s : steps) {
            int32_t most = 0;  // row tiles right of a pivot
            for (const ElimEnt<T>& x : s) most = std::max(most, x.R - 1 - x.r);
            p.steps.push_back(ElimPlan::Step{ents.size(), (int32_t)s.size(), most});
            ents.insert(ents.end(), s.begin(), s.end());
        }
        p.words = words;
        p.nrun = (int32_t)runs.size();
        p.o_off = o_off;
        p.o_out = o_out;
        p.o_ent = o_ent;
        p.diag = diag;
        if ((e = cudaMemcpyAsync(p.mem + o_off, off.data(), off.size() * 8, cudaMemcpyHostToDevice, st)) == cudaSuccess)
            e = cudaMemcpyAsync(p.mem + o_ent, ents.data(), ents.size() * sizeof(ElimEnt<T>), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) {
            p.release(st);
            return e;
        }
    }
    const ElimEnt<T>* d_ents = reinterpret_cast<const ElimEnt<T>*>(p.mem + p.o_ent);
    unsigned long long* out = reinterpret_cast<unsigned long long*>(p.mem + p.o_out);
    if ((e = cudaMemsetAsync(p.mem, 0, (size_t)p.words * 4, st)) == cudaSuccess) e = cudaMemsetAsync(out, 0, 16, st);
    std::vector<cudaEvent_t> evs;  // around every phase 3 (profiling only)
    if (prof && e == cudaSuccess) {
        evs.resize(2 * p.steps.size(), nullptr);
        for (auto& ev : evs)
            if (e == cudaSuccess) e = cudaEventCreate(&ev);
    }
    for (size_t i = 0; i < p.steps.size() && e == cudaSuccess; ++i) {
        const ElimPlan::Step& s = p.steps[i];
        const ElimEnt<T>* en = d_ents + s.first;
        // CTAs per run: two per SM side by side, or as many as its strips could use; a list
        // is much shorter than the row (about 10 tiles on planar boundary graphs)
        for (int32_t y0 = 0; y0 < s.count; y0 += 65535) {
            const unsigned gy = (unsigned)std::min(s.count - y0, 65535);
            const int64_t share = std::max<int64_t>(8, (4 * (int64_t)sms() + gy - 1) / gy);
            const unsigned g2 = (unsigned)std::min<int64_t>(std::max<int64_t>(1, (int64_t)kStrips * s.most), std::min<int64_t>(share, 2 * sms()));
            const unsigned g3 = (unsigned)std::min<int64_t>(2 * share, 2 * sms());
            k_elim_phase1<T><<<dim3(2, gy), 1024, T_ * T_ * sizeof(T), st>>>(en + y0);
            count_launches(1);
            if (s.most > 0) {
                k_elim_phase2<T><<<dim3(g2, gy), NTH, psm, st>>>(en + y0, skip_inf ? 1 : 0);
                if (!evs.empty() && y0 == 0) cudaEventRecord(evs[2 * i], st);
                k_elim_phase3<T><<<dim3(g3, gy), NTH, psm, st>>>(en + y0, skip_inf ? 1 : 0);
                count_launches(2);
            }
        }
        if (!evs.empty()) cudaEventRecord(evs[2 * i + 1], st);
        e = cudaGetLastError();
    }
    if (!replay && e == cudaSuccess) {
        k_elim_tiles<<<1, 256, 0, st>>>(reinterpret_cast<const uint32_t*>(p.mem),
                                        reinterpret_cast<const int64_t*>(p.mem + p.o_off), p.nrun, out);
        count_launches(1);
        unsigned long long htv[2] = {0, 0};
        e = cudaMemcpyAsync(htv, out, sizeof(htv), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        const double t3 = (double)T_ * T_ * T_;
        p.updates = ((double)htv[0] + (double)htv[1] + p.diag) * t3;  // phase 3, phase 2, phase 1 tiles
        if (prof) {
            prof->p3_ms = 0.0;
            prof->p3_launches = 0;
            for (size_t i = 0; e == cudaSuccess && i < p.steps.size(); ++i) {
                float t = 0.f;
                if (p.steps[i].most > 0 && cudaEventElapsedTime(&t, evs[2 * i], evs[2 * i + 1]) == cudaSuccess) {
                    prof->p3_ms += t;
                    prof->p3_launches += 1;
                }
            }
            prof->p3_updates = (double)htv[0] * t3;
        }
    }
    for (auto& ev : evs)
        if (ev) cudaEventDestroy(ev);
    if (updates) *updates = p.updates;
    if (!replay) {
        if (keep && e == cudaSuccess) {
            p.ready = true;
            *keep = std::move(p);
        } else {
            p.release(st);
        }
    }
    return e;
}

template <typename T>
cudaError_t fw_batched(T* base, const MatDesc* d_descs, const MatDesc* h_descs, int32_t nmat, int32_t max_n,
                       cudaStream_t st, int32_t** keep_buf) {
    if (nmat <= 0 || max_n <= 0) return cudaSuccess;
    cudaError_t e = set_smem_attrs<T>();
    if (e != cudaSuccess) return e;
    const int32_t R = (max_n + T_ - 1) / T_;
    // per round: the matrices still active (more than r tile rows), in one host buffer
    //   [sel_0 | p3off_0 (as two int32 words each) | sel_1 | ...]
    std::vector<int64_t> start(R + 1, 0);
    std::vector<int32_t> nsel(R, 0);
    std::vector<int32_t> buf;
    for (int32_t r = 0; r < R; ++r) {
        start[r] = (int64_t)buf.size();
        std::vector<int32_t> sel;
        for (int32_t m = 0; m < nmat; ++m)
            if ((h_descs[m].n + T_ - 1) / T_ > r) sel.push_back(m);
        nsel[r] = (int32_t)sel.size();
        buf.insert(buf.end(), sel.begin(), sel.end());
        if (buf.size() & 1) buf.push_back(0);  // 8-byte alignment of the offsets
        int64_t acc = 0;
        for (size_t i = 0; i <= sel.size(); ++i) {
            int32_t w2[2];
            memcpy(w2, &acc, 8);
            buf.push_back(w2[0]);
            buf.push_back(w2[1]);
            if (i < sel.size()) {
                const int64_t Rm = (h_descs[sel[i]].n + T_ - 1) / T_ - 1;
                acc += Rm * (Rm + 1) / 2;
            }
        }
    }
    int32_t* d_buf = keep_buf ? *keep_buf : nullptr;
    if (!d_buf) {
        e = scratch_alloc((void**)&d_buf, buf.size() * sizeof(int32_t), st);
        if (e != cudaSuccess) return e;
        e = cudaMemcpyAsync(d_buf, buf.data(), buf.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st);
        if (keep_buf) *keep_buf = d_buf;
    }
    const size_t psm = sizeof(PanelSmem<T>);
    const int p3_grid = sms() * 2;
    for (int32_t r = 0; r < R && e == cudaSuccess; ++r) {
        const int32_t ns = nsel[r];
        if (ns == 0) break;
        const int32_t* sel = d_buf + start[r];
        const int64_t* p3off = reinterpret_cast<const int64_t*>(d_buf + start[r] + ns + (ns & 1));
        const unsigned gy = (unsigned)(ns < 65535 ? ns : 65535);
        k_phase1<T><<<dim3(1, gy), NTH, T_ * T_ * sizeof(T), st>>>(base, d_descs, ns, r, sel);
        count_launches(1);
        if (R > 1) {
            k_phase2<T><<<dim3(R - 1, gy), NTH, psm, st>>>(base, d_descs, ns, r, nullptr, 0, sel);
            k_phase3_sel<T><<<p3_grid, NTH, psm, st>>>(base, d_descs, sel, ns, p3off, r);
            count_launches(2);
        }
        e = cudaGetLastError();
    }
    if (!keep_buf) cudaFreeAsync(d_buf, st);  // (the pageable upload above completed before it returned)
    return e;
}

int64_t fw_single_scratch_words(int64_t N) {
    int64_t R = (N + T_ - 1) / T_;
    return 2 * R + 8;  // flags[R], list[1 + R] (+1 pad), two tile counters (u64)
}

template <typename T>
cudaError_t fw_single(T* M, int64_t N, bool skip_inf, uint32_t* scratch, double* updates, FwProfile* prof,
                      cudaStream_t st) {
    if (updates) *updates = 0.0;
    if (N <= 0) return cudaSuccess;
    cudaError_t e = set_smem_attrs<T>();
    if (e != cudaSuccess) return e;
    const int32_t R = (int32_t)((N + T_ - 1) / T_);
    uint32_t* flags = scratch;
    uint32_t* list = scratch + R;
    unsigned long long* tiles = reinterpret_cast<unsigned long long*>(scratch + 2 * R + 2);
    e = cudaMemsetAsync(scratch, 0, fw_single_scratch_words(N) * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    MatDesc h{0, (int32_t)N, 0};
    MatDesc* dd = nullptr;
    e = scratch_alloc((void**)&dd, sizeof(MatDesc), st);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(dd, &h, sizeof(MatDesc), cudaMemcpyHostToDevice, st);
    const size_t psm = sizeof(PanelSmem<T>);
    const int p3_grid = sms() * 2;
    // optional per-launch timing of phase 3 (one event pair per round)
    std::vector<cudaEvent_t> evs;
    if (prof && R > 1) {
        evs.resize(2 * (size_t)R, nullptr);
        for (auto& ev : evs)
            if (e == cudaSuccess) e = cudaEventCreate(&ev);
    }
    for (int32_t r = 0; r < R && e == cudaSuccess; ++r) {
        k_phase1<T><<<dim3(1, 1), NTH, T_ * T_ * sizeof(T), st>>>(M, dd, 1, r, nullptr);
        count_launches(1);
        if (R > 1) {
            k_phase2<T><<<dim3(R - 1, 1), NTH, psm, st>>>(M, dd, 1, r, flags, 0, nullptr);
            if (!skip_inf) {
                // mark every tile: the compaction then lists all J != r
                cudaMemsetAsync(flags, 0xff, R * sizeof(uint32_t), st);
            }
            k_compact<<<1, 1024, 0, st>>>(flags, R, r, list, tiles);
            if (!evs.empty()) cudaEventRecord(evs[2 * r], st);
            k_phase3_list<T><<<p3_grid, NTH, psm, st>>>(M, N, r, list);
            if (!evs.empty()) cudaEventRecord(evs[2 * r + 1], st);
            count_launches(3);
        }
        e = cudaGetLastError();
    }
    unsigned long long htv[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(htv, tiles, sizeof(htv), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFreeAsync(dd, st);
    if (prof) {
        prof->p3_ms = 0.0;
        prof->p3_launches = 0;
        for (size_t r = 0; e == cudaSuccess && 2 * r + 1 < evs.size(); ++r) {
            float t = 0.f;
            if (cudaEventElapsedTime(&t, evs[2 * r], evs[2 * r + 1]) == cudaSuccess) {
                prof->p3_ms += t;
                prof->p3_launches += 1;
            }
        }
        prof->p3_updates = (double)htv[0] * (double)T_ * T_ * T_;
    }
    for (auto& ev : evs)
        if (ev) cudaEventDestroy(ev);
    if (updates) {
        double t3 = (double)T_ * T_ * T_;
        *updates = ((double)htv[0] + (double)htv[1] + (double)R) * t3;  // phase 3, phase 2, phase 1 tiles
    }
    return e;
}

int64_t fw_many_scratch_words(int32_t nmat, int32_t max_n) {
    const int64_t R = (max_n + T_ - 1) / T_;
    // flags, lists, offsets, (alignment), two u64 counters, row masks (4 words per tile)
    return (int64_t)nmat * R + (int64_t)nmat * (R + 1) + nmat + 1 + 1 + 4 + (int64_t)nmat * R * 4;
}

template <typename T>
cudaError_t fw_many_skip(T* base, const MatDesc* d_descs, int32_t nmat, int32_t max_n, uint32_t* scratch,
                         double* updates, cudaStream_t st, bool trail, bool stats) {
    if (updates && stats) *updates = 0.0;
    if (nmat <= 0 || max_n <= 0) return cudaSuccess;
    cudaError_t e = set_smem_attrs<T>();
    if (e != cudaSuccess) return e;
    const int32_t R = (max_n + T_ - 1) / T_;
    uint32_t* flags = scratch;
    uint32_t* lists = flags + (int64_t)nmat * R;
    uint32_t* offs = lists + (int64_t)nmat * (R + 1);
    int64_t toff = (int64_t)nmat * R + (int64_t)nmat * (R + 1) + nmat + 1;
    toff += toff & 1;  // 8-byte alignment of the counters
    unsigned long long* tiles = reinterpret_cast<unsigned long long*>(scratch + toff);
    uint32_t* kmask = scratch + toff + 4;  // per matrix R x 4 words
    const int32_t kstride = 4 * R;
    e = cudaMemsetAsync(scratch, 0, (size_t)(toff + 4) * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    const unsigned gy = (unsigned)(nmat < 65535 ? nmat : 65535);
    const size_t psm = sizeof(PanelSmem<T>);
    const int p3_grid = sms() * 2;
    for (int32_t r = 0; r < R && e == cudaSuccess; ++r) {
        k_phase1<T><<<dim3(1, gy), NTH, T_ * T_ * sizeof(T), st>>>(base, d_descs, nmat, r, nullptr);
        count_launches(1);
        if (R > 1 && (!trail || r + 1 < R)) {
            // (elimination form: the flags of the tiles left of r stay clear, so the lists
            //  and phase 3 hold only tiles right of / below the pivot block)
            // (row masks: phase 3 skips the pivot-row chunks infinite in either row tile)
            if (trail)
                k_phase2<T><<<dim3(R - 1 - r, gy), NTH, psm, st>>>(base, d_descs, nmat, r, flags, R, nullptr, 1,
                                                                    kmask, kstride);
            else
                k_phase2<T><<<dim3(R - 1, gy), NTH, psm, st>>>(base, d_descs, nmat, r, flags, R, nullptr, 0, kmask,
                                                                kstride);
            k_compact_many<<<nmat, 1024, 0, st>>>(flags, R, d_descs, nmat, r, lists, R + 1, offs, tiles);
            launch_scan_excl(offs, nmat + 1, st);
            k_phase3_many<T><<<p3_grid, NTH, psm, st>>>(base, d_descs, nmat, r, lists, R + 1, offs, kmask, kstride);
            count_launches(4);
        }
        e = cudaGetLastError();
    }
    if (!stats) return e;
    unsigned long long htv[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(htv, tiles, sizeof(htv), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    // phase-3 and phase-2 tiles; the caller adds the phase-1 (diagonal) tiles
    if (updates) *updates = ((double)htv[0] + (double)htv[1]) * (double)T_ * T_ * T_;
    return e;
}

template cudaError_t fw_many_skip<int32_t>(int32_t*, const MatDesc*, int32_t, int32_t, uint32_t*, double*,
                                           cudaStream_t, bool, bool);
template cudaError_t fw_many_skip<float>(float*, const MatDesc*, int32_t, int32_t, uint32_t*, double*, cudaStream_t,
                                         bool, bool);

template cudaError_t fw_batched<int32_t>(int32_t*, const MatDesc*, const MatDesc*, int32_t, int32_t, cudaStream_t,
                                         int32_t**);
template cudaError_t fw_batched<float>(float*, const MatDesc*, const MatDesc*, int32_t, int32_t, cudaStream_t,
                                       int32_t**);
template cudaError_t fw_single<int32_t>(int32_t*, int64_t, bool, uint32_t*, double*, FwProfile*, cudaStream_t);
template cudaError_t fw_single<float>(float*, int64_t, bool, uint32_t*, double*, FwProfile*, cudaStream_t);
template cudaError_t elim_forward<int32_t>(const std::vector<ElimMat<int32_t>>&, bool, double*, FwProfile*, cudaStream_t,
                                           ElimPlan*);
template cudaError_t elim_forward<float>(const std::vector<ElimMat<float>>&, bool, double*, FwProfile*, cudaStream_t,
                                         ElimPlan*);

}  // namespace spq
