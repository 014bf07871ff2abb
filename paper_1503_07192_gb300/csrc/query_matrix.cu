// Many-to-many distances: dist(s, w) for every source s and target w (row-major ns x nt).
//
// Algorithm 2 in two stages (its first loop depends on the source and the target's
// component only): for a source v1 in C1 and a target component C2,
//   t(b2) = min over b1 in B(C1) of dist_C1(v1, b1) + dist_BG(b1, b2)          (once)
// and then for every target v2 in C2
//   dist = min over b2 of t(b2) + dist_C2(b2, v2), and dist_C1(v1, v2) if C1 = C2,
// so a (source, target component) pair costs |B1||B2| updates once plus |B2| per target
// instead of |B1||B2| per pair.
//
// Stage 1 (k_matrix_t) is bound by the sources' rows of the boundary matrix (64 sources on
// 2^18 vertices: 1.2 GB): a warp per source and target component, four rows x four columns
// of loads in flight, t written once.  Stage 2 (k_matrix_out) is a min-plus matrix product
// per target component, (sources x |B2|) by (|B2| x targets): tiles of 64 sources x 128
// targets, both operands in rows along b2 staged by 16-byte asynchronous copies, so the
// targets' rows of APSP(C2) are read once per 64 sources and in whole lines (one target per
// lane, walking its own row, read a sector per value: 1.39 ms for 64 x 2^18 where the two
// stages take 0.4); the tile goes out through shared memory, so that runs of neighbouring
// targets are written together.  The targets are sorted by component; the tiles, and the
// components that have targets (the only ones t is computed and has columns for: 20,000
// sources x 1 target 2.4 ms with columns for all 256 components, 512 sources at a time, 0.40
// with one component's), are listed on the device, and nothing waits on the host.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "fw_tile.cuh"
#include "handle.h"

namespace spq {

namespace {

constexpr int MTH = 256;
constexpr int MT = 128;      // targets per tile: 16 groups of 8
constexpr int MS = 64;       // sources per tile: 16 groups of 4
constexpr int MK = 32;       // boundary vertices per staged chunk
constexpr int MLD = MK + 4;  // row stride in shared memory: 16-byte rows on different banks

template <typename T>
__device__ __forceinline__ T tmin2(T a, T b) {
    return a < b ? a : b;
}
__device__ __forceinline__ int32_t add_min(int32_t a, int32_t b, int32_t t) { return __viaddmin_s32(a, b, t); }
__device__ __forceinline__ float add_min(float a, float b, float t) { return fminf(t, a + b); }

// key = component of the vertex (k for an id out of range: sorted last), val = position
__global__ void k_comp_keys(const int32_t* __restrict__ ids, int64_t n, int32_t nv, const int32_t* __restrict__ comp,
                            uint32_t k, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t v = ids[i];
    keys[i] = (v >= 0 && v < nv) ? (uint32_t)comp[v] : k;
    vals[i] = (uint32_t)i;
}

// A tile of the sorted targets: positions [start, start + count) of component c (k: ids out
// of range), whose values of t start at column toff (a multiple of 4).
struct MTile {
    uint32_t c, start, count, toff;
};

// What the targets need on the device: the number of tiles, of components with targets, and
// of columns of t (only those components have any: a row of t over every component would leave
// room for few sources at a time where the targets are few).
struct MCount {
    uint32_t ntiles, ncomp, width, pad_;
};

// The tiles of every component (thread c): its run of the sorted keys by two binary
// searches, cut into pieces of MT; comps: the components with a run and their columns of t.
__global__ void k_matrix_tiles(const uint32_t* __restrict__ keys, int64_t n, uint32_t k, MTile* __restrict__ tiles,
                               MCount* __restrict__ count, uint2* __restrict__ comps,
                               const int32_t* __restrict__ nb) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c > k) return;
    auto lower = [&](uint32_t x) {  // first position with keys >= x
        int64_t lo = 0, hi = n;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (keys[mid] < x) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    const int64_t a = lower(c), b = lower(c + 1);
    if (a == b) return;
    uint32_t toff = 0;
    if (c < k) {
        toff = atomicAdd(&count->width, (uint32_t)(nb[c] + 3) & ~3u);
        comps[atomicAdd(&count->ncomp, 1u)] = make_uint2(c, toff);
    }
    const uint32_t m = (uint32_t)((b - a + MT - 1) / MT), at = atomicAdd(&count->ntiles, m);
    for (uint32_t i = 0; i < m; ++i)
        tiles[at + i] = MTile{c, (uint32_t)(a + (int64_t)i * MT), (uint32_t)std::min<int64_t>(MT, b - a - (int64_t)i * MT), toff};
}

// Stage 1: t of the sources sid[s0 .. s0 + ns) for the components with targets, a warp per
// (source, component); values past |B2| up to a multiple of 4 are infinite.  Only components
// with targets are enumerated: over all k of them, a grid whose warps are a multiple of k gives
// each warp one component for good, so that with few targets most warps had nothing to do.
template <typename T>
__global__ void __launch_bounds__(MTH) k_matrix_t(const QueryCtx<T> ctx, const int32_t* __restrict__ sid,
                                                  int64_t s0, int64_t ns, const MCount* __restrict__ count,
                                                  const uint2* __restrict__ comps, int64_t ldt,
                                                  T* __restrict__ t) {
    const int lane = threadIdx.x & 31;
    const T inf = Inf<T>::value();
    const int64_t nw = ((int64_t)gridDim.x * MTH) >> 5, nc = count->ncomp;
    for (int64_t x = ((int64_t)blockIdx.x * MTH + threadIdx.x) >> 5; x < ns * nc; x += nw) {
        const int64_t s = x / nc;
        const uint2 ct = comps[x - s * nc];
        const int32_t c2 = (int32_t)ct.x;
        const int32_t v1 = sid[s0 + s];
        if (v1 < 0 || v1 >= ctx.n) continue;
        const int32_t c1 = ctx.comp[v1];
        const MatDesc d1 = ctx.descs[c1];
        const int32_t nb1 = ctx.nb[c1], nb2 = ctx.nb[c2], nb4 = (nb2 + 3) & ~3;
        const int32_t* pos1 = ctx.bgpos + ctx.bg_off[c1];
        const int32_t* pos2 = ctx.bgpos + ctx.bg_off[c2];
        const T* a1 = ctx.apsp + d1.off + (int64_t)ctx.local[v1] * d1.n;
        T* tr = t + s * ldt + ct.y;
        for (int32_t jb = 0; jb < nb4; jb += 128) {
            int32_t col[4];
            T y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t j = jb + 32 * q + lane;
                col[q] = j < nb2 ? pos2[j] : -1;
                y[q] = inf;
            }
            for (int32_t ib = 0; ib < nb1; ib += 32) {
                const T areg = ib + lane < nb1 ? a1[ib + lane] : inf;
                const int32_t preg = ib + lane < nb1 ? pos1[ib + lane] : 0;
                const int iend = (nb1 - ib) < 32 ? (nb1 - ib) : 32;
#pragma unroll 4
                for (int ii = 0; ii < iend; ++ii) {
                    const T a = __shfl_sync(0xffffffffu, areg, ii);
                    const T* drow = ctx.D + (int64_t)__shfl_sync(0xffffffffu, preg, ii) * ctx.N;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (col[q] >= 0) y[q] = add_min(a, drow[col[q]], y[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t j = jb + 32 * q + lane;
                if (j < nb4) tr[j] = y[q];
            }
        }
    }
}

template <typename T>
struct MSmem {
    union {
        struct {
            T a[2][MT][MLD];  // the targets' rows of APSP(C2)
            T t[2][MS][MLD];  // the sources' rows of t
        };
        T out[MS][MT + 1];
    };
    int32_t tv[MT];        // the targets' vertices
    uint32_t tp[MT];       // and positions in the caller's list
    int32_t sv[MS];        // the sources' vertices (-1: out of range)
    int64_t arow[MT];
};

// Stage 2: items (target tile, group of MS sources), persistent.
template <typename T, bool OUT_F32>
__global__ void __launch_bounds__(MTH, 2)
    k_matrix_out(const QueryCtx<T> ctx, uint32_t k, const int32_t* __restrict__ sid, int64_t s0, int64_t ns,
                 const int32_t* __restrict__ tid_, const uint32_t* __restrict__ tval, const MTile* __restrict__ tiles,
                 const MCount* __restrict__ count, int64_t nt, int64_t ldt, const T* __restrict__ t,
                 void* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MSmem<T>& sm = *reinterpret_cast<MSmem<T>*>(smem_raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const T inf = Inf<T>::value();
    const int64_t ntiles = count->ntiles, nsg = (ns + MS - 1) / MS;
    for (int64_t item = blockIdx.x; item < ntiles * nsg; item += gridDim.x) {
        const MTile tl = tiles[item % ntiles];
        const int64_t sb = (item / ntiles) * MS;
        const int nsrc = (int)((ns - sb) < MS ? (ns - sb) : MS);
        const int nt_ = (int)tl.count;
        const bool valid = tl.c < k;
        MatDesc d2{0, 0, 0};
        int32_t nb4 = 0;
        int64_t to = 0;
        if (valid) {
            d2 = ctx.descs[tl.c];
            nb4 = (ctx.nb[tl.c] + 3) & ~3;
            to = tl.toff;
        }
        if (tid < MT) {
            const uint32_t p = tid < nt_ ? tval[tl.start + tid] : 0u;
            const int32_t v = tid < nt_ ? tid_[p] : -1;
            sm.tv[tid] = v;
            sm.tp[tid] = p;
            sm.arow[tid] = valid && tid < nt_ ? d2.off + (int64_t)ctx.local[v] * d2.n : d2.off;
        } else if (tid < MT + MS) {
            const int s = tid - MT;
            const int32_t v = s < nsrc ? sid[s0 + sb + s] : -1;
            sm.sv[s] = v >= 0 && v < ctx.n ? v : -1;
        }
        __syncthreads();
        // (rows past the tile's targets repeat a row of the table, sources past the group's a
        //  row of t: neither is written out)
        auto stage = [&](int32_t k0) {
            const int b = (k0 / MK) & 1;
            const int q = tid & 7;
            if (k0 + 4 * q < nb4) {
                for (int r = tid >> 3; r < MT; r += MTH / 8) cp_async16(&sm.a[b][r][4 * q], ctx.apsp + sm.arow[r] + k0 + 4 * q);
                for (int r = tid >> 3; r < MS; r += MTH / 8)
                    cp_async16(&sm.t[b][r][4 * q], t + (sb + (r < nsrc ? r : 0)) * ldt + to + k0 + 4 * q);
            }
            cp_async_commit();
        };
        T acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = inf;
        if (nb4 > 0) stage(0);
        for (int32_t k0 = 0; k0 < nb4; k0 += MK) {
            if (k0 + MK < nb4) {
                stage(k0 + MK);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncthreads();
            const int b = (k0 / MK) & 1;
            const int kend = nb4 - k0 < MK ? nb4 - k0 : MK;
#pragma unroll 1
            for (int kk = 0; kk < kend; kk += 4) {
                int4 tv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) tv[j] = *reinterpret_cast<const int4*>(&sm.t[b][tx + 16 * j][kk]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int4 av = *reinterpret_cast<const int4*>(&sm.a[b][ty + 16 * i][kk]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if constexpr (std::is_same<T, float>::value) {
                            const float2 x = __fadd2_rn(make_float2(__int_as_float(av.x), __int_as_float(av.y)),
                                                        make_float2(__int_as_float(tv[j].x), __int_as_float(tv[j].y)));
                            const float2 y = __fadd2_rn(make_float2(__int_as_float(av.z), __int_as_float(av.w)),
                                                        make_float2(__int_as_float(tv[j].z), __int_as_float(tv[j].w)));
                            acc[i][j] = fmin3(fmin3(acc[i][j], x.x, x.y), y.x, y.y);
                        } else {
                            acc[i][j] = __viaddmin_s32(av.x, tv[j].x, acc[i][j]);
                            acc[i][j] = __viaddmin_s32(av.y, tv[j].y, acc[i][j]);
                            acc[i][j] = __viaddmin_s32(av.z, tv[j].z, acc[i][j]);
                            acc[i][j] = __viaddmin_s32(av.w, tv[j].w, acc[i][j]);
                        }
                    }
                }
            }
            __syncthreads();  // (the buffer's next chunk; after the last one, `out` below)
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sm.out[tx + 16 * j][ty + 16 * i] = acc[i][j];
        __syncthreads();
        const int tt = tid & (MT - 1);
        if (tt < nt_) {
            const int32_t v2 = sm.tv[tt];
            const int32_t l2 = valid ? ctx.local[v2] : 0;
            for (int s = tid / MT; s < nsrc; s += MTH / MT) {
                const int32_t v1 = sm.sv[s];
                const int64_t at = (s0 + sb + s) * nt + sm.tp[tt];
                if (!valid || v1 < 0) {
                    if (OUT_F32)
                        ((float*)out)[at] = __int_as_float(0x7fc00000);
                    else
                        ((int32_t*)out)[at] = -1;
                    continue;
                }
                T y = sm.out[s][tt];
                if (ctx.comp[v1] == (int32_t)tl.c)
                    y = tmin2(y, ctx.apsp[d2.off + (int64_t)ctx.local[v1] * d2.n + l2]);
                if (v1 == v2) y = T(0);
                if (OUT_F32)
                    ((float*)out)[at] = (float)y;
                else
                    ((int32_t*)out)[at] = (int32_t)tmin2<int32_t>((int32_t)y, SPQ_INF_I32);
            }
        }
        if ((!valid && tid == 0) || (tid < nsrc && sm.sv[tid] < 0)) atomicOr(ctx.err, kErrPair);
        __syncthreads();  // the tile's records are rewritten by the next item
    }
}

int g_msms = 0;
int msms() {
    if (g_msms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_msms, cudaDevAttrMultiProcessorCount, dev);
        if (g_msms <= 0) g_msms = 1;
    }
    return g_msms;
}

// Most boundary vertices of a component: the entry point's documented limit.  (It dates from a
// kernel that kept t of eight sources in shared memory; the kernels here need no such buffer.)
constexpr int32_t kMatrixMaxNb = 6400;
constexpr int64_t kTElems = 1 << 24;  // most values of t at a time (64 MB), at least MS rows

template <typename T, bool OUT_F32>
cudaError_t matrix_launch(const QueryCtx<T>& ctx, uint32_t k, const int32_t* src, int64_t ns,
                          const int32_t* tgt, const uint32_t* tval, const MTile* tiles, const MCount* count,
                          const uint2* comps, int64_t nt, int64_t ldt, int64_t rows, T* t, void* out,
                          cudaStream_t st) {
    auto kern = k_matrix_out<T, OUT_F32>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MSmem<T>));
    for (int64_t s0 = 0; s0 < ns && e == cudaSuccess; s0 += rows) {
        const int64_t n = std::min(rows, ns - s0);
        const int64_t warps = n * std::min<int64_t>(k, nt);  // at most
        k_matrix_t<T><<<(unsigned)std::min<int64_t>((warps + 7) / 8, (int64_t)msms() * 32), MTH, 0, st>>>(
            ctx, src, s0, n, count, comps, ldt, t);
        const int64_t items = ((nt + MT - 1) / MT + k + 1) * ((n + MS - 1) / MS);
        kern<<<(unsigned)std::min<int64_t>(items, (int64_t)msms() * 2), MTH, sizeof(MSmem<T>), st>>>(
            ctx, k, src, s0, n, tgt, tval, tiles, count, nt, ldt, t, out);
        count_launches(2);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace
}  // namespace spq

extern "C" spq_status spq_query_matrix(spq_handle* h, const int32_t* sources, int64_t ns, const int32_t* targets,
                                       int64_t nt, void* dist_out, void* stream) {
    using namespace spq;
    if (!h || ns < 0 || nt < 0 || !on_handle_device(h)) return SPQ_EINVAL;
    if (ns == 0 || nt == 0) return SPQ_OK;
    if (!sources || !targets || !dist_out) return SPQ_EINVAL;
    if (ns > INT32_MAX || nt > INT32_MAX) return SPQ_EINVAL;
    if (h->arena) return SPQ_EUNSUPPORTED;
    cudaPointerAttributes a;
    auto on_dev = [&](const void* p) {
        if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
    };
    const bool ds = on_dev(sources), dt = on_dev(targets), dd = on_dev(dist_out);
    if (ds != dt || ds != dd) return SPQ_EINVAL;
    if (!ds && (ns * nt > ((int64_t)1 << 31))) return SPQ_EINVAL;  // host output: bounded
    cudaStream_t st = (cudaStream_t)stream;
    QueryCtx<int32_t> ci;
    QueryCtx<float> cf;
    bool f32store = false, out_f32 = false;
    int32_t k = 0;
    handle_query_view(h, &ci, &cf, &f32store, &out_f32, &k);
    if (h->max_nb > kMatrixMaxNb) return SPQ_EUNSUPPORTED;
    std::vector<void*> tmp;
    auto alloc = [&](void** p, size_t bytes) {
        cudaError_t e = scratch_alloc(p, bytes ? bytes : 4, st);
        if (e == cudaSuccess) tmp.push_back(*p);
        return e;
    };
    auto finish = [&](spq_status s) {
        for (void* p : tmp) cudaFreeAsync(p, st);
        return s;
    };
    auto fail = [&](cudaError_t err) {
        note_cuda_error(err);
        return finish(SPQ_ECUDA);
    };
    const int32_t *d_s = sources, *d_t = targets;
    void* d_out = dist_out;
    cudaError_t e = cudaSuccess;
    if (!ds) {
        void *p1, *p2, *p3;
        if ((e = alloc(&p1, (size_t)ns * 4)) != cudaSuccess || (e = alloc(&p2, (size_t)nt * 4)) != cudaSuccess ||
            (e = alloc(&p3, (size_t)(ns * nt) * 4)) != cudaSuccess)
            return fail(e);
        cudaMemcpyAsync(p1, sources, (size_t)ns * 4, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(p2, targets, (size_t)nt * 4, cudaMemcpyHostToDevice, st);
        d_s = (const int32_t*)p1;
        d_t = (const int32_t*)p2;
        d_out = p3;
    }
    // the targets sorted by component, their tiles, t of a batch of sources
    // (its rows: the components with targets, at most nt of them)
    const int64_t ldt = std::min(round_up(h->nbg + 3 * (int64_t)k, 4), std::min<int64_t>(nt, k) * round_up(h->max_nb, 4)) + 4;
    int64_t rows = std::min(round_up(ns, MS), std::max<int64_t>(MS, kTElems / ldt / MS * MS));
    const int64_t max_tiles = (nt + MT - 1) / MT + k + 1;
    uint32_t* buf;
    MCount* count;  // then the components with targets
    MTile* tiles;
    void* t;
    if ((e = alloc((void**)&buf, (size_t)(4 * nt + radix_hist_words(nt)) * 4)) != cudaSuccess ||
        (e = alloc((void**)&count, sizeof(MCount) + (size_t)k * sizeof(uint2))) != cudaSuccess ||
        (e = alloc((void**)&tiles, (size_t)max_tiles * sizeof(MTile))) != cudaSuccess)
        return fail(e);
    // (fewer sources at a time where t of that many does not fit)
    while ((e = alloc(&t, (size_t)(rows * ldt) * 4)) == cudaErrorMemoryAllocation && rows > 1) {
        cudaGetLastError();
        rows = (rows + 1) / 2;
    }
    if (e != cudaSuccess) return fail(e);
    uint2* comps = reinterpret_cast<uint2*>(count + 1);
    k_comp_keys<<<(unsigned)((nt + 255) / 256), 256, 0, st>>>(d_t, nt, h->n, h->comp, (uint32_t)k, buf, buf + nt);
    int bits = 0;
    while (bits < 32 && ((uint64_t)k >> bits)) ++bits;
    bool in_k1 = false;
    if ((e = radix_sort_pairs(buf, buf + nt, buf + 2 * nt, buf + 3 * nt, buf + 4 * nt, nt, bits, &in_k1, st)) !=
            cudaSuccess ||
        (e = cudaMemsetAsync(count, 0, sizeof(MCount), st)) != cudaSuccess)
        return fail(e);
    k_matrix_tiles<<<(unsigned)((k + 1 + 127) / 128), 128, 0, st>>>(in_k1 ? buf + 2 * nt : buf, nt, (uint32_t)k, tiles,
                                                                    count, comps, h->nb);
    count_launches(2);
    const uint32_t* tval = in_k1 ? buf + 3 * nt : buf + nt;
    if (f32store)
        e = out_f32 ? matrix_launch<float, true>(cf, (uint32_t)k, d_s, ns, d_t, tval, tiles, count, comps, nt,
                                                 ldt, rows, (float*)t, d_out, st)
                    : matrix_launch<float, false>(cf, (uint32_t)k, d_s, ns, d_t, tval, tiles, count, comps, nt,
                                                  ldt, rows, (float*)t, d_out, st);
    else
        e = out_f32 ? matrix_launch<int32_t, true>(ci, (uint32_t)k, d_s, ns, d_t, tval, tiles, count, comps, nt,
                                                   ldt, rows, (int32_t*)t, d_out, st)
                    : matrix_launch<int32_t, false>(ci, (uint32_t)k, d_s, ns, d_t, tval, tiles, count, comps,
                                                    nt, ldt, rows, (int32_t*)t, d_out, st);
    if (e != cudaSuccess) return fail(e);
    if (!ds) {
        if ((e = cudaMemcpyAsync(dist_out, d_out, (size_t)(ns * nt) * 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
            return fail(e);
        uint32_t f = 0;
        cudaMemcpyAsync(&f, h->err, sizeof(f), cudaMemcpyDeviceToHost, st);
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return fail(e);
        if (f & kErrPair) {
            cudaMemsetAsync(h->err, 0, sizeof(uint32_t), st);
            cudaStreamSynchronize(st);
            return finish(SPQ_EINVAL);
        }
    }
    return finish(SPQ_OK);
}
