// Gradients of query distances with respect to edge weights (float32 graphs).
//
// Forward (spq_query_saved): Algorithm 2 as in query.cu, keeping the minimising boundary
// pair (b1*, b2*) (local boundary indices; ties broken towards the smallest (b1, b2) so the
// choice does not depend on the launch), or a marker: -1 the same-component distance
// dist_C1(v1, v2) won, -2 v1 = v2, -3 no path.  One warp per pair, or for large batches
// grouped by component pair (query_blocks.cu: the distance, then the witness that attains it).
//
// Backward (spq_query_backward): the distance is the length of a shortest path, so its
// derivative with respect to the weight of a CSR slot is the number of times the path
// uses that slot (where the path is unique).  Each pair's path is walked again without
// having been stored: inside a component, from x towards target t, the next slot is the
// one minimising w(x, u) + dist_C(u, t) over the slots x -> u staying in the component
// (the APSP(C) tables hold dist_C); across the boundary graph, from boundary vertex b
// towards b2*, the next move minimises either dist_C(b, y) + dist_BG(y, b2*) over the
// other boundary vertices y of b's component (a clique edge, expanded into its path
// inside the component) or w(b, u) + dist_BG(u, b2*) over the slots b -> u into other
// components.  Each slot on the path receives the pair's upstream gradient (atomicAdd).
// Where a batch's moves are worth it, those minima are first computed once for the whole graph
// and the walks follow the records (walk.cuh); the form here finds each move on the way.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <new>
#include <vector>

#include "common.cuh"
#include "handle.h"
#include "walk.cuh"

namespace spq {
namespace {

constexpr int GTH = 256;
constexpr int kNoPath = -3, kSame = -2, kDirect = -1;

// Warp-wide lexicographic argmin of (value, index).
template <typename T>
__device__ __forceinline__ void warp_argmin(T& v, int64_t& i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const T v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const int64_t i2 = __shfl_xor_sync(0xffffffffu, i, o);
        if (less_lex(v2, i2, v, i)) {
            v = v2;
            i = i2;
        }
    }
}

// Forward with the minimising boundary pair.  dist_out: T[q]; saved: int2[q].
template <typename T>
__global__ void __launch_bounds__(GTH) k_query_saved(const View<T> V, const int2* __restrict__ pairs, int64_t q,
                                                     T* __restrict__ dist_out, int2* __restrict__ saved,
                                                     uint32_t* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * GTH) >> 5;
    const T inf = Inf<T>::value();
    for (int64_t qi = ((int64_t)blockIdx.x * GTH + threadIdx.x) >> 5; qi < q; qi += nw) {
        const int2 pr = pairs[qi];
        const int32_t v = pr.x, w = pr.y;
        if (v < 0 || v >= V.n || w < 0 || w >= V.n) {
            if (lane == 0) {
                dist_out[qi] = (T)-1;
                saved[qi] = make_int2(kNoPath, kNoPath);
                atomicOr(err, kErrPair);
            }
            continue;
        }
        if (v == w) {
            if (lane == 0) {
                dist_out[qi] = T(0);
                saved[qi] = make_int2(kSame, kSame);
            }
            continue;
        }
        const int32_t c1 = V.comp[v], c2 = V.comp[w];
        const MatDesc d1 = V.descs[c1], d2 = V.descs[c2];
        const T* A1 = V.apsp + d1.off + (int64_t)V.local[v] * d1.n;
        const T* A2 = V.apsp + d2.off + (int64_t)V.local[w] * d2.n;
        const int32_t nb1 = V.nb[c1], nb2 = V.nb[c2];
        const int32_t* pos1 = V.bgpos + V.bg_off[c1];
        const int32_t* pos2 = V.bgpos + V.bg_off[c2];
        // lane-owned columns j; per column the best row i (smallest on ties)
        T best = inf;
        int64_t bidx = INT64_MAX;  // (i << 32) + j
        for (int32_t j = lane; j < nb2; j += 32) {
            const T cj = A2[j];
            const int64_t colp = pos2[j];
            T t = inf;
            int32_t ti = 0;
            for (int32_t i = 0; i < nb1; ++i) {
                const T cand = A1[i] + V.D[(int64_t)pos1[i] * V.N + colp];
                if (cand < t) {
                    t = cand;
                    ti = i;
                }
            }
            const T tot = t + cj;
            const int64_t idx = ((int64_t)ti << 32) + j;
            if (less_lex(tot, idx, best, bidx)) {
                best = tot;
                bidx = idx;
            }
        }
        warp_argmin(best, bidx);
        if (lane == 0) {
            int2 sv = best < inf ? make_int2((int32_t)(bidx >> 32), (int32_t)(bidx & 0xffffffff))
                                 : make_int2(kNoPath, kNoPath);
            if (c1 == c2) {
                const T direct = A1[V.local[w]];
                if (direct <= best && direct < inf) {
                    best = direct;
                    sv = make_int2(kDirect, kDirect);
                }
            }
            dist_out[qi] = best;
            saved[qi] = sv;
        }
    }
}

// Walk inside component c from vertex x to the vertex of local index tl, adding g to
// every slot taken.  All lanes of the warp take part; returns false if the walk did not
// reach its target within `limit` steps.
// Visitors of the slots a walk takes (called by lane 0 only).
struct AddGrad {
    float g;
    float* grad;
    __device__ void operator()(int64_t e, int32_t /*to*/) const { atomicAdd(&grad[e], g); }
};
struct RecordPath {
    int32_t* verts;  // this pair's row of max_len vertices
    int32_t max_len;
    int32_t* len;    // vertices written so far (may exceed max_len: the path did not fit)
    __device__ void operator()(int64_t /*e*/, int32_t to) const {
        const int32_t i = (*len)++;
        if (i < max_len) verts[i] = to;
    }
};

template <typename T, typename Visit>
__device__ bool walk_in_component(const View<T>& V, int32_t c, int32_t x, int32_t tl, const Visit& visit,
                                  int64_t limit, int lane) {
    const MatDesc d = V.descs[c];
    const T* A = V.apsp + d.off;
    const T inf = Inf<T>::value();
    for (int64_t step = 0; V.local[x] != tl; ++step) {
        if (step >= limit) return false;
        T best = inf;
        int64_t be = INT64_MAX;
        for (int64_t e = V.rp[x] + lane; e < V.rp[x + 1]; e += 32) {
            const int32_t u = V.col[e];
            if (u == x || V.comp[u] != c) continue;
            const T cand = V.w[e] + A[(int64_t)V.local[u] * d.n + tl];
            if (less_lex(cand, e, best, be)) {
                best = cand;
                be = e;
            }
        }
        warp_argmin(best, be);
        if (be == INT64_MAX) return false;
        x = V.col[be];
        if (lane == 0) visit(be, x);
    }
    return true;
}

// Walk through the boundary graph from boundary vertex b to boundary vertex b2.
template <typename T, typename Visit>
__device__ bool walk_boundary_graph(const View<T>& V, int32_t b, int32_t b2, const Visit& visit, int64_t limit,
                                    int lane) {
    const T inf = Inf<T>::value();
    const int64_t pb2 = V.bgpos[V.bg_off[V.comp[b2]] + V.local[b2]];
    const int64_t kInter = (int64_t)1 << 40;
    for (int64_t step = 0; b != b2; ++step) {
        if (step >= limit) return false;
        const int32_t cb = V.comp[b], lb = V.local[b];
        const MatDesc d = V.descs[cb];
        const T* Ab = V.apsp + d.off + (int64_t)lb * d.n;
        const int32_t* posb = V.bgpos + V.bg_off[cb];
        T best = inf;
        int64_t bi = INT64_MAX;
        for (int32_t y = lane; y < V.nb[cb]; y += 32) {  // clique edges of b's component
            if (y == lb) continue;
            const T cand = Ab[y] + V.D[(int64_t)posb[y] * V.N + pb2];
            if (less_lex(cand, (int64_t)y, best, bi)) {
                best = cand;
                bi = y;
            }
        }
        for (int64_t e = V.rp[b] + lane; e < V.rp[b + 1]; e += 32) {  // edges into other components
            const int32_t u = V.col[e];
            const int32_t cu = V.comp[u];
            if (cu == cb) continue;
            const T cand = V.w[e] + V.D[(int64_t)V.bgpos[V.bg_off[cu] + V.local[u]] * V.N + pb2];
            if (less_lex(cand, kInter + e, best, bi)) {
                best = cand;
                bi = kInter + e;
            }
        }
        warp_argmin(best, bi);
        if (bi == INT64_MAX) return false;
        if (bi < kInter) {
            const int32_t y = (int32_t)bi;
            if (!walk_in_component(V, cb, b, y, visit, limit, lane)) return false;
            b = V.vorder[V.vstart[cb] + y];
        } else {
            const int64_t e = bi - kInter;
            b = V.col[e];
            if (lane == 0) visit(e, b);
        }
    }
    return true;
}

// The whole path of one pair: v1 -> b1* inside C1, b1* -> b2* through the boundary
// graph, b2* -> v2 inside C2 (or v1 -> v2 inside C1 when the direct distance won).
template <typename T, typename Visit>
__device__ bool walk_pair(const View<T>& V, int32_t v, int32_t w, int2 sv, const Visit& visit, int64_t limit,
                          int lane) {
    const int32_t c1 = V.comp[v], c2 = V.comp[w];
    // a witness that is not one this handle's forward call can produce fails the walk
    if (sv.x == kDirect) return c1 == c2 && walk_in_component(V, c1, v, V.local[w], visit, limit, lane);
    if (sv.x < 0 || sv.x >= V.nb[c1] || sv.y < 0 || sv.y >= V.nb[c2]) return false;
    const int32_t b1 = V.vorder[V.vstart[c1] + sv.x];
    const int32_t b2 = V.vorder[V.vstart[c2] + sv.y];
    return walk_in_component(V, c1, v, sv.x, visit, limit, lane) &&
           walk_boundary_graph(V, b1, b2, visit, limit, lane) &&
           walk_in_component(V, c2, b2, V.local[w], visit, limit, lane);
}

template <typename T>
__global__ void __launch_bounds__(GTH) k_query_backward(const View<T> V, const int2* __restrict__ pairs,
                                                        const int2* __restrict__ saved, int64_t q,
                                                        const float* __restrict__ gdist, float* __restrict__ grad,
                                                        uint32_t* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * GTH) >> 5;
    const int64_t limit = (int64_t)V.n + 1;
    for (int64_t qi = ((int64_t)blockIdx.x * GTH + threadIdx.x) >> 5; qi < q; qi += nw) {
        const int2 pr = pairs[qi];
        const int2 sv = saved[qi];
        const float g = gdist[qi];
        if (sv.x == kSame || sv.x == kNoPath || g == 0.0f) continue;
        if (pr.x < 0 || pr.x >= V.n || pr.y < 0 || pr.y >= V.n) continue;
        const AddGrad visit{g, grad};
        if (!walk_pair(V, pr.x, pr.y, sv, visit, limit, lane) && lane == 0) atomicOr(err, kErrWalk);
    }
}

// Vertex sequence of each pair's shortest path: verts[i][0] = v1, ..., up to v2;
// lens[i] = number of vertices (-1: no path; > max_len: did not fit, truncated).
template <typename T>
__global__ void __launch_bounds__(GTH) k_query_paths(const View<T> V, const int2* __restrict__ pairs,
                                                     const int2* __restrict__ saved, int64_t q, int32_t max_len,
                                                     int32_t* __restrict__ verts, int32_t* __restrict__ lens,
                                                     uint32_t* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * GTH) >> 5;
    const int64_t limit = (int64_t)V.n + 1;
    for (int64_t qi = ((int64_t)blockIdx.x * GTH + threadIdx.x) >> 5; qi < q; qi += nw) {
        const int2 pr = pairs[qi];
        const int2 sv = saved[qi];
        int32_t* row = verts + qi * (int64_t)max_len;
        if (sv.x == kNoPath || pr.x < 0 || pr.x >= V.n || pr.y < 0 || pr.y >= V.n) {
            if (lane == 0) lens[qi] = -1;
            continue;
        }
        int32_t len = 1;
        if (lane == 0 && max_len > 0) row[0] = pr.x;
        if (sv.x != kSame) {
            const RecordPath visit{row, max_len, &len};
            if (!walk_pair(V, pr.x, pr.y, sv, visit, limit, lane) && lane == 0) atomicOr(err, kErrWalk);
        }
        if (lane == 0) lens[qi] = len;
    }
}

// ---------------- large batches: walks by the records of walk.cuh ----------------

// Part of a backward walk: the moves of pair i through the boundary graph.  A clique edge
// adds the pair's upstream gradient to its flow, an edge between components to its slot.
template <typename T, int H>
__global__ void __launch_bounds__(GTH, 5) k_backward_bg(const View<T> V, const WalkCtx<T> W,
                                                     const uint32_t* __restrict__ order, const int2* __restrict__ pairs, const int2* __restrict__ saved,
                                                     int64_t q, const float* __restrict__ gdist,
                                                     float* __restrict__ grad, uint32_t* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * GTH) >> 5;
    const int64_t limit = (int64_t)V.n + 1;
    for (int64_t p = ((int64_t)blockIdx.x * GTH + threadIdx.x) >> 5; p < q; p += nw) {
        const int64_t qi = order ? order[p] : p;
        const int2 pr = pairs[qi];
        const int2 sv = saved[qi];
        const float g = gdist[qi];
        if (sv.x == kSame || sv.x == kNoPath || sv.x == kDirect || g == 0.0f) continue;
        if (pr.x < 0 || pr.x >= V.n || pr.y < 0 || pr.y >= V.n) continue;
        const int32_t c1 = V.comp[pr.x], c2 = V.comp[pr.y];
        if (sv.x < 0 || sv.x >= V.nb[c1] || sv.y < 0 || sv.y >= V.nb[c2]) continue;  // (marked by k_backward_ends)
        const bool ok = walk_bg<T, H>(
            V, W, c1, sv.x, c2, sv.y, limit, lane,
            [&](int32_t c, int32_t b, int32_t y, int32_t nb) {
                if (lane == 0) atomicAdd(W.flow + W.foff[c] + (int64_t)b * nb + y, g);
            },
            [&](int32_t e, int32_t) {
                if (lane == 0) atomicAdd(grad + e, g);
            });
        if (!ok && lane == 0) atomicOr(err, kErrWalk);
    }
}

// The rest of it: v1 -> b1* inside C1 (by the hop table) and b2* -> v2 inside C2 (or v1 ->
// v2 directly), searched slot by slot: v2 is any vertex.  Eight lanes a pair.
constexpr int ESUB = 8;
template <typename T>
__global__ void __launch_bounds__(GTH, 6) k_backward_ends(const View<T> V, const WalkCtx<T> W,
                                                       const uint32_t* __restrict__ order, const int2* __restrict__ pairs, const int2* __restrict__ saved,
                                                       int64_t q, const float* __restrict__ gdist,
                                                       float* __restrict__ grad, uint32_t* __restrict__ err) {
    const int lane = threadIdx.x & 31, g8 = lane & (ESUB - 1);
    const unsigned mask = ((1u << ESUB) - 1u) << (lane & ~(ESUB - 1));
    const int64_t nw = ((int64_t)gridDim.x * GTH) / ESUB;
    const int64_t limit = (int64_t)V.n + 1;
    for (int64_t p = ((int64_t)blockIdx.x * GTH + threadIdx.x) / ESUB; p < q; p += nw) {
        const int64_t qi = order ? order[p] : p;
        const int2 pr = pairs[qi];
        const int2 sv = saved[qi];
        const float g = gdist[qi];
        if (sv.x == kSame || sv.x == kNoPath || g == 0.0f) continue;
        if (pr.x < 0 || pr.x >= V.n || pr.y < 0 || pr.y >= V.n) continue;
        const int32_t c1 = V.comp[pr.x], c2 = V.comp[pr.y], lw = V.local[pr.y];
        int32_t x = V.local[pr.x];
        bool ok;
        if (sv.x == kDirect) {
            ok = c1 == c2;
        } else {
            ok = sv.x >= 0 && sv.x < V.nb[c1] && sv.y >= 0 && sv.y < V.nb[c2];
            if (ok) {
                const int32_t vs1 = V.vstart[c1];
                ok = walk_hops<T, ESUB>(V, W, c1, x, sv.x, limit, g8, mask,
                                        [&](int32_t from, int32_t slot, int32_t) {
                                            if (g8 == 0) atomicAdd(grad + W.vrange[vs1 + from].x + slot, g);
                                        });
                x = sv.y;
            }
        }
        if (ok) {
            const MatDesc d = V.descs[c2];
            const T* A = V.apsp + d.off;
            const int32_t vs = V.vstart[c2];
            for (int64_t step = 0; x != lw; ++step) {
                const int32_t e = step < limit ? best_slot<T, ESUB>(V, W, A, d.n, vs, x, lw, g8, mask) : -1;
                if (e < 0) {
                    ok = false;
                    break;
                }
                if (g8 == 0) atomicAdd(grad + e, g);
            }
        }
        if (!ok && g8 == 0) atomicOr(err, kErrWalk);
    }
}

// Every clique edge's flow onto the slots of its path inside the component, one thread each.
template <typename T>
__global__ void __launch_bounds__(GTH) k_backward_flow(const View<T> V, const WalkCtx<T> W, int32_t k, int64_t total,
                                                       float* __restrict__ grad, uint32_t* __restrict__ err) {
    const int64_t i = (int64_t)blockIdx.x * GTH + threadIdx.x;
    if (i >= total) return;
    const float g = W.flow[i];
    if (g == 0.0f) return;
    int32_t lo = 0, hi = k;  // the component whose range holds i
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (W.foff[mid] <= i) lo = mid; else hi = mid;
    }
    const int32_t nb = V.nb[lo], vs = V.vstart[lo];
    // (64 bits: |B|^2 passes 2^31 from 46,341 boundary vertices on)
    const int64_t r = i - W.foff[lo], b = r / nb;
    const bool ok = walk_hops<T, 1>(V, W, lo, (int32_t)b, (int32_t)(r - b * nb), (int64_t)V.n + 1, 0,
                                    1u << (threadIdx.x & 31),
                                    [&](int32_t from, int32_t slot, int32_t) {
                                        atomicAdd(grad + W.vrange[vs + from].x + slot, g);
                                    });
    if (!ok) atomicOr(err, kErrWalk);
}

// Vertex sequences: as k_query_paths, a warp per pair.  The moves through the boundary graph
// are collected 32 at a time, and each lane expands one of them: once to count its hops
// (its place in the row is the sum of the earlier ones'), once to write its vertices.
template <typename T, int H>
__global__ void __launch_bounds__(GTH, 4) k_paths_hops(const View<T> V, const WalkCtx<T> W,
                                                    const uint32_t* __restrict__ order, const int2* __restrict__ pairs, const int2* __restrict__ saved,
                                                    int64_t q, int32_t max_len, int32_t* __restrict__ verts,
                                                    int32_t* __restrict__ lens, uint32_t* __restrict__ err) {
    // collected moves: (component, from, to) or (-1, vertex, 0)
    __shared__ int32_t sc[GTH / 32][32], sx[GTH / 32][32], st[GTH / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nw = ((int64_t)gridDim.x * GTH) >> 5;
    const int64_t limit = (int64_t)V.n + 1;
    for (int64_t p = ((int64_t)blockIdx.x * GTH + threadIdx.x) >> 5; p < q; p += nw) {
        const int64_t qi = order ? order[p] : p;
        const int2 pr = pairs[qi];
        const int2 sv = saved[qi];
        int32_t* row = verts + qi * (int64_t)max_len;
        if (sv.x == kNoPath || pr.x < 0 || pr.x >= V.n || pr.y < 0 || pr.y >= V.n) {
            if (lane == 0) lens[qi] = -1;
            continue;
        }
        int32_t len = 1;
        if (lane == 0 && max_len > 0) row[0] = pr.x;
        bool ok = true;
        if (sv.x != kSame) {
            const int32_t c1 = V.comp[pr.x], c2 = V.comp[pr.y], lw = V.local[pr.y];
            int32_t x = V.local[pr.x];
            int n = 0;
            auto flush = [&]() {  // expands the n collected moves; false if one did not arrive
                __syncwarp();
                const int32_t c = lane < n ? sc[warp][lane] : -1;
                const int32_t a = lane < n ? sx[warp][lane] : 0, b = lane < n ? st[warp][lane] : 0;
                int32_t cnt = lane < n ? 1 : 0;
                bool good = true;
                if (c >= 0) {
                    cnt = 0;
                    good = walk_hops<T, 1>(V, W, c, a, b, limit, 0, 1u << lane,
                                           [&](int32_t, int32_t, int32_t) { ++cnt; });
                }
                const unsigned bad = __ballot_sync(0xffffffffu, !good);
                const int last = bad ? __ffs(bad) - 1 : 31;  // the moves after a failed one are not made
                if (lane > last) cnt = 0;
                int32_t incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                int32_t at = len + incl - cnt;
                if (cnt > 0 && c < 0) {
                    if (at < max_len) row[at] = a;
                } else if (cnt > 0) {
                    const int32_t vs = V.vstart[c];
                    const int64_t lim = cnt < max_len - at ? cnt : max_len - at;
                    if (lim > 0)
                        walk_hops<T, 1>(V, W, c, a, b, lim, 0, 1u << lane, [&](int32_t, int32_t, int32_t y) {
                            row[at++] = V.vorder[vs + y];
                        });
                }
                len += __shfl_sync(0xffffffffu, incl, 31);
                n = 0;
                __syncwarp();
                return bad == 0;
            };
            auto add = [&](int32_t c, int32_t a, int32_t b) {
                if (lane == 0) {
                    sc[warp][n] = c;
                    sx[warp][n] = a;
                    st[warp][n] = b;
                }
                if (++n == 32) ok = flush() && ok;
            };
            if (sv.x == kDirect) {
                ok = c1 == c2;
            } else if (sv.x < 0 || sv.x >= V.nb[c1] || sv.y < 0 || sv.y >= V.nb[c2]) {
                ok = false;
            } else {
                add(c1, x, sv.x);
                const bool there = walk_bg<T, H>(
                    V, W, c1, sv.x, c2, sv.y, limit, lane,
                    [&](int32_t c, int32_t b, int32_t y, int32_t) {
                        if (ok) add(c, b, y);
                    },
                    [&](int32_t, int32_t at) {
                        if (ok) add(-1, V.vorder[at], 0);
                    });
                if (ok && n > 0) ok = flush();
                ok = ok && there;
                x = sv.y;
            }
            if (ok) {
                const MatDesc d = V.descs[c2];
                const T* A = V.apsp + d.off;
                const int32_t vs = V.vstart[c2];
                for (int64_t step = 0; x != lw; ++step) {
                    const int32_t e = step < limit ? best_slot<T, 32>(V, W, A, d.n, vs, x, lw, lane, 0xffffffffu) : -1;
                    if (e < 0) {
                        ok = false;
                        break;
                    }
                    if (lane == 0 && len < max_len) row[len] = V.vorder[vs + x];
                    ++len;
                }
            }
            if (!ok && lane == 0) atomicOr(err, kErrWalk);
        }
        if (lane == 0) lens[qi] = len;
    }
}

constexpr int64_t kSavedSlice = 1 << 22;

// Whether q pairs are answered with their witnesses in groups: what a group's block, a pair in
// a group and a pair on its own take, in ns of the whole GPU, as functions of the mean |B(C)| =
// nb that fit measurements of random pairs (at nb 28, 56, 118 and 235: a block 10, 16, 31 and
// 108 ns, a pair on its own 2.1, 7.3, 29 and 97), and 60 us of launches for the sort.  Random
// pairs make k^2 (1 - e^(-q / k^2)) groups.  0.95: many tying columns cost a few ns a pair.
// (256 components with nb 118: 20,000 pairs 645 us a warp per pair and 644 grouped, 40,000 1,220
// and 1,035, a million 28,400 and 4,240; 1,024 components with nb 28: a million 2,060 and 7,800.)
bool saved_groups(const spq_handle* h, int64_t q) {
    if (q < 4096 || h->k > 65535 || h->max_nb > query_blocks_max_nb()) return false;
    const double n = (double)q, k2 = (double)h->k * h->k, nb = (double)h->nbg / h->k;
    const double groups = k2 * -expm1(-n / k2);
    return groups * std::max(4.0 + 0.225 * nb, 0.00195 * nb * nb) + n * (0.5 + 0.014 * nb) + 6e4 <
           0.95 * n * (0.035 * nb + 0.00176 * nb * nb);
}

bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return true;
}

int grad_sms() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

template <typename T>
View<T> view_of(const spq_handle* h) {
    return View<T>{h->n,       h->comp,         h->local, h->descs, h->nb,    h->bg_off, h->bgpos, (const T*)h->apsp,
                   (const T*)h->D, h->N, h->csr_rp, h->csr_col, (const T*)h->csr_w, h->vorder, h->vstart};
}

bool on_device(const void* p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// The records of walk.cuh for handle h, in one stream-ordered allocation (freed by the caller
// with cudaFreeAsync(*mem)); false if it does not fit, or if a walk's loop over slots, in 32
// bits and steps of up to 32, could pass INT32_MAX (the caller walks without them).
template <typename T>
bool walk_records(const spq_handle* h, bool want_flow, cudaStream_t st, WalkCtx<T>* W, void** mem, int64_t* nflow) {
    const int32_t k = h->k;
    if (h->m > INT32_MAX - 32) return false;
    std::vector<int64_t> off;
    try {
        off.assign(2 * ((size_t)k + 1), 0);
    } catch (const std::bad_alloc&) {
        return false;
    }
    for (int32_t c = 0; c < k; ++c) {
        off[c + 1] = off[c] + (int64_t)h->h_csize[c] * h->h_nb[c];
        off[k + 2 + c] = off[k + 1 + c] + (int64_t)h->h_nb[c] * h->h_nb[c];
    }
    const int64_t nt = off[k], nf = want_flow ? off[2 * (size_t)k + 1] : 0;
    const int64_t o_out = h->nbg * (2 * kOut * 16);
    const int64_t o_sl = o_out, o_sr = o_sl + h->m * 8, o_off = o_sr + (int64_t)h->n * 8;
    const int64_t o_sc = o_off + (int64_t)off.size() * 8;
    const int64_t o_hop = o_sc + h->nbg * 4, o_fl = o_hop + nt * 4;
    unsigned char* p = nullptr;
    if (scratch_alloc((void**)&p, (size_t)(o_fl + nf * 4), st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    *mem = p;
    *nflow = nf;
    int64_t* d_off = (int64_t*)(p + o_off);
    *W = WalkCtx<T>{(int2*)(p + o_sl), (int2*)(p + o_sr), (int32_t*)(p + o_sc),    (int4*)p,
                    d_off,             d_off + (k + 1),   (uint32_t*)(p + o_hop), (float*)(p + o_fl)};
    const View<T> V = view_of<T>(h);
    cudaMemcpyAsync(d_off, off.data(), off.size() * 8, cudaMemcpyHostToDevice, st);
    if (nf > 0) cudaMemsetAsync(p + o_fl, 0, (size_t)nf * 4, st);
    k_walk_slots<T><<<(unsigned)((h->n + 255) / 256), 256, 0, st>>>(V, (int2*)(p + o_sl), (int2*)(p + o_sr),
                                                                       (int32_t*)(p + o_sc), (int4*)p);
    k_walk_hops<T><<<(unsigned)(((int64_t)h->n * 32 + 255) / 256), 256, 0, st>>>(V, *W, (uint32_t*)(p + o_hop));
    count_launches(2);
    return true;
}

// Whether q walks pay for the records: a hop searched on the spot costs about 0.17 ns of the
// GPU (measured: 1M pairs on 2^18 vertices 86 ms, 100k on 2^14 1.96 ms; the hops of a pair
// grow with sqrt(n)), the records about 60 us plus 8 ps per table entry.  Never inside a
// stream capture: a captured call allocates nothing.
bool walks_pay(const spq_handle* h, int64_t q, cudaStream_t st) {
    if (capturing(st)) return false;
    double nt = 0.0;
    for (int32_t c = 0; c < h->k; ++c) nt += (double)h->h_csize[c] * h->h_nb[c];
    return 21.0 * (double)q * sqrt((double)h->n) > 7.5e6 + nt;
}

__global__ void k_target_keys(const int2* __restrict__ pairs, int64_t q, int32_t n, const int32_t* __restrict__ comp,
                              uint32_t k, uint32_t* __restrict__ keys, uint32_t* __restrict__ idx) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= q) return;
    const int32_t w = pairs[i].y;
    keys[i] = w >= 0 && w < n ? (uint32_t)comp[w] : k;
    idx[i] = (uint32_t)i;
}

// The order the walks are taken in: by the target's component, so that the matrix rows and
// the table that a component's walks read (22 MB and 4 MB for 1,024 vertices) stay in L2
// while they do (1M pairs on 2^18 vertices in their own order: 11.1 + 5.6 ms, 7 TB/s of it
// from DRAM for the most part).  Null (the pairs' own order) where the tables fit L2 anyway,
// for small batches, or where the sort's scratch does not fit.
const uint32_t* walk_order(const spq_handle* h, const int32_t* pairs, int64_t q, cudaStream_t st, void** mem) {
    *mem = nullptr;
    if (h->bytes < (size_t)64 << 20 || q < 16384 || q > (int64_t)UINT32_MAX) return nullptr;
    uint32_t* b = nullptr;
    if (scratch_alloc((void**)&b, (size_t)(4 * q + radix_hist_words(q)) * 4, st) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    *mem = b;
    k_target_keys<<<(unsigned)((q + 255) / 256), 256, 0, st>>>((const int2*)pairs, q, h->n, h->comp, (uint32_t)h->k, b,
                                                               b + q);
    count_launches(1);
    int bits = 0;
    while (bits < 32 && ((uint64_t)h->k >> bits)) ++bits;
    bool in_k1 = false;
    if (radix_sort_pairs(b, b + q, b + 2 * q, b + 3 * q, b + 4 * q, q, bits, &in_k1, st) != cudaSuccess) return nullptr;
    return in_k1 ? b + 3 * q : b + q;
}

template <typename T>
bool backward_by_records(const spq_handle* h, const int32_t* pairs, int64_t q, const int32_t* saved,
                         const float* grad_dist, float* grad_w, cudaStream_t st) {
    WalkCtx<T> W;
    void* mem = nullptr;
    int64_t nf = 0;
    if (!walk_records<T>(h, true, st, &W, &mem, &nf)) return false;
    void* omem = nullptr;
    const uint32_t* order = walk_order(h, pairs, q, st, &omem);
    const View<T> V = view_of<T>(h);
    const int64_t cap = (int64_t)grad_sms() * 8;
    const int2 *p2 = (const int2*)pairs, *s2 = (const int2*)saved;
    auto bg = h->max_nb <= 128 ? k_backward_bg<T, 4> : (h->max_nb <= 192 ? k_backward_bg<T, 6> : k_backward_bg<T, 8>);
    bg<<<(unsigned)std::min<int64_t>((q + 7) / 8, cap), GTH, 0, st>>>(V, W, order, p2, s2, q, grad_dist, grad_w, h->err);
    k_backward_ends<T><<<(unsigned)std::min<int64_t>((q + GTH / ESUB - 1) / (GTH / ESUB), cap), GTH, 0, st>>>(
        V, W, order, p2, s2, q, grad_dist, grad_w, h->err);
    count_launches(2);
    if (nf > 0) {
        k_backward_flow<T><<<(unsigned)((nf + GTH - 1) / GTH), GTH, 0, st>>>(V, W, h->k, nf, grad_w, h->err);
        count_launches(1);
    }
    cudaFreeAsync(mem, st);
    if (omem) cudaFreeAsync(omem, st);
    return true;
}

template <typename T>
bool paths_by_records(const spq_handle* h, const int32_t* pairs, int64_t q, const int32_t* saved, int32_t max_len,
                      int32_t* verts, int32_t* lens, cudaStream_t st) {
    WalkCtx<T> W;
    void* mem = nullptr;
    int64_t nf = 0;
    if (!walk_records<T>(h, false, st, &W, &mem, &nf)) return false;
    void* omem = nullptr;
    const uint32_t* order = walk_order(h, pairs, q, st, &omem);
    const int64_t cap = (int64_t)grad_sms() * 8;
    auto hops = h->max_nb <= 128 ? k_paths_hops<T, 4> : (h->max_nb <= 192 ? k_paths_hops<T, 6> : k_paths_hops<T, 8>);
    hops<<<(unsigned)std::min<int64_t>((q + 7) / 8, cap), GTH, 0, st>>>(
        view_of<T>(h), W, order, (const int2*)pairs, (const int2*)saved, q, max_len, verts, lens, h->err);
    count_launches(1);
    cudaFreeAsync(mem, st);
    if (omem) cudaFreeAsync(omem, st);
    return true;
}

}  // namespace
}  // namespace spq

extern "C" {

spq_status spq_query_saved(spq_handle* h, const int32_t* pairs, int64_t q, void* dist_out, int32_t* saved,
                           void* stream) {
    using namespace spq;
    if (!h || q < 0 || !on_handle_device(h)) return SPQ_EINVAL;
    if (q == 0) return SPQ_OK;
    if (!h->vorder || !h->csr_rp) return SPQ_EUNSUPPORTED;
    if (!on_device(pairs) || !on_device(dist_out) || !on_device(saved)) return SPQ_EINVAL;
    if (((uintptr_t)pairs & 7u) || ((uintptr_t)saved & 7u) || ((uintptr_t)dist_out & 3u)) return SPQ_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    // Large batches grouped by component pair, each block of the boundary matrix read once per
    // group (1M pairs on 2^18 vertices: a warp per pair 28.3 ms, most of it the block's rows
    // from DRAM again for every pair; grouped 4.2 ms); at most kSavedSlice pairs at a time (39
    // words of scratch a pair).  Not inside a stream capture: a captured call allocates nothing.
    if (saved_groups(h, q) && !capturing(st)) {
        uint32_t* scratch = nullptr;
        const int64_t slice = std::min(q, kSavedSlice);
        if (scratch_alloc((void**)&scratch, (size_t)query_saved_scratch_words(slice) * 4, st) == cudaSuccess) {
            QueryCtx<int32_t> ci;
            QueryCtx<float> cf;
            bool f32store = false, out_f32 = false;
            int32_t k = 0;
            const bool ran = h->qprof_ran;  // (the query profile covers spq_query only)
            handle_query_view(h, &ci, &cf, &f32store, &out_f32, &k);
            h->qprof_ran = ran;
            cudaError_t e = cudaSuccess;
            for (int64_t a = 0; a < q && e == cudaSuccess; a += slice) {
                const int64_t n = std::min(slice, q - a);
                e = f32store ? launch_query_saved_grouped<float>(cf, pairs + 2 * a, n, (float*)dist_out + a,
                                                                 saved + 2 * a, (uint32_t)k, scratch, st)
                             : launch_query_saved_grouped<int32_t>(ci, pairs + 2 * a, n, (int32_t*)dist_out + a,
                                                                   saved + 2 * a, (uint32_t)k, scratch, st);
            }
            cudaFreeAsync(scratch, st);
            if (e != cudaSuccess) note_cuda_error(e);
            return e == cudaSuccess ? SPQ_OK : SPQ_ECUDA;
        }
        cudaGetLastError();  // (no room: a warp per pair needs none)
    }
    int64_t blocks = (q + 7) / 8;
    const int64_t cap = (int64_t)grad_sms() * 16;
    if (blocks > cap) blocks = cap;
    if (h->f32store)
        k_query_saved<float><<<(unsigned)blocks, GTH, 0, st>>>(view_of<float>(h), (const int2*)pairs, q,
                                                                (float*)dist_out, (int2*)saved, h->err);
    else
        k_query_saved<int32_t><<<(unsigned)blocks, GTH, 0, st>>>(view_of<int32_t>(h), (const int2*)pairs, q,
                                                                  (int32_t*)dist_out, (int2*)saved, h->err);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? SPQ_OK : SPQ_ECUDA;
}

spq_status spq_query_backward(spq_handle* h, const int32_t* pairs, int64_t q, const int32_t* saved,
                              const float* grad_dist, float* grad_w, void* stream) {
    using namespace spq;
    if (!h || q < 0 || !on_handle_device(h)) return SPQ_EINVAL;
    if (q == 0) return SPQ_OK;
    if (!h->vorder || !h->csr_rp) return SPQ_EUNSUPPORTED;
    if (!on_device(pairs) || !on_device(saved) || !on_device(grad_dist) || !on_device(grad_w)) return SPQ_EINVAL;
    if (((uintptr_t)pairs & 7u) || ((uintptr_t)saved & 7u)) return SPQ_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (walks_pay(h, q, st) &&
        (h->f32store ? backward_by_records<float>(h, pairs, q, saved, grad_dist, grad_w, st)
                     : backward_by_records<int32_t>(h, pairs, q, saved, grad_dist, grad_w, st)))
        return cudaGetLastError() == cudaSuccess ? SPQ_OK : SPQ_ECUDA;
    int64_t blocks = (q + 7) / 8;
    const int64_t cap = (int64_t)grad_sms() * 16;
    if (blocks > cap) blocks = cap;
    if (h->f32store)
        k_query_backward<float><<<(unsigned)blocks, GTH, 0, st>>>(view_of<float>(h), (const int2*)pairs,
                                                                   (const int2*)saved, q, grad_dist, grad_w, h->err);
    else
        k_query_backward<int32_t><<<(unsigned)blocks, GTH, 0, st>>>(view_of<int32_t>(h), (const int2*)pairs,
                                                                     (const int2*)saved, q, grad_dist, grad_w,
                                                                     h->err);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? SPQ_OK : SPQ_ECUDA;
}

spq_status spq_query_paths(spq_handle* h, const int32_t* pairs, int64_t q, const int32_t* saved, int32_t max_len,
                           int32_t* verts, int32_t* lens, void* stream) {
    using namespace spq;
    if (!h || q < 0 || max_len < 0 || !on_handle_device(h)) return SPQ_EINVAL;
    if (q == 0) return SPQ_OK;
    if (!h->vorder || !h->csr_rp) return SPQ_EUNSUPPORTED;
    if (!on_device(pairs) || !on_device(saved) || !on_device(lens) || (max_len > 0 && !on_device(verts)))
        return SPQ_EINVAL;
    if (((uintptr_t)pairs & 7u) || ((uintptr_t)saved & 7u)) return SPQ_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (walks_pay(h, q, st) &&
        (h->f32store ? paths_by_records<float>(h, pairs, q, saved, max_len, verts, lens, st)
                     : paths_by_records<int32_t>(h, pairs, q, saved, max_len, verts, lens, st)))
        return cudaGetLastError() == cudaSuccess ? SPQ_OK : SPQ_ECUDA;
    int64_t blocks = (q + 7) / 8;
    const int64_t cap = (int64_t)grad_sms() * 16;
    if (blocks > cap) blocks = cap;
    if (h->f32store)
        k_query_paths<float><<<(unsigned)blocks, GTH, 0, st>>>(view_of<float>(h), (const int2*)pairs,
                                                                (const int2*)saved, q, max_len, verts, lens, h->err);
    else
        k_query_paths<int32_t><<<(unsigned)blocks, GTH, 0, st>>>(view_of<int32_t>(h), (const int2*)pairs,
                                                                  (const int2*)saved, q, max_len, verts, lens,
                                                                  h->err);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? SPQ_OK : SPQ_ECUDA;
}

}  // extern "C"
