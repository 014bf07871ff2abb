// Path walks for large batches (gradients and path retrieval, grad.cu): the same moves as
// walk_pair's, one by one, from records made once per call.
//
// What bounds a walk is latency: a warp that looks at every slot of every vertex on the way
// waits for five dependent loads a hop (0.2 ns of the whole GPU per hop: 86 ms for a million
// pairs of 400 hops).  Four records shorten it:
//   slots   per CSR slot its target's local index (same component) or boundary slot and
//           matrix position (another component): no comp / local / bgpos look-ups on the way;
//   out     per boundary slot its slots into other components with all that a move needs
//           (slot, target, position, weight; the target's component, |B|, first slot, first
//           vertex): one load where the CSR is three deep, and none of the look-ups by
//           component after the move;
//   hops    per component, vertex x and boundary vertex t: the slot that the walk from x
//           towards t takes first and the vertex it leads to (4 bytes; sum of |C||B(C)|), so a
//           hop towards a boundary vertex is one load;
//   flow    (gradients) per component and pair (b, y) of boundary vertices: the upstream
//           gradients of all pairs whose walk takes the clique edge b -> y, so that each
//           clique edge is expanded into its slots once and not once per pair.
// In the boundary graph a warp holds the distances D(y, b2) of a component's boundary
// vertices y in registers for as long as the walk stays in the component, and reads them
// along row b2 of D.  D is symmetric bit for bit outside its diagonal 128 x 128 tiles (the
// kernels store such a tile and its mirror from the same registers); inside them the walk
// reads D(y, b2) itself, so that each comparison sees the value it always saw.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace spq {
namespace {

// Read-only tables of a handle, as the walks use them.
template <typename T>
struct View {
    int32_t n;
    const int32_t* comp;
    const int32_t* local;
    const MatDesc* descs;
    const int32_t* nb;
    const int32_t* bg_off;
    const int32_t* bgpos;
    const T* apsp;
    const T* D;
    int64_t N;
    const int64_t* rp;
    const int32_t* col;
    const T* w;
    const int32_t* vorder;
    const int32_t* vstart;
};

// (value, index) order: ties to the smallest index.
template <typename T>
__device__ __forceinline__ bool less_lex(T a, int64_t ai, T b, int64_t bi) {
    return a < b || (a == b && ai < bi);
}

constexpr int kOut = 4;  // slots into other components in a boundary slot's record
constexpr uint32_t kNoHop = 0xffffffffu;  // no entry of the table (searched on the spot)

template <typename T>
struct WalkCtx {
    const int2* slots;        // [m]: (local index, 0) inside the component; (~slot, position); (INT_MIN, 0) self-loop
    const int2* vrange;       // [n]: CSR range of the vertex at vstart[c] + local index
    const int32_t* scomp;     // [|BG|]: a boundary slot's component
    const int4* out;          // [|BG| x kOut x 2]: a boundary slot's slots into other components
    const int64_t* toff;      // [k + 1]: hops of component c at toff[c] + x * |B| + t
    const int64_t* foff;      // [k + 1]: flow of component c at foff[c] + b * |B| + y
    const uint32_t* hops;
    float* flow;
};

// Values compared as unsigned words: distances are never negative (word_of: nor -0).
__device__ __forceinline__ uint32_t key_of(int32_t v) { return (uint32_t)v; }
__device__ __forceinline__ uint32_t key_of(float v) { return (uint32_t)__float_as_int(v + 0.0f); }
__device__ __forceinline__ uint32_t word_of(int32_t v) { return (uint32_t)v; }
__device__ __forceinline__ uint32_t word_of(float v) { return (uint32_t)__float_as_int(v); }

template <typename T>
__global__ void __launch_bounds__(256) k_walk_slots(const View<T> V, int2* __restrict__ slots,
                                                    int2* __restrict__ vrange, int32_t* __restrict__ scomp,
                                                    int4* __restrict__ out) {
    const int32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= V.n) return;
    const int32_t c = V.comp[u], l = V.local[u];
    const int64_t e0 = V.rp[u], e1 = V.rp[u + 1];
    const bool bnd = l < V.nb[c];
    int4* o = out + (int64_t)(bnd ? V.bg_off[c] + l : 0) * (2 * kOut);
    int n = 0;
    for (int64_t e = e0; e < e1; ++e) {
        const int32_t v = V.col[e];
        const int32_t cv = V.comp[v];
        if (cv != c && bnd) {
            if (n < kOut) {
                const int32_t s = V.bg_off[cv] + V.local[v];
                const T w = V.w[e];
                o[2 * n] = make_int4((int32_t)e, s, V.bgpos[s], *reinterpret_cast<const int32_t*>(&w));
                o[2 * n + 1] = make_int4(cv, V.nb[cv], V.bg_off[cv], V.vstart[cv]);
            }
            ++n;
        }
        if (cv == c) {
            slots[e] = v == u ? make_int2(INT32_MIN, 0) : make_int2(V.local[v], 0);
        } else {
            const int32_t s = V.bg_off[cv] + V.local[v];
            slots[e] = make_int2(~s, V.bgpos[s]);
        }
    }
    vrange[V.vstart[c] + l] = make_int2((int32_t)e0, (int32_t)e1);
    if (bnd) {
        scomp[V.bg_off[c] + l] = c;
        // (unused places: position -1; too many slots: -2 in all, the CSR is searched)
        for (int i = n > kOut ? 0 : n; i < kOut; ++i) o[2 * i] = make_int4(0, 0, n > kOut ? -2 : -1, 0);
    }
}

// The slot a walk inside component c takes at local vertex x towards local vertex t: the one
// minimising w + dist_C(u, t), ties to the smallest slot.  sub lanes of the warp (lane g of
// them) share the slots; every one of them returns the slot (-1: none) and, in x, the vertex.
template <typename T, int SUB>
__device__ __forceinline__ int32_t best_slot(const View<T>& V, const WalkCtx<T>& W, const T* A, int32_t ld,
                                             int32_t vs, int32_t& x, int32_t t, int g, unsigned mask) {
    const int2 er = W.vrange[vs + x];
    T best = Inf<T>::value();
    int32_t be = INT32_MAX, to = -1;  // (a graph has fewer than INT32_MAX slots)
    for (int32_t e = er.x + g; e < er.y; e += SUB) {
        const int32_t u = W.slots[e].x;
        if (u < 0) continue;
        const T cand = V.w[e] + A[(int64_t)u * ld + t];
        if (less_lex(cand, e, best, be)) {
            best = cand;
            be = e;
            to = u;
        }
    }
#pragma unroll
    for (int o = SUB / 2; o > 0; o >>= 1) {
        const T b2 = __shfl_xor_sync(mask, best, o);
        const int32_t e2 = __shfl_xor_sync(mask, be, o);
        const int32_t t2 = __shfl_xor_sync(mask, to, o);
        if (less_lex(b2, e2, best, be)) {
            best = b2;
            be = e2;
            to = t2;
        }
    }
    if (be == INT32_MAX) return -1;
    x = to;
    return be;
}

// hops: a warp per vertex, lanes over the boundary vertices (consecutive columns of the
// neighbours' rows of APSP(C)).  An entry is (slot - first slot) << 16 | local target, or
// kNoHop where either needs more than 16 bits (or no slot leads on).
template <typename T>
__global__ void __launch_bounds__(256) k_walk_hops(const View<T> V, const WalkCtx<T> W, uint32_t* __restrict__ hops) {
    const int lane = threadIdx.x & 31;
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (v >= V.n) return;
    const int32_t c = V.comp[v], x = V.local[v], nb = V.nb[c];
    const MatDesc d = V.descs[c];
    const T* A = V.apsp + d.off;
    const int64_t e0 = V.rp[v], e1 = V.rp[v + 1];
    uint32_t* row = hops + W.toff[c] + (int64_t)x * nb;
    for (int32_t t0 = 0; t0 < nb; t0 += 128) {
        T best[4];
        int64_t be[4];
        int32_t to[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            best[q] = Inf<T>::value();
            be[q] = INT64_MAX;
            to[q] = 0;
        }
        for (int64_t e = e0; e < e1; ++e) {
            const int32_t u = W.slots[e].x;
            if (u < 0) continue;
            const T we = V.w[e];
            const T* Au = A + (int64_t)u * d.n;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t t = t0 + 32 * q + lane;
                if (t < nb) {
                    const T cand = we + Au[t];
                    if (less_lex(cand, e, best[q], be[q])) {
                        best[q] = cand;
                        be[q] = e;
                        to[q] = u;
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int32_t t = t0 + 32 * q + lane;
            if (t < nb) {
                const bool ok = be[q] != INT64_MAX && be[q] - e0 < 0xffff && to[q] < 0x10000;
                row[t] = ok ? ((uint32_t)(be[q] - e0) << 16) | (uint32_t)to[q] : kNoHop;
            }
        }
    }
}

// Walk inside component c from local vertex x to boundary vertex t along the hop table;
// visit(from, slot - first slot of from, to) each hop.  SUB lanes walk together (all of them call visit).
template <typename T, int SUB, typename Visit>
__device__ __forceinline__ bool walk_hops(const View<T>& V, const WalkCtx<T>& W, int32_t c, int32_t x, int32_t t,
                                          int64_t limit, int g, unsigned mask, const Visit& visit) {
    const int32_t nb = V.nb[c], vs = V.vstart[c];
    const uint32_t* tab = W.hops + W.toff[c] + t;
    for (int64_t step = 0; x != t; ++step) {
        if (step >= limit) return false;
        const uint32_t h = tab[(int64_t)x * nb];
        if (h != kNoHop) {
            const int32_t from = x;
            x = (int32_t)(h & 0xffffu);
            visit(from, (int32_t)(h >> 16), x);
        } else {
            const int32_t from = x;
            const MatDesc d = V.descs[c];
            const int32_t e = best_slot<T, SUB>(V, W, V.apsp + d.off, d.n, vs, x, t, g, mask);
            if (e < 0) return false;
            visit(from, e - W.vrange[vs + from].x, x);
        }
    }
    return true;
}

// Walk through the boundary graph from boundary vertex (c, l) to (c2, l2), the whole warp
// together: clique(c, l, y, nb) or edge(e, the target's place in vorder) for every move (all
// lanes call them).  As
// walk_boundary_graph: the move minimising dist_C(b, y) + D(y, b2) over the component's other
// boundary vertices y or w(e) + D(u, b2) over the slots into other components, ties to the
// smallest y, then to the smallest slot.
// H: boundary vertices held per lane (components of up to 32 H; wider ones look the rest up).
template <typename T, int H, typename Clique, typename Edge>
__device__ __forceinline__ bool walk_bg(const View<T>& V, const WalkCtx<T>& W, int32_t c, int32_t l, int32_t c2,
                                        int32_t l2, int64_t limit, int lane, const Clique& clique, const Edge& edge) {
    const uint32_t kinf = key_of(Inf<T>::value());
    const int32_t s2 = V.bg_off[c2] + l2;
    const int64_t p2 = V.bgpos[s2];
    const T* Drow = V.D + p2 * V.N;
    auto dist = [&](int64_t p) {  // D(p, p2)
        return (p >> 7) == (p2 >> 7) ? V.D[p * V.N + p2] : Drow[p];
    };
    int64_t step = 0;
    bool fresh = true;
    T dv[H];
    int32_t nb = V.nb[c], off = V.bg_off[c], vs = V.vstart[c], ld = 0;
    const T* A = nullptr;
    for (;;) {
        if (c == c2 && l == l2) return true;
        if (step++ >= limit) return false;
        if (fresh) {  // another component: its slots' distances to b2
            const MatDesc d = V.descs[c];
            A = V.apsp + d.off;
            ld = d.n;
#pragma unroll
            for (int q = 0; q < H; ++q) {
                const int32_t y = lane + 32 * q;
                // (+ 0: a sum with it is never -0, whose pattern is the largest)
                dv[q] = y < nb ? dist(V.bgpos[off + y]) + T(0) : Inf<T>::value();
            }
            fresh = false;
        }
        const int4* o = W.out + (int64_t)(off + l) * (2 * kOut);
        const int4 oa = lane < kOut ? o[2 * lane] : make_int4(0, 0, -1, 0);
        const int4 ob = lane < kOut ? o[2 * lane + 1] : make_int4(0, 0, 0, 0);
        const T* Ab = A + (int64_t)l * ld;
        // the sums over the component's other boundary vertices, as words that order like them
        uint32_t key[H], bk = kinf;
        T av[H];
#pragma unroll
        for (int q = 0; q < H; ++q) {
            const int32_t y = lane + 32 * q;
            av[q] = y < nb && y != l ? Ab[y] : Inf<T>::value();
        }
        // ... and over the slots into other components
        uint32_t ek = kinf;
        int32_t ei = 0;
        if (oa.z >= 0) {
            const T w = *reinterpret_cast<const T*>(&oa.w);
            ek = word_of((T)(w + (dist(oa.z) + T(0))));
            ei = oa.x;
        }
        const bool many = __any_sync(0xffffffffu, oa.z == -2);
        if (many) {
            const int2 er = W.vrange[vs + l];
            for (int32_t e = er.x + lane; e < er.y; e += 32) {
                const int2 s = W.slots[e];
                if (s.x >= 0 || s.x == INT32_MIN) continue;
                const uint32_t k = word_of((T)(V.w[e] + (dist(s.y) + T(0))));
                if (k < ek) {
                    ek = k;
                    ei = e;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < H; ++q) {
            key[q] = word_of((T)(av[q] + dv[q]));
            bk = min(bk, key[q]);
        }
        uint32_t wk = kinf;
        int32_t wi = 0;
        for (int32_t y = lane + 32 * H; y < nb; y += 32) {
            if (y == l) continue;
            const uint32_t k = word_of((T)(Ab[y] + (dist(V.bgpos[off + y]) + T(0))));
            if (k < wk) {
                wk = k;
                wi = y;
            }
        }
        const uint32_t mk = __reduce_min_sync(0xffffffffu, min(min(bk, wk), ek));
        if (mk >= kinf) return false;
        // the smallest y attaining it, else the smallest slot
        uint32_t yi = wk == mk ? (uint32_t)wi : 0xffffffffu;
#pragma unroll
        for (int q = H - 1; q >= 0; --q)
            if (key[q] == mk) yi = (uint32_t)(lane + 32 * q);
        const int32_t y = (int32_t)__reduce_min_sync(0xffffffffu, yi);
        if (y >= 0) {
            clique(c, l, y, nb);
            l = y;
        } else {
            const int32_t e = (int32_t)__reduce_min_sync(0xffffffffu, ek == mk ? (uint32_t)ei : 0xffffffffu);
            int32_t s;
            if (many) {
                s = ~W.slots[e].x;
                c = W.scomp[s];
                nb = V.nb[c];
                off = V.bg_off[c];
                vs = V.vstart[c];
            } else {
                const int src = __ffs(__ballot_sync(0xffffffffu, oa.z >= 0 && oa.x == e)) - 1;
                s = __shfl_sync(0xffffffffu, oa.y, src);
                c = __shfl_sync(0xffffffffu, ob.x, src);
                nb = __shfl_sync(0xffffffffu, ob.y, src);
                off = __shfl_sync(0xffffffffu, ob.z, src);
                vs = __shfl_sync(0xffffffffu, ob.w, src);
            }
            edge(e, vs + s - off);
            l = s - off;
            fresh = true;
        }
    }
}

}  // namespace
}  // namespace spq
