// Evaluation of one work item from a genome record staged in shared memory:
// the node rule of Section 3.3 applied level by level.  Shared by the
// single-population forward kernel, the multi-population persistent kernel
// and the CPPN query kernel.
#pragma once

#include "neat_device.cuh"
#include "neat_internal.h"

namespace neat {

// Barrier among the G threads of group `gi` (G a power of two).  Groups of
// at most a warp use a warp-level barrier on their lanes; larger groups use
// a named barrier (id 1 + gi) unless the group is the whole block.
__device__ __forceinline__ void group_sync(int G, int gi)
{
    if (G < 32) {
        const unsigned base = (threadIdx.x & 31u) & ~(unsigned)(G - 1);
        __syncwarp(((1u << G) - 1u) << base);
    } else if (G == 32) {
        __syncwarp();
    } else if (G == (int)blockDim.x) {
        __syncthreads();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(gi + 1), "r"(G) : "memory");
    }
}

// Value slot of position p, column col.  T1: one column (tile 1).
template <bool T1>
__device__ __forceinline__ int vslot(uint32_t p, int lgT, int col)
{
    return T1 ? (int)p : (int)(p << lgT) + col;
}

// Aggregation order.  A node's incoming edges i = 0..ec-1 (record order) are
// dealt round-robin into four partials, partial k = edges k, k+4, k+8, ...,
// each accumulated in increasing i (sum and mean with fused multiply-add);
// the aggregate is ((p0 . p1) . (p2 . p3)) with . the aggregation's binary
// operation, divided by ec for the mean, and 0 when ec = 0.  The order is a
// function of the genome alone: one thread, two or four threads per node
// (combined through warp shuffles along the same tree) give identical bits.
enum : uint32_t { kAggSum = 0, kAggProduct = 1, kAggMax = 2, kAggMean = 3 };

__device__ __forceinline__ float agg_identity(uint32_t agg)
{
    // max starts from NaN: fmaxf(NaN, x) = x, and an all-NaN set stays NaN
    return agg == kAggProduct ? 1.0f : (agg == kAggMax ? __int_as_float(0x7fc00000) : 0.0f);
}

__device__ __forceinline__ float agg_combine(uint32_t agg, float a, float b)
{
    return agg == kAggProduct ? a * b : (agg == kAggMax ? fmaxf(a, b) : a + b);
}

__device__ __forceinline__ float agg_step(uint32_t agg, float acc, float w, float x)
{
    return agg == kAggProduct ? acc * (w * x) : (agg == kAggMax ? fmaxf(acc, w * x) : fmaf(w, x, acc));
}

// Partials k0 .. k0+nk-1 of one node for one column, combined along the tree.
template <bool T1, bool SUM>
__device__ __forceinline__ float partials(uint32_t agg, const uint2 *__restrict__ e, uint32_t ec,
                                          const float *__restrict__ v, int lgT, int col, int k0, int nk)
{
    if (SUM) agg = kAggSum;
    const float id = SUM ? 0.0f : agg_identity(agg);
    if (nk == 4) {
        float q0 = id, q1 = id, q2 = id, q3 = id;
        uint32_t i = 0;
        // not unrolled further: nodes have few edges (about 8 in the Ant
        // workload), where a second copy of the body costs more issue than
        // it saves (measured 8.27 -> 8.09 us per Ant step without it)
#pragma unroll 1
        for (; i + 4 <= ec; i += 4) {
            const uint2 t0 = e[i], t1 = e[i + 1], t2 = e[i + 2], t3 = e[i + 3];
            q0 = agg_step(agg, q0, __uint_as_float(t0.x), v[vslot<T1>(t0.y, lgT, col)]);
            q1 = agg_step(agg, q1, __uint_as_float(t1.x), v[vslot<T1>(t1.y, lgT, col)]);
            q2 = agg_step(agg, q2, __uint_as_float(t2.x), v[vslot<T1>(t2.y, lgT, col)]);
            q3 = agg_step(agg, q3, __uint_as_float(t3.x), v[vslot<T1>(t3.y, lgT, col)]);
        }
        if (i < ec) { const uint2 t = e[i]; q0 = agg_step(agg, q0, __uint_as_float(t.x), v[vslot<T1>(t.y, lgT, col)]); }
        if (i + 1 < ec) { const uint2 t = e[i + 1]; q1 = agg_step(agg, q1, __uint_as_float(t.x), v[vslot<T1>(t.y, lgT, col)]); }
        if (i + 2 < ec) { const uint2 t = e[i + 2]; q2 = agg_step(agg, q2, __uint_as_float(t.x), v[vslot<T1>(t.y, lgT, col)]); }
        return agg_combine(agg, agg_combine(agg, q0, q1), agg_combine(agg, q2, q3));
    }
    if (nk == 2) {
        float q0 = id, q1 = id;
        for (uint32_t i = (uint32_t)k0; i < ec; i += 4) {
            const uint2 t0 = e[i];
            q0 = agg_step(agg, q0, __uint_as_float(t0.x), v[vslot<T1>(t0.y, lgT, col)]);
            if (i + 1 < ec) {
                const uint2 t1 = e[i + 1];
                q1 = agg_step(agg, q1, __uint_as_float(t1.x), v[vslot<T1>(t1.y, lgT, col)]);
            }
        }
        return agg_combine(agg, q0, q1);
    }
    float q = id;
    for (uint32_t i = (uint32_t)k0; i < ec; i += 4) {
        const uint2 t = e[i];
        q = agg_step(agg, q, __uint_as_float(t.x), v[vslot<T1>(t.y, lgT, col)]);
    }
    return q;
}

// Finish a node from its combined aggregate: mean division, empty set, node rule.
__device__ __forceinline__ float node_output(const uint4 ne, uint32_t agg, uint32_t act, uint32_t ec, float a)
{
    if (agg == kAggMean) a = a / (float)ec;
    if (ec == 0) a = 0.0f;
    return activate(act, fmaf(__uint_as_float(ne.y), a, __uint_as_float(ne.x)));
}

// The four partials of one node for one column of a tile, combined along
// the tree, for a compile-time aggregation AGG (sum also serves mean): the
// operations of `partials` with all four partials, in the same order, so the
// bits are those of every other shape.  One loop per aggregation instead of
// a select among the three per edge.
template <uint32_t AGG>
__device__ __forceinline__ float partials_agg(const uint2 *__restrict__ e, uint32_t ec,
                                              const float *__restrict__ v, int lgT, int col)
{
    const float id = agg_identity(AGG);
    float q0 = id, q1 = id, q2 = id, q3 = id;
    uint32_t i = 0;
#pragma unroll 2
    for (; i + 4 <= ec; i += 4) {
        const uint2 t0 = e[i], t1 = e[i + 1], t2 = e[i + 2], t3 = e[i + 3];
        q0 = agg_step(AGG, q0, __uint_as_float(t0.x), v[vslot<false>(t0.y, lgT, col)]);
        q1 = agg_step(AGG, q1, __uint_as_float(t1.x), v[vslot<false>(t1.y, lgT, col)]);
        q2 = agg_step(AGG, q2, __uint_as_float(t2.x), v[vslot<false>(t2.y, lgT, col)]);
        q3 = agg_step(AGG, q3, __uint_as_float(t3.x), v[vslot<false>(t3.y, lgT, col)]);
    }
    if (i < ec) { const uint2 t = e[i]; q0 = agg_step(AGG, q0, __uint_as_float(t.x), v[vslot<false>(t.y, lgT, col)]); }
    if (i + 1 < ec) { const uint2 t = e[i + 1]; q1 = agg_step(AGG, q1, __uint_as_float(t.x), v[vslot<false>(t.y, lgT, col)]); }
    if (i + 2 < ec) { const uint2 t = e[i + 2]; q2 = agg_step(AGG, q2, __uint_as_float(t.x), v[vslot<false>(t.y, lgT, col)]); }
    return agg_combine(AGG, agg_combine(AGG, q0, q1), agg_combine(AGG, q2, q3));
}

// The four partials of an aggregation AGG over exactly EC edges (EC known
// at compile time), for one column, combined along the tree: straight-line
// code with the operations of `partials` in the same order (partial i mod 4,
// edges in increasing i, from the aggregation's identity), so the same bits.
template <bool T1, uint32_t AGG, int EC>
__device__ __forceinline__ float agg_edges_fixed(const uint2 *__restrict__ e, const float *__restrict__ v, int lgT,
                                                 int col)
{
    const float id = agg_identity(AGG);
    float q[4] = {id, id, id, id};
#pragma unroll
    for (int i = 0; i < EC; ++i) {
        const uint2 t = e[i];
        q[i & 3] = agg_step(AGG, q[i & 3], __uint_as_float(t.x), v[vslot<T1>(t.y, lgT, col)]);
    }
    return agg_combine(AGG, agg_combine(AGG, q[0], q[1]), agg_combine(AGG, q[2], q[3]));
}

// The aggregate of a node's ec edges for one column: one dispatch on ec
// into straight-line code for up to 8 edges (instead of a loop test per
// four edges and three remainder tests), the loop of `partials` beyond.
// For callers whose warp is on one node (a tile row of 32 or more columns,
// a CPPN's queries): lanes on different nodes would run the cases one after
// another.
template <bool T1, uint32_t AGG>
__device__ __forceinline__ float agg_edges(const uint2 *__restrict__ e, uint32_t ec, const float *__restrict__ v,
                                           int lgT, int col)
{
    switch (ec) {
    case 0: return agg_edges_fixed<T1, AGG, 0>(e, v, lgT, col);
    case 1: return agg_edges_fixed<T1, AGG, 1>(e, v, lgT, col);
    case 2: return agg_edges_fixed<T1, AGG, 2>(e, v, lgT, col);
    case 3: return agg_edges_fixed<T1, AGG, 3>(e, v, lgT, col);
    case 4: return agg_edges_fixed<T1, AGG, 4>(e, v, lgT, col);
    case 5: return agg_edges_fixed<T1, AGG, 5>(e, v, lgT, col);
    case 6: return agg_edges_fixed<T1, AGG, 6>(e, v, lgT, col);
    case 7: return agg_edges_fixed<T1, AGG, 7>(e, v, lgT, col);
    case 8: return agg_edges_fixed<T1, AGG, 8>(e, v, lgT, col);
    default:
        if (T1) return partials<T1, AGG == kAggSum>(AGG, e, ec, v, lgT, col, 0, 4);
        return partials_agg<AGG>(e, ec, v, lgT, col);
    }
}

// One whole node for one column of a tile (one thread), the aggregation
// dispatched once per node: the threads of a node row take the same branch.
template <bool FAST>
__device__ __forceinline__ void eval_node_tile(const uint4 ne, const uint2 *__restrict__ edges,
                                               float *__restrict__ v, int p, int lgT, int col)
{
    const uint32_t act = ne.w & 0xffu;
    if (act == kInputAct) return;
    const uint32_t agg = FAST ? kAggSum : ((ne.w >> 8) & 0xffu);
    const uint32_t ec = ne.z >> 16;
    const uint2 *e = edges + (ne.z & 0xffffu);
    float a;
    if (lgT >= 5) {
        // a tile row fills whole warps: every lane of a warp is on this node,
        // so the dispatch on its edge count does not diverge
        if (FAST || agg == kAggSum || agg == kAggMean) a = agg_edges<false, kAggSum>(e, ec, v, lgT, col);
        else if (agg == kAggProduct) a = agg_edges<false, kAggProduct>(e, ec, v, lgT, col);
        else a = agg_edges<false, kAggMax>(e, ec, v, lgT, col);
    } else {
        if (FAST || agg == kAggSum || agg == kAggMean) a = partials_agg<kAggSum>(e, ec, v, lgT, col);
        else if (agg == kAggProduct) a = partials_agg<kAggProduct>(e, ec, v, lgT, col);
        else a = partials_agg<kAggMax>(e, ec, v, lgT, col);
    }
    v[vslot<false>(p, lgT, col)] = FAST ? node_tanh(fmaf(__uint_as_float(ne.y), ec ? a : 0.0f, __uint_as_float(ne.x)))
                                        : node_output(ne, agg, act, ec, a);
}

// walk_levels for 2^lg columns, from position `first` (the inputs before it have
// their values).  One loop for every width: beside one compiled for 32 columns, 2
// to 4% faster there, it took 4 to 10% longer (launches of 4 and 16 vectors, 10
// 000 genomes of 50 rows: 24.6 and 37.7 us, 26.5 and 41.6 with both; six fused
// steps of 300 rows, 1000 genomes, 8 and 16 vectors: 94 and 130, 101 and 136).
template <bool FAST>
__device__ __forceinline__ void walk_tile(const uint4 *nodes, const uint2 *edges, const uint16_t *lev, float *v,
                                          int first, int n_nodes, int n_levels, int G, int gi, int lane, int lg,
                                          bool col_ok)
{
    const int col = lane & ((1 << lg) - 1);
    const int sub = lane >> lg;
    const int nsub = G >> lg;
    if (nsub == 1) {
        if (col_ok)
            for (int p = first; p < n_nodes; ++p) eval_node_tile<FAST>(nodes[p], edges, v, p, lg, col);
    } else {
        int p0 = first;
        for (int l = 0; l < n_levels; ++l) {
            const int p1 = lev[l + 1];
            if (col_ok)
                for (int p = p0 + sub; p < p1; p += nsub) eval_node_tile<FAST>(nodes[p], edges, v, p, lg, col);
            p0 = p1;
            group_sync(G, gi);
        }
    }
}

// ---- two adjacent columns per thread
//
// A tile row of 64 columns is evaluated by 32 threads, columns 2 l and 2 l + 1 in
// thread l: the node's entry, its dispatches and its edges are read once for
// both, their values are one 8-byte read and their sums run as a packed pair.
// Each column's operations are those of eval_node_tile in the same order, so
// the bits are too.
constexpr int kLgPairTile = 6;

template <int EC>
__device__ __forceinline__ f2 sum_edges_pair(const uint2 *__restrict__ e, const char *__restrict__ v)
{
    f2 q[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int i = 0; i < EC; ++i) {
        const uint2 t = e[i];
        const f2 x = *reinterpret_cast<const f2 *>(v + (t.y << (kLgPairTile + 2)));
        q[i & 3] = fma2(pack2(__uint_as_float(t.x), __uint_as_float(t.x)), x, q[i & 3]);
    }
    return add2(add2(q[0], q[1]), add2(q[2], q[3]));
}

__device__ __forceinline__ f2 sum_edges_pair_any(const uint2 *__restrict__ e, uint32_t ec, const char *__restrict__ v)
{
    f2 q[4] = {0ull, 0ull, 0ull, 0ull};
    for (uint32_t i = 0; i < ec; i += 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < ec) {
                const uint2 t = e[i + k];
                const f2 x = *reinterpret_cast<const f2 *>(v + (t.y << (kLgPairTile + 2)));
                q[k] = fma2(pack2(__uint_as_float(t.x), __uint_as_float(t.x)), x, q[k]);
            }
        }
    }
    return add2(add2(q[0], q[1]), add2(q[2], q[3]));
}

template <uint32_t AGG>
__device__ __forceinline__ float2 fold_edges_pair(const uint2 *__restrict__ e, uint32_t ec, const char *__restrict__ v)
{
    float q[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k][0] = q[k][1] = agg_identity(AGG);
    for (uint32_t i = 0; i < ec; i += 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < ec) {
                const uint2 t = e[i + k];
                const float2 x = *reinterpret_cast<const float2 *>(v + (t.y << (kLgPairTile + 2)));
                q[k][0] = agg_step(AGG, q[k][0], __uint_as_float(t.x), x.x);
                q[k][1] = agg_step(AGG, q[k][1], __uint_as_float(t.x), x.y);
            }
        }
    }
    return make_float2(agg_combine(AGG, agg_combine(AGG, q[0][0], q[1][0]), agg_combine(AGG, q[2][0], q[3][0])),
                       agg_combine(AGG, agg_combine(AGG, q[0][1], q[1][1]), agg_combine(AGG, q[2][1], q[3][1])));
}

// Node p for the thread's columns; v: the thread's place in row 0.
template <bool FAST>
__device__ __forceinline__ void eval_node_pair(const uint4 ne, const uint2 *__restrict__ edges, char *__restrict__ v,
                                               int p)
{
    const uint32_t act = ne.w & 0xffu;
    if (act == kInputAct) return;
    const uint32_t agg = FAST ? kAggSum : ((ne.w >> 8) & 0xffu);
    const uint32_t ec = ne.z >> 16;
    const uint2 *e = edges + (ne.z & 0xffffu);
    float2 a;
    if (FAST || agg == kAggSum || agg == kAggMean) {
        f2 s;
        switch (ec) {
        case 0: s = 0ull; break;
        case 1: s = sum_edges_pair<1>(e, v); break;
        case 2: s = sum_edges_pair<2>(e, v); break;
        case 3: s = sum_edges_pair<3>(e, v); break;
        case 4: s = sum_edges_pair<4>(e, v); break;
        case 5: s = sum_edges_pair<5>(e, v); break;
        case 6: s = sum_edges_pair<6>(e, v); break;
        default: s = sum_edges_pair_any(e, ec, v);
        }
        a = unpack2(s);
        if (!FAST && agg == kAggMean && ec > 0) {
            a.x = a.x / (float)ec;
            a.y = a.y / (float)ec;
        }
    } else {
        a = agg == kAggProduct ? fold_edges_pair<kAggProduct>(e, ec, v) : fold_edges_pair<kAggMax>(e, ec, v);
        if (ec == 0) a = make_float2(0.0f, 0.0f);
    }
    const float r = __uint_as_float(ne.y), b = __uint_as_float(ne.x);
    const float z0 = fmaf(r, a.x, b), z1 = fmaf(r, a.y, b);
    float2 y;
    if (FAST) {
        y = make_float2(node_tanh(z0), node_tanh(z1));
    } else {
        switch (act) {                            // one dispatch for both
        case 1: y = make_float2(activate(1, z0), activate(1, z1)); break;
        case 2: y = make_float2(activate(2, z0), activate(2, z1)); break;
        case 3: y = make_float2(activate(3, z0), activate(3, z1)); break;
        case 4: y = make_float2(activate(4, z0), activate(4, z1)); break;
        case 5: y = make_float2(activate(5, z0), activate(5, z1)); break;
        case 6: y = make_float2(activate(6, z0), activate(6, z1)); break;
        default: y = make_float2(z0, z1);
        }
    }
    *reinterpret_cast<float2 *>(v + (p << (kLgPairTile + 2))) = y;
}

// walk_levels for two columns per thread, of which the first `cols` are asked for.
template <bool FAST>
__device__ __forceinline__ void walk_pairs(const uint4 *srec, float *v, int G, int gi, int lane, int cols)
{
    const uint4 h0 = srec[0], h1 = srec[1];
    const int n_levels = (int)(h0.x >> 16);
    const uint4 *nodes = srec + 2;
    const uint2 *edges = reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(srec) + h1.y);
    const uint16_t *lev = reinterpret_cast<const uint16_t *>(reinterpret_cast<const char *>(srec) + h1.z);
    const int pair = lane & 31, sub = lane >> 5, nsub = G >> 5;
    char *mine = reinterpret_cast<char *>(v + 2 * pair);
    const bool ok = 2 * pair < cols;
    int p0 = (int)(h0.w >> 16);
    for (int l = 0; l < n_levels; ++l) {
        const int p1 = lev[l + 1];
        if (ok)
            for (int p = p0 + sub; p < p1; p += nsub) eval_node_pair<FAST>(nodes[p], edges, mine, p);
        p0 = p1;
        group_sync(G, gi);
    }
}

// All non-input nodes of a staged record, for the columns this thread owns.
//  Columns (T > 1): thread `lane` = (sub, col) computes column col of nodes
//  sub, sub + nsub, ... of every level, nsub = G / T.
//  One column (T1): per level, `split` threads (1, 2 or 4, at most
//  2^lg_split_max) share each node, lane = (slot, part); slots = G / split
//  nodes of the level are in flight at once.
// A group barrier separates levels.  Every thread of the group must call it.
// FAST: every non-input node uses sum aggregation and tanh activation (the
// setting of the paper's experiments), decoded once per genome.
template <bool T1, bool FAST>
__device__ __forceinline__ void walk_levels(const uint4 *srec, float *v, int G, int gi, int lane, int lgT,
                                            int lg_split_max, bool col_ok)
{
    const uint4 h0 = srec[0], h1 = srec[1];
    const int n_nodes = (int)(h0.x & 0xffffu), n_levels = (int)(h0.x >> 16);
    const uint4 *nodes = srec + 2;
    const uint2 *edges = reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(srec) + h1.y);
    const uint16_t *lev = reinterpret_cast<const uint16_t *>(reinterpret_cast<const char *>(srec) + h1.z);
    if (T1) {
        // the leading input positions of level 0 are skipped
        int p0 = (int)(h0.w >> 16);
        if (lg_split_max == 0) {                 // one thread per node, no shuffles
            // the node entry of a thread's first node in the next level is
            // read before the level barrier (entries do not depend on values)
            int p1 = lev[1];
            uint4 ne = (p0 + lane < n_nodes) ? nodes[p0 + lane] : make_uint4(0u, 0u, 0u, (uint32_t)kInputAct);
            for (int l = 0; l < n_levels; ++l) {
                const int p2 = lev[l + 2 <= n_levels ? l + 2 : n_levels];
                for (int p = p0 + lane; p < p1; p += G) {
                    if (p != p0 + lane) ne = nodes[p];
                    const uint32_t act = ne.w & 0xffu;
                    if (act == kInputAct) continue;
                    const uint32_t agg = FAST ? kAggSum : ((ne.w >> 8) & 0xffu);
                    const uint32_t ec = ne.z >> 16;
                    const float a = partials<true, FAST>(agg, edges + (ne.z & 0xffffu), ec, v, 0, 0, 0, 4);
                    v[p] = FAST ? node_tanh(fmaf(__uint_as_float(ne.y), ec ? a : 0.0f, __uint_as_float(ne.x)))
                                : node_output(ne, agg, act, ec, a);
                }
                const int pn = p1 + lane;
                if (pn < n_nodes) ne = nodes[pn];
                p0 = p1;
                p1 = p2;
                group_sync(G, gi);
            }
            group_sync(G, gi);
            return;
        }
        // threads per node chosen per level: 4 when the level has at most
        // G/4 nodes, 2 when at most G/2, else 1 (capped by lg_split_max)
        for (int l = 0; l < n_levels; ++l) {
            const int p1 = lev[l + 1];
            const int cnt = p1 - p0;
            const int lg_split = min(lg_split_max, (cnt * 4 <= G) ? 2 : ((cnt * 2 <= G) ? 1 : 0));
            const int split = 1 << lg_split;
            const int slot = lane >> lg_split, part = lane & (split - 1);
            const int slots = G >> lg_split;
            const int nk = 4 >> lg_split;
            const unsigned mask = ((1u << split) - 1u) << ((threadIdx.x & 31u) & ~(unsigned)(split - 1));
            for (int p = p0 + slot; p < p1; p += slots) {
                const uint4 ne = nodes[p];
                const uint32_t act = ne.w & 0xffu;
                if (act == kInputAct) continue;              // same for every part of the slot
                const uint32_t agg = FAST ? kAggSum : ((ne.w >> 8) & 0xffu);
                const uint32_t ec = ne.z >> 16;
                float a = partials<true, FAST>(agg, edges + (ne.z & 0xffffu), ec, v, 0, 0, part * nk, nk);
                for (int m = 1; m < split; m <<= 1) a = agg_combine(agg, a, __shfl_xor_sync(mask, a, m));
                if (part == 0)
                    v[p] = FAST ? node_tanh(fmaf(__uint_as_float(ne.y), ec ? a : 0.0f, __uint_as_float(ne.x)))
                                : node_output(ne, agg, act, ec, a);
            }
            p0 = p1;
            group_sync(G, gi);
        }
    } else {
        walk_tile<FAST>(nodes, edges, lev, v, (int)(h0.w >> 16), n_nodes, n_levels, G, gi, lane, lgT, col_ok);
    }
    group_sync(G, gi);
}

// Record traits word (header word 3): uniform activation | uniform aggregation << 8.
constexpr uint32_t kTraitsSumTanh = 1u | (0u << 8);

__device__ __forceinline__ int ilog2(int x) { return 31 - __clz(x); }

constexpr int kInputRegs = 8;   // inputs prefetched into registers per thread
constexpr uint32_t kNoBar = 0xffffffffu;

// Records and nodes of the sizes that the shapes were made for.
struct AlwaysFits {
    __device__ __forceinline__ bool operator()(uint32_t, int) const { return true; }
};

// Everything of one work item after its record copy was issued by lane 0
// (mbarrier `bar` initialised and armed, `flag` set to 0, both before the
// call; bar kNoBar: the record is read where it is, nothing to wait for): inputs
// are read into registers while the copy is in flight, the group waits for
// the record (a bounded wait; on expiry the device error word gets
// kErrWaitExpired and the outputs NaN), scatters the inputs into the value
// tile, walks the levels and writes the outputs.
//   xb: inputs of the item [bt][I]; yb: its outputs [bt][O]; vcap: floats of
//   the value tile, at least one column of the genome's nodes (a genome with
//   more nodes than the tile has rows takes fewer columns at a time; WHOLE: the
//   tile has the rows, all columns at once, vcap is not read).
//   fits(bytes of the record, values of its columns): asked once the record is
//   there; where it is false, run_item returns false with nothing evaluated.
// PAIRS: two columns per thread (tile 64, WHOLE).
template <bool T1, bool PAIRS = false, bool WHOLE = false, typename Fits>
__device__ __forceinline__ bool run_item(const uint4 *srec, float *v, uint32_t bar, volatile int *flag, int G,
                                         int gi, int lane, const float *__restrict__ xb, float *__restrict__ yb,
                                         int I, int O, int bt, int tile, int lg_split, int vcap, const Fits &fits,
                                         unsigned int *err)
{
    int lgT = T1 ? 0 : ilog2(tile);
    const int nx = bt * I;
    float xr[kInputRegs];
#pragma unroll
    for (int k = 0; k < kInputRegs; ++k) {
        const int i = lane + k * G;
        xr[k] = (i < nx) ? __ldg(xb + i) : 0.0f;
    }
    group_sync(G, gi);                    // barrier initialised before anyone waits on it
    if (bar != kNoBar && !mbar_wait(bar, 0)) *flag = 1;
    group_sync(G, gi);
    if (*flag) {                          // uniform over the group
        if (lane == 0) atomicOr(err, kErrWaitExpired);
        mbar_wait(bar, 0);                // let the copy land before the region is reused
        for (int i = lane; i < bt * O; i += G) yb[i] = __int_as_float(0x7fc00000);
        return true;
    }
    const uint4 h0 = srec[0], h1 = srec[1];
    if (h0.z & NEAT_G_ERROR_MASK) {
        for (int i = lane; i < bt * O; i += G) yb[i] = __int_as_float(0x7fc00000);
        return true;
    }
    if (!fits(h1.x, (int)(h0.x & 0xffffu) << lgT)) return false;
    const uint16_t *io = reinterpret_cast<const uint16_t *>(reinterpret_cast<const char *>(srec) + h1.w);
    if constexpr (!T1 && !WHOLE)
        while (lgT > 0 && ((int)(h0.x & 0xffffu) << lgT) > vcap) --lgT;
    const int step = T1 ? 1 : 1 << lgT;
    constexpr bool kOnce = T1 || WHOLE;
    for (int c0 = 0; c0 < (kOnce ? 1 : bt); c0 += step) {   // once, unless the nodes outgrow the tile's rows
        const int cols = T1 ? 1 : WHOLE ? bt : min(bt - c0, step);
        const int ni = cols * I;
        if (c0 > 0) {
            group_sync(G, gi);                              // the last columns' outputs were read
#pragma unroll
            for (int k = 0; k < kInputRegs; ++k) {
                const int i = lane + k * G;
                xr[k] = (i < ni) ? __ldg(xb + (size_t)c0 * I + i) : 0.0f;
            }
        }
#pragma unroll
        for (int k = 0; k < kInputRegs; ++k) {
            const int i = lane + k * G;
            if (i < ni) {
                if (T1) v[io[i]] = xr[k];
                else {
                    const int b = i / I, j = i - b * I;
                    v[((int)io[j] << lgT) + b] = xr[k];
                }
            }
        }
        for (int i = lane + kInputRegs * G; i < ni; i += G) {
            if (T1) v[io[i]] = __ldg(xb + i);
            else {
                const int b = i / I, j = i - b * I;
                v[((int)io[j] << lgT) + b] = __ldg(xb + (size_t)c0 * I + i);
            }
        }
        group_sync(G, gi);
        const bool col_ok = T1 || (lane & (step - 1)) < cols;
        const bool fast = (h0.w & 0xffffu) == kTraitsSumTanh;
        if constexpr (PAIRS) {
            if (fast) walk_pairs<true>(srec, v, G, gi, lane, cols);
            else walk_pairs<false>(srec, v, G, gi, lane, cols);
        } else if (fast) walk_levels<T1, true>(srec, v, G, gi, lane, lgT, lg_split, col_ok);
        else walk_levels<T1, false>(srec, v, G, gi, lane, lgT, lg_split, col_ok);
        for (int i = lane; i < cols * O; i += G) {
            if (T1) yb[i] = v[io[I + i]];
            else {
                const int b = i / O, j = i - b * O;
                yb[(size_t)c0 * O + i] = v[((int)io[I + j] << lgT) + b];
            }
        }
    }
    return true;
}

}  // namespace neat
