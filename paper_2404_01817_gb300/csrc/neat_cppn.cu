// CPPN query of a HyperNEAT substrate (the CPPN / HyperNEAT extensions of
// Section 4.3): every CPPN genome is evaluated at every (source, target) node
// pair of consecutive substrate layers, with inputs (x_s, y_s, x_t, y_t, 1),
// and its output becomes the connection weight, zeroed when |w| < threshold.
//
// Substrate: `layers` layers of res x res nodes on the grid -1 + 2 i / (res-1)
// of [-1,1]^2, node index = res * iy + ix.  Output layout
// weights[genome][block][source][target], block l joining layer l to l+1.
//
// Every block of the weights has the same value for the same (source, target)
// pair: the layers share one grid and a query holds no layer coordinate.  Each
// pair is evaluated once and its weight written to every block.
//
// GB300 mapping: a block takes (genome, chunk of pairs), bulk-copies the
// genome's record into shared memory once (TMA + mbarrier), and lists the
// nodes that the output depends on, walking the levels back from it; only
// these are evaluated and have a row in the value tile.  Each thread evaluates
// 4 consecutive pairs at a time in its own four adjacent columns.  Node and
// edge reads are the same for the whole warp (broadcasts), the four values of
// a source are one 16-byte read, and the sums run as packed pairs
// (fma.rn.f32x2: two IEEE fused multiply-adds per instruction, each rounded as
// the scalar one, so the bits are those of every other path).  No barrier is
// needed between nodes.  A block has as many threads at work as its tile has
// room for: 256 up to 16 rows, 128 at 32.
//
// Bound by issue (66% of the slots at 22 warps per SM): the edges' shared
// memory reads, the dispatches and the transcendentals; the only traffic is 4
// bytes written per weight.  1000 genomes (up to 32 nodes, 96 connections), 3
// layers of 16 x 16: 0.33 to 0.38 ms by population, the benchmark's 0.41 (perf/
// cases.py seed 5: 0.36 ms and 0.23 G warp instructions, 1.45 TB/s written).
// One pair per thread and column, every node, every block evaluated: 2.70 ms
// and 3.07 G; four columns and one evaluation per pair, without the list of
// needed nodes and with a fixed 128 threads: 1.29 ms and 0.75 G at 12 warps.
#include <algorithm>

#include "neat_device.cuh"
#include "neat_internal.h"
#include "neat_trace.h"
#include "neat_item.cuh"

namespace neat {
namespace {

constexpr int kCppnThreads = 256;
constexpr int kCppnMaxNodes = 256;   // above what shared memory admits (195)

struct CppnArgs {
    const uint8_t *rec;
    size_t stride;
    float *out;
    int pop, N;
    int res, blocks;         // weight blocks (layers - 1)
    int pairs;               // res^4: weights per block
    int chunk, chunks;       // pairs per thread block, thread blocks per genome
    float threshold;
    int rec_words;           // 16-byte words of the record region
    int edge_words;          // 16-byte words of the widened edges (0: edges stay as they are in the record)
    int tile_bytes;          // value tile
    int use_xy;              // node coordinate table in shared memory (res^2 <= 4096)
    int vec_out;             // weights written 16 bytes at a time
};

__device__ unsigned int g_cppn_error;

// An edge as staged: weight (twice, when widened) and the byte offset of its
// source's row of the value tile.
template <bool WIDE>
struct Edge;
template <>
struct Edge<true> {
    using T = uint4;
    static __device__ __forceinline__ f2 ww(const uint4 &e) { return pack2(__uint_as_float(e.x), __uint_as_float(e.y)); }
    static __device__ __forceinline__ float w(const uint4 &e) { return __uint_as_float(e.x); }
    static __device__ __forceinline__ uint32_t at(const uint4 &e) { return e.z; }
};
template <>
struct Edge<false> {
    using T = uint2;
    static __device__ __forceinline__ f2 ww(const uint2 &e) { return pack2(__uint_as_float(e.x), __uint_as_float(e.x)); }
    static __device__ __forceinline__ float w(const uint2 &e) { return __uint_as_float(e.x); }
    static __device__ __forceinline__ uint32_t at(const uint2 &e) { return e.y; }
};

// The thread's four values of the tile row at byte offset `at` (v: the
// thread's columns).
struct Four {
    f2 lo, hi;
};
__device__ __forceinline__ Four load4(const char *v, uint32_t at)
{
    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(v + at);
    return Four{x.x, x.y};
}

// Sums of a node's edges for the thread's four columns: edge i into partial
// i mod 4 from +0 with fused multiply-adds, then (p0 + p1) + (p2 + p3), the
// order of every evaluation path.
template <bool WIDE, int EC>
__device__ __forceinline__ Four sum_fixed(const typename Edge<WIDE>::T *__restrict__ e, const char *__restrict__ v)
{
    Four q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = Four{0ull, 0ull};
#pragma unroll
    for (int i = 0; i < EC; ++i) {
        const auto t = e[i];
        const f2 w = Edge<WIDE>::ww(t);
        const Four x = load4(v, Edge<WIDE>::at(t));
        q[i & 3].lo = fma2(w, x.lo, q[i & 3].lo);
        q[i & 3].hi = fma2(w, x.hi, q[i & 3].hi);
    }
    return Four{add2(add2(q[0].lo, q[1].lo), add2(q[2].lo, q[3].lo)),
                add2(add2(q[0].hi, q[1].hi), add2(q[2].hi, q[3].hi))};
}

template <bool WIDE>
__device__ __forceinline__ Four sum_any(const typename Edge<WIDE>::T *__restrict__ e, int ec, const char *__restrict__ v)
{
    Four q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = Four{0ull, 0ull};
    for (int i = 0; i < ec; i += 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k >= ec) break;                        // uniform over the block
            const auto t = e[i + k];
            const f2 w = Edge<WIDE>::ww(t);
            const Four x = load4(v, Edge<WIDE>::at(t));
            q[k].lo = fma2(w, x.lo, q[k].lo);
            q[k].hi = fma2(w, x.hi, q[k].hi);
        }
    }
    return Four{add2(add2(q[0].lo, q[1].lo), add2(q[2].lo, q[3].lo)),
                add2(add2(q[0].hi, q[1].hi), add2(q[2].hi, q[3].hi))};
}

template <bool WIDE>
__device__ __forceinline__ Four sum_edges(const typename Edge<WIDE>::T *__restrict__ e, int ec,
                                          const char *__restrict__ v)
{
    switch (ec) {
    case 0: return Four{0ull, 0ull};
    case 1: return sum_fixed<WIDE, 1>(e, v);
    case 2: return sum_fixed<WIDE, 2>(e, v);
    case 3: return sum_fixed<WIDE, 3>(e, v);
    case 4: return sum_fixed<WIDE, 4>(e, v);
    case 5: return sum_fixed<WIDE, 5>(e, v);
    case 6: return sum_fixed<WIDE, 6>(e, v);
    case 7: return sum_fixed<WIDE, 7>(e, v);
    case 8: return sum_fixed<WIDE, 8>(e, v);
    default: return sum_any<WIDE>(e, ec, v);
    }
}

// Products or maxima, the same partials.
template <bool WIDE, uint32_t AGG>
__device__ __forceinline__ void fold_edges(const typename Edge<WIDE>::T *__restrict__ e, int ec,
                                           const char *__restrict__ v, float out[4])
{
    float q[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) q[k][j] = agg_identity(AGG);
    for (int i = 0; i < ec; i += 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k >= ec) break;
            const auto t = e[i + k];
            const float w = Edge<WIDE>::w(t);
            const float4 x = *reinterpret_cast<const float4 *>(v + Edge<WIDE>::at(t));
            q[k][0] = agg_step(AGG, q[k][0], w, x.x);
            q[k][1] = agg_step(AGG, q[k][1], w, x.y);
            q[k][2] = agg_step(AGG, q[k][2], w, x.z);
            q[k][3] = agg_step(AGG, q[k][3], w, x.w);
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        out[j] = agg_combine(AGG, agg_combine(AGG, q[0][j], q[1][j]), agg_combine(AGG, q[2][j], q[3][j]));
}

// NaN for the pairs [q0, qend) of every weight block of a genome.
__device__ __forceinline__ void write_nan(float *out, const CppnArgs &a, int q0, int qend)
{
    for (int l = 0; l < a.blocks; ++l)
        for (int q = q0 + (int)threadIdx.x; q < qend; q += blockDim.x)
            out[(size_t)l * a.pairs + q] = __int_as_float(0x7fc00000);
}

// The needed nodes of a record with one level, which tells nothing of the order
// (neat_transform_recurrent's: positions follow node rows): a warp's passes over
// the nodes marked last (1; 2 once their sources are), until none is added.  True,
// in some lane, when a node does not come after the nodes it reads.
__device__ __noinline__ bool close_over_edges(uint8_t *need, const uint4 *nodes, const uint2 *packed, int n_nodes, int lane)
{
    bool unordered = false;
    for (bool more = true; more;) {
        more = false;
        for (int p = lane; p < n_nodes; p += 32) {
            if (need[p] != 1) continue;
            need[p] = 2;
            const uint32_t z = nodes[p].z;
            for (uint32_t i = z & 0xffffu, e = i + (z >> 16); i < e; ++i) {
                const uint32_t src = packed[i].y;
                if (need[src] == 0) need[src] = 1;
                unordered |= (int)src >= p && (nodes[src].w & 0xffu) != kInputAct;
                more = true;
            }
        }
        __syncwarp();
        more = __any_sync(0xffffffffu, more);
    }
    return unordered;
}

template <bool WIDE>
__global__ void __launch_bounds__(kCppnThreads) cppn_kernel(const CppnArgs a)
{
    extern __shared__ __align__(16) uint4 smem[];
    __shared__ uint64_t bar_mem;
    __shared__ float coord[256];
    __shared__ uint8_t need[kCppnMaxNodes], slot_of[kCppnMaxNodes];
    __shared__ int failed, n_prog;                         // n_prog: -1 where the rows are in no order to follow
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int g = (int)(blockIdx.x / a.chunks);
    const int q0 = (int)(blockIdx.x - (unsigned)g * a.chunks) * a.chunk;
    uint4 *srec = smem;
    uint4 *prog = srec + a.rec_words;                      // [N] the nodes to evaluate
    uint4 *wide = prog + a.N;
    char *tile = reinterpret_cast<char *>(wide + a.edge_words);
    float2 *nodexy = reinterpret_cast<float2 *>(tile + a.tile_bytes);   // (x, y) of node i
    const uint32_t bar = smem_addr(&bar_mem);
    const uint8_t *grec = a.rec + (size_t)g * a.stride;
    if (tid == 0) {
        const uint32_t bytes = min(align16(__ldg(reinterpret_cast<const uint32_t *>(grec) + 4)),
                                   (uint32_t)a.rec_words * 16u);
        failed = 0;
        mbar_init(bar, 1);
        mbar_arrive_expect_tx(bar, bytes);
        bulk_g2s(smem_addr(srec), grec, bytes, bar);
    }
    for (int i = tid; i < a.res; i += nt) coord[i] = (float)(-1.0 + 2.0 * (double)i / (double)(a.res - 1));
    for (int i = tid; i < kCppnMaxNodes; i += nt) need[i] = 0;
    __syncthreads();
    const int rr = a.res * a.res;
    if (a.use_xy)
        for (int i = tid; i < rr; i += nt) nodexy[i] = make_float2(coord[i % a.res], coord[i / a.res]);
    if (!mbar_wait(bar, 0)) failed = 1;
    __syncthreads();
    float *out = a.out + (size_t)g * a.blocks * (size_t)a.pairs;
    const int qend = min(a.pairs, q0 + a.chunk);
    const uint4 h0 = srec[0], h1 = srec[1];
    if (failed || (h0.z & NEAT_G_ERROR_MASK)) {
        if (failed && tid == 0) atomicOr(&g_cppn_error, kErrWaitExpired);
        if (failed) mbar_wait(bar, 0);                     // let the copy land before the block's memory is released
        write_nan(out, a, q0, qend);
        return;
    }
    const int n_nodes = (int)(h0.x & 0xffffu), n_levels = (int)(h0.x >> 16), n_edges = (int)h0.y;
    const uint4 *nodes = srec + 2;
    uint2 *packed = reinterpret_cast<uint2 *>(reinterpret_cast<char *>(srec) + h1.y);
    const uint16_t *lev = reinterpret_cast<const uint16_t *>(reinterpret_cast<const char *>(srec) + h1.z);
    const uint16_t *io = reinterpret_cast<const uint16_t *>(reinterpret_cast<const char *>(srec) + h1.w);
    const int p_out = io[5];
    if (tid < 32) {
        // the nodes that the output depends on, from the last level back
        if (lane == 0) need[p_out] = 1;
        __syncwarp();
        const bool unordered = n_levels == 1 && close_over_edges(need, nodes, packed, n_nodes, lane);
        for (int l = n_levels - 1; l > 0; --l) {
            for (int p = lev[l] + lane; p < lev[l + 1]; p += 32)
                if (need[p]) {
                    const uint32_t z = nodes[p].z;
                    for (uint32_t i = z & 0xffffu, e = i + (z >> 16); i < e; ++i) need[packed[i].y] = 1;
                }
            __syncwarp();
        }
        // tile rows: the inputs, then the nodes to evaluate in their order
        if (lane < 5) slot_of[io[lane]] = (uint8_t)lane;
        int count = 0;
        for (int p = lane; p - lane < n_nodes; p += 32) {
            const uint4 ne = p < n_nodes ? nodes[p] : make_uint4(0u, 0u, 0u, (uint32_t)kInputAct);
            const bool used = (ne.w & 0xffu) != kInputAct && need[p];
            const unsigned m = __ballot_sync(0xffffffffu, used);
            if (used) {
                const int k = count + __popc(m & ((1u << lane) - 1u));
                prog[k] = ne;
                slot_of[p] = (uint8_t)(5 + k);
            }
            count += __popc(m);
        }
        const unsigned none = __ballot_sync(0xffffffffu, unordered);
        if (lane == 0) n_prog = none ? -1 : count;
    }
    __syncthreads();
    const int np = n_prog;
    if (np < 0) {
        write_nan(out, a, q0, qend);
        return;
    }
    // four columns per thread, as many threads as the rows leave room for
    const int active = min(nt, (a.tile_bytes / (16 * (5 + np))) & ~31);
    const int row = 16 * active;                           // bytes of a tile row
    // sources become byte offsets of their rows (a node that is not evaluated
    // has edges no one reads)
    for (int i = tid; i < n_edges; i += nt) {
        const uint2 e = packed[i];
        const uint32_t at = (uint32_t)(slot_of[e.y] * row);
        if (WIDE) wide[i] = make_uint4(e.x, e.x, at, 0u);
        else packed[i].y = at;
    }
    __syncthreads();
    if (tid >= active) return;
    using E = typename Edge<WIDE>::T;
    const E *edges = WIDE ? reinterpret_cast<const E *>(wide) : reinterpret_cast<const E *>(packed);
    char *v = tile + 16 * tid;                             // the thread's columns
    *reinterpret_cast<float4 *>(v + 4 * row) = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
    for (int q = q0 + 4 * tid; q < qend; q += 4 * active) {
        {
            int s = q / rr, t = q - s * rr;
            float2 ps[4], pt[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (a.use_xy) {
                    ps[j] = nodexy[s];
                    pt[j] = nodexy[t];
                } else {
                    ps[j] = make_float2(coord[s % a.res], coord[s / a.res]);
                    pt[j] = make_float2(coord[t % a.res], coord[t / a.res]);
                }
                if (++t == rr) {
                    t = 0;
                    if (s + 1 < rr) ++s;                   // past the last pair: any source will do
                }
            }
            *reinterpret_cast<float4 *>(v) = make_float4(ps[0].x, ps[1].x, ps[2].x, ps[3].x);
            *reinterpret_cast<float4 *>(v + row) = make_float4(ps[0].y, ps[1].y, ps[2].y, ps[3].y);
            *reinterpret_cast<float4 *>(v + 2 * row) = make_float4(pt[0].x, pt[1].x, pt[2].x, pt[3].x);
            *reinterpret_cast<float4 *>(v + 3 * row) = make_float4(pt[0].y, pt[1].y, pt[2].y, pt[3].y);
        }
        char *vp = v + 5 * row;
        float4 y = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        uint4 next = prog[0];
        for (int p = 0; p < np; ++p, vp += row) {
            const uint4 ne = next;
            next = prog[min(p + 1, np - 1)];               // read ahead of this node's sums
            const uint32_t act = ne.w & 0xffu, agg = (ne.w >> 8) & 0xffu;
            const int ec = (int)(ne.z >> 16);
            const E *e = edges + (ne.z & 0xffffu);
            f2 lo, hi;
            if (agg == kAggSum) {
                const Four sum = sum_edges<WIDE>(e, ec, v);
                lo = sum.lo;
                hi = sum.hi;
            } else {
                float x[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (ec > 0) {
                    if (agg == kAggProduct) fold_edges<WIDE, kAggProduct>(e, ec, v, x);
                    else if (agg == kAggMax) fold_edges<WIDE, kAggMax>(e, ec, v, x);
                    else {
                        const Four sum = sum_edges<WIDE>(e, ec, v);
                        const float2 l2 = unpack2(sum.lo), h2 = unpack2(sum.hi);
                        x[0] = l2.x / (float)ec;
                        x[1] = l2.y / (float)ec;
                        x[2] = h2.x / (float)ec;
                        x[3] = h2.y / (float)ec;
                    }
                }
                lo = pack2(x[0], x[1]);
                hi = pack2(x[2], x[3]);
            }
            const f2 rr2 = pack2(__uint_as_float(ne.y), __uint_as_float(ne.y));
            const f2 bb2 = pack2(__uint_as_float(ne.x), __uint_as_float(ne.x));
            const float2 z0 = unpack2(fma2(rr2, lo, bb2)), z1 = unpack2(fma2(rr2, hi, bb2));
            switch (act) {                                 // one dispatch for the four columns
            case 1: y = make_float4(activate(1, z0.x), activate(1, z0.y), activate(1, z1.x), activate(1, z1.y)); break;
            case 2: y = make_float4(activate(2, z0.x), activate(2, z0.y), activate(2, z1.x), activate(2, z1.y)); break;
            case 3: y = make_float4(activate(3, z0.x), activate(3, z0.y), activate(3, z1.x), activate(3, z1.y)); break;
            case 4: y = make_float4(activate(4, z0.x), activate(4, z0.y), activate(4, z1.x), activate(4, z1.y)); break;
            case 5: y = make_float4(activate(5, z0.x), activate(5, z0.y), activate(5, z1.x), activate(5, z1.y)); break;
            case 6: y = make_float4(activate(6, z0.x), activate(6, z0.y), activate(6, z1.x), activate(6, z1.y)); break;
            default: y = make_float4(z0.x, z0.y, z1.x, z1.y);
            }
            *reinterpret_cast<float4 *>(vp) = y;
        }
        // the output is the last node that anything needed is evaluated for
        float4 w = y;
        w.x = fabsf(w.x) < a.threshold ? 0.0f : w.x;
        w.y = fabsf(w.y) < a.threshold ? 0.0f : w.y;
        w.z = fabsf(w.z) < a.threshold ? 0.0f : w.z;
        w.w = fabsf(w.w) < a.threshold ? 0.0f : w.w;
        for (int l = 0; l < a.blocks; ++l) {
            float *o = out + (size_t)l * a.pairs + q;
            if (a.vec_out) {
                *reinterpret_cast<float4 *>(o) = w;
            } else {
                o[0] = w.x;
                if (q + 1 < qend) o[1] = w.y;
                if (q + 2 < qend) o[2] = w.z;
                if (q + 3 < qend) o[3] = w.w;
            }
        }
    }
}

}  // namespace
}  // namespace neat

using namespace neat;

extern "C" int neat_cppn_query(const void *transformed_dev, int32_t pop, neat_dims d, neat_substrate sub,
                               float threshold, float *weights_dev, void *stream)
{
    TraceRange trace_range("neat_cppn_query");
    clear_error();
    if (!dims_ok(d)) return invalid("neat_cppn_query: invalid dims");
    if (d.num_inputs != 5 || d.num_outputs != 1)
        return invalid("neat_cppn_query: a CPPN has 5 inputs (x_s, y_s, x_t, y_t, 1) and 1 output");
    if (sub.resolution < 2 || sub.resolution > 181 || sub.layers < 2)
        return invalid("neat_cppn_query: substrate resolution must be in 2..181 and layers >= 2");
    if (pop < 0) return invalid("neat_cppn_query: pop < 0");
    if (pop == 0) return NEAT_OK;
    if (!transformed_dev || !weights_dev) return invalid("neat_cppn_query: null pointer");
    if (reinterpret_cast<uintptr_t>(transformed_dev) & 15u)
        return invalid("neat_cppn_query: transformed must be 16-byte aligned");
    CppnArgs a;
    a.rec = static_cast<const uint8_t *>(transformed_dev);
    a.stride = record_stride(d);
    a.out = weights_dev;
    a.pop = pop;
    a.N = d.max_nodes;
    a.res = sub.resolution;
    a.blocks = sub.layers - 1;
    const long r2 = (long)sub.resolution * sub.resolution;
    a.pairs = (int)(r2 * r2);                              // at most 181^4 < 2^31
    // pairs per block: fewer prologues, but about eight blocks per resident
    // one (three per SM) before blocks grow
    a.chunk = 16384;
    while (a.chunk > 1024 && (long)pop * ((a.pairs + a.chunk - 1) / a.chunk) < 8L * 3 * 152) a.chunk >>= 1;
    a.chunks = (a.pairs + a.chunk - 1) / a.chunk;
    a.threshold = threshold;
    a.rec_words = (int)(record_max_bytes(5, 1, d.max_nodes, d.max_conns) / 16);
    a.use_xy = (r2 <= 4096) ? 1 : 0;
    a.vec_out = (a.pairs % 4 == 0 && (reinterpret_cast<uintptr_t>(weights_dev) & 15u) == 0) ? 1 : 0;
    // the value tile: 64 KB (three blocks per SM), or 128 columns of every
    // node where that is more; edges widened where there is room
    a.tile_bytes = std::max(64 * 1024, 512 * d.max_nodes);
    const size_t limit = 200u * 1024u;
    auto smem_for = [&](bool wide) {
        return 16u * ((size_t)a.rec_words + (size_t)d.max_nodes + (wide ? (size_t)d.max_conns : 0u)) +
               (size_t)a.tile_bytes + (a.use_xy ? 8u * (size_t)r2 : 0u);
    };
    if ((size_t)a.rec_words * 16 + 1024u * (size_t)d.max_nodes + (a.use_xy ? 8u * (size_t)r2 : 0u) > limit)
        return invalid("neat_cppn_query: genome too large for one block (max_nodes <= 160)");
    const bool wide = smem_for(true) <= limit;
    a.edge_words = wide ? d.max_conns : 0;
    const size_t smem = smem_for(wide);
    const long blocks = (long)pop * a.chunks;
    if (blocks > 0x7fffffffL) return invalid("neat_cppn_query: too many queries");
    auto kern = wide ? cppn_kernel<true> : cppn_kernel<false>;
    int rc = allow_dynamic_smem(reinterpret_cast<const void *>(kern), smem, "neat_cppn_query: shared memory per block");
    if (rc) return rc;
    kern<<<(unsigned)blocks, kCppnThreads, smem, as_stream(stream)>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_cppn_query: launch");
    return NEAT_OK;
}

namespace neat {
int read_cppn_error(unsigned int *v, int clear)
{
    cudaError_t e = cudaMemcpyFromSymbol(v, g_cppn_error, sizeof(*v));
    if (e != cudaSuccess) return cuda_fail(e, "cppn error word: read");
    if (clear) {
        const unsigned int zero = 0;
        e = cudaMemcpyToSymbol(g_cppn_error, &zero, sizeof(zero));
        if (e != cudaSuccess) return cuda_fail(e, "cppn error word: clear");
    }
    return NEAT_OK;
}
}  // namespace neat
