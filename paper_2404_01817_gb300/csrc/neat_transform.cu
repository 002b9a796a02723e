// Transformation stage of tensorized NEAT inference (Section 3.3): turns a
// genome's padded node/connection tensors (Section 3.1) into a record holding
// the layered Kahn order and, in place of the dense expanded-connection tensor
// C_exp, the enabled incoming edges of every node packed by destination
// position (layout in include/neat.h).
//
// Two forms build the same record:
//   transform_warp_kernel  genomes of at most 128 node rows and 512
//                          connection rows: one warp per genome, node sets
//                          as bit masks, no block barrier;
//   transform_block_kernel larger ones: one block per genome.
// Both keep all per-genome state in shared memory, stage the record there and
// write it with coalesced 16-byte stores.
#include <algorithm>

#include "neat_device.cuh"
#include "neat_internal.h"
#include "neat_hash.cuh"
#include "neat_trace.h"

namespace neat {
namespace {

struct TransformArgs {
    const float *nodes;
    const float *conns;
    uint8_t *out;
    uint32_t *status;
    size_t stride;
    int pop, I, O, N, C;
    int Np2, Cp2;   // powers of two >= N and >= max(C, 1)
    int recurrent;  // cycles allowed: no Kahn order, every present node in level 0 (row order)
    int record_bytes;   // warp form: shared memory of a warp's staged record
    int smem_per_warp;  // warp form: shared memory of a warp
};

__device__ __forceinline__ bool is_enum(float v, int n)
{
    return !isnan(v) && floorf(v) == v && v >= 0.0f && v < (float)n;
}

// Exclusive prefix sums of a[0..n) (n <= 1024) in chunks of 32: afterwards
// the prefix of i is a[i] + tot[i >> 5].  Every thread of the block calls it;
// ends with a barrier.
__device__ void chunked_exclusive_scan(int *a, int *tot, int n)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int ch = warp; ch * 32 < n; ch += nw) {
        const int i = ch * 32 + lane;
        const int x = (i < n) ? a[i] : 0;
        int incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (i < n) a[i] = incl - x;
        if (lane == 31) tot[ch] = incl;
    }
    __syncthreads();
    if (warp == 0) {
        const int x = (lane * 32 < n) ? tot[lane] : 0;
        int incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        tot[lane] = incl - x;
    }
    __syncthreads();
}

// A connection row's checked endpoints: kRowAbsent (no connection), kRowBad
// (a key is no key), else present.
enum : int { kRowAbsent = 0, kRowBad = 1, kRowPresent = 2 };
__device__ __forceinline__ int conn_row(const float4 row)
{
    if (isnan(row.x) || isnan(row.y) || isnan(row.z)) return kRowAbsent;
    return is_key(row.x) && is_key(row.y) ? kRowPresent : kRowBad;
}

__device__ __forceinline__ void write_error_record(uint8_t *rec, int n, uint32_t status)
{
    uint4 *h = reinterpret_cast<uint4 *>(rec);
    h[0] = make_uint4((unsigned)n, 0u, status, 0xffffu);
    h[1] = make_uint4(kHeaderBytes, kHeaderBytes, kHeaderBytes, kHeaderBytes);
}

struct RecordOffsets {
    uint32_t edge, level, io, used;
};
__device__ __forceinline__ RecordOffsets record_offsets(int n, int E, int nl, int nio)
{
    RecordOffsets o;
    o.edge = kHeaderBytes + kNodeBytes * (uint32_t)n;
    o.level = align16(o.edge + kEdgeBytes * (uint32_t)E);
    o.io = align16(o.level + 2u * (uint32_t)(nl + 1));
    o.used = align16(o.io + 2u * (uint32_t)nio);
    return o;
}

// ------------------------------------------------------------ warp form
//
// Rows r = lane + 32 i (i < RN) of the node tensor belong to lane; a set of
// node rows is RN 32-bit words.  Keys resolve through a 32-bit open-addressing
// table (key << 8 | row); a pair (source row, destination row) already seen
// shows in a bit matrix; the enabled sources of every node are a bit mask, so
// one Kahn level is a mask test per row and RN ballots, and a position is a
// population count.  So is an edge's place among its node's edges: each
// 32 connection rows leave a bit mask per destination row.  (Ranks from
// __match_any_sync instead cost one round per distinct value, 133 cycles for 8
// and 397 for 32: 70 us against 33 below.)
//
// Bound by instruction issue (61% of the slots; 2180 warp instructions per
// Ant-sized genome) at 28 warps per SM, the staged record and the tables
// taking 7.5 KB each.  10 000 Ant-sized genomes (50 node rows, 200 connection
// rows): 33 us, where a block of 128 threads per genome took 117 us and 9400
// instructions, most of them hash probes, barriers and a serial counting sort;
// 1001 genomes of 101 / 403 rows: 18 us against 29.  The bytes alone (42 MB
// read, 19 MB written) take 9 us at the measured copy rate.
constexpr int kWarpNodes = 128, kWarpConns = 512;

__host__ __device__ inline int warp_record_bytes(size_t record_bytes) { return (int)((record_bytes + 15) & ~(size_t)15); }

// A warp's shared memory, after its staged record: the key table, what starts
// as zeros, the rest (16-byte words where the warp clears them).  The matrix
// of pairs seen lives in the record region, which is free until the order is
// known.
struct WarpLayout {
    int zero, place, before, edge_of, total;   // byte offsets from the key table's start; zero .. place is cleared
};
__host__ __device__ inline WarpLayout warp_layout(int N, int C, int RN, int Np2)
{
    const int cw = (C + 31) / 32;
    WarpLayout l;
    l.zero = 8 * Np2;                                             // key table: 2 Np2 words
    l.place = (l.zero + 4 * N * RN + 4 * cw * N + 15) & ~15;      // enabled sources; edges into a row, a mask per
                                                                  // 32 connection rows
    l.before = l.place + 4 * N;                                   // position | first edge << 16
    l.edge_of = (l.before + 2 * cw * N + 7) & ~7;                 // edges into a row from earlier connection rows
    l.total = (l.edge_of + 8 * C + 15) & ~15;                     // (rows), weight
    return l;
}

// Connections to or from absent keys: the bit matrix cannot hold them, so
// their duplicates are found by a set of (in, out) pairs in the record region
// (free until the record is built; room for C + 4 pairs).
__device__ __noinline__ bool duplicate_dangling(const float4 *cn, int C, const uint32_t *tab, uint32_t mask, int shift,
                                                unsigned long long *set, int cap, int lane)
{
    for (int i = lane; i < cap; i += 32) set[i] = kFree;
    __syncwarp();
    bool dup = false;
    for (int c = lane; c < C; c += 32) {
        const float4 row = __ldg(cn + c);
        if (conn_row(row) != kRowPresent) continue;
        const uint32_t ki = (uint32_t)row.x, ko = (uint32_t)row.y;
        if (find32(tab, mask, shift, ki) >= 0 && find32(tab, mask, shift, ko) >= 0) continue;
        const unsigned long long pair = ((unsigned long long)ki << 24) | ko;
        int s = (int)(tslot(pair, 0xffffffffu) % (uint32_t)cap);
        for (int probe = 0; probe < cap; ++probe) {
            const unsigned long long old = atomicCAS(set + s, kFree, pair);
            if (old == kFree) break;
            if (old == pair) { dup = true; break; }
            s = (s + 1 == cap) ? 0 : s + 1;
        }
    }
    __syncwarp();
    return dup;
}

template <int RN>
__global__ void __launch_bounds__(128) transform_warp_kernel(const TransformArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = blockIdx.x * (blockDim.x >> 5) + warp;
    if (g >= a.pop) return;
    const int N = a.N, C = a.C, I = a.I, O = a.O;
    const unsigned below = (1u << lane) - 1u, all = 0xffffffffu;
    const uint32_t kmask = 2u * (uint32_t)a.Np2 - 1u;
    const int kshift = __clz(kmask);
    const int cw = (C + 31) >> 5;
    uint4 *rec4 = reinterpret_cast<uint4 *>(sm + (size_t)warp * a.smem_per_warp);
    unsigned char *srec = reinterpret_cast<unsigned char *>(rec4);
    unsigned char *work = srec + a.record_bytes;
    const WarpLayout lay = warp_layout(N, C, RN, a.Np2);
    uint32_t *ktab = reinterpret_cast<uint32_t *>(work);                      // [2 Np2]
    uint32_t *preds = reinterpret_cast<uint32_t *>(work + lay.zero);          // [N][RN] enabled sources of a row
    uint32_t *emask = preds + N * RN;                                         // [cw][N]
    uint32_t *place = reinterpret_cast<uint32_t *>(work + lay.place);         // [N]
    uint16_t *before = reinterpret_cast<uint16_t *>(work + lay.before);       // [cw][N]
    uint2 *edge_of = reinterpret_cast<uint2 *>(work + lay.edge_of);           // [C] (s | d << 8, or none), weight
    uint32_t *pairs = reinterpret_cast<uint32_t *>(srec);                     // [N][RN] sources seen, enabled or not
    const float *nd = a.nodes + (size_t)g * N * 5;
    const float4 *cn = reinterpret_cast<const float4 *>(a.conns + (size_t)g * C * 4);

    // the node rows and the first connection rows are in flight together
    float key[RN], bias[RN], resp[RN], agg[RN], act[RN];
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        const int r = lane + 32 * i;
        key[i] = __int_as_float(0x7fc00000);
        bias[i] = resp[i] = agg[i] = act[i] = 0.0f;
        if (r < N) {
            key[i] = __ldg(nd + r * 5);
            bias[i] = __ldg(nd + r * 5 + 1);
            resp[i] = __ldg(nd + r * 5 + 2);
            agg[i] = __ldg(nd + r * 5 + 3);
            act[i] = __ldg(nd + r * 5 + 4);
        }
    }
    constexpr int kAhead = 4;                                                // connection rows loaded ahead per lane
    float4 rows[kAhead];
    auto load_rows = [&](int base) {
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int c = base + 32 * j + lane;
            rows[j] = make_float4(__int_as_float(0x7fc00000), 0.0f, 0.0f, 0.0f);
            if (c < C) rows[j] = __ldg(cn + c);
        }
    };
    load_rows(0);
    {
        const uint4 free4 = make_uint4(all, all, all, all), zero4 = make_uint4(0u, 0u, 0u, 0u);
        uint4 *w4 = reinterpret_cast<uint4 *>(work);
        for (int i = lane; i < a.Np2 / 2; i += 32) w4[i] = free4;             // Np2 >= 4 wherever this form runs
        for (int i = (lay.zero >> 4) + lane; i < lay.place >> 4; i += 32) w4[i] = zero4;
        for (int i = lane; i < (4 * N * RN + 15) >> 4; i += 32) rec4[i] = zero4;
    }
    __syncwarp();

    // 1. node rows
    uint32_t st = 0, acts = 0, aggs = 0;
    uint32_t present[RN];
    int n = 0;
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        const int r = lane + 32 * i;
        bool here = false;
        if (!isnan(key[i])) {
            if (!is_key(key[i])) {
                st |= NEAT_G_BADKEY;
            } else {
                here = true;
                if (!is_enum(agg[i], 4) || !is_enum(act[i], 7)) st |= NEAT_G_BADENUM;
                else if (key[i] >= (float)I) {
                    acts |= 1u << (int)act[i];
                    aggs |= 1u << (int)agg[i];
                }
                if (isnan(bias[i]) || isnan(resp[i])) st |= NEAT_G_BADATTR;
                if (insert32(ktab, kmask, kshift, (uint32_t)key[i], (uint32_t)r)) st |= NEAT_G_DUPKEY;
            }
        }
        present[i] = __ballot_sync(all, here);
        n += __popc(present[i]);
    }
    __syncwarp();
    int io_row[RN];                                                          // I + O <= N: at most RN per lane
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        const int j = lane + 32 * i;
        io_row[i] = -1;
        if (j < I + O) {
            io_row[i] = find32(ktab, kmask, kshift, (uint32_t)j);
            if (io_row[i] < 0) st |= NEAT_G_MISSING_IO;
        }
    }

    // 2. connection rows; disabled ones only count towards duplicate pairs
    bool dangling = false;
    for (int base = 0; base < C; base += 32 * kAhead) {
        if (base) load_rows(base);
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            if (base + 32 * j >= C) break;                                   // uniform over the warp
            const int c = base + 32 * j + lane;
            const float4 row = rows[j];
            const int kind = conn_row(row);
            int s = -1, d = -1;
            bool active = false;
            if (kind == kRowBad) st |= NEAT_G_BADKEY;
            if (kind == kRowPresent) {
                const uint32_t ki = (uint32_t)row.x, ko = (uint32_t)row.y;
                s = find32(ktab, kmask, kshift, ki);
                d = find32(ktab, kmask, kshift, ko);
                const bool both = s >= 0 && d >= 0;
                const uint32_t bit = 1u << (s & 31);
                if (both) {
                    if (atomicOr(pairs + d * RN + (s >> 5), bit) & bit) st |= NEAT_G_DUPCONN;
                } else {
                    dangling = true;
                }
                if (row.z != 0.0f) {
                    if (isnan(row.w)) st |= NEAT_G_BADATTR;
                    if (!both) st |= NEAT_W_DANGLING;
                    else if (ko < (uint32_t)I) st |= NEAT_W_INTO_INPUT;
                    else {
                        active = true;
                        atomicOr(preds + d * RN + (s >> 5), bit);
                        atomicOr(emask + (c >> 5) * N + d, 1u << lane);
                    }
                }
            }
            if (c < C)
                edge_of[c] = make_uint2(active ? (uint32_t)s | ((uint32_t)d << 8) : kFree32, __float_as_uint(row.w));
        }
    }
    __syncwarp();
    if (__any_sync(all, dangling) &&
        duplicate_dangling(cn, C, ktab, kmask, kshift, reinterpret_cast<unsigned long long *>(srec), a.record_bytes / 8, lane))
        st |= NEAT_G_DUPCONN;

    // 3. layered Kahn on the masks; a row's position is its rank by (level,
    //    row).  The level starts go straight to their place in the record
    uint32_t pred[RN][RN];
    int pos[RN], deg[RN], E = 0;
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        const int r = lane + 32 * i;
        pos[i] = -1;
        deg[i] = 0;
        if (r < N)
            for (int k = 0; k < cw; ++k) {
                before[k * N + r] = (uint16_t)deg[i];
                deg[i] += __popc(emask[k * N + r]);
            }
        E += deg[i];
#pragma unroll
        for (int j = 0; j < RN; ++j) pred[i][j] = (r < N && !a.recurrent) ? preds[r * RN + j] : 0u;
    }
    E = __reduce_add_sync(all, E);
    uint16_t *lev = reinterpret_cast<uint16_t *>(srec + record_offsets(n, E, 0, 0).level);
    uint32_t left[RN];
    int placed = 0, nl = 0;
#pragma unroll
    for (int i = 0; i < RN; ++i) left[i] = present[i];
    while (placed < n) {
        uint32_t now[RN];
        int joined = 0;
#pragma unroll
        for (int i = 0; i < RN; ++i) {
            uint32_t wait = 0;
#pragma unroll
            for (int j = 0; j < RN; ++j) wait |= pred[i][j] & left[j];
            const bool ready = ((left[i] >> lane) & 1u) && wait == 0u;
            now[i] = __ballot_sync(all, ready);
            if (ready) pos[i] = placed + joined + __popc(now[i] & below);
            joined += __popc(now[i]);
        }
        if (joined == 0) break;                                              // a cycle
        if (lane == 0) lev[nl] = (uint16_t)placed;
        placed += joined;
        ++nl;
#pragma unroll
        for (int i = 0; i < RN; ++i) left[i] &= ~now[i];
    }
    st = __reduce_or_sync(all, st);
    if (placed < n) st |= NEAT_G_CYCLE;
    uint8_t *rec = a.out + (size_t)g * a.stride;
    if (a.status && lane == 0) a.status[g] = st;
    if (st & NEAT_G_ERROR_MASK) {
        if (lane == 0) write_error_record(rec, n, st);
        return;
    }

    // 4. first edges in position order
    const RecordOffsets o = record_offsets(n, E, nl, I + O);
#pragma unroll
    for (int i = 0; i < RN; ++i)
        if (pos[i] >= 0) place[pos[i]] = (uint32_t)deg[i];
    __syncwarp();
    int carry = 0;
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        const int p = lane + 32 * i;
        const int x = p < n ? (int)place[p] : 0;
        int incl = x;
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const int y = __shfl_up_sync(all, incl, k);
            if (lane >= k) incl += y;
        }
        if (p < n) place[p] = (uint32_t)(carry + incl - x);
        carry += __shfl_sync(all, incl, 31);
    }
    __syncwarp();
    int first[RN];
#pragma unroll
    for (int i = 0; i < RN; ++i) first[i] = pos[i] >= 0 ? (int)place[pos[i]] : 0;
    __syncwarp();

    // 5. node entries, (position, first edge) by row
    acts = __reduce_or_sync(all, acts);
    aggs = __reduce_or_sync(all, aggs);
    unsigned lead = (unsigned)n;                                             // leading positions that are inputs
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        if (pos[i] >= 0) {
            const int r = lane + 32 * i;
            const bool input = key[i] < (float)I;
            if (!input) lead = min(lead, (unsigned)pos[i]);
            place[r] = (uint32_t)pos[i] | ((uint32_t)first[i] << 16);
            rec4[2 + pos[i]] = make_uint4(__float_as_uint(bias[i]), __float_as_uint(resp[i]),
                                          (uint32_t)first[i] | ((uint32_t)deg[i] << 16),
                                          (input ? (uint32_t)kInputAct : (uint32_t)act[i]) |
                                              ((uint32_t)agg[i] << 8) | ((uint32_t)r << 16));
        }
    }
    lead = __reduce_min_sync(all, lead);
    __syncwarp();

    // 6. edges, input and output positions, header; the gaps hold zeros
    uint2 *edges = reinterpret_cast<uint2 *>(srec + o.edge);
    for (int c = lane; c < C; c += 32) {
        const uint2 e = edge_of[c];
        if (e.x == kFree32) continue;
        const int at = (c >> 5) * N + (int)(e.x >> 8);
        edges[(place[e.x >> 8] >> 16) + before[at] + __popc(emask[at] & below)] =
            make_uint2(e.y, place[e.x & 0xffu] & 0xffffu);
    }
    uint16_t *io = reinterpret_cast<uint16_t *>(srec + o.io);
#pragma unroll
    for (int i = 0; i < RN; ++i) {
        const int j = lane + 32 * i;
        if (j < I + O) io[j] = (uint16_t)(place[io_row[i]] & 0xffffu);
    }
    if (lane == 0) {
        lev[nl] = (uint16_t)n;
        if (E & 1) edges[E] = make_uint2(0u, 0u);
        const uint32_t ua = __popc(acts) == 1 ? (uint32_t)(__ffs(acts) - 1) : 0xffu;
        const uint32_t ug = __popc(aggs) == 1 ? (uint32_t)(__ffs(aggs) - 1) : 0xffu;
        rec4[0] = make_uint4((unsigned)n | ((unsigned)nl << 16), (unsigned)E, st, ua | (ug << 8) | (lead << 16));
        rec4[1] = make_uint4(o.used, o.edge, o.level, o.io);
    }
    if (lane < 8) {
        const uint32_t lend = o.level + 2u * (uint32_t)(nl + 1) + 2u * lane;
        if (lend < o.io) *reinterpret_cast<uint16_t *>(srec + lend) = 0;
        const uint32_t iend = o.io + 2u * (uint32_t)(I + O) + 2u * lane;
        if (iend < o.used) *reinterpret_cast<uint16_t *>(srec + iend) = 0;
    }
    __syncwarp();
    uint4 *out4 = reinterpret_cast<uint4 *>(rec);
    for (uint32_t i = lane; i < o.used / 16u; i += 32) out4[i] = rec4[i];
}

// ----------------------------------------------------------- block form
//
//   1. node rows: presence, key and attribute checks; keys into an
//      open-addressing table key -> lowest row;
//   2. connection rows: checks, endpoint lookup, duplicate pairs by insertion
//      of (source row, destination row) into a hash set (rows with an absent
//      end by their keys, in a pass of their own where there are any); an edge
//      takes the next free place among its destination's edges, in whatever
//      order they arrive, and the next place of a list of all edges;
//   3. layered Kahn: one pass over the active edges per level;
//   4. positions = rank of (level, row): every 32 rows count their levels,
//      the counts are summed over the rows before;
//   5. edges in (destination position, connection row) order: every edge
//      counts the edges of its destination with a lower row (a node has a few
//      edges); the rows of a destination with more than kHubEdges are sorted
//      first, by a warp through a bit per connection row, and searched;
//      the record staged in shared memory and written in one coalesced pass.
// Bound by issue and barriers (57% of the issue slots at 30 warps per SM).
// 4096 genomes of 500 / 2000 rows: 172 us in blocks of 256 threads (four per
// SM by 48 KB of shared memory each), against 411 us for the form whose one
// warp placed all edges in chunks of 32, waiting for each chunk's weights, and
// 253 us for that placement spread over 16 warps with match-based ranks.  608
// genomes of 1000 inputs, each feeding 8 outputs: 165 us (768 where every edge
// counts through its output's 1000; that warp 497); 2000 of 500 inputs and 4
// outputs 111 (347; 652).
constexpr int kHubEdges = 128;   // above 128 node rows the bits of one destination always fit two words per row

struct BlockLayout {
    size_t ktab, ptab, edge_of, ints, list, rows, io, total;
    int level, indeg, cnt, place, tot;       // offsets in `ints` (words)
};

__host__ __device__ inline size_t align_up(size_t x) { return (x + 15u) & ~(size_t)15u; }

__host__ __device__ inline BlockLayout block_layout(int N, int C, int nio, int Np2, int Cp2)
{
    BlockLayout l;
    const size_t nseg = (size_t)(N + 31) / 32;
    // the tables' memory is used again: the key table for the staged node
    // entries; the pair set for pairs with an absent end, the level counts,
    // then the staged edges
    const size_t pairs = 8u * (size_t)Cp2 + 16u, levels = 2u * nseg * (size_t)N;
    l.ktab = 0;
    l.ptab = 16u * (size_t)Np2;
    l.edge_of = align_up(l.ptab + (pairs > levels ? pairs : levels));
    l.ints = align_up(l.edge_of + 4u * (size_t)C);
    l.level = 0;
    l.indeg = N;
    l.cnt = 2 * N;
    l.place = 3 * N;
    l.tot = 4 * N + 1;
    l.list = l.ints + 4u * (size_t)(4 * N + 1 + 32);
    l.rows = l.list + 2u * (size_t)C;
    l.io = l.rows + 2u * (size_t)C;
    l.total = align_up(l.io + 2u * (size_t)nio);
    return l;
}

// Key -> lowest row (entries key << 32 | row), slots as in the warp form.
// True when the key was already present.
__device__ __forceinline__ bool insert64(unsigned long long *tab, uint32_t mask, int shift, uint32_t key, uint32_t row)
{
    const unsigned long long v = ((unsigned long long)key << 32) | row;
    uint32_t s = slot32(key, shift);
    for (;;) {                               // at most half the slots are taken
        const unsigned long long old = atomicCAS(tab + s, kFree, v);
        if (old == kFree) return false;
        if ((uint32_t)(old >> 32) == key) {
            atomicMin(tab + s, v);
            return true;
        }
        s = (s + 1u) & mask;
    }
}

__device__ __forceinline__ int find64(const unsigned long long *tab, uint32_t mask, int shift, uint32_t key)
{
    uint32_t s = slot32(key, shift);
    for (;;) {
        const unsigned long long v = tab[s];
        if (v == kFree) return -1;
        if ((uint32_t)(v >> 32) == key) return (int)(uint32_t)v;
        s = (s + 1u) & mask;
    }
}

// Duplicates among the present connections with an absent end, whose pairs
// have no rows: their keys in a set of `cap` >= C entries.
__device__ __noinline__ bool duplicate_dangling_block(const float4 *cn, int C, const unsigned long long *tab,
                                                      uint32_t mask, int shift, unsigned long long *set, int cap)
{
    for (int i = threadIdx.x; i < cap; i += blockDim.x) set[i] = kFree;
    __syncthreads();
    bool dup = false;
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        const float4 row = __ldg(cn + c);
        if (conn_row(row) != kRowPresent) continue;
        const uint32_t ki = (uint32_t)row.x, ko = (uint32_t)row.y;
        if (find64(tab, mask, shift, ki) >= 0 && find64(tab, mask, shift, ko) >= 0) continue;
        const unsigned long long pair = ((unsigned long long)ki << 24) | ko;
        int s = (int)(tslot(pair, 0xffffffffu) % (uint32_t)cap);
        for (int probe = 0; probe < cap; ++probe) {
            const unsigned long long old = atomicCAS(set + s, kFree, pair);
            if (old == kFree) break;
            if (old == pair) { dup = true; break; }
            s = (s + 1 == cap) ? 0 : s + 1;
        }
    }
    return dup;
}

// The connection rows list[0 .. m) in ascending order, by one warp; bits: a word
// for every 32 of the C connection rows.  (As a function of its own, or the search
// too: the call alone cost genomes without such a destination 1 to 5%.)
__device__ __forceinline__ void sort_rows(uint16_t *list, int m, uint32_t *bits, int C, int lane)
{
    const int words = (C + 31) >> 5;
    for (int i = lane; i < words; i += 32) bits[i] = 0u;
    __syncwarp();
    for (int i = lane; i < m; i += 32) atomicOr(bits + (list[i] >> 5), 1u << (list[i] & 31u));
    __syncwarp();
    int carry = 0;
    for (int base = 0; base < words; base += 32) {
        const uint32_t mine = base + lane < words ? bits[base + lane] : 0u;
        int incl = __popc(mine);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        int at = carry + incl - __popc(mine);
        for (uint32_t b = mine; b; b &= b - 1u) list[at++] = (uint16_t)(32 * (base + lane) + __ffs(b) - 1);
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
}

__global__ void __launch_bounds__(512, 2) transform_block_kernel(const TransformArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int g = blockIdx.x;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int N = a.N, C = a.C, I = a.I, O = a.O;
    const unsigned below = (1u << lane) - 1u, all = 0xffffffffu;
    const uint32_t kmask = 2u * (uint32_t)a.Np2 - 1u, pmask = 2u * (uint32_t)a.Cp2 - 1u;
    const int kshift = __clz(kmask), pshift = __clz(pmask);
    const BlockLayout lay = block_layout(N, C, I + O, a.Np2, a.Cp2);
    unsigned long long *ktab = reinterpret_cast<unsigned long long *>(sm + lay.ktab);
    uint32_t *ptab = reinterpret_cast<uint32_t *>(sm + lay.ptab);            // [2 Cp2] s | d << 10
    uint32_t *edge_of = reinterpret_cast<uint32_t *>(sm + lay.edge_of);      // [E] s | d << 10 | arrival << 20
    uint16_t *rows_of = reinterpret_cast<uint16_t *>(sm + lay.rows);         // [E] its connection row
    uint16_t *list = reinterpret_cast<uint16_t *>(sm + lay.list);            // [E] rows, those of a destination together
    int *ints = reinterpret_cast<int *>(sm + lay.ints);
    int *level = ints + lay.level;                                           // -2 absent, -1 unplaced
    int *indeg = ints + lay.indeg;
    int *cnt = ints + lay.cnt;                                               // [N] in-degree by row
    int *place = ints + lay.place;                                           // [N + 1] level starts, first edges, then
                                                                             // position | first edge << 16 by row
    int *tot = ints + lay.tot;                                               // [32] scan totals
    uint16_t *io_row = reinterpret_cast<uint16_t *>(sm + lay.io);

    __shared__ unsigned int st, acts_seen, aggs_seen, lead_inputs;
    __shared__ int n_present, n_edges, max_level, hubs;
    if (tid == 0) {
        hubs = 0;
        st = 0;
        acts_seen = 0;
        aggs_seen = 0;
        lead_inputs = (unsigned)NEAT_MAX_NODES;
        n_present = 0;
        n_edges = 0;
        max_level = -1;
    }
    const float *nd = a.nodes + (size_t)g * N * 5;
    const float4 *cn = reinterpret_cast<const float4 *>(a.conns + (size_t)g * C * 4);
    {
        const uint4 free4 = make_uint4(all, all, all, all);
        uint4 *k4 = reinterpret_cast<uint4 *>(ktab), *p4 = reinterpret_cast<uint4 *>(ptab);
        for (int i = tid; i < a.Np2; i += nt) k4[i] = free4;
        for (int i = tid; i < (a.Cp2 + 1) / 2; i += nt) p4[i] = free4;
    }
    __syncthreads();

    // 1. node rows (Section 3.1 encoding; an absent row is NaN)
    unsigned int lst = 0;
    for (int r = tid; r < N; r += nt) {
        const float k = __ldg(nd + r * 5);
        level[r] = -2;
        cnt[r] = 0;
        if (isnan(k)) continue;
        if (!is_key(k)) { lst |= NEAT_G_BADKEY; continue; }
        const float bias = __ldg(nd + r * 5 + 1), resp = __ldg(nd + r * 5 + 2);
        const float agg = __ldg(nd + r * 5 + 3), act = __ldg(nd + r * 5 + 4);
        if (!is_enum(agg, 4) || !is_enum(act, 7)) lst |= NEAT_G_BADENUM;
        else if (k >= (float)I) {
            atomicOr(&acts_seen, 1u << (int)act);
            atomicOr(&aggs_seen, 1u << (int)agg);
        }
        if (isnan(bias) || isnan(resp)) lst |= NEAT_G_BADATTR;
        level[r] = -1;
        if (insert64(ktab, kmask, kshift, (uint32_t)k, (uint32_t)r)) lst |= NEAT_G_DUPKEY;
        atomicAdd(&n_present, 1);
    }
    __syncthreads();
    const int n = n_present;
    for (int j = tid; j < I + O; j += nt) {
        const int r = find64(ktab, kmask, kshift, (uint32_t)j);
        io_row[j] = (uint16_t)max(r, 0);
        if (r < 0) lst |= NEAT_G_MISSING_IO;
    }

    // 2. connection rows; disabled ones only count towards duplicate pairs
    constexpr int kAhead = 4;                                                // rows loaded ahead per thread
    bool dangling = false;
    for (int base = warp * 32; base < C; base += nt * kAhead) {
        float4 rows[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int c = base + nt * j + lane;
            rows[j] = make_float4(__int_as_float(0x7fc00000), 0.0f, 0.0f, 0.0f);
            if (c < C) rows[j] = __ldg(cn + c);
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            if (base + nt * j >= C) break;                                   // uniform over the warp
            const float4 row = rows[j];
            const int kind = conn_row(row);
            bool active = false;
            int s = -1, d = -1;
            if (kind == kRowBad) lst |= NEAT_G_BADKEY;
            if (kind == kRowPresent) {
                const uint32_t ki = (uint32_t)row.x, ko = (uint32_t)row.y;
                s = find64(ktab, kmask, kshift, ki);
                d = find64(ktab, kmask, kshift, ko);
                const bool both = s >= 0 && d >= 0;
                if (both) {
                    const uint32_t v = (uint32_t)s | ((uint32_t)d << 10);
                    uint32_t at = slot32(v, pshift);
                    for (;;) {
                        const uint32_t old = atomicCAS(ptab + at, kFree32, v);
                        if (old == kFree32) break;
                        if (old == v) { lst |= NEAT_G_DUPCONN; break; }
                        at = (at + 1u) & pmask;
                    }
                } else {
                    dangling = true;
                }
                if (row.z != 0.0f) {
                    if (isnan(row.w)) lst |= NEAT_G_BADATTR;
                    if (!both) lst |= NEAT_W_DANGLING;
                    else if (ko < (uint32_t)I) lst |= NEAT_W_INTO_INPUT;
                    else active = true;
                }
            }
            __syncwarp();
            const unsigned on = __ballot_sync(all, active);
            if (on == 0u) continue;
            int at = 0;
            if (lane == 0) at = atomicAdd(&n_edges, __popc(on));
            at = __shfl_sync(all, at, 0) + __popc(on & below);
            if (active) {
                // an arrival of 1024 or more needs a duplicate pair: an error,
                // and the arrival is not used
                edge_of[at] = (uint32_t)s | ((uint32_t)d << 10) | (((uint32_t)atomicAdd(&cnt[d], 1) & 1023u) << 20);
                rows_of[at] = (uint16_t)(base + nt * j + lane);
            }
        }
    }
    const bool any_dangling = __syncthreads_or(dangling);
    if (any_dangling) {
        if (duplicate_dangling_block(cn, C, ktab, kmask, kshift, reinterpret_cast<unsigned long long *>(ptab), a.Cp2))
            lst |= NEAT_G_DUPCONN;
    }
    const int E = n_edges;

    // 3. layered Kahn: level 0 = present nodes without enabled incoming edges
    for (int r = tid; r < N; r += nt) {
        indeg[r] = cnt[r];
        if (level[r] == -1 && (cnt[r] == 0 || a.recurrent)) level[r] = 0;
    }
    // one barrier per level: it also tells every thread whether any node
    // joined the next level
    __syncthreads();
    for (int L = 0; !a.recurrent; ++L) {
        int joined = 0;
        for (int k = tid; k < E; k += nt) {
            const uint32_t e = edge_of[k];
            if (level[e & 1023u] == L) {
                const int d = (int)((e >> 10) & 1023u);
                if (atomicSub(&indeg[d], 1) == 1) {
                    level[d] = L + 1;
                    joined = 1;
                }
            }
        }
        if (!__syncthreads_or(joined)) break;
    }
    int lmax = -1;
    for (int r = tid; r < N; r += nt) {
        if (level[r] == -1) lst |= NEAT_G_CYCLE;
        lmax = max(lmax, level[r]);
    }
    lst = __reduce_or_sync(all, lst);
    lmax = __reduce_max_sync(all, lmax);
    if (lane == 0) {
        if (lst) atomicOr(&st, lst);
        atomicMax(&max_level, lmax);
    }
    __syncthreads();

    const uint32_t status = st;
    uint8_t *rec = a.out + (size_t)g * a.stride;
    if (tid == 0 && a.status) a.status[g] = status;
    if (status & NEAT_G_ERROR_MASK) {
        if (tid == 0) write_error_record(rec, n, status);
        return;
    }

    // 4. positions = rank of (level, row)
    const int nl = max_level + 1;
    const RecordOffsets o = record_offsets(n, E, nl, I + O);
    uint16_t *lcount = reinterpret_cast<uint16_t *>(ptab);                   // [ceil(N/32)][nl]
    const int nseg = (N + 31) / 32;
    for (int i = tid; i < nseg * nl; i += nt) lcount[i] = 0;
    __syncthreads();
    for (int ch = warp; ch < nseg; ch += nw) {
        const int r = ch * 32 + lane;
        const int lv = r < N ? level[r] : -2;
        const unsigned m = __match_any_sync(all, lv >= 0 ? lv : -1 - lane);
        if (lv >= 0 && lane == 31 - __clz(m)) lcount[ch * nl + lv] = (uint16_t)__popc(m);
        if (lv >= 0) indeg[r] = __popc(m & below);                           // rank within the 32 rows
    }
    __syncthreads();
    for (int L = tid; L < nl; L += nt) {
        int sum = 0;
        for (int ch = 0; ch < nseg; ++ch) {
            const int x = lcount[ch * nl + L];
            lcount[ch * nl + L] = (uint16_t)sum;
            sum += x;
        }
        place[L] = sum;
    }
    __syncthreads();
    chunked_exclusive_scan(place, tot, nl);
    uint16_t *lev_out = reinterpret_cast<uint16_t *>(rec + o.level);
    for (int L = tid; L <= nl; L += nt) lev_out[L] = (uint16_t)(L < nl ? place[L] + tot[L >> 5] : n);
    for (int r = tid; r < N; r += nt) {
        const int lv = level[r];
        if (lv >= 0) indeg[r] += place[lv] + tot[lv >> 5] + lcount[(r >> 5) * nl + lv];   // the row's position
    }
    __syncthreads();
    for (int r = tid; r < N; r += nt)
        if (level[r] >= 0) place[indeg[r]] = cnt[r];
    __syncthreads();
    chunked_exclusive_scan(place, tot, n);
    // first edge by row, over the levels (no longer needed but for presence)
    for (int r = tid; r < N; r += nt)
        if (level[r] >= 0) level[r] = place[indeg[r]] + tot[indeg[r] >> 5];
    __syncthreads();

    // 5. node entries and edges, staged; (position | first edge << 16) by row
    uint4 *nodes_st = reinterpret_cast<uint4 *>(ktab);
    unsigned lead = (unsigned)n;
    for (int r = tid; r < N; r += nt) {
        if (level[r] < 0) continue;
        const int p = indeg[r], first = level[r];
        place[r] = p | (first << 16);
        const float key = __ldg(nd + r * 5);
        const float bias = __ldg(nd + r * 5 + 1), resp = __ldg(nd + r * 5 + 2);
        const uint32_t agg = (uint32_t)__ldg(nd + r * 5 + 3);
        const bool input = key < (float)I;
        const uint32_t act = input ? (uint32_t)kInputAct : (uint32_t)__ldg(nd + r * 5 + 4);
        if (!input) lead = min(lead, (unsigned)p);                           // leading positions that are inputs
        if (cnt[r] > kHubEdges) hubs = 1;
        nodes_st[p] = make_uint4(__float_as_uint(bias), __float_as_uint(resp),
                                 (uint32_t)first | ((uint32_t)cnt[r] << 16), act | (agg << 8) | ((uint32_t)r << 16));
    }
    lead = __reduce_min_sync(all, lead);
    if (lane == 0) atomicMin(&lead_inputs, lead);
    __syncthreads();
    for (int k = tid; k < E; k += nt) {
        const uint32_t e = edge_of[k];
        list[(uint32_t)(place[(e >> 10) & 1023u] >> 16) + (e >> 20)] = rows_of[k];
    }
    __syncthreads();
    if (hubs) {
        // the levels and positions by row have been used: their memory holds the bits
        const int words = (C + 31) >> 5, sorters = min(nw, 2 * N / words);
        if (warp < sorters) {
            int seen = 0;
            for (int base = 0; base < N; base += 32) {
                unsigned m = __ballot_sync(all, base + lane < N && cnt[base + lane] > kHubEdges);
                for (; m; m &= m - 1u) {
                    const int d = base + __ffs(m) - 1;
                    if (seen++ % sorters == warp)
                        sort_rows(list + (place[d] >> 16), cnt[d], reinterpret_cast<uint32_t *>(ints) + warp * words, C, lane);
                }
            }
        }
        __syncthreads();
    }
    uint2 *edges_st = reinterpret_cast<uint2 *>(ptab);
    for (int k = tid; k < E; k += nt) {
        const uint32_t e = edge_of[k];
        const int c = rows_of[k];
        const float w = __ldg(a.conns + ((size_t)g * C + c) * 4 + 3);
        const int d = (int)((e >> 10) & 1023u);
        const int first = place[d] >> 16, m = cnt[d];
        int rank = 0;
        if (m > kHubEdges) {
            for (int above = m; rank + 1 < above;) {                         // list[first + rank] <= c < list[first + above]
                const int mid = (rank + above) >> 1;
                if ((int)list[first + mid] <= c) rank = mid; else above = mid;
            }
        } else {
            for (int i = 0; i < m; ++i) rank += (int)list[first + i] < c ? 1 : 0;
        }
        edges_st[first + rank] = make_uint2(__float_as_uint(w), (uint32_t)place[e & 1023u] & 0xffffu);
    }
    uint16_t *io_out = reinterpret_cast<uint16_t *>(rec + o.io);
    for (int j = tid; j < I + O; j += nt) io_out[j] = (uint16_t)(place[io_row[j]] & 0xffff);
    __syncthreads();
    uint4 *out4 = reinterpret_cast<uint4 *>(rec);
    for (int p = tid; p < n; p += nt) out4[2 + p] = nodes_st[p];
    const uint4 *e4 = reinterpret_cast<const uint4 *>(edges_st);
    uint4 *eo4 = reinterpret_cast<uint4 *>(rec + o.edge);
    for (int i = tid; i < E / 2; i += nt) eo4[i] = e4[i];
    if (tid == 0) {
        if (E & 1) reinterpret_cast<uint2 *>(rec + o.edge)[E - 1] = edges_st[E - 1];
        uint4 *h = reinterpret_cast<uint4 *>(rec);
        const uint32_t ua = __popc(acts_seen) == 1 ? (uint32_t)(__ffs(acts_seen) - 1) : 0xffu;
        const uint32_t ug = __popc(aggs_seen) == 1 ? (uint32_t)(__ffs(aggs_seen) - 1) : 0xffu;
        h[0] = make_uint4((unsigned)n | ((unsigned)nl << 16), (unsigned)E, status, ua | (ug << 8) | (lead_inputs << 16));
        h[1] = make_uint4(o.used, o.edge, o.level, o.io);
    }
}

int next_pow2(int x)
{
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

}  // namespace

}  // namespace neat

using namespace neat;

extern "C" size_t neat_record_stride(neat_dims d)
{
    return dims_ok(d) ? record_stride(d) : 0;
}

extern "C" size_t neat_transformed_bytes(int32_t pop, neat_dims d)
{
    if (!dims_ok(d) || pop < 0) return 0;
    return record_stride(d) * (size_t)pop;
}

static int transform_impl(const float *nodes_dev, const float *conns_dev, int32_t pop, neat_dims d,
                          void *transformed_dev, size_t transformed_bytes, uint32_t *status_dev, void *stream,
                          int recurrent)
{
    TraceRange trace_range(recurrent ? "neat_transform_recurrent" : "neat_transform");
    clear_error();
    if (!dims_ok(d)) return invalid("neat_transform: invalid dims");
    if (pop < 0) return invalid("neat_transform: pop < 0");
    if (pop == 0) return NEAT_OK;
    if (!nodes_dev || (!conns_dev && d.max_conns > 0) || !transformed_dev)
        return invalid("neat_transform: null pointer");
    if ((reinterpret_cast<uintptr_t>(conns_dev) & 15u) || (reinterpret_cast<uintptr_t>(transformed_dev) & 15u))
        return invalid("neat_transform: conns and transformed must be 16-byte aligned");
    const size_t stride = record_stride(d);
    if (transformed_bytes < stride * (size_t)pop) {
        set_error("neat_transform: transformed buffer too small");
        return NEAT_ENOMEM;
    }
    TransformArgs a;
    a.nodes = nodes_dev;
    a.conns = conns_dev;
    a.out = static_cast<uint8_t *>(transformed_dev);
    a.status = status_dev;
    a.stride = stride;
    a.pop = pop;
    a.I = d.num_inputs;
    a.O = d.num_outputs;
    a.N = d.max_nodes;
    a.C = d.max_conns;
    a.Np2 = next_pow2(a.N);
    a.Cp2 = next_pow2(a.C > 0 ? a.C : 1);
    a.recurrent = recurrent;
    a.record_bytes = a.smem_per_warp = 0;
    // a warp's masks grow with the square of the node rows and its chain with
    // the connection rows: up to 128 / 512 it beats a block (18 against 29 us
    // at 101 / 403), beyond, a warp's shared memory leaves too few per SM
    if (a.N <= kWarpNodes && a.C <= kWarpConns) {
        const int rn = a.N <= 32 ? 1 : (a.N <= 64 ? 2 : 4);
        a.record_bytes = warp_record_bytes(record_max_bytes(a.I, a.O, a.N, a.C));
        a.Np2 = std::max(a.Np2, 4);                        // the key table is cleared by 16-byte words
        a.smem_per_warp = a.record_bytes + warp_layout(a.N, a.C, rn, a.Np2).total;
        // four genomes per block; one where the population leaves SMs idle
        const int warps = pop > 4 * 152 ? 4 : 1;
        const size_t smem = (size_t)warps * a.smem_per_warp;
        auto kern = rn == 1 ? transform_warp_kernel<1> : (rn == 2 ? transform_warp_kernel<2> : transform_warp_kernel<4>);
        int rc = allow_dynamic_smem(reinterpret_cast<const void *>(kern), smem, "neat_transform: shared memory per block");
        if (rc) return rc;
        kern<<<(pop + warps - 1) / warps, 32 * warps, smem, as_stream(stream)>>>(a);
    } else {
        const int threads = (a.N <= 512 && a.C <= 4096) ? 256 : 512;
        const size_t smem = block_layout(a.N, a.C, a.I + a.O, a.Np2, a.Cp2).total;
        int rc = allow_dynamic_smem(reinterpret_cast<const void *>(transform_block_kernel), smem,
                                    "neat_transform: shared memory per block");
        if (rc) return rc;
        transform_block_kernel<<<pop, threads, smem, as_stream(stream)>>>(a);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_transform: launch");
    return NEAT_OK;
}

extern "C" int neat_transform(const float *nodes_dev, const float *conns_dev, int32_t pop, neat_dims d,
                              void *transformed_dev, size_t transformed_bytes, uint32_t *status_dev,
                              void *stream)
{
    return transform_impl(nodes_dev, conns_dev, pop, d, transformed_dev, transformed_bytes, status_dev, stream, 0);
}

extern "C" int neat_transform_recurrent(const float *nodes_dev, const float *conns_dev, int32_t pop, neat_dims d,
                                        void *transformed_dev, size_t transformed_bytes, uint32_t *status_dev,
                                        void *stream)
{
    return transform_impl(nodes_dev, conns_dev, pop, d, transformed_dev, transformed_bytes, status_dev, stream, 1);
}
