// Batched evaluation of several populations in one persistent launch per
// step (the data-parallel forward of Section 3.3 over uneven populations).
//
// Every call first copies the records to compact ones, without the nodes that
// no output depends on (compact_kernel), where that saves more than it costs.
//
// Plan creation (host, once): the headers of the records to be evaluated are
// read back, each population is split into size buckets by node count (powers
// of two from 16), and each bucket gets a launch shape: group size G, tile T
// and split (threads per node), chosen by a heuristic or timed on the plan's
// own data.  A bucket's work is cut into block items of `gpc` work items each
// (gpc = threads per block / G); block items are numbered bucket by bucket,
// largest records first, so the most expensive items start first.
//
// Kernel (per step): persistent blocks pull block items from a per-step
// device counter.  For a block item every group of G threads bulk-copies its
// genome's record into its shared-memory region (TMA, completion on an
// mbarrier) and then runs the same item evaluation as the single-population
// kernel (run_item), so results match neat_forward bit for bit.
//
// Four populations of 2048 genomes (up to 16, 64, 256 and 1024 nodes), 64
// inputs each: 181 us a step with compact records (509 us without), the copies'
// 36 us included.
#include <algorithm>
#include <climits>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "neat_device.cuh"
#include "neat_internal.h"
#include "neat_trace.h"
#include "neat_item.cuh"

namespace neat {
namespace {

__device__ unsigned int g_plan_error;

// ---- compact records
//
// Nothing reads a node that reaches no output.  Before its steps, a plan
// copies every record to a workspace of its own with only the nodes that the
// outputs depend on (and the inputs), in the record format: positions, levels,
// edge sources and input/output lists renumbered, every remaining node's edges
// in their order, so its value has the same bits.  In random graphs a large
// genome shrinks most: of 1024 node rows and 4 outputs, 23% of the nodes and
// 12% of the edges remain, of 64 rows 54% and 44%.  The copy is made anew by
// every call from the records as they are then; only the launch shapes come
// from the records at creation.
//
// One warp per genome, straight from memory: marks the needed nodes from the
// outputs back, ranks them by population counts, writes the copy.  Bound by
// the latency of a chain of L2 reads per round, hidden by the warps of other
// genomes.  (Marking inside
// the forward kernel, by the threads that then walk the item, cost as much as
// it saved: 541 against 509 us for the uneven plan.)
struct CompactPop {
    const uint8_t *src;
    uint8_t *dst;
    uint64_t stride;
    int first;               // first genome's number over all populations
    int I, O;
};

constexpr int kCompactWarps = 4;
// A node's edges that one lane goes through by itself; the warp shares more (2000
// genomes of 500 inputs, 4 outputs that read them all and 300 unneeded nodes, 8
// vectors: 146 us a step, 252 with a lane for each output's 500 edges, 165 without
// copies).
constexpr int kLaneEdges = 32;

// Whether a header describes a record of these sizes (a plan may be created
// before its records are written; whatever lies there then is not followed).
__device__ __forceinline__ bool header_holds(const uint4 &h0, const uint4 &h1, int I, int O, uint64_t stride)
{
    const uint32_t n = h0.x & 0xffffu, nl = h0.x >> 16, E = h0.y;
    const uint32_t off_edge = kHeaderBytes + kNodeBytes * n, off_level = align16(off_edge + kEdgeBytes * E);
    const uint32_t off_io = align16(off_level + 2u * (nl + 1u));
    return n >= (uint32_t)(I + O) && n <= (uint32_t)NEAT_MAX_NODES && E <= (uint32_t)NEAT_MAX_CONNS && nl >= 1u &&
           nl <= n && h1.y == off_edge && h1.z == off_level && h1.w == off_io &&
           h1.x == align16(off_io + 2u * (uint32_t)(I + O)) && h1.x <= stride;
}

__global__ void __launch_bounds__(32 * kCompactWarps)
compact_kernel(const CompactPop *__restrict__ pops, int np, const CompactPop one, int total, unsigned int *counters,
               int nc, unsigned int *largest)
{
    __shared__ uint32_t s_bits[kCompactWarps][32];
    __shared__ int s_pre[kCompactWarps][32];
    __shared__ uint16_t s_list[kCompactWarps][NEAT_MAX_NODES];
    constexpr unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == 0)                       // the steps' work counters, for the launches that follow
        for (int i = threadIdx.x; i < nc; i += blockDim.x) counters[i] = 0u;
    const int w = blockIdx.x * kCompactWarps + warp;
    if (w >= total) return;
    int lo = 0, hi = np - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pops[mid].first <= w) lo = mid; else hi = mid - 1;
    }
    const CompactPop P = np > 0 ? pops[lo] : one;
    const uint8_t *src = P.src + (size_t)(w - P.first) * P.stride;
    uint8_t *dst = P.dst + (size_t)(w - P.first) * P.stride;
    const int I = P.I, O = P.O;
    const uint4 h0 = __ldg(reinterpret_cast<const uint4 *>(src)), h1 = __ldg(reinterpret_cast<const uint4 *>(src) + 1);
    uint4 *out = reinterpret_cast<uint4 *>(dst);
    if ((h0.z & NEAT_G_ERROR_MASK) || !header_holds(h0, h1, I, O, P.stride)) {
        // nothing to evaluate: outputs NaN
        if (lane == 0) {
            out[0] = make_uint4(0u, 0u, h0.z & NEAT_G_ERROR_MASK ? h0.z : h0.z | NEAT_G_MISSING_IO, 0xffffu);
            out[1] = make_uint4(kHeaderBytes, kHeaderBytes, kHeaderBytes, kHeaderBytes);
        }
        return;
    }
    const int n_levels = (int)(h0.x >> 16);
    const uint4 *nodes = reinterpret_cast<const uint4 *>(src + kHeaderBytes);
    const uint2 *edges = reinterpret_cast<const uint2 *>(src + h1.y);
    const uint16_t *lev = reinterpret_cast<const uint16_t *>(src + h1.z);
    const uint16_t *io = reinterpret_cast<const uint16_t *>(src + h1.w);
    uint32_t *bits = s_bits[warp];
    int *pre = s_pre[warp];
    uint16_t *list = s_list[warp];
    bits[lane] = 0u;
    __syncwarp();
    int last = 0;
    for (int j = lane; j < O; j += 32) {
        const int p = __ldg(io + I + j);
        last = max(last, p);
        atomicOr(bits + (p >> 5), 1u << (p & 31));
    }
    last = __reduce_max_sync(all, last);
    __syncwarp();
    // the sources of edges i, i + step, ... below e
    auto mark = [&](int i, int e, int step) {
        for (; i < e; i += 4 * step) {
            uint32_t s[4];
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) s[k4] = i + k4 * step < e ? __ldg(&edges[i + k4 * step].y) : all;
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4)
                if (s[k4] != all) atomicOr(bits + (s[k4] >> 5), 1u << (s[k4] & 31u));
        }
    };
    // from the outputs back, a round for all nodes marked since the last one:
    // a node each lane, whatever its level (rounds of one level each leave
    // most lanes idle)
    uint32_t done = 0u;                                        // of word `lane`
    for (;;) {
        const uint32_t fresh = bits[lane] & ~done;
        done |= fresh;
        int incl = __popc(fresh);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(all, incl, o);
            if (lane >= o) incl += y;
        }
        const int count = __shfl_sync(all, incl, 31);
        if (count == 0) break;
        int k = incl - __popc(fresh);
        for (uint32_t m = fresh; m; m &= m - 1u) list[k++] = (uint16_t)(32 * lane + __ffs(m) - 1);
        __syncwarp();
        for (int q0 = 0; q0 < count; q0 += 32) {
            const uint32_t z = q0 + lane < count ? __ldg(&nodes[list[q0 + lane]].z) : 0u;
            const int b = (int)(z & 0xffffu), e = b + (int)(z >> 16);
            for (unsigned many = __ballot_sync(all, e - b > kLaneEdges); many; many &= many - 1u) {
                const int from = __ffs(many) - 1, wb = __shfl_sync(all, b, from), we = __shfl_sync(all, e, from);
                mark(wb + lane, we, 32);
            }
            if (e - b <= kLaneEdges) mark(b, e, 1);
        }
        __syncwarp();
    }
    int top = n_levels - 1;
    while ((int)__ldg(lev + top) > last) --top;                // the levels above every output
    for (int j = lane; j < I; j += 32) {
        const int p = __ldg(io + j);
        atomicOr(bits + (p >> 5), 1u << (p & 31));
    }
    __syncwarp();
    const uint32_t mine = bits[lane];
    int incl = __popc(mine);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(all, incl, o);
        if (lane >= o) incl += y;
    }
    const int n = __shfl_sync(all, incl, 31);
    pre[lane] = incl - __popc(mine);
    {
        int k = incl - __popc(mine);
        for (uint32_t m = mine; m; m &= m - 1u) list[k++] = (uint16_t)(32 * lane + __ffs(m) - 1);
    }
    __syncwarp();
    auto rank = [&](uint32_t p) { return (uint32_t)(pre[p >> 5] + __popc(bits[p >> 5] & ((1u << (p & 31u)) - 1u))); };
    const uint32_t off_edge = kHeaderBytes + kNodeBytes * (uint32_t)n;
    uint2 *edges_out = reinterpret_cast<uint2 *>(dst + off_edge);
    // edges i, i + step, ... below ec of a node whose edges begin at b, to begin at `to`
    auto copy = [&](int b, int to, int i, int ec, int step) {
        for (; i < ec; i += 4 * step) {
            uint2 e[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + q * step < ec) e[q] = __ldg(edges + b + i + q * step);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + q * step < ec) edges_out[to + i + q * step] = make_uint2(e[q].x, rank(e[q].y));
        }
    };
    int carry = 0;
    unsigned lead = (unsigned)n;                               // leading positions that are inputs
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int k = k0 + lane;
        uint4 ne = make_uint4(0u, 0u, 0u, (uint32_t)kInputAct);
        if (k < n) ne = __ldg(nodes + list[k]);
        const int ec = (int)(ne.z >> 16), b = (int)(ne.z & 0xffffu);
        int sum = ec;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(all, sum, o);
            if (lane >= o) sum += y;
        }
        const int to = carry + sum - ec;
        carry += __shfl_sync(all, sum, 31);
        for (unsigned many = __ballot_sync(all, k < n && ec > kLaneEdges); many; many &= many - 1u) {
            const int from = __ffs(many) - 1, wb = __shfl_sync(all, b, from), we = __shfl_sync(all, ec, from);
            copy(wb, __shfl_sync(all, to, from), lane, we, 32);
        }
        if (k >= n) continue;
        if ((ne.w & 0xffu) != kInputAct) lead = min(lead, (unsigned)k);
        out[2 + k] = make_uint4(ne.x, ne.y, (uint32_t)to | ((uint32_t)ec << 16), ne.w);
        if (ec <= kLaneEdges) copy(b, to, 0, ec, 1);
    }
    lead = __reduce_min_sync(all, lead);
    const uint32_t off_level = align16(off_edge + kEdgeBytes * (uint32_t)carry);
    const uint32_t off_io = align16(off_level + 2u * (uint32_t)(top + 2));
    uint16_t *lev_out = reinterpret_cast<uint16_t *>(dst + off_level);
    for (int l = lane; l <= top; l += 32) lev_out[l] = (uint16_t)rank(__ldg(lev + l));
    uint16_t *io_out = reinterpret_cast<uint16_t *>(dst + off_io);
    for (int j = lane; j < I + O; j += 32) io_out[j] = (uint16_t)rank(__ldg(io + j));
    if (lane == 0) {
        lev_out[top + 1] = (uint16_t)n;
        out[0] = make_uint4((uint32_t)n | ((uint32_t)(top + 1) << 16), (uint32_t)carry, h0.z,
                            (h0.w & 0xffffu) | (lead << 16));
        const uint32_t used = align16(off_io + 2u * (uint32_t)(I + O));
        out[1] = make_uint4(used, off_edge, off_level, off_io);
        if (largest) {                                         // most bytes and nodes of a copy
            atomicMax(largest, used);
            atomicMax(largest + 1, (unsigned int)n);
        }
    }
}

// The items of a block item whose record or nodes outgrow their group's region
// (records changed since the plan chose its shapes): one after the other, the
// record read where it lies, the values in the memory of all regions, which
// holds a column of any genome of the population (`spare` floats).  So a region
// is no larger than its bucket's genomes need: with room for max_nodes values
// in every group, 4000 genomes of 14 nodes in 1024 rows and 64 vectors took
// 16.4 us a step instead of 15.3.  Every thread of the block calls it.
__device__ __noinline__ void run_outgrown(const BucketDev &d, int ci, int step, bool late, float *v, int *flags,
                                          unsigned int *err)
{
    const int G = d.G, gi = threadIdx.x >> d.lgG, lane = threadIdx.x & (G - 1);
    const long item = (long)(ci - d.cta_begin) * d.gpc + gi;
    const int k = late ? (int)(item / d.tiles) : 0, g = __ldg(d.gidx + k);
    const int b0 = (int)(item - (long)k * d.tiles) * d.tile;
    const uint4 *rec = reinterpret_cast<const uint4 *>(d.rec + (size_t)g * d.stride);
    const float *xb = d.x + d.x_step * step + ((size_t)g * d.B + b0) * d.I;
    float *yb = d.y + d.y_step * step + ((size_t)g * d.B + b0) * d.O;
    for (int turn = 0; turn < d.gpc; ++turn) {
        if (late && turn == gi) {
            if (d.tile == 1)
                run_item<true>(rec, v, kNoBar, flags + gi, G, gi, lane, xb, yb, d.I, d.O, 1, 1, d.lg_split, d.spare,
                               AlwaysFits{}, err);
            else
                run_item<false>(rec, v, kNoBar, flags + gi, G, gi, lane, xb, yb, d.I, d.O, min(d.tile, d.B - b0), d.tile, 0,
                                d.spare, AlwaysFits{}, err);
        }
        __syncthreads();
    }
}

// A work item whose record's copy is on its way; false, with nothing evaluated,
// when the record or its nodes outgrow the group's region.  The walk of one
// vector is a function of its own: beside the tiles' in one body its loop came
// out slower (a launch of one vector each, 231 genomes of 26 and of 77 rows 18.5
// us, 14.5 as a function; the tiles' as a function too: 8 to 31 vectors 3 to 8%
// slower).
template <bool T1>
__device__ __forceinline__ bool staged_item(const BucketDev &d, uint4 *srec, uint32_t bar, int *flag, int gi, int lane,
                                            int g, int b0, int step)
{
    const float *xb = d.x + d.x_step * step + ((size_t)g * d.B + b0) * d.I;
    float *yb = d.y + d.y_step * step + ((size_t)g * d.B + b0) * d.O;
    const auto fits = [&](uint32_t bytes, int values) {
        return bytes <= (uint32_t)d.rec_words * 16u && values <= (d.region_words - d.rec_words) * 4;
    };
    return run_item<T1, false, true>(srec, reinterpret_cast<float *>(srec + d.rec_words), bar, flag, d.G, gi, lane, xb, yb,
                                     d.I, d.O, T1 ? 1 : min(d.tile, d.B - b0), T1 ? 1 : d.tile, T1 ? d.lg_split : 0, 0, fits,
                                     &g_plan_error);
}

__device__ __noinline__ bool staged_vector(const BucketDev &d, uint4 *srec, uint32_t bar, int *flag, int gi, int lane,
                                           int g, int b0, int step)
{
    return staged_item<true>(d, srec, bar, flag, gi, lane, g, b0, step);
}

template <bool PDL>
__global__ void __launch_bounds__(1024, 1)
plan_kernel(const BucketDev *__restrict__ buckets, int nb, int item_lo, int item_hi, unsigned int *counter, int step)
{
    extern __shared__ __align__(16) uint4 smem[];
    __shared__ int s_ci, s_late;
    const int NT = blockDim.x;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    int *flags = reinterpret_cast<int *>(bars + NT);
    uint4 *regions = smem + forward_header_words(NT);
    bool waited = !PDL;
    if (threadIdx.x == 0) s_late = 0;
    for (;;) {
        if (threadIdx.x == 0) s_ci = item_lo + (int)atomicAdd(counter, 1u);
        __syncthreads();
        const int ci = s_ci;
        if (ci >= item_hi) break;
        int lo = 0, hi = nb - 1;                       // bucket holding block item ci
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (buckets[mid].cta_begin <= ci) lo = mid; else hi = mid - 1;
        }
        const BucketDev &d = buckets[lo];
        const int G = d.G, lgG = d.lgG;
        const int gi = threadIdx.x >> lgG;
        const int lane = threadIdx.x & (G - 1);
        const long item = (long)(ci - d.cta_begin) * d.gpc + gi;
        const bool active = gi < d.gpc && item < (long)d.n_genomes * d.tiles;
        uint4 *srec = regions + (size_t)gi * d.region_words;
        const uint32_t bar = smem_addr(bars + gi);
        int g = 0, b0 = 0;
        bool staged = active;
        if (active) {
            const int k = (int)(item / d.tiles);
            g = __ldg(d.gidx + k);
            b0 = (int)(item - (long)k * d.tiles) * d.tile;
            const uint8_t *grec = d.rec + (size_t)g * d.stride;
            uint32_t bytes = (uint32_t)d.rec_copy_bytes;
            if (bytes == 0) {                          // a compact record's own size
                bytes = align16(__ldg(reinterpret_cast<const uint32_t *>(grec) + 4));
                staged = bytes <= (uint32_t)d.rec_words * 16u;
            }
            if (lane == 0) {
                flags[gi] = 0;
                if (staged) {
                    fence_proxy_async_smem();          // the region was read by the previous item
                    mbar_init(bar, 1);
                    mbar_arrive_expect_tx(bar, bytes);
                    bulk_g2s(smem_addr(srec), grec, bytes, bar);
                }
            }
        }
        if (PDL && !waited) {                          // inputs of this step may come from the previous kernel
            pdl_wait();
            pdl_trigger();
            waited = true;
        }
        bool late = active && !staged;
        if (staged)
            late = !(d.tile == 1 ? staged_vector(d, srec, bar, flags + gi, gi, lane, g, b0, step)
                                 : staged_item<false>(d, srec, bar, flags + gi, gi, lane, g, b0, step));
        if (late) s_late = 1;
        __syncthreads();
        if (staged && lane == 0) mbar_inval(bar);      // re-initialised by the next item using this slot
        if (s_late) {                                  // the same for all: cleared behind run_outgrown's barriers
            run_outgrown(d, ci, step, late, reinterpret_cast<float *>(regions), flags, &g_plan_error);
            if (threadIdx.x == 0) s_late = 0;
        }
    }
}

struct Shape {
    int G = 0, tile = 0, split = 1;
};

struct HostBucket {
    int pop_index = 0;
    int n_class = 0;         // node-count bound of the bucket
    int max_used = 0;        // largest record (bytes) in the bucket
    int max_rows = 0;        // value tile rows: most nodes of a record in the bucket
    std::vector<int32_t> gidx;
    Shape shape;
};

int lg(int x)
{
    int l = 0;
    while ((1 << l) < x) ++l;
    return l;
}

// A shape the kernels can index: G and tile powers of two, tile <= G <= NT,
// split 1, 2 or 4 (a bad shape would mis-index shared memory, so it is
// refused on the host before any launch).
bool shape_ok(const Shape &s, int NT)
{
    const auto p2 = [](int x) { return x > 0 && (x & (x - 1)) == 0; };
    return p2(s.G) && s.G <= NT && p2(s.tile) && s.tile <= s.G && (s.split == 1 || s.split == 2 || s.split == 4);
}

// Floats of a block's regions (a multiple of 16 bytes), at least a column of the
// population's largest genome (run_outgrown).
int spare_floats(size_t regions, int max_nodes) { return std::max((int)(regions / 4), (max_nodes + 3) & ~3); }

// Launch shape without timing: as neat_default_launch, with groups of at
// most NT threads (the persistent block).
Shape heuristic_shape(int n_class, int batch, int NT)
{
    Shape s;
    s.split = 1;
    if (batch <= 1) {
        s.tile = 1;
        s.G = std::min(NT, n_class <= 64 ? 8 : (n_class <= 256 ? 16 : 32));
    } else {
        int t = 1;
        while (t < batch && t < 32 && t < NT) t <<= 1;
        s.tile = t;
        int nsub = tile_row_threads(n_class);
        while (nsub > 1 && t * nsub > NT) nsub >>= 1;
        s.G = t * nsub;
    }
    return s;
}

}  // namespace
}  // namespace neat

using namespace neat;

struct neat_plan {
    std::vector<neat_pop_desc> pops;
    neat_plan_options opt;
    std::vector<HostBucket> hb;
    std::vector<BucketDev> bd;
    BucketDev *d_buckets = nullptr;
    int32_t *d_gidx = nullptr;
    unsigned int *d_counters = nullptr;
    int n_counters = 0;
    int block_threads = 256;
    size_t smem = 0;
    int grid = 0;
    int total_items = 0;
    cudaStream_t cap = nullptr;
    cudaGraphExec_t exec = nullptr;
    int graph_first = -1, graph_steps = -1;
    std::string autotune_log;
    int max_footprint_bucket = -1;    // host bucket whose groups take the most shared memory
    size_t smem_override = 0;         // while timing one bucket: its own footprint
    uint8_t *d_compact = nullptr;     // compact records (null: the records themselves are evaluated)
    CompactPop *d_cpops = nullptr;
    std::vector<uint8_t *> compact_of;   // by population
    int n_cpops = 0, n_genomes = 0;
};

namespace neat {
namespace {

size_t region_bytes(const HostBucket &b)
{
    const size_t rec = (size_t)align16((uint32_t)b.max_used);
    return (rec + 4u * (size_t)((b.max_rows * b.shape.tile + 3) & ~3) + 15) & ~(size_t)15;
}

// Compact records from the records as they are now, and `counters` cleared.
int launch_compact(neat_plan *P, int counters, cudaStream_t s)
{
    if (!P->d_compact) {
        const cudaError_t e = cudaMemsetAsync(P->d_counters, 0, sizeof(unsigned int) * (size_t)counters, s);
        return e == cudaSuccess ? NEAT_OK : cuda_fail(e, "plan: counter reset");
    }
    const int blocks = (P->n_genomes + kCompactWarps - 1) / kCompactWarps;
    compact_kernel<<<blocks, 32 * kCompactWarps, 0, s>>>(P->d_cpops, P->n_cpops, CompactPop{}, P->n_genomes,
                                                         P->d_counters, counters, nullptr);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NEAT_OK : cuda_fail(e, "plan: compact launch");
}

// Lay out the block items and the device bucket table for the current shapes.
int layout(neat_plan *P, cudaStream_t s)
{
    const int NT = P->block_threads;
    // largest records first
    std::vector<int> order(P->hb.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        const size_t ca = (size_t)P->hb[a].max_used * P->hb[a].shape.tile;
        const size_t cb = (size_t)P->hb[b].max_used * P->hb[b].shape.tile;
        return ca > cb;
    });
    std::vector<BucketDev> bd;
    size_t smem_regions = 0;
    int cta = 0;
    size_t goff = 0;
    std::vector<size_t> goffs(P->hb.size());
    for (size_t i = 0; i < P->hb.size(); ++i) {
        goffs[i] = goff;
        goff += P->hb[i].gidx.size();
    }
    for (int bi : order) {
        const HostBucket &h = P->hb[bi];
        const neat_pop_desc &pd = P->pops[h.pop_index];
        BucketDev d;
        d.rec = P->d_compact ? P->compact_of[h.pop_index] : static_cast<const uint8_t *>(pd.transformed_dev);
        d.gidx = P->d_gidx + goffs[bi];
        d.x = pd.inputs_dev;
        d.y = pd.outputs_dev;
        d.x_step = pd.in_step_stride;
        d.y_step = pd.out_step_stride;
        d.stride = record_stride(pd.dims);
        d.n_genomes = (int)h.gidx.size();
        d.I = pd.dims.num_inputs;
        d.O = pd.dims.num_outputs;
        d.B = pd.batch;
        d.tile = h.shape.tile;
        d.tiles = (pd.batch + d.tile - 1) / d.tile;
        d.lg_split = lg(h.shape.split);
        if (!shape_ok(h.shape, NT)) return invalid("plan: invalid bucket launch shape");
        d.G = h.shape.G;
        d.lgG = lg(d.G);
        const size_t reg = region_bytes(h);
        int gpc = NT / d.G;
        if (d.G > 32) gpc = std::min(gpc, 15);
        while (gpc > 1 && reg * gpc > 200u * 1024u) --gpc;
        if (reg * gpc + 16u * forward_header_words(NT) > 227u * 1024u)
            return invalid("plan: a bucket's region exceeds shared memory; use a smaller tile");
        d.gpc = gpc;
        d.region_words = (int)(reg / 16);
        d.rec_words = (int)(align16((uint32_t)h.max_used) / 16);
        d.rec_copy_bytes = P->d_compact ? 0 : (int)align16((uint32_t)h.max_used);
        const long items = (long)d.n_genomes * d.tiles;
        d.cta_begin = cta;
        d.cta_items = (int)((items + gpc - 1) / gpc);
        cta += d.cta_items;
        d.spare = spare_floats(reg * gpc, pd.dims.max_nodes);
        smem_regions = std::max(smem_regions, 4u * (size_t)d.spare);
        bd.push_back(d);
    }
    P->bd = bd;
    P->total_items = cta;
    P->smem = smem_regions + 16u * forward_header_words(NT);
    P->max_footprint_bucket = -1;
    {
        size_t best = 0;
        for (size_t i = 0; i < bd.size(); ++i) {
            const size_t f = 4u * (size_t)bd[i].spare;
            if (f > best) {
                best = f;
                P->max_footprint_bucket = order[i];
            }
        }
    }
    if (P->d_buckets) cudaFree(P->d_buckets);
    cudaError_t e = cudaMalloc(&P->d_buckets, sizeof(BucketDev) * std::max<size_t>(bd.size(), 1));
    if (e != cudaSuccess) return cuda_fail(e, "plan: cudaMalloc buckets");
    e = cudaMemcpyAsync(P->d_buckets, bd.data(), sizeof(BucketDev) * bd.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "plan: copy buckets");
    // persistent grid: as many resident blocks as the shared memory allows
    int dev = 0, sms = 152, smem_sm = 233472;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    int per_sm = (int)(smem_sm / (P->smem + 1024));
    per_sm = std::max(1, std::min(per_sm, 2048 / NT));
    P->grid = std::max(1, std::min(sms * per_sm, P->total_items));
    for (auto f : {plan_kernel<true>, plan_kernel<false>}) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, f);
        if (e != cudaSuccess) return cuda_fail(e, "plan: cudaFuncGetAttributes");
        if (P->smem + fa.sharedSizeBytes > 227u * 1024u)
            return invalid("plan: shared memory per block exceeds 227 KB; use a smaller tile");
        const int rc = allow_dynamic_smem(reinterpret_cast<const void *>(f), P->smem, "plan: shared memory per block");
        if (rc) return rc;
    }
    if (P->exec) {
        cudaGraphExecDestroy(P->exec);
        P->exec = nullptr;
    }
    return NEAT_OK;
}

int ensure_counters(neat_plan *P, int n)
{
    if (P->n_counters >= n) return NEAT_OK;
    if (P->d_counters) cudaFree(P->d_counters);
    P->d_counters = nullptr;
    cudaError_t e = cudaMalloc(&P->d_counters, sizeof(unsigned int) * (size_t)n);
    if (e != cudaSuccess) return cuda_fail(e, "plan: cudaMalloc counters");
    P->n_counters = n;
    return NEAT_OK;
}

// One step of block items [lo, hi) using counter `ctr` (reset first).
int launch_step(neat_plan *P, int lo, int hi, unsigned int *ctr, int step, bool pdl, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::max(1, std::min(P->grid, hi - lo)));
    cfg.blockDim = dim3((unsigned)P->block_threads);
    cfg.dynamicSmemBytes = P->smem_override ? P->smem_override : P->smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (pdl) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    cudaError_t e = pdl ? cudaLaunchKernelEx(&cfg, plan_kernel<true>, (const BucketDev *)P->d_buckets,
                                             (int)P->bd.size(), lo, hi, ctr, step)
                        : cudaLaunchKernelEx(&cfg, plan_kernel<false>, (const BucketDev *)P->d_buckets,
                                             (int)P->bd.size(), lo, hi, ctr, step);
    if (e != cudaSuccess) return cuda_fail(e, "plan: launch");
    return NEAT_OK;
}

// Time `reps` launches of bucket index `bi` (position in P->bd) alone.
float time_bucket(neat_plan *P, int bi, cudaStream_t s, int reps)
{
    const BucketDev &d = P->bd[bi];
    P->smem_override = 4u * (size_t)d.spare + 16u * forward_header_words(P->block_threads);
    const int grid_saved = P->grid;
    {
        int dev = 0, sms = 152, smem_sm = 233472;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        int per_sm = (int)(smem_sm / (P->smem_override + 1024));
        per_sm = std::max(1, std::min(per_sm, 2048 / P->block_threads));
        P->grid = sms * per_sm;
    }
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    float best = 1e30f;
    for (int r = 0; r < reps + 1; ++r) {
        cudaMemsetAsync(P->d_counters, 0, sizeof(unsigned int), s);
        cudaEventRecord(a, s);
        if (launch_step(P, d.cta_begin, d.cta_begin + d.cta_items, P->d_counters, 0, false, s) != NEAT_OK) {
            best = 1e30f;
            break;
        }
        cudaEventRecord(b, s);
        cudaEventSynchronize(b);
        float ms = 0;
        cudaEventElapsedTime(&ms, a, b);
        if (r > 0) best = std::min(best, ms);
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    P->smem_override = 0;
    P->grid = grid_saved;
    return best;
}

// Time one whole step of the laid-out plan (best of reps).
float time_plan(neat_plan *P, cudaStream_t s, int reps)
{
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    float best = 1e30f;
    for (int r = 0; r < reps + 1; ++r) {
        cudaMemsetAsync(P->d_counters, 0, sizeof(unsigned int), s);
        cudaEventRecord(a, s);
        if (launch_step(P, 0, P->total_items, P->d_counters, 0, false, s) != NEAT_OK) break;
        cudaEventRecord(b, s);
        cudaEventSynchronize(b);
        float ms = 0;
        cudaEventElapsedTime(&ms, a, b);
        if (r > 0) best = std::min(best, ms);
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return best;
}

std::vector<Shape> candidates(int n_class, int batch, int NT)
{
    std::vector<Shape> c;
    if (batch <= 1) {
        for (int G : {4, 8, 16, 32})
            for (int split : {1, 2})
                if (G <= NT) c.push_back(Shape{G, 1, split});
    } else {
        for (int t : {4, 8, 16, 32}) {
            if (t > 2 * batch && t > 4) continue;
            for (int nsub : {1, 2, 4, 8, 16, 32}) {
                if (t * nsub > NT || t * nsub < 8) continue;
                if (nsub > 1 && nsub * 4 > n_class) continue;       // more threads than a level can use
                c.push_back(Shape{t * nsub, t, 1});
            }
        }
    }
    return c;
}

// Footprint in shared memory of a bucket's groups in one block.
size_t footprint(const neat_plan *P, const HostBucket &h)
{
    int gpc = P->block_threads / h.shape.G;
    if (h.shape.G > 32) gpc = std::min(gpc, 15);
    return region_bytes(h) * gpc;
}

int autotune(neat_plan *P, cudaStream_t s, float *step_ms)
{
    char line[256];
    auto position_of = [&](size_t hbi) {
        size_t goff = 0;
        for (size_t i = 0; i < hbi; ++i) goff += P->hb[i].gidx.size();
        for (size_t i = 0; i < P->bd.size(); ++i)
            if (P->bd[i].gidx == P->d_gidx + goff) return (int)i;
        return -1;
    };
    // 1. each bucket alone, at its own shared-memory footprint
    std::vector<std::vector<std::pair<float, Shape>>> timed(P->hb.size());
    for (size_t hbi = 0; hbi < P->hb.size(); ++hbi) {
        HostBucket &h = P->hb[hbi];
        const neat_pop_desc &pd = P->pops[h.pop_index];
        const Shape keep = h.shape;
        for (const Shape &c : candidates(h.n_class, pd.batch, P->block_threads)) {
            h.shape = c;
            if (layout(P, s) != NEAT_OK) {
                cudaGetLastError();
                continue;
            }
            const int pos = position_of(hbi);
            if (pos < 0) continue;
            timed[hbi].push_back({time_bucket(P, pos, s, 2), c});
        }
        cudaGetLastError();
        std::sort(timed[hbi].begin(), timed[hbi].end(),
                  [](const std::pair<float, Shape> &a, const std::pair<float, Shape> &b) { return a.first < b.first; });
        h.shape = timed[hbi].empty() ? keep : timed[hbi][0].second;
    }
    // 2. the whole step: shrink the bucket that sets the block's shared
    //    memory (it limits every bucket's residency) while that pays
    int rc = layout(P, s);
    if (rc) return rc;
    float best_ms = time_plan(P, s, 2);
    for (int round = 0; round < 8; ++round) {
        const int hbi = P->max_footprint_bucket;
        if (hbi < 0) break;
        HostBucket &h = P->hb[hbi];
        const Shape cur = h.shape;
        const size_t cur_fp = footprint(P, h);
        bool improved = false;
        for (const auto &cand : timed[hbi]) {
            h.shape = cand.second;
            if (footprint(P, h) >= cur_fp) continue;
            if (layout(P, s) != NEAT_OK) {
                cudaGetLastError();
                continue;
            }
            const float ms = time_plan(P, s, 2);
            if (ms < best_ms) {
                best_ms = ms;
                improved = true;
                break;
            }
        }
        if (!improved) {
            h.shape = cur;
            break;
        }
    }
    for (size_t hbi = 0; hbi < P->hb.size(); ++hbi) {
        const HostBucket &h = P->hb[hbi];
        snprintf(line, sizeof(line), "%s{\"pop\":%d,\"n_class\":%d,\"G\":%d,\"tile\":%d,\"split\":%d}",
                 hbi ? "," : "", h.pop_index, h.n_class, h.shape.G, h.shape.tile, h.shape.split);
        P->autotune_log += line;
    }
    snprintf(line, sizeof(line), ",{\"block_threads\":%d,\"step_ms\":%.5f}", P->block_threads, best_ms);
    P->autotune_log += line;
    if (step_ms) *step_ms = best_ms;
    return layout(P, s);
}

// Autotune at each persistent block size and keep the fastest: large
// groups (a tile row of many threads for genomes of hundreds of nodes) need
// large blocks, many small groups share smaller ones well.
int autotune_block_threads(neat_plan *P, cudaStream_t s)
{
    struct Best {
        float ms = -1.0f;
        int NT = 0;
        std::vector<Shape> shapes;
        std::string log;
    } best;
    for (int NT : {256, 512, 1024}) {
        P->block_threads = NT;
        P->autotune_log.clear();
        for (HostBucket &b : P->hb) b.shape = heuristic_shape(b.n_class, P->pops[b.pop_index].batch, NT);
        int rc = layout(P, s);
        float ms = -1.0f;
        if (rc == NEAT_OK) rc = autotune(P, s, &ms);
        if (rc != NEAT_OK) {
            cudaGetLastError();
            clear_error();
            continue;
        }
        if (best.ms < 0.0f || ms < best.ms) {
            best.ms = ms;
            best.NT = NT;
            best.shapes.clear();
            for (const HostBucket &b : P->hb) best.shapes.push_back(b.shape);
            best.log = P->autotune_log;
        }
    }
    if (best.NT == 0) return invalid("neat_plan_create: no block size could be tuned");
    P->block_threads = best.NT;
    P->opt.block_threads = best.NT;
    for (size_t i = 0; i < P->hb.size(); ++i) P->hb[i].shape = best.shapes[i];
    P->autotune_log = best.log;
    return layout(P, s);
}

// The workspace of the compact records, and a first copy.  Without memory for
// it the plan evaluates the records themselves.
int make_compact(neat_plan *P, cudaStream_t s)
{
    size_t bytes = 0;
    std::vector<CompactPop> cp;
    std::vector<int> order(P->pops.size());
    P->compact_of.assign(P->pops.size(), nullptr);
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    // the largest records' long chains first
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return record_stride(P->pops[a].dims) > record_stride(P->pops[b].dims);
    });
    for (const neat_pop_desc &pd : P->pops)
        if (pd.pop > 0 && pd.batch > 0) bytes += record_stride(pd.dims) * (size_t)pd.pop;
    if (bytes == 0) return NEAT_OK;
    if (cudaMalloc(&P->d_compact, bytes) != cudaSuccess) {
        cudaGetLastError();
        P->d_compact = nullptr;
        return NEAT_OK;
    }
    size_t off = 0;
    for (int p : order) {
        const neat_pop_desc &pd = P->pops[p];
        if (pd.pop == 0 || pd.batch == 0) continue;
        CompactPop c;
        c.src = static_cast<const uint8_t *>(pd.transformed_dev);
        c.dst = P->compact_of[p] = P->d_compact + off;
        c.stride = record_stride(pd.dims);
        c.first = P->n_genomes;
        c.I = pd.dims.num_inputs;
        c.O = pd.dims.num_outputs;
        off += c.stride * (size_t)pd.pop;
        P->n_genomes += pd.pop;
        cp.push_back(c);
    }
    P->n_cpops = (int)cp.size();
    cudaError_t e = cudaMalloc(&P->d_cpops, sizeof(CompactPop) * cp.size());
    if (e != cudaSuccess) return cuda_fail(e, "neat_plan_create: cudaMalloc");
    e = cudaMemcpyAsync(P->d_cpops, cp.data(), sizeof(CompactPop) * cp.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "neat_plan_create: copy");
    const int rc = launch_compact(P, 1, s);
    if (rc) return rc;
    e = cudaStreamSynchronize(s);              // cp goes out of scope
    return e == cudaSuccess ? NEAT_OK : cuda_fail(e, "neat_plan_create: synchronize");
}

void free_compact(neat_plan *P)
{
    if (P->d_compact) cudaFree(P->d_compact);
    if (P->d_cpops) cudaFree(P->d_cpops);
    P->d_compact = nullptr;
    P->d_cpops = nullptr;
}

int read_headers(neat_plan *P, bool compact, cudaStream_t s, std::vector<std::vector<uint32_t>> *out)
{
    out->assign(P->pops.size(), {});
    for (size_t p = 0; p < P->pops.size(); ++p) {
        const neat_pop_desc &pd = P->pops[p];
        if (pd.pop == 0 || pd.batch == 0) continue;
        (*out)[p].resize((size_t)pd.pop * 8);
        const void *src = compact ? P->compact_of[p] : pd.transformed_dev;
        const cudaError_t e = cudaMemcpy2DAsync((*out)[p].data(), 32, src, record_stride(pd.dims), 32, (size_t)pd.pop,
                                                cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return cuda_fail(e, "neat_plan_create: header copy");
    }
    return NEAT_OK;
}

// Whether the nodes saved are worth the copy that every call makes.  A warp
// takes a node for 32 columns, or several nodes for fewer, in about 130
// instructions; 100 000 of those are what the copy and its wait cost.  Small
// batches save little per node: 248 genomes each of 56 to 441 rows and 8
// vectors, 32 us a step as they are and 49 with copies; 425 of 26 to 284 rows
// and 3 vectors 32 and 47; 1 669 of 20 to 509 rows and 3 vectors 59 and 62.
// (Some small batches of large genomes would gain and stay as they are: 1 723
// of 216 and 700 rows and 2 vectors, 94 and 69.)
bool compact_pays(const neat_plan *P, const std::vector<std::vector<uint32_t>> &full,
                  const std::vector<std::vector<uint32_t>> &compact)
{
    double saved = 0.0;
    for (size_t p = 0; p < full.size(); ++p) {
        const int batch = P->pops[p].batch;
        const double per_node = batch > 16 ? (double)((batch + 31) / 32) : std::max(4, 1 << lg(batch)) / 32.0;
        for (size_t g = 0; g * 8 < full[p].size(); ++g)
            saved += per_node * ((double)(full[p][g * 8] & 0xffffu) - (double)(compact[p][g * 8] & 0xffffu));
    }
    return saved > 100000.0;
}

}  // namespace
}  // namespace neat

extern "C" int neat_plan_create(const neat_pop_desc *pops, int32_t npops, const neat_plan_options *opt,
                                void *stream, neat_plan **out)
{
    TraceRange trace_range("neat_plan_create");
    clear_error();
    if (!out) return invalid("neat_plan_create: null output pointer");
    *out = nullptr;
    if (!pops || npops < 1) return invalid("neat_plan_create: no populations");
    cudaStream_t s = as_stream(stream);
    neat_plan_options o = {0, 1, 0, 1};
    if (opt) o = *opt;
    const bool tune_block = o.autotune && o.block_threads == 0;
    if (o.block_threads == 0) o.block_threads = 256;
    if (o.block_threads < 32 || o.block_threads > 1024 || (o.block_threads & (o.block_threads - 1)))
        return invalid("neat_plan_create: block_threads must be a power of two in 32..1024");
    for (int p = 0; p < npops; ++p) {
        const neat_pop_desc &pd = pops[p];
        if (!dims_ok(pd.dims)) return invalid("neat_plan_create: invalid dims");
        if (pd.pop < 0 || pd.batch < 0) return invalid("neat_plan_create: pop and batch must be >= 0");
        if (pd.pop > 0 && pd.batch > 0 && (!pd.transformed_dev || !pd.outputs_dev ||
                                            (pd.dims.num_inputs > 0 && !pd.inputs_dev)))
            return invalid("neat_plan_create: null pointer");
        if (reinterpret_cast<uintptr_t>(pd.transformed_dev) & 15u)
            return invalid("neat_plan_create: transformed must be 16-byte aligned");
    }
    neat_plan *P = new neat_plan();
    P->pops.assign(pops, pops + npops);
    P->opt = o;
    P->block_threads = o.block_threads;
    // read every header once, and those of the compact records
    std::vector<std::vector<uint32_t>> hdrs, chdrs;
    int rc = ensure_counters(P, 1);
    if (rc == NEAT_OK) rc = make_compact(P, s);
    if (rc == NEAT_OK) rc = read_headers(P, false, s, &hdrs);
    if (rc == NEAT_OK && P->d_compact) rc = read_headers(P, true, s, &chdrs);
    cudaError_t e = cudaSuccess;
    if (rc == NEAT_OK && (e = cudaStreamSynchronize(s)) != cudaSuccess) rc = cuda_fail(e, "neat_plan_create: synchronize");
    if (rc != NEAT_OK) {
        neat_plan_destroy(P);
        return rc;
    }
    if (P->d_compact) {
        if (compact_pays(P, hdrs, chdrs)) hdrs.swap(chdrs);
        else free_compact(P);
    }
    for (int p = 0; p < npops; ++p) {
        const neat_pop_desc &pd = pops[p];
        if (hdrs[p].empty()) continue;
        const int max_class = 1 << lg(pd.dims.max_nodes);
        std::vector<int> slot_of_class(12, -1);
        for (int g = 0; g < pd.pop; ++g) {
            const uint32_t *h = &hdrs[p][(size_t)g * 8];
            const int n = std::min((int)(h[0] & 0xffffu), pd.dims.max_nodes);
            int cls = o.size_buckets ? std::max(16, 1 << lg(std::max(n, 1))) : max_class;
            cls = std::min(cls, std::max(16, max_class));
            int key = lg(cls);
            if (slot_of_class[key] < 0) {
                slot_of_class[key] = (int)P->hb.size();
                HostBucket b;
                b.pop_index = p;
                b.n_class = std::min(cls, pd.dims.max_nodes);
                b.max_used = 32;
                P->hb.push_back(b);
            }
            HostBucket &b = P->hb[slot_of_class[key]];
            b.gidx.push_back(g);
            b.max_rows = P->d_compact ? std::max(b.max_rows, n) : b.n_class;
            const uint32_t used = std::min<uint32_t>(h[4], record_max_bytes(pd.dims.num_inputs, pd.dims.num_outputs,
                                                                            pd.dims.max_nodes, pd.dims.max_conns));
            b.max_used = std::max<int>(b.max_used, (int)align16(used));
        }
    }
    // within a bucket, deepest and largest genomes first: groups that share
    // a warp then have similar level counts (a warp walks as many levels as
    // its deepest genome), and the longest items start first
    for (HostBucket &b : P->hb) {
        const std::vector<uint32_t> &h = hdrs[b.pop_index];
        std::stable_sort(b.gidx.begin(), b.gidx.end(), [&](int32_t x, int32_t y) {
            const uint32_t lx = h[(size_t)x * 8] >> 16, ly = h[(size_t)y * 8] >> 16;
            if (lx != ly) return lx > ly;
            return h[(size_t)x * 8 + 1] > h[(size_t)y * 8 + 1];
        });
        b.shape = heuristic_shape(b.n_class, P->pops[b.pop_index].batch, P->block_threads);
    }
    size_t total = 0;
    for (const HostBucket &b : P->hb) total += b.gidx.size();
    if (total > 0) {
        e = cudaMalloc(&P->d_gidx, sizeof(int32_t) * total);
        if (e != cudaSuccess) {
            neat_plan_destroy(P);
            return cuda_fail(e, "neat_plan_create: cudaMalloc indices");
        }
        size_t off = 0;
        for (const HostBucket &b : P->hb) {
            e = cudaMemcpyAsync(P->d_gidx + off, b.gidx.data(), sizeof(int32_t) * b.gidx.size(),
                                cudaMemcpyHostToDevice, s);
            if (e != cudaSuccess) {
                neat_plan_destroy(P);
                return cuda_fail(e, "neat_plan_create: copy indices");
            }
            off += b.gidx.size();
        }
    }
    rc = layout(P, s);
    if (rc == NEAT_OK && o.autotune && !P->hb.empty())
        rc = tune_block ? autotune_block_threads(P, s) : autotune(P, s, nullptr);
    if (rc == NEAT_OK) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_fail(e, "neat_plan_create: synchronize");
    }
    if (rc != NEAT_OK) {
        neat_plan_destroy(P);
        return rc;
    }
    *out = P;
    return NEAT_OK;
}

extern "C" int neat_plan_forward(neat_plan *P, int32_t step, void *stream)
{
    TraceRange trace_range("neat_plan_forward");
    clear_error();
    if (!P) return invalid("neat_plan_forward: null plan");
    if (step < 0) return invalid("neat_plan_forward: step < 0");
    if (P->total_items == 0) return NEAT_OK;
    cudaStream_t s = as_stream(stream);
    const int rc = launch_compact(P, 1, s);
    if (rc) return rc;
    return launch_step(P, 0, P->total_items, P->d_counters, step, false, s);
}

extern "C" int neat_plan_forward_steps(neat_plan *P, int32_t first_step, int32_t steps, void *stream)
{
    TraceRange trace_range("neat_plan_forward_steps");
    clear_error();
    if (!P) return invalid("neat_plan_forward_steps: null plan");
    if (first_step < 0 || steps < 0) return invalid("neat_plan_forward_steps: negative step");
    if (steps == 0 || P->total_items == 0) return NEAT_OK;
    if (!P->exec || P->graph_first != first_step || P->graph_steps != steps) {
        if (P->exec) {
            cudaGraphExecDestroy(P->exec);
            P->exec = nullptr;
        }
        int rc = ensure_counters(P, steps);
        if (rc) return rc;
        cudaError_t e;
        if (!P->cap) {
            e = cudaStreamCreateWithFlags(&P->cap, cudaStreamNonBlocking);
            if (e != cudaSuccess) return cuda_fail(e, "neat_plan_forward_steps: stream");
        }
        e = cudaStreamBeginCapture(P->cap, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(e, "neat_plan_forward_steps: begin capture");
        rc = launch_compact(P, steps, P->cap);
        for (int k = 0; k < steps && rc == NEAT_OK; ++k)
            rc = launch_step(P, 0, P->total_items, P->d_counters + k, first_step + k, P->opt.pdl && k > 0, P->cap);
        cudaGraph_t graph = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(P->cap, &graph);
        if (rc != NEAT_OK || e2 != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            if (rc) return rc;
            return cuda_fail(e2, "neat_plan_forward_steps: capture");
        }
        e = cudaGraphInstantiate(&P->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            P->exec = nullptr;
            return cuda_fail(e, "neat_plan_forward_steps: instantiate");
        }
        P->graph_first = first_step;
        P->graph_steps = steps;
    }
    cudaError_t e = cudaGraphLaunch(P->exec, as_stream(stream));
    if (e != cudaSuccess) return cuda_fail(e, "neat_plan_forward_steps: launch");
    return NEAT_OK;
}

extern "C" int neat_plan_describe(const neat_plan *P, char *buf, int32_t len)
{
    if (!P) return invalid("neat_plan_describe: null plan");
    std::string js = "{\"block_threads\":" + std::to_string(P->block_threads) +
                     ",\"grid\":" + std::to_string(P->grid) + ",\"smem\":" + std::to_string(P->smem) +
                     ",\"block_items\":" + std::to_string(P->total_items) + ",\"buckets\":[";
    for (size_t i = 0; i < P->bd.size(); ++i) {
        const BucketDev &d = P->bd[i];
        char tmp[320];
        snprintf(tmp, sizeof(tmp),
                 "%s{\"genomes\":%d,\"batch\":%d,\"G\":%d,\"tile\":%d,\"split\":%d,\"groups_per_block\":%d,"
                 "\"record_bytes\":%d,\"region_bytes\":%d,\"block_items\":%d}",
                 i ? "," : "", d.n_genomes, d.B, d.G, d.tile, 1 << d.lg_split, d.gpc, d.rec_words * 16,
                 d.region_words * 16, d.cta_items);
        js += tmp;
    }
    js += "],\"autotune\":[" + P->autotune_log + "]}";
    if (buf && len > 0) {
        const size_t n = std::min<size_t>(js.size(), (size_t)len - 1);
        memcpy(buf, js.data(), n);
        buf[n] = 0;
    }
    return (int)js.size() + 1;
}

extern "C" void neat_plan_destroy(neat_plan *P)
{
    if (!P) return;
    if (P->exec) cudaGraphExecDestroy(P->exec);
    if (P->cap) cudaStreamDestroy(P->cap);
    if (P->d_buckets) cudaFree(P->d_buckets);
    if (P->d_gidx) cudaFree(P->d_gidx);
    if (P->d_counters) cudaFree(P->d_counters);
    free_compact(P);
    delete P;
}

namespace neat {
int read_plan_error(unsigned int *v, int clear)
{
    cudaError_t e = cudaMemcpyFromSymbol(v, g_plan_error, sizeof(*v));
    if (e != cudaSuccess) return cuda_fail(e, "plan error word: read");
    if (clear) {
        const unsigned int zero = 0;
        e = cudaMemcpyToSymbol(g_plan_error, &zero, sizeof(zero));
        if (e != cudaSuccess) return cuda_fail(e, "plan error word: clear");
    }
    return NEAT_OK;
}
}  // namespace neat

// ------------------------------------------------------------------------
// Allocation-free batched forward: the persistent plan kernel, fed from a
// fixed scratch array in device memory instead of buffers the plan
// allocates.  For callers that cannot call cudaMalloc (see neat.h).
//
// Scratch layout (file-scope, 256-byte aligned, held by every GPU that loads
// the library until the process exits):
//   [0, 256)             the work counter, cleared by every call
//   [256, idx_off)       the bucket table, written by every call
//   [idx_off, end)       genome indices 0 .. kNoallocMaxGenomes-1, written once
// Host code only knows the array through a host-side stand-in, so its device
// address is fetched with cudaGetSymbolAddress once per device.
namespace neat {
namespace {

constexpr int kNoallocMaxPops = 64;
constexpr int kNoallocMaxGenomes = 32768;
constexpr size_t kNoallocTableOff = 256;
constexpr size_t kNoallocIdxOff = kNoallocTableOff + ((sizeof(BucketDev) * kNoallocMaxPops + 255) & ~(size_t)255);
constexpr size_t kNoallocScratchBytes = kNoallocIdxOff + sizeof(int32_t) * kNoallocMaxGenomes;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

__global__ void noalloc_fill_indices(int32_t *idx, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) idx[i] = i;
}

// The call's bucket table travels as a kernel argument (no host-to-device
// copy); one small kernel writes it into the scratch array and clears the
// work counter.
struct NoallocTable {
    BucketDev b[kNoallocMaxPops];
};

__global__ void noalloc_set_table(const NoallocTable t, int nb, BucketDev *dst, unsigned int *counter)
{
    const uint32_t *src = reinterpret_cast<const uint32_t *>(t.b);
    uint32_t *out = reinterpret_cast<uint32_t *>(dst);
    const int words = nb * (int)(sizeof(BucketDev) / sizeof(uint32_t));
    for (int i = threadIdx.x; i < words; i += blockDim.x) out[i] = src[i];
    if (threadIdx.x == 0) *counter = 0u;
}
static_assert(sizeof(BucketDev) % sizeof(uint32_t) == 0, "bucket entries copy as words");

std::mutex g_noalloc_mu;
unsigned char *g_noalloc_base[256] = {};   // device address of the scratch array, per device id

// Per-device set-up, on the first call made with that device current: the
// array's device address (cudaGetSymbolAddress) and its index list.
int noalloc_setup(cudaStream_t s, unsigned char **base)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= 256) return invalid("neat_forward_multi_noalloc: device id out of range");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (g_noalloc_base[dev]) {
        *base = g_noalloc_base[dev];
        return NEAT_OK;
    }
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: cudaGetSymbolAddress");
    noalloc_fill_indices<<<64, 256, 0, s>>>(reinterpret_cast<int32_t *>(static_cast<unsigned char *>(p) + kNoallocIdxOff),
                                            kNoallocMaxGenomes);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: index fill");
    // the index list is complete before any call (on any stream or thread)
    // can see the cached address
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: index fill");
    g_noalloc_base[dev] = static_cast<unsigned char *>(p);
    *base = g_noalloc_base[dev];
    return NEAT_OK;
}

}  // namespace
}  // namespace neat

extern "C" int neat_forward_multi_noalloc(const neat_pop_desc *pops, int32_t npops, int32_t step, void *stream)
{
    TraceRange trace_range("neat_forward_multi_noalloc");
    clear_error();
    if (!pops) return invalid("neat_forward_multi_noalloc: null populations");
    if (npops < 1 || npops > kNoallocMaxPops)
        return invalid("neat_forward_multi_noalloc: npops must be in 1..64 (the scratch table holds 64 populations)");
    if (step < 0) return invalid("neat_forward_multi_noalloc: step < 0");
    for (int p = 0; p < npops; ++p) {
        const neat_pop_desc &pd = pops[p];
        if (!dims_ok(pd.dims)) return invalid("neat_forward_multi_noalloc: invalid dims");
        if (pd.pop < 0 || pd.batch < 0) return invalid("neat_forward_multi_noalloc: pop and batch must be >= 0");
        if (pd.pop > kNoallocMaxGenomes)
            return invalid("neat_forward_multi_noalloc: at most 32768 genomes per population (scratch index list)");
        if (pd.pop > 0 && pd.batch > 0 &&
            (!pd.transformed_dev || !pd.outputs_dev || (pd.dims.num_inputs > 0 && !pd.inputs_dev)))
            return invalid("neat_forward_multi_noalloc: null pointer");
        if (reinterpret_cast<uintptr_t>(pd.transformed_dev) & 15u)
            return invalid("neat_forward_multi_noalloc: transformed must be 16-byte aligned");
    }
    cudaStream_t s = as_stream(stream);
    unsigned char *base = nullptr;
    int rc = noalloc_setup(s, &base);
    if (rc) return rc;

    // one bucket per population, shapes from the heuristic, reserved record size
    const int NT = 256;
    NoallocTable tab;
    BucketDev *table = tab.b;
    int order[kNoallocMaxPops];
    int nb = 0;
    for (int p = 0; p < npops; ++p)
        if (pops[p].pop > 0 && pops[p].batch > 0) order[nb++] = p;
    for (int i = 1; i < nb; ++i)                    // largest records first
        for (int j = i; j > 0; --j) {
            const neat_dims &a = pops[order[j]].dims, &b = pops[order[j - 1]].dims;
            if (record_max_bytes(a.num_inputs, a.num_outputs, a.max_nodes, a.max_conns) <=
                record_max_bytes(b.num_inputs, b.num_outputs, b.max_nodes, b.max_conns))
                break;
            std::swap(order[j], order[j - 1]);
        }
    size_t smem_regions = 0;
    int64_t cta = 0;
    for (int i = 0; i < nb; ++i) {
        const neat_pop_desc &pd = pops[order[i]];
        const Shape sh = heuristic_shape(pd.dims.max_nodes, pd.batch, NT);
        const uint32_t rec = record_max_bytes(pd.dims.num_inputs, pd.dims.num_outputs, pd.dims.max_nodes,
                                              pd.dims.max_conns);
        const size_t reg = ((size_t)rec + 4u * (size_t)((pd.dims.max_nodes * sh.tile + 3) & ~3) + 15) & ~(size_t)15;
        if (!shape_ok(sh, NT)) return invalid("neat_forward_multi_noalloc: invalid launch shape");
        int gpc = NT / sh.G;
        if (sh.G > 32) gpc = std::min(gpc, 15);
        while (gpc > 1 && reg * gpc > 200u * 1024u) --gpc;
        if (reg * gpc + 16u * forward_header_words(NT) > 227u * 1024u)
            return invalid("neat_forward_multi_noalloc: a population's genome is too large for one block");
        BucketDev &d = table[i];
        d.rec = static_cast<const uint8_t *>(pd.transformed_dev);
        d.gidx = reinterpret_cast<const int32_t *>(base + kNoallocIdxOff);
        d.x = pd.inputs_dev;
        d.y = pd.outputs_dev;
        d.x_step = pd.in_step_stride;
        d.y_step = pd.out_step_stride;
        d.stride = record_stride(pd.dims);
        d.n_genomes = pd.pop;
        d.I = pd.dims.num_inputs;
        d.O = pd.dims.num_outputs;
        d.B = pd.batch;
        d.tile = sh.tile;
        d.tiles = (pd.batch + sh.tile - 1) / sh.tile;
        d.lg_split = lg(sh.split);
        d.G = sh.G;
        d.lgG = lg(sh.G);
        d.gpc = gpc;
        d.region_words = (int)(reg / 16);
        d.rec_words = (int)(rec / 16);
        d.rec_copy_bytes = (int)rec;
        const int64_t items = ((int64_t)d.n_genomes * d.tiles + gpc - 1) / gpc;
        if (items > INT_MAX || cta + items > INT_MAX)
            return invalid("neat_forward_multi_noalloc: more than 2^31 - 1 block work items in one call");
        d.cta_begin = (int)cta;
        d.cta_items = (int)items;
        cta += items;
        d.spare = spare_floats(reg * gpc, pd.dims.max_nodes);
        smem_regions = std::max(smem_regions, 4u * (size_t)d.spare);
    }
    if (nb == 0) return NEAT_OK;
    const size_t smem = smem_regions + 16u * forward_header_words(NT);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, plan_kernel<false>);
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: cudaFuncGetAttributes");
    if (smem + fa.sharedSizeBytes > 227u * 1024u)
        return invalid("neat_forward_multi_noalloc: shared memory per block exceeds 227 KB");
    {
        const int rc = allow_dynamic_smem(reinterpret_cast<const void *>(plan_kernel<false>), smem,
                                          "neat_forward_multi_noalloc: shared memory per block");
        if (rc) return rc;
    }
    // the bucket table and a zero work counter, by one small kernel
    noalloc_set_table<<<1, 256, 0, s>>>(tab, nb, reinterpret_cast<BucketDev *>(base + kNoallocTableOff),
                                        reinterpret_cast<unsigned int *>(base));
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: table");
    int dev = 0, sms = 152, smem_sm = 233472;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    int per_sm = std::max(1, std::min((int)(smem_sm / (smem + 1024)), 2048 / NT));
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm, cta));
    plan_kernel<false><<<grid, NT, smem, s>>>(reinterpret_cast<const BucketDev *>(base + kNoallocTableOff), nb, 0,
                                              (int)cta, reinterpret_cast<unsigned int *>(base), step);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_forward_multi_noalloc: launch");
    return NEAT_OK;
}

// ------------------------------------------------------------------------
// Internal helpers for other translation units (the serving runtime).
namespace neat {

int launch_compact_population(const void *src, void *dst, int pop, const neat_dims &d, unsigned int *largest_dev,
                              cudaStream_t s)
{
    if (pop == 0) return NEAT_OK;
    const CompactPop one{static_cast<const uint8_t *>(src), static_cast<uint8_t *>(dst), record_stride(d), 0,
                         d.num_inputs, d.num_outputs};
    compact_kernel<<<(pop + kCompactWarps - 1) / kCompactWarps, 32 * kCompactWarps, 0, s>>>(nullptr, 0, one, pop, nullptr,
                                                                                             0, largest_dev);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NEAT_OK : cuda_fail(e, "compact records: launch");
}

int fill_population_bucket(const neat_pop_desc &pd, const int32_t *gidx_dev, int block_threads, int cta_begin,
                           BucketDev *out, size_t *footprint, bool own_size, int max_used, int max_rows)
{
    const int rows = max_rows > 0 ? std::min(max_rows, pd.dims.max_nodes) : pd.dims.max_nodes;
    // (the threads of a tile row halve below a power of two: 504 of 512 rows left
    // do not count as fewer)
    const Shape sh = heuristic_shape(10 * rows >= 9 * pd.dims.max_nodes ? pd.dims.max_nodes : rows, pd.batch, block_threads);
    uint32_t rec = record_max_bytes(pd.dims.num_inputs, pd.dims.num_outputs, pd.dims.max_nodes, pd.dims.max_conns);
    if (max_used > 0) rec = std::min(rec, align16((uint32_t)max_used));
    const size_t reg = ((size_t)rec + 4u * (size_t)((rows * sh.tile + 3) & ~3) + 15) & ~(size_t)15;
    if (!shape_ok(sh, block_threads)) return invalid("invalid launch shape for a population bucket");
    int gpc = block_threads / sh.G;
    if (sh.G > 32) gpc = std::min(gpc, 15);
    while (gpc > 1 && reg * gpc > 200u * 1024u) --gpc;
    if (gpc < 1 || reg * gpc + 16u * forward_header_words(block_threads) > 227u * 1024u)
        return invalid("a genome of this size does not fit one block");
    BucketDev &d = *out;
    d.rec = static_cast<const uint8_t *>(pd.transformed_dev);
    d.gidx = gidx_dev;
    d.x = pd.inputs_dev;
    d.y = pd.outputs_dev;
    d.x_step = pd.in_step_stride;
    d.y_step = pd.out_step_stride;
    d.stride = record_stride(pd.dims);
    d.n_genomes = pd.pop;
    d.I = pd.dims.num_inputs;
    d.O = pd.dims.num_outputs;
    d.B = pd.batch;
    d.tile = sh.tile;
    d.tiles = (pd.batch + sh.tile - 1) / sh.tile;
    d.lg_split = lg(sh.split);
    d.G = sh.G;
    d.lgG = lg(sh.G);
    d.gpc = gpc;
    d.region_words = (int)(reg / 16);
    d.rec_words = (int)(rec / 16);
    d.rec_copy_bytes = own_size ? 0 : (int)rec;
    d.cta_begin = cta_begin;
    d.cta_items = (int)(((long)d.n_genomes * d.tiles + gpc - 1) / gpc);
    d.spare = spare_floats(reg * gpc, pd.dims.max_nodes);
    *footprint = 4u * (size_t)d.spare;
    return NEAT_OK;
}

int launch_plan_table(const BucketDev *table_dev, int nb, int total_items, unsigned int *counter_dev, int step,
                      size_t smem_regions, int block_threads, cudaStream_t s)
{
    if (nb == 0 || total_items == 0) return NEAT_OK;
    const size_t smem = smem_regions + 16u * forward_header_words(block_threads);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, plan_kernel<false>);
    if (e != cudaSuccess) return cuda_fail(e, "plan table: cudaFuncGetAttributes");
    if (smem + fa.sharedSizeBytes > 227u * 1024u) return invalid("plan table: shared memory exceeds 227 KB");
    {
        const int rc = allow_dynamic_smem(reinterpret_cast<const void *>(plan_kernel<false>), smem,
                                          "plan table: shared memory per block");
        if (rc) return rc;
    }
    int dev = 0, sms = 152, smem_sm = 233472;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    const int per_sm = std::max(1, std::min((int)(smem_sm / (smem + 1024)), 2048 / block_threads));
    const int grid = std::max(1, std::min(sms * per_sm, total_items));
    plan_kernel<false><<<grid, block_threads, smem, s>>>(table_dev, nb, 0, total_items, counter_dev, step);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "plan table: launch");
    return NEAT_OK;
}

}  // namespace neat
