// Tensorized mutation and crossover (Section 3.2): node addition writes the
// first NaN row, removal writes NaN over a row, attribute modification
// overwrites one column, and the NEAT operators are built from these, for a
// whole population at once.  The operator hyperparameters are the
// appendix's list; the rules (declared with neat_mutate in neat.h) take
// every random number from caller-supplied inputs: uint32 words decide
// (u < T(p), T(p) = min(floor(p 2^32), 2^32)) and choose (floor(u k / 2^32)),
// float normals give the perturbations.
//
// GB300 mapping: one warp per genome up to 128 node rows and 512 connection
// rows (mutate_warp_kernel, crossover_warp_kernel; above 288 and 208
// connection rows for large populations only), else one block per genome.
// The block forms work in place on the population tensors: the node
// keys and the connections' (in, out, enabled) columns are kept in shared
// memory while the four structural steps run one after another (block-wide
// counts, rank selection by a block scan, first-free-row searches, and for
// feedforward networks a key -> row hash table and a breadth-first
// reachability sweep over the connections); the attribute step then updates
// every present row in parallel.  Crossover: the second parent's node keys and
// (in, out) pairs in shared-memory hash tables (lowest row per key or pair)
// looked up for every row of the first parent.
//
// The warp forms are bound by memory latency (long-scoreboard stalls at 36 to
// 45% of the warps, 45 to 47% of the issue slots).  10 000 Ant-sized genomes:
// mutation 34 us (block of 64 threads per genome: 80 us, 3490 against 1520
// warp instructions per genome; with loops whose remainders wait for each row
// 44 us), crossover 38 us (block of 128: 75 us, 4900 against 1710; with its
// lookups' rows loaded together, which takes 64 registers, no faster).
#include <algorithm>

#include "neat_device.cuh"
#include "neat_internal.h"
#include "neat_hash.cuh"
#include "neat_trace.h"

namespace neat {
namespace {

constexpr int kEvoThreads = 256;
constexpr int kStructWords = 16;
constexpr int kStructNormals = 4;

struct MutArgs {
    float *nodes;
    float *conns;
    const uint32_t *words;
    const float *normals;
    const int32_t *new_keys;
    int pop, N, C, I, O, Np2;
    size_t W, Z;                               // words / normals per genome
    unsigned long long t_node_add, t_node_delete, t_conn_add, t_conn_delete;
    unsigned long long t_bias_m, t_bias_mr, t_resp_m, t_resp_mr, t_w_m, t_w_mr, t_act, t_agg, t_en;
    float bias_mean, bias_std, bias_power, resp_mean, resp_std, resp_power, w_mean, w_std, w_power;
    int act_default, agg_default, n_act, n_agg;
    int act_opt[8], agg_opt[4];
    int feedforward;
};

__device__ __forceinline__ bool below(uint32_t u, unsigned long long t) { return (unsigned long long)u < t; }
__device__ __forceinline__ int choose(uint32_t u, int k)
{
    return (int)(((unsigned long long)u * (unsigned long long)k) >> 32);
}

__device__ __forceinline__ float qnan() { return __int_as_float(0x7fc00000); }

// Block-wide rank selection: rows [0, R) in order, `pred(row)` the
// candidates.  One block scan counts them; then, with the count known to
// every thread, the rows of ranks rank_of(total) (and rank2_of(total), when
// asked for) among the candidates are found (-1 where there are not that
// many).  Returns the first row, the second through *row2, the count
// through *total_out.
template <typename Pred, typename RankOf, typename Rank2Of>
__device__ int select_ranks(int R, Pred pred, RankOf rank_of, Rank2Of rank2_of, int *s_cnt, int *s_row,
                            int *total_out, int *row2)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    const int chunk = (R + nt - 1) / nt;
    const int r0 = min(R, tid * chunk), r1 = min(R, r0 + chunk);
    int c = 0;
    for (int r = r0; r < r1; ++r) c += pred(r) ? 1 : 0;
    // exclusive scan of the per-thread counts: warp scan, then warp totals
    const int lane = tid & 31, warp = tid >> 5;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_cnt[warp] = incl;
    if (tid == 0) s_row[0] = s_row[1] = -1;
    __syncthreads();
    int base = 0, total = 0;
    for (int w = 0; w < nt / 32; ++w) {
        if (w < warp) base += s_cnt[w];
        total += s_cnt[w];
    }
    const int excl = base + incl - c;
    auto find = [&](int rank, int *out) {
        if (rank >= 0 && rank >= excl && rank < excl + c) {
            int k = rank - excl;
            for (int r = r0; r < r1; ++r)
                if (pred(r) && k-- == 0) {
                    *out = r;
                    break;
                }
        }
    };
    find(rank_of(total), s_row);
    find(rank2_of(total), s_row + 1);
    __syncthreads();
    const int row = s_row[0];
    if (row2) *row2 = s_row[1];
    *total_out = total;
    __syncthreads();
    return row;
}

// The candidate of rank `rank` (-1 if there are not that many).
template <typename Pred>
__device__ int select_rank(int R, Pred pred, int rank, int *s_cnt, int *s_row, int *total_out)
{
    return select_ranks(
        R, pred, [=](int) { return rank; }, [](int) { return -1; }, s_cnt, s_row, total_out, nullptr);
}

// The candidate chosen by the random word u among all of them (-1 if none).
template <typename Pred>
__device__ int select_choose(int R, Pred pred, uint32_t u, int *s_cnt, int *s_row, int *total_out)
{
    return select_ranks(
        R, pred, [=](int total) { return total > 0 ? choose(u, total) : -1; }, [](int) { return -1; }, s_cnt,
        s_row, total_out, nullptr);
}

// ------------------------------------------------ a warp per genome
//
// Genomes of at most 128 node rows and 512 connection rows (predecessor masks
// of four words, at most 14 KB a genome): one warp stages the whole genome in shared memory, so that the structural steps need warp
// barriers only and the tensors are read and written once, in full sectors.
// Candidate sets are bit masks (lane k holds rows 32k .. 32k+31), the cycle
// check a sweep over predecessor masks.
constexpr int kWarpNodes = 128, kWarpConns = 512;
constexpr unsigned kAll = 0xffffffffu;
constexpr int kBatch = 4;                // rows a lane has in flight at once

// The mask of rows 32k .. 32k+31 of [0, R) that satisfy pred, on lane k.
template <typename Pred>
__device__ __forceinline__ uint32_t row_mask(int R, Pred pred, int lane)
{
    uint32_t mine = 0;
    for (int k = 0; k * 32 < R; ++k) {
        const int r = k * 32 + lane;
        const unsigned m = __ballot_sync(kAll, r < R && pred(r));
        if (lane == k) mine = m;
    }
    return mine;
}

__device__ __forceinline__ int mask_count(uint32_t mine) { return __reduce_add_sync(kAll, __popc(mine)); }

// The row of rank `rank` (0 <= rank < count) in such a mask.
__device__ __forceinline__ int mask_pick(uint32_t mine, int rank, int lane)
{
    int incl = __popc(mine);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += v;
    }
    const int owner = __ffs(__ballot_sync(kAll, rank < incl)) - 1;
    int row = 0;
    if (lane == owner) {
        uint32_t m = mine;
        for (int k = rank - (incl - __popc(mine)); k > 0; --k) m &= m - 1u;
        row = lane * 32 + __ffs(m) - 1;
    }
    return __shfl_sync(kAll, row, owner);
}

// The lowest row of such a mask (-1 if none).
__device__ __forceinline__ int mask_first(uint32_t mine)
{
    const unsigned some = __ballot_sync(kAll, mine != 0u);
    if (some == 0u) return -1;
    const int owner = __ffs(some) - 1;
    return owner * 32 + __shfl_sync(kAll, __ffs(mine) - 1, owner);
}

struct MutWarpLayout {
    int nodes, preds, ktab, total;           // byte offsets in a warp's shared memory (connections at 0)
};
__host__ __device__ inline MutWarpLayout mut_warp_layout(int N, int C, int Np2)
{
    MutWarpLayout l;
    const int RN = (N + 31) / 32;
    l.nodes = 16 * C;
    l.preds = l.nodes + 20 * N;
    l.ktab = l.preds + 4 * RN * N;
    l.total = (l.ktab + 8 * Np2 + 15) & ~15;
    return l;
}

__global__ void __launch_bounds__(128) mutate_warp_kernel(const MutArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = blockIdx.x * (blockDim.x >> 5) + warp;
    if (g >= a.pop) return;
    const int N = a.N, C = a.C;
    const MutWarpLayout lay = mut_warp_layout(N, C, a.Np2);
    unsigned char *mine = sm + (size_t)warp * lay.total;
    float4 *cs = reinterpret_cast<float4 *>(mine);                // [C] (in, out, enabled, weight)
    float *ns = reinterpret_cast<float *>(mine + lay.nodes);      // [N][5]
    float *nodes = a.nodes + (size_t)g * N * 5;
    float4 *conns = reinterpret_cast<float4 *>(a.conns + (size_t)g * C * 4);
    const uint32_t *u = a.words + (size_t)g * a.W;
    const float *z = a.normals + (size_t)g * a.Z;

    const uint32_t word = lane < 9 ? __ldg(u + lane) : 0u;        // the structural words
    // loads in whole batches, past the last row too (predicated off): a loop's
    // remainder would wait for every row by itself
    for (int base = lane; base < C; base += 32 * kBatch) {
        float4 row[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
            if (base + 32 * j < C) row[j] = conns[base + 32 * j];
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
            if (base + 32 * j < C) cs[base + 32 * j] = row[j];
    }
    for (int base = lane; base < 5 * N; base += 64 * kBatch) {
        float x[2 * kBatch];
#pragma unroll
        for (int j = 0; j < 2 * kBatch; ++j)
            if (base + 32 * j < 5 * N) x[j] = nodes[base + 32 * j];
#pragma unroll
        for (int j = 0; j < 2 * kBatch; ++j)
            if (base + 32 * j < 5 * N) ns[base + 32 * j] = x[j];
    }
    __syncwarp();
    auto u_at = [&](int k) { return __shfl_sync(kAll, word, k); };
    auto node_present = [&](int r) { return !isnan(ns[5 * r]); };
    auto conn_present = [&](int c) { return !(isnan(cs[c].x) || isnan(cs[c].y) || isnan(cs[c].z)); };
    const float4 none = make_float4(qnan(), qnan(), qnan(), qnan());

    // 1. node addition: split a present enabled connection
    if (below(u_at(0), a.t_node_add)) {
        const float nkey = (float)__ldg(a.new_keys + g);
        const uint32_t enabled = row_mask(C, [&](int c) { return conn_present(c) && cs[c].z != 0.0f; }, lane);
        uint32_t free = row_mask(C, [&](int c) { return !conn_present(c); }, lane);
        const int total = mask_count(enabled);
        const int rn = mask_first(row_mask(N, [&](int r) { return !node_present(r); }, lane));
        const int ra = mask_first(free);
        if (ra >= 0 && lane == (ra >> 5)) free &= free - 1u;
        const int rb = mask_first(free);
        bool used = false;
        for (int r = lane; r < N; r += 32) used |= node_present(r) && ns[5 * r] == nkey;
        used = __any_sync(kAll, used);
        if (total > 0 && rn >= 0 && ra >= 0 && rb >= 0 && !used) {
            const int pick = mask_pick(enabled, choose(u_at(1), total), lane);
            __syncwarp();
            if (lane == 0) {
                const float4 old = cs[pick];
                cs[pick].z = 0.0f;
                cs[ra] = make_float4(old.x, nkey, 1.0f, 1.0f);
                cs[rb] = make_float4(nkey, old.y, 1.0f, old.w);
                float *n = ns + 5 * rn;
                n[0] = nkey;
                n[1] = a.bias_mean;
                n[2] = a.resp_mean;
                n[3] = (float)a.agg_default;
                n[4] = (float)a.act_default;
            }
        }
        __syncwarp();
    }

    // 2. node deletion: a hidden node and every connection touching it
    if (below(u_at(2), a.t_node_delete)) {
        const float io_end = (float)(a.I + a.O);
        const uint32_t hidden = row_mask(N, [&](int r) { return node_present(r) && ns[5 * r] >= io_end; }, lane);
        const int total = mask_count(hidden);
        if (total > 0) {
            const int rd = mask_pick(hidden, choose(u_at(3), total), lane);
            const float q = ns[5 * rd];
            for (int c = lane; c < C; c += 32)
                if (conn_present(c) && (cs[c].x == q || cs[c].y == q)) cs[c] = none;
            __syncwarp();
            if (lane < 5) ns[5 * rd + lane] = qnan();
            __syncwarp();
        }
    }

    // 3. connection addition
    if (below(u_at(4), a.t_conn_add)) {
        const float in_end = (float)a.I;
        const uint32_t here = row_mask(N, node_present, lane);
        const uint32_t target = row_mask(N, [&](int r) { return node_present(r) && ns[5 * r] >= in_end; }, lane);
        const int n_src = mask_count(here), n_dst = mask_count(target);
        if (n_src > 0 && n_dst > 0) {
            const float s = ns[5 * mask_pick(here, choose(u_at(5), n_src), lane)];
            const float t = ns[5 * mask_pick(target, choose(u_at(6), n_dst), lane)];
            const int existing = mask_first(
                row_mask(C, [&](int c) { return conn_present(c) && cs[c].x == s && cs[c].y == t; }, lane));
            __syncwarp();
            if (existing >= 0) {
                if (lane == 0) cs[existing].z = 1.0f;
                __syncwarp();
            } else {
                bool reject = false;
                if (a.feedforward && s == t) reject = true;
                else if (a.feedforward) {
                    // rows by key, then every row's predecessors among the
                    // present nodes, then a sweep from t
                    const int RN = (N + 31) >> 5;
                    uint32_t *ktab = reinterpret_cast<uint32_t *>(mine + lay.ktab);    // [2 Np2]
                    uint32_t *preds = reinterpret_cast<uint32_t *>(mine + lay.preds);  // [RN][N]
                    const uint32_t kmask = 2u * (uint32_t)a.Np2 - 1u;
                    const int kshift = __clz(kmask);
                    for (int i = lane; i < 2 * a.Np2; i += 32) ktab[i] = kFree32;
                    for (int i = lane; i < RN * N; i += 32) preds[i] = 0u;
                    __syncwarp();
                    // (a malformed genome's node keys beyond 24 bits do not fit the table:
                    // its rows are searched, by the whole key as in the block form)
                    bool wide = false;
                    for (int r = lane; r < N; r += 32)
                        if (node_present(r)) {
                            const uint32_t key = (uint32_t)ns[5 * r];
                            wide |= key > 0xffffffu;
                            insert32(ktab, kmask, kshift, key & 0xffffffu, (uint32_t)r);
                        }
                    wide = __any_sync(kAll, wide);
                    __syncwarp();                        // the votes order no memory
                    auto row_of = [&](float k) {
                        const uint32_t key = (uint32_t)k;
                        if (!wide) return find32(ktab, kmask, kshift, key);
                        for (int r = 0; r < N; ++r)
                            if (node_present(r) && (uint32_t)ns[5 * r] == key) return r;
                        return -1;
                    };
                    for (int c = lane; c < C; c += 32) {
                        if (!conn_present(c)) continue;
                        const int x = row_of(cs[c].x), y = row_of(cs[c].y);
                        if (x >= 0 && y >= 0) atomicOr(preds + (x >> 5) * N + y, 1u << (x & 31));
                    }
                    __syncwarp();
                    const int row_s = row_of(s), row_t = row_of(t);
                    uint32_t seen = lane == (row_t >> 5) ? 1u << (row_t & 31) : 0u;    // lane k: rows 32k ..
                    for (;;) {
                        uint32_t next = seen;
                        for (int k = 0; k < RN; ++k) {
                            const int r = 32 * k + lane;
                            uint32_t hit = 0;
                            for (int j = 0; j < RN; ++j) {
                                const uint32_t from = __shfl_sync(kAll, seen, j);
                                if (r < N) hit |= preds[j * N + r] & from;
                            }
                            const unsigned m = __ballot_sync(kAll, hit != 0u);
                            if (lane == k) next |= m;
                        }
                        const bool grown = __any_sync(kAll, next != seen);
                        seen = next;
                        reject = (__shfl_sync(kAll, seen, row_s >> 5) >> (row_s & 31)) & 1u;
                        if (reject || !grown) break;
                    }
                }
                if (!reject) {
                    const int rf = mask_first(row_mask(C, [&](int c) { return !conn_present(c); }, lane));
                    __syncwarp();
                    if (rf >= 0 && lane == 0) cs[rf] = make_float4(s, t, 1.0f, fmaf(a.w_std, __ldg(z), a.w_mean));
                    __syncwarp();
                }
            }
        }
    }

    // 4. connection deletion
    if (below(u_at(7), a.t_conn_delete)) {
        const uint32_t present = row_mask(C, conn_present, lane);
        const int total = mask_count(present);
        if (total > 0) {
            const int rc = mask_pick(present, choose(u_at(8), total), lane);
            __syncwarp();
            if (lane == 0) cs[rc] = none;
            __syncwarp();
        }
    }

    // attributes of every present row
    const float in_end = (float)a.I;
    const uint32_t *wc = u + kStructWords + 6 * (size_t)N;
    const float *zc = z + kStructNormals + 2 * (size_t)N;
    for (int base = lane; base < C; base += 32 * kBatch) {
        uint32_t w0[kBatch], w1[kBatch];
        float zz[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int c = base + 32 * j;
            w0[j] = w1[j] = 0xffffffffu;
            zz[j] = 0.0f;
            if (c < C) {
                w0[j] = __ldg(wc + 2 * (size_t)c);
                if (a.t_en) w1[j] = __ldg(wc + 2 * (size_t)c + 1);
                zz[j] = __ldg(zc + c);
            }
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int c = base + 32 * j;
            if (c >= C) break;
            float4 x = cs[c];
            if (!(isnan(x.x) || isnan(x.y) || isnan(x.z))) {
                if (below(w0[j], a.t_w_m)) x.w = fmaf(a.w_power, zz[j], x.w);
                else if (below(w0[j], a.t_w_mr)) x.w = fmaf(a.w_std, zz[j], a.w_mean);
                if (a.t_en && below(w1[j], a.t_en)) x.z = (x.z != 0.0f) ? 0.0f : 1.0f;
            }
            conns[c] = x;
        }
    }
    for (int base = lane; base < N; base += 64) {
        // two rows a lane; only the words that some rate can use
        uint32_t wr[2][6];
        float zr[2][2];
        bool on[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = base + 32 * j;
            on[j] = r < N && !isnan(ns[5 * min(r, N - 1)]) && ns[5 * min(r, N - 1)] >= in_end;
            const uint32_t *w = u + kStructWords + 6 * (size_t)r;
            const float *zz = z + kStructNormals + 2 * (size_t)r;
#pragma unroll
            for (int k = 0; k < 6; ++k) wr[j][k] = 0xffffffffu;
            zr[j][0] = zr[j][1] = 0.0f;
            if (on[j]) {
                if (a.t_bias_m | a.t_bias_mr) {
                    wr[j][0] = __ldg(w);
                    zr[j][0] = __ldg(zz);
                }
                if (a.t_resp_m | a.t_resp_mr) {
                    wr[j][1] = __ldg(w + 1);
                    zr[j][1] = __ldg(zz + 1);
                }
                if (a.t_act && a.n_act > 0) {
                    wr[j][2] = __ldg(w + 2);
                    wr[j][3] = __ldg(w + 3);
                }
                if (a.t_agg && a.n_agg > 0) {
                    wr[j][4] = __ldg(w + 4);
                    wr[j][5] = __ldg(w + 5);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (!on[j]) continue;
            float *n = ns + 5 * (base + 32 * j);
            if (below(wr[j][0], a.t_bias_m)) n[1] = fmaf(a.bias_power, zr[j][0], n[1]);
            else if (below(wr[j][0], a.t_bias_mr)) n[1] = fmaf(a.bias_std, zr[j][0], a.bias_mean);
            if (below(wr[j][1], a.t_resp_m)) n[2] = fmaf(a.resp_power, zr[j][1], n[2]);
            else if (below(wr[j][1], a.t_resp_mr)) n[2] = fmaf(a.resp_std, zr[j][1], a.resp_mean);
            if (a.t_act && a.n_act > 0 && below(wr[j][2], a.t_act)) n[4] = (float)a.act_opt[choose(wr[j][3], a.n_act)];
            if (a.t_agg && a.n_agg > 0 && below(wr[j][4], a.t_agg)) n[3] = (float)a.agg_opt[choose(wr[j][5], a.n_agg)];
        }
    }
    __syncwarp();
#pragma unroll 4
    for (int i = lane; i < 5 * N; i += 32) nodes[i] = ns[i];
}

// ------------------------------------------------ larger: a block per genome
__global__ void __launch_bounds__(kEvoThreads) mutate_kernel(const MutArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    unsigned long long *map = reinterpret_cast<unsigned long long *>(sm);   // [2 Np2] key -> lowest row table
    float *nk = reinterpret_cast<float *>(map + 2 * a.Np2);                  // [N] node keys
    float *ci = nk + a.N;                                                     // [C] in keys
    float *co = ci + a.C;                                                     // [C] out keys
    float *ce = co + a.C;                                                     // [C] enabled
    short *inr = reinterpret_cast<short *>(ce + a.C);                        // [C] rows of the endpoints
    short *outr = inr + a.C;
    unsigned char *seen = reinterpret_cast<unsigned char *>(outr + a.C);     // [N]
    __shared__ int s_cnt[kEvoThreads / 32], s_row[2];
    const int g = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int N = a.N, C = a.C;
    float *nodes = a.nodes + (size_t)g * N * 5;
    float *conns = a.conns + (size_t)g * C * 4;
    const uint32_t *u = a.words + (size_t)g * a.W;
    const float *z = a.normals + (size_t)g * a.Z;

    for (int r = tid; r < N; r += nt) nk[r] = nodes[(size_t)r * 5];
    for (int c = tid; c < C; c += nt) {
        const float4 x = *reinterpret_cast<const float4 *>(conns + (size_t)c * 4);
        ci[c] = x.x;
        co[c] = x.y;
        ce[c] = x.z;
    }
    __syncthreads();
    auto node_present = [&](int r) { return !isnan(nk[r]); };
    auto conn_present = [&](int c) { return !(isnan(ci[c]) || isnan(co[c]) || isnan(ce[c])); };
    auto conn_free = [&](int c) { return !conn_present(c); };
    auto node_free = [&](int r) { return !node_present(r); };
    int total = 0;

    // 1. node addition: split a present enabled connection
    if (below(u[0], a.t_node_add)) {
        const float nkey = (float)__ldg(a.new_keys + g);
        auto enabled = [&](int c) { return conn_present(c) && ce[c] != 0.0f; };
        const int pick = select_choose(C, enabled, u[1], s_cnt, s_row, &total);
        const int rn = select_rank(N, node_free, 0, s_cnt, s_row, &total);
        int rb = -1;
        const int ra = select_ranks(
            C, conn_free, [](int) { return 0; }, [](int) { return 1; }, s_cnt, s_row, &total, &rb);
        bool used = false;
        for (int r = tid; r < N; r += nt) used |= node_present(r) && nk[r] == nkey;
        used = __syncthreads_or(used);
        if (pick >= 0 && rn >= 0 && ra >= 0 && rb >= 0 && !used) {
            if (tid == 0) {
                const float in = ci[pick], out = co[pick], w = conns[(size_t)pick * 4 + 3];
                ce[pick] = 0.0f;
                conns[(size_t)pick * 4 + 2] = 0.0f;
                nk[rn] = nkey;
                float *n = nodes + (size_t)rn * 5;
                n[0] = nkey;
                n[1] = a.bias_mean;
                n[2] = a.resp_mean;
                n[3] = (float)a.agg_default;
                n[4] = (float)a.act_default;
                *reinterpret_cast<float4 *>(conns + (size_t)ra * 4) = make_float4(in, nkey, 1.0f, 1.0f);
                *reinterpret_cast<float4 *>(conns + (size_t)rb * 4) = make_float4(nkey, out, 1.0f, w);
                ci[ra] = in; co[ra] = nkey; ce[ra] = 1.0f;
                ci[rb] = nkey; co[rb] = out; ce[rb] = 1.0f;
            }
        }
        __syncthreads();
    }

    // 2. node deletion: a hidden node and every connection touching it
    if (below(u[2], a.t_node_delete)) {
        const float io_end = (float)(a.I + a.O);
        auto hidden = [&](int r) { return node_present(r) && nk[r] >= io_end; };
        const int rd = select_choose(N, hidden, u[3], s_cnt, s_row, &total);
        if (total > 0) {
            const float q = nk[rd];
            for (int c = tid; c < C; c += nt)
                if (conn_present(c) && (ci[c] == q || co[c] == q)) {
                    *reinterpret_cast<float4 *>(conns + (size_t)c * 4) = make_float4(qnan(), qnan(), qnan(), qnan());
                    ci[c] = co[c] = ce[c] = qnan();
                }
            __syncthreads();
            if (tid == 0) {
                for (int j = 0; j < 5; ++j) nodes[(size_t)rd * 5 + j] = qnan();
                nk[rd] = qnan();
            }
            __syncthreads();
        }
    }

    // 3. connection addition
    if (below(u[4], a.t_conn_add)) {
        const float in_end = (float)a.I;
        auto target = [&](int r) { return node_present(r) && nk[r] >= in_end; };
        int ks = 0, kt = 0;
        const int rs = select_choose(N, node_present, u[5], s_cnt, s_row, &ks);
        const int rt = select_choose(N, target, u[6], s_cnt, s_row, &kt);
        if (ks > 0 && kt > 0) {
            const float s = nk[rs], t = nk[rt];
            const int existing =
                select_rank(C, [&](int c) { return conn_present(c) && ci[c] == s && co[c] == t; }, 0, s_cnt, s_row,
                            &total);
            if (existing >= 0) {
                if (tid == 0) {
                    ce[existing] = 1.0f;
                    conns[(size_t)existing * 4 + 2] = 1.0f;
                }
                __syncthreads();
            } else {
                bool reject = false;
                if (a.feedforward) {
                    if (s == t) {
                        reject = true;
                    } else {
                        // key -> lowest row table of the present nodes, endpoint
                        // rows of the connections, then a sweep from t until s is seen
                        const uint32_t kmask = 2u * (uint32_t)a.Np2 - 1u;
                        for (int i = tid; i < 2 * a.Np2; i += nt) map[i] = kFree;
                        __syncthreads();
                        for (int r = tid; r < N; r += nt)
                            if (node_present(r)) key_insert(map, kmask, (uint32_t)nk[r], (uint32_t)r);
                        __syncthreads();
                        for (int c = tid; c < C; c += nt) {
                            inr[c] = outr[c] = -1;
                            if (conn_present(c)) {
                                inr[c] = (short)key_row(map, kmask, (uint32_t)ci[c]);
                                outr[c] = (short)key_row(map, kmask, (uint32_t)co[c]);
                            }
                        }
                        for (int r = tid; r < N; r += nt) seen[r] = 0;
                        __syncthreads();
                        const int row_s = key_row(map, kmask, (uint32_t)s);
                        const int row_t = key_row(map, kmask, (uint32_t)t);
                        if (tid == 0) seen[row_t] = 1;
                        __syncthreads();
                        for (int it = 0; it <= N; ++it) {
                            bool changed = false;
                            for (int c = tid; c < C; c += nt) {
                                const int x = inr[c], y = outr[c];
                                if (x >= 0 && y >= 0 && seen[x] && !seen[y]) {
                                    seen[y] = 1;
                                    changed = true;
                                }
                            }
                            changed = __syncthreads_or(changed);
                            // read by one thread between two barriers, so the next
                            // pass's writes cannot race with the exit decision
                            const bool hit = __syncthreads_or(tid == 0 && seen[row_s]);
                            if (hit || !changed) break;
                        }
                        reject = seen[row_s] != 0;
                        __syncthreads();
                    }
                }
                if (!reject) {
                    const int rf = select_rank(C, conn_free, 0, s_cnt, s_row, &total);
                    if (rf >= 0 && tid == 0) {
                        const float w = fmaf(a.w_std, z[0], a.w_mean);
                        *reinterpret_cast<float4 *>(conns + (size_t)rf * 4) = make_float4(s, t, 1.0f, w);
                        ci[rf] = s; co[rf] = t; ce[rf] = 1.0f;
                    }
                    __syncthreads();
                }
            }
        }
    }

    // 4. connection deletion
    if (below(u[7], a.t_conn_delete)) {
        const int rc = select_choose(C, conn_present, u[8], s_cnt, s_row, &total);
        if (total > 0) {
            if (tid == 0) {
                *reinterpret_cast<float4 *>(conns + (size_t)rc * 4) = make_float4(qnan(), qnan(), qnan(), qnan());
                ci[rc] = co[rc] = ce[rc] = qnan();
            }
            __syncthreads();
        }
    }

    // attributes of every present row
    const float in_end = (float)a.I;
    for (int r = tid; r < N; r += nt) {
        if (!node_present(r) || nk[r] < in_end) continue;
        float *n = nodes + (size_t)r * 5;
        const uint32_t *w = u + kStructWords + 6 * (size_t)r;
        const float *zz = z + kStructNormals + 2 * (size_t)r;
        if (below(w[0], a.t_bias_m)) n[1] = fmaf(a.bias_power, zz[0], n[1]);
        else if (below(w[0], a.t_bias_mr)) n[1] = fmaf(a.bias_std, zz[0], a.bias_mean);
        if (below(w[1], a.t_resp_m)) n[2] = fmaf(a.resp_power, zz[1], n[2]);
        else if (below(w[1], a.t_resp_mr)) n[2] = fmaf(a.resp_std, zz[1], a.resp_mean);
        if (a.n_act > 0 && below(w[2], a.t_act)) n[4] = (float)a.act_opt[choose(w[3], a.n_act)];
        if (a.n_agg > 0 && below(w[4], a.t_agg)) n[3] = (float)a.agg_opt[choose(w[5], a.n_agg)];
    }
    for (int c = tid; c < C; c += nt) {
        if (!conn_present(c)) continue;
        float *x = conns + (size_t)c * 4;
        const uint32_t *w = u + kStructWords + 6 * (size_t)N + 2 * (size_t)c;
        const float zz = z[kStructNormals + 2 * (size_t)N + c];
        if (below(w[0], a.t_w_m)) x[3] = fmaf(a.w_power, zz, x[3]);
        else if (below(w[0], a.t_w_mr)) x[3] = fmaf(a.w_std, zz, a.w_mean);
        if (below(w[1], a.t_en)) x[2] = (ce[c] != 0.0f) ? 0.0f : 1.0f;
    }
}

struct CrossArgs {
    const float *nodes;
    const float *conns;
    const int32_t *parents;
    const uint32_t *words;
    float *nodes_out;
    float *conns_out;
    int pop, K, N, C, Np2, Cp2;
};

// A child whose parent index lies outside [0, pop) is written empty (every
// row NaN) by threads i, i + step, ...
__device__ __forceinline__ void write_empty_child(float *no, float4 *co, int N, int C, int lane, int step)
{
    for (int e = lane; e < N * 5; e += step) no[e] = __int_as_float(0x7fc00000);
    const float q = __int_as_float(0x7fc00000);
    for (int c = lane; c < C; c += step) co[c] = make_float4(q, q, q, q);
}

// One warp per child, for parents of at most 128 node rows and 512 connection
// rows.  The second parent's connections sit in a 32-bit table (22 bits of the
// pair's hash | row); a lookup that matches reads the row it names, whose keys
// decide and whose attributes are what the child takes.
struct CrossWarpLayout {
    int ntab, ctab, total;                   // byte offsets in a warp's shared memory (child's nodes at 0)
};
__host__ __device__ inline CrossWarpLayout cross_warp_layout(int N, int Np2, int Cp2)
{
    CrossWarpLayout l;
    l.ntab = (20 * N + 15) & ~15;
    l.ctab = l.ntab + 8 * Np2;               // 2 Np2 words
    l.total = (l.ctab + 8 * Cp2 + 15) & ~15; // 2 Cp2 words
    return l;
}

__device__ __forceinline__ uint32_t pair_hash(uint32_t ki, uint32_t ko)
{
    // finalised with a multiplier of Wellons's hash prospector (2c1b3c6d)
    uint32_t h = ki * 0x9E3779B1u + ko * 0x85EBCA6Bu;
    h ^= h >> 15;
    h *= 0x2C1B3C6Du;
    return h ^ (h >> 13);
}

__global__ void __launch_bounds__(128) crossover_warp_kernel(const CrossArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * (blockDim.x >> 5) + warp;
    if (k >= a.K) return;
    const int N = a.N, C = a.C;
    const CrossWarpLayout lay = cross_warp_layout(N, a.Np2, a.Cp2);
    unsigned char *mine = sm + (size_t)warp * lay.total;
    float *ns = reinterpret_cast<float *>(mine);                             // [N][5]
    uint32_t *ntab = reinterpret_cast<uint32_t *>(mine + lay.ntab);          // key << 8 | lowest row of p2
    uint32_t *ctab = reinterpret_cast<uint32_t *>(mine + lay.ctab);          // hash bits << 10 | lowest row of p2
    const uint32_t nmask = 2u * (uint32_t)a.Np2 - 1u, cmask = 2u * (uint32_t)a.Cp2 - 1u;
    const int nshift = __clz(nmask), cshift = __clz(cmask);
    float *no = a.nodes_out + (size_t)k * N * 5;
    float4 *co = reinterpret_cast<float4 *>(a.conns_out + (size_t)k * C * 4);
    const int p1 = __ldg(a.parents + 2 * k), p2 = __ldg(a.parents + 2 * k + 1);
    if (p1 < 0 || p1 >= a.pop || p2 < 0 || p2 >= a.pop) {
        write_empty_child(no, co, N, C, lane, 32);
        return;
    }
    const float *n1 = a.nodes + (size_t)p1 * N * 5, *n2 = a.nodes + (size_t)p2 * N * 5;
    const float4 *c1 = reinterpret_cast<const float4 *>(a.conns + (size_t)p1 * C * 4);
    const float4 *c2 = reinterpret_cast<const float4 *>(a.conns + (size_t)p2 * C * 4);
    const uint32_t *w = a.words + (size_t)k * (N + C);
    constexpr int kAhead = 4;                                                // rows loaded ahead per lane
    float4 row[kAhead];
    auto load_rows = [&](const float4 *from, int base) {
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int c = base + 32 * j + lane;
            row[j] = make_float4(qnan(), 0.0f, 0.0f, 0.0f);
            if (c < C) row[j] = __ldg(from + c);
        }
    };
    load_rows(c2, 0);
#pragma unroll 4
    for (int i = lane; i < 5 * N; i += 32) ns[i] = __ldg(n1 + i);
    for (int i = lane; i < 2 * (a.Np2 + a.Cp2); i += 32) ntab[i] = kFree32;  // both tables
    __syncwarp();
    for (int r = lane; r < N; r += 32) {
        const float key = __ldg(n2 + (size_t)r * 5);
        if (is_key(key)) insert32(ntab, nmask, nshift, (uint32_t)key, (uint32_t)r);
    }
    for (int base = 0; base < C; base += 32 * kAhead) {
        if (base) load_rows(c2, base);
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int c = base + 32 * j + lane;
            const float4 y = row[j];
            if (!(is_key(y.x) && is_key(y.y) && !isnan(y.z))) continue;      // NaN past the last row
            const uint32_t h = pair_hash((uint32_t)y.x, (uint32_t)y.y);
            const uint32_t v = (h << 10) | (uint32_t)c;
            uint32_t s = h >> cshift;
            for (;;) {                                                       // at most half the slots are taken
                const uint32_t old = atomicCAS(ctab + s, kFree32, v);
                if (old == kFree32) break;
                if ((old >> 10) == (v >> 10)) {
                    const float4 o = __ldg(c2 + (old & 0x3ffu));
                    if (o.x == y.x && o.y == y.y) {                          // the pair's lowest row stays
                        atomicMin(ctab + s, v);
                        break;
                    }
                }
                s = (s + 1u) & cmask;
            }
        }
    }
    load_rows(c1, 0);
    __syncwarp();
    for (int base = 0; base < C; base += 32 * kAhead) {
        if (base) load_rows(c1, base);
        uint32_t word[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int c = base + 32 * j + lane;
            word[j] = c < C ? __ldg(w + N + c) : 0u;
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int c = base + 32 * j + lane;
            float4 x = row[j];
            if (word[j] >= 0x80000000u && is_key(x.x) && is_key(x.y) && !isnan(x.z)) {
                const uint32_t h = pair_hash((uint32_t)x.x, (uint32_t)x.y);
                const uint32_t bits = h & 0x3fffffu;
                uint32_t s = h >> cshift;
                for (;;) {
                    const uint32_t v = ctab[s];
                    if (v == kFree32) break;
                    if ((v >> 10) == bits) {
                        const float4 y = __ldg(c2 + (v & 0x3ffu));
                        if (y.x == x.x && y.y == x.y) {
                            x.z = y.z;
                            x.w = y.w;
                            break;
                        }
                    }
                    s = (s + 1u) & cmask;
                }
            }
            if (c < C) co[c] = x;
        }
    }
    for (int r = lane; r < N; r += 32) {
        const float key = ns[5 * r];
        if (__ldg(w + r) >= 0x80000000u && is_key(key)) {
            const int q = find32(ntab, nmask, nshift, (uint32_t)key);        // p2's lowest row with the key
            if (q >= 0) {
                const float *y = n2 + (size_t)q * 5;
#pragma unroll
                for (int j = 1; j < 5; ++j) ns[5 * r + j] = __ldg(y + j);
            }
        }
    }
    __syncwarp();
#pragma unroll 4
    for (int i = lane; i < 5 * N; i += 32) no[i] = ns[i];
}

__global__ void __launch_bounds__(kEvoThreads) crossover_kernel(const CrossArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    unsigned long long *ntab = reinterpret_cast<unsigned long long *>(sm);   // key -> lowest row of p2
    unsigned long long *ctab = ntab + 2 * a.Np2;                              // (in, out) -> lowest row of p2
    const uint32_t nmask = 2u * (uint32_t)a.Np2 - 1u, cmask = 2u * (uint32_t)a.Cp2 - 1u;
    const int k = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int N = a.N, C = a.C;
    const int p1 = __ldg(a.parents + 2 * k), p2 = __ldg(a.parents + 2 * k + 1);
    if (p1 < 0 || p1 >= a.pop || p2 < 0 || p2 >= a.pop) {
        write_empty_child(a.nodes_out + (size_t)k * N * 5, reinterpret_cast<float4 *>(a.conns_out + (size_t)k * C * 4),
                          N, C, tid, nt);
        return;
    }
    const float *n1 = a.nodes + (size_t)p1 * N * 5, *n2 = a.nodes + (size_t)p2 * N * 5;
    const float *c1 = a.conns + (size_t)p1 * C * 4, *c2 = a.conns + (size_t)p2 * C * 4;
    float *no = a.nodes_out + (size_t)k * N * 5;
    float *co = a.conns_out + (size_t)k * C * 4;
    const uint32_t *w = a.words + (size_t)k * (N + C);
    for (int i = tid; i < 2 * a.Np2; i += nt) ntab[i] = kFree;
    for (int i = tid; i < 2 * a.Cp2; i += nt) ctab[i] = kFree;
    __syncthreads();
    for (int r = tid; r < N; r += nt) {
        const float key = __ldg(n2 + (size_t)r * 5);
        if (is_key(key)) key_insert(ntab, nmask, (uint32_t)key, (uint32_t)r);
    }
    for (int c = tid; c < C; c += nt) {
        const float4 y = __ldg(reinterpret_cast<const float4 *>(c2) + c);
        if (is_key(y.x) && is_key(y.y) && !isnan(y.z))
            pair_row_insert(ctab, cmask, ((unsigned long long)(uint32_t)y.x << 24) | (uint32_t)y.y, (uint32_t)c);
    }
    __syncthreads();
    for (int r = tid; r < N; r += nt) {
        const float *x = n1 + (size_t)r * 5;
        float v[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = __ldg(x + j);
        if (is_key(v[0]) && w[r] >= 0x80000000u) {
            const int q = key_row(ntab, nmask, (uint32_t)v[0]);     // p2's lowest row with the key
            if (q >= 0) {
                const float *y = n2 + (size_t)q * 5;
#pragma unroll
                for (int j = 1; j < 5; ++j) v[j] = __ldg(y + j);
            }
        }
#pragma unroll
        for (int j = 0; j < 5; ++j) no[(size_t)r * 5 + j] = v[j];
    }
    for (int c = tid; c < C; c += nt) {
        float4 x = __ldg(reinterpret_cast<const float4 *>(c1) + c);
        if (is_key(x.x) && is_key(x.y) && !isnan(x.z) && w[N + c] >= 0x80000000u) {
            const int q = pair_row(ctab, cmask, ((unsigned long long)(uint32_t)x.x << 24) | (uint32_t)x.y);
            if (q >= 0) {
                const float4 y = __ldg(reinterpret_cast<const float4 *>(c2) + q);
                x.z = y.z;
                x.w = y.w;
            }
        }
        reinterpret_cast<float4 *>(co)[c] = x;
    }
}

unsigned long long threshold(double p)
{
    if (!(p > 0.0)) return 0ull;
    const double t = std::floor(p * 4294967296.0);
    return t >= 4294967296.0 ? 4294967296ull : (unsigned long long)t;
}

int pow2_at_least(int x)
{
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

}  // namespace
}  // namespace neat

using namespace neat;

extern "C" int neat_mutation_sizes(neat_dims d, int64_t *words, int64_t *normals)
{
    if (!dims_ok(d) || !words || !normals) return invalid("neat_mutation_sizes: invalid argument");
    *words = kStructWords + 6 * (int64_t)d.max_nodes + 2 * (int64_t)d.max_conns;
    *normals = kStructNormals + 2 * (int64_t)d.max_nodes + (int64_t)d.max_conns;
    return NEAT_OK;
}

extern "C" int neat_mutate(float *nodes_dev, float *conns_dev, int32_t pop, neat_dims d, const neat_mutation *m,
                           const uint32_t *words_dev, const float *normals_dev, const int32_t *new_keys_dev,
                           void *stream)
{
    TraceRange trace_range("neat_mutate");
    clear_error();
    if (!dims_ok(d) || !m) return invalid("neat_mutate: invalid dims or config");
    if (pop < 0) return invalid("neat_mutate: pop < 0");
    if (pop == 0) return NEAT_OK;
    if (!nodes_dev || (!conns_dev && d.max_conns > 0) || !words_dev || !normals_dev || !new_keys_dev)
        return invalid("neat_mutate: null pointer");
    if (reinterpret_cast<uintptr_t>(conns_dev) & 15u) return invalid("neat_mutate: conns must be 16-byte aligned");
    if (m->n_activation_options < 0 || m->n_activation_options > 8 || m->n_aggregation_options < 0 ||
        m->n_aggregation_options > 4)
        return invalid("neat_mutate: option counts out of range");
    MutArgs a;
    a.nodes = nodes_dev;
    a.conns = conns_dev;
    a.words = words_dev;
    a.normals = normals_dev;
    a.new_keys = new_keys_dev;
    a.pop = pop;
    a.N = d.max_nodes;
    a.C = d.max_conns;
    a.I = d.num_inputs;
    a.O = d.num_outputs;
    a.Np2 = pow2_at_least(a.N);
    a.W = kStructWords + 6 * (size_t)a.N + 2 * (size_t)a.C;
    a.Z = kStructNormals + 2 * (size_t)a.N + (size_t)a.C;
    a.t_node_add = threshold(m->node_add);
    a.t_node_delete = threshold(m->node_delete);
    a.t_conn_add = threshold(m->conn_add);
    a.t_conn_delete = threshold(m->conn_delete);
    a.t_bias_m = threshold(m->bias_mutate_rate);
    a.t_bias_mr = threshold((double)m->bias_mutate_rate + (double)m->bias_replace_rate);
    a.t_resp_m = threshold(m->response_mutate_rate);
    a.t_resp_mr = threshold((double)m->response_mutate_rate + (double)m->response_replace_rate);
    a.t_w_m = threshold(m->weight_mutate_rate);
    a.t_w_mr = threshold((double)m->weight_mutate_rate + (double)m->weight_replace_rate);
    a.t_act = threshold(m->activation_replace_rate);
    a.t_agg = threshold(m->aggregation_replace_rate);
    a.t_en = threshold(m->enabled_mutate_rate);
    a.bias_mean = m->bias_init_mean;
    a.bias_std = m->bias_init_std;
    a.bias_power = m->bias_mutate_power;
    a.resp_mean = m->response_init_mean;
    a.resp_std = m->response_init_std;
    a.resp_power = m->response_mutate_power;
    a.w_mean = m->weight_init_mean;
    a.w_std = m->weight_init_std;
    a.w_power = m->weight_mutate_power;
    a.act_default = m->activation_default;
    a.agg_default = m->aggregation_default;
    a.n_act = m->n_activation_options;
    a.n_agg = m->n_aggregation_options;
    for (int i = 0; i < 8; ++i) a.act_opt[i] = m->activation_options[i];
    for (int i = 0; i < 4; ++i) a.agg_opt[i] = m->aggregation_options[i];
    a.feedforward = m->feedforward != 0;
    // above 288 rows a lone warp's chain is the longer one until there are
    // genomes enough to hide it (97 / 388 rows: 500 genomes 17.5 us, 14.7 by
    // blocks; 2000: 17.3 and 24.0)
    if (a.N <= kWarpNodes && a.C <= kWarpConns && (a.C <= 288 || pop >= 1500)) {
        const int warps = pop > 4 * 152 ? 4 : 1;
        const size_t bytes = (size_t)warps * mut_warp_layout(a.N, a.C, a.Np2).total;
        const int rw = allow_dynamic_smem(reinterpret_cast<const void *>(mutate_warp_kernel), bytes,
                                          "neat_mutate: shared memory");
        if (rw) return rw;
        mutate_warp_kernel<<<(pop + warps - 1) / warps, 32 * warps, bytes, as_stream(stream)>>>(a);
        const cudaError_t ew = cudaGetLastError();
        if (ew != cudaSuccess) return cuda_fail(ew, "neat_mutate: launch");
        return NEAT_OK;
    }
    const size_t smem = 16u * (size_t)a.Np2 + 4u * (size_t)a.N + 12u * (size_t)a.C + 4u * (size_t)a.C +
                        (size_t)a.N + 16u;
    int rc = allow_dynamic_smem(reinterpret_cast<const void *>(mutate_kernel), smem, "neat_mutate: shared memory");
    if (rc) return rc;
    mutate_kernel<<<pop, kEvoThreads, smem, as_stream(stream)>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_mutate: launch");
    return NEAT_OK;
}

extern "C" int neat_crossover(const float *nodes_dev, const float *conns_dev, int32_t pop, neat_dims d,
                              const int32_t *parents_dev, int32_t n_children, const uint32_t *words_dev,
                              float *nodes_out_dev, float *conns_out_dev, void *stream)
{
    TraceRange trace_range("neat_crossover");
    clear_error();
    if (!dims_ok(d)) return invalid("neat_crossover: invalid dims");
    if (pop < 0 || n_children < 0) return invalid("neat_crossover: sizes must be >= 0");
    if (n_children == 0) return NEAT_OK;
    if (!nodes_dev || (!conns_dev && d.max_conns > 0) || !parents_dev || !words_dev || !nodes_out_dev ||
        (!conns_out_dev && d.max_conns > 0))
        return invalid("neat_crossover: null pointer");
    if ((reinterpret_cast<uintptr_t>(conns_dev) & 15u) || (reinterpret_cast<uintptr_t>(conns_out_dev) & 15u))
        return invalid("neat_crossover: connection tensors must be 16-byte aligned");
    CrossArgs a;
    a.nodes = nodes_dev;
    a.conns = conns_dev;
    a.parents = parents_dev;
    a.words = words_dev;
    a.nodes_out = nodes_out_dev;
    a.conns_out = conns_out_dev;
    a.pop = pop;
    a.K = n_children;
    a.N = d.max_nodes;
    a.C = d.max_conns;
    a.Np2 = pow2_at_least(a.N);
    a.Cp2 = pow2_at_least(a.C > 0 ? a.C : 1);
    // the same from 208 rows on, with the longer chain of lookups (72 / 289
    // rows: 1000 children 20.7 us, 12.7 by blocks; 4000: 24.8 and 30.6; 128 /
    // 512: 4000 51.7 and 50.8)
    if (a.N <= kWarpNodes && a.C <= kWarpConns && (a.C <= 208 || n_children >= 12 * a.C)) {
        const int warps = n_children > 4 * 152 ? 4 : 1;
        const size_t bytes = (size_t)warps * cross_warp_layout(a.N, a.Np2, a.Cp2).total;
        const int rw = allow_dynamic_smem(reinterpret_cast<const void *>(crossover_warp_kernel), bytes,
                                          "neat_crossover: shared memory");
        if (rw) return rw;
        crossover_warp_kernel<<<(n_children + warps - 1) / warps, 32 * warps, bytes, as_stream(stream)>>>(a);
        const cudaError_t ew = cudaGetLastError();
        if (ew != cudaSuccess) return cuda_fail(ew, "neat_crossover: launch");
        return NEAT_OK;
    }
    const size_t smem = 16u * ((size_t)a.Np2 + (size_t)a.Cp2);
    int rc = allow_dynamic_smem(reinterpret_cast<const void *>(crossover_kernel), smem, "neat_crossover: shared memory");
    if (rc) return rc;
    crossover_kernel<<<n_children, kEvoThreads, smem, as_stream(stream)>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_crossover: launch");
    return NEAT_OK;
}
