// HyperNEAT substrate evaluation (the CPPN / HyperNEAT extensions of Section
// 4.3): the weight blocks written by neat_cppn_query define a layered
// network over the substrate grid, evaluated here for a batch of input
// vectors per genome: layer 0 = the R = res^2 inputs, layer l+1 node
// t = act(sum_s W_l[s][t] v_l[s]) (no bias; hidden_act inside, output_act on
// the last layer).
//
// GB300 mapping: for the control setting (one or a few input vectors per
// genome) this is a batched matrix-vector product whose cost is reading the
// fp32 weight blocks once from HBM (2 x 256 KB per genome at 16 x 16), so it
// runs on the FP32 pipes at the bandwidth roofline rather than on tensor
// cores, which would also round the weights below the float tolerance.  One
// block per (genome, batch chunk of NB vectors): each thread owns VEC
// adjacent target columns of one slice of the sources (the slices are
// equal runs of consecutive rows), keeps NB x VEC accumulators in registers,
// and the slices are summed in a fixed order through shared memory, where
// the layer's values also stay, so the result is a function of the inputs
// alone.  The weights stream through shared memory by TMA bulk copies of
// whole source rows (substrate_tma_kernel, tiles of up to 4 vectors, near
// the HBM roofline at one vector per genome); shapes it cannot take (R not a
// multiple of 4) use per-thread VEC-wide read-only loads (substrate_kernel).
// Both accumulate compensated dot products and give the same bits.
//
// Bounds: at one vector per genome the weights' stream (1000 genomes of 3
// layers of 16 x 16: 90 us, 5.8 TB/s); at 16 the ten FP32 operations of a
// compensated step, run as packed pairs so that they take half the issue
// slots: 0.74 ms, 74% of the FP32 lanes (scalar 0.92 ms, 59%).
#include <algorithm>

#include "neat_device.cuh"
#include "neat_internal.h"
#include "neat_trace.h"

namespace neat {
namespace {

constexpr int kSubThreads = 256;

struct SubArgs {
    const float *w;        // [pop][L-1][R][R]
    const float *x;        // [pop][B][R]
    float *y;              // [pop][B][R]
    int R, L, B;
    int hidden_act, output_act;
    int groups;            // slices of the source range (threads per column group)
    int cols;              // column groups per pass (cols * groups <= threads)
    int stage_rows;        // bulk-copy path: source rows per shared-memory stage
    int tiles;             // vector tiles per genome
};

__device__ unsigned int g_substrate_error;

// Compensated dot products.  Error-free transformations of Ogita, Rump and
// Oishi ("Accurate sum and dot product", SIAM J. Sci. Comput. 26(6), 2005):
// TwoSum (after Knuth) and TwoProduct by one FMA.  dot2_step adds x*w to the
// pair (s, c), s the rounded running sum and c the sum of the rounding
// errors; s + c is as accurate as the dot product in twice the working
// precision, so sums of large weights stay within the float tolerance.  The
// _rn intrinsics keep the compiler from contracting or reassociating them.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}

__device__ __forceinline__ void dot2_step(float &s, float &c, float x, float w)
{
    const float p = __fmul_rn(x, w);
    const float pe = __fmaf_rn(x, w, -p);                  // x*w - p, exactly
    float t, e;
    two_sum(s, p, t, e);
    s = t;
    c = __fadd_rn(c, __fadd_rn(e, pe));
}

// dot2_step on two accumulators at once, x2 * w2 half by half, nw2 = -w2: the
// operations of dot2_step with the product's error held negated (p - x*w
// exactly), so c takes e - (-pe); the same bits in half the issue slots.
__device__ __forceinline__ void dot2_step2(f2 &s, f2 &c, f2 x2, f2 w2, f2 nw2)
{
    const f2 p = mul2(x2, w2);
    const f2 npe = fma2(x2, nw2, p);
    const f2 t = add2(s, p);
    const f2 z = sub2(t, s);
    const f2 e = add2(sub2(s, sub2(t, z)), sub2(p, z));
    s = t;
    c = add2(c, sub2(e, npe));
}

// The slices' (s, c) pairs added in slice order, rounded once at the end.
__device__ __forceinline__ float combine_slices(const float *ps, const float *pc, size_t stride, int groups)
{
    float S = ps[0], C = pc[0];
    for (int j = 1; j < groups; ++j) {
        float t, e;
        two_sum(S, ps[(size_t)j * stride], t, e);
        S = t;
        C = __fadd_rn(C, __fadd_rn(e, pc[(size_t)j * stride]));
    }
    return __fadd_rn(S, C);
}

template <int VEC>
struct VecT;
template <>
struct VecT<1> {
    using T = float;
    static __device__ __forceinline__ float get(const float &v, int) { return v; }
};
template <>
struct VecT<4> {
    using T = float4;
    static __device__ __forceinline__ float get(const float4 &v, int i)
    {
        return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
    }
};

template <int NB, int VEC>
__global__ void __launch_bounds__(kSubThreads) substrate_kernel(const SubArgs a)
{
    extern __shared__ __align__(16) float sm[];
    const int R = a.R;
    float *cur = sm;                       // [NB][R]
    float *nxt = cur + NB * R;             // [NB][R]
    float *ps = nxt + NB * R;              // [groups][NB][R] slice sums
    float *pc = ps + (size_t)a.groups * NB * R;   // [groups][NB][R] their rounding errors
    // a genome's vector tiles are neighbours in the grid: they share its weights in L2
    const int g = blockIdx.x / a.tiles, b0 = (blockIdx.x - g * a.tiles) * NB;
    const int nb = min(NB, a.B - b0);
    const int tid = threadIdx.x;
    const float *xg = a.x + ((size_t)g * a.B + b0) * R;
    for (int i = tid; i < NB * R; i += kSubThreads) cur[i] = (i < nb * R) ? __ldg(xg + i) : 0.0f;
    __syncthreads();
    const int ncols = R / VEC;                              // column groups in a row
    const int slice = (R + a.groups - 1) / a.groups;        // sources per slice
    const int col_in_pass = tid % a.cols, grp = tid / a.cols;
    using V = typename VecT<VEC>::T;
    for (int l = 0; l + 1 < a.L; ++l) {
        const float *Wl = a.w + ((size_t)g * (a.L - 1) + l) * (size_t)R * R;
        const int act = (l + 2 == a.L) ? a.output_act : a.hidden_act;
        for (int c0 = 0; c0 < ncols; c0 += a.cols) {
            const int c = c0 + col_in_pass;
            if (grp < a.groups && c < ncols) {
                // accumulators in pairs: of columns, or of vectors where a thread
                // has one column and sixteen.  With one column and fewer vectors
                // the pairs of vectors cost registers (125 instead of 48 at
                // eight) and what they save is not what bounds it: scalar sums
                // (427 substrates of 15 x 15, 8 vectors: 102 us, 151 in pairs)
                constexpr bool kPairs = VEC > 1 || NB > 8;
                constexpr int kAcc = kPairs ? NB * VEC / 2 : 1;
                f2 as[kAcc], ac[kAcc];
                constexpr int kOne = kPairs ? 1 : NB;
                float s1f[kOne], c1f[kOne];
#pragma unroll
                for (int b = 0; b < kOne; ++b) s1f[b] = c1f[b] = 0.0f;
#pragma unroll
                for (int k = 0; k < kAcc; ++k) as[k] = ac[k] = 0ull;
                const int s0 = grp * slice, s1 = min(R, s0 + slice);
                const V *col = reinterpret_cast<const V *>(Wl) + c;
#pragma unroll 8
                for (int s = s0; s < s1; ++s) {
                    const V wv = __ldg(col + (size_t)s * ncols);
                    if constexpr (!kPairs) {
#pragma unroll
                        for (int b = 0; b < NB; ++b) dot2_step(s1f[b], c1f[b], cur[b * R + s], VecT<VEC>::get(wv, 0));
                    } else if constexpr (VEC == 1) {
                        const f2 w2 = pack2(VecT<VEC>::get(wv, 0), VecT<VEC>::get(wv, 0)), nw2 = neg2(w2);
#pragma unroll
                        for (int b = 0; b < NB; b += 2)
                            dot2_step2(as[b / 2], ac[b / 2], pack2(cur[b * R + s], cur[(b + 1) * R + s]), w2, nw2);
                    } else {
                        f2 w2[VEC / 2], nw2[VEC / 2];
#pragma unroll
                        for (int v = 0; v < VEC; v += 2) {
                            w2[v / 2] = pack2(VecT<VEC>::get(wv, v), VecT<VEC>::get(wv, v + 1));
                            nw2[v / 2] = neg2(w2[v / 2]);
                        }
#pragma unroll
                        for (int b = 0; b < NB; ++b) {
                            const f2 x2 = pack2(cur[b * R + s], cur[b * R + s]);
#pragma unroll
                            for (int k = 0; k < VEC / 2; ++k)
                                dot2_step2(as[b * (VEC / 2) + k], ac[b * (VEC / 2) + k], x2, w2[k], nw2[k]);
                        }
                    }
                }
                auto put = [&](int b, int v, float sum, float err) {
                    ps[((size_t)grp * NB + b) * R + c * VEC + v] = sum;
                    pc[((size_t)grp * NB + b) * R + c * VEC + v] = err;
                };
                if constexpr (!kPairs) {
#pragma unroll
                    for (int b = 0; b < NB; ++b) put(b, 0, s1f[b], c1f[b]);
                } else {
#pragma unroll
                    for (int k = 0; k < kAcc; ++k) {
                        const float2 sk = unpack2(as[k]), ck = unpack2(ac[k]);
                        if constexpr (VEC == 1) {
                            put(2 * k, 0, sk.x, ck.x);
                            put(2 * k + 1, 0, sk.y, ck.y);
                        } else {
                            const int b = k / (VEC / 2), v = 2 * (k % (VEC / 2));
                            put(b, v, sk.x, ck.x);
                            put(b, v + 1, sk.y, ck.y);
                        }
                    }
                }
            }
            __syncthreads();
            // sum the slices in order, apply the activation
            for (int i = tid; i < NB * a.cols * VEC; i += kSubThreads) {
                const int b = i / (a.cols * VEC), t = c0 * VEC + i % (a.cols * VEC);
                if (t >= R) continue;
                nxt[b * R + t] = activate((uint32_t)act, combine_slices(ps + (size_t)b * R + t, pc + (size_t)b * R + t,
                                                                         (size_t)NB * R, a.groups));
            }
            __syncthreads();
        }
        float *tmp = cur;
        cur = nxt;
        nxt = tmp;
    }
    float *yg = a.y + ((size_t)g * a.B + b0) * R;
    for (int i = tid; i < nb * R; i += kSubThreads) yg[i] = cur[i];
}

// The same layers with the weights streamed through shared memory by bulk
// copies (TMA): each stage is `stage_rows` consecutive source rows, which
// are contiguous in the source-major block; two stages are in flight, each
// completing on its own mbarrier (bounded waits).  The sources are split
// into `groups` slices (equal runs of consecutive rows) and a stage holds
// the next stage_rows / groups rows of every slice, one bulk copy each, so
// every thread works on every stage: thread (col, grp) owns the 4 target
// columns col*4 .. col*4+3 and adds the rows of slice grp, in increasing s,
// for its NB vectors; the slices' partial sums are added in order through
// shared memory.  The operations and their order are those of
// substrate_kernel, so the bits are the same.  Needs R % 4 == 0, R / 4
// dividing the block, and the per-slice stage rows dividing the slice.
template <int NB>
__global__ void __launch_bounds__(kSubThreads) substrate_tma_kernel(const SubArgs a)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int failed;
    const int R = a.R, rows = a.stage_rows;
    float *stage = sm;                                      // [2][rows][R]
    // values, each twice (both halves of a pair)
    float2 *cur = reinterpret_cast<float2 *>(stage + 2 * (size_t)rows * R);   // [NB][R]
    float2 *nxt = cur + NB * R;                                               // [NB][R]
    // slice sums and their rounding errors [groups][NB][R], in the stages'
    // memory once a layer's stages are used up
    float *ps = stage, *pc = ps + (size_t)(kSubThreads / (R / 4)) * NB * R;
    // a genome's vector tiles are neighbours in the grid: they share its weights in L2
    const int g = blockIdx.x / a.tiles, b0 = (blockIdx.x - g * a.tiles) * NB;
    const int nb = min(NB, a.B - b0);
    const int tid = threadIdx.x;
    const int ncols = R / 4, groups = kSubThreads / ncols;
    const int slen = R / groups;                            // sources per slice (R % groups == 0)
    const int col = tid % ncols, grp = tid / ncols;
    const uint32_t bar0 = smem_addr(&bars[0]), bar1 = smem_addr(&bars[1]);
    const int rps = rows / groups;                          // rows of each slice per stage
    const uint32_t slice_bytes = (uint32_t)rps * (uint32_t)R * 4u;
    const uint32_t stage_bytes = slice_bytes * (uint32_t)groups;
    const int nstages = slen / rps;
    if (tid == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar1, 1);
        failed = 0;
    }
    const float *xg = a.x + ((size_t)g * a.B + b0) * R;
    for (int i = tid; i < NB * R; i += kSubThreads) {
        const float v = (i < nb * R) ? __ldg(xg + i) : 0.0f;
        cur[i] = make_float2(v, v);
    }
    __syncthreads();
    // copies issued into and completions seen on each buffer (every thread
    // counts; thread 0 issues)
    uint32_t issued0 = 0u, issued1 = 0u, seen0 = 0u, seen1 = 0u;
    // stage st of layer block Wl: rows st*rps .. st*rps+rps-1 of every slice
    // (one bulk copy per slice), slice j's rows at buffer rows j*rps ..
    auto issue = [&](int buf, const float *Wl, int st) {
        if (tid == 0) {
            fence_proxy_async_smem();                       // the buffer's earlier reads come first
            const uint32_t bar = buf ? bar1 : bar0;
            mbar_arrive_expect_tx(bar, stage_bytes);
            for (int j = 0; j < groups; ++j)
                bulk_g2s(smem_addr(stage + (size_t)buf * rows * R + (size_t)j * rps * R),
                         Wl + ((size_t)j * slen + (size_t)st * rps) * R, slice_bytes, bar);
        }
        if (buf) ++issued1; else ++issued0;
    };
    for (int l = 0; l + 1 < a.L && !failed; ++l) {
        const float *Wl = a.w + ((size_t)g * (a.L - 1) + l) * (size_t)R * R;
        const int act = (l + 2 == a.L) ? a.output_act : a.hidden_act;
        for (int st = 0; st < 2 && st < nstages; ++st) issue(st, Wl, st);
        f2 as[NB][2], ac[NB][2];
#pragma unroll
        for (int b = 0; b < NB; ++b) as[b][0] = as[b][1] = ac[b][0] = ac[b][1] = 0ull;
        for (int st = 0; st < nstages; ++st) {
            const int buf = st & 1;
            if (mbar_wait(buf ? bar1 : bar0, (buf ? seen1 : seen0) & 1u)) {
                if (buf) ++seen1; else ++seen0;
            } else {
                failed = 1;
            }
            // this thread's rows: sources grp*slen + st*rps .. + rps - 1
            const ulonglong2 *W4 = reinterpret_cast<const ulonglong2 *>(stage + (size_t)buf * rows * R +
                                                                        (size_t)grp * rps * R) + col;
            const f2 *xs = reinterpret_cast<const f2 *>(cur) + grp * slen + st * rps;
#pragma unroll 2
            for (int r = 0; r < rps; ++r) {
                const ulonglong2 w = W4[(size_t)r * ncols];
                const f2 nx = neg2(w.x), ny = neg2(w.y);
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const f2 x2 = xs[b * R + r];
                    dot2_step2(as[b][0], ac[b][0], x2, w.x, nx);
                    dot2_step2(as[b][1], ac[b][1], x2, w.y, ny);
                }
            }
            __syncthreads();                                // every thread is done with the buffer
            if (failed) break;
            if (st + 2 < nstages) issue(buf, Wl, st + 2);
        }
        if (failed) break;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const size_t at = ((size_t)grp * NB + b) * R + col * 4;
            *reinterpret_cast<ulonglong2 *>(ps + at) = make_ulonglong2(as[b][0], as[b][1]);
            *reinterpret_cast<ulonglong2 *>(pc + at) = make_ulonglong2(ac[b][0], ac[b][1]);
        }
        __syncthreads();
        for (int i = tid; i < NB * R; i += kSubThreads) {
            const float v = activate((uint32_t)act, combine_slices(ps + i, pc + i, (size_t)NB * R, groups));
            nxt[i] = make_float2(v, v);
        }
        __syncthreads();
        float2 *tmp = cur;
        cur = nxt;
        nxt = tmp;
    }
    float *yg = a.y + ((size_t)g * a.B + b0) * R;
    if (failed) {
        // a stage did not arrive in time: let every copy in flight land
        // before the block's shared memory is released, then report
        for (; seen0 < issued0; ++seen0) mbar_wait(bar0, seen0 & 1u);
        for (; seen1 < issued1; ++seen1) mbar_wait(bar1, seen1 & 1u);
        if (tid == 0) atomicOr(&g_substrate_error, kErrWaitExpired);
        for (int i = tid; i < nb * R; i += kSubThreads) yg[i] = __int_as_float(0x7fc00000);
        return;
    }
    for (int i = tid; i < nb * R; i += kSubThreads) yg[i] = cur[i].x;
}

template <int NB, int VEC>
int launch_sub(SubArgs a, int pop, cudaStream_t s)
{
    const size_t smem = sizeof(float) * ((size_t)2 * NB * a.R + 2 * (size_t)a.groups * NB * a.R);
    auto kern = substrate_kernel<NB, VEC>;
    int rc = allow_dynamic_smem(reinterpret_cast<const void *>(kern), smem, "neat_substrate_forward: shared memory");
    if (rc) return rc;
    a.tiles = (a.B + NB - 1) / NB;
    const long blocks = (long)pop * a.tiles;
    if (blocks > 0x7fffffffL) return invalid("neat_substrate_forward: too many blocks");
    kern<<<(unsigned)blocks, kSubThreads, smem, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_substrate_forward: launch");
    return NEAT_OK;
}

// Shared memory of the bulk-copy kernel: two stages (or the slice sums, which
// take their place), two value tiles of pairs.
size_t tma_smem_bytes(int R, int stage_rows, int nb)
{
    const size_t stages = 2 * (size_t)stage_rows * R, sums = 2 * (size_t)(kSubThreads / (R / 4)) * nb * R;
    return sizeof(float) * (std::max(stages, sums) + 4 * (size_t)nb * R);
}

template <int NB>
int launch_tma(SubArgs a, int pop, cudaStream_t s)
{
    const size_t smem = tma_smem_bytes(a.R, a.stage_rows, NB);
    auto kern = substrate_tma_kernel<NB>;
    int rc = allow_dynamic_smem(reinterpret_cast<const void *>(kern), smem, "neat_substrate_forward: shared memory");
    if (rc) return rc;
    a.tiles = (a.B + NB - 1) / NB;
    const long blocks = (long)pop * a.tiles;
    if (blocks > 0x7fffffffL) return invalid("neat_substrate_forward: too many blocks");
    kern<<<(unsigned)blocks, kSubThreads, smem, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "neat_substrate_forward: launch");
    return NEAT_OK;
}

template <int VEC>
int launch_vec(const SubArgs &a, int pop, int nb, cudaStream_t s)
{
    switch (nb) {
    case 1: return launch_sub<1, VEC>(a, pop, s);
    case 2: return launch_sub<2, VEC>(a, pop, s);
    case 4: return launch_sub<4, VEC>(a, pop, s);
    case 8: return launch_sub<8, VEC>(a, pop, s);
    default: return launch_sub<16, VEC>(a, pop, s);
    }
}

}  // namespace
}  // namespace neat

using namespace neat;

extern "C" int neat_substrate_forward(const float *weights_dev, int32_t pop, neat_substrate sub, const float *inputs_dev,
                                      int32_t batch, int32_t hidden_act, int32_t output_act, float *outputs_dev,
                                      void *stream)
{
    TraceRange trace_range("neat_substrate_forward");
    clear_error();
    if (sub.resolution < 2 || sub.resolution > 181 || sub.layers < 2)
        return invalid("neat_substrate_forward: substrate resolution must be in 2..181 and layers >= 2");
    if (pop < 0 || batch < 0) return invalid("neat_substrate_forward: sizes must be >= 0");
    if (hidden_act < 0 || hidden_act > 6 || output_act < 0 || output_act > 6)
        return invalid("neat_substrate_forward: activation ids are 0..6");
    if (pop == 0 || batch == 0) return NEAT_OK;
    if (!weights_dev || !inputs_dev || !outputs_dev) return invalid("neat_substrate_forward: null pointer");
    if ((batch + 15) / 16 > 65535) return invalid("neat_substrate_forward: batch too large");
    SubArgs a;
    a.w = weights_dev;
    a.x = inputs_dev;
    a.y = outputs_dev;
    a.R = sub.resolution * sub.resolution;
    a.L = sub.layers;
    a.B = batch;
    a.hidden_act = hidden_act;
    a.output_act = output_act;
    const bool vec4 = (a.R % 4 == 0) && (reinterpret_cast<uintptr_t>(weights_dev) % 16 == 0);
    const int ncols = vec4 ? a.R / 4 : a.R;
    a.cols = std::min(ncols, kSubThreads);
    a.groups = std::max(1, kSubThreads / a.cols);
    int nb = 1;
    while (nb < batch && nb < 16) nb <<= 1;
    // shared memory: two value tiles and the slice partials
    while (sizeof(float) * ((size_t)2 * nb * a.R + 2 * (size_t)a.groups * nb * a.R) > 200u * 1024u && a.groups > 1)
        a.groups >>= 1;
    while (sizeof(float) * ((size_t)2 * nb * a.R + 2 * (size_t)a.groups * nb * a.R) > 200u * 1024u && nb > 1)
        nb >>= 1;
    if (sizeof(float) * ((size_t)4 * nb * a.R) > 200u * 1024u)
        return invalid("neat_substrate_forward: substrate too large for one block");
    // bulk-copy path: 32 KB stages of whole source rows, tiles of up to 4
    // vectors (with the compensated sums, larger batches are bound by
    // arithmetic, not by streaming the weights once per tile), when R / 4
    // divides the block and a block takes at most 112 KB (two or more per SM;
    // 16 KB stages and a third block at 4 vectors measured the same).  Both
    // kernels split the sources into the same slices, so their
    // results are identical
    if (vec4 && kSubThreads % (a.R / 4) == 0) {
        const int groups = kSubThreads / (a.R / 4);
        const int nbt = std::min(nb, 4);
        // stage rows: a multiple of the slices, each slice's share dividing
        // the slice
        const int slen = a.R / groups;
        int rows = std::max(groups, std::min(a.R, (32 * 1024) / (4 * a.R)));
        while (rows > groups && (rows % groups || slen % (rows / groups))) --rows;
        // the same slices as substrate_kernel: groups = kSubThreads / (R / 4)
        // there too while its shared memory needs no fewer (true for nb <= 4)
        if (a.R % groups == 0 && rows % groups == 0 && slen % (rows / groups) == 0 && groups == a.groups &&
            tma_smem_bytes(a.R, rows, nbt) <= 112u * 1024u) {
            a.stage_rows = rows;
            switch (nbt) {
            case 1: return launch_tma<1>(a, pop, as_stream(stream));
            case 2: return launch_tma<2>(a, pop, as_stream(stream));
            default: return launch_tma<4>(a, pop, as_stream(stream));
            }
        }
    }
    return vec4 ? launch_vec<4>(a, pop, nb, as_stream(stream)) : launch_vec<1>(a, pop, nb, as_stream(stream));
}

namespace neat {
int read_substrate_error(unsigned int *v, int clear)
{
    cudaError_t e = cudaMemcpyFromSymbol(v, g_substrate_error, sizeof(*v));
    if (e != cudaSuccess) return cuda_fail(e, "substrate error word: read");
    if (clear) {
        const unsigned int zero = 0;
        e = cudaMemcpyToSymbol(g_substrate_error, &zero, sizeof(zero));
        if (e != cudaSuccess) return cuda_fail(e, "substrate error word: clear");
    }
    return NEAT_OK;
}
}  // namespace neat
