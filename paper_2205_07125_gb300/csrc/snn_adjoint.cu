// Surrogate-gradient adjoint of the partitioned LIF step (sm_103a).
//
// No counterpart in the paper (arXiv 2205.07125 simulates, it does not
// train).  The differentiable form keeps the step's routing and integer
// delivery and adds population-pair gains G and per-population drive rates
// lam as parameters:
//   populations  pop(j) = 2 vn(j) + (1 if j is inhibitory), n_pop = 2 n_vn;
//   inputs       A_jb(t) = int32 sum of the weights from population b
//                arriving at j at step t (delivered through the two-level
//                route's tables, kept per source population);
//   current      I_j = (((G[a][0] A_j0 + G[a][1] A_j1) + ...) + w_ext (lam_a
//                + sigma xi_j(t)), fp32, fixed order, no FMA; xi_j(t) =
//                (sum of 12 bytes of Philox4x32-10 (j, t, 0xAD, 0) - 1530) / 256;
//   membrane     as the plain step (hard threshold, reset, refractory).
// Forward: T steps from the initial state with checkpoints of (V, ref, ring)
// every K steps; population spike counts give the rates.  Backward
// (surrogate 1 / (1 + beta |V_pre - theta|)^2, reset detached): segment by
// segment from the last checkpoint, the segment's steps are recomputed with
// their V_pre, spike/refractory flags and inputs recorded, then walked
// backwards: every neuron gathers the adjoints of its targets along its own
// level-2 entries and synapse segments (the transpose of the routed
// delivery), and the parameter gradients accumulate in float64.
//
// The term of a synapse (j -> k, delay d) of step t is w G[pop k][pop j] g_k(t +
// d), g the adjoint of V_pre.  The synapses of delay d >= 3 are read every
// third step only, when the planes of three steps are complete, and gather the
// three at once (for the steps d earlier); delay 2 every second step two,
// delay 1 every step one: 0.44 of the synapses per step for delays uniform in
// 1..8, and one index per three gathered planes.  The planes are
// kept interleaved (three or two steps of a neuron in one 16- or 8-byte word),
// the slice of a source's own partition (most targets) staged in shared
// memory.  Every segment's steps run as one CUDA graph whose kernels read the
// segment's first step from device memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <vector>

#include "snn_internal.h"

using namespace snn;

namespace {

constexpr int kAThreads = 256;
constexpr int kBThreads = 1024;  // backward: one block per SM, up to 64 registers (32 warps hide latency)
constexpr int kBWarps = kBThreads / 32;
constexpr int kBGroups = 2;      // k_adj_backward_runs: groups of 4 synapses per lane per batch
constexpr int kBUnroll = 8;      // synapses of a source in flight
constexpr int64_t kBatchedNeurons = 25000;  // see adj_batched
constexpr int kParts = 2;        // parts of a partition staged one after the other; other targets are part kParts
constexpr int kKinds = kParts + 1;
constexpr int kBatch = 3;        // steps gathered at once by a synapse of delay >= kBatch
constexpr int kItemSources = 1024;  // sources per work unit, at most (their sums are in shared memory)
constexpr int kDWarps = 4;       // forward delivery: warps per spike
constexpr int kDUnroll = 4;
constexpr int kMaxPop = 8;
constexpr uint32_t kNoiseTag = 0xAD;

// A backward block's unit of work: sources j0..j1-1 of one partition, whose
// first n_stage neurons (from base) are staged, cap of them at a time; slices
// of 32 sources from sl0.
struct BItem {
    uint32_t j0, j1, base, n_stage;
    uint32_t sl0, n_sl, plane0, pad;  // (plane0: first plane of the partition's VN, k_adj_backward_runs)
};

struct AdjDev {
    long long M;
    int n_pop, D, t_ref;
    float alpha, e_l, v_th, v_reset, w_ext, sigma, beta;
    uint32_t key0, key1;
    // state
    float *V;
    uint8_t *ref;
    int32_t *ring;          // [D][M][n_pop]
    const uint8_t *pop;     // [M] internal order
    const uint32_t *gid;    // internal -> global id (nullptr: identical)
    // tables (internal order)
    const unsigned long long *run;  // [M+1] first synapse of each neuron's run: the run its
                                    // level-2 entries tile (one segment per destination partition)
    const uint32_t *syn_td; // [E] target | (delay - 1) << 28
    const int16_t *syn_w;   // [E]
    // step
    uint32_t *spk;          // [2][M] spikes of a step, by parity
    unsigned int *spk_n;    // [2]
    unsigned long long *pop_cnt;  // [n_pop] spikes per population (forward)
    unsigned long long *raster;   // [raster_cap] (t << 32 | global id)
    unsigned long long *raster_n;
    long long raster_cap;
    // parameters
    const float *G;         // [n_pop][n_pop]
    const float *lam;       // [n_pop]
    // recorded segment
    float *seg_vpre;        // [K][M]
    uint8_t *seg_flag;      // [K][M] bit 0 spike, bit 1 refractory
    int32_t *seg_A;         // [K][M][n_pop]
    // backward
    // The backward's synapses, by item, kind (part of the source's partition
    // that holds the target, or none), delay, slice of 32 sources; inside a slice column k holds the k-th synapse of every source that
    // has one, so a lane per source reads whole columns.
    const uint2 *rec;       // [E] target | pop << 28, weight (float bits)
    const uint32_t *cnt;    // [kKinds S M] synapses by (item, kind, delay, source)
    const unsigned long long *col;  // [kKinds S slices] first record of each (item, kind, delay, slice)
    // k_adj_backward_runs: planes [2][n_pop][M] by step parity, G[pop k][b] * (adjoint of V_pre of k); partial sums
    // [S][M] by step slot
    float *hbuf, *rpart;
    float *g1;              // [2][M] adjoint of V_pre by step parity
    float2 *g2;             // [2][M] the same of steps 2 m, 2 m + 1 (m mod 2)
    float4 *g3;             // [2][M] the same of steps 3 m .. 3 m + 2 (m mod 2)
    float *part;            // [R][M] gathered terms of steps to come (step mod R)
    float2 *gacc;           // [n_pop + 1][M] float pairs: a neuron's sums of g c A_b and of g c w_ext
    int S, R;               // largest delay; steps a step's gathers reach (at least 2)
    const BItem *items;     // [n_items] backward work units
    int n_items, cap, src_cap;  // neurons staged at a time, sources per item (shared memory)
    int ways;               // warps that share a slice's delays
    const int *tb;          // first step of the running segment
    float *gV;              // [M]
    const float *direct;    // [n_pop] dL/dr_a / (T N_a)
    double *dG;             // [n_pop][n_pop]
    double *dlam;           // [n_pop]
};

__device__ __forceinline__ uint4 philox_ctr(uint32_t k0, uint32_t k1, uint32_t c0, uint32_t c1, uint32_t c2,
                                            uint32_t c3)
{
    uint32_t x0 = c0, x1 = c1, x2 = c2, x3 = c3;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, x0), lo0 = 0xD2511F53u * x0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, x2), lo1 = 0xCD9E8D57u * x2;
        const uint32_t y0 = hi1 ^ x1 ^ k0, y2 = hi0 ^ x3 ^ k1;
        x0 = y0;
        x1 = lo1;
        x2 = y2;
        x3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(x0, x1, x2, x3);
}

// Programmatic dependent launch (the kernels of a segment's graph): wait for
// the kernel before this one.  The next kernel's blocks start as this one's
// exit, which saves the gap between them.  Asking for the next kernel at the
// start puts its waiting blocks in the way of this one's: forward and backward
// of 138 steps of 22,888 neurons x 450 synapses 7.06 ms without the early
// start, 7.09 with the next kernel asked for at once (7.29 on another device),
// 6.97 as here; 60,000 x 100 7.20, 7.28, 7.13; 120 steps of 4,096 x 64 3.69,
// 3.55, 3.55.
__device__ __forceinline__ void pdl_enter() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ int byte_sum(uint32_t w)
{
    return (int)(w & 0xFFu) + (int)((w >> 8) & 0xFFu) + (int)((w >> 16) & 0xFFu) + (int)(w >> 24);
}

// xi_j(t): exact multiple of 2^-8
__device__ __forceinline__ float noise_of(const AdjDev &a, uint32_t g, uint32_t t)
{
    const uint4 w = philox_ctr(a.key0, a.key1, g, t, kNoiseTag, 0u);
    const int n = byte_sum(w.x) + byte_sum(w.y) + byte_sum(w.z) - 1530;
    return __fdiv_rn((float)n, 256.0f);
}

// One step t = (segment start) + toff of the forward for every neuron
// (thread per neuron).  rec >= 0:
// record V_pre, flags and inputs in segment slot rec; count: add the spikes
// to the population counts and the raster.
template <int NP>
__global__ void __launch_bounds__(kAThreads) k_adj_update(const AdjDev a, int toff, int rec, int count)
{
    pdl_enter();
    const int t = *a.tb + toff;
    __shared__ unsigned long long s_cnt[kMaxPop];
    if (threadIdx.x < kMaxPop) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int par = t & 1;
    const int slot = t % a.D;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.spk_n[par ^ 1] = 0;  // the next step's list
    for (long long k = (long long)blockIdx.x * kAThreads + threadIdx.x; k < a.M;
         k += (long long)gridDim.x * kAThreads) {
        // every load first: the neuron's ring row (NP int32, 8-byte aligned),
        // population, state, id
        int2 *rg = reinterpret_cast<int2 *>(a.ring + ((long long)slot * a.M + k) * NP);
        int32_t A[NP];
#pragma unroll
        for (int b = 0; b < NP / 2; ++b) {
            const int2 v = rg[b];
            A[2 * b] = v.x;
            A[2 * b + 1] = v.y;
        }
        const int p = a.pop[k];
        const uint8_t r = a.ref[k];
        const float v = a.V[k];
        const uint32_t g = a.gid ? a.gid[k] : (uint32_t)k;
#pragma unroll
        for (int b = 0; b < NP / 2; ++b) rg[b] = make_int2(0, 0);
        if (rec >= 0) {
            int2 *sa = reinterpret_cast<int2 *>(a.seg_A + ((long long)rec * a.M + k) * NP);
#pragma unroll
            for (int b = 0; b < NP / 2; ++b) sa[b] = make_int2(A[2 * b], A[2 * b + 1]);
        }
        float irec = __fmul_rn(a.G[p * NP], (float)A[0]);
#pragma unroll
        for (int b = 1; b < NP; ++b) irec = __fadd_rn(irec, __fmul_rn(a.G[p * NP + b], (float)A[b]));
        const float x1 = __fmul_rn(a.sigma, noise_of(a, g, (uint32_t)t));
        const float x2 = __fadd_rn(a.lam[p], x1);
        const float drv = __fmul_rn(a.w_ext, x2);
        const float I = __fadd_rn(irec, drv);
        const bool refr = r > 0;
        const float u = __fsub_rn(v, a.e_l);
        const float au = __fmul_rn(a.alpha, u);
        float vp = __fadd_rn(a.e_l, au);
        vp = __fadd_rn(vp, __fmul_rn(I, 0.0009765625f));
        const bool S = !refr && vp >= a.v_th;
        if (rec >= 0) {
            a.seg_vpre[(long long)rec * a.M + k] = vp;
            a.seg_flag[(long long)rec * a.M + k] = (uint8_t)((S ? 1 : 0) | (refr ? 2 : 0));
        }
        a.V[k] = (refr || S) ? a.v_reset : vp;
        a.ref[k] = refr ? (uint8_t)(r - 1) : (S ? (uint8_t)a.t_ref : (uint8_t)0);
        if (S) {
            const unsigned int pos = atomicAdd(&a.spk_n[par], 1u);
            a.spk[(long long)par * a.M + pos] = (uint32_t)k;
            if (count) {
                atomicAdd(&s_cnt[p], 1ull);
                const unsigned long long rp = atomicAdd(a.raster_n, 1ull);
                if ((long long)rp < a.raster_cap) a.raster[rp] = ((unsigned long long)t << 32) | g;
            }
        }
    }
    __syncthreads();
    if (count && threadIdx.x < NP && s_cnt[threadIdx.x]) atomicAdd(&a.pop_cnt[threadIdx.x], s_cnt[threadIdx.x]);
}

// Delivery of step t's spikes through the routing tables: a spike's level-2
// entries tile its synapse run, which kDWarps warps share (a contiguous
// quarter each, kDUnroll loads per lane in flight); every weight is added
// to the ring slot of its delay, column = the source population.
__global__ void __launch_bounds__(kAThreads) k_adj_deliver(const AdjDev a, int toff)
{
    pdl_enter();
    const int t = *a.tb + toff;
    const int par = t & 1;
    const unsigned int n = *(volatile unsigned int *)&a.spk_n[par];
    const int lane = threadIdx.x & 31;
    const unsigned int nw = (gridDim.x * kAThreads) >> 5;
    for (unsigned int wq = (blockIdx.x * kAThreads + threadIdx.x) >> 5; wq < n * kDWarps; wq += nw) {
        const uint32_t i = a.spk[(long long)par * a.M + wq / kDWarps];
        const int q = (int)(wq % kDWarps);
        const int pi = a.pop[i];
        const unsigned long long r0 = a.run[i], len = a.run[i + 1] - r0;
        const unsigned long long b0 = r0 + len * q / kDWarps, b1 = r0 + len * (q + 1) / kDWarps;
        for (unsigned long long x0 = b0 + lane; x0 < b1; x0 += 32 * kDUnroll) {
            uint32_t td[kDUnroll];
            int32_t w[kDUnroll];
#pragma unroll
            for (int u = 0; u < kDUnroll; ++u) {
                const unsigned long long x = x0 + 32ull * u;
                td[u] = x < b1 ? __ldg(a.syn_td + x) : 0u;
                w[u] = x < b1 ? (int32_t)__ldg(a.syn_w + x) : 0;
            }
#pragma unroll
            for (int u = 0; u < kDUnroll; ++u) {
                if (x0 + 32ull * u >= b1) break;
                int sl = t + (int)(td[u] >> kTgtBits) + 1;
                sl %= a.D;
                atomicAdd(&a.ring[((long long)sl * a.M + (td[u] & kTgtMask)) * a.n_pop + pi], w[u]);
            }
        }
    }
}

// A float sum kept as an unevaluated pair hi + lo (Dekker / Knuth two-sum):
// adds the exact product gd * x (two-product with one fused multiply-add) and
// keeps the rounding errors in lo, so hi + lo carries about 48 significant
// bits.  The float64 pipe of this GPU is slow, so the per-neuron terms stay in
// the float pipe; k_adj_reduce adds the pairs in float64.
__device__ __forceinline__ float2 pair_add(float2 a, float gd, float x)
{
    const float p = __fmul_rn(gd, x);
    const float q = __fmaf_rn(gd, x, -p);  // p + q == gd * x exactly
    const float s = __fadd_rn(a.x, p);
    const float bp = __fsub_rn(s, a.x);
    const float err = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bp)), __fsub_rn(p, bp));
    return make_float2(s, __fadd_rn(a.y, __fadd_rn(err, q)));
}

// Places of an item's entries in cnt and col.
__device__ __forceinline__ size_t cnt_at(const AdjDev &a, const BItem &it, int kind, int d)
{
    return (size_t)kKinds * a.S * it.j0 + ((size_t)kind * a.S + (d - 1)) * (it.j1 - it.j0);
}

__device__ __forceinline__ size_t col_at(const AdjDev &a, const BItem &it, int kind, int d, uint32_t sl)
{
    return (size_t)kKinds * a.S * it.sl0 + ((size_t)kind * a.S + (d - 1)) * it.n_sl + sl;
}

// Build the backward's synapse order (targets and weights).  A block per
// item.  The k-th synapse of a source is the k-th of its kind in the table's
// order, so the sums' rounding does not change from run to run.
__global__ void __launch_bounds__(kAThreads) k_adj_sort(const AdjDev a, uint2 *rec, uint32_t *cnt,
                                                        unsigned long long *col)
{
    constexpr int kW = kAThreads / 32;
    __shared__ uint32_t s_n[kW][kKinds * kMaxDelay];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nk = kKinds * a.S;
    uint32_t *n = s_n[wid];
    for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        const BItem it = a.items[item];
        const uint32_t ns = it.j1 - it.j0;
        auto key = [&](uint32_t td) {
            const uint32_t rel = (td & kTgtMask) - it.base;
            return (rel < it.n_stage ? (int)(rel / (uint32_t)a.cap) : kParts) * a.S + (int)(td >> kTgtBits);
        };
        for (uint32_t si = wid; si < ns; si += kW) {
            const unsigned long long r0 = a.run[it.j0 + si], r1 = a.run[it.j0 + si + 1];
            for (int k = lane; k < nk; k += 32) n[k] = 0u;
            __syncwarp();
            for (unsigned long long x = r0 + lane; x < r1; x += 32) atomicAdd(&n[key(a.syn_td[x])], 1u);
            __syncwarp();
            for (int k = lane; k < nk; k += 32) cnt[cnt_at(a, it, 0, 1 + k) + si] = n[k];
            __syncwarp();
        }
        __syncthreads();
        const uint32_t ne = (uint32_t)nk * it.n_sl;  // entries of col, (kind, delay, slice) in order
        unsigned long long *co = col + col_at(a, it, 0, 1, 0);
        for (uint32_t e = wid; e < ne; e += kW) {
            const uint32_t sl = e % it.n_sl, si = sl * 32 + lane;
            const uint32_t c = si < ns ? cnt[cnt_at(a, it, 0, 1 + (int)(e / it.n_sl)) + si] : 0u;
            unsigned long long v = c;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
            if (lane == 0) co[e] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long at = a.run[it.j0];
            for (uint32_t e = 0; e < ne; ++e) {
                const unsigned long long c = co[e];
                co[e] = at;
                at += c;
            }
        }
        __syncthreads();
        for (uint32_t si = wid; si < ns; si += kW) {
            const unsigned long long r0 = a.run[it.j0 + si], r1 = a.run[it.j0 + si + 1];
            const uint32_t sl = si >> 5, in = si & 31u, left = min(32u, ns - sl * 32);
            for (int k = lane; k < nk; k += 32) n[k] = 0u;
            __syncwarp();
            for (unsigned long long x0 = r0; x0 < r1; x0 += 32) {
                const unsigned long long x = x0 + lane;
                const uint32_t td = x < r1 ? a.syn_td[x] : 0u;
                const int k = x < r1 ? key(td) : -1;
                const uint32_t same = __match_any_sync(0xFFFFFFFFu, k);
                const uint32_t rank = __popc(same & ((1u << lane) - 1u));
                uint32_t c = 0;
                if (k >= 0) c = n[k] + rank;
                __syncwarp();
                if (k >= 0) {
                    if (rank == 0) n[k] += __popc(same);
                    // column c of the slice: the columns before it, the sources before this one in it
                    const uint32_t *len = cnt + cnt_at(a, it, 0, 1 + k) + sl * 32;
                    unsigned long long pos = co[(size_t)k * it.n_sl + sl];
                    for (uint32_t u = 0; u < left; ++u) {
                        const uint32_t m = len[u];
                        pos += min(m, c) + (u < in && m > c ? 1u : 0u);
                    }
                    const uint32_t t = td & kTgtMask;
                    rec[pos] = make_uint2(t | (uint32_t)a.pop[t] << kTgtBits, __float_as_uint((float)a.syn_w[x]));
                }
                __syncwarp();
            }
        }
        __syncthreads();
    }
}

// One backward step t = (segment start) + toff, segment slot rec.  A block
// takes the sources of an item.  For the planes that are complete at step t
// (the last one always: delay 1; two at odd t: delay 2; three when t + 1 is a
// multiple of 3: delays from 3) a warp takes a slice of 32 sources, a lane per
// source, and walks the columns of those delays: first the targets in the
// parts of its own partition, each part's slice of the planes staged in shared
// memory for the block, then the other targets from global memory.  The sums
// go to the steps t, t - 1, .. of the source (acc, carried in part).  Step t's
// sum is then complete and a thread per source runs the adjoint recursion,
// writes the plane entries of step t and adds the parameter-gradient terms to
// the neuron's own pairs.
//
// The gathers from global memory are bound by the lines that L1 can hold in
// flight: staging half a partition at a time (98 KB) instead of all of it (196
// KB) leaves four times as many.  Measured at the adjoint workload (131,072
// neurons, 500 synapses, delays 1-8): 99 us per step against 191 for
// k_adj_backward_runs; 132 with the whole partition staged.
//
// A term is w (G g): the gain times the adjoint rounded by itself, as
// k_adj_backward_runs does.  Rounding w G ahead instead gives every synapse of
// one weight and population pair the same error in every step, which adds up.
template <int B>
__device__ __forceinline__ void adj_gather(const AdjDev &a, const BItem &it, int d0, int d1, const float *h1,
                                           const float2 *h2, const float4 *h3, const float *s_G, float *hs, float *acc)
{
    const uint32_t ns = it.j1 - it.j0;
    const int lane = threadIdx.x & 31, np = a.n_pop;
    const uint32_t cap = (uint32_t)a.cap, stride = cap + 1u, ways = (uint32_t)a.ways;
#pragma unroll 1
    for (int kind = 0; kind < kKinds; ++kind) {
        const uint32_t from = (uint32_t)kind * cap;  // first staged neuron of the part
        if (kind < kParts && from >= it.n_stage) continue;
        if (kind < kParts) {
            const uint32_t n = min(cap, it.n_stage - from);
            __syncthreads();
#pragma unroll 4
            for (uint32_t x = threadIdx.x; x < n; x += kBThreads) {
                const uint32_t j = it.base + from + x;
                if constexpr (B == 1) {
                    hs[x] = h1[j];
                } else if constexpr (B == 2) {
                    const float2 v = h2[j];
                    hs[x] = v.x;
                    hs[stride + x] = v.y;
                } else {
                    const float4 v = h3[j];
                    hs[x] = v.x;
                    hs[stride + x] = v.y;
                    hs[2 * stride + x] = v.z;
                }
            }
            // (a plane's last entry stays 0: what a lane without a synapse multiplies)
            if (threadIdx.x < B) hs[threadIdx.x * stride + cap] = 0.0f;
            __syncthreads();
        }
        // a warp per slice; with few slices several, which share the delays (each with sums of its own)
        for (uint32_t wu = threadIdx.x >> 5; wu < it.n_sl * ways; wu += kBThreads / 32) {
            const uint32_t sl = wu / ways, way = wu - sl * ways;
            const uint32_t si = sl * 32 + lane;
            if (d0 + (int)way > d1) continue;
            // gains of the source's population; its partition's targets are of two populations
            const int pj = si < ns ? a.pop[it.j0 + si] : (int)it.plane0;
            const float *gain = s_G + pj;
            const float g0 = gain[it.plane0 * np], g1 = gain[(it.plane0 + 1u) * np];
            // synapses of a delay and their first records, those of the next delay in flight
            uint32_t n0 = 0;
            unsigned long long c0;
            auto bounds = [&](int d) {
                if (si < ns) n0 = a.cnt[cnt_at(a, it, kind, d) + si];
                c0 = a.col[col_at(a, it, kind, d, sl)];
            };
            bounds(d0 + (int)way);
#pragma unroll 1
            for (int d = d0 + (int)way; d <= d1; d += (int)ways) {
                const uint32_t n = n0;
                const uint2 *r = a.rec + c0;
                if (d + (int)ways <= d1) {
                    bounds(d + (int)ways);
                    // the slice's records of the next delay into L2
                    const uint32_t tot = __reduce_add_sync(0xFFFFFFFFu, n0);
                    for (uint32_t x = 16u * lane; x < tot; x += 512u)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.rec + c0 + x));
                }
                float sum[B];
#pragma unroll
                for (int b = 0; b < B; ++b) sum[b] = 0.0f;
                const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, n);
#pragma unroll 1
                for (uint32_t k = 0; k < most; k += kBUnroll) {
                    // records of columns [k, k + kBUnroll) (none past a source's last)
                    uint2 q[kBUnroll];
#pragma unroll
                    for (int u = 0; u < kBUnroll; ++u) {
                        const bool in = n > k + u;
                        const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
                        q[u] = in ? __ldcs(r + __popc(m & ((1u << lane) - 1u)))
                                  : make_uint2(it.base + from + cap, 0u);
                        r += __popc(m);
                    }
                    float part[B];  // (the terms of a batch by themselves: short chains round less)
#pragma unroll
                    for (int b = 0; b < B; ++b) part[b] = 0.0f;
                    if (kind < kParts) {
#pragma unroll
                        for (int u = 0; u < kBUnroll; ++u) {
                            const float *h = hs + ((q[u].x & kTgtMask) - it.base - from);
                            const float gn = q[u].x & (1u << kTgtBits) ? g1 : g0;
#pragma unroll
                            for (int b = 0; b < B; ++b)
                                part[b] = __fmaf_rn(__uint_as_float(q[u].y), __fmul_rn(gn, h[b * stride]), part[b]);
                        }
                    } else {
                        float v[kBUnroll][B];
#pragma unroll
                        for (int u = 0; u < kBUnroll; ++u) {
                            const uint32_t x = q[u].x & kTgtMask;
#pragma unroll
                            for (int b = 0; b < B; ++b) v[u][b] = 0.0f;
                            if (n <= k + u) continue;
                            if constexpr (B == 1) {
                                v[u][0] = __ldg(h1 + x);
                            } else if constexpr (B == 2) {
                                const float2 w = __ldg(h2 + x);
                                v[u][0] = w.x;
                                v[u][1] = w.y;
                            } else {
                                const float4 w = __ldg(h3 + x);
                                v[u][0] = w.x;
                                v[u][1] = w.y;
                                v[u][2] = w.z;
                            }
                        }
#pragma unroll
                        for (int u = 0; u < kBUnroll; ++u) {
                            const float gn = gain[(q[u].x >> kTgtBits) * np];
#pragma unroll
                            for (int b = 0; b < B; ++b)
                                part[b] = __fmaf_rn(__uint_as_float(q[u].y), __fmul_rn(gn, v[u][b]), part[b]);
                        }
                    }
#pragma unroll
                    for (int b = 0; b < B; ++b) sum[b] = __fadd_rn(sum[b], part[b]);
                }
                // the last of the planes is gathered by step t - (d - d0), the one before it by the step before
                if (si < ns)
#pragma unroll
                    for (int b = 0; b < B; ++b)
                        acc[((int)way * a.R + d - d0 + B - 1 - b) * a.src_cap + si] += sum[b];
            }
        }
    }
}

__global__ void __launch_bounds__(kBThreads, 1) k_adj_backward(const AdjDev a, int toff, int rec)
{
    extern __shared__ __align__(16) float bsm[];
    pdl_enter();
    const int t = *a.tb + toff;
    const long long M = a.M;
    const int np = a.n_pop, R = a.R;
    float *hs = bsm;                       // [kBatch][cap + 1] staged planes
    float *acc = bsm + kBatch * (a.cap + 1);    // [ways][R][src_cap] sums of steps t, t - 1, ..
    const float c = 0.0009765625f;
    __shared__ float s_G[kMaxPop * kMaxPop];
    if (threadIdx.x < np * np) s_G[threadIdx.x] = a.G[threadIdx.x];  // (the item loop begins with a barrier)
    const bool triple = a.S >= kBatch && (t + 1) % kBatch == 0;  // planes t + 1 .. t + 3 are complete
    const int nacc = triple ? R : 2;       // steps that get terms
    for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        const BItem it = a.items[item];
        const uint32_t ns = it.j1 - it.j0;
        __syncthreads();
        for (int i = 0; i < nacc; ++i)
            for (uint32_t x = threadIdx.x; x < ns; x += kBThreads)
                acc[i * a.src_cap + x] = t >= i ? a.part[(size_t)((t - i) % R) * M + it.j0 + x] : 0.0f;
        for (int x = R * a.src_cap + threadIdx.x; x < a.ways * R * a.src_cap; x += kBThreads) acc[x] = 0.0f;
        adj_gather<1>(a, it, 1, 1, a.g1 + (size_t)((t + 1) & 1) * M, nullptr, nullptr, s_G, hs, acc);
        if (a.S >= 2 && (t & 1))
            adj_gather<2>(a, it, 2, 2, nullptr, a.g2 + (size_t)(((t + 1) / 2) & 1) * M, nullptr, s_G, hs, acc);
        if (triple)
            adj_gather<3>(a, it, 3, a.S, nullptr, nullptr, a.g3 + (size_t)(((t + 1) / kBatch) & 1) * M, s_G, hs, acc);
        __syncthreads();
        if (a.ways > 1) {
            for (int x = threadIdx.x; x < nacc * a.src_cap; x += kBThreads)
                for (int w = 1; w < a.ways; ++w) acc[x] += acc[w * R * a.src_cap + x];
            __syncthreads();
        }
        for (int i = 1; i < nacc; ++i)
            for (uint32_t x = threadIdx.x; x < ns; x += kBThreads)
                if (t >= i) a.part[(size_t)((t - i) % R) * M + it.j0 + x] = acc[i * a.src_cap + x];
        for (uint32_t x = threadIdx.x; x < ns; x += kBThreads) {
            const uint32_t j = it.j0 + x;
            const int pj = a.pop[j];
            const uint8_t fl = a.seg_flag[(long long)rec * M + j];
            const float vpre = a.seg_vpre[(long long)rec * M + j];
            float g = 0.0f;
            if (!(fl & 2)) {
                const float gS = __fadd_rn(a.direct[pj], __fmul_rn(c, acc[x]));
                const float dv = __fsub_rn(vpre, a.v_th);
                const float den = __fadd_rn(1.0f, __fmul_rn(a.beta, fabsf(dv)));
                const float sg = __frcp_rn(__fmul_rn(den, den));
                const float keep = (fl & 1) ? 0.0f : a.gV[j];
                g = __fadd_rn(keep, __fmul_rn(gS, sg));
            }
            a.gV[j] = __fmul_rn(a.alpha, g);
            a.g1[(size_t)(t & 1) * M + j] = g;
            reinterpret_cast<float *>(a.g2 + (size_t)((t / 2) & 1) * M + j)[t & 1] = g;
            reinterpret_cast<float *>(a.g3 + (size_t)((t / kBatch) & 1) * M + j)[t % kBatch] = g;
            // step t's slot is step t - R's from now on
            a.part[(size_t)(t % R) * M + j] = 0.0f;
            // parameter-gradient terms g c A_b and g c w_ext: exact products on the neuron's float pairs
            if (g != 0.0f) {
                const float gd = __fmul_rn(g, c);
                const int32_t *A = a.seg_A + ((long long)rec * M + j) * np;
                for (int b = 0; b < np; ++b) {
                    const int32_t xi = A[b];
                    if (xi < (1 << 24) && xi > -(1 << 24))
                        a.gacc[(size_t)b * M + j] = pair_add(a.gacc[(size_t)b * M + j], gd, (float)xi);
                    else
                        atomicAdd(&a.dG[pj * np + b], (double)g * (double)c * (double)xi);
                }
                a.gacc[(size_t)np * M + j] = pair_add(a.gacc[(size_t)np * M + j], gd, a.w_ext);
            }
        }
    }
}

// A float sum kept as an unevaluated pair hi + lo (Dekker / Knuth two-sum):
// add() takes the exact product gd * x (two-product with one fused
// multiply-add) and keeps the rounding errors in lo, so hi + lo carries about
// 48 significant bits; flush() adds hi + lo in float64 and clears the pair.
// The float64 pipe of this GPU is slow, so the per-neuron terms stay in the
// float pipe.
struct FloatPairSum {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float gd, float x)
    {
        const float p = __fmul_rn(gd, x);
        const float q = __fmaf_rn(gd, x, -p);  // p + q == gd * x exactly
        const float s = __fadd_rn(hi, p);
        const float bp = __fsub_rn(s, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(p, bp));
        hi = s;
        lo = __fadd_rn(lo, __fadd_rn(err, q));
    }
    __device__ __forceinline__ void flush(double *dst)
    {
        const double v = (double)hi + (double)lo;
        if (v != 0.0) atomicAdd(dst, v);
        hi = lo = 0.0f;
    }
};

// One backward step t = (segment start) + toff, segment slot rec, for every
// neuron, a warp each (networks too small for k_adj_backward, see adj_batched).  The warp of source j walks j's synapse run (the
// transpose of the routed delivery) and takes, for every synapse (k, d),
// w * h_k(t + 1) from plane pop(j) of step t + 1: a term of j's input adjoint
// at step t + 1 - d.  The terms collect per lane and delay in shared memory,
// are summed over the warp and added to the partial sums of those steps;
// the sum of step t is then complete (d = 1 is the last term it gets) and
// gives j's adjoint recursion, its plane entries for step t and its
// parameter-gradient terms.  A block works on sources of one partition with
// that partition's slice of the two planes its sources read staged in
// shared memory; a warp's next source has its run bounds and first batch of
// synapses in flight while the current source finishes.
template <int NDL>
__global__ void __launch_bounds__(kBThreads, 1) k_adj_backward_runs(const AdjDev a, int toff, int rec)
{
    extern __shared__ __align__(16) float bsm[];
    pdl_enter();
    __shared__ double s_dG[kMaxPop * kMaxPop];
    __shared__ double s_dl[kMaxPop];
    const int t = *a.tb + toff;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long M = a.M;
    const int np = a.n_pop;
    float *hs = bsm;                                          // [2][cap]
    float *col = bsm + 2 * a.cap + warp * (NDL * 32) + lane;  // this lane's column, stride 32 per delay
    for (int x = threadIdx.x; x < kMaxPop * kMaxPop; x += kBThreads) s_dG[x] = 0.0;
    if (threadIdx.x < kMaxPop) s_dl[threadIdx.x] = 0.0;
#pragma unroll
    for (int dd = 0; dd < NDL; ++dd) col[dd * 32] = 0.0f;
    const float c = 0.0009765625f;
    const float *hn = a.hbuf + (size_t)((t + 1) & 1) * np * M;  // step t + 1
    float *ho = a.hbuf + (size_t)(t & 1) * np * M;              // step t
    // the lanes that hold the warp's sum of delay index dd = lane >> sh
    constexpr int sh = NDL == 8 ? 2 : 1;
    const int dd = lane >> sh;
    const bool holder = (lane & ((1 << sh) - 1)) == 0 && dd < a.S && t - dd >= 0;
    const int slot = (t - dd + a.S) % a.S;  // meaningful where holder
    FloatPairSum acc0, acc1;
    for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        const BItem it = a.items[item];
        __syncthreads();
        {
            const float *s0 = hn + (size_t)it.plane0 * M + it.base;
            const float *s1 = s0 + M;
            for (uint32_t x0 = threadIdx.x; x0 < it.n_stage; x0 += 4 * kBThreads) {
                float v0[4], v1[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t x = x0 + u * kBThreads;
                    v0[u] = x < it.n_stage ? s0[x] : 0.0f;
                    v1[u] = x < it.n_stage ? s1[x] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t x = x0 + u * kBThreads;
                    if (x < it.n_stage) {
                        hs[x] = v0[u];
                        hs[a.cap + x] = v1[u];
                    }
                }
            }
        }
        __syncthreads();
        uint32_t j = it.j0 + warp;
        // the first source's run and batch.  A batch is kBGroups groups of 4
        // synapses per lane from the run's start rounded down to a multiple
        // of 4 (one 16-byte load of target words and one 8-byte load of
        // weights per group); weights outside the run count as 0.
        unsigned long long r0 = 0, r1 = 0;
        int pj = 0;
        if (j < it.j1) {
            r0 = a.run[j];
            r1 = a.run[j + 1];
            pj = a.pop[j];
        }
        uint4 tv[kBGroups];
        uint2 wv[kBGroups];
        auto load_batch = [&](unsigned long long g0, unsigned long long end) {
#pragma unroll
            for (int u = 0; u < kBGroups; ++u) {
                const unsigned long long e = g0 + 4ull * (lane + 32 * u);
                const bool in = e < end;
                tv[u] = in ? __ldg(reinterpret_cast<const uint4 *>(a.syn_td + e)) : make_uint4(0, 0, 0, 0);
                wv[u] = in ? __ldg(reinterpret_cast<const uint2 *>(a.syn_w + e)) : make_uint2(0, 0);
            }
        };
        load_batch(r0 & ~3ull, r1);
        for (; j < it.j1; j += kBWarps) {
            // the next source's run; this source's epilogue inputs
            const uint32_t jn = j + kBWarps;
            unsigned long long n0 = 0, n1 = 0;
            int pn = 0;
            if (jn < it.j1) {
                n0 = a.run[jn];
                n1 = a.run[jn + 1];
                pn = a.pop[jn];
            }
            const float pin = holder ? a.rpart[(size_t)slot * M + j] : 0.0f;
            const int32_t Ab = lane < np ? a.seg_A[((long long)rec * M + j) * np + lane] : 0;
            const float Gb = lane < np ? a.G[pj * np + lane] : 0.0f;
            uint8_t fl = 0;
            float vpre = 0.0f, gVj = 0.0f, dir = 0.0f;
            if (lane == 0) {
                fl = a.seg_flag[(long long)rec * M + j];
                vpre = a.seg_vpre[(long long)rec * M + j];
                gVj = a.gV[j];
                dir = a.direct[pj];
            }
            const float *hsp = hs + (pj & 1) * a.cap;
            const float *hgp = hn + (size_t)pj * M;
            for (unsigned long long g0 = r0 & ~3ull;;) {
#pragma unroll
                for (int u = 0; u < kBGroups; ++u) {
                    const unsigned long long e = g0 + 4ull * (lane + 32 * u);
                    const uint32_t tdu[4] = {tv[u].x, tv[u].y, tv[u].z, tv[u].w};
                    const int32_t wu[4] = {(int32_t)(int16_t)(wv[u].x & 0xFFFFu), (int32_t)(int16_t)(wv[u].x >> 16),
                                           (int32_t)(int16_t)(wv[u].y & 0xFFFFu), (int32_t)(int16_t)(wv[u].y >> 16)};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const bool in = e + i >= r0 && e + i < r1;
                        const uint32_t k = tdu[i] & kTgtMask;
                        const uint32_t rel = k - it.base;
                        const float hk = rel < it.n_stage ? hsp[rel] : __ldg(hgp + k);
                        float *cp = col + (tdu[i] >> kTgtBits) * 32;
                        *cp = __fadd_rn(*cp, __fmul_rn((float)(in ? wu[i] : 0), hk));
                    }
                }
                g0 += 4ull * 32 * kBGroups;
                if (g0 >= r1) break;
                load_batch(g0, r1);
            }
            // the next source's first batch, in flight during the epilogue
            load_batch(n0 & ~3ull, n1);
            // the warp's sum per delay: halve the delays held per lane over
            // lane bits 4, 3, ..., then sum the rest of the warp
            float r[NDL];
#pragma unroll
            for (int x = 0; x < NDL; ++x) {
                r[x] = col[x * 32];
                col[x * 32] = 0.0f;
            }
#pragma unroll
            for (int half = NDL / 2, sft = 16; half >= 1; half >>= 1, sft >>= 1) {
                const bool up = (lane & sft) != 0;
#pragma unroll
                for (int q = 0; q < half; ++q) {
                    const float keep = up ? r[half + q] : r[q];
                    const float give = up ? r[q] : r[half + q];
                    r[q] = __fadd_rn(keep, __shfl_xor_sync(0xFFFFFFFFu, give, sft));
                }
            }
#pragma unroll
            for (int sft = (1 << sh) >> 1; sft > 0; sft >>= 1)
                r[0] = __fadd_rn(r[0], __shfl_xor_sync(0xFFFFFFFFu, r[0], sft));
            const float sum = __fadd_rn(pin, r[0]);
            // step t's slot is consumed (and cleared for step t - S); the
            // earlier steps' slots take their terms
            if (holder) a.rpart[(size_t)slot * M + j] = dd == 0 ? 0.0f : sum;
            float gvp = 0.0f;
            if (lane == 0 && !(fl & 2)) {
                const float gS = __fadd_rn(dir, __fmul_rn(c, sum));
                const float x = __fsub_rn(vpre, a.v_th);
                const float den = __fadd_rn(1.0f, __fmul_rn(a.beta, fabsf(x)));
                const float sg = __frcp_rn(__fmul_rn(den, den));
                const float keep = (fl & 1) ? 0.0f : gVj;
                gvp = __fadd_rn(keep, __fmul_rn(gS, sg));
            }
            gvp = __shfl_sync(0xFFFFFFFFu, gvp, 0);
            // the products each source population gathers at step t - 1
            if (lane < np) ho[(size_t)lane * M + j] = __fmul_rn(Gb, gvp);
            if (lane == 0) a.gV[j] = __fmul_rn(a.alpha, gvp);
            // parameter-gradient terms gvp * c * A_jb (lane b) and gvp * c * w_ext
            // (lane 31): exact products, summed per warp as float pairs
            if (gvp != 0.0f && (lane < np || lane == 31)) {
                const int32_t xi = lane < np ? Ab : 0;
                if (lane == 31 || (xi < (1 << 24) && xi > -(1 << 24))) {
                    const float gd = __fmul_rn(gvp, c);
                    const float x = lane == 31 ? a.w_ext : (float)xi;
                    if (pj & 1) acc1.add(gd, x);
                    else acc0.add(gd, x);
                } else {
                    atomicAdd(&s_dG[pj * np + lane], (double)gvp * (double)c * (double)xi);
                }
            }
            r0 = n0;
            r1 = n1;
            pj = pn;
        }
        // the warp's sums of this item (populations plane0, plane0 + 1)
        if (lane < np) {
            acc0.flush(&s_dG[it.plane0 * np + lane]);
            acc1.flush(&s_dG[(it.plane0 + 1) * np + lane]);
        } else if (lane == 31) {
            acc0.flush(&s_dl[it.plane0]);
            acc1.flush(&s_dl[it.plane0 + 1]);
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < np * np; x += kBThreads)
        if (s_dG[x] != 0.0) atomicAdd(&a.dG[x], s_dG[x]);
    if (threadIdx.x < np && s_dl[threadIdx.x] != 0.0) atomicAdd(&a.dlam[threadIdx.x], s_dl[threadIdx.x]);
}

// The parameter gradients: every neuron's pairs in float64 by population
// (blockIdx.y: the column, n_pop for the drive rates).
__global__ void __launch_bounds__(kAThreads) k_adj_reduce(const AdjDev a)
{
    __shared__ double s[kMaxPop];
    if (threadIdx.x < kMaxPop) s[threadIdx.x] = 0.0;
    __syncthreads();
    const int col = blockIdx.y, np = a.n_pop;
    const float2 *g = a.gacc + (size_t)col * a.M;
    double v = 0.0;
    int p = -1;
    for (long long j = (long long)blockIdx.x * kAThreads + threadIdx.x; j < a.M; j += (long long)gridDim.x * kAThreads) {
        const int pj = a.pop[j];
        if (pj != p) {
            if (p >= 0) atomicAdd(&s[p], v);
            p = pj;
            v = 0.0;
        }
        v += (double)g[j].x + (double)g[j].y;
    }
    if (p >= 0) atomicAdd(&s[p], v);
    __syncthreads();
    if (threadIdx.x < np) atomicAdd(col < np ? &a.dG[threadIdx.x * np + col] : &a.dlam[threadIdx.x], s[threadIdx.x]);
}

__global__ void k_adj_set_step(int *tb, int t)
{
    *tb = t;
}

struct Region {
    size_t off = 0, bytes = 0;
};

struct ALayout {
    Region V, ref, ring, pop, gid, run, syn_td, syn_w, spk, spk_n, pop_cnt, raster, raster_n;
    Region G, lam, seg_vpre, seg_flag, seg_A, rec, cnt, col, hbuf, rpart, g1, g2, g3, part, gacc, items, tb, gV, direct, dG, dlam;
    Region ck_V, ck_ref, ck_ring;  // [n_ckpt] checkpoints
    size_t total = 0;
    int D = 2, n_pop = 2, n_ckpt = 1, S = 1, R = 2, n_items = 1;
    int64_t n_slices = 0;
    bool batched = false;  // k_adj_backward, else k_adj_backward_runs
};

void aplace(ALayout &L, Region &r, size_t bytes)
{
    r.off = L.total;
    r.bytes = bytes;
    L.total += (bytes + 255) & ~(size_t)255;
}

bool adj_params_ok(const snn_adjoint_params *ap)
{
    return ap && ap->T >= 1 && ap->ckpt_every >= 1 && std::isfinite(ap->sigma) && std::isfinite(ap->beta) &&
           ap->beta > 0.0f;
}

int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                   cudaSuccess)
        sms = 0;
    cudaGetLastError();
    return std::max(1, sms);
}

// The backward's work units: every partition cut into chunks of at most
// kItemSources sources, about one chunk per SM in all (at least one per
// partition).  Returns the count and the slices of 32 sources; fills `out` when given (n_stage is capped at create).
int backward_items(const snn_routing *rt, std::vector<BItem> *out, int64_t *slices)
{
    const int sms = sm_count();
    const int64_t M = rt->M;
    int n = 0;
    *slices = 0;
    for (int32_t ip = 0; ip < rt->P; ++ip) {
        const int64_t a = rt->pbase[ip], b = rt->pbase[ip + 1];
        if (b <= a) continue;
        const int64_t c = std::max<int64_t>((b - a + kItemSources - 1) / kItemSources,
                                            (int64_t)sms * (b - a) / std::max<int64_t>(1, M));
        for (int64_t x = 0; x < c; ++x) {
            BItem it;
            std::memset(&it, 0, sizeof(it));
            it.j0 = (uint32_t)(a + (b - a) * x / c);
            it.j1 = (uint32_t)(a + (b - a) * (x + 1) / c);
            it.base = (uint32_t)a;
            it.n_stage = (uint32_t)(b - a);
            it.plane0 = (uint32_t)(2 * (ip / (rt->P / rt->n_vn)));
            it.sl0 = (uint32_t)*slices;
            it.n_sl = (it.j1 - it.j0 + 31) / 32;
            *slices += it.n_sl;
            if (out) out->push_back(it);
            ++n;
        }
    }
    return std::max(1, n);
}

// Whether the backward batches steps (k_adj_backward) or walks every run each
// step (k_adj_backward_runs).  A batched step has several phases in a row, each
// some loads deep, that pay from about 25,000 neurons.  A lane walks its
// source's synapses of a delay by itself, so its chain grows with the
// synapses, and with few delays there is little to share out between warps
// and nothing to batch: then more neurons are needed, growing about as the
// root of the synapses per neuron.  Measured, backward of 60 steps in ms, runs
// / batched: 26,000 neurons x 50 synapses, delays 1-8 1.92 / 1.47; 40,000 x
// 150, delay 1 2.48 / 2.46; 26,000 x 400, 1-8 2.47 / 2.66, 40,000 x 400 3.64 /
// 2.94; 50,000 x 400, 1-3 4.19 / 4.47, 1-4 4.23 / 3.87; 65,536 x 400, 1 5.00 /
// 5.19; 65,536 x 800, 1-3 7.76 / 7.81; 131,072 x 400, 1 9.94 / 6.82, 1-8 11.4 /
// 5.91.  SNN_ADJ_BATCHED=0|1 overrides (tests).
bool adj_batched(const snn_routing *rt)
{
    const char *e = std::getenv("SNN_ADJ_BATCHED");
    if (e && (e[0] == '0' || e[0] == '1')) return e[0] == '1';
    const double root = std::sqrt((double)rt->E / (double)std::max<int64_t>(1, rt->M));
    const double per_root = rt->max_delay <= 3 ? 3300 : rt->max_delay <= 5 ? 2400 : 1600;
    return (double)rt->M >= std::max((double)kBatchedNeurons, per_root * root);
}

int adj_layout(const snn_routing *rt, const snn_sim_params *p, const snn_adjoint_params *ap, ALayout &L)
{
    const int64_t M = rt->M, E = rt->E;
    L = ALayout();
    L.D = rt->max_delay + 1;
    L.S = std::max(1, (int)rt->max_delay);
    L.R = std::max(2, L.S);
    L.n_items = backward_items(rt, nullptr, &L.n_slices);
    L.n_pop = 2 * rt->n_vn;
    if (L.n_pop > kMaxPop) return SNN_E_RANGE;
    L.n_ckpt = (ap->T + ap->ckpt_every - 1) / ap->ckpt_every;
    const int K = std::min(ap->T, ap->ckpt_every);
    const size_t ring_b = sizeof(int32_t) * (size_t)L.D * M * L.n_pop;
    aplace(L, L.V, sizeof(float) * M);
    aplace(L, L.ref, M);
    aplace(L, L.ring, ring_b);
    aplace(L, L.pop, M);
    aplace(L, L.gid, rt->identity ? 0 : sizeof(uint32_t) * M);
    aplace(L, L.run, sizeof(unsigned long long) * (M + 1));
    // (k_adj_backward_runs reads synapses in aligned groups of 4: up to 3 past the end, zero-filled)
    aplace(L, L.syn_td, sizeof(uint32_t) * (E + 4));
    aplace(L, L.syn_w, sizeof(int16_t) * (E + 4));
    aplace(L, L.spk, sizeof(uint32_t) * 2 * M);
    aplace(L, L.spk_n, 2 * sizeof(unsigned int));
    aplace(L, L.pop_cnt, sizeof(unsigned long long) * kMaxPop);
    aplace(L, L.raster, sizeof(unsigned long long) * (size_t)std::max<int64_t>(0, p->raster_cap));
    aplace(L, L.raster_n, sizeof(unsigned long long));
    aplace(L, L.G, sizeof(float) * kMaxPop * kMaxPop);
    aplace(L, L.lam, sizeof(float) * kMaxPop);
    aplace(L, L.seg_vpre, sizeof(float) * (size_t)K * M);
    aplace(L, L.seg_flag, (size_t)K * M);
    aplace(L, L.seg_A, sizeof(int32_t) * (size_t)K * M * L.n_pop);
    L.batched = adj_batched(rt);
    if (L.batched) {
        aplace(L, L.rec, sizeof(uint2) * (size_t)E);
        aplace(L, L.cnt, sizeof(uint32_t) * (size_t)M * kKinds * L.S);
        aplace(L, L.col, sizeof(unsigned long long) * kKinds * L.S * (size_t)L.n_slices);
        aplace(L, L.g1, sizeof(float) * 2 * M);
        aplace(L, L.g2, sizeof(float2) * 2 * M);
        aplace(L, L.g3, sizeof(float4) * 2 * M);
        aplace(L, L.part, sizeof(float) * (size_t)L.R * M);
        aplace(L, L.gacc, sizeof(float2) * (size_t)(L.n_pop + 1) * M);
    } else {
        aplace(L, L.hbuf, sizeof(float) * 2 * (size_t)L.n_pop * M);
        aplace(L, L.rpart, sizeof(float) * (size_t)L.S * M);
    }
    aplace(L, L.items, sizeof(BItem) * (size_t)L.n_items);
    aplace(L, L.tb, sizeof(int));
    aplace(L, L.gV, sizeof(float) * M);
    aplace(L, L.direct, sizeof(float) * kMaxPop);
    aplace(L, L.dG, sizeof(double) * kMaxPop * kMaxPop);
    aplace(L, L.dlam, sizeof(double) * kMaxPop);
    aplace(L, L.ck_V, sizeof(float) * M * (size_t)L.n_ckpt);
    aplace(L, L.ck_ref, (size_t)M * L.n_ckpt);
    aplace(L, L.ck_ring, ring_b * L.n_ckpt);
    return SNN_OK;
}

}  // namespace

struct snn_adjoint {
    const snn_routing *rt = nullptr;
    snn_sim_params prm;
    snn_adjoint_params ap;
    ALayout L;
    AdjDev dev;
    char *ws = nullptr;
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;  // graph capture
    unsigned grid_n = 1, grid_w = 1, grid_b = 1;
    size_t bsmem = 0;                   // dynamic shared memory of the backward
    int ndl = 8;                        // delay columns of k_adj_backward_runs (8 or 16)
    std::vector<double> pop_size;
    bool have_forward = false;
    // one graph per (kind, segment length): 0 forward counted, 1 forward
    // recorded, 2 backward
    std::map<std::pair<int, int>, cudaGraphExec_t> graphs;

    ~snn_adjoint()
    {
        for (auto &g : graphs) cudaGraphExecDestroy(g.second);
        if (cap_stream) cudaStreamDestroy(cap_stream);
    }
};

#define ACK(x)                                    \
    do {                                          \
        cudaError_t e_ = (x);                     \
        if (e_ != cudaSuccess) return SNN_E_CUDA; \
    } while (0)

extern "C" void snn_adjoint_params_default(snn_adjoint_params *ap)
{
    if (!ap) return;
    std::memset(ap, 0, sizeof(*ap));
    ap->T = 500;
    ap->ckpt_every = 50;
    ap->sigma = 0.9f;
    ap->beta = 5.0f;
}

extern "C" int snn_adjoint_workspace_bytes(const snn_routing *rt, const snn_sim_params *p,
                                           const snn_adjoint_params *ap, size_t *bytes)
{
    if (!rt || !p || !bytes || !adj_params_ok(ap)) return SNN_E_ARG;
    ALayout L;
    int rc = adj_layout(rt, p, ap, L);
    if (rc) return rc;
    *bytes = L.total;
    return SNN_OK;
}

extern "C" int snn_adjoint_create(const snn_network *net, const uint8_t *is_exc, const snn_routing *rt,
                                  const snn_sim_params *p, const snn_adjoint_params *ap, void *workspace,
                                  size_t ws_bytes, void *stream, snn_adjoint **out)
{
    if (!out) return SNN_E_ARG;
    *out = nullptr;
    if (!net || !is_exc || !rt || !p || !adj_params_ok(ap) || !workspace || ((uintptr_t)workspace & 255))
        return SNN_E_ARG;
    if (net->n_neurons != rt->M || p->raster_cap < 0) return SNN_E_ARG;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) return SNN_E_NODEV;
    snn_adjoint *a = new (std::nothrow) snn_adjoint();
    if (!a) return SNN_E_NOMEM;
    a->rt = rt;
    a->prm = *p;
    a->ap = *ap;
    int rc = adj_layout(rt, p, ap, a->L);
    if (rc) {
        delete a;
        return rc;
    }
    if (ws_bytes < a->L.total) {
        delete a;
        return SNN_E_NOMEM;
    }
    a->ws = (char *)workspace;
    a->stream = (cudaStream_t)stream;
    const ALayout &L = a->L;
    const int64_t M = rt->M;
    char *w = a->ws;
    AdjDev &d = a->dev;
    std::memset(&d, 0, sizeof(d));
    d.M = M;
    d.n_pop = L.n_pop;
    d.D = L.D;
    d.t_ref = p->t_ref;
    d.alpha = (float)std::exp(-p->dt_ms / p->tau_ms);
    d.e_l = p->e_l;
    d.v_th = p->v_th;
    d.v_reset = p->v_reset;
    d.w_ext = (float)p->w_ext;
    d.sigma = ap->sigma;
    d.beta = ap->beta;
    d.key0 = (uint32_t)p->drive_seed;
    d.key1 = (uint32_t)(p->drive_seed >> 32);
    d.V = (float *)(w + L.V.off);
    d.ref = (uint8_t *)(w + L.ref.off);
    d.ring = (int32_t *)(w + L.ring.off);
    d.pop = (const uint8_t *)(w + L.pop.off);
    d.gid = rt->identity ? nullptr : (const uint32_t *)(w + L.gid.off);
    d.run = (const unsigned long long *)(w + L.run.off);
    d.syn_td = (const uint32_t *)(w + L.syn_td.off);
    d.syn_w = (const int16_t *)(w + L.syn_w.off);
    d.spk = (uint32_t *)(w + L.spk.off);
    d.spk_n = (unsigned int *)(w + L.spk_n.off);
    d.pop_cnt = (unsigned long long *)(w + L.pop_cnt.off);
    d.raster = (unsigned long long *)(w + L.raster.off);
    d.raster_n = (unsigned long long *)(w + L.raster_n.off);
    d.raster_cap = p->raster_cap;
    d.G = (const float *)(w + L.G.off);
    d.lam = (const float *)(w + L.lam.off);
    d.seg_vpre = (float *)(w + L.seg_vpre.off);
    d.seg_flag = (uint8_t *)(w + L.seg_flag.off);
    d.seg_A = (int32_t *)(w + L.seg_A.off);
    d.rec = (const uint2 *)(w + L.rec.off);
    d.cnt = (const uint32_t *)(w + L.cnt.off);
    d.col = (const unsigned long long *)(w + L.col.off);
    d.g1 = (float *)(w + L.g1.off);
    d.g2 = (float2 *)(w + L.g2.off);
    d.g3 = (float4 *)(w + L.g3.off);
    d.gacc = (float2 *)(w + L.gacc.off);
    d.hbuf = (float *)(w + L.hbuf.off);
    d.rpart = (float *)(w + L.rpart.off);
    d.part = (float *)(w + L.part.off);
    d.S = L.S;
    d.R = L.R;
    d.items = (const BItem *)(w + L.items.off);
    d.tb = (const int *)(w + L.tb.off);
    d.gV = (float *)(w + L.gV.off);
    d.direct = (const float *)(w + L.direct.off);
    d.dG = (double *)(w + L.dG.off);
    d.dlam = (double *)(w + L.dlam.off);
    // populations (internal order) and their sizes
    std::vector<uint8_t> pop((size_t)M);
    const int32_t s = rt->P / rt->n_vn;
    a->pop_size.assign((size_t)L.n_pop, 0.0);
    for (int32_t ip = 0; ip < rt->P; ++ip)
        for (int64_t k = rt->pbase[ip]; k < rt->pbase[ip + 1]; ++k) {
            const uint32_t g = rt->perm_inv[k];
            pop[k] = (uint8_t)(2 * (ip / s) + (is_exc[g] ? 0 : 1));
            a->pop_size[pop[k]] += 1.0;
        }
    // each neuron's level-2 entries tile its synapse run (one segment per
    // destination partition, partitions ascending): check, keep the bounds
    for (int64_t i = 0; i < M; ++i) {
        uint64_t at = (uint64_t)rt->csr[i];
        for (uint32_t f = rt->l1_l2[rt->l1_ptr[i]]; f < rt->l1_l2[rt->l1_ptr[i + 1]]; ++f) {
            if ((rt->l2[f].off & kOffMask) != at) {
                delete a;
                return SNN_E_STATE;
            }
            at += rt->l2[f].len;
        }
        if (at != (uint64_t)rt->csr[i + 1]) {
            delete a;
            return SNN_E_STATE;
        }
    }
    // on the object's stream, as the kernel below that reads them (the legacy stream's copies and clears are not
    // ordered before a non-blocking stream's kernels); the host arrays outlive the synchronisation at the end
    auto copy = [&](size_t off, const void *src, size_t bytes) -> cudaError_t {
        return bytes ? cudaMemcpyAsync(w + off, src, bytes, cudaMemcpyHostToDevice, a->stream) : cudaSuccess;
    };
    auto up = [&](const Region &r, const void *src) { return copy(r.off, src, r.bytes); };
    if (up(L.pop, pop.data()) || up(L.run, rt->csr.data()) ||
        cudaMemsetAsync(w + L.syn_td.off, 0, L.syn_td.bytes, a->stream) ||
        cudaMemsetAsync(w + L.syn_w.off, 0, L.syn_w.bytes, a->stream) ||
        copy(L.syn_td.off, rt->syn_td.data(), sizeof(uint32_t) * rt->E) ||
        copy(L.syn_w.off, rt->syn_w.data(), sizeof(int16_t) * rt->E) ||
        (!rt->identity && up(L.gid, rt->perm_inv.data()))) {
        delete a;
        return SNN_E_CUDA;
    }
    const int sms = sm_count();
    a->grid_n = (unsigned)std::max<int64_t>(1, std::min<int64_t>((M + kAThreads - 1) / kAThreads, 65535));
    a->grid_w = (unsigned)std::max(1, sms * 8);
    // backward: the sums of an item's sources, then as much of a partition's
    // slice of three planes as shared memory holds
    {
        std::vector<BItem> items;
        int64_t slices = 0;
        backward_items(rt, &items, &slices);
        int dev = 0, optin = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
            delete a;
            return SNN_E_CUDA;
        }
        int64_t widest = 0, most = 0;
        for (const BItem &it : items) {
            widest = std::max<int64_t>(widest, it.n_stage);
            most = std::max<int64_t>(most, it.j1 - it.j0);
        }
        d.n_items = (int)items.size();
        const void *fn;
        if (L.batched) {
            d.ways = (int)std::max<int64_t>(1, std::min<int64_t>(8, kBThreads / std::max<int64_t>(32, (most + 31) / 32 * 32)));
            const size_t sums = sizeof(float) * (size_t)d.ways * L.R * (size_t)most, fixed = 1024;
            // (parts of at most 8192 neurons, 96 KB of staged planes: the rest of the SM's memory is L1's, for the
            // gathers from global memory)
            int64_t cap = std::min<int64_t>(8192, (int64_t)(((size_t)optin - sums - fixed) / (kBatch * sizeof(float))) - 1);
            cap = std::min<int64_t>(cap, widest);
            for (BItem &it : items) it.n_stage = (uint32_t)std::min<int64_t>(it.n_stage, kParts * cap);
            d.cap = (int)cap;
            d.src_cap = (int)most;
            a->bsmem = sums + sizeof(float) * kBatch * (size_t)(cap + 1);
            fn = (const void *)k_adj_backward;
        } else {
            // the delay columns, then as much of a partition's two planes as fits
            a->ndl = rt->max_delay <= 8 ? 8 : 16;
            const size_t cols = sizeof(float) * (size_t)kBWarps * a->ndl * 32;
            const size_t fixed = sizeof(double) * (kMaxPop * kMaxPop + kMaxPop) + 1024;
            int64_t cap = 0;
            if ((size_t)optin > cols + fixed) cap = (int64_t)(((size_t)optin - cols - fixed) / (2 * sizeof(float))) & ~3ll;
            cap = std::min<int64_t>(cap, (widest + 3) & ~3ll);
            for (BItem &it : items) it.n_stage = (uint32_t)std::min<int64_t>(it.n_stage, cap);
            d.cap = (int)cap;
            a->bsmem = cols + 2 * sizeof(float) * (size_t)cap;
            fn = a->ndl == 8 ? (const void *)k_adj_backward_runs<8> : (const void *)k_adj_backward_runs<16>;
        }
        if ((int)items.size() != L.n_items ||
            !snn::allow_dynamic_smem(fn, a->bsmem) ||
            copy(L.items.off, items.data(), sizeof(BItem) * items.size()) != cudaSuccess ||
            cudaStreamCreateWithFlags(&a->cap_stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete a;
            return SNN_E_CUDA;
        }
        if (L.batched)
            k_adj_sort<<<(unsigned)std::max(1, d.n_items), kAThreads, 0, a->stream>>>(
                d, (uint2 *)(w + L.rec.off), (uint32_t *)(w + L.cnt.off), (unsigned long long *)(w + L.col.off));
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(a->stream) != cudaSuccess) {
            delete a;
            return SNN_E_CUDA;
        }
        a->grid_b = (unsigned)std::min(d.n_items, sms);
    }
    *out = a;
    return SNN_OK;
}

// Initial state (V = v0, ref = 0, empty ring), empty spike lists and counts.
static int adj_reset(snn_adjoint *a)
{
    const ALayout &L = a->L;
    char *w = a->ws;
    cudaStream_t st = a->stream;
    ACK(cudaMemcpyAsync(w + L.V.off, a->rt->v0.data(), L.V.bytes, cudaMemcpyHostToDevice, st));
    ACK(cudaMemsetAsync(w + L.ref.off, 0, L.ref.bytes, st));
    ACK(cudaMemsetAsync(w + L.ring.off, 0, L.ring.bytes, st));
    ACK(cudaMemsetAsync(w + L.spk_n.off, 0, L.spk_n.bytes, st));
    ACK(cudaMemsetAsync(w + L.pop_cnt.off, 0, L.pop_cnt.bytes, st));
    ACK(cudaMemsetAsync(w + L.raster_n.off, 0, L.raster_n.bytes, st));
    return SNN_OK;
}

// The steps of one segment of `len` steps from the step base in device
// memory: kind 0 the counted forward, 1 the recorded forward, 2 the
// backward (last step first).  Captured once per (kind, len) and replayed.
static int adj_segment(snn_adjoint *a, int kind, int len)
{
    cudaGraphExec_t &ex = a->graphs[std::make_pair(kind, len)];
    if (!ex) {
        cudaStream_t cs = a->cap_stream;
        ACK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.stream = cs;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t le = cudaSuccess;
        for (int i = 0; i < len && le == cudaSuccess; ++i) {
            cfg.dynamicSmemBytes = 0;
            cfg.blockDim = dim3(kAThreads);
            if (kind == 2) {
                const int toff = len - 1 - i;
                cfg.gridDim = dim3(a->grid_b);
                cfg.blockDim = dim3(kBThreads);
                cfg.dynamicSmemBytes = a->bsmem;
                if (a->L.batched) le = cudaLaunchKernelEx(&cfg, k_adj_backward, a->dev, toff, toff);
                else if (a->ndl == 8) le = cudaLaunchKernelEx(&cfg, k_adj_backward_runs<8>, a->dev, toff, toff);
                else le = cudaLaunchKernelEx(&cfg, k_adj_backward_runs<16>, a->dev, toff, toff);
            } else {
                const int rec = kind == 1 ? i : -1, cnt = kind == 0 ? 1 : 0;
                cfg.gridDim = dim3(a->grid_n);
                switch (a->dev.n_pop) {
                case 2: le = cudaLaunchKernelEx(&cfg, k_adj_update<2>, a->dev, i, rec, cnt); break;
                case 4: le = cudaLaunchKernelEx(&cfg, k_adj_update<4>, a->dev, i, rec, cnt); break;
                case 6: le = cudaLaunchKernelEx(&cfg, k_adj_update<6>, a->dev, i, rec, cnt); break;
                default: le = cudaLaunchKernelEx(&cfg, k_adj_update<8>, a->dev, i, rec, cnt); break;
                }
                cfg.gridDim = dim3(a->grid_w);
                if (le == cudaSuccess) le = cudaLaunchKernelEx(&cfg, k_adj_deliver, a->dev, i);
            }
        }
        cudaGraph_t g = nullptr;
        const cudaError_t e = cudaStreamEndCapture(cs, &g);
        if (le != cudaSuccess || e != cudaSuccess || !g) {
            if (g) cudaGraphDestroy(g);
            a->graphs.erase(std::make_pair(kind, len));
            return SNN_E_CUDA;
        }
        const cudaError_t e2 = cudaGraphInstantiate(&ex, g, 0);
        cudaGraphDestroy(g);
        if (e2 != cudaSuccess) {
            a->graphs.erase(std::make_pair(kind, len));
            return SNN_E_CUDA;
        }
    }
    ACK(cudaGraphLaunch(ex, a->stream));
    return SNN_OK;
}

static int adj_set_step(snn_adjoint *a, int t)
{
    k_adj_set_step<<<1, 1, 0, a->stream>>>((int *)a->dev.tb, t);
    ACK(cudaGetLastError());
    return SNN_OK;
}

extern "C" int snn_adjoint_forward(snn_adjoint *a, const float *G, const float *lam, float *rates,
                                   int64_t *spikes)
{
    if (!a || !G || !lam) return SNN_E_ARG;
    const ALayout &L = a->L;
    char *w = a->ws;
    cudaStream_t st = a->stream;
    const int np = L.n_pop;
    ACK(cudaMemcpyAsync(w + L.G.off, G, sizeof(float) * np * np, cudaMemcpyHostToDevice, st));
    ACK(cudaMemcpyAsync(w + L.lam.off, lam, sizeof(float) * np, cudaMemcpyHostToDevice, st));
    int rc = adj_reset(a);
    if (rc) return rc;
    const int T = a->ap.T, K = a->ap.ckpt_every;
    const int64_t M = a->rt->M;
    const size_t ring_b = L.ring.bytes;
    for (int t0 = 0; t0 < T; t0 += K) {
        const int c = t0 / K;
        ACK(cudaMemcpyAsync(w + L.ck_V.off + (size_t)c * sizeof(float) * M, w + L.V.off, L.V.bytes,
                            cudaMemcpyDeviceToDevice, st));
        ACK(cudaMemcpyAsync(w + L.ck_ref.off + (size_t)c * M, w + L.ref.off, L.ref.bytes, cudaMemcpyDeviceToDevice,
                            st));
        ACK(cudaMemcpyAsync(w + L.ck_ring.off + (size_t)c * ring_b, w + L.ring.off, ring_b, cudaMemcpyDeviceToDevice,
                            st));
        if ((rc = adj_set_step(a, t0)) != SNN_OK || (rc = adj_segment(a, 0, std::min(K, T - t0))) != SNN_OK)
            return rc;
    }
    unsigned long long cnt[kMaxPop];
    ACK(cudaMemcpyAsync(cnt, w + L.pop_cnt.off, sizeof(cnt), cudaMemcpyDeviceToHost, st));
    ACK(cudaStreamSynchronize(st));
    int64_t tot = 0;
    for (int b = 0; b < np; ++b) {
        if (rates) rates[b] = (float)((double)cnt[b] / ((double)T * a->pop_size[b]));
        tot += (int64_t)cnt[b];
    }
    if (spikes) *spikes = tot;
    a->have_forward = true;
    return SNN_OK;
}

extern "C" int snn_adjoint_backward(snn_adjoint *a, const double *grates, double *dG, double *dlam)
{
    if (!a || !grates || !dG || !dlam) return SNN_E_ARG;
    if (!a->have_forward) return SNN_E_STATE;
    const ALayout &L = a->L;
    char *w = a->ws;
    cudaStream_t st = a->stream;
    const int np = L.n_pop, T = a->ap.T, K = a->ap.ckpt_every;
    const int64_t M = a->rt->M;
    float direct[kMaxPop] = {0};
    for (int b = 0; b < np; ++b) direct[b] = (float)(grates[b] / ((double)T * a->pop_size[b]));
    ACK(cudaMemcpyAsync(w + L.direct.off, direct, sizeof(direct), cudaMemcpyHostToDevice, st));
    if (L.batched) {
        // (g1 .. gacc are one range: planes from step T on and all sums are 0)
        ACK(cudaMemsetAsync(w + L.g1.off, 0, L.gacc.off + L.gacc.bytes - L.g1.off, st));
    } else {
        ACK(cudaMemsetAsync(w + L.hbuf.off, 0, L.hbuf.bytes, st));
        ACK(cudaMemsetAsync(w + L.rpart.off, 0, L.rpart.bytes, st));
    }
    ACK(cudaMemsetAsync(w + L.gV.off, 0, L.gV.bytes, st));
    ACK(cudaMemsetAsync(w + L.dG.off, 0, L.dG.bytes, st));
    ACK(cudaMemsetAsync(w + L.dlam.off, 0, L.dlam.bytes, st));
    const size_t ring_b = L.ring.bytes;
    for (int c = L.n_ckpt - 1; c >= 0; --c) {
        const int t0 = c * K, t1 = std::min(T, t0 + K);
        // the segment's forward again, from its checkpoint, recorded
        ACK(cudaMemcpyAsync(w + L.V.off, w + L.ck_V.off + (size_t)c * sizeof(float) * M, L.V.bytes,
                            cudaMemcpyDeviceToDevice, st));
        ACK(cudaMemcpyAsync(w + L.ref.off, w + L.ck_ref.off + (size_t)c * M, L.ref.bytes, cudaMemcpyDeviceToDevice,
                            st));
        ACK(cudaMemcpyAsync(w + L.ring.off, w + L.ck_ring.off + (size_t)c * ring_b, ring_b, cudaMemcpyDeviceToDevice,
                            st));
        ACK(cudaMemsetAsync(w + L.spk_n.off, 0, L.spk_n.bytes, st));
        int rc = adj_set_step(a, t0);
        if (rc == SNN_OK) rc = adj_segment(a, 1, t1 - t0);
        if (rc == SNN_OK) rc = adj_segment(a, 2, t1 - t0);
        if (rc != SNN_OK) return rc;
    }
    if (L.batched)
        k_adj_reduce<<<dim3((unsigned)std::max(1, std::min(64, (int)((M + kAThreads - 1) / kAThreads))), np + 1), kAThreads, 0,
                   st>>>(a->dev);
    ACK(cudaGetLastError());
    ACK(cudaMemcpyAsync(dG, w + L.dG.off, sizeof(double) * np * np, cudaMemcpyDeviceToHost, st));
    ACK(cudaMemcpyAsync(dlam, w + L.dlam.off, sizeof(double) * np, cudaMemcpyDeviceToHost, st));
    ACK(cudaStreamSynchronize(st));
    return SNN_OK;
}

extern "C" int snn_adjoint_read_spikes(snn_adjoint *a, uint64_t *out, int64_t cap, int64_t *n)
{
    if (!a || !n) return SNN_E_ARG;
    unsigned long long cnt = 0;
    ACK(cudaStreamSynchronize(a->stream));
    ACK(cudaMemcpy(&cnt, a->ws + a->L.raster_n.off, sizeof(cnt), cudaMemcpyDeviceToHost));
    *n = (int64_t)cnt;
    const int64_t m = std::min<int64_t>((int64_t)cnt, std::min<int64_t>(cap, a->prm.raster_cap));
    if (m > 0 && out) ACK(cudaMemcpy(out, a->ws + a->L.raster.off, sizeof(uint64_t) * m, cudaMemcpyDeviceToHost));
    if ((int64_t)cnt > a->prm.raster_cap) return SNN_E_CAPACITY;
    return SNN_OK;
}

extern "C" void snn_adjoint_destroy(snn_adjoint *a)
{
    delete a;
}
