// Device partitioner (sm_103a): Algorithm 1 (Sec. IV.A) with batched
// growth, the parallel form of the greedy that the paper leaves as future
// work (Sec. VII, parallelization of algorithms).
//
// A cooperative launch runs two iterations t side by side, each on one half of
// the blocks with its own state and barrier; iteration t grows parts 0..P-2
// one after the other, the last part takes the rest; the host keeps the
// iteration with the smallest objective.  A part grows in rounds:
//   scatter  the members that joined in the last round add their weight W_a
//            to acc[j] of every neuron j they share a synapse with (either
//            direction, with multiplicity): gain(j) = W_j * acc[j] is
//            sum_{i in part} (c_ij + c_ji) W_i W_j;
//   select   a histogram of the unassigned neurons' gains on a logarithmic
//            scale gives a bound that the `need` largest unique 64-bit keys
//            (gain << idbits | (2^idbits - 1 - j): ties to the lowest id) all
//            reach and at most kMaxBatch keys do (further histograms split
//            the bound's bin while more do); those keys are listed;
//   join     every block sorts the listed keys by itself, and the first
//            `need` join in that order until the part's weight reaches
//            sum(W)/P: each block keeps the labels of its own neurons and
//            the part's size and weight, so nothing is sent after the join.
// need = min(B, unassigned, max(1, n_k / g)) (g = 0 drops the last term),
// n_k = the part's size so far.  Every step is integer arithmetic, so the
// result does not depend on the order of the atomic additions: it equals the
// sequential reading with the same rounds bit for bit, and with B = 1 the
// one-neuron-at-a-time greedy.  Grid barriers are bounded (a block that
// waits past the limit records a timeout and the launch ends).
//
// The rounds are short (65,536 neurons of 200 synapses into 16 parts: 1,260
// rounds over 4 iterations), so what bounds them is the chain of barriers and
// of steps between them, not the memory.  Hence three barriers per round
// (after the scatter, the histogram and the listing), one block per SM, and
// two iterations at once.  Building that network up to its first 100 steps
// (lists, this partition, routing tables, sim) takes 25 ms; 68 with seven
// barriers per round (four histogram passes over the keys, the join on one
// block), two blocks per SM and one iteration at a time.
#include <cuda_runtime.h>

#include "snn_internal.h"

namespace {

constexpr int kPT = 1024;                // threads per block
constexpr int kPW = kPT / 32;
constexpr int kDigit = 11;               // digit bits of the histograms
constexpr int kBins = 1 << kDigit;
constexpr int kHists = 3;                // global histograms in turn: filled, read, cleared
constexpr int kGroups = 2;               // iterations side by side
constexpr int kMaxBatch = 2048;          // largest round
constexpr int kChunk = 256;              // synapses per scatter task
constexpr int kPUnroll = kChunk / 32;    // loads in flight per lane

constexpr uint32_t kPStTimeout = 1u, kPStRange = 2u, kPStFault = 4u;

struct PCtl {
    alignas(128) unsigned long long bar;  // barrier arrivals of the running launch
    alignas(128) unsigned int nsel;       // keys listed by the selection
    alignas(128) unsigned int status;
    unsigned int seed_id[3];              // seed of part k at k % 3: lowest unassigned id (t == 1, atomicMin) or
                                          // the drawn one (t > 1); all ones until then
    unsigned long long obj;               // objective of the iteration
    // setup results (group 0)
    unsigned long long gain_max;          // largest possible gain
    unsigned long long deg_max;           // largest out- or in-degree
};

// State of one iteration.
struct PGroup {
    unsigned long long *acc;    // [M] weight shared with the growing part
    int32_t *lab;               // [M] part of each neuron (-1: unassigned)
    uint32_t *hist;             // [kHists][kBins]
    unsigned long long *sel;    // [kMaxBatch] keys listed by the selection
    uint32_t *cnt;              // [blocks] unassigned neurons per block
    unsigned long long *wpart;  // [P] part weights
    PCtl *c;
};

struct PDev {
    const long long *ptr;       // [M+1] out-synapses of each neuron
    const uint32_t *tgt;        // [E]
    long long *in_ptr;          // [M+1] in-synapses of each neuron
    uint32_t *in_src;           // [E]
    uint32_t *W;                // [M] out-degree
    uint32_t *fill;             // [M] in-degree counters of the in-list build
    PGroup g[kGroups];
    long long M, E, Wtot;
    int P, B, grow, idbits, mbits, chunks;
    int t0, groups, blocks;     // the launch runs iterations t0 .. t0 + groups - 1 on `blocks` blocks each
    uint64_t seed;
    unsigned long long limit_ns;
};

__device__ __forceinline__ unsigned long long p_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded barrier number k of an iteration's blocks (cooperative launch: every
// block is resident).  A block-wide barrier, a release add and acquire loads at GPU
// scope make the writes of every block before it visible after it.  Returns
// false (after recording kPStTimeout) when the wait runs out or another
// block's did.
__device__ __forceinline__ bool p_sync(PCtl *c, unsigned long long k, int blocks, unsigned long long limit_ns)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned long long target = (k + 1ull) * (unsigned long long)blocks;
        asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(&c->bar) : "memory");
        const unsigned long long deadline = p_ns() + limit_ns;
        unsigned int spins = 0;
        for (;;) {
            unsigned long long v;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&c->bar) : "memory");
            if (v >= target) break;
            if ((++spins & 63u) == 0u) {
                if (*(volatile unsigned int *)&c->status & kPStTimeout) {
                    ok = 0;
                    break;
                }
                if (p_ns() > deadline) {
                    atomicOr(&c->status, kPStTimeout);
                    ok = 0;
                    break;
                }
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <class T>
__device__ __forceinline__ T p_block_sum(T v, T *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    T s = 0;
#pragma unroll
    for (int w = 0; w < kPW; ++w) s += sh[w];
    return s;
}

// Exclusive block scan of one value per thread (thread order).
template <class T>
__device__ __forceinline__ T p_block_excl(T v, T *sh, T &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    T base = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kPW; ++w) {
        if (w < wid) base += sh[w];
        tot += sh[w];
    }
    total = tot;
    return base + x - v;
}

// ------------------------------------------------------------------ setup
// Out-degrees, in-degree counts and the target range check.
__global__ void k_part_degrees(PDev d)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < d.M; i += stride)
        d.W[i] = (uint32_t)(d.ptr[i + 1] - d.ptr[i]);
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < d.E; e += stride) {
        const uint32_t j = d.tgt[e];
        if (j < (unsigned long long)d.M) atomicAdd(&d.fill[j], 1u);
        else atomicOr(&d.g[0].c->status, kPStRange);
    }
}

// in_ptr = exclusive scan of the in-degrees (one block); fill goes back to
// zero for the per-target cursors of k_part_in_lists.
__global__ void __launch_bounds__(1024) k_part_scan(PDev d)
{
    __shared__ long long sh[32];
    const long long n = d.M;
    const long long per = (n + blockDim.x - 1) / blockDim.x;
    const long long a = min(n, (long long)threadIdx.x * per), b = min(n, a + per);
    long long s = 0;
    for (long long i = a; i < b; ++i) s += d.fill[i];
    // block-wide exclusive scan of the thread sums
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long x = s;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    long long base = 0;
    for (int w = 0; w < wid; ++w) base += sh[w];
    long long run = base + x - s;
    for (long long i = a; i < b; ++i) {
        d.in_ptr[i] = run;
        run += d.fill[i];
        d.fill[i] = 0;
    }
    if (threadIdx.x == blockDim.x - 1) d.in_ptr[n] = run;
}

// in_src: the sources of every neuron's in-synapses (list order is the
// atomics' order, which no later step depends on).  One warp per source.
__global__ void k_part_in_lists(PDev d)
{
    const int lane = threadIdx.x & 31;
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = w0; i < d.M; i += nw)
        for (long long e = d.ptr[i] + lane; e < d.ptr[i + 1]; e += 32) {
            const uint32_t j = d.tgt[e];
            if (j >= (unsigned long long)d.M) continue;
            const uint32_t pos = atomicAdd(&d.fill[j], 1u);
            d.in_src[d.in_ptr[j] + pos] = (uint32_t)i;
        }
}

// Largest possible gain W_j * sum of W over j's synapses in both directions
// and the largest degree (for the selection key width and the scatter's
// chunking).  A gain that would not fit 64 bits records kPStRange.
__global__ void k_part_bounds(PDev d)
{
    const int lane = threadIdx.x & 31;
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long j = w0; j < d.M; j += nw) {
        unsigned long long s = 0;
        for (long long e = d.ptr[j] + lane; e < d.ptr[j + 1]; e += 32) {
            const uint32_t x = d.tgt[e];
            if (x < (unsigned long long)d.M) s += d.W[x];
        }
        for (long long e = d.in_ptr[j] + lane; e < d.in_ptr[j + 1]; e += 32) s += d.W[d.in_src[e]];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        if (lane == 0) {
            const unsigned long long wj = d.W[j];
            if (__umul64hi(wj, s) != 0ull) atomicOr(&d.g[0].c->status, kPStRange);
            atomicMax(&d.g[0].c->gain_max, wj * s);
            const unsigned long long dg = max(d.ptr[j + 1] - d.ptr[j], d.in_ptr[j + 1] - d.in_ptr[j]);
            atomicMax(&d.g[0].c->deg_max, dg);
        }
    }
}

// ------------------------------------------------------------------ growth
// Word 0 of Philox4x32-10 at counter (c0, c1, c2, 0).
__device__ __noinline__ uint32_t p_philox_word0(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2)
{
    uint32_t x[4] = {c0, c1, c2, 0u};
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        const uint32_t h0 = __umulhi(0xD2511F53u, x[0]), l0 = 0xD2511F53u * x[0];
        const uint32_t h1 = __umulhi(0xCD9E8D57u, x[2]), l1 = 0xCD9E8D57u * x[2];
        x[0] = h1 ^ x[1] ^ k0;
        x[1] = l1;
        x[2] = h0 ^ x[3] ^ k1;
        x[3] = l0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return x[0];
}

struct PShared {
    uint32_t hist[kBins];
    unsigned long long key[kMaxBatch];  // listed keys, then sorted
    uint32_t added[kMaxBatch];          // members that joined in the last round
    uint32_t cut;                       // bin of the need-th largest key, keys in the bins above it, in it
    uint32_t above, in;
    uint32_t n, base, seed;
    unsigned long long redu[kPW];
    uint32_t red32[kPW];
};

// Bin of a gain: exact below 2^mb, then 2^mb bins per power of two (an
// increasing function); p_bin_range inverts it to a range of keys.
__device__ __forceinline__ uint32_t p_bin(unsigned long long gain, int mb)
{
    if (gain < (1ull << mb)) return (uint32_t)gain;
    const int e = 63 - __clzll((long long)gain);
    return ((uint32_t)(e - mb) << mb) + (uint32_t)(gain >> (e - mb));
}
__device__ __forceinline__ void p_bin_range(uint32_t bin, int mb, int idbits, unsigned long long &base, int &width)
{
    // (bins e << mb | m of e >= 1 stand for gains (2^mb + m) << (e - 1))
    const int e = (int)(bin >> mb);
    const unsigned long long m = bin & ((1u << mb) - 1u);
    const int sh = max(0, e - 1);
    base = ((e ? m + (1ull << mb) : m) << sh) << idbits;
    width = sh + idbits;
}

// Adds the block's histogram to the global one h, clears `next` (this block's
// share), passes the barrier and finds the bin of the need-th largest key.
__device__ __forceinline__ bool p_cut(const PDev &d, const PGroup &g, PShared &sh, int rank, uint32_t *h,
                                      uint32_t *next, uint32_t need, unsigned long long &bk)
{
    __syncthreads();
    for (int x = threadIdx.x; x < kBins; x += kPT)
        if (sh.hist[x]) atomicAdd(h + x, sh.hist[x]);
    for (int x = rank * kPT + threadIdx.x; x < kBins; x += d.blocks * kPT) next[x] = 0u;
    if (!p_sync(g.c, bk++, d.blocks, d.limit_ns)) return false;
    constexpr int kPer = kBins / kPT;
    uint32_t v[kPer], s = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        v[q] = __ldcg(h + threadIdx.x * kPer + q);
        s += v[q];
    }
    uint32_t tot;
    const uint32_t ex = p_block_excl(s, sh.red32, tot);
    uint32_t above = tot - ex - s;  // keys in the bins above this thread's
#pragma unroll
    for (int q = kPer - 1; q >= 0; --q) {
        if (above < need && above + v[q] >= need) {
            sh.cut = (uint32_t)(threadIdx.x * kPer + q);
            sh.above = above;
            sh.in = v[q];
        }
        above += v[q];
    }
    __syncthreads();
    return true;
}

// Sorts key[0 .. n2), n2 a power of two >= 64, in decreasing order.  A warp
// holds the pairs of 64 keys in a row, so strides up to 32 need no block
// barrier.
__device__ __forceinline__ void p_sort(unsigned long long *key, int n2)
{
    static_assert(kMaxBatch <= 2 * kPT, "one pair per thread");
    const int x = threadIdx.x;
    const bool mine = x < (n2 >> 1);
    for (int size = 2; size <= n2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride > 32 || (stride == 32 && size > 64)) __syncthreads();
            else __syncwarp();
            if (mine) {
                const int i = ((x & ~(stride - 1)) << 1) | (x & (stride - 1)), j = i + stride;
                const unsigned long long a = key[i], b = key[j];
                if ((i & size) == 0 ? a < b : a > b) {
                    key[i] = b;
                    key[j] = a;
                }
            }
        }
    __syncthreads();
}

__global__ void __launch_bounds__(kPT, 1) k_part_grow(const PDev d)
{
    __shared__ PShared sh;
    const int grp = blockIdx.x / d.blocks, rank = blockIdx.x - grp * d.blocks, t = d.t0 + grp;
    const PGroup g = d.g[grp];
    PCtl *c = g.c;
    // this block's neurons
    const long long lo = d.M * rank / d.blocks, hi = d.M * (rank + 1) / d.blocks;
    const int lane = threadIdx.x & 31, tid = threadIdx.x;
    const long long gwarp = ((long long)rank * kPT + tid) >> 5, nwarp = ((long long)d.blocks * kPT) >> 5;
    const unsigned long long idmask = (1ull << d.idbits) - 1ull;
    unsigned long long bk = 0;  // barriers passed
    int hcur = 0;               // histogram to fill next
    long long n_un = d.M;       // unassigned neurons (the same in every block, as all of the part's state)
    bool ok = true;

    for (int k = 0; k < d.P - 1 && ok && n_un > 0; ++k) {
        // a new part: clear the shared weights; find the seed
        unsigned int m = 0xFFFFFFFFu, n = 0;
        for (long long j = lo + tid; j < hi; j += kPT) {
            g.acc[j] = 0ull;
            if (__ldcg(g.lab + j) < 0) {
                ++n;
                m = min(m, (unsigned int)j);
            }
        }
        unsigned int *seed_id = &c->seed_id[k % 3];
        if (t == 1) {
            m = __reduce_min_sync(0xFFFFFFFFu, m);
            if (lane == 0 && m != 0xFFFFFFFFu) atomicMin(seed_id, m);
        } else {
            n = p_block_sum(n, sh.red32);
            if (tid == 0) g.cnt[rank] = n;
        }
        if (!(ok = p_sync(c, bk++, d.blocks, d.limit_ns))) break;
        if (t != 1) {
            // the r-th unassigned neuron in id order, r = word mod unassigned
            const unsigned long long r =
                (unsigned long long)p_philox_word0(d.seed, (uint32_t)t, (uint32_t)k, 0xA1u) % (unsigned long long)n_un;
            unsigned long long pre = 0;
            for (int x = tid; x < rank; x += kPT) pre += __ldcg(g.cnt + x);
            pre = p_block_sum(pre, sh.redu);
            const unsigned long long mine = __ldcg(g.cnt + rank);
            if (r >= pre && r < pre + mine) {
                // walk the slice in blocks of kPT ids, scanning the flags
                unsigned long long want = r - pre;
                for (long long j0 = lo; j0 < hi; j0 += kPT) {
                    const long long j = j0 + tid;
                    const unsigned int f = (j < hi && __ldcg(g.lab + j) < 0) ? 1u : 0u;
                    unsigned int tot;
                    const unsigned int ex = p_block_excl(f, sh.red32, tot);
                    if (f && ex == want) *(volatile unsigned int *)seed_id = (unsigned int)j;
                    if (want < tot) break;
                    want -= tot;
                }
            }
            if (!(ok = p_sync(c, bk++, d.blocks, d.limit_ns))) break;
        }
        const unsigned int seed = __ldcg(seed_id);
        // (the word of part k + 2: last read before this part's first barrier)
        if (rank == 0 && tid == 0) *(volatile unsigned int *)&c->seed_id[(k + 2) % 3] = 0xFFFFFFFFu;
        if (seed >= (unsigned long long)d.M) {
            // no seed found (the same in every block): record it and end
            if (tid == 0) atomicOr(&c->status, kPStFault);
            return;
        }
        if (tid == 0) {
            sh.added[0] = seed;
            if (seed >= lo && seed < hi) g.lab[seed] = k;
        }
        __syncthreads();
        long long wk = d.W[seed], nk = 1;  // weight and size of part k
        int na = 1;                        // members that joined in the last round
        --n_un;

        while (wk * (long long)d.P < d.Wtot && n_un > 0) {
            // scatter: (member, direction, chunk of kChunk synapses) per warp
            const long long tasks = (long long)na * 2 * d.chunks;
            for (long long x = gwarp; x < tasks; x += nwarp) {
                const long long mem = x / (2 * d.chunks);
                const uint32_t a = sh.added[mem];
                const int rem = (int)(x - mem * (2 * d.chunks));
                const bool in = rem >= d.chunks;
                const long long ch = rem - (in ? d.chunks : 0);
                const long long *ptr = in ? d.in_ptr : d.ptr;
                const uint32_t *list = in ? d.in_src : d.tgt;
                const long long s0 = ptr[a] + ch * kChunk, s1 = min(ptr[a + 1], s0 + kChunk);
                const unsigned long long wa = d.W[a];
                uint32_t j[kPUnroll];
#pragma unroll
                for (int q = 0; q < kPUnroll; ++q)
                    if (s0 + lane + 32 * q < s1) j[q] = list[s0 + lane + 32 * q];
#pragma unroll
                for (int q = 0; q < kPUnroll; ++q)
                    if (s0 + lane + 32 * q < s1) atomicAdd(g.acc + j[q], wa);
            }
            uint32_t need = (uint32_t)min((long long)d.B, n_un);
            if (d.grow > 0) need = (uint32_t)min((long long)need, max(1ll, nk / d.grow));
            for (int x = tid; x < kBins; x += kPT) sh.hist[x] = 0u;
            if (!(ok = p_sync(c, bk++, d.blocks, d.limit_ns))) break;
            if (rank == 0 && tid == 0) *(volatile unsigned int *)&c->nsel = 0u;

            // select: bins of the gains; neurons without gain count per warp
            const auto key_of = [&](long long j) -> unsigned long long {
                return __ldcg(g.lab + j) >= 0 ? 0ull
                                              : (unsigned long long)d.W[j] * __ldcg(g.acc + j) << d.idbits |
                                                    (idmask - (unsigned long long)j);
            };
            for (long long j0 = lo; j0 < hi; j0 += kPT) {
                const long long j = j0 + tid;
                const unsigned long long kj = j < hi ? key_of(j) : 0ull;
                const uint32_t bin = p_bin(kj >> d.idbits, d.mbits);
                const unsigned int zero = __ballot_sync(0xFFFFFFFFu, kj != 0ull && bin == 0u);
                if (kj != 0ull && bin != 0u) atomicAdd(&sh.hist[bin], 1u);
                if (lane == 0 && zero) atomicAdd(&sh.hist[0], (uint32_t)__popc(zero));
            }
            int hnext = hcur == kHists - 1 ? 0 : hcur + 1;
            if (!(ok = p_cut(d, g, sh, rank, g.hist + hcur * kBins, g.hist + hnext * kBins, need, bk))) break;
            hcur = hnext;
            unsigned long long base;  // the bound's bin: keys base .. base + 2^width - 1
            int width;
            p_bin_range(sh.cut, d.mbits, d.idbits, base, width);
            uint32_t above = sh.above, in = sh.in;
            while (above + in > (uint32_t)kMaxBatch && width > 0) {
                // more keys reach the bin than a round's list holds: split it
                const int shift = max(0, width - kDigit);
                __syncthreads();
                for (int x = tid; x < kBins; x += kPT) sh.hist[x] = 0u;
                __syncthreads();
                for (long long j = lo + tid; j < hi; j += kPT) {
                    const unsigned long long off = key_of(j) - base;
                    // (an assigned neuron's key 0 lies below every bin's keys but those of base 0, where key 0
                    // is excluded by itself)
                    if (off >> width == 0ull && off + base != 0ull) atomicAdd(&sh.hist[off >> shift], 1u);
                }
                hnext = hcur == kHists - 1 ? 0 : hcur + 1;
                if (!(ok = p_cut(d, g, sh, rank, g.hist + hcur * kBins, g.hist + hnext * kBins, need - above, bk)))
                    break;
                hcur = hnext;
                base += (unsigned long long)sh.cut << shift;
                width = shift;
                above += sh.above;
                in = sh.in;
            }
            if (!ok) break;
            const uint32_t ns = above + in;
            // list the keys >= base: this block's into shared memory, then one place in the list for them
            if (tid == 0) sh.n = 0u;
            __syncthreads();
            for (long long j = lo + tid; j < hi; j += kPT) {
                const unsigned long long kj = key_of(j);
                if (kj != 0ull && kj >= base) {
                    const uint32_t pos = atomicAdd(&sh.n, 1u);
                    if (pos < (uint32_t)kMaxBatch) sh.key[pos] = kj;  // (more is a fault, flagged below)
                }
            }
            __syncthreads();
            if (tid == 0 && sh.n) sh.base = atomicAdd(&c->nsel, sh.n);
            __syncthreads();
            for (uint32_t x = tid; x < min(sh.n, (uint32_t)kMaxBatch); x += kPT)
                if (sh.base + x < (uint32_t)kMaxBatch) g.sel[sh.base + x] = sh.key[x];
            if (!(ok = p_sync(c, bk++, d.blocks, d.limit_ns))) break;

            // join: the listed keys in decreasing order; the first `need`
            // join while the part's weight is below sum(W)/P
            if (__ldcg(&c->nsel) != ns || ns < need || ns > (uint32_t)kMaxBatch) {
                // not the round's size (the same in every block): record it and end
                if (tid == 0) atomicOr(&c->status, kPStFault);
                return;
            }
            int n2 = 64;
            while (n2 < (int)ns) n2 <<= 1;
            for (int x = tid; x < n2; x += kPT) sh.key[x] = x < (int)ns ? __ldcg(g.sel + x) : 0ull;
            __syncthreads();
            p_sort(sh.key, n2);
            // inclusive prefix sums of the members' weights, kPer per thread
            constexpr int kPer = kMaxBatch / kPT;
            long long w[kPer], s = 0;
            uint32_t id[kPer];
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int x = tid * kPer + q;
                w[q] = 0;
                if (x < (int)need) {
                    id[q] = (uint32_t)(idmask - (sh.key[x] & idmask));
                    w[q] = (long long)d.W[id[q]];
                }
                s += w[q];
            }
            unsigned long long tot;
            long long run = (long long)p_block_excl((unsigned long long)s, sh.redu, tot);
            // members before the first one whose join fills the part
            unsigned int cont = 0;
            long long pre[kPer];
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                run += w[q];
                pre[q] = run;
                const int x = tid * kPer + q;
                cont += x < (int)need && (wk + run) * (long long)d.P < d.Wtot && n_un - x - 1 > 0;
            }
            na = min((int)need, (int)p_block_sum(cont, sh.red32) + 1);
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int x = tid * kPer + q;
                if (x >= na) continue;
                sh.added[x] = id[q];
                if (id[q] >= lo && id[q] < hi) g.lab[id[q]] = k;
                if (x == na - 1) sh.redu[0] = (unsigned long long)pre[q];
            }
            __syncthreads();
            wk += (long long)sh.redu[0];
            nk += na;
            n_un -= na;
        }
    }
    if (!ok) return;
    // the last part takes the rest
    __syncthreads();
    for (long long j = lo + tid; j < hi; j += kPT)
        if (__ldcg(g.lab + j) < 0) g.lab[j] = d.P - 1;
    if (!p_sync(c, bk++, d.blocks, d.limit_ns)) return;
    // objective (sum over cut synapses of W_i W_j) and part weights; one
    // warp per source neuron
    unsigned long long cut = 0;
    for (long long i = gwarp; i < d.M; i += nwarp) {
        const int li = __ldcg(g.lab + i);
        const unsigned long long wi = d.W[i];
        if (lane == 0) atomicAdd(g.wpart + li, wi);
        for (long long e0 = d.ptr[i] + lane; e0 < d.ptr[i + 1]; e0 += 32 * kPUnroll) {
            uint32_t j[kPUnroll];
            int lj[kPUnroll];
#pragma unroll
            for (int q = 0; q < kPUnroll; ++q) j[q] = e0 + 32 * q < d.ptr[i + 1] ? d.tgt[e0 + 32 * q] : (uint32_t)i;
#pragma unroll
            for (int q = 0; q < kPUnroll; ++q) lj[q] = __ldcg(g.lab + j[q]);
#pragma unroll
            for (int q = 0; q < kPUnroll; ++q)
                if (lj[q] != li) cut += wi * d.W[j[q]];
        }
    }
    cut = p_block_sum(cut, sh.redu);
    if (tid == 0 && cut) atomicAdd(&c->obj, cut);
}

// ------------------------------------------------------------------ host
struct PLayout {
    size_t ctl, ptr, in_ptr, tgt, in_src, W, fill, best, acc[kGroups], lab[kGroups], hist, sel, cnt, wpart, total;
};

constexpr int kMaxGrid = 4096;

PLayout p_layout(long long M, long long E, int P)
{
    PLayout L;
    size_t o = 0;
    auto put = [&](size_t &f, size_t bytes) {
        f = o;
        o += (bytes + 255) & ~(size_t)255;
    };
    put(L.ctl, sizeof(PCtl) * kGroups);
    put(L.ptr, 8 * (size_t)(M + 1));
    put(L.in_ptr, 8 * (size_t)(M + 1));
    put(L.tgt, 4 * (size_t)(E > 0 ? E : 1));
    put(L.in_src, 4 * (size_t)(E > 0 ? E : 1));
    put(L.W, 4 * (size_t)M);
    put(L.best, 4 * (size_t)M);
    for (int g = 0; g < kGroups; ++g) {
        put(L.acc[g], 8 * (size_t)M);
        put(L.lab[g], 4 * (size_t)M);
    }
    L.fill = L.lab[0];  // (the in-list build ends before the growth begins)
    put(L.hist, 4 * (size_t)kGroups * kHists * kBins);
    put(L.sel, 8 * (size_t)kGroups * kMaxBatch);
    put(L.cnt, 4 * (size_t)kMaxGrid);
    put(L.wpart, 8 * (size_t)P * kGroups);
    L.total = o;
    return L;
}

int bit_length(unsigned long long x)
{
    int n = 0;
    while (x) {
        ++n;
        x >>= 1;
    }
    return n;
}

#define PCK(x)                                    \
    do {                                          \
        cudaError_t e_ = (x);                     \
        if (e_ != cudaSuccess) return SNN_E_CUDA; \
    } while (0)

}  // namespace

extern "C" void snn_partition_device_params_default(snn_partition_device_params *p)
{
    if (!p) return;
    std::memset(p, 0, sizeof(*p));
    p->iters = 4;
    p->batch = 2048;
    p->grow = 2;
    p->seed = 7;
}

extern "C" int snn_partition_device_workspace_bytes(const snn_network *net, int32_t P, size_t *bytes)
{
    if (!net || !net->syn_ptr || net->n_neurons <= 0 || !bytes || P < 1 || P > net->n_neurons) return SNN_E_ARG;
    *bytes = p_layout(net->n_neurons, net->syn_ptr[net->n_neurons], P).total;
    return SNN_OK;
}

extern "C" int snn_partition_device(const snn_network *net, int32_t P, const snn_partition_device_params *prm,
                                    void *workspace, size_t workspace_bytes, void *stream, int32_t *part_of,
                                    snn_partition_stats *stats)
{
    if (!net || !net->syn_ptr || !prm || !part_of || !workspace) return SNN_E_ARG;
    const long long M = net->n_neurons;
    if (M <= 0 || P < 1 || P > M) return SNN_E_ARG;
    if (M >= (1ll << snn::kTgtBits)) return SNN_E_RANGE;
    if (prm->iters < 1 || prm->batch < 1 || prm->batch > kMaxBatch || prm->grow < 0) return SNN_E_ARG;
    const long long E = net->syn_ptr[M];
    if (net->syn_ptr[0] != 0 || E < 0 || (E > 0 && !net->syn_tgt)) return SNN_E_ARG;
    const PLayout L = p_layout(M, E, P);
    if (workspace_bytes < L.total || ((uintptr_t)workspace & 255)) return SNN_E_NOMEM;
    cudaStream_t st = (cudaStream_t)stream;
    char *w = (char *)workspace;

    int dev = 0, sms = 0, coop = 0, occ = 0;
    PCK(cudaGetDevice(&dev));
    PCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PCK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return SNN_E_NODEV;
    PCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_part_grow, kPT, 0));
    if (occ < 1) return SNN_E_NODEV;
    // one block per SM, shared out among the iterations that run side by side
    const int grid = std::min(kMaxGrid, sms);

    PDev d;
    std::memset(&d, 0, sizeof(d));
    d.ptr = (const long long *)(w + L.ptr);
    d.tgt = (const uint32_t *)(w + L.tgt);
    d.in_ptr = (long long *)(w + L.in_ptr);
    d.in_src = (uint32_t *)(w + L.in_src);
    d.W = (uint32_t *)(w + L.W);
    d.fill = (uint32_t *)(w + L.fill);
    for (int g = 0; g < kGroups; ++g) {
        PGroup &x = d.g[g];
        x.acc = (unsigned long long *)(w + L.acc[g]);
        x.lab = (int32_t *)(w + L.lab[g]);
        x.hist = (uint32_t *)(w + L.hist) + (size_t)g * kHists * kBins;
        x.sel = (unsigned long long *)(w + L.sel) + (size_t)g * kMaxBatch;
        x.cnt = (uint32_t *)(w + L.cnt) + (size_t)g * (kMaxGrid / kGroups);
        x.wpart = (unsigned long long *)(w + L.wpart) + (size_t)g * P;
        x.c = (PCtl *)(w + L.ctl) + g;
    }
    d.M = M;
    d.E = E;
    d.Wtot = E;
    d.P = P;
    d.B = prm->batch;
    d.grow = prm->grow;
    d.seed = prm->seed;
    d.limit_ns = 2000000000ull;

    // tables to the device; in-lists and the key width on the device
    PCK(cudaMemcpyAsync((void *)d.ptr, net->syn_ptr, 8 * (size_t)(M + 1), cudaMemcpyHostToDevice, st));
    if (E > 0) PCK(cudaMemcpyAsync((void *)d.tgt, net->syn_tgt, 4 * (size_t)E, cudaMemcpyHostToDevice, st));
    PCK(cudaMemsetAsync(w + L.ctl, 0, sizeof(PCtl), st));
    PCK(cudaMemsetAsync(d.fill, 0, 4 * (size_t)M, st));
    const int g2 = sms * 8;
    k_part_degrees<<<g2, 256, 0, st>>>(d);
    k_part_scan<<<1, 1024, 0, st>>>(d);
    k_part_in_lists<<<g2, 256, 0, st>>>(d);
    k_part_bounds<<<g2, 256, 0, st>>>(d);
    PCK(cudaGetLastError());
    PCtl ctl[kGroups];
    PCK(cudaMemcpyAsync(ctl, w + L.ctl, sizeof(PCtl), cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
    if (ctl[0].status & kPStRange) return SNN_E_ARG;
    d.idbits = std::max(1, bit_length((unsigned long long)M));
    const int gbits = bit_length(ctl[0].gain_max);
    if (gbits + d.idbits > 64) return SNN_E_RANGE;
    d.mbits = kDigit;  // as many bins per power of two as the gains' range leaves
    while ((std::max(0, gbits - d.mbits) + 1) << d.mbits > kBins) --d.mbits;
    d.chunks = (int)std::max(1ull, (ctl[0].deg_max + kChunk - 1) / kChunk);

    std::vector<unsigned long long> wp((size_t)P);
    unsigned long long best = 0;
    for (int t = 1; t <= prm->iters; t += d.groups) {
        d.t0 = t;
        d.groups = std::min(kGroups, prm->iters - t + 1);
        d.blocks = std::max(1, grid / d.groups);
        std::memset(ctl, 0, sizeof(ctl));
        for (PCtl &c : ctl)
            for (unsigned int &x : c.seed_id) x = 0xFFFFFFFFu;
        PCK(cudaMemcpyAsync(w + L.ctl, ctl, sizeof(ctl), cudaMemcpyHostToDevice, st));
        for (int g = 0; g < d.groups; ++g) PCK(cudaMemsetAsync(d.g[g].lab, 0xFF, 4 * (size_t)M, st));
        PCK(cudaMemsetAsync(w + L.hist, 0, 4 * (size_t)kGroups * kHists * kBins, st));
        PCK(cudaMemsetAsync(w + L.wpart, 0, 8 * (size_t)P * kGroups, st));
        void *args[] = {&d};
        PCK(cudaLaunchCooperativeKernel((const void *)k_part_grow, dim3(d.blocks * d.groups), dim3(kPT), args, 0, st));
        PCK(cudaMemcpyAsync(ctl, w + L.ctl, sizeof(ctl), cudaMemcpyDeviceToHost, st));
        PCK(cudaStreamSynchronize(st));
        for (int g = 0; g < d.groups; ++g) {
            if (ctl[g].status & kPStTimeout) return SNN_E_TIMEOUT;
            if (ctl[g].status & kPStFault) return SNN_E_STATE;
        }
        for (int g = 0; g < d.groups; ++g)
            if (t + g == 1 || ctl[g].obj < best) {
                best = ctl[g].obj;
                PCK(cudaMemcpyAsync(w + L.best, d.g[g].lab, 4 * (size_t)M, cudaMemcpyDeviceToDevice, st));
                PCK(cudaMemcpyAsync(wp.data(), d.g[g].wpart, 8 * (size_t)P, cudaMemcpyDeviceToHost, st));
            }
    }
    PCK(cudaMemcpyAsync(part_of, w + L.best, 4 * (size_t)M, cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
    if (stats) {
        stats->objective = (int64_t)best;
        stats->min_weight = (int64_t)*std::min_element(wp.begin(), wp.end());
        stats->max_weight = (int64_t)*std::max_element(wp.begin(), wp.end());
    }
    return SNN_OK;
}
