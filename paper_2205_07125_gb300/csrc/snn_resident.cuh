// Resident step kernel (sm_103a), included by snn_sim.cu after snn_step.cuh:
// the whole dynamic state of a network on the chip, one exchange between
// blocks per step.
//
// Block b owns the contiguous run of N neurons from b N: their membrane
// potentials, refractory counters and next drive in registers, their pending
// input of the next S = max delay steps in shared memory.  A step t is
//   update    input slot t mod S is consumed (and becomes the slot of step
//             t + S), LIF update and threshold;
//   publish   the block's spikes go to every block's mailbox as 8-byte words
//             that carry a tag of the step: a reader that sees the tag has
//             the ids with it, so no fence and no flag is needed;
//   drive     the drive and leak of step t + 1 while the words travel;
//   gather    the block reads its mailbox: the step's spike list;
//   deliver   the synapses of the step's spikes that end in this block, of
//             every delay, with shared-memory reductions.
// Only the gather waits for other blocks.  A block that has every block's
// spikes of step t needs nothing else of them: its input is its own.  Hence
// one exchange per step where the push form (k_persist) needs two grid
// barriers, and shared-memory reductions where it needs L2 reductions.
// The mailboxes are in the blocks' shared memory when the blocks fit in one
// cluster (CLU), else in global memory (L2).
//
// The exchange of the two-level route (arXiv 2205.07125, Sec. IV.B: buckets
// per destination VN, inboxes per destination partition) and the raster run
// beside the steps on r.walkers warps of their own: each source partition's
// pairs belong to one block, which keeps their fill counters in shared
// memory and walks the partition's spikes of step t while step t + 1 updates.
//
// What bounds it: the chain of a step's dependent parts, not bandwidth.  At
// 4,096 neurons (8 blocks, 2.8 us per step): update 0.35, publish 0.5, gather
// 1.1 (the drive of the next step inside it), two dependent loads and the
// reductions of the delivery 0.75.  At 1,048,576 neurons and 1,000 synapses
// (152 blocks, 13.7 us): a lookup per (spike, block), 137,000 of 32 bytes per
// step, takes 3.9 us and the waits on the block with the most synapses 3.
// Measured against k_persist with the delay ring, us per step (GB300, 10 Hz):
//   4,096 neurons, 100 synapses, delay 1          8.3 -> 2.8
//   16,384 neurons, 100 synapses, delays 1-8      9.0 -> 3.0
//   65,536 neurons, 200 synapses, reordered ids  10.6 -> 4.1
//   200,003 neurons, 137 synapses                15.1 -> 5.7
//   1,048,576 neurons, 1,000 synapses            17.1 -> 13.7
//
// Delivery by target block needs each neuron's synapses grouped by the block
// that owns the target: k_res_build makes that copy, 4 bytes per synapse
// (input index (delay - 1) N + local target, below 2^16 because the input
// slots fit in shared memory, and the int16 weight) and {first, length} of
// each (neuron, block) run.
#pragma once

namespace {

constexpr int kResMaxThreads = 1024;
constexpr int kResMaxCluster = 8;   // (the portable cluster size)
constexpr uint32_t kResNone = 0xFFFFFFFFu;
constexpr uint32_t kResEmpty = 0xFFFFu;  // empty id place in a mailbox word (local ids are below 2^14)
constexpr uint32_t kResShort = 4;      // runs of at most this many synapses: one lane
constexpr uint32_t kResPiece = 128;    // longer ones in pieces, a warp each
constexpr int kResEntries = 3;         // routing entries in flight per lane of a walking warp

// Offsets in k_resident's shared memory: exchange regions of the block's
// pairs, mailbox (CLU), pieces, step's list, own lists and duty lists (by step parity),
// fill counters, drive counts, spike counts per block (by parity).
struct ResSmem {
    uint32_t slot, mail, piece, list, own, duty, pc, kb, cnt;
};

struct Res {
    const uint2 *ptr;           // [M * G] {first synapse, synapses} of each (neuron, target block) run
    const uint32_t *syn;        // [E] input index << 16 | uint16 weight, by (neuron, target block)
    unsigned long long *mail;   // [2][G][G][W] mailbox words of each block from each block, by the tag's parity
    uint32_t *dovf;             // [2][2 M] spikes past the blocks' duty lists (a block's from a1 + a2)
    unsigned long long *ovf;    // [2][G * N] ids that the words have no place for, {id, tag}
    const long long *pbase;     // [P + 1] first internal neuron of each internal partition
    const uint32_t *bptr, *iptr;  // [P + 1] first exchange pair of each source partition (levels 1, 2)
    int G, N, S;                // blocks, neurons per block (a multiple of 4), input slots
    int W, wsh;                 // words per message: 4 or 8; log2(W / 2)
    int lcap, ocap, dcap, pcap; // entries of the step's list, a block's own list, duty list, pieces
    int npair;                  // exchange pairs a block keeps, at most
    int walkers;                // warps beside the steps
    int kbytes;                 // drive arrivals in shared memory (a byte per neuron; reordered ids)
    int prefetch;               // pull the spikes' rows into L2 (tables larger than it)
    unsigned int few;           // spikes per step up to which 4 to 32 lanes take one each
    unsigned int most;          // mean spikes per step above which another kernel is faster
    int first;                  // the first launch of a call of several (Dev::t_base)
    uint32_t tag0;              // tag of the launch's first step
    uint32_t key[20];           // Philox round keys of a single network's drive
    ResSmem o;
};

// Ids that fit in a message of W words, each {tag, 3 ids} of 16 bits, the
// first id's place taken by the count.  The words are written and read in
// pairs by L = W / 2 lanes: place f (0..5) of lane l holds id f L + l - 1, so
// that a block's few spikes spread over the lanes.
__host__ __device__ constexpr int res_pub(int W)
{
    return 3 * W - 1;
}

// Places the arrays of k_resident's shared memory after the input slots.
__host__ inline size_t res_smem(Res &r, bool clu)
{
    size_t o = ((size_t)r.S * r.N * 4 + 15) / 16 * 16;
    auto place = [&](size_t bytes) {
        const size_t at = o;
        o += bytes;
        return (uint32_t)at;
    };
    r.o.slot = place((size_t)r.npair * 16);
    r.o.mail = place(clu ? (size_t)2 * r.G * r.W * 8 : 0);
    r.o.piece = place((size_t)r.pcap * 8);
    r.o.list = place((size_t)r.lcap * 4);
    r.o.own = place((size_t)2 * r.ocap * 4);
    r.o.duty = place((size_t)2 * r.dcap * 4);
    r.o.pc = place((size_t)r.npair * 4);
    r.o.kb = place(r.kbytes ? (size_t)r.N : 0);
    r.o.cnt = place((size_t)2 * r.G * 2);
    return (o + 15) / 16 * 16;
}

// Exchange units: 2 p = level 1 of source partition p, 2 p + 1 = level 2.
// Block b keeps units [b U / G, (b + 1) U / G), U = 2 P: partitions
// [pa1, pb1) at level 1 and [pa2, pb2) at level 2.
struct ResDuty {
    int pa1, pb1, pa2, pb2;
};

__host__ __device__ inline ResDuty res_duty(int b, int G, int P)
{
    const long long U = 2ll * P;
    const int ua = (int)(U * b / G), ub = (int)(U * (b + 1) / G);
    ResDuty r;
    r.pa1 = (ua + 1) / 2;
    r.pb1 = (ub + 1) / 2;
    r.pa2 = ua / 2;
    r.pb2 = ub / 2;
    return r;
}

// The synapses of every neuron grouped by target block, a warp per neuron:
// count per block, bounds, placement (order inside a run is free: the
// deliveries are integer sums).  E < 2^32.
__global__ void __launch_bounds__(kThreads) k_res_build(const unsigned long long *csr, const uint32_t *syn_td,
                                                        const int16_t *syn_w, long long M, int G, int N,
                                                        uint2 *ptr, uint32_t *syn)
{
    extern __shared__ uint32_t s_hist[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *h = s_hist + (size_t)wid * G;
    const long long nw = ((long long)gridDim.x * kThreads) >> 5;
    for (long long i = ((long long)blockIdx.x * kThreads + threadIdx.x) >> 5; i < M; i += nw) {
        const unsigned long long o0 = csr[i], o1 = csr[i + 1];
        for (int c = lane; c < G; c += 32) h[c] = 0u;
        __syncwarp();
        for (unsigned long long x = o0 + lane; x < o1; x += 32)
            atomicAdd(&h[(syn_td[x] & kTgtMask) / (uint32_t)N], 1u);
        __syncwarp();
        uint32_t carry = 0;
        for (int c0 = 0; c0 < G; c0 += 32) {
            const int c = c0 + lane;
            const uint32_t v = c < G ? h[c] : 0u;
            uint32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= o) inc += y;
            }
            if (c < G) {
                ptr[(size_t)i * G + c] = make_uint2((uint32_t)o0 + carry + inc - v, v);
                h[c] = carry + inc - v;
            }
            carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        __syncwarp();
        for (unsigned long long x = o0 + lane; x < o1; x += 32) {
            const uint32_t td = syn_td[x];
            const uint32_t tgt = td & kTgtMask, c = tgt / (uint32_t)N;
            const uint32_t pos = atomicAdd(&h[c], 1u);
            const uint32_t idx = (td >> kTgtBits) * (uint32_t)N + (tgt - c * (uint32_t)N);
            syn[o0 + pos] = (idx << 16) | (uint32_t)(uint16_t)syn_w[x];
        }
        __syncwarp();
    }
}

__device__ __forceinline__ ulonglong2 ld_words(const unsigned long long *p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ ulonglong2 ld_words_shared(uint32_t a)
{
    ulonglong2 v;
    asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void st_words(unsigned long long *p, unsigned long long x, unsigned long long y)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}

// Two words to shared address a (this block's view) of block `rank` of the cluster.
__device__ __forceinline__ void st_words_cluster(uint32_t a, int rank, unsigned long long x, unsigned long long y)
{
    asm volatile(
        "{ .reg .u32 q; mapa.shared::cluster.u32 q, %0, %1; st.relaxed.cluster.shared::cluster.v2.u64 [q], {%2, %3}; }" ::
            "r"(a), "r"(rank), "l"(x), "l"(y)
        : "memory");
}

__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_word(unsigned long long *p, uint32_t x, uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)tag << 32) | x) : "memory");
}

// (Each barrier is taken by whole warps.)
__device__ __forceinline__ void cluster_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void bar_sync(int id, int n)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

__device__ __forceinline__ void bar_arrive(int id, int n)
{
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Named barriers of k_resident: the step warps; own list and duty list
// ready, both free again (by step parity); the walking warps.
enum { kBarMain = 1, kBarReady = 2, kBarFree = 4, kBarWalk = 6 };

// Loops are not unrolled unless their loads are to be in flight together: a step walks its code once, so the
// code's length is latency.
#define RES_COLD __device__ __forceinline__

// Drive arrivals (finite thresholds <= word, as drive_units) of the words of w, a byte each, by every threshold.
RES_COLD uint32_t drive_counts_slow(const uint32_t *th, int fin, uint4 w)
{
    uint32_t kc = 0;
#pragma unroll 1
    for (int e = 0; e < 4; ++e) {
        const uint32_t u = uint4_word(w, (uint32_t)e);
        int k = 0;
#pragma unroll 1
        while (k < fin && u >= th[k]) ++k;
        kc |= (uint32_t)k << (8 * e);
    }
    return kc;
}

// The drive of a network: its first six thresholds (absent ones 2^32 - 1), all of them, its Philox key and
// first id.
struct ResDrive {
    uint32_t t[6];
    const uint32_t *th;
    int fin;
    uint32_t key0, key1, off;
};

__device__ __forceinline__ ResDrive res_drive(const Dev &d, uint32_t g)
{
    ResDrive r;
    if (!d.net_of) {
#pragma unroll
        for (int k = 0; k < 6; ++k) r.t[k] = d.th32[k];
        r.th = d.th32;
        r.fin = d.th_fin;
        r.key0 = d.key0;
        r.key1 = d.key1;
        r.off = 0;
    } else {
        const NetDrive *nd = d.net_drive + __ldg(d.net_of + (g >> 2));
#pragma unroll
        for (int k = 0; k < 6; ++k) r.t[k] = __ldg(nd->th + k);
        r.th = nd->th;
        r.fin = __ldg(&nd->fin);
        r.key0 = __ldg(&nd->key0);
        r.key1 = __ldg(&nd->key1);
        r.off = (uint32_t)__ldg(&nd->off);
    }
    return r;
}

// philox4 with the round keys given (constant operands).
__device__ __forceinline__ uint4 philox4_keys(const uint32_t *key, uint32_t c0, uint32_t c1)
{
    uint32_t x0 = c0, x1 = c1, x2 = 0u, x3 = 0u;
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, x0), lo0 = 0xD2511F53u * x0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, x2), lo1 = 0xCD9E8D57u * x2;
        x0 = hi1 ^ x1 ^ key[2 * i];
        x1 = lo1;
        x2 = hi0 ^ x3 ^ key[2 * i + 1];
        x3 = lo0;
    }
    return make_uint4(x0, x1, x2, x3);
}

// Drive arrivals of four words, a byte each: five thresholds compared at once; a word past the sixth (0.02 % of
// them at 0.8 arrivals per step) takes the loop.
__device__ __forceinline__ uint32_t drive_counts(const ResDrive &r, uint4 w)
{
    if (__builtin_expect(max(max(w.x, w.y), max(w.z, w.w)) >= r.t[5], 0)) return drive_counts_slow(r.th, r.fin, w);
    uint32_t c[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        c[0] += w.x >= r.t[k];
        c[1] += w.y >= r.t[k];
        c[2] += w.z >= r.t[k];
        c[3] += w.w >= r.t[k];
    }
    return (c[0] | c[1] << 8) | (c[2] | c[3] << 8) << 16;
}

// Hash terms and the input record of the quad from internal id j (nv neurons) at step t.
RES_COLD ulonglong2 res_record(const Dev &d, bool do_hash, int32_t *cur, uint32_t j, int nv, int4 i4, float4 v4)
{
    unsigned long long hc = 0, hv = 0;
#pragma unroll 1
    for (int e = 0; e < 4 && e < nv; ++e) {
        const int32_t i = e == 0 ? i4.x : e == 1 ? i4.y : e == 2 ? i4.z : i4.w;
        const float v = e == 0 ? v4.x : e == 1 ? v4.y : e == 2 ? v4.z : v4.w;
        const uint32_t g = d.gid ? d.gid[j + e] : j + e;
        if (do_hash) {
            hc += mix64(((unsigned long long)g << 32) | (uint32_t)i);
            hv += mix64(((unsigned long long)g << 32) | __float_as_uint(v));
        }
        if (cur) cur[j + e] = i;
    }
    return make_ulonglong2(hc, hv);
}

RES_COLD void res_hash(const Dev &d, long long t, unsigned long long hc, unsigned long long hv)
{
    hc = warp_sum(hc);
    hv = warp_sum(hv);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&d.hash[2 * t], hc);
        atomicAdd(&d.hash[2 * t + 1], hv);
    }
}

// Whether both words of v carry the tag.
__device__ __forceinline__ bool tagged(ulonglong2 v, uint32_t tag)
{
    return !((((uint32_t)v.x ^ tag) | ((uint32_t)v.y ^ tag)) & 0xFFFFu);
}

// Mailbox words at p (global) or, with p == nullptr, at shared address a: wait until they carry the tag,
// at most limit_ns (then kStTimeout, *abort and empty words).
RES_COLD ulonglong2 res_wait_words(const unsigned long long *p, uint32_t a, uint32_t tag, unsigned int *status,
                                   unsigned int *abort, unsigned long long limit_ns)
{
    const unsigned long long deadline = global_ns() + limit_ns;
    unsigned int spins = 0;
#pragma unroll 1
    for (;;) {
        const ulonglong2 v = p ? ld_words(p) : ld_words_shared(a);
        if (tagged(v, tag)) return v;
        if ((++spins & 255u) == 0u) {
            if (global_ns() > deadline) atomicOr(status, kStTimeout);
            if (*(volatile unsigned int *)status & kStTimeout) {
                *abort = 1u;
                return make_ulonglong2(~0ull, ~0ull);
            }
        }
    }
}

// Id at p (an {id, tag} word), waiting for its tag as res_wait_words.
RES_COLD uint32_t res_fetch(const unsigned long long *p, uint32_t tag, unsigned int *status, unsigned int *abort,
                            unsigned long long limit_ns)
{
    const unsigned long long deadline = global_ns() + limit_ns;
    unsigned int spins = 0;
#pragma unroll 1
    for (;;) {
        const unsigned long long v = ld_word(p);
        if ((uint32_t)(v >> 32) == tag) return (uint32_t)v;
        if ((++spins & 255u) == 0u) {
            if (global_ns() > deadline) atomicOr(status, kStTimeout);
            if (*(volatile unsigned int *)status & kStTimeout) {
                *abort = 1u;
                return kResNone;
            }
        }
    }
}

// What a block keeps of the exchange: id ranges of its source partitions at
// both levels, their pairs' regions and fill counters.
struct ResWalk {
    uint32_t a1, b1, a2, b2;   // internal ids of the partitions at level 1 and 2
    uint32_t bp0, ip0, nb, np; // first pair of each level; level-1 pairs (level-2 ones follow in slot / pc), all
    const ulonglong2 *slot;
    uint32_t *pc;
    uint32_t *more;            // spikes past the duty list (even steps)
};

// Messages by kind (slots C_EVENTS .. of the tally row).
struct ResTally {
    unsigned long long ev = 0;
    unsigned int c[6] = {0, 0, 0, 0, 0, 0};  // l1 local, l1 cross-VN, l2 by class
};

// Add a thread's tallies to the block's.
__device__ __forceinline__ void res_tally(const ResTally &ty, unsigned long long *tally)
{
    if (ty.ev) atomicAdd(&tally[0], ty.ev);
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (ty.c[k]) atomicAdd(&tally[1 + k], (unsigned long long)ty.c[k]);
}

// a4 + a5 for n spikes whose source partition the block keeps, list[0, ..) in
// shared memory and past cap entries more[0, ..) in global memory, by warps
// [0, ww): 32 spikes per warp, a lane per entry.  The fill counters are the
// block's own, so a reservation is a shared-memory add.
__device__ __forceinline__ void res_walk(const Dev &d, const ResWalk &w, const uint32_t *list, const uint32_t *more,
                                         unsigned int cap, unsigned int n, int wid, int ww, ResTally &ty,
                                         unsigned int *status)
{
    const int lane = threadIdx.x & 31;
    unsigned int ovf = 0;
#pragma unroll 1
    for (unsigned int x0 = 0; x0 < n; x0 += 32u * (unsigned int)ww) {
        const unsigned int x = x0 + (unsigned int)(lane * ww + wid);
        const uint32_t id = x >= n ? kResNone : x < cap ? list[x] : *(const volatile uint32_t *)(more + (x - cap));
        const bool d1 = id >= w.a1 && id < w.b1, d2 = id >= w.a2 && id < w.b2;
        uint32_t e0 = 0, n1 = 0, f0 = 0, n2 = 0;
        int vn0 = 0;
        if (d1 || d2) {
            const uint2 ra = d.row[id], rb = d.row[id + 1];
            e0 = ra.x;
            n1 = d1 ? rb.x - ra.x : 0u;
            f0 = ra.y;
            n2 = d2 ? rb.y - ra.y : 0u;
            vn0 = d.src_part[id] / d.vn_size;
        }
        // the entries of the warp's spikes numbered through (level 1: pass 0, level 2: pass 1), several per
        // lane in flight; a lane finds the spike of its entry by a search over the lanes' prefix sums
#pragma unroll 1
        for (int level = 0; level < 2; ++level) {
            const uint32_t c = level ? n2 : n1, first = level ? f0 : e0;
            uint32_t inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= o) inc += y;
            }
            const uint32_t ex = inc - c, tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
#pragma unroll 1
            for (uint32_t y0 = 0; y0 < tot; y0 += 32u * kResEntries) {
                uint32_t f[kResEntries], q[kResEntries];
                int vs[kResEntries];
                DevL2 l[kResEntries];
                int g[kResEntries];
#pragma unroll
                for (int u = 0; u < kResEntries; ++u) {
                    const uint32_t y = y0 + 32u * (uint32_t)u + (uint32_t)lane;
                    int src = 0;
#pragma unroll
                    for (int h = 16; h > 0; h >>= 1) {
                        const uint32_t v = __shfl_sync(0xFFFFFFFFu, ex, src + h);
                        if (v <= y) src += h;
                    }
                    f[u] = __shfl_sync(0xFFFFFFFFu, first, src) + (y - __shfl_sync(0xFFFFFFFFu, ex, src));
                    vs[u] = __shfl_sync(0xFFFFFFFFu, vn0, src);
                    q[u] = kResNone;
                    if (y < tot) {
                        if (level) {
                            l[u] = d.l2[f[u]];
                            q[u] = d.l2_pair[f[u]] - w.ip0 + w.nb;
                        } else {
                            g[u] = d.l1_vn[f[u]];
                            q[u] = d.l1_pair[f[u]] - w.bp0;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < kResEntries; ++u) {
                    if (q[u] == kResNone) continue;
                    const unsigned int pos = atomicAdd(&w.pc[q[u]], 1u);
                    const ulonglong2 sl = w.slot[q[u]];
                    if (level) {
                        // a5: the relay expands the entry into inbox (p, q) of partition q
                        if (pos < sl.y)
                            d.inbox[sl.x + pos] =
                                ((l[u].off & kOffMask) << kLenBits) | (unsigned long long)l[u].len;
                        else ovf |= kStInbox;
                        ty.ev += l[u].len;
                        ty.c[2] += l[u].cls == 0;
                        ty.c[3] += l[u].cls == 1;
                        ty.c[4] += l[u].cls == 2;
                        ty.c[5] += l[u].cls == 3;
                    } else {
                        // a4: one level-1 entry per destination VN, appended to bucket (p, g)
                        if (pos < sl.y) d.bucket[sl.x + pos] = f[u];
                        else ovf |= kStBucket;
                        ty.c[0] += g[u] == vs[u];
                        ty.c[1] += g[u] != vs[u];
                    }
                }
            }
        }
    }
    if (ovf) atomicOr(status, ovf);
}

// Add a synapse word to the input slots (rot: the slot of delay 1).
__device__ __forceinline__ void res_add(int32_t *ring, uint32_t rot, uint32_t SN, uint32_t x)
{
    uint32_t a = (x >> 16) + rot;
    if (a >= SN) a -= SN;
    atomicAdd(ring + a, (int32_t)(int16_t)(x & 0xFFFFu));
}

// Pending input of the block's neurons, steps t0 .. t0 + S - 1, from the delay ring into the input slots.  What a
// short call costs beside its steps: several loads in flight per thread, in 16 bytes where the rows are aligned.
__device__ __forceinline__ void res_load(const int32_t *rows, int D, long long M, int32_t *ring, long long t0, int S, int N, int nloc)
{
    const int all = blockDim.x, r0 = (int)(t0 % D), s0 = (int)(t0 % S);
    auto go = [&](auto *to, const auto *from, int n, int have, long long row) {
        constexpr int kU = 8;
#pragma unroll 1
        for (int x0 = threadIdx.x; x0 < S * n; x0 += kU * all) {
            typename std::remove_reference<decltype(*to)>::type v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int x = x0 + u * all, s = x / n, y = x - s * n;
                v[u] = {};
                if (s < S && y < have) v[u] = from[(r0 + s >= D ? r0 + s - D : r0 + s) * row + y];
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int x = x0 + u * all, s = x / n, y = x - s * n;
                if (s < S) to[(s0 + s >= S ? s0 + s - S : s0 + s) * n + y] = v[u];
            }
        }
    };
    if (M % 4 == 0)  // (jb, N and so nloc are multiples of 4 then)
        go(reinterpret_cast<int4 *>(ring), reinterpret_cast<const int4 *>(rows), N / 4, nloc / 4, M / 4);
    else
        go(ring, rows, N, nloc, M);
}

// The input slots back as the pending input of steps te .. te + S - 1; the delay ring's other slots are empty.  Out
// of line: in line it made the step loop of 4,096 neurons 2.5 % slower.
__device__ __noinline__ void res_store(int32_t *rows, int D, long long M, const int32_t *ring, long long te, int S, int N,
                                       int nloc)
{
    const int all = blockDim.x, r0 = (int)(te % D), s0 = (int)(te % S);
    auto go = [&](auto *to, const auto *from, int n, int have, long long row) {
#pragma unroll 4
        for (int x = threadIdx.x; x < D * n; x += all) {
            const int s = x / n, y = x - s * n;
            if (y < have)
                to[(r0 + s >= D ? r0 + s - D : r0 + s) * row + y] =
                    s < S ? from[(s0 + s >= S ? s0 + s - S : s0 + s) * n + y]
                          : typename std::remove_reference<decltype(*to)>::type{};
        }
    };
    if (M % 4 == 0)
        go(reinterpret_cast<int4 *>(rows), reinterpret_cast<const int4 *>(ring), N / 4, nloc / 4, M / 4);
    else
        go(rows, ring, N, nloc, M);
}

// T steps, one launch (cooperative, or one cluster: CLU).  QPT: quads of
// neurons per step thread, at most; REC: hashes and input records.  Waits are bounded as in k_persist
// (limit_ns each, kStTimeout); skip (tests of the bounded wait): block 0 does
// not publish the first step.
template <int QPT, bool CLU, bool REC>
__global__ void __launch_bounds__(kResMaxThreads, 1)
    k_resident(const __grid_constant__ Dev d, const __grid_constant__ Res r, int T, unsigned long long limit_ns,
               int skip)
{
    extern __shared__ __align__(128) unsigned char s_dyn[];
    // by step parity: own spikes, list entries, a message was too small, duty entries, pieces, the step was
    // given up
    __shared__ unsigned int s_on[2], s_ln[2], s_over[2], s_dn[2], s_pn[2], s_quit[2];
    // a wait of the step ran out: in the gather, in the delivery.  Each word is read behind a barrier that all
    // writers of it have passed and before the next one, so the warps agree and no barrier loses some of them.
    __shared__ unsigned int s_abort, s_abort2;
    __shared__ unsigned int s_done;
    __shared__ unsigned long long s_ph[kPhases], s_spikes;
    __shared__ long long s_head;  // raster head (walking warps)
    __shared__ unsigned long long s_tally[kTally];
    int32_t *const ring = reinterpret_cast<int32_t *>(s_dyn);
    Ctrl *c = d.ctrl;
    // a later launch of a call: another kernel's turn, or the call was given up
    if (d.t_base && !r.first && (*(volatile unsigned int *)d.hot || call_left(d) != T)) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int all = blockDim.x, nt = all - 32 * r.walkers, nw = nt >> 5;  // step threads, step warps
    const int G = r.G, b = blockIdx.x, N = r.N, S = r.S;
    const uint32_t SN = (uint32_t)(S * N);
    const uint32_t jb = (uint32_t)b * (uint32_t)N;
    const int nloc = (int)max(0ll, min((long long)N, d.M - (long long)jb)), nq = (nloc + 3) / 4;
    const long long t0 = *(volatile long long *)&c->t;

    // the state into registers and shared memory
    float4 V[QPT];
    uint32_t ref[QPT], kc[QPT];
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int q = tid + k * nt;
        V[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        ref[k] = 0u;
        kc[k] = 0u;
        if (tid < nt && q < nq) {
            const long long j = (long long)jb + 4 * q;
            if (j + 4 <= d.M) {
                V[k] = *reinterpret_cast<const float4 *>(d.V + j);
                ref[k] = *reinterpret_cast<const uint32_t *>(d.ref + j);
            } else {
                float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 3; ++e)
                    if (j + e < d.M) {
                        v[e] = d.V[j + e];
                        ref[k] |= (uint32_t)d.ref[j + e] << (8 * e);
                    }
                V[k] = make_float4(v[0], v[1], v[2], 0.f);
            }
        }
    }
    res_load(d.ring + jb, d.D, d.M, ring, t0, S, N, nloc);
    // the exchange pairs this block keeps
    ulonglong2 *const slot = reinterpret_cast<ulonglong2 *>(s_dyn + r.o.slot);
    uint32_t *const pc = reinterpret_cast<uint32_t *>(s_dyn + r.o.pc);
    __shared__ ResWalk wk;
    if (tid == 0) {
        const ResDuty du = res_duty(b, G, d.P);
        wk.a1 = (uint32_t)r.pbase[du.pa1];
        wk.b1 = (uint32_t)r.pbase[du.pb1];
        wk.a2 = (uint32_t)r.pbase[du.pa2];
        wk.b2 = (uint32_t)r.pbase[du.pb2];
        wk.bp0 = r.bptr[du.pa1];
        wk.ip0 = r.iptr[du.pa2];
        wk.nb = r.bptr[du.pb1] - wk.bp0;
        wk.np = wk.nb + r.iptr[du.pb2] - wk.ip0;
        wk.slot = slot;
        wk.pc = pc;
        wk.more = r.dovf + (size_t)wk.a1 + wk.a2;
    }
    __syncthreads();
    const uint32_t np = wk.np;
#pragma unroll 1
    for (uint32_t x = tid; x < np; x += all) {
        slot[x] = x < wk.nb ? d.bucket_slot[wk.bp0 + x] : d.inbox_slot[wk.ip0 + (x - wk.nb)];
        pc[x] = 0u;
    }
    if constexpr (CLU) {
        // mailbox words with a tag that no step near the launch's start has
        unsigned long long *mb = reinterpret_cast<unsigned long long *>(s_dyn + r.o.mail);
#pragma unroll 1
        for (int x = tid; x < 2 * G * r.W; x += all) mb[x] = (unsigned long long)((r.tag0 + 0x8000u) & 0xFFFFu);
    }
    if (tid < kTally) s_tally[tid] = 0ull;
    if (tid < 2) s_on[tid] = s_ln[tid] = s_over[tid] = s_dn[tid] = s_pn[tid] = s_quit[tid] = 0u;
    if (tid < kPhases) s_ph[tid] = 0ull;
    if (tid == 0) {
        s_abort = s_abort2 = 0u;
        s_head = *(volatile long long *)&c->head[slot3(t0)];
        s_spikes = 0ull;
    }
    __syncthreads();
    if constexpr (CLU) cluster_sync();  // every mailbox is ready

    uint32_t *const own0 = reinterpret_cast<uint32_t *>(s_dyn + r.o.own);
    uint32_t *const duty0 = reinterpret_cast<uint32_t *>(s_dyn + r.o.duty);
    uint16_t *const cnt0 = reinterpret_cast<uint16_t *>(s_dyn + r.o.cnt);
    if (wid >= nw) {
        // ------------------------------------------------ walking warps: raster, exchange
        const int ww = wid - nw;
        ResTally ty;
#pragma unroll 1
        for (int s = 0; s < T; ++s) {
            const int par = s & 1;
            const uint32_t *own = own0 + par * r.ocap;
            bar_sync(kBarReady + par, all);
            const unsigned int mine = s_on[par], nd = s_dn[par];
            if (s_quit[par]) break;
            if (ww == r.walkers - 1) {
                // raster: the block's spikes at the head plus the counts of the blocks before it
                const long long t = t0 + s;
                const uint16_t *cnt = cnt0 + par * G;
                unsigned int before = 0, tot = mine;
                if (G > 1) {
                    tot = 0;
#pragma unroll 1
                    for (int g = lane; g < G; g += 32) {
                        tot += cnt[g];
                        if (g < b) before += cnt[g];
                    }
                    tot = __reduce_add_sync(0xFFFFFFFFu, tot);
                    before = __reduce_add_sync(0xFFFFFFFFu, before);
                }
                const long long head = s_head;
                if (head >= 0)
#pragma unroll 1
                    for (unsigned int k = lane; k < mine; k += 32)
                        d.spk[head + before + k] =
                            k < (unsigned int)r.ocap
                                ? own[k]
                                : (uint32_t)ld_word(r.ovf + ((size_t)((r.tag0 + (uint32_t)s) & 1u) * G + b) * N + k);
                const long long hn = next_head(d, head, tot, t);
                __syncwarp();
                if (lane == 0) {
                    if (b == 0) {
                        if (hn >= 0) {
                            d.raster_off[t + 1] = hn;
                            c->rec_steps = t + 1;
                        } else if (head >= 0) {
                            atomicOr(&c->status, kStRaster);
                        }
                    }
                    s_head = hn;
                    s_spikes += tot;
                }
            }
#pragma unroll 1
            for (uint32_t x = tid - nt; x < np; x += 32 * r.walkers) pc[x] = 0u;
            bar_sync(kBarWalk, 32 * r.walkers);
            if (tid == nt) s_on[par] = s_dn[par] = 0u;
            res_walk(d, wk, duty0 + par * r.dcap, wk.more + (size_t)par * 2 * d.M, (unsigned int)r.dcap, nd, ww, r.walkers,
                     ty, &c->status);
            if ((s & 255) == 255 || s + 1 == T) {  // (32-bit tallies)
                res_tally(ty, s_tally);
                ty = ResTally();
            }
            bar_arrive(kBarFree + par, all);
        }
    } else {
        // ------------------------------------------------ step warps
        uint32_t *const list0 = reinterpret_cast<uint32_t *>(s_dyn + r.o.list);
        unsigned long long *const piece = reinterpret_cast<unsigned long long *>(s_dyn + r.o.piece);
        uint8_t *const kb = s_dyn + r.o.kb;
        const uint32_t mail_s = smem_u32(s_dyn + r.o.mail);
        const int nm = G << r.wsh;  // pairs of words of a step's messages into one mailbox
        const int pub = res_pub(r.W);

        // drive and leak of step t, ahead of its input.  With reordered ids a
        // neuron's drive word comes from a Philox block of its own: then a
        // thread per neuron, the counts through kb.
        auto prepare = [&](uint32_t t) {
            if (r.kbytes)
#pragma unroll 1
                for (int x = tid; x < nloc; x += nt) {
                    const uint32_t g = __ldg(d.gid + jb + x);
                    const ResDrive dr = res_drive(d, g);
                    const uint32_t u = uint4_word(d.net_of ? philox4(dr.key0, dr.key1, (g - dr.off) >> 2, t)
                                                           : philox4_keys(r.key, g >> 2, t),
                                                  g & 3u);
                    kb[x] = (uint8_t)drive_counts(dr, make_uint4(u, 0u, 0u, 0u));
                }
#pragma unroll
            for (int k = 0; k < QPT; ++k) {
                const int q = tid + k * nt;
                if (q < nq) {
                    if (!r.kbytes) {
                        const uint32_t j = jb + 4u * (uint32_t)q;
                        const ResDrive dr = res_drive(d, j);
                        kc[k] = drive_counts(dr, d.net_of ? philox4(dr.key0, dr.key1, (j - dr.off) >> 2, t)
                                                          : philox4_keys(r.key, j >> 2, t));
                    }
                    V[k] = make_float4(lif_leak(d, V[k].x), lif_leak(d, V[k].y), lif_leak(d, V[k].z),
                                       lif_leak(d, V[k].w));
                }
            }
        };
        // profiling: block 0's time per part (snn_profile_phases)
        const bool prof = d.phase_ns != nullptr && b == 0 && tid == 0;
        unsigned long long stamp = prof ? global_ns() : 0ull;
        auto part = [&](int k) {
            if (prof) {
                const unsigned long long now = global_ns();
                s_ph[k] += now - stamp;
                stamp = now;
            }
        };
        // the next step with an input record
        long long cur_next = -1;
        if (REC && d.cur_every > 0) cur_next = (t0 + d.cur_every - 1) / d.cur_every * d.cur_every;

        prepare((uint32_t)t0);
        bar_sync(kBarMain, nt);
        int ts = (int)(t0 % S), done = 0;
        int nfree = 0;  // steps whose lists the walking warps have handed back
        auto wait_free = [&](int upto) {
#pragma unroll 1
            for (; nfree <= upto; ++nfree) bar_sync(kBarFree + (nfree & 1), all);
        };
#pragma unroll 1
        for (int s = 0; s < T; ++s) {
            // lp: the half of the mailboxes, by the tag.  Tags only go up, so a half is written again every second
            // tag whatever the step numbers do (a reset or a restored state takes them back), and no word is old
            // enough for its 16 bits to come round.
            const uint32_t tag = r.tag0 + (uint32_t)s;
            const int par = s & 1, lp = (int)(tag & 1u);
            uint32_t *own = own0 + par * r.ocap;
            uint16_t *cnt = cnt0 + par * G;
            // records of the step
            bool do_hash = false;
            int32_t *cur = nullptr;
            unsigned long long hc = 0, hv = 0;
            if constexpr (REC) {
                if (t0 + s < d.hash_steps) do_hash = true;
                if (t0 + s == cur_next) {
                    const long long k = cur_next / d.cur_every;
                    if (k < d.cur_slots) cur = d.cur_rec + k * d.M;
                    cur_next += d.cur_every;
                }
            }
            // the lists of this parity are free again (the walk of step s - 2 is over)
            wait_free(s - 2);
            // update: consume input slot ts, finish the LIF step, note the spikes
            // (the arithmetic of lif_finish; the refractory bytes of a quad together)
            uint32_t spikes = 0;
#pragma unroll
            for (int k = 0; k < QPT; ++k) {
                const int q = tid + k * nt;
                if (q < nq) {
                    int4 *ip = reinterpret_cast<int4 *>(ring + ts * N) + q;
                    const int4 i4 = *ip;
                    *ip = make_int4(0, 0, 0, 0);
                    const uint32_t kk = r.kbytes ? reinterpret_cast<const uint32_t *>(kb)[q] : kc[k];
                    float vv[4] = {V[k].x, V[k].y, V[k].z, V[k].w};
                    const int32_t ii[4] = {i4.x, i4.y, i4.z, i4.w};
                    const uint32_t rf = ref[k];
                    uint32_t m = 0, rn = __vsubus4(rf, 0x01010101u);
                    const int nv = nloc - 4 * q;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t ext = ((kk >> (8 * e)) & 0xFFu) * (uint32_t)d.w_ext + (uint32_t)d.i_bias;
                        const float x = __fadd_rn(
                            vv[e], __fmul_rn(__int2float_rn((int32_t)((uint32_t)ii[e] + ext)), 0.0009765625f));
                        const bool held = (rf & (0xFFu << (8 * e))) != 0u, spk = !held && x >= d.v_th && e < nv;
                        vv[e] = (held || spk) ? d.v_reset : x;
                        if (spk) {
                            m |= 1u << e;
                            rn |= (uint32_t)d.t_ref << (8 * e);
                        }
                    }
                    V[k] = make_float4(vv[0], vv[1], vv[2], vv[3]);
                    ref[k] = rn;
                    spikes |= m << (4 * k);
                    if (REC && (do_hash || cur)) {
                        const ulonglong2 h = res_record(d, do_hash, cur, jb + 4u * (uint32_t)q, nv, i4, V[k]);
                        hc += h.x;
                        hv += h.y;
                    }
                }
            }
            if (spikes) {
                unsigned int pos = atomicAdd(&s_on[par], (unsigned int)__popc(spikes));
#pragma unroll 1
                for (; spikes; spikes &= spikes - 1u, ++pos) {
                    const uint32_t e = (uint32_t)__ffs(spikes) - 1u;
                    const uint32_t x = 4u * ((uint32_t)tid + (e >> 2) * (uint32_t)nt) + (e & 3u);
                    if (pos < (unsigned int)r.ocap) own[pos] = jb + x;
                    if (pos >= (unsigned int)(G == 1 ? r.ocap : pub))
                        st_word(r.ovf + ((size_t)lp * G + b) * N + pos, jb + x, tag);
                }
            }
            if (REC && do_hash) res_hash(d, t0 + s, hc, hv);
            part(0);
            bar_sync(kBarMain, nt);
            const unsigned int mine = s_on[par];
            // publish: the count and the first ids to every block's mailbox, two words per thread
            if (G > 1 && !(skip && s == 0 && b == 0)) {
#pragma unroll 1
                for (int i = tid; i < nm; i += nt) {
                    const int dst = i >> r.wsh, jj = i - (dst << r.wsh);
                    uint32_t id[6];
#pragma unroll
                    for (int e = 0; e < 6; ++e) {
                        const int x = (e << r.wsh) + jj - 1;
                        id[e] = x < 0 ? mine : (unsigned int)x < mine ? own[x] - jb : kResEmpty;
                    }
                    const uint32_t h = tag & 0xFFFFu;
                    const unsigned long long x = (h | id[0] << 16) | (unsigned long long)(id[1] | id[2] << 16) << 32;
                    const unsigned long long y = (h | id[3] << 16) | (unsigned long long)(id[4] | id[5] << 16) << 32;
                    if constexpr (CLU)
                        st_words_cluster(mail_s + (uint32_t)((lp * G + b) * r.W + 2 * jj) * 8u, dst, x, y);
                    else
                        st_words(r.mail + (((size_t)lp * G + dst) * G + b) * r.W + 2 * jj, x, y);
                }
            }
            if (tid == 0) s_ln[par ^ 1] = s_over[par ^ 1] = s_pn[par ^ 1] = 0u;
            part(1);
            // while the words travel: the rows of the block's spikes into L2 (a warp per spike), and the next step's
            // drive and leak
            const uint32_t pid = r.prefetch && (unsigned int)wid < min(mine, (unsigned int)r.ocap) ? own[wid] : kResNone;
            uint32_t pf0 = 0, pf1 = 0;
            unsigned long long pc0 = 0, pc1 = 0;
            if (pid != kResNone) {
                const uint2 *p = r.ptr + (size_t)pid * G;
                prefetch_span(p, p + G, lane);
                pc0 = d.csr[pid];
                pc1 = d.csr[pid + 1];
                pf0 = d.row[pid].y;
                pf1 = d.row[pid + 1].y;
            }
            if (s + 1 < T) prepare((uint32_t)t0 + (uint32_t)s + 1u);
            if (pid != kResNone) {
                prefetch_span(r.syn + pc0, r.syn + pc1, lane);
                prefetch_span(d.l2 + pf0, d.l2 + pf1, lane);
                prefetch_span(d.l2_pair + pf0, d.l2_pair + pf1, lane);
            }
            part(2);
            // gather: every block's message, two words per lane, the ids onto the list.  The last warps read first:
            // with few neurons per block they have no drive to compute.
            auto message = [&](int i, bool wait, uint32_t (&id)[6]) {  // words 2 i, 2 i + 1; id[0] the count of lane 0
                const unsigned long long *p = CLU ? nullptr : r.mail + ((size_t)lp * G + b) * G * r.W + 2 * i;
                const uint32_t a = mail_s + (uint32_t)(lp * G * r.W + 2 * i) * 8u;
                ulonglong2 v;
                if constexpr (CLU) v = ld_words_shared(a);
                else v = ld_words(p);
                if (wait && !tagged(v, tag)) v = res_wait_words(p, a, tag & 0xFFFFu, &c->status, &s_abort, limit_ns);
                id[0] = (uint32_t)v.x >> 16;
                id[1] = (uint32_t)(v.x >> 32) & 0xFFFFu;
                id[2] = (uint32_t)(v.x >> 48);
                id[3] = (uint32_t)v.y >> 16;
                id[4] = (uint32_t)(v.y >> 32) & 0xFFFFu;
                id[5] = (uint32_t)(v.y >> 48);
            };
            if (G > 1) {
#pragma unroll 1
                for (int i0 = (nw - 1 - wid) * 32; i0 < nm; i0 += nt) {
                    const int i = i0 + lane, g = i >> r.wsh;
                    uint32_t id[6] = {kResEmpty, kResEmpty, kResEmpty, kResEmpty, kResEmpty, kResEmpty};
                    if (i < nm) {
                        message(i, true, id);
                        if (i == g << r.wsh) {
                            if (id[0] == kResEmpty) id[0] = 0u;  // (a message given up)
                            cnt[g] = (uint16_t)id[0];
                            if (id[0] > (uint32_t)pub) s_over[par] = 1u;
                            id[0] = kResEmpty;
                        }
                    }
                    __syncwarp();
                    unsigned int mask[6], tot = 0;
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        mask[k] = __ballot_sync(0xFFFFFFFFu, id[k] != kResEmpty);
                        tot += __popc(mask[k]);
                    }
                    if (tot) {
                        unsigned int pos = 0;
                        if (lane == 0) pos = atomicAdd(&s_ln[par], tot);
                        pos = __shfl_sync(0xFFFFFFFFu, pos, 0);
#pragma unroll
                        for (int k = 0; k < 6; ++k) {
                            const unsigned int x = pos + lane_rank(mask[k]);
                            if (id[k] != kResEmpty && x < (unsigned int)r.lcap)
                                list0[x] = (uint32_t)g * (uint32_t)N + id[k];
                            pos += __popc(mask[k]);
                        }
                    }
                }
                bar_sync(kBarMain, nt);
                if (__builtin_expect(s_over[par] != 0u, 0)) {
                    // blocks with more spikes than a message holds: the rest, a warp per block
#pragma unroll 1
                    for (int g = wid; g < G; g += nw) {
                        const unsigned int cg = cnt[g];
#pragma unroll 1
                        for (unsigned int k0 = pub; k0 < cg; k0 += 32u) {
                            const unsigned int m = min(32u, cg - k0);
                            unsigned int pos = 0;
                            if (lane == 0) pos = atomicAdd(&s_ln[par], m);
                            pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + lane;
                            if ((unsigned int)lane < m && pos < (unsigned int)r.lcap)
                                list0[pos] = res_fetch(r.ovf + ((size_t)lp * G + g) * N + k0 + lane, tag, &c->status,
                                                       &s_abort, limit_ns);
                            __syncwarp();
                        }
                    }
                    bar_sync(kBarMain, nt);
                }
            }
            if (s_abort) break;
            part(3);
            const uint32_t *list = G == 1 ? own : list0;
            const unsigned int n = G == 1 ? mine : s_ln[par];
            const unsigned int fit = (unsigned int)(G == 1 ? r.ocap : r.lcap);
            // deliver
            const uint32_t rot = ts + 1 == S ? 0u : (uint32_t)((ts + 1) * N);  // delay 1: the slot after ts
            auto duty = [&](uint32_t id) {  // the spikes whose partition this block keeps go on the duty list
                if ((id >= wk.a1 && id < wk.b1) || (id >= wk.a2 && id < wk.b2)) {
                    const unsigned int pos = atomicAdd(&s_dn[par], 1u);
                    if (pos < (unsigned int)r.dcap) duty0[par * r.dcap + pos] = id;
                    else wk.more[(size_t)par * 2 * d.M + pos - r.dcap] = id;
                }
            };
            if (n <= min(fit, r.few)) {
                // few spikes: 4 to 32 lanes each walk its run of synapses into this block
                const int sh = n > (unsigned int)(4 * nw)   ? 2
                               : n > (unsigned int)(2 * nw) ? 3
                               : n > (unsigned int)nw       ? 4
                                                            : 5;
                const unsigned int x = (unsigned int)tid >> sh, l = (unsigned int)tid & ((1u << sh) - 1u);
                if (x < n) {
                    const uint32_t id = list[x];
                    const uint2 run = __ldg(r.ptr + (size_t)id * G + b);
                    const uint32_t p1 = run.x + run.y;
#pragma unroll 1
                    for (uint32_t k = run.x + l; k < p1; k += 4u << sh) {
                        uint32_t v[4];
#pragma unroll
                        for (uint32_t u = 0; u < 4u; ++u)
                            if (k + (u << sh) < p1) v[u] = __ldg(r.syn + k + (u << sh));
#pragma unroll
                        for (uint32_t u = 0; u < 4u; ++u)
                            if (k + (u << sh) < p1) res_add(ring, rot, SN, v[u]);
                    }
                    if (l == 0) duty(id);
                }
            } else {
            // many: a spike is one lane's.  Its run is walked at once when it is short, a longer one cut into pieces
            // for the warps.  The words of a short run stay in flight until the lane's next spike.
            uint32_t sw[kResShort], slen = 0;
            auto flush = [&]() {
#pragma unroll
                for (uint32_t k = 0; k < kResShort; ++k)
                    if (k < slen) res_add(ring, rot, SN, sw[k]);
            };
            auto spike = [&](uint32_t id, uint2 run) {  // (whole warp; id kResNone: none)
                uint32_t len = 0, v[kResShort];
                if (id != kResNone) {
                    len = run.y;
                    duty(id);
                }
                const bool sh = len <= kResShort;
#pragma unroll
                for (uint32_t k = 0; k < kResShort; ++k)
                    if (sh && k < len) v[k] = __ldg(r.syn + run.x + k);
                if (__any_sync(0xFFFFFFFFu, !sh)) {
                    const uint32_t c0 = sh ? 0u : (len + kResPiece - 1u) / kResPiece;
                    uint32_t inc = c0;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                        if (lane >= o) inc += y;
                    }
                    uint32_t pos = 0;
                    if (lane == 31) pos = atomicAdd(&s_pn[par], inc);
                    pos = __shfl_sync(0xFFFFFFFFu, pos, 31) + inc - c0;
                    const bool fits = pos + c0 <= (uint32_t)r.pcap;
#pragma unroll 1
                    for (uint32_t k = 0; k < c0; ++k, ++pos) {
                        const uint32_t o = k * kResPiece, w = min(kResPiece, len - o);
                        if (pos < (uint32_t)r.pcap)
                            piece[pos] = fits ? ((unsigned long long)w << 32) | (run.x + o) : 0ull;
                    }
                    // runs that the list has no room for: the warp at once, one after another
#pragma unroll 1
                    for (uint32_t y = __ballot_sync(0xFFFFFFFFu, c0 && !fits); y; y &= y - 1u) {
                        const int src = __ffs(y) - 1;
                        const uint32_t o = __shfl_sync(0xFFFFFFFFu, run.x, src), w = __shfl_sync(0xFFFFFFFFu, len, src);
#pragma unroll 2
                        for (uint32_t k = lane; k < w; k += 32u) res_add(ring, rot, SN, __ldg(r.syn + o + k));
                    }
                }
                flush();
                slen = sh ? len : 0u;
#pragma unroll
                for (uint32_t k = 0; k < kResShort; ++k) sw[k] = v[k];
            };
            // From the list, a spike per lane; when it does not hold the step, batches of up to six spikes per lane
            // from the messages again (one block: its own list), then the spikes that had no place there, a warp
            // per block.
            const bool listed = n <= fit;
            const int lim = listed ? (int)n : G == 1 ? r.ocap : nm;
            int i0 = wid * 32, g1 = wid;
            unsigned int k0 = (unsigned int)(G == 1 ? r.ocap : pub);
#pragma unroll 1
            for (;;) {
                uint32_t id[6] = {kResNone, kResNone, kResNone, kResNone, kResNone, kResNone};
                const int i = i0 + lane;
                if (i0 < lim) {
                    if (listed || G == 1) {
                        if (i < lim) id[0] = list[i];
                    } else if (i < lim) {
                        message(i, false, id);
                        if ((i & ((1 << r.wsh) - 1)) == 0) id[0] = kResEmpty;
#pragma unroll
                        for (int k = 0; k < 6; ++k)
                            id[k] = id[k] == kResEmpty ? kResNone : (uint32_t)(i >> r.wsh) * (uint32_t)N + id[k];
                    }
                    i0 += nt;
                } else if (listed) {
                    break;
                } else {
                    unsigned int cg = 0;
#pragma unroll 1
                    while (g1 < G && k0 >= (cg = G == 1 ? mine : cnt[g1])) {
                        g1 += nw;
                        k0 = (unsigned int)(G == 1 ? r.ocap : pub);
                    }
                    if (g1 >= G) break;
                    if (k0 + lane < cg)
                        id[0] = res_fetch(r.ovf + ((size_t)lp * G + g1) * N + k0 + lane, tag, &c->status, &s_abort2,
                                          limit_ns);
                    k0 += 32u;
                }
                __syncwarp();
                // (places are filled in order: the first one empty in every lane ends the batch)
#pragma unroll 1
                do {
                    spike(id[0], id[0] != kResNone ? __ldg(r.ptr + (size_t)id[0] * G + b) : make_uint2(0u, 0u));
#pragma unroll
                    for (int x = 0; x < 5; ++x) id[x] = id[x + 1];
                    id[5] = kResNone;
                } while (__any_sync(0xFFFFFFFFu, id[0] != kResNone));
            }
            flush();
            part(4);
            bar_sync(kBarMain, nt);
            if (s_abort2) break;
            // the pieces, a warp each, the loads of two in flight
            const unsigned int np2 = min(s_pn[par], (unsigned int)r.pcap);
#pragma unroll 1
            for (unsigned int u0 = wid; u0 < np2; u0 += 2u * (unsigned int)nw) {
                uint32_t v[8], w[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const unsigned int u = u0 + (unsigned int)(k * nw);
                    const unsigned long long pd = u < np2 ? piece[u] : 0ull;
                    w[k] = (uint32_t)(pd >> 32);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if ((uint32_t)(lane + 32 * e) < w[k])
                            v[4 * k + e] = __ldg(r.syn + (uint32_t)pd + (uint32_t)(lane + 32 * e));
                }
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if ((uint32_t)(lane + 32 * e) < w[k]) res_add(ring, rot, SN, v[4 * k + e]);
            }
            }
            part(5);
            bar_sync(kBarMain, nt);
            bar_arrive(kBarReady + par, all);
            part(6);
            if (++ts == S) ts = 0;
            ++done;
        }
        if (done < T) {
            // step `done` was given up: the walking warps wait for its duty list
            if (tid == 0) s_quit[done & 1] = 1u;
            bar_arrive(kBarReady + (done & 1), all);
        }
        wait_free(done - 1);
        if (tid == 0) s_done = (unsigned int)done;
    }
    __syncthreads();

    // the state back: potentials, refractory counters, pending input as the delay ring
    const long long te = t0 + s_done;
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int q = tid + k * nt;
        if (tid < nt && q < nq) {
            const long long j = (long long)jb + 4 * q;
            if (j + 4 <= d.M) {
                *reinterpret_cast<float4 *>(d.V + j) = V[k];
                *reinterpret_cast<uint32_t *>(d.ref + j) = ref[k];
            } else {
                const float v[3] = {V[k].x, V[k].y, V[k].z};
#pragma unroll
                for (int e = 0; e < 3; ++e)
                    if (j + e < d.M) {
                        d.V[j + e] = v[e];
                        d.ref[j + e] = (uint8_t)(ref[k] >> (8 * e));
                    }
            }
        }
    }
    res_store(d.ring + jb, d.D, d.M, ring, te, S, N, nloc);
    // the last step's exchange fill counters (the other parity is the next step's)
    const int pl = (int)((te + 1) & 1);
#pragma unroll 1
    for (uint32_t x = tid; x < np; x += all) {
        const bool l1 = x < wk.nb;
        const size_t k = (size_t)(l1 ? wk.bp0 + x : wk.ip0 + (x - wk.nb)) * kPairStride;
        uint32_t *a = l1 ? bucket_cnt_of(d, pl) : inbox_cnt_of(d, pl);
        uint32_t *z = l1 ? bucket_cnt_of(d, pl ^ 1) : inbox_cnt_of(d, pl ^ 1);
        a[k] = pc[x];
        z[k] = 0u;
    }
    if (tid < kTally && s_tally[tid]) atomicAdd(&d.tally[(size_t)b * C_N + C_EVENTS + tid], s_tally[tid]);
    if (b == 0 && tid == 0) {
        c->head[slot3(te)] = s_head;
        for (int k = 0; k < 3; ++k) c->S_acc[k] = 0u;
        d.counters[C_STEPS] += (unsigned long long)s_done;
        d.counters[C_SPIKES] += s_spikes;
        c->t = te;
        if (s_done < (unsigned int)T) {
            if (d.t_base) *d.t_base = kNoBase;
        } else {
            if (r.first) *d.t_base = t0;
            if (T >= kHotSteps) set_hot(d, s_spikes > (unsigned long long)r.most * (unsigned long long)T);
        }
        for (int k = 0; k < kPhases && d.phase_ns; ++k) d.phase_ns[k] += s_ph[k];
    }
    if constexpr (CLU) cluster_sync();  // no block leaves while another may write to its mailbox
}

}  // namespace
