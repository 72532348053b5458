// queue.cuh -- device side of the cost-bucketed work queue for ragged batches
// (the batch mode of Section 4 for messages of mixed lengths and variants),
// shared by the translation units that instantiate its kernels.
//
// A message's cost is its number of Keccak-f permutations: floor(len/r) + 1
// absorbed blocks plus ceil(d/r) - 1 extra squeezes.  Costs fall into cost
// buckets (exact below 64, 32 per octave above, so the messages of one warp
// differ in cost by at most 1/32; costs of 2^40 and more share the top one),
// and each cost bucket is split by the variant's rate (five rates), so that a
// warp's 32 messages normally share one rate and the absorb can use the
// rate's compile-time form.  The work order lists the buckets longest first.
//   1. k_prep: digest-offset tile sums and a bucket histogram;
//   2. k_scatter: lays the buckets out longest first, digest offsets, and each
//      message's slot in the work order; its first block splits the order between
//      the next two kernels;
//   3. k_sha3_queue: a persistent grid; each warp takes a group of 32
//      consecutive entries of the order with one atomic and hashes one
//      message per thread.  Warps run messages of nearly equal cost.  The
//      queue has two parts of equal work, the costlier with a group for every SM
//      sub-partition at least: on every sub-partition the warp in the lowest
//      hardware slot starts with the costlier (the longest chains start first),
//      the others with the cheaper; either goes on to the other's part when its
//      own is handed out.  Both parts run longest first.
//   k_sha3_lanes runs the first K entries of the order (the K costliest
//   messages; K from the plan, or given) one warp per message, concurrently with
//   the queue kernel, which covers the entries from K on: it is launched first and
//   lets the queue kernel start as soon as its own blocks have.
//
// Why two parts.  Measured on GB300: when two warps of one sub-partition both
// have ALU work ready, the one in the lower hardware warp slot (%warpid)
// issues, and once blocks are prefetched a warp rarely stalls, so the other
// warp only runs in its partner's gaps.  With one queue, a long chain of
// permutations that landed in a higher slot waited behind its partner's
// stream of groups and finished milliseconds after everything else.  With two
// parts the long chains go to the slots that issue first, a warp in a higher
// slot starts with chains of half the work's median at most, and what is handed
// out last, by then to every warp, is the cheapest, so the warps end together.
// (With the higher slots going up from the cheapest group instead, the two met
// in groups of middling cost: 2^20 messages log-uniform to 64 KiB 11.60 ms
// against 11.21, 300,000 4.24 against 4.11.)  Three warps a sub-partition take
// 11.28 and 4.66 ms, the chains of each being slower.  The order of the slots
// affects only speed: every group is taken exactly once, whichever warp takes it.
#pragma once

#include <cstdint>

#include "../../include/sha3gb.h"
#include "coop_sponge.cuh"
#include "keccak_core.cuh"
#include "runtime.cuh"
#include "scan.cuh"
#include "sponge.cuh"
#include "sponge_staged.cuh"

namespace kb {

constexpr int kBucketsPerOctave = 32;
constexpr int kCostBuckets = 64 + 34 * kBucketsPerOctave;  // costs below 2^40 apart; above, one bucket
constexpr int kRateClasses = 5;                              // rates 72, 104, 136, 144, 168 bytes
constexpr int kBuckets = kCostBuckets * kRateClasses;

// How the queue kernel reads message blocks (low two bits) and whether its
// permutation loops over all 24 rounds (kLooped).
constexpr int kStageDirect = 0;  // each thread loads its block's words when it absorbs them
constexpr int kStageAsync = 1;   // the next block is copied into shared memory during the permutation
constexpr int kStageRegs = 2;    // the next block is loaded into registers before the permutation
constexpr int kLooped = 4;

// Permutations a message costs (0 for an invalid variant, which the hashing
// kernel flags and skips).
__device__ __forceinline__ uint64_t message_cost(uint64_t len, int v, uint32_t dlen) {
    if (v > 5) return 0;
    const uint32_t rate = uint32_t(variant_rate(v));
    return len / rate + 1 + (dlen > rate ? (dlen - 1) / rate : 0);
}

__device__ __forceinline__ uint32_t cost_bucket(uint64_t c) {
    if (c < 64) return uint32_t(c);
    const int e = 63 - __clzll(static_cast<long long>(c));  // >= 6
    if (e >= 40) return uint32_t(kCostBuckets - 1);
    return uint32_t(64 + (e - 6) * kBucketsPerOctave + int((c >> (e - 5)) & (kBucketsPerOctave - 1)));
}

// 0..4 by increasing rate; SHA3-256 and SHAKE256 share a rate.
__device__ __forceinline__ uint32_t rate_class(int v) {
    return v == 3 ? 0u : v == 2 ? 1u : (v == 1 || v == 5) ? 2u : v == 0 ? 3u : 4u;
}

// Bucket of a message: cost bucket x rate class, or (for the per-variant
// control schedule) its variant, 6 standing for an invalid one.
template <bool BY_VARIANT>
__device__ __forceinline__ uint32_t bucket_key(uint64_t len, int v, uint32_t dlen) {
    if constexpr (BY_VARIANT) return v > 5 ? 6u : uint32_t(v);
    else return cost_bucket(message_cost(len, v, dlen)) * kRateClasses + (v > 5 ? 0u : rate_class(v));
}

constexpr uint32_t kSlotWords = 48;  // SMs told apart: 192 (beyond, they share bytes, which affects speed only)

struct Control {
    uint32_t count[kBuckets];        // messages per bucket
    uint32_t cursor[kBuckets];       // slots of each bucket in the order that are taken
    unsigned long long head;         // warp-per-message schedule: next entry of the order
    unsigned long long lane_head;    // hybrid: next of the first K entries (one warp each)
    unsigned long long ends;         // queue: groups taken from the cheaper part (high 32 bits) and the costlier (low)
    unsigned long long queue_start;  // queue: first entry of the order it covers (K)
    unsigned long long queue_mid;    // queue: first entry of its cheaper part
    uint32_t slots[kSlotWords];      // queue: a byte per SM, a bit per group of four hardware warp slots in use
    uint32_t ready;                  // 1: k_sha3_lanes has seen the end of k_scatter
};

// The hand-off from k_scatter to a k_sha3_queue that starts beside k_sha3_lanes.
// griddepcontrol.wait covers the kernel before (k_sha3_lanes), whose end the queue
// kernel must not wait for; that kernel's own wait makes k_scatter's writes visible
// to itself alone.  So a thread of k_sha3_lanes that has waited releases a flag, and
// a warp of every block of the queue kernel acquires it for the block.
__device__ __forceinline__ void hand_over(uint32_t *flag) {
    asm volatile("st.release.gpu.b32 [%0], %1;" ::"l"(flag), "r"(1u) : "memory");
}
// False where the flag is not seen within some tens of microseconds (it is set before
// the last block of k_sha3_lanes lets the queue kernel start, so it is there or on its
// way): the caller then waits for the whole of k_sha3_lanes.
__device__ __forceinline__ bool taken_over(const uint32_t *flag) {
    uint32_t v = 0;
    for (int i = 0; i < 64 && v == 0; ++i)
        asm volatile("ld.acquire.gpu.b32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    return v != 0;
}

template <bool BY_VARIANT>
__global__ void __launch_bounds__(kScanThreads)
    k_prep(const uint64_t *lens, const uint8_t *variants,
           const uint32_t *out_lens, uint64_t n, uint64_t *tile_sums, Control *ctl) {
    __shared__ uint32_t hist[kBuckets];
    launch_next();
    for (int b = threadIdx.x; b < kBuckets; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    launch_wait();
    const uint64_t base = uint64_t(blockIdx.x) * kScanTile + uint64_t(threadIdx.x) * kScanItems;
    uint64_t s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const uint64_t i = base + j;
        if (i < n) {
            const uint32_t d = out_lens[i];
            s += d;
            atomicAdd(&hist[bucket_key<BY_VARIANT>(lens[i], variants[i], d)], 1u);
        }
    }
    uint64_t excl;
    const uint64_t total = block_exclusive_scan(s, excl);
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
    __syncthreads();
    for (int b = threadIdx.x; b < kBuckets; b += blockDim.x)
        if (hist[b]) atomicAdd(&ctl->count[b], hist[b]);
}

// Permutations of a message of bucket b (the middle of the bucket's range).
__device__ __forceinline__ uint64_t bucket_cost(int b) {
    const int cb = b / kRateClasses;
    if (cb < 64) return uint64_t(cb);
    const int e = 6 + (cb - 64) / kBucketsPerOctave, m = (cb - 64) % kBucketsPerOctave;
    return (uint64_t(2 * (kBucketsPerOctave + m) + 1) << e) / (2 * kBucketsPerOctave);
}

// How the batch is split between one warp per message (the costliest) and one
// thread per message (the rest), in picoseconds of a GB300: a permutation takes
// kThreadChain in a thread of the queue kernel and kWarpChain in a warp of its
// own; with the GPU full the queue kernel needs kThreadWork for each (4.65 G/s), and
// the kLanesPerSm warps per SM beside it kWarpWork, alone kWarpAlone: the two kernels
// share the issue slots.  kWarpWork is fitted on lengths log-uniform to 64 KiB, us
// before, at 2200 and at 3000: 2,000 messages 4123, 1706, 1727; 20,000 4120, 2335,
// 2386; 100,000 4127, 2813, 2904; 200,000 4201, 3659, 3522; 300,000 4215, 4145, 4196.
// A larger kThreadChain (6000000, 7500000) gains a tenth at 20,000 and loses a tenth
// to a quarter at 300,000.
constexpr uint64_t kThreadChain = 4800000, kWarpChain = 1700000, kThreadWork = 215, kWarpWork = 3000, kWarpAlone = 1750;
constexpr uint64_t kAutoSplit = ~uint64_t(0);

// About how long the batch lasts when the costliest messages, `moved` of the `all`
// permutations, go to warps, the costliest left takes `next` permutations (0: none is
// left) and the costliest of all `top`.  The warps keep kWarpWork while the queue
// kernel runs and kWarpAlone from then on.
__device__ __forceinline__ uint64_t split_time(uint64_t next, uint64_t moved, uint64_t all, uint64_t top) {
    const uint64_t chain = next * kThreadChain, work = all * kThreadWork;
    const uint64_t queue = next == 0 ? 0 : chain > work ? chain : work;
    const uint64_t beside = moved * kWarpWork;
    const uint64_t after = moved * kWarpAlone + queue / kWarpWork * (kWarpWork - kWarpAlone);
    uint64_t t = beside < after ? beside : after;
    if (t < queue) t = queue;
    return moved && t < top * kWarpChain ? top * kWarpChain : t;
}

// The least of a warp's values into a shared word, one atomic a warp.
__device__ __forceinline__ void warp_min_into(unsigned long long &word, uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t other = __shfl_xor_sync(0xffffffffu, v, o);
        v = other < v ? other : v;
    }
    if ((threadIdx.x & 31) == 0) atomicMin(&word, (unsigned long long)v);
}

// The queue kernel's first entry where the plan chooses it: the number of messages
// that are better off with a warp each.  The candidates are the edges between the
// buckets, from none to all; of equal ones the first.  A split has to save an eighth
// by the model to be taken: where it promises less, the warps' share of the issue
// slots slows the chains beside them by as much (20,000 messages of lengths uniform to
// 64 KiB 2434 us split for a promised 4%, 2171 in threads).  (The first edge at which
// the next chain is no longer the longest term, without a look at what the moved work
// takes, gave whole batches of one cost to warps: 20,000 messages of 64 KiB 16353 us,
// 3942 in threads, 10,000 of 4 KiB 594 and 175.)  Called by a whole block; thread t
// holds the counts of buckets kBuckets-1 - (kPer t + j) and, in the buckets above
// them, `before` messages of w permutations out of the batch's `all`.
constexpr int kPer = (kBuckets + kScanThreads - 1) / kScanThreads;
__device__ __forceinline__ uint64_t plan_split(const uint32_t (&count)[kPer], uint64_t before, uint64_t w,
                                               uint64_t all, uint64_t n) {
    __shared__ unsigned long long top_cost, unsplit, best, cut;
    if (threadIdx.x == 0) {
        top_cost = 0;
        unsplit = 0;
        best = ~0ull;
        cut = n;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPer; ++j) {  // the first bucket that is not empty, in descending order of cost
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        if (b >= 0 && count[j] && before == 0) {
            top_cost = bucket_cost(b);
            break;
        }
    }
    __syncthreads();
    uint64_t time[kPer], m = before;  // of the edge before each bucket
    uint64_t least = threadIdx.x == 0 ? split_time(0, all, all, top_cost) : ~0ull;  // every message to a warp
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        time[j] = ~0ull;
        if (b >= 0 && count[j]) {
            const uint64_t c = bucket_cost(b);
            time[j] = split_time(c, w, all, top_cost);
            if (m == 0) unsplit = time[j];
            else least = time[j] < least ? time[j] : least;
            m += count[j];
            w += count[j] * c;
        }
    }
    warp_min_into(best, least);
    __syncthreads();
    if (best >= unsplit - unsplit / 8) return 0;
    m = before;
    least = n;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        if (time[j] == best && m > 0 && m < least) least = m;
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        if (b >= 0) m += count[j];
    }
    warp_min_into(cut, least);
    __syncthreads();
    return cut;
}

// The entry where the queue kernel's cheaper part begins: entries [first, mid) have
// half of the permutations of [first, n).  Where the line lies matters little between
// 3/8 and 5/8 (2^20 messages log-uniform to 64 KiB 11.21 ms at each, 2^19 5.63 ms); at
// 1/4 and 3/4 2^19 messages take 5.89, at 3/4 and 7/8 2^20 take 11.47 and 11.35.
// But the costlier part has at least `least` entries, a group for every SM
// sub-partition: where the batch lasts as long as its longest chains, each of them
// has to start in a slot that issues first, and a back-slot warp given one finishes
// last (6,000 messages of 60,000 bytes beside 44,000 of 200, all in threads: 3647 us
// at half of the work alone, 2041 with 304 groups at least, 2039 with 608, one per
// sub-partition; 20,000 of lengths uniform to 64 KiB 3296, 2888, 2171 and with 1216
// 2876).  Called as plan_split.
__device__ __forceinline__ uint64_t plan_mid(const uint32_t (&count)[kPer], uint64_t before, uint64_t first,
                                             uint64_t w, uint64_t all, uint64_t n, uint64_t least) {
    __shared__ unsigned long long skipped, mid;
    if (threadIdx.x == 0) {
        skipped = 0;
        mid = first;
    }
    __syncthreads();
    uint64_t m = before, u = w;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        if (b >= 0 && count[j]) {
            const uint64_t c = bucket_cost(b);
            if (first > m && first <= m + count[j]) skipped = u + (first - m) * c;
            m += count[j];
            u += count[j] * c;
        }
    }
    __syncthreads();
    const uint64_t target = skipped + (all - skipped) / 2;
    m = before;
    u = w;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        if (b >= 0 && count[j]) {
            const uint64_t c = bucket_cost(b);
            if (c && target > u && target <= u + count[j] * c) mid = m + (target - u + c - 1) / c;
            m += count[j];
            u += count[j] * c;
        }
    }
    __syncthreads();
    const uint64_t left = n > first ? n - first : 0;
    const uint64_t floor = first + (left < least ? left : least);
    return mid < floor ? floor : mid;
}

// Tile sums to the messages' exclusive sums, for batches of so many tiles that each
// block of k_scatter would take long to add up those before its own.
constexpr uint64_t kSumTiles = 4096;
static __global__ void __launch_bounds__(kScanThreads) k_plan_tiles(uint64_t *tile_sums, uint64_t ntiles) {
    launch_next();
    launch_wait();
    uint64_t carry = 0;
    for (uint64_t start = 0; start < ntiles; start += kScanThreads) {
        const uint64_t i = start + threadIdx.x;
        const uint64_t v = i < ntiles ? tile_sums[i] : 0;
        uint64_t excl;
        const uint64_t total = block_exclusive_scan(v, excl);
        if (i < ntiles) tile_sums[i] = carry + excl;
        carry += total;
    }
}

// Digest offsets, and each message's slot in the work order.  Every block lays the
// buckets out by itself, in descending order (bucket kBuckets-1 first), and block 0
// chooses the queue kernel's first entry (`split`, or by plan_split for kAutoSplit): a
// launch of one block for that in between took 9 to 11 us.
template <bool BY_VARIANT>
__global__ void __launch_bounds__(kScanThreads)
    k_scatter(const uint64_t *lens, const uint8_t *variants,
              const uint32_t *out_lens, uint64_t n, const uint64_t *tile_sums,
              uint64_t ntiles, uint64_t *out_off, uint32_t *order, Control *ctl,
              uint64_t split, uint32_t sub_partitions) {
    __shared__ uint32_t hist[kBuckets];
    __shared__ uint32_t start[kBuckets];
    for (int b = threadIdx.x; b < kBuckets; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    launch_wait();
    const uint64_t base = uint64_t(blockIdx.x) * kScanTile + uint64_t(threadIdx.x) * kScanItems;
    uint32_t d[kScanItems], key[kScanItems], rank[kScanItems];
    uint64_t s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const uint64_t i = base + j;
        d[j] = 0;
        key[j] = 0;
        rank[j] = 0;
        if (i < n) {
            d[j] = out_lens[i];
            key[j] = bucket_key<BY_VARIANT>(lens[i], variants[i], d[j]);
            rank[j] = atomicAdd(&hist[key[j]], 1u);
        }
        s += d[j];
    }
    // Bytes of output before this block's messages.
    uint64_t tile = 0, excl;
    if (ntiles > kSumTiles) {
        tile = tile_sums[blockIdx.x];  // k_plan_tiles has added them up
    } else {
        uint64_t mine = 0;
        for (uint64_t t = threadIdx.x; t < blockIdx.x; t += kScanThreads) mine += tile_sums[t];
        tile = block_exclusive_scan(mine, excl);
    }
    block_exclusive_scan(s, excl);
    uint64_t acc = tile + excl;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        if (base + j < n) out_off[base + j] = acc;
        acc += d[j];
    }
    // The buckets' first slots.
    uint32_t count[kPer];
    uint64_t messages = 0, m0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        count[j] = b >= 0 ? ctl->count[b] : 0u;
        messages += count[j];
    }
    block_exclusive_scan(messages, m0);
    uint32_t m = uint32_t(m0);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
        if (b >= 0) start[b] = m + (hist[b] ? atomicAdd(&ctl->cursor[b], hist[b]) : 0u);
        m += count[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        if (base + j < n) order[start[key[j]] + rank[j]] = uint32_t(base + j);
    if (blockIdx.x == 0) {
        uint64_t work = 0, w;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int b = kBuckets - 1 - (int(threadIdx.x) * kPer + j);
            if (b >= 0) work += count[j] * bucket_cost(b);
        }
        const uint64_t all = block_exclusive_scan(work, w);
        const uint64_t first = split == kAutoSplit ? plan_split(count, m0, w, all, n) : split;
        const uint64_t mid = plan_mid(count, m0, first, w, all, n, 32ull * sub_partitions);
        if (threadIdx.x == 0) {
            ctl->queue_start = first;
            ctl->queue_mid = mid;
        }
    }
}

// The persistent queue kernel: one thread per message, 32 messages per
// dequeue.  STAGE picks how blocks are read and the permutation's form
// (kStage* | kLooped).  `beside`: launched to run beside k_sha3_lanes.  No pointer is
// __restrict__: loads of what k_scatter wrote stay behind the hand-off.
template <int MINB, int STAGE>
__global__ void __launch_bounds__(kThreads, MINB)
    k_sha3_queue(const uint8_t *msgs, const uint64_t *offsets,
                 const uint64_t *lens, const uint8_t *variants,
                 const uint32_t *out_lens, const uint64_t *out_off,
                 const uint32_t *order, uint8_t *digests, uint64_t n, Control *ctl,
                 unsigned int *status, bool beside) {
    static_assert(kThreads == 128, "the stage layout assumes 128 threads per block");
    constexpr int kRead = STAGE & 3;
    constexpr bool kLoop = (STAGE & kLooped) != 0;
    __shared__ uint32_t stage_mem[kRead == kStageAsync ? 2 * kStageWords * kThreads : 1];
    const int lane = threadIdx.x & 31;
    // One warp a block asks, so that the block's warps go on together: with each for
    // itself some were late for the look at the slots below and took the longest
    // chains into slots that issue second (2^20 messages at 3 blocks per SM 11.1 to
    // 14.0 ms from call to call, now 11.1).
    if (beside) {
        if (threadIdx.x < 32 && !taken_over(&ctl->ready)) launch_wait();
        __syncthreads();
    }
    const uint64_t start = ctl->queue_start;
    const unsigned long long ngroups = n > start ? (n - start + 31) / 32 : 0;
    const unsigned long long nfront = min((unsigned long long)(ctl->queue_mid - start) / 32, ngroups);
    // Whether this warp is in the lowest hardware slot of its sub-partition that a
    // warp of this kernel holds: warps of k_sha3_lanes may sit below.
    bool front;
    {
        unsigned slot, sm;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
        sm %= 4 * kSlotWords;
        const uint32_t bit = 1u << (slot < 28 ? slot / 4 : 7u);
        uint32_t *word = &ctl->slots[sm / 4];
        uint32_t held = 0;
        if (lane == 0) {
            atomicOr(word, bit << (8 * (sm & 3)));
            __nanosleep(400);  // the SM's other blocks start within this time, if they start now
            held = atomicOr(word, 0u) >> (8 * (sm & 3));
        }
        front = (__shfl_sync(0xffffffffu, held, 0) & 0xffu & (bit - 1)) == 0;
    }
    // One atomic per group; a warp that finds its part handed out goes on to the other.
    for (int parts = 2; parts > 0;) {
        unsigned long long old = 0;
        if (lane == 0) old = atomicAdd(&ctl->ends, front ? 1ull : (1ull << 32));
        old = __shfl_sync(0xffffffffu, old, 0);
        const unsigned long long g = front ? old & 0xffffffffull : nfront + (old >> 32);
        if (g >= (front ? nfront : ngroups)) {
            front = !front;
            --parts;
            continue;
        }
        const uint64_t idx = start + g * 32 + lane;
        if (idx < n) {
            if constexpr (STAGE == kStageDirect) {
                hash_ragged_message(msgs, offsets, lens, variants, out_lens, out_off, digests, order[idx], status);
            } else {
                const uint32_t i = order[idx];
                const int v = variants[i];
                const uint32_t dlen = out_lens[i];
                if (v > 5) {
                    atomicOr(status, KB_DEV_BAD_VARIANT);
                } else if (v < 4 && dlen != uint32_t(variant_digest(v))) {
                    atomicOr(status, KB_DEV_BAD_OUTLEN);
                } else if constexpr (kRead == kStageAsync) {
                    const Stage st = make_stage(stage_mem);
                    sponge_rt_staged<kLoop>(st, msgs + offsets[i], lens[i], v, digests + out_off[i], dlen);
                } else if constexpr (kRead == kStageRegs) {
                    sponge_rt_prefetch<kLoop>(msgs + offsets[i], lens[i], v, digests + out_off[i], dlen);
                } else {
                    sponge_rt_direct<kLoop>(msgs + offsets[i], lens[i], v, digests + out_off[i], dlen);
                }
            }
        }
    }
    launch_wait();  // for k_sha3_lanes, beside which this kernel runs
}

// Device scratch of one call for n messages (the layout queue_issue carves):
// the control block, the digest offsets (8 B per message), the digest scan's
// tile sums (8 B per kScanTile messages) and the work order (4 B per
// message), each part 256-byte aligned where it starts a region.
constexpr size_t queue_scratch_size(uint64_t n) {
    return (sizeof(Control) + 255) / 256 * 256 + 8 * n + 8 * ((n + kScanTile - 1) / kScanTile) +
           (4 * n + 255) / 256 * 256;
}

// Kernel entry points of the staged instances (sha3_queue_staged.cu); nullptr
// for a combination that is not compiled.
const void *queue_kernel_staged(int minb, int stage);

}  // namespace kb
