// sha3_uniform.cu -- fixed-stride batch kernel: one thread per message
// (the paper's granularity of a thread per message, Section 4.1), every
// message the same length and variant (Section 4.3).
//
// Specialisations: for each variant, a compile-time 64-byte message read with
// four 16-byte loads (one rate block: the padding folds into constants and
// round 0 runs on mostly-zero lanes), a runtime length below the rate (one
// block, round 0 on zero capacity lanes), and a general runtime length; the
// runtime forms with 8-byte aligned loads or at any alignment.  The state representation is
// a template parameter: plain 32-bit halves by default, bit-interleaved
// halves as the measured control for SHA3-256.  A thread takes one message, and the
// grid as many blocks as that takes.  Batches that give an SM sub-partition two warps or fewer
// go to sha3_small.cu first.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "keccak_core.cuh"
#include "keccak_interleaved.cuh"
#include "runtime.cuh"
#include "sponge.cuh"
#include "tma.cuh"

namespace kb {
namespace {

// Blocks per SM a kernel is compiled for.  With rotations on the multiply pipe more
// warps keep both pipes fed, as long as nothing spills: 2^24 64-byte messages staged
// by bulk copies 3143 us at 5, 3179 at 6, 3135 at 7; 2^22 messages of 32 bytes 824 at 4,
// 815 at 5 and 6, 805 at 7, of 135 bytes 861, 842, 840 and 830 (at 8 these spill: 3355,
// 867 and 893).  The 64-byte kernel that loads directly takes 868 at 6 and 908 at 7, the
// multi-block kernel is best at kMinBlocks (2^18 messages of 1023 bytes 820; 837 at 5,
// 851 at 6, spilling).
constexpr int min_blocks(int len) { return len == -1 ? kMinBlocks : len == -2 ? 7 : 6; }
constexpr int kStagedMinBlocks = 7;

// LEN >= 0: compile-time message length; -1: runtime; -2: runtime, below the
// rate, with at most one block of output.  A8: base and stride are multiples
// of 8 (16 when LEN == 64).
template <int V, int LEN, bool A8, class Rep>
__global__ void __launch_bounds__(kThreads, min_blocks(LEN))
    k_sha3_uniform(const uint8_t *msgs, uint64_t stride, uint64_t len_rt,
                   uint8_t *out, uint32_t out_len, uint64_t n) {
    using P = Variant<V>;
    launch_wait();
    constexpr int kOut = P::digest ? P::digest : P::rate;
    const uint64_t len = LEN >= 0 ? uint64_t(LEN) : len_rt;
    const uint32_t dlen = P::digest ? uint32_t(P::digest) : out_len;
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t m = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; m < n; m += step) {
        const uint8_t *p = msgs + m * stride;
        uint8_t *dst = out + m * dlen;
        if constexpr (LEN == 64) {
            static_assert(64 < P::rate, "a 64-byte message is one block for every variant");
            uint32_t A[25], B[25];
#pragma unroll
            for (int i = 0; i < 25; ++i) A[i] = B[i] = 0;
            const uint4 *q = reinterpret_cast<const uint4 *>(p);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 v = q[j];
                Rep::set_word(A[2 * j], B[2 * j], v.x, v.y);
                Rep::set_word(A[2 * j + 1], B[2 * j + 1], v.z, v.w);
            }
            // Domain byte at offset 64 (lane 8, byte 0); 0x80 at byte rate-1.
            A[8] ^= Rep::word_a(uint64_t(P::domain));
            B[8] ^= Rep::word_b(uint64_t(P::domain));
            constexpr uint64_t kEnd = uint64_t(0x80) << 56;
            A[P::rate / 8 - 1] ^= Rep::word_a(kEnd);
            B[P::rate / 8 - 1] ^= Rep::word_b(kEnd);
            const uint32_t nsq = dlen > uint32_t(P::rate) ? (dlen - 1) / P::rate : 0;
            for (uint32_t i = 0; i <= nsq; ++i) {
                if (i > 0) squeeze<P::rate, Rep>(A, B, dst + uint64_t(i - 1) * P::rate, P::rate);
                Rep::template permute<true>(A, B);
            }
            squeeze<P::rate, Rep, kOut>(A, B, dst + uint64_t(nsq) * P::rate, dlen - nsq * P::rate);
        } else if constexpr (LEN == -2) {
            // A runtime length below the rate and at most one output block:
            // the message is the padded last block and one permutation,
            // with round 0 on the known-zero capacity lanes folded.
            uint32_t A[25], B[25];
#pragma unroll
            for (int i = 0; i < 25; ++i) A[i] = B[i] = 0;
            absorb_last_same<P::rate, P::domain, A8, Rep>(A, B, p, uint32_t(len));
            keccak_f1600_plain<true, 23, 2>(A, B);
            squeeze<P::rate, Rep, kOut>(A, B, dst, dlen);
        } else {
            sponge<P::rate, P::domain, A8, Rep, true>(p, len, dst, dlen);
        }
    }
}

// The 64-byte form with its messages staged through shared memory by a bulk
// asynchronous copy (cp.async.bulk, completed on an mbarrier): a block takes one
// tile of kThreads consecutive messages (8 KiB, copied by thread 0) and ends; the
// other blocks of its SM hash while its copy is in flight.  Needs stride 64 and a
// 16-byte aligned base in device memory.  A wait that outlasts kWaitNs sets
// KB_DEV_TIMEOUT; the thread then waits (bounded) once more for the copy and stops
// without writing its digest.
//
// What bounds it is the round (keccak_core.cuh); why one tile a block: the warp in
// a sub-partition's lowest slot issues first, so blocks with equal shares of the
// tiles finish one after the other and leave the last alone, with too few warps to
// fill the pipes, while blocks that take a tile at a time are replaced until the
// tiles run out.  2^24 messages: 3258 us with 912 blocks that share all tiles and
// load two ahead, 3173 with 16 tiles a block, 3164 with 4 and 3169 with 1; 119,040
// messages 41.3, 82.3, 41.2 and 35.5.
constexpr uint32_t kTileBytes = kThreads * 64;  // 8 KiB
constexpr uint64_t kWaitNs = 1000000000ull;     // 1 s

template <int V, class Rep>
__global__ void __launch_bounds__(kThreads, kStagedMinBlocks)
    k_sha3_uniform64_tma(const uint8_t *msgs, uint8_t *out, uint32_t out_len, uint64_t n,
                         unsigned int *status) {
    using P = Variant<V>;
    static_assert(64 < P::rate, "a 64-byte message is one block for every variant");
    constexpr int kOut = P::digest ? P::digest : P::rate;
    __shared__ __align__(128) uint8_t buf[kTileBytes];
    __shared__ __align__(8) uint64_t bar;
    const uint64_t first = uint64_t(blockIdx.x) * kThreads;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
        launch_wait();
        const uint32_t bytes = uint32_t(n - first < kThreads ? n - first : uint64_t(kThreads)) * 64;
        mbar_arrive_expect_tx(&bar, bytes);
        bulk_copy_g2s(buf, msgs + first * 64, bytes, &bar);
    }
    __syncthreads();
    launch_wait();
    if (!mbar_wait_bounded(&bar, 0, kWaitNs)) {
        atomicOr(status, KB_DEV_TIMEOUT);
        mbar_wait_bounded(&bar, 0, kWaitNs);  // the copy may still land: not into another block's memory
        return;
    }
    const uint64_t m = first + threadIdx.x;
    if (m >= n) return;
    uint32_t A[25], B[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) A[i] = B[i] = 0;
    const uint4 *q = reinterpret_cast<const uint4 *>(buf + threadIdx.x * 64);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint4 v = q[j];
        Rep::set_word(A[2 * j], B[2 * j], v.x, v.y);
        Rep::set_word(A[2 * j + 1], B[2 * j + 1], v.z, v.w);
    }
    A[8] ^= Rep::word_a(uint64_t(P::domain));
    B[8] ^= Rep::word_b(uint64_t(P::domain));
    constexpr uint64_t kEnd = uint64_t(0x80) << 56;
    A[P::rate / 8 - 1] ^= Rep::word_a(kEnd);
    B[P::rate / 8 - 1] ^= Rep::word_b(kEnd);
    const uint32_t dlen = P::digest ? uint32_t(P::digest) : out_len;
    uint8_t *dst = out + m * dlen;
    const uint32_t nsq = dlen > uint32_t(P::rate) ? (dlen - 1) / P::rate : 0;
    for (uint32_t i = 0; i <= nsq; ++i) {
        if (i > 0) squeeze<P::rate, Rep>(A, B, dst + uint64_t(i - 1) * P::rate, P::rate);
        Rep::template permute<true>(A, B);
    }
    squeeze<P::rate, Rep, kOut>(A, B, dst + uint64_t(nsq) * P::rate, dlen - nsq * P::rate);
}

template <int V, int LEN, bool A8, class Rep>
int launch_one(const uint8_t *msgs, uint64_t stride, uint64_t len, uint32_t out_len, uint8_t *digests,
               uint64_t n, cudaStream_t stream) {
    // A message per thread and as many blocks as that takes, so that the block
    // scheduler balances the sub-partitions' shares (k_sha3_uniform64_tma).  One-block
    // messages with (occupancy x SMs) blocks striding over them, against this: 2^22 of
    // 32 bytes 851 us -> 816, of 135 bytes 929 -> 841, of 64 at a stride of 80 903 -> 868.
    const uint64_t grid = std::min<uint64_t>((n + kThreads - 1) / kThreads, uint64_t(INT32_MAX));
    return cuda_status(launch_overlapped(k_sha3_uniform<V, LEN, A8, Rep>, unsigned(grid), kThreads, 0, stream, msgs,
                                         stride, len, digests, out_len, n));
}

template <int V>
int launch_tma(const uint8_t *msgs, uint32_t out_len, uint8_t *digests, uint64_t n, cudaStream_t stream,
               const DeviceInfo &dev) {
    const uint64_t grid = (n + kThreads - 1) / kThreads;  // device memory holds fewer than 2^31 tiles
    return cuda_status(launch_overlapped(k_sha3_uniform64_tma<V, PlainRep>, unsigned(grid), kThreads, 0, stream, msgs,
                                         digests, out_len, n, dev.d_status));
}

// True when p is device memory of this device (not host-mapped, not a peer's).
bool device_resident(const void *p, int device) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice && a.device == device;
}

template <int V>
int launch_variant(const uint8_t *msgs, uint64_t stride, uint64_t len, uint32_t out_len, uint8_t *digests,
                   uint64_t n, cudaStream_t stream, const DeviceInfo &dev) {
    const uintptr_t base = reinterpret_cast<uintptr_t>(msgs);
    const bool a16 = ((base | stride) & 15) == 0;
    const bool a8 = ((base | stride) & 7) == 0;
    if constexpr (V == 1) {
        // The bit-interleaved control, selected through the tuning interface.
        if (tuning_get(KB_TUNE_REPRESENTATION) == KB_REP_INTERLEAVED) {
            if (len == 64 && a16)
                return launch_one<V, 64, true, InterleavedRep>(msgs, stride, len, out_len, digests, n, stream);
            if (a8) return launch_one<V, -1, true, InterleavedRep>(msgs, stride, len, out_len, digests, n, stream);
        }
    }
    if (len == 64 && stride == 64 && a16 && tuning_get(KB_TUNE_STAGING) == KB_STAGING_TMA &&
        device_resident(msgs, dev.device))
        return launch_tma<V>(msgs, out_len, digests, n, stream, dev);
    if (len == 64 && a16) return launch_one<V, 64, true, PlainRep>(msgs, stride, len, out_len, digests, n, stream);
    constexpr int rate = Variant<V>::rate;
    if (len < uint64_t(rate) && (Variant<V>::digest || out_len <= uint32_t(rate))) {
        if (a8) return launch_one<V, -2, true, PlainRep>(msgs, stride, len, out_len, digests, n, stream);
        return launch_one<V, -2, false, PlainRep>(msgs, stride, len, out_len, digests, n, stream);
    }
    if (a8) return launch_one<V, -1, true, PlainRep>(msgs, stride, len, out_len, digests, n, stream);
    return launch_one<V, -1, false, PlainRep>(msgs, stride, len, out_len, digests, n, stream);
}

}  // namespace

int launch_uniform(const uint8_t *msgs, uint64_t stride, uint64_t len, int variant, uint32_t out_len,
                   uint8_t *digests, uint64_t n, cudaStream_t stream, const DeviceInfo &dev) {
    int rc = KB_OK;
    if (tuning_get(KB_TUNE_REPRESENTATION) == KB_REP_PLAIN &&
        launch_uniform_small(msgs, stride, len, variant, out_len, digests, n, stream, dev, &rc))
        return rc;
    switch (variant) {
        case 0: return launch_variant<0>(msgs, stride, len, out_len, digests, n, stream, dev);
        case 1: return launch_variant<1>(msgs, stride, len, out_len, digests, n, stream, dev);
        case 2: return launch_variant<2>(msgs, stride, len, out_len, digests, n, stream, dev);
        case 3: return launch_variant<3>(msgs, stride, len, out_len, digests, n, stream, dev);
        case 4: return launch_variant<4>(msgs, stride, len, out_len, digests, n, stream, dev);
        case 5: return launch_variant<5>(msgs, stride, len, out_len, digests, n, stream, dev);
        default: return KB_ERR_INVALID;
    }
}

}  // namespace kb
