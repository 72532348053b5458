// sha3_small.cu -- fixed-stride batches too small to fill the GPU with a thread per
// message: the same messages with thirty or two threads each (coop.cuh, pair.cuh), so
// that the chain of permutations that a message is takes less time.
#include <cuda_runtime.h>

#include "coop_sponge.cuh"
#include "pair.cuh"
#include "runtime.cuh"

namespace kb {
namespace {

// One message per warp and one warp per block: the block scheduler then spreads
// the warps over the SMs first.  (Four warps to a block measured 1.79 us a
// permutation instead of 1.55: the warps of an SM share one path to its shared
// memory.)
__global__ void __launch_bounds__(32)
    k_sha3_uniform_coop(const uint8_t *msgs, uint64_t stride, uint64_t len, int variant,
                        uint8_t *out, uint32_t out_len, bool few) {
    __shared__ __align__(16) uint32_t mem[Coop::kWarpWords];
    const Coop c(mem);
    const uint64_t m = blockIdx.x;
    launch_wait();
    coop_sponge<-1, true>(c, msgs + m * stride, len, variant, out + m * out_len, out_len, few);
}

template <int V>
__global__ void __launch_bounds__(kThreads)
    k_sha3_uniform_pair(const uint8_t *msgs, uint64_t stride, uint64_t len, uint8_t *out,
                        uint32_t out_len, uint64_t n) {
    const uint64_t m = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 1;
    launch_wait();
    pair_sponge<Variant<V>::rate, Variant<V>::domain>(m < n, msgs + m * stride, len, out + m * out_len, out_len);
}

// The same for messages of one block, which need no loop over blocks and only the
// output's lanes of the last round.
template <int V>
__global__ void __launch_bounds__(kThreads)
    k_sha3_uniform_pair_one(const uint8_t *msgs, uint64_t stride, uint64_t len, uint8_t *out,
                            uint32_t out_len, uint64_t n) {
    using P = Variant<V>;
    const uint64_t m = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 1;
    launch_wait();
    launch_next();
    pair_one_block<P::rate, P::domain, P::digest ? (P::digest + 7) / 8 : P::rate / 8>(
        m < n, msgs + m * stride, uint32_t(len), out + m * out_len, out_len);
}

// A thread per message where that gives a sub-partition one warp or two: few warps
// do not hide each other's loads, so each thread's next block is loaded into
// registers before the permutation, which for a lone warp keeps to funnel shifts
// (keccak_core.cuh).
template <int V, bool MUL>
__global__ void __launch_bounds__(kThreads, 2)
    k_sha3_uniform_thin(const uint8_t *msgs, uint64_t stride, uint64_t len, uint8_t *out,
                        uint32_t out_len, uint64_t n) {
    using P = Variant<V>;
    constexpr int kWords = P::rate / 4;
    const uint64_t m = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    launch_wait();
    if (m >= n) return;
    const uint8_t *p = msgs + m * stride;
    const uint32_t dlen = P::digest ? uint32_t(P::digest) : out_len;
    uint8_t *dst = out + m * dlen;
    const uint64_t nfull = len / P::rate;
    const uint32_t nsq = dlen > uint32_t(P::rate) ? (dlen - 1) / P::rate : 0;
    const uint32_t sh = uint32_t(reinterpret_cast<uintptr_t>(p) & 3) * 8;  // the same for every block (rate % 4 == 0)
    uint32_t A[25], B[25], w[kWords + 1];
#pragma unroll
    for (int k = 0; k < 25; ++k) A[k] = B[k] = 0;
    auto fetch = [&](uint64_t i) {
        const uint32_t *a = reinterpret_cast<const uint32_t *>((reinterpret_cast<uintptr_t>(p) & ~uintptr_t(3)) +
                                                               i * P::rate);
#pragma unroll
        for (int k = 0; k < kWords; ++k) w[k] = a[k];
        w[kWords] = sh ? a[kWords] : 0u;
    };
    if (nfull) fetch(0);
    for (uint64_t i = 0; i <= nfull + nsq; ++i) {
        if (i < nfull) {
#pragma unroll
            for (int k = 0; k < P::rate / 8; ++k)
                PlainRep::xor_word(A[k], B[k], __funnelshift_r(w[2 * k], w[2 * k + 1], sh),
                                   __funnelshift_r(w[2 * k + 1], w[2 * k + 2], sh));
            if (i + 1 < nfull) fetch(i + 1);
        } else if (i == nfull) {
            absorb_last_same<P::rate, P::domain, false, PlainRep>(A, B, p + nfull * P::rate,
                                                                  uint32_t(len - nfull * P::rate));
        } else {
            squeeze<P::rate, PlainRep>(A, B, dst + (i - nfull - 1) * P::rate, P::rate);
        }
        keccak_f1600_plain<false, 24, 4, MUL>(A, B);
    }
    squeeze<P::rate, PlainRep>(A, B, dst + uint64_t(nsq) * P::rate, dlen - nsq * P::rate);
}

template <int V, bool MUL>
int launch_thin(const uint8_t *msgs, uint64_t stride, uint64_t len, uint32_t out_len, uint8_t *digests, uint64_t n,
                cudaStream_t stream) {
    return cuda_status(launch_overlapped(k_sha3_uniform_thin<V, MUL>, unsigned((n + kThreads - 1) / kThreads), kThreads, 0,
                                         stream, msgs, stride, len, digests, out_len, n));
}

template <int V>
int launch_pair(const uint8_t *msgs, uint64_t stride, uint64_t len, uint32_t out_len, uint8_t *digests, uint64_t n,
                cudaStream_t stream) {
    const uint64_t per_block = kThreads / 2;
    const bool one = len < uint64_t(Variant<V>::rate) && out_len <= uint32_t(Variant<V>::rate);
    return cuda_status(launch_overlapped(one ? k_sha3_uniform_pair_one<V> : k_sha3_uniform_pair<V>, unsigned((n + per_block - 1) / per_block), kThreads, 0,
                                         stream, msgs, stride, len, digests, out_len, n));
}

}  // namespace

bool launch_uniform_small(const uint8_t *msgs, uint64_t stride, uint64_t len, int variant, uint32_t out_len,
                          uint8_t *digests, uint64_t n, cudaStream_t stream, const DeviceInfo &dev, int *rc) {
    const uint64_t sms = uint64_t(dev.sm_count > 0 ? dev.sm_count : 1);
    const uint32_t rate = uint32_t(variant_rate(variant));
    const bool one = len < rate && out_len <= rate;
    if (n <= (one ? kCoopOnePerSm : kCoopPerSm) * sms) {
        *rc = cuda_status(launch_overlapped(k_sha3_uniform_coop, unsigned(n), 32, 0, stream, msgs, stride, len, variant,
                                            digests, out_len, few_warps(n, dev.sm_count)));
        return true;
    }
    // One-block messages: a thread each folds round 0 and most of the last, so two
    // threads gain less, and lose where their many 4-byte loads queue ahead of the
    // shuffles (4096 messages, us a call: 10 bytes 4.68 against 5.83, 64 bytes 5.04
    // against 5.64, 135 bytes 7.04 against 5.82).
    if (n > (one ? kPairPerSm : kThinPerSm) * sms || (one && len > 72)) return false;
    const bool pair = n <= kPairPerSm * sms, lone = n <= kThinPerSm / 2 * sms;
#define KB_FEW(V) \
    *rc = pair   ? launch_pair<V>(msgs, stride, len, out_len, digests, n, stream) \
          : lone ? launch_thin<V, false>(msgs, stride, len, out_len, digests, n, stream) \
                 : launch_thin<V, true>(msgs, stride, len, out_len, digests, n, stream); \
    return true
    switch (variant) {
        case 0: KB_FEW(0);
        case 1: KB_FEW(1);
        case 2: KB_FEW(2);
        case 3: KB_FEW(3);
        case 4: KB_FEW(4);
        case 5: KB_FEW(5);
        default: return false;
    }
#undef KB_FEW
}

}  // namespace kb
