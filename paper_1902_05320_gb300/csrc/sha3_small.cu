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
    k_sha3_uniform_coop(const uint8_t *__restrict__ msgs, uint64_t stride, uint64_t len, int variant,
                        uint8_t *__restrict__ out, uint32_t out_len) {
    __shared__ __align__(16) uint32_t mem[Coop::kWarpWords];
    const Coop c(mem);
    const uint64_t m = blockIdx.x;
    launch_wait();
    coop_sponge<-1, true>(c, msgs + m * stride, len, variant, out + m * out_len, out_len);
}

template <int V>
__global__ void __launch_bounds__(kThreads)
    k_sha3_uniform_pair(const uint8_t *__restrict__ msgs, uint64_t stride, uint64_t len, uint8_t *__restrict__ out,
                        uint32_t out_len, uint64_t n) {
    const uint64_t m = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 1;
    launch_wait();
    pair_sponge<Variant<V>::rate, Variant<V>::domain>(m < n, msgs + m * stride, len, out + m * out_len, out_len);
}

template <int V>
int launch_pair(const uint8_t *msgs, uint64_t stride, uint64_t len, uint32_t out_len, uint8_t *digests, uint64_t n,
                cudaStream_t stream) {
    const uint64_t per_block = kThreads / 2;
    return cuda_status(launch_overlapped(k_sha3_uniform_pair<V>, unsigned((n + per_block - 1) / per_block), kThreads, 0,
                                         stream, msgs, stride, len, digests, out_len, n));
}

}  // namespace

bool launch_uniform_small(const uint8_t *msgs, uint64_t stride, uint64_t len, int variant, uint32_t out_len,
                          uint8_t *digests, uint64_t n, cudaStream_t stream, const DeviceInfo &dev, int *rc) {
    const uint64_t sms = uint64_t(dev.sm_count > 0 ? dev.sm_count : 1);
    // A message of one permutation: a thread each folds round 0 and most of the
    // last, and beats two threads (6.1 against 6.5 us a launch).
    const uint32_t rate = uint32_t(variant_rate(variant));
    const bool one = len < rate && out_len <= rate;
    if (n <= (one ? kCoopOnePerSm : kCoopPerSm) * sms) {
        *rc = cuda_status(launch_overlapped(k_sha3_uniform_coop, unsigned(n), 32, 0, stream, msgs, stride, len, variant,
                                            digests, out_len));
        return true;
    }
    if (one || n > kPairPerSm * sms) return false;
    switch (variant) {
        case 0: *rc = launch_pair<0>(msgs, stride, len, out_len, digests, n, stream); return true;
        case 1: *rc = launch_pair<1>(msgs, stride, len, out_len, digests, n, stream); return true;
        case 2: *rc = launch_pair<2>(msgs, stride, len, out_len, digests, n, stream); return true;
        case 3: *rc = launch_pair<3>(msgs, stride, len, out_len, digests, n, stream); return true;
        case 4: *rc = launch_pair<4>(msgs, stride, len, out_len, digests, n, stream); return true;
        case 5: *rc = launch_pair<5>(msgs, stride, len, out_len, digests, n, stream); return true;
        default: return false;
    }
}

}  // namespace kb
