// runtime.cuh -- host-side runtime shared by the library's translation units:
// per-device state (SM count, the device status word), per-stream scratch
// arenas, and the launch helpers.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <cstddef>
#include <cstdint>

#include "../../include/sha3gb.h"

namespace kb {

// NVTX range for the host side of an entry point (visible in Nsight tools;
// free when no tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Threads per block of the thread-per-message kernels.
constexpr int kThreads = 128;
// Minimum resident blocks per SM asked of ptxas for the sponge kernels: caps
// them at 128 registers per thread (16 warps per SM).
constexpr int kMinBlocks = 4;

struct DeviceInfo {
    int device = -1;
    int sm_count = 0;
    unsigned int *d_status = nullptr;  // device status word (KB_DEV_* bits)
};

// State of the calling thread's current device, created on first use.
// Returns nullptr (and sets *err) when the CUDA runtime fails.
DeviceInfo *device_info(int *err);

// A scratch arena cached per (device, stream): returns at least `bytes` of
// device memory reserved for work enqueued on `stream`.  Growing the arena
// synchronises the stream before the old block is freed.
void *stream_scratch(cudaStream_t stream, size_t bytes, int *err);

// Frees all cached state of the current device.
void release_device();

// Blocks of `threads` that keep every SM busy for kernel `fn` (occupancy x SMs),
// capped by the number of blocks the work needs.
uint64_t persistent_grid(const void *fn, int threads, size_t smem, uint64_t work_items,
                         const DeviceInfo &dev);

// The status of a runtime call.  Its error is cleared with it: the caller hears of it
// here, and the thread's last error would be taken for that of a later plain launch.
inline int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return KB_OK;
    cudaGetLastError();
    return KB_ERR_CUDA;
}

// A launch that may be set up while the kernel before it in the stream still runs
// (programmatic dependent launch).  The kernel calls launch_wait() before it
// touches memory, so what it reads and writes is ordered as by a plain launch;
// only the launch itself and the kernel's own set-up leave the critical path.
// Back to back in one stream a plain launch costs about 2 us between two kernels.
template <class... P, class... A>
cudaError_t launch_overlapped(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                              A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // as cuda_status
    return e;
}

#ifdef __CUDACC__
// Lets the next kernel of the stream be set up from here on (it waits for this
// one to end before it touches memory, when it is launched to overlap at all);
// without it that happens as this kernel's blocks exit.  Not for kernels whose
// blocks need an SM, or a share of one, to themselves: the next kernel's blocks are
// placed while this one's still stand, several to an SM where others are free (89
// blocks of 128 threads, call after call: 45 us each became 137).
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Returns when every earlier kernel of the stream has ended and its writes are
// visible; at once in a plain launch.  Only plain loads stay behind it: no kernel that
// calls it has __restrict__ parameters or read-only loads.
__device__ __forceinline__ void launch_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

// Process-wide tuning knobs (kb_tune_key values of sha3gb.h).
int64_t tuning_get(int key);
int tuning_set(int key, int64_t value);

// Whether a launch of `blocks` one-warp blocks is small enough (four to an SM) for the
// next kernel of the stream to be set up as soon as these have started (coop_sponge).
inline bool few_warps(uint64_t blocks, int sm_count) { return blocks <= 4 * uint64_t(sm_count > 0 ? sm_count : 1); }

// Launchers (one per translation unit of kernels).
int launch_uniform(const uint8_t *msgs, uint64_t stride, uint64_t len, int variant, uint32_t out_len,
                   uint8_t *digests, uint64_t n, cudaStream_t stream, const DeviceInfo &dev);
// Fixed-stride batches of up to kThinPerSm messages per SM (sha3_small.cu): true when
// one of its kernels took the batch (*rc is the launch's status).
//
// The lines between the forms, in messages per SM, from us a permutation on a
// GB300 of 152 SMs: thirty threads a message 1.55 at 0.4, 1.80 at 8 and 2.58 at
// 12; two threads 2.82 up to 64 (one warp per sub-partition) and 4.97 beyond; a
// thread each 4.5 up to 128 (the same).  Up to 256 the kernel that loads the next
// block ahead (k_sha3_uniform_thin) beats the general one: 23,907 bytes a message,
// 17,800 messages 754 us against 966, 38,912 1384 against 1535; beyond, with three
// warps a sub-partition, it does not (1000 bytes: 102 us either way).
constexpr uint64_t kCoopOnePerSm = 8, kCoopPerSm = 12, kPairPerSm = 64, kThinPerSm = 256;
bool launch_uniform_small(const uint8_t *msgs, uint64_t stride, uint64_t len, int variant, uint32_t out_len,
                          uint8_t *digests, uint64_t n, cudaStream_t stream, const DeviceInfo &dev, int *rc);
int launch_ragged(const uint8_t *msgs, const uint64_t *offsets, const uint64_t *lens, const uint8_t *variants,
                  const uint32_t *out_lens, uint8_t *digests, uint64_t n, cudaStream_t stream,
                  const DeviceInfo &dev);
uint64_t digest_offsets_tiles(uint64_t n);
int launch_digest_offsets(const uint32_t *out_lens, uint64_t n, uint64_t *out_off, uint64_t *tile_sums,
                          cudaStream_t stream);
// Streaming states (stream.cu).
int launch_stream_init(uint8_t *states, const uint8_t *variants, uint64_t n, cudaStream_t stream,
                       const DeviceInfo &dev);
int launch_stream_absorb(uint8_t *states, const uint8_t *msgs, const uint64_t *offsets, const uint64_t *lens,
                         uint64_t n, cudaStream_t stream, const DeviceInfo &dev);
int launch_stream_final(uint8_t *states, const uint32_t *out_lens, uint8_t *digests, uint64_t n,
                        cudaStream_t stream, const DeviceInfo &dev);
// One fused step: optionally start from fresh states (init, variants read),
// absorb a piece (msgs may be null for none), optionally pad and squeeze
// (final_, outputs at the exclusive scan of out_lens).
int launch_stream_step(bool init, bool final_, uint8_t *states, const uint8_t *variants, const uint8_t *msgs,
                       const uint64_t *offsets, const uint64_t *lens, const uint32_t *out_lens, uint8_t *digests,
                       uint64_t n, cudaStream_t stream, const DeviceInfo &dev);
// The cost-bucketed persistent path is declared in queue_host.h.
uint64_t merkle_nodes(uint64_t n_leaves);
int launch_merkle_levels(const uint8_t *buf, uint64_t n_leaves, uint64_t leaf_bytes, uint8_t *nodes,
                         cudaStream_t stream, const DeviceInfo &dev);
uint64_t merkle_message_leaves(uint64_t len, uint64_t chunk_bytes);
int launch_keccak_p(uint64_t *states, int b, int nr, uint64_t n, cudaStream_t stream, const DeviceInfo &dev);
int launch_merkle_many(const uint8_t *buf, uint64_t n_trees, uint64_t leaves_per_tree, uint64_t leaf_bytes,
                       uint8_t *roots, cudaStream_t stream, const DeviceInfo &dev);
int launch_merkle_message(const uint8_t *msg, uint64_t len, uint64_t chunk_bytes, uint8_t *nodes,
                          cudaStream_t stream, const DeviceInfo &dev);

}  // namespace kb
