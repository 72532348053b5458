// queue_host.h -- host-side interface of the ragged-batch work queue
// (sha3_queue.cu): its configuration, its launch sequence on caller-owned
// scratch, and the autotuner.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "runtime.cuh"

namespace kb {

// One configuration of the queue schedule (the dimensions the autotuner
// searches).  stage is a kStage* value of queue.cuh.
struct QueueConfig {
    int minb = 2;               // register budget: blocks of 128 threads per SM compiled for
    int blocks_per_sm = 0;      // blocks per SM of the launch (0: as many as fit)
    int stage = 2 | 4;          // how message blocks are read: registers, looped permutation (kStageRegs | kLooped)
    int64_t warp_messages = 0;  // the K costliest messages run one warp each, unless auto_split
    bool auto_split = true;     // K from the batch's costs (plan_split)
    bool lanes = false;         // control: every message one warp
    bool per_variant = false;   // control: one launch per variant, unsorted
    float ms = 0;               // the autotuner's time for this configuration
};

// The fixed splits the autotuner tries on its best configuration beside the plan's
// own: one warp each for the 32 or the 608 (4 per SM on 152 SMs) costliest messages.
constexpr int64_t kHybridChoices[] = {32, 608};

// Warps per SM of the kernel that gives the costliest messages a warp each.  On
// 100,000 messages to 64 KiB: 3.5 ms at 4, 3.2 to 3.4 at 6, 2.8 at 8, 2.9 at 12.
constexpr uint64_t kLanesPerSm = 8;

// Messages per SM up to which a ragged batch takes the single launch of one warp
// per message, in input order.  Long messages of one length bound it: with every SM
// busy 1.4 to 1.6 ns a permutation, against 4.6 us in threads for any number up to 128
// per SM, cross at 18 to 21.  3,040 messages, us alone and by the queue: of 4 KiB 170
// and 167, of 64 KiB 2334 and 2136; of 64 bytes 10 and 34, of lengths log-uniform to
// 600 bytes 23 and 53, to 64 KiB 1545 and 1684.
constexpr uint64_t kRaggedCoopPerSm = 20;

// Device scratch of one call for n messages: the queue's control block, the
// digest offsets (8 B per message), the scan's tile sums and the work order
// (4 B per message).
size_t queue_scratch_bytes(uint64_t n);

// Whether the configuration names a compiled kernel.
bool queue_config_valid(const QueueConfig &cfg);

// Blocks of the hashing launch for n messages on a device of sm_count SMs
// (occupancy queried once per kernel and device).
uint64_t queue_grid_for(const QueueConfig &cfg, uint64_t n, int device, int sm_count);

// Enqueues the whole pipeline on `stream` using `scratch`
// (queue_scratch_bytes(n) bytes, 256-byte aligned): no allocation, no
// synchronisation.  status is the device status word per-message errors go
// to.
int queue_issue(const uint8_t *msgs, const uint64_t *offsets, const uint64_t *lens, const uint8_t *variants,
                const uint32_t *out_lens, uint8_t *digests, uint64_t n, uint8_t *scratch, const QueueConfig &cfg,
                uint64_t grid, int sm_count, unsigned int *status, cudaStream_t stream);

// Whether a batch of n messages takes the single launch of one warp per message:
// few enough messages, and no knob that asks for the queue.
bool ragged_small(uint64_t n, int sm_count);

// Enqueues that launch: no scratch, no allocation, no synchronisation.
int ragged_small_issue(const uint8_t *msgs, const uint64_t *offsets, const uint64_t *lens, const uint8_t *variants,
                       const uint32_t *out_lens, uint8_t *digests, uint64_t n, unsigned int *status,
                       int sm_count, cudaStream_t stream);

// keccak_batch's queue path: configuration from knobs, tuned entries and the
// cache file; graph capture and replay.
int launch_ragged_queue(const uint8_t *msgs, const uint64_t *offsets, const uint64_t *lens, const uint8_t *variants,
                        const uint32_t *out_lens, uint8_t *digests, uint64_t n, cudaStream_t stream,
                        const DeviceInfo &dev);

// The autotuner; writes the chosen configuration (with its time) to *chosen
// when not null.
int autotune_ragged_queue(const uint8_t *msgs, const uint64_t *offsets, const uint64_t *lens, const uint8_t *variants,
                          const uint32_t *out_lens, uint8_t *digests, uint64_t n, cudaStream_t stream,
                          const DeviceInfo &dev, QueueConfig *chosen);

// The tuning knobs applied over a configuration.
void apply_knobs(QueueConfig &cfg);

// The configuration keccak_batch would use for n messages on this device.
QueueConfig queue_config_for(uint64_t n, const DeviceInfo &dev);

// The KB_QUEUE_STAGING_* value of a configuration.
int queue_staging_value(const QueueConfig &cfg);

void release_queue_graphs(int device);
void forget_tuning(int device);
// keccak_batch_noalloc: forget the cached device address of its array.
void forget_noalloc_setup();

}  // namespace kb
