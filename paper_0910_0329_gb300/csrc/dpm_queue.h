// dpm_queue.h -- persistent transport kernel with device-wide particle queues.
#pragma once

#include <cuda_runtime.h>

#include <string>

#include "dpm_internal.h"

namespace dpm {

struct QueueState {
  void *mem = nullptr;     // one device allocation holding queues and control words
  size_t bytes = 0;
  int K = 0, log2_cap = 0;  // the layout in `mem` (K = 0: none yet), in order between launches
  int per_sm = 0;           // resident blocks per SM of the queue kernels on the context's device
  uint64_t budget = 0;          // the owning context's device-memory budget (0 = none)
  uint64_t *in_use = nullptr;   // the owning context's bytes in use (the queues' included)
};

// Launch the persistent kernel for one run; returns a dpm_status code.
// `start` (may be NULL) is recorded on the stream just before the transport kernel.
int queue_run(QueueState &q, const RunParams &R, uint64_t batch_size, const dpm_run_opts &o, int sm_count,
              cudaStream_t st, cudaEvent_t start, std::string &err);
void queue_free(QueueState &q);

// Launch shape for the options (K shards = blocks, laid out with 2^log2cs slots
// each, of which the launch uses 2^log2use), the context's queue memory
// allocated for it and, if the layout is a new one, the queues made ready on the
// stream (never while it is being captured: what is captured relies on the layout).
int queue_prepare(QueueState &q, const dpm_run_opts &o, int sm_count, cudaStream_t st, int &K, int &log2cs, int &log2use,
                  std::string &err);

// Jobs one shared (batch) launch of the queue kernel takes: their step
// records are kept in shared memory.
constexpr int kSharedJobs = 64;

// A launch pauses refills that found nothing (dpm_run_opts.refill_pause = 0)
// with shards of at least 2^kPauseMinLog2 slots: small queues (the
// no-allocation entry point's, or a small queue_log2) need every refill to keep
// the producers' shards from overflowing.
constexpr int kPauseMinLog2 = 13;

// Resident blocks per SM of the queue kernel (occupancy query), or 0 on error.
int queue_blocks_per_sm();
// Load the queue kernels on the current device now (they are otherwise
// loaded at their first launch under lazy module loading); returns
// queue_blocks_per_sm(), or 0 on error.
int queue_preload();
// Device bytes the queues of K shards of 2^log2cs slots occupy.
size_t queue_bytes(int K, int log2cs);
// Make the queues of a fresh layout ready: K shards of 2^log2cs slots in `mem`
// (at least queue_bytes(K, log2cs) bytes of device memory, any alignment).
int queue_fresh(void *mem, int K, int log2cs, int sm_count, cudaStream_t st, std::string &err);
// Launch on queues that are ready, using 2^log2use slots of each shard: allocates
// nothing, and leaves the queues ready for the next launch.
int queue_launch(void *mem, int K, int log2cs, int log2use, const RunParams &R, uint64_t batch_size,
                 const dpm_run_opts &o, cudaStream_t st, cudaEvent_t start, std::string &err);

}  // namespace dpm
