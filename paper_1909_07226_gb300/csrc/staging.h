// Hand-over of staged batches between one loader and several readers through two buffers.
//
// Batch b sits in buffer staging_buffer(b).  Batch 0 is staged by the readers themselves; for
// every later batch the loader waits until the readers have left the batch before it in the
// same buffer, fills the buffer and arrives on the buffer's "full" barrier, on which every
// reader waits; every reader arrives on the buffer's "free" barrier when it has left a batch.
// Barriers are waited for by the parity of their phase, so no barrier may complete two phases
// between two waits of one thread.  With a pair of barriers per buffer none can: the next phase
// of a "full" barrier follows a wait of the loader on the buffer's "free" barrier, to which
// every reader has arrived after its own wait, and the other way round.  (One pair for both
// buffers could run two phases ahead of a late thread, which would then wait for ever.)
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define IDG_HD __host__ __device__
#else
#define IDG_HD
#endif

namespace idg {

constexpr int kStagingBuffers = 2;
constexpr int kStagingBarriers = kStagingBuffers;      // of each kind

// the buffer of batch b, and the barrier (of either kind) of batch b
IDG_HD constexpr int staging_buffer(int b) { return b & 1; }
IDG_HD constexpr int staging_barrier(int b) { return b & 1; }
// parity a reader waits for before it reads batch b >= 1 (batches 1, 3, 5 .. and 2, 4, 6 .. are
// the phases 0, 1, 2 .. of their barriers)
IDG_HD constexpr uint32_t staging_full_parity(int b) { return (uint32_t)(((b - 1) >> 1) & 1); }
// parity the loader waits for before it fills batch b >= 2: batch b - 2 was left
IDG_HD constexpr uint32_t staging_free_parity(int b) { return (uint32_t)(((b - 2) >> 1) & 1); }

}  // namespace idg
