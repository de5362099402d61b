// creutz_queue.cuh -- per-warp shared-memory queues of the Creutz phase
// kernels (single lattice and batches): links whose first two trials were
// rejected wait for further Philox blocks; links with an accepted trial wait
// for their a0 (deferred_a0), direction and store, 32 at a time.
#pragma once

#include <cuda_runtime.h>

namespace su2 {

// Both queues share one array: the direction queue grows from its start, the
// retry queue from kCrRetryTop down.  A push finds at most 31 entries in each
// and adds at most 32 in all, so 94 hold them; lanes that push nothing write to
// entry kCrNobody, which nobody reads, so the stores need no branch.
constexpr int kCrRetryTop = 93;
constexpr int kCrNobody = 94;
constexpr int kCrEntries = 95;

struct CrQueues {
    float4 ut[kCrEntries];  // U~^dag
    float ibk[kCrEntries];  // 1/(beta k) (0 on the Haar branch); beta k for Kennedy-Pendleton
    float x[kCrEntries];    // waiting for a trial: exp(-2 beta k); accepted: x of the trial (a0 on the Haar branch)
    int eo[kCrEntries], blk[kCrEntries];  // index, next Philox block
    // when the phase measures the plaquette: the staple terms of the directions nu < mu
    float4 sp[kCrEntries];
};

}  // namespace su2
