// batch.cuh -- in-place batch edit of the device graph (Sec. 3.2).
#pragma once
#include "graph.cuh"

namespace dfpr {

// endpoint arrays are device pointers in user ids; validated unless `validated`
int apply_batch_device(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is,
                       const int32_t* id, int64_t ni, bool validated);

// the same in two phases, so that the batches of many graphs are queued before
// the host waits for any: a small batch (at most 16384 edges) is queued by
// apply_batch_launch and finished by apply_batch_complete (which waits for the
// graph's stream); a larger one is applied whole by apply_batch_launch.
struct EditStatus;
struct EditBufs;
struct SmallApply {
  EditBufs* B = nullptr;   // set while a small batch is pending
  int32_t* S[2] = {nullptr, nullptr};
};
// a host batch's endpoint arrays where the device can read them (up to 16384
// edges the graph's pinned host memory, else device scratch, the copy queued on
// the graph's stream): *out holds nd deletion sources, nd targets, ni insertion
// sources, ni targets
int stage_host_batch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is, const int32_t* id,
                     int64_t ni, int32_t** out);
int apply_batch_launch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is,
                       const int32_t* id, int64_t ni, bool validated, SmallApply* pending);
int apply_batch_complete(Graph* g, SmallApply* pending);

}  // namespace dfpr
