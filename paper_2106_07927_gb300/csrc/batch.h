// Batch engine: many pairs of uneven W, H, D in persistent kernels fed by device work queues.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "batch_dev.cuh"
#include "common.cuh"

namespace r2t {

// Most bytes the batch scratch takes beyond the sums' layout for path planes: with none, a batch whose
// planes do not fit runs a few pairs at a time, and small pairs then wait for one another's chains
// (5 x 160x120, D = 32, P2 = 200: 193 us, 53 with room for all; the persistent kernels 97). Small
// batches fit; larger ones fill the GPU a few pairs at a time (with 512 MB: 8 x 640x480, D = 32, P2 =
// 200 571 -> 425 us, 8 x 320x240, D = 128 367 -> 335, the others within 5 %).
constexpr size_t kBatchExtra = (size_t)256 << 20;

struct BatchEngine;

// Device bytes of the descriptor tables for n pairs (upper bound, excluding per-pair scratch).
size_t batch_fixed_bytes(int n);

// Creates or grows the engine so it holds `need` bytes of per-pair scratch and n pairs. The scratch is
// allocated anew only when it is smaller than need, and then takes `want` bytes (what path planes can
// use) where half of the device's memory stays free with them: a batch that ran once never moves
// it again, whatever memory has become free since, so captured batches keep their addresses until a
// larger batch arrives. planar: the method's route (batch_planar_method), for the default settings.
// Returns 0, -2 when device memory is short, -3 on another CUDA error.
int batch_reserve(BatchEngine** e, size_t need, size_t want, int n, bool planar);

// Device bytes the engine holds (0 without one).
size_t batch_bytes(const BatchEngine* e);

// Base of the per-pair scratch (valid after batch_reserve).
char* batch_scratch(BatchEngine* e);

// Runs the batch on stream s: uploads the descriptors, clears the queue counters and replays
// the captured graph (capturing it first when the capacities changed). Returns 0 or -3.
int batch_run(BatchEngine* e, const Problem* probs, int n, const Method& mt, cudaStream_t s,
              int* launches);

// The route of batches whose method has path planes (batch_planar_method): groups of pairs of one D
// run stage by stage on up to 4 streams, each stream's groups in one part of the scratch after
// another. Uses the engine's scratch as it is; a pair whose planes do not fit it runs with its sums
// in place. Returns 0 or -3.
bool batch_planar_method(const Method& mt);
int batch_run_planar(BatchEngine* e, const Problem* probs, int n, const Method& mt, cudaStream_t s,
                     int* launches);

// Kernel settings per bucket of pairs (tune_bucket: D / 16 and the size class): the defaults,
// their validity, and the engine's table (set returns -1 for an invalid setting).
BatchTune batch_default_tune(int bucket, bool planar);
// The settings t stands for in a batch of that many rows in all: itself, or, for a default on path
// planes, what such a batch runs, as an explicit setting.
BatchTune batch_resolved_tune(int bucket, const BatchTune& t, bool planar, int64_t rows);
// True when the two settings run the same kernels (on path planes the sheared settings have no effect
// and the selection's tile is capped).
bool batch_tune_same(int bucket, const BatchTune& a, const BatchTune& b, bool planar);
bool batch_tune_valid(int bucket, const BatchTune& t);
int batch_set_tune(BatchEngine* e, int bucket, const BatchTune& t);
BatchTune batch_get_tune(BatchEngine* e, int bucket, bool planar);

const char* batch_error(BatchEngine* e);
void batch_destroy(BatchEngine* e);

}  // namespace r2t
