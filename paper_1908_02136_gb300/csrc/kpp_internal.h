// kpp_internal.h -- declarations shared by the host-side translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kpp_device.cuh"

namespace kpp {

// One streamed-form specialisation chosen for (dtype, d, lanes).
struct StreamedKernel {
    const void *fn;
    int rows_align; // per-CTA row ranges are multiples of this
    int lanes;      // lanes per row (0 for the generic kernel)
    bool generic;
};

bool streamed_lookup(int dt, int d, int lanes, StreamedKernel *out);
int streamed_threads();
int streamed_segments();
size_t streamed_smem(const StreamedKernel &k, int d);
cudaError_t streamed_launch(const StreamedKernel &k, int grid, const Problem &p, int m,
                            cudaStream_t stream);
// Point-sharded seeding (kpp_shard_*): first seed, draw after a pass, phi.
cudaError_t shard_first_launch(const Problem &p, int64_t row0, long long *xchg, int eb,
                               cudaStream_t stream);
cudaError_t shard_pick_launch(const Problem &p, int m, int rank, int world, const float *totals,
                              int64_t row0, long long *xchg, int eb, cudaStream_t stream);
cudaError_t shard_phi_launch(const float *totals, int world, double *phi, cudaStream_t stream);

// Small form (kpp_small.cu): one CTA, everything in shared memory.
const void *small_lookup(int dt, int d);
int small_threads();
size_t small_smem(int64_t N, int d, int dt);
cudaError_t small_launch(const void *fn, size_t smem, const Problem &p, cudaStream_t stream);

// Runtime arguments of the persistent kernel.
struct PersistArgs {
    int64_t cache_supers; // super-iterations of each warp's segment kept in smem
    int32_t reverse;     // walk rows backwards on odd passes
    int32_t l2_hint;     // global point loads: 0 none, 1 evict_last, 2 evict_first
    uint64_t timeout_ns; // bound of every grid-barrier wait
};

struct PersistentKernel {
    const void *fn_smem;   // D^2 in shared memory
    const void *fn_global; // D^2 in the output array
    const void *prune_smem;   // the same with passes that skip rows, or null
    const void *prune_global;
    int rows_align;          // rows per super-iteration; blocks are multiples of it
    int row_bytes;
    int lanes;
};

// any_d: the kernel for every d (no fn_smem / fn_global) where d has no
// specialisation.
bool persistent_lookup(int dt, int d, int lanes, bool any_d, PersistentKernel *out);
int persistent_threads();
int persistent_max_blocks();
int persistent_segments();
cudaError_t persistent_launch(const void *fn, int grid, size_t smem, const Problem &p,
                              const PersistArgs &a, cudaStream_t stream);

// The options the autotuner (kpp_tune) recorded for this shape on the
// current device, if `asked` leaves every knob to the automatic choice.
bool tuned_options(int64_t N, int32_t d, int32_t K, int dt, const kpp_options &asked,
                   kpp_options *out);

// For the autotuner: what kpp_seed does under these options, given the room,
// and the first `passes` passes of that seeding (the plan is the one for K).
struct PlanFacts {
    kpp_plan plan;
    bool skips;    // its passes skip rows (kpp_pass.cuh)
    size_t bytes;  // workspace it needs to run as planned
};
kpp_status plan_facts(int64_t N, int32_t d, int32_t K, kpp_dtype dtype, const kpp_options *opts,
                      PlanFacts *out);
kpp_status seed_passes(const void *points, const float *row_scales, int64_t N, int32_t d,
                       int32_t K, int32_t passes, kpp_dtype dtype, uint64_t seed,
                       uint64_t stream_id, const int64_t *forced_prefix, int32_t n_forced,
                       int64_t *indices_out, float *d2_out, double *phi_out, void *workspace,
                       size_t workspace_bytes, kpp_stream_t stream, const kpp_options *opts);

} // namespace kpp

namespace kpp {

// kpp_lloyd_assign for centres whose first row and count are known only on
// the device: rows [*row0, *row0 + *kdev) of `centres` (*kdev <= kmax; 0 is
// a no-op), for points prepared by kpp_lloyd_prepare(..., kmax, ...).
kpp_status lloyd_assign_device_count(const float *centres, const long long *row0,
                                     const int32_t *kdev, int32_t kmax, int64_t N, int32_t d,
                                     int32_t *labels_out, void *workspace, size_t workspace_bytes,
                                     cudaStream_t stream);

// Workspace of kpp_lloyd_prepare and the assignments alone (0 if invalid).
size_t lloyd_assign_workspace(int64_t N, int32_t d, int32_t K);

cudaError_t quantize_bf16(const float *x, int64_t n, uint16_t *out, cudaStream_t stream);
cudaError_t quantize_fp8(const float *x, int64_t N, int d, uint8_t *q, float *scales,
                         cudaStream_t stream);

} // namespace kpp
