// fmb_ac_walk.cuh -- host interface of the thread-per-ray alpha-compositing forward
// (fmb_ac_walk.cu).
#pragma once

#include "fmb_internal.cuh"

namespace fmb {

// Columns of ac_walk_run pixels, one per thread, for batches of whole images; 0 if the
// batch (its rays, launches, largest K and shortest focal length) is not for this kernel.
// Work items of ac_walk_threads() columns.
int ac_walk_threads();
int ac_walk_run(long long total_rays, int launches, int maxK, float min_f, int sms);
cudaError_t launch_forward_ac_walk(const Batch& b, const Scene& s, const Consts& c, const float4* records, bool normals,
                                   int n_flow, int maxK, const FwdOut& o, int run, int* counter, cudaStream_t st);

}  // namespace fmb
