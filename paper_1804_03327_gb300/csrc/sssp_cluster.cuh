// gbx_sssp on meshes (sssp_cluster.cu) and its hand-over to the grid-wide kernel (sssp.cu).
#pragma once

#include "gbx_internal.cuh"

namespace gbx {

// After the weights are set: the records the cluster kernel reads, and the step of its
// threshold (G->sp_step, negative where the kernel does not apply).  Synchronises s.
gbx_status sssp_cluster_prepare(Graph* G, cudaStream_t s);
gbx_status sssp_cluster_wanted(Graph* G, const gbx_desc& d, bool* wanted);
// Initialises dist and relaxes until it is done or hands over (ws.handoff->done): the
// grid-wide kernel has to follow on the same stream.
gbx_status sssp_cluster_launch(Graph* G, int32_t source, float* dist, cudaStream_t s);
// One launch in which a block withholds its counts: every block's wait runs out after timeout_ns.
gbx_status sssp_cluster_selftest(Graph* G, uint64_t timeout_ns, cudaStream_t s);

}  // namespace gbx
