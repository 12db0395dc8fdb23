// The small-frontier phase of gbx_bfs (bfs_cluster.cu) and what it hands over to the
// grid-wide kernel (bfs.cu).
#pragma once

#include "gbx_internal.cuh"

namespace gbx {

// Whether a search on G with descriptor d starts in the cluster kernel.
gbx_status cluster_bfs_wanted(Graph* G, const gbx_desc& d, bool* wanted);

// Initialises the outputs and runs levels until the search ends or its frontier outgrows the
// cluster; *complete: it always ends there.  Otherwise the grid-wide kernel has to follow on
// the same stream with ws.handoff.
gbx_status cluster_bfs_launch(Graph* G, int32_t source, int32_t* depth, int32_t* parent, cudaStream_t s,
                              bool* complete);

// One launch in which a block withholds its queue length: every block's wait runs out after
// timeout_ns.
gbx_status cluster_bfs_selftest(Graph* G, uint64_t timeout_ns, cudaStream_t s);

// out[i] = fill for all i < n except out[special] = special_value; 16-byte stores when aligned.
__device__ __forceinline__ void fill_i32(int32_t* out, int32_t n, int32_t fill, int32_t special, int32_t special_value,
                                         long long gtid, long long gstride) {
    if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
        const long long n4 = n >> 2;
        int4* o4 = reinterpret_cast<int4*>(out);
        for (long long q = gtid; q < n4; q += gstride) {
            int4 v = make_int4(fill, fill, fill, fill);
            const long long b = q << 2;
            if (special >= b && special < b + 4) {
                const int r = (int)(special - b);
                if (r == 0) v.x = special_value;
                if (r == 1) v.y = special_value;
                if (r == 2) v.z = special_value;
                if (r == 3) v.w = special_value;
            }
            o4[q] = v;
        }
        for (long long i = (n4 << 2) + gtid; i < n; i += gstride) out[i] = i == special ? special_value : fill;
    } else {
        for (long long i = gtid; i < n; i += gstride) out[i] = i == special ? special_value : fill;
    }
}

}  // namespace gbx
