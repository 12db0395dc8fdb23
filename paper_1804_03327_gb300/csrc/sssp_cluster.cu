// gbx_sssp on meshes with non-negative weights: one thread-block cluster that relaxes near
// vertices first, instead of the whole grid's Bellman-Ford iterations (sssp.cu).
//
// On a road-like graph Bellman-Ford runs as many iterations as the longest shortest path has
// edges, and each vertex improves many times on the way: 1001 x 777 vertices with real lengths
// take 1,346 iterations of 25K improved vertices, 43 relaxations of every vertex.  Here the
// improved vertices at most T away from the source go on at once (the near queue) and the
// others wait (the far pile); when no near vertex is left, T moves to the nearest far one plus
// a step.  Vertices then improve about twice, the frontier stays as long as the wavefront (a
// few thousand vertices), and it lives in the cluster's shared memory like that of the BFS
// (bfs_cluster.cu).  This is the near-far form of delta-stepping (Davidson, Baxter, Garland
// and Owens 2014; Meyer and Sanders 2003).
//
// Any order of relaxations ends in the same distances: with non-negative weights each vertex's
// smallest left-to-right rounded path sum, because binary32 addition is monotonic and every
// decrease of a distance is followed by a relaxation of the vertex's edges from it (or a
// smaller one).
//
// A phase is bound by two dependent round trips (the vertex's record and distance, the atomic
// minima of its neighbours) and the exchange of the queue lengths.  1001 x 777
// grid: 25.4-26.2 -> 3.6-3.7 ms.  With a fixed step of 2, 4, 8 and 16 mean weights: 4.8, 3.9, 3.6 and
// 3.5 ms there; a 200 x 200 grid 1.04, 0.85, 0.74 and 0.66 ms, with the moving step 0.63.
#include <algorithm>

#include "cluster.cuh"
#include "sssp_cluster.cuh"

namespace gbx {

constexpr int kSpThreads = 512;
constexpr int kSpLanes = 4;                         // lanes per vertex, one neighbour of its record each
constexpr int kSpPerRound = kSpThreads / kSpLanes;  // vertices a block takes at a time
constexpr int kSpCap = 6144;                        // near queue entries a block holds
// The near queue at which the grid takes over: the edges of that many average rows, at most
// kSpMaxNear vertices.  A phase of the cluster takes its edges' time on 16 SMs, the hand-over pulls
// every row.  With 32,768 vertices as the only limit the random 16-regular graph of 30,000 vertices took
// 170 us (the grid alone 127, now 118); with 128K edges and no share of the entries the 8-regular
// one of 2M 738 (688, 689), and the 126 x 126 x 126 grid 10.1 ms (13.0, 5.6): it was handed over at its
// widest.  16K and 32K edges take 2-D grids off the cluster too early (777K vertices 21.5 ms, not 3.7).
constexpr int32_t kSpMaxNear = 32768;
constexpr int64_t kSpMaxEdges = 96 * 1024;
constexpr int64_t kSpMaxShare = 80;  // ... and this fraction of the stored entries
// T first moves on by this many mean weights; the step is doubled while the near queue keeps
// below kSpFew vertices from one move to the next (a phase then has idle lanes, and moves cost
// phases of their own) and halved when it exceeds kSpMany (vertices would improve too often).
constexpr float kSpStep = 8.0f;
constexpr int32_t kSpFew = 1024;
constexpr int32_t kSpMany = 4096;

struct SpArgs {
    int32_t n, source;
    const int32_t* ptr;
    const int32_t* col;
    const float* val;
    const int4* rcol;
    const float4* rval;
    float* dist;
    int32_t* farv[2];  // far piles: vertices ...
    float* fard[2];    // ... and the distance each was put there with; block r's part is [r seg, r seg + seg)
    int32_t seg, max_near;
    float step;
    ClHandoff* ho;
    int32_t* status;
    unsigned long long timeout_ns;
};

// What each block tells the others after a phase.
enum { SP_NEAR = 0, SP_FAR = 1, SP_MIN = 2, SP_WORDS = 3 };

struct SpSmem {
    int2 q[2][kSpCap];  // near vertices and the distance each was put there with (bits)
    unsigned long long bar[2];
    int32_t told[2][SP_WORDS][kClusterMax];
    int32_t cnt[2];    // entries in q[.] (may count past kSpCap: those went to the far pile)
    int32_t fcnt[2];   // entries in the far piles
    uint32_t fmin;     // smallest distance in the current far pile (bits)
    int32_t lost;      // a far entry found no room
    int32_t abort;
};

__global__ void __launch_bounds__(512) sp_fill_kernel(float* dist, int32_t n, int32_t source) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dist[i] = i == source ? 0.0f : INFINITY;
}

// Adds the lanes with `take` to the far pile f of this block.
__device__ __forceinline__ void sp_far(const SpArgs& a, SpSmem& sm, int f, int32_t base, bool take, int32_t v, float d) {
    const uint32_t m = __ballot_sync(0xffffffffu, take);
    if (!m) return;
    int32_t pos = 0;
    if ((threadIdx.x & 31) == 0) pos = atomicAdd(&sm.fcnt[f], __popc(m));
    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m & lanemask_lt());
    const uint32_t least = __reduce_min_sync(0xffffffffu, take ? __float_as_uint(d) : 0xffffffffu);
    if ((threadIdx.x & 31) == 0) atomicMin(&sm.fmin, least);
    if (!take) return;
    if (pos < a.seg) {
        a.farv[f][base + pos] = v;
        a.fard[f][base + pos] = d;
    } else {
        sm.lost = 1;
    }
}

// Adds the lanes with `take` to the near queue np, or to the far pile where that is full.
__device__ __forceinline__ void sp_near(const SpArgs& a, SpSmem& sm, int np, int f, int32_t base, bool take, int32_t v,
                                        float d) {
    const uint32_t m = __ballot_sync(0xffffffffu, take);
    if (!m) return;
    int32_t pos = 0;
    if ((threadIdx.x & 31) == 0) pos = atomicAdd(&sm.cnt[np], __popc(m));
    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m & lanemask_lt());
    const bool fits = pos < kSpCap;
    if (take && fits) sm.q[np][pos] = make_int2(v, __float_as_int(d));
    if (__any_sync(0xffffffffu, take && !fits)) sp_far(a, sm, f, base, take && !fits, v, d);
}

// Lowers the distance of v to d (take: whether the lane has one) and queues v if that did.
__device__ __forceinline__ void sp_relax(const SpArgs& a, SpSmem& sm, int np, int f, int32_t base, bool take, int32_t v,
                                         float d, float T) {
    // non-negative binary32 values order like their bits
    const bool lowered =
        take && d < __int_as_float(atomicMin(reinterpret_cast<int*>(a.dist + v), __float_as_int(d)));
    sp_near(a, sm, np, f, base, lowered && d <= T, v, d);
    sp_far(a, sm, f, base, lowered && !(d <= T), v, d);
}

// kWithhold: block 1 keeps its counts to itself, so that every block's wait runs out.
template <bool kWithhold>
__global__ void __launch_bounds__(kSpThreads, 1) sssp_cluster_kernel(const __grid_constant__ SpArgs a) {
    extern __shared__ __align__(16) unsigned char raw[];
    SpSmem& sm = *reinterpret_cast<SpSmem*>(raw);
    const int t = threadIdx.x, lane = t & 31, j = t & (kSpLanes - 1);
    const int rank = (int)cluster_rank(), C = (int)cluster_size();
    const int shift = 31 - __clz(C);
    const int32_t base = rank * a.seg;
    const int pending = t == 0 ? ld_volatile_i32(a.status + ST_ERROR) : 0;
    if (__syncthreads_or(pending)) {
        if (rank == 0 && t == 0) a.ho->done = 1;
        return;
    }
    if (t == 0) {
        sm.q[0][0] = make_int2(a.source, __float_as_int(0.0f));
        mbar_init(&sm.bar[0], 1u);
        mbar_init(&sm.bar[1], 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.cnt[0] = sm.cnt[1] = sm.fcnt[0] = sm.fcnt[1] = 0;
        sm.fmin = 0xffffffffu;
        sm.lost = sm.abort = 0;
    }
    if (t < kClusterMax) {
        sm.told[0][SP_NEAR][t] = t == 0 ? 1 : 0;
        sm.told[0][SP_FAR][t] = 0;
        sm.told[0][SP_MIN][t] = -1;
    }
    __syncthreads();
    cluster_barrier();
    float step = a.step, T = step;
    int32_t top = 0;  // longest near queue since T moved
    int f = 0;        // current far pile
    for (int32_t ph = 0;; ++ph) {
        const int p = ph & 1, np = p ^ 1;
        const int32_t c = lane < C ? sm.told[p][SP_NEAR][lane] : 0;
        const int32_t fc = lane < C ? sm.told[p][SP_FAR][lane] : 0;
        const int32_t total = (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)c);
        const bool over = __any_sync(0xffffffffu, fc < 0);  // a far pile overflowed
        const bool far = __any_sync(0xffffffffu, fc > 0);
        if (over || total > a.max_near || (total == 0 && !far)) {
            if (rank == 0 && t == 0) {
                // handed over: the distances are those of paths; the grid's pull iterations finish them
                a.ho->done = over || total > a.max_near ? 0 : 1;
                a.status[ST_LEVELS] = ph;
            }
            cluster_barrier();  // no block leaves while another may still write to its shared memory
            return;
        }
        if (t == 0) sm.cnt[p] = 0;  // filled again at the next phase
        if (total == 0) {
            // no near vertex left: T moves on, and the far pile is split anew (stale entries, whose vertex
            // has come closer since, go)
            const uint32_t fm = lane < C ? (uint32_t)sm.told[p][SP_MIN][lane] : 0xffffffffu;
            if (top < kSpFew)
                step = fminf(2.0f * step, 1024.0f * a.step);
            else if (top > kSpMany)
                step = fmaxf(0.5f * step, 0.25f * a.step);
            top = 0;
            T = __uint_as_float(__reduce_min_sync(0xffffffffu, fm)) + step;
            const int32_t m = sm.fcnt[f];
            __syncthreads();
            if (t == 0) {
                sm.fmin = 0xffffffffu;
                sm.fcnt[f] = 0;
            }
            __syncthreads();
            for (int32_t i0 = 0; i0 < m; i0 += kSpThreads) {
                const int32_t i = i0 + t;
                bool live = false;
                int32_t v = 0;
                float d = 0.0f;
                if (i < m) {
                    v = a.farv[f][base + i];
                    d = a.fard[f][base + i];
                    live = !(__ldcg(a.dist + v) < d);
                }
                sp_near(a, sm, np, f ^ 1, base, live && d <= T, v, d);
                sp_far(a, sm, f ^ 1, base, live && !(d <= T), v, d);
            }
            f ^= 1;
        } else {
            top = max(top, total);
            const int32_t most = (int32_t)__reduce_max_sync(0xffffffffu, (uint32_t)c);
            const bool share = most > kSpPerRound && ((long long)most << shift) > (long long)total + (total >> 2);
            int32_t g0 = 0, m = sm.told[p][SP_NEAR][rank], inc = 0;
            if (share) {
                inc = (int32_t)warp_inclusive_sum((uint32_t)c);
                const int32_t each = (total + C - 1) >> shift;
                g0 = rank * each;
                m = max(0, min(total - g0, each));
                cluster_barrier();  // the other blocks' queues are complete
                if (ld_volatile_i32(&sm.abort)) return;
            }
            for (int32_t i0 = 0; i0 < m; i0 += kSpPerRound) {
                const int32_t i = i0 + t / kSpLanes;
                int32_t u = -1;
                float x = 0.0f;
                if (share) {
                    int32_t o, at;
                    cluster_locate(inc, g0 + i, o, at);
                    if (i < m) {
                        const uint32_t r = remote_smem(&sm.q[p][at], (uint32_t)o);
                        u = ld_remote(r);
                        x = __int_as_float(ld_remote(r + 4u));
                    }
                } else if (i < m) {
                    const int2 e = sm.q[p][i];
                    u = e.x;
                    x = __int_as_float(e.y);
                }
                int32_t w = -1;
                float len = 0.0f;
                bool live = false;
                if (u >= 0) {
                    live = !(__ldcg(a.dist + u) < x);  // else a smaller distance of u is queued, too
                    w = __ldg(reinterpret_cast<const int32_t*>(a.rcol + u) + j);
                    len = __ldg(reinterpret_cast<const float*>(a.rval + u) + j);
                }
                const bool more = live && w < -1;  // the last lane's neighbour is coded when the row goes on
                if (w < -1) w = -2 - w;
                sp_relax(a, sm, np, f, base, live && w >= 0, w, x + len, T);
                const uint32_t mm = __ballot_sync(0xffffffffu, more);
                if (mm) {
                    int32_t beg = 0, deg = 0;
                    if ((mm >> (lane | (kSpLanes - 1))) & 1u) {
                        beg = __ldg(a.ptr + u);
                        deg = __ldg(a.ptr + u + 1) - beg;
                    }
                    for (int32_t k = kSpLanes + j; __any_sync(0xffffffffu, k < deg); k += kSpLanes) {
                        const bool in = k < deg;
                        const int32_t v = in ? __ldg(a.col + beg + k) : 0;
                        const float d = in ? x + __ldg(a.val + beg + k) : 0.0f;
                        sp_relax(a, sm, np, f, base, in, v, d, T);
                    }
                }
            }
        }
        __syncthreads();
        if (t < C * SP_WORDS && !(kWithhold && rank == 1)) {
            const int to = t / SP_WORDS, what = t - to * SP_WORDS;
            const int32_t v = what == SP_NEAR ? min(sm.cnt[np], kSpCap)
                              : what == SP_FAR ? (sm.lost ? -1 : sm.fcnt[f])
                                               : (int32_t)sm.fmin;
            st_async(remote_smem(&sm.told[np][what][rank], (uint32_t)to), v, remote_smem(&sm.bar[np], (uint32_t)to));
        }
        if (t == 0) mbar_expect(&sm.bar[np], 4u * SP_WORDS * (uint32_t)C);
        if (!mbar_wait_block(&sm.bar[np], (uint32_t)(ph >> 1) & 1u, a.timeout_ns)) {
            if (t == 0) a.ho->done = 1;
            cluster_give_up(&sm.abort, C, a.status);
            return;
        }
    }
}

// ---------------------------------------------------------------- records

// rcol[v] / rval[v]: the first four out-edges of v (-1 past the row's end); the fourth
// neighbour w of a longer row is coded as -2 - w.
__global__ void sp_records_kernel(const int32_t* __restrict__ ptr, const int32_t* __restrict__ col,
                                  const float* __restrict__ val, int32_t n, int4* __restrict__ rcol,
                                  float4* __restrict__ rval) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t b = ptr[i], d = ptr[i + 1] - b;
        int4 c = make_int4(-1, -1, -1, -1);
        float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (d > 0) c.x = col[b], x.x = val[b];
        if (d > 1) c.y = col[b + 1], x.y = val[b + 1];
        if (d > 2) c.z = col[b + 2], x.z = val[b + 2];
        if (d > 3) c.w = d > 4 ? -2 - col[b + 3] : col[b + 3], x.w = val[b + 3];
        rcol[i] = c;
        rval[i] = x;
    }
}

// stats[0]: sum of the finite weights, stats[1]: their number, stats[2]: the negative ones.
__global__ void __launch_bounds__(256) sp_stats_kernel(const float* __restrict__ val, int64_t nnz, double* stats) {
    double sum = 0.0;
    unsigned long long fin = 0, neg = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
        const float x = val[i];
        if (x < INFINITY) {
            sum += (double)x;
            fin += 1;
        }
        neg += x < 0.0f ? 1 : 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    fin = warp_sum_u64(fin);
    neg = warp_sum_u64(neg);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(stats, sum);
        atomicAdd(stats + 1, (double)fin);
        if (neg) atomicAdd(stats + 2, (double)neg);
    }
}

// Which searches run here: rows of at most kSpMeshDegree entries.  On meshes the near queue stays
// short; random regular graphs and small worlds (10K to 2M vertices, 4 to 16 entries a row, integer
// and real weights) are handed over early and take 0.31 to 1.04 of the grid's time.  A graph with
// hubs reaches most of its vertices in a few iterations of the whole GPU.
constexpr int32_t kSpMeshDegree = 32;

gbx_status sssp_cluster_prepare(Graph* G, cudaStream_t s) {
    G->sp_step = -1.0f;
    if (G->max_out_degree > kSpMeshDegree || G->nnz == 0) return GBX_OK;
    if (!G->sp_rec) {
        const cudaError_t e = cudaMalloc(&G->sp_rec, 32 * (size_t)G->n);
        if (e == cudaErrorMemoryAllocation) {  // the weights are in; searches run on the whole grid
            G->sp_rec = nullptr;
            cudaGetLastError();
            return GBX_OK;
        }
        GBX_CUDA_TRY(e);
    }
    int4* rcol = static_cast<int4*>(G->sp_rec);
    const unsigned grid = std::min<unsigned>(div_up(G->n, 256), (unsigned)G->num_sms * 8u);
    sp_records_kernel<<<grid, 256, 0, s>>>(G->out_ptr, G->out_col, G->out_val, G->n, rcol,
                                           reinterpret_cast<float4*>(rcol + G->n));
    double* stats = reinterpret_cast<double*>(G->ws.flag + 12);  // 8-byte aligned words of the scratch
    GBX_CUDA_TRY(cudaMemsetAsync(stats, 0, 3 * sizeof(double), s));
    sp_stats_kernel<<<std::min<unsigned>(div_up(G->nnz, 256), (unsigned)G->num_sms * 8u), 256, 0, s>>>(G->out_val, G->nnz,
                                                                                                stats);
    GBX_CUDA_TRY(cudaGetLastError());
    double h[3] = {0.0, 0.0, 0.0};
    GBX_CUDA_TRY(cudaMemcpyAsync(h, stats, sizeof(h), cudaMemcpyDeviceToHost, s));
    GBX_CUDA_TRY(cudaStreamSynchronize(s));
    if (h[2] == 0.0 && h[1] > 0.0) G->sp_step = (float)(h[0] / h[1]) * kSpStep;
    return GBX_OK;
}

gbx_status sssp_cluster_wanted(Graph* G, const gbx_desc& d, bool* wanted) {
    *wanted = false;
    if (d.trace || d.direction == GBX_DIR_PULL || !(G->sp_step >= 0.0f)) return GBX_OK;
    if (G->sp_cluster_blocks == 0)
        GBX_TRY(cluster_fit((const void*)sssp_cluster_kernel<false>, kSpThreads, sizeof(SpSmem), &G->sp_cluster_blocks));
    *wanted = G->sp_cluster_blocks > 0;
    return GBX_OK;
}

static void sssp_cluster_args(Graph* G, int32_t source, float* dist, SpArgs& a) {
    a.n = G->n;
    a.source = source;
    a.ptr = G->out_ptr;
    a.col = G->out_col;
    a.val = G->out_val;
    a.rcol = static_cast<const int4*>(G->sp_rec);
    a.rval = reinterpret_cast<const float4*>(a.rcol + G->n);
    a.dist = dist;
    for (int i = 0; i < 2; ++i) {
        a.farv[i] = G->ws.q[i];
        a.fard[i] = reinterpret_cast<float*>(G->ws.qp[i]);
    }
    a.seg = G->n / G->sp_cluster_blocks;
    a.max_near = (int32_t)std::min<int64_t>(
        kSpMaxNear, (kSpMaxEdges + G->nnz / kSpMaxShare) * G->n / std::max<int64_t>(G->nnz, 1));
    a.step = G->sp_step;
    a.ho = G->ws.handoff;
    a.status = G->ws.status;
    a.timeout_ns = wait_timeout_ns();
}

gbx_status sssp_cluster_launch(Graph* G, int32_t source, float* dist, cudaStream_t s) {
    SpArgs a;
    sssp_cluster_args(G, source, dist, a);
    sp_fill_kernel<<<std::min<unsigned>(div_up(G->n, 512), (unsigned)G->num_sms * 4u), 512, 0, s>>>(dist, G->n, source);
    GBX_CUDA_TRY(cudaGetLastError());
    void* args[] = {&a};
    return cluster_launch((const void*)sssp_cluster_kernel<false>, G->sp_cluster_blocks, kSpThreads, sizeof(SpSmem), args,
                          s);
}

gbx_status sssp_cluster_selftest(Graph* G, uint64_t timeout_ns, cudaStream_t s) {
    bool wanted = false;
    gbx_desc d;
    gbx_desc_init(&d);
    GBX_TRY(sssp_cluster_wanted(G, d, &wanted));
    GBX_CHECK(wanted, GBX_ERR_NOT_SUPPORTED, "searches on this graph do not start in a cluster (or it has no weights)");
    const void* fn = (const void*)sssp_cluster_kernel<true>;
    int blocks = 0;
    GBX_TRY(cluster_fit(fn, kSpThreads, sizeof(SpSmem), &blocks));
    GBX_CHECK(blocks == G->sp_cluster_blocks, GBX_ERR_NOT_SUPPORTED, "the cluster does not fit");
    SpArgs a;
    float* const dist = reinterpret_cast<float*>(G->ws.qd[0]);
    sssp_cluster_args(G, 0, dist, a);
    a.timeout_ns = timeout_ns;
    sp_fill_kernel<<<std::min<unsigned>(div_up(G->n, 512), (unsigned)G->num_sms * 4u), 512, 0, s>>>(dist, G->n, 0);
    GBX_CUDA_TRY(cudaGetLastError());
    void* args[] = {&a};
    return cluster_launch(fn, blocks, kSpThreads, sizeof(SpSmem), args, s);
}

}  // namespace gbx
