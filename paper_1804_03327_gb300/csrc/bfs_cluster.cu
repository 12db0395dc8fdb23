// The small-frontier phase of gbx_bfs: one thread-block cluster walks the levels while the
// frontier is small, instead of the whole grid of bfs.cu.
//
// A level of a few thousand frontier vertices has no bandwidth to be bound by: it costs its
// chain of dependent memory round trips and its barrier.  In the grid-wide kernel that
// chain is nine trips long (prefix search, queue entry, neighbour, visited probe, claim, row
// offsets, queue slot, counters) and the barrier goes through the L2.  Here one trip is left:
//   - the frontier lives in the blocks' shared memory, each vertex with its first five
//     neighbours, and four lanes take a vertex;
//   - a neighbour is claimed by an atomicOr on the visited bitmap, which deduplicates exactly
//     (Eq 5) and is spread over the blocks' shared memory (a graph too large for that keeps
//     it in global memory), while the neighbour's own neighbours are loaded from the dense
//     first-entry and next-entries arrays (no row offsets).  On a large level only the
//     claimed ones load;
//   - the level ends when every block has the length of every block's new queue, sent with
//     st.async to an mbarrier of each.  The cluster's hardware barrier (release, acquire)
//     would also wait for the level's stores to global memory: 1,100 cycles of 3,100 on an
//     8-wide grid.  It is used only before a block reads another one's queue.  No other
//     order is needed between levels: exactly one claim of a bit returns it clear.
// The blocks keep what they found; a level whose blocks are unequal is split evenly, reading
// the other blocks' queues through distributed shared memory.  Rows with more than five
// entries take the rest from the column array, split evenly over the block's threads.
//
// 2048 x 2048 grid (1 % of the edges deleted, 3,375 levels of 1,250 vertices): 8.0 us a level
// in the grid-wide kernel, 1.7 here (26.2-27.0 -> 5.5-5.9 ms); an 8 x 20,000 grid 6.1 and 1.14 us.  A
// level then takes 3,800 cycles: 1,900 claims and loads, 300 waiting for the block's other
// warps, 1,000 for the other blocks.  Blocks of 256 threads: 2.10 us; clusters of 8: 3.1 us;
// neighbours only ever loaded after the claim: the 8-wide grid 1.22 us.
//
// Every level pushes.  Section 6.3's rule would pull on some levels of a small graph; depths
// do not depend on it, and the traced kernel (which reports the schedule) follows the rule.
#include "bfs_cluster.cuh"
#include "cluster.cuh"

#include <algorithm>

namespace gbx {

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClLanes = 4;                         // lanes per frontier vertex
constexpr int kClPerRound = kClThreads / kClLanes;  // frontier vertices a block takes at a time
constexpr int kClLongUnroll = 4;                    // entries of long rows in flight per thread
constexpr int kClCap = 8192;                        // queue entries a block holds
constexpr int kClNear = 1024;                       // ... of which with neighbours and parent
constexpr int kClBmWords = 15360;                   // bitmap words a block holds (n up to 7.8M in 16 blocks)
constexpr int kClAhead = 2 * kClPerRound;            // block share up to which neighbours are loaded ahead
constexpr int kClShareWhole = 16;                   // queue length from which a small graph's levels are shared
// The frontier at which the cluster hands over to the grid: the edges of that many average rows, at
// most kClMaxFrontier vertices.  The cluster takes about 5,000 edges a microsecond, a grid-wide
// level 8 to 10 us.  Random 16-regular graph of 30,000 vertices: 62 us, on the grid alone 79, with
// 24,576 vertices as the only limit 155; 126 x 126 x 126 grid 2.61 ms, 2.70 and 2.86.  48K edges: 2.49
// there, but a ring of 500,000 vertices with one edge in a thousand rewired 1.87 ms instead of 1.33;
// 96K and 128K: 2.87 on the 3-D grid.  2-D grids keep below it (a 2000 x 2000 one 5.58 ms with all).
constexpr int kClMaxFrontier = 24576;
constexpr int64_t kClMaxEdges = 64 * 1024;

struct ClArgs {
    int32_t n, nwords, source;
    const int32_t* ptr;
    const int32_t* col;
    const int32_t* first;
    const int4* next;
    int32_t* depth;
    int32_t* parent;
    uint32_t* vis;
    int32_t* list;   // hand-over: the frontier
    int32_t* spill;  // ... and the entries no queue had room for
    ClHandoff* ho;
    int32_t* status;
    int32_t fill;   // initialise the outputs and the bitmap here (else cl_fill_kernel did)
    int32_t whole;  // the graph fits: never hand over
    int32_t max_frontier;  // ... else above this many vertices
    unsigned long long timeout_ns;
    int32_t shared_bm;  // the visited bitmap is in shared memory (block r: words w with w mod blocks = r)
};

// Outputs and visited bitmap of a new search (Algorithm 1, lines 2-5), by threads
// [tid, stride) of the launch.
__device__ __forceinline__ void cl_fill(const ClArgs& a, long long tid, long long stride) {
    fill_i32(a.depth, a.n, -1, a.source, 0, tid, stride);
    if (a.parent) fill_i32(a.parent, a.n, -1, a.source, a.source, tid, stride);
    if (a.shared_bm) return;
    for (long long w = tid; w < a.nwords; w += stride)
        a.vis[w] = w == (a.source >> 5) ? 1u << (a.source & 31) : 0u;
}

__global__ void __launch_bounds__(512) cl_fill_kernel(ClArgs a) {
    cl_fill(a, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

struct ClSmem {
    int32_t q[2][kClCap];       // this block's part of the frontier, and of the next one
    int32_t nb[2][5][kClNear];  // the first kClNear entries' neighbours 0..4 (-1 past the row's end) ...
    int32_t par[2][kClNear];    // ... and parents (a neighbour that needs no claim)
    int32_t lq[kClCap];         // frontier vertices with entries past the fifth
    int32_t pre[kClThreads];    // long rows: exclusive prefix of the entries left, start, vertex
    int32_t beg[kClThreads];
    int32_t own[kClThreads];
    unsigned long long bar[2];  // mbarriers of the queue lengths, by level parity
    int32_t counts[2][kClusterMax];      // every block's queue length, by level parity
    int32_t cnt[2];             // entries in q[.]
    int32_t lcnt[2];            // entries in lq, by level parity
    int32_t abort;              // a block's wait ran out
    int32_t wsum[kClWarps];
    uint32_t bm[1];             // the block's words of the visited bitmap (as many as the launch asks for)
};

// The cluster's shape, as every thread keeps it.
struct ClShape {
    int rank, shift;  // this block, log2 of the number of blocks
};

// Claims w[k] for frontier vertices u[k] at level L (w < 0: nothing to claim) and queues them
// with their neighbours, which are loaded for every candidate while the claims are under
// way (ahead) or for the claimed ones only; all lanes of the warp call this.
template <int K>
__device__ __forceinline__ void cl_claim(const ClArgs& a, ClSmem& sm, const ClShape& cs, int32_t L, int np,
                                         const int32_t (&u)[K], const int32_t (&w)[K], bool ahead) {
    const int lane = threadIdx.x & 31;
    uint32_t old[K];
    int32_t f[K];
    int4 x[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        old[k] = 0xffffffffu;
        if (w[k] < 0) continue;
        const uint32_t word = (uint32_t)w[k] >> 5, bit = 1u << (w[k] & 31);
        if (a.shared_bm)
            old[k] = or_remote(remote_smem(sm.bm + (word >> cs.shift), word & ((1u << cs.shift) - 1u)), bit);
        else
            old[k] = atomicOr(a.vis + word, bit);
    }
    if (ahead) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (w[k] >= 0) {
                f[k] = __ldg(a.first + w[k]);
                x[k] = __ldg(a.next + w[k]);
            }
    }
    uint32_t m[K];
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        m[k] = __ballot_sync(0xffffffffu, w[k] >= 0 && !((old[k] >> (w[k] & 31)) & 1u));
        cnt += __popc(m[k]);
    }
    if (cnt == 0) return;
    int32_t pos = 0;
    if (lane == 0) pos = atomicAdd(&sm.cnt[np], cnt);
    pos = __shfl_sync(0xffffffffu, pos, 0);
    int32_t at[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        at[k] = (m[k] >> lane) & 1u ? pos + __popc(m[k] & lanemask_lt()) : -1;
        pos += __popc(m[k]);
        if (!ahead && at[k] >= 0 && at[k] < kClNear) {
            f[k] = __ldg(a.first + w[k]);
            x[k] = __ldg(a.next + w[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (at[k] < 0) continue;
        if (at[k] < kClCap)
            sm.q[np][at[k]] = w[k];
        else
            a.spill[atomicAdd(&a.ho->spilled, 1)] = w[k];  // the level ends in a hand-over
        if (at[k] < kClNear) {
            sm.nb[np][0][at[k]] = f[k];
            sm.nb[np][1][at[k]] = x[k].x;
            sm.nb[np][2][at[k]] = x[k].y;
            sm.nb[np][3][at[k]] = x[k].z;
            sm.nb[np][4][at[k]] = x[k].w;
            sm.par[np][at[k]] = u[k];
        }
        a.depth[w[k]] = L + 1;
        if (a.parent) a.parent[w[k]] = u[k];
    }
}

// The entries past the fifth of the block's nl long rows, split evenly over its threads.
__device__ __forceinline__ void cl_long_rows(const ClArgs& a, ClSmem& sm, const ClShape& cs, int32_t L, int np,
                                             int32_t nl) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
    for (int32_t b = 0; b < nl; b += kClThreads) {
        int32_t v = 0, beg = 0, left = 0;
        if (b + t < nl) {
            v = sm.lq[b + t];
            beg = __ldg(a.ptr + v) + 5;
            left = max(0, __ldg(a.ptr + v + 1) - beg);
        }
        const int32_t inc = (int32_t)warp_inclusive_sum((uint32_t)left);
        if (lane == 31) sm.wsum[wid] = inc;
        __syncthreads();
        const int32_t wv = lane < kClWarps ? sm.wsum[lane] : 0;
        const int32_t winc = (int32_t)warp_inclusive_sum((uint32_t)wv);
        const int32_t total = __shfl_sync(0xffffffffu, winc, 31);
        sm.pre[t] = __shfl_sync(0xffffffffu, winc - wv, wid) + inc - left;
        sm.beg[t] = beg;
        sm.own[t] = v;
        __syncthreads();
        for (int32_t i0 = 0; i0 < total; i0 += kClThreads * kClLongUnroll) {
            int32_t u[kClLongUnroll], w[kClLongUnroll];
#pragma unroll
            for (int k = 0; k < kClLongUnroll; ++k) {
                const int32_t i = i0 + k * kClThreads + t;
                u[k] = 0;
                w[k] = -1;
                if (i < total) {
                    int32_t lo = 0;  // last entry whose prefix is <= i
#pragma unroll
                    for (int s = kClThreads / 2; s > 0; s >>= 1)
                        if (sm.pre[lo + s] <= i) lo += s;
                    u[k] = sm.own[lo];
                    w[k] = __ldg(a.col + sm.beg[lo] + (i - sm.pre[lo]));
                }
            }
            cl_claim<kClLongUnroll>(a, sm, cs, L, np, u, w, false);
        }
        __syncthreads();
    }
}

// A block's part of a level: its own queue, or entries [g0, g0 + m) of all queues one after
// another (lane r of a warp holds where block r's ends in inc).
struct ClPart {
    bool share;
    int32_t inc, g0, m;
};

// Takes the block's part of level L, kClLanes lanes per vertex and K rounds in flight.
template <int K>
__device__ __forceinline__ void cl_take(const ClArgs& a, ClSmem& sm, const ClShape& cs, int32_t L, const ClPart& part) {
    const int t = threadIdx.x, lane = t & 31, j = t & (kClLanes - 1);
    const int p = L & 1, np = p ^ 1;
    const bool ahead = part.m <= kClAhead;
    for (int32_t i0 = 0; i0 < part.m; i0 += kClPerRound * K) {
        int32_t u[K], w[K], w5[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int32_t i = i0 + k * kClPerRound + t / kClLanes;
            u[k] = w[k] = w5[k] = -1;
            int32_t parent = -1;
            bool near = true;
            if (part.share) {
                int32_t o, x;
                cluster_locate(part.inc, part.g0 + i, o, x);
                if (i < part.m) {
                    near = x < kClNear;
                    u[k] = ld_remote(remote_smem(&sm.q[p][x], (uint32_t)o));
                    if (near) {
                        w[k] = ld_remote(remote_smem(&sm.nb[p][j][x], (uint32_t)o));
                        if (j == 3) w5[k] = ld_remote(remote_smem(&sm.nb[p][4][x], (uint32_t)o));
                        parent = ld_remote(remote_smem(&sm.par[p][x], (uint32_t)o));
                    }
                }
            } else if (i < part.m) {
                near = i < kClNear;
                u[k] = sm.q[p][i];
                if (near) {
                    w[k] = sm.nb[p][j][i];
                    if (j == 3) w5[k] = sm.nb[p][4][i];
                    parent = sm.par[p][i];
                }
            }
            if (!near) {
                if (j == 0) {
                    w[k] = __ldg(a.first + u[k]);
                } else if (j < 3) {
                    w[k] = __ldg(reinterpret_cast<const int32_t*>(a.next + u[k]) + (j - 1));
                } else {
                    const int2 y = __ldg(reinterpret_cast<const int2*>(a.next + u[k]) + 1);
                    w[k] = y.x;
                    w5[k] = y.y;
                }
            }
            if (w[k] == parent) w[k] = -1;  // visited
        }
        bool more = false;
#pragma unroll
        for (int k = 0; k < K; ++k) more |= w5[k] >= 0;
        cl_claim<K>(a, sm, cs, L, np, u, w, ahead);
        if (__any_sync(0xffffffffu, more)) {
            cl_claim<K>(a, sm, cs, L, np, u, w5, false);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const uint32_t mm = __ballot_sync(0xffffffffu, w5[k] >= 0);
                int32_t base = 0;
                if (lane == 0 && mm) base = atomicAdd(&sm.lcnt[p], __popc(mm));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (w5[k] >= 0) sm.lq[base + __popc(mm & lanemask_lt())] = u[k];
            }
        }
    }
}

// kWithhold: block 1 keeps its queue length to itself, so that every block's wait runs out.
template <bool kWithhold>
__global__ void __launch_bounds__(kClThreads, 1) bfs_cluster_kernel(const __grid_constant__ ClArgs a) {
    extern __shared__ __align__(16) unsigned char raw[];
    ClSmem& sm = *reinterpret_cast<ClSmem*>(raw);
    const int t = threadIdx.x, lane = t & 31;
    const int rank = (int)cluster_rank(), C = (int)cluster_size();
    const ClShape cs{rank, 31 - __clz(C)};
    // an error of an earlier launch not yet read by the host: this launch does nothing
    const int pending = t == 0 ? ld_volatile_i32(a.status + ST_ERROR) : 0;
    if (__syncthreads_or(pending)) {
        if (rank == 0 && t == 0) a.ho->done = 1;
        return;
    }
    if (a.fill) cl_fill(a, (long long)rank * kClThreads + t, (long long)C * kClThreads);
    if (t == 0) {
        sm.q[0][0] = a.source;  // its depth and parent come with the initialisation
        sm.par[0][0] = a.source;
        const int4 x = __ldg(a.next + a.source);
        sm.nb[0][0][0] = __ldg(a.first + a.source);
        sm.nb[0][1][0] = x.x;
        sm.nb[0][2][0] = x.y;
        sm.nb[0][3][0] = x.z;
        sm.nb[0][4][0] = x.w;
        mbar_init(&sm.bar[0], 1u);
        mbar_init(&sm.bar[1], 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.abort = 0;
        sm.cnt[0] = sm.cnt[1] = sm.lcnt[0] = sm.lcnt[1] = 0;
        if (rank == 0) a.ho->spilled = 0;
    }
    if (t < kClusterMax) sm.counts[0][t] = t == 0 ? 1 : 0;
    if (a.shared_bm) {
        const int32_t sw = a.source >> 5;
        for (int32_t i = t; rank + (i << cs.shift) < a.nwords; i += kClThreads)
            sm.bm[i] = rank + (i << cs.shift) == sw ? 1u << (a.source & 31) : 0u;
    }
    __syncthreads();
    cluster_barrier();
    int32_t last = 0;  // size of the frontier one level up
    for (int32_t L = 0;; ++L) {
        const int p = L & 1, np = p ^ 1;
        const int32_t c = lane < C ? sm.counts[p][lane] : 0;
        const int32_t total = (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)c);
        const int32_t most = (int32_t)__reduce_max_sync(0xffffffffu, (uint32_t)c);
        if (total == 0 || L >= a.n) {
            if (rank == 0 && t == 0) {
                a.status[ST_LEVELS] = L;
                if (total) atomicCAS(a.status + ST_ERROR, 0, (int)GBX_ERR_OVERFLOW);  // more than n levels
                a.ho->done = 1;
            }
            cluster_barrier();  // no block leaves while another may still write to its shared memory
            return;
        }
        int32_t inc = 0;  // the blocks' queues one after another: where each one ends
        if (!a.whole && (total > a.max_frontier || most > kClCap)) {
            // hand over: the queues one after another (the spilled entries are listed already)
            cluster_barrier();  // every claim is in the bitmap
            if (ld_volatile_i32(&sm.abort)) return;
            inc = (int32_t)warp_inclusive_sum((uint32_t)min(c, kClCap));
            const int32_t m = min(sm.counts[p][rank], kClCap);
            const int32_t at = __shfl_sync(0xffffffffu, inc, rank) - m;
            for (int32_t i = t; i < m; i += kClThreads) a.list[at + i] = sm.q[p][i];
            if (rank == 0 && t == 0) {
                a.ho->done = 0;
                a.ho->level = L;
                a.ho->frontier = total;
                a.ho->before = last;
            }
            if (rank == C - 1 && t == 0) a.ho->listed = at + m;
            if (a.shared_bm)
                for (int32_t i = t; rank + (i << cs.shift) < a.nwords; i += kClThreads)
                    a.vis[rank + (i << cs.shift)] = sm.bm[i];
            cluster_barrier();
            return;
        }
        if (t == 0) {
            sm.cnt[p] = 0;   // filled again at the next level
            sm.lcnt[np] = 0;
        }
        // each block its own queue, or an equal share of all when the blocks are unequal
        // (rows of a small dense graph are long: even a few are worth sharing)
        const bool share = most > (a.whole ? kClShareWhole : kClPerRound) &&
                           ((long long)most << cs.shift) > (long long)total + (total >> 2);
        int32_t g0 = 0, m = sm.counts[p][rank];
        if (share) {
            inc = (int32_t)warp_inclusive_sum((uint32_t)c);
            const int32_t each = (total + C - 1) >> cs.shift;
            g0 = rank * each;
            m = max(0, min(total - g0, each));
            cluster_barrier();  // the other blocks' queues are complete
            if (ld_volatile_i32(&sm.abort)) return;
        }
        const ClPart part{share, inc, g0, m};
        if (m <= kClPerRound)
            cl_take<1>(a, sm, cs, L, part);
        else
            cl_take<2>(a, sm, cs, L, part);
        __syncthreads();
        const int32_t nl = sm.lcnt[p];
        if (nl) {
            cl_long_rows(a, sm, cs, L, np, nl);
            __syncthreads();
        }
        // this block's queue length to every block, theirs from them
        if (t < C && !(kWithhold && rank == 1))
            st_async(remote_smem(&sm.counts[np][rank], (uint32_t)t), sm.cnt[np], remote_smem(&sm.bar[np], (uint32_t)t));
        if (t == 0) mbar_expect(&sm.bar[np], 4u * (uint32_t)C);
        last = total;
        if (!mbar_wait_block(&sm.bar[np], (uint32_t)(L >> 1) & 1u, a.timeout_ns)) {
            if (t == 0) a.ho->done = 1;
            cluster_give_up(&sm.abort, C, a.status);
            return;
        }
    }
}

// ---------------------------------------------------------------- host side

static_assert(sizeof(ClSmem) + 4 * kClBmWords <= 232448, "fits a block's shared memory");
static size_t cl_smem(int32_t bm_words) { return sizeof(ClSmem) + sizeof(uint32_t) * (size_t)bm_words; }

static gbx_status cl_geometry(Graph* G) {
    if (G->cluster_blocks != 0) return GBX_OK;
    return cluster_fit((const void*)bfs_cluster_kernel<false>, kClThreads, cl_smem(kClBmWords), &G->cluster_blocks);
}

// Which searches start in the cluster: those of graphs whose levels stay small.
//  - no row longer than kClMeshDegree.  On grids, meshes and roads there are many small levels.  A
//    graph of short rows whose frontier grows fast (random regular, small world) is handed
//    over after a few levels, each still cheaper here: 16 entries a row 63 us for 10,000 vertices
//    (82 on the grid alone), 80 for 100,000 (109), 91 for 500,000 (96), 235 for 2M (247).  A graph with
//    hubs reaches most of its vertices in a few levels, which need the whole GPU: RMAT-22 takes 107 us.
//  - a graph that one block's queue holds (n <= kClCap) with few entries: every level is
//    small.  RMAT-10 (edge factor 16) takes 25 us here and 41 on the grid (one block per SM).  Of 112 RMAT
//    graphs (500 to 8,000 vertices, edge factors 2 to 24, directed and not) all 89 of up to 72K
//    entries are faster here (69-72K: 41-43 us and 43-45), and of those with 74K to 95K the grid is:
//    4,000 vertices of edge factor 12 43.7 and 41.4, of 16 49.2 and 42.0.
constexpr int32_t kClMeshDegree = 32;
constexpr int64_t kClTinyEntries = 72 * 1024;

static bool cl_tiny(const Graph* G) { return G->n <= kClCap && G->nnz <= kClTinyEntries; }

gbx_status cluster_bfs_wanted(Graph* G, const gbx_desc& d, bool* wanted) {
    *wanted = false;
    if (d.trace || d.direction == GBX_DIR_PULL || d.heuristic != GBX_HEUR_RATIO) return GBX_OK;
    // the switches of Sections 5.2-5.4 change what a pull level does: they are measured in the grid-wide kernel
    if (d.direction == GBX_DIR_AUTO && !(d.early_exit && d.masking && d.operand_reuse)) return GBX_OK;
    if (!cl_tiny(G) && G->max_out_degree > kClMeshDegree) return GBX_OK;
    GBX_TRY(cl_geometry(G));
    *wanted = G->cluster_blocks > 0;
    return GBX_OK;
}

static void cluster_bfs_args(Graph* G, int32_t source, int32_t* depth, int32_t* parent, ClArgs& a, int32_t* bm_words) {
    a.n = G->n;
    a.nwords = G->nwords;
    a.source = source;
    a.ptr = G->out_ptr;
    a.col = G->out_col;
    a.first = G->first_out;
    a.next = G->next_out;
    a.depth = depth;
    a.parent = parent;
    a.vis = G->ws.bm[0];
    a.list = G->ws.q[1];
    a.spill = G->ws.list;
    a.ho = G->ws.handoff;
    a.status = G->ws.status;
    a.whole = cl_tiny(G) ? 1 : 0;
    a.max_frontier = (int32_t)std::min<int64_t>(kClMaxFrontier, kClMaxEdges * G->n / std::max<int64_t>(G->nnz, 1));
    a.timeout_ns = wait_timeout_ns();
    a.fill = G->n <= (1 << 16) ? 1 : 0;  // 16 blocks write 0.5 MB faster than a launch takes
    *bm_words = (G->nwords + G->cluster_blocks - 1) / G->cluster_blocks;
    a.shared_bm = *bm_words <= kClBmWords ? 1 : 0;
    if (!a.shared_bm) *bm_words = 0;
}

gbx_status cluster_bfs_launch(Graph* G, int32_t source, int32_t* depth, int32_t* parent, cudaStream_t s,
                              bool* complete) {
    ClArgs a;
    int32_t bm_words = 0;
    cluster_bfs_args(G, source, depth, parent, a, &bm_words);
    *complete = a.whole != 0;
    if (!a.fill) {
        const unsigned blocks = std::min<unsigned>(div_up(G->n, 512 * 4), (unsigned)G->num_sms * 4u);
        cl_fill_kernel<<<blocks, 512, 0, s>>>(a);
        GBX_CUDA_TRY(cudaGetLastError());
    }
    void* args[] = {&a};
    GBX_TRY(cluster_launch((const void*)bfs_cluster_kernel<false>, G->cluster_blocks, kClThreads, cl_smem(bm_words), args,
                           s));
    return GBX_OK;
}

gbx_status cluster_bfs_selftest(Graph* G, uint64_t timeout_ns, cudaStream_t s) {
    bool wanted = false;
    gbx_desc d;
    gbx_desc_init(&d);
    GBX_TRY(cluster_bfs_wanted(G, d, &wanted));
    GBX_CHECK(wanted, GBX_ERR_NOT_SUPPORTED, "searches on this graph do not start in a cluster");
    const void* fn = (const void*)bfs_cluster_kernel<true>;
    int blocks = 0;
    GBX_TRY(cluster_fit(fn, kClThreads, cl_smem(kClBmWords), &blocks));
    GBX_CHECK(blocks == G->cluster_blocks, GBX_ERR_NOT_SUPPORTED, "the cluster does not fit");
    ClArgs a;
    int32_t bm_words = 0;
    cluster_bfs_args(G, 0, G->ws.qp[0], nullptr, a, &bm_words);
    a.fill = 1;
    a.timeout_ns = timeout_ns;
    void* args[] = {&a};
    return cluster_launch(fn, blocks, kClThreads, cl_smem(bm_words), args, s);
}

}  // namespace gbx
