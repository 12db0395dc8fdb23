// Masked matvec over the (min, +) semiring (R u {+inf}, +, min, +inf) that
// Section 5.6 names for SSSP: the generalised-semiring form of Eq 2-5 with
// x = + and + = min, no early exit (it exists only for Boolean semirings) and no
// structure-only shortcut (the values are read).  Same two directions as the
// Boolean operator: pull computes each passing row's minimum over its entries
// (Algorithm 2 without the break), push expands the columns of u's finite
// entries and folds them into w with an atomic minimum (Eq 5 / Algorithm 3's
// reduction, done in place).  All sums are binary32.
//
// A call is three kernels, four under AUTO (a push then needs a queue first): mask and u, the
// matvec, the rows a pull deferred.  A call that can only pull reads a dense mask itself and
// needs the last one only if the graph has rows that are deferred.  The scratch is that of the
// Boolean operator (mxv.cu), left zero.
#include <algorithm>
#include <cmath>

#include "frontier.cuh"
#include "gbx_internal.cuh"
#include "mxv.cuh"

namespace gbx {

constexpr int kMpUnroll = 4;          // entries a lane has in flight
constexpr int32_t kMpChunk = 512;     // entries of a deferred row a warp takes at a time
constexpr int32_t kMpLongSteps = 4;   // steps left beyond which a row is deferred ...
constexpr int32_t kMpWarpSteps = 16;  // ... with a whole warp to a row

struct MpArgs {
    int32_t n, nwords;
    MxvVec mask;
    uint32_t invert;
    int32_t accum, dir, group;
    int32_t rows;       // rows a warp of the pull takes at a time: 32, fewer where that leaves warps without any
    int32_t push_most;  // finite entries of u up to which AUTO pushes
    const float* u;
    float* w;
    const int32_t* pull_ptr;
    const int32_t* pull_col;
    const float* pull_val;
    const int32_t* push_ptr;
    const int32_t* push_col;
    const float* push_val;
    uint32_t* ubm;
    uint32_t* pass;
    LevelCtr* ctr;  // q: the push queue; n_new: finite entries of u
    int32_t* q[2];  // [0] the push queue, [1] deferred rows: row, next entry, prefix of the chunk counts
    int32_t* qp[2];
    int32_t* qd[2];
    int32_t nothing;
    const uint8_t* bytes;  // the dense mask, where the pull reads it as it is
    int32_t shorts;        // every row is short: a lane each
    int32_t dirty;         // the bitmaps have been written
    unsigned long long* huge;  // deferred rows and their chunks; zero when the pull starts
    int32_t longest;       // entries left beyond which a row is deferred
};

__device__ __forceinline__ int mp_dir(const MpArgs& a) {
    if (a.dir != GBX_DIR_AUTO) return a.dir;
    return (int32_t)a.ctr->n_new <= a.push_most ? GBX_DIR_PUSH : GBX_DIR_PULL;
}

__device__ __forceinline__ bool mp_pass(const MpArgs& a, int32_t i) {
    return a.mask.format < 0 || (((a.pass[i >> 5] ^ a.invert) >> (i & 31)) & 1u);
}

// ... of a pull, which may read the mask's bytes
__device__ __forceinline__ bool mp_pull_pass(const MpArgs& a, int32_t i) {
    return a.bytes ? (a.bytes[i] != 0) != (a.invert != 0u) : mp_pass(a, i);
}

__device__ __forceinline__ Stage mp_stage(const MpArgs& a, StageBuf* sb, Acc* acc) {
    return Stage{sb + (threadIdx.x >> 5), 0, a.ctr, a.q[0], a.qp[0], a.qd[0], a.push_ptr, a.push_ptr, 0, 0, acc};
}

// The mask as a bitmap; u's finite entries as the push queue (dir == PUSH) or as a bitmap and
// their number (AUTO); w = +inf where a push without accumulation starts from that.
__global__ void __launch_bounds__(kMxvThreads) mp_prep_kernel(const __grid_constant__ MpArgs a) {
    pdl_begin();
    __shared__ StageBuf sb[kMxvThreads / 32];
    __shared__ unsigned long long bsm[kMxvThreads / 32];
    __shared__ unsigned long long csm[kMxvThreads / 32][4];
    const int lane = threadIdx.x & 31;
    const int64_t gtid = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x, gs = (int64_t)gridDim.x * kMxvThreads;
    if (gtid == 0) *a.huge = 0ull;
    if (a.mask.format == GBX_DENSE) {
        for (int64_t w = gtid; w < a.nwords; w += gs)
            a.pass[w] = pack_word(static_cast<const uint8_t*>(a.mask.data), a.n, (int32_t)w);
    } else if (a.mask.format == GBX_SPARSE) {
        const int32_t* list = static_cast<const int32_t*>(a.mask.data);
        const int32_t count = min(*a.mask.count, a.mask.cap);
        for (int64_t i = gtid; i < count; i += gs) {
            const int32_t v = list[i];
            if (v >= 0 && v < a.n) atomicOr(a.pass + (v >> 5), 1u << (v & 31));
        }
    }
    if (a.dir == GBX_DIR_PULL && !a.nothing) return;
    if ((a.dir == GBX_DIR_PUSH || a.nothing) && !a.accum)
        for (int64_t i = gtid; i < a.n; i += gs) a.w[i] = INFINITY;
    if (a.nothing) return;
    Acc acc;
    Stage st = mp_stage(a, sb, &acc);
    uint32_t cnt = 0;
    for (int64_t b = gtid - lane; b < a.n; b += gs) {  // warp-uniform
        const int32_t i = (int32_t)b + lane;
        const bool fin = i < a.n && a.u[i] < INFINITY;
        if (a.dir == GBX_DIR_PUSH) {
            st.put(fin, i);
        } else {
            const uint32_t word = __ballot_sync(0xffffffffu, fin);
            if (lane == 0) a.ubm[b >> 5] = word;
            cnt += fin ? 1u : 0u;
        }
    }
    if (a.dir == GBX_DIR_PUSH) st.flush_block<kMxvThreads / 32>(bsm);
    block_add_counts<kMxvThreads / 32>(csm, cnt, 0ull, 0ull, 0ull, &a.ctr->n_new, nullptr, nullptr, nullptr);
}

// Push: w(i) <- min(w(i), a(j, i) + u(j)) for every entry of the columns of u's finite
// entries j, rows that pass the mask only; the edges are split evenly over all warps.
__device__ __forceinline__ void mp_push(const MpArgs& a) {
    const unsigned long long qv = a.ctr->q;
    const uint32_t qcount = (uint32_t)qv;
    const int32_t E = (int32_t)(qv >> 32);
    const int gwarp = (int)((blockIdx.x * kMxvThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMxvThreads) >> 5);
    constexpr int kStep = 32 * kMpUnroll;
    int32_t chunk = (int32_t)(((long long)E + nwarps - 1) / nwarps);
    chunk = chunk <= 32 ? 32 : ((chunk + kStep - 1) / kStep) * kStep;
    for (long long e0l = (long long)gwarp * chunk; e0l < E; e0l += (long long)nwarps * chunk) {
        const int32_t e0 = (int32_t)e0l;
        const int32_t e1 = E - e0 > chunk ? e0 + chunk : E;
        PushCursorT<kMpUnroll> cur;
        cur.k = warp_find_entry(a.qp[0], (int32_t)qcount, e0);
        cur.wlast = -1;
        for (int32_t base = e0; base < e1; base += kStep) {
            const PushStepT<kMpUnroll> ps = cur.gather(a.push_col, a.q[0], a.qp[0], a.qd[0], qcount, base, e1);
            float x[kMpUnroll], old[kMpUnroll];
            bool ok[kMpUnroll];
#pragma unroll
            for (int t = 0; t < kMpUnroll; ++t) {
                const bool in = ps.u[t] >= 0;
                x[t] = in ? a.u[ps.u[t]] + a.push_val[ps.k[t]] : INFINITY;
                old[t] = in ? a.w[ps.v[t]] : 0.0f;
                ok[t] = in && mp_pass(a, ps.v[t]);
            }
#pragma unroll
            for (int t = 0; t < kMpUnroll; ++t)  // a stale w only costs an atomic: w falls
                if (ok[t] && x[t] < old[t]) atomic_min_f32(a.w + ps.v[t], x[t]);
        }
    }
}

// The minimum over entries [beg, beg + len) of a row, by a warp.
__device__ __forceinline__ float mp_chunk(const MpArgs& a, int32_t beg, int32_t len) {
    float m = INFINITY;
    for (int32_t o = threadIdx.x & 31; o < len; o += 32 * kMpUnroll) {
        int32_t j[kMpUnroll];
        float x[kMpUnroll];
#pragma unroll
        for (int t = 0; t < kMpUnroll; ++t) {
            const bool in = o + 32 * t < len;
            j[t] = in ? __ldg(a.pull_col + beg + o + 32 * t) : -1;
            x[t] = in ? __ldg(a.pull_val + beg + o + 32 * t) : INFINITY;
        }
#pragma unroll
        for (int t = 0; t < kMpUnroll; ++t)
            if (j[t] >= 0) m = fminf(m, x[t] + __ldg(a.u + j[t]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
    return m;
}

// The long rows of a small graph a block finishes itself (mp_pull<true>): no launch for them.  A pull of
// 50,000 rows that a mask lets 1 % of through, 9.8-12.3 us with that launch, takes 7.5; one of 5,000
// rows 12.3, now 10.3.  A block that meets more than kMpLongs leaves the rest to the groups that have them.
// Above 58,000 rows (fewer than four lanes each) a block meets too many: 388,799 rows, 4 directed
// edges each, 30 us with the launch and 48 without.
constexpr int kMpLongs = 64;
constexpr int32_t kMpBlockRow = 16384;
struct MpLong {
    int2 row[kMpLongs];  // row, next entry
    float part[kMxvThreads / 32];
    int count;
};

// Pull: groups of a.group lanes take a row each, kMpUnroll entries a lane in flight, and go on to
// the next row as soon as their own is done.  A warp's row offsets come 32 rows at a time,
// the next 32 loaded ahead.  A row with more than a.longest entries left is deferred:
// mp_last_kernel spreads its chunks over all warps, or (kBlock) the block's warps take them in the end.
//
// Bound by the gathers of u (4 bytes of a 32-byte L2 sector per entry).  A lane per row of up to
// 32 entries, one load at a time, and a warp for each longer row had taken 316 us on a
// directed graph of 700,001 rows and 11.2M entries whose longest rows hold tens of thousands
// (the whole call 373-382 us, now 82-90; rows deferred after 8, 16 and 64 steps 2, 9 and 39 us
// more).  The group is 8 lanes from 12 entries a row on, 4 from 6, else 1: rows shorter
// than the group's step leave lanes idle, longer ones take several dependent steps.  On small graphs
// it grows to a warp while a quarter of the lanes are enough, and a row of up to 2,176 entries is not
// deferred then: 3,537 vertices and 24 edges each 11.2 us with a launch for the deferred rows, so 7.6.
template <bool kBlock>
__device__ __forceinline__ void mp_pull(const MpArgs& a, uint8_t* list, MpLong& lo) {
    if constexpr (kBlock) {
        if (threadIdx.x == 0) lo.count = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int G = a.group, sub = lane & (G - 1), first = lane & ~(G - 1);
    const int32_t nwarps = (int32_t)((gridDim.x * kMxvThreads) >> 5);
    const int32_t R = a.rows, ntiles = (a.n + R - 1) / R;
    int32_t tile = (int32_t)((blockIdx.x * kMxvThreads + threadIdx.x) >> 5);
    // a tile's rows: lane l holds row R tile + l
    auto load = [&](int32_t t, int32_t& b, int32_t& e) {
        const int64_t i = (int64_t)t * R + lane;
        b = e = 0;
        if (t < ntiles && lane < R && i < a.n && mp_pull_pass(a, (int32_t)i)) {
            b = __ldg(a.pull_ptr + i);
            e = __ldg(a.pull_ptr + i + 1);
        }
    };
    int32_t b0, e0, b1, e1;
    load(tile, b0, e0);
    load(tile + nwarps, b1, e1);
    int32_t base = -1;        // first row of the tile in b0 / e0
    int open = 0, next = 0;   // its rows with entries (list: their lanes), and how many are handed out
    bool fresh = true;        // the tile has not been looked at
    int32_t v = -1, k = 0, end = 0;
    float m = INFINITY;
    for (;;) {
        const uint32_t need = __ballot_sync(0xffffffffu, v < 0 && sub == 0);
        if (need && next == open && tile < ntiles) {
            if (!fresh) {
                tile += nwarps;
                b0 = b1;
                e0 = e1;
                load(tile + nwarps, b1, e1);
            }
            fresh = false;
            base = tile * R;
            const uint32_t with = __ballot_sync(0xffffffffu, e0 > b0);  // none past the last tile
            __syncwarp();
            if (e0 > b0) list[__popc(with & lanemask_lt())] = (uint8_t)lane;
            __syncwarp();
            open = __popc(with);
            next = 0;
            // rows without entries (or that do not pass) are settled here; min(NaN, +inf) is +inf where a
            // row passes
            if (tile < ntiles && e0 == b0 && lane < R && base + lane < a.n) {
                if (!a.accum)
                    a.w[base + lane] = INFINITY;
                else if (mp_pull_pass(a, base + lane) && isnan(a.w[base + lane]))
                    a.w[base + lane] = INFINITY;
            }
        }
        if (need && next < open) {
            const int r = next + __popc(need & ((1u << first) - 1u));  // the group's place among those without a row
            const bool got = v < 0 && r < open;
            const int from = got ? (int)list[r] : 0;
            const int32_t nb = __shfl_sync(0xffffffffu, b0, from);
            const int32_t ne = __shfl_sync(0xffffffffu, e0, from);
            if (got) {
                v = base + from;
                k = nb;
                end = ne;
                m = INFINITY;
            }
            next = min(open, next + __popc(need));
        }
        if (__ballot_sync(0xffffffffu, v >= 0) == 0u) {
            if (tile >= ntiles) break;
            continue;
        }
        // one step of every group: G * kMpUnroll entries
        int32_t c[kMpUnroll];
        float x[kMpUnroll];
#pragma unroll
        for (int t = 0; t < kMpUnroll; ++t) {
            const int32_t o = sub + G * t;
            const bool in = v >= 0 && o < end - k;  // (a position past the row's end need not fit 32 bits)
            c[t] = in ? __ldg(a.pull_col + k + o) : -1;
            x[t] = in ? __ldg(a.pull_val + k + o) : INFINITY;
        }
#pragma unroll
        for (int t = 0; t < kMpUnroll; ++t)
            if (c[t] >= 0) m = fminf(m, x[t] + __ldg(a.u + c[t]));
        k = end - k > G * kMpUnroll ? k + G * kMpUnroll : end;
        const bool done = v >= 0 && k >= end;
        bool defer = v >= 0 && end - k > a.longest;
        if (kBlock && __any_sync(0xffffffffu, defer)) {  // to the block, as long as its list has room
            int slot = kMpLongs;
            if (defer && sub == 0) slot = atomicAdd(&lo.count, 1);
            slot = __shfl_sync(0xffffffffu, slot, first);
            defer = defer && slot < kMpLongs;
            if (defer && sub == 0) lo.row[slot] = make_int2(v, k);
        }
        if (!__any_sync(0xffffffffu, done || defer)) continue;
        float t = m;
        for (int o = 1; o < G; o <<= 1) t = fminf(t, __shfl_xor_sync(0xffffffffu, t, o));
        if ((done || defer) && sub == 0) {
            if (a.accum) t = fminf(t, a.w[v]);
            a.w[v] = t;
        }
        const uint32_t dm = kBlock ? 0u : __ballot_sync(0xffffffffu, defer && sub == 0);
        if (dm) {
            const uint32_t nch = defer && sub == 0 ? (uint32_t)(end - k + kMpChunk - 1) / kMpChunk : 0u;
            const uint32_t inc = warp_inclusive_sum(nch);
            const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
            unsigned long long old = 0ull;
            if (lane == 0)
                old = atomicAdd(a.huge, ((unsigned long long)tot << 32) | (unsigned long long)__popc(dm));
            old = __shfl_sync(0xffffffffu, old, 0);
            if (defer && sub == 0) {
                const uint32_t slot = (uint32_t)old + __popc(dm & lanemask_lt());
                a.q[1][slot] = v;
                a.qp[1][slot] = k;
                a.qd[1][slot] = (int32_t)((uint32_t)(old >> 32) + inc - nch);
            }
        }
        if (done || defer) v = -1;
    }
    if constexpr (!kBlock) return;
    // the block's long rows, one after another, its warps taking kMpChunk entries at a time
    __syncthreads();
    const int wib = threadIdx.x >> 5, count = min(lo.count, kMpLongs);
    for (int h = 0; h < count; ++h) {
        const int32_t row = lo.row[h].x, beg = lo.row[h].y, len = __ldg(a.pull_ptr + row + 1) - beg;
        float least = INFINITY;
        for (int32_t o = kMpChunk * wib; o < len; o += kMpChunk * (kMxvThreads / 32))
            least = fminf(least, mp_chunk(a, beg + o, len - o < kMpChunk ? len - o : kMpChunk));
        if (lane == 0) lo.part[wib] = least;
        __syncthreads();
        if (threadIdx.x == 0) {
            least = a.w[row];
#pragma unroll
            for (int x = 0; x < kMxvThreads / 32; ++x) least = fminf(least, lo.part[x]);
            a.w[row] = least;
        }
        __syncthreads();
    }
}

// Pull where every row has at most kMpShortRow entries and six on average: a lane per row.
// Handing such rows out to lanes (mp_pull) only costs: a pull of the 1001 x 777 grid 14.4 us, with
// a lane per row and one launch instead of three 7.5 (the launch itself).
constexpr int32_t kMpShortRow = 32;

__device__ __forceinline__ void mp_pull_short(const MpArgs& a) {
    for (int64_t i = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kMxvThreads) {
        float t = INFINITY;
        if (!mp_pull_pass(a, (int32_t)i)) {
            if (a.accum) continue;
        } else {
            const int32_t beg = __ldg(a.pull_ptr + i), len = __ldg(a.pull_ptr + i + 1) - beg;
            for (int32_t k = 0; k < len; k += kMpUnroll) {
                int32_t c[kMpUnroll];
                float x[kMpUnroll];
#pragma unroll
                for (int q = 0; q < kMpUnroll; ++q) {
                    c[q] = k + q < len ? __ldg(a.pull_col + beg + k + q) : -1;
                    x[q] = k + q < len ? __ldg(a.pull_val + beg + k + q) : INFINITY;
                }
#pragma unroll
                for (int q = 0; q < kMpUnroll; ++q)
                    if (c[q] >= 0) t = fminf(t, x[q] + __ldg(a.u + c[q]));
            }
            if (a.accum) t = fminf(t, a.w[i]);
        }
        a.w[i] = t;
    }
}

// Pull, push, or -- AUTO found u sparse -- the queue (and w = +inf) for mp_push_kernel.
template <bool kBlock>
__global__ void __launch_bounds__(kMxvThreads, 6) mp_main_kernel(const __grid_constant__ MpArgs a) {
    pdl_begin();
    __shared__ StageBuf sb[kMxvThreads / 32];
    __shared__ unsigned long long bsm[kMxvThreads / 32];
    __shared__ MpLong longs;
    if (mp_dir(a) == GBX_DIR_PULL) {
        if (a.shorts)
            mp_pull_short(a);
        else
            mp_pull<kBlock>(a, reinterpret_cast<uint8_t*>(sb + (threadIdx.x >> 5)), longs);
    } else if (a.dir == GBX_DIR_PUSH) {
        mp_push(a);
    } else {
        const int lane = threadIdx.x & 31;
        const int64_t gtid = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x, gs = (int64_t)gridDim.x * kMxvThreads;
        if (!a.accum)
            for (int64_t i = gtid; i < a.n; i += gs) a.w[i] = INFINITY;
        Acc acc;
        Stage st = mp_stage(a, sb, &acc);
        for (int64_t w0 = gtid - lane; w0 < a.nwords; w0 += gs) {
            const uint32_t mine = w0 + lane < a.nwords ? a.ubm[w0 + lane] : 0u;
            uint32_t todo = __ballot_sync(0xffffffffu, mine != 0u);
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                const uint32_t word = __shfl_sync(0xffffffffu, mine, j);
                st.put((word >> lane) & 1u, (int32_t)((w0 + j) << 5) + lane);
            }
        }
        st.flush_block<kMxvThreads / 32>(bsm);
    }
}

__global__ void __launch_bounds__(kMxvThreads) mp_push_kernel(const __grid_constant__ MpArgs a) {
    pdl_begin();
    if (mp_dir(a) == GBX_DIR_PUSH) mp_push(a);
}

// The chunks of the rows a pull deferred, and the scratch left zero for the next call.
__global__ void __launch_bounds__(kMxvThreads) mp_last_kernel(const __grid_constant__ MpArgs a) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t gtid = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x, gs = (int64_t)gridDim.x * kMxvThreads;
    const unsigned long long huge = *a.huge;
    const int32_t entries = (int32_t)(uint32_t)huge, chunks = (int32_t)(huge >> 32);
    for (int64_t c = gtid >> 5; c < chunks; c += gs >> 5) {
        const int32_t h = warp_find_entry(a.qd[1], entries, c);
        const int32_t v = a.q[1][h];
        const int32_t rend = __ldg(a.pull_ptr + v + 1);
        const int32_t beg = a.qp[1][h] + (int32_t)(c - a.qd[1][h]) * kMpChunk;
        const int32_t len = rend - beg < kMpChunk ? rend - beg : kMpChunk;
        const float m = mp_chunk(a, beg, len);
        if (lane == 0 && m < a.w[v]) atomic_min_f32(a.w + v, m);
    }
    if (a.dirty) {
        for (int64_t w = gtid; w < a.nwords; w += gs) {
            a.ubm[w] = 0u;
            if (a.mask.format >= 0) a.pass[w] = 0u;
        }
        if (gtid == 0) {
            a.ctr->q = 0ull;
            a.ctr->n_new = 0ull;
        }
        return;
    }
    // nothing clears the number before the next such call: the last block to have read it does
    if (huge == 0ull) return;
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&a.ctr->list, 1ull) == gridDim.x - 1) {
        *a.huge = 0ull;
        a.ctr->list = 0ull;
    }
}

gbx_status mxv_scratch(Graph* G, cudaStream_t s);

gbx_status mxv_minplus(Graph* G, float* w, const MxvVec& mask, const float* u, const gbx_desc& d, cudaStream_t s) {
    MpArgs a;
    a.n = G->n;
    a.nwords = G->nwords;
    a.mask = mask;
    a.invert = d.mask_complement ? 0xffffffffu : 0u;
    a.accum = d.accum ? 1 : 0;
    a.dir = d.direction;
    a.group = G->nnz > 12ll * G->n ? 8 : (G->nnz > 6ll * G->n ? 4 : 1);
    a.push_most = a.dir == GBX_DIR_AUTO ? mxv_push_most(G->n, d.alpha) : 0;
    a.u = u;
    a.w = w;
    a.pull_ptr = d.transpose ? G->in_ptr : G->out_ptr;
    a.pull_col = d.transpose ? G->in_col : G->out_col;
    a.pull_val = d.transpose ? G->in_val : G->out_val;
    a.push_ptr = d.transpose ? G->out_ptr : G->in_ptr;
    a.push_col = d.transpose ? G->out_col : G->in_col;
    a.push_val = d.transpose ? G->out_val : G->in_val;
    a.ubm = G->ws.mx_bm[0];
    a.pass = G->ws.mx_bm[1];
    a.ctr = G->ws.mx_ctr;
    for (int i = 0; i < 2; ++i) {
        a.q[i] = G->ws.q[i];
        a.qp[i] = G->ws.qp[i];
        a.qd[i] = G->ws.qd[i];
    }
    a.nothing = mask.format < 0 && d.mask_complement;
    const bool direct = a.dir == GBX_DIR_PULL && !a.nothing && mask.format != GBX_SPARSE;
    const int32_t longest = d.transpose ? G->max_in_degree : G->max_out_degree;
    a.bytes = direct && mask.format == GBX_DENSE ? static_cast<const uint8_t*>(mask.data) : nullptr;
    a.shorts = a.group == 1 && longest <= kMpShortRow;
    a.dirty = direct ? 0 : 1;
    a.huge = direct ? &G->ws.mx_ctr->mf_new : &G->ws.mx_ctr->huge;
    const unsigned full = (unsigned)G->num_sms * 6u;
    const long long lanes = (long long)full * kMxvThreads;
    if (!a.shorts)
        while (a.group < 32 && 4ll * a.group * a.n <= lanes) a.group *= 2;
    a.longest = kMpUnroll * a.group * (a.group == 32 ? kMpWarpSteps : kMpLongSteps);
    const bool block = direct && !a.shorts && longest <= kMpBlockRow && 4ll * a.n <= lanes;
    const bool deferring = !a.shorts && !block && longest > a.longest + kMpUnroll * a.group;
    // 5,000 vertices of 30 entries (157 warps of 32 rows): 18.5 us, with 4 rows a warp and one launch fewer 12.3
    a.rows = 32;
    while (a.rows * a.group > 32 && (long long)a.n * 2 < (long long)a.rows * full * (kMxvThreads / 32)) a.rows /= 2;
    const unsigned grid = direct ? std::min(full, div_up(a.n, (kMxvThreads / 32) * (a.shorts ? 32 : a.rows))) : full;
    const unsigned small = std::max(1u, std::min(div_up(a.n, kMxvThreads), (unsigned)G->num_sms * 4u));
    GBX_TRY(mxv_scratch(G, s));
    G->ws.mx_dirty = true;  // until every kernel of the call is issued
    if (!direct) GBX_TRY(pdl_launch(mp_prep_kernel, small, a, false, s));
    if (!a.nothing) {
        GBX_TRY(pdl_launch(block ? mp_main_kernel<true> : mp_main_kernel<false>, grid, a, !direct, s));
        if (a.dir == GBX_DIR_AUTO) GBX_TRY(pdl_launch(mp_push_kernel, grid, a, true, s));
    }
    if (!direct || deferring) GBX_TRY(pdl_launch(mp_last_kernel, small, a, true, s));
    G->ws.mx_dirty = false;
    return GBX_OK;
}

}  // namespace gbx
