// GrB_mxv over the Boolean semiring: the four matvec variants of Table 1.
//
//   row-based (pull, Eq 2 / Eq 4, Algorithm 2): a warp takes the rows of up to 32
//     result words that the mask test passes; each row ORs u over its
//     entries, stopping at the first hit when early exit is on (Section 5.3).
//   column-based (push, Eq 3 / Eq 5): the columns selected by u's nonzeros
//     are expanded with their edges split evenly over warps (exclusive prefix
//     of the selected columns' lengths); every hit that passes the mask sets
//     its bit in a result bitmap with atomicOr, which merges the columns
//     exactly (the multiway merge of Section 3.1, done by a bitmap instead of
//     the radix sort of Algorithm 3).
// The result bitmap is then written out as a dense byte vector or as a sorted
// index list (Section 3: sparse vectors are sorted lists).
//
// A call is three kernels, one more for a sparse result and one more where AUTO has to count a
// dense u before it can push: mxv_prep_kernel reads u and the mask into bitmaps, or u into a queue
// with its degree prefix; mxv_main_kernel pulls or pushes, by a decision each block takes
// from the count of u; the output kernels write w and leave the scratch bitmaps zero for the
// next call.  A small call is bound by its launches: the separate conversions, scans and
// decisions of 17 captured launches took 38 us for a sparse step of 100 vertices on RMAT-20
// (and a capture for every new set of buffers); now 14-16 us, launched directly (a first
// call on new buffers 154 -> 46 us).
#include <algorithm>

#include "frontier.cuh"
#include "gbx_internal.cuh"
#include "mxv.cuh"

namespace gbx {

constexpr int kMxvProbe = 16;

// Row-based matvec over the rows the mask lets through (Eq 2 / Eq 4).  A warp
// takes a tile of a.tile_words result words (at most 32: 1,024 rows) and lists the
// passing nonempty rows in shared memory (each lane its word's rows, at its prefix of
// the words' counts).  A fuller tile first tests every row's entry 0 from the dense
// first-entry array (one coalesced read instead of a random sector); then a lane takes
// a row at a time: entries 1..4 from the dense next-entries array (one 16-byte read),
// then up to kMxvProbe entries four at a time.  Longer rows are finished by the whole
// warp 128 entries at a time, and those with more than kMxvLongRow left by the whole
// block after its tiles.  With early exit a row stops at its first hit (Section 5.3); the
// result is the same either way.
//
// Bound by dependent gathers: RMAT-22 with half its rows masked and a fifth of its vertices in
// u reads 117 MB.  Rounds of 64 rows in lockstep took as long as their slowest row, 8 us longer;
// the call takes 51-55 us (107-109 in rounds, with 17 launches and tiles of 32 words).
//
// A tile's words lie ntiles apart, not side by side: the unvisited rows of a mesh are one band of
// the numbering, which would be the work of a few warps (the 2048 x 2048 grid's BFS levels pulled at
// 40, 60 and 80 % of the levels 61.5, 51 and 30 us, so 40, 25 and 17).  A warp then reads its words'
// masks from as many sectors, 1 us of the RMAT-22 call.  Pieces of 4 words side by side: 45, 29
// and 19, and the same 1 us.
constexpr int kMxvP1 = 4;  // first-pass rows per lane per round

// The rows of a tile whose bits are set in the lane words m (lane l: word l), in
// row order, as offsets in the tile, written at the lane's prefix excl.
__device__ __forceinline__ void mxv_tile_list(uint16_t* list, uint32_t m, uint32_t excl) {
    __syncwarp();
    const uint32_t rowbase = (threadIdx.x & 31) << 5;
    while (m) {
        const uint32_t b = __ffs(m) - 1;
        m &= m - 1;
        list[excl++] = (uint16_t)(rowbase + b);
    }
    __syncwarp();
}

// The block's deferred rows: its warps take 512-entry pieces of a row, four loads in flight a
// lane.  With early exit the pieces after a known hit are skipped.  exam counts the entries
// read (every lane adds its own).
__device__ __forceinline__ void mxv_long_rows(const PullArgs& a, PullSmem& sm, unsigned long long& exam) {
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int cnt = sm.nlong < kMxvLongs ? sm.nlong : kMxvLongs;
    for (int h = 0; h < cnt; ++h) {
        const int32_t i = sm.longs[h].x, beg = sm.longs[h].y, end = a.ptr[i + 1];
        if (threadIdx.x == 0) sm.hit = 0;
        __syncthreads();
        // (offsets from beg and entries left: positions past a row's end need not fit 32 bits)
        for (int64_t o = 512 * wib; o < end - beg; o += 512 * (kMxvThreads / 32)) {
            // the whole warp stops or goes on: another warp, or its own lane 0, may just be writing the word
            if (a.early_exit && __any_sync(0xffffffffu, *(volatile int*)&sm.hit)) break;
            const int32_t k0 = beg + (int32_t)o, len = end - k0 < 512 ? end - k0 : 512;
            for (int32_t kk = 0; kk < len; kk += 128) {
                int32_t j[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) j[q] = kk + 32 * q + lane < len ? a.col[k0 + kk + 32 * q + lane] : -1;
                bool hit = false;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    exam += j[q] >= 0 ? 1u : 0u;
                    hit |= j[q] >= 0 && bit_test(a.ubm, j[q]);
                }
                if (__any_sync(0xffffffffu, hit)) {
                    if (lane == 0) sm.hit = 1;
                    if (a.early_exit) break;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && sm.hit) atomicOr(a.R + (i >> 5), 1u << (i & 31));
        __syncthreads();
    }
}

__device__ __forceinline__ void mxv_pull(const PullArgs& a, PullSmem& sm) {
    const int32_t* __restrict__ ptr = a.ptr;
    const int32_t* __restrict__ col = a.col;
    const int32_t* __restrict__ first = a.first;
    const int4* __restrict__ next = a.next;
    const uint32_t* __restrict__ multi = a.multi;
    const uint32_t* __restrict__ ubm = a.ubm;
    const int32_t nwords = a.nwords, tw = a.tile_words;
    const int early_exit = a.early_exit;
    uint32_t* hits = sm.hits[threadIdx.x >> 5];
    uint16_t* list = sm.rows[threadIdx.x >> 5];
    if (threadIdx.x == 0) sm.nlong = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    const int32_t ntiles = (nwords + tw - 1) / tw;
    unsigned long long rows = 0, exam = 0;
    for (int32_t tile = gwarp; tile < ntiles; tile += nwarps) {
        const int32_t w = tile + lane * ntiles;
        // the row of an entry of the list
        auto row_at = [&](int off) { return ((tile + (off >> 5) * ntiles) << 5) + (off & 31); };
        const bool wok = lane < tw && w < nwords;
        const uint32_t cand0 = wok ? ((a.pass ? a.pass[w] ^ a.invert : 0xffffffffu) & a.nz[w]) : 0u;
        hits[lane] = 0u;
        __syncwarp();
        // a tile with more candidates than one round first tests every candidate's first entry
        // (the dense first-entry array: no row offsets loaded); the rest goes on with the rows it
        // left open that have more entries
        const uint32_t cnt0 = __popc(cand0);
        const uint32_t incl0 = warp_inclusive_sum(cnt0);
        const uint32_t total0 = __shfl_sync(0xffffffffu, incl0, 31);
        const bool two_pass = first != nullptr && total0 > 64u;
        if (two_pass) {
            mxv_tile_list(list, cand0, incl0 - cnt0);
            for (uint32_t base = 0; base < total0; base += 32 * kMxvP1) {
                int32_t off[kMxvP1], f0[kMxvP1];
#pragma unroll
                for (int r = 0; r < kMxvP1; ++r) {
                    const uint32_t c = base + 32 * r + lane;
                    off[r] = c < total0 ? (int)list[c] : -1;
                }
#pragma unroll
                for (int r = 0; r < kMxvP1; ++r) f0[r] = off[r] >= 0 ? first[row_at(off[r])] : -1;
#pragma unroll
                for (int r = 0; r < kMxvP1; ++r) {
                    if (off[r] < 0) continue;
                    rows += 1;
                    exam += 1;
                    if (bit_test(ubm, f0[r])) atomicOr(hits + (off[r] >> 5), 1u << (off[r] & 31));
                }
            }
            __syncwarp();
        }
        const uint32_t f1 = hits[lane];  // rows the first pass found
        const uint32_t cand =
            two_pass ? cand0 & (multi ? (wok ? multi[w] : 0u) : 0xffffffffu) & (early_exit ? ~f1 : 0xffffffffu) : cand0;
        const uint32_t cntw = __popc(cand);
        const uint32_t incl = warp_inclusive_sum(cntw);
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (total) mxv_tile_list(list, cand, incl - cntw);
        // a row per lane, each lane going on to the next one as soon as its row is settled
        uint32_t nxt = 0;  // rows of the list handed out
        int32_t i = -1, at = 0, beg = 0, end = 0, k = 0;  // row, its place in the tile
        bool found = false;
        for (;;) {
            const uint32_t need = __ballot_sync(0xffffffffu, i < 0);
            int32_t x[4] = {-1, -1, -1, -1}, f0 = -1;
            bool fresh = false;
            if (need != 0u && nxt < total) {
                const uint32_t c = nxt + __popc(need & lanemask_lt());
                fresh = i < 0 && c < total;
                const int off = fresh ? (int)list[c] : 0;
                const uint32_t f1j = __shfl_sync(0xffffffffu, f1, off >> 5);
                nxt += __popc(need);
                if (fresh) {
                    i = row_at(off);
                    at = off;
                    found = two_pass && ((f1j >> (off & 31)) & 1u);  // only without early exit can it be set here
                }
            }
            if (!__any_sync(0xffffffffu, i >= 0)) break;
            if (fresh) {
                beg = __ldg(ptr + i);
                end = __ldg(ptr + i + 1);
                if (next) {
                    const int4 nx = ld_stream(next + i);
                    x[0] = nx.x;
                    x[1] = nx.y;
                    x[2] = nx.z;
                    x[3] = nx.w;
                }
                k = beg + 1;
                if (!two_pass) {
                    rows += 1;
                    exam += 1;
                    f0 = first ? __ldg(first + i) : __ldg(col + beg);
                }
            }
            if (i >= 0 && !(fresh && next)) {
                const int32_t own = (end - beg < kMxvProbe ? end - beg : kMxvProbe) - (k - beg);  // left to the lane
#pragma unroll
                for (int t = 0; t < 4; ++t) x[t] = t < own ? ld_stream(col + k + t) : -1;
            }
            const bool hit0 = f0 >= 0 && bit_test(ubm, f0);
            bool h[4];
            int nv = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                h[t] = x[t] >= 0 && bit_test(ubm, x[t]);
                nv += x[t] >= 0 ? 1 : 0;
            }
            bool done = false;
            if (i >= 0) {
                found |= hit0;
                done = hit0 && early_exit;
                if (!done) {
                    const int hit = h[0] ? 0 : (h[1] ? 1 : (h[2] ? 2 : (h[3] ? 3 : -1)));
                    found |= hit >= 0;
                    done = hit >= 0 && early_exit;
                    const int used = done ? hit + 1 : nv;
                    exam += (unsigned long long)used;
                    k += used;
                }
                done |= k >= end;
            }
            // past the lane probe: the whole warp, or the whole block once its tiles are done
            const bool past = i >= 0 && !done && k - beg >= kMxvProbe;
            if (past && end - k > kMxvLongRow) {
                const int slot = atomicAdd(&sm.nlong, 1);
                if (slot < kMxvLongs) {
                    sm.longs[slot] = make_int2(i, k);
                    done = true;  // a found row keeps its bit
                }
            }
            uint32_t pend = __ballot_sync(0xffffffffu, past && !done);
            while (pend) {
                const int t = __ffs(pend) - 1;
                pend &= pend - 1;
                const int32_t kk = __shfl_sync(0xffffffffu, k, t);
                int32_t ahead = __shfl_sync(0xffffffffu, end, t) - kk;  // entries left
                bool tf = __shfl_sync(0xffffffffu, found, t);
                unsigned long long tx = 0;
                // 128 entries per round (four independent loads per lane)
                for (int64_t o = kk; ahead > 0; o += 128, ahead -= 128) {
                    int32_t jq[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) jq[q] = 32 * q + lane < ahead ? col[o + 32 * q + lane] : -1;
                    bool stop = false;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (stop) break;
                        const uint32_t hb = __ballot_sync(0xffffffffu, jq[q] >= 0 && bit_test(ubm, jq[q]));
                        const int32_t left = ahead - 32 * q;
                        if (left <= 0) break;
                        if (hb) {
                            tf = true;
                            if (early_exit) {
                                tx += (unsigned long long)__ffs(hb);
                                stop = true;
                                break;
                            }
                        }
                        tx += (unsigned long long)(left < 32 ? left : 32);
                    }
                    if (stop) break;
                }
                if (lane == t) {
                    found = tf;
                    exam += tx;
                    done = true;
                }
            }
            if (done) {
                if (found) atomicOr(hits + (at >> 5), 1u << (at & 31));
                i = -1;
            }
        }
        __syncwarp();
        if (wok) a.R[w] = a.accum ? a.R[w] | hits[lane] : hits[lane];
        __syncwarp();
    }
    mxv_long_rows(a, sm, exam);
    if (a.stats) {
        rows = warp_sum_u64(rows);
        exam = warp_sum_u64(exam);
        if (lane == 0) {
            if (rows) atomicAdd(&a.stats->rows, rows);
            if (exam) atomicAdd(&a.stats->exam, exam);
        }
    }
}


__global__ void __launch_bounds__(kMxvThreads, 4) mxv_pull_kernel(PullArgs a) {
    __shared__ PullSmem sm;
    mxv_pull(a, sm);
}

// ---------------------------------------------------------------- one call's arguments

struct MxvArgs {
    int32_t n, nwords;
    MxvVec u, mask, w;
    uint32_t invert;  // the mask's complement: all ones
    int32_t accum, dir, early_exit;
    int32_t push_most;  // nonzeros of u up to which AUTO pushes
    PullArgs pull;
    const int32_t* push_ptr;
    const int32_t* push_col;
    // scratch, zero between calls: u, mask and result bitmaps; ctr->q: the push queue's length
    // and edges, ctr->n_new: nonzeros of a dense u
    uint32_t* ubm;
    uint32_t* pass;
    uint32_t* R;
    LevelCtr* ctr;
    int32_t* q;
    int32_t* qp;
    int32_t* qd;
    int32_t* sums;  // set bits of each block's words (sparse result)
    int32_t per;    // words per thread of the sparse result's kernels
    int32_t nothing;  // no row passes
    MxvStats* stats;
};

__device__ __forceinline__ int mxv_dir(const MxvArgs& a) {
    if (a.dir != GBX_DIR_AUTO) return a.dir;
    const int32_t c = a.u.format == GBX_SPARSE ? *a.u.count : (int32_t)a.ctr->n_new;
    return c <= a.push_most ? GBX_DIR_PUSH : GBX_DIR_PULL;
}

// A queue of the columns a push expands: vertex, exclusive prefix of the columns' lengths, column
// start minus prefix (frontier.cuh); empty columns are left out.
__device__ __forceinline__ Stage mxv_stage(const MxvArgs& a, StageBuf* sb, Acc* acc) {
    return Stage{sb + (threadIdx.x >> 5), 0, a.ctr, a.q, a.qp, a.qd, a.push_ptr, a.push_ptr, 0, 0, acc};
}

// Stages the set bits of the warp's 32 words (lane l holds word w0 + l); all lanes call.
__device__ __forceinline__ void mxv_stage_words(Stage& st, uint32_t mine, int32_t w0) {
    const int lane = threadIdx.x & 31;
    uint32_t todo = __ballot_sync(0xffffffffu, mine != 0u);
    while (todo) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t word = __shfl_sync(0xffffffffu, mine, k);
        st.put((word >> lane) & 1u, ((w0 + k) << 5) + lane);
    }
}

__global__ void __launch_bounds__(kMxvThreads) mxv_prep_kernel(const __grid_constant__ MxvArgs a) {
    pdl_begin();
    __shared__ StageBuf sb[kMxvThreads / 32];
    __shared__ unsigned long long bsm[kMxvThreads / 32];
    __shared__ unsigned long long csm[kMxvThreads / 32][4];
    const int lane = threadIdx.x & 31;
    const int64_t gtid = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x, gs = (int64_t)gridDim.x * kMxvThreads;
    if (a.stats && gtid == 0) *a.stats = MxvStats{};
    const bool u_sparse = a.u.format == GBX_SPARSE;
    // a dense u under AUTO is counted here and decided by the next kernel
    const int dir = u_sparse || a.dir != GBX_DIR_AUTO ? mxv_dir(a) : GBX_DIR_AUTO;
    Acc acc;
    Stage st = mxv_stage(a, sb, &acc);
    uint32_t cnt = 0;
    if (!u_sparse || a.mask.format == GBX_DENSE) {
        for (int64_t w0 = gtid - lane; w0 < a.nwords; w0 += gs) {  // warp-uniform
            const int32_t w = (int32_t)w0 + lane;
            const bool ok = w < a.nwords;
            if (a.mask.format == GBX_DENSE && ok)
                a.pass[w] = pack_word(static_cast<const uint8_t*>(a.mask.data), a.n, w);
            if (u_sparse) continue;
            const uint32_t word = ok ? pack_word(static_cast<const uint8_t*>(a.u.data), a.n, w) : 0u;
            if (dir == GBX_DIR_PUSH) {
                mxv_stage_words(st, word, (int32_t)w0);
            } else if (ok) {
                a.ubm[w] = word;
            }
            cnt += (uint32_t)__popc(word);
        }
    }
    if (u_sparse) {
        const int32_t* list = static_cast<const int32_t*>(a.u.data);
        const int32_t count = min(min(*a.u.count, a.u.cap), a.n);
        for (int64_t b = gtid - lane; b < count; b += gs) {  // entries outside [0, n) expand nothing
            const int32_t v = b + lane < count ? list[b + lane] : -1;
            const bool ok = v >= 0 && v < a.n;
            if (dir == GBX_DIR_PUSH)
                st.put(ok, v);
            else if (ok)
                atomicOr(a.ubm + (v >> 5), 1u << (v & 31));
        }
    }
    if (a.mask.format == GBX_SPARSE) {
        const int32_t* list = static_cast<const int32_t*>(a.mask.data);
        const int32_t count = min(*a.mask.count, a.mask.cap);
        for (int64_t i = gtid; i < count; i += gs) {
            const int32_t v = list[i];
            if (v >= 0 && v < a.n) atomicOr(a.pass + (v >> 5), 1u << (v & 31));
        }
    }
    if (a.accum && a.w.format == GBX_SPARSE) {  // the result keeps w's entries
        const int32_t* list = static_cast<const int32_t*>(a.w.data);
        const int32_t count = min(*a.w.count, a.w.cap);
        for (int64_t i = gtid; i < count; i += gs) {
            const int32_t v = list[i];
            if (v >= 0 && v < a.n) atomicOr(a.R + (v >> 5), 1u << (v & 31));
        }
    }
    if (dir == GBX_DIR_PUSH) st.flush_block<kMxvThreads / 32>(bsm);
    block_add_counts<kMxvThreads / 32>(csm, cnt, 0ull, 0ull, 0ull, &a.ctr->n_new, nullptr, nullptr, nullptr);
}

// The queue's edges, evenly over all warps, kMxvPushIlp per lane in flight: a target that
// passes the mask sets its bit (a reduction) unless the L1-cached word already has it.
constexpr int kMxvPushIlp = 4;

__device__ __forceinline__ void mxv_push(const MxvArgs& a) {
    const unsigned long long qv = a.ctr->q;
    const uint32_t qcount = (uint32_t)qv;
    const int32_t E = (int32_t)(qv >> 32);
    const int gwarp = (int)((blockIdx.x * kMxvThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMxvThreads) >> 5);
    if (a.stats && blockIdx.x == 0 && threadIdx.x == 0) {
        a.stats->ucount = a.u.format == GBX_SPARSE ? (unsigned long long)max(0, min(*a.u.count, a.n)) : a.ctr->n_new;
        a.stats->edges = (unsigned long long)E;
    }
    constexpr int kStep = 32 * kMxvPushIlp;
    int32_t chunk = (int32_t)(((long long)E + nwarps - 1) / nwarps);
    chunk = chunk <= 32 ? 32 : ((chunk + kStep - 1) / kStep) * kStep;
    for (long long e0l = (long long)gwarp * chunk; e0l < E; e0l += (long long)nwarps * chunk) {
        const int32_t e0 = (int32_t)e0l;
        const int32_t e1 = E - e0 > chunk ? e0 + chunk : E;
        PushCursorT<kMxvPushIlp> cur;
        cur.k = warp_find_entry(a.qp, (int32_t)qcount, e0);
        cur.wlast = -1;
        for (int32_t base = e0; base < e1; base += kStep) {
            const PushStepT<kMxvPushIlp> ps = cur.gather(a.push_col, a.q, a.qp, a.qd, qcount, base, e1);
            uint32_t p[kMxvPushIlp], r[kMxvPushIlp];
#pragma unroll
            for (int t = 0; t < kMxvPushIlp; ++t) {
                p[t] = ps.u[t] >= 0 ? (a.mask.format >= 0 ? a.pass[ps.v[t] >> 5] ^ a.invert : 0xffffffffu) : 0u;
                r[t] = ps.u[t] >= 0 ? __ldca(a.R + (ps.v[t] >> 5)) : 0xffffffffu;
            }
#pragma unroll
            for (int t = 0; t < kMxvPushIlp; ++t)
                if (((p[t] & ~r[t]) >> (ps.v[t] & 31)) & 1u) atomicOr(a.R + (ps.v[t] >> 5), 1u << (ps.v[t] & 31));
        }
    }
}

// Pull, push, or -- a dense u that AUTO found sparse -- the queue for mxv_push_kernel.
__global__ void __launch_bounds__(kMxvThreads, 4) mxv_main_kernel(const __grid_constant__ MxvArgs a) {
    pdl_begin();
    union MainSmem {
        PullSmem pull;
        StageBuf sb[kMxvThreads / 32];
    };
    __shared__ MainSmem sm;
    __shared__ unsigned long long bsm[kMxvThreads / 32];
    if (mxv_dir(a) == GBX_DIR_PULL) {
        mxv_pull(a.pull, sm.pull);
    } else if (a.u.format == GBX_SPARSE || a.dir == GBX_DIR_PUSH) {
        mxv_push(a);
    } else {
        Acc acc;
        Stage st = mxv_stage(a, sm.sb, &acc);
        const int lane = threadIdx.x & 31;
        const int64_t gtid = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x, gs = (int64_t)gridDim.x * kMxvThreads;
        for (int64_t w0 = gtid - lane; w0 < a.nwords; w0 += gs)
            mxv_stage_words(st, w0 + lane < a.nwords ? a.ubm[w0 + lane] : 0u, (int32_t)w0);
        st.flush_block<kMxvThreads / 32>(bsm);
    }
}

__global__ void __launch_bounds__(kMxvThreads) mxv_push_kernel(const __grid_constant__ MxvArgs a) {
    pdl_begin();
    if (mxv_dir(a) == GBX_DIR_PUSH) mxv_push(a);
}

// ---------------------------------------------------------------- output

// Leaves word w of the scratch bitmaps zero for the next call and returns the result's.
__device__ __forceinline__ uint32_t mxv_take_word(const MxvArgs& a, int32_t w) {
    const uint32_t word = a.R[w];
    if (word) a.R[w] = 0u;
    a.ubm[w] = 0u;
    if (a.mask.format >= 0) a.pass[w] = 0u;
    return word;
}

// One thread per word writes its 32 bytes (two 16-byte stores where w is aligned), ORing in the
// old values when accumulating.
__global__ void __launch_bounds__(kMxvThreads) mxv_dense_kernel(const __grid_constant__ MxvArgs a) {
    pdl_begin();
    uint8_t* out = static_cast<uint8_t*>(const_cast<void*>(a.w.data));
    const bool vec = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctr->q = 0ull;
        a.ctr->n_new = 0ull;
    }
    for (int64_t w = (int64_t)blockIdx.x * kMxvThreads + threadIdx.x; w < a.nwords; w += (int64_t)gridDim.x * kMxvThreads) {
        const uint32_t word = mxv_take_word(a, (int32_t)w);
        const int64_t base = w << 5;
        if (vec && base + 32 <= a.n) {
            uint32_t v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = (((word >> (4 * q)) & 0xfu) * 0x00204081u) & 0x01010101u;
            if (a.accum) {
                const uint4 x = reinterpret_cast<const uint4*>(out + base)[0];
                const uint4 y = reinterpret_cast<const uint4*>(out + base)[1];
                const uint32_t o[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int t = 0; t < 4; ++t) v[q] |= (((o[q] >> (8 * t)) & 0xffu) != 0u ? 1u : 0u) << (8 * t);
            }
            reinterpret_cast<uint4*>(out + base)[0] = make_uint4(v[0], v[1], v[2], v[3]);
            reinterpret_cast<uint4*>(out + base)[1] = make_uint4(v[4], v[5], v[6], v[7]);
        } else {
            for (int t = 0; t < 32 && base + t < a.n; ++t) {
                uint8_t x = (uint8_t)((word >> t) & 1u);
                if (a.accum) x |= out[base + t] != 0 ? 1 : 0;
                out[base + t] = x;
            }
        }
    }
}

// Set bits of each block's words (a.per consecutive words a thread).
__global__ void __launch_bounds__(kMxvThreads) mxv_count_kernel(const __grid_constant__ MxvArgs a) {
    pdl_begin();
    __shared__ int32_t part[kMxvThreads / 32];
    const int64_t w0 = ((int64_t)blockIdx.x * kMxvThreads + threadIdx.x) * a.per;
    uint32_t c = 0;
    for (int k = 0; k < a.per; ++k) c += w0 + k < a.nwords ? (uint32_t)__popc(a.R[w0 + k]) : 0u;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = (int32_t)c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t s = 0;
#pragma unroll
        for (int k = 0; k < kMxvThreads / 32; ++k) s += part[k];
        a.sums[blockIdx.x] = s;
    }
}

// The sorted list of the set bits: a block's place is the sum of the blocks before it.
__global__ void __launch_bounds__(kMxvThreads) mxv_list_kernel(const __grid_constant__ MxvArgs a) {
    pdl_begin();
    __shared__ uint32_t part[2][kMxvThreads / 32];
    int32_t* out = static_cast<int32_t*>(const_cast<void*>(a.w.data));
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t before = 0;
    for (int32_t b = threadIdx.x; b < (int32_t)blockIdx.x; b += kMxvThreads) before += (uint32_t)a.sums[b];
    const int64_t w0 = ((int64_t)blockIdx.x * kMxvThreads + threadIdx.x) * a.per;
    uint32_t c = 0;
    for (int k = 0; k < a.per; ++k) c += w0 + k < a.nwords ? (uint32_t)__popc(a.R[w0 + k]) : 0u;
    const uint32_t inc = warp_inclusive_sum(c);
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 31) part[0][wib] = inc;
    if (lane == 0) part[1][wib] = before;
    __syncthreads();
    uint32_t at = inc - c;
#pragma unroll
    for (int k = 0; k < kMxvThreads / 32; ++k) at += part[1][k] + (k < wib ? part[0][k] : 0u);
    for (int k = 0; k < a.per && w0 + k < a.nwords; ++k) {
        uint32_t word = mxv_take_word(a, (int32_t)(w0 + k));
        for (; word; word &= word - 1) out[at++] = (int32_t)((w0 + k) << 5) + __ffs(word) - 1;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kMxvThreads - 1) {
        *const_cast<int32_t*>(a.w.count) = (int32_t)at;
        a.ctr->q = 0ull;
        a.ctr->n_new = 0ull;
    }
}

// ---------------------------------------------------------------- host side

__global__ void zero_stats_kernel(MxvStats* s) {
    MxvStats z = {};
    *s = z;
}

__global__ void set_push_stats_kernel(MxvStats* s, int32_t ucount, int64_t edges) {
    s->ucount = (unsigned long long)ucount;
    s->edges = (unsigned long long)edges;
}

static gbx_status check_vec(const gbx_vector* v, int32_t n, const char* name, bool output) {
    GBX_CHECK(v->format == GBX_DENSE || v->format == GBX_SPARSE || v->format == GBX_DENSE_F32, GBX_ERR_INVALID_VALUE,
              std::string(name) + ": unknown format");
    GBX_CHECK(v->size == n, GBX_ERR_DIMENSION_MISMATCH, std::string(name) + ": size differs from the graph's n");
    GBX_CHECK(v->data != nullptr, GBX_ERR_NULL_POINTER, std::string(name) + ": data is NULL");
    if (v->format == GBX_SPARSE) {
        GBX_CHECK(v->nnz != nullptr, GBX_ERR_NULL_POINTER, std::string(name) + ": nnz is NULL");
        GBX_CHECK(v->capacity >= 0, GBX_ERR_INVALID_VALUE, std::string(name) + ": capacity < 0");
        if (output)
            GBX_CHECK(v->capacity >= v->size, GBX_ERR_INVALID_VALUE,
                      std::string(name) + ": a sparse output needs capacity >= size");
    }
    return GBX_OK;
}

// desc.push_sort: Algorithm 3 on the host's decision (mxv_push_sorted); *done: w is written, else
// the call pulls.
static gbx_status mxv_sorted(Graph* G, gbx_vector* w, const gbx_vector* mask, const gbx_vector* u, const gbx_desc& d,
                             cudaStream_t s, bool* done) {
    const int32_t n = G->n;
    *done = false;
    if (d.direction == GBX_DIR_PULL || (!mask && d.mask_complement)) return GBX_OK;
    const int32_t* ulist = (const int32_t*)u->data;
    const int32_t* ucount = u->nnz;
    int32_t ucap = u->capacity < n ? u->capacity : n;
    uint32_t* ubm = G->ws.bm[0];
    uint32_t* pass = mask ? G->ws.bm[1] : nullptr;
    uint32_t* R = G->ws.bm[2];
    if (u->format == GBX_DENSE) {
        GBX_TRY(pack_dense_to_bitmap((const uint8_t*)u->data, n, 0, ubm, s));
        GBX_TRY(bitmap_to_list(ubm, n, G->ws.list, G->ws.flag + 0, G->ws.qd[0], G->ws.scan_tmp, s));
        ulist = G->ws.list;
        ucount = G->ws.flag + 0;
        ucap = n;
    }
    if (mask && mask->format == GBX_DENSE) {
        GBX_TRY(pack_dense_to_bitmap((const uint8_t*)mask->data, n, d.mask_complement ? 1u : 0u, pass, s));
    } else if (mask) {
        GBX_TRY(fill_bitmap(pass, n, 0u, s));
        GBX_TRY(scatter_list_to_bitmap((const int32_t*)mask->data, mask->nnz, mask->capacity, n, pass, s));
        if (d.mask_complement) GBX_TRY(invert_bitmap(pass, n, s));
    }
    int32_t hc = 0;
    GBX_CUDA_TRY(cudaMemcpyAsync(&hc, ucount, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    GBX_CUDA_TRY(cudaStreamSynchronize(s));
    if (d.direction == GBX_DIR_AUTO && !((double)hc / (double)n <= (double)d.alpha)) return GBX_OK;
    const int32_t count = hc < 0 ? 0 : (hc > n ? n : hc);
    const bool direct = w->format == GBX_SPARSE && !d.accum;  // the sorted list is w itself
    if (!direct) GBX_TRY(fill_bitmap(R, n, 0u, s));
    int64_t edges = 0;
    GBX_TRY(mxv_push_sorted(G, d.transpose ? G->out_ptr : G->in_ptr, d.transpose ? G->out_col : G->in_col, ulist, count,
                            ucap, pass, direct ? nullptr : R, direct ? (int32_t*)w->data : nullptr,
                            direct ? w->nnz : nullptr, &edges, s));
    if (d.trace) {
        MxvStats* stats = reinterpret_cast<MxvStats*>(G->ws.ctr + 3);
        zero_stats_kernel<<<1, 1, 0, s>>>(stats);
        set_push_stats_kernel<<<1, 1, 0, s>>>(stats, count, edges);
    }
    if (!direct && w->format == GBX_DENSE) {
        GBX_TRY(bitmap_to_dense(R, n, d.accum ? (const uint8_t*)w->data : nullptr, (uint8_t*)w->data, s));
    } else if (!direct) {
        GBX_TRY(scatter_list_to_bitmap((const int32_t*)w->data, w->nnz, w->capacity, n, R, s));
        GBX_TRY(bitmap_to_list(R, n, (int32_t*)w->data, w->nnz, G->ws.qd[1], G->ws.scan_tmp, s));
    }
    GBX_CUDA_TRY(cudaGetLastError());
    G->ws.last_stream = s;
    *done = true;
    return GBX_OK;
}

static MxvVec mxv_vec(const gbx_vector* v) {
    if (!v) return MxvVec{-1, nullptr, nullptr, 0};
    return MxvVec{v->format, v->data, v->nnz, v->capacity};
}

// Zeroes the call scratch after a call that could not be issued whole (the output kernels leave it zero).
gbx_status mxv_scratch(Graph* G, cudaStream_t s) {
    if (!G->ws.mx_dirty) return GBX_OK;
    GBX_CUDA_TRY(cudaMemsetAsync(G->ws.mx_bm[0], 0, sizeof(uint32_t) * 3 * ((size_t)G->nwords + 1), s));
    GBX_CUDA_TRY(cudaMemsetAsync(G->ws.mx_ctr, 0, sizeof(LevelCtr), s));
    return GBX_OK;
}

static gbx_status mxv_bool(Graph* G, gbx_vector* w, const gbx_vector* mask, const gbx_vector* u, const gbx_desc& d,
                           cudaStream_t s) {
    // w = A' u with A' = A^T (transpose) or A.  Pull reads rows of A' (CSR of A'),
    // push reads the columns of A' selected by u, i.e. rows of (A')^T.
    MxvArgs a;
    a.n = G->n;
    a.nwords = G->nwords;
    a.u = mxv_vec(u);
    a.mask = mxv_vec(mask);
    a.w = mxv_vec(w);
    a.invert = d.mask_complement ? 0xffffffffu : 0u;
    a.accum = d.accum ? 1 : 0;
    a.dir = d.direction;
    a.push_most = a.dir == GBX_DIR_AUTO ? mxv_push_most(G->n, d.alpha) : 0;
    a.early_exit = d.early_exit ? 1 : 0;
    a.stats = d.trace ? reinterpret_cast<MxvStats*>(G->ws.ctr + 3) : nullptr;
    a.push_ptr = d.transpose ? G->out_ptr : G->in_ptr;
    a.push_col = d.transpose ? G->out_col : G->in_col;
    a.ubm = G->ws.mx_bm[0];
    a.pass = G->ws.mx_bm[1];
    a.R = G->ws.mx_bm[2];
    a.ctr = G->ws.mx_ctr;
    a.q = G->ws.q[0];
    a.qp = G->ws.qp[0];
    a.qd = G->ws.qd[0];
    a.sums = G->ws.scan_tmp;
    a.nothing = !mask && d.mask_complement;
    const unsigned main_blocks = (unsigned)G->num_sms * 4u;
    PullArgs& p = a.pull;
    p.ptr = d.transpose ? G->in_ptr : G->out_ptr;
    p.col = d.transpose ? G->in_col : G->out_col;
    p.first = d.transpose ? G->first_in : G->first_out;
    p.next = d.transpose ? G->next_in : G->next_out;
    p.nz = d.transpose ? G->nz_in : G->nz_out;
    p.multi = d.transpose ? G->multi_in : G->multi_out;
    p.ubm = a.ubm;
    p.pass = mask ? a.pass : nullptr;
    p.invert = a.invert;
    p.R = a.R;
    p.accum = a.accum && w->format == GBX_SPARSE ? 1 : 0;
    p.nwords = a.nwords;
    p.tile_words = mxv_tile_words(a.nwords, (long long)main_blocks * (kMxvThreads / 32));
    p.early_exit = a.early_exit;
    p.stats = a.stats;
    if (!(G->l1_set & 1024u)) {
        GBX_TRY(prefer_l1((const void*)mxv_main_kernel, 4));
        G->l1_set |= 1024u;
    }
    GBX_TRY(mxv_scratch(G, s));
    G->ws.mx_dirty = true;  // until every kernel of the call is issued
    const int32_t most = std::max(std::max(a.nwords, u->format == GBX_SPARSE ? std::min(u->capacity, G->n) : 0),
                                  std::max(mask && mask->format == GBX_SPARSE ? std::min(mask->capacity, G->n) : 0,
                                           p.accum ? G->n : 0));
    const unsigned prep_blocks = std::max(1u, std::min(div_up(most, kMxvThreads), (unsigned)G->num_sms * 4u));
    GBX_TRY(pdl_launch(mxv_prep_kernel, prep_blocks, a, false, s));
    if (!a.nothing) {
        GBX_TRY(pdl_launch(mxv_main_kernel, main_blocks, a, true, s));
        if (u->format == GBX_DENSE && a.dir == GBX_DIR_AUTO)
            GBX_TRY(pdl_launch(mxv_push_kernel, main_blocks, a, true, s));
    }
    if (w->format == GBX_DENSE) {
        const unsigned blocks = std::max(1u, std::min(div_up(a.nwords, kMxvThreads), (unsigned)G->num_sms * 16u));
        GBX_TRY(pdl_launch(mxv_dense_kernel, blocks, a, true, s));
    } else {
        a.per = std::max(4, (int)(((int64_t)a.nwords + kMxvThreads * 4096ll - 1) / (kMxvThreads * 4096ll)));
        const unsigned blocks = div_up(a.nwords, (int64_t)kMxvThreads * a.per);
        GBX_TRY(pdl_launch(mxv_count_kernel, blocks, a, true, s));
        GBX_TRY(pdl_launch(mxv_list_kernel, blocks, a, true, s));
    }
    G->ws.mx_dirty = false;
    G->ws.last_stream = s;
    return GBX_OK;
}

gbx_status mxv_minplus(Graph* G, float* w, const MxvVec& mask, const float* u, const gbx_desc& d, cudaStream_t s);

}  // namespace gbx

using namespace gbx;

extern "C" gbx_status gbx_mxv(gbx_vector* w, const gbx_vector* mask, int32_t semiring, const gbx_graph* A,
                              const gbx_vector* u, const gbx_desc* desc, void* stream) {
    clear_error();
    GBX_TRY(check_graph(A));
    GBX_CHECK(w != nullptr && u != nullptr, GBX_ERR_NULL_POINTER, "w or u is NULL");
    GBX_CHECK(semiring == GBX_LOR_LAND || semiring == GBX_MIN_PLUS_F32, GBX_ERR_NOT_SUPPORTED,
              "semiring must be GBX_LOR_LAND or GBX_MIN_PLUS_F32");
    Graph* G = const_cast<Graph*>(as_impl(A));
    const int32_t n = G->n;
    GBX_TRY(check_vec(u, n, "u", false));
    GBX_TRY(check_vec(w, n, "w", true));
    if (mask) GBX_TRY(check_vec(mask, n, "mask", false));
    GBX_CHECK(w->data != u->data && (!mask || w->data != mask->data), GBX_ERR_INVALID_VALUE,
              "w must not alias u or mask");
    gbx_desc d;
    if (desc)
        d = *desc;
    else
        gbx_desc_init(&d);
    GBX_CHECK(d.direction >= GBX_DIR_AUTO && d.direction <= GBX_DIR_PULL, GBX_ERR_INVALID_VALUE, "desc.direction");
    GBX_CHECK(d.alpha >= 0.0f && d.alpha == d.alpha, GBX_ERR_INVALID_VALUE, "desc.alpha must be >= 0");
    GBX_CHECK(d.push_sort == 0 || d.push_sort == 1, GBX_ERR_INVALID_VALUE, "desc.push_sort must be 0 or 1");
    for (int k = 0; k < 2; ++k) GBX_CHECK(d.reserved[k] == 0, GBX_ERR_INVALID_VALUE, "desc.reserved must be 0");
    GBX_CHECK(!mask || mask->format != GBX_DENSE_F32, GBX_ERR_INVALID_VALUE, "mask: GBX_DENSE or GBX_SPARSE");
    if (semiring == GBX_MIN_PLUS_F32) {
        GBX_CHECK(u->format == GBX_DENSE_F32 && w->format == GBX_DENSE_F32, GBX_ERR_INVALID_VALUE,
                  "the (min, +) semiring takes GBX_DENSE_F32 u and w");
        GBX_CHECK(d.push_sort == 0, GBX_ERR_NOT_SUPPORTED, "desc.push_sort is for the Boolean semiring");
        GBX_CHECK(G->out_val != nullptr, GBX_ERR_INVALID_VALUE,
                  "the (min, +) semiring needs edge weights (gbx_graph_set_weights)");
    } else {
        GBX_CHECK(u->format != GBX_DENSE_F32 && w->format != GBX_DENSE_F32, GBX_ERR_INVALID_VALUE,
                  "GBX_DENSE_F32 vectors belong to the (min, +) semiring");
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (semiring == GBX_MIN_PLUS_F32) {
        GBX_TRY(mxv_minplus(G, (float*)w->data, mxv_vec(mask), (const float*)u->data, d, s));
        G->ws.last_stream = s;
        return GBX_OK;
    }
    if (d.push_sort) {
        bool done = false;
        GBX_TRY(mxv_sorted(G, w, mask, u, d, s, &done));
        if (done) return GBX_OK;
        d.direction = GBX_DIR_PULL;
    }
    return mxv_bool(G, w, mask, u, d, s);
}

extern "C" gbx_status gbx_mxv_stats(const gbx_graph* A, int64_t* rows, int64_t* examined, int64_t* u_nnz,
                                    int64_t* edges) {
    clear_error();
    GBX_TRY(check_graph(A));
    const Graph* G = as_impl(A);
    if (G->ws.last_stream) GBX_CUDA_TRY(cudaStreamSynchronize(G->ws.last_stream));
    MxvStats st;
    GBX_CUDA_TRY(cudaMemcpy(&st, G->ws.ctr + 3, sizeof(st), cudaMemcpyDeviceToHost));
    if (rows) *rows = (int64_t)st.rows;
    if (examined) *examined = (int64_t)st.exam;
    if (u_nnz) *u_nnz = (int64_t)st.ucount;
    if (edges) *edges = (int64_t)st.edges;
    return GBX_OK;
}
