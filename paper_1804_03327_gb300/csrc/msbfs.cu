// Batched multi-source BFS: S sources at once as bit lanes (Algorithm 1 run for
// S frontier vectors together), with the Boolean semiring acting lane-wise on
// uint64 words (OR = bitwise OR, AND = bitwise AND).  Lane b of vertex v is
// bit b % 64 of word b / 64 of v's W-word row.
//
// State (vertex-major, W words per vertex, W padded to a multiple of the chunk):
//   V[v]      lanes in which v has been visited,
//   F_k[v]    lanes in which v was found at level L (k = L mod 3): level L reads
//             F_{L mod 3} of its active list, writes F_{(L+1) mod 3}, and clears
//             F_{(L+2) mod 3} for the list of level L - 1 (read one level earlier,
//             written again one level later), so no extra barrier is needed;
//   D         one bit per vertex: every lane visited (pull skips it without loads);
//   T_k       one bit per vertex: listed for level L + 1 (W > 1), rotating like F.
// Each level runs in the direction chosen for the whole batch:
//   push (Eq 5 lane-wise): the active list's edges are split evenly over warps.
//     One word per vertex (S <= 64): each edge claims the lanes F[u] & ~V[v] with a
//     64-bit atomicOr on V[v]; the lanes it gained are new (unique claimant): their
//     depth is written, they are ORed into F_next[v], and the first claimant of v
//     lists it -- one phase.  Wider batches: each edge ORs F[u] & ~V[v] into
//     F_next[v] with reductions and lists v once; after a grid barrier a finalising
//     pass over the touched vertices keeps new = F_next & ~V, sets V |= new and
//     writes the depths (one returning atomic per word and edge would cost more).
//   pull (Eq 4 lane-wise, masking + early exit + operand reuse): every vertex with
//     an unvisited lane ORs V of its in-neighbours (V is the state before this
//     level) and stops as soon as every unvisited lane is covered; new = acc & ~V.
//     Long rows are deferred and spread over the whole grid.
// New lanes get depth L + 1.  Depths are not stored as they are found (2-byte
// stores scattered over S rows leave partial sectors that are evicted and merged
// again level after level): a depth below 16 is recorded as bits in four per-vertex
// planes of lane words (plane p holds bit p), larger ones are stored at once, and
// after the last level one pass emits every other entry of the S rows exactly once,
// coalesced along the vertices (-1 where a lane never arrived).
#include <algorithm>
#include <cmath>

#include "frontier.cuh"
#include "gbx_internal.cuh"

namespace gbx {

constexpr int kMsThreads = 512;
// Register budgets of the persistent batched kernel: the default build fits two
// 512-thread blocks on an SM (64 registers a thread: twice the resident warps of an
// unbounded build at 114, for 24-222 bytes of spills), the lean build three (40
// registers, more spills; lane words 1 and 2 only).  Lean pays on graphs with few
// wide levels and loses on long chains of small ones (a grid), so a descriptor
// chooses it (blocks_per_sm >= 3) and the autotuner times both.
constexpr int kMsOcc = 2;
constexpr int kMsOccLean = 3;
constexpr int kMsProbe = 8;  // default a.probe; with two words and more a long row is deferred after four times as many
constexpr int kMsPlanes = 4;  // depth bit planes: bit p of depths below 16

struct MsArgs {
    int32_t n, S, W, nwords;
    long long nnz;
    const int32_t* out_ptr;
    const int32_t* out_col;
    const int32_t* in_ptr;
    const int32_t* in_col;
    const uint32_t* nz_in;
    const int32_t* first_in;
    const int4* next_in;
    unsigned long long* V;
    unsigned long long* Fb[3];  // rotating found-lane buffers
    unsigned long long* P[4];   // depth bit planes (see record_depth)
    uint32_t* D;                // all lanes visited
    uint32_t* Tb[3];            // rotating "listed" bitmaps
    int32_t* tlist;             // vertices touched by a wide push level
    void* depth;        // [S][n], used when rows is NULL
    void* const* rows;  // optional: lane b writes its n depths to rows[b]
    int depth16;
    const int32_t* src;
    int32_t* ids[3];  // active lists, rotating like Fb
    int32_t* qp[2];
    int32_t* qd[2];
    LevelCtr* ctr;
    GridBar* bar;
    unsigned int bar_parity;
    LevelRec* trace;
    int32_t* status;
    uint32_t push_most;  // active edges up to which AUTO pushes: floor(alpha * nnz)
    int32_t mode, trace_cap, symmetric, probe;
    // kMesh: every level pushes, and a vertex may be listed more than once: lists 0 and 1 alternate (ids[0]
    // and ids[1], from entry more_from on more[]), as do Fb[0] and Fb[1]
    int32_t never_pull;
    uint32_t more_from;
    int32_t* more[2];
    int32_t group;  // warp lanes that hold a vertex's words (a power of two)
    int32_t team;   // warp lanes per row of a pull (ms_pull_few); 0: ms_pull
    unsigned long long timeout_ns;
};

__device__ __forceinline__ unsigned long long lane_mask(int32_t S, int32_t w) {
    const int32_t lo = w * 64;
    if (lo + 64 <= S) return ~0ull;
    if (lo >= S) return 0ull;
    return (1ull << (S - lo)) - 1ull;
}

__device__ __forceinline__ void store_depth(const MsArgs& a, int32_t lane_b, int32_t v, int32_t d) {
    if (a.rows) {
        if (a.depth16)
            static_cast<int16_t*>(a.rows[lane_b])[v] = (int16_t)d;
        else
            static_cast<int32_t*>(a.rows[lane_b])[v] = d;
        return;
    }
    const size_t idx = (size_t)lane_b * (size_t)a.n + (size_t)v;
    if (a.depth16)
        static_cast<int16_t*>(a.depth)[idx] = (int16_t)d;
    else
        static_cast<int32_t*>(a.depth)[idx] = d;
}

// Records depth d for the lanes nw of word w of vertex v.  Depths below 16 go to
// the bit planes (atomically when several edges may record lanes of one word in the
// same level, as the one-phase push does); larger ones are stored now.  A visited
// lane with no plane bit is either its own source (depth 0) or such a deep one,
// which the emission pass tells apart by the source.
__device__ __forceinline__ void record_depth(const MsArgs& a, int32_t v, int32_t w, unsigned long long nw, int32_t d,
                                             bool atomic) {
    if (!nw) return;
    if (d < 16) {
        const size_t iv = (size_t)v * a.W + w;
#pragma unroll
        for (int p = 0; p < kMsPlanes; ++p) {
            if (!((d >> p) & 1)) continue;
            if (atomic)
                atomicOr(a.P[p] + iv, nw);
            else
                a.P[p][iv] |= nw;
        }
        return;
    }
    unsigned long long m = nw;
    while (m) {
        const int b = __ffsll((long long)m) - 1;
        m &= m - 1;
        store_depth(a, w * 64 + b, v, d);
    }
}

// After the last level: every (lane, vertex) entry of the output rows, once.  A warp
// takes 128 consecutive vertices and 32 rows (half a lane word), four vertices a lane,
// and each row's 128 entries leave together: four entries of a lane are one 8- or
// 16-byte store where the rows allow it (aligned, a full group), else four stores whose
// 32 lanes are consecutive.  Lanes never visited get -1; lanes found at depth 16 or more
// were stored when found and are left alone (emit_rows).
//
// Bound by the stores: S rows of n entries, written once, many rows at a time.  With 32
// vertices a warp (one 64- or 128-byte piece of a row per store, ten instructions an
// entry) the RMAT-20 batch of 1,000 int16 rows spent 2.0 ms here and the RMAT-21 batch of
// 64 int32 rows 0.25 ms; now 0.8 and 0.14 ms, of which 0.31 and 0.08 are the rows' 2.1 and
// 0.54 GB at the measured copy rate.
constexpr int kEmitV = 4;               // vertices a lane
constexpr int kEmitTile = 32 * kEmitV;  // vertices a warp

// Bits 0..3 of x as the low bits of bytes 0..3.
__device__ __forceinline__ uint32_t spread4(uint32_t x) { return ((x & 0xfu) * 0x00204081u) & 0x01010101u; }

// Byte-wise selection of (lo, hi) with sign replication (selector bit 3 of a nibble).
__device__ __forceinline__ uint32_t prmt_sext(uint32_t lo, uint32_t hi, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(sel));
    return r;
}

// The address of entry 0 of output row b.
__device__ __forceinline__ char* depth_row(const MsArgs& a, int32_t b) {
    if (a.rows) return static_cast<char*>(a.rows[b]);
    return static_cast<char*>(a.depth) + (size_t)b * (size_t)a.n * (a.depth16 ? 2u : 4u);
}

// Rows [b0, b1) of half word h for 32 consecutive vertices, a lane each: entry by entry, a row's
// 32 entries per store.  Lanes found at depth 16 or more were stored when found.
__device__ __noinline__ void emit_rows(const MsArgs& a, int32_t v, int32_t h, int b0, int b1) {
    if (v >= a.n) return;
    const size_t iw = (size_t)v * a.W * 2 + h;
    const uint32_t vis = reinterpret_cast<const uint32_t*>(a.V)[iw];
    uint32_t p[kMsPlanes];
#pragma unroll
    for (int q = 0; q < kMsPlanes; ++q) p[q] = reinterpret_cast<const uint32_t*>(a.P[q])[iw];
    for (int b = b0; b < b1; ++b) {
        int32_t d = -1;
        if ((vis >> b) & 1u) {
            d = (int32_t)(((p[0] >> b) & 1u) | (((p[1] >> b) & 1u) << 1) | (((p[2] >> b) & 1u) << 2) |
                          (((p[3] >> b) & 1u) << 3));
            if (d == 0 && __ldg(a.src + 32 * h + b) != v) continue;  // deep: already stored
        }
        store_depth(a, 32 * h + b, v, d);
    }
}

// One half word of a group: the lane's visited and plane bits of vertices v + stride * j.
struct EmitBits {
    uint32_t vis[kEmitV], p[kMsPlanes][kEmitV];
};

// Writes the rows of one half word (rows 32 h + lane's row address in `row`).
__device__ __forceinline__ void emit_half(const MsArgs& a, const EmitBits& e, char* row, int nrows, int32_t v,
                                          bool wide) {
    for (int b = 0; b < nrows; b += 4) {
        // byte r of d[j]: depth of (row b + r, vertex j), 0xff where it was never visited
        uint32_t d[kEmitV];
#pragma unroll
        for (int j = 0; j < kEmitV; ++j)
            d[j] = (spread4(e.p[0][j] >> b) | (spread4(e.p[1][j] >> b) << 1) | (spread4(e.p[2][j] >> b) << 2) |
                    (spread4(e.p[3][j] >> b) << 3)) |
                   ~(spread4(e.vis[j] >> b) * 0xffu);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            char* const rp = reinterpret_cast<char*>(
                __shfl_sync(0xffffffffu, (unsigned long long)reinterpret_cast<uintptr_t>(row), b + r));
            if (b + r >= nrows) continue;
            if (a.depth16) {
                const uint32_t sel = 0xc480u + 0x1111u * r;  // bytes r, sign of r, 4 + r, its sign
                const uint32_t lo = prmt_sext(d[0], d[1], sel), hi = prmt_sext(d[2], d[3], sel);
                int16_t* const o = reinterpret_cast<int16_t*>(rp) + v;
                if (wide) {
                    *reinterpret_cast<uint2*>(o) = make_uint2(lo, hi);
                } else {
                    if (v < a.n) o[0] = (int16_t)lo;
                    if (v + 32 < a.n) o[32] = (int16_t)(lo >> 16);
                    if (v + 64 < a.n) o[64] = (int16_t)hi;
                    if (v + 96 < a.n) o[96] = (int16_t)(hi >> 16);
                }
            } else {
                const uint32_t sel = 0x8880u + 0x1111u * r;  // byte r, its sign three times
                int32_t* const o = reinterpret_cast<int32_t*>(rp) + v;
                const int32_t x0 = (int32_t)prmt_sext(d[0], 0u, sel), x1 = (int32_t)prmt_sext(d[1], 0u, sel);
                const int32_t x2 = (int32_t)prmt_sext(d[2], 0u, sel), x3 = (int32_t)prmt_sext(d[3], 0u, sel);
                if (wide) {
                    *reinterpret_cast<int4*>(o) = make_int4(x0, x1, x2, x3);
                } else {
                    if (v < a.n) o[0] = x0;
                    if (v + 32 < a.n) o[32] = x1;
                    if (v + 64 < a.n) o[64] = x2;
                    if (v + 96 < a.n) o[96] = x3;
                }
            }
        }
    }
}

// W >= 4: the block stages 128 vertices x 8 words of V and the planes in shared memory
// (16-byte loads, 64 consecutive bytes a vertex), one array of 128 32-bit halves per half
// word, and each of its 16 warps writes the rows of one half.  Loading a half straight
// from the vertex-major words would touch 32 lines with every load (stride 8 W bytes).
constexpr int kEmitWords = 8;
constexpr int kEmitPad = kEmitTile + 2;  // staging writes 8 vertices x 4 halves: distinct banks
constexpr int kEmitSmem = (1 + kMsPlanes) * 2 * kEmitWords * kEmitPad * 4;  // bytes
static_assert(kMsThreads / 32 == 2 * kEmitWords, "one warp per half word of the staged tile");

// smem: kEmitSmem bytes (16-byte aligned), used by the block from here on.
template <bool kStaged>
__device__ __forceinline__ void emit_depths(const MsArgs& a, uint32_t* smem) {
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int32_t ngroups = (a.n + kEmitTile - 1) / kEmitTile;
    const int32_t nhalf = (a.S + 31) >> 5;  // half words holding real lanes
    const uint32_t esz = a.depth16 ? 2u : 4u;
    // staged: a block takes a tile of 16 halves; else a warp takes one half
    const int32_t per = kStaged ? 2 * kEmitWords : 1;
    const int32_t ntile = (nhalf + per - 1) / per;
    const long long items = (long long)ngroups * ntile;
    const long long nwarps = ((long long)gridDim.x * kMsThreads) >> 5;
    if ((long long)ngroups * nhalf < nwarps) {
        // fewer pieces than warps: 32 vertices and as few rows as keep every warp busy, at least 4 (1,000
        // vertices, what a batch takes beside its levels: 20 sources 40 -> 25 us, 100 sources 56 -> 25)
        const int32_t nv = (a.n + 31) >> 5;
        int rows = 32;
        while (rows > 4 && (long long)nv * nhalf * (64 / rows) <= nwarps) rows >>= 1;
        const int32_t parts = 32 / rows;
        for (long long it = (long long)wib * gridDim.x + blockIdx.x; it < (long long)nv * nhalf * parts; it += nwarps) {
            const int32_t r = (int32_t)(it % parts), i = (int32_t)(it / parts), h = i % nhalf;
            const int b1 = a.S - 32 * h < (r + 1) * rows ? a.S - 32 * h : (r + 1) * rows;
            emit_rows(a, 32 * (i / nhalf) + lane, h, r * rows, b1);
        }
        return;
    }
    const long long first = kStaged ? blockIdx.x : (((long long)blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const long long nstep = kStaged ? gridDim.x : nwarps;
    for (long long it = first; it < items; it += nstep) {
        const int32_t g = (int32_t)(it / ntile);
        const int32_t h0 = (int32_t)(it - (long long)g * ntile) * per;
        if (kStaged) {
            __syncthreads();  // the last tile has been read
            const int32_t w0 = h0 >> 1;
            for (int i = threadIdx.x; i < (1 + kMsPlanes) * kEmitTile * (kEmitWords / 2); i += kMsThreads) {
                const int q = i / (kEmitTile * (kEmitWords / 2)), r = i - q * (kEmitTile * (kEmitWords / 2));
                const int vl = r / (kEmitWords / 2), c = r - vl * (kEmitWords / 2);  // vertex, pair of words
                const int32_t v = g * kEmitTile + vl, w = w0 + 2 * c;
                uint4 x = make_uint4(0u, 0u, 0u, 0u);
                if (v < a.n && w < a.W)
                    x = *reinterpret_cast<const uint4*>((q == 0 ? a.V : a.P[q - 1]) + (size_t)v * a.W + w);
                uint32_t* const o = smem + (q * 2 * kEmitWords + 4 * c) * kEmitPad + vl;
                o[0] = x.x;
                o[kEmitPad] = x.y;
                o[2 * kEmitPad] = x.z;
                o[3 * kEmitPad] = x.w;
            }
            __syncthreads();
        }
        const int32_t h = kStaged ? h0 + wib : h0;
        if (h >= nhalf) continue;
        const int nrows = a.S - 32 * h < 32 ? a.S - 32 * h : 32;
        char* const row = depth_row(a, 32 * h + (lane < nrows ? lane : 0));  // lane r: row 32 h + r
        const bool wide = __all_sync(0xffffffffu, (reinterpret_cast<uintptr_t>(row) & (kEmitV * esz - 1)) == 0) &&
                          (long long)(g + 1) * kEmitTile <= a.n;
        const int32_t stride = wide ? 1 : 32, vl = wide ? kEmitV * lane : lane;
        const int32_t v = g * kEmitTile + vl;
        EmitBits e;
        uint32_t deep = 0u;
#pragma unroll
        for (int j = 0; j < kEmitV; ++j) {
            const int32_t vj = v + stride * j;
            if (kStaged) {
                const uint32_t* const sp = smem + wib * kEmitPad + vl + stride * j;
                e.vis[j] = sp[0];
#pragma unroll
                for (int q = 0; q < kMsPlanes; ++q) e.p[q][j] = sp[(q + 1) * 2 * kEmitWords * kEmitPad];
            } else {
                const size_t iw = (size_t)(vj < a.n ? vj : 0) * a.W * 2 + h;  // 32-bit half of the word
                e.vis[j] = vj < a.n ? reinterpret_cast<const uint32_t*>(a.V)[iw] : 0u;
#pragma unroll
                for (int q = 0; q < kMsPlanes; ++q)
                    e.p[q][j] = vj < a.n ? reinterpret_cast<const uint32_t*>(a.P[q])[iw] : 0u;
            }
            deep |= e.vis[j] & ~(e.p[0][j] | e.p[1][j] | e.p[2][j] | e.p[3][j]);
        }
        if (__any_sync(0xffffffffu, deep != 0u))  // or a lane's own source
            for (int j = 0; j < kEmitV; ++j) emit_rows(a, g * kEmitTile + 32 * j + lane, h, 0, nrows);
        else
            emit_half(a, e, row, nrows, v, wide);
    }
}

// ---------------------------------------------------------------- lane-word groups

// A vertex's W lane words are handled by a group of a.group consecutive warp lanes,
// WL words a lane (one 8- or 16-byte access): W = 1 is one lane and one word, W = 16
// eight lanes whose 16-byte loads make one 128-byte line per vertex.  W above 64 goes
// through the group in chunks of 64 words.
template <int WL>
struct Words {
    unsigned long long x[WL];
    __device__ __forceinline__ bool any() const {
        unsigned long long o = 0ull;
#pragma unroll
        for (int j = 0; j < WL; ++j) o |= x[j];
        return o != 0ull;
    }
};

template <int WL>
__device__ __forceinline__ Words<WL> ld_words(const unsigned long long* p) {
    Words<WL> r;
    if (WL == 2) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
        r.x[0] = t.x;
        r.x[WL - 1] = t.y;
    } else {
        r.x[0] = *p;
    }
    return r;
}

template <int WL>
__device__ __forceinline__ void st_words(unsigned long long* p, const Words<WL>& w) {
    if (WL == 2)
        *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(w.x[0], w.x[WL - 1]);
    else
        *p = w.x[0];
}

template <int WL>
__device__ __forceinline__ Words<WL> zero_words() {
    Words<WL> r;
#pragma unroll
    for (int j = 0; j < WL; ++j) r.x[j] = 0ull;
    return r;
}

// The calling lane's place in its group.
struct Group {
    int size, sub, first;  // lanes, this lane's index, warp lane of index 0
    uint32_t mask;         // the group's lanes
    __device__ __forceinline__ explicit Group(int n) {
        const int lane = threadIdx.x & 31;
        size = n;
        sub = lane & (n - 1);
        first = lane & ~(n - 1);
        mask = (n == 32 ? 0xffffffffu : (1u << n) - 1u) << first;
    }
    __device__ __forceinline__ bool any(bool p) const { return (__ballot_sync(0xffffffffu, p) & mask) != 0u; }
    __device__ __forceinline__ bool all(bool p) const { return (__ballot_sync(0xffffffffu, p) & mask) == mask; }
};

// Records depth d for this lane's new words nw of vertex v (one writer per word); was: its
// words of V before.  With two words a lane the planes are not zeroed at the start: the
// first lanes found in a word write all four of its plane words.
template <int WL>
__device__ __forceinline__ void record_words(const MsArgs& a, int32_t v, int32_t w, const Words<WL>& nw,
                                             const Words<WL>& was, int32_t d) {
    if (!nw.any()) return;
    const size_t iv = (size_t)v * a.W + w;
    if (WL == 2) {
        const bool fresh = (nw.x[0] && !was.x[0]) || (nw.x[WL - 1] && !was.x[WL - 1]);
        const int32_t bits = d < 16 ? d : 0;
#pragma unroll
        for (int p = 0; p < kMsPlanes; ++p) {
            const bool set = (bits >> p) & 1;
            if (!set && !fresh) continue;
            Words<WL> t = was.any() ? ld_words<WL>(a.P[p] + iv) : zero_words<WL>();
#pragma unroll
            for (int j = 0; j < WL; ++j) t.x[j] = (was.x[j] ? t.x[j] : 0ull) | (set ? nw.x[j] : 0ull);
            st_words<WL>(a.P[p] + iv, t);
        }
        if (d < 16) return;
    }
#pragma unroll
    for (int j = 0; j < WL; ++j) record_depth(a, v, w + j, nw.x[j], d, false);
}

// ---------------------------------------------------------------- pull level

constexpr int kMsUnroll = 4;        // in-neighbours a group ORs per step (loads in flight)
constexpr int32_t kMsLongRow = 64;   // in-edges left after the probe beyond which a row is deferred
// Steps of a whole warp on a row before it is deferred, with one word (128 in-neighbours a step):
// a deferred row costs two more grid barriers and the chain of its chunks, 11 us.  RMAT graphs of
// 300,000, 600,000 and 2M vertices (20, 20 and 64 sources): 170, 276 and 725 us with 8 steps, 161, 285
// and 726 with 16.
constexpr int kMsScan = 16;
constexpr int32_t kMsChunk = 512;   // in-edges of a deferred row a warp takes at a time
constexpr int32_t kMsCheck = 128;   // ... between two tests whether they cover the row (a power of two)

// Rows of a pull level left to the grid: vertex, first in-edge left, ascending prefix
// of their chunk counts.
struct MsLong {
    int32_t* row;
    int32_t* k;
    int32_t* base;
};

// Leaves the rows v of the lanes with `take`, from in-edge k on (left of them), to the grid; all lanes call.
__device__ __forceinline__ void ms_defer(const MsLong& lr, bool take, int32_t v, int32_t k, int32_t left,
                                         LevelCtr* cout) {
    const uint32_t dm = __ballot_sync(0xffffffffu, take);
    const uint32_t nch = take ? (uint32_t)(left - 1) / kMsChunk + 1u : 0u;
    const uint32_t inc = warp_inclusive_sum(nch);
    const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
    unsigned long long old = 0ull;
    if ((threadIdx.x & 31) == 0)
        old = atomicAdd(&cout->huge, ((unsigned long long)tot << 32) | (unsigned long long)__popc(dm));
    old = __shfl_sync(0xffffffffu, old, 0);
    if (take) {
        const uint32_t slot = (uint32_t)old + __popc(dm & lanemask_lt());
        lr.row[slot] = v;
        lr.k[slot] = k;
        lr.base[slot] = (int32_t)((uint32_t)(old >> 32) + inc - nch);
    }
}

// A row of a pull level is settled: the lane's new words nw of vertex v (unv: the lanes v missed
// before).  F_next is zero before the level: only words with new lanes are written.
template <int WL>
__device__ __forceinline__ void ms_settle(const MsArgs& a, int32_t L, int32_t v, int32_t w, bool sink,
                                          const Words<WL>& nw, const Words<WL>& unv, const Words<WL>& lm,
                                          unsigned long long* Fn, Acc& acc) {
    if (!nw.any()) return;
    const size_t iv = (size_t)v * a.W + w;
    if (sink) {
        // nobody's in-neighbour: no other row reads its V, and it never joins the active list
        Words<WL> t = ld_words<WL>(a.V + iv);
#pragma unroll
        for (int j = 0; j < WL; ++j) t.x[j] |= nw.x[j];
        st_words<WL>(a.V + iv, t);
    } else {
        st_words<WL>(Fn + iv, nw);
    }
    Words<WL> was;
#pragma unroll
    for (int j = 0; j < WL; ++j) {
        acc.n_new += (uint32_t)__popcll(nw.x[j]);
        was.x[j] = ~unv.x[j] & lm.x[j];
    }
    record_words<WL>(a, v, w, nw, was, L + 1);
}

// Two words and more: every vertex with an unvisited lane ORs V of its in-neighbours (V as of
// the level's start), kMsUnroll at a time, until all its unvisited lanes are covered.  A warp
// lists the open vertices of 32 of its bitmap words in shared memory and its groups take them
// one after another, each going on to the next as soon as its own is settled, so a long
// row holds up nobody else's.  A row that is still open after 4 a.probe in-neighbours with
// more than kMsLongRow left is deferred: its chunks are spread over all warps
// (ms_pull_long) and it is settled after that (ms_finalize).
//
// Bound by the gathers of V (W words per examined in-neighbour, mostly L2).  A lane per
// row with its V words in 32-byte chunks, and one warp for a long row, had made the first
// pull level of the RMAT-20 batch of 1,000 sources 7.1 ms: every gather touched 32 rows at
// once and a hub row held one warp for milliseconds.  Now 0.76 ms (31.4M in-neighbours x
// 128 B, 5.3 TB/s).  kMsLongRow 64, 128 and 512 give that level 0.76, 0.78 and 1.0 ms;
// kMsChunk 256 instead of 512 cost the RMAT-21 batch of 64 6 % (more of a row's chunks run before
// one covers it).
template <int WL>
__device__ __forceinline__ void ms_pull(const MsArgs& a, int32_t L, int32_t c0, unsigned long long* Fn, uint32_t* Tn,
                                        uint16_t* list, const MsLong& lr, bool defer, Stage& st,
                                        unsigned long long* bsm, Acc& acc) {
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)((blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMsThreads) >> 5);
    const Group gr(a.group);
    const int32_t w = c0 + WL * gr.sub;
    const bool wok = w < a.W;
    const bool one = a.W <= WL * gr.size;  // one chunk: a row is settled in one go
    const uint32_t chunks256 = (uint32_t)(a.W + 3) >> 2;
    Words<WL> lm;
#pragma unroll
    for (int j = 0; j < WL; ++j) lm.x[j] = wok ? lane_mask(a.S, w + j) : 0ull;
    const int32_t own = 4 * a.probe;
    for (long long wb = gwarp; wb < a.nwords; wb += 32ll * nwarps) {
        const long long tw = wb + (long long)lane * nwarps;
        const uint32_t m = tw < a.nwords ? (a.nz_in[tw] & ~a.D[tw]) : 0u;
        const uint32_t cnt = __popc(m);
        const uint32_t incl = warp_inclusive_sum(cnt);
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (total == 0u) continue;
        __syncwarp();
        // a word's rows at a time, a lane per row (a warp has a few words only on all but huge graphs)
        for (uint32_t wm = __ballot_sync(0xffffffffu, m != 0u); wm; wm &= wm - 1) {
            const int j = __ffs(wm) - 1;
            const uint32_t word = __shfl_sync(0xffffffffu, m, j), at = __shfl_sync(0xffffffffu, incl - cnt, j);
            if ((word >> lane) & 1u) list[at + __popc(word & lanemask_lt())] = (uint16_t)((j << 5) + lane);
        }
        __syncwarp();
        uint32_t next = 0;
        int32_t v = -1, k = 0, end = 0, lim = 0;
        int32_t u[kMsUnroll] = {-1, -1, -1, -1};  // the in-neighbours of this step; the next step's are loaded meanwhile
        bool sink = false;
        Words<WL> unv = zero_words<WL>(), ac = zero_words<WL>();
        for (;;) {
            const uint32_t need = __ballot_sync(0xffffffffu, v < 0 && gr.sub == 0);
            if (need) {
                const uint32_t idx = next + __popc(need & ((1u << gr.first) - 1u));
                if (v < 0 && idx < total) {
                    const uint32_t off = list[idx];
                    v = (int32_t)((wb + (long long)(off >> 5) * nwarps) << 5) + (int32_t)(off & 31u);
                    k = __ldg(a.in_ptr + v);
                    end = __ldg(a.in_ptr + v + 1);
                    lim = end - k > own + kMsLongRow ? k + own : end;
                    sink = !a.symmetric && __ldg(a.out_ptr + v + 1) == __ldg(a.out_ptr + v);
                    unv = wok ? ld_words<WL>(a.V + (size_t)v * a.W + w) : zero_words<WL>();
#pragma unroll
                    for (int j = 0; j < WL; ++j) {
                        unv.x[j] = ~unv.x[j] & lm.x[j];
                        ac.x[j] = 0ull;
                    }
#pragma unroll
                    for (int t = 0; t < kMsUnroll; ++t) u[t] = t < end - k ? __ldg(a.in_col + k + t) : -1;
                }
                next += __popc(need);
            }
            if (__ballot_sync(0xffffffffu, v >= 0) == 0u) break;
            Words<WL> x[kMsUnroll];
#pragma unroll
            for (int t = 0; t < kMsUnroll; ++t)
                x[t] = u[t] >= 0 && wok ? ld_words<WL>(a.V + (size_t)u[t] * a.W + w) : zero_words<WL>();
            const int32_t left = end - k;
            k = left > kMsUnroll ? k + kMsUnroll : end;
#pragma unroll
            for (int t = 0; t < kMsUnroll; ++t) u[t] = v >= 0 && t < end - k ? __ldg(a.in_col + k + t) : -1;
            bool cov = true;
#pragma unroll
            for (int j = 0; j < WL; ++j) {
#pragma unroll
                for (int t = 0; t < kMsUnroll; ++t) ac.x[j] |= x[t].x[j];
                cov &= (ac.x[j] & unv.x[j]) == unv.x[j];
            }
            const bool covered = gr.all(cov);
            if (v >= 0 && gr.sub == 0) acc.exam += chunks256 * (uint32_t)(left < kMsUnroll ? left : kMsUnroll);
            const bool done = v >= 0 && (covered || k >= end);
            const bool put_off = defer && v >= 0 && !done && k >= lim && lim != end;
            if (!__any_sync(0xffffffffu, done || put_off)) continue;
            Words<WL> nw;
#pragma unroll
            for (int j = 0; j < WL; ++j) nw.x[j] = done || put_off ? ac.x[j] & unv.x[j] : 0ull;
            const bool any_new = gr.any(nw.any());
            const bool full = gr.all(!done || (nw.x[0] == unv.x[0] && nw.x[WL - 1] == unv.x[WL - 1]));
            if (done)
                ms_settle<WL>(a, L, v, w, sink, nw, unv, lm, Fn, acc);
            else if (nw.any())
                st_words<WL>(Fn + (size_t)v * a.W + w, nw);
            bool take = done && gr.sub == 0 && any_new && !sink;
            if (done && sink && full && one && gr.sub == 0) atomicOr(a.D + (v >> 5), 1u << (v & 31));
            if (!one && take) take = !(atomicOr(Tn + (v >> 5), 1u << (v & 31)) & (1u << (v & 31)));
            st.put(take, v);
            if (__any_sync(0xffffffffu, put_off)) ms_defer(lr, put_off && gr.sub == 0, v, k, end - k, st.cout);
            if (done || put_off) v = -1;
        }
    }
    st.flush_block<kMsThreads / 32>(bsm);
}

// The pull with one word: a lane per row of the warp's bitmap word, the first five in-neighbours
// from the dense arrays, then up to a.probe more, four at a time, or all if kMsOwnRow more end the
// row; the rows still open are taken by the whole warp one after another, kMsScan steps each, and
// what is open then is deferred.  Rows of a mesh (kMesh: at most kMsMeshDegree entries) are left
// to their lanes.
//
// Bound by its instructions where the rows are short: handing rows out to lanes as ms_pull does took
// 710M instructions and 1.85 ms for the 46 x 46 x 46 grid and 64 sources, so 1.32 ms; the first pull
// level of an RMAT graph of 300,000 vertices and 20 sources 68 us, so 39.  Without kMsOwnRow a
// random graph of 100,000 vertices and 16 edges each 193 us, with 16 or 24 152.
constexpr int32_t kMsOwnRow = 24;

template <bool kMesh>
__device__ __forceinline__ void ms_pull_one(const MsArgs& a, int32_t L, unsigned long long* Fn, const MsLong& lr,
                                            Stage& st, unsigned long long* bsm, Acc& acc) {
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)((blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMsThreads) >> 5);
    const unsigned long long full0 = lane_mask(a.S, 0);
    for (int32_t tile = gwarp; tile < a.nwords; tile += nwarps) {
        const uint32_t m = a.nz_in[tile] & ~a.D[tile];
        if (m == 0u) continue;
        const int32_t v = (tile << 5) + lane;
        unsigned long long ac = 0ull, unv = 0ull;
        int32_t beg = 0, left = 0, k = 0;  // the row: where it starts, its length, in-neighbours looked at
        bool sink = false;
        if ((m >> lane) & 1u) {
            const int4 x = __ldg(a.next_in + v);
            const int32_t u[5] = {__ldg(a.first_in + v), x.x, x.y, x.z, x.w};
            beg = __ldg(a.in_ptr + v);
            left = __ldg(a.in_ptr + v + 1) - beg;
            if (!kMesh) sink = !a.symmetric && __ldg(a.out_ptr + v + 1) == __ldg(a.out_ptr + v);
            unv = ~a.V[v] & full0;
#pragma unroll
            for (int t = 0; t < 5; ++t) ac |= u[t] >= 0 ? a.V[u[t]] : 0ull;
            const int32_t lim = kMesh || left <= 5 + a.probe + kMsOwnRow ? left : 5 + a.probe;
            for (k = 5; k < lim && (ac & unv) != unv; k += kMsUnroll) {
                int32_t y[kMsUnroll];
#pragma unroll
                for (int t = 0; t < kMsUnroll; ++t) y[t] = k + t < left ? __ldg(a.in_col + beg + k + t) : -1;
#pragma unroll
                for (int t = 0; t < kMsUnroll; ++t) ac |= y[t] >= 0 ? a.V[y[t]] : 0ull;
            }
            k = min(k, left);
            acc.exam += (uint32_t)k;
        }
        bool open = !kMesh && k < left && (ac & unv) != unv;
        if (!kMesh) {
            for (uint32_t pm = __ballot_sync(0xffffffffu, open); pm; pm &= pm - 1) {
                const int t0 = __ffs(pm) - 1;
                const int32_t kt = __shfl_sync(0xffffffffu, beg + k, t0), lt = __shfl_sync(0xffffffffu, left - k, t0);
                const unsigned long long ut = __shfl_sync(0xffffffffu, unv, t0);
                unsigned long long at = __shfl_sync(0xffffffffu, ac, t0);
                const int32_t len = lt > kMsScan * 32 * kMsUnroll ? kMsScan * 32 * kMsUnroll : lt;
                int32_t o = 0;
                for (; o < len && (at & ut) != ut; o += 32 * kMsUnroll) {
                    int32_t y[kMsUnroll];
#pragma unroll
                    for (int t = 0; t < kMsUnroll; ++t)
                        y[t] = o + 32 * t + lane < len ? __ldg(a.in_col + kt + o + 32 * t + lane) : -1;
                    unsigned long long z = 0ull;
#pragma unroll
                    for (int t = 0; t < kMsUnroll; ++t) z |= y[t] >= 0 ? a.V[y[t]] : 0ull;
                    at |= ((unsigned long long)__reduce_or_sync(0xffffffffu, (uint32_t)(z >> 32)) << 32) |
                          __reduce_or_sync(0xffffffffu, (uint32_t)z);
                }
                if (lane == t0) {
                    ac = at;
                    acc.exam += (uint32_t)min(o, len);
                    k += min(o, lt);
                    open = k < left && (ac & unv) != unv;
                }
            }
        }
        const unsigned long long nw = ac & unv;
        if (nw) {
            if (sink && !open)  // nobody's in-neighbour: no other row reads its V, and it never joins the active list
                a.V[v] |= nw;
            else
                Fn[v] = nw;  // zero before the level
            if (!open) {
                acc.n_new += (uint32_t)__popcll(nw);
                record_depth(a, v, 0, nw, L + 1, false);
            }
        }
        if (!kMesh && sink && !open && nw == unv) atomicOr(a.D + (v >> 5), 1u << (v & 31));
        st.put(nw != 0ull && !open && !sink, v);
        if (!kMesh && __any_sync(0xffffffffu, open))
            ms_defer(lr, open, v, beg + k, left - k, st.cout);
    }
    st.flush_block<kMsThreads / 32>(bsm);
}

// A block's open rows of a pull level on a small graph: those with up to kMsFewWarp in-neighbours
// left from the front of row, longer ones from its back, those with more than kMsFewBlock in most.
// (20,000 vertices, 64 sources: listed after 2, 4 and 8 steps 129, 130 and 138 us; a warp each from
// 96, 256 and 1,024 left 128, 129 and 133.)
constexpr int32_t kMsFewWarp = 256;
constexpr int32_t kMsFewBlock = 2048;
constexpr int kMsFewSteps = 2;  // steps of a row's team before it is listed
constexpr int kMsFewMost = 32;  // rows of most (further ones are taken as longer)
struct MsFew {
    int32_t row[kMsThreads], most[kMsFewMost];
    int32_t cnt[3];
    unsigned long long acc[64];
};

// ORs V of the in-neighbours [k, end) of a row into ac, team lanes (a power of two, at least the
// group's) taking kMsUnroll a group and step, until what it misses (unv) is covered or `stop` is
// reached.  All lanes of the warp call; row < 0: nothing to do.  Returns whether it is covered.
template <int WL>
__device__ __forceinline__ bool ms_team_scan(const MsArgs& a, const Group& gr, int team, int32_t row, int32_t& k,
                                             int32_t end, int32_t stop, const Words<WL>& unv, Words<WL>& ac) {
    const int lane = threadIdx.x & 31, tg = (lane & (team - 1)) / gr.size, step = kMsUnroll * (team / gr.size);
    const uint32_t tmask = (team == 32 ? 0xffffffffu : (1u << team) - 1u) << (lane & ~(team - 1));
    const int32_t w = WL * gr.sub;
    bool covered = false;
    int32_t u[kMsUnroll];  // the in-neighbours of this step; the next step's are loaded meanwhile
#pragma unroll
    for (int t = 0; t < kMsUnroll; ++t)
        u[t] = row >= 0 && kMsUnroll * tg + t < end - k ? __ldg(a.in_col + k + kMsUnroll * tg + t) : -1;
    while (__any_sync(0xffffffffu, row >= 0 && !covered && k < stop)) {
        const bool go = row >= 0 && !covered && k < stop;
        Words<WL> x[kMsUnroll];
#pragma unroll
        for (int t = 0; t < kMsUnroll; ++t)
            x[t] = go && u[t] >= 0 && w < a.W ? ld_words<WL>(a.V + (size_t)u[t] * a.W + w) : zero_words<WL>();
        if (go) k = end - k > step ? k + step : end;
#pragma unroll
        for (int t = 0; t < kMsUnroll; ++t)
            u[t] = go && kMsUnroll * tg + t < end - k ? __ldg(a.in_col + k + kMsUnroll * tg + t) : -1;
        bool cov = true;
#pragma unroll
        for (int j = 0; j < WL; ++j) {
#pragma unroll
            for (int t = 0; t < kMsUnroll; ++t) ac.x[j] |= x[t].x[j];
            for (int o = gr.size; o < team; o <<= 1) ac.x[j] |= __shfl_xor_sync(0xffffffffu, ac.x[j], o);
            cov &= (ac.x[j] & unv.x[j]) == unv.x[j];
        }
        const bool all = (__ballot_sync(0xffffffffu, cov) & tmask) == tmask;
        covered |= go && all;
    }
    return covered;
}

// The pull on a small graph: every row its own team of a.team lanes, spread over the blocks.  A
// level then lasts as long as its longest row, and ms_pull with its deferred rows (two more
// grid barriers and a finalising pass) as long as several: rows still open after kMsFewSteps
// steps are listed by the block and taken by as many lanes as there are for each, by a warp
// each, or by the whole block.
//
// Batches on RMAT graphs with ms_pull and so: 1,000 vertices, 100 sources 208 and 102 us (a level 35 and
// 10.5); 6,000 vertices, 100 sources 328 and 152; 20,000, 64 sources 175 and 125; 1,000, 700 sources 449
// and 171.
template <int WL>
__device__ __forceinline__ void ms_pull_few(const MsArgs& a, int32_t L, unsigned long long* Fn, MsFew& few, Stage& st,
                                            unsigned long long* bsm, Acc& acc) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const Group gr(a.group);
    const int32_t w = WL * gr.sub;
    const bool wok = w < a.W;
    const uint32_t chunks256 = (uint32_t)(a.W + 3) >> 2;
    Words<WL> lm;
#pragma unroll
    for (int j = 0; j < WL; ++j) lm.x[j] = wok ? lane_mask(a.S, w + j) : 0ull;
    struct Row {
        int32_t k, end;
        bool sink;
        Words<WL> unv, ac;
    };
    auto open = [&](int32_t v) {
        Row r{0, 0, false, zero_words<WL>(), zero_words<WL>()};
        if (v >= 0) {
            r.k = __ldg(a.in_ptr + v);
            r.end = __ldg(a.in_ptr + v + 1);
            r.sink = !a.symmetric && __ldg(a.out_ptr + v + 1) == __ldg(a.out_ptr + v);
            if (wok) r.unv = ld_words<WL>(a.V + (size_t)v * a.W + w);
#pragma unroll
            for (int j = 0; j < WL; ++j) r.unv.x[j] = ~r.unv.x[j] & lm.x[j];
        }
        return r;
    };
    // the row's first group writes what is new; all lanes call (v < 0: nothing)
    auto settle = [&](int32_t v, const Row& r, bool first_group) {
        Words<WL> nw;
        const bool mine = v >= 0 && first_group;
#pragma unroll
        for (int j = 0; j < WL; ++j) nw.x[j] = mine ? r.ac.x[j] & r.unv.x[j] : 0ull;
        const bool any_new = gr.any(nw.any());
        const bool full = gr.all(nw.x[0] == r.unv.x[0] && nw.x[WL - 1] == r.unv.x[WL - 1]);
        ms_settle<WL>(a, L, v, w, r.sink, nw, r.unv, lm, Fn, acc);
        const bool lead = mine && gr.sub == 0;
        if (lead && r.sink && full) atomicOr(a.D + (v >> 5), 1u << (v & 31));
        st.put(lead && any_new && !r.sink, v);
    };
    if (threadIdx.x < 3) few.cnt[threadIdx.x] = 0;
    __syncthreads();
    {
        const int team = a.team;
        const long long id = (((long long)wib * gridDim.x + blockIdx.x) * 32 + lane) / team;
        int32_t v = id < a.n ? (int32_t)id : -1;
        if (v >= 0 && !(((a.nz_in[v >> 5] & ~a.D[v >> 5]) >> (v & 31)) & 1u)) v = -1;
        Row r = open(v);
        const int32_t beg = r.k, own = max(a.probe, kMsFewSteps * kMsUnroll * (team / gr.size));
        const bool leader = (lane & (team - 1)) == 0;
        const bool list = r.end - beg > (team == 32 ? own + kMsFewBlock : 2 * own);
        const bool covered = ms_team_scan<WL>(a, gr, team, v, r.k, r.end, list ? beg + own : r.end, r.unv, r.ac);
        if (v >= 0 && leader) acc.exam += chunks256 * (uint32_t)(r.k - beg);
        const bool done = covered || r.k >= r.end;
        if (v >= 0 && !done && leader) {
            const int32_t left = r.end - r.k;
            const int at = left > kMsFewBlock ? atomicAdd(&few.cnt[2], 1) : kMsFewMost;
            if (at < kMsFewMost)
                few.most[at] = v;
            else if (left > kMsFewWarp)
                few.row[kMsThreads - 1 - atomicAdd(&few.cnt[1], 1)] = v;
            else
                few.row[atomicAdd(&few.cnt[0], 1)] = v;
        }
        settle(done ? v : -1, r, (lane & (team - 1)) < gr.size);
    }
    __syncthreads();
    // listed rows are read from their start: what their team found is not kept
    for (int part = 0; part < 2; ++part) {
        const int32_t count = few.cnt[part];
        int team = 32;
        while (part == 0 && team > max(8, gr.size) && count * team > kMsThreads) team >>= 1;
        for (int32_t h0 = wib * (32 / team); h0 < count; h0 += kMsThreads / team) {
            const int32_t h = h0 + lane / team;
            const int32_t v = h < count ? few.row[part ? kMsThreads - 1 - h : h] : -1;
            Row r = open(v);
            const int32_t beg = r.k;
            ms_team_scan<WL>(a, gr, team, v, r.k, r.end, r.end, r.unv, r.ac);
            if (v >= 0 && (lane & (team - 1)) == 0) acc.exam += chunks256 * (uint32_t)(r.k - beg);
            settle(v, r, (lane & (team - 1)) < gr.size);
        }
    }
    const int32_t most = min(few.cnt[2], kMsFewMost);
    for (int32_t h = 0; h < most; ++h) {
        const int32_t v = few.most[h];
        Row r = open(v);
        const int32_t piece = 4 * kMsUnroll * (32 / gr.size), first = r.k;  // in-neighbours a warp takes at a time
        if ((int)threadIdx.x < a.W) few.acc[threadIdx.x] = 0ull;
        __syncthreads();
        for (int32_t o = wib * piece; o < r.end - first; o += piece * (kMsThreads / 32)) {
            r.k = first + o;
            const int32_t e = r.end - r.k < piece ? r.end : r.k + piece;
            const int32_t beg = r.k;
            ms_team_scan<WL>(a, gr, 32, v, r.k, e, e, r.unv, r.ac);
            if (lane == 0) acc.exam += chunks256 * (uint32_t)(r.k - beg);
            // with what the other warps have found meanwhile
            if (wok) {
#pragma unroll
                for (int j = 0; j < WL; ++j) {
                    if (gr.first == 0 && r.ac.x[j]) atomicOr(few.acc + w + j, r.ac.x[j]);
                    r.ac.x[j] |= *(volatile unsigned long long*)(few.acc + w + j);
                }
            }
            bool cov = true;
#pragma unroll
            for (int j = 0; j < WL; ++j) cov &= (r.ac.x[j] & r.unv.x[j]) == r.unv.x[j];
            if (__all_sync(0xffffffffu, cov)) break;
        }
        __syncthreads();
        if (wib == h % (kMsThreads / 32)) {
#pragma unroll
            for (int j = 0; j < WL; ++j) r.ac.x[j] = wok ? few.acc[w + j] : 0ull;
            settle(v, r, gr.first == 0);
        }
        __syncthreads();
    }
    st.flush_block<kMsThreads / 32>(bsm);
}

// The deferred rows' chunks, round-robin over the warps: the groups of a warp take
// kMsUnroll in-neighbours each per step, their results are ORed together and folded into
// F_next (which already holds what the probe found).  A chunk of a row that is covered by
// then is skipped.
template <int WL>
__device__ __forceinline__ void ms_pull_long(const MsArgs& a, unsigned long long* Fn, const MsLong& lr,
                                             int32_t entries, int32_t chunks, Acc& acc) {
    const int gwarp = (int)((blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMsThreads) >> 5);
    const Group gr(a.group);
    const int32_t w = WL * gr.sub;
    const bool wok = w < a.W;
    const int32_t step = kMsUnroll * (32 / gr.size);
    const uint32_t chunks256 = (uint32_t)(a.W + 3) >> 2;
    for (int32_t c = gwarp; c < chunks; c += nwarps) {
        const int32_t e = warp_find_entry(lr.base, entries, c);
        const int32_t v = lr.row[e];
        const int32_t rend = __ldg(a.in_ptr + v + 1);
        const int32_t beg = lr.k[e] + (c - lr.base[e]) * kMsChunk;
        const int32_t len = rend - beg < kMsChunk ? rend - beg : kMsChunk;
        const size_t iv = (size_t)v * a.W + w;
        Words<WL> unv = zero_words<WL>(), ac = zero_words<WL>();
        if (wok) {
            const Words<WL> vis = ld_words<WL>(a.V + iv);
#pragma unroll
            for (int j = 0; j < WL; ++j)  // what the row still misses (the fold of another chunk may have come in)
                unv.x[j] = ~(vis.x[j] | __ldcg(Fn + iv + j)) & lane_mask(a.S, w + j);
        }
        if (!__any_sync(0xffffffffu, unv.any())) continue;
        int32_t k0 = 0;
        const int32_t kofs = kMsUnroll * (gr.first / gr.size);
        int32_t u[kMsUnroll];  // the group's in-neighbours of this step; the next step's are loaded meanwhile
#pragma unroll
        for (int t = 0; t < kMsUnroll; ++t) u[t] = kofs + t < len ? __ldg(a.in_col + beg + kofs + t) : -1;
        while (k0 < len) {
            Words<WL> x[kMsUnroll];
#pragma unroll
            for (int t = 0; t < kMsUnroll; ++t)
                x[t] = u[t] >= 0 && wok ? ld_words<WL>(a.V + (size_t)u[t] * a.W + w) : zero_words<WL>();
            k0 += step;
#pragma unroll
            for (int t = 0; t < kMsUnroll; ++t) u[t] = k0 + kofs + t < len ? __ldg(a.in_col + beg + k0 + kofs + t) : -1;
#pragma unroll
            for (int j = 0; j < WL; ++j)
#pragma unroll
                for (int t = 0; t < kMsUnroll; ++t) ac.x[j] |= x[t].x[j];
            if (k0 < len && (k0 & (kMsCheck - 1)) != 0) continue;
            bool cov = true;
#pragma unroll
            for (int j = 0; j < WL; ++j) {
                for (int o = gr.size; o < 32; o <<= 1) ac.x[j] |= __shfl_xor_sync(0xffffffffu, ac.x[j], o);
                cov &= (ac.x[j] & unv.x[j]) == unv.x[j];
            }
            if (__all_sync(0xffffffffu, cov)) break;
        }
        if ((threadIdx.x & 31) == 0) acc.exam += chunks256 * (uint32_t)(k0 < len ? k0 : len);
        if (gr.first == 0)
#pragma unroll
            for (int j = 0; j < WL; ++j)
                if (ac.x[j] & unv.x[j]) atomicOr(Fn + iv + j, ac.x[j] & unv.x[j]);
    }
}

// V |= F for the vertices found by the pull level; mark vertices with all lanes visited.
template <int WL>
__device__ __forceinline__ void ms_pull_commit(const MsArgs& a, const int32_t* list, uint32_t count,
                                               const unsigned long long* Fn) {
    const Group gr(a.group);
    const int per = 32 / gr.size;  // vertices a warp takes at a time
    const long long gwarp = ((long long)blockIdx.x * kMsThreads + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * kMsThreads) >> 5;
    for (long long b = gwarp * per; b < count; b += nwarps * per) {  // warp-uniform
        const long long i = b + gr.first / gr.size;
        const int32_t v = i < count ? list[i] : -1;
        bool full = v >= 0;
        for (int32_t w = WL * gr.sub; v >= 0 && w < a.W; w += WL * gr.size) {
            const size_t iv = (size_t)v * a.W + w;
            Words<WL> x = ld_words<WL>(a.V + iv);
            const Words<WL> f = ld_words<WL>(Fn + iv);
#pragma unroll
            for (int j = 0; j < WL; ++j) {
                x.x[j] |= f.x[j];
                full &= (x.x[j] & lane_mask(a.S, w + j)) == lane_mask(a.S, w + j);
            }
            if (f.any()) st_words<WL>(a.V + iv, x);
        }
        if (gr.all(full) && gr.sub == 0) atomicOr(a.D + (v >> 5), 1u << (v & 31));
    }
}

// ---------------------------------------------------------------- push level

// W == 1, one phase: each edge (u, v) of the active list claims the lanes F_cur[u] & ~V[v]
// with an atomicOr on V[v]; the lanes it gained (not set before) are new at level
// L + 1 and this edge is their only claimant, so it writes their depth and ORs them
// into F_next[v]; the first edge to gain anything at v (the previous F_next word tells)
// lists v.  It claims without probing V[v] first (a dependent load per edge costs more
// than the extra atomics).
__device__ __forceinline__ void ms_push_one(const MsArgs& a, int32_t L, const int32_t* q, const int32_t* qp,
                                            const int32_t* qd, uint32_t qcount, uint32_t qedges,
                                            const unsigned long long* Fc, unsigned long long* Fn, Stage& st,
                                            unsigned long long* bsm, Acc& acc) {
    const int gwarp = (int)((blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMsThreads) >> 5);
    const int32_t E = (int32_t)qedges;
    const unsigned long long full0 = lane_mask(a.S, 0);
    int32_t chunk = (int32_t)(((long long)E + nwarps - 1) / nwarps);
    chunk = chunk < kPushStep ? kPushStep : ((chunk + kPushStep - 1) / kPushStep) * kPushStep;
    for (long long e0l = (long long)gwarp * chunk; e0l < E; e0l += (long long)nwarps * chunk) {
        const int32_t e0 = (int32_t)e0l;
        const int32_t e1 = E - e0 > chunk ? e0 + chunk : E;
        PushCursor cur_;
        cur_.k = warp_find_entry(qp, (int32_t)qcount, e0);
        cur_.wlast = -1;
        for (int32_t base = e0; base < e1; base += kPushStep) {
            const PushStep ps = cur_.gather(a.out_col, q, qp, qd, qcount, base, e1);
#pragma unroll
            for (int t = 0; t < kPushIlp; ++t) {
                const int32_t u = ps.u[t], v = ps.v[t];
                bool first = false;
                if (u >= 0 && !((a.D[v >> 5] >> (v & 31)) & 1u)) {
                    const unsigned long long cand = Fc[u];
                    if (cand) {
                        const unsigned long long old = atomicOr(a.V + v, cand);
                        const unsigned long long gained = cand & ~old;
                        if (gained) {
                            first = atomicOr(Fn + v, gained) == 0ull;
                            if (((old | cand) & full0) == full0) atomicOr(a.D + (v >> 5), 1u << (v & 31));
                            acc.n_new += (uint32_t)__popcll(gained);
                            record_depth(a, v, 0, gained, L + 1, true);
                        }
                    }
                }
                st.put(first, v);
            }
        }
    }
    // few edges: no more warps have something than there are blocks (a level of a few hundred vertices
    // 5.9 -> 5.0 us)
    if (E <= (long long)kPushStep * gridDim.x)
        st.flush();
    else
        st.flush_block<kMsThreads / 32>(bsm);
}

// A list of vertices in two pieces of memory: entries [0, cap) and the rest.
struct IdList {
    int32_t* first;
    int32_t* rest;
    uint32_t cap;
    __device__ __forceinline__ int32_t& at(uint32_t i) const { return i < cap ? first[i] : rest[i - cap]; }
};

// A level's next active list without degrees: vertices staged per warp, published with one
// atomic per full stage and one per block at the end.
struct IdStage {
    StageBuf* sb;
    int cnt;  // warp-uniform
    LevelCtr* cout;
    IdList ids;

    __device__ __forceinline__ void write(unsigned long long at) {
        __syncwarp();
        for (int i = threadIdx.x & 31; i < cnt; i += 32) ids.at((uint32_t)at + i) = sb->v[i];
        __syncwarp();
        cnt = 0;
    }
    __device__ __forceinline__ void put(bool take, int32_t v) {
        const uint32_t m = __ballot_sync(0xffffffffu, take);
        if (!m) return;
        if (cnt + __popc(m) > kStage) {
            unsigned long long at = 0ull;
            if ((threadIdx.x & 31) == 0) at = atomicAdd(&cout->q, (unsigned long long)cnt);
            write(__shfl_sync(0xffffffffu, at, 0));
        }
        if (take) sb->v[cnt + __popc(m & lanemask_lt())] = v;
        cnt += __popc(m);
    }
    template <int kWarps>
    __device__ __forceinline__ void flush_block(unsigned long long* bsm) {
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (lane == 0) bsm[w] = (unsigned long long)cnt;
        __syncthreads();
        if (w == 0) {
            const uint32_t own = lane < kWarps ? (uint32_t)bsm[lane] : 0u;
            const uint32_t inc = warp_inclusive_sum(own);
            unsigned long long at = 0ull;
            if (lane == 31 && inc) at = atomicAdd(&cout->q, (unsigned long long)inc);
            at = __shfl_sync(0xffffffffu, at, 31);
            if (lane < kWarps) bsm[lane] = at + inc - own;
        }
        __syncthreads();
        write(bsm[w]);
    }
};

// W == 1 on a mesh (a symmetric graph whose rows are short): ms_push_one without the queue's
// degree prefix.  Four lanes take a vertex and read its first five neighbours from the dense
// first-entry and next-entries arrays; a warp has up to kMsMeshIlp x 8 vertices in flight and
// the level's work is spread over all warps before one takes more than 8.  The degrees (the
// direction rule and the trace want their sum) are loaded when a vertex is claimed and added
// a step later.
//
// A mesh level (the 1024 x 1024 grid, 64 sources: 2,000 levels of about 30K active vertices)
// is bound by its chain of dependent round trips: list, neighbours, claim, F_next, list slot,
// barrier; the prefix search, the queue's row starts, the probe of D and the degrees of the
// flush are off it, and one atomic per block instead of one per warp reserves the list slots.
// A level 11.7 -> 8.5 us on the whole GPU (the batch 23.8 -> 18.4 ms); on the quarter that a
// server slot gets 14 -> 11 us, and to 10.2 with the clearing of the level before last off the
// chain, too.
constexpr int kMsMeshIlp = 4;
constexpr int32_t kMsMeshDegree = 32;  // longest row of a mesh

__device__ __forceinline__ bool ms_mesh_gain(const MsArgs& a, int32_t L, int32_t v, unsigned long long cand,
                                             unsigned long long old, unsigned long long was, char* const* rows,
                                             Acc& acc) {
    const unsigned long long gained = cand & ~old;
    if (!gained) return false;
    const unsigned long long full0 = lane_mask(a.S, 0);
    if (((old | cand) & full0) == full0) atomicOr(a.D + (v >> 5), 1u << (v & 31));
    acc.n_new += (uint32_t)__popcll(gained);
    if (L + 1 < 16) {
        record_depth(a, v, 0, gained, L + 1, true);
    } else {
        for (unsigned long long m = gained; m; m &= m - 1) {
            char* const r = rows[__ffsll((long long)m) - 1];
            if (a.depth16)
                reinterpret_cast<int16_t*>(r)[v] = (int16_t)(L + 1);
            else
                reinterpret_cast<int32_t*>(r)[v] = L + 1;
        }
    }
    return was == 0ull;  // the first edge to gain a lane at v lists it
}

// rows: the output rows' addresses (shared memory).
// once: v is listed by the first edge that gains a lane there, which the word of F_next tells it
// (a round trip before the list).  Else every edge that gains one lists v -- 7 % more entries on
// the grid, where a vertex has 1.07 new lanes a level -- and whoever takes an entry takes its
// lanes with it, leaving F_cur zero (which needs no clearing later) and nothing for the others;
// those entries are counted (exam, indeg: their number and degrees).  The first form is for graphs that
// may pull or whose lists could grow too long; against ms_push_one it takes 0.64 to 1.0 of the time of
// a batch of 64 on grids of 4, 6 and 8 neighbours and small worlds, 1.04 and 1.07 on two of 15 (2M
// vertices, nearly all of them active).
__device__ __forceinline__ void ms_push_mesh(const MsArgs& a, int32_t L, const IdList& ids, uint32_t qcount,
                                             unsigned long long* Fc, unsigned long long* Fn, char* const* rows,
                                             bool once, IdStage& st, unsigned long long* bsm, Acc& acc) {
    constexpr int K = kMsMeshIlp;
    const int lane = threadIdx.x & 31, j = lane & 3;
    const uint32_t gwarp = (uint32_t)((blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const uint32_t nwarps = (uint32_t)((gridDim.x * kMsThreads) >> 5);
    const uint32_t steps = (qcount + 8u * nwarps - 1u) / (8u * nwarps);  // steps of 8 vertices a warp has
    const uint32_t per = 8u * (steps < (uint32_t)K ? (steps ? steps : 1u) : (uint32_t)K);
    int32_t da[K], db[K];
#pragma unroll
    for (int k = 0; k < K; ++k) da[k] = db[k] = 0;
    for (unsigned long long base = (unsigned long long)gwarp * per; base < qcount;
         base += (unsigned long long)nwarps * per) {
        int32_t u[K], w[K];
        unsigned long long f[K], old[K], was[K];
        bool more = false;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t o = 8u * k + (lane >> 2);
            u[k] = o < per && base + o < qcount ? ids.at((uint32_t)base + o) : -1;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) acc.mf += (uint32_t)(db[k] - da[k]);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            w[k] = -1;
            f[k] = 0ull;
            if (u[k] < 0) continue;
            if (once)
                f[k] = Fc[u[k]];
            else if (j == 0)
                f[k] = atomicExch(Fc + u[k], 0ull);
            if (j == 0) {
                w[k] = __ldg(a.first_in + u[k]);
            } else if (j < 3) {
                w[k] = __ldg(reinterpret_cast<const int32_t*>(a.next_in + u[k]) + (j - 1));
            } else {
                const int2 x = __ldg(reinterpret_cast<const int2*>(a.next_in + u[k]) + 1);
                w[k] = x.x;
                more |= x.y >= 0;
            }
        }
        if (!once) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                f[k] = __shfl_sync(0xffffffffu, f[k], lane & ~3);
                if (u[k] >= 0 && f[k] == 0ull) {  // listed before
                    if (j == 0) {
                        acc.exam += 1;
                        acc.indeg += (uint32_t)(__ldg(a.out_ptr + u[k] + 1) - __ldg(a.out_ptr + u[k]));
                    }
                    u[k] = w[k] = -1;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) old[k] = w[k] >= 0 ? atomicOr(a.V + w[k], f[k]) : ~0ull;
        if (once) {
#pragma unroll
            for (int k = 0; k < K; ++k) was[k] = (f[k] & ~old[k]) ? atomicOr(Fn + w[k], f[k] & ~old[k]) : ~0ull;
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                was[k] = 0ull;
                if (f[k] & ~old[k]) atomicOr(Fn + w[k], f[k] & ~old[k]);  // a reduction
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool first = ms_mesh_gain(a, L, w[k], f[k], old[k], was[k], rows, acc);
            da[k] = first ? __ldg(a.out_ptr + w[k]) : 0;
            db[k] = first ? __ldg(a.out_ptr + w[k] + 1) : 0;
            st.put(first, w[k]);
        }
        if (__any_sync(0xffffffffu, more)) {  // rows of more than four entries: the rest, four lanes each
#pragma unroll
            for (int k = 0; k < K; ++k) {
                int32_t beg = 0, deg = 0;
                if (u[k] >= 0) {
                    beg = __ldg(a.out_ptr + u[k]);
                    deg = __ldg(a.out_ptr + u[k] + 1) - beg;
                }
                for (int32_t x = 4 + j; __any_sync(0xffffffffu, x < deg); x += 4) {
                    bool first = false;
                    int32_t v = 0;
                    if (x < deg) {
                        v = __ldg(a.out_col + beg + x);
                        const unsigned long long o = atomicOr(a.V + v, f[k]);
                        const unsigned long long p = (f[k] & ~o) ? atomicOr(Fn + v, f[k] & ~o) : ~0ull;
                        first = ms_mesh_gain(a, L, v, f[k], o, once ? p : 0ull, rows, acc);
                        if (first) acc.mf += (uint32_t)(__ldg(a.out_ptr + v + 1) - __ldg(a.out_ptr + v));
                    }
                    st.put(first, v);
                }
            }
        }
    }
    st.flush_block<kMsThreads / 32>(bsm);
#pragma unroll
    for (int k = 0; k < K; ++k) acc.mf += (uint32_t)(db[k] - da[k]);
}

// Wide batches, first phase: a warp takes 32 edges (u, v) of the active list and its
// groups OR F_cur[u] & ~V[v] into F_next[v] with reductions, one edge a group and
// kMsUnroll in flight; a touched v is listed once (the T_next bit).  The probe of V[v]
// only saves reductions (bits are only ever set).  A lane per edge walking its W words
// instead touched 32 rows with every load: level 0 of the RMAT-20 batch of 1,000 sources
// (55.7K edges), with the zeroing of the state, 276 us, now 128.
template <int WL>
__device__ __forceinline__ void ms_push_wide(const MsArgs& a, const int32_t* q, const int32_t* qp, const int32_t* qd,
                                             uint32_t qcount, uint32_t qedges, const unsigned long long* Fc,
                                             unsigned long long* Fn, uint32_t* Tn, StageBuf* sb, LevelCtr* cout) {
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)((blockIdx.x * kMsThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * kMsThreads) >> 5);
    const Group gr(a.group);
    const int per = 32 / gr.size;  // edges the warp's groups take at a time
    const int32_t E = (int32_t)qedges;
    int32_t chunk = (int32_t)(((long long)E + nwarps - 1) / nwarps);
    chunk = chunk < 32 ? 32 : ((chunk + 31) / 32) * 32;
    int staged = 0;  // touched vertices waiting in sb (warp-uniform)
    auto publish = [&]() {
        __syncwarp();
        unsigned long long pos = 0ull;
        if (lane == 0) pos = atomicAdd(&cout->list, (unsigned long long)staged);
        pos = __shfl_sync(0xffffffffu, pos, 0);
        for (int i = lane; i < staged; i += 32) a.tlist[pos + i] = sb->v[i];
        staged = 0;
        __syncwarp();
    };
    for (long long e0l = (long long)gwarp * chunk; e0l < E; e0l += (long long)nwarps * chunk) {
        const int32_t e0 = (int32_t)e0l;
        const int32_t e1 = E - e0 > chunk ? e0 + chunk : E;
        PushCursorT<1> cur_;
        cur_.k = warp_find_entry(qp, (int32_t)qcount, e0);
        cur_.wlast = -1;
        for (int32_t base = e0; base < e1; base += 32) {
            const PushStepT<1> ps = cur_.gather(a.out_col, q, qp, qd, qcount, base, e1);
            const int32_t v = ps.v[0];
            const int32_t u = ps.u[0] >= 0 && !((a.D[v >> 5] >> (v & 31)) & 1u) ? ps.u[0] : -1;
            bool touched = false;
            for (int32_t w = WL * gr.sub; w - WL * gr.sub < a.W; w += WL * gr.size) {
                for (int j0 = 0; j0 < gr.size; j0 += kMsUnroll) {
                    int32_t vv[kMsUnroll];
                    Words<WL> f[kMsUnroll], x[kMsUnroll];
#pragma unroll
                    for (int t = 0; t < kMsUnroll; ++t) {
                        const int e = (j0 + t) * per + gr.first / gr.size;  // the group's edge (a lane of the warp)
                        const int32_t uu = __shfl_sync(0xffffffffu, u, e & 31);
                        vv[t] = __shfl_sync(0xffffffffu, v, e & 31);
                        const bool ok = j0 + t < gr.size && uu >= 0 && w < a.W;
                        f[t] = ok ? ld_words<WL>(Fc + (size_t)uu * a.W + w) : zero_words<WL>();
                        x[t] = ok ? ld_words<WL>(a.V + (size_t)vv[t] * a.W + w) : zero_words<WL>();
                    }
#pragma unroll
                    for (int t = 0; t < kMsUnroll; ++t) {
                        bool hit = false;
#pragma unroll
                        for (int j = 0; j < WL; ++j) {
                            const unsigned long long cand = f[t].x[j] & ~x[t].x[j];
                            if (cand) {
                                atomicOr(Fn + (size_t)vv[t] * a.W + w + j, cand);  // result unused: a reduction
                                hit = true;
                            }
                        }
                        const uint32_t hm = __ballot_sync(0xffffffffu, hit);
                        // this lane's edge was taken by group lane % per in round lane / per
                        const uint32_t gm = gr.size == 32 ? 0xffffffffu : (1u << gr.size) - 1u;
                        if (lane / per == j0 + t) touched |= ((hm >> ((lane % per) * gr.size)) & gm) != 0u;
                    }
                }
            }
            const bool first = touched && !(atomicOr(Tn + (v >> 5), 1u << (v & 31)) & (1u << (v & 31)));
            const uint32_t fm = __ballot_sync(0xffffffffu, first);
            if (fm) {
                if (staged + __popc(fm) > kStage) publish();
                if (first) sb->v[staged + __popc(fm & lanemask_lt())] = v;
                staged += __popc(fm);
            }
        }
    }
    if (staged) publish();
}

// Vertices whose F_next words were gathered by several warps (a wide push level's touched
// ones, a pull level's deferred rows), after a barrier: new = F_next & ~V; V |= new,
// F_next = new, depth, "all lanes" map; those with new lanes join the next active list.
// Every T_next bit belongs to a touched vertex, so the words are cleared whole (racing
// writers all store zero).
template <int WL>
__device__ __forceinline__ void ms_finalize(const MsArgs& a, int32_t L, const int32_t* list, uint32_t count,
                                            unsigned long long* Fn, uint32_t* Tn, Stage& st, unsigned long long* bsm,
                                            Acc& acc) {
    const Group gr(a.group);
    const int per = 32 / gr.size;
    const long long gwarp = ((long long)blockIdx.x * kMsThreads + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * kMsThreads) >> 5;
    for (long long b = gwarp * per; b < count; b += nwarps * per) {  // warp-uniform: st.put needs all lanes
        const long long i = b + gr.first / gr.size;
        const int32_t v = i < count ? list[i] : -1;
        bool any_new = false, full = v >= 0;
        for (int32_t w = WL * gr.sub; v >= 0 && w < a.W; w += WL * gr.size) {
            const size_t iv = (size_t)v * a.W + w;
            Words<WL> x = ld_words<WL>(a.V + iv);
            const Words<WL> was = x, f = ld_words<WL>(Fn + iv);
            Words<WL> nw;
            bool changed = false;
#pragma unroll
            for (int j = 0; j < WL; ++j) {
                const unsigned long long lm = lane_mask(a.S, w + j);
                nw.x[j] = f.x[j] & ~x.x[j] & lm;
                changed |= nw.x[j] != f.x[j];
                x.x[j] |= nw.x[j];
                full &= (x.x[j] & lm) == lm;
                acc.n_new += (uint32_t)__popcll(nw.x[j]);
            }
            if (changed) st_words<WL>(Fn + iv, nw);
            if (nw.any()) st_words<WL>(a.V + iv, x);
            any_new |= nw.any();
            record_words<WL>(a, v, w, nw, was, L + 1);
        }
        const bool allfull = gr.all(full);
        any_new = gr.any(any_new);
        if (v >= 0 && gr.sub == 0) {
            Tn[v >> 5] = 0u;
            if (allfull) atomicOr(a.D + (v >> 5), 1u << (v & 31));
        }
        st.put(v >= 0 && gr.sub == 0 && any_new, v);
    }
    st.flush_block<kMsThreads / 32>(bsm);
}

// Clear F_{(L+2) mod 3} and T_{(L+2) mod 3} for the active list of level L - 1:
// those buffers were last read at level L - 1 and are written again at level L + 1.
template <int WL>
__device__ __forceinline__ void ms_clear_prev(const MsArgs& a, const int32_t* ids, uint32_t count,
                                              unsigned long long* F, uint32_t* T) {
    const Group gr(a.group);
    const int per = 32 / gr.size;
    const long long gwarp = ((long long)blockIdx.x * kMsThreads + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * kMsThreads) >> 5;
    for (long long b = gwarp * per; b < count; b += nwarps * per) {
        const long long i = b + gr.first / gr.size;
        if (i >= count) continue;
        const int32_t v = ids[i];
        for (int32_t w = WL * gr.sub; w < a.W; w += WL * gr.size)
            st_words<WL>(F + (size_t)v * a.W + w, zero_words<WL>());
        // every bit of T_{(L+2) mod 3} belongs to that list: racing writers all store zero
        if (gr.sub == 0) T[v >> 5] = 0u;
    }
}

// ---------------------------------------------------------------- kernel

// kMesh (WL = 1): push levels run ms_push_mesh.
template <int WL, int kOcc, bool kMesh = false>
__global__ void __launch_bounds__(kMsThreads, kOcc) ms_bfs_kernel(const __grid_constant__ MsArgs a) {
    const long long gtid = (long long)blockIdx.x * kMsThreads + threadIdx.x;
    // an error of an earlier launch not yet read by the host: this launch does nothing
    const int pending = threadIdx.x == 0 ? ld_volatile_i32(a.status + ST_ERROR) : 0;
    const long long gstride = (long long)gridDim.x * kMsThreads;
    // per warp: staged vertices, open rows of a pull level; after the last level the
    // emission's staging area
    struct WarpMem {
        StageBuf stage;
        uint16_t open_list[1024];
    };
    union BlockMem {
        WarpMem warp[kMsThreads / 32];
        uint32_t emit[WL == 2 ? kEmitSmem / 4 : 1];
    };
    __shared__ __align__(16) BlockMem mem;
    __shared__ MsFew few_mem;
    __shared__ unsigned long long stage_sum[kMsThreads / 32];  // per-warp queue ranges of a block flush
    __shared__ unsigned long long lvl[6];
    // of the level under way: its queue (entries, out-edges), the entries of the one before, the pairs found by
    // that one and when it ended; kept here rather than in every thread's registers
    __shared__ unsigned long long now_q, now_pairs, now_mark;
    __shared__ uint32_t now_prev;
    __shared__ unsigned long long acc_mem[kMsThreads / 32][4];
    const int wib = threadIdx.x >> 5;
    unsigned int* barc = a.bar->count + a.bar_parity;
    unsigned int bar_round = 0;
    if (threadIdx.x == 0) now_mark = global_timer_ns();
    // ---- init: V = F_k = 0, depth planes = 0, D = T_k = 0 (the output rows are written at the end)
    const size_t nw_total = (size_t)a.n * (size_t)a.W;
    for (size_t i = gtid; i < nw_total; i += gstride) {
        a.V[i] = 0ull;
        a.Fb[0][i] = 0ull;
        a.Fb[1][i] = 0ull;
        a.Fb[2][i] = 0ull;
        if (WL == 1)
#pragma unroll
            for (int p = 0; p < kMsPlanes; ++p) a.P[p][i] = 0ull;
    }
    for (long long w = gtid; w < a.nwords; w += gstride) {
        a.D[w] = 0u;
        a.Tb[0][w] = 0u;
        a.Tb[1][w] = 0u;
        a.Tb[2][w] = 0u;
    }
    if (gtid == 0) {
        LevelCtr z = {};
        a.ctr[0] = z;
        a.ctr[1] = z;
        a.ctr[2] = z;
        a.status[ST_LEVELS] = 0;
        a.bar->count[a.bar_parity ^ 1u] = 0u;
    }
    if (__syncthreads_or(pending)) return;
    if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
    // ---- sources: lane b starts at src[b] with depth 0
    for (long long b = gtid; b < a.S; b += gstride) {
        const int32_t s = a.src[b];
        atomicOr(a.V + (size_t)s * a.W + (b >> 6), 1ull << (b & 63));  // depth 0: no plane bit
        if (WL == 2)
#pragma unroll
            for (int p = 0; p < kMsPlanes; ++p) a.P[p][(size_t)s * a.W + (b >> 6)] = 0ull;
    }
    if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
    // F = V for the (distinct) source vertices; they form the first active list
    {
        Acc acc0;
        Stage st{&mem.warp[wib].stage, 0, a.ctr + 0, a.ids[0], a.qp[0], a.qd[0], a.out_ptr, a.in_ptr, 1, 0, &acc0};
        const long long rounds = ((long long)a.S + gstride - 1) / gstride;
        for (long long r = 0; r < rounds; ++r) {
            const long long b = r * gstride + gtid;
            bool take = false;
            int32_t s = 0;
            if (b < a.S) {
                s = a.src[b];
                take = !(atomicOr(a.Tb[0] + (s >> 5), 1u << (s & 31)) & (1u << (s & 31)));
                if (take)
                    for (int32_t w = 0; w < a.W; ++w) a.Fb[0][(size_t)s * a.W + w] = a.V[(size_t)s * a.W + w];
            }
            st.put(take, s);
        }
        st.flush();
        const unsigned long long m = warp_sum_u64(acc0.mf);
        if ((threadIdx.x & 31) == 0 && m) atomicAdd(&a.ctr[0].mf_new, m);
    }
    if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
    for (long long b = gtid; b < a.S; b += gstride) {
        const int32_t s = a.src[b];
        a.Tb[0][s >> 5] = 0u;  // racing writers all store zero
    }
    __shared__ char* row_mem[kMesh ? 64 : 1];  // the output rows' addresses
    if (kMesh && threadIdx.x < 64) row_mem[threadIdx.x] = depth_row(a, (int)threadIdx.x < a.S ? threadIdx.x : 0);
    if (threadIdx.x == 0) {
        now_q = ld_volatile_u64(&a.ctr[0].q);
        now_pairs = (unsigned long long)a.S;
        now_prev = 0u;
    }
    if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
    for (int32_t L = 0;; ++L) {
        const int r0 = L % 3, r1 = (L + 1) % 3, r2 = (L + 2) % 3, p0 = L & 1, p1 = p0 ^ 1;
        LevelCtr* cout = a.ctr + ((L + 1) % 3);
        if (gtid == 0) {
            LevelCtr z = {};
            a.ctr[(L + 2) % 3] = z;
        }
        const uint32_t qcount = (uint32_t)now_q, qedges = (uint32_t)(now_q >> 32);  // active vertices, their out-edges
        const uint32_t prev_count = now_prev;  // entries of the list of level L - 1
        // direction for the whole batch: pull once the active edges exceed alpha * nnz
        int dir = a.mode;
        if (dir == GBX_DIR_AUTO) dir = qedges > a.push_most ? GBX_DIR_PULL : GBX_DIR_PUSH;
        if (kMesh && a.never_pull) dir = GBX_DIR_PUSH;
        if (a.depth16 && L + 1 > 32767) {
            if (gtid == 0) atomicCAS(a.status + ST_ERROR, 0, (int)GBX_ERR_OVERFLOW);
            return;
        }
        Acc acc;
        Stage st{&mem.warp[wib].stage, 0, cout, a.ids[r1], a.qp[p1], a.qd[p1], a.out_ptr, a.in_ptr, 1, 0, &acc};
        if (!kMesh) ms_clear_prev<WL>(a, a.ids[r2], prev_count, a.Fb[r2], a.Tb[r2]);
        const MsLong lr{a.tlist, a.qp[p0], a.qd[p0]};  // a pull level does not read the queue's prefix
        if (dir == GBX_DIR_PUSH) {
            if (kMesh) {
                if (a.never_pull) {
                    const IdList now{a.ids[L & 1], a.more[L & 1], a.more_from};
                    IdStage ist{&mem.warp[wib].stage, 0, cout, IdList{a.ids[p1], a.more[p1], a.more_from}};
                    ms_push_mesh(a, L, now, qcount, a.Fb[p0], a.Fb[p1], row_mem, false, ist, stage_sum, acc);
                } else {
                    // the words of level L - 1's list are cleared here, their ids loaded before the push so that
                    // nothing waits for them
                    const long long c1 = gtid + gstride;
                    const int32_t v0 = gtid < prev_count ? a.ids[r2][gtid] : -1;
                    const int32_t v1 = c1 < prev_count ? a.ids[r2][c1] : -1;
                    IdStage ist{&mem.warp[wib].stage, 0, cout, IdList{a.ids[r1], nullptr, 0xffffffffu}};
                    ms_push_mesh(a, L, IdList{a.ids[r0], nullptr, 0xffffffffu}, qcount, a.Fb[r0], a.Fb[r1], row_mem,
                                 true, ist, stage_sum, acc);
                    if (v0 >= 0) a.Fb[r2][v0] = 0ull;
                    if (v1 >= 0) a.Fb[r2][v1] = 0ull;
                    for (long long k = c1 + gstride; k < prev_count; k += gstride) a.Fb[r2][a.ids[r2][k]] = 0ull;
                }
            } else if (WL == 1) {
                ms_push_one(a, L, a.ids[r0], a.qp[p0], a.qd[p0], qcount, qedges, a.Fb[r0], a.Fb[r1], st,
                            stage_sum, acc);
            } else {
                ms_push_wide<WL>(a, a.ids[r0], a.qp[p0], a.qd[p0], qcount, qedges, a.Fb[r0], a.Fb[r1], a.Tb[r1],
                                 &mem.warp[wib].stage, cout);
                if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
                if (threadIdx.x == 0) lvl[5] = ld_volatile_u64(&cout->list);
                __syncthreads();
                ms_finalize<WL>(a, L, a.tlist, (uint32_t)lvl[5], a.Fb[r1], a.Tb[r1], st, stage_sum, acc);
            }
        } else {
            if (kMesh) {
                ms_clear_prev<WL>(a, a.ids[r2], prev_count, a.Fb[r2], a.Tb[r2]);
                ms_pull_one<true>(a, L, a.Fb[r1], lr, st, stage_sum, acc);
            } else if (a.team) {
                ms_pull_few<WL>(a, L, a.Fb[r1], few_mem, st, stage_sum, acc);
            } else if (WL == 1) {
                ms_pull_one<false>(a, L, a.Fb[r1], lr, st, stage_sum, acc);
            } else {
                const bool one = a.W <= WL * a.group;  // one chunk of words: long rows can be deferred
                for (int32_t c0 = 0; c0 < a.W; c0 += WL * a.group)
                    ms_pull<WL>(a, L, c0, a.Fb[r1], a.Tb[r1], mem.warp[wib].open_list, lr, one, st, stage_sum, acc);
            }
        }
        block_add_counts<kMsThreads / 32>(acc_mem, acc.n_new, acc.mf, acc.exam, kMesh ? acc.indeg : 0ull, &cout->n_new,
                                          &cout->mf_new, &cout->e_exam, kMesh ? &cout->indeg_new : nullptr);
        if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
        if (threadIdx.x == 0) {
            lvl[0] = ld_volatile_u64(&cout->n_new);
            lvl[1] = ld_volatile_u64(&cout->mf_new);
            lvl[2] = ld_volatile_u64(&cout->huge);
            if (kMesh) lvl[5] = ld_volatile_u64(&cout->indeg_new);
            lvl[3] = ld_volatile_u64(&cout->e_exam);
            lvl[4] = ld_volatile_u64(&cout->q);
        }
        __syncthreads();
        if (!kMesh && dir == GBX_DIR_PULL && lvl[2] != 0ull) {  // the level deferred long rows: the grid takes them now
            const uint32_t rows = (uint32_t)lvl[2];
            Acc acc2;
            Stage st2{&mem.warp[wib].stage, 0, cout, a.ids[r1], a.qp[p1], a.qd[p1], a.out_ptr, a.in_ptr, 1, 0, &acc2};
            ms_pull_long<WL>(a, a.Fb[r1], lr, (int32_t)rows, (int32_t)(lvl[2] >> 32), acc2);
            if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
            ms_finalize<WL>(a, L, lr.row, rows, a.Fb[r1], a.Tb[r1], st2, stage_sum, acc2);
            block_add_counts<kMsThreads / 32>(acc_mem, acc2.n_new, acc2.mf, acc2.exam, 0ull, &cout->n_new,
                                              &cout->mf_new, &cout->e_exam, nullptr);
            if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
            if (threadIdx.x == 0) {
                lvl[0] = ld_volatile_u64(&cout->n_new);
                lvl[1] = ld_volatile_u64(&cout->mf_new);
                lvl[3] = ld_volatile_u64(&cout->e_exam);
                lvl[4] = ld_volatile_u64(&cout->q);
            }
            __syncthreads();
        }
        if (dir == GBX_DIR_PULL) {
            // V |= F for the vertices the pull found (their new lanes were kept apart so the
            // level read V as it was before it started)
            ms_pull_commit<WL>(a, a.ids[r1], (uint32_t)lvl[4], a.Fb[r1]);
            if (!grid_barrier(barc, gridDim.x, bar_round, a.status, a.timeout_ns)) return;
        }
        const long long n_new = (long long)lvl[0];
        if (gtid == 0 && L < a.trace_cap) {
            LevelRec r;
            r.direction = dir;
            r.level = L;
            r.nf = (long long)(uint32_t)now_q;
            r.mf = (long long)(now_q >> 32);
            r.mu = (long long)now_pairs;
            r.e_exam = dir == GBX_DIR_PULL ? (long long)lvl[3] : -1;
            r.n_new = n_new;
            r.mf_new = (long long)lvl[1];
            if (kMesh && a.never_pull) {  // without the entries that were listed again
                r.nf -= (long long)lvl[3];
                r.mf -= (long long)lvl[5];
                if (L > 0) a.trace[L - 1].mf_new = r.mf;
            }
            const unsigned long long now = global_timer_ns();
            r.t_ns = (long long)(now - now_mark);
            now_mark = now;
            a.trace[L] = r;
        }
        if (n_new == 0) {
            if (gtid == 0) a.status[ST_LEVELS] = L + 1;
            if (WL == 2 && a.W >= 4)
                emit_depths<true>(a, mem.emit);
            else
                emit_depths<false>(a, mem.emit);
            return;
        }
        if (L + 1 >= a.n) {
            if (gtid == 0) atomicCAS(a.status + ST_ERROR, 0, (int)GBX_ERR_OVERFLOW);
            return;
        }
        if (threadIdx.x == 0) {
            now_prev = (uint32_t)now_q;
            now_pairs = lvl[0];
            now_q = lvl[4] | (kMesh && dir == GBX_DIR_PUSH ? lvl[1] << 32 : 0ull);  // a mesh push lists without the degrees
        }
        __syncthreads();
    }
}

gbx_status ms_reserve(Workspace& w, int32_t n, int32_t S, cudaStream_t s) {
    const int32_t w_raw = (S + 63) / 64;
    const int cw = w_raw >= 4 ? 4 : (w_raw >= 2 ? 2 : 1);
    const int64_t need = (int64_t)n * ((w_raw + cw - 1) / cw * cw);
    if (w.ms_cap_words < need) {
        if (w.msV || w.msP || w.msF[0] || w.msF[1] || w.msF[2]) {
            GBX_CUDA_TRY(cudaStreamSynchronize(s));
            cudaFree(w.msV);
            w.msV = nullptr;
            for (auto& p : w.msF) {
                cudaFree(p);
                p = nullptr;
            }
            cudaFree(w.msP);
            w.msP = nullptr;
            w.ms_cap_words = 0;
        }
        GBX_CUDA_TRY(cudaMalloc((void**)&w.msV, sizeof(unsigned long long) * (size_t)need));
        for (auto& p : w.msF) GBX_CUDA_TRY(cudaMalloc((void**)&p, sizeof(unsigned long long) * (size_t)need));
        GBX_CUDA_TRY(cudaMalloc((void**)&w.msP, sizeof(unsigned long long) * (size_t)need * kMsPlanes));
        w.ms_cap_words = need;  // only once every buffer exists
    }
    if (w.ms_t_cap < (int64_t)n + 1) {
        if (w.msT) {
            GBX_CUDA_TRY(cudaStreamSynchronize(s));
            cudaFree(w.msT);
            w.msT = nullptr;
            w.ms_t_cap = 0;
        }
        GBX_CUDA_TRY(cudaMalloc((void**)&w.msT, sizeof(int32_t) * ((size_t)n + 1)));
        w.ms_t_cap = (int64_t)n + 1;
    }
    return GBX_OK;
}

int64_t ms_scratch_bytes(int32_t n, int32_t S) {
    const int32_t w_raw = (S + 63) / 64;
    const int cw = w_raw >= 4 ? 4 : (w_raw >= 2 ? 2 : 1);
    return (4ll + kMsPlanes) * 8ll * (int64_t)n * ((w_raw + cw - 1) / cw * cw) + 4ll * ((int64_t)n + 1);
}

template <int WL, int kOcc, bool kMesh = false>
static gbx_status ms_launch(Graph* G, const MsArgs& a0, int blocks, int per_sm_cap, cudaStream_t s) {
    const uint32_t which = 32u << (WL == 2 ? kOcc - kMsOcc : 2 + (kMesh ? 2 : kOcc - kMsOcc));
    if (!(G->l1_set & which)) {
        GBX_TRY(prefer_l1((const void*)ms_bfs_kernel<WL, kOcc, kMesh>, kOcc));
        G->l1_set |= which;
    }
    int per_sm = 0;
    GBX_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ms_bfs_kernel<WL, kOcc, kMesh>, kMsThreads, 0));
    GBX_CHECK(per_sm >= 1, GBX_ERR_CUDA, "batched BFS kernel cannot be resident");
    if (per_sm_cap > 0 && per_sm_cap < per_sm) per_sm = per_sm_cap;
    const int full = per_sm * G->num_sms;
    const int nb = blocks > 1 ? (full / blocks > 0 ? full / blocks : 1) : full;  // a 1/blocks share of the GPU
    MsArgs a = a0;
    // a team of lanes for every row where there are as many; with one word four a row, since a lane walks
    // short rows well by itself (80,000 vertices, 20 sources: 108 us with a lane or two a row, 103
    // without; 40,000: 101 and 99; 20,000 and 64 sources, four: 131 and 132)
    const long long lanes = (long long)nb * kMsThreads;
    a.team = 0;
    if (a.W <= WL * a.group && (WL == 1 ? 4ll : (long long)a.group) * a.n <= lanes)
        for (a.team = a.group; a.team < 32 && 2ll * a.team * a.n <= lanes;) a.team *= 2;
    void* args[] = {&a};
    GBX_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)ms_bfs_kernel<WL, kOcc, kMesh>, dim3(nb), dim3(kMsThreads), args, 0,
                                             s));
    return GBX_OK;
}

// One batched BFS on G: sources already on the device (src_dev), depth either a
// [S][n] buffer or a device table of S row pointers.  `blocks` > 1 runs the
// persistent kernel on 1/blocks of the GPU's resident blocks (so that many
// batches of other graphs fit alongside); scratch must be reserved for S lanes.
gbx_status ms_run(Graph* G, Workspace& w, int32_t S, const int32_t* src_dev, void* depth, void* const* rows,
                  int depth16, const gbx_desc& d, int blocks, cudaStream_t s) {
    const int32_t w_raw = (S + 63) / 64;
    const int cw = w_raw >= 4 ? 4 : (w_raw >= 2 ? 2 : 1);
    const int32_t W = (w_raw + cw - 1) / cw * cw;
    GBX_CHECK(w.ms_cap_words >= (int64_t)G->n * W && w.n_cap >= G->n && w.ms_t_cap > G->n, GBX_ERR_INVALID_VALUE,
              "batch scratch not reserved");
    MsArgs a;
    a.n = G->n;
    a.S = S;
    a.W = W;
    a.nwords = G->nwords;
    a.nnz = G->nnz;
    a.out_ptr = G->out_ptr;
    a.out_col = G->out_col;
    a.in_ptr = G->in_ptr;
    a.in_col = G->in_col;
    a.nz_in = G->nz_in;
    a.first_in = G->first_in;
    a.next_in = G->next_in;
    a.V = w.msV;
    for (int k = 0; k < 3; ++k) a.Fb[k] = w.msF[k];
    for (int k = 0; k < kMsPlanes; ++k) a.P[k] = w.msP + (size_t)k * (size_t)G->n * (size_t)W;
    a.D = w.bm[2];
    a.Tb[0] = w.bm[3];
    a.Tb[1] = w.bm[0];
    a.Tb[2] = w.bm[1];
    a.tlist = w.msT;
    a.depth = depth;
    a.rows = rows;
    a.depth16 = depth16;
    a.src = src_dev;
    a.ids[0] = w.q[0];
    a.ids[1] = w.q[1];
    a.ids[2] = w.list;
    for (int i = 0; i < 2; ++i) {
        a.qp[i] = w.qp[i];
        a.qd[i] = w.qd[i];
    }
    a.ctr = w.ctr;
    a.bar = w.bar;
    a.bar_parity = w.bar_parity;
    a.trace = w.trace;
    a.status = w.status;
    // (the product in binary64 in every thread took 0.7 us of each level)
    a.push_most = (uint32_t)std::min(4294967295.0, std::floor((double)d.alpha * (double)G->nnz));
    a.mode = d.direction;
    a.symmetric = G->symmetric;
    a.trace_cap = kTraceCap;
    a.probe = d.pull_probe > 0 ? d.pull_probe : kMsProbe;
    a.timeout_ns = wait_timeout_ns();
    // the lean build only when this batch has the GPU to itself: concurrent cooperative
    // grids of one register budget tile the SMs exactly, mixed budgets need not
    const bool lean = blocks <= 1 && d.blocks_per_sm >= kMsOccLean && cw <= 2;
    // few vertices: barriers among half the blocks are cheaper (8K vertices, 436 sources 515 -> 423 us, 45
    // sources 171 -> 149; 20K, 516 sources 622 -> 563, 38 sources 183 -> 171; 125K, 36 sources 182 -> 186)
    const bool small = blocks <= 1 && d.blocks_per_sm == 0 && G->n <= 32768;
    const int cap = lean ? 0 : small ? 1 : d.blocks_per_sm;
    gbx_status st;
    // A threshold of one and more never pulls: at most every edge is active.  A level lists at most one
    // vertex per edge; the queue arrays q, qp and qd of one side lie one after another (workspace_carve)
    // and the third lane buffer, not needed then, holds n more entries of each of two lists.
    a.never_pull = G->nnz <= 4ll * G->n && G->n <= (1 << 30) &&
                   (d.direction == GBX_DIR_PUSH || (d.direction == GBX_DIR_AUTO && d.alpha >= 1.0f));
    a.more_from = 3u * (uint32_t)G->n;
    a.more[0] = reinterpret_cast<int32_t*>(w.msF[2]);
    a.more[1] = a.more[0] + G->n;
    a.group = 1;
    while (2 * a.group < W && a.group < 32) a.group *= 2;
    if (W > 1)
        st = lean ? ms_launch<2, kMsOccLean>(G, a, blocks, cap, s) : ms_launch<2, kMsOcc>(G, a, blocks, cap, s);
    else if (!lean && G->symmetric && G->max_out_degree <= kMsMeshDegree)
        st = ms_launch<1, kMsOcc, true>(G, a, blocks, cap, s);
    else
        st = lean ? ms_launch<1, kMsOccLean>(G, a, blocks, cap, s) : ms_launch<1, kMsOcc>(G, a, blocks, cap, s);
    if (st != GBX_OK) return st;
    w.bar_parity ^= 1u;
    w.last_stream = s;
    w.last_traced = 2;  // batched trace
    return GBX_OK;
}

}  // namespace gbx

using namespace gbx;

extern "C" gbx_status gbx_bfs_batch(gbx_graph* g, const int32_t* sources, int32_t S, void* depth, int32_t depth_type,
                                    const gbx_desc* desc, void* stream) {
    clear_error();
    GBX_TRY(check_graph(g));
    Graph* G = as_impl(g);
    GBX_CHECK(S >= 1, GBX_ERR_INVALID_VALUE, "S must be >= 1");
    GBX_CHECK(sources != nullptr && depth != nullptr, GBX_ERR_NULL_POINTER, "sources or depth is NULL");
    GBX_CHECK(depth_type == GBX_DEPTH_I32 || depth_type == GBX_DEPTH_I16, GBX_ERR_INVALID_VALUE, "depth_type");
    for (int32_t k = 0; k < S; ++k)
        GBX_CHECK(sources[k] >= 0 && sources[k] < G->n, GBX_ERR_INVALID_INDEX, "source outside [0, n)");
    gbx_desc d;
    if (desc)
        d = *desc;
    else
        gbx_desc_init(&d);
    GBX_CHECK(d.direction >= GBX_DIR_AUTO && d.direction <= GBX_DIR_PULL, GBX_ERR_INVALID_VALUE, "desc.direction");
    GBX_CHECK(d.alpha >= 0.0f && d.alpha == d.alpha, GBX_ERR_INVALID_VALUE, "desc.alpha must be >= 0");
    GBX_CHECK(d.pull_probe == 0 || (d.pull_probe >= 4 && d.pull_probe <= 1024), GBX_ERR_INVALID_VALUE,
              "desc.pull_probe must be 0 or in [4, 1024]");
    GBX_CHECK(d.push_sort == 0, GBX_ERR_NOT_SUPPORTED, "desc.push_sort applies to gbx_mxv only");
    GBX_CHECK(d.blocks_per_sm >= 0, GBX_ERR_INVALID_VALUE, "desc.blocks_per_sm must be >= 0");
    cudaStream_t s = (cudaStream_t)stream;
    GBX_TRY(ms_reserve(G->ws, G->n, S, s));
    if (G->ws.ms_src_cap < S) {
        if (G->ws.ms_src) {
            GBX_CUDA_TRY(cudaStreamSynchronize(s));
            cudaFree(G->ws.ms_src);
            cudaFreeHost(G->ws.ms_src_pinned);
            G->ws.ms_src = nullptr;
            G->ws.ms_src_pinned = nullptr;
        }
        GBX_CUDA_TRY(cudaMalloc((void**)&G->ws.ms_src, sizeof(int32_t) * (size_t)S));
        GBX_CUDA_TRY(cudaMallocHost((void**)&G->ws.ms_src_pinned, sizeof(int32_t) * (size_t)S));
        G->ws.ms_src_cap = S;
    }
    if (!G->ws.ms_src_ready) GBX_CUDA_TRY(cudaEventCreateWithFlags(&G->ws.ms_src_ready, cudaEventDisableTiming));
    // sources: pinned staging, then one async copy (the staging buffer is reused only
    // after the previous copy has completed)
    GBX_CUDA_TRY(cudaEventSynchronize(G->ws.ms_src_ready));
    for (int32_t k = 0; k < S; ++k) G->ws.ms_src_pinned[k] = sources[k];
    GBX_CUDA_TRY(cudaMemcpyAsync(G->ws.ms_src, G->ws.ms_src_pinned, sizeof(int32_t) * (size_t)S, cudaMemcpyHostToDevice, s));
    GBX_CUDA_TRY(cudaEventRecord(G->ws.ms_src_ready, s));
    return ms_run(G, G->ws, S, G->ws.ms_src, depth, nullptr, depth_type == GBX_DEPTH_I16 ? 1 : 0, d, 0, s);
}

extern "C" gbx_status gbx_bfs_batch_trace(gbx_graph* g, gbx_level* levels, int32_t cap, int32_t* nlevels) {
    clear_error();
    GBX_TRY(check_graph(g));
    Graph* G = as_impl(g);
    GBX_CHECK(nlevels != nullptr, GBX_ERR_NULL_POINTER, "nlevels is NULL");
    GBX_CHECK(cap == 0 || levels != nullptr, GBX_ERR_NULL_POINTER, "levels is NULL");
    GBX_CHECK(G->ws.last_traced == 2, GBX_ERR_INVALID_VALUE, "the last run on this graph was not a batched BFS");
    if (G->ws.last_stream) GBX_CUDA_TRY(cudaStreamSynchronize(G->ws.last_stream));
    int32_t st[ST_WORDS];
    GBX_CUDA_TRY(cudaMemcpy(st, G->ws.status, sizeof(st), cudaMemcpyDeviceToHost));
    GBX_CHECK(st[ST_ERROR] == 0, (gbx_status)st[ST_ERROR], "the last batched BFS recorded a device-side error");
    *nlevels = st[ST_LEVELS];
    const int32_t L = st[ST_LEVELS] < kTraceCap ? st[ST_LEVELS] : kTraceCap;
    const int32_t ncopy = L < cap ? L : cap;
    if (ncopy <= 0) return GBX_OK;
    LevelRec* recs = new LevelRec[ncopy];
    const cudaError_t e = cudaMemcpy(recs, G->ws.trace, sizeof(LevelRec) * ncopy, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        delete[] recs;
        GBX_CUDA_TRY(e);
    }
    for (int32_t l = 0; l < ncopy; ++l) {
        const LevelRec& r = recs[l];
        gbx_level o = {};
        o.direction = r.direction;
        o.level = r.level;
        o.nf = r.nf;          // active vertices (any lane)
        o.mf = r.mf;          // their out-edges
        o.nu = -1;
        o.nu_nz = -1;
        o.mu = r.mu;          // (vertex, lane) pairs found at the previous level
        o.e_exam = r.e_exam;  // pull: edges examined (per 256-lane chunk)
        o.n_new = r.n_new;    // (vertex, lane) pairs found at this level
        o.mf_new = r.mf_new;  // out-edges of the next active list
        o.time_ns = r.t_ns;
        levels[l] = o;
    }
    delete[] recs;
    return GBX_OK;
}
