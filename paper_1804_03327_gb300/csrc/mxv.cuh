// Shared by the matvec translation units: the row-based (pull) matvec on bitmaps.
#pragma once

#include "gbx_internal.cuh"

namespace gbx {

constexpr int kMxvThreads = 256;

// Per-call counters of gbx_mxv (desc.trace): [0] rows computed by pull, [1]
// entries examined by pull, [2] nonzeros of u expanded by push, [3] edges expanded.
struct MxvStats {
    unsigned long long rows, exam, ucount, edges, pad[4];
};

constexpr int32_t kMxvLongRow = 1024;  // entries left after the lane probe beyond which a row is the block's
constexpr int kMxvLongs = 64;          // such rows a block holds (further ones stay with their warp)

struct PullArgs {
    const int32_t* ptr;
    const int32_t* col;
    const int32_t* first;   // entry 0 of each row, or NULL
    const int4* next;       // entries 1..4 of each row, or NULL
    const uint32_t* nz;     // nonempty rows
    const uint32_t* multi;  // rows of at least two entries, or NULL
    const uint32_t* ubm;
    const uint32_t* pass;  // rows that pass, XOR invert; NULL: all
    uint32_t invert;       // 0 or all ones
    uint32_t* R;
    int32_t accum;  // R holds bits to be kept
    int32_t nwords, tile_words, early_exit;
    MxvStats* stats;
};

struct PullSmem {
    uint32_t hits[kMxvThreads / 32][32];
    uint16_t rows[kMxvThreads / 32][1024];
    int2 longs[kMxvLongs];  // row, next entry
    int nlong, hit;
};

// Bitmap words a warp takes at a time: an even share of the words over as many rounds as 32
// words a warp need.  Tiles of 32 words (1,024 rows) leave most warps without any on a graph
// of a million rows.
inline int32_t mxv_tile_words(int32_t nwords, long long nwarps) {
    const long long rounds = (nwords + 32 * nwarps - 1) / (32 * nwarps);
    const long long tw = (nwords + nwarps * rounds - 1) / (nwarps * rounds);
    return (int32_t)(tw < 2 ? 2 : tw);
}

// The row-based matvec alone (mxv.cu), for the allocation-free entry point; kMxvThreads a block.
__global__ void mxv_pull_kernel(PullArgs a);

// The kernels of one call depend on one another and each is short: a later one is launched
// while the one before still runs (programmatic dependent launch), its blocks take their
// places as soon as every block of that one has started, and pdl_begin waits there until
// the one before has ended and its writes are visible.  Saves about 2 us of the 4 between
// two dependent launches.
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename A>
gbx_status pdl_launch(void (*fn)(A), unsigned blocks, const A& a, bool dependent, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kMxvThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = dependent ? 1 : 0;
    GBX_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, a));
    return GBX_OK;
}

// AUTO pushes while count / n <= alpha (input sparsity, Section 6.3): the largest such count.  The
// division is the host's: binary64 is slow here, and every thread of a kernel dividing took 8 of the
// 12 us of an otherwise empty one.
inline int32_t mxv_push_most(int32_t n, float alpha) {
    const double a = (double)alpha;
    if (a * (double)n >= 2147483647.0) return INT32_MAX;
    int32_t c = (int32_t)(a * (double)n);
    while (c < INT32_MAX && (double)(c + 1) / (double)n <= a) ++c;
    while (c > 0 && (double)c / (double)n > a) --c;
    return c;
}

// What gbx_mxv reads, as bitmaps and queues (mxv.cu).
struct MxvVec {
    int32_t format;  // GBX_DENSE, GBX_SPARSE or GBX_DENSE_F32; -1: none
    const void* data;
    const int32_t* count;
    int32_t cap;
};

// Word w of a dense byte vector (bits past n clear): two 16-byte loads where it is aligned.
__device__ __forceinline__ uint32_t pack_word(const uint8_t* __restrict__ dense, int32_t n, int32_t w) {
    const int64_t base = (int64_t)w << 5;
    uint32_t word = 0;
    if ((reinterpret_cast<uintptr_t>(dense) & 15u) == 0 && base + 32 <= n) {
        const uint4 x = reinterpret_cast<const uint4*>(dense + base)[0];
        const uint4 y = reinterpret_cast<const uint4*>(dense + base)[1];
        const uint32_t v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int t = 0; t < 4; ++t) word |= (((v[q] >> (8 * t)) & 0xffu) != 0u ? 1u : 0u) << (4 * q + t);
    } else {
        for (int t = 0; t < 32 && base + t < n; ++t) word |= (dense[base + t] != 0 ? 1u : 0u) << t;
    }
    return word;
}

}  // namespace gbx
