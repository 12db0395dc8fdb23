// Graph construction on the device: edge list -> CSR of A and CSR of A^T.
//
// Section 7.1: every dataset is made undirected and has self-loops and
// duplicate edges removed.  The build packs each directed entry (row, col)
// into one 64-bit key row << b | col (b = bits of n), radix-sorts the keys,
// drops repeats, and derives row offsets from the sorted rows.  Neighbour lists
// therefore come out ascending (Section 3 assumes sorted index lists).
#include <algorithm>
#include <new>

#include "gbx_internal.cuh"

namespace gbx {

static int bits_for(int64_t v) {  // smallest b >= 1 with 2^b > v
    int b = 1;
    while (b < 31 && ((int64_t)1 << b) <= v) ++b;
    return b;
}

// A dropped self-loop's key is `none`, all ones in 2b bits: the largest key.  It is no valid
// pair's then -- the pair of ones is (n - 1, n - 1) at most, a self-loop -- and without the
// drop no key is invalid.
__global__ void make_keys_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int64_t m,
                                 int32_t n, int b, int symmetrize, int drop_self, int reverse,
                                 unsigned long long* __restrict__ keys, int32_t* status) {
    const unsigned long long none = (1ull << (2 * b)) - 1ull;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        int32_t u = src[e], v = dst[e];
        if (reverse) {
            const int32_t t = u;
            u = v;
            v = t;
        }
        unsigned long long k0 = none, k1 = none;
        if (u < 0 || u >= n || v < 0 || v >= n) {
            atomicCAS(status + ST_BADINDEX, -1, (int)(e < INT32_MAX ? e : INT32_MAX));
        } else if (!(drop_self && u == v)) {
            k0 = ((unsigned long long)u << b) | (unsigned long long)v;
            k1 = ((unsigned long long)v << b) | (unsigned long long)u;
        }
        keys[e] = k0;
        if (symmetrize) keys[m + e] = k1;
    }
}

// The sorted keys a thread owns (kUniqItems consecutive ones) and which of them are kept: valid
// and different from the one before.
constexpr int kUniqThreads = 256;
constexpr int kUniqItems = 8;
constexpr int kUniqTile = kUniqThreads * kUniqItems;

__device__ __forceinline__ uint32_t load_unique(const unsigned long long* __restrict__ keys, int64_t K,
                                                unsigned long long none, int64_t i0, unsigned long long (&x)[kUniqItems],
                                                unsigned long long& prev) {
    prev = i0 > 0 && i0 <= K ? keys[i0 - 1] : ~0ull;
    if (i0 + kUniqItems <= K) {
#pragma unroll
        for (int t = 0; t < kUniqItems / 2; ++t) {
            const ulonglong2 y = reinterpret_cast<const ulonglong2*>(keys + i0)[t];
            x[2 * t] = y.x;
            x[2 * t + 1] = y.y;
        }
    } else {
#pragma unroll
        for (int t = 0; t < kUniqItems; ++t) x[t] = i0 + t < K ? keys[i0 + t] : none;
    }
    uint32_t keep = 0u;
    unsigned long long p = prev;
#pragma unroll
    for (int t = 0; t < kUniqItems; ++t) {
        if (i0 + t < K && x[t] != none && x[t] != p) keep |= 1u << t;
        p = x[t];
    }
    return keep;
}

// counts[b] = keys kept in tile b.  (none: ~0 when every key is valid)
__global__ void __launch_bounds__(kUniqThreads)
    count_unique_kernel(const unsigned long long* __restrict__ keys, int64_t K, unsigned long long none,
                        int32_t* __restrict__ counts) {
    __shared__ uint32_t part[kUniqThreads / 32];
    unsigned long long x[kUniqItems], prev;
    const int64_t i0 = ((int64_t)blockIdx.x * kUniqThreads + threadIdx.x) * kUniqItems;
    const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(load_unique(keys, K, none, i0, x, prev)));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < kUniqThreads / 32; ++w) s += part[w];
        counts[blockIdx.x] = (int32_t)s;
    }
}

// The kept keys' columns, and row_ptr[r] = first position whose row is >= r: the first key of
// a row writes its own entry and those of the empty rows before it, the last key those after it.
__global__ void __launch_bounds__(kUniqThreads)
    emit_csr_kernel(const unsigned long long* __restrict__ keys, int64_t K, unsigned long long none,
                    const int32_t* __restrict__ before, int b, int32_t n, int32_t nnz, int32_t* __restrict__ col,
                    int32_t* __restrict__ row_ptr) {
    __shared__ uint32_t part[kUniqThreads / 32];
    __shared__ int32_t tile[kUniqTile];  // the tile's columns, so that they leave coalesced
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x[kUniqItems], prev;
    const int64_t i0 = ((int64_t)blockIdx.x * kUniqThreads + threadIdx.x) * kUniqItems;
    const uint32_t keep = load_unique(keys, K, none, i0, x, prev);
    const uint32_t inc = warp_inclusive_sum((uint32_t)__popc(keep));
    if (lane == 31) part[wid] = inc;
    __syncthreads();
    const uint32_t base = (uint32_t)before[blockIdx.x];
    uint32_t at = inc - (uint32_t)__popc(keep), kept = 0;
#pragma unroll
    for (int w = 0; w < kUniqThreads / 32; ++w) {
        at += w < wid ? part[w] : 0u;
        kept += part[w];
    }
    const unsigned long long cmask = (1ull << b) - 1ull;
    int32_t row = prev == ~0ull && i0 == 0 ? -1 : (int32_t)(prev >> b);
#pragma unroll
    for (int t = 0; t < kUniqItems; ++t) {
        if (!((keep >> t) & 1u)) continue;
        const int32_t r = (int32_t)(x[t] >> b);
        for (int32_t q = row + 1; q <= r; ++q) row_ptr[q] = (int32_t)(base + at);
        row = r;
        tile[at++] = (int32_t)(x[t] & cmask);
        if ((int32_t)(base + at) == nnz)  // the last key
            for (int32_t q = r + 1; q <= n; ++q) row_ptr[q] = nnz;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < kept; i += kUniqThreads) col[base + i] = tile[i];
}

// What the kernels read of each row beside the CSR: its first entry, entries 1..4 (-1 past the
// row's end), whether it has any entry and whether it has two, and the longest row's length.
__global__ void __launch_bounds__(256)
    row_heads_kernel(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int32_t n,
                     int32_t* __restrict__ first, int4* __restrict__ next, uint32_t* __restrict__ nz,
                     uint32_t* __restrict__ multi, int32_t* longest) {
    const int lane = threadIdx.x & 31;
    int32_t most = 0;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < n; i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + lane;
        int32_t d = 0;
        if (i < n) {
            const int32_t b = row_ptr[i];
            d = row_ptr[i + 1] - b;
            first[i] = d > 0 ? col[b] : -1;
            next[i] = make_int4(d > 1 ? col[b + 1] : -1, d > 2 ? col[b + 2] : -1, d > 3 ? col[b + 3] : -1,
                                d > 4 ? col[b + 4] : -1);
        }
        const uint32_t w1 = __ballot_sync(0xffffffffu, d >= 1), w2 = __ballot_sync(0xffffffffu, d >= 2);
        if (lane == 0) {
            nz[i0 >> 5] = w1;
            multi[i0 >> 5] = w2;
        }
        most = max(most, d);
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0 && most > 0) atomicMax(longest, most);
}

static unsigned grid_for(int64_t work) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, 152 * 32)); }

// Temporaries of a build, one allocation: cudaMalloc and cudaFree take about 0.1 ms together
// whatever the size, the stream-ordered pool gives its memory back at every synchronisation
// and takes 1.2 ms for these 540 MB.
struct BuildTemp {
    void* p = nullptr;
    ~BuildTemp() {
        if (p) cudaFree(p);
    }
};

// Sorts the K keys and produces the CSR: row_ptr (given) and col (allocated here).  counts
// needs an int per tile of kUniqTile keys and one more, and room for the scan of those.
static gbx_status keys_to_csr(unsigned long long* keys, unsigned long long* alt, int64_t K, int32_t n, int b, bool drop,
                              int32_t* sort_tmp, int32_t* counts, const int32_t* status, int32_t* row_ptr,
                              int32_t** col_out, int64_t* nnz_out, cudaStream_t s) {
    unsigned long long* k1 = keys;
    unsigned long long* k2 = alt;
    const unsigned long long none = drop ? (1ull << (2 * b)) - 1ull : ~0ull;
    const int64_t tiles = (K + kUniqTile - 1) / kUniqTile;
    int32_t nnz32 = 0, bad = -1;
    if (K > 0) {
        GBX_TRY(radix_sort_u64(&k1, &k2, K, 2 * b, sort_tmp, s));
        count_unique_kernel<<<(unsigned)tiles, kUniqThreads, 0, s>>>(k1, K, none, counts);
        GBX_TRY(exclusive_scan_i32(counts, counts, tiles, nullptr, counts + tiles + 1, s));
        GBX_CUDA_TRY(cudaMemcpyAsync(&nnz32, counts + tiles, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    }
    GBX_CUDA_TRY(cudaMemcpyAsync(&bad, status + ST_BADINDEX, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    GBX_CUDA_TRY(cudaStreamSynchronize(s));
    if (bad >= 0) {
        set_error("edge " + std::to_string(bad) + " has an endpoint outside [0, n)");
        return GBX_ERR_INVALID_INDEX;
    }
    const int64_t nnz = (uint32_t)nnz32;  // K < 2^32 entries; counts below 2^31 checked below
    GBX_CHECK(nnz < ((int64_t)1 << 31), GBX_ERR_OVERFLOW, "graph has 2^31 or more stored edges");
    int32_t* col = nullptr;
    GBX_CUDA_TRY(cudaMalloc((void**)&col, sizeof(int32_t) * (size_t)(nnz + kColPad)));
    *col_out = col;  // the graph's from here on
    *nnz_out = nnz;
    if (nnz > 0)
        emit_csr_kernel<<<(unsigned)tiles, kUniqThreads, 0, s>>>(k1, K, none, counts, b, n, (int32_t)nnz, col, row_ptr);
    else
        GBX_CUDA_TRY(cudaMemsetAsync(row_ptr, 0, sizeof(int32_t) * ((size_t)n + 1), s));
    GBX_CUDA_TRY(cudaGetLastError());
    return GBX_OK;
}

// Hands out 256-byte aligned parts of one allocation: first with base NULL for the size, then again.
struct Carve {
    char* base = nullptr;
    size_t used = 0;
    template <typename T>
    T* take(size_t count) {
        T* r = reinterpret_cast<T*>(base + used);
        used += (sizeof(T) * count + 255) & ~(size_t)255;
        return r;
    }
};

void workspace_release(Workspace& w) {
    auto f = [](void* p) {
        if (p) cudaFree(p);
    };
    f(w.slab);
    f(w.msV);
    for (auto& p : w.msF) f(p);
    f(w.msP);
    f(w.msT);
    f(w.ms_src);
    if (w.ms_src_pinned) cudaFreeHost(w.ms_src_pinned);
    if (w.ms_src_ready) cudaEventDestroy(w.ms_src_ready);
    w = Workspace{};
}

static void graph_release(Graph* g) {
    if (!g) return;
    auto f = [](void* p) {
        if (p) cudaFree(p);
    };
    if (g->in_col != g->out_col) f(g->in_col);
    f(g->out_col);
    f(g->slab);
    if (g->in_val != g->out_val) f(g->in_val);
    f(g->out_val);
    f(g->nzr_in);
    f(g->sp_rec);
    workspace_release(g->ws);
    for (int i = 0; i < 2; ++i) {
        f(g->hdepth[i]);
        f(g->hparent[i]);
        if (g->ev_done[i]) cudaEventDestroy(g->ev_done[i]);
        if (g->ev_copied[i]) cudaEventDestroy(g->ev_copied[i]);
    }
    if (g->copy_stream) cudaStreamDestroy(g->copy_stream);
    delete g;
}

// The parts of a workspace for n vertices; those that start out zero come first (*zero bytes).
static void workspace_carve(Workspace& w, int32_t n, Carve& c, size_t* zero) {
    const size_t nw = (size_t)(n + 31) / 32 + 1;
    const size_t nn = (size_t)n + 1;
    w.bar = c.take<GridBar>(1);
    w.status = c.take<int32_t>(ST_WORDS);
    w.flag = c.take<int32_t>(64);
    w.mx_ctr = c.take<LevelCtr>(1);
    w.mx_bm[0] = c.take<uint32_t>(3 * nw);
    w.mx_bm[1] = w.mx_bm[0] + nw;
    w.mx_bm[2] = w.mx_bm[1] + nw;
    *zero = c.used;
    for (auto& p : w.bm) p = c.take<uint32_t>(nw);
    for (int i = 0; i < 2; ++i) {  // one after another: the batched BFS on meshes uses the three as one list
        w.q[i] = c.take<int32_t>(nn);
        w.qp[i] = c.take<int32_t>(nn);
        w.qd[i] = c.take<int32_t>(nn);
    }
    w.list = c.take<int32_t>(nn);
    w.scan_tmp = c.take<int32_t>(scan_tmp_ints((int64_t)nn));
    w.ctr = c.take<LevelCtr>(4);
    w.trace = c.take<LevelRec>(kTraceCap);
    w.handoff = c.take<ClHandoff>(1);
}

static gbx_status workspace_alloc_all(Workspace& w, int32_t n, cudaStream_t s) {
    Carve c;
    size_t zero = 0;
    workspace_carve(w, n, c, &zero);
    GBX_CUDA_TRY(cudaMalloc(&w.slab, c.used));
    c.base = static_cast<char*>(w.slab);
    c.used = 0;
    workspace_carve(w, n, c, &zero);
    GBX_CUDA_TRY(cudaMemsetAsync(w.slab, 0, zero, s));
    w.n_cap = n;  // only once every buffer exists
    return GBX_OK;
}

// All or nothing: a failed allocation releases what was allocated, so no half-built
// workspace (one that claims capacity n but holds null buffers) is ever left behind.
gbx_status workspace_alloc(Workspace& w, int32_t n, cudaStream_t s) {
    const gbx_status st = workspace_alloc_all(w, n, s);
    if (st != GBX_OK) workspace_release(w);
    return st;
}

static gbx_status build_impl(Graph* g, int32_t n, int64_t m, const int32_t* src, const int32_t* dst, uint32_t flags,
                             cudaStream_t s) {
    const int sym = (flags & GBX_SYMMETRIZE) ? 1 : 0;
    const int drop = (flags & GBX_DROP_SELF_LOOPS) ? 1 : 0;
    GBX_CUDA_TRY(cudaGetDevice(&g->device));
    GBX_CUDA_TRY(cudaDeviceGetAttribute(&g->num_sms, cudaDevAttrMultiProcessorCount, g->device));
    g->n = n;
    g->nwords = (n + 31) / 32;
    g->symmetric = sym;
    g->drop_self_loops = drop;
    GBX_TRY(workspace_alloc(g->ws, n, s));

    const int64_t K = sym ? 2 * m : m;
    GBX_CHECK(K < ((int64_t)1 << 32), GBX_ERR_OVERFLOW, "too many edge entries (2^32 or more)");
    const int b = bits_for((int64_t)n - 1);

    // the arrays whose size follows from n
    for (int pass = 0; pass < 2; ++pass) {
        Carve c;
        c.base = static_cast<char*>(g->slab);
        g->out_ptr = c.take<int32_t>((size_t)n + 1);
        g->in_ptr = sym ? g->out_ptr : c.take<int32_t>((size_t)n + 1);
        g->nz_in = c.take<uint32_t>((size_t)g->nwords + 1);
        g->multi_in = c.take<uint32_t>((size_t)g->nwords + 1);
        g->first_in = c.take<int32_t>((size_t)n + 1);
        g->next_in = c.take<int4>((size_t)n + 1);
        g->nz_out = sym ? g->nz_in : c.take<uint32_t>((size_t)g->nwords + 1);
        g->multi_out = sym ? g->multi_in : c.take<uint32_t>((size_t)g->nwords + 1);
        g->first_out = sym ? g->first_in : c.take<int32_t>((size_t)n + 1);
        g->next_out = sym ? g->next_in : c.take<int4>((size_t)n + 1);
        if (pass == 0) GBX_CUDA_TRY(cudaMalloc(&g->slab, c.used));
    }

    // temporaries: two key buffers, the sort's and the deduplication's scratch, a device copy of a host edge list
    const bool on_host = !(flags & GBX_DEVICE_EDGES) && m > 0;
    const int64_t tiles = (K + kUniqTile - 1) / kUniqTile;
    BuildTemp temp;
    unsigned long long* keys = nullptr;
    unsigned long long* alt = nullptr;
    int32_t* sort_tmp = nullptr;
    int32_t* counts = nullptr;
    int32_t* own = nullptr;
    for (int pass = 0; pass < 2; ++pass) {
        Carve c;
        c.base = static_cast<char*>(temp.p);
        keys = c.take<unsigned long long>((size_t)K + 1);
        alt = c.take<unsigned long long>((size_t)K + 1);
        sort_tmp = c.take<int32_t>(radix_tmp_ints(K));
        counts = c.take<int32_t>((size_t)tiles + 1 + scan_tmp_ints(tiles));
        own = c.take<int32_t>(on_host ? 2 * (size_t)m : 0);
        if (pass == 0) GBX_CUDA_TRY(cudaMalloc(&temp.p, c.used));
    }
    const int32_t* dsrc = src;
    const int32_t* ddst = dst;
    if (on_host) {
        GBX_CUDA_TRY(cudaMemcpyAsync(own, src, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, s));
        GBX_CUDA_TRY(cudaMemcpyAsync(own + m, dst, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, s));
        dsrc = own;
        ddst = own + m;
    }
    GBX_CUDA_TRY(cudaMemsetAsync(g->ws.status + ST_BADINDEX, 0xff, sizeof(int32_t), s));
    if (m > 0) make_keys_kernel<<<grid_for(m), 256, 0, s>>>(dsrc, ddst, m, n, b, sym, drop, 0, keys, g->ws.status);
    GBX_TRY(keys_to_csr(keys, alt, K, n, b, drop != 0, sort_tmp, counts, g->ws.status, g->out_ptr, &g->out_col, &g->nnz, s));
    if (sym) {
        g->in_col = g->out_col;
    } else {
        // A^T: the same entries with row and column exchanged
        if (m > 0) make_keys_kernel<<<grid_for(m), 256, 0, s>>>(dsrc, ddst, m, n, b, 0, drop, 1, keys, g->ws.status);
        int64_t nnz_t = 0;
        GBX_TRY(keys_to_csr(keys, alt, K, n, b, drop != 0, sort_tmp, counts, g->ws.status, g->in_ptr, &g->in_col, &nnz_t, s));
        GBX_CHECK(nnz_t == g->nnz, GBX_ERR_CUDA, "internal: transpose has a different edge count");
    }
    int32_t* const longest = g->ws.flag + 10;  // of the out-rows and of the in-rows: zero since the workspace was made
    row_heads_kernel<<<grid_for(n), 256, 0, s>>>(g->out_ptr, g->out_col, n, g->first_out, g->next_out, g->nz_out,
                                                 g->multi_out, longest);
    if (!sym)
        row_heads_kernel<<<grid_for(n), 256, 0, s>>>(g->in_ptr, g->in_col, n, g->first_in, g->next_in, g->nz_in,
                                                     g->multi_in, longest + 1);
    GBX_CUDA_TRY(cudaGetLastError());
    int32_t most[2] = {0, 0};
    GBX_CUDA_TRY(cudaMemcpyAsync(most, longest, sizeof(most), cudaMemcpyDeviceToHost, s));
    GBX_CUDA_TRY(cudaStreamSynchronize(s));
    g->max_out_degree = most[0];
    g->max_in_degree = sym ? most[0] : most[1];
    return GBX_OK;
}

}  // namespace gbx

using namespace gbx;

extern "C" gbx_status gbx_graph_build(gbx_graph** out, int32_t n, int64_t m, const int32_t* src, const int32_t* dst,
                                      uint32_t flags, void* stream) {
    clear_error();
    GBX_CHECK(out != nullptr, GBX_ERR_NULL_POINTER, "out is NULL");
    *out = nullptr;
    GBX_CHECK(n >= 1, GBX_ERR_INVALID_VALUE, "n must be >= 1");
    GBX_CHECK(m >= 0, GBX_ERR_INVALID_VALUE, "m must be >= 0");
    GBX_CHECK((flags & ~(GBX_SYMMETRIZE | GBX_DROP_SELF_LOOPS | GBX_DEVICE_EDGES)) == 0, GBX_ERR_INVALID_VALUE,
              "unknown flag bits");
    GBX_CHECK(m == 0 || (src != nullptr && dst != nullptr), GBX_ERR_NULL_POINTER, "src or dst is NULL");
    Graph* g = new (std::nothrow) Graph();
    GBX_CHECK(g != nullptr, GBX_ERR_OUT_OF_MEMORY, "host allocation failed");
    const gbx_status st = build_impl(g, n, m, src, dst, flags, (cudaStream_t)stream);
    if (st != GBX_OK) {
        graph_release(g);
        return st;
    }
    *out = reinterpret_cast<gbx_graph*>(g);
    return GBX_OK;
}

extern "C" gbx_status gbx_graph_free(gbx_graph* g) {
    clear_error();
    if (!g) return GBX_OK;
    Graph* G = as_impl(g);
    cudaDeviceSynchronize();
    graph_release(G);
    return GBX_OK;
}

extern "C" gbx_status gbx_graph_info(const gbx_graph* g, int32_t* n, int64_t* nnz, int32_t* symmetric) {
    clear_error();
    GBX_TRY(check_graph(g));
    const Graph* G = as_impl(g);
    if (n) *n = G->n;
    if (nnz) *nnz = G->nnz;
    if (symmetric) *symmetric = G->symmetric;
    return GBX_OK;
}

extern "C" gbx_status gbx_graph_csr(const gbx_graph* g, int32_t transpose, const int32_t** row_ptr,
                                    const int32_t** col) {
    clear_error();
    GBX_TRY(check_graph(g));
    GBX_CHECK(row_ptr != nullptr && col != nullptr, GBX_ERR_NULL_POINTER, "row_ptr or col is NULL");
    const Graph* G = as_impl(g);
    *row_ptr = transpose ? G->in_ptr : G->out_ptr;
    *col = transpose ? G->in_col : G->out_col;
    return GBX_OK;
}

extern "C" gbx_status gbx_graph_copy_csr(const gbx_graph* g, int32_t transpose, int32_t* row_ptr_dst,
                                         int32_t* col_dst) {
    clear_error();
    GBX_TRY(check_graph(g));
    GBX_CHECK(row_ptr_dst != nullptr && col_dst != nullptr, GBX_ERR_NULL_POINTER, "destination is NULL");
    const Graph* G = as_impl(g);
    GBX_CUDA_TRY(cudaDeviceSynchronize());
    GBX_CUDA_TRY(cudaMemcpy(row_ptr_dst, transpose ? G->in_ptr : G->out_ptr, sizeof(int32_t) * ((size_t)G->n + 1),
                            cudaMemcpyDefault));
    if (G->nnz > 0)
        GBX_CUDA_TRY(cudaMemcpy(col_dst, transpose ? G->in_col : G->out_col, sizeof(int32_t) * (size_t)G->nnz,
                                cudaMemcpyDefault));
    return GBX_OK;
}

extern "C" gbx_status gbx_graph_sync(gbx_graph* g, void* stream) {
    clear_error();
    GBX_TRY(check_graph(g));
    Graph* G = as_impl(g);
    cudaStream_t s = (cudaStream_t)stream;
    GBX_CUDA_TRY(cudaStreamSynchronize(s));
    if (G->ws.last_stream && G->ws.last_stream != s) GBX_CUDA_TRY(cudaStreamSynchronize(G->ws.last_stream));
    int32_t err = 0;
    GBX_CUDA_TRY(cudaMemcpy(&err, G->ws.status + ST_ERROR, sizeof(int32_t), cudaMemcpyDeviceToHost));
    if (err != 0) {
        // a kernel gave up: clear the error and the barrier it may have left half-arrived
        GBX_CUDA_TRY(cudaMemset(G->ws.status + ST_ERROR, 0, sizeof(int32_t)));
        GBX_CUDA_TRY(cudaMemset(G->ws.bar, 0, sizeof(GridBar)));
        set_error(err == GBX_ERR_TIMEOUT ? "a bounded device-side wait ran out" : "device-side error");
        return (gbx_status)err;
    }
    return GBX_OK;
}
