// Graph pre-processing (Sec. 3.1): index partitions, PNG layout of Alg. 3 with
// destination lists written once, SC bin capacities, gather/scatter task lists.
// Runs once per graph on the GPU; CUB radix sorts and scans are used as
// library primitives here (this step is outside the iteration hot path).
#include <cub/cub.cuh>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <functional>
#include <mutex>
#include <utility>
#include <vector>

#include "gpop_internal.cuh"

namespace gpop {

static thread_local std::string g_last_error;

void set_error(const std::string &msg) { g_last_error = msg; }

gpop_status fail(gpop_status st, const std::string &msg) {
    if (st == GPOP_ERR_OOM) cudaGetLastError();  // reported here: not the next call's error too
    g_last_error = msg;
    return st;
}

void free_graph(Graph *g) {
    release_run_state(g);
    void *ptrs[] = {g->rowptr, g->col, g->w, g->esub, g->row_bin, g->bin_q,
                    g->png, g->pdata, g->png_dst, g->pc_blk_src, g->pc_blk_nval, g->pc_blk_prange,
                    g->pc_task, g->pc_tsp, g->pc_rng, g->pc_merge, g->col_ntask, g->col_part0, g->pc_part, g->pe, g->pw,
                    g->scpair, g->sccnt, g->sub_cap, g->sub_task, g->row_sub, g->task_sub_ptr,
                    g->Ep, g->npng_p, g->gtask, g->col_task, g->stask, g->pc_state,
                    g->sm_range, g->sm_edge, g->sm_w, g->in_off, g->in_edge, g->in_span};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete[] g->h_Ep;
    delete[] g->h_npng;
    *g = Graph();
}

namespace {

// Temporary device buffers of one build, in stream order out of a memory pool of the build's own: a buffer that a step
// no longer needs is released for the next one without waiting for the device (cudaMalloc and cudaFree took a third of
// a small graph's build, 1.7 of 2.9 ms, and kept the host from running ahead of the device).  The pool ends with the
// build.  A large buffer (kTrimBytes) goes back to the device when it is released, so that the build's peak footprint
// stays a few steps' buffers besides the layout; the others go back when an allocation fails without them.
struct Temps {
    static constexpr uint64_t kTrimBytes = 2ull << 30;
    cudaStream_t s;
    cudaMemPool_t pool = nullptr;
    std::vector<std::pair<void *, uint64_t>> ptrs;
    explicit Temps(cudaStream_t stream) : s(stream) {}
    Temps(const Temps &) = delete;
    template <typename T>
    cudaError_t alloc(T **p, uint64_t count) {
        cudaError_t e = cudaSuccess;
        if (!pool) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            e = cudaGetDevice(&props.location.id);
            if (e == cudaSuccess) e = cudaMemPoolCreate(&pool, &props);
            uint64_t keep = ~0ull;  // freed memory stays in the pool until the build ends
            if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) return e;
        }
        const uint64_t bytes = sizeof(T) * std::max<uint64_t>(count, 1);
        e = cudaMallocFromPoolAsync((void **)p, bytes, pool, s);
        if (e == cudaErrorMemoryAllocation && again()) e = cudaMallocFromPoolAsync((void **)p, bytes, pool, s);
        if (e == cudaSuccess) ptrs.emplace_back(*p, bytes);
        return e;
    }
    // an array of the graph's own (which does not come out of the pool)
    template <typename T>
    cudaError_t keep(Graph *g, T **p, uint64_t count) {
        cudaError_t e = dalloc(g, p, count);
        if (e == cudaErrorMemoryAllocation && again()) e = dalloc(g, p, count);
        return e;
    }
    // gives what has been released back to the device
    bool trim() { return cudaStreamSynchronize(s) == cudaSuccess && cudaMemPoolTrimTo(pool, 0) == cudaSuccess; }
    // whether to try an allocation once more that has failed
    bool again() {
        cudaGetLastError();
        return pool && trim();
    }
    void release(void *p) {
        for (size_t i = 0; i < ptrs.size(); ++i)
            if (ptrs[i].first == p) {
                const bool large = ptrs[i].second >= kTrimBytes;
                cudaFreeAsync(p, s);
                ptrs.erase(ptrs.begin() + (long)i);
                if (large) trim();
                return;
            }
    }
    ~Temps() {
        for (auto &p : ptrs) cudaFreeAsync(p.first, s);
        if (pool) {
            cudaStreamSynchronize(s);
            cudaMemPoolDestroy(pool);
        }
    }
};

struct MaxOp {
    __host__ __device__ uint32_t operator()(uint32_t a, uint32_t b) const { return a > b ? a : b; }
};

constexpr int kThreads = 256;

inline unsigned blocks_for(uint64_t n, int per = kThreads) {
    uint64_t b = (n + per - 1) / per;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(b, 1u << 22));
}

// --- validation --------------------------------------------------------------------------------

__global__ void k_validate(uint32_t V, uint64_t E, const uint64_t *rp, const uint32_t *col,
                           const int32_t *w, uint32_t *err) {  // err[1]: the largest weight
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    int32_t wmax = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= V; i += stride) {
        if (i == 0 && rp[0] != 0) atomicOr(err, 1u);
        if (i == V && rp[V] != E) atomicOr(err, 2u);
        if (i < V && rp[i] > rp[i + 1]) atomicOr(err, 4u);
    }
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        if (col[e] >= V) atomicOr(err, 8u);
        if (w && w[e] < 0) atomicOr(err, 16u);
        if (w) wmax = max(wmax, w[e]);
    }
    if (wmax > 0) atomicMax(&err[1], (uint32_t)wmax);
}

__global__ void k_rowptr32(uint32_t V, const uint64_t *rp, uint32_t *out) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= V; i += stride)
        out[i] = (uint32_t)rp[i];
}

// source vertex of every edge: largest u with rowptr[u] <= e.  A CTA takes a tile of edges and searches the tile's first
// and last source in all rows, the others between them: the searches stay short and in L1.  Raises *unsorted when a
// row's destinations are not in ascending order.
constexpr uint32_t kSrcTile = 8 * kThreads;
__global__ void __launch_bounds__(kThreads) k_edge_src(uint32_t V, uint64_t E, const uint32_t *rowptr, const uint32_t *col,
                                                       uint32_t *src, uint32_t *unsorted) {
    __shared__ uint32_t s_row[2];
    auto row_of = [&](uint64_t e, uint32_t lo, uint32_t hi) {  // rowptr[lo] <= e < rowptr[hi]
        while (hi - lo > 1) {
            const uint32_t mid = lo + (hi - lo) / 2;
            if (rowptr[mid] <= (uint32_t)e) lo = mid; else hi = mid;
        }
        return lo;
    };
    for (uint64_t base = blockIdx.x * (uint64_t)kSrcTile; base < E; base += gridDim.x * (uint64_t)kSrcTile) {
        const uint64_t end = min(base + kSrcTile, E);
        if (threadIdx.x < 2) s_row[threadIdx.x] = row_of(threadIdx.x ? end - 1 : base, 0, V);
        __syncthreads();
        const uint32_t lo = s_row[0], hi = s_row[1] + 1;
        for (uint64_t e = base + threadIdx.x; e < end; e += kThreads) {
            const uint32_t u = row_of(e, lo, hi);
            src[e] = u;
            if (e > rowptr[u] && col[e] < col[e - 1]) atomicOr(unsorted, 1u);
        }
        __syncthreads();
    }
}

__global__ void k_pack_src_dst(uint64_t E, const uint32_t *src, const uint32_t *col, uint64_t *key) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride)
        key[e] = ((uint64_t)src[e] << 32) | col[e];
}

__global__ void k_unpack_dst(uint64_t E, const uint64_t *key, uint32_t *col) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride)
        col[e] = (uint32_t)key[e];
}

// A message (Sec. 3.1.2) is one (source, destination partition) pair; its first
// edge in the destination-sorted row is the head.
__global__ void k_heads(uint64_t E, uint32_t shift, uint32_t k, const uint32_t *rowptr, const uint32_t *src,
                        const uint32_t *col, uint8_t *head, uint64_t *mkey, uint32_t *head_idx) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        uint32_t u = src[e], q = col[e] >> shift;
        bool h = (e == rowptr[u]) || ((col[e - 1] >> shift) != q);
        head[e] = h;
        uint32_t p = u >> shift, ul = u & ((1u << shift) - 1);
        mkey[e] = ((((uint64_t)p * k + q)) << shift) | ul;  // sort key (bin, local source)
        head_idx[e] = h ? (uint32_t)e : 0u;                 // for the max-scan
    }
}

// per sorted message j: does it start a new bin?
__global__ void k_msg_bins(uint64_t nmsg, uint32_t shift, const uint64_t *skey, uint32_t *newbin) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < nmsg; j += stride)
        newbin[j] = (j == 0) || ((skey[j - 1] >> shift) != (skey[j] >> shift));
}

// Segment starts of keys sorted by seg(i) = (key[i] >> sh) / div, seg < nseg: start[s] = first index with
// seg >= s for s in [0, nseg], start[nseg] = n.  Each boundary writes the starts it crosses (no atomics).
__global__ void k_seg_starts(uint64_t n, const uint64_t *key, uint32_t sh, uint64_t div, uint32_t nseg,
                             uint32_t *start) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= n; i += stride) {
        const uint32_t hi = i < n ? (uint32_t)((key[i] >> sh) / div) : nseg;
        const uint32_t lo = i == 0 ? 0u : (uint32_t)((key[i - 1] >> sh) / div) + 1;
        for (uint32_t sg = lo; sg <= hi && sg <= nseg; ++sg) start[sg] = (uint32_t)i;
    }
}

// per row p: messages and bins, from the row's message range and the inclusive scan of new-bin flags
__global__ void k_row_counts(uint32_t k, const uint32_t *row_start, const uint32_t *binscan, uint32_t *msgs_row,
                             uint32_t *bins_row) {
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < k; p += gridDim.x * blockDim.x) {
        const uint32_t a = row_start[p], b = row_start[p + 1];
        msgs_row[p] = b - a;
        bins_row[p] = b > a ? binscan[b - 1] - (a > 0 ? binscan[a - 1] : 0u) : 0u;
    }
}

__global__ void k_pad8(uint32_t k, const uint32_t *m, uint32_t *mp) {
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < k; p += gridDim.x * blockDim.x)
        mp[p] = (m[p] + kPngAlign - 1) / kPngAlign * kPngAlign;
}

// first message (sorted order), destination partition and source partition of every bin
__global__ void k_bin_starts(uint64_t nmsg, uint32_t shift, uint32_t k, const uint64_t *skey, const uint32_t *binscan,
                             uint32_t *bin_j0, uint32_t *bin_q, uint32_t *bin_p) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < nmsg; j += stride) {
        uint64_t pk = skey[j] >> shift;
        if (j == 0 || (skey[j - 1] >> shift) != pk) {
            uint32_t b = binscan[j] - 1;
            bin_j0[b] = (uint32_t)j;
            bin_q[b] = (uint32_t)(pk % k);
            bin_p[b] = (uint32_t)(pk / k);
        }
    }
}

// every bin occupies its message count rounded up to kBinAlign slots of its PNG row (so that each bin,
// and each block of a column's message sequence, starts 16-byte aligned); per row, the padded length
__global__ void k_bin_pad(uint32_t nb, const uint32_t *bin_j0, const uint32_t *bin_p, uint32_t *cnt4,
                          uint32_t *row_len4) {
    for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        uint32_t c = (bin_j0[b + 1] - bin_j0[b] + kBinAlign - 1) / kBinAlign * kBinAlign;
        cnt4[b] = c;
        atomicAdd(&row_len4[bin_p[b]], c);
    }
}

// places every message in its PNG slot (row start + padded offset of its bin + rank in the bin) and records the
// column-major slot of its value (bin_cslot0: the bin's first), per head edge and per group of 8 PNG slots
__global__ void k_place_msgs(uint64_t nmsg, uint32_t shift, const uint64_t *skey, const uint32_t *shead,
                             const uint32_t *binscan, const uint32_t *bin_j0, const uint32_t *bin_p,
                             const uint32_t *binoff, const uint32_t *row_bin, const uint32_t *row_png,
                             const uint32_t *bin_cslot0, uint16_t *png, uint32_t *png_dst, uint32_t *cslot_of_head) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < nmsg; j += stride) {
        const uint32_t b = binscan[j] - 1, p = bin_p[b], i = (uint32_t)j - bin_j0[b], cslot = bin_cslot0[b] + i;
        const uint32_t slot = row_png[p] + (binoff[b] - binoff[row_bin[p]]) + i;
        png[slot] = (uint16_t)(skey[j] & ((1u << shift) - 1));
        cslot_of_head[shead[j]] = cslot;
        if (i % kBinAlign == 0) png_dst[slot / kBinAlign] = cslot / kBinAlign;
    }
}

// padded lengths of the bins in column order
__global__ void k_col_lengths(uint64_t nb, const uint32_t *col_bins, const uint32_t *cnt4, uint32_t *len) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < nb; i += stride) len[i] = cnt4[col_bins[i]];
}
// column-major slots: first of every bin and of every column, from the scanned lengths (coff: nb + 1)
__global__ void k_col_slots(uint64_t nb, uint32_t k, const uint32_t *col_bins, const uint32_t *col_bin, const uint32_t *coff,
                            uint32_t *bin_cslot0, uint32_t *col_off) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x, t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    for (uint64_t i = t; i < nb; i += stride) bin_cslot0[col_bins[i]] = coff[i];
    for (uint64_t q = t; q <= k; q += stride) col_off[q] = coff[col_bin[q]];
}
// first and last source partition of every gather block's bins (prange starts as (0xFFFFFFFF, 0))
__global__ void k_blk_prange(uint64_t nb, const uint32_t *bin_q, const uint32_t *bin_p, const uint32_t *cnt4,
                             const uint32_t *bin_cslot0, const uint32_t *col_off, const uint32_t *col_blk0, uint2 *prange) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b < nb; b += stride) {
        const uint32_t q = bin_q[b], s0 = bin_cslot0[b] - col_off[q], s1 = s0 + cnt4[b] - 1;
        for (uint32_t blk = s0 / kPcBlock; blk <= s1 / kPcBlock; ++blk) {
            atomicMin(&prange[col_blk0[q] + blk].x, bin_p[b]);
            atomicMax(&prange[col_blk0[q] + blk].y, bin_p[b]);
        }
    }
}

// key of every PC in-entry: (gather block << 32) | (local destination << 16) | index in the block,
// where the message of edge e is the one of its head (same source, same destination partition)
__global__ void k_pc_keys(uint64_t E, uint32_t shift, uint32_t P, const uint32_t *head_of, const uint32_t *cslot_of_head,
                          const uint32_t *col, const uint32_t *col_off, const uint32_t *col_blk0, uint64_t *key) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        const uint32_t v = col[e], q = v >> shift, cseq = cslot_of_head[head_of[e]] - col_off[q];
        key[e] = ((uint64_t)(col_blk0[q] + cseq / kPcBlock) << 32) | ((uint64_t)(v & (P - 1)) << 16) | (cseq % kPcBlock);
    }
}

__global__ void k_pc_unpack(uint64_t E, const uint64_t *key, uint32_t *pe) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < E; i += stride) pe[i] = (uint32_t)key[i];
}

// gather task of every destination
__global__ void k_task_of(const GatherTask *gtask, uint32_t shift, uint32_t V, uint32_t *task_of) {
    const GatherTask gt = gtask[blockIdx.x];
    const uint32_t lo = (gt.q << shift) + gt.d0, hi = min((gt.q << shift) + gt.d1, V);
    for (uint32_t v = lo + threadIdx.x; v < hi; v += blockDim.x) task_of[v] = blockIdx.x;
}

// SC bins are (source partition p, gather task t) pairs: key p * tasks + t per edge
template <typename K>
__global__ void k_sub_keys(uint64_t E, uint32_t shift, uint32_t ngt, const uint32_t *src, const uint32_t *col,
                           const uint32_t *task_of, K *key) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride)
        key[e] = (K)(src[e] >> shift) * ngt + task_of[col[e]];
}

template <typename K>
__global__ void k_sub_split(uint64_t nsub, uint32_t ngt, const K *ukey, uint32_t *sub_task, uint32_t *row_hist,
                            uint32_t *task_hist) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < nsub; s += stride) {
        const uint32_t tsk = (uint32_t)(ukey[s] % ngt);
        sub_task[s] = tsk;
        atomicAdd(&row_hist[(uint32_t)(ukey[s] / ngt)], 1u);
        atomicAdd(&task_hist[tsk], 1u);
    }
}

// index of every edge's SC bin within its bin row (binary search of its task in the row)
__global__ void k_edge_sub(uint64_t E, uint32_t shift, const uint32_t *src, const uint32_t *col,
                           const uint32_t *task_of, const uint32_t *row_sub, const uint32_t *sub_task, uint16_t *esub) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        uint32_t p = src[e] >> shift, tsk = task_of[col[e]];
        uint32_t lo = row_sub[p], hi = row_sub[p + 1];  // sub_task[lo..hi) ascending, contains tsk
        while (hi - lo > 1) {
            uint32_t mid = (lo + hi) >> 1;
            if (sub_task[mid] <= tsk) lo = mid; else hi = mid;
        }
        esub[e] = (uint16_t)(lo - row_sub[p]);
    }
}

// splitmix64's output function (Steele, Lea, Flood 2014): a bijective 64-bit mix
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
// Fingerprint of the graph for checkpoints: the sum (mod 2^64) over edges of a mixed (source, destination,
// weight) key, so it depends on the edge multiset only, not on the order of the sums
__global__ void k_fingerprint(uint64_t E, const uint32_t *src, const uint32_t *col, const int32_t *w,
                              unsigned long long *out) {
    unsigned long long acc = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        const uint64_t wt = w ? (uint32_t)w[e] : 0u;
        acc += mix64((((uint64_t)src[e] << 32) | col[e]) ^ mix64(wt + 0x9E3779B97F4A7C15ull));
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

// first entry of [l, h) (sorted by destination) whose destination is at least D
__device__ __forceinline__ uint32_t first_dest_at_least(const uint32_t *pe, uint32_t l, uint32_t h, uint32_t D) {
    while (l < h) {
        const uint32_t m = l + (h - l) / 2;
        if ((pe[m] >> 16) < D) l = m + 1; else h = m;
    }
    return l;
}

// in-degree of every 32-vertex block of destinations (where the gather tasks are cut), from the sorted entries: one
// thread per (gather block, 32 destinations of its column)
__global__ void k_block_indeg(uint64_t nblocks, uint32_t P, const uint32_t *blk_col, const uint32_t *blk_ent,
                              const uint32_t *pe, uint32_t *cnt) {
    const uint32_t per = P / 32;
    const uint64_t n = nblocks * per, stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t b = (uint32_t)(i / per), j = (uint32_t)(i % per), lo = blk_ent[b], hi = blk_ent[b + 1];
        const uint32_t e0 = first_dest_at_least(pe, lo, hi, j * 32), e1 = first_dest_at_least(pe, e0, hi, j * 32 + 32);
        if (e1 > e0) atomicAdd(&cnt[(uint64_t)blk_col[b] * per + j], e1 - e0);
    }
}

// Destination cuts of the PC gather's warps, one set per task: the w-th cut (w = 1 .. kPcGatherWarps - 1)
// of task t is the smallest destination D such that at least w / kPcGatherWarps of the task's entries (over
// all its blocks, rows [row0[t], row0[t + 1]) with entries [lo, hi) each, sorted by destination) go to
// destinations below D.  Warp w then owns destinations [D_w, D_w+1) in every block of the task, so that
// gather warps working on different blocks never touch one destination.
__global__ void k_task_cuts(uint32_t ntask, uint32_t P, const uint32_t *row0, const uint32_t *lo, const uint32_t *hi,
                            const uint32_t *pe, uint32_t *cut) {
    constexpr uint32_t kW = kPcGatherWarps;
    const uint64_t n = (uint64_t)ntask * (kW - 1), stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t t = (uint32_t)(i / (kW - 1)), w = (uint32_t)(i % (kW - 1)) + 1;
        uint64_t total = 0;
        for (uint32_t r = row0[t]; r < row0[t + 1]; ++r) total += hi[r] - lo[r];
        const uint64_t target = (total * w + kW - 1) / kW;
        uint32_t a = 0, b = P;  // smallest D in [0, P] with count(dest < D) >= target
        while (a < b) {
            const uint32_t D = a + (b - a) / 2;
            uint64_t c = 0;
            for (uint32_t r = row0[t]; r < row0[t + 1]; ++r) c += first_dest_at_least(pe, lo[r], hi[r], D) - lo[r];
            if (c >= target) b = D; else a = D + 1;
        }
        cut[i] = a;
    }
}

// Warp splits of the PC gather: for every task block (entries [lo, hi), sorted by destination) and w in
// 0..kPcGatherWarps, the first entry of warp w's destinations [D_w, D_w+1) under its task's cuts.
__global__ void k_warp_splits(uint32_t nrow, const uint32_t *lo, const uint32_t *hi, const uint32_t *row_task,
                              const uint32_t *cut, const uint32_t *pe, uint32_t *out) {
    constexpr uint32_t kSp = kPcGatherWarps + 1;
    uint64_t n = (uint64_t)nrow * kSp, stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t r = (uint32_t)(i / kSp), w = (uint32_t)(i % kSp);
        const uint32_t l = lo[r], h = hi[r];
        uint32_t a = w == 0 ? l : h;
        if (w > 0 && w < kPcGatherWarps)
            a = first_dest_at_least(pe, l, h, cut[(uint64_t)row_task[r] * (kPcGatherWarps - 1) + w - 1]);
        out[i] = a;
    }
}

// Quads of every range (the entries of one gather warp in one task block; see kPcRunA): one CTA per range walks its
// entries, sorted by destination, in tiles; the thread at a run's first entry finds the run's length.  Without WRITE
// it counts the range's runs of the classes A, B, C and quads of class D (cls) and its quads; with WRITE it places every run at its rank in its class.  Ranks come from block scans, so the layout
// does not depend on timing.  A class's first quad takes the slack of the last: its unused places come before the
// run they name, so that the gather, which reads the accumulator words of a quad before it writes them in order,
// ends with that run's result.
// Place of piece x of a range's n pieces of class D: rows of 64 quads, of which a gather lane takes number l and
// 32 + l; consecutive pieces fill the lanes in order, two in each of the first lanes.
__device__ __forceinline__ uint32_t piece_place(uint32_t x, uint32_t n) {
    const uint32_t row = x / 64 * 64, t = x - row, m = min(64u, n - row), two = m > 32 ? m - 32 : 0u;
    return row + (t < 2 * two ? (t & 1) * 32 + t / 2 : t - two);
}
constexpr int kQuadThreads = 128;
constexpr uint32_t kPieceSelf = 16;  // a D run of more pieces is written by the whole CTA

template <bool WRITE>
__global__ void __launch_bounds__(kQuadThreads) k_range_quads(uint32_t nrange, const uint32_t *sp, const uint32_t *pe,
                                                              const int32_t *pw, uint4 *cls, uint32_t *nquad,
                                                              const uint32_t *qoff, uint4 *rng, uint4 *pe2, uint4 *pw2, bool w16) {
    using ScanC = cub::BlockScan<unsigned long long, kQuadThreads>;
    using ScanD = cub::BlockScan<uint32_t, kQuadThreads>;
    __shared__ typename ScanC::TempStorage s_c;
    __shared__ typename ScanD::TempStorage s_d;
    __shared__ uint32_t s_cnt[4], s_nbig, s_bi[kQuadThreads], s_bl[kQuadThreads], s_bq[kQuadThreads];
    constexpr uint32_t kW = kPcGatherWarps, kPad = kPcPadIdx * 4u;
    const uint32_t tid = threadIdx.x;
    for (uint32_t r = blockIdx.x; r < nrange; r += gridDim.x) {
        const uint32_t row = r / kW, w = r % kW;
        const uint32_t a = sp[(uint64_t)row * (kW + 1) + w], b = sp[(uint64_t)row * (kW + 1) + w + 1];
        uint32_t qA = 0, qB = 0, qC = 0, qD = 0, padA = 0, padB = 0, q0 = 0;
        uint32_t rA = 0, rB = 0, rC = 0, rD = 0;  // runs (quads of D) before the tile; without WRITE: this thread's
        if (WRITE) {
            const uint4 c = cls[r];
            qA = (c.x + 3) / 4; qB = (c.y + 1) / 2; qC = c.z; qD = c.w;
            padA = qA * 4 - c.x; padB = qB * 2 - c.y;
            q0 = qoff[r];
            if (tid == 0) rng[r] = make_uint4(q0, qA | qB << 16, qC, 0u);
        } else if (tid < 4) {
            s_cnt[tid] = 0;
        }
        uint32_t *const words = reinterpret_cast<uint32_t *>(pe2 + q0);
        uint4 *const wq = pw2 ? pw2 + (w16 ? 1ull : 2ull) * q0 : nullptr;  // one or two weight quads for each quad
        for (uint32_t off = 0; off < b - a; off += kQuadThreads) {
            const uint32_t i = a + off + tid;
            uint32_t d = 0, L = 0;  // the run that starts at entry i (L = 0: none)
            if (off + tid < b - a) {
                d = pe[i] >> 16;
                if (i == a || (pe[i - 1] >> 16) != d) {
                    if (b - i <= kPcRunC || (pe[i + kPcRunC] >> 16) != d) {
                        L = 1;
                        while (L < b - i && (pe[i + L] >> 16) == d) ++L;
                    } else {
                        L = first_dest_at_least(pe, i + kPcRunC + 1, b, d + 1) - i;
                    }
                }
            }
            const bool isA = L == kPcRunA, isB = L > kPcRunA && L <= kPcRunB, isC = L > kPcRunB && L <= kPcRunC;
            const uint32_t nD = L > kPcRunC ? (L + kPcRunC - 1) / kPcRunC : 0u;
            if (!WRITE) {
                rA += isA; rB += isB; rC += isC; rD += nD;
                continue;
            }
            unsigned long long cx = (unsigned long long)isA | (unsigned long long)isB << 16 | (unsigned long long)isC << 32, ct;
            uint32_t dx = nD, dt;
            ScanC(s_c).ExclusiveSum(cx, cx, ct);
            ScanD(s_d).ExclusiveSum(dx, dx, dt);
            if (tid == 0) s_nbig = 0;
            __syncthreads();
            const uint32_t dest = pc_swz(d) * 4u;  // byte offset of the accumulator word
            auto idx = [&](uint32_t j) { return j < L ? (pe[i + j] & 0xFFFFu) * 4u : kPad; };
            auto wt = [&](uint32_t j) { return j < L ? (uint32_t)pw[i + j] : 0u; };
            if (isA) {
                const uint32_t j = rA + (uint32_t)(cx & 0xFFFFu);
                words[padA + j] = dest << 16 | idx(0);
                if (j == 0) for (uint32_t x = 0; x < padA; ++x) words[x] = dest << 16 | kPad;
                if (wq) {  // 32-bit: word j of a quad's first weight quad; the second is not read
                    uint32_t *ww = reinterpret_cast<uint32_t *>(wq);
                    auto at = [&](uint32_t x) { return w16 ? x : x / 4 * 8 + x % 4; };
                    ww[at(padA + j)] = wt(0);
                    if (j == 0) for (uint32_t x = 0; x < padA; ++x) ww[at(x)] = 0u;
                }
            } else if (isB) {
                const uint32_t j = rB + (uint32_t)(cx >> 16 & 0xFFFFu), h = padB + j;  // half quad of class B
                uint2 *halves = reinterpret_cast<uint2 *>(pe2 + q0 + qA);
                halves[h] = make_uint2(dest << 16 | idx(0), idx(2) << 16 | idx(1));
                if (j == 0 && padB) halves[0] = make_uint2(dest << 16 | kPad, kPad << 16 | kPad);
                if (wq) {
                    if (w16) {
                        uint2 *wh = reinterpret_cast<uint2 *>(wq + qA);
                        wh[h] = make_uint2(wt(0), wt(2) << 16 | wt(1));
                        if (j == 0 && padB) wh[0] = make_uint2(0u, 0u);
                    } else {
                        wq[2 * qA + h] = make_uint4(wt(0), wt(1), wt(2), 0u);
                        if (j == 0 && padB) wq[2 * qA] = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
            } else if (isC || (nD && nD <= kPieceSelf)) {
                for (uint32_t pc = 0; pc * kPcRunC < L; ++pc) {
                    const uint32_t o = pc * kPcRunC;  // x: the quad's place in the range
                    const uint32_t x = qA + qB + (isC ? rC + (uint32_t)(cx >> 32 & 0xFFFFu) : qC + piece_place(rD + dx + pc, qD));
                    pe2[q0 + x] = make_uint4(dest << 16 | idx(o), idx(o + 2) << 16 | idx(o + 1),
                                                        idx(o + 4) << 16 | idx(o + 3),
                                                        idx(o + 6) << 16 | idx(o + 5));
                    if (wq) {
                        if (w16) {
                            wq[x] = make_uint4(wt(o), wt(o + 2) << 16 | wt(o + 1), wt(o + 4) << 16 | wt(o + 3), wt(o + 6) << 16 | wt(o + 5));
                        } else {
                            wq[2 * x] = make_uint4(wt(o), wt(o + 1), wt(o + 2), wt(o + 3));
                            wq[2 * x + 1] = make_uint4(wt(o + 4), wt(o + 5), wt(o + 6), 0u);
                        }
                    }
                }
            } else if (nD) {
                const uint32_t k = atomicAdd(&s_nbig, 1u);
                s_bi[k] = i;
                s_bl[k] = L;
                s_bq[k] = rD + dx;
            }
            __syncthreads();
            for (uint32_t k = 0; k < s_nbig; ++k) {  // long runs: a piece per thread
                const uint32_t bi = s_bi[k], bl = s_bl[k], x0 = s_bq[k], bd = pc_swz(pe[bi] >> 16) * 4u;
                auto bidx = [&](uint32_t j) { return j < bl ? (pe[bi + j] & 0xFFFFu) * 4u : kPad; };
                auto bwt = [&](uint32_t j) { return j < bl ? (uint32_t)pw[bi + j] : 0u; };
                for (uint32_t pc = tid; pc * kPcRunC < bl; pc += kQuadThreads) {
                    const uint32_t o = pc * kPcRunC, x = qA + qB + qC + piece_place(x0 + pc, qD);
                    pe2[q0 + x] = make_uint4(bd << 16 | bidx(o), bidx(o + 2) << 16 | bidx(o + 1),
                                                        bidx(o + 4) << 16 | bidx(o + 3), bidx(o + 6) << 16 | bidx(o + 5));
                    if (wq) {
                        if (w16) {
                            wq[x] = make_uint4(bwt(o), bwt(o + 2) << 16 | bwt(o + 1), bwt(o + 4) << 16 | bwt(o + 3), bwt(o + 6) << 16 | bwt(o + 5));
                        } else {
                            wq[2 * x] = make_uint4(bwt(o), bwt(o + 1), bwt(o + 2), bwt(o + 3));
                            wq[2 * x + 1] = make_uint4(bwt(o + 4), bwt(o + 5), bwt(o + 6), 0u);
                        }
                    }
                }
            }
            rA += (uint32_t)(ct & 0xFFFFu); rB += (uint32_t)(ct >> 16 & 0xFFFFu); rC += (uint32_t)(ct >> 32 & 0xFFFFu);
            rD += dt;
            __syncthreads();  // the list and the scans' storage are used again
        }
        if (!WRITE) {
            __syncthreads();
            if (rA) atomicAdd(&s_cnt[0], rA);
            if (rB) atomicAdd(&s_cnt[1], rB);
            if (rC) atomicAdd(&s_cnt[2], rC);
            if (rD) atomicAdd(&s_cnt[3], rD);
            __syncthreads();
            if (tid == 0) {
                const uint4 c = make_uint4(s_cnt[0], s_cnt[1], s_cnt[2], s_cnt[3]);
                cls[r] = c;
                nquad[r] = (c.x + 3) / 4 + (c.y + 1) / 2 + c.z + c.w;
            }
            __syncthreads();
        }
    }
    if (WRITE && blockIdx.x == 0 && tid == 0) rng[nrange] = make_uint4(qoff[nrange], 0u, 0u, 0u);
}

// Small graphs: the edges' destinations as sort keys and their numbers as values
__global__ void k_small_keys(uint64_t E, const uint32_t *col, uint32_t *key, uint32_t *num) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        key[e] = col[e];
        num[e] = (uint32_t)e;
    }
}
// ... the first entry of every destination in that order (start[V] = E)
__global__ void k_small_starts(uint64_t E, uint32_t V, const uint32_t *key, uint32_t *start) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= E; i += stride) {
        const uint32_t hi = i < E ? key[i] : V, lo = i == 0 ? 0u : key[i - 1] + 1;
        for (uint32_t v = lo; v <= hi; ++v) start[v] = (uint32_t)i;
    }
}
// In-edges as (source, destination), and a span for every destination that shares cut, made at the first cut
__global__ void k_in_edges(uint64_t E, uint32_t share, const uint32_t *key, const uint32_t *src, const uint32_t *off,
                           uint2 *edge, uint4 *span, uint32_t *nspan) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < E; e += stride) {
        const uint32_t d = key[e];
        edge[e] = make_uint2(src[e], d);
        if (e % share == 0 && e > 0 && key[e - 1] == d && off[d] >= e - share)
            span[atomicAdd(nspan, 1u)] = make_uint4(d, (uint32_t)(e / share) - 1, (off[d + 1] - 1) / share - (uint32_t)(e / share) + 2, 0u);
    }
}
// ... the n + 1 cuts of the destinations into ranges of equal work, in-edges + vcost * vertices, and their first entries:
// cut j is the first destination with at least j / n of the work before it
__global__ void k_small_cuts(uint32_t n, uint32_t V, uint64_t E, uint64_t vcost, const uint32_t *start, uint2 *cut) {
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j <= n; j += gridDim.x * blockDim.x) {
        const uint64_t want = (E + vcost * V) * j / n;
        uint32_t lo = 0, hi = V;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) / 2;
            if (start[mid] + vcost * mid >= want) hi = mid; else lo = mid + 1;
        }
        cut[j] = make_uint2(j == n ? V : lo, j == n ? (uint32_t)E : start[lo]);
    }
}
// ... and every range's words and weights, one CTA per range: entry i of the range is edge num[first[r] + i] of the order
// by destination; the last quad is filled up with the padding's source
__global__ void k_small_words(uint32_t n, uint32_t V, const uint4 *range, const uint32_t *first, const uint32_t *num,
                              const uint32_t *src, const uint32_t *col, const int32_t *w, uint32_t *word, uint32_t *wword) {
    for (uint32_t r = blockIdx.x; r < n; r += gridDim.x) {
        const uint4 g = range[r];
        const uint32_t a = first[r], m = first[r + 1] - a;
        for (uint32_t i = threadIdx.x; i < g.w * 4; i += blockDim.x) {  // (no quads: no entries)
            const uint32_t e = num[a + min(i, m - 1)];
            word[(uint64_t)g.z * 4 + i] = (col[e] - g.x) << kSmallSrcBits | (i < m ? src[e] : V);
            if (wword) wword[(uint64_t)g.z * 4 + i] = i < m ? (uint32_t)w[e] : 0u;
        }
    }
}

__global__ void k_colbin_keys(uint64_t nb, uint32_t k, const uint32_t *bin_q, const uint32_t *row_bin,
                              uint64_t *key, uint32_t *val, uint32_t *bins_per_col) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b < nb; b += stride) {
        // row of bin b: largest p with row_bin[p] <= b
        uint32_t lo = 0, hi = k;
        while (hi - lo > 1) {
            uint32_t mid = lo + (hi - lo) / 2;
            if (row_bin[mid] <= (uint32_t)b) lo = mid; else hi = mid;
        }
        key[b] = (uint64_t)bin_q[b] * k + lo;
        val[b] = (uint32_t)b;
        atomicAdd(&bins_per_col[bin_q[b]], 1u);
    }
}

__global__ void k_part_edges(uint32_t k, uint32_t V, uint32_t shift, const uint32_t *rowptr, uint32_t *Ep) {
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < k; p += gridDim.x * blockDim.x) {
        uint64_t a = (uint64_t)p << shift, b = (uint64_t)(p + 1) << shift;
        if (b > V) b = V;
        Ep[p] = rowptr[b] - rowptr[a];
    }
}

template <typename F>
cudaError_t cub_run(Temps &t, F f) {
    size_t bytes = 0;
    cudaError_t e = f(nullptr, bytes);
    if (e != cudaSuccess) return e;
    void *tmp = nullptr;
    e = t.alloc((char **)&tmp, bytes);
    if (e != cudaSuccess) return e;
    e = f(tmp, bytes);
    t.release(tmp);
    return e;
}

int bits_for(uint64_t x) {  // number of bits to represent values < x
    int b = 0;
    while (b < 64 && (1ull << b) < x) ++b;
    return std::max(b, 1);
}

}  // namespace

static gpop_status build_impl(Graph *g, uint32_t V, uint64_t E, const uint64_t *row_ptr, const uint32_t *col,
                              const int32_t *weights, uint32_t P, int mem_is_device, cudaStream_t s) {
    GPOP_CUDA_TRY(cudaGetDevice(&g->device));
    GPOP_CUDA_TRY(cudaDeviceGetAttribute(&g->num_sms, cudaDevAttrMultiProcessorCount, g->device));
    g->V = V;
    g->E = E;
    g->P = P;
    g->shift = 0;
    while ((1u << g->shift) < P) ++g->shift;
    g->k = (uint32_t)(((uint64_t)V + P - 1) / P);
    g->weighted = weights != nullptr;
    const uint32_t k = g->k, shift = g->shift;
    Temps t(s);

    // 1. inputs on the device
    const uint64_t *d_rp = row_ptr;
    const uint32_t *d_col = col;
    const int32_t *d_w = weights;
    if (!mem_is_device) {
        uint64_t *a; uint32_t *b; int32_t *c = nullptr;
        GPOP_CUDA_TRY(t.alloc(&a, (uint64_t)V + 1));
        GPOP_CUDA_TRY(t.alloc(&b, E));
        GPOP_CUDA_TRY(cudaMemcpyAsync(a, row_ptr, sizeof(uint64_t) * (V + 1), cudaMemcpyHostToDevice, s));
        if (E) GPOP_CUDA_TRY(cudaMemcpyAsync(b, col, sizeof(uint32_t) * E, cudaMemcpyHostToDevice, s));
        if (weights) {
            GPOP_CUDA_TRY(t.alloc(&c, E));
            if (E) GPOP_CUDA_TRY(cudaMemcpyAsync(c, weights, sizeof(int32_t) * E, cudaMemcpyHostToDevice, s));
        }
        d_rp = a; d_col = b; d_w = c;
    }
    {
        uint32_t *d_err;
        GPOP_CUDA_TRY(t.alloc(&d_err, 2));
        GPOP_CUDA_TRY(cudaMemsetAsync(d_err, 0, 8, s));
        k_validate<<<blocks_for(std::max<uint64_t>(E, V + 1ull)), kThreads, 0, s>>>(V, E, d_rp, d_col, d_w, d_err);
        uint32_t hval[2] = {0, 0};
        GPOP_CUDA_TRY(cudaMemcpyAsync(hval, d_err, 8, cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
        const uint32_t herr = hval[0];
        g->w16 = g->weighted && hval[1] <= 0xFFFFu;
        if (herr) {
            char buf[200];
            snprintf(buf, sizeof buf, "malformed CSR (flags 0x%x: 1 row_ptr[0]!=0, 2 row_ptr[V]!=E, 4 decreasing "
                     "row_ptr, 8 col>=V, 16 negative weight)", herr);
            return fail(GPOP_ERR_INVALID_ARG, buf);
        }
    }

    // 2. CSR with destination-sorted rows (u32 offsets)
    GPOP_CUDA_TRY(t.keep(g, &g->rowptr, (uint64_t)V + 1));
    GPOP_CUDA_TRY(t.keep(g, &g->col, E));
    if (g->weighted) GPOP_CUDA_TRY(t.keep(g, &g->w, E));
    k_rowptr32<<<blocks_for(V + 1ull), kThreads, 0, s>>>(V, d_rp, g->rowptr);
    uint32_t *src, *d_unsorted, unsorted = 0;
    GPOP_CUDA_TRY(t.alloc(&src, E));
    GPOP_CUDA_TRY(t.alloc(&d_unsorted, 1));
    GPOP_CUDA_TRY(cudaMemsetAsync(d_unsorted, 0, 4, s));
    if (E) {
        k_edge_src<<<blocks_for(E, (int)kSrcTile), kThreads, 0, s>>>(V, E, g->rowptr, d_col, src, d_unsorted);
        GPOP_CUDA_TRY(cudaMemcpyAsync(&unsorted, d_unsorted, 4, cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
        if (unsorted) {
            uint64_t *k0, *k1;
            GPOP_CUDA_TRY(t.alloc(&k0, E));
            GPOP_CUDA_TRY(t.alloc(&k1, E));
            k_pack_src_dst<<<blocks_for(E), kThreads, 0, s>>>(E, src, d_col, k0);
            int end_bit = 32 + bits_for(V);
            if (g->weighted) {
                GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                    return cub::DeviceRadixSort::SortPairs(tmp, bytes, k0, k1, d_w, g->w, E, 0, end_bit, s);
                }));
            } else {
                GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                    return cub::DeviceRadixSort::SortKeys(tmp, bytes, k0, k1, E, 0, end_bit, s);
                }));
            }
            k_unpack_dst<<<blocks_for(E), kThreads, 0, s>>>(E, k1, g->col);
            t.release(k0);
            t.release(k1);
        } else {  // every row is in order, as CSR usually comes: what the (stable) sort would leave
            GPOP_CUDA_TRY(cudaMemcpyAsync(g->col, d_col, 4ull * E, cudaMemcpyDeviceToDevice, s));
            if (g->weighted) GPOP_CUDA_TRY(cudaMemcpyAsync(g->w, d_w, 4ull * E, cudaMemcpyDeviceToDevice, s));
        }
    }
    {  // the graph's fingerprint (checkpoints of another graph are refused)
        unsigned long long *d_fp, h_fp = 0;
        GPOP_CUDA_TRY(t.alloc(&d_fp, 1));
        GPOP_CUDA_TRY(cudaMemsetAsync(d_fp, 0, 8, s));
        if (E) k_fingerprint<<<std::min<uint64_t>(blocks_for(E), 8ull * g->num_sms), kThreads, 0, s>>>(E, src, g->col, g->w, d_fp);
        GPOP_CUDA_TRY(cudaMemcpyAsync(&h_fp, d_fp, 8, cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
        g->fingerprint = h_fp ^ ((uint64_t)V << 32) ^ (E * 0x9E3779B97F4A7C15ull) ^ (uint64_t)g->weighted;
    }

    // 3. messages: one per (source, destination partition), sorted by (p, q, source)
    uint8_t *head;
    uint64_t *mkey, *skey = nullptr;
    uint32_t *head_idx, *shead = nullptr, *d_nmsg;
    GPOP_CUDA_TRY(t.alloc(&head, E));
    GPOP_CUDA_TRY(t.alloc(&mkey, E));
    GPOP_CUDA_TRY(t.alloc(&head_idx, E));
    GPOP_CUDA_TRY(t.alloc(&d_nmsg, 1));
    GPOP_CUDA_TRY(cudaMemsetAsync(d_nmsg, 0, 4, s));
    uint64_t nmsg = 0;
    if (E) {
        k_heads<<<blocks_for(E), kThreads, 0, s>>>(E, shift, k, g->rowptr, src, g->col, head, mkey, head_idx);
        uint64_t *hkey;
        uint32_t *hidx;
        GPOP_CUDA_TRY(t.alloc(&hkey, E));
        GPOP_CUDA_TRY(t.alloc(&hidx, E));
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceSelect::Flagged(tmp, bytes, mkey, head, hkey, d_nmsg, (int64_t)E, s);
        }));
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceSelect::Flagged(tmp, bytes, head_idx, head, hidx, d_nmsg, (int64_t)E, s);
        }));
        t.release(mkey);
        uint32_t h_nmsg = 0;
        GPOP_CUDA_TRY(cudaMemcpyAsync(&h_nmsg, d_nmsg, 4, cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
        nmsg = h_nmsg;
        GPOP_CUDA_TRY(t.alloc(&skey, nmsg));
        GPOP_CUDA_TRY(t.alloc(&shead, nmsg));
        int end_bit = bits_for((uint64_t)k * k) + (int)shift;
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceRadixSort::SortPairs(tmp, bytes, hkey, skey, hidx, shead, nmsg, 0, end_bit, s);
        }));
        t.release(hkey);
        t.release(hidx);
    }
    t.release(head);
    g->npng = nmsg;

    // 4. bins, rows, padded PNG slots
    uint32_t *newbin, *binscan, *msgs_row, *msgs_row_pad, *row_start;
    GPOP_CUDA_TRY(t.alloc(&row_start, (uint64_t)k + 1));
    GPOP_CUDA_TRY(t.alloc(&newbin, nmsg));
    GPOP_CUDA_TRY(t.alloc(&binscan, nmsg));
    GPOP_CUDA_TRY(t.alloc(&msgs_row, (uint64_t)k + 1));
    GPOP_CUDA_TRY(t.alloc(&msgs_row_pad, (uint64_t)k + 1));
    uint32_t *nbins_p;
    GPOP_CUDA_TRY(t.alloc(&nbins_p, (uint64_t)k + 1));
    GPOP_CUDA_TRY(t.keep(g, &g->npng_p, (uint64_t)k + 1));
    GPOP_CUDA_TRY(t.keep(g, &g->row_bin, (uint64_t)k + 1));
    uint32_t *row_png;
    GPOP_CUDA_TRY(t.alloc(&row_png, (uint64_t)k + 1));
    GPOP_CUDA_TRY(cudaMemsetAsync(msgs_row, 0, 4ull * (k + 1), s));
    GPOP_CUDA_TRY(cudaMemsetAsync(nbins_p, 0, 4ull * (k + 1), s));
    if (nmsg) {
        k_msg_bins<<<blocks_for(nmsg), kThreads, 0, s>>>(nmsg, shift, skey, newbin);
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceScan::InclusiveSum(tmp, bytes, newbin, binscan, nmsg, s);
        }));
    }
    t.release(newbin);
    // messages are sorted by (row p, column q, source): row p = (key >> shift) / k
    k_seg_starts<<<blocks_for(nmsg + 1), kThreads, 0, s>>>(nmsg, skey, shift, k, k, row_start);
    k_row_counts<<<blocks_for(k), kThreads, 0, s>>>(k, row_start, binscan, msgs_row, nbins_p);
    GPOP_CUDA_TRY(cudaMemsetAsync(msgs_row + k, 0, 4, s));
    GPOP_CUDA_TRY(cudaMemcpyAsync(g->npng_p, msgs_row, 4ull * (k + 1), cudaMemcpyDeviceToDevice, s));
    GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
        return cub::DeviceScan::ExclusiveSum(tmp, bytes, nbins_p, g->row_bin, (uint64_t)k + 1, s);
    }));
    uint32_t h_nb = 0;
    GPOP_CUDA_TRY(cudaMemcpyAsync(&h_nb, g->row_bin + k, 4, cudaMemcpyDeviceToHost, s));
    GPOP_CUDA_TRY(cudaStreamSynchronize(s));
    g->nb = h_nb;
    // bins padded to kBinAlign slots, rows to kPngAlign
    uint32_t *bin_j0, *bin_p, *cnt4, *binoff, *row_len4;
    GPOP_CUDA_TRY(t.alloc(&bin_j0, g->nb + 1));
    GPOP_CUDA_TRY(t.alloc(&bin_p, g->nb + 1));
    GPOP_CUDA_TRY(t.alloc(&cnt4, g->nb + 1));
    GPOP_CUDA_TRY(t.alloc(&binoff, g->nb + 1));
    GPOP_CUDA_TRY(t.alloc(&row_len4, (uint64_t)k + 1));
    GPOP_CUDA_TRY(t.keep(g, &g->bin_q, g->nb));
    GPOP_CUDA_TRY(cudaMemsetAsync(row_len4, 0, 4ull * (k + 1), s));
    const uint32_t nmsg32 = (uint32_t)nmsg;  // messages <= edges < 2^32
    GPOP_CUDA_TRY(cudaMemcpyAsync(bin_j0 + g->nb, &nmsg32, 4, cudaMemcpyHostToDevice, s));
    GPOP_CUDA_TRY(cudaMemsetAsync(cnt4 + g->nb, 0, 4, s));
    if (nmsg) {
        k_bin_starts<<<blocks_for(nmsg), kThreads, 0, s>>>(nmsg, shift, k, skey, binscan, bin_j0, g->bin_q, bin_p);
        k_bin_pad<<<blocks_for(g->nb), kThreads, 0, s>>>((uint32_t)g->nb, bin_j0, bin_p, cnt4, row_len4);
    }
    GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
        return cub::DeviceScan::ExclusiveSum(tmp, bytes, cnt4, binoff, g->nb + 1, s);
    }));
    k_pad8<<<blocks_for(k), kThreads, 0, s>>>(k, row_len4, msgs_row_pad);
    GPOP_CUDA_TRY(cudaMemsetAsync(msgs_row_pad + k, 0, 4, s));
    GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
        return cub::DeviceScan::ExclusiveSum(tmp, bytes, msgs_row_pad, row_png, (uint64_t)k + 1, s);
    }));
    uint32_t h_npad = 0;
    GPOP_CUDA_TRY(cudaMemcpyAsync(&h_npad, row_png + k, 4, cudaMemcpyDeviceToHost, s));
    GPOP_CUDA_TRY(cudaStreamSynchronize(s));
    g->npng_pad = h_npad;

    // 5. bins per column in ascending source partition, and the column-major slots of the message values: column by
    //    column, each bin padded as in its row
    uint32_t *bin_cslot0, *d_col_off;
    GPOP_CUDA_TRY(t.alloc(&bin_cslot0, g->nb + 1));
    GPOP_CUDA_TRY(t.alloc(&d_col_off, (uint64_t)k + 1));
    uint32_t *col_bins;
    GPOP_CUDA_TRY(t.alloc(&col_bins, g->nb));
    uint32_t *col_bin;
    GPOP_CUDA_TRY(t.alloc(&col_bin, (uint64_t)k + 1));
    {
        uint64_t *bk, *bk2;
        uint32_t *bv, *bpc;
        GPOP_CUDA_TRY(t.alloc(&bk, g->nb));
        GPOP_CUDA_TRY(t.alloc(&bk2, g->nb));
        GPOP_CUDA_TRY(t.alloc(&bv, g->nb));
        GPOP_CUDA_TRY(t.alloc(&bpc, (uint64_t)k + 1));
        GPOP_CUDA_TRY(cudaMemsetAsync(bpc, 0, 4ull * (k + 1), s));
        if (g->nb) {
            k_colbin_keys<<<blocks_for(g->nb), kThreads, 0, s>>>(g->nb, k, g->bin_q, g->row_bin, bk, bv, bpc);
            GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                return cub::DeviceRadixSort::SortPairs(tmp, bytes, bk, bk2, bv, col_bins, g->nb, 0,
                                                       bits_for((uint64_t)k * k), s);
            }));
        }
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceScan::ExclusiveSum(tmp, bytes, bpc, col_bin, (uint64_t)k + 1, s);
        }));
        uint32_t *len, *coff;
        GPOP_CUDA_TRY(t.alloc(&len, g->nb + 1));
        GPOP_CUDA_TRY(t.alloc(&coff, g->nb + 1));
        GPOP_CUDA_TRY(cudaMemsetAsync(len + g->nb, 0, 4, s));
        if (g->nb) k_col_lengths<<<blocks_for(g->nb), kThreads, 0, s>>>(g->nb, col_bins, cnt4, len);
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceScan::ExclusiveSum(tmp, bytes, len, coff, g->nb + 1, s);
        }));
        k_col_slots<<<blocks_for(std::max<uint64_t>(g->nb, k + 1ull)), kThreads, 0, s>>>(g->nb, k, col_bins, col_bin, coff,
                                                                                         bin_cslot0, d_col_off);
    }

    GPOP_CUDA_TRY(t.keep(g, &g->png, g->npng_pad));
    GPOP_CUDA_TRY(t.keep(g, &g->pdata, g->npng_pad));
    // padding slots keep local source 0: their values are staged but no entry refers to them
    GPOP_CUDA_TRY(cudaMemsetAsync(g->png, 0, 2ull * std::max<uint64_t>(g->npng_pad, 1), s));
    GPOP_CUDA_TRY(cudaMemsetAsync(g->pdata, 0xFF, 4ull * std::max<uint64_t>(g->npng_pad, 1), s));
    GPOP_CUDA_TRY(t.keep(g, &g->png_dst, g->npng_pad / kBinAlign));
    uint32_t *cslot_of_head;
    GPOP_CUDA_TRY(t.alloc(&cslot_of_head, E));
    if (nmsg)
        k_place_msgs<<<blocks_for(nmsg), kThreads, 0, s>>>(nmsg, shift, skey, shead, binscan, bin_j0, bin_p, binoff,
                                                           g->row_bin, row_png, bin_cslot0, g->png, g->png_dst,
                                                           cslot_of_head);
    t.release(skey);
    t.release(shead);
    t.release(binscan);

    // 6. message head of every edge (its first edge to the same destination partition)
    uint32_t *head_of;
    GPOP_CUDA_TRY(t.alloc(&head_of, E));
    if (E) {
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceScan::InclusiveScan(tmp, bytes, head_idx, head_of, MaxOp(), E, s);
        }));
    }
    t.release(head_idx);

    const uint32_t nblk = (V + 31) / 32;
    uint32_t *d_in;  // in-edges of every 32 destinations
    GPOP_CUDA_TRY(t.alloc(&d_in, nblk));
    GPOP_CUDA_TRY(cudaMemsetAsync(d_in, 0, 4ull * nblk, s));

    // 7. PC gather blocks.  The messages of column q (its bins (p, q), p ascending, each bin's
    //    messages in source order) form the column sequence; it is cut into blocks of kPcBlock messages
    //    that the gather stages in shared memory by one copy each (the values are stored in column order).
    //    Every PC in-entry is a word (local destination << 16 | index in its block), sorted by (block,
    //    destination, index), before it becomes part of a quad.
    //    Gather tasks cover consecutive entries of one column: at most the entries chosen below and at most
    //    kPcTaskBlocks blocks each, a block's entries split over several
    //    tasks when it is larger; a column with several tasks leaves one partial vector per task,
    //    merged in column order by the filter.  Tasks are listed largest first.
    {
        std::vector<uint32_t> hcol_off(k + 1), col_blk0(k + 1), blk_src, blk_nval, blk_col;
        GPOP_CUDA_TRY(cudaMemcpyAsync(hcol_off.data(), d_col_off, 4ull * (k + 1), cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
        for (uint32_t q = 0; q < k; ++q) {
            col_blk0[q] = (uint32_t)blk_src.size();
            for (uint32_t x = hcol_off[q]; x < hcol_off[q + 1]; x += std::min(kPcBlock, hcol_off[q + 1] - x)) {
                blk_src.push_back(x);
                blk_col.push_back(q);
                blk_nval.push_back(std::min(kPcBlock, hcol_off[q + 1] - x));
            }
        }
        const uint32_t nblocks = (uint32_t)blk_src.size();
        col_blk0[k] = nblocks;
        g->npcb = nblocks;
        uint32_t *pc_blk_ent;
        GPOP_CUDA_TRY(t.alloc(&pc_blk_ent, (uint64_t)nblocks + 1));
        GPOP_CUDA_TRY(t.keep(g, &g->col_ntask, k));
        GPOP_CUDA_TRY(t.keep(g, &g->col_part0, k));
        uint32_t *spe;            // entries (destination << 16 | index), sorted by block, destination, index
        int32_t *spw = nullptr;   // their weights
        GPOP_CUDA_TRY(t.alloc(&spe, E));
        if (g->weighted) GPOP_CUDA_TRY(t.alloc(&spw, E));
        GPOP_CUDA_TRY(t.keep(g, &g->pc_blk_src, (uint64_t)nblocks + 1));
        GPOP_CUDA_TRY(t.keep(g, &g->pc_blk_nval, (uint64_t)nblocks + 1));
        GPOP_CUDA_TRY(t.keep(g, &g->pc_blk_prange, (uint64_t)nblocks + 1));
        uint32_t *d_colblk0;
        GPOP_CUDA_TRY(t.alloc(&d_colblk0, (uint64_t)k + 1));
        GPOP_CUDA_TRY(cudaMemcpyAsync(d_colblk0, col_blk0.data(), 4ull * (k + 1), cudaMemcpyHostToDevice, s));
        const std::vector<uint2> prange0(nblocks, make_uint2(0xFFFFFFFFu, 0u));
        if (nblocks) {
            GPOP_CUDA_TRY(cudaMemcpyAsync(g->pc_blk_src, blk_src.data(), 4ull * nblocks, cudaMemcpyHostToDevice, s));
            GPOP_CUDA_TRY(cudaMemcpyAsync(g->pc_blk_nval, blk_nval.data(), 4ull * nblocks, cudaMemcpyHostToDevice, s));
            GPOP_CUDA_TRY(cudaMemcpyAsync(g->pc_blk_prange, prange0.data(), sizeof(uint2) * nblocks, cudaMemcpyHostToDevice, s));
            k_blk_prange<<<blocks_for(g->nb), kThreads, 0, s>>>(g->nb, g->bin_q, bin_p, cnt4, bin_cslot0, d_col_off, d_colblk0,
                                                                g->pc_blk_prange);
        }
        // entries: sort keys (block, local destination, index in block)
        if (E) {
            uint64_t *pk, *pk2;
            GPOP_CUDA_TRY(t.alloc(&pk, E));
            GPOP_CUDA_TRY(t.alloc(&pk2, E));
            k_pc_keys<<<blocks_for(E), kThreads, 0, s>>>(E, shift, P, head_of, cslot_of_head, g->col, d_col_off, d_colblk0, pk);
            t.release(head_of);
            t.release(cslot_of_head);
            // from the destination up: edges come by ascending source, which is the order of the messages of a block, so
            // the stable sort leaves equal destinations by index
            const int first_bit = 16, end_bit = 32 + bits_for((uint64_t)nblocks + 1);
            if (g->weighted) {
                GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                    return cub::DeviceRadixSort::SortPairs(tmp, bytes, pk, pk2, g->w, spw, E, first_bit, end_bit, s);
                }));
            } else {
                GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                    return cub::DeviceRadixSort::SortKeys(tmp, bytes, pk, pk2, E, first_bit, end_bit, s);
                }));
            }
            k_pc_unpack<<<blocks_for(E), kThreads, 0, s>>>(E, pk2, spe);
            k_seg_starts<<<blocks_for(E + 1), kThreads, 0, s>>>(E, pk2, 32, 1, nblocks, pc_blk_ent);
            t.release(pk);
            t.release(pk2);
            uint32_t *d_blkcol;
            GPOP_CUDA_TRY(t.alloc(&d_blkcol, nblocks));
            GPOP_CUDA_TRY(cudaMemcpyAsync(d_blkcol, blk_col.data(), 4ull * nblocks, cudaMemcpyHostToDevice, s));
            k_block_indeg<<<blocks_for((uint64_t)nblocks * (P / 32)), kThreads, 0, s>>>(nblocks, P, d_blkcol, pc_blk_ent, spe,
                                                                                       d_in);
        } else {
            GPOP_CUDA_TRY(cudaMemsetAsync(pc_blk_ent, 0, 4ull * (nblocks + 1), s));
        }
        std::vector<uint32_t> hbe(nblocks + 1);
        GPOP_CUDA_TRY(cudaMemcpyAsync(hbe.data(), pc_blk_ent, 4ull * (nblocks + 1), cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));

        // gather tasks over each column's entries, a column's tasks sharing its entries evenly: at most `target`
        // entries each, or `fine` in the smallest columns, those after the first `tail` entries of the columns in
        // falling order of size; prng: each task's entries
        std::vector<uint32_t> by_col(k);  // columns in falling order of size
        std::vector<uint64_t> before(k);  // entries of the columns before each in that order
        for (uint32_t q = 0; q < k; ++q) by_col[q] = q;
        auto col_ents = [&](uint32_t q) { return (uint64_t)hbe[col_blk0[q + 1]] - hbe[col_blk0[q]]; };
        std::stable_sort(by_col.begin(), by_col.end(), [&](uint32_t x, uint32_t y) { return col_ents(x) > col_ents(y); });
        uint64_t ents = 0;
        for (uint32_t q : by_col) {
            before[q] = ents;
            ents += col_ents(q);
        }
        auto cut_tasks = [&](uint64_t target, uint64_t fine, uint64_t tail, std::vector<uint4> &ptasks, std::vector<uint2> &prng,
                             std::vector<uint32_t> &col_ntask, std::vector<uint32_t> &col_part0) -> uint32_t {
            ptasks.clear();
            prng.clear();
            uint32_t nparts = 0;
            for (uint32_t q = 0; q < k; ++q) {
                const uint32_t b_end = col_blk0[q + 1];
                uint32_t b = col_blk0[q];
                uint64_t pos = hbe[b];
                const uint64_t most = before[q] >= tail ? fine : target;
                const uint64_t end = hbe[b_end], pieces = (end - pos + most - 1) / most;
                const uint64_t share = pieces ? (end - pos + pieces - 1) / pieces : 0;
                const size_t first_task = ptasks.size();
                for (;;) {
                    while (b < b_end && pos >= hbe[b + 1]) ++b;  // skip exhausted blocks
                    if (b == b_end || pos >= end) break;
                    const uint32_t tb = b;
                    const uint64_t ea = pos;
                    uint64_t cnt = 0;
                    uint32_t tb_end;
                    for (;;) {
                        const uint64_t avail = hbe[b + 1] - pos, room = share - cnt;
                        if (avail >= room) {  // task full; the block may continue in the next task
                            pos += room;
                            tb_end = b + 1;
                            break;
                        }
                        cnt += avail;
                        pos = hbe[b + 1];
                        ++b;
                        if (b - tb == kPcTaskBlocks || b == b_end) {
                            tb_end = b;
                            break;
                        }
                    }
                    ptasks.push_back(make_uint4(q, tb, tb_end, kNull));
                    prng.push_back(make_uint2((uint32_t)ea, (uint32_t)pos));
                    b = tb_end - 1;
                }
                const uint32_t ntq = (uint32_t)(ptasks.size() - first_task);
                col_ntask[q] = ntq;
                col_part0[q] = nparts;
                if (ntq > 1) {
                    for (uint32_t j = 0; j < ntq; ++j) ptasks[first_task + j].w = nparts + j;
                    nparts += ntq;
                }
            }
            return nparts;
        };
        // largest tasks first, so that the persistent CTAs finish together
        auto by_size = [](const std::vector<uint2> &prng) {
            std::vector<uint32_t> order(prng.size());
            for (uint32_t i = 0; i < order.size(); ++i) order[i] = i;
            std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) {
                return prng[x].y - prng[x].x > prng[y].y - prng[y].x;
            });
            return order;
        };
        // Task sizes: at most E / (d SMs) entries, d = 2 .. 32, and a quarter of that in the smallest columns, which hold
        // 0, 1/8, 1/4 or 1/2 of the entries: the choice for which an all-active gather should take the least time.
        // The tasks go to the CTAs largest first; a CTA's time is modelled as kTaskNs a task (slot, result vector),
        // kBlockNs a staged block and kEntryNs an entry, and every partial vector of a split column costs its trip
        // through memory in the merge, whose launch costs kMergeNs.  A few large columns otherwise leave the last wave
        // nearly empty: 367 equal columns on 152 CTAs (a uniform graph of 6 M vertices) ran 3 rounds for 2.4 rounds' work.
        constexpr double kTaskNs = 2000, kBlockNs = 400, kEntryNs = 0.2, kMergeNs = 4000, kPartNsPerWord = 0.002;
        const uint64_t sms = (uint64_t)std::max(1, g->num_sms);
        std::vector<uint4> ptasks;
        std::vector<uint2> prng;
        std::vector<uint32_t> col_ntask(k, 0), col_part0(k, 0);
        uint64_t best[3] = {0, 0, 0};
        double best_ns = 0, ideal_ns = 0;  // ideal: the tasks' time spread evenly
        for (uint64_t d : {2, 3, 4, 6, 8, 12, 16, 24, 32}) {
            const uint64_t target = std::max<uint64_t>(kPcTaskMinEntries, E / (d * sms));
            const uint64_t fine = std::max<uint64_t>(kPcTaskMinEntries, target / 4);
            for (uint64_t eighths : {0, 1, 2, 4}) {
                const uint64_t tail = E - E / 8 * eighths;
                if (eighths && fine == target) break;
                const uint32_t parts = cut_tasks(target, fine, tail, ptasks, prng, col_ntask, col_part0);
                std::vector<double> busy(sms, 0.0);  // a heap: the CTA that is free first takes the next task
                double sum = 0;
                for (uint32_t i : by_size(prng)) {
                    const double ns = kTaskNs + kBlockNs * (ptasks[i].z - ptasks[i].y) + kEntryNs * (prng[i].y - prng[i].x);
                    std::pop_heap(busy.begin(), busy.end(), std::greater<double>());
                    busy.back() += ns;
                    std::push_heap(busy.begin(), busy.end(), std::greater<double>());
                    sum += ns;
                }
                if (ideal_ns == 0) ideal_ns = sum / (double)sms;
                const double ns = *std::max_element(busy.begin(), busy.end()) +
                                  (parts ? kMergeNs + kPartNsPerWord * (double)parts * P : 0.0);
                if (best[0] == 0 || ns < best_ns) {
                    best[0] = target; best[1] = fine; best[2] = tail;
                    best_ns = ns;
                }
            }
            // little left to gain, more tasks than the CTAs' imbalance could gain from, or none smaller to be had
            if (best_ns < 1.04 * ideal_ns || target == kPcTaskMinEntries || ptasks.size() > 8 * sms) break;
        }
        const uint32_t nparts = cut_tasks(best[0], best[1], best[2], ptasks, prng, col_ntask, col_part0);
        const std::vector<uint32_t> order = by_size(prng);
        std::vector<uint4> stasks(ptasks.size());
        std::vector<uint2> srng(ptasks.size());
        for (size_t i = 0; i < order.size(); ++i) {
            stasks[i] = ptasks[order[i]];
            srng[i] = prng[order[i]];
        }
        // warp splits: per task block, kPcGatherWarps entry ranges of about equal size cut at
        // destination boundaries
        constexpr uint32_t kSp = kPcGatherWarps + 1;
        {
            std::vector<uint32_t> tsp(stasks.size() + 1), rlo, rhi, rtask;
            for (size_t ti = 0; ti < stasks.size(); ++ti) {
                tsp[ti] = (uint32_t)rlo.size();
                const uint4 tk = stasks[ti];
                for (uint32_t b = tk.y; b < tk.z; ++b) {
                    rlo.push_back(b == tk.y ? srng[ti].x : hbe[b]);
                    rhi.push_back(b + 1 == tk.z ? srng[ti].y : hbe[b + 1]);
                    rtask.push_back((uint32_t)ti);
                }
            }
            tsp[stasks.size()] = (uint32_t)rlo.size();
            const uint32_t nrow = (uint32_t)rlo.size(), ntask = (uint32_t)stasks.size();
            uint32_t *d_lo, *d_hi, *d_rtask, *d_row0, *d_cut;
            GPOP_CUDA_TRY(t.alloc(&d_lo, (uint64_t)nrow + 1));
            GPOP_CUDA_TRY(t.alloc(&d_hi, (uint64_t)nrow + 1));
            GPOP_CUDA_TRY(t.alloc(&d_rtask, (uint64_t)nrow + 1));
            GPOP_CUDA_TRY(t.alloc(&d_row0, (uint64_t)ntask + 1));
            GPOP_CUDA_TRY(t.alloc(&d_cut, (uint64_t)ntask * (kPcGatherWarps - 1) + 1));
            uint32_t *d_sp;
            GPOP_CUDA_TRY(t.alloc(&d_sp, (uint64_t)nrow * kSp + 1));
            GPOP_CUDA_TRY(t.keep(g, &g->pc_tsp, (uint64_t)ntask + 1));
            if (nrow) {
                GPOP_CUDA_TRY(cudaMemcpyAsync(d_lo, rlo.data(), 4ull * nrow, cudaMemcpyHostToDevice, s));
                GPOP_CUDA_TRY(cudaMemcpyAsync(d_hi, rhi.data(), 4ull * nrow, cudaMemcpyHostToDevice, s));
                GPOP_CUDA_TRY(cudaMemcpyAsync(d_rtask, rtask.data(), 4ull * nrow, cudaMemcpyHostToDevice, s));
                GPOP_CUDA_TRY(cudaMemcpyAsync(d_row0, tsp.data(), 4ull * (ntask + 1), cudaMemcpyHostToDevice, s));
                GPOP_CUDA_TRY(cudaMemcpyAsync(g->pc_tsp, tsp.data(), 4ull * ntask, cudaMemcpyHostToDevice, s));
                k_task_cuts<<<blocks_for((uint64_t)ntask * (kPcGatherWarps - 1)), kThreads, 0, s>>>(
                    ntask, g->P, d_row0, d_lo, d_hi, spe, d_cut);
                k_warp_splits<<<blocks_for((uint64_t)nrow * kSp), kThreads, 0, s>>>(nrow, d_lo, d_hi, d_rtask, d_cut,
                                                                                    spe, d_sp);
            }
            // the entries of every range as quads: counted, placed by a scan over the ranges, written
            const uint32_t nrange = nrow * kPcGatherWarps;
            uint4 *d_cls;
            uint32_t *d_nq, *d_qoff, nquads = 0;
            GPOP_CUDA_TRY(t.alloc(&d_cls, (uint64_t)nrange + 1));
            GPOP_CUDA_TRY(t.alloc(&d_nq, (uint64_t)nrange + 1));
            GPOP_CUDA_TRY(t.alloc(&d_qoff, (uint64_t)nrange + 1));
            GPOP_CUDA_TRY(t.keep(g, &g->pc_rng, (uint64_t)nrange + 1));
            GPOP_CUDA_TRY(cudaMemsetAsync(d_nq + nrange, 0, 4, s));
            if (nrange)
                k_range_quads<false><<<nrange, kQuadThreads, 0, s>>>(nrange, d_sp, spe, spw, d_cls, d_nq, nullptr, nullptr,
                                                                     nullptr, nullptr, false);
            GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                return cub::DeviceScan::ExclusiveSum(tmp, bytes, d_nq, d_qoff, (uint64_t)nrange + 1, s);
            }));
            GPOP_CUDA_TRY(cudaMemcpyAsync(&nquads, d_qoff + nrange, 4, cudaMemcpyDeviceToHost, s));
            GPOP_CUDA_TRY(cudaStreamSynchronize(s));
            // + 64: the gather reads whole rows
            GPOP_CUDA_TRY(t.keep(g, &g->pe, (uint64_t)nquads + 64));
            GPOP_CUDA_TRY(cudaMemsetAsync(g->pe + nquads, 0, 64 * sizeof(uint4), s));
            if (g->weighted) {
                const uint64_t per = g->w16 ? 1 : 2;
                GPOP_CUDA_TRY(t.keep(g, &g->pw, per * ((uint64_t)nquads + 64)));
                GPOP_CUDA_TRY(cudaMemsetAsync(g->pw + per * nquads, 0, per * 64 * sizeof(uint4), s));
            }
            k_range_quads<true><<<std::max(1u, nrange), kQuadThreads, 0, s>>>(nrange, d_sp, spe, spw, d_cls, nullptr,
                                                                               d_qoff, g->pc_rng, g->pe, g->pw, g->w16 != 0);
            GPOP_CUDA_TRY(cudaStreamSynchronize(s));
            t.release(spe);
            if (spw) t.release(spw);
        }
        // merge items: 1024-destination chunks of every column split over several tasks
        {
            std::vector<uint2> items;
            for (uint32_t q = 0; q < k; ++q)
                if (col_ntask[q] > 1) {
                    const uint32_t wq = (uint32_t)std::min<uint64_t>(P, V - ((uint64_t)q << shift));
                    for (uint32_t d0 = 0; d0 < wq; d0 += 1024) items.push_back(make_uint2(q, d0));
                }
            g->nmerge = (uint32_t)items.size();
            GPOP_CUDA_TRY(t.keep(g, &g->pc_merge, items.size()));
            if (!items.empty())
                GPOP_CUDA_TRY(cudaMemcpyAsync(g->pc_merge, items.data(), sizeof(uint2) * items.size(), cudaMemcpyHostToDevice, s));
        }
        g->npct = (uint32_t)stasks.size();
        g->npart = nparts;
        GPOP_CUDA_TRY(t.keep(g, &g->pc_task, stasks.size()));
        GPOP_CUDA_TRY(t.keep(g, &g->pc_part, (uint64_t)nparts * P));
        if (!stasks.empty()) {
            GPOP_CUDA_TRY(cudaMemcpyAsync(g->pc_task, stasks.data(), sizeof(uint4) * stasks.size(), cudaMemcpyHostToDevice, s));
        }
        GPOP_CUDA_TRY(cudaMemcpyAsync(g->col_ntask, col_ntask.data(), 4ull * k, cudaMemcpyHostToDevice, s));
        GPOP_CUDA_TRY(cudaMemcpyAsync(g->col_part0, col_part0.data(), 4ull * k, cudaMemcpyHostToDevice, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
    }

    // 8. per-partition statics
    GPOP_CUDA_TRY(t.keep(g, &g->Ep, (uint64_t)k + 1));
    k_part_edges<<<blocks_for(k), kThreads, 0, s>>>(k, V, shift, g->rowptr, g->Ep);
    std::vector<uint32_t> hEp(k), hnp(k), hnb(k), hrow_png(k + 1);
    GPOP_CUDA_TRY(cudaMemcpyAsync(hEp.data(), g->Ep, 4ull * k, cudaMemcpyDeviceToHost, s));
    GPOP_CUDA_TRY(cudaMemcpyAsync(hnp.data(), g->npng_p, 4ull * k, cudaMemcpyDeviceToHost, s));
    GPOP_CUDA_TRY(cudaMemcpyAsync(hnb.data(), nbins_p, 4ull * k, cudaMemcpyDeviceToHost, s));
    GPOP_CUDA_TRY(cudaMemcpyAsync(hrow_png.data(), row_png, 4ull * (k + 1), cudaMemcpyDeviceToHost, s));

    // 9. static gather tasks: ranges of whole 32-vertex blocks of one column, at most kGatherWidth
    //    destinations and (unless one block alone has more) at most `tgt` in-edges, so that the SC pairs
    //    of a hub column, which one task folds alone, are spread over several
    std::vector<uint32_t> hin(nblk);
    GPOP_CUDA_TRY(cudaMemcpyAsync(hin.data(), d_in, 4ull * nblk, cudaMemcpyDeviceToHost, s));
    GPOP_CUDA_TRY(cudaStreamSynchronize(s));
    g->h_Ep = new uint64_t[k];
    g->h_npng = new uint64_t[k];
    g->max_row_bins = 0;
    for (uint32_t p = 0; p < k; ++p) {
        g->h_Ep[p] = hEp[p];
        g->h_npng[p] = hnp[p];
        g->max_row_bins = std::max(g->max_row_bins, hnb[p]);
    }
    if (g->max_row_bins > kMaxRowBins)
        return fail(GPOP_ERR_INVALID_ARG, "a bin row has more non-empty bins than the SC scatter supports; "
                                          "use a larger partition size");
    std::vector<GatherTask> gt;
    std::vector<uint32_t> col_task(k + 1);
    const uint32_t width_blocks = std::min(P, kGatherWidth) / 32;
    const uint64_t tgt = std::max<uint64_t>(kGatherTaskMinEdges, E / (4ull * (uint64_t)std::max(1, g->num_sms)));
    for (uint32_t q = 0; q < k; ++q) {
        col_task[q] = (uint32_t)gt.size();
        uint32_t b0 = (uint32_t)(((uint64_t)q << shift) / 32);
        uint32_t b1 = (uint32_t)std::min<uint64_t>((((uint64_t)q + 1) << shift) / 32, nblk);
        uint32_t base = b0;
        while (b0 < b1) {
            uint32_t b = b0;
            uint64_t in = 0;
            while (b < b1 && b - b0 < width_blocks && (b == b0 || in + hin[b] <= tgt)) in += hin[b++];
            gt.push_back(GatherTask{q, (b0 - base) * 32, (b - base) * 32, (uint32_t)std::min<uint64_t>(in, 0xFFFFFFFFu)});
            b0 = b;
        }
    }
    col_task[k] = (uint32_t)gt.size();
    g->ngt = (uint32_t)gt.size();
    GPOP_CUDA_TRY(t.keep(g, &g->gtask, g->ngt));
    GPOP_CUDA_TRY(t.keep(g, &g->col_task, (uint64_t)k + 1));
    GPOP_CUDA_TRY(cudaMemcpyAsync(g->gtask, gt.data(), sizeof(GatherTask) * gt.size(), cudaMemcpyHostToDevice, s));
    GPOP_CUDA_TRY(cudaMemcpyAsync(g->col_task, col_task.data(), 4ull * (k + 1), cudaMemcpyHostToDevice, s));

    // 10. static PC scatter tasks: padded rows in chunks of about 1/6 of an SM's share of the slots, so that a hub
    //     partition's row spreads over the SMs also in a graph of few rows; a chunk stages its partition's P values,
    //     so it has at least P / 2 slots (a slot costs 6.5 bytes, a staged value 4), and at most kScatterChunk.
    //     R-MAT 20 (6.7 M slots, P = 4096): 42 us a launch with 131072-slot chunks, 15 us now (16.5 us when the chunk was
    //     a multiple of 4096).  Tasks of 65536 slots or more get CTAs of 1024 threads: with 1024 and 512 threads R-MAT 24
    //     (131072 slots) took 162 and 167 us, R-MAT 22 with BF16 messages (24576) 36.6 and 35.0, R-MAT 20 (6144) 20.8 and 15.1
    const uint64_t share = g->npng_pad / (6ull * (uint64_t)std::max(1, g->num_sms));
    const uint32_t chunk = (uint32_t)std::min<uint64_t>(kScatterChunk, std::max<uint64_t>({share, P / 2, kScatterMin}) / kScatterUnit * kScatterUnit);
    g->st_threads = chunk >= 65536 ? 1024 : 512;
    std::vector<ScatterTask> st;
    for (uint32_t p = 0; p < k; ++p)
        for (uint64_t b = hrow_png[p]; b < hrow_png[p + 1]; b += chunk)
            st.push_back(ScatterTask{p, (uint32_t)b, (uint32_t)std::min<uint64_t>(b + chunk, hrow_png[p + 1]), b == hrow_png[p]});
    g->nst = (uint32_t)st.size();
    GPOP_CUDA_TRY(t.keep(g, &g->stask, g->nst));
    if (g->nst)
        GPOP_CUDA_TRY(cudaMemcpyAsync(g->stask, st.data(), sizeof(ScatterTask) * st.size(), cudaMemcpyHostToDevice, s));

    // 11. SC bins at gather-task granularity: bin (p, t) receives the SC pairs from partition p to the
    //     destinations of gather task t (capacity = edges p -> t), so each gather task reads only its own
    {
        uint32_t *d_task_of, *row_hist, *task_hist, *d_nsub;
        GPOP_CUDA_TRY(t.alloc(&d_task_of, V));
        GPOP_CUDA_TRY(t.alloc(&row_hist, (uint64_t)k + 1));
        GPOP_CUDA_TRY(t.alloc(&task_hist, (uint64_t)g->ngt + 1));
        GPOP_CUDA_TRY(t.alloc(&d_nsub, 1));
        k_task_of<<<g->ngt, kThreads, 0, s>>>(g->gtask, shift, V, d_task_of);
        GPOP_CUDA_TRY(cudaMemsetAsync(row_hist, 0, 4ull * (k + 1), s));
        GPOP_CUDA_TRY(cudaMemsetAsync(task_hist, 0, 4ull * (g->ngt + 1), s));
        GPOP_CUDA_TRY(cudaMemsetAsync(d_nsub, 0, 4, s));
        uint32_t nsub = 0;
        // the distinct keys, ascending, with the edges of each: 32-bit keys (3 sort passes over 4 B an edge for 4 M
        // pairs of partition and task) wherever the pairs allow it
        auto sub_bins = [&](auto zero) -> gpop_status {
            using K = decltype(zero);
            K *skey, *skey2, *ukey;
            uint32_t *counts;
            GPOP_CUDA_TRY(t.alloc(&skey, E));
            GPOP_CUDA_TRY(t.alloc(&skey2, E));
            GPOP_CUDA_TRY(t.alloc(&counts, E + 1));
            if (E) {
                k_sub_keys<<<blocks_for(E), kThreads, 0, s>>>(E, shift, g->ngt, src, g->col, d_task_of, skey);
                GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                    return cub::DeviceRadixSort::SortKeys(tmp, bytes, skey, skey2, E, 0, bits_for((uint64_t)k * g->ngt), s);
                }));
            }
            ukey = skey;  // the unsorted keys are no longer needed
            if (E) {
                GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                    return cub::DeviceRunLengthEncode::Encode(tmp, bytes, skey2, ukey, counts, d_nsub, (int64_t)E, s);
                }));
                GPOP_CUDA_TRY(cudaMemcpyAsync(&nsub, d_nsub, 4, cudaMemcpyDeviceToHost, s));
                GPOP_CUDA_TRY(cudaStreamSynchronize(s));
            }
            g->nsub = nsub;
            GPOP_CUDA_TRY(t.keep(g, &g->sub_cap, (uint64_t)nsub + 1));
            GPOP_CUDA_TRY(t.keep(g, &g->sub_task, nsub));
            GPOP_CUDA_TRY(cudaMemsetAsync(counts + nsub, 0, 4, s));
            GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
                return cub::DeviceScan::ExclusiveSum(tmp, bytes, counts, g->sub_cap, (uint64_t)nsub + 1, s);
            }));
            if (nsub) k_sub_split<<<blocks_for(nsub), kThreads, 0, s>>>(nsub, g->ngt, ukey, g->sub_task, row_hist, task_hist);
            return GPOP_OK;
        };
        const gpop_status sst = (uint64_t)k * g->ngt <= 0xFFFFFFFFull ? sub_bins(uint32_t{0}) : sub_bins(uint64_t{0});
        if (sst != GPOP_OK) return sst;
        GPOP_CUDA_TRY(t.keep(g, &g->row_sub, (uint64_t)k + 1));
        GPOP_CUDA_TRY(t.keep(g, &g->task_sub_ptr, (uint64_t)g->ngt + 1));
        GPOP_CUDA_TRY(t.keep(g, &g->esub, E));
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceScan::ExclusiveSum(tmp, bytes, row_hist, g->row_sub, (uint64_t)k + 1, s);
        }));
        GPOP_CUDA_TRY(cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceScan::ExclusiveSum(tmp, bytes, task_hist, g->task_sub_ptr, (uint64_t)g->ngt + 1, s);
        }));
        std::vector<uint32_t> hrow(k);
        GPOP_CUDA_TRY(cudaMemcpyAsync(hrow.data(), row_hist, 4ull * k, cudaMemcpyDeviceToHost, s));
        GPOP_CUDA_TRY(cudaStreamSynchronize(s));
        g->max_row_subs = 0;
        for (uint32_t p = 0; p < k; ++p) g->max_row_subs = std::max(g->max_row_subs, hrow[p]);
        if (g->max_row_subs > kMaxRowBins)
            return fail(GPOP_ERR_INVALID_ARG, "a partition sends SC messages to more gather tasks than the SC "
                                              "scatter supports; use a larger partition size");
        if (E) k_edge_sub<<<blocks_for(E), kThreads, 0, s>>>(E, shift, src, g->col, d_task_of, g->row_sub,
                                                             g->sub_task, g->esub);
    }
    GPOP_CUDA_TRY(t.keep(g, &g->scpair, E));
    GPOP_CUDA_TRY(t.keep(g, &g->sccnt, g->nsub));
    GPOP_CUDA_TRY(t.keep(g, &g->pc_state, k));
    GPOP_CUDA_TRY(cudaMemsetAsync(g->pc_state, 0, k, s));
    // 12. small graphs: a range of destinations for each CTA of k_small, two per SM less one, of equal work (in-edges, and
    //     a vertex as vcost of them: its own, and enough that no range has more than kSmallDest).  Not where a hub would
    //     leave one CTA several times its share of the messages, nor without memory for it: the iteration's kernels run any
    //     graph.  Ten PageRank iterations and a BFS, one launch / the iteration's kernels (us), with a hub of the given
    //     in-degree: 100,000 vertices and 2 M edges, 30,000: 206 / 388, 110 / 226; 60,000: 306 / 403, 153 / 215; 120,000:
    //     497 / 406, 243 / 228; 20,000 vertices and 200,000 edges, 10,000: 110 / 327, 65 / 246; 50,000: 242 / 336, 153 / 253;
    //     100,000: 405 / 348, 279 / 298.  The line (34,600 and 10,800 there) lies well inside.
    const uint64_t nrg = 2ull * (uint64_t)std::max(1, g->num_sms) - 1;
    if (E && E <= kSmallEdges && V < kSmallSrc && nrg * kSmallDest > 2ull * V) {
        ArrayGroup arrays(g);
        auto small_layout = [&]() -> cudaError_t {
            const uint64_t vcost = std::max<uint64_t>(4, E / (nrg * kSmallDest - V) + 1);
            uint32_t *key, *key2, *num, *num2, *start, *d_first;
            uint2 *d_cut;
            cudaError_t e = cudaSuccess;
            auto A = [&](auto **p, uint64_t n) {
                if (e == cudaSuccess) e = t.alloc(p, n);
            };
            A(&key, E); A(&key2, E); A(&num, E); A(&num2, E);
            A(&start, (uint64_t)V + 1);
            A(&d_cut, nrg + 1);
            if (e != cudaSuccess) return e;
            k_small_keys<<<blocks_for(E), kThreads, 0, s>>>(E, g->col, key, num);
            e = cub_run(t, [&](void *tmp, size_t &bytes) {
                return cub::DeviceRadixSort::SortPairs(tmp, bytes, key, key2, num, num2, E, 0, bits_for(V), s);
            });
            if (e != cudaSuccess) return e;
            k_small_starts<<<blocks_for(E + 1), kThreads, 0, s>>>(E, V, key2, start);
            k_small_cuts<<<blocks_for(nrg + 1), kThreads, 0, s>>>((uint32_t)nrg, V, E, vcost, start, d_cut);
            std::vector<uint2> cut(nrg + 1);
            e = cudaMemcpyAsync(cut.data(), d_cut, sizeof(uint2) * (nrg + 1), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return e;
            std::vector<uint4> rg;
            std::vector<uint32_t> first;
            uint32_t quads = 0, largest = 0, widest = 0;
            for (uint64_t j = 0; j < nrg; ++j) {
                const uint32_t nd = cut[j + 1].x - cut[j].x, in = cut[j + 1].y - cut[j].y;
                if (nd == 0) continue;
                rg.push_back(make_uint4(cut[j].x, nd, quads, (in + 3) / 4));
                first.push_back(cut[j].y);
                quads += (in + 3) / 4;
                largest = std::max(largest, in);
                widest = std::max(widest, nd);
            }
            first.push_back((uint32_t)E);
            if (widest > kSmallDest || largest > 4 * (E / nrg) + 8192) return cudaSuccess;
            A(&d_first, first.size());
            arrays.add(&g->sm_range, rg.size());
            arrays.add(&g->sm_edge, quads);
            if (g->weighted) arrays.add(&g->sm_w, quads);
            if (e == cudaSuccess) e = arrays.error;
            if (e == cudaSuccess) e = cudaMemcpyAsync(g->sm_range, rg.data(), sizeof(uint4) * rg.size(), cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess) e = cudaMemcpyAsync(d_first, first.data(), 4ull * first.size(), cudaMemcpyHostToDevice, s);
            if (e != cudaSuccess) return e;
            g->sm_n = (uint32_t)rg.size();
            g->sm_wide = widest;
            k_small_words<<<g->sm_n, kThreads, 0, s>>>(g->sm_n, V, g->sm_range, d_first, num2, src, g->col, g->w,
                                                       reinterpret_cast<uint32_t *>(g->sm_edge), reinterpret_cast<uint32_t *>(g->sm_w));
            return cudaStreamSynchronize(s);
        };
        const cudaError_t e = small_layout();
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            arrays.give_back();
            g->sm_n = 0;
        } else {
            GPOP_CUDA_TRY(e);
        }
    }
    GPOP_CUDA_TRY(cudaStreamSynchronize(s));
    GPOP_CUDA_TRY(cudaGetLastError());
    return GPOP_OK;
}

}  // namespace gpop

// In-edges by destination for the batched PPR: 8 bytes an edge and 4 a vertex, made once per graph.  A share is what a
// quarter of a warp takes: half an SM's part over its 256 quarters, 64 to 512 edges.
gpop_status gpop::make_in_edges(Graph *g, cudaStream_t s) {
    static std::mutex once;  // calls on one graph from several threads
    const std::lock_guard<std::mutex> lock(once);
    const uint64_t E = g->E;
    if (g->in_off) return GPOP_OK;
    Temps t(s);
    uint32_t *src, *src2, *key2, *none, *off = nullptr, *d_n, n = 0;
    uint2 *edge = nullptr;
    uint4 *span = nullptr;
    const uint32_t share = (uint32_t)std::min<uint64_t>(512, std::max<uint64_t>(64, E / (512ull * (uint64_t)std::max(1, g->num_sms)) / 8 * 8));
    const uint32_t shares = (uint32_t)((E + share - 1) / share);
    cudaError_t e = cudaSuccess;
    auto A = [&](auto **p, uint64_t m) {
        if (e == cudaSuccess) e = t.alloc(p, m);
    };
    A(&src, E); A(&src2, E); A(&key2, E); A(&none, 1); A(&d_n, 1);
    ArrayGroup arrays(g);
    arrays.add(&off, (uint64_t)g->V + 1);
    arrays.add(&edge, E);
    arrays.add(&span, shares);
    if (e == cudaSuccess) e = arrays.error;
    if (e == cudaSuccess) e = cudaMemsetAsync(d_n, 0, 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(none, 0, 4, s);
    if (e == cudaSuccess && E) {
        k_edge_src<<<blocks_for(E, (int)kSrcTile), kThreads, 0, s>>>(g->V, E, g->rowptr, g->col, src, none);
        e = cub_run(t, [&](void *tmp, size_t &bytes) {
            return cub::DeviceRadixSort::SortPairs(tmp, bytes, g->col, key2, src, src2, E, 0, bits_for(g->V), s);
        });
        if (e == cudaSuccess) {  // (unsorted keys would send the kernels' stores anywhere)
            k_small_starts<<<blocks_for(E + 1), kThreads, 0, s>>>(E, g->V, key2, off);
            k_in_edges<<<blocks_for(E), kThreads, 0, s>>>(E, share, key2, src2, off, edge, span, d_n);
            e = cudaMemcpyAsync(&n, d_n, 4, cudaMemcpyDeviceToHost, s);
        }
    } else if (e == cudaSuccess) {
        e = cudaMemsetAsync(off, 0, 4ull * (g->V + 1ull), s);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        arrays.give_back();
        return fail(e == cudaErrorMemoryAllocation ? GPOP_ERR_OOM : GPOP_ERR_CUDA, std::string("in-edges: ") + cudaGetErrorString(e));
    }
    g->in_off = off; g->in_edge = edge; g->in_span = span;
    g->in_share = share; g->n_share = shares; g->n_span = n;
    return GPOP_OK;
}

using namespace gpop;

extern "C" gpop_status gpop_graph_build(uint32_t num_vertices, uint64_t num_edges, const uint64_t *row_ptr,
                                        const uint32_t *col, const int32_t *weights, uint32_t partition_size,
                                        int mem_is_device, void *cuda_stream, gpop_graph **out) {
    set_error("");
    if (!out) return fail(GPOP_ERR_INVALID_ARG, "out is NULL");
    if (num_vertices == 0 || num_vertices >= (1u << 31)) return fail(GPOP_ERR_INVALID_ARG, "num_vertices out of range");
    if (num_edges >= (1ull << 32)) return fail(GPOP_ERR_INVALID_ARG, "num_edges must be < 2^32");
    if (!row_ptr || (num_edges && !col)) return fail(GPOP_ERR_INVALID_ARG, "row_ptr/col is NULL");
    uint32_t P = partition_size;
    if (P == 0) {
        P = 32;
        while (P < 16384 && P < num_vertices) P <<= 1;
    }
    if (P < 32 || P > 16384 || (P & (P - 1))) return fail(GPOP_ERR_INVALID_ARG, "partition_size must be a power of two in [32, 16384]");
    if (((uint64_t)num_vertices + P - 1) / P > 65536) return fail(GPOP_ERR_INVALID_ARG, "more than 65536 partitions");
    gpop_graph *h = new (std::nothrow) gpop_graph();
    if (!h) return fail(GPOP_ERR_OOM, "host allocation failed");
    gpop_status st = build_impl(&h->g, num_vertices, num_edges, row_ptr, col, weights, P, mem_is_device,
                                (cudaStream_t)cuda_stream);
    if (st != GPOP_OK) {
        cudaGetLastError();
        free_graph(&h->g);
        delete h;
        if (st == GPOP_ERR_CUDA && std::string(gpop_last_error()).find("out of memory") != std::string::npos)
            st = GPOP_ERR_OOM;
        return st;
    }
    *out = h;
    return GPOP_OK;
}

extern "C" gpop_status gpop_graph_build_union(uint32_t num_graphs, const uint32_t *num_vertices,
                                              const uint64_t *num_edges, const uint64_t *const *row_ptrs,
                                              const uint32_t *const *cols, const int32_t *const *weights,
                                              uint32_t partition_size, void *cuda_stream, gpop_graph **out) {
    set_error("");
    if (!out || !num_vertices || !num_edges || !row_ptrs || !cols) return fail(GPOP_ERR_INVALID_ARG, "NULL argument");
    if (num_graphs == 0) return fail(GPOP_ERR_INVALID_ARG, "no graphs");
    // the union's CSR: graph i's vertices follow graph i-1's, its edges shifted by its first vertex
    std::vector<uint32_t> goff(num_graphs + 1, 0);
    uint64_t V = 0, E = 0;
    for (uint32_t i = 0; i < num_graphs; ++i) {
        if (num_vertices[i] == 0) return fail(GPOP_ERR_INVALID_ARG, "a graph without vertices");
        if (!row_ptrs[i] || (num_edges[i] && !cols[i])) return fail(GPOP_ERR_INVALID_ARG, "a graph's row_ptr/col is NULL");
        if ((weights != nullptr) && !weights[i] && num_edges[i]) return fail(GPOP_ERR_INVALID_ARG, "weights for some graphs only");
        if (row_ptrs[i][0] != 0 || row_ptrs[i][num_vertices[i]] != num_edges[i])
            return fail(GPOP_ERR_INVALID_ARG, "a graph's row_ptr does not span its edges");
        goff[i] = (uint32_t)std::min<uint64_t>(V, 0xFFFFFFFFull);
        V += num_vertices[i];
        E += num_edges[i];
        if (V >= (1ull << 31)) return fail(GPOP_ERR_INVALID_ARG, "the union has 2^31 vertices or more");
        if (E >= (1ull << 32)) return fail(GPOP_ERR_INVALID_ARG, "the union has 2^32 edges or more");
    }
    goff[num_graphs] = (uint32_t)V;
    std::vector<uint64_t> rp(V + 1);
    std::vector<uint32_t> col(std::max<uint64_t>(E, 1));
    std::vector<int32_t> w(weights ? std::max<uint64_t>(E, 1) : 0);
    uint64_t eo = 0;
    for (uint32_t i = 0; i < num_graphs; ++i) {
        const uint32_t n = num_vertices[i], base = goff[i];
        for (uint32_t v = 0; v < n; ++v) rp[base + v] = eo + row_ptrs[i][v];
        for (uint64_t e = 0; e < num_edges[i]; ++e) {
            if (cols[i][e] >= n) return fail(GPOP_ERR_INVALID_ARG, "a destination outside its graph");
            col[eo + e] = base + cols[i][e];
            if (weights) w[eo + e] = weights[i][e];
        }
        eo += num_edges[i];
    }
    rp[V] = E;
    gpop_status st = gpop_graph_build((uint32_t)V, E, rp.data(), col.data(), weights ? w.data() : nullptr,
                                      partition_size, 0, cuda_stream, out);
    if (st == GPOP_OK) (*out)->g.goff = std::move(goff);
    return st;
}

extern "C" gpop_status gpop_graph_union_offsets(const gpop_graph *h, uint32_t *offsets, uint32_t *num_graphs) {
    if (!h || !num_graphs) return fail(GPOP_ERR_INVALID_ARG, "NULL argument");
    const uint32_t n = h->g.goff.empty() ? 0u : (uint32_t)h->g.goff.size() - 1;
    *num_graphs = n;
    if (offsets)
        for (uint32_t i = 0; i <= n && n; ++i) offsets[i] = h->g.goff[i];
    return GPOP_OK;
}

extern "C" gpop_status gpop_graph_get_info(const gpop_graph *h, gpop_graph_info *info) {
    if (!h || !info) return fail(GPOP_ERR_INVALID_ARG, "NULL argument");
    const Graph &g = h->g;
    memset(info, 0, sizeof *info);
    info->num_vertices = g.V;
    info->partition_size = g.P;
    info->num_partitions = g.k;
    info->weighted = (uint32_t)g.weighted;
    info->num_edges = g.E;
    info->num_bins = g.nb;
    info->num_png = g.npng;
    info->num_png_padded = g.npng_pad;
    info->num_gather_tasks = g.ngt;
    info->num_scatter_tasks = g.nst;
    info->max_row_bins = g.max_row_bins;
    info->device_bytes = g.device_bytes;
    info->num_pc_blocks = g.npcb;
    info->num_pc_tasks = g.npct;
    info->num_pc_partials = g.npart;
    return GPOP_OK;
}

extern "C" gpop_status gpop_graph_partition_stats(const gpop_graph *h, uint64_t *edges, uint64_t *png) {
    if (!h) return fail(GPOP_ERR_INVALID_ARG, "NULL graph");
    for (uint32_t p = 0; p < h->g.k; ++p) {
        if (edges) edges[p] = h->g.h_Ep[p];
        if (png) png[p] = h->g.h_npng[p];
    }
    return GPOP_OK;
}

extern "C" void gpop_graph_destroy(gpop_graph *h) {
    if (!h) return;
    free_graph(&h->g);
    delete h;
}

extern "C" const char *gpop_last_error(void) { return gpop::g_last_error.c_str(); }
