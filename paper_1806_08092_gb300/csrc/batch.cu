// Batched seeded personalized PageRank (gpop_run_ppr_batch): up to 32 seeds per pass through the
// partition-centric gather of Alg. 2 on the PC layout of Alg. 3, every message carrying one FP32 value per
// seed (lane j of a warp holds seed j).
//
// A message is 128 bytes against the 4 of its index, and its value is the same for every destination partition:
// it is read where its source keeps it instead of being copied into a bin per partition.  The hub sources'
// messages, which most entries name, then stay in L2.  One pass = per iteration:
//   k_bmark     the columns that partitions with an active vertex (for any seed: the union frontier) send to;
//   k_bpull     a quarter of a warp takes an equal share of the in-edges, sorted by destination, four seeds a lane: 16
//               bytes of a message each, eight messages in flight per quarter, the sum of a destination in registers
//               (compensated, so its length costs no accuracy), a fixed order;
//   k_bfix      the destinations that shares cut: their partial sums in order;
//   k_bfilter   x_j = alpha [v = s_j] + (1 - alpha) sum_j, the next message (where the sum was), the active flags and
//               each seed's L1 change.
// L1 changes are added as 62-bit fixed point, exact in any order.
// Bound by the 128 bytes an in-edge reads through L2.  Measured on R-MAT 20 (48 seeds in two passes of 40 iterations):
// a call took 195 ms with a bin slot per (source, destination partition) written and read back; 82.6 ms with the
// messages read at their sources by CTAs that each fold a column's block, where a hub's warp keeps the others waiting
// at the block's barrier; now 27 ms (pull
// 0.19 ms an iteration, 10.7 TB/s out of L2).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "gpop_internal.cuh"

namespace gpop {
namespace {

constexpr uint32_t kSeeds = 32;                  // seeds per pass, one lane each
constexpr uint32_t kBatchMaxP = 1024;            // the interface's limit on the partition size
constexpr int kBThreads = 256;
constexpr int kBWarps = kBThreads / 32;
constexpr double kFixOne = 0x1p62, kFixUnit = 0x1p-62;  // fixed point of the L1 change (at most 2)

struct BParams {
    uint32_t V, shift, k;
    const uint32_t *rowptr, *Ep, *row_bin, *bin_q;
    const uint32_t *in_off;  // in-edges by destination, and the destinations that shares cut (Graph::in_off)
    const uint2 *in_edge;
    const uint4 *in_span;
    uint32_t share, n_share, n_span;
    uint64_t E;
    const uint32_t *seed;     // [32]: the pass's seeds, kNull for unused lanes
    float *X, *M, *Mnext;     // V x 32 each: values, this iteration's messages, the next one's
    float *part;              // two partial sums of 32 per share: of its first and of its last destination
    uint8_t *pact, *pact_prev, *pact_next;  // partitions with an active vertex: now, last iteration, next
    uint32_t *gflag;          // column received messages this iteration (== epoch)
    unsigned long long *edges;  // out-edges of the scattered partitions, summed over iterations
    unsigned long long *res;  // per seed: L1 change of the iteration (fixed point)
    float c0, c1;             // alpha, 1 - alpha
    uint32_t epoch;
};

// seeds: value 1 and message 1 / deg on their own lane (FP32, as the single-seed run computes it)
__global__ void k_binit(BParams p) {
    const uint32_t j = threadIdx.x;
    if (j >= kSeeds) return;
    const uint32_t s = p.seed[j];
    if (s == kNull) return;
    const uint32_t deg = p.rowptr[s + 1] - p.rowptr[s];
    p.X[(uint64_t)s * kSeeds + j] = 1.f;
    p.M[(uint64_t)s * kSeeds + j] = deg ? 1.f / (float)deg : 0.f;
    p.pact[s >> p.shift] = 1;
}

// columns that receive messages (bin row of every active partition), and the iteration's counters
__global__ void __launch_bounds__(kBThreads) k_bmark(BParams p) {
    if (blockIdx.x == 0 && threadIdx.x < kSeeds) p.res[threadIdx.x] = 0ull;
    for (uint32_t q = blockIdx.x; q < p.k; q += gridDim.x) {
        if (threadIdx.x == 0) p.pact_next[q] = 0;
        if (!p.pact[q]) continue;
        for (uint32_t b = p.row_bin[q] + threadIdx.x; b < p.row_bin[q + 1]; b += kBThreads)
            p.gflag[p.bin_q[b]] = p.epoch;
        if (threadIdx.x == 0) atomicAdd(p.edges, (unsigned long long)p.Ep[q]);
    }
}

// whether a column's vertices can change: it receives messages or has, or had, active vertices (otherwise its values
// and both its message buffers are zero)
__device__ __forceinline__ bool column_live(const BParams &p, uint32_t q) {
    return p.gflag[q] == p.epoch || p.pact[q] || p.pact_prev[q];
}

// One quarter of a warp per share of the in-edges (see the top of the file); the sums go to the rows of the next messages
__global__ void __launch_bounds__(kBThreads, 4) k_bpull(BParams p) {
    const uint32_t lane = threadIdx.x & 31, l8 = lane & 7, q0 = lane & 24;
    const uint32_t c = (blockIdx.x * kBThreads + threadIdx.x) / 8;  // share
    const uint64_t e0 = (uint64_t)c * p.share;
    uint32_t n = c < p.n_share ? (uint32_t)min((uint64_t)p.share, p.E - e0) : 0u;
    const uint2 *edge = p.in_edge + e0;
    uint32_t d = kNull, dl = kNull;
    bool cut = false;   // the first destination began in an earlier share
    bool more = false;  // the last one goes on in the next
    if (n) {
        d = edge[0].y;
        dl = edge[n - 1].y;
        cut = e0 > 0 && edge[-1].y == d;
        more = e0 + n < p.E && edge[n].y == dl;
        bool live = false;  // any column of its destinations may change
        for (uint32_t q = d >> p.shift; q <= dl >> p.shift; ++q) live |= column_live(p, q);
        if (!live) n = 0;
    }
    const uint32_t dA = d;
    const float4 *M = reinterpret_cast<const float4 *>(p.M);
    float4 *S = reinterpret_cast<float4 *>(p.Mnext), *part = reinterpret_cast<float4 *>(p.part) + (uint64_t)c * 16 + l8;
    float sum[4] = {0.f, 0.f, 0.f, 0.f}, lost[4] = {0.f, 0.f, 0.f, 0.f};
    auto put = [&](float4 *to) { *to = make_float4(sum[0], sum[1], sum[2], sum[3]); };
    uint2 en = l8 < n ? edge[l8] : make_uint2(0u, kNull);
    for (uint32_t base = 0; __any_sync(0xffffffffu, base < n); base += 8) {
        const uint2 ec = en;
        en = base + 8 + l8 < n ? edge[base + 8 + l8] : make_uint2(0u, kNull);
        float4 v[8];
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
            const uint32_t u = __shfl_sync(0xffffffffu, ec.x, (int)(q0 + k));
            v[k] = base + k < n ? M[(uint64_t)u * 8 + l8] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
            const uint32_t dk = __shfl_sync(0xffffffffu, ec.y, (int)(q0 + k));
            if (dk != kNull && dk != d) {  // a later destination
                put(d == dA && cut ? part : S + (uint64_t)d * 8 + l8);
                d = dk;
                sum[0] = sum[1] = sum[2] = sum[3] = 0.f;
                lost[0] = lost[1] = lost[2] = lost[3] = 0.f;
            }
            const float x[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float y = x[j] - lost[j], t = sum[j] + y;
                lost[j] = (t - sum[j]) - y;
                sum[j] = t;
            }
        }
    }
    if (n) put(d == dA && cut ? part : more ? part + 8 : S + (uint64_t)d * 8 + l8);
}

// One warp per destination that shares cut: its sum to the row of its next message
__global__ void __launch_bounds__(kBThreads) k_bfix(BParams p) {
    const int lane = threadIdx.x & 31;
    const uint32_t i = blockIdx.x * kBWarps + (threadIdx.x >> 5);
    if (i >= p.n_span) return;
    const uint4 sp = p.in_span[i];
    if (!column_live(p, sp.x >> p.shift)) return;
    const float *part = p.part + (uint64_t)sp.y * 2 * kSeeds + lane;
    float sum = part[kSeeds], lost = 0.f;  // its first share: the last destination there
    for (uint32_t c0 = 1; c0 < sp.z; c0 += 8) {
        float x[8];
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u) x[u] = c0 + u < sp.z ? part[(uint64_t)(c0 + u) * 2 * kSeeds] : 0.f;
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u) {
            const float y = x[u] - lost, t = sum + y;
            lost = (t - sum) - y;
            sum = t;
        }
    }
    p.Mnext[(uint64_t)sp.x * kSeeds + lane] = sum;
}

// PPR's filterFunc of every vertex of the live columns: a warp takes 8 vertices at a time, lane j for seed j
__global__ void __launch_bounds__(kBThreads, 4) k_bfilter(BParams p) {
    __shared__ unsigned long long s_res[kSeeds];
    const int lane = threadIdx.x & 31;
    const uint32_t seed = p.seed[lane];
    unsigned long long res = 0;
    if (threadIdx.x < kSeeds) s_res[threadIdx.x] = 0ull;
    __syncthreads();
    for (uint64_t w = blockIdx.x * (uint64_t)kBWarps + (threadIdx.x >> 5); w * 8 < p.V; w += (uint64_t)gridDim.x * kBWarps) {
        const uint32_t v0 = (uint32_t)w * 8;
        if (!column_live(p, v0 >> p.shift)) continue;  // (a partition has a multiple of 8 vertices)
        const uint32_t n = min(8u, p.V - v0), at = v0 + min((uint32_t)lane, n);
        const uint32_t rp = p.rowptr[at], io = p.in_off[at];  // offsets, one per lane
        // vertices with in-edges; the others keep zero rows, and are passed over, unless a seed is near
        const uint32_t has = __ballot_sync(0xffffffffu, __shfl_down_sync(0xffffffffu, io, 1) != io) & 0xFFu;
        const uint32_t todo = (__any_sync(0xffffffffu, seed >> 3 == v0 >> 3) ? 0xFFu : has) & ((1u << n) - 1u);
        if (!todo) continue;
        float acc[8], xo[8], fres = 0.f;
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
            const uint64_t o = (uint64_t)(v0 + k) * kSeeds + lane;
            acc[k] = (has >> k) & (todo >> k) & 1u ? p.Mnext[o] : 0.f;
            xo[k] = (todo >> k) & 1u ? p.X[o] : 0.f;
        }
        bool on = false;
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
            const uint32_t deg = __shfl_sync(0xffffffffu, rp, (int)k + 1) - __shfl_sync(0xffffffffu, rp, (int)k);
            if (!((todo >> k) & 1u)) continue;
            const uint64_t o = (uint64_t)(v0 + k) * kSeeds + lane;
            const float xn = fmaf(p.c1, acc[k], v0 + k == seed ? p.c0 : 0.f);
            p.X[o] = xn;
            p.Mnext[o] = deg ? xn / (float)deg : 0.f;
            fres += fabsf(xn - xo[k]);
            on |= xn > 0.f;
        }
        if (__any_sync(0xffffffffu, on) && lane == 0) p.pact_next[v0 >> p.shift] = 1;
        res += __double2ull_rn((double)fres * kFixOne);
    }
    if (res) atomicAdd(&s_res[lane], res);
    __syncthreads();
    if (threadIdx.x < kSeeds && s_res[lane]) atomicAdd(&p.res[lane], s_res[lane]);
}

// rows of the result: out[j][v] = X[v][j] for the pass's seeds, through 32 x 32 shared tiles
__global__ void k_btranspose(const float *X, float *out, uint32_t V, uint32_t nseeds) {
    __shared__ float tile[32][33];
    const uint32_t v0 = blockIdx.x * 32;
    for (uint32_t r = threadIdx.y; r < 32; r += blockDim.y) {
        const uint32_t v = v0 + r;
        tile[r][threadIdx.x] = v < V ? X[(uint64_t)v * kSeeds + threadIdx.x] : 0.f;
    }
    __syncthreads();
    for (uint32_t j = threadIdx.y; j < nseeds; j += blockDim.y) {
        const uint32_t v = v0 + threadIdx.x;
        if (v < V) out[(uint64_t)j * V + v] = tile[threadIdx.x][j];
    }
}

struct BatchBuffers {
    std::vector<void *> ptrs;
    ~BatchBuffers() {
        for (void *q : ptrs) cudaFree(q);
    }
    template <typename T>
    cudaError_t alloc(T **q, uint64_t n) {
        void *r = nullptr;
        cudaError_t e = cudaMalloc(&r, std::max<uint64_t>(n, 1) * sizeof(T));
        if (e == cudaSuccess) ptrs.push_back(r);
        *q = static_cast<T *>(r);
        return e;
    }
};

}  // namespace
}  // namespace gpop

using namespace gpop;

extern "C" gpop_status gpop_run_ppr_batch(gpop_graph *h, const gpop_run_opts *o, const uint32_t *seeds,
                                          uint32_t num_seeds, float *out_values, int out_is_device,
                                          gpop_run_stats *stats) {
    set_error("");
    if (!h || !o) return fail(GPOP_ERR_INVALID_ARG, "NULL graph or options");
    Graph *g = &h->g;
    if (num_seeds && (!seeds || !out_values)) return fail(GPOP_ERR_INVALID_ARG, "NULL seeds or output buffer");
    for (uint32_t j = 0; j < num_seeds; ++j)
        if (seeds[j] >= g->V) return fail(GPOP_ERR_INVALID_ARG, "seed out of range");
    if (!(o->damping > 0.0 && o->damping < 1.0)) return fail(GPOP_ERR_INVALID_ARG, "damping must be in (0, 1)");
    if (o->msg_bf16 || o->resume) return fail(GPOP_ERR_INVALID_ARG, "batched PPR: msg_bf16 and resume must be 0");
    if (g->P > kBatchMaxP)
        return fail(GPOP_ERR_INVALID_ARG, "batched PPR: partition size must be at most 1024");
    gpop_run_stats total;
    memset(&total, 0, sizeof total);
    total.converged = 1;
    if (num_seeds == 0) {
        if (stats) *stats = total;
        return GPOP_OK;
    }
    cudaStream_t s = (cudaStream_t)o->cuda_stream;
    const gpop_status ins = make_in_edges(g, s);
    if (ins != GPOP_OK) return ins;
    BatchBuffers bb;
    BParams p{};
    p.V = g->V; p.shift = g->shift; p.k = g->k; p.E = g->E;
    p.rowptr = g->rowptr; p.Ep = g->Ep; p.row_bin = g->row_bin; p.bin_q = g->bin_q;
    p.in_off = g->in_off; p.in_edge = g->in_edge; p.in_span = g->in_span;
    p.share = g->in_share; p.n_share = g->n_share; p.n_span = g->n_span;
    p.c0 = (float)(1.0 - o->damping);
    p.c1 = (float)o->damping;
    const uint64_t V32 = (uint64_t)g->V * kSeeds;
    const uint32_t grid_p = (uint32_t)(((uint64_t)g->n_share * 8 + kBThreads - 1) / kBThreads);
    const uint32_t grid_x = (g->n_span + kBWarps - 1) / kBWarps;
    const uint32_t grid_f = (uint32_t)std::min<uint64_t>((g->V + 8ull * kBWarps - 1) / (8 * kBWarps), 16ull * g->num_sms);
    const uint32_t grid_k = std::min<uint32_t>(g->k, 8u * g->num_sms);
    uint32_t *d_seed = nullptr;
    uint8_t *pa[3] = {};
    float *staging = nullptr, *msg[2] = {};
    cudaError_t e = cudaSuccess;
    auto A = [&](auto **ptr, uint64_t n) {
        if (e == cudaSuccess) e = bb.alloc(ptr, n);
    };
    A(&p.X, V32); A(&msg[0], V32); A(&msg[1], V32);
    A(&p.part, (uint64_t)g->n_share * 2 * kSeeds);
    A(&pa[0], g->k); A(&pa[1], g->k); A(&pa[2], g->k);
    A(&p.gflag, g->k);
    A(&p.edges, 1);
    A(&p.res, kSeeds);
    A(&d_seed, kSeeds);
    if (!out_is_device) A(&staging, V32);
    if (e != cudaSuccess)
        return fail(e == cudaErrorMemoryAllocation ? GPOP_ERR_OOM : GPOP_ERR_CUDA,
                    std::string("batched PPR buffers: ") + cudaGetErrorString(e));
    p.seed = d_seed;
    const bool prof = o->profile_kernels != 0;
    cudaEvent_t ev0, ev1, kev[2];
    GPOP_CUDA_TRY(cudaEventCreate(&ev0));
    GPOP_CUDA_TRY(cudaEventCreate(&ev1));
    GPOP_CUDA_TRY(cudaEventCreate(&kev[0]));
    GPOP_CUDA_TRY(cudaEventCreate(&kev[1]));
    auto timed = [&](int kind, auto launch) {
        if (prof) cudaEventRecord(kev[0], s);
        launch();
        if (prof) {
            cudaEventRecord(kev[1], s);
            cudaEventSynchronize(kev[1]);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, kev[0], kev[1]);
            total.kernel_ms[kind] += ms;
            total.kernel_launches[kind] += 1;
        }
    };
    gpop_status status = GPOP_OK;
    uint32_t epoch = 0;
    GPOP_CUDA_TRY(cudaMemsetAsync(p.gflag, 0, 4ull * g->k, s));
    GPOP_CUDA_TRY(cudaMemsetAsync(p.edges, 0, 8, s));
    GPOP_CUDA_TRY(cudaEventRecord(ev0, s));
    for (uint32_t b0 = 0; b0 < num_seeds && status == GPOP_OK; b0 += kSeeds) {
        const uint32_t n = std::min(kSeeds, num_seeds - b0);
        uint32_t hs[kSeeds];
        for (uint32_t j = 0; j < kSeeds; ++j) hs[j] = j < n ? seeds[b0 + j] : kNull;
        cudaError_t ce = cudaMemcpyAsync(d_seed, hs, sizeof hs, cudaMemcpyHostToDevice, s);
        // a pass starts from zero values, messages and frontier
        if (ce == cudaSuccess) ce = cudaMemsetAsync(p.X, 0, 4 * V32, s);
        for (int i = 0; i < 2 && ce == cudaSuccess; ++i) ce = cudaMemsetAsync(msg[i], 0, 4 * V32, s);
        for (int i = 0; i < 3 && ce == cudaSuccess; ++i) ce = cudaMemsetAsync(pa[i], 0, g->k, s);
        if (ce != cudaSuccess) {
            status = fail(GPOP_ERR_CUDA, cudaGetErrorString(ce));
            break;
        }
        p.pact = pa[0]; p.pact_prev = pa[1]; p.pact_next = pa[2];
        p.M = msg[0]; p.Mnext = msg[1];
        k_binit<<<1, kSeeds, 0, s>>>(p);
        uint32_t it = 0;
        unsigned long long hres[kSeeds] = {};
        bool conv = false;
        for (; it < o->max_iters; ++it) {
            p.epoch = ++epoch;
            timed(1, [&] { k_bmark<<<grid_k, kBThreads, 0, s>>>(p); });
            if (grid_p) timed(4, [&] { k_bpull<<<grid_p, kBThreads, 0, s>>>(p); });
            if (grid_x) timed(5, [&] { k_bfix<<<grid_x, kBThreads, 0, s>>>(p); });
            timed(3, [&] { k_bfilter<<<grid_f, kBThreads, 0, s>>>(p); });
            std::swap(p.M, p.Mnext);
            uint8_t *old_prev = p.pact_prev;  // partitions active now become last iteration's
            p.pact_prev = p.pact;
            p.pact = p.pact_next;
            p.pact_next = old_prev;
            // the seeds' L1 changes decide only when there is a tolerance; otherwise the last ones are read
            if (o->tol_l1 <= 0.0 && it + 1 < o->max_iters) continue;
            ce = cudaMemcpyAsync(hres, p.res, sizeof hres, cudaMemcpyDeviceToHost, s);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
            if (ce == cudaSuccess) ce = cudaGetLastError();
            if (ce != cudaSuccess) {
                status = fail(GPOP_ERR_CUDA, std::string("batched PPR: ") + cudaGetErrorString(ce));
                break;
            }
            double mx = 0.0;
            for (uint32_t j = 0; j < n; ++j) mx = std::max(mx, (double)hres[j] * kFixUnit);
            total.residual = mx;
            if (o->tol_l1 > 0.0 && mx < o->tol_l1) {  // every seed's L1 change below the tolerance
                ++it;
                conv = true;
                break;
            }
        }
        if (status != GPOP_OK) break;
        total.iterations += it;
        total.converged &= conv ? 1 : 0;
        float *rows = out_values + (uint64_t)b0 * g->V;
        k_btranspose<<<(g->V + 31) / 32, dim3(32, 8), 0, s>>>(p.X, out_is_device ? rows : staging, g->V, n);
        if (!out_is_device) {
            ce = cudaMemcpyAsync(rows, staging, 4ull * n * g->V, cudaMemcpyDeviceToHost, s);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
            if (ce != cudaSuccess) status = fail(GPOP_ERR_CUDA, cudaGetErrorString(ce));
        }
    }
    cudaEventRecord(ev1, s);
    cudaEventSynchronize(ev1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev0, ev1);
    unsigned long long edges = 0;
    cudaMemcpy(&edges, p.edges, 8, cudaMemcpyDeviceToHost);
    cudaEventDestroy(ev0);
    cudaEventDestroy(ev1);
    cudaEventDestroy(kev[0]);
    cudaEventDestroy(kev[1]);
    if (status != GPOP_OK) return status;
    GPOP_CUDA_TRY(cudaStreamSynchronize(s));
    total.device_ms = ms;
    total.edges_scattered = edges;
    total.pc_partition_steps = 0;
    if (stats) *stats = total;
    return GPOP_OK;
}
