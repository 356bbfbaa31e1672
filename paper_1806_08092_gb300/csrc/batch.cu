// Batched seeded personalized PageRank (gpop_run_ppr_batch): up to 32 seeds per pass through the
// partition-centric gather of Alg. 2 on the PC layout of Alg. 3, every message carrying one FP32 value per
// seed (lane j of a warp holds seed j).
//
// A message is 128 bytes against the 4 of its index, and its value is the same for every destination partition:
// it is read where its source keeps it instead of being copied into a bin per partition.  The hub sources'
// messages, which most entries name, then stay in L2.  One pass = per iteration:
//   k_bmark     the columns that partitions with an active vertex (for any seed: the union frontier) send to;
//   k_bgather   one CTA per PC gather task (a range of one column's blocks): the sources of a block's messages are
//               staged in shared memory, and each warp folds the entries of its destination slice (the same slice
//               in every block of the task) into the column accumulator acc[P][32], lane j adding seed j's values:
//               128-byte loads, no bank conflicts, no atomics, a fixed order.  A column of one task is filtered
//               right there: x_j = alpha [v = s_j] + (1 - alpha) acc_j, the next messages, the active flag and
//               each seed's L1 change;
//   k_bfilter   the same for columns split over several tasks, whose partial vectors it sums in task order, and
//               for columns that lost or did not receive messages.
// L1 changes are added as 62-bit fixed point, exact in any order.
// Measured on R-MAT 20 (P = 1024, 48 seeds in two passes of 40 iterations): 82.6 ms a call, against 195 ms with a
// bin slot per (source, destination partition) written and read back and separate merge and filter passes.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "gpop_internal.cuh"

namespace gpop {
namespace {

constexpr uint32_t kSeeds = 32;                  // seeds per pass, one lane each
constexpr uint32_t kBatchMaxP = 1024;            // acc[P][32] floats must fit in shared memory
constexpr int kBThreads = 256;
constexpr int kBWarps = kBThreads / 32;
constexpr uint32_t kBRows = 8 * kBWarps;         // vertices per CTA of the filter, 8 a warp
constexpr int kBGWarps = kPcGatherWarps;         // gather warps: one destination slice of each task each
constexpr int kBGThreads = 32 * kBGWarps;
constexpr double kFixOne = 0x1p62, kFixUnit = 0x1p-62;  // fixed point of the L1 change (at most 2)

struct BParams {
    uint32_t V, P, shift, k, npct;
    const uint32_t *rowptr, *Ep;
    const uint16_t *png;
    const uint32_t *row_png, *row_bin, *bin_q;
    const uint4 *pc_task, *pc_rng, *pe;
    const uint32_t *png_dst, *pc_tsp, *pc_blk_src, *pc_blk_nval, *col_ntask, *col_part0;
    const uint32_t *seed;     // [32]: the pass's seeds, kNull for unused lanes
    uint32_t *src;            // source vertex of every (column-major) message slot
    float *X, *M, *Mnext;     // V x 32 each: values, this iteration's messages, the next one's
    float *part;              // partial vectors of split columns (npart x P x 32)
    uint8_t *pact, *pact_prev, *pact_next;  // partitions with an active vertex: now, last iteration, next
    uint32_t *gflag;          // column received messages this iteration (== epoch)
    uint32_t *counter;        // gather task counter
    unsigned long long *edges;  // out-edges of the scattered partitions, summed over iterations
    unsigned long long *res;  // per seed: L1 change of the iteration (fixed point)
    float c0, c1;             // alpha, 1 - alpha
    uint32_t epoch;
};

// source vertex of every message slot in the gather's column-major order (once per call: 4 bytes a slot)
__global__ void __launch_bounds__(kBThreads) k_bsources(BParams p) {
    for (uint32_t q = blockIdx.x; q < p.k; q += gridDim.x) {
        const uint32_t g0 = q << p.shift;
        for (uint32_t i = p.row_png[q] + threadIdx.x; i < p.row_png[q + 1]; i += kBThreads)
            p.src[p.png_dst[i / kBinAlign] * kBinAlign + i % kBinAlign] = g0 + p.png[i];
    }
}

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
    if (blockIdx.x == 0) {
        if (threadIdx.x < kSeeds) p.res[threadIdx.x] = 0ull;
        if (threadIdx.x == kSeeds) *p.counter = 0u;
    }
    for (uint32_t q = blockIdx.x; q < p.k; q += gridDim.x) {
        if (threadIdx.x == 0) p.pact_next[q] = 0;
        if (!p.pact[q]) continue;
        for (uint32_t b = p.row_bin[q] + threadIdx.x; b < p.row_bin[q + 1]; b += kBThreads)
            p.gflag[p.bin_q[b]] = p.epoch;
        if (threadIdx.x == 0) atomicAdd(p.edges, (unsigned long long)p.Ep[q]);
    }
}

// PPR's filterFunc of eight consecutive vertices v0 .. by one warp, lane j for seed j, from their combined messages:
// values, next messages, the partition's active flag; returns the lane's L1 change
__device__ __forceinline__ float bfilter8(const BParams &p, uint32_t v0, const float (&acc)[8], uint32_t seed, int lane) {
    const uint32_t n = min(8u, p.V - v0);
    const uint32_t rp = p.rowptr[v0 + min((uint32_t)lane, n)];  // row offsets, one per lane
    float xo[8], res = 0.f;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) xo[k] = k < n ? p.X[(uint64_t)(v0 + k) * kSeeds + lane] : 0.f;
    bool any = false;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
        const uint32_t deg = __shfl_sync(0xffffffffu, rp, (int)k + 1) - __shfl_sync(0xffffffffu, rp, (int)k);
        if (k >= n) continue;
        const uint64_t o = (uint64_t)(v0 + k) * kSeeds + lane;
        const float xn = fmaf(p.c1, acc[k], v0 + k == seed ? p.c0 : 0.f);
        p.X[o] = xn;
        p.Mnext[o] = deg ? xn / (float)deg : 0.f;
        res += fabsf(xn - xo[k]);
        any |= xn > 0.f;
    }
    if (__any_sync(0xffffffffu, any) && lane == 0) p.pact_next[v0 >> p.shift] = 1;
    return res;
}

// PC gather: one CTA per task (1 per SM, persistent), acc[P][32] and the sources of a block's messages in shared
// memory.  Bound by the 128-byte messages it reads through L2: one per entry, fourteen loads in flight per warp.
__global__ void __launch_bounds__(kBGThreads, 1) k_bgather(BParams p) {
    extern __shared__ __align__(16) float s_acc[];                                 // P x 32 (swizzled destinations)
    uint32_t *s_src = reinterpret_cast<uint32_t *>(s_acc + (size_t)p.P * kSeeds);  // kPcBlock sources
    __shared__ uint32_t s_task;
    __shared__ unsigned long long s_res[kSeeds];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t seed = p.seed[lane];
    unsigned long long res = 0;  // the lane's L1 change in the columns this CTA filters
    if (threadIdx.x < kSeeds) s_res[threadIdx.x] = 0ull;
    for (;;) {
        if (threadIdx.x == 0) s_task = atomicAdd(p.counter, 1u);
        __syncthreads();
        const uint32_t t = s_task;
        __syncthreads();
        if (t >= p.npct) break;
        const uint4 tk = p.pc_task[t];  // column, first block, end block, partial slot
        if (p.gflag[tk.x] != p.epoch) continue;
        for (uint32_t i = threadIdx.x; i < p.P * kSeeds; i += kBGThreads) s_acc[i] = 0.f;
        const uint32_t tsp = p.pc_tsp[t];
        for (uint32_t b = tk.y; b < tk.z; ++b) {
            const uint32_t *bs = p.src + p.pc_blk_src[b];  // 32-byte aligned, a multiple of 8 sources
            const uint32_t nv = p.pc_blk_nval[b];
            __syncthreads();  // the accumulator is cleared and the previous block's sources are no longer read
            for (uint32_t i = threadIdx.x; i < nv / 4; i += kBGThreads)
                reinterpret_cast<uint4 *>(s_src)[i] = reinterpret_cast<const uint4 *>(bs)[i];
            __syncthreads();
            // the warp's entries (it alone owns their destinations), quad by quad (layout at kPcRunA): lane j adds
            // seed j's values of a run in registers and the run's sum to the accumulator, a fixed order
            const uint4 *rg = p.pc_rng + (uint64_t)(tsp + (b - tk.y)) * kPcGatherWarps + wid;
            const uint4 g = rg[0];
            const uint32_t n = rg[1].x - g.x, nA = g.y & 0xFFFFu, nAB = nA + (g.y >> 16);
            uint32_t cur_d = 0xFFFFFFFFu;  // class C and D: the run being summed (byte offset of its word)
            float cur = 0.f, lost = 0.f;   // its sum over the pieces, compensated (Kahan): a run can have thousands
            uint4 q_next = (uint32_t)lane < n ? p.pe[g.x + lane] : make_uint4(0, 0, 0, 0);
            for (uint32_t r0 = 0; r0 < n; r0 += 32) {
                const uint4 q = q_next;
                if (r0 + 32 < n) q_next = (uint32_t)lane < n - r0 - 32 ? p.pe[g.x + r0 + 32 + lane] : make_uint4(0, 0, 0, 0);
                const uint32_t m = min(32u, n - r0);
                for (uint32_t t0 = 0; t0 < m; t0 += 2) {
                    float v[2][7];
                    uint4 e[2];
#pragma unroll
                    for (uint32_t u = 0; u < 2; ++u) {
                        const int t = (int)min(t0 + u, m - 1);
                        e[u].x = __shfl_sync(0xffffffffu, q.x, t);
                        e[u].y = __shfl_sync(0xffffffffu, q.y, t);
                        e[u].z = __shfl_sync(0xffffffffu, q.z, t);
                        e[u].w = __shfl_sync(0xffffffffu, q.w, t);
                        const bool a = r0 + t < nA, ab = r0 + t < nAB;  // the fields that are indices, by class
                        constexpr uint32_t kPad = 4u * kPcPadIdx;
                        const uint32_t x[7] = {e[u].x & 0xFFFFu, e[u].y & 0xFFFFu, a ? kPad : e[u].y >> 16,
                                               e[u].z & 0xFFFFu, ab ? kPad : e[u].z >> 16, e[u].w & 0xFFFFu,
                                               a ? kPad : e[u].w >> 16};
#pragma unroll
                        for (uint32_t k = 0; k < 7; ++k)
                            v[u][k] = x[k] < kPad ? p.M[(uint64_t)s_src[x[k] / 4] * kSeeds + lane] : 0.f;
                    }
#pragma unroll
                    for (uint32_t u = 0; u < 2; ++u) {
                        if (t0 + u >= m) break;
                        const uint32_t i = r0 + t0 + u;
                        auto add = [&](uint32_t word, float s) { s_acc[(word >> 16) * (kSeeds / 4) + lane] += s; };
                        if (i < nA) {
                            add(e[u].x, v[u][0]);
                            add(e[u].y, v[u][1]);
                            add(e[u].z, v[u][3]);
                            add(e[u].w, v[u][5]);
                        } else if (i < nAB) {
                            add(e[u].x, v[u][0] + v[u][1] + v[u][2]);
                            add(e[u].z, v[u][3] + v[u][5] + v[u][6]);
                        } else {
                            if ((e[u].x >> 16) != cur_d) {
                                if (cur_d != 0xFFFFFFFFu) add(cur_d << 16, cur);
                                cur_d = e[u].x >> 16;
                                cur = lost = 0.f;
                            }
                            const float y = ((v[u][0] + v[u][1]) + (v[u][2] + v[u][3])) + ((v[u][4] + v[u][5]) + v[u][6]) - lost;
                            const float t = cur + y;
                            lost = (t - cur) - y;
                            cur = t;
                        }
                    }
                }
            }
            if (cur_d != 0xFFFFFFFFu) s_acc[cur_d * (kSeeds / 4) + lane] += cur;
        }
        __syncthreads();
        const uint32_t gq = tk.x << p.shift, wq = min(p.P, p.V - gq);
        if (tk.w == kNull) {  // the column's only task: filter it
            double dres = 0.0;
            for (uint32_t d = (uint32_t)wid * 8; d < wq; d += kBGWarps * 8) {
                float acc[8];
#pragma unroll
                for (uint32_t k = 0; k < 8; ++k) acc[k] = d + k < wq ? s_acc[pc_swz(d + k) * kSeeds + lane] : 0.f;
                dres += (double)bfilter8(p, gq + d, acc, seed, lane);
            }
            res += __double2ull_rn(dres * kFixOne);
        } else {
            float *out = p.part + (uint64_t)tk.w * p.P * kSeeds;
            for (uint32_t i = threadIdx.x; i < wq * kSeeds; i += kBGThreads)
                out[i] = s_acc[pc_swz(i / kSeeds) * kSeeds + (i % kSeeds)];
        }
        __syncthreads();
    }
    if (res) atomicAdd(&s_res[lane], res);
    __syncthreads();
    if (wid == 0 && s_res[lane]) atomicAdd(&p.res[lane], s_res[lane]);
}

// columns the gather did not filter: those split over several tasks (their partial vectors, summed in task order)
// and those without messages that are or were active (a skipped column's values and both its message buffers are
// zero); 8 vertices a warp, kBRows a CTA
__global__ void __launch_bounds__(kBThreads) k_bfilter(BParams p) {
    __shared__ unsigned long long s_res[kSeeds];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t seed = p.seed[lane], per = (p.P + kBRows - 1) / kBRows;
    unsigned long long res = 0;
    if (threadIdx.x < kSeeds) s_res[threadIdx.x] = 0ull;
    __syncthreads();
    for (uint64_t it = blockIdx.x; it < (uint64_t)p.k * per; it += gridDim.x) {
        const uint32_t q = (uint32_t)(it / per), d = (uint32_t)(it % per) * kBRows + (uint32_t)wid * 8;
        const uint32_t nt = p.col_ntask[q], gq = q << p.shift, wq = min(p.P, p.V - gq);
        const bool got = p.gflag[q] == p.epoch && nt > 0;
        if (got ? nt == 1 : !(p.pact[q] | p.pact_prev[q])) continue;
        if (d >= wq) continue;
        float acc[8] = {};
        if (got) {
            const float *src = p.part + ((uint64_t)p.col_part0[q] * p.P + d) * kSeeds + lane;
            for (uint32_t t0 = 0; t0 < nt; t0 += 4) {  // 32 loads in flight
                float v[4][8];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u)
#pragma unroll
                    for (uint32_t k = 0; k < 8; ++k)
                        v[u][k] = (t0 + u < nt && d + k < wq) ? src[((uint64_t)(t0 + u) * p.P + k) * kSeeds] : 0.f;
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u)
#pragma unroll
                    for (uint32_t k = 0; k < 8; ++k) acc[k] += v[u][k];
            }
        }
        res += __double2ull_rn((double)bfilter8(p, gq + d, acc, seed, lane) * kFixOne);
    }
    if (res) atomicAdd(&s_res[lane], res);
    __syncthreads();
    if (wid == 0 && s_res[lane]) atomicAdd(&p.res[lane], s_res[lane]);
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
        return fail(GPOP_ERR_INVALID_ARG, "batched PPR keeps 32 values per destination in shared memory: partition "
                                          "size must be at most 1024");
    gpop_run_stats total;
    memset(&total, 0, sizeof total);
    total.converged = 1;
    if (num_seeds == 0) {
        if (stats) *stats = total;
        return GPOP_OK;
    }
    cudaStream_t s = (cudaStream_t)o->cuda_stream;
    const size_t gsmem = sizeof(float) * (size_t)g->P * kSeeds + sizeof(uint32_t) * kPcBlock;
    {
        int optin = 0, dev = 0;
        GPOP_CUDA_TRY(cudaGetDevice(&dev));
        GPOP_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        cudaFuncAttributes fa;
        GPOP_CUDA_TRY(cudaFuncGetAttributes(&fa, k_bgather));
        if (gsmem + fa.sharedSizeBytes > (size_t)optin) return fail(GPOP_ERR_INVALID_ARG, "batched PPR: shared memory too small");
        GPOP_CUDA_TRY(cudaFuncSetAttribute(k_bgather, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsmem));
    }
    BatchBuffers bb;
    BParams p{};
    p.V = g->V; p.P = g->P; p.shift = g->shift; p.k = g->k; p.npct = g->npct;
    p.rowptr = g->rowptr; p.Ep = g->Ep; p.png = g->png; p.row_png = g->row_png; p.row_bin = g->row_bin;
    p.bin_q = g->bin_q; p.png_dst = g->png_dst; p.pc_task = g->pc_task; p.pc_tsp = g->pc_tsp; p.pc_rng = g->pc_rng;
    p.pc_blk_src = g->pc_blk_src; p.pc_blk_nval = g->pc_blk_nval; p.pe = g->pe; p.col_ntask = g->col_ntask;
    p.col_part0 = g->col_part0;
    p.c0 = (float)(1.0 - o->damping);
    p.c1 = (float)o->damping;
    const uint64_t V32 = (uint64_t)g->V * kSeeds;
    const int grid_f = (int)std::min<uint64_t>((uint64_t)g->k * ((g->P + kBRows - 1) / kBRows), 8u * (uint32_t)g->num_sms);
    const uint32_t grid_k = std::min<uint32_t>(g->k, 8u * g->num_sms);
    uint32_t *d_seed = nullptr;
    uint8_t *pa[3] = {};
    float *staging = nullptr, *msg[2] = {};
    cudaError_t e = cudaSuccess;
    auto A = [&](auto **ptr, uint64_t n) {
        if (e == cudaSuccess) e = bb.alloc(ptr, n);
    };
    A(&p.X, V32); A(&msg[0], V32); A(&msg[1], V32);
    A(&p.src, g->npng_pad);
    A(&p.part, (uint64_t)g->npart * g->P * kSeeds);
    A(&pa[0], g->k); A(&pa[1], g->k); A(&pa[2], g->k);
    A(&p.gflag, g->k);
    A(&p.counter, 1);
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
    k_bsources<<<grid_k, kBThreads, 0, s>>>(p);
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
            timed(4, [&] { k_bgather<<<g->num_sms, kBGThreads, gsmem, s>>>(p); });
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
