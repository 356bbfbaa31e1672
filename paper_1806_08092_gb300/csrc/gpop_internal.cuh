// Internal declarations of the GB300 GPOP engine (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <utility>
#include <vector>

#include "../../include/gpop.h"

namespace gpop {

// Reserved message value: a partition-centric message from an inactive source
// (and the "no message" state of a vertex).  As FP32 it is a NaN that no
// arithmetic of the applications produces; as uint32 it is above every vertex
// ID, distance and label.
constexpr uint32_t kNull = 0xFFFFFFFFu;
constexpr uint32_t kInf = 0xFFFFFFFFu;
constexpr uint32_t kMsBfsWidth = 32;  // sources per multi-source BFS pass (bits of a 32-bit message)

constexpr int kPngAlign = 8;           // PNG rows padded to 8 entries (16-byte u16 vectors)
constexpr uint32_t kBinAlign = 8;      // every bin padded to 8 slots: its values move as aligned 16-byte vectors (BF16)
constexpr uint32_t kGatherWidth = 4096;  // max destinations per gather task (smem accumulator)
constexpr uint64_t kGatherTaskMinEdges = 65536;  // in-edges a gather task may take before it is cut
constexpr uint32_t kScatterChunk = 131072;  // most PNG slots per PC scatter task (one staging of the partition's values)
constexpr uint32_t kScatterMin = 4096;      // fewest
constexpr uint32_t kScatterUnit = 2048;     // and their unit
constexpr uint32_t kMaxRowBins = 40960;     // SC scatter keeps one cursor per row bin in smem
// messages staged in shared memory per PC gather block: a multiple of kBinAlign, and such that the byte offset of the
// padding value after them (4 kPcBlock) fits the 16-bit index field of a destination entry
constexpr uint32_t kPcBlock = 16376;
constexpr uint32_t kPcTaskBlocks = 20;      // at most this many blocks per PC gather task (static smem per block)
constexpr uint32_t kPcGatherWarps = 19;     // consumer warps of the PC gather, one destination slice of each task each
constexpr uint32_t kPcPadIdx = kPcBlock;    // block index of the padding value
constexpr uint32_t kPcTaskMinEntries = 8192;  // PC gather tasks are not cut below this many entries

// A gather warp's entries of a block (those of its destination slice) are grouped into runs: all entries of one
// destination.  The runs are stored as 16-byte quads, one quad per lane and step, in four classes by length:
//   A  1 entry         4 runs a quad: words (destination << 16 | index)
//   B  2 or 3 entries  2 runs a quad: words (destination << 16 | index), (index << 16 | index)
//   C  4 to 7 entries  1 run a quad:  word (destination << 16 | index) and three words (index << 16 | index)
//   D  8 or more       pieces of up to 7 entries, laid out as C, a run's pieces in consecutive quads
// "destination" is the byte offset of the accumulator word, "index" that of the message in the block (as FP32);
// places left over hold the offset of the padding value (the identity).  Every destination is in one run of a block, so
// only the pieces of a D run meet in one accumulator word.  Runs of equal length side by side let a lane fold its
// run in registers and touch the accumulator once per run, and an entry costs 2 bytes plus its share of the run's
// destination: 2.8 B an entry on R-MAT of scale 22, 3.7 B on a uniform graph of degree 20, against the 4 B
// (destination, index) words of a plain sorted list.
constexpr uint32_t kPcRunA = 1, kPcRunB = 3, kPcRunC = 7;  // longest run of each class

// Position of destination d in the gather's shared accumulator: bits 5-9 XORed into bits 0-4, a bijection
// on every aligned 32-word group that spreads the lanes of one fold step (destinations a near-constant
// stride apart) over distinct banks.  Destination entries carry the swizzled position.
__host__ __device__ constexpr uint32_t pc_swz(uint32_t d) { return d ^ ((d >> 5) & 31u); }

// Small graphs (k_small): the in-edges of a range of destinations as words (destination in the range << kSmallSrcBits |
// source), so at most 2^19 - 1 vertices (one more source is the padding's) and 8192 destinations a range
constexpr uint32_t kSmallSrcBits = 19, kSmallSrc = 1u << kSmallSrcBits, kSmallDest = 1u << (32 - kSmallSrcBits);
// Wall time of a call, one launch / the iteration's kernels, on uniform graphs of 500,000 vertices: 8 M edges ten PageRank
// iterations 520 / 621 us, BFS 283 / 348, SSSP 1135 / 1341; 16 M edges 804 / 795, 409 / 322, 1776 / 1462.  On R-MAT 18 the
// two cross later (14.5 M edges: 556 / 665, 278 / 290, 665 / 599).
constexpr uint64_t kSmallEdges = 8u << 20;

enum Mode : uint8_t { kModeNone = 0, kModeSC = 1, kModePC = 2 };
enum Action : uint8_t { kActSkip = 0, kActPC = 1, kActNull = 2 };

// Per-iteration control block written by the plan kernel and read by the host.
struct Control {
    unsigned long long frontier_v;   // sum of V_a entering the iteration
    unsigned long long frontier_e;   // sum of E_a
    double residual;                 // L1 change of the previous iteration (PR/PPR)
    double model_bytes;              // Sec. 3.2 bytes of this iteration's chosen modes
    uint32_t n_pc, n_sc, n_null;     // partitions per action
    uint32_t done;                   // 1 = stop before scattering this iteration
    uint32_t n_fallback;             // learned mode: partitions that fell back to Eq. (mode)
    uint32_t error;                  // device check flags
    uint32_t n_sc_units;             // SC scatter work units (split hub partitions count several)
    uint32_t seq;                    // the plan's epoch, written last (the host waits for it)
    unsigned long long sc_v, sc_e;   // V_a and E_a of the partitions scattered in SC mode
    unsigned long long gathered;     // destinations the run's task gathers visited so far
    uint32_t go, pad;                // 1 = PC scatter and gather are all this iteration needs (see Params::spec)
};

// Static gather task: destinations [d0, d1) (local IDs) of column q, which have `entries` in-edges.
struct GatherTask {
    uint32_t q, d0, d1, entries;
};

// Static PC scatter task: PNG slots [beg, end) of partition p (padded row layout).
struct ScatterTask {
    uint32_t p, beg, end, first;  // first = 1 for the chunk that starts the row
};

struct Graph {
    uint32_t V = 0, P = 0, shift = 0, k = 0;
    uint64_t E = 0;
    int weighted = 0;
    uint64_t nb = 0, npng = 0, npng_pad = 0;
    uint32_t max_row_bins = 0;

    // CSR with rows sorted by destination
    uint32_t *rowptr = nullptr;   // V+1
    uint32_t *col = nullptr;      // E
    int32_t *w = nullptr;         // E or null
    uint16_t *esub = nullptr;     // E: index of the edge's SC bin within its bin row

    // bins bin[p][q] (non-empty), row-major
    uint32_t *row_bin = nullptr;  // k+1
    uint32_t *bin_q = nullptr;    // nb

    // PNG (Alg. 3) and PC data bins, padded rows
    uint16_t *png = nullptr;      // npng_pad: local source ID per message slot
    uint32_t *pdata = nullptr;    // npng_pad: message values, column by column (a column's bins in ascending source
                                  // partition, each padded to kBinAlign)
    uint32_t *png_dst = nullptr;  // npng_pad / 8: where the values of each group of 8 PNG slots go (slot / 8)

    // PC gather blocks: each column's message sequence (bins (p, q), p ascending) cut into blocks of
    // kPcBlock messages, each a contiguous piece of pdata; destination lists as quads (kPcRunA)
    uint32_t *pc_blk_src = nullptr;  // npcb: first value slot of each block
    uint32_t *pc_blk_nval = nullptr; // npcb: staged values of each block (a multiple of kBinAlign)
    uint2 *pc_blk_prange = nullptr;  // npcb: first and last source partition of each block's bins
    uint4 *pc_task = nullptr;     // npct: (column, first block, end block, partial slot or kNull), largest first
    uint32_t *pc_tsp = nullptr;   // npct: first of the task's blocks in pc_rng
    uint4 *pc_rng = nullptr;      // per task block and gather warp, the entries of the warp's destination slice
                                  // (the same slice in every block of the task): (first quad, quads of class A |
                                  // quads of class B << 16, quads of class C, 0); the quads end where the
                                  // next range's start
    uint32_t *col_ntask = nullptr;   // k: PC gather tasks of the column (0 = no PC in-edges)
    uint32_t *col_part0 = nullptr;   // k: first partial slot of a multi-task column
    uint32_t *pc_part = nullptr;  // npart x P partial results
    uint2 *pc_merge = nullptr;    // nmerge: (column, first destination) of each 1024-destination chunk of a
                                  // column split over several tasks (its partials are merged into pc_sum)
    uint32_t nmerge = 0;
    uint4 *pe = nullptr;          // destination entries of every range as quads, class by class
    uint4 *pw = nullptr;          // null or their weights.  w16 (no weight above 65535): one quad for each quad, the
                                  // weight of each index in the same field; else two quads for each quad, 32-bit
                                  // weights of its first four places (class B: the first run's three), of the rest
    uint32_t w16 = 0;
    uint32_t npcb = 0, npct = 0, npart = 0;

    // SC bins, one per (source partition p, gather task t) with edges p -> t
    uint2 *scpair = nullptr;      // E: (local destination, value), regions of capacity edges(p, t)
    uint32_t *sccnt = nullptr;    // nsub: pairs written this iteration
    uint32_t *sub_cap = nullptr;  // nsub+1: region offsets
    uint32_t *sub_task = nullptr; // nsub: gather task of the bin
    uint32_t *row_sub = nullptr;  // k+1: bins of each source partition
    uint32_t *task_sub_ptr = nullptr;  // ngt+1: capacity of each task's fresh-bin list
    uint32_t nsub = 0, max_row_subs = 0;

    // per partition statics
    uint32_t *Ep = nullptr, *npng_p = nullptr;  // device, k each
    uint64_t *h_Ep = nullptr, *h_npng = nullptr;                      // host copies

    // small graphs: the whole run in one launch (k_small)
    uint32_t sm_n = 0, sm_wide = 0;  // ranges (0: not a small graph), most destinations of one
    uint4 *sm_range = nullptr;    // (first destination, destinations, first quad, quads)
    uint4 *sm_edge = nullptr, *sm_w = nullptr;  // the ranges' in-edges by destination, padded to whole quads; weights

    // batched PPR (made by its first call): in-edges by destination, sources ascending, in shares of in_share edges
    uint32_t *in_off = nullptr;    // V + 1 offsets
    uint2 *in_edge = nullptr;      // E: (source, destination)
    uint4 *in_span = nullptr;      // destinations cut by shares: (destination, first share, shares, 0)
    uint32_t in_share = 0, n_share = 0, n_span = 0;

    // tasks
    uint32_t ngt = 0, nst = 0, st_threads = 512;  // st_threads: threads of a PC scatter task's CTA
    GatherTask *gtask = nullptr;  // ngt
    uint32_t *col_task = nullptr; // k+1
    ScatterTask *stask = nullptr; // nst

    // persistent run state (allocated lazily, reused across runs)
    uint8_t *pc_state = nullptr;  // k: row of pdata holds non-NULL values
    uint32_t epoch = 0;           // iteration stamp, never reused within the handle
    bool pdata_dirty = false;
    bool pdata_set = false;  // rows may hold values of a run by the iteration's kernels
    int pdata_fmt = 0;  // message format of the data rows: 0 FP32/u32, 1 BF16

    uint64_t device_bytes = 0;
    uint64_t fingerprint = 0;     // of the edge multiset with weights, V and E (checkpoints name their graph)
    std::vector<uint32_t> goff;   // graphs built as one disjoint union: first vertex of each (+ V at the end)
    int device = 0, num_sms = 0;
    void *run = nullptr;          // cached per-run buffers (engine.cu)
};

// error reporting (thread-local last error)
void set_error(const std::string &msg);
gpop_status fail(gpop_status st, const std::string &msg);

#define GPOP_CUDA_TRY(expr)                                                                       \
    do {                                                                                          \
        cudaError_t _e = (expr);                                                                  \
        if (_e != cudaSuccess)                                                                    \
            return ::gpop::fail(GPOP_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(_e)); \
    } while (0)

// device allocation helper tracked in Graph::device_bytes
template <typename T>
cudaError_t dalloc(Graph *g, T **p, uint64_t count) {
    if (count == 0) count = 1;
    cudaError_t e = cudaMalloc((void **)p, sizeof(T) * count);
    if (e == cudaSuccess) g->device_bytes += sizeof(T) * count;
    return e;
}

// Device arrays that are needed together: once one cannot be had, the others are given back, null and no longer counted
struct ArrayGroup {
    Graph *g;
    cudaError_t error = cudaSuccess;
    std::vector<std::pair<void **, uint64_t>> had;  // the arrays so far, with their bytes
    explicit ArrayGroup(Graph *graph) : g(graph) {}
    template <typename T>
    void add(T **p, uint64_t count) {
        if (error != cudaSuccess) return;
        const uint64_t before = g->device_bytes;
        error = dalloc(g, p, count);
        if (error == cudaSuccess) had.emplace_back(reinterpret_cast<void **>(p), g->device_bytes - before);
        else *p = nullptr;
    }
    void give_back() {
        for (auto &a : had) {
            cudaFree(*a.first);
            *a.first = nullptr;
            g->device_bytes -= a.second;
        }
        had.clear();
    }
};

void free_graph(Graph *g);
gpop_status make_in_edges(Graph *g, cudaStream_t s);  // build.cu: Graph::in_off and the rest
void release_run_state(Graph *g);   // engine.cu
const float *selector_device_params();             // selector.cu: installed MLP parameters or null
const float *selector_device_params_transposed();  // the same with W1, W2 transposed (inference layout)

}  // namespace gpop

struct gpop_graph {
    gpop::Graph g;
};
