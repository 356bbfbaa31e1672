// A small graph's whole run in one launch (part of engine.cu).
//
// An iteration of a graph whose edges and values stay in L2 costs the engine's kernels 40 to 60 us of launches, plans
// and host round trips for a few microseconds of work.  k_small runs all iterations in one cooperative launch instead:
// every CTA owns the in-edges of a range of consecutive destinations (sorted by destination, at most kSmallDest of
// them, cut so that the CTAs have about equal work) and reads the message of an edge at its source, out of a buffer
// that stays in L2 for the whole iteration; it combines the messages in shared memory, applies the user functions to
// its own destinations and writes their next messages to the other buffer.  One grid barrier ends an iteration.  One
// more CTA keeps the run's statistics (Eq. (mode) per partition) a phase behind the others.
//  * A warp takes an equal share of its CTA's edges, 4 per lane and step: the lane's inner runs go straight to the
//    accumulator, the open runs through a segmented warp scan, as in pc_fold.  A run that began in the share of an
//    earlier warp goes to a word of the warp's own, added after the barrier in warp order.  No atomics, a fixed order.
//  * Sums are pairs of FP32 words (SmallSum) that lose nothing beyond the messages' own rounding, so that a value is rounded
//    once, as after the SC scatter's fixed point, and a hub's in-degree costs no accuracy; NULL messages count as the
//    identity.
// Bound by the latency of a step (edges, then messages out of L2) and of the barrier.  Wall time of a call, iteration
// kernels -> one launch: ten PageRank iterations on R-MAT 12 256 -> 95 us, R-MAT 16 329 -> 123 us, R-MAT 18 with 7.6 M
// edges 580 -> 381 us; BFS 171 -> 47, 214 -> 57, 281 -> 167 us; SSSP on a uniform graph of 500,000 vertices and 8 M edges
// 1341 -> 1135 us.
constexpr int kSmallThreads = 512;
constexpr uint32_t kSmallWarps = kSmallThreads / 32;

// What the run leaves for the host (mapped memory)
struct SmallReport {
    uint32_t iterations, error;
    double residual, model_bytes;
    unsigned long long frontier_v, edges, vertices, pc, sc, sc_v, sc_e;
};

struct SmallParams {
    const uint4 *edge, *w;    // words (destination in the range << kSmallSrcBits | source), padded to whole quads; weights
    const uint4 *range;       // per CTA: first destination, destinations, first quad, quads
    uint32_t n;               // ranges
    uint32_t *sval[2];        // messages of this iteration and the next (V + 1 words, the last NULL)
    unsigned long long *cnt;  // small_counters(k) words, zero at launch
    SmallReport *report;
    uint32_t *out, *out_parent;  // device results, or null
    uint32_t resume, base;
};

// Counters: the abort flag, then three slots in turn (small_barrier.h), each for one iteration's frontier: the word of the
// barrier before the iteration (with the graph's V_a), E_a and L1 change of the graph, V_a and E_a of its partitions
constexpr uint32_t kSmallHead = 1;
__host__ __device__ constexpr uint64_t small_slot(uint32_t k) { return 3 + 2ull * k; }
__host__ __device__ constexpr uint64_t small_counters(uint32_t k) { return kSmallHead + kSmallSlots * small_slot(k); }

// Arrival of one CTA, with `active` vertices, at the grid barrier of a round (its word) and the wait for the others, by one
// thread after a barrier of its CTA.  *frontier: the vertices active after the round.  False when the wait ran out (2 s) or
// another CTA's did.
__device__ __forceinline__ bool small_arrive_wait(unsigned long long *word, unsigned long long *abort, uint32_t active,
                                                  uint32_t *frontier) {
    __threadfence();
    unsigned long long w = atomicAdd(word, small_arrival(active)) + small_arrival(active);
    bool go = true;
    const unsigned long long t0 = globaltimer();
    for (uint32_t it = 0; !small_all_arrived(w, gridDim.x); ++it) {
        if ((it & 63u) == 63u && (*(volatile unsigned long long *)abort || globaltimer() - t0 > kPcWaitNs)) {
            atomicExch(abort, 1ull);
            go = false;
            break;
        }
        w = *(volatile unsigned long long *)word;
    }
    __threadfence();
    *frontier = small_active(w);
    return go;
}

// What a CTA keeps of the messages of a destination: a word of the monoid, or for the sums an FP32 sum and what its
// roundings have lost (their sum is the value: a relative error of at most 2^-48 per addition).  Fixed point, as in the
// task gather's SC pass, would cost small values their last digits: most messages of a small graph's run are in partitions
// that the iteration's kernels scatter in PC mode and sum in FP32.  Against plain FP32 sums: ten PageRank iterations on
// R-MAT 16 141 -> 148 us.
struct SmallSum {
    float sum, lost;
};
template <int ALGO>
struct SmallAcc {
    static constexpr bool kSum = sums(ALGO);
    using T = typename std::conditional<kSum, SmallSum, uint32_t>::type;
    static __device__ __forceinline__ T of(uint32_t m) {
        if constexpr (kSum) return SmallSum{u2f(m), 0.f};
        else return m;
    }
    static __device__ __forceinline__ T identity() { return of(Op<ALGO>::identity()); }
    static __device__ __forceinline__ T combine(T a, T b) {
        if constexpr (kSum) {  // Knuth's exact addition of two numbers: s and its error
            const float s = a.sum + b.sum, t = s - a.sum, e = (a.sum - (s - t)) + (b.sum - t);
            return SmallSum{s, (a.lost + b.lost) + e};
        } else {
            return Op<ALGO>::combine(a, b);
        }
    }
    static __device__ __forceinline__ T shfl_up(T a, uint32_t o) {
        if constexpr (kSum) return SmallSum{__shfl_up_sync(0xffffffffu, a.sum, o), __shfl_up_sync(0xffffffffu, a.lost, o)};
        else return __shfl_up_sync(0xffffffffu, a, o);
    }
    static __device__ __forceinline__ uint32_t message(T a) {
        if constexpr (kSum) return f2u(a.sum + a.lost);
        else return a;
    }
};

// Statistics of the iteration that the counters in slot cur describe, as k_plan takes them; the slot of the iteration after
// the next is cleared.  Thread 0 keeps the run's totals in rep.
template <int ALGO>
__device__ void small_statistics(const Params &p, const SmallParams &sp, const unsigned long long *cur,
                                 unsigned long long *clear, SmallReport &rep) {
    __shared__ unsigned long long s_sum[7][kSmallWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x[7] = {0, 0, 0, 0, 0, 0, 0};  // n_pc, n_sc, bytes, two fractions, V_a and E_a in SC mode
    for (uint32_t q = threadIdx.x; q < p.k; q += kSmallThreads) {
        const uint64_t Va = __ldcg(cur + 3 + 2 * (uint64_t)q), Ea = __ldcg(cur + 4 + 2 * (uint64_t)q);
        const uint32_t Ep = p.Ep[q], np = p.npng_p[q];
        const uint8_t m = analytic_mode(p.k, Ep, np, Va, Ea, p.bw_num, p.bw_den);
        if (m == kModePC) {
            x[0]++;
            x[2] += pc_mode_bytes(p.k, Ep, np);
        } else if (m == kModeSC) {
            unsigned long long d1, d2;
            x[1]++;
            x[2] += sc_mode_bytes(Ep, np, Va, Ea, &d1, &d2);
            x[3] += d1;
            x[4] += d2;
            x[5] += Va;
            x[6] += Ea;
        }
        p.pc_state[q] = m == kModePC;  // as the iteration's kernels would leave it (the rows themselves are NULL)
    }
    for (uint64_t i = threadIdx.x; i < small_slot(p.k); i += kSmallThreads) clear[i] = 0ull;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const unsigned long long y = warp_sum_u64(x[i]);
        if (lane == 0) s_sum[i][wid] = y;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t[7];
        for (int i = 0; i < 7; ++i) {
            t[i] = 0;
            for (uint32_t w = 0; w < kSmallWarps; ++w) t[i] += s_sum[i][w];
        }
        rep.vertices += small_active(__ldcg(cur));
        rep.edges += __ldcg(cur + 1);
        rep.pc += t[0];
        rep.sc += t[1];
        rep.model_bytes += (double)t[2] + (double)t[3] * 0x1p-29 + (double)t[4] * 0x1p-61;
        rep.sc_v += t[5];
        rep.sc_e += t[6];
    }
    __syncthreads();
}

template <int ALGO, bool B16>
__global__ void __launch_bounds__(kSmallThreads, 2) k_small(Params p, SmallParams sp) {
    using O = Op<ALGO>;
    using A = SmallAcc<ALGO>;
    using T = typename A::T;
    extern __shared__ __align__(8) unsigned char s_small_dyn[];
    T *const s_acc = reinterpret_cast<T *>(s_small_dyn);  // the range's destinations
    __shared__ T s_carry[kSmallWarps];
    __shared__ uint32_t s_cd[kSmallWarps];
    __shared__ unsigned long long s_va, s_ea;
    __shared__ double s_res[kSmallWarps];
    __shared__ uint32_t s_go, s_frontier;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool keeper = blockIdx.x == sp.n;  // the CTA that keeps the statistics
    const uint4 rg = keeper ? make_uint4(0, 0, 0, 0) : sp.range[blockIdx.x];
    const uint32_t d0 = rg.x, nd = rg.y;
    // this warp's share of the range's quads, and the destination it shares with an earlier warp (kSent: none)
    // (the warps without one come last, so that warps that share a destination are neighbours)
    const uint32_t per = (rg.w + kSmallWarps - 1) / kSmallWarps, q0 = min(rg.w, per * (uint32_t)wid), q1 = min(rg.w, q0 + per);
    uint32_t cfd = kSent;
    if (q0 > 0 && q0 < q1) {
        const uint32_t a = sp.edge[rg.z + q0 - 1].w >> kSmallSrcBits, b = sp.edge[rg.z + q0].x >> kSmallSrcBits;
        if (a == b) cfd = a;
    }
    if (lane == 0) s_cd[wid] = cfd;
    const uint64_t slot = small_slot(p.k);
    unsigned long long *const slots = sp.cnt + kSmallHead;
    __shared__ SmallReport rep;  // the keeper's, by its thread 0
    if (threadIdx.x == 0) rep = SmallReport{};

    // a warp's statistics of 32 consecutive destinations (one partition) into the slot of the next iteration; the
    // graph's totals go through shared memory
    auto count = [&](unsigned long long *to, uint32_t g, bool act, uint32_t deg) {
        const uint32_t word = __ballot_sync(0xffffffffu, act);
        if (word) {
            const uint32_t va = __popc(word), ea = __reduce_add_sync(0xffffffffu, act ? deg : 0u);
            if (lane == 0) {
                const uint32_t q = g >> p.shift;
                atomicAdd(to + 3 + 2 * (uint64_t)q, (unsigned long long)va);
                atomicAdd(to + 4 + 2 * (uint64_t)q, (unsigned long long)ea);
                atomicAdd(&s_va, (unsigned long long)va);
                atomicAdd(&s_ea, (unsigned long long)ea);
            }
        }
    };
    // the CTA's totals into the slot `to`, then the grid barrier
    auto finish = [&](unsigned long long *to, double res) -> bool {
        if (sums(ALGO)) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) res += __shfl_xor_sync(0xffffffffu, res, o);
            if (lane == 0) s_res[wid] = res;
        }
        __syncthreads();
        if (wid == 0) {
            if (sums(ALGO)) {
                res = lane < (int)kSmallWarps ? s_res[lane] : 0.0;
#pragma unroll
                for (int o = kSmallWarps / 2; o > 0; o >>= 1) res += __shfl_xor_sync(0xffffffffu, res, o);
            }
            if (lane == 0) {
                const uint32_t va = (uint32_t)s_va;
                if (va) atomicAdd(to + 1, s_ea);
                if (sums(ALGO) && !keeper) atomicAdd(to + 2, __double2ull_rn(res * kResOne));
                s_va = s_ea = 0ull;
                uint32_t now;
                s_go = small_arrive_wait(to, sp.cnt, va, &now);
                s_frontier = now;
            }
        }
        __syncthreads();
        return s_go != 0;
    };

    // initial values and frontier, or those of the saved state
    if (threadIdx.x == 0) s_va = s_ea = 0ull;
    __syncthreads();
    // destinations in groups of 32 from a multiple of 32 (so of one partition), one per lane
    const uint32_t gb = d0 & ~31u, ge = d0 + nd;
    for (uint32_t g = gb + threadIdx.x; g - (uint32_t)lane < ge; g += kSmallThreads) {
        uint32_t deg = 0;
        bool act = false;
        if (g >= d0 && g < ge) {
            deg = p.rowptr[g + 1] - p.rowptr[g];
            if (sp.resume) {
                act = (p.bits[g >> 5] >> (g & 31)) & 1u;
            } else {
                uint32_t v, lv, sv;
                act = init_vertex<ALGO>(p, g, deg, v, lv, sv);
                if (ALGO == ALG_MSBFS) {
                    for (uint32_t j = 0; j < p.nsrc; ++j) {
                        const bool here = p.msrc[j] == g;
                        if (here) v |= 1u << j;
                        p.lvl_ms[(uint64_t)j * p.V + g] = here ? 0u : kInf;
                    }
                    act = v != 0u;
                    sv = act ? ~v : kNull;
                }
                p.val[g] = v;
                if (ALGO == ALG_BFS) p.lvl[g] = lv;
                sp.sval[0][g] = sv;
            }
        }
        count(slots, g, act, deg);
    }
    if (keeper && threadIdx.x == 0) {
        sp.sval[0][p.V] = sp.sval[1][p.V] = kNull;
        if (sums(ALGO)) atomicAdd(slots + 2, __double2ull_rn(p.t_res0 * kResOne));
    }
    // what stays the same over the iterations or is this thread's alone is kept in registers: the warp's first quads (all
    // of them in the smallest graphs) and the first destination's degree, value, level and message
    const uint4 none = make_uint4(0, 0, 0, 0);
    const uint4 e_first = q0 + (uint32_t)lane < q1 ? sp.edge[rg.z + q0 + lane] : none;
    const uint4 w_first = (ALGO == ALG_SSSP && q0 + (uint32_t)lane < q1) ? sp.w[rg.z + q0 + lane] : none;
    const uint32_t g1 = gb + threadIdx.x;
    const bool own = g1 >= d0 && g1 < ge;
    uint32_t deg1 = 0, v1 = 0, lv1 = kInf, m1 = kNull;
    if (own) {
        deg1 = p.rowptr[g1 + 1] - p.rowptr[g1];
        v1 = p.val[g1];
        if (ALGO == ALG_BFS) lv1 = p.lvl[g1];
        m1 = sp.sval[0][g1];
    }
    uint32_t it = 0;
    bool ok = finish(slots, 0.0);
    for (; ok; ++it) {
        unsigned long long *cur = slots + small_slot_of(it) * slot, *next = slots + small_slot_of(it + 1) * slot;
        const uint32_t iter = sp.base + it + 1;
        const uint32_t fv = s_frontier;
        const double r = sums(ALGO) ? (double)__ldcg(cur + 2) * kResUnit : 0.0;
        bool done = fv == 0 || iter > p.max_iters;
        if ((ALGO == ALG_PR || ALGO == ALG_PPR) && iter > 1 && r < p.tol) done = true;
        if (done) {
            rep.frontier_v = fv;
            rep.residual = r;
            break;
        }
        if (keeper) {
            small_statistics<ALGO>(p, sp, cur, slots + small_slot_to_clear(it + 1) * slot, rep);
        } else {
            const uint32_t *msg = sp.sval[it & 1];
            uint32_t *nmsg = sp.sval[(it + 1) & 1];
            for (uint32_t i = threadIdx.x; i < nd; i += kSmallThreads) s_acc[i] = A::identity();
            if (lane == 0) s_carry[wid] = A::identity();
            __syncthreads();
            uint4 en = e_first, wn = w_first;
            for (uint32_t qb = q0; qb < q1; qb += 32) {
                const uint4 e = en, w = wn;
                const bool in = qb + (uint32_t)lane < q1;
                if (qb + 32 + (uint32_t)lane < q1) {
                    en = sp.edge[rg.z + qb + 32 + lane];
                    if (ALGO == ALG_SSSP) wn = sp.w[rg.z + qb + 32 + lane];
                }
                auto value = [&](uint32_t word, uint32_t wt) -> T {
                    uint32_t x = msg[word & (kSmallSrc - 1)];
                    if (x == kNull) return A::identity();
                    if (B16) x = from_bf16(to_bf16(x));
                    return A::of(O::weigh(x, (int32_t)wt));
                };
                T v0 = A::identity(), v1 = v0, v2 = v0, v3 = v0;
                uint32_t a0 = kSent, a1 = kSent, a2 = kSent, a3 = kSent;
                if (in) {
                    v0 = value(e.x, w.x); v1 = value(e.y, w.y); v2 = value(e.z, w.z); v3 = value(e.w, w.w);
                    a0 = e.x >> kSmallSrcBits; a1 = e.y >> kSmallSrcBits; a2 = e.z >> kSmallSrcBits; a3 = e.w >> kSmallSrcBits;
                }
                auto put = [&](uint32_t d, T v) {
                    T *to = d == cfd ? &s_carry[wid] : &s_acc[d];
                    *to = A::combine(*to, v);
                };
                const bool one = a0 == a3;  // the lane is inside one run
                T head = v0, open = v3;  // the first run's part (when it ends here), the open run's
                if (one) {
                    open = A::combine(A::combine(v0, v1), A::combine(v2, v3));
                } else {
                    if (a1 == a0) head = A::combine(head, v1);
                    if (a2 == a0) head = A::combine(head, v2);
                    if (a2 == a3) open = A::combine(v2, open);
                    if (a1 == a3) open = A::combine(v1, open);
                    if (a1 != a0 && a1 != a3) put(a1, a2 == a1 ? A::combine(v1, v2) : v1);
                    if (a2 != a1 && a2 != a3) put(a2, v2);  // a2 > a1 >= a0
                }
                const uint32_t pd = __shfl_up_sync(0xffffffffu, a3, 1), nx = __shfl_down_sync(0xffffffffu, a0, 1);
                const bool joins = lane > 0 && pd == a0;
                const uint32_t heads = __ballot_sync(0xffffffffu, !(joins && one));
                const uint32_t h = (uint32_t)lane - (31u - __clz(heads & (0xffffffffu >> (31 - lane))));
                const uint32_t hmax = __reduce_max_sync(0xffffffffu, in ? h : 0u);
                for (uint32_t o = 1; o <= hmax; o <<= 1) {
                    const T t = A::shfl_up(open, o);
                    if (h >= o) open = A::combine(t, open);
                }
                const T before = A::shfl_up(open, 1);
                __syncwarp();  // the words of a run that goes on from the step before are written
                if (in) {
                    if (!one) put(a0, joins ? A::combine(before, head) : head);
                    if (lane == 31 || nx != a3) put(a3, open);
                }
                __syncwarp();
            }
            __syncthreads();
            if (wid == 0) {  // the parts of runs that began in an earlier warp's share, in warp order
                const uint32_t cd = lane < (int)kSmallWarps ? s_cd[lane] : kSent;
                T x = lane < (int)kSmallWarps ? s_carry[lane] : A::identity();
                const uint32_t pd = __shfl_up_sync(0xffffffffu, cd, 1), nx = __shfl_down_sync(0xffffffffu, cd, 1);
                const uint32_t heads = __ballot_sync(0xffffffffu, lane == 0 || pd != cd);
                const uint32_t h = (uint32_t)lane - (31u - __clz(heads & (0xffffffffu >> (31 - lane))));
#pragma unroll
                for (uint32_t o = 1; o < kSmallWarps; o <<= 1) {
                    const T t = A::shfl_up(x, o);
                    if (h >= o) x = A::combine(t, x);
                }
                if (cd != kSent && (lane == 31 || nx != cd)) s_acc[cd] = A::combine(s_acc[cd], x);
            }
            __syncthreads();
            double res = 0.0;
            for (uint32_t g = g1; g - (uint32_t)lane < ge; g += kSmallThreads) {
                uint32_t deg = 0, fresh = 0;
                bool act = false;
                if (g >= d0 && g < ge) {
                    uint32_t v = v1, lv = lv1, m0 = m1;
                    deg = deg1;
                    if (g != g1) {
                        deg = p.rowptr[g + 1] - p.rowptr[g];
                        v = p.val[g];
                        if (ALGO == ALG_BFS) lv = p.lvl[g];
                        if (ALGO == ALG_PPR || ALGO == ALG_NIBBLE) m0 = msg[g];
                    }
                    // a vertex is active exactly when it has a message
                    const bool was = (ALGO == ALG_PPR || ALGO == ALG_NIBBLE) && m0 != kNull;
                    const Applied ap = apply_vertex<ALGO>(p, iter, g >> p.shift, g, v, lv, A::message(s_acc[g - d0]), deg, was);
                    if (ap.val != v) p.val[g] = ap.val;
                    nmsg[g] = ap.msg;
                    if (ALGO == ALG_BFS && ap.act) p.lvl[g] = iter;
                    if (g == g1) {
                        v1 = ap.val;
                        m1 = ap.msg;
                        if (ALGO == ALG_BFS && ap.act) lv1 = iter;
                    }
                    if (sums(ALGO)) res += (double)ap.change;
                    act = ap.act;
                    fresh = ap.fresh;
                }
                if (ALGO == ALG_MSBFS) {  // level rows: the stores to one row come from consecutive lanes
                    uint32_t wall = __reduce_or_sync(0xffffffffu, fresh);
                    while (wall) {
                        const int j = __ffs(wall) - 1;
                        wall &= wall - 1;
                        if ((fresh >> j) & 1u) p.lvl_ms[(uint64_t)j * p.V + g] = iter;
                    }
                }
                count(next, g, act, deg);
            }
            ok = finish(next, res);
        }
        if (keeper) ok = finish(next, 0.0);
    }
    // results, and the messages and the frontier where a later run looks for them
    for (uint32_t w = blockIdx.x * kSmallWarps + wid; w < (p.V + 31) / 32; w += gridDim.x * kSmallWarps) {
        const uint32_t g = w * 32 + (uint32_t)lane;
        const uint32_t word = __ballot_sync(0xffffffffu, g < p.V && sp.sval[it & 1][g] != kNull);
        if (lane == 0) p.bits[w] = word;
    }
    for (uint32_t i = threadIdx.x; i < nd; i += kSmallThreads) {
        const uint32_t g = d0 + i;
        if (it & 1) sp.sval[0][g] = sp.sval[1][g];
        if (sp.out) sp.out[g] = ALGO == ALG_BFS ? p.lvl[g] : p.val[g];
        if (ALGO == ALG_BFS && sp.out_parent) sp.out_parent[g] = p.val[g];
    }
    if (keeper && threadIdx.x == 0) {
        rep.iterations = it;
        rep.error = !ok || __ldcg(sp.cnt) != 0ull;
        *sp.report = rep;  // read by the host after it has synchronised with the stream
    }
}
