// FP64 epilogue of an evaluation at given poses, and the small kernels around the levels: set-up,
// top-K, selection.
//
//   tile sums     FP64 sum of the build pass' FP32 partial records, fixed order
//   gravity term  Eq. 3: r = R gamma^W - gamma^imu, J = [0 | -[a]x], a = R gamma^W
//   range term    Eq. 4-6: P = R^T (q - t), r = P_z - D(P_x, P_y), J = [-n | n x q]
//                 with n = R (-D_x, -D_y, 1) and q = d v
//   assembly      Supp. "Sensor-Prior Fusion in LM": H, g are sums over the terms
//   LM step       Eq. 8: (H + lambda I) dxi = -g by 6x6 Cholesky, Eq. 9: T' = exp(dxi) T
//   acceptance    keep T' iff its objective is lower and enough anchors stay visible
//   top-K         Supp. "Multi-Hypothesis Refinement": keep the K lowest objectives
//   selection     Sec. IV-E: argmin of the final objective over usable hypotheses
#include <math.h>

#include "pilot_fp64.cuh"
#include "pilot_internal.cuh"

namespace pilot {

namespace {

// One block of 256 threads per pose: FP64 sum of the tile records (8 partial chains per value,
// combined in a fixed order), then the priors on warp 0.  Launched while the build pass before it
// still runs.
__global__ void epilogue_kernel(const EpilogueParams p) {
    const int slot = blockIdx.x;
    __shared__ double part[8][kAcc];
    __shared__ double E[kAcc];
    const int v = threadIdx.x & 31, c = threadIdx.x >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float* src = p.partial + (size_t)slot * p.n_tiles * kAcc + v;
    part[c][v] = chain_sum([&](int t) { return __ldcg(src + (size_t)t * kAcc); }, c, p.n_tiles);
    __syncthreads();
    if (threadIdx.x >= 32) return;                 // warp 0
    double sum = part[0][v];
    for (int k = 1; k < min(8, p.n_tiles); ++k) sum += part[k][v];
    E[v] = sum;
    __syncwarp();
    lm_update(p.state[slot], kEpiEval, 0, p.damping_mode, p.prior, E, 0.0, nullptr,
              p.eval_out + (size_t)slot * kNumSums, v);
}

// LM state of hypothesis m at the start of a solve, by one warp.
__device__ __forceinline__ void init_hyp(HypState& s, const double* T_cw, int lane) {
    if (lane < 12) s.T[lane] = s.Tc[lane] = T_cw[lane];
    if (lane < 21) s.H[lane] = 0.0;
    else if (lane < 27) s.g[lane - 21] = 0.0;
    if (lane == 0) {
        s.cost = 0.0;
        s.lambda = 0.0;
        s.n_valid = 0;
        s.has_cand = 0;
        s.last_fail = 0;
        s.active = 1;
        s.status = PILOT_HYP_OK;
    }
}

// Number of set flags among N, by the whole block (blockDim.x a multiple of 32, at most 1024; 16
// flags per load between 16-byte boundaries); on every thread.
__device__ __forceinline__ int count_flags(const uint8_t* valid, int N) {
    __shared__ int part[32];
    int c = 0;
    const int head = min(N, (int)((0u - (unsigned)(uintptr_t)valid) & 15u)), n16 = (N - head) / 16;
    const uint4* w = reinterpret_cast<const uint4*>(valid + head);
    auto set4 = [](unsigned v) { return ((v & 0xffu) != 0) + ((v & 0xff00u) != 0) + ((v & 0xff0000u) != 0) + ((v >> 24) != 0); };
#pragma unroll 4
    for (int k = threadIdx.x; k < n16; k += blockDim.x) {
        const uint4 v = w[k];
        c += set4(v.x) + set4(v.y) + set4(v.z) + set4(v.w);
    }
    // the bytes before and behind (fewer than 32)
    for (int j = threadIdx.x; j < N - 16 * n16; j += blockDim.x) c += valid[j < head ? j : j + 16 * n16] != 0;
    c = __reduce_add_sync(0xffffffffu, c);
    __syncthreads();                                   // a count before this one has been read
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
    __syncthreads();
    c = 0;
    for (int k = 0; k < (int)blockDim.x / 32; ++k) c += part[k];
    return c;
}

// Threshold on visible anchors for the fraction frac of c; never -0.0 (a fraction of -0.0 is accepted
// as 0), because the LM step compares it with a count by their words.
__device__ __forceinline__ double visible_threshold(double frac, int c) { return fabs(frac) * (double)c; }

// Start of a plain solve: the hypotheses' states, one per warp; the tickets; and, by the last
// block, the threshold on visible anchors.  One launch for what were three (5.7 + 5.5 us alone at
// 65536 anchors and 64 hypotheses, 2.8 + 7.7 us at 500 and 1210).
constexpr int kInitThreads = 256;
__global__ void __launch_bounds__(kInitThreads)
solve_init_kernel(HypState* st, const double* T_cw, int* active_idx, int M, unsigned* tickets, unsigned* done_ticket,
                  const uint8_t* valid, int N, double frac, double* min_valid) {
    if (blockIdx.x == gridDim.x - 1) {
        const int c = valid ? count_flags(valid, N) : N;
        if (threadIdx.x == 0) {
            *min_valid = visible_threshold(frac, c);
            *done_ticket = 0u;
        }
        return;
    }
    const int m = blockIdx.x * (kInitThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (m >= M) return;
    init_hyp(st[m], T_cw + 12 * (size_t)m, lane);
    if (lane == 0) {
        active_idx[m] = m;
        tickets[m] = 0u;
    }
}

__global__ void level_init_kernel(HypState* st, float* pose32, const int* active_idx, int n_active,
                                  double lambda0) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_active) return;
    const int m = active_idx[s];
    st[m].lambda = lambda0;
    st[m].last_fail = 0;
    st[m].has_cand = 1;
    store_pose32(pose32 + 12 * m, st[m].T);
}

// Ranking key of a hypothesis: (unusable, cost, index), unusable = non-finite objective or
// too few visible anchors; unusable ones compare by index only.  The cost is compared as an
// order-preserving 64-bit integer image of the double (both zeros map to one value), which
// orders exactly as the doubles do but keeps the n^2 comparisons off the FP64 pipe.
__device__ __forceinline__ void rank_key(const HypState& h, double min_valid, int* bad,
                                         unsigned long long* c) {
    *bad = !(isfinite(h.cost) && h.n_valid >= min_valid);
    const unsigned long long u = (unsigned long long)__double_as_longlong((isfinite(h.cost) ? h.cost : 0.0) + 0.0);
    *c = (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// The (unusable, cost image, index) order as one lexicographic comparison of two 64-bit
// words: hi = unusable bit | cost image >> 1, lo = lowest cost-image bit | index.
__device__ __forceinline__ ulonglong2 order_key(int bad, unsigned long long c, int idx) {
    return make_ulonglong2(((unsigned long long)(bad != 0) << 63) | (c >> 1),
                           ((c & 1ull) << 63) | (unsigned long long)(unsigned)idx);
}

// Top-K (Supp. "Multi-Hypothesis Refinement") over the n hypotheses listed in act[0, n) of
// S, in two passes.  rank_mark: LANES lanes of a block share one listed hypothesis of
// [s_begin, s_begin + kRankThreads / LANES), count the listed hypotheses that rank before it (keys
// streamed through shared memory kRankThreads at a time) and mark it pruned if that count is
// K or more.  compact_active (one block, blockDim.x a multiple of 32, at most 1024, after every
// rank_mark block has finished): writes the survivors' indices, in their order in act, to
// act_out[0, K) (act_out may be act) by a block-wide prefix count.
// The n^2 comparisons are spread over LANES lanes per hypothesis since five blocks of one thread
// per hypothesis took 28.6 us for 1210 (alone); a warp each, with the compaction of the survivors (6 us)
// in the same launch: 16 us.
constexpr int kRankThreads = 256;

template <int LANES>
__device__ void rank_mark(HypState* S, const int* act, int n, int K, double min_valid, int s_begin) {
    __shared__ ulonglong2 kk[kRankThreads];      // order keys of the current chunk
    const int tid = threadIdx.x, sub = tid % LANES;
    const int s = s_begin + tid / LANES;
    int m = -1, rank = 0;
    ulonglong2 key = make_ulonglong2(~0ull, ~0ull);
    if (s < n) {
        int bad;
        unsigned long long c;
        m = act[s];
        rank_key(S[m], min_valid, &bad, &c);
        key = order_key(bad, c, m);
    }
    for (int c0 = 0; c0 < n; c0 += kRankThreads) {
        __syncthreads();
        if (c0 + tid < n) {
            int bad;
            unsigned long long c;
            const int m2 = act[c0 + tid];
            rank_key(S[m2], min_valid, &bad, &c);
            kk[tid] = order_key(bad, c, m2);
        }
        __syncthreads();
        if (s < n) {
            const int lim = min(kRankThreads, n - c0);
#pragma unroll 4
            for (int j = sub; j < lim; j += LANES) {
                const ulonglong2 o = kk[j];
                rank += (o.x < key.x) | ((o.x == key.x) & (o.y < key.y));
            }
        }
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (s < n && rank >= K && sub == 0) {
        S[m].active = 0;
        S[m].status = PILOT_HYP_PRUNED;
    }
}

__device__ void compact_active(const HypState* S, const int* act, int* act_out, int n) {
    __shared__ int wsum[32];
    __shared__ int s_base;
    const int bd = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_base = 0;
    __syncthreads();
    for (int c0 = 0; c0 < n; c0 += bd) {
        const int s = c0 + tid;
        int m = -1;
        bool keep = false;
        if (s < n) {
            m = act[s];
            keep = __ldcg(&S[m].active) != 0;        // other blocks of the launch may have marked it
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) wsum[warp] = __popc(bal);
        __syncthreads();
        int off = s_base;
        for (int w = 0; w < warp; ++w) off += wsum[w];
        if (keep) act_out[off + __popc(bal & ((1u << lane) - 1u))] = m;
        __syncthreads();
        if (tid == 0) {
            int t = 0;
            for (int w = 0; w < bd / 32; ++w) t += wsum[w];
            s_base += t;
        }
        __syncthreads();
    }
}

// Whether this block is the last of the launch to get here (ticket zero before the launch and left
// zero); what the other blocks wrote before is then visible.
__device__ __forceinline__ bool last_block(unsigned* ticket, unsigned blocks) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(ticket, 1u) == blocks - 1u;
        if (last) *ticket = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Plain form: the last block lists the survivors, in their order in active_in, in active_out.  A warp
// per listed hypothesis, but eight lanes beyond kWideRank of them and one beyond kThinRank: every
// block reads every key, n^2 LANES / 256 reads, and they are then what the launch takes.  Solves of
// 100 anchors, one iteration per level, with a warp and as it is: 8193 hypotheses 479 and 469 us,
// 20000 1373 and 1115, 60000 6406 and 4209 (4616 with eight lanes), 150000 30.9 and 14.1 ms
// (18.1).
constexpr int kWideRank = 8192, kThinRank = 32768;
template <int LANES>
__global__ void __launch_bounds__(kRankThreads)
prune_kernel(HypState* st, const int* active_in, int* active_out, int n, int K, const double* min_valid_ptr,
             unsigned* ticket) {
    rank_mark<LANES>(st, active_in, n, K, *min_valid_ptr, blockIdx.x * (kRankThreads / LANES));
    if (last_block(ticket, gridDim.x)) compact_active(st, active_in, active_out, n);
}

// Final status and outputs of one hypothesis, by one warp (output index o).
__device__ __forceinline__ void finish_hyp(HypState& s, double min_valid, size_t o, double* T, double* cost, int* nv,
                                           int* status, int lane) {
    const double t = lane < 12 ? s.T[lane] : 0.0;
    const double c = s.cost;
    const bool finite = __all_sync(0xffffffffu, isfinite(t)) && isfinite(c);
    if (lane < 12) T[12 * o + lane] = t;
    if (lane == 0) {
        int code = s.status;
        if (s.active) {
            if (!finite) code = PILOT_HYP_NONFINITE;
            else if (s.n_valid < min_valid) code = PILOT_HYP_FEW_VALID;
            else if (s.last_fail) code = PILOT_HYP_NOT_PD;
            else code = PILOT_HYP_OK;
            s.status = code;
        }
        cost[o] = c;
        nv[o] = s.n_valid;
        status[o] = code;
    }
}

// Index of the lowest cost among M hypotheses with status OK (ties: the lowest index), or -1; by
// the whole block of kFinishThreads, on thread 0.  Outputs other blocks wrote are read from L2.
constexpr int kFinishThreads = 256;
__device__ __forceinline__ int best_of(const double* cost, const int* status, int M) {
    __shared__ double bc[kFinishThreads];
    __shared__ int bi[kFinishThreads];
    const int tid = threadIdx.x;
    double my_c = 0.0;
    int my_i = -1;
    for (int m = tid; m < M; m += kFinishThreads) {
        const double c = __ldcg(cost + m);
        if (__ldcg(status + m) == PILOT_HYP_OK && (my_i < 0 || c < my_c)) {
            my_c = c;
            my_i = m;
        }
    }
    bc[tid] = my_c;
    bi[tid] = my_i;
    __syncthreads();
    for (int s = kFinishThreads / 2; s > 0; s >>= 1) {
        if (tid < s) {
            const int j = tid + s;
            const bool take = bi[j] >= 0 &&
                              (bi[tid] < 0 || bc[j] < bc[tid] || (bc[j] == bc[tid] && bi[j] < bi[tid]));
            if (take) {
                bc[tid] = bc[j];
                bi[tid] = bi[j];
            }
        }
        __syncthreads();
    }
    return bi[0];
}

// Plain form: statuses and the result block, one hypothesis per warp; the last block selects.  One
// block of a thread per hypothesis, each reading its 560-byte state alone, took 26.7 us for
// 1210 hypotheses (alone); now 8.0 us.
__global__ void __launch_bounds__(kFinishThreads)
finalize_kernel(HypState* st, int M, const double* min_valid_ptr, unsigned char* res, ResultLayout lay, unsigned* ticket) {
    double* cost = reinterpret_cast<double*>(res + lay.off_cost);
    int* status = reinterpret_cast<int*>(res + lay.off_status);
    const int m = blockIdx.x * (kFinishThreads / 32) + (threadIdx.x >> 5);
    if (m < M)
        finish_hyp(st[m], *min_valid_ptr, m, reinterpret_cast<double*>(res + lay.off_T), cost,
                   reinterpret_cast<int*>(res + lay.off_nvalid), status, threadIdx.x & 31);
    if (!last_block(ticket, gridDim.x)) return;
    const int best = best_of(cost, status, M);
    if (threadIdx.x == 0) *reinterpret_cast<int*>(res + lay.off_best) = best;
}

// ---- batched form and serving rounds ----

// The hypotheses of one frame from the first-th on, one per warp, every stride-th.
__device__ void init_frame(const FrameDesc& f, HypState* st, int* active, int first, int stride) {
    const int lane = threadIdx.x & 31;
    for (int m = first; m < f.M; m += stride) {
        init_hyp(st[f.hyp_offset + m], f.T_cw + 12 * (size_t)m, lane);
        if (lane == 0) active[f.hyp_offset + m] = m;
    }
}

// Statuses and outputs (at the global hypothesis index) of one frame's hypotheses from the first-th
// on, one per warp, every stride-th.
__device__ void finish_frame(const FrameDesc& f, HypState* st, double mv, unsigned char* res, int max_hyps, int first,
                             int stride) {
    const ResultLayout lay = ResultLayout::make(max_hyps);
    for (int m = first; m < f.M; m += stride)
        finish_hyp(st[f.hyp_offset + m], mv, (size_t)f.hyp_offset + m, reinterpret_cast<double*>(res + lay.off_T),
                   reinterpret_cast<double*>(res + lay.off_cost), reinterpret_cast<int*>(res + lay.off_nvalid),
                   reinterpret_cast<int*>(res + lay.off_status), threadIdx.x & 31);
}

// The selection of one frame whose outputs are written.
__device__ void select_frame(const FrameDesc& f, int fi, unsigned char* res, int max_hyps) {
    const ResultLayout lay = ResultLayout::make(max_hyps);
    const int best = best_of(reinterpret_cast<double*>(res + lay.off_cost) + f.hyp_offset,
                             reinterpret_cast<int*>(res + lay.off_status) + f.hyp_offset, f.M);
    if (threadIdx.x == 0) reinterpret_cast<int*>(res + lay.bytes)[fi] = best;     // one int per frame after the block
}

// Grids over the frames (x) and over one frame's hypotheses (y).  A handle's or a server's launches
// are captured for all the frames it may hold, so their grids are bounded: blocks that find no work
// still take their turn (eight frames in a handle for 65536: 2234 us with a block per frame, 10275
// with every block of every frame, 719 so).
constexpr int kFrameBlocks = 16;
constexpr int kMaxFrameBlocks = 1024;      // frames side by side; more take turns

// Set-up and results, a warp per hypothesis, and one more block: sixteen blocks per frame (with one,
// 1210 hypotheses took 54 us to set up and 28.6 us to finish, alone) while a few thousand are enough.
dim3 frame_grid(int max_frames) {
    const int x = max_frames < kMaxFrameBlocks ? max_frames : kMaxFrameBlocks;
    return dim3(x, (x <= 256 ? kFrameBlocks : 4096 / x) + 1);
}

// Ranking, kRankHyps hypotheses per turn of a block.  Turns are numbered frame after frame, as if every
// frame had max_frame_hyps; block b takes turns b, b + gridDim.x, ... of those a frame has, so that a
// frame's turns go to different blocks, and by the blocks' prime number different frames' first turns
// too.
constexpr int kRankLanes = 8, kRankHyps = kRankThreads / kRankLanes;   // batched and served forms
constexpr int kRankBlocks = 2039;
int rank_turns(int max_frame_hyps) { return (max_frame_hyps + kRankHyps - 1) / kRankHyps; }
int rank_blocks(int max_frames, int turns) {
    const long long n = (long long)max_frames * turns;
    return n < kRankBlocks ? (int)n : kRankBlocks;
}

// body(frame, first hypothesis) for this block's turns, count(frame) being a frame's hypotheses to
// rank; a thread looks up one turn.  All threads of the block of kRankThreads.
template <typename Count, typename Body>
__device__ __forceinline__ void each_rank_turn(int n_frames, int turns, Count count, Body body) {
    __shared__ int2 list[kRankThreads];
    __shared__ int listed;
    const long long all = (long long)n_frames * turns;
    for (long long w0 = blockIdx.x; w0 < all; w0 += (long long)gridDim.x * kRankThreads) {
        __syncthreads();
        if (threadIdx.x == 0) listed = 0;
        __syncthreads();
        const long long w = w0 + (long long)threadIdx.x * gridDim.x;
        if (w < all) {
            const int fi = (int)(w / turns), s0 = (int)(w % turns) * kRankHyps;
            if (s0 < count(fi)) list[atomicAdd(&listed, 1)] = make_int2(fi, s0);
        }
        __syncthreads();
        for (int i = 0; i < listed; ++i) body(list[i].x, list[i].y);
    }
}

__global__ void __launch_bounds__(kInitThreads)
batch_init_kernel(const BatchHeader* hdr, const FrameDesc* frames, HypState* st, int* active, double frac,
                  double* min_valid, unsigned* tickets) {
    const int warps = kInitThreads / 32, parts = gridDim.y - 1;
    for (int fi = blockIdx.x; fi < hdr->n_frames; fi += gridDim.x) {
        const FrameDesc& f = frames[fi];
        if ((int)blockIdx.y < parts) {
            init_frame(f, st, active, blockIdx.y * warps + (threadIdx.x >> 5), parts * warps);
        } else {
            const int c = f.valid ? count_flags(f.valid, f.N) : f.N;
            if (threadIdx.x == 0) {
                min_valid[fi] = visible_threshold(frac, c);
                tickets[fi] = 0u;
            }
        }
    }
}

// Batched form, top-K after a level (frames whose count is at most K keep all of them).
__global__ void __launch_bounds__(kRankThreads)
batch_rank_kernel(const BatchHeader* hdr, const FrameDesc* frames, HypState* st, const int* active,
                  const int* n_active, int turns, int K, const double* min_valid) {
    if (K <= 0) return;
    each_rank_turn(hdr->n_frames, turns, [&](int fi) { return K < n_active[fi] ? n_active[fi] : 0; }, [&](int fi, int s0) {
        const FrameDesc& f = frames[fi];
        rank_mark<kRankLanes>(st + f.hyp_offset, active + f.hyp_offset, n_active[fi], K, min_valid[fi], s0);
    });
}

// Batched form: each pruned frame's active list compacted in place.
__global__ void batch_compact_kernel(const BatchHeader* hdr, const FrameDesc* frames, const HypState* st,
                                     int* active, const int* n_active, int K) {
    for (int fi = blockIdx.x; fi < hdr->n_frames; fi += gridDim.x) {
        const int n = n_active[fi];
        if (K <= 0 || K >= n) continue;
        const FrameDesc& f = frames[fi];
        compact_active(st + f.hyp_offset, active + f.hyp_offset, active + f.hyp_offset, n);
    }
}

__global__ void __launch_bounds__(kFinishThreads)
batch_finalize_kernel(const BatchHeader* hdr, const FrameDesc* frames, HypState* st, const double* min_valid,
                      unsigned char* res, int max_hyps, unsigned* tickets) {
    const int warps = kFinishThreads / 32, parts = gridDim.y;
    for (int fi = blockIdx.x; fi < hdr->n_frames; fi += gridDim.x) {
        finish_frame(frames[fi], st, min_valid[fi], res, max_hyps, blockIdx.y * warps + (threadIdx.x >> 5), parts * warps);
        if (last_block(tickets + fi, parts)) select_frame(frames[fi], fi, res, max_hyps);
    }
}

// Serving rounds, blocks as frame_grid lays them out: of a frame's, all but the last take its hypotheses
// and the last one its count of valid anchors.
__global__ void __launch_bounds__(kInitThreads)
round_prepare_kernel(const BatchHeader* hdr, const FrameDesc* frames, HypState* st, int* active, double frac,
                     double* min_valid, unsigned* tickets) {
    const int warps = kInitThreads / 32, parts = gridDim.y - 1;
    for (int fi = blockIdx.x; fi < hdr->n_frames; fi += gridDim.x) {
        const FrameDesc& f = frames[fi];
        if (!(f.flags & kFlagInit)) continue;
        if ((int)blockIdx.y < parts) {
            init_frame(f, st, active, blockIdx.y * warps + (threadIdx.x >> 5), parts * warps);
        } else {
            const int c = f.valid ? count_flags(f.valid, f.N) : f.N;
            if (threadIdx.x == 0) {
                min_valid[fi] = visible_threshold(frac, c);
                tickets[fi] = 0u;
            }
        }
    }
}

// Serving round, top-K of the frames that finished a pruning level (as batch_rank_kernel).
__global__ void __launch_bounds__(kRankThreads)
round_rank_kernel(const BatchHeader* hdr, const FrameDesc* frames, HypState* st, const int* active, int turns,
                  const double* min_valid) {
    each_rank_turn(hdr->n_frames, turns, [&](int fi) { return frames[fi].flags & kFlagPrune ? frames[fi].n_active : 0; },
                   [&](int fi, int s0) {
        const FrameDesc& f = frames[fi];
        rank_mark<kRankLanes>(st + f.hyp_offset, active + f.hyp_offset, f.n_active, f.keep, min_valid[fi], s0);
    });
}

// The end of a round's level, blocks as in round_prepare_kernel: the last one of a frame's compacts the
// active list after a pruning level, the others write a finished frame's results, and the last of
// those to be done selects.
__global__ void __launch_bounds__(kFinishThreads)
round_finish_kernel(const BatchHeader* hdr, const FrameDesc* frames, HypState* st, int* active, const double* min_valid,
                    unsigned char* res, int max_hyps, unsigned* tickets) {
    const int warps = kFinishThreads / 32, parts = gridDim.y - 1;
    for (int fi = blockIdx.x; fi < hdr->n_frames; fi += gridDim.x) {
        const FrameDesc& f = frames[fi];
        if ((int)blockIdx.y == parts) {
            if (f.flags & kFlagPrune)
                compact_active(st + f.hyp_offset, active + f.hyp_offset, active + f.hyp_offset, f.n_active);
        } else if (f.flags & kFlagFinalize) {
            finish_frame(f, st, min_valid[fi], res, max_hyps, blockIdx.y * warps + (threadIdx.x >> 5), parts * warps);
            if (last_block(tickets + fi, parts)) select_frame(f, fi, res, max_hyps);
        }
    }
}

// Serving round with several levels: after a level's finish, every listed frame moves on to
// its next level on the device (what the host does between one-level rounds): a frame that
// finished level 0 (finalised), or that has used its quota of levels for the round, drops out
// with no jobs; the others take their top-K, step to the next finer level and get that
// level's flags; the job and item tables are rebuilt in list order.  One thread: at most
// max_slots frames.
__global__ void round_advance_kernel(const BatchHeader* hdr, FrameDesc* frames, const int* fr_list, int* fr_item,
                                     int* fr_job, LevelKeep keep, int tile, int tpi) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    const int nl = hdr->n_listed[0];
    if (hdr->tiles_per_item > 0) tpi = hdr->tiles_per_item;   // the round's own work-item size
    fr_item[0] = 0;
    fr_job[0] = 0;
    for (int i = 0; i < nl; ++i) {
        FrameDesc& f = frames[fr_list[i]];
        f.quota -= 1;
        if (f.n_active > 0 && f.quota <= 0) {
            // this frame's levels for the round are done: it idles until the next round (the
            // host carries its level and active count over)
            f.n_active = 0;
            f.flags = 0;
        } else if (f.n_active > 0) {
            if (f.level == 0) {
                f.n_active = 0;
                f.flags = 0;
            } else {
                if (f.flags & kFlagPrune) f.n_active = f.keep;
                f.level -= 1;
                const int K = keep.k[f.level];
                f.keep = K;
                f.flags = ((f.level > 0 && K > 0 && K < f.n_active) ? kFlagPrune : 0) | (f.level == 0 ? kFlagFinalize : 0);
            }
        } else {
            f.flags = 0;
        }
        fr_job[i + 1] = fr_job[i] + f.n_active;
        fr_item[i + 1] = fr_item[i] + frame_items(f.n_active, f.N, tile, tpi);
    }
}

}  // namespace

cudaError_t launch_round_advance(const BatchHeader* hdr, FrameDesc* frames, const int* fr_list, int* fr_item,
                                 int* fr_job, const LevelKeep& keep, int tile, int tpi, cudaStream_t s) {
    round_advance_kernel<<<1, 32, 0, s>>>(hdr, frames, fr_list, fr_item, fr_job, keep, tile, tpi);
    return cudaGetLastError();
}

cudaError_t launch_batch_init(const BatchHeader* hdr, const FrameDesc* frames, HypState* st,
                              int* active, double frac, double* min_valid, unsigned* tickets, int max_frames,
                              cudaStream_t s) {
    batch_init_kernel<<<frame_grid(max_frames), kInitThreads, 0, s>>>(hdr, frames, st, active, frac, min_valid, tickets);
    return cudaGetLastError();
}

cudaError_t launch_batch_prune(const BatchHeader* hdr, const FrameDesc* frames, HypState* st,
                               int* active, const int* n_active, int keep, const double* min_valid,
                               int max_frames, int max_frame_hyps, cudaStream_t s) {
    const int turns = rank_turns(max_frame_hyps);
    batch_rank_kernel<<<rank_blocks(max_frames, turns), kRankThreads, 0, s>>>(hdr, frames, st, active, n_active, turns, keep,
                                                                              min_valid);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    batch_compact_kernel<<<frame_grid(max_frames).x, 1024, 0, s>>>(hdr, frames, st, active, n_active, keep);
    return cudaGetLastError();
}

cudaError_t launch_batch_finalize(const BatchHeader* hdr, const FrameDesc* frames, HypState* st,
                                  const double* min_valid, unsigned char* result, int max_hyps,
                                  unsigned* tickets, int max_frames, cudaStream_t s) {
    const dim3 grid = frame_grid(max_frames);
    batch_finalize_kernel<<<dim3(grid.x, grid.y - 1), kFinishThreads, 0, s>>>(hdr, frames, st, min_valid, result, max_hyps,
                                                                              tickets);
    return cudaGetLastError();
}

cudaError_t launch_round_prepare(const BatchHeader* hdr, const FrameDesc* frames, HypState* st,
                                 int* active, double frac, double* min_valid, unsigned* tickets, int max_frames,
                                 cudaStream_t s) {
    round_prepare_kernel<<<frame_grid(max_frames), kInitThreads, 0, s>>>(hdr, frames, st, active, frac, min_valid, tickets);
    return cudaGetLastError();
}

cudaError_t launch_round_finish(const BatchHeader* hdr, const FrameDesc* frames, HypState* st,
                                int* active, const double* min_valid, unsigned char* result,
                                int max_hyps, unsigned* tickets, int max_frames, int max_frame_hyps, cudaStream_t s) {
    const int turns = rank_turns(max_frame_hyps);
    round_rank_kernel<<<rank_blocks(max_frames, turns), kRankThreads, 0, s>>>(hdr, frames, st, active, turns, min_valid);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    round_finish_kernel<<<frame_grid(max_frames), kFinishThreads, 0, s>>>(hdr, frames, st, active, min_valid, result, max_hyps,
                                                                          tickets);
    return cudaGetLastError();
}

cudaError_t launch_epilogue(const EpilogueParams& p, cudaStream_t s) {
    if (p.n_active <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(p.n_active);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, epilogue_kernel, p);
}

cudaError_t launch_solve_init(HypState* st, const double* T_cw, int* active_idx, int M, unsigned* tickets,
                              unsigned* done_ticket, const uint8_t* valid, int N, double frac, double* min_valid,
                              cudaStream_t s) {
    solve_init_kernel<<<(M + kInitThreads / 32 - 1) / (kInitThreads / 32) + 1, kInitThreads, 0, s>>>(
        st, T_cw, active_idx, M, tickets, done_ticket, valid, N, frac, min_valid);
    return cudaGetLastError();
}

cudaError_t launch_level_init(HypState* st, float* pose32, const int* active_idx, int n_active,
                              double lambda0, cudaStream_t s) {
    if (n_active <= 0) return cudaSuccess;
    level_init_kernel<<<(n_active + 127) / 128, 128, 0, s>>>(st, pose32, active_idx, n_active, lambda0);
    return cudaGetLastError();
}

cudaError_t launch_prune(HypState* st, const int* active_in, int* active_out, int n_active,
                         int keep, const double* min_valid, unsigned* ticket, cudaStream_t s) {
    if (n_active <= 0) return cudaSuccess;
    auto launch = [&](auto kernel, int lanes) {
        const int per_block = kRankThreads / lanes;
        kernel<<<(n_active + per_block - 1) / per_block, kRankThreads, 0, s>>>(st, active_in, active_out, n_active, keep,
                                                                              min_valid, ticket);
    };
    if (n_active <= kWideRank) launch(prune_kernel<32>, 32);
    else if (n_active <= kThinRank) launch(prune_kernel<8>, 8);
    else launch(prune_kernel<1>, 1);
    return cudaGetLastError();
}

cudaError_t launch_finalize(HypState* st, int M, const double* min_valid, unsigned char* result,
                            ResultLayout lay, unsigned* ticket, cudaStream_t s) {
    constexpr int per_block = kFinishThreads / 32;
    finalize_kernel<<<(M + per_block - 1) / per_block, kFinishThreads, 0, s>>>(st, M, min_valid, result, lay, ticket);
    return cudaGetLastError();
}

}  // namespace pilot
