// Geo-anchor sampling on the GPU (Supp. "TDOM/DSM Reference Crop": the valid geo-anchors
// the solver uses are sampled from the reference crop).
//
// Pixel j of the crop gets the key (upper 32 bits of the (j+1)-th output of the SplitMix64
// generator started at `seed`) * 2^32 + j -- unique per pixel, uniformly ordered over the
// pixels by the generator -- and the n_select valid pixels with the smallest keys are
// taken: a uniform draw without replacement, decided in integer arithmetic only.
// SplitMix64 (Steele, Lea and Flood, "Fast splittable pseudorandom number generators",
// OOPSLA 2014): state += 0x9E3779B97F4A7C15, then
//   z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9; z = (z ^ (z >> 27)) * 0x94D049BB133111EB;
//   output z ^ (z >> 31).
//
// One cluster of 8 CTAs (one CTA for small crops).  A pass over an 11-bit digit of the keys (one shared-memory histogram
// per CTA, summed through distributed shared memory) finds the bin that holds the n_select-th
// smallest key; with uniform keys the first digit leaves about n / 2048 candidates, which are
// gathered and ranked against one another (more digits follow only while more than 1024 keys
// share the prefix, e.g. a crop of millions of pixels).  Every warp owns a run of consecutive
// pixels, so the selected pixels are listed in increasing order from ballots and one scan over
// the warps and CTAs.
//
// What bounds it: latency, not bytes (64 KB of mask).  One CTA of 1024 threads making 8 digit
// passes and re-hashing every pixel in each took 162 us for 500 of 65536 pixels (174 us alone
// under ncu); a cluster of 8 CTAs that keeps the hashed halves of the keys in shared memory (up to
// 20 per thread, 163840 pixels; larger crops hash again per pass) takes 18.4 us, most of
// it the launch, five cluster barriers and the scans between them.  Crops of up to 4096 pixels need no
// second CTA: 500 of 1000 pixels 8.5 us (12.6 with the cluster, 26.8 before it), all of 1000 6.5
// (11.4, 6.3), 500 of 4096 12.5 (12.6, 22.9), all of 4096 8.5 (10.6, 10.4).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pilot_internal.cuh"

namespace cg = cooperative_groups;

namespace pilot {
namespace {

constexpr int kSampleCtas = 8;                    // one cluster (one CTA for small crops)
constexpr int kSampleThreads = 1024;
constexpr int kSampleWarps = kSampleThreads / 32;
constexpr int kSampleBins = 2048;                 // 11-bit digits
constexpr int kSampleList = 1024;                 // candidates ranked directly
static_assert(kSampleBins == 2 * kSampleThreads, "two bins per thread");

__device__ __forceinline__ unsigned long long splitmix64_output(unsigned long long seed, unsigned long long j) {
    unsigned long long z = seed + (j + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Inclusive scan over the CTA (v per thread); *total receives the sum.  Two barriers.
__device__ __forceinline__ unsigned cta_scan(unsigned v, unsigned* s_warp, unsigned* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) s_warp[warp] = v;
    __syncthreads();
    unsigned before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kSampleWarps; ++w) {
        const unsigned c = s_warp[w];
        before += w < warp ? c : 0u;
        all += c;
    }
    __syncthreads();
    *total = all;
    return v + before;
}

constexpr int kSampleKeep = 20;                   // most steps whose keys are kept
constexpr int kSampleOne = 4096;                  // most pixels that one CTA takes

// KEEP: at most kSampleKeep steps of CTAS kSampleThreads pixels, the hashed halves of the keys kept in
// (dynamic) shared memory; else any number, hashed again where they are read.  One CTA counts the
// valid pixels before it hashes: where all of them are taken it lists them at once.
template <bool KEEP, int CTAS>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(kSampleThreads)
sample_anchors_kernel(const uint8_t* valid, const float* points, int n, int k, unsigned long long seed,
                      int* out_idx, float* out_pts, int* out_count) {
    static_assert(KEEP || CTAS > 1, "one CTA keeps its keys");
    constexpr int kStep = CTAS * kSampleThreads;   // pixels taken per step of all threads
    __shared__ __align__(16) unsigned hist[kSampleBins];
    __shared__ unsigned long long list[kSampleList], all[kSampleList];
    __shared__ unsigned s_warp[kSampleWarps];
    __shared__ unsigned s_n, s_bin, s_before, s_count, s_total;
    __shared__ unsigned long long s_kth;
    cg::cluster_group cluster = cg::this_cluster();
    auto all_ctas = [&]() {
        if constexpr (CTAS > 1) cluster.sync();
        else __syncthreads();
    };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = CTAS > 1 ? (int)cluster.block_rank() : 0;
    // warp gw owns pixels [gw run, (gw + 1) run), lane l of step i pixel 32 i + l of them
    const unsigned steps = (unsigned)(((long long)n + kStep - 1) / kStep);
    const unsigned first = (unsigned)(rank * kSampleWarps + warp) * steps * 32u + (unsigned)lane;
    extern __shared__ unsigned keys[];             // [step][thread] (KEEP)
    unsigned long long ok = 0;                     // bit i: pixel of step i is valid (KEEP)
    auto hash = [&](unsigned i) {
        keys[i * kSampleThreads + tid] = (unsigned)(splitmix64_output(seed, first + 32u * i) >> 32);
    };
    unsigned take = 0, want = 0;                   // want: 1-based rank within the prefix
    bool every = false;                            // every valid pixel is taken
    if constexpr (KEEP) {
        for (unsigned i0 = 0; i0 < steps; i0 += 8) {
            uint8_t v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = first + 32u * (i0 + u) < (unsigned)n && i0 + u < steps ? valid[first + 32u * (i0 + u)] : 0;
            if constexpr (CTAS > 1) {
#pragma unroll 2
                for (int u = 0; u < 8; ++u) {
                    if (i0 + u >= steps) break;
                    hash(i0 + u);
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) ok |= (unsigned long long)(v[u] != 0) << (i0 + u);
        }
        if constexpr (CTAS == 1) {
            unsigned total;
            cta_scan((unsigned)__popcll(ok), s_warp, &total);
            take = (unsigned)k < total ? (unsigned)k : total;
            every = take == total;
            if (!every)
                for (unsigned i = 0; i < steps; ++i) hash(i);
        }
    }
    // key of this thread's pixel of step i; false when it is not valid
    auto key_of = [&](unsigned i, unsigned long long& key) {
        const unsigned j = first + 32u * i;
        if constexpr (KEEP) {
            key = ((unsigned long long)keys[i * kSampleThreads + tid] << 32) | j;
            return ((ok >> i) & 1ull) != 0ull;
        } else {
            key = (splitmix64_output(seed, j) >> 32 << 32) | j;
            return j < (unsigned)n && valid[j] != 0;
        }
    };
    auto each_valid = [&](auto f) {
#pragma unroll 4
        for (unsigned i = 0; i < steps; ++i) {
            unsigned long long key;
            if (key_of(i, key)) f(key);
        }
    };

    // the take-th smallest key (all valid pixels when take is their number)
    unsigned long long kth = ~0ull, prefix = 0, mask = 0;
    if (tid == 0) s_n = 0;
    for (int shift = 53; shift >= 0 && !every; shift = shift > 11 ? shift - 11 : (shift > 0 ? 0 : -1)) {
        // digits of the key's bits 63-53, 52-42, 41-31, 30-20, 19-9 (11 bits each) and 8-0
        const unsigned digit_mask = shift == 0 ? 0x1ffu : 0x7ffu;
        reinterpret_cast<uint2*>(hist)[tid] = make_uint2(0u, 0u);
        __syncthreads();
        each_valid([&](unsigned long long key) {
            if ((key & mask) == prefix) atomicAdd(&hist[(unsigned)(key >> shift) & digit_mask], 1u);
        });
        all_ctas();
        uint2 c = make_uint2(0u, 0u);              // bins 2 tid and 2 tid + 1 over the cluster
        if constexpr (CTAS > 1) {
#pragma unroll
            for (int r = 0; r < CTAS; ++r) {
                const uint2 o = reinterpret_cast<const uint2*>(cluster.map_shared_rank(hist, r))[tid];
                c.x += o.x, c.y += o.y;
            }
        } else {
            c = reinterpret_cast<const uint2*>(hist)[tid];
        }
        const unsigned sum = c.x + c.y;
        unsigned total;
        const unsigned incl = cta_scan(sum, s_warp, &total);
        if (shift == 53) {
            take = (unsigned)k < total ? (unsigned)k : total;
            want = take;
            every = take == total;
            if (take == 0 || every) break;
        }
        const unsigned before = incl - sum;
        if (before < want && want <= incl) {       // exactly one thread
            const bool second = before + c.x < want;
            s_bin = 2u * tid + second;
            s_before = before + (second ? c.x : 0u);
            s_count = second ? c.y : c.x;
        }
        __syncthreads();
        prefix |= (unsigned long long)s_bin << shift;
        mask |= (unsigned long long)digit_mask << shift;
        want -= s_before;
        if (s_count <= kSampleList) {
            // few candidates: gathered in every CTA and ranked against one another
            each_valid([&](unsigned long long key) {
                if ((key & mask) == prefix) list[atomicAdd(&s_n, 1u)] = key;
            });
            all_ctas();
            unsigned at = s_n;
            const unsigned long long* found = list;
            if constexpr (CTAS > 1) {
                // warp r copies CTA r's list behind those of the CTAs before it
                const unsigned held = lane < CTAS ? *cluster.map_shared_rank(&s_n, lane) : 0u;
                at = __reduce_add_sync(0xffffffffu, held);
                if (warp < CTAS) {
                    const unsigned m = __shfl_sync(0xffffffffu, held, warp);
                    const unsigned to = __reduce_add_sync(0xffffffffu, lane < warp ? held : 0u);
                    const unsigned long long* src = cluster.map_shared_rank(list, warp);
                    for (unsigned i = lane; i < m; i += 32) all[to + i] = src[i];
                }
                found = all;
                __syncthreads();
            }
            for (unsigned i = tid; i < at; i += kSampleThreads) {
                const unsigned long long key = found[i];
                unsigned less = 0;
                for (unsigned q = 0; q < at; ++q) less += found[q] < key;
                if (less + 1u == want) s_kth = key;
            }
            __syncthreads();
            kth = s_kth;
            break;
        }
        if (shift == 0) kth = prefix;              // cannot happen: keys are distinct
        all_ctas();                                // every CTA has read the histograms
    }

    // selected pixels in increasing order: counts per warp, then a scan over warps and CTAs
    const unsigned lanes_below = (1u << lane) - 1u;
    auto selected = [&](unsigned i) {
        unsigned long long key;
        return key_of(i, key) && take > 0 && (every || key <= kth);
    };
    unsigned mine = 0;
    unsigned long long sel = 0;                    // bit i: pixel of step i is selected (KEEP)
#pragma unroll 4
    for (unsigned i = 0; i < steps; ++i) {
        const bool b = selected(i);
        mine += b;
        if constexpr (KEEP) sel |= (unsigned long long)b << i;
    }
    const unsigned in_warp = __reduce_add_sync(0xffffffffu, mine);
    unsigned total;
    const unsigned upto = cta_scan(lane == 0 ? in_warp : 0u, s_warp, &total);
    unsigned pos = __shfl_sync(0xffffffffu, upto, 0) - in_warp;    // of this warp within the CTA
    if constexpr (CTAS > 1) {
        if (tid == 0) s_total = total;
        cluster.sync();
        pos += __reduce_add_sync(0xffffffffu, lane < rank ? *cluster.map_shared_rank(&s_total, lane) : 0u);
        cluster.sync();                            // the shared totals have been read
    }
    auto put = [&](bool s, unsigned i) {
        const unsigned bal = __ballot_sync(0xffffffffu, s);
        if (s) {
            const unsigned at = pos + __popc(bal & lanes_below), j = first + 32u * i;
            out_idx[at] = (int)j;
            if (out_pts) {
                out_pts[at] = points[j];
                out_pts[(size_t)k + at] = points[(size_t)n + j];
                out_pts[2 * (size_t)k + at] = points[2 * (size_t)n + j];
            }
        }
        pos += __popc(bal);
    };
#pragma unroll 1
    for (unsigned i = 0; i < steps; ++i) put(KEEP ? ((sel >> i) & 1ull) != 0ull : selected(i), i);
    if (rank == 0 && tid == 0) *out_count = (int)take;
}

}  // namespace
}  // namespace pilot

using namespace pilot;

extern "C" pilot_status pilot_sample_anchors(const unsigned char* valid, const float* points, int n_pixels, int n_select,
                                             unsigned long long seed, int* out_idx, float* out_points,
                                             int* out_count, void* stream) {
    if (n_pixels < 0 || n_select < 0) {
        record_error("pilot_sample_anchors: n_pixels and n_select must be >= 0");
        return PILOT_EINVAL;
    }
    if (!out_count || (n_pixels > 0 && !valid) || (n_select > 0 && !out_idx) || (out_points && !points)) {
        record_error("pilot_sample_anchors: valid, out_idx and out_count are required (points with out_points)");
        return PILOT_EINVAL;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kernel, int ctas, bool keep) {
        const int steps = (int)(((long long)n_pixels + ctas * kSampleThreads - 1) / (ctas * kSampleThreads));
        const size_t bytes = keep ? sizeof(unsigned) * kSampleThreads * (size_t)steps : 0;
        if (keep && ctas > 1)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(unsigned) * kSampleThreads * kSampleKeep);
        if (e == cudaSuccess)
            kernel<<<ctas, kSampleThreads, bytes, s>>>(valid, points, n_pixels, n_select, seed, out_idx, out_points, out_count);
    };
    if (n_pixels <= kSampleOne) launch(sample_anchors_kernel<true, 1>, 1, true);
    else if (n_pixels <= kSampleKeep * kSampleCtas * kSampleThreads)
        launch(sample_anchors_kernel<true, kSampleCtas>, kSampleCtas, true);
    else launch(sample_anchors_kernel<false, kSampleCtas>, kSampleCtas, false);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        record_error(cudaGetErrorString(e));
        return PILOT_ECUDA;
    }
    return PILOT_OK;
}
