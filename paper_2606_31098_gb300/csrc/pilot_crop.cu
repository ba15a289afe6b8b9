// TDOM/DSM reference crop on the GPU (Supp. "TDOM/DSM Reference Crop"): the step before
// the pose solver that turns the global maps and a pose prior into a pixel-aligned 2.5D
// reference and its geo-anchors.
//
//   footprint   crop_rays_kernel: one thread-block cluster per image corner; its threads walk the
//               corner ray's samples s_k = s_min + k s_step (metres along the unit ray),
//               read the DSM bilinearly under each, and reduce to the sample whose height is
//               closest to the surface, arg-min |z_ray(s) - h_DSM(x_ray(s), y_ray(s))|
//               (ties: the nearest sample)
//   homography  the origin is the footprint's centroid; the homography mapping the normalised
//               crop square's corners (0,0), (1,0), (1,1), (0,1) to the footprint offsets, in
//               closed form (FP64; one warp of every CTA of the warp kernel)
//   warp + lift crop_warp_kernel: one thread per crop pixel: the homography at the pixel
//               centre gives its map coordinates (the warped coordinate grids); the DSM and the
//               TDOM are read bilinearly there (the same warp for every layer), and the pixel is
//               lifted to the geo-anchor (x - ox, y - oy, D)
//
// Geometry is FP64 throughout (every integer decision is the FP64 one); the map is read in
// place from device memory (an L2/HBM gather of 4 cells per layer and pixel).
//
// What bounds it: the FP64 pipe.  A sub-partition of an SM takes one FP64 warp instruction per 64
// cycles, arithmetic, comparison or conversion, however few lanes it has (a division is about
// ten of them), so the footprint's 32 000 samples and the S^2 pixels are counted in FP64
// instructions, not in bytes.  Hence: quotients by the map's cell size, the crop side and the
// homography's w are products with a reciprocal and a correction by the remainder (one product
// where the divisor is a power of two); conversions, comparisons and truncations are integer
// operations on the FP64 words; the rays' directions come from the host; each ray is spread over
// a 16-CTA cluster; the homography's two rows run on two lanes, without a launch of their own.
// 256^2 crop of a 4096^2 map, with colours: 57.0 us -> 24.0 us (alone under ncu, caches flushed: footprint
// 26.2 -> 10.4, homography 4.7 -> 0, warp 22.9 -> 14.5).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <math.h>

#include "pilot_bits.cuh"
#include "pilot_internal.cuh"

namespace cg = cooperative_groups;

namespace pilot {
namespace {

constexpr int kRayThreads = 128;
constexpr int kRayCluster = 16;     // CTAs per corner ray (a thread-block cluster of the largest size)
constexpr int kWarpMaxThreads = 1024;

// Threads per CTA of crop_warp_kernel for n pixels.  A sub-partition's time is its number of warps
// (the FP64 pipe), and every CTA works the homography out once more, the other warps waiting for
// it: the pixels spread evenly over the SMs in one CTA each, of at least one warp per sub-partition.
// Crops of more warps per SM than a CTA takes run in CTAs of 14 warps, three to an SM by their
// registers, so that one CTA's homography falls into another's pixels.  Whole crop of a 4096^2 map
// in a row of calls, against 448 threads at every size (us): 64^2 23.2 -> 18.4, 96^2 25.0 -> 18.8,
// 128^2 24.2 -> 20.9, 192^2 25.1 -> 25.2, 256^2 25.0 (the same 448), 320^2 35.5 -> 31.2, 384^2
// 47.6 -> 37.5; with 256 threads beyond 394^2, 512^2 54.0, 768^2 115, 2048^2 659; with 448 55.8,
// 113, 648.
int warp_threads(long long n) {
    constexpr int kSms = 152;
    const long long per_sm = ((n + 31) / 32 + kSms - 1) / kSms;
    return per_sm > kWarpMaxThreads / 32 ? 448 : 32 * (int)(per_sm > 4 ? per_sm : 4);
}

// A divisor and its correctly rounded reciprocal; exact: a power of two, whose quotients are
// products with the reciprocal.
struct Divisor {
    double b, inv;
    int exact;
};

struct MapView {
    const float* dsm;
    const unsigned char* tdom;
    int H, W;
    double x0, y0, wmax, hmax;      // wmax, hmax = W - 1, H - 1
    Divisor gsd;
};

// The camera centre and the corners' unit rays, world frame.
struct Rays {
    double C[3], d[4][3];
};

__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ double divide(double a, const Divisor& d) {
    if (d.exact) return a * d.inv;
    if ((__double2hiint(d.inv) & 0x7fffffff) >= 0x7c300000) return a / d.b;   // a reciprocal near overflow
    return quotient(a, d.b, d.inv);
}

// 1 / w to within an ulp for w of moderate size (three FP64 instructions after an FP32 seed, by
// Newton's iteration of third order); the division itself elsewhere.
__device__ __forceinline__ double reciprocal(double w) {
    const float f = narrow(w);
    const unsigned e = (__float_as_uint(f) >> 23) & 0xffu;
    if (e < 32u || e > 222u) return 1.0 / w;
    const double y = widen(1.0f / f);
    const double r = fma(-w, y, 1.0);
    return fma(fma(r, r, r), y, y);
}

// Bilinear read between cell centres at array coordinates (col, row).  The cell is
// (min(floor(col), W - 2), min(floor(row), H - 2)).
struct Cell {
    int c0, r0;
    double ax, ay;
};

// false outside [0, W-1] x [0, H-1]
__device__ __forceinline__ bool find_cell(const MapView& m, double col, double row, Cell* c) {
    if (!(within(col, m.wmax) && within(row, m.hmax))) return false;
    c->c0 = min(whole_part(col), m.W - 2);
    c->r0 = min(whole_part(row), m.H - 2);
    c->ax = col - as_double(c->c0);
    c->ay = row - as_double(c->r0);
    return true;
}

__device__ __forceinline__ double bilinear(double t00, double t01, double t10, double t11, const Cell& c) {
    const double ax = c.ax, ay = c.ay;
    return (1.0 - ay) * ((1.0 - ax) * t00 + ax * t01) + ay * ((1.0 - ax) * t10 + ax * t11);
}

template <typename T>
__device__ __forceinline__ double read_cell(const T* f, int W, int C, int k, const Cell& c) {
    const size_t i00 = ((size_t)c.r0 * W + c.c0) * C + k;
    const size_t i10 = i00 + (size_t)W * C;
    return bilinear(widen(__ldg(f + i00)), widen(__ldg(f + i00 + C)), widen(__ldg(f + i10)), widen(__ldg(f + i10 + C)), c);
}

__device__ __forceinline__ void map_coords(const MapView& m, double x, double y, double* col, double* row) {
    *col = divide(x - m.x0, m.gsd) - 0.5;
    *row = divide(y - m.y0, m.gsd) - 0.5;
}

// geometry layout: H[9], origin[2], quad[12], sample index per corner (as double, -1: none),
// then 1.0 when the crop is valid (27 values + flag)
constexpr int kGeoH = 0, kGeoOrigin = 9, kGeoQuad = 11, kGeoIdx = 23, kGeoOk = 27;

// Smaller distance first, then the nearer sample.  Distances are compared by their words: they
// are not negative, and a NaN's word is above every other.
__device__ __forceinline__ void argmin_merge(unsigned long long& best, int& arg, unsigned long long eo, int ko) {
    if (ko >= 0 && (arg < 0 || eo < best || (eo == best && ko < arg))) {
        best = eo;
        arg = ko;
    }
}

// One cluster of kRayCluster CTAs per image corner: CTA r of the cluster takes the samples
// k = r kRayThreads + tid + j kRayCluster kRayThreads (increasing k per thread), reduces to
// its own arg-min, and CTA 0 merges the cluster's results through distributed shared memory.
__global__ void __launch_bounds__(kRayThreads)
crop_rays_kernel(const MapView m, const __grid_constant__ Rays rays, double s_min, double s_step, int n_samples, double* geometry) {
    __shared__ unsigned long long s_e[kRayThreads / 32];
    __shared__ int s_k[kRayThreads / 32];
    __shared__ unsigned long long blk_e;
    __shared__ int blk_k;
    start_next();
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int corner = blockIdx.x / kRayCluster, lane = threadIdx.x & 31;
    const double* Cw = rays.C;
    const double* d = rays.d[corner];
    unsigned long long best = kInfBits;
    int arg = -1;
    auto merge_warp = [&]() {
        for (int off = 16; off > 0; off >>= 1)
            argmin_merge(best, arg, __shfl_down_sync(0xffffffffu, best, off), __shfl_down_sync(0xffffffffu, arg, off));
    };
    // four samples at a time, their map reads in flight together
    constexpr int kAhead = 4, kStep = kRayCluster * kRayThreads;
    for (int k0 = rank * kRayThreads + threadIdx.x; k0 < n_samples; k0 += kAhead * kStep) {
        Cell c[kAhead];
        bool in[kAhead];
        float h[kAhead][4];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const double t = s_min + as_double(min(k0 + i * kStep, n_samples - 1)) * s_step;
            double col, row;
            map_coords(m, Cw[0] + t * d[0], Cw[1] + t * d[1], &col, &row);
            in[i] = k0 + i * kStep < n_samples && find_cell(m, col, row, &c[i]);
            const float* f = m.dsm + (in[i] ? (size_t)c[i].r0 * m.W + c[i].c0 : 0);
            h[i][0] = __ldg(f);
            h[i][1] = __ldg(f + 1);
            h[i][2] = __ldg(f + m.W);
            h[i][3] = __ldg(f + m.W + 1);
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            if (!in[i]) continue;
            const int k = k0 + i * kStep;
            const double t = s_min + as_double(k) * s_step;
            const double z = bilinear(widen(h[i][0]), widen(h[i][1]), widen(h[i][2]), widen(h[i][3]), c[i]);
            const unsigned long long e = bits(Cw[2] + t * d[2] - z) & 0x7fffffffffffffffull;
            if (e < best) {
                best = e;
                arg = k;
            }
        }
    }
    merge_warp();
    if (lane == 0) {
        s_e[threadIdx.x >> 5] = best;
        s_k[threadIdx.x >> 5] = arg;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kRayThreads / 32; ++w) argmin_merge(best, arg, s_e[w], s_k[w]);
        blk_e = best;
        blk_k = arg;
    }
    cluster.sync();                       // every CTA's result is in its shared memory
    if (rank == 0 && threadIdx.x < 32) {  // lane r reads CTA r's result
        best = kInfBits;
        arg = -1;
        if (lane < kRayCluster) {
            best = *cluster.map_shared_rank(&blk_e, lane);
            arg = *cluster.map_shared_rank(&blk_k, lane);
        }
        merge_warp();
        if (lane == 0) {
            double* q = geometry + kGeoQuad + 3 * corner;
            const double t = s_min + as_double(max(arg, 0)) * s_step;
            for (int i = 0; i < 3; ++i) q[i] = arg < 0 ? 0.0 : Cw[i] + t * d[i];
            geometry[kGeoIdx + corner] = (double)arg;
        }
    }
    cluster.sync();                       // keep the shared results alive until they are read
}

// The homography from the unit square's corners (0,0), (1,0), (1,1), (0,1) to the footprint
// offsets p0..p3 in closed form (the square-to-quadrilateral projective map, Heckbert 1989,
// "Fundamentals of Texture Mapping and Image Warping", Sec. 2.2.3), with H[8] = 1; it is the
// unique homography through the four correspondences, the one the 8 x 8 DLT system defines.
// One warp, all lanes: even lanes compute the x row, odd lanes the y row; lane 0 and 1 write
// them to out[0, 9) and the origin to out[9, 11).  Returns whether the crop is valid.
__device__ __forceinline__ bool crop_geometry(const double* g, double* out) {
    const int lane = threadIdx.x & 31, c = lane & 1;
    bool ok = true;
    for (int k = 0; k < 4; ++k) ok = ok && __double2hiint(g[kGeoIdx + k]) >= 0;      // an index or -1
    double p[4], o = 0.0;
    for (int k = 0; k < 4; ++k) p[k] = g[kGeoQuad + 3 * k + c];
    for (int k = 0; k < 4; ++k) o += p[k];
    o *= 0.25;
    for (int k = 0; k < 4; ++k) p[k] -= o;
    auto of = [](double v, int coord) { return __shfl_sync(0xffffffffu, v, coord); };
    const double s = p[0] - p[1] + p[2] - p[3];
    const double sx = of(s, 0), sy = of(s, 1);
    double gg = 0.0, hh = 0.0, e1, e2;     // e1, e2: a, b on the x row and d, e on the y row
    if (sx == 0.0 && sy == 0.0) {          // a parallelogram: affine
        e1 = p[1] - p[0];
        e2 = p[3] - p[0];
    } else {
        const double d1 = p[1] - p[2], d2 = p[3] - p[2];
        const double dx1 = of(d1, 0), dx2 = of(d2, 0), dy1 = of(d1, 1), dy2 = of(d2, 1);
        const double den = dx1 * dy2 - dx2 * dy1;
        if (den == 0.0) ok = false;
        // g on even lanes, h on odd ones
        const double num = c == 0 ? sx * dy2 - dx2 * sy : dx1 * sy - sx * dy1;
        const double v = ok ? num / den : 0.0;
        gg = of(v, 0);
        hh = of(v, 1);
        e1 = p[1] - p[0] + gg * p[1];
        e2 = p[3] - p[0] + hh * p[3];
    }
    if (lane < 2) {
        out[3 * c] = ok ? e1 : 0.0;
        out[3 * c + 1] = ok ? e2 : 0.0;
        out[3 * c + 2] = ok ? p[0] : 0.0;
        out[6 + c] = ok ? (c ? hh : gg) : 0.0;
        out[9 + c] = ok ? o : 0.0;
        if (c == 0) out[8] = ok ? 1.0 : 0.0;
    }
    return ok;
}

__global__ void __launch_bounds__(kWarpMaxThreads)
crop_warp_kernel(const MapView m, int S, const Divisor side, double* geometry, float* points, unsigned char* valid,
                 float* rgb) {
    __shared__ double H[11];
    __shared__ int s_ok;
    const long long NP = (long long)S * S;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    // pixel centres (2 i + 1) / 2: an exact conversion, halved exactly (S^2 <= 2^26)
    const int u = (int)((unsigned)j % (unsigned)S), v = (int)((unsigned)j / (unsigned)S);
    auto half_past = [](int i) {
        const double t = widen((float)(2 * i + 1));
        return __hiloint2double(__double2hiint(t) - 0x100000, __double2loint(t));
    };
    const double a = divide(half_past(u), side), b = divide(half_past(v), side);
    wait_previous();
    if (threadIdx.x < 32) {
        const bool g = crop_geometry(geometry, H);
        __syncwarp();
        if (threadIdx.x == 0) s_ok = g;
        if (blockIdx.x == 0) {
            if (threadIdx.x < 9) geometry[kGeoH + threadIdx.x] = H[threadIdx.x];
            else if (threadIdx.x < 11) geometry[kGeoOrigin + threadIdx.x - 9] = H[threadIdx.x];
            else if (threadIdx.x == 11) geometry[kGeoOk] = g ? 1.0 : 0.0;
        }
    }
    __syncthreads();
    if (j >= NP) return;
    bool ok = s_ok != 0;
    double dx = 0.0, dy = 0.0, h = 0.0;
    Cell cell{};
    if (ok) {
        const double w = H[6] * a + H[7] * b + H[8], inv = reciprocal(w);
        dx = quotient(H[0] * a + H[1] * b + H[2], w, inv);
        dy = quotient(H[3] * a + H[4] * b + H[5], w, inv);
        double col, row;
        map_coords(m, H[9] + dx, H[10] + dy, &col, &row);
        ok = __double2hiint(w) > 0 && find_cell(m, col, row, &cell);
        if (ok) h = read_cell(m.dsm, m.W, 1, 0, cell);
    }
    valid[j] = ok ? 1 : 0;
    points[j] = ok ? narrow(dx) : 0.0f;
    points[NP + j] = ok ? narrow(dy) : 0.0f;
    points[2 * NP + j] = ok ? narrow(h) : 0.0f;
    if (rgb)
        for (int k = 0; k < 3; ++k)
            rgb[3 * j + k] = ok && m.tdom ? narrow(read_cell(m.tdom, m.W, 3, k, cell)) : 0.0f;
}

Divisor divisor(double b) {
    int e;
    const double inv = 1.0 / b;
    return Divisor{b, inv, frexp(b, &e) == 0.5 && inv > 1e-290 && inv < 1e290 ? 1 : 0};
}

// The camera centre -R^T t and the unit rays R^T K^-1 (u, v, 1) through the image corners.
Rays corner_rays(const pilot_crop_params& p) {
    Rays r;
    const double* T = p.T_cw;
    for (int i = 0; i < 3; ++i) r.C[i] = -fma(T[8 + i], T[11], fma(T[4 + i], T[7], T[i] * T[3]));
    for (int corner = 0; corner < 4; ++corner) {
        const double u = (corner == 1 || corner == 2) ? (double)p.img_w : 0.0;
        const double v = (corner >= 2) ? (double)p.img_h : 0.0;
        const double dc[3] = {(u - p.cx) / p.fx, (v - p.cy) / p.fy, 1.0};
        double* d = r.d[corner];
        for (int i = 0; i < 3; ++i) d[i] = fma(T[8 + i], dc[2], fma(T[4 + i], dc[1], T[i] * dc[0]));
        const double n = sqrt(fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])));
        for (int i = 0; i < 3; ++i) d[i] /= n;
    }
    return r;
}

pilot_status crop_fail(pilot_status st, const char* m) {
    record_error(m);
    return st;
}

}  // namespace
}  // namespace pilot

using namespace pilot;

extern "C" pilot_status pilot_crop_reference(const pilot_map* map, const pilot_crop_params* p, float* points,
                                             unsigned char* valid, float* rgb, double* geometry, void* stream) {
    if (!map || !p) return crop_fail(PILOT_EINVAL, "map or params is NULL");
    if (!map->dsm) return crop_fail(PILOT_EINVAL, "the map has no DSM");
    if (map->H < 2 || map->W < 2 || !(map->gsd > 0.0)) return crop_fail(PILOT_EINVAL, "map must be at least 2 x 2 with gsd > 0");
    if (p->S < 1 || p->S > 8192) return crop_fail(PILOT_EINVAL, "crop side S must be in [1, 8192]");
    if (p->n_samples < 1 || p->n_samples > (1 << 22)) return crop_fail(PILOT_EINVAL, "n_samples must be in [1, 4194304]");
    if (!(p->s_step > 0.0) || !(p->fx > 0.0) || !(p->fy > 0.0) || p->img_w < 1 || p->img_h < 1)
        return crop_fail(PILOT_EINVAL, "s_step, fx, fy and the image size must be positive");
    if (!points || !valid || !geometry) return crop_fail(PILOT_EINVAL, "points, valid or geometry is NULL");
    if (((uintptr_t)geometry & 7) != 0 || ((uintptr_t)points & 3) != 0 || (rgb && ((uintptr_t)rgb & 3) != 0))
        return crop_fail(PILOT_EINVAL, "outputs must be naturally aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const MapView m{map->dsm, map->tdom, map->H, map->W, map->x0, map->y0, map->W - 1.0, map->H - 1.0,
                    divisor(map->gsd)};
    const long long NP = (long long)p->S * p->S;
    // the footprint: a cluster of more than 8 CTAs has to be asked for
    cudaError_t e = cudaFuncSetAttribute(crop_rays_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (e == cudaSuccess) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kRayCluster;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(4 * kRayCluster);
        cfg.blockDim = dim3(kRayThreads);
        e = cudaLaunchKernelEx(&cfg, crop_rays_kernel, m, corner_rays(*p), p->s_min, p->s_step, p->n_samples, geometry);
    }
    if (e == cudaSuccess) {
        // may start while the footprint runs; it waits for it before it reads its results
        attr[0] = cudaLaunchAttribute{};
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        const int threads = warp_threads(NP);
        cfg.gridDim = dim3((unsigned)((NP + threads - 1) / threads));
        cfg.blockDim = dim3(threads);
        e = cudaLaunchKernelEx(&cfg, crop_warp_kernel, m, p->S, divisor(p->S), geometry, points, valid, rgb);
    }
    if (e != cudaSuccess) return crop_fail(PILOT_ECUDA, cudaGetErrorString(e));
    return PILOT_OK;
}
