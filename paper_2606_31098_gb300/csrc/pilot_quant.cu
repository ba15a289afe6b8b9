// Feature quantiser: FP32 rows of C channels -> BF16 / FP16 / FP8-E4M3 storage with one
// FP32 scale per channel, stored value = round(x / s_c), value used = stored x s_c.
//
//   s_c = absmax_c / q_max   (q_max = 448 for E4M3; 65504 for FP16; 1 for BF16, i.e. unit
//                             absmax) when per-channel scaling is requested or the storage
//                             is E4M3; otherwise s_c = 1.
//   rounding: to nearest, ties to even; E4M3 saturates to +-448 (no infinities in E4M3).
//
// The absmax is reduced into the caller's scale array (as the bit patterns of the
// non-negative floats, whose unsigned order is their numeric order); the conversion derives the
// scales from it, and a last one-block launch turns the array into the scales in place: no
// memory is allocated.  Without scaling (unscaled BF16 / FP16) there is one launch only.
//
// What bounds it: HBM and L2 (the conversion re-reads a map that fits the 129 MB L2), and at a
// map's size still the launches.  480 x 640 x 32 FP32 to FP8: 28.7 us in a row of calls (31 to 33
// alone) with four shared-memory atomics per 16 bytes, a division per element and byte stores;
// 20.5 us (25 to 28 alone) with running maxima in registers (a thread's channels stay the same: its
// stride is a multiple of C), one reciprocal per channel, packed conversions and programmatic
// dependent launches.  As many values in 48 channels 27.2 -> 25.1 us, in 12 32.9 -> 20.5, in 2048
// 37.1 -> 18.6.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <string>

#include "pilot_internal.cuh"

namespace pilot {
namespace {

constexpr int kQuantThreads = 256;
constexpr int kQuantUnroll = 4;      // 16-byte loads in flight per thread

// Waits for the launch before this one in the stream (launched while it still ran).
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Both passes: `stride` threads work (the launch's, less a remainder), a multiple of C / 4, each
// taking every stride-th vector of four values, so that its four channels never change.

// The maxima are kept in registers.
__global__ void __launch_bounds__(kQuantThreads)
absmax_kernel(const float* __restrict__ src, long long rows, int C, long long stride, unsigned* __restrict__ bits) {
    extern __shared__ unsigned smax[];
    start_next();
    for (int c = threadIdx.x; c < C; c += blockDim.x) smax[c] = 0u;
    __syncthreads();
    const long long n4 = rows * C / 4;
    const uint4* s4 = reinterpret_cast<const uint4*>(src);
    const long long k0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    uint4 m = make_uint4(0u, 0u, 0u, 0u);
    auto take = [&](const uint4& v) {
        m.x = max(m.x, v.x & 0x7fffffffu);
        m.y = max(m.y, v.y & 0x7fffffffu);
        m.z = max(m.z, v.z & 0x7fffffffu);
        m.w = max(m.w, v.w & 0x7fffffffu);
    };
    long long k = k0 < stride ? k0 : n4;
    for (; k + (kQuantUnroll - 1) * stride < n4; k += kQuantUnroll * stride) {
        uint4 v[kQuantUnroll];
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) v[u] = __ldg(s4 + k + u * stride);
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) take(v[u]);
    }
    for (; k < n4; k += stride) take(__ldg(s4 + k));
    // lanes that hold the same channels (uniform over the warp), then one atomic per channel
    int holders = 32;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if ((4 * o) % C != 0) break;
        m.x = max(m.x, __shfl_xor_sync(0xffffffffu, m.x, o));
        m.y = max(m.y, __shfl_xor_sync(0xffffffffu, m.y, o));
        m.z = max(m.z, __shfl_xor_sync(0xffffffffu, m.z, o));
        m.w = max(m.w, __shfl_xor_sync(0xffffffffu, m.w, o));
        holders = o;
    }
    if ((int)(threadIdx.x & 31) < holders) {
        const int c = (int)(4u * (unsigned)k0 % (unsigned)C);
        atomicMax(&smax[c], m.x);
        atomicMax(&smax[c + 1], m.y);
        atomicMax(&smax[c + 2], m.z);
        atomicMax(&smax[c + 3], m.w);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < C; c += blockDim.x)
        if (smax[c] != 0u) atomicMax(bits + c, smax[c]);
}

// The scale of a channel whose absmax has these bits.
__device__ __forceinline__ float scale_of(unsigned bits, float qmax, int use_absmax) {
    const float amax = __uint_as_float(bits);
    return (use_absmax && amax > 0.0f && isfinite(amax)) ? amax / qmax : 1.0f;
}

__global__ void scales_kernel(float* scale, int C, float qmax, int use_absmax) {
    wait_previous();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < C) scale[c] = scale_of(reinterpret_cast<unsigned*>(scale)[c], qmax, use_absmax);
}

// Four values as stored: 8 bytes (16-bit types) or 4 (FP8).
template <pilot_dtype DT>
__device__ __forceinline__ void store4(void* dst, long long k, bool wide, float y0, float y1, float y2, float y3) {
    if constexpr (DT == PILOT_FP8E4M3) {
        const unsigned lo = __nv_cvt_float2_to_fp8x2(make_float2(y0, y1), __NV_SATFINITE, __NV_E4M3);
        const unsigned hi = __nv_cvt_float2_to_fp8x2(make_float2(y2, y3), __NV_SATFINITE, __NV_E4M3);
        static_cast<unsigned*>(dst)[k] = lo | (hi << 16);
    } else {
        uint2 o;
        if constexpr (DT == PILOT_BF16) {
            const __nv_bfloat162 a = __floats2bfloat162_rn(y0, y1), b = __floats2bfloat162_rn(y2, y3);
            memcpy(&o.x, &a, 4);
            memcpy(&o.y, &b, 4);
        } else {
            const __half2 a = __floats2half2_rn(y0, y1), b = __floats2half2_rn(y2, y3);
            memcpy(&o.x, &a, 4);
            memcpy(&o.y, &b, 4);
        }
        if (wide) {
            static_cast<uint2*>(dst)[k] = o;
        } else {                         // dst is only 4-byte aligned
            static_cast<unsigned*>(dst)[2 * k] = o.x;
            static_cast<unsigned*>(dst)[2 * k + 1] = o.y;
        }
    }
}

// SCALED: the scales derived from the absmax bits in `scale` (by absmax_kernel); else the values
// as they are, and `scale` is set to ones.
template <pilot_dtype DT, bool SCALED>
__global__ void __launch_bounds__(kQuantThreads, 6)
convert_kernel(const float* __restrict__ src, long long rows, int C, long long stride, float* scale, float qmax,
               void* __restrict__ dst) {
    start_next();
    const long long n4 = rows * C / 4;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    const long long k0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool wide = ((uintptr_t)dst & 7) == 0;
    if constexpr (!SCALED) {
        if (blockIdx.x == 0)
            for (int c = threadIdx.x; c < C; c += blockDim.x) scale[c] = 1.0f;
    } else {
        wait_previous();
    }
    // the products are with the reciprocals of the scales
    float i0 = 1.0f, i1 = 1.0f, i2 = 1.0f, i3 = 1.0f;
    if constexpr (SCALED) {
        const unsigned* bits = reinterpret_cast<const unsigned*>(scale) + 4u * (unsigned)k0 % (unsigned)C;
        auto inverse = [&](int c) { return 1.0f / scale_of(__ldcg(bits + c), qmax, 1); };
        i0 = inverse(0), i1 = inverse(1), i2 = inverse(2), i3 = inverse(3);
    }
    auto convert = [&](long long k, const float4& v) {
        if constexpr (SCALED) store4<DT>(dst, k, wide, v.x * i0, v.y * i1, v.z * i2, v.w * i3);
        else store4<DT>(dst, k, wide, v.x, v.y, v.z, v.w);
    };
    long long k = k0 < stride ? k0 : n4;
    for (; k + (kQuantUnroll - 1) * stride < n4; k += kQuantUnroll * stride) {
        float4 v[kQuantUnroll];
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) v[u] = __ldg(s4 + k + u * stride);
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) convert(k + u * stride, v[u]);
    }
    for (; k < n4; k += stride) convert(k, __ldg(s4 + k));
}

int grid_for(long long n4, int per_sm) {
    long long b = (n4 + kQuantThreads - 1) / kQuantThreads;
    if (b > 152 * per_sm) b = 152 * per_sm;
    return b < 1 ? 1 : (int)b;
}

// The threads of `grid` CTAs that take part: a multiple of C / 4, and of 8 too (whole 128-byte lines
// per step) where that leaves most of them.
long long stride_for(int grid, int C) {
    const long long threads = (long long)grid * kQuantThreads, quads = C / 4, lines = 8 * quads;
    return threads >= 8 * lines ? threads / lines * lines : threads / quads * quads;
}

// One launch that may begin while the kernel before it in the stream still runs; the kernels
// launched so (the scaled conversion, the scales) wait for that one before they touch memory.
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <pilot_dtype DT>
cudaError_t launch_convert(const float* src, long long rows, int C, bool scaled, float* scale, float qmax, void* dst,
                           cudaStream_t s) {
    const int grid = grid_for(rows * C / 4, 6);    // one wave
    if (!scaled) {
        convert_kernel<DT, false><<<grid, kQuantThreads, 0, s>>>(src, rows, C, (long long)grid * kQuantThreads, scale, qmax, dst);
        return cudaGetLastError();
    }
    return launch_after(convert_kernel<DT, true>, grid, kQuantThreads, 0, s, src, rows, C, stride_for(grid, C), scale, qmax,
                        dst);
}

pilot_status qfail(pilot_status st, const std::string& m) {
    record_error(m.c_str());
    return st;
}

}  // namespace
}  // namespace pilot

using namespace pilot;

extern "C" pilot_status pilot_quantize_features(const float* src, long long rows, int C,
                                                pilot_dtype dtype, int per_channel, void* dst,
                                                float* scale, void* stream) {
    if (!src || !dst || !scale) return qfail(PILOT_EINVAL, "src, dst or scale is NULL");
    if (rows < 0 || C < 4 || C % 4 != 0 || C > 4096) return qfail(PILOT_EINVAL, "rows >= 0 and C a multiple of 4 in [4, 4096]");
    if (dtype != PILOT_BF16 && dtype != PILOT_F16 && dtype != PILOT_FP8E4M3)
        return qfail(PILOT_EINVAL, "dtype must be BF16, F16 or FP8E4M3");
    if (((uintptr_t)src & 15) != 0) return qfail(PILOT_EINVAL, "src must be 16-byte aligned");
    if (((uintptr_t)dst & 3) != 0) return qfail(PILOT_EINVAL, "dst must be 4-byte aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const long long n4 = rows * C / 4;
    const bool use_absmax = per_channel != 0 || dtype == PILOT_FP8E4M3;
    const float qmax = dtype == PILOT_FP8E4M3 ? 448.0f : (dtype == PILOT_F16 ? 65504.0f : 1.0f);
    cudaError_t e = cudaSuccess;
    // absmax: four CTAs per SM (each adds one atomic per channel at its end)
    if (use_absmax || n4 == 0) e = cudaMemsetAsync(scale, 0, sizeof(float) * C, s);
    if (e == cudaSuccess && use_absmax && n4 > 0) {
        const int grid = grid_for(n4, 4);
        absmax_kernel<<<grid, kQuantThreads, sizeof(unsigned) * C, s>>>(src, rows, C, stride_for(grid, C),
                                                                        reinterpret_cast<unsigned*>(scale));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && n4 > 0) {
        if (dtype == PILOT_BF16) e = launch_convert<PILOT_BF16>(src, rows, C, use_absmax, scale, qmax, dst, s);
        else if (dtype == PILOT_F16) e = launch_convert<PILOT_F16>(src, rows, C, use_absmax, scale, qmax, dst, s);
        else e = launch_convert<PILOT_FP8E4M3>(src, rows, C, use_absmax, scale, qmax, dst, s);
    }
    if (e == cudaSuccess && n4 == 0) {
        scales_kernel<<<(C + 127) / 128, 128, 0, s>>>(scale, C, qmax, 0);
        e = cudaGetLastError();
    } else if (e == cudaSuccess && use_absmax) {
        e = launch_after(scales_kernel, (C + 127) / 128, 128, 0, s, scale, C, qmax, 1);
    }
    if (e != cudaSuccess) return qfail(PILOT_ECUDA, std::string("quantiser launch: ") + cudaGetErrorString(e));
    return PILOT_OK;
}
