// Build pass: for one level, every (anchor tile, tile of hypotheses) evaluates the photo
// term of the objective and its normal equations at the hypotheses' candidate poses.
//
//   Eq. 1  r_j = f^q(pi(K_l, T, P_j)) - f^r(p_j)   (bilinear read of C channels)
//   Eq. 2  cost += rho(w_j ||r_j||^2)              (Huber on the squared norm)
//   Eq. 8  H += w_j rho' J_j^T J_j, g += w_j rho' J_j^T r_j
//
// with J_j = G_j A_j: G_j (C x 2) the analytic gradient of the bilinear interpolant and
// A_j (2 x 6) = d(u,v)/dp [I | -[p]x] the projection Jacobian times the se(3)
// generators (left perturbation, camera frame).  The dense C x 6 Jacobian is never
// formed: per anchor only the 2x2 Gram matrix M = G^T G, b = G^T r and s = ||r||^2 are
// summed over channels, then H_j = w A^T M A and g_j = w A^T b.
//
// Thread mapping.  A CTA holds kHypTile (HT) hypotheses over one anchor tile.  A group of
// LP consecutive lanes reads one tap with one load per lane, 32 bytes for FP32 and 16-bit
// maps and 16 bytes for FP8 and for maps with per-channel scales (LP = C x element size /
// load width, at most 8: 4 lanes for FP32 at C = 32, 2 for BF16, 2 for FP8), i.e. one L1
// wavefront per record and tap, where a record is one (anchor, hypothesis) pair.  A group works on LP
// records at a time: APB anchors under HG = min(HT, LP) hypotheses (APB HG = LP); with
// LP < HT, HT / HG neighbouring groups take the same anchors under the other hypotheses.
// Each lane projects one record (lane q of the group: anchor q mod APB under the group's
// hypothesis q div APB) and broadcasts its tap offset and bilinear weights to the group; the
// group then reads the 4 taps of every record and the reference row of every anchor
// together -- once for all the hypotheses of the CTA (vector k of lane q holds channels
// VW (q + k LP) .. + VW).  A butterfly reduce-scatter over the group leaves in lane q the
// channel sums of record q, and each lane finishes its own record (Huber weight, A, 21 + 6
// sums) exactly once.  An invisible record's partial sums stay in its own reduce-scatter
// slot and are discarded by its owner.  The hypothesis slot of a lane is read from lane bits
// log2 APB .. log2 (APB HT) - 1; the CTA reduces the lanes of each slot over the other lane
// bits, then the warps, in a fixed order.  A hypothesis' sums do not depend on which slot
// it takes or on the other hypotheses (the lanes of all slots run the same anchors in the
// same order, and the reduction trees are translates of one another), so the result is
// deterministic and independent of the grid shape and of how hypotheses are grouped.
//
// What bounds it: issue and the latency of the L1 gathers, at two CTAs (16 warps) per SM, which 128
// registers allow; the frame's maps stay in L2, and DRAM is idle.  So the taps and reference rows
// stay in registers as they were loaded and are widened where they are used, and two records of an
// anchor whose hypotheses agree to a pixel -- most, once a solve converges -- share one cell's
// loads and tap differences (64 hypotheses x 65536 anchors: a solve 4158 -> 3738 us, one
// evaluation 163.8 -> 156.5 us; uneven BF16 batch 15.06 -> 13.60 ms).  Not faster: a third or
// fourth CTA per SM with the sums in tensor memory (solve 4.3 - 4.6 ms, read-modify-write of 29
// words per record), the same with the loads of a cell shared by all four hypotheses (4.2 ms), the
// shared taps held for the second pair (4.1 ms, spills), L1 prefetches a batch ahead (no change).
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "pilot_fp64.cuh"
#include "pilot_internal.cuh"

namespace pilot {

template <pilot_dtype DT> struct Storage;
template <> struct Storage<PILOT_F32> { using T = float; static constexpr int VEC = 8; };   // 32-byte loads
template <> struct Storage<PILOT_BF16> { using T = uint16_t; static constexpr int VEC = 16; };  // 32-byte loads
template <> struct Storage<PILOT_F16> { using T = uint16_t; static constexpr int VEC = 16; };
template <> struct Storage<PILOT_FP8E4M3> { using T = uint8_t; static constexpr int VEC = 16; };

// W (4, 8 or 16) consecutive channels at p as they are stored (one load of W elements: 4 to 32
// bytes).
template <pilot_dtype DT, int W> struct RawVec {
    static constexpr int NW = W * (int)sizeof(typename Storage<DT>::T) / 4;
    uint32_t w[NW];
};

template <pilot_dtype DT, int W>
__device__ __forceinline__ void load_raw(const typename Storage<DT>::T* p, RawVec<DT, W>& o) {
    constexpr int NW = RawVec<DT, W>::NW;
    static_assert(NW == 1 || NW == 2 || NW == 4 || NW == 8, "vector width");
    if constexpr (NW == 8) {
        // one 256-bit load (32-byte aligned: device feature pointers are validated for it)
        asm("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(o.w[0]), "=r"(o.w[1]), "=r"(o.w[2]), "=r"(o.w[3]), "=r"(o.w[4]), "=r"(o.w[5]), "=r"(o.w[6]),
              "=r"(o.w[7])
            : "l"(p));
    } else if constexpr (NW == 4) {
        asm("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
            : "=r"(o.w[0]), "=r"(o.w[1]), "=r"(o.w[2]), "=r"(o.w[3]) : "l"(p));
    } else if constexpr (NW == 2) {
        asm("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(o.w[0]), "=r"(o.w[1]) : "l"(p));
    } else {
        asm("ld.global.nc.u32 %0, [%1];" : "=r"(o.w[0]) : "l"(p));
    }
}

// One row of a pose (16-byte aligned), by a volatile load: a loop reads it again in every pass
// instead of holding it in registers.
__device__ __forceinline__ void load_row(const float* p, float& x, float& y, float& z, float& t) {
    asm volatile("ld.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x), "=f"(y), "=f"(z), "=f"(t) : "l"(p));
}

// Channels e and e + 1 (e even) widened to FP32.
template <pilot_dtype DT, int W>
__device__ __forceinline__ void raw_pair(const RawVec<DT, W>& v, int e, float& lo, float& hi) {
    if constexpr (DT == PILOT_F32) {
        lo = __uint_as_float(v.w[e]);
        hi = __uint_as_float(v.w[e + 1]);
    } else if constexpr (DT == PILOT_BF16) {
        // bfloat16 is the upper half of an IEEE binary32: widening is a 16-bit shift
        lo = __uint_as_float(v.w[e / 2] << 16);
        hi = __uint_as_float(v.w[e / 2] & 0xffff0000u);
    } else if constexpr (DT == PILOT_F16) {
        __half2 h;
        memcpy(&h, &v.w[e / 2], 4);
        const float2 f = __half22float2(h);
        lo = f.x;
        hi = f.y;
    } else {
        const __half2_raw h =
            __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)((v.w[e / 4] >> (8 * (e & 2))) & 0xffffu), __NV_E4M3);
        const float2 f = __half22float2(__half2(h));
        lo = f.x;
        hi = f.y;
    }
}

// ---- two channels per instruction: packed FP32x2 arithmetic (each lane of the pair is
// rounded exactly like the scalar operation) ----
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Six sums over channel pairs: lane .lo of each accumulates even channels, .hi odd ones.
struct ChanSums2 {
    f2 s, m00, m01, m11, b0, b1;
};

// Two channels at once.  The differences of the taps of a cell ...
struct CellDiffs {
    f2 t00, bq, cq, dq;
};
__device__ __forceinline__ CellDiffs cell_diffs(f2 t00, f2 t01, f2 t10, f2 t11) {
    const f2 bq = sub2(t01, t00);                    // d/dx along the upper row
    const f2 cq = sub2(t10, t00);                    // d/dy along the left column
    return CellDiffs{t00, bq, cq, sub2(sub2(t11, t10), bq)};   // bilinear cross term
}
// ... and the value, in-cell gradient, residual (fr: the reference value, scaled) and six sums of
// one position in it.
template <bool SCALED>
__device__ __forceinline__ void channel_pair(ChanSums2& a, const CellDiffs& d, f2 fr, f2 ax, f2 ay, f2 sq) {
    f2 fu = fma2(d.dq, ay, d.bq);                    // df/du inside the cell
    f2 fv = fma2(d.dq, ax, d.cq);                    // df/dv inside the cell
    f2 f = fma2(ax, fu, fma2(ay, d.cq, d.t00));
    if constexpr (SCALED) {
        f = mul2(f, sq);
        fu = mul2(fu, sq);
        fv = mul2(fv, sq);
    }
    const f2 r = sub2(f, fr);
    a.s = fma2(r, r, a.s);
    a.m00 = fma2(fu, fu, a.m00);
    a.m01 = fma2(fu, fv, a.m01);
    a.m11 = fma2(fv, fv, a.m11);
    a.b0 = fma2(fu, r, a.b0);
    a.b1 = fma2(fv, r, a.b1);
}

__device__ __forceinline__ float hsum(f2 v) {
    float lo, hi;
    upk(v, lo, hi);
    return lo + hi;
}

// Lane layout of the build pass for C channels stored as DT (see the top of the file): LP
// lanes per tap = records per group batch, HG hypotheses per group, NS = kHypTile / HG
// groups over the same anchors, APB anchors per group batch.  The slot of lane l is
// (l / APB) mod kHypTile.  Maps with per-channel scales keep 16-byte loads: the wider lane
// share of channels would hold twice the scale registers and spill.
template <pilot_dtype DT, int C, bool SCALED> struct GroupShape {
    static constexpr int VEC = SCALED ? 16 / (int)sizeof(typename Storage<DT>::T) : Storage<DT>::VEC;  // per load
    static constexpr int VW = (C < VEC) ? C : VEC;            // channels per vector load
    static constexpr int LP = (C / VW < 8) ? C / VW : 8;      // lanes per tap
    static constexpr int HG = LP < kHypTile ? LP : kHypTile;  // hypotheses per group
    static constexpr int NS = kHypTile / HG;                  // groups over the same anchors
    static constexpr int APB = LP / HG;                       // anchors per group batch
    static constexpr int NV = C / LP / VW;                    // vector loads per lane and tap
    static_assert(APB * kHypTile <= 32, "a warp holds every slot of an anchor");
};

// The CTA's hypotheses: their FP32 poses and whether each slot has one to evaluate.
struct SlotPoses {
    const float* p[kHypTile];
    bool act[kHypTile];
};

// The level-specific inputs of the anchor loop.
struct LevelView {
    const float* px;
    const float* py;
    const float* pz;
    const float* weight;
    const uint8_t* valid;
    const void* qry;
    const void* ref;
    const float* qscale;
    const float* rscale;
    const float* conf;
    int H, W;
    float fx, fy, cx, cy, huber;
};

__device__ __forceinline__ LevelView level_view(const BuildParams& p) {
    return LevelView{p.px, p.py, p.pz, p.weight, p.valid, p.qry, p.ref, p.qscale, p.rscale, p.conf,
                     p.H, p.W, p.fx, p.fy, p.cx, p.cy, p.huber};
}

// The 4 taps of one record in this lane's channels (vector k covers VW (q + k LP) .. + VW).
template <pilot_dtype DT, int C, bool SCALED> struct TapBuf {
    using G = GroupShape<DT, C, SCALED>;
    RawVec<DT, G::VW> t[G::NV][4];

    __device__ __forceinline__ void load(const typename Storage<DT>::T* t00, int WC, int q) {
#pragma unroll
        for (int k = 0; k < G::NV; ++k) {
            const typename Storage<DT>::T* p = t00 + G::VW * (q + k * G::LP);
            load_raw<DT, G::VW>(p, t[k][0]);
            load_raw<DT, G::VW>(p + C, t[k][1]);
            load_raw<DT, G::VW>(p + WC, t[k][2]);
            load_raw<DT, G::VW>(p + WC + C, t[k][3]);
        }
    }
};

// This lane's channels of one anchor's reference row.
template <pilot_dtype DT, int C, bool SCALED> struct RefBuf {
    using G = GroupShape<DT, C, SCALED>;
    RawVec<DT, G::VW> r[G::NV];

    __device__ __forceinline__ void load(const typename Storage<DT>::T* row, int q) {
#pragma unroll
        for (int k = 0; k < G::NV; ++k) load_raw<DT, G::VW>(row + G::VW * (q + k * G::LP), r[k]);
    }
};

// Channel sums of R records of one cell over this lane's channels: the 4 taps against the anchor's
// reference values: bilinear value and in-cell gradient at each record's (ax, ay), residual, and
// the six partial sums p[record].
template <pilot_dtype DT, int C, bool SCALED, int R>
__device__ __forceinline__ void record_partials(const TapBuf<DT, C, SCALED>& b, const RefBuf<DT, C, SCALED>& rr,
                                                const float (&ax)[R], const float (&ay)[R], const float* qs,
                                                const float* rs, float (*p)[6]) {
    using G = GroupShape<DT, C, SCALED>;
    constexpr int VW = G::VW;
    const f2 z2 = pk(0.f, 0.f);
    f2 ax2[R], ay2[R];
    ChanSums2 cs[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        ax2[i] = pk(ax[i], ax[i]);
        ay2[i] = pk(ay[i], ay[i]);
        cs[i] = ChanSums2{z2, z2, z2, z2, z2, z2};
    }
#pragma unroll
    for (int k = 0; k < G::NV; ++k) {
#pragma unroll
        for (int e = 0; e < VW; e += 2) {
            float a[4][2], r[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) raw_pair<DT, VW>(b.t[k][i], e, a[i][0], a[i][1]);
            raw_pair<DT, VW>(rr.r[k], e, r[0], r[1]);
            const CellDiffs d = cell_diffs(pk(a[0][0], a[0][1]), pk(a[1][0], a[1][1]), pk(a[2][0], a[2][1]), pk(a[3][0], a[3][1]));
            f2 fr = pk(r[0], r[1]);
            const f2 sq = pk(qs[k * VW + e], qs[k * VW + e + 1]);
            if constexpr (SCALED) fr = mul2(fr, pk(rs[k * VW + e], rs[k * VW + e + 1]));
#pragma unroll
            for (int i = 0; i < R; ++i) channel_pair<SCALED>(cs[i], d, fr, ax2[i], ay2[i], sq);
        }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
        p[i][0] = hsum(cs[i].s);
        p[i][1] = hsum(cs[i].m00);
        p[i][2] = hsum(cs[i].m01);
        p[i][3] = hsum(cs[i].m11);
        p[i][4] = hsum(cs[i].b0);
        p[i][5] = hsum(cs[i].b1);
    }
}

// Whether reading the pose again per batch (REREAD, below) may pay: not where one lane reads a 32-byte
// tap of 16 channels by itself (uneven batch, confidence maps: BF16 2152 us with it, 2057 without).
template <pilot_dtype DT, int C, bool SCALED>
constexpr bool kPoseReread = !(GroupShape<DT, C, SCALED>::LP == 1 && C == 16);

// Accumulate anchors [j_begin, j_end) under the CTA's kHypTile hypotheses into this lane's
// 29 sums (the lane's own slot, see GroupShape).  sp: the slots' poses (12 FP32 values each)
// and whether each has a pose to evaluate (an inactive slot's lanes finish nothing).  Every
// thread of the CTA calls it with the same arguments; threads are grouped as described at
// the top of the file.
// PREFETCH: read the next batch's anchor coordinates one batch ahead (four more registers
// through the loop; the sums are the same either way).  FRESH_TID: read the thread index
// through a volatile move, so that the lane layout derived from it is recomputed at each call
// instead of being hoisted into an enclosing loop and held across that loop's function calls.
// REREAD: read the pose again for every batch (three 16-byte loads) instead of holding it in
// twelve registers through the gathers.  Held against read again, 64 hypotheses x 65536 anchors:
// 16-bit maps 3739 -> 3703 us a solve, an uneven batch 13.54 -> 13.31 ms, eight frames of the
// paper's schedule 1212 -> 1160 us; FP32 evaluation 158.5 -> 153.6 us, but FP32 solves 3824 ->
// 3846 us and FP8 ones 4433 -> 4480 us, which therefore hold it.
template <pilot_dtype DT, int C, bool SCALED, bool CONF, int NTHREADS, bool PREFETCH = true, bool FRESH_TID = false,
          bool REREAD = (DT == PILOT_BF16 || DT == PILOT_F16) && kPoseReread<DT, C, SCALED>>
__device__ __forceinline__ void accumulate_anchors(const LevelView& v, const SlotPoses& sp, int j_begin, int j_end,
                                                   float* acc) {
    using Elem = typename Storage<DT>::T;
    using G = GroupShape<DT, C, SCALED>;
    constexpr int VW = G::VW, LP = G::LP, HG = G::HG, NS = G::NS, APB = G::APB, NV = G::NV;
    constexpr int CPL = C / LP;                      // channels per lane
    constexpr int ASTEP = NTHREADS / (LP * NS) * APB;   // anchors per CTA batch
    static_assert(C % 4 == 0 && C >= 4 && C <= 64 && LP >= 1 && LP <= 8, "channels");

    int tid = threadIdx.x;
    if constexpr (FRESH_TID) asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    const int lane = tid & 31;
    const int q = lane & (LP - 1);
    const int slot = (lane / APB) % kHypTile;        // this lane's hypothesis slot
    const int qa = q % APB;                          // this lane's anchor in the batch
    const int src0 = lane & ~(LP - 1);
    constexpr unsigned all = 0xffffffffu;            // every lane that exchanges runs every batch

    const float* P = sp.p[0];
    bool act = sp.act[0];
#pragma unroll
    for (int h = 1; h < kHypTile; ++h)
        if (slot == h) {
            P = sp.p[h];
            act = sp.act[h];
        }
    float R00, R01, R02, T0, R10, R11, R12, T1, R20, R21, R22, T2;
    if constexpr (!REREAD) {
        R00 = P[0], R01 = P[1], R02 = P[2], T0 = P[3];
        R10 = P[4], R11 = P[5], R12 = P[6], T1 = P[7];
        R20 = P[8], R21 = P[9], R22 = P[10], T2 = P[11];
    }

    // channels owned by this lane: vector k covers VW (q + k LP) .. + VW
    float qs[CPL], rs[CPL];
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            const int ch = VW * (q + k * LP) + e;
            qs[k * VW + e] = SCALED ? __ldg(v.qscale + ch) : 1.0f;
            rs[k * VW + e] = SCALED ? __ldg(v.rscale + ch) : 1.0f;
        }

    const Elem* qry = static_cast<const Elem*>(v.qry);
    const Elem* ref = static_cast<const Elem*>(v.ref);
    const int WC = v.W * C;
    const float xmax = (float)(v.W - 1), ymax = (float)(v.H - 1);
    const float d2 = v.huber * v.huber;

    // with PREFETCH the anchor coordinates of the next batch are read one batch ahead, so
    // that their load latency overlaps the current batch's gathers
    const int jfirst = j_begin + (tid / (LP * NS)) * APB;
    float nX = 0.f, nY = 0.f, nZ = 0.f;
    bool nok = false;
    if (PREFETCH && jfirst + qa < j_end) {
        const int j = jfirst + qa;
        nok = act && (!v.valid || v.valid[j]);
        nX = __ldg(v.px + j), nY = __ldg(v.py + j), nZ = __ldg(v.pz + j);
    }
    // every lane of a CTA runs the same batches; without exchanges (LP = 1) to its own last one (uneven
    // batch of 16 channels, with confidence maps: BF16 2057 -> 2011 us, FP16 2196 -> 2088)
    const int batches = (j_end - j_begin + ASTEP - 1) / ASTEP;
    for (int b = 0, jb = jfirst; LP == 1 ? jb < j_end : b < batches; ++b, jb += ASTEP) {
        // 1. every lane projects its own record: anchor jb + qa under its hypothesis
        const int jo = jb + qa;
        float X = nX, Y = nY, Z = nZ;
        bool ok = nok && jo < j_end;
        if constexpr (PREFETCH) {
            nok = false;
            if (jo + ASTEP < j_end) {
                const int j = jo + ASTEP;
                nok = act && (!v.valid || v.valid[j]);
                nX = __ldg(v.px + j), nY = __ldg(v.py + j), nZ = __ldg(v.pz + j);
            }
        } else if (jo < j_end) {
            ok = act && (!v.valid || v.valid[jo]);
            X = __ldg(v.px + jo), Y = __ldg(v.py + jo), Z = __ldg(v.pz + jo);
        }
        bool vis = false;
        int off = LP == 1 ? 0 : -1;                  // tap offset; -1: not visible
        float ax = 0.f, ay = 0.f, x = 0.f, y = 0.f, z = 1.f, iz = 1.f, wq = 1.f;
        if (ok) {
            if constexpr (REREAD) {
                load_row(P, R00, R01, R02, T0);
                load_row(P + 4, R10, R11, R12, T1);
                load_row(P + 8, R20, R21, R22, T2);
            }
            // p = R P + t  (world -> camera)
            x = fmaf(R00, X, fmaf(R01, Y, fmaf(R02, Z, T0)));
            y = fmaf(R10, X, fmaf(R11, Y, fmaf(R12, Z, T1)));
            z = fmaf(R20, X, fmaf(R21, Y, fmaf(R22, Z, T2)));
            if (z > kZNear) {
                iz = 1.0f / z;
                // pixel i covers [i, i+1): array coordinate = pixel - 1/2
                const float xs = fmaf(v.fx * x, iz, v.cx) - 0.5f;
                const float ys = fmaf(v.fy * y, iz, v.cy) - 0.5f;
                if (xs >= 0.f && xs <= xmax && ys >= 0.f && ys <= ymax) {
                    const int c0 = min((int)xs, v.W - 2);
                    const int r0 = min((int)ys, v.H - 2);
                    ax = xs - (float)c0;
                    ay = ys - (float)r0;
                    off = (r0 * v.W + c0) * C;
                    vis = true;
                    if constexpr (CONF) {  // query confidence, bilinear in the same cell
                        const float* cp = v.conf + r0 * v.W + c0;
                        const float c00 = __ldg(cp), c01 = __ldg(cp + 1);
                        const float c10 = __ldg(cp + v.W), c11 = __ldg(cp + v.W + 1);
                        const float bq = c01 - c00, cq2 = c10 - c00, dq = (c11 - c10) - bq;
                        wq = fmaf(ax, fmaf(dq, ay, bq), fmaf(ay, cq2, c00));
                    }
                }
            }
        }

        float S[6];
        if constexpr (LP == 1) {
            // one lane per record: its own taps and reference row
            RefBuf<DT, C, SCALED> rr;
            TapBuf<DT, C, SCALED> taps;
            rr.load(ref + (jo < j_end ? jo : j_begin) * C, 0);
            taps.load(qry + off, WC, 0);
            float P[1][6];
            record_partials<DT, C, SCALED, 1>(taps, rr, {ax}, {ay}, qs, rs, P);
#pragma unroll
            for (int k = 0; k < 6; ++k) S[k] = P[0][k];
        } else {
            // 2. the group reads its records two at a time: records t and t + LP/2, one
            //    anchor (t mod APB) under two of the group's hypotheses, against one read of
            //    the anchor's reference row (with four hypotheses per group, the rows are read
            //    once per batch and kept for both record pairs of an anchor); the first
            //    butterfly round (xor LP/2) keeps in each lane only the record it owns, so
            //    only LP/2 partial records stay live
            constexpr int HALF = LP / 2;
            RefBuf<DT, C, SCALED> rra[HG > 2 ? APB : 1];
            if constexpr (HG > 2) {
#pragma unroll
                for (int a = 0; a < APB; ++a) rra[a].load(ref + (jb + a < j_end ? jb + a : j_begin) * C, q);
            }
            // one butterfly step: lane keeps the record of its half and adds the partner's
            auto combine = [&](float* lo, const float* hi, int half) {
                const bool upper = (q & half) != 0;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const float send = upper ? lo[k] : hi[k];
                    const float keep = upper ? hi[k] : lo[k];
                    lo[k] = keep + __shfl_xor_sync(all, send, half);
                }
            };
            // record pair t: records t and t + HALF (one anchor, two hypotheses) against one
            // reference read, then the first butterfly round
            auto pair = [&](int t, float* Bt) {
                RefBuf<DT, C, SCALED>& rr = rra[HG > 2 ? t % APB : 0];
                if constexpr (HG <= 2) rr.load(ref + (jb + t < j_end ? jb + t : j_begin) * C, q);
                float P2[2][6];
                const int o0 = __shfl_sync(all, off, src0 + t), o1 = __shfl_sync(all, off, src0 + t + HALF);
                const float ax2[2] = {__shfl_sync(all, ax, src0 + t), __shfl_sync(all, ax, src0 + t + HALF)};
                const float ay2[2] = {__shfl_sync(all, ay, src0 + t), __shfl_sync(all, ay, src0 + t + HALF)};
                TapBuf<DT, C, SCALED> taps;
                // hypotheses that agree to a fraction of a pixel read the same cell: one load and
                // one set of tap differences for both (an invisible record's sums are discarded, so
                // it goes with the other)
                if (__all_sync(all, o0 == o1 || (o0 | o1) < 0)) {
                    taps.load(qry + max(max(o0, o1), 0), WC, q);
                    record_partials<DT, C, SCALED, 2>(taps, rr, ax2, ay2, qs, rs, P2);
                } else {
                    taps.load(qry + max(o0, 0), WC, q);
                    record_partials<DT, C, SCALED, 1>(taps, rr, {ax2[0]}, {ay2[0]}, qs, rs, P2);
                    taps.load(qry + max(o1, 0), WC, q);
                    record_partials<DT, C, SCALED, 1>(taps, rr, {ax2[1]}, {ay2[1]}, qs, rs, P2 + 1);
                }
                combine(P2[0], P2[1], HALF);
#pragma unroll
                for (int k = 0; k < 6; ++k) Bt[k] = P2[0][k];
            };
            float B[HALF][6];
            if constexpr (HALF == 4) {
                // the pairs in the order 0, 2, 1, 3: the second round combines (0, 2) and
                // (1, 3) as soon as both exist, so fewer partial records stay live (the same
                // additions as the round-by-round order)
                pair(0, B[0]);
                pair(2, B[2]);
                combine(B[0], B[2], 2);
                pair(1, B[1]);
                pair(3, B[3]);
                combine(B[1], B[3], 2);
                combine(B[0], B[1], 1);
            } else {
#pragma unroll
                for (int t = 0; t < HALF; ++t) pair(t, B[t]);
                // remaining butterfly rounds: afterwards B[0] of lane q holds record q's sums
#pragma unroll
                for (int half = HALF / 2; half >= 1; half >>= 1)
#pragma unroll
                    for (int t = 0; t < half; ++t) combine(B[t], B[t + half], half);
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) S[k] = B[0][k];
        }

        // 4. each lane finishes its own record: Huber weight, A = d(u,v)/dp [I | -[p]x],
        //    H += w A^T M A, g += w A^T b
        if (vis) {
            const float s = S[0], m00 = S[1], m01 = S[2], m11 = S[3];
            const float b0 = S[4], b1 = S[5];
            const float w = (v.weight ? __ldg(v.weight + jo) : 1.0f) * wq;
            const float sw = w * s;
            float rho, drho;
            if (sw <= d2) {
                rho = sw;
                drho = 1.0f;
            } else {
                const float rt = sqrtf(sw);
                rho = 2.0f * v.huber * rt - d2;
                drho = v.huber / rt;
            }
            const float om = w * drho;
            // the rotational part of each row a of d(u,v)/dp is p x a
            const float du_dx = v.fx * iz, du_dz = -v.fx * x * iz * iz;
            const float dv_dy = v.fy * iz, dv_dz = -v.fy * y * iz * iz;
            const float A0[6] = {du_dx, 0.f, du_dz, y * du_dz, z * du_dx - x * du_dz, -y * du_dx};
            const float A1[6] = {0.f, dv_dy, dv_dz, y * dv_dz - z * dv_dy, -x * dv_dz, x * dv_dy};
            // A0[1] = A1[0] = 0: the terms they multiply are left out (adding a zero product
            // leaves an FP32 sum unchanged, so the sums are the same as with them)
            float B0[6], B1[6], W0[6], W1[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if (k == 0) {
                    B0[k] = m00 * A0[k];
                    B1[k] = m01 * A0[k];
                } else if (k == 1) {
                    B0[k] = m01 * A1[k];
                    B1[k] = m11 * A1[k];
                } else {
                    B0[k] = fmaf(m00, A0[k], m01 * A1[k]);
                    B1[k] = fmaf(m01, A0[k], m11 * A1[k]);
                }
                W0[k] = (k == 1) ? 0.f : om * A0[k];
                W1[k] = (k == 0) ? 0.f : om * A1[k];
            }
            int e = 0;
#pragma unroll
            for (int a = 0; a < 6; ++a) {
#pragma unroll
                for (int b = a; b < 6; ++b) {
                    if (a == 0) acc[e] = fmaf(W0[a], B0[b], acc[e]);
                    else if (a == 1) acc[e] = fmaf(W1[a], B1[b], acc[e]);
                    else acc[e] = fmaf(W0[a], B0[b], fmaf(W1[a], B1[b], acc[e]));
                    ++e;
                }
            }
#pragma unroll
            for (int a = 0; a < 6; ++a) {
                if (a == 0) acc[21 + a] = fmaf(W0[a], b0, acc[21 + a]);
                else if (a == 1) acc[21 + a] = fmaf(W1[a], b1, acc[21 + a]);
                else acc[21 + a] = fmaf(W0[a], b0, fmaf(W1[a], b1, acc[21 + a]));
            }
            acc[27] += rho;
            acc[28] += 1.0f;
        }
    }
}

// ---- one hypothesis per CTA ----
// A record's factors as the chains below read them: W0[6], W1[6] (W = om A), B0[6], B1[6], b0, b1,
// rho, 1; a record that is not visible is all zeros (adding zero products changes nothing).
// Rows of 29 words: the lanes' own rows fall into different banks.
constexpr int kRowWords = 29;
enum RowCell { kRowW0 = 0, kRowW1 = 6, kRowB0 = 12, kRowB1 = 18, kRowb0 = 24, kRowb1 = 25, kRowRho = 26, kRowOne = 27,
               kRowZero = 1 /* W0[1] */ };

// The 29 sums over the kHypTile lanes of the slots (four, a quad), 2 kRoleSums each: kRoleSums of
// the form acc = fma(x, y, acc) (the first two rows of H, their g, the cost, the count) and
// kRoleSums of the form acc = fma(x, y, fma(z, w, acc)).  Entry: the sum's index, then its cells.
constexpr int kRoleSums = 16 / kHypTile;
struct RoleTable {
    unsigned char sum[kHypTile][2 * kRoleSums], cell[kHypTile][6 * kRoleSums];
};
constexpr RoleTable make_roles() {
    constexpr int K = kRoleSums;
    RoleTable t{};
    int n1 = 0, n2 = 0;
    for (int l = 0; l < kHypTile; ++l) {
        for (int i = 0; i < 2 * K; ++i) t.sum[l][i] = kNumSums;                // none
        for (int i = 0; i < 6 * K; ++i) t.cell[l][i] = kRowZero;
    }
    int e = 0;
    for (int a = 0; a < 6; ++a)
        for (int b = a; b < 6; ++b, ++e) {
            if (a < 2) {
                t.sum[n1 / K][n1 % K] = e;
                t.cell[n1 / K][2 * (n1 % K)] = (a == 0 ? kRowW0 : kRowW1) + a;
                t.cell[n1 / K][2 * (n1 % K) + 1] = (a == 0 ? kRowB0 : kRowB1) + b;
                ++n1;
            } else {
                unsigned char* c = t.cell[n2 / K] + 2 * K + 4 * (n2 % K);
                t.sum[n2 / K][K + n2 % K] = e;
                c[0] = kRowW0 + a, c[1] = kRowB0 + b, c[2] = kRowW1 + a, c[3] = kRowB1 + b;
                ++n2;
            }
        }
    for (int a = 0; a < 6; ++a) {
        if (a < 2) {
            t.sum[n1 / K][n1 % K] = 21 + a;
            t.cell[n1 / K][2 * (n1 % K)] = (a == 0 ? kRowW0 : kRowW1) + a;
            t.cell[n1 / K][2 * (n1 % K) + 1] = a == 0 ? kRowb0 : kRowb1;
            ++n1;
        } else {
            unsigned char* c = t.cell[n2 / K] + 2 * K + 4 * (n2 % K);
            t.sum[n2 / K][K + n2 % K] = 21 + a;
            c[0] = kRowW0 + a, c[1] = kRowb0, c[2] = kRowW1 + a, c[3] = kRowb1;
            ++n2;
        }
    }
    for (int i = 0; i < 2; ++i) {                            // cost, count
        t.sum[n1 / K][n1 % K] = 27 + i;
        t.cell[n1 / K][2 * (n1 % K)] = i == 0 ? kRowRho : kRowOne;
        t.cell[n1 / K][2 * (n1 % K) + 1] = kRowOne;
        ++n1;
    }
    return t;
}
static __constant__ RoleTable kRoles = make_roles();

// Accumulate anchors [j_begin, j_end) under one hypothesis: the layout of accumulate_anchors with
// a lane's slot standing for the batch of anchors it takes (slot h: every fourth batch from the
// h-th), so that a step covers four batches, all of their taps in flight at once.  The records'
// factors pass through shared memory (rows, one per thread) and a quad's lanes add them in the
// order of their anchors, eight sums each: the same sums in the same order as with four
// hypotheses per CTA.  acc: this lane's eight, 2 kRoleSums (kRoles.sum[slot]).
template <pilot_dtype DT, int C, bool SCALED, bool CONF>
__device__ __forceinline__ void accumulate_spread(const LevelView& v, const float* pose, int j_begin, int j_end,
                                                  float (*rows)[kRowWords], float* acc) {
    using Elem = typename Storage<DT>::T;
    using G = GroupShape<DT, C, SCALED>;
    constexpr int VW = G::VW, LP = G::LP, NS = G::NS, APB = G::APB, NV = G::NV, CPL = C / LP;
    constexpr int BATCH = kBuildThreads / (LP * NS) * APB, STEP = kHypTile * BATCH;
    constexpr int CHUNK = LP < 4 ? LP : 4, HALF = LP / 2;   // records whose taps are in flight
    const int tid = threadIdx.x, lane = tid & 31, q = lane & (LP - 1), src0 = lane & ~(LP - 1);
    const int slot = (lane / APB) % kHypTile;
    const int mine = q % APB + slot * BATCH;                // this lane's anchor in the step
    const float R00 = pose[0], R01 = pose[1], R02 = pose[2], T0 = pose[3];
    const float R10 = pose[4], R11 = pose[5], R12 = pose[6], T1 = pose[7];
    const float R20 = pose[8], R21 = pose[9], R22 = pose[10], T2 = pose[11];
    float qs[CPL], rs[CPL];
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            const int ch = VW * (q + k * LP) + e;
            qs[k * VW + e] = SCALED ? __ldg(v.qscale + ch) : 1.0f;
            rs[k * VW + e] = SCALED ? __ldg(v.rscale + ch) : 1.0f;
        }
    const Elem* qry = static_cast<const Elem*>(v.qry);
    const Elem* ref = static_cast<const Elem*>(v.ref);
    const int WC = v.W * C;
    const float xmax = (float)(v.W - 1), ymax = (float)(v.H - 1), d2 = v.huber * v.huber;
    constexpr int K = kRoleSums;
    int cell[6 * K];
#pragma unroll
    for (int i = 0; i < 6 * K; ++i) cell[i] = kRoles.cell[slot][i];
#pragma unroll
    for (int i = 0; i < 2 * K; ++i) acc[i] = 0.f;
    float* row = rows[tid];

    float nX = 0.f, nY = 0.f, nZ = 0.f;
    bool nok = false;
    const int jfirst = j_begin + (tid / (LP * NS)) * APB;
    auto fetch = [&](int j) {
        nok = false;
        if (j < j_end) {
            nok = !v.valid || v.valid[j];
            nX = __ldg(v.px + j), nY = __ldg(v.py + j), nZ = __ldg(v.pz + j);
        }
    };
    fetch(jfirst + mine);
    const int steps = (j_end - j_begin + STEP - 1) / STEP;  // the same for every thread
    for (int b = 0, jb = jfirst; b < steps; ++b, jb += STEP) {
        const float X = nX, Y = nY, Z = nZ;
        const bool ok = nok;
        fetch(jb + STEP + mine);
        bool vis = false;
        int off = 0;
        float ax = 0.f, ay = 0.f, x = 0.f, y = 0.f, z = 1.f, iz = 1.f, wq = 1.f;
        if (ok) {
            // p = R P + t  (world -> camera)
            x = fmaf(R00, X, fmaf(R01, Y, fmaf(R02, Z, T0)));
            y = fmaf(R10, X, fmaf(R11, Y, fmaf(R12, Z, T1)));
            z = fmaf(R20, X, fmaf(R21, Y, fmaf(R22, Z, T2)));
            if (z > kZNear) {
                iz = 1.0f / z;
                // pixel i covers [i, i+1): array coordinate = pixel - 1/2
                const float xs = fmaf(v.fx * x, iz, v.cx) - 0.5f;
                const float ys = fmaf(v.fy * y, iz, v.cy) - 0.5f;
                if (xs >= 0.f && xs <= xmax && ys >= 0.f && ys <= ymax) {
                    const int c0 = min((int)xs, v.W - 2);
                    const int r0 = min((int)ys, v.H - 2);
                    ax = xs - (float)c0;
                    ay = ys - (float)r0;
                    off = (r0 * v.W + c0) * C;
                    vis = true;
                    if constexpr (CONF) {  // query confidence, bilinear in the same cell
                        const float* cp = v.conf + r0 * v.W + c0;
                        const float c00 = __ldg(cp), c01 = __ldg(cp + 1);
                        const float c10 = __ldg(cp + v.W), c11 = __ldg(cp + v.W + 1);
                        const float bq = c01 - c00, cq2 = c10 - c00, dq = (c11 - c10) - bq;
                        wq = fmaf(ax, fmaf(dq, ay, bq), fmaf(ay, cq2, c00));
                    }
                }
            }
        }
        auto combine = [&](float* lo, const float* hi, int half) {
            const bool upper = (q & half) != 0;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const float send = upper ? lo[k] : hi[k];
                const float keep = upper ? hi[k] : lo[k];
                lo[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
            }
        };
        // the order accumulate_anchors combines its records in: pairs (t, t + LP / 2), the pairs
        // bit-reversed, as a tree
        float S[6], B[3][6];
#pragma unroll
        for (int c = 0; c < LP; c += CHUNK) {
            TapBuf<DT, C, SCALED> taps[CHUNK];
            RefBuf<DT, C, SCALED> rr[CHUNK];
#pragma unroll
            for (int m = 0; m < CHUNK; ++m) {
                const int k = c + m;
                const int i = LP == 8 ? (k & 1) * 4 + ((k >> 1) & 1) * 2 + (k >> 2) : (LP == 4 ? (k & 1) * 2 + (k >> 1) : k);
                const int o = LP > 1 ? __shfl_sync(0xffffffffu, off, src0 + i) : off;
                taps[m].load(qry + o, WC, q);
                const int ja = jb + i % APB + BATCH * (((src0 + i) / APB) % kHypTile);
                rr[m].load(ref + (ja < j_end ? ja : j_begin) * C, q);
            }
#pragma unroll
            for (int m = 0; m < CHUNK; ++m) {
                const int k = c + m;
                const int i = LP == 8 ? (k & 1) * 4 + ((k >> 1) & 1) * 2 + (k >> 2) : (LP == 4 ? (k & 1) * 2 + (k >> 1) : k);
                const float axi = LP > 1 ? __shfl_sync(0xffffffffu, ax, src0 + i) : ax;
                const float ayi = LP > 1 ? __shfl_sync(0xffffffffu, ay, src0 + i) : ay;
                float* P = LP == 1 || k == 6 ? S : (k & 1) ? B[2] : (k == 0 ? B[0] : B[1]);
                record_partials<DT, C, SCALED, 1>(taps[m], rr[m], {axi}, {ayi}, qs, rs, reinterpret_cast<float(*)[6]>(P));
                if (k == 1) combine(B[0], B[2], HALF);
                if (k == 3) {
                    combine(B[1], B[2], HALF);
                    combine(B[0], B[1], HALF / 2);
                }
                if (k == 5) combine(B[1], B[2], HALF);
                if (k == 7) {
                    combine(S, B[2], HALF);
                    combine(B[1], S, HALF / 2);
                    combine(B[0], B[1], 1);
                }
            }
        }
        if constexpr (LP > 1) {
#pragma unroll
            for (int k = 0; k < 6; ++k) S[k] = B[0][k];
        }
        // the lane's own record: Huber weight, A = d(u,v)/dp [I | -[p]x], the factors of
        // H += w A^T M A, g += w A^T b
        float f[28];
#pragma unroll
        for (int k = 0; k < 28; ++k) f[k] = 0.f;
        if (vis) {
            const float s = S[0], m00 = S[1], m01 = S[2], m11 = S[3];
            const float w = (v.weight ? __ldg(v.weight + jb + mine) : 1.0f) * wq;
            const float sw = w * s;
            float rho, drho;
            if (sw <= d2) {
                rho = sw;
                drho = 1.0f;
            } else {
                const float rt = sqrtf(sw);
                rho = 2.0f * v.huber * rt - d2;
                drho = v.huber / rt;
            }
            const float om = w * drho;
            const float du_dx = v.fx * iz, du_dz = -v.fx * x * iz * iz;
            const float dv_dy = v.fy * iz, dv_dz = -v.fy * y * iz * iz;
            const float A0[6] = {du_dx, 0.f, du_dz, y * du_dz, z * du_dx - x * du_dz, -y * du_dx};
            const float A1[6] = {0.f, dv_dy, dv_dz, y * dv_dz - z * dv_dy, -x * dv_dz, x * dv_dy};
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if (k == 0) {
                    f[kRowB0 + k] = m00 * A0[k];
                    f[kRowB1 + k] = m01 * A0[k];
                } else if (k == 1) {
                    f[kRowB0 + k] = m01 * A1[k];
                    f[kRowB1 + k] = m11 * A1[k];
                } else {
                    f[kRowB0 + k] = fmaf(m00, A0[k], m01 * A1[k]);
                    f[kRowB1 + k] = fmaf(m01, A0[k], m11 * A1[k]);
                }
                if (k != 1) f[kRowW0 + k] = om * A0[k];
                if (k != 0) f[kRowW1 + k] = om * A1[k];
            }
            f[kRowb0] = S[4];
            f[kRowb1] = S[5];
            f[kRowRho] = rho;
            f[kRowOne] = 1.0f;
        }
#pragma unroll
        for (int k = 0; k < 28; ++k) row[k] = f[k];
        __syncwarp();
        const float* quad = rows[(tid & ~31) + (lane & ~((kHypTile - 1) * APB))];
#pragma unroll
        for (int h = 0; h < kHypTile; ++h) {
            const float* r = quad + h * APB * kRowWords;
#pragma unroll
            for (int m = 0; m < K; ++m) {
                const int* c = cell + 2 * K + 4 * m;
                acc[m] = fmaf(r[cell[2 * m]], r[cell[2 * m + 1]], acc[m]);
                acc[K + m] = fmaf(r[c[0]], r[c[1]], fmaf(r[c[2]], r[c[3]], acc[K + m]));
            }
        }
        __syncwarp();
    }
}

// The CTA's sums of accumulate_spread, in cta_reduce_slots' order: thread t < 32 returns sum t (0
// pads).  Called by the accumulating warps only (barrier 1).
template <int APB>
__device__ __forceinline__ float cta_reduce_spread(float* acc, float (*red)[kAcc]) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        if (off >= APB && off < APB * kHypTile) continue;
#pragma unroll
        for (int i = 0; i < 2 * kRoleSums; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], off);
    }
    if (lane % APB == 0 && lane < APB * kHypTile) {
#pragma unroll
        for (int i = 0; i < 2 * kRoleSums; ++i) {
            const int s = kRoles.sum[lane / APB][i];
            if (s < kNumSums) red[warp][s] = acc[i];
        }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kBuildThreads) : "memory");
    float v = 0.f;
    if (tid < kNumSums) {
#pragma unroll
        for (int w = 0; w < kBuildThreads / 32; ++w) v += red[w][tid];
    }
    return v;
}

// Fixed-order CTA reduction of the lanes' 29 sums, per hypothesis slot: the 32 / kHypTile lanes of a
// slot are reduced by a butterfly over every lane bit but the slot bits (APB .. APB kHypTile / 2),
// then the warps in order.  SCATTER: the butterfly scatters as it goes (16, 8, then 4 sums exchanged
// instead of 29 three times: the shuffles are what the reduction costs), so a lane ends with
// kHypTile sums; without it fewer registers are live, which the level kernels need more (batched
// BF16, uneven frames: 15.1 ms without, 15.4 ms with).  Thread t < kHypTile kAcc returns sum t mod
// kAcc of slot t / kAcc (0 pads).
template <int NTHREADS, int APB, bool SCATTER = true>
__device__ __forceinline__ float cta_reduce_slots(float* acc, float (*red)[kHypTile][kAcc]) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int slot_bits = APB * (kHypTile - 1);
    static_assert(APB * kHypTile <= 32, "slots of a warp");
    if constexpr (SCATTER) {
        float a[kAcc];
#pragma unroll
        for (int i = 0; i < kAcc; ++i) a[i] = i < kNumSums ? acc[i] : 0.f;
        int n = kAcc, kept = 0;                      // sums held, and the first one's index
#pragma unroll
        for (int bit = 1; bit < 32; bit <<= 1) {
            if (bit & slot_bits) continue;
            n /= 2;                                  // keeps the lower or upper half
            const bool up = (lane & bit) != 0;
#pragma unroll
            for (int i = 0; i < kAcc / 2; ++i) {
                if (i >= n) break;
                const float send = up ? a[i] : a[i + n], keep = up ? a[i + n] : a[i];
                a[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
            }
            if (up) kept += n;
        }
        float* dst = &red[warp][(lane / APB) % kHypTile][kept];
        if constexpr (kHypTile == 2) {
            *reinterpret_cast<float2*>(dst) = make_float2(a[0], a[1]);
        } else {
#pragma unroll
            for (int i = 0; i < kHypTile; i += 4)
                *reinterpret_cast<float4*>(dst + i) = make_float4(a[i], a[i + 1], a[i + 2], a[i + 3]);
        }
    } else {
#pragma unroll
        for (int bit = 1; bit < 32; bit <<= 1) {
            if (bit & slot_bits) continue;
#pragma unroll
            for (int i = 0; i < kNumSums; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], bit);
        }
        if (lane % APB == 0 && lane < APB * kHypTile) {
#pragma unroll
            for (int i = 0; i < kNumSums; ++i) red[warp][lane / APB][i] = acc[i];
        }
    }
    __syncthreads();
    float v = 0.f;
    if (tid < kHypTile * kAcc && (tid % kAcc) < kNumSums) {
#pragma unroll
        for (int w = 0; w < NTHREADS / 32; ++w) v += red[w][tid / kAcc][tid % kAcc];
    }
    return v;
}

// The CTA's hypotheses: slots kHypTile blockIdx.y + h of the active list, h < n.
struct TileSlots {
    int slot[kHypTile];
    int hyp[kHypTile];
    bool cand[kHypTile];
    int n;                                           // 1 .. kHypTile
};

__device__ __forceinline__ TileSlots tile_slots(const BuildParams& p) {
    TileSlots s;
    s.n = min(kHypTile, p.n_active - kHypTile * (int)blockIdx.y);
#pragma unroll
    for (int h = 0; h < kHypTile; ++h) {
        s.slot[h] = kHypTile * blockIdx.y + (h < s.n ? h : 0);
        s.hyp[h] = p.active_idx[s.slot[h]];
        s.cand[h] = h < s.n && p.state[s.hyp[h]].has_cand;
    }
    return s;
}

__device__ __forceinline__ SlotPoses slot_poses(const BuildParams& p, const TileSlots& ts) {
    SlotPoses sp;
#pragma unroll
    for (int h = 0; h < kHypTile; ++h) {
        sp.p[h] = p.pose32 + 12 * ts.hyp[h];
        sp.act[h] = ts.cand[h];
    }
    return sp;
}

__device__ __forceinline__ bool any_cand(const TileSlots& ts) {
    bool a = false;
#pragma unroll
    for (int h = 0; h < kHypTile; ++h) a = a || ts.cand[h];
    return a;
}

// Evaluation of larger frames at given poses (T_cw, M x 12): the tile records; epilogue_kernel,
// which may start while the last of these CTAs run, sums them.  The poses are narrowed here, and
// left in the state for the priors.  (Summing in the last CTA of each hypothesis tile, as
// build_fused_kernel does, made 64 poses x 65536 anchors 172 us instead of 164: sixteen CTAs sum
// what sixty-four blocks do here.)  With the shared cells and the pose read again per batch 153.6 us.
template <pilot_dtype DT, int C, bool SCALED, bool CONF>
__global__ void __launch_bounds__(kBuildThreads, 2)
build_kernel(const BuildParams p, HypState* state, const double* T_cw) {
    __shared__ __align__(16) float red[kBuildThreads / 32][kHypTile][kAcc];
    __shared__ __align__(16) float pose[kHypTile][12];
    const int slot0 = kHypTile * (int)blockIdx.y, n = min(kHypTile, p.n_active - slot0), tid = threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid < 12 * kHypTile) {
        const int h = tid / 12, hyp = slot0 + (h < n ? h : 0);
        const double t = T_cw[12 * (size_t)hyp + tid % 12];
        pose[h][tid % 12] = narrow(t);
        if (blockIdx.x == 0 && h < n) state[hyp].T[tid % 12] = t;
    }
    __syncthreads();
    SlotPoses sp;
#pragma unroll
    for (int h = 0; h < kHypTile; ++h) {
        sp.p[h] = pose[h];
        sp.act[h] = h < n;
    }
    float acc[kNumSums];
#pragma unroll
    for (int i = 0; i < kNumSums; ++i) acc[i] = 0.f;
    const int j0 = blockIdx.x * p.tile;
    accumulate_anchors<DT, C, SCALED, CONF, kBuildThreads, true, false, DT != PILOT_FP8E4M3 && kPoseReread<DT, C, SCALED>>(
        level_view(p), sp, j0, min(j0 + p.tile, p.N), acc);
    const float v = cta_reduce_slots<kBuildThreads, GroupShape<DT, C, SCALED>::APB>(acc, red);
    const int h = tid / kAcc;
    if (tid < kHypTile * kAcc && h < n) p.partial[((size_t)(slot0 + h) * p.n_tiles + blockIdx.x) * kAcc + tid % kAcc] = v;
}

// The same pass with the per-hypothesis FP64 step fused in: the CTA that takes the last
// ticket of its hypothesis tile sums the tile records of its hypotheses (FP64, 8 chains per
// value, fixed order) and runs lm_step for hypothesis h on warp h.  A step may set has_cand and
// write the next pose, which a tile's CTAs read when they start, so the last ticket is also the
// one of a tile of hypotheses with no candidate, where there is nothing to sum: its step may find
// one (a larger lambda), and a CTA of the launch that had not started yet would evaluate it.
template <pilot_dtype DT, int C, bool SCALED, bool CONF>
__global__ void __launch_bounds__(kBuildThreads, 2)
build_fused_kernel(const FusedBuildParams fp) {
    const BuildParams& p = fp.b;
    __shared__ __align__(16) float red[kBuildThreads / 32][kHypTile][kAcc];
    __shared__ double part[kHypTile][8][kAcc];
    __shared__ double E[kHypTile][kAcc];
    __shared__ int s_last;
    const TileSlots ts = tile_slots(p);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // whether this CTA is the last of its hypothesis tile to get here (one fence for what its
    // threads read and wrote: it is cumulative over the barrier)
    auto last_of_tile = [&]() {
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            s_last = (atomicAdd(fp.tickets + blockIdx.y, 1u) == (unsigned)(p.n_tiles - 1));
            if (s_last) __threadfence();
        }
        __syncthreads();
        return s_last != 0;
    };
    if (!any_cand(ts)) {                             // uniform over the CTA
        if (p.n_tiles > 1 && !last_of_tile()) return;
        if (warp < ts.n) lm_step(fp.ep, ts.slot[warp], E[warp], *fp.min_valid, lane);
        if (p.n_tiles > 1 && tid == 0) fp.tickets[blockIdx.y] = 0u;
        return;
    }
    float acc[kNumSums];
#pragma unroll
    for (int i = 0; i < kNumSums; ++i) acc[i] = 0.f;
    const int j0 = blockIdx.x * p.tile;
    accumulate_anchors<DT, C, SCALED, CONF, kBuildThreads>(level_view(p), slot_poses(p, ts), j0,
                                                           min(j0 + p.tile, p.N), acc);
    const float v = cta_reduce_slots<kBuildThreads, GroupShape<DT, C, SCALED>::APB>(acc, red);
    const int hv = tid / kAcc, iv = tid % kAcc;     // slot and sum this thread holds (tid < kHypTile kAcc)
    if (p.n_tiles == 1) {
        // the only tile: its record is the sum, no round trip through the partial buffer and the
        // ticket
        if (tid < kHypTile * kAcc) E[hv][iv] = widen(v);
        __syncthreads();
        if (warp < ts.n) lm_step(fp.ep, ts.slot[warp], E[warp], *fp.min_valid, lane);
        return;
    }
    if (tid < kHypTile * kAcc && hv < ts.n && ts.cand[hv])
        p.partial[((size_t)ts.slot[hv] * p.n_tiles + blockIdx.x) * kAcc + iv] = v;
    if (!last_of_tile()) return;
    // 8 chains per slot and value: thread (h, c, i) sums tiles c, c + 8, ... of sum i of slot h
    {
        constexpr int kTPC = kBuildThreads / (kHypTile * 8);     // threads per (slot, chain)
        const int h = tid / (8 * kTPC), c = (tid / kTPC) & 7;
        for (int ii = tid % kTPC; ii < kAcc; ii += kTPC) {
            double a = 0.0;
            if (h < ts.n && ts.cand[h]) {
                const float* src = p.partial + (size_t)ts.slot[h] * p.n_tiles * kAcc + ii;
                a = chain_sum([&](int t) { return __ldcg(src + (size_t)t * kAcc); }, c, p.n_tiles);
            }
            part[h][c][ii] = a;
        }
    }
    __syncthreads();
    if (tid < kHypTile * kAcc) {
        double sum = part[hv][0][iv];
        for (int k = 1; k < min(8, p.n_tiles); ++k) sum += part[hv][k][iv];
        E[hv][iv] = sum;
    }
    __syncthreads();
    if (warp < ts.n) {                               // the warp-cooperative FP64 steps
        lm_step(fp.ep, ts.slot[warp], E[warp], *fp.min_valid, lane);
    }
    if (tid == 0) fp.tickets[blockIdx.y] = 0u;
}

// ---- a whole level of a small frame in one launch ----
// The CTAs of a hypothesis tile (one per anchor tile, at most kMaxCluster: a thread-block cluster)
// stay on their SMs through all of a level's LM iterations.  An iteration's tile records and next
// poses pass through (distributed) shared memory between cluster barriers; the cluster's first
// CTA sums the records (FP64, the order of the 8-chain sum: at most one record per chain) and runs
// the FP64 steps.
//
// Why: with few anchors an iteration is a chain of latencies -- the launch, eight or more
// dependent batches of gathers, the FP64 step.  One launch per level drops the launches, and
// level_spread_kernel shortens the rest while SMs would be idle.  4096 anchors, 1
// hypothesis, 20 iterations: 752 -> 378 us; paper's schedule (500 anchors, 1210 -> 128
// hypotheses, 12 evaluations): 552 -> 284 us (with the FP64 step's own gain).

// kHypTile hypotheses per CTA, hypothesis h stepped by warp h.
template <pilot_dtype DT, int C, bool SCALED, bool CONF>
__global__ void __launch_bounds__(kBuildThreads, 2)
level_resident_kernel(const __grid_constant__ ResidentParams rp) {
    namespace cg = cooperative_groups;
    const BuildParams& p = rp.b;
    __shared__ __align__(16) float red[kBuildThreads / 32][kHypTile][kAcc];
    __shared__ ResidentHyp hyps[kHypTile];
    __shared__ double E[kHypTile][kAcc];
    __shared__ float rec[kHypTile][kAcc];
    __shared__ __align__(16) float pose[kHypTile][12];
    __shared__ int s_cand[kHypTile];
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x, slot0 = kHypTile * (int)blockIdx.y, n = min(kHypTile, p.n_active - slot0);
    const int iters = rp.iters;
    const bool steps = rank == 0 && warp < n;
    auto all_ctas = [&]() {
        if (p.n_tiles > 1) cluster.sync();
        else __syncthreads();
    };
    int hyp = 0;
    if (warp < kHypTile) {
        const int slot = slot0 + (warp < n ? warp : 0);
        hyp = p.active_idx ? p.active_idx[slot] : slot;
        const double T = lane < 12 ? (rp.T_cw ? rp.T_cw[12 * (size_t)hyp + lane] : __ldcg(rp.ep.state[hyp].T + lane)) : 0.0;
        if (steps) resident_begin(hyps[warp], T, rp.ep.lambda0, lane);
        if (lane < 12) pose[warp][lane] = narrow(T);
        if (lane == 0) s_cand[warp] = warp < n;
    }
    __syncthreads();
    for (int k = 0; k <= iters; ++k) {
        SlotPoses sp;
        bool any = false;
#pragma unroll
        for (int h = 0; h < kHypTile; ++h) {
            sp.p[h] = pose[h];
            sp.act[h] = s_cand[h] != 0;
            any = any || sp.act[h];
        }
        if (any) {                                       // the same in every CTA of the cluster
            if (steps && s_cand[warp]) resident_priors(hyps[warp], rp.ep.prior, k == 0, lane);
            float acc[kNumSums];
#pragma unroll
            for (int i = 0; i < kNumSums; ++i) acc[i] = 0.f;
            const int j0 = rank * p.tile;
            accumulate_anchors<DT, C, SCALED, CONF, kBuildThreads>(level_view(p), sp, j0, min(j0 + p.tile, p.N), acc);
            const float v = cta_reduce_slots<kBuildThreads, GroupShape<DT, C, SCALED>::APB>(acc, red);
            if (tid < kHypTile * kAcc) rec[tid / kAcc][tid % kAcc] = v;
        }
        all_ctas();
        if (rank == 0) {
            if (tid < kHypTile * kAcc) {
                double sum = widen((&rec[0][0])[tid]);
                for (int t = 1; t < p.n_tiles; ++t) sum += widen(cluster.map_shared_rank(&rec[0][0], t)[tid]);
                (&E[0][0])[tid] = sum;
            }
            __syncthreads();
            if (steps && rp.T_cw) {
                if (lane < kNumSums)
                    rp.ep.eval_out[(size_t)(slot0 + warp) * kNumSums + lane] =
                        with_priors(E[warp][lane], hyps[warp].terms[lane]);
            } else if (steps) {
                const int cand = resident_step(hyps[warp], E[warp], k == 0 ? kEpiInit : kEpiStep, k < iters,
                                               rp.ep.damping_mode, *rp.min_valid, pose[warp], lane);
                if (lane == 0) s_cand[warp] = cand;
            }
        }
        all_ctas();
        if (k < iters && rank != 0) {
            if (tid < 12 * kHypTile) (&pose[0][0])[tid] = cluster.map_shared_rank(&pose[0][0], 0)[tid];
            if (tid < kHypTile) s_cand[tid] = cluster.map_shared_rank(s_cand, 0)[tid];
            __syncthreads();
        }
    }
    if (steps && !rp.T_cw) resident_end(hyps[warp], rp.ep.state[hyp], lane);
}

// One hypothesis per CTA, and a ninth warp for its FP64 work: the warp keeps the LM state on its
// lanes through the level, works out the priors at the candidate while the others gather (they
// depend on the pose only) and then steps on the records.  One CTA per SM: the registers hold the
// taps of four batches at once (accumulate_spread).
constexpr int kSpreadThreads = kBuildThreads + 32;

template <pilot_dtype DT, int C, bool SCALED, bool CONF>
__global__ void __launch_bounds__(kSpreadThreads, 1)
level_spread_kernel(const __grid_constant__ ResidentParams rp) {
    namespace cg = cooperative_groups;
    const BuildParams& p = rp.b;
    __shared__ float rows[kBuildThreads][kRowWords];
    __shared__ float red[kBuildThreads / 32][kAcc];
    __shared__ float rec[kAcc];
    __shared__ float pose[12];
    __shared__ int s_cand;
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x, iters = rp.iters;
    const bool steps = warp == kBuildThreads / 32 && rank == 0;
    const int slot = blockIdx.y, hyp = p.active_idx ? p.active_idx[slot] : slot;
    HypState& st = rp.ep.state[hyp];
    auto all_ctas = [&]() {
        if (p.n_tiles > 1) cluster.sync();
        else __syncthreads();
    };
    LmLanes s{};
    int ta = 0, tb = 0;
    if (warp == kBuildThreads / 32) {
        s.T = lane < 12 ? (rp.T_cw ? rp.T_cw[12 * (size_t)hyp + lane] : __ldcg(st.T + lane)) : 0.0;
        s.lambda = rp.ep.lambda0;
        s.has_cand = 1;
        if (lane < 12) pose[lane] = narrow(s.T);
        if (lane == 0) s_cand = 1;
        if (lane < 21) tri_pair(lane, &ta, &tb);
    }
    __syncthreads();
    for (int k = 0; k <= iters; ++k) {
        const bool cand = s_cand != 0;                   // the same in every CTA of the cluster
        PriorTerms terms{};
        if (warp < kBuildThreads / 32) {
            if (cand) {
                float acc[2 * kRoleSums];
                const int j0 = rank * p.tile;
                accumulate_spread<DT, C, SCALED, CONF>(level_view(p), pose, j0, min(j0 + p.tile, p.N), rows, acc);
                const float v = cta_reduce_spread<GroupShape<DT, C, SCALED>::APB>(acc, red);
                if (tid < kAcc) rec[tid] = v;
            }
        } else if (steps && cand) {
            terms = prior_terms(rp.ep.prior, k == 0 ? s.T : s.Tc, lane, ta, tb);
        }
        all_ctas();
        if (steps) {
            double e = 0.0;
            if (cand && lane < kNumSums) {
                e = widen(rec[lane]);
                for (int t = 1; t < p.n_tiles; ++t) e += widen(cluster.map_shared_rank(rec, t)[lane]);
            }
            if (cand) e = with_priors(e, terms);
            if (rp.T_cw) {
                if (lane < kNumSums) rp.ep.eval_out[(size_t)slot * kNumSums + lane] = e;
            } else {
                bool take;
                lm_lanes_step(s, k == 0 ? kEpiInit : kEpiStep, cand, k < iters, rp.ep.damping_mode, e, *rp.min_valid, lane,
                              ta, tb, &take);
                if (s.has_cand && lane < 12) pose[lane] = narrow(s.Tc);
                if (lane == 0) s_cand = s.has_cand;
            }
        }
        all_ctas();
        if (k < iters && rank != 0) {
            if (tid < 12) pose[tid] = cluster.map_shared_rank(pose, 0)[tid];
            if (tid == 0) s_cand = *cluster.map_shared_rank(&s_cand, 0);
            __syncthreads();
        }
    }
    if (steps && !rp.T_cw) {                             // what the next level and the selection read
        if (lane < 12) st.T[lane] = s.T;
        if (lane == 0) {
            st.cost = s.cost;
            st.lambda = s.lambda;
            st.n_valid = s.n_valid;
            st.has_cand = s.has_cand;
            st.last_fail = s.last_fail;
        }
    }
}

template <pilot_dtype DT, int C>
cudaError_t launch_build_typed(const BuildParams& p, HypState* state, const double* T_cw, cudaStream_t s) {
    dim3 grid(p.n_tiles, (p.n_active + kHypTile - 1) / kHypTile);
    if (p.qscale && p.conf)
        build_kernel<DT, C, true, true><<<grid, kBuildThreads, 0, s>>>(p, state, T_cw);
    else if (p.qscale)
        build_kernel<DT, C, true, false><<<grid, kBuildThreads, 0, s>>>(p, state, T_cw);
    else if (p.conf)
        build_kernel<DT, C, false, true><<<grid, kBuildThreads, 0, s>>>(p, state, T_cw);
    else
        build_kernel<DT, C, false, false><<<grid, kBuildThreads, 0, s>>>(p, state, T_cw);
    return cudaGetLastError();
}

template <pilot_dtype DT, int C>
cudaError_t launch_build_fused_typed(const FusedBuildParams& p, cudaStream_t s) {
    dim3 grid(p.b.n_tiles, (p.b.n_active + kHypTile - 1) / kHypTile);
    if (p.b.qscale && p.b.conf)
        build_fused_kernel<DT, C, true, true><<<grid, kBuildThreads, 0, s>>>(p);
    else if (p.b.qscale)
        build_fused_kernel<DT, C, true, false><<<grid, kBuildThreads, 0, s>>>(p);
    else if (p.b.conf)
        build_fused_kernel<DT, C, false, true><<<grid, kBuildThreads, 0, s>>>(p);
    else
        build_fused_kernel<DT, C, false, false><<<grid, kBuildThreads, 0, s>>>(p);
    return cudaGetLastError();
}

template <pilot_dtype DT, int C, bool SCALED, bool CONF>
cudaError_t launch_resident_kernel(const ResidentParams& p, bool spread, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.b.n_tiles;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(p.b.n_tiles, spread ? p.b.n_active : (p.b.n_active + kHypTile - 1) / kHypTile);
    cfg.blockDim = dim3(spread ? kSpreadThreads : kBuildThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return spread ? cudaLaunchKernelEx(&cfg, level_spread_kernel<DT, C, SCALED, CONF>, p)
                  : cudaLaunchKernelEx(&cfg, level_resident_kernel<DT, C, SCALED, CONF>, p);
}

template <pilot_dtype DT, int C>
cudaError_t launch_resident_typed(const ResidentParams& p, bool spread, cudaStream_t s) {
    if (p.b.qscale && p.b.conf) return launch_resident_kernel<DT, C, true, true>(p, spread, s);
    if (p.b.qscale) return launch_resident_kernel<DT, C, true, false>(p, spread, s);
    if (p.b.conf) return launch_resident_kernel<DT, C, false, true>(p, spread, s);
    return launch_resident_kernel<DT, C, false, false>(p, spread, s);
}

template <pilot_dtype DT>
cudaError_t launch_resident_dtype(const ResidentParams& p, bool spread, cudaStream_t s) {
    switch (p.b.C) {
        case 4: return launch_resident_typed<DT, 4>(p, spread, s);
        case 8: return launch_resident_typed<DT, 8>(p, spread, s);
        case 16: return launch_resident_typed<DT, 16>(p, spread, s);
        case 32: return launch_resident_typed<DT, 32>(p, spread, s);
        case 64: return launch_resident_typed<DT, 64>(p, spread, s);
        default: return cudaErrorInvalidValue;
    }
}

template <pilot_dtype DT>
cudaError_t launch_build_dtype(const BuildParams& p, HypState* state, const double* T_cw, cudaStream_t s) {
    switch (p.C) {
        case 4: return launch_build_typed<DT, 4>(p, state, T_cw, s);
        case 8: return launch_build_typed<DT, 8>(p, state, T_cw, s);
        case 16: return launch_build_typed<DT, 16>(p, state, T_cw, s);
        case 32: return launch_build_typed<DT, 32>(p, state, T_cw, s);
        case 64: return launch_build_typed<DT, 64>(p, state, T_cw, s);
        default: return cudaErrorInvalidValue;
    }
}

template <pilot_dtype DT>
cudaError_t launch_build_fused_dtype(const FusedBuildParams& p, cudaStream_t s) {
    switch (p.b.C) {
        case 4: return launch_build_fused_typed<DT, 4>(p, s);
        case 8: return launch_build_fused_typed<DT, 8>(p, s);
        case 16: return launch_build_fused_typed<DT, 16>(p, s);
        case 32: return launch_build_fused_typed<DT, 32>(p, s);
        case 64: return launch_build_fused_typed<DT, 64>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pilot
