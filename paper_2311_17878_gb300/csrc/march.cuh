// The voxel walk of Alg. 1 / Alg. 2 ("NextVoxel") and the grid-box clip, shared by the
// ray march (bounds.cu) and the ray-casting fusion (integrate.cu).  Every operation is an
// explicitly rounded IEEE binary32 operation (no contraction), so the walk is the same
// voxel sequence wherever it runs.
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"

namespace tsdfs {
namespace {

struct GridDev {
    const void* V;
    int f16;
    int n[3];
    float org[3];
    float vs;
    float trunc;
};

// V at a voxel of the grid by its linear index
__device__ __forceinline__ float vat(const GridDev& g, int64_t idx) {
    return g.f16 ? __half2float(__ldg(reinterpret_cast<const __half*>(g.V) + idx))
                 : __ldg(reinterpret_cast<const float*>(g.V) + idx);
}
// linear index of a voxel of the grid; SMALL: the grid has under 2^31 voxels
template <bool SMALL>
__device__ __forceinline__ int64_t vidx(const GridDev& g, int i, int j, int k) {
    if constexpr (SMALL) return (uint32_t)((k * g.n[1] + j) * g.n[0] + i);
    return ((int64_t)k * g.n[1] + j) * g.n[0] + i;
}

// whether a grid's voxels and boundaries have 32-bit linear indexes and exact FP32 numbers
inline bool small_grid(const int32_t n[3]) {
    return (int64_t)n[0] * n[1] * n[2] <= (int64_t)INT32_MAX && n[0] < (1 << 23) && n[1] < (1 << 23) && n[2] < (1 << 23);
}

// The walk.  Per axis: the number b of the boundary it crosses next and what turns that into the
// crossing's parameter, t = ((org + b vs) - o) / d; how far the linear index moves; how many voxels are
// left ahead.  An axis without a step has o = -inf and 1 / d = inf, so its crossing is at +inf.
// A step is issue-bound code that every voxel pays for, so it converts nothing between integers and
// floats: SMALL, b is counted in FP32 (exact), otherwise in integers and converted.
template <bool SMALL>
struct Walk {
    float b[3], sf[3], o[3], inv[3];
    int st[3];          // -1, 0, 1
    int left[3];        // voxels ahead along the axis
    int64_t stride[3];  // of the linear index per step (SMALL: fits 32 bits)
    int64_t idx;
    int ib[3];          // !SMALL: b
    float t;            // entry parameter of the voxel

    __device__ __forceinline__ void place(const GridDev& g, const int X[3], float t_entry) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ib[a] = X[a] + (st[a] > 0 ? 1 : 0);
            b[a] = (float)ib[a];
            left[a] = st[a] > 0 ? g.n[a] - 1 - X[a] : (st[a] < 0 ? X[a] : INT32_MAX);
        }
        idx = vidx<SMALL>(g, X[0], X[1], X[2]);
        t = t_entry;
    }
    // at parameter t0 (a point inside the grid box): the voxel that holds origin + t0 d, clamped into the grid
    __device__ __forceinline__ void start(const GridDev& g, const float org[3], const float d[3], float t0) {
        const float kInf = __int_as_float(0x7f800000);
        int X[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            st[a] = d[a] > 0.0f ? 1 : (d[a] < 0.0f ? -1 : 0);
            sf[a] = (float)st[a];
            o[a] = st[a] ? org[a] : -kInf;
            inv[a] = st[a] ? __fdiv_rn(1.0f, d[a]) : kInf;
            const float pa = __fadd_rn(org[a], __fmul_rn(t0, d[a]));
            const float gg = floorf(__fdiv_rn(__fsub_rn(pa, g.org[a]), g.vs));
            X[a] = gg >= 0.0f ? (gg > (float)(g.n[a] - 1) ? g.n[a] - 1 : (int)gg) : 0;
        }
        stride[0] = st[0];
        stride[1] = (int64_t)st[1] * g.n[0];
        stride[2] = (int64_t)st[2] * g.n[0] * g.n[1];
        place(g, X, t0);
    }
    // the voxel's coordinates
    __device__ __forceinline__ void voxel(int X[3]) const {
#pragma unroll
        for (int a = 0; a < 3; ++a) X[a] = (SMALL ? (int)b[a] : ib[a]) - (st[a] > 0 ? 1 : 0);
    }
    // its centre along axis a, in voxels from the grid's corner
    __device__ __forceinline__ float centre(int a) const {
        if constexpr (SMALL) return b[a] + (st[a] > 0 ? -0.5f : 0.5f);
        return __fadd_rn((float)(ib[a] - (st[a] > 0 ? 1 : 0)), 0.5f);
    }
    // one step: the first crossing in the order (parameter, axis); `axis` receives its axis; false: the
    // walk left the grid
    __device__ __forceinline__ bool next(const GridDev& g, int& axis) {
        float tc[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) tc[a] = __fmul_rn(__fsub_rn(__fadd_rn(g.org[a], __fmul_rn(b[a], g.vs)), o[a]), inv[a]);
        int ax = 0;
        float tm = tc[0];
        if (tc[1] < tm) { ax = 1; tm = tc[1]; }
        if (tc[2] < tm) { ax = 2; tm = tc[2]; }
        t = tm;
        axis = ax;
        // the axis is a run-time value: the three components are updated by selection, so the
        // state stays in registers
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const bool m = ax == a;
            if constexpr (SMALL) {
                b[a] += m ? sf[a] : 0.0f;
                idx = (uint32_t)((int32_t)idx + (m ? (int32_t)stride[a] : 0));
            } else {
                ib[a] += m ? st[a] : 0;
                b[a] = (float)ib[a];
                idx += m ? stride[a] : 0;
            }
            left[a] -= m && st[a] != 0;
            in = in && left[a] >= 0;
        }
        return in;
    }
    __device__ __forceinline__ bool next(const GridDev& g) {
        int axis;
        return next(g, axis);
    }
};

__device__ __forceinline__ void point_at(const float o[3], const float d[3], float t, float p[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) p[a] = __fadd_rn(o[a], __fmul_rn(t, d[a]));
}

// clip a ray to the grid box ("RenderingCube") within [t_near, t_far]: [t0, t_end]
__device__ __forceinline__ bool clip_box(const GridDev& g, const float o[3], const float d[3], float t_near, float t_far,
                                         float& t0, float& t_end) {
    const float kInf = __int_as_float(0x7f800000);
    float tmin = -kInf, tmax = kInf;
    bool hit = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float lo = g.org[a], hi = __fadd_rn(g.org[a], __fmul_rn((float)g.n[a], g.vs));
        if (d[a] == 0.0f) {
            if (o[a] < lo || o[a] > hi) hit = false;
            continue;
        }
        const float inv = __fdiv_rn(1.0f, d[a]);
        const float t1 = __fmul_rn(__fsub_rn(lo, o[a]), inv), t2 = __fmul_rn(__fsub_rn(hi, o[a]), inv);
        const float tl = t1 < t2 ? t1 : t2, th = t1 < t2 ? t2 : t1;
        if (tl > tmin) tmin = tl;
        if (th < tmax) tmax = th;
    }
    t0 = t_near > tmin ? t_near : tmin;
    t_end = t_far < tmax ? t_far : tmax;
    return hit && t0 < t_end;
}

}  // namespace
}  // namespace tsdfs
