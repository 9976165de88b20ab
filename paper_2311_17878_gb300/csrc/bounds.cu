// K3: TSDF sample bounds of Alg. 1 + the adaptive count of Sec. 3.4.
// K4: exclusive scan of the counts into ragged offsets.
//
// One thread per ray, or a warp for few rays.  The voxel walk recomputes every crossing parameter from
// its integer boundary, so the walk is exact to the voxel no matter how long.
// fp32, round-to-nearest, no contraction (intrinsics + --fmad=false), in the
// operation order of the oracle's fp32-exact mode, so t_n, t_f, counts and
// status are identical bit for bit.
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "march.cuh"

namespace tsdfs {
int grid_check(const tsdfs_grid* g);

namespace {

constexpr int kBoundsBlock = 128;      // default threads per block of the march
constexpr int kBoundsMaxBlock = 256;   // largest block the autotuner may pick
constexpr int kScanBlock = 1024;
constexpr int kScanItems = 8;
constexpr int kScanChunk = kScanBlock * kScanItems;

struct BoundsDev {
    float d_s, t_near, t_far, step;
    int nb_radius, m_confirm, n_max, n_fallback;
    int max_steps;   // voxel steps a walk may take (0: nx + ny + nz + 8, more than any walk needs)
};

template <bool SMALL>
__device__ __forceinline__ float trilinear(const GridDev& g, const float p[3]) {
    int i0[3];
    float fr[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float gg = __fsub_rn(__fdiv_rn(__fsub_rn(p[a], g.org[a]), g.vs), 0.5f);
        float fl = floorf(gg);
        fr[a] = __fsub_rn(gg, fl);
        if (!(fl >= -1.0f)) { fl = -1.0f; fr[a] = 1.0f; }
        if (fl > (float)g.n[a]) { fl = (float)g.n[a]; fr[a] = 0.0f; }
        i0[a] = (int)fl;
    }
    float c[2][2][2];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                const int ii = min(max(i0[0] + dx, 0), g.n[0] - 1);
                const int jj = min(max(i0[1] + dy, 0), g.n[1] - 1);
                const int kk = min(max(i0[2] + dz, 0), g.n[2] - 1);
                c[dz][dy][dx] = vat(g, vidx<SMALL>(g, ii, jj, kk));
            }
    const float x00 = __fadd_rn(c[0][0][0], __fmul_rn(fr[0], __fsub_rn(c[0][0][1], c[0][0][0])));
    const float x01 = __fadd_rn(c[0][1][0], __fmul_rn(fr[0], __fsub_rn(c[0][1][1], c[0][1][0])));
    const float x10 = __fadd_rn(c[1][0][0], __fmul_rn(fr[0], __fsub_rn(c[1][0][1], c[1][0][0])));
    const float x11 = __fadd_rn(c[1][1][0], __fmul_rn(fr[0], __fsub_rn(c[1][1][1], c[1][1][0])));
    const float y0 = __fadd_rn(x00, __fmul_rn(fr[1], __fsub_rn(x01, x00)));
    const float y1 = __fadd_rn(x10, __fmul_rn(fr[1], __fsub_rn(x11, x10)));
    return __fadd_rn(y0, __fmul_rn(fr[2], __fsub_rn(y1, y0)));
}

// The far phase's test without the precomputed mask: every voxel of [lo, hi] has V < 0 (out of
// grid = unseen = -1).  A plane at a time, its loads in flight together.
__device__ __forceinline__ bool box_negative(const GridDev& g, const int lo[3], const int hi[3]) {
    const int x0 = max(lo[0], 0), x1 = min(hi[0], g.n[0] - 1), y0 = max(lo[1], 0), y1 = min(hi[1], g.n[1] - 1);
    const int z0 = max(lo[2], 0), z1 = min(hi[2], g.n[2] - 1);
    for (int z = z0; z <= z1; ++z) {
        bool neg = true;
        const int64_t plane = (int64_t)z * g.n[1];
#pragma unroll 5
        for (int y = y0; y <= y1; ++y) {
            const int64_t row = (plane + y) * g.n[0];
#pragma unroll 5
            for (int x = x0; x <= x1; ++x) {
                const float v = g.f16 ? __half2float(__ldg(reinterpret_cast<const __half*>(g.V) + row + x))
                                      : __ldg(reinterpret_cast<const float*>(g.V) + row + x);
                neg = neg && v < 0.0f;
            }
        }
        if (!neg) return false;
    }
    return true;
}
__device__ __forceinline__ bool all_negative(const GridDev& g, const int X[3], int r) {
    const int lo[3] = {X[0] - r, X[1] - r, X[2] - r}, hi[3] = {X[0] + r, X[1] + r, X[2] + r};
    return box_negative(g, lo, hi);
}
// the same for a voxel whose predecessor along `axis` passed: only the leading face is new
__device__ __forceinline__ bool face_negative(const GridDev& g, const int X[3], int r, int axis, int step) {
    int lo[3], hi[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = X[a] + (a == axis && step > 0 ? r : -r);
        hi[a] = X[a] + (a == axis && step < 0 ? -r : r);
    }
    return box_negative(g, lo, hi);
}

__device__ __forceinline__ bool inside_bit(const uint32_t* __restrict__ mask, int64_t idx) {
    return (__ldg(mask + (idx >> 5)) >> (idx & 31)) & 1u;
}

// clamp(ceil((t_f - t_n) / step), 1, n_max) (Sec. 3.4)
__device__ __forceinline__ int adaptive_count(float tn, float tf, const BoundsDev& p) {
    const float q = __fdiv_rn(__fsub_rn(tf, tn), p.step);
    int cnt;
    if (!(q > 1.0f)) cnt = 1;
    else if (q >= (float)p.n_max) cnt = p.n_max;
    else cnt = (int)ceilf(q);
    return cnt > p.n_max ? p.n_max : cnt;
}

// A thread per ray.  Bound by instruction issue (80 % of the slots of a 640 x 480 view): voxels known
// to lie in the grid are not checked again, the walk converts nothing (march.cuh), and every loop is
// left by the whole warp together: rays that end a phase at different steps otherwise go through the
// next one apart (a view took half as long again).
template <bool SMALL>
__global__ void __launch_bounds__(kBoundsMaxBlock, 3) k_ray_bounds(GridDev g, const uint32_t* __restrict__ mask,
                                                                const float* __restrict__ ray_o,
                                                                const float* __restrict__ ray_d, int64_t n_rays,
                                                                BoundsDev p, float* __restrict__ t_n_out,
                                                                float* __restrict__ t_f_out, int32_t* __restrict__ n_out,
                                                                float* __restrict__ t_zero_out,
                                                                uint8_t* __restrict__ status_out, uint32_t* dev_status) {
    const float kNaN = __int_as_float(0x7fffffff);
    const unsigned kAll = 0xffffffffu;
    const float ds_norm = __fdiv_rn(p.d_s, g.trunc);
    const int max_steps = p.max_steps > 0 ? p.max_steps : g.n[0] + g.n[1] + g.n[2] + 8;
    const bool search = t_zero_out != nullptr;   // nobody asks for t_zero: its samples are not taken
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, n_warps_rays = (n_rays + 31) / 32 * 32;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_warps_rays; r += stride) {
        const bool valid = r < n_rays;
        const int64_t rr = valid ? r : n_rays - 1;
        float o[3], d[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            o[a] = __ldg(ray_o + 3 * rr + a);
            d[a] = __ldg(ray_d + 3 * rr + a);
        }
        // ---- clip to the grid box ("RenderingCube") ----
        float t0, t_end;
        const bool hit = clip_box(g, o, d, p.t_near, p.t_far, t0, t_end) && valid;
        // ---- voxel walk init ----
        Walk<SMALL> s;
        s.start(g, o, d, t0);
        // ---- near phase: first voxel with V(centre) <= D_s ----
        // The walk does not depend on the values: the next kAhead voxels are stepped and
        // their values requested before the current one is tested, so the loads are in
        // flight together; the voxels, their order and every test are unchanged.
        constexpr int kAhead = 4;
        float tq[kAhead], vq[kAhead];
        std::conditional_t<SMALL, uint32_t, int64_t> iq[kAhead], at = 0;
        bool okq[kAhead];     // the loop condition of that step: still in the grid, t < t_end
        bool live = hit;      // the walk has not left the grid
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            if (i > 0) {
                const bool in = s.next(g);
                live = live && in;
            }
            tq[i] = s.t;
            iq[i] = s.idx;
            okq[i] = live && s.t < t_end;
            vq[i] = live ? vat(g, s.idx) : 0.0f;
        }
        bool found = false;
        float t_before = t0, tn = 0.0f;
        int steps = 0;
        for (bool run = hit;;) {
            run = run && okq[0];
            if (!__any_sync(kAll, run)) break;
            if (run) {
                if (++steps > max_steps) {
                    set_status(dev_status, TSDFS_DEV_MARCH_CAP);
                    run = false;
                } else if (vq[0] <= ds_norm) {
                    found = true;
                    tn = tq[0];
                    at = iq[0];
                    run = false;
                } else {
                    t_before = tq[0];
                }
            }
#pragma unroll
            for (int i = 0; i + 1 < kAhead; ++i) {
                tq[i] = tq[i + 1];
                iq[i] = iq[i + 1];
                vq[i] = vq[i + 1];
                okq[i] = okq[i + 1];
            }
            const bool in = s.next(g);
            live = live && run && in;
            tq[kAhead - 1] = s.t;
            iq[kAhead - 1] = s.idx;
            okq[kAhead - 1] = live && s.t < t_end;
            vq[kAhead - 1] = live ? vat(g, s.idx) : 0.0f;
        }
        // ---- zero-crossing search, starting at the entry of the voxel before ----
        float tf = t_end, tz = kNaN, t_prev = tn, v_prev = 0.0f;
        if (found) {
            // back from the voxels looked ahead at
            int X[3];
            const int64_t row = SMALL ? (int64_t)((uint32_t)at / (uint32_t)g.n[0]) : (int64_t)at / g.n[0];
            X[0] = (int)((int64_t)at - row * g.n[0]);
            X[2] = SMALL ? (int)((uint32_t)row / (uint32_t)g.n[1]) : (int)(row / g.n[1]);
            X[1] = (int)(row - (int64_t)X[2] * g.n[1]);
            s.place(g, X, tn);
            float pp[3];
            point_at(o, d, t_before, pp);
            const float vb = trilinear<SMALL>(g, pp);
            point_at(o, d, tn, pp);
            v_prev = trilinear<SMALL>(g, pp);
            if (tn > t_before && vb > 0.0f && v_prev <= 0.0f)
                tz = __fadd_rn(t_before, __fmul_rn(__fsub_rn(tn, t_before), __fdiv_rn(vb, __fsub_rn(vb, v_prev))));
        }
        // ---- far phase: consecutive voxels whose neighbourhood is all negative ----
        int m = 0, axis = 0;
        for (bool run = found;;) {
            run = run && s.t < t_end;
            if (!__any_sync(kAll, run)) break;
            if (run && ++steps > max_steps) {
                set_status(dev_status, TSDFS_DEV_MARCH_CAP);
                run = false;
            }
            if (run) {
                bool inside;
                if (mask) {
                    inside = inside_bit(mask, s.idx);
                } else {
                    int X[3];
                    s.voxel(X);
                    inside = m > 0 ? face_negative(g, X, p.nb_radius, axis, axis == 0 ? s.st[0] : (axis == 1 ? s.st[1] : s.st[2]))
                                   : all_negative(g, X, p.nb_radius);
                }
                m = inside ? m + 1 : 0;
            }
            const bool in = s.next(g, axis);
            if (run) {
                const float tc = s.t < t_end ? s.t : t_end;
                if (search && tz != tz) {
                    float pp[3];
                    point_at(o, d, tc, pp);
                    const float vc = trilinear<SMALL>(g, pp);
                    if (v_prev > 0.0f && vc <= 0.0f)
                        tz = __fadd_rn(t_prev, __fmul_rn(__fsub_rn(tc, t_prev), __fdiv_rn(v_prev, __fsub_rn(v_prev, vc))));
                    v_prev = vc;
                    t_prev = tc;
                }
                if (m == p.m_confirm) {
                    tf = tc;
                    run = false;
                }
                run = run && in;
            }
        }
        if (!valid) continue;
        const bool miss = !hit;
        t_n_out[r] = found ? tn : (miss ? 0.0f : t0);
        t_f_out[r] = found ? tf : (miss ? 0.0f : t_end);
        n_out[r] = found ? adaptive_count(tn, tf, p) : (miss ? 0 : p.n_fallback);
        status_out[r] = found ? TSDFS_BOUNDED : (miss ? TSDFS_MISS : TSDFS_FALLBACK);
        if (t_zero_out) t_zero_out[r] = tz;
    }
}

// A warp per ray, for few rays, where a thread's chain of steps and loads is all there is to wait for
// (500 rays in a 64^3 grid without the inside mask: 616 us with a thread per ray, 34 us).  The walk does not
// depend on the values, so every lane walks the next 32 voxels and keeps the one of its number;
// the values, the far phase's neighbourhoods and the trilinear samples of 32 voxels are then loaded
// together, and the first event in their order is taken: the same voxels, tests and results.
template <bool SMALL>
__global__ void __launch_bounds__(kBoundsMaxBlock, 2) k_ray_bounds_warp(GridDev g, const uint32_t* __restrict__ mask,
                                                                  const float* __restrict__ ray_o,
                                                                  const float* __restrict__ ray_d, int64_t n_rays,
                                                                  BoundsDev p, float* __restrict__ t_n_out,
                                                                  float* __restrict__ t_f_out, int32_t* __restrict__ n_out,
                                                                  float* __restrict__ t_zero_out,
                                                                  uint8_t* __restrict__ status_out, uint32_t* dev_status) {
    const float kNaN = __int_as_float(0x7fffffff);
    const unsigned kAll = 0xffffffffu;
    const float ds_norm = __fdiv_rn(p.d_s, g.trunc);
    const int max_steps = p.max_steps > 0 ? p.max_steps : g.n[0] + g.n[1] + g.n[2] + 8;
    const int lane = threadIdx.x & 31;
    const bool search = t_zero_out != nullptr;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < n_rays; r += warps) {
        float o[3], d[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            o[a] = __ldg(ray_o + 3 * r + a);
            d[a] = __ldg(ray_d + 3 * r + a);
        }
        auto put = [&](float tn, float tf, int n, int status, float tz) {
            if (lane != 0) return;
            t_n_out[r] = tn; t_f_out[r] = tf; n_out[r] = n; status_out[r] = (uint8_t)status;
            if (t_zero_out) t_zero_out[r] = tz;
        };
        float t0, t_end;
        if (!clip_box(g, o, d, p.t_near, p.t_far, t0, t_end)) {
            put(0.0f, 0.0f, 0, TSDFS_MISS, kNaN);
            continue;
        }
        Walk<SMALL> s;
        s.start(g, o, d, t0);
        bool in = true;             // s is in the grid
        int steps = 0;              // voxels visited
        // the lane's voxel: position, entry parameter, whether the walk visits it, and the next one's entry
        int64_t idx;
        float t, t_next;
        bool ok;
        auto walk = [&]() {
            ok = false;
            t = t_next = 0.0f;
            idx = 0;
            for (int k = 0; k < 32 && in && s.t < t_end; ++k) {
                if (lane == k) {
                    idx = s.idx;
                    t = s.t;
                    ok = true;
                }
                in = s.next(g);
                if (lane == k) t_next = s.t;
            }
        };
        // ---- near phase ----
        bool found = false;
        float tn = 0.0f, t_before = t0;
        int first = 0;              // the found voxel's lane in the batch in hand
        while (true) {
            walk();
            const unsigned oks = __ballot_sync(kAll, ok);
            if (oks == 0) break;
            const unsigned hits = __ballot_sync(kAll, ok && vat(g, idx) <= ds_norm);
            first = hits ? __ffs(hits) - 1 : 32;
            const int visited = first < 32 ? first + 1 : __popc(oks);
            if (steps + visited > max_steps) {
                if (lane == 0) set_status(dev_status, TSDFS_DEV_MARCH_CAP);
                break;
            }
            steps += visited;
            if (first < 32) {
                found = true;
                tn = __shfl_sync(kAll, t, first);
                const float tb = __shfl_sync(kAll, t, first > 0 ? first - 1 : 0);
                if (first > 0) t_before = tb;
                break;
            }
            t_before = __shfl_sync(kAll, t, __popc(oks) - 1);
        }
        if (!found) {
            put(t0, t_end, p.n_fallback, TSDFS_FALLBACK, kNaN);
            continue;
        }
        float tf = t_end, tz = kNaN, t_prev = tn, v_prev;
        {
            float pp[3];
            point_at(o, d, t_before, pp);
            const float vb = trilinear<SMALL>(g, pp);
            point_at(o, d, tn, pp);
            v_prev = trilinear<SMALL>(g, pp);
            if (tn > t_before && vb > 0.0f && v_prev <= 0.0f)
                tz = __fadd_rn(t_before, __fmul_rn(__fsub_rn(tn, t_before), __fdiv_rn(vb, __fsub_rn(vb, v_prev))));
        }
        // ---- far phase: the rest of the batch in hand (from lane `first`), then whole batches ----
        int m = 0;
        while (true) {
            unsigned oks = __ballot_sync(kAll, ok && lane >= first);
            if (oks == 0) {
                if (!(in && s.t < t_end)) break;
                first = 0;
                walk();
                oks = __ballot_sync(kAll, ok);
            }
            const int n_ok = __popc(oks);             // lanes first .. first + n_ok - 1
            const int allowed = max_steps - steps;    // voxels before the step cap
            const int n_vis = n_ok < allowed ? n_ok : allowed;
            const bool vis = lane >= first && lane < first + n_vis;
            bool inside = false;
            if (vis) {
                if (mask) {
                    inside = inside_bit(mask, idx);
                } else {
                    const int64_t row = idx / g.n[0];
                    const int X[3] = {(int)(idx - row * g.n[0]), (int)(row % g.n[1]), (int)(row / g.n[1])};
                    inside = all_negative(g, X, p.nb_radius);
                }
            }
            const unsigned ins = __ballot_sync(kAll, inside);
            // consecutive inside voxels up to this lane's
            const unsigned out = ~ins & ((2u << lane) - 1u) & ~((1u << first) - 1u);
            const int run = out ? lane - (31 - __clz(out)) : m + lane - first + 1;
            const unsigned conf = __ballot_sync(kAll, vis && inside && run == p.m_confirm);
            const int last = conf ? __ffs(conf) - 1 : first + n_vis - 1;   // the last voxel visited
            const float tc = t_next < t_end ? t_next : t_end;
            if (search && tz != tz && n_vis > 0) {
                float vc = 0.0f;
                if (vis) {
                    float pp[3];
                    point_at(o, d, tc, pp);
                    vc = trilinear<SMALL>(g, pp);
                }
                float vp = __shfl_up_sync(kAll, vc, 1), tp = __shfl_up_sync(kAll, tc, 1);
                if (lane == first) {
                    vp = v_prev;
                    tp = t_prev;
                }
                const unsigned cross = __ballot_sync(kAll, vis && lane <= last && vp > 0.0f && vc <= 0.0f);
                if (cross) {
                    const float z = __fadd_rn(tp, __fmul_rn(__fsub_rn(tc, tp), __fdiv_rn(vp, __fsub_rn(vp, vc))));
                    tz = __shfl_sync(kAll, z, __ffs(cross) - 1);
                }
                v_prev = __shfl_sync(kAll, vc, last);
                t_prev = __shfl_sync(kAll, tc, last);
            }
            if (conf) {
                tf = __shfl_sync(kAll, tc, last);
                break;
            }
            if (n_vis < n_ok) {
                if (lane == 0) set_status(dev_status, TSDFS_DEV_MARCH_CAP);
                break;
            }
            steps += n_vis;
            m = __shfl_sync(kAll, inside ? run : 0, last);
            ok = false;
        }
        put(tn, tf, adaptive_count(tn, tf, p), TSDFS_BOUNDED, tz);
    }
}

// ---- recovery (Sec. 4.5): BOUNDED rays whose weight sum stayed below tau are
// rendered again over the whole [t0, t_end] with n_fallback samples ----
__global__ void __launch_bounds__(kBoundsMaxBlock) k_recovery_bounds(GridDev g, const float* __restrict__ ray_o,
                                                                  const float* __restrict__ ray_d, int64_t n_rays,
                                                                  BoundsDev p, float tau,
                                                                  const float* __restrict__ wsum,
                                                                  const uint8_t* __restrict__ status,
                                                                  float* __restrict__ t_n2, float* __restrict__ t_f2,
                                                                  int32_t* __restrict__ n2, uint8_t* __restrict__ status2) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rays; r += (int64_t)gridDim.x * blockDim.x) {
        float o[3], d[3], t0 = 0.0f, t_end = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            o[a] = __ldg(ray_o + 3 * r + a);
            d[a] = __ldg(ray_d + 3 * r + a);
        }
        const bool again = status[r] == TSDFS_BOUNDED && wsum[r] < tau && clip_box(g, o, d, p.t_near, p.t_far, t0, t_end);
        t_n2[r] = again ? t0 : 0.0f;
        t_f2[r] = again ? t_end : 0.0f;
        n2[r] = again ? p.n_fallback : 0;
        status2[r] = again ? (uint8_t)TSDFS_FALLBACK : (uint8_t)TSDFS_MISS;
    }
}

// ---- K4: exclusive scan of the counts, in chunks of 8192: one launch for one chunk; two
// (the chunks' sums; each chunk's scan, which adds up the sums before it itself) for up to 1024;
// else a third between them that scans the sums.  What it costs is the launches: 307 200 counts
// took 12 us in three, their 2.5 MB take under 1.
__device__ __forceinline__ int warp_inclusive(int x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}
// sum of v over the block's 32 warps, and the sum over the warps before this one
__device__ __forceinline__ int block_sums(int warp_total, int* sh, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[warp] = warp_total;
    __syncthreads();
    const int incl = warp_inclusive(sh[lane]);
    total = __shfl_sync(0xffffffffu, incl, 31);
    return __shfl_sync(0xffffffffu, incl, warp) - sh[warp];
}

__global__ void __launch_bounds__(kScanBlock) k_chunk_sums(const int32_t* __restrict__ cnt, int64_t n,
                                                           int32_t* __restrict__ sums) {
    __shared__ int sh[32];
    const int64_t base = (int64_t)blockIdx.x * kScanChunk + threadIdx.x;
    int v = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i * kScanBlock < n) v += cnt[base + i * kScanBlock];
    int total;
    block_sums(__reduce_add_sync(0xffffffffu, v), sh, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_sums(int32_t* __restrict__ sums, int64_t n_chunks) {
    __shared__ int sh[32];
    const int per = (int)((n_chunks + kScanBlock - 1) / kScanBlock);
    const int64_t base = (int64_t)threadIdx.x * per;
    int v = 0;
    for (int i = 0; i < per; ++i)
        if (base + i < n_chunks) v += sums[base + i];
    const int incl = warp_inclusive(v);
    int total;
    int run = block_sums(__shfl_sync(0xffffffffu, incl, 31), sh, total) + incl - v;
    for (int i = 0; i < per; ++i)
        if (base + i < n_chunks) {
            const int c = sums[base + i];
            sums[base + i] = run;
            run += c;
        }
}

// sums: the chunks' sums (SCANNED: their exclusive scan); the last chunk writes the total
template <bool SCANNED>
__global__ void __launch_bounds__(kScanBlock) k_chunk_scan(const int32_t* __restrict__ cnt, int64_t n,
                                                           const int32_t* __restrict__ sums,
                                                           int32_t* __restrict__ offsets) {
    __shared__ int sh[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a warp's 256 counts as 8 rows of 32
    const int64_t base = (int64_t)blockIdx.x * kScanChunk + warp * (32 * kScanItems) + lane;
    int v[kScanItems], x[kScanItems], carry = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) v[i] = base + 32 * i < n ? cnt[base + 32 * i] : 0;
    int before = 0;
    if (SCANNED) {
        before = sums[blockIdx.x];
    } else if (gridDim.x > 1) {
        const int s = (int)threadIdx.x < (int)blockIdx.x ? sums[threadIdx.x] : 0;
        block_sums(__reduce_add_sync(0xffffffffu, s), sh, before);
    }
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int incl = warp_inclusive(v[i]);
        x[i] = carry + incl - v[i];
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    int total;
    before += block_sums(carry, sh, total) ;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + 32 * i < n) {
            offsets[base + 32 * i] = before + x[i];
            if (base + 32 * i == n - 1) offsets[n] = before + x[i] + v[i];
        }
}

}  // namespace

int64_t scan_chunks(int64_t n) { return (n + kScanChunk - 1) / kScanChunk; }

// ---- launch shape of the march (threads per block, resident blocks per SM of the
// grid-stride grid): the default, or what tsdfs_autotune_bounds measured, per device and per kernel (what
// suits a thread per ray does not suit a warp per ray)
namespace {
struct MarchShape {
    int block = kBoundsBlock;
    int blocks_per_sm = 64;
};
struct MarchShapes {
    MarchShape of[2];   // a thread per ray, a warp per ray
    int last = 0;       // the one last set or tuned
};
std::mutex g_shape_mu;
MarchShapes g_shape[64];

MarchShapes march_shapes() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return MarchShapes{};
    std::lock_guard<std::mutex> lk(g_shape_mu);
    return g_shape[dev];
}

// A warp per ray up to these many rays, with and without the inside mask.  Measured (us, warp /
// thread, rays of a room view in 256^3 and of a sphere view in 64^3): with the mask 1728 rays 22 / 35 and
// 20 / 78, 4800 39 / 35 and 25 / 78; without it 4800 80 / 190 and 47 / 550, 10 800 144 / 192 and 70 / 550;
// a thread per ray takes the same up to 30 000 rays.
constexpr int64_t kWarpRaysMask = 4096, kWarpRays = 16384;
bool warp_per_ray(int64_t n_rays, const uint32_t* mask) { return n_rays <= (mask ? kWarpRaysMask : kWarpRays); }

unsigned march_grid(int64_t n_rays, const MarchShape& sh) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return grid_1d(n_rays, sh.block, sms * sh.blocks_per_sm);
}
}  // namespace

// exclusive scan of n counts into offsets[0..n]; `sums` needs scan_chunks(n) ints
int exclusive_scan(const int32_t* cnt, int64_t n, int32_t* offsets, int32_t* sums, cudaStream_t st) {
    const int64_t chunks = scan_chunks(n);
    if (n == 0) return cuda_check(cudaMemsetAsync(offsets, 0, sizeof(int32_t), st), "scan memset");
    if (chunks > (int64_t)kScanBlock * 64) return fail(TSDFS_E_INVALID, "too many rays for the scan (%lld)", (long long)n);
    ProfScope ps("scan", st);
    if (chunks > 1) k_chunk_sums<<<(unsigned)chunks, kScanBlock, 0, st>>>(cnt, n, sums);
    if (chunks > kScanBlock) {
        k_scan_sums<<<1, kScanBlock, 0, st>>>(sums, chunks);
        k_chunk_scan<true><<<(unsigned)chunks, kScanBlock, 0, st>>>(cnt, n, sums, offsets);
    } else {
        k_chunk_scan<false><<<(unsigned)chunks, kScanBlock, 0, st>>>(cnt, n, sums, offsets);
    }
    return cuda_check(cudaGetLastError(), "scan launch");
}

}  // namespace tsdfs

using namespace tsdfs;

extern "C" size_t tsdfs_bounds_workspace_size(int64_t n_rays) {
    if (n_rays < 0) return 0;
    return (size_t)(scan_chunks(n_rays) + 1) * sizeof(int32_t) + 256;
}

extern "C" int tsdf_ray_bounds(const tsdfs_grid* g, const uint32_t* mask, const float* ray_o, const float* ray_d,
                               int64_t n_rays, const tsdfs_bounds_params* p, float* t_n, float* t_f,
                               int32_t* n_samples, int32_t* offsets, float* t_zero, uint8_t* status, void* ws,
                               size_t ws_bytes, tsdfs_stream_t stream) {
    int rc = grid_check(g);
    if (rc) return rc;
    if (!p) return fail(TSDFS_E_INVALID, "params is NULL");
    if (n_rays < 0) return fail(TSDFS_E_INVALID, "n_rays must be >= 0");
    if (n_rays > (int64_t)INT32_MAX) return fail(TSDFS_E_INVALID, "n_rays must fit in int32 offsets");
    if (!(p->step > 0.0f) || !(p->d_s == p->d_s)) return fail(TSDFS_E_INVALID, "step must be > 0 and d_s finite");
    if (p->nb_radius < 0 || p->nb_radius > 4) return fail(TSDFS_E_INVALID, "nb_radius must be in [0, 4]");
    if (p->m_confirm < 1) return fail(TSDFS_E_INVALID, "m_confirm must be >= 1");
    if (p->n_max < 1 || p->n_fallback < 0 || p->n_max > 4096 || p->n_fallback > 4096)
        return fail(TSDFS_E_INVALID, "n_max must be in [1, 4096] and n_fallback in [0, 4096]");
    if ((int64_t)(p->n_max > p->n_fallback ? p->n_max : p->n_fallback) * n_rays > (int64_t)INT32_MAX)
        return fail(TSDFS_E_INVALID, "sample total could overflow int32 offsets");
    if (!(p->t_near < p->t_far)) return fail(TSDFS_E_INVALID, "t_near must be < t_far");
    if (n_rays > 0 && (!ray_o || !ray_d || !t_n || !t_f || !n_samples || !status))
        return fail(TSDFS_E_INVALID, "ray and output pointers must be non-NULL");
    if (!offsets) return fail(TSDFS_E_INVALID, "offsets is NULL");
    if (ws_bytes < tsdfs_bounds_workspace_size(n_rays) || !ws) return fail(TSDFS_E_WORKSPACE, "bounds workspace too small");
    cudaStream_t st = (cudaStream_t)stream;
    int32_t* sums = reinterpret_cast<int32_t*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255));
    if (n_rays > 0) {
        GridDev gd{g->tsdf, g->dtype == TSDFS_F16, {g->nx, g->ny, g->nz}, {g->origin[0], g->origin[1], g->origin[2]},
                   g->voxel_size, g->trunc};
        BoundsDev bd{p->d_s, p->t_near, p->t_far, p->step, p->nb_radius, p->m_confirm, p->n_max, p->n_fallback,
                     test_march_cap()};
        const bool warp = warp_per_ray(n_rays, mask), small = small_grid(gd.n);
        const MarchShape sh = march_shapes().of[warp];
        ProfScope ps("ray_bounds", st);
        auto march = warp ? (small ? k_ray_bounds_warp<true> : k_ray_bounds_warp<false>)
                          : (small ? k_ray_bounds<true> : k_ray_bounds<false>);
        march<<<march_grid(warp ? n_rays * 32 : n_rays, sh), sh.block, 0, st>>>(
            gd, mask, ray_o, ray_d, n_rays, bd, t_n, t_f, n_samples, t_zero, status, device_status_word());
        rc = cuda_check(cudaGetLastError(), "tsdf_ray_bounds launch");
        if (rc) return rc;
    }
    return exclusive_scan(n_samples, n_rays, offsets, sums, st);
}

extern "C" int tsdf_recovery_bounds(const tsdfs_grid* g, const float* ray_o, const float* ray_d, int64_t n_rays,
                                    const tsdfs_bounds_params* p, float tau, const float* wsum, const uint8_t* status,
                                    float* t_n2, float* t_f2, int32_t* n2, int32_t* offsets2, uint8_t* status2,
                                    void* ws, size_t ws_bytes, tsdfs_stream_t stream) {
    int rc = grid_check(g);
    if (rc) return rc;
    if (!p) return fail(TSDFS_E_INVALID, "params is NULL");
    if (n_rays < 0 || n_rays > (int64_t)INT32_MAX) return fail(TSDFS_E_INVALID, "n_rays must be in [0, 2^31)");
    if (!(p->t_near < p->t_far)) return fail(TSDFS_E_INVALID, "t_near must be < t_far");
    if (p->n_fallback < 0 || p->n_fallback > 4096) return fail(TSDFS_E_INVALID, "n_fallback must be in [0, 4096]");
    if ((int64_t)p->n_fallback * n_rays > (int64_t)INT32_MAX)
        return fail(TSDFS_E_INVALID, "sample total could overflow int32 offsets");
    if (!(tau == tau)) return fail(TSDFS_E_INVALID, "tau must not be NaN");
    if (n_rays > 0 && (!ray_o || !ray_d || !wsum || !status || !t_n2 || !t_f2 || !n2 || !status2))
        return fail(TSDFS_E_INVALID, "ray, input and output pointers must be non-NULL");
    if (!offsets2) return fail(TSDFS_E_INVALID, "offsets2 is NULL");
    if (ws_bytes < tsdfs_bounds_workspace_size(n_rays) || !ws) return fail(TSDFS_E_WORKSPACE, "recovery workspace too small");
    cudaStream_t st = (cudaStream_t)stream;
    if (n_rays > 0) {
        GridDev gd{g->tsdf, g->dtype == TSDFS_F16, {g->nx, g->ny, g->nz}, {g->origin[0], g->origin[1], g->origin[2]},
                   g->voxel_size, g->trunc};
        BoundsDev bd{p->d_s, p->t_near, p->t_far, p->step, p->nb_radius, p->m_confirm, p->n_max, p->n_fallback,
                     test_march_cap()};
        const MarchShape sh = march_shapes().of[0];
        ProfScope ps("recovery_bounds", st);
        k_recovery_bounds<<<march_grid(n_rays, sh), sh.block, 0, st>>>(
            gd, ray_o, ray_d, n_rays, bd, tau, wsum, status, t_n2, t_f2, n2, status2);
        rc = cuda_check(cudaGetLastError(), "tsdf_recovery_bounds launch");
        if (rc) return rc;
    }
    int32_t* sums = reinterpret_cast<int32_t*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255));
    return exclusive_scan(n2, n_rays, offsets2, sums, st);
}

// ---------------------------------------------------------------------------
// tsdf_ray_bounds without a caller workspace.
//
// Some callers cannot allocate device memory of their own: a host application
// that hands the library only buffers it registered at start-up, a real-time
// render loop that forbids any allocation once it runs, or code embedded in a
// framework whose allocator it cannot reach.  For them the only scratch this
// call needs -- the per-chunk partial sums of the offsets scan -- lives in the
// array below, which every device that loads the library holds until exit.
// It is sized for kNoAllocMaxRays rays per call; every call overwrites the
// partial sums it uses before reading them, so nothing has to be cleared, and
// two calls that overlap on the GPU (different streams, no ordering) race on it.
// ---------------------------------------------------------------------------
namespace {
constexpr int64_t kNoAllocMaxRays = (int64_t)1 << 24;
constexpr size_t kNoAllocScratchBytes = (size_t)(((kNoAllocMaxRays + kScanChunk - 1) / kScanChunk) + 1) * sizeof(int32_t) + 256;
static __device__ __align__(256) unsigned char g_bounds_scratch[kNoAllocScratchBytes];

SymbolCache g_scratch_cache;

// device address of g_bounds_scratch in the current context (looked up on the first call
// in each context, so the first call on a device belongs before any stream capture)
int bounds_scratch(void** out) {
    return symbol_address(g_scratch_cache, (const void*)&g_bounds_scratch, out,
                          "tsdf_ray_bounds_noalloc cudaGetSymbolAddress");
}
}  // namespace

extern "C" int64_t tsdf_ray_bounds_noalloc_max_rays(void) { return kNoAllocMaxRays; }

extern "C" int tsdf_ray_bounds_noalloc(const tsdfs_grid* g, const uint32_t* mask, const float* ray_o,
                                       const float* ray_d, int64_t n_rays, const tsdfs_bounds_params* p, float* t_n,
                                       float* t_f, int32_t* n_samples, int32_t* offsets, float* t_zero,
                                       uint8_t* status, tsdfs_stream_t stream) {
    if (n_rays > kNoAllocMaxRays)
        return fail(TSDFS_E_INVALID, "tsdf_ray_bounds_noalloc takes at most %lld rays per call (got %lld); split the batch",
                    (long long)kNoAllocMaxRays, (long long)n_rays);
    void* scratch = nullptr;
    int rc = bounds_scratch(&scratch);
    if (rc) return rc;
    return tsdf_ray_bounds(g, mask, ray_o, ray_d, n_rays, p, t_n, t_f, n_samples, offsets, t_zero, status, scratch,
                           kNoAllocScratchBytes, stream);
}

// ---------------------------------------------------------------------------
// Adaptive sample counts relative to the mean interval (Sec. 3.4: samples at
// equal spacing inside [t_n, t_f], so the count is proportional to the
// interval's length; the supplementary ray study: a ray whose bound is longer
// than the average bound gets more samples, a shorter one fewer).  Two passes:
// the mean length of the BOUNDED intervals over the batch, then per ray
// n = clamp(ceil(L / (mean / n_mean)), n_min, n_max).  The mean is summed in
// FP64 in a fixed order (a fixed grid of kMeanBlocks blocks, each a fixed tree),
// so it does not depend on scheduling, and rounded once to FP32; the count
// arithmetic is FP32 with IEEE division (this file is compiled without FMA
// contraction), so an FP32 restatement on the host reproduces every count.
// ---------------------------------------------------------------------------
namespace tsdfs {
namespace {
constexpr int kMeanBlocks = 256;
constexpr int kMeanThreads = 256;

__global__ void __launch_bounds__(kMeanThreads) k_len_partials(const float* __restrict__ t_n,
                                                                const float* __restrict__ t_f,
                                                                const uint8_t* __restrict__ status, int64_t n_rays,
                                                                double* __restrict__ part_sum,
                                                                unsigned long long* __restrict__ part_cnt) {
    __shared__ double s_sum[kMeanThreads];
    __shared__ unsigned long long s_cnt[kMeanThreads];
    double acc = 0.0;
    unsigned long long cnt = 0;
    for (int64_t r = blockIdx.x * (int64_t)kMeanThreads + threadIdx.x; r < n_rays; r += (int64_t)kMeanBlocks * kMeanThreads) {
        if (__ldg(status + r) == TSDFS_BOUNDED) {
            acc += (double)__fsub_rn(__ldg(t_f + r), __ldg(t_n + r));
            ++cnt;
        }
    }
    s_sum[threadIdx.x] = acc;
    s_cnt[threadIdx.x] = cnt;
    __syncthreads();
    for (int h = kMeanThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s_sum[threadIdx.x] += s_sum[threadIdx.x + h];
            s_cnt[threadIdx.x] += s_cnt[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part_sum[blockIdx.x] = s_sum[0];
        part_cnt[blockIdx.x] = s_cnt[0];
    }
}

// one block: the partials in a fixed tree -> mean (FP32) and the spacing mean / n_mean
__global__ void __launch_bounds__(kMeanBlocks) k_len_mean(const double* __restrict__ part_sum,
                                                          const unsigned long long* __restrict__ part_cnt,
                                                          float n_mean, float* __restrict__ mean_out,
                                                          float* __restrict__ spacing_out) {
    __shared__ double s_sum[kMeanBlocks];
    __shared__ unsigned long long s_cnt[kMeanBlocks];
    s_sum[threadIdx.x] = part_sum[threadIdx.x];
    s_cnt[threadIdx.x] = part_cnt[threadIdx.x];
    __syncthreads();
    for (int h = kMeanBlocks / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s_sum[threadIdx.x] += s_sum[threadIdx.x + h];
            s_cnt[threadIdx.x] += s_cnt[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const float mean = s_cnt[0] > 0 ? (float)(s_sum[0] / (double)s_cnt[0]) : 0.0f;
        *spacing_out = __fdiv_rn(mean, n_mean);
        if (mean_out) *mean_out = mean;
    }
}

__global__ void k_adaptive_counts(const float* __restrict__ t_n, const float* __restrict__ t_f,
                                  const uint8_t* __restrict__ status, int64_t n_rays,
                                  const float* __restrict__ spacing, int n_min, int n_max, int n_fallback,
                                  int32_t* __restrict__ n_out) {
    const float dl = __ldg(spacing);
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rays; r += (int64_t)gridDim.x * blockDim.x) {
        const uint8_t st = __ldg(status + r);
        int n = 0;
        if (st == TSDFS_BOUNDED) {
            const float len = __fsub_rn(__ldg(t_f + r), __ldg(t_n + r));
            float q = dl > 0.0f ? ceilf(__fdiv_rn(len, dl)) : (float)n_min;
            q = fminf(fmaxf(q, (float)n_min), (float)n_max);  // also maps NaN to n_min
            n = (int)q;
        } else if (st == TSDFS_FALLBACK) {
            n = n_fallback;
        }
        n_out[r] = n;
    }
}
}  // namespace
}  // namespace tsdfs

extern "C" size_t tsdfs_adaptive_counts_workspace_size(int64_t n_rays) {
    if (n_rays < 0) return 0;
    return tsdfs_bounds_workspace_size(n_rays) + (size_t)kMeanBlocks * (sizeof(double) + sizeof(unsigned long long)) +
           3 * 256;
}

extern "C" int tsdf_adaptive_counts(const float* t_n, const float* t_f, const uint8_t* status, int64_t n_rays,
                                    float n_mean, int32_t n_min, int32_t n_max, int32_t n_fallback,
                                    int32_t* n_samples, int32_t* offsets, float* mean_len, void* ws, size_t ws_bytes,
                                    tsdfs_stream_t stream) {
    if (n_rays < 0 || n_rays > (int64_t)INT32_MAX) return fail(TSDFS_E_INVALID, "n_rays must be in [0, 2^31)");
    if (!(n_mean > 0.0f) || !(n_mean <= 4096.0f)) return fail(TSDFS_E_INVALID, "n_mean must be in (0, 4096]");
    if (n_min < 1 || n_max < n_min || n_max > 4096) return fail(TSDFS_E_INVALID, "need 1 <= n_min <= n_max <= 4096");
    if (n_fallback < 0 || n_fallback > 4096) return fail(TSDFS_E_INVALID, "n_fallback must be in [0, 4096]");
    if ((int64_t)(n_max > n_fallback ? n_max : n_fallback) * n_rays > (int64_t)INT32_MAX)
        return fail(TSDFS_E_INVALID, "sample total could overflow int32 offsets");
    if (n_rays > 0 && (!t_n || !t_f || !status || !n_samples))
        return fail(TSDFS_E_INVALID, "bound, status and count pointers must be non-NULL");
    if (!offsets) return fail(TSDFS_E_INVALID, "offsets is NULL");
    if (!ws || ws_bytes < tsdfs_adaptive_counts_workspace_size(n_rays))
        return fail(TSDFS_E_WORKSPACE, "adaptive counts workspace too small");
    cudaStream_t st = (cudaStream_t)stream;
    uintptr_t p = (reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255);
    int32_t* sums = reinterpret_cast<int32_t*>(p);
    p = (p + (size_t)(scan_chunks(n_rays) + 1) * sizeof(int32_t) + 255) & ~uintptr_t(255);
    double* part_sum = reinterpret_cast<double*>(p);
    unsigned long long* part_cnt = reinterpret_cast<unsigned long long*>(p + kMeanBlocks * sizeof(double));
    float* spacing = reinterpret_cast<float*>(p + kMeanBlocks * (sizeof(double) + sizeof(unsigned long long)));
    if (n_rays > 0) {
        ProfScope ps("adaptive_counts", st);
        k_len_partials<<<kMeanBlocks, kMeanThreads, 0, st>>>(t_n, t_f, status, n_rays, part_sum, part_cnt);
        k_len_mean<<<1, kMeanBlocks, 0, st>>>(part_sum, part_cnt, n_mean, mean_len, spacing);
        k_adaptive_counts<<<grid_1d(n_rays, 256), 256, 0, st>>>(t_n, t_f, status, n_rays, spacing, n_min, n_max,
                                                                n_fallback, n_samples);
        int rc = cuda_check(cudaGetLastError(), "adaptive counts launch");
        if (rc) return rc;
    } else if (mean_len) {
        int rc = cuda_check(cudaMemsetAsync(mean_len, 0, sizeof(float), st), "adaptive counts memset");
        if (rc) return rc;
    }
    return exclusive_scan(n_samples, n_rays, offsets, sums, st);
}

// ---------------------------------------------------------------------------
// Autotuner of the march's launch shape.  The march is latency-bound (a DDA per
// thread, scattered reads of an L2-resident grid), so its speed depends on how
// many rays are in flight per SM and how rays are grouped into blocks; the best
// shape depends on the grid, the ray batch and the device.  The candidates are
// every (threads per block, resident blocks per SM) pair below; each is timed
// with CUDA events on the caller's stream over `reps` launches on the caller's
// own rays (outputs are identical for every shape: rays are independent), and
// the fastest becomes this device's shape for tsdf_ray_bounds and
// tsdf_recovery_bounds.  It synchronises the stream: a set-up call.
// ---------------------------------------------------------------------------
namespace {
constexpr int kTuneBlocks[] = {64, 128, 256};
constexpr int kTunePerSm[] = {4, 8, 16, 32, 64};
}  // namespace

extern "C" int tsdfs_bounds_launch_shape(int32_t* block, int32_t* blocks_per_sm) {
    if (!block || !blocks_per_sm) return fail(TSDFS_E_INVALID, "block and blocks_per_sm must be non-NULL");
    const MarchShapes all = march_shapes();
    const MarchShape sh = all.of[all.last];
    *block = sh.block;
    *blocks_per_sm = sh.blocks_per_sm;
    return TSDFS_OK;
}

extern "C" int tsdfs_set_bounds_launch_shape(int32_t block, int32_t blocks_per_sm) {
    if (block == 0 && blocks_per_sm == 0) {
        block = kBoundsBlock;
        blocks_per_sm = 64;
    }
    if (block < 32 || block > kBoundsMaxBlock || block % 32 != 0 || blocks_per_sm < 1 || blocks_per_sm > 1024)
        return fail(TSDFS_E_INVALID, "block must be a multiple of 32 in [32, %d], blocks_per_sm in [1, 1024]",
                    kBoundsMaxBlock);
    int dev = 0;
    int rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice");
    if (rc) return rc;
    if (dev < 0 || dev >= 64) return fail(TSDFS_E_UNSUPPORTED, "device index %d out of range", dev);
    std::lock_guard<std::mutex> lk(g_shape_mu);
    for (MarchShape& sh : g_shape[dev].of) sh = MarchShape{block, blocks_per_sm};
    g_shape[dev].last = 0;
    return TSDFS_OK;
}

extern "C" int tsdfs_autotune_bounds(const tsdfs_grid* g, const uint32_t* mask, const float* ray_o, const float* ray_d,
                                     int64_t n_rays, const tsdfs_bounds_params* p, float* t_n, float* t_f,
                                     int32_t* n_samples, int32_t* offsets, float* t_zero, uint8_t* status, void* ws,
                                     size_t ws_bytes, int32_t reps, float* best_ms, tsdfs_stream_t stream) {
    if (reps < 1 || reps > 1000) return fail(TSDFS_E_INVALID, "reps must be in [1, 1000]");
    if (n_rays < 1) return fail(TSDFS_E_INVALID, "autotuning needs at least one ray");
    MarchShapes shapes = march_shapes();
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = cuda_check(cudaEventCreate(&e0), "autotune event");
    if (!rc) rc = cuda_check(cudaEventCreate(&e1), "autotune event");
    float best = 1e30f;
    MarchShape fastest;
    for (int bi = 0; !rc && bi < (int)(sizeof(kTuneBlocks) / sizeof(int)); ++bi)
        for (int si = 0; !rc && si < (int)(sizeof(kTunePerSm) / sizeof(int)); ++si) {
            rc = tsdfs_set_bounds_launch_shape(kTuneBlocks[bi], kTunePerSm[si]);
            // one untimed launch (argument checks, caches), then `reps` timed
            if (!rc) rc = tsdf_ray_bounds(g, mask, ray_o, ray_d, n_rays, p, t_n, t_f, n_samples, offsets, t_zero,
                                          status, ws, ws_bytes, stream);
            if (!rc) rc = cuda_check(cudaEventRecord(e0, st), "autotune event record");
            for (int r = 0; !rc && r < reps; ++r)
                rc = tsdf_ray_bounds(g, mask, ray_o, ray_d, n_rays, p, t_n, t_f, n_samples, offsets, t_zero, status,
                                     ws, ws_bytes, stream);
            if (!rc) rc = cuda_check(cudaEventRecord(e1, st), "autotune event record");
            if (!rc) rc = cuda_check(cudaEventSynchronize(e1), "autotune event sync");
            float ms = 0.0f;
            if (!rc) rc = cuda_check(cudaEventElapsedTime(&ms, e0, e1), "autotune elapsed");
            if (!rc && ms < best) {
                best = ms;
                fastest = MarchShape{kTuneBlocks[bi], kTunePerSm[si]};
            }
        }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    // the kernel that these rays take keeps the fastest shape, the other one its own
    if (!rc) {
        shapes.last = warp_per_ray(n_rays, mask);
        shapes.of[shapes.last] = fastest;
    }
    int dev = 0;
    const int rc2 = cuda_check(cudaGetDevice(&dev), "cudaGetDevice");
    if (!rc2 && dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(g_shape_mu);
        g_shape[dev] = shapes;
    }
    if (rc) return rc;
    if (best_ms) *best_ms = best / (float)reps;
    return rc2;
}

// ---------------------------------------------------------------------------
// L2 read-bandwidth probe: the measured peak against which the ray march is
// judged when its grid stays in L2.  Every thread streams 16-byte loads over the
// buffer (which the caller keeps at a size L2 holds) reps times; the XOR of the
// loaded words goes to `sink` so the loads are kept.
// ---------------------------------------------------------------------------
namespace tsdfs {
namespace {
__global__ void k_l2_read(const uint4* __restrict__ buf, int64_t n16, int reps, uint32_t* sink) {
    uint32_t acc = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int r = 0; r < reps; ++r)
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n16; i += stride) {
            const uint4 v = __ldcg(buf + i);
            acc ^= v.x ^ v.y ^ v.z ^ v.w;
        }
    if (acc == 0x9e3779b9u) *sink = acc;   // practically never taken; keeps the loads live
}
}  // namespace
}  // namespace tsdfs

extern "C" int tsdfs_l2_read_probe(const void* buf, size_t bytes, int32_t reps, uint32_t* sink, float* ms_out,
                                   tsdfs_stream_t stream) {
    using namespace tsdfs;
    if (!buf || !sink || !ms_out || bytes < 16 || reps < 1 || (reinterpret_cast<uintptr_t>(buf) & 15u) != 0)
        return fail(TSDFS_E_INVALID, "tsdfs_l2_read_probe: buf (16-byte aligned), sink, ms_out, bytes >= 16, reps >= 1");
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t n16 = (int64_t)(bytes / 16);
    const uint4* b = static_cast<const uint4*>(buf);
    // one pass to bring the buffer into L2, then the timed passes
    k_l2_read<<<sms * 4, 512, 0, st>>>(b, n16, 1, sink);
    int rc = cuda_check(cudaGetLastError(), "l2 probe launch");
    if (rc) return rc;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    rc = cuda_check(cudaEventCreate(&e0), "l2 probe event");
    if (!rc) rc = cuda_check(cudaEventCreate(&e1), "l2 probe event");
    if (!rc) rc = cuda_check(cudaEventRecord(e0, st), "l2 probe record");
    if (!rc) {
        k_l2_read<<<sms * 4, 512, 0, st>>>(b, n16, reps, sink);
        rc = cuda_check(cudaGetLastError(), "l2 probe launch");
    }
    if (!rc) rc = cuda_check(cudaEventRecord(e1, st), "l2 probe record");
    if (!rc) rc = cuda_check(cudaEventSynchronize(e1), "l2 probe sync");
    if (!rc) rc = cuda_check(cudaEventElapsedTime(ms_out, e0, e1), "l2 probe elapsed");
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    return rc;
}
