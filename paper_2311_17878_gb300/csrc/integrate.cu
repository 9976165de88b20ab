// K1: projective TSDF fusion (Sec. 3.2, Eq. 3, Alg. 2 in its per-voxel form)
// K2: the far-phase neighbourhood test of Alg. 1 as a bit mask.
//
// K1 arithmetic is IEEE fp32 round-to-nearest with no contraction (explicit
// __f*_rn intrinsics, and this file is compiled with --fmad=false), in the
// operation order that tsdfs.h documents, so pixel choices, weights and
// values are reproducible bit for bit.
#include "common.cuh"
#include "march.cuh"

namespace tsdfs {

namespace {

constexpr int kFuseBlock = 256;

__device__ __forceinline__ float load_v(const void* V, int f16, int64_t idx) {
    return f16 ? __half2float(reinterpret_cast<const __half*>(V)[idx]) : reinterpret_cast<const float*>(V)[idx];
}
__device__ __forceinline__ void store_v(void* V, int f16, int64_t idx, float v) {
    if (f16) reinterpret_cast<__half*>(V)[idx] = __float2half_rn(v);
    else reinterpret_cast<float*>(V)[idx] = v;
}

__global__ void k_grid_init(void* V, int f16, uint8_t* W, int64_t n) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        store_v(V, f16, q, -1.0f);
        W[q] = 0;
    }
}

// Projective fusion, brick by brick.  A camera inside a room sees about a tenth of its voxels, and
// what a voxel-view costs is the projection's IEEE divisions and square root (~170 instructions in
// all).  So:
//  - a block takes a brick of 8 x 8 x 8 voxels and first tests every view against it (a view per
//    thread; the image's four side planes and the camera plane as linear functions over a box); only
//    the views that may see it are run per voxel, in their order, and a brick that no view sees is not
//    read.  A view is left out only if every voxel of the brick fails the per-voxel tests: a plane's
//    bound is widened by 1e-5 of the sum of its terms' magnitudes, some 20 times the FP32 rounding
//    of the per-voxel arithmetic, and a NaN keeps the view;
//  - the pixel comes from an approximate reciprocal wherever u and v are not within its error of a
//    whole number, and from the divisions elsewhere (the same pixel either way);
//  - a depth that is more than D_T (and the rounding) in front of or behind the voxel needs no
//    projection onto the ray: the voxel is skipped, or s is D_T and s / D_T is 1; and a voxel whose
//    mean is 1 keeps it.
// The camera table of all views is staged in shared memory once per block (20 floats per view:
// c2w[12], fx, fy, cx, cy and what the tests use), the list of the brick's views after it.  256^3
// voxels, 100 views of the room: 2816 us without any of it, 950 with bricks of 32 x 4 x 4, 844 as it
// is in 152 x 8 blocks and 645 in kFuseBlocks; what is left is the ~40 instructions of a voxel-view and
// the divisions near the surface.
constexpr int kBX = 8, kBY = 8, kBZ = 8;
constexpr int kBrickVoxels = kBX * kBY * kBZ;
constexpr int kCam = 20;
// Blocks at most.  Five are resident on an SM, and bricks differ in their views: 152 x 8 blocks are
// 1.6 rounds of equal shares (the SMs idle for 15 % of the time), 20 rounds even out, and staging the
// table once per block still costs less than that.  256^3, 100 views / 300 x 225 x 121, 3 views: 152 x 5
// blocks 770 / 102 us, x 8 846 / 72, x 32 680 / 56, x 108 645 / 56, x 216 648 / 56.
constexpr int kFuseBlocks = 152 * 5 * 20;
// k_integrate_few (figures there): views staged at a time; the voxels up to which and the views above which it
// is taken.  640 views' table is 52 KB: four blocks of k_integrate on an SM instead of five.
constexpr int kViewChunk = 256;
constexpr int64_t kFewVoxels = 64 * 64 * 64;
constexpr int kManyViews = 640;

// whether view P can see a voxel centre within h[3] of c[3]
__device__ __forceinline__ bool brick_visible(const float* P, const float c[3], const float h[3], float fW, float fH) {
    float x = 0.0f, y = 0.0f, z = 0.0f;          // camera coordinates of the centre
    float ax = 0.0f, ay = 0.0f, az = 0.0f;       // sums of their terms' magnitudes over the brick
    float d[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        d[k] = c[k] - P[4 * k + 3];
        const float m = fabsf(c[k]) + fabsf(P[4 * k + 3]) + h[k];
        x += P[4 * k] * d[k];
        y += P[4 * k + 1] * d[k];
        z += P[4 * k + 2] * d[k];
        ax += fabsf(P[4 * k]) * m;
        ay += fabsf(P[4 * k + 1]) * m;
        az += fabsf(P[4 * k + 2]) * m;
    }
    const float fx = P[12], fy = P[13], cx = P[14], cy = P[15];
    float rz = 0.0f, rl = 0.0f, rr = 0.0f, rt = 0.0f, rb = 0.0f;   // half ranges over the brick
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        rz += fabsf(P[4 * k + 2]) * h[k];
        rl += fabsf(fx * P[4 * k] + cx * P[4 * k + 2]) * h[k];
        rr += fabsf(fx * P[4 * k] + (cx - fW) * P[4 * k + 2]) * h[k];
        rt += fabsf(fy * P[4 * k + 1] + cy * P[4 * k + 2]) * h[k];
        rb += fabsf(fy * P[4 * k + 1] + (cy - fH) * P[4 * k + 2]) * h[k];
    }
    constexpr float kSlack = 1e-5f;
    const float su = kSlack * (fabsf(fx) * ax + (fabsf(cx) + fW) * az), sv = kSlack * (fabsf(fy) * ay + (fabsf(cy) + fH) * az);
    if (z + rz + kSlack * az < 0.0f) return false;                        // behind the camera
    if (fx * x + cx * z + rl + su < 0.0f) return false;                   // u < 0 throughout
    if (fx * x + (cx - fW) * z - rr - su > 0.0f) return false;            // u > W
    if (fy * y + cy * z + rt + sv < 0.0f) return false;
    if (fy * y + (cy - fH) * z - rb - sv > 0.0f) return false;
    return true;
}

__global__ void __launch_bounds__(kFuseBlock) k_integrate(int nx, int ny, int nz, float ox, float oy, float oz,
                                                          float vs, float trunc, void* V, int f16, uint8_t* W,
                                                          const float* __restrict__ depth, int nv, int H, int Wd,
                                                          const float* __restrict__ Kc, const float* __restrict__ c2w) {
    extern __shared__ float cam[];
    uint16_t* list = reinterpret_cast<uint16_t*>(cam + nv * kCam);
    __shared__ int s_warp[kFuseBlock / 32];
    for (int v = threadIdx.x; v < nv; v += blockDim.x) {
        float* P = cam + v * kCam;
        for (int c = 0; c < 12; ++c) P[c] = c2w[v * 12 + c];
        for (int c = 0; c < 4; ++c) P[12 + c] = Kc[v * 4 + c];
        // the voxel's range times cos(angle to its pixel's ray) is the projection: the pixel's half
        // diagonal bounds the angle, 1e-5 the rounding
        const float hx = 0.5f / P[12], hy = 0.5f / P[13];
        P[16] = 1.0f - 1.1f * (hx * hx + hy * hy) - 1e-5f;     // least (projection / range)^2
        P[17] = 1e-5f * fabsf(P[14]) + 1e-4f;                  // error of the approximate u, v: plus 1e-5 of them
        P[18] = 1e-5f * fabsf(P[15]) + 1e-4f;
    }
    const int bx = (nx + kBX - 1) / kBX, by = (ny + kBY - 1) / kBY, bz = (nz + kBZ - 1) / kBZ;
    const int64_t bricks = (int64_t)bx * by * bz;
    const float fW = (float)Wd, fH = (float)H;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t br = blockIdx.x; br < bricks; br += gridDim.x) {
        const int i0 = (int)(br % bx) * kBX, j0 = (int)((br / bx) % by) * kBY, k0 = (int)(br / ((int64_t)bx * by)) * kBZ;
        const float h[3] = {0.5f * kBX * vs, 0.5f * kBY * vs, 0.5f * kBZ * vs};
        const float c[3] = {ox + ((float)i0 + 0.5f * kBX) * vs, oy + ((float)j0 + 0.5f * kBY) * vs,
                            oz + ((float)k0 + 0.5f * kBZ) * vs};
        // the brick's views, in order
        int n_list = 0;
        for (int v0 = 0; v0 < nv; v0 += kFuseBlock) {
            __syncthreads();   // the table; the last brick's list; s_warp
            const int v = v0 + (int)threadIdx.x;
            const bool keep = v < nv && brick_visible(cam + v * kCam, c, h, fW, fH);
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) s_warp[warp] = __popc(m);
            __syncthreads();
            int before = n_list, all = 0;
#pragma unroll
            for (int w = 0; w < kFuseBlock / 32; ++w) {
                const int n = s_warp[w];
                before += w < warp ? n : 0;
                all += n;
            }
            if (keep) list[before + __popc(m & ((1u << lane) - 1u))] = (uint16_t)v;
            n_list += all;
        }
        if (n_list == 0) continue;
        __syncthreads();
        for (int e = threadIdx.x; e < kBrickVoxels; e += kFuseBlock) {
            const int i = i0 + (e % kBX), j = j0 + (e / kBX) % kBY, k = k0 + e / (kBX * kBY);
            if (i >= nx || j >= ny || k >= nz) continue;
            const int64_t q = ((int64_t)k * ny + j) * nx + i;
            const float cx = __fadd_rn(ox, __fmul_rn(__fadd_rn((float)i, 0.5f), vs));
            const float cy = __fadd_rn(oy, __fmul_rn(__fadd_rn((float)j, 0.5f), vs));
            const float cz = __fadd_rn(oz, __fmul_rn(__fadd_rn((float)k, 0.5f), vs));
            float Vv = load_v(V, f16, q);
            int Wv = W[q];
            for (int l = 0; l < n_list; ++l) {
                const int view = list[l];
                const float* P = cam + view * kCam;
                const float dx = __fsub_rn(cx, P[3]), dy = __fsub_rn(cy, P[7]), dz = __fsub_rn(cz, P[11]);
                const float zc = __fadd_rn(__fadd_rn(__fmul_rn(P[2], dx), __fmul_rn(P[6], dy)), __fmul_rn(P[10], dz));
                if (!(zc > 0.0f)) continue;
                const float xc = __fadd_rn(__fadd_rn(__fmul_rn(P[0], dx), __fmul_rn(P[4], dy)), __fmul_rn(P[8], dz));
                const float yc = __fadd_rn(__fadd_rn(__fmul_rn(P[1], dx), __fmul_rn(P[5], dy)), __fmul_rn(P[9], dz));
                const float fx = P[12], fy = P[13], ccx = P[14], ccy = P[15];
                // the pixel: floor(u), floor(v)
                const float rz = __fdividef(1.0f, zc);
                const float ua = fmaf(fx * xc, rz, ccx), va = fmaf(fy * yc, rz, ccy);
                float fu = floorf(ua), fv = floorf(va);
                const float eu = fmaf(1e-5f, fabsf(ua), P[17]), ev = fmaf(1e-5f, fabsf(va), P[18]);
                const float ru = ua - fu, rv = va - fv;
                if (!(ru > eu && ru < 1.0f - eu && rv > ev && rv < 1.0f - ev)) {
                    const float u = __fadd_rn(__fmul_rn(fx, __fdiv_rn(xc, zc)), ccx);
                    const float v = __fadd_rn(__fmul_rn(fy, __fdiv_rn(yc, zc)), ccy);
                    if (!(u >= 0.0f && u < fW && v >= 0.0f && v < fH)) continue;
                    fu = floorf(u);
                    fv = floorf(v);
                }
                if (!(fu >= 0.0f && fu < fW && fv >= 0.0f && fv < fH)) continue;
                const int px = min((int)fu, Wd - 1), py = min((int)fv, H - 1);
                const float D = __ldg(depth + ((int64_t)view * H + py) * Wd + px);
                // far behind the surface: proj >= range * cos > D + D_T
                const float range2 = fmaf(xc, xc, fmaf(yc, yc, zc * zc)), reach = D + trunc;
                if (reach >= 0.0f && reach * reach < range2 * P[16]) continue;
                float sn = 1.0f;
                // far before it: proj <= range < D - D_T, so s is cut to D_T
                const float room = D - trunc;
                if (!(room > 0.0f && room * room > range2 * 1.00001f)) {
                    const float a = __fdiv_rn(__fsub_rn(__fadd_rn((float)px, 0.5f), ccx), fx);
                    const float b = __fdiv_rn(__fsub_rn(__fadd_rn((float)py, 0.5f), ccy), fy);
                    const float nrm = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)), 1.0f));
                    const float proj = __fdiv_rn(__fadd_rn(__fadd_rn(__fmul_rn(a, xc), __fmul_rn(b, yc)), zc), nrm);
                    float s = __fsub_rn(D, proj);
                    if (s > trunc) s = trunc;
                    if (s < -trunc) s = -trunc;
                    if (!(s > -trunc)) continue;
                    sn = __fdiv_rn(s, trunc);
                }
                const float Wf = (float)Wv;
                // (W + 1) / (W + 1)
                if (!(sn == 1.0f && Vv == 1.0f))
                    Vv = __fdiv_rn(__fadd_rn(__fmul_rn(Wf, Vv), sn), __fadd_rn(Wf, 1.0f));
                if (Wv < 255) ++Wv;
            }
            store_v(V, f16, q, Vv);
            W[q] = (uint8_t)Wv;
        }
    }
}

// Few voxels, thin grids, many views: a brick of 2^lx x 2^ly x 2^(8 - lx - ly) voxels, one to a thread, shaped to
// the grid (bricks of 8 x 8 x 8 leave 7 of 8 threads idle in a grid one voxel thick, and a grid of 16^3 is 8 of
// them: then a voxel's chain of views is all there is to wait for); and at most kViewChunk views staged at a
// time, so that their table does not cost resident blocks.  The pixel and the projection are taken at once by the
// divisions: that chain is shorter than the approximations' with their branches, and the projection's is done
// while the depth is on its way.
// Measured (us, k_integrate / this; 100 views unless said otherwise; a sphere that all views see whole): 16^3 125 /
// 53, 48^3 137 / 75, 64^3 174 / 152 and with 12 views 28.7 / 28.8, 512 x 512 x 1 182 / 144, 1 x 512 x 512 694 / 146,
// 64^3 with 2048 views 6919 / 2877, 192^3 with 1000 38.5 / 31.8 ms; the room: 48^3 45 / 23, 64^3 47 / 30, 192^3 with
// 1000 views 3.72 / 3.25 ms.  Above 64^3 voxels it depends on the views (80^3 of the room, 12 views 18.5 / 19.8,
// 100 views 51 / 43), and soon no more: 96^3 with 12 views 22.6 / 28.7, 256^3 with 100 665 / 814.
__global__ void __launch_bounds__(kFuseBlock) k_integrate_few(int nx, int ny, int nz, int lx, int ly, float ox, float oy,
                                                              float oz, float vs, float trunc, void* V, int f16, uint8_t* W,
                                                              const float* __restrict__ depth, int nv, int H, int Wd,
                                                              const float* __restrict__ Kc, const float* __restrict__ c2w) {
    __shared__ float cam[kViewChunk * 16];
    __shared__ uint16_t list[kViewChunk];
    __shared__ int s_warp[kFuseBlock / 32];
    static_assert(kViewChunk == kFuseBlock, "a view per thread");
    const int sx = 1 << lx, sy = 1 << ly, sz = kFuseBlock >> (lx + ly);
    const int bx = (nx - 1) / sx + 1, by = (ny - 1) / sy + 1, bz = (nz - 1) / sz + 1;
    const int64_t bricks = (int64_t)bx * by * bz;
    const float fW = (float)Wd, fH = (float)H;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t br = blockIdx.x; br < bricks; br += gridDim.x) {
        const int i0 = (int)(br % bx) * sx, j0 = (int)((br / bx) % by) * sy, k0 = (int)(br / ((int64_t)bx * by)) * sz;
        const float h[3] = {0.5f * (float)sx * vs, 0.5f * (float)sy * vs, 0.5f * (float)sz * vs};
        const float c[3] = {ox + ((float)i0 + 0.5f * (float)sx) * vs, oy + ((float)j0 + 0.5f * (float)sy) * vs,
                            oz + ((float)k0 + 0.5f * (float)sz) * vs};
        const int i = i0 + ((int)threadIdx.x & (sx - 1)), j = j0 + (((int)threadIdx.x >> lx) & (sy - 1));
        const int k = k0 + ((int)threadIdx.x >> (lx + ly));
        const bool voxel = i < nx && j < ny && k < nz;
        const int64_t q = ((int64_t)k * ny + j) * nx + i;
        const float cx = __fadd_rn(ox, __fmul_rn(__fadd_rn((float)i, 0.5f), vs));
        const float cy = __fadd_rn(oy, __fmul_rn(__fadd_rn((float)j, 0.5f), vs));
        const float cz = __fadd_rn(oz, __fmul_rn(__fadd_rn((float)k, 0.5f), vs));
        float Vv = 0.0f;
        int Wv = 0;
        bool seen = false;   // by a view; the voxel stays in registers from chunk to chunk
        for (int v0 = 0; v0 < nv; v0 += kViewChunk) {
            const int views = nv - v0 < kViewChunk ? nv - v0 : kViewChunk;
            __syncthreads();   // the last list and its table; s_warp
            if (nv > kViewChunk || br == blockIdx.x) {
                for (int e = threadIdx.x; e < views * 16; e += kFuseBlock) {
                    const int v = v0 + (e >> 4), a = e & 15;
                    cam[e] = a < 12 ? c2w[v * 12 + a] : Kc[v * 4 + (a - 12)];
                }
                __syncthreads();
            }
            const bool keep = (int)threadIdx.x < views && brick_visible(cam + threadIdx.x * 16, c, h, fW, fH);
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) s_warp[warp] = __popc(m);
            __syncthreads();
            int before = 0, n_list = 0;
#pragma unroll
            for (int w = 0; w < kFuseBlock / 32; ++w) {
                const int n = s_warp[w];
                before += w < warp ? n : 0;
                n_list += n;
            }
            if (n_list == 0) continue;
            if (keep) list[before + __popc(m & ((1u << lane) - 1u))] = (uint16_t)threadIdx.x;
            __syncthreads();
            if (voxel && !seen) {
                Vv = load_v(V, f16, q);
                Wv = W[q];
            }
            seen = true;
            for (int l = 0; voxel && l < n_list; ++l) {
                const int view = list[l];
                const float* P = cam + view * 16;
                const float dx = __fsub_rn(cx, P[3]), dy = __fsub_rn(cy, P[7]), dz = __fsub_rn(cz, P[11]);
                const float zc = __fadd_rn(__fadd_rn(__fmul_rn(P[2], dx), __fmul_rn(P[6], dy)), __fmul_rn(P[10], dz));
                if (!(zc > 0.0f)) continue;
                const float xc = __fadd_rn(__fadd_rn(__fmul_rn(P[0], dx), __fmul_rn(P[4], dy)), __fmul_rn(P[8], dz));
                const float yc = __fadd_rn(__fadd_rn(__fmul_rn(P[1], dx), __fmul_rn(P[5], dy)), __fmul_rn(P[9], dz));
                const float fx = P[12], fy = P[13], ccx = P[14], ccy = P[15];
                const float u = __fadd_rn(__fmul_rn(fx, __fdiv_rn(xc, zc)), ccx);
                const float v = __fadd_rn(__fmul_rn(fy, __fdiv_rn(yc, zc)), ccy);
                if (!(u >= 0.0f && u < fW && v >= 0.0f && v < fH)) continue;
                const int px = min((int)floorf(u), Wd - 1), py = min((int)floorf(v), H - 1);
                const float D = __ldg(depth + ((int64_t)(v0 + view) * H + py) * Wd + px);
                const float a = __fdiv_rn(__fsub_rn(__fadd_rn((float)px, 0.5f), ccx), fx);
                const float b = __fdiv_rn(__fsub_rn(__fadd_rn((float)py, 0.5f), ccy), fy);
                const float nrm = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)), 1.0f));
                const float proj = __fdiv_rn(__fadd_rn(__fadd_rn(__fmul_rn(a, xc), __fmul_rn(b, yc)), zc), nrm);
                float s = __fsub_rn(D, proj);
                if (s > trunc) s = trunc;
                if (s < -trunc) s = -trunc;
                if (!(s > -trunc)) continue;
                const float sn = __fdiv_rn(s, trunc), Wf = (float)Wv;
                Vv = __fdiv_rn(__fadd_rn(__fmul_rn(Wf, Vv), sn), __fadd_rn(Wf, 1.0f));
                if (Wv < 255) ++Wv;
            }
        }
        if (seen && voxel) {
            store_v(V, f16, q, Vv);
            W[q] = (uint8_t)Wv;
        }
    }
}

// K2: inside bit of voxel X = all voxels within Chebyshev radius r have V < 0.
//
// Only the signs matter, so the erosion runs on words of 32 voxels: a warp reads 32 voxels of a
// row and one ballot makes their word; an x erosion is an AND of the word's shifts (with the
// neighbour words' bits), the y and z erosions ANDs of whole words.  A block takes kMW words x
// kMY x kMZ rows (8 x 16, small grids 4 x 4) with a halo of r rows (and, at a tile's end inside the grid, one word); the volume is
// read once from memory, the halo (1.9 x at r = 2) from L2.  Bound: the instructions of those reads.
// 256^3 FP32, r = 2: 592 us as a running maximum of values over shared-memory tiles, 37 us so.  A NaN voxel
// counts as negative unless its whole neighbourhood is NaN (a maximum of the values ignores a NaN):
// a tile that has one goes through its neighbourhoods again.  Rows that are no multiple of 32 voxels
// long put their words into the bit array with two atomic ORs each.
constexpr int kMW = 8, kMaxR = 4;
constexpr int kMThreads = 256;
// Tiles of 4 x 4 rows where those of 8 x 16 would be fewer blocks than this (a block's rows are all there is to wait
// for then), and in grids of at most 4 rows at r = 0, where half of a tile's are out of the grid.  Measured (us, 8 x 16 / 4 x
// 4): 16^3, r = 2 19 / 8.4; 64^3, r = 0 10.3 / 7.1, r = 2 18.5 / 8.3; 96^3 (72 blocks), r = 4 28.7 / 24.6; 256 x 5 x 256 16.5 /
// 7.2; 128^3 (128 blocks), r = 2 18.5 / 18.5, r = 4 28.7 / 36.9; 160^3, r = 2 22.6 / 26.7; 4 x 4 x 100000, r = 0 154 / 109, r = 2
// 282 / 330.
constexpr int64_t kSmallMask = 128;

template <int kMY, int kMZ>
__global__ void __launch_bounds__(kMThreads) k_inside_mask(const void* __restrict__ V, int f16, int nx, int ny, int nz,
                                                           int r, uint32_t* __restrict__ bits, int aligned_rows) {
    constexpr int RY = kMY + 2 * kMaxR, RZ = kMZ + 2 * kMaxR;
    __shared__ uint32_t s_neg[RZ * RY][kMW + 2];   // not (V >= 0): word w - 1 of the tile's row; then its x erosion
    const int w0 = blockIdx.x * kMW, y0 = blockIdx.y * kMY, z0 = blockIdx.z * kMZ;
    const int words = (nx + 31) / 32;
    const int hy = kMY + 2 * r, hz = kMZ + 2 * r;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool left = w0 > 0, right = w0 + kMW < words;   // words beyond the tile inside the grid
    bool nan = false;
    int ly = warp % hy, lz = warp / hy;
    for (int row = warp; row < hy * hz; row += kMThreads / 32) {
        const int gy = y0 + ly - r, gz = z0 + lz - r;
        const bool in = gy >= 0 && gz >= 0 && gy < ny && gz < nz;
        const int64_t base = in ? ((int64_t)gz * ny + gy) * nx : 0;
        const int x0 = w0 * 32 + lane;
        float v[kMW], vl = -1.0f, vr = -1.0f;   // out of grid = unseen
#pragma unroll
        for (int w = 0; w < kMW; ++w) {
            v[w] = -1.0f;
            if (in && x0 + 32 * w < nx) v[w] = load_v(V, f16, base + x0 + 32 * w);
        }
        if (in && left && lane >= 32 - r) vl = load_v(V, f16, base + x0 - 32);
        if (in && right && lane < r && x0 + 32 * kMW < nx) vr = load_v(V, f16, base + x0 + 32 * kMW);
        nan = nan || vl != vl || vr != vr;
        uint32_t mine = 0xffffffffu;
#pragma unroll
        for (int w = 0; w < kMW; ++w) {
            nan = nan || v[w] != v[w];
            const unsigned neg = __ballot_sync(0xffffffffu, !(v[w] >= 0.0f));
            if (lane == w + 1) mine = neg;
        }
        const unsigned nl = __ballot_sync(0xffffffffu, !(vl >= 0.0f)), nr = __ballot_sync(0xffffffffu, !(vr >= 0.0f));
        if (lane == 0) mine = nl;
        if (lane == kMW + 1) mine = nr;
        if (lane < kMW + 2) s_neg[row][lane] = mine;
        ly += kMThreads / 32;
        while (ly >= hy) {
            ly -= hy;
            ++lz;
        }
    }
    const bool any_nan = __syncthreads_or(nan);
    // x erosion: each thread keeps its words in registers, then they replace the rows' words
    constexpr int kPer = (RZ * RY * kMW + kMThreads - 1) / kMThreads;
    uint32_t ew[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int e = threadIdx.x + i * kMThreads, row = e / kMW, w = e % kMW;
        ew[i] = 0;
        if (row >= hy * hz) continue;
        const uint32_t l = s_neg[row][w], c = s_neg[row][w + 1], h = s_neg[row][w + 2];
        uint32_t m = c;
        for (int d = 1; d <= r; ++d) m &= __funnelshift_l(l, c, d) & __funnelshift_r(c, h, d);
        ew[i] = m;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int e = threadIdx.x + i * kMThreads, row = e / kMW, w = e % kMW;
        if (row < hy * hz) s_neg[row][w] = ew[i];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kMW * kMY * kMZ; e += kMThreads) {
        const int w = e % kMW, ty = (e / kMW) % kMY, tz = e / (kMW * kMY);
        const int gw = w0 + w, gy = y0 + ty, gz = z0 + tz;
        if (gw >= words || gy >= ny || gz >= nz) continue;
        uint32_t m = 0xffffffffu;
        for (int dz = 0; dz <= 2 * r; ++dz)
            for (int dy = 0; dy <= 2 * r; ++dy) m &= s_neg[(tz + dz) * hy + ty + dy][w];
        const int rest = nx - gw * 32;   // voxels of this word inside the row
        if (rest < 32) m &= (1u << rest) - 1u;
        if (any_nan) {
            // drop voxels whose neighbourhood holds no V < 0 (it is all NaN then)
            for (uint32_t todo = m; todo; todo &= todo - 1) {
                const int b = __ffs(todo) - 1, gx = gw * 32 + b;
                bool lt = false;
                for (int z = gz - r; z <= gz + r && !lt; ++z)
                    for (int y = gy - r; y <= gy + r && !lt; ++y)
                        for (int x = gx - r; x <= gx + r && !lt; ++x)
                            lt = x < 0 || y < 0 || z < 0 || x >= nx || y >= ny || z >= nz ||
                                 load_v(V, f16, ((int64_t)z * ny + y) * nx + x) < 0.0f;
                if (!lt) m &= ~(1u << b);
            }
        }
        const int64_t idx = ((int64_t)gz * ny + gy) * nx + (int64_t)gw * 32;
        if (aligned_rows) {
            bits[idx >> 5] = m;
        } else if (m) {
            const int sh = (int)(idx & 31);
            atomicOr(bits + (idx >> 5), m << sh);
            if (sh && (m >> (32 - sh))) atomicOr(bits + (idx >> 5) + 1, m >> (32 - sh));
        }
    }
}

// ---- Alg. 2 as printed, one view at a time: march every pixel's ray ---------------
// Thread per pixel of view `view`: unit ray through the pixel centre, clipped to the grid
// box from t = 0; voxel walk of Alg. 1; at each voxel s = clamp(v . (p* - c), -D_T, D_T),
// p* = o + D v (D = +inf: s = D_T); stop at the first s <= -D_T, else the voxel gets one count and
// s / D_T in fixed point (2^-32 units: integer sums, so the result does not depend on the order in
// which the rays arrive).  k_raycast_apply folds the view's sums in.
//
// The bound is the atomics: 40 M visits of a 640 x 480 view, 922 us with a 64-bit sum and a count
// for each.  Nearly all of them are in free space, where s / D_T is exactly 1: so the sum is kept
// as what is missing to the count, 2^32 - s / D_T 2^32, which is 0 there and needs no atomic.  And
// rays of neighbouring pixels cross the same voxels in step: a warp takes 8 x 4 pixels, and
// lanes in one voxel at the same step add their counts with one atomic.  144 us a view so; what is
// left is the walk.
constexpr double kFix = 4294967296.0;   // 2^32
constexpr int64_t kFewCounts = 1 << 19;   // k_raycast_apply_few
constexpr int kRayW = 8, kRayH = 4;     // pixels of a warp

// Whether rays of neighbouring pixels share voxels where they enter the grid: kMergePixels of them and more to a
// voxel's side.  A match in every step lengthens the chain of steps, and pays only where lanes meet.  Measured (us,
// merged / not, a sphere seen from outside): 64^3 from 160 x 160 pixels (1.7 to a voxel) 55 / 40, from 640 x 640 (6.7) 70 /
// 74; 128^3 from 160 x 160 147 / 117; the room, from inside, 64^3 from 320 x 240 41 / 198.  The test costs large images 2.5 %
// (its branch stands in the loop), so those merge always.
constexpr float kMergePixels = 4.0f;
__device__ __forceinline__ bool rays_meet(const GridDev& g, const float* __restrict__ Kc, const float* __restrict__ c2w,
                                          int view) {
    float away = 0.0f;   // the camera's distance from the grid, squared
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float o = __ldg(c2w + 12 * view + 4 * k + 3), hi = g.org[k] + (float)g.n[k] * g.vs;
        const float d = fmaxf(fmaxf(g.org[k] - o, o - hi), 0.0f);
        away += d * d;
    }
    return sqrtf(away) * kMergePixels < g.vs * fabsf(__ldg(Kc + 4 * view));
}

// FEW: an image of few tiles, whose time is its rays' chains of steps
template <bool SMALL, bool FEW>
__global__ void __launch_bounds__(kFuseBlock) k_raycast_view(GridDev g, const float* __restrict__ depth, int H, int Wd,
                                                             const float* __restrict__ Kc, const float* __restrict__ c2w,
                                                             int view, unsigned long long* __restrict__ lack,
                                                             uint32_t* __restrict__ cnt) {
    const bool merge = SMALL && (!FEW || __any_sync(0xffffffffu, rays_meet(g, Kc, c2w, view)));
    const float kInf = __int_as_float(0x7f800000);
    const float* P = c2w + 12 * view;
    const float fx = __ldg(Kc + 4 * view), fy = __ldg(Kc + 4 * view + 1);
    const float cx = __ldg(Kc + 4 * view + 2), cy = __ldg(Kc + 4 * view + 3);
    const float o[3] = {__ldg(P + 3), __ldg(P + 7), __ldg(P + 11)};
    const int max_steps = g.n[0] + g.n[1] + g.n[2] + 8;
    const int lane = threadIdx.x & 31;
    const int tx = (Wd + kRayW - 1) / kRayW, ty = (H + kRayH - 1) / kRayH;
    const int64_t tiles = (int64_t)tx * ty, warps = (int64_t)gridDim.x * (blockDim.x / 32);
    for (int64_t q = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5); q < tiles; q += warps) {
        const int px = (int)(q % tx) * kRayW + lane % kRayW, py = (int)(q / tx) * kRayH + lane / kRayW;
        bool act = px < Wd && py < H;
        const float a = __fdiv_rn(__fsub_rn(__fadd_rn((float)px, 0.5f), cx), fx);
        const float b = __fdiv_rn(__fsub_rn(__fadd_rn((float)py, 0.5f), cy), fy);
        float d[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            d[k] = __fadd_rn(__fadd_rn(__fmul_rn(__ldg(P + 4 * k), a), __fmul_rn(__ldg(P + 4 * k + 1), b)),
                             __ldg(P + 4 * k + 2));
        const float nn = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(d[0], d[0]), __fmul_rn(d[1], d[1])), __fmul_rn(d[2], d[2])));
#pragma unroll
        for (int k = 0; k < 3; ++k) d[k] = __fdiv_rn(d[k], nn);
        const float D = act ? __ldg(depth + ((int64_t)view * H + py) * Wd + px) : 0.0f;
        float t0 = 0.0f, t_end = 0.0f;
        act = act && clip_box(g, o, d, 0.0f, kInf, t0, t_end);
        float ps[3];   // p* = o + D v
#pragma unroll
        for (int k = 0; k < 3; ++k) ps[k] = __fadd_rn(o[k], __fmul_rn(D, d[k]));
        const bool free_ray = isinf(D);
        // before this parameter s = v . (p* - c) is above D_T whatever the voxel: its centre is within
        // 1.74 voxels of the ray's point at t along v, and 1e-5 of the lengths cover the rounding
        const float t_free = D - g.trunc - 2.0f * g.vs - 1e-5f * (fabsf(D) + fabsf(o[0]) + fabsf(o[1]) + fabsf(o[2]) + g.trunc);
        Walk<SMALL> s;
        s.start(g, o, d, t0);
        for (int st = 0; st < max_steps; ++st) {
            act = act && s.t < t_end;
            float sx = g.trunc;
            if (act && !free_ray && !(s.t < t_free)) {
                float e[3];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    e[k] = __fsub_rn(ps[k], __fadd_rn(g.org[k], __fmul_rn(s.centre(k), g.vs)));
                const float dot = __fadd_rn(__fadd_rn(__fmul_rn(d[0], e[0]), __fmul_rn(d[1], e[1])), __fmul_rn(d[2], e[2]));
                sx = dot > g.trunc ? g.trunc : (dot < -g.trunc ? -g.trunc : dot);
            }
            act = act && sx > -g.trunc;
            const unsigned live = __ballot_sync(0xffffffffu, act);
            if (live == 0) break;
            if (act) {
                const int64_t idx = s.idx;
                const unsigned same = merge ? __match_any_sync(live, (unsigned)idx) : 1u << lane;
                if (lane == __ffs(same) - 1) atomicAdd(cnt + idx, (unsigned)__popc(same));
                if (sx != g.trunc) {
                    const long long qv = __double2ll_rn((double)__fdiv_rn(sx, g.trunc) * kFix);
                    atomicAdd(lack + idx, (unsigned long long)((1ll << 32) - qv));
                }
                act = s.next(g);
            }
        }
    }
}

// the view's k visits of a voxel: V <- (W V + sum) / (W + k) in FP64, rounded once to the
// storage type; W <- min(W + k, 255); the accumulators are cleared for the next view.  Most voxels
// have no count, and reading the counts is the bound.
__device__ __forceinline__ void raycast_apply(void* V, int f16, uint8_t* W, unsigned long long* lack, uint32_t* cnt,
                                              int64_t q, uint32_t k) {
    const long long sum = ((long long)k << 32) - (long long)lack[q];
    const float v = load_v(V, f16, q);
    const uint32_t w = W[q];
    const double vn = ((double)w * (double)v + (double)sum / kFix) / (double)(w + k);
    store_v(V, f16, q, (float)vn);
    W[q] = (uint8_t)(w + k > 255u ? 255u : w + k);
    lack[q] = 0ull;
    cnt[q] = 0u;
}

// few voxels: one to a thread (eight counts to a lane are eight FP64 divisions in series: the fusion of a 64 x 64 view
// into 32^3 46 us, 36 so, and 31 without merging as well)
__global__ void k_raycast_apply_few(void* V, int f16, uint8_t* W, unsigned long long* __restrict__ lack,
                                    uint32_t* __restrict__ cnt, int64_t n) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const uint32_t k = q < n ? cnt[q] : 0u;
    if (k) raycast_apply(V, f16, W, lack, cnt, q, k);
}

__global__ void k_raycast_apply(void* V, int f16, uint8_t* W, unsigned long long* __restrict__ lack,
                                uint32_t* __restrict__ cnt, int64_t n) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
    // a warp looks at 256 counts (16-byte aligned); where any is set it takes them 32 by 32
    for (int64_t i = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5); i * 256 < n; i += warps) {
        const int64_t q0 = i * 256;
        bool any = true;
        if (q0 + 256 <= n) {
            const uint4 a = reinterpret_cast<const uint4*>(cnt + q0)[lane], b = reinterpret_cast<const uint4*>(cnt + q0)[32 + lane];
            any = (a.x | a.y | a.z | a.w | b.x | b.y | b.z | b.w) != 0;
        }
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll 4
        for (int j = 0; j < 8; ++j) {
            const int64_t q = q0 + 32 * j + lane;
            if (q >= n) break;
            const uint32_t k = cnt[q];
            if (k) raycast_apply(V, f16, W, lack, cnt, q, k);
        }
    }
}

}  // namespace

int grid_check(const tsdfs_grid* g) {
    if (!g) return fail(TSDFS_E_INVALID, "grid is NULL");
    if (g->nx <= 0 || g->ny <= 0 || g->nz <= 0) return fail(TSDFS_E_INVALID, "grid dimensions must be positive");
    if ((int64_t)g->nx * g->ny * g->nz > ((int64_t)1 << 40)) return fail(TSDFS_E_INVALID, "grid too large");
    if (!(g->voxel_size > 0.0f) || !(g->trunc > 0.0f)) return fail(TSDFS_E_INVALID, "voxel_size and trunc must be > 0");
    if (g->dtype != TSDFS_F32 && g->dtype != TSDFS_F16) return fail(TSDFS_E_INVALID, "grid dtype must be TSDFS_F32 or TSDFS_F16");
    if (!g->tsdf) return fail(TSDFS_E_INVALID, "grid tsdf pointer is NULL");
    return TSDFS_OK;
}

}  // namespace tsdfs

using namespace tsdfs;

extern "C" int tsdfs_grid_init(const tsdfs_grid* g, tsdfs_stream_t stream) {
    int rc = grid_check(g);
    if (rc) return rc;
    if (!g->weight) return fail(TSDFS_E_INVALID, "grid weight pointer is NULL");
    int64_t n = (int64_t)g->nx * g->ny * g->nz;
    k_grid_init<<<grid_1d(n, 256), 256, 0, (cudaStream_t)stream>>>(g->tsdf, g->dtype == TSDFS_F16, g->weight, n);
    return cuda_check(cudaGetLastError(), "tsdfs_grid_init launch");
}

extern "C" int tsdf_integrate(const tsdfs_grid* g, const float* depth, int32_t n_views, int32_t H, int32_t W,
                              const float* K, const float* c2w, tsdfs_stream_t stream) {
    int rc = grid_check(g);
    if (rc) return rc;
    if (!g->weight) return fail(TSDFS_E_INVALID, "grid weight pointer is NULL");
    if (n_views < 0 || H <= 0 || W <= 0) return fail(TSDFS_E_INVALID, "n_views must be >= 0 and H, W > 0");
    if (n_views == 0) return TSDFS_OK;
    if (n_views > 2048) return fail(TSDFS_E_INVALID, "at most 2048 views per call (split larger sets)");
    if (!depth || !K || !c2w) return fail(TSDFS_E_INVALID, "depth, K and c2w must be non-NULL");
    ProfScope ps("integrate", (cudaStream_t)stream);
    const int n[3] = {g->nx, g->ny, g->nz};
    const bool thin = n[0] < kBX || n[1] < kBY || n[2] < kBZ;
    if (thin || n_views > kManyViews || (int64_t)n[0] * n[1] * n[2] <= kFewVoxels) {
        // 8 x 8 x 4 voxels; an axis with fewer gives its share to those with the most bricks
        int lg[3] = {3, 3, 2}, spare = 0;
        for (int a = 0; a < 3; ++a)
            for (; lg[a] > 0 && (1 << (lg[a] - 1)) >= n[a]; --lg[a]) ++spare;
        for (; spare > 0; --spare) {
            int most = 0;
            for (int a = 1; a < 3; ++a)
                if (n[a] >> lg[a] > n[most] >> lg[most]) most = a;
            ++lg[most];
        }
        int64_t bricks = 1;
        for (int a = 0; a < 3; ++a) bricks *= ((n[a] - 1) >> lg[a]) + 1;
        k_integrate_few<<<grid_1d(bricks, 1, kFuseBlocks), kFuseBlock, 0, (cudaStream_t)stream>>>(
            g->nx, g->ny, g->nz, lg[0], lg[1], g->origin[0], g->origin[1], g->origin[2], g->voxel_size, g->trunc, g->tsdf,
            g->dtype == TSDFS_F16, g->weight, depth, n_views, H, W, K, c2w);
        return cuda_check(cudaGetLastError(), "tsdf_integrate launch");
    }
    const int64_t bricks = (int64_t)((g->nx + kBX - 1) / kBX) * ((g->ny + kBY - 1) / kBY) * ((g->nz + kBZ - 1) / kBZ);
    size_t smem = (size_t)n_views * (kCam * sizeof(float) + sizeof(uint16_t));
    if (smem > 48 * 1024) {
        rc = cuda_check(cudaFuncSetAttribute(k_integrate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                        "tsdf_integrate smem attribute");
        if (rc) return rc;
    }
    k_integrate<<<grid_1d(bricks, 1, kFuseBlocks), kFuseBlock, smem, (cudaStream_t)stream>>>(
        g->nx, g->ny, g->nz, g->origin[0], g->origin[1], g->origin[2], g->voxel_size, g->trunc, g->tsdf,
        g->dtype == TSDFS_F16, g->weight, depth, n_views, H, W, K, c2w);
    return cuda_check(cudaGetLastError(), "tsdf_integrate launch");
}

extern "C" size_t tsdfs_raycast_workspace_size(const tsdfs_grid* g) {
    if (!g || g->nx <= 0 || g->ny <= 0 || g->nz <= 0) return 0;
    const int64_t n = (int64_t)g->nx * g->ny * g->nz;
    return (size_t)n * (sizeof(unsigned long long) + sizeof(uint32_t)) + 512;
}

extern "C" int tsdf_integrate_raycast(const tsdfs_grid* g, const float* depth, int32_t n_views, int32_t H, int32_t W,
                                      const float* K, const float* c2w, void* ws, size_t ws_bytes,
                                      tsdfs_stream_t stream) {
    int rc = grid_check(g);
    if (rc) return rc;
    if (!g->weight) return fail(TSDFS_E_INVALID, "grid weight pointer is NULL");
    if (n_views < 0 || H <= 0 || W <= 0) return fail(TSDFS_E_INVALID, "n_views must be >= 0 and H, W > 0");
    if (n_views == 0) return TSDFS_OK;
    if (!depth || !K || !c2w) return fail(TSDFS_E_INVALID, "depth, K and c2w must be non-NULL");
    if ((int64_t)H * W > (int64_t)1 << 21)
        return fail(TSDFS_E_INVALID, "at most 2^21 pixels per view (the fixed-point sums hold 2^21 visits)");
    if (!ws || ws_bytes < tsdfs_raycast_workspace_size(g)) return fail(TSDFS_E_WORKSPACE, "raycast workspace too small");
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = (int64_t)g->nx * g->ny * g->nz;
    uintptr_t p = (reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255);
    unsigned long long* lack = reinterpret_cast<unsigned long long*>(p);
    // 16-byte aligned for the apply kernel's vector loads
    uint32_t* cnt = reinterpret_cast<uint32_t*>((p + (size_t)n * sizeof(unsigned long long) + 15) & ~uintptr_t(15));
    ProfScope ps("integrate_raycast", st);
    rc = cuda_check(cudaMemsetAsync(lack, 0, (size_t)((uint8_t*)(cnt + n) - (uint8_t*)lack), st),
                    "raycast workspace clear");
    if (rc) return rc;
    GridDev gd{g->tsdf, g->dtype == TSDFS_F16, {g->nx, g->ny, g->nz}, {g->origin[0], g->origin[1], g->origin[2]},
               g->voxel_size, g->trunc};
    const int f16 = g->dtype == TSDFS_F16;
    const int64_t tiles = (int64_t)((W + kRayW - 1) / kRayW) * ((H + kRayH - 1) / kRayH);
    // few warps: one to a block, so that each has an SM's issue slots for its chain of steps
    const bool few = tiles < 152 * 16, small = small_grid(gd.n);
    const int block = few ? 32 : kFuseBlock;
    for (int v = 0; v < n_views; ++v) {
        auto view = !small ? k_raycast_view<false, false> : (few ? k_raycast_view<true, true> : k_raycast_view<true, false>);
        view<<<grid_1d(tiles * 32, block, 152 * 16), block, 0, st>>>(gd, depth, H, W, K, c2w, v, lack, cnt);
        if (n <= kFewCounts)
            k_raycast_apply_few<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(g->tsdf, f16, g->weight, lack, cnt, n);
        else
            k_raycast_apply<<<grid_1d((n + 7) / 8, 256, 152 * 8), 256, 0, st>>>(g->tsdf, f16, g->weight, lack, cnt, n);
    }
    return cuda_check(cudaGetLastError(), "tsdf_integrate_raycast launch");
}

extern "C" int64_t tsdfs_inside_mask_words(const tsdfs_grid* g) {
    if (!g || g->nx <= 0 || g->ny <= 0 || g->nz <= 0) return 0;
    return ((int64_t)g->nx * g->ny * g->nz + 31) / 32;
}

extern "C" int tsdfs_inside_mask(const tsdfs_grid* g, int32_t r, uint32_t* bits, tsdfs_stream_t stream) {
    int rc = grid_check(g);
    if (rc) return rc;
    if (r < 0 || r > kMaxR) return fail(TSDFS_E_INVALID, "nb_radius must be in [0, %d]", kMaxR);
    if (!bits) return fail(TSDFS_E_INVALID, "mask_bits is NULL");
    if (g->ny > 4 * 65535 || g->nz > 4 * 65535) return fail(TSDFS_E_INVALID, "grid too large for the mask kernel");
    int aligned = (g->nx % 32) == 0;
    if (!aligned) {
        rc = cuda_check(cudaMemsetAsync(bits, 0, (size_t)tsdfs_inside_mask_words(g) * 4, (cudaStream_t)stream),
                        "tsdfs_inside_mask memset");
        if (rc) return rc;
    }
    const int64_t nx = g->nx, ny = g->ny, nz = g->nz;
    const int64_t blocks = ((nx - 1) / (32 * kMW) + 1) * ((ny - 1) / 8 + 1) * ((nz - 1) / 16 + 1);
    const bool small = blocks < kSmallMask || (ny <= 4 && r == 0);
    const int my = small ? 4 : 8, mz = small ? 4 : 16;
    dim3 grid((unsigned)((nx - 1) / (32 * kMW) + 1), (unsigned)((ny - 1) / my + 1), (unsigned)((nz - 1) / mz + 1));
    ProfScope ps("inside_mask", (cudaStream_t)stream);
    auto inside = small ? k_inside_mask<4, 4> : k_inside_mask<8, 16>;
    inside<<<grid, kMThreads, 0, (cudaStream_t)stream>>>(g->tsdf, g->dtype == TSDFS_F16, g->nx, g->ny, g->nz, r, bits,
                                                         aligned);
    return cuda_check(cudaGetLastError(), "tsdfs_inside_mask launch");
}
