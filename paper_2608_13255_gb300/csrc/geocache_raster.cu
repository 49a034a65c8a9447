// Position-map rasteriser: the per-pixel world positions and validity masks
// that a geometry-conditioned texturing pipeline renders for each view
// (Sec. 3.1), from which the correspondence operator of Sec. 3.2 is built.
//
// A z-buffer over pixel centres, in two kernels:
//  raster_faces_kernel: one thread per face (fewer per warp in small renders of
//    large faces), looping over the CTA's views (the
//    face's vertices are loaded once; a CTA's faces normally belong to one
//    asset, whose cameras are staged in shared memory).  For each view the
//    face is projected; every pixel centre inside or on it (three
//    sign-normalised edge functions) gets the camera z of the ray /
//    face-plane intersection, and
//    the key (depth bits << 32 | face index) is min-combined into the
//    pixel's z-buffer word with a 64-bit atomicMin (nearest face wins, ties
//    to the lower face index; positive floats order like their bits).  The
//    pixel boxes of a warp's 32 faces are concatenated and the 32 lanes
//    stride over the concatenation, so that the work is balanced whatever
//    the mix of small and large faces; the pixels found covered are queued
//    and their depths formed 32 at a time.
//    Bound by instruction issue (75% of the slots busy; XU and DRAM far
//    below).  A blob of 81,920 noisy faces has 5.7 box pixels per face and
//    view at 128 x 128, 0.7 of them covered, so the test of a box pixel is
//    what was made short: its face comes from a population count over the
//    ballot of box starts (not a binary search), its row from a float
//    reciprocal (not an integer division), its edge functions from the
//    differences stored with the face, without a branch; and the three IEEE
//    divisions of a depth run with full warps (with one lane in eight when
//    each warp formed the depths as it met them).  16 meshes x 6 views at
//    128 x 128: 454 -> 241 us; 4 smooth ones at 512 x 512: 134 -> 83 us.
//    4 resident CTAs per SM (64 registers); 3, 5 and 6: 6%, 9% and 20%
//    slower.
//  raster_resolve_kernel: one thread per pixel; the key's depth gives the
//    world position of the intersection.
// Super-sampled maps (the pipeline's image-resolution render brought to the
// latent token grid): the faces are rasterised at s times the token
// resolution with the cameras' focal lengths and principal point scaled by
// s, and raster_pool_kernel resolves each token's s x s pixels and pools
// them (mean of the valid pixels' positions, foreground when at least half
// are valid).  pool_posmaps_kernel pools maps the caller rendered itself.
// Every decision and the position are binary32 with one rounding per
// operation in a fixed order (explicit __f*_rn intrinsics), so the maps are
// reproducible bit for bit.
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "geocache.h"
#include "geocache_device.cuh"
#include "geocache_internal.h"

namespace geocache {

namespace {

// Status word of this translation unit (the library is linked without
// relocatable device code): bit 3 = a face index outside [0, nv).  Read and
// cleared together with the transport's word by geocache_device_status.
__device__ unsigned int g_raster_error = 0;

constexpr int kRasterThreads = 256;
constexpr int kRasterBlocks = 4;  // resident CTAs per SM of the face kernel

// How a render is split over CTAs: `views` consecutive views per CTA (each CTA
// loads its faces again) and `faces` faces per warp (32 or fewer; all 32 lanes
// still share the warp's pixels).
struct RasterSplit {
    int views, faces;
};
constexpr unsigned long long kEmpty = ~0ull;  // z-buffer word of an uncovered pixel

struct Cam32 {
    float R[9], t[3], fx, fy, cx, cy;
};

// c points to global or shared memory (generic loads); the intrinsics are
// multiplied by `scale` (binary32), the camera of an s-times finer pixel grid
__device__ __forceinline__ Cam32 load_cam(const geocache_camera* c, float scale = 1.0f) {
    Cam32 k;
    const float* p = reinterpret_cast<const float*>(c);
#pragma unroll
    for (int i = 0; i < 9; ++i) k.R[i] = p[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) k.t[i] = p[9 + i];
    k.fx = __fmul_rn(p[12], scale);
    k.fy = __fmul_rn(p[13], scale);
    k.cx = __fmul_rn(p[14], scale);
    k.cy = __fmul_rn(p[15], scale);
    return k;
}

// x_c = R X + t, each row summed ((R0 X0 + R1 X1) + R2 X2) + t
__device__ __forceinline__ void cam_point(const Cam32& c, const float (&X)[3], float* xc) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        float s = __fmul_rn(c.R[3 * r], X[0]);
        s = __fadd_rn(s, __fmul_rn(c.R[3 * r + 1], X[1]));
        s = __fadd_rn(s, __fmul_rn(c.R[3 * r + 2], X[2]));
        xc[r] = __fadd_rn(s, c.t[r]);
    }
}

// One projected face: screen vertices, signed area, camera-space plane
// n . x = nd, and the clamped pixel box (whole numbers).
struct Face {
    float u[3], v[3], area, n[3], nd;
    float ilo, ihi, jlo, jhi;
};

// false when the face covers no pixel centre: a vertex not in front
// (z <= 1e-6), zero area, or a box outside the image
__device__ __forceinline__ bool setup_face(const Cam32& c, const float (&X)[3][3], int H, int W, Face& o) {
    float P[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        cam_point(c, X[k], P[k]);
        o.u[k] = __fadd_rn(__fmul_rn(c.fx, __fdiv_rn(P[k][0], P[k][2])), c.cx);
        o.v[k] = __fadd_rn(__fmul_rn(c.fy, __fdiv_rn(P[k][1], P[k][2])), c.cy);
    }
    o.area = __fsub_rn(__fmul_rn(__fsub_rn(o.u[1], o.u[0]), __fsub_rn(o.v[2], o.v[0])),
                       __fmul_rn(__fsub_rn(o.v[1], o.v[0]), __fsub_rn(o.u[2], o.u[0])));
    const float umin = fminf(o.u[0], fminf(o.u[1], o.u[2])), umax = fmaxf(o.u[0], fmaxf(o.u[1], o.u[2]));
    const float vmin = fminf(o.v[0], fminf(o.v[1], o.v[2])), vmax = fmaxf(o.v[0], fmaxf(o.v[1], o.v[2]));
    o.ilo = fmaxf(ceilf(__fsub_rn(umin, 0.5f)), 0.0f);
    o.ihi = fminf(floorf(__fsub_rn(umax, 0.5f)), (float)(W - 1));
    o.jlo = fmaxf(ceilf(__fsub_rn(vmin, 0.5f)), 0.0f);
    o.jhi = fminf(floorf(__fsub_rn(vmax, 0.5f)), (float)(H - 1));
    float e1[3], e2[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        e1[r] = __fsub_rn(P[1][r], P[0][r]);
        e2[r] = __fsub_rn(P[2][r], P[0][r]);
    }
    o.n[0] = __fsub_rn(__fmul_rn(e1[1], e2[2]), __fmul_rn(e1[2], e2[1]));
    o.n[1] = __fsub_rn(__fmul_rn(e1[2], e2[0]), __fmul_rn(e1[0], e2[2]));
    o.n[2] = __fsub_rn(__fmul_rn(e1[0], e2[1]), __fmul_rn(e1[1], e2[0]));
    float nd = __fmul_rn(o.n[0], P[0][0]);
    nd = __fadd_rn(nd, __fmul_rn(o.n[1], P[0][1]));
    o.nd = __fadd_rn(nd, __fmul_rn(o.n[2], P[0][2]));
    // one test without branches: most of a warp's faces cover a pixel in most views
    return (P[0][2] > 1e-6f) & (P[1][2] > 1e-6f) & (P[2][2] > 1e-6f) & ((o.area > 0.0f) | (o.area < 0.0f)) &
           (o.ilo <= o.ihi) & (o.jlo <= o.jhi);
}

// camera-space ray direction through the pixel centre (pu, pv)
__device__ __forceinline__ void ray(const Cam32& c, float pu, float pv, float& d0, float& d1) {
    d0 = __fdiv_rn(__fsub_rn(pu, c.cx), c.fx);
    d1 = __fdiv_rn(__fsub_rn(pv, c.cy), c.fy);
}

// Faces of a warp published for its pixel loop: 20 words each, so that eight
// different faces read by 16-byte loads fall into different banks.
//   [0..2]  edge k = 0, 1, 2 from vertex a to vertex b ((1,2), (2,0), (0,1)):
//           (u_b - u_a, v_b - v_a), both negated when the area is negative
//           (which negates the edge function exactly), and (u_a, v_a)
//   [3]     first pixel of the face in the warp's concatenated boxes,
//           1 / box width (to an ulp), centre of the box's first pixel
//   [4]     n, nd
// and beside them (SlotInfo) the box width and the face's lane.
constexpr int kSlotQuads = 5;
struct SlotInfo {
    float width;
    int lane;
};

__device__ __forceinline__ void publish_face(float4* q, SlotInfo* info, const Face& o, int start, int lane) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int a = (k + 1) % 3, b = (k + 2) % 3;
        const float du = __fsub_rn(o.u[b], o.u[a]), dv = __fsub_rn(o.v[b], o.v[a]);
        q[k] = make_float4(o.area < 0.0f ? -du : du, o.area < 0.0f ? -dv : dv, o.u[a], o.v[a]);
    }
    const float width = o.ihi - o.ilo + 1.0f;
    q[3] = make_float4(__int_as_float(start), __fdividef(1.0f, width), o.ilo + 0.5f, o.jlo + 0.5f);
    q[4] = make_float4(o.n[0], o.n[1], o.n[2], o.nd);
    *info = SlotInfo{width, lane};
}

// whether the centre (pu, pv) lies inside or on the published face: its three
// edge functions (u_b - u_a)(pv - v_a) - (v_b - v_a)(pu - u_a) have the sign
// of the area or are zero
__device__ __forceinline__ bool covers(const float4* q, float pu, float pv) {
    const float4 e[3] = {q[0], q[1], q[2]};
    float w[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        w[k] = __fsub_rn(__fmul_rn(e[k].x, __fsub_rn(pv, e[k].w)), __fmul_rn(e[k].y, __fsub_rn(pu, e[k].z)));
    return (w[0] >= 0.0f) & (w[1] >= 0.0f) & (w[2] >= 0.0f);
}

// depth key of the covered pixel with centre (pu, pv), or kEmpty when the ray
// meets the face's plane (n, nd) at no positive finite depth
__device__ __forceinline__ unsigned long long depth_key(const Cam32& c, const float4& n, float pu, float pv,
                                                        unsigned int face) {
    float d0, d1;
    ray(c, pu, pv, d0, d1);
    float den = __fmul_rn(n.x, d0);
    den = __fadd_rn(den, __fmul_rn(n.y, d1));
    den = __fadd_rn(den, n.z);
    if (den == 0.0f) return kEmpty;
    const float s = __fdiv_rn(n.w, den);
    if (!(s > 0.0f && s <= 3.0e38f)) return kEmpty;
    return ((unsigned long long)__float_as_uint(s) << 32) | face;
}

// asset of face f: face_off[b] <= f < face_off[b + 1] (clamped to [0, B))
__device__ __forceinline__ int asset_of(const int64_t* __restrict__ face_off, int B, long long f) {
    int lo = 0, hi = B - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(face_off + mid) <= f) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Boxes of more pixels than this are rasterised one at a time by the whole
// warp, row by row; smaller ones are concatenated, so that the 32 boxes of a
// warp hold fewer than 2^22 pixels (the float quotient below is then exact).
constexpr int kLargeBox = 1 << 16;

// A warp's share of the CTA's shared memory.
struct WarpFaces {
    float4 slot[32 * kSlotQuads];
    SlotInfo info[32];
    float2 centre[64];  // queue of covered pixels
    uint8_t of[64];
};

// integer in [0, 2^23) to float and back by the float whose low bits it is
constexpr float kTwo23 = 8388608.0f;
__device__ __forceinline__ float small_float(int x) { return __int_as_float(x | 0x4b000000) - kTwo23; }

// The faces of one warp (lane l: face f_warp + l with vertices X, of asset b)
// in every view.  ONE: the CTA's faces belong to one asset, whose cameras
// are at s_cam with their intrinsics scaled.
template <bool ONE>
__device__ __forceinline__ void raster_warp(const float (&X)[3][3], bool ok, int b, unsigned int f_warp,
                                            const geocache_camera* s_cam, const geocache_camera* __restrict__ cams,
                                            const int* b_w, WarpFaces& sh, int N, int view0, int view1, int H, int W,
                                            float scale, unsigned long long* __restrict__ zbuf) {
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    for (int view = view0; view < view1; ++view) {
        // depth and z-buffer update of the pixel with centre (pu, pv), covered by the face of a slot
        auto resolve = [&](int slot, float pu, float pv) {
            const int src = sh.info[slot].lane;
            const int qb = ONE ? b : b_w[src];
            const Cam32 qc = ONE ? load_cam(s_cam + view) : load_cam(cams + (size_t)qb * N + view, scale);
            const unsigned long long key = depth_key(qc, sh.slot[slot * kSlotQuads + 4], pu, pv, f_warp + src);
            if (key != kEmpty)
                atomicMin(zbuf + ((size_t)qb * N + view) * (size_t)H * W + (size_t)(int)pv * W + (int)pu, key);
        };
        Face o;
        const bool live =
            ok && setup_face(ONE ? load_cam(s_cam + view) : load_cam(cams + (size_t)b * N + view, scale), X, H, W, o);
        const float pixels = live ? (o.ihi - o.ilo + 1.0f) * (o.jhi - o.jlo + 1.0f) : 0.0f;
        const int box = pixels > (float)kLargeBox ? 0 : (int)pixels;  // exact up to 2^24
        // first pixel of each face in the concatenation
        int incl = box;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31), start = box ? incl - box : INT_MAX;
        // the faces with a box take the slots in lane order, so the slot of
        // concatenated pixel k is the number of starts at or before k, less one
        const uint32_t boxed = __ballot_sync(0xffffffffu, box > 0);
        if (box > 0) {
            const int slot = __popc(boxed & below);
            publish_face(sh.slot + slot * kSlotQuads, sh.info + slot, o, start, lane);
        }
        __syncwarp();
        int n_started = -1, n_queued = 0;
        for (int k0 = 0; k0 < total; k0 += 32) {
            const uint32_t rel = (uint32_t)(start - k0);
            const uint32_t starts = __reduce_or_sync(0xffffffffu, rel < 32u ? 1u << rel : 0u);
            const int k = min(k0 + lane, total - 1);  // lanes past the end repeat the last pixel, uncounted
            const int slot = n_started + __popc(starts & (2u * below + 1u));
            n_started += __popc(starts);
            const float4* q = sh.slot + slot * kSlotQuads;
            const float4 h = q[3];
            const float local = small_float(k - __float_as_int(h.x));
            // row of the box: local / width by the reciprocal, exact since the box has at most 2^16
            // pixels (the quotient is at least 0.5 / width from an integer, its error below 2^-4 /
            // width); rounding the sum with 2^23 down leaves its integer part
            const float row = __fadd_rd((local + 0.5f) * h.y, kTwo23) - kTwo23;
            const float pu = h.z + __fmaf_rn(-row, sh.info[slot].width, local), pv = h.w + row;
            const bool in = covers(q, pu, pv) & (k0 + lane < total);
            const uint32_t hits = __ballot_sync(0xffffffffu, in);
            if (in) {
                const int at = n_queued + __popc(hits & below);
                sh.centre[at] = make_float2(pu, pv);
                sh.of[at] = (uint8_t)slot;
            }
            n_queued += __popc(hits);
            if (n_queued >= 32) {
                __syncwarp();
                const float2 c = sh.centre[lane];
                resolve(sh.of[lane], c.x, c.y);
                n_queued -= 32;
                const float2 rest = sh.centre[32 + lane];
                const uint8_t rest_of = sh.of[32 + lane];
                __syncwarp();
                if (lane < n_queued) {
                    sh.centre[lane] = rest;
                    sh.of[lane] = rest_of;
                }
            }
        }
        __syncwarp();
        if (lane < n_queued) {
            const float2 c = sh.centre[lane];
            resolve(sh.of[lane], c.x, c.y);
        }
        __syncwarp();  // the slots are rewritten for the next view
        for (uint32_t big = __ballot_sync(0xffffffffu, pixels > (float)kLargeBox); big; big &= big - 1) {
            const int src = __ffs(big) - 1;
            if (lane == src) publish_face(sh.slot, sh.info, o, 0, lane);
            const float ilo = __shfl_sync(0xffffffffu, o.ilo, src), ihi = __shfl_sync(0xffffffffu, o.ihi, src);
            const float jlo = __shfl_sync(0xffffffffu, o.jlo, src), jhi = __shfl_sync(0xffffffffu, o.jhi, src);
            __syncwarp();
            for (float j = jlo; j <= jhi; j += 1.0f)
                for (float i = ilo + (float)lane; i <= ihi; i += 32.0f)
                    if (covers(sh.slot, i + 0.5f, j + 0.5f)) resolve(0, i + 0.5f, j + 0.5f);
            __syncwarp();
        }
    }
}

__global__ void __launch_bounds__(kRasterThreads, kRasterBlocks) raster_faces_kernel(
    const float* __restrict__ V, long long nv, const int32_t* __restrict__ F, long long nf,
    const int64_t* __restrict__ face_off, int B, const geocache_camera* __restrict__ cams, int N, RasterSplit split, int H, int W,
    float scale, unsigned long long* __restrict__ zbuf) {
    __shared__ geocache_camera s_cam[GEOCACHE_MAX_VIEWS];
    __shared__ int s_asset[2];
    __shared__ WarpFaces s_faces[kRasterThreads / 32];
    __shared__ int s_b[kRasterThreads];
    const int w0 = threadIdx.x & ~31, lane = threadIdx.x & 31;
    const int per_cta = split.faces * (kRasterThreads / 32);
    const long long f0 = blockIdx.x * (long long)per_cta, f_warp = f0 + (w0 >> 5) * split.faces;
    const long long f = f_warp + lane;
    // the CTA's faces belong to one asset unless it straddles a boundary
    if (threadIdx.x == 0) s_asset[0] = asset_of(face_off, B, f0);
    if (threadIdx.x == 1) s_asset[1] = asset_of(face_off, B, min(f0 + per_cta, nf) - 1);
    __syncthreads();
    const bool one_asset = s_asset[0] == s_asset[1];
    for (int i = threadIdx.x; i < N * 16; i += kRasterThreads) {
        const float x = __ldg(reinterpret_cast<const float*>(cams + (size_t)s_asset[0] * N) + i);
        reinterpret_cast<float*>(s_cam)[i] = (i & 15) >= 12 ? __fmul_rn(x, scale) : x;  // fx, fy, cx, cy
    }
    int b = s_asset[0];
    bool ok = lane < split.faces && f < nf;
    float X[3][3];
    if (ok) {
        if (!one_asset) b = asset_of(face_off, B, f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int32_t vi = __ldg(F + 3 * f + k);
            if (vi < 0 || vi >= nv) {
                atomicOr(&g_raster_error, 8u);
                ok = false;
                break;
            }
            X[k][0] = __ldg(V + 3 * (size_t)vi);
            X[k][1] = __ldg(V + 3 * (size_t)vi + 1);
            X[k][2] = __ldg(V + 3 * (size_t)vi + 2);
        }
    }
    s_b[threadIdx.x] = b;
    __syncthreads();
    // the CTA's views
    const int view0 = blockIdx.y * split.views, view1 = min(view0 + split.views, N);
    if (one_asset)
        raster_warp<true>(X, ok, b, (unsigned int)f_warp, s_cam, cams, s_b + w0, s_faces[w0 >> 5], N,
                          view0, view1, H, W, scale, zbuf);
    else
        raster_warp<false>(X, ok, b, (unsigned int)f_warp, s_cam, cams, s_b + w0, s_faces[w0 >> 5], N,
                          view0, view1, H, W, scale, zbuf);
}

// World position of the surface point of pixel (i, j) whose z-buffer key is
// `key` (not kEmpty): the ray through the pixel centre at the key's depth,
// x_w = R^T (x_c - t).
__device__ __forceinline__ void ray_position(const Cam32& c, unsigned long long key, float d0, float d1, float (&X)[3]) {
    const float s = __uint_as_float((unsigned int)(key >> 32));
    const float xc[3] = {__fsub_rn(__fmul_rn(s, d0), c.t[0]), __fsub_rn(__fmul_rn(s, d1), c.t[1]),
                         __fsub_rn(s, c.t[2])};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        float x = __fmul_rn(c.R[r], xc[0]);
        x = __fadd_rn(x, __fmul_rn(c.R[3 + r], xc[1]));
        X[r] = __fadd_rn(x, __fmul_rn(c.R[6 + r], xc[2]));
    }
}

__device__ __forceinline__ void key_position(const Cam32& c, unsigned long long key, int i, int j, float (&X)[3]) {
    float d0, d1;
    ray(c, __fadd_rn((float)i, 0.5f), __fadd_rn((float)j, 0.5f), d0, d1);
    ray_position(c, key, d0, d1, X);
}

__global__ void __launch_bounds__(kRasterThreads) raster_resolve_kernel(const unsigned long long* __restrict__ zbuf,
                                                                         const geocache_camera* __restrict__ cams,
                                                                         int N, int H, int W, long long n_pix,
                                                                         float* __restrict__ pos,
                                                                         uint8_t* __restrict__ valid) {
    const long long HW = (long long)H * W;
    for (long long p = blockIdx.x * (long long)kRasterThreads + threadIdx.x; p < n_pix;
         p += (long long)gridDim.x * kRasterThreads) {
        const unsigned long long key = zbuf[p];
        float X[3] = {0.0f, 0.0f, 0.0f};
        if (key != kEmpty) {
            const int pix = (int)(p % HW);
            key_position(load_cam(cams + p / HW), key, pix % W, pix / W, X);  // [B, N] cameras, one per map
        }
        pos[3 * p] = X[0];
        pos[3 * p + 1] = X[1];
        pos[3 * p + 2] = X[2];
        valid[p] = key != kEmpty;
    }
}

// Token (i, j) of a token-grid map from its s x s pixels (i s + sx, j s + sy)
// of the fine map: positions of the valid pixels summed componentwise in
// binary32, pixel rows sy ascending and sx ascending within a row, divided
// once by their number n; foreground when 2 n >= s * s.
struct PoolAcc {
    float sum[3] = {0.0f, 0.0f, 0.0f};
    int n = 0;
    __device__ __forceinline__ void add(const float (&X)[3]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[c] = __fadd_rn(sum[c], X[c]);
        ++n;
    }
    __device__ __forceinline__ void store(int s, float* __restrict__ pos, uint8_t* __restrict__ valid, long long p) const {
        const bool fg = n > 0 && 2 * n >= s * s;
#pragma unroll
        for (int c = 0; c < 3; ++c) pos[3 * p + c] = fg ? __fdiv_rn(sum[c], (float)n) : 0.0f;
        valid[p] = fg;
    }
};

// resolve + pool of a z-buffer rendered at s x the token grid: one thread per
// token, grid-stride over the B * N * H * W tokens.  S: s where it is 2, 4 or
// 8, 0 otherwise.  With S the key words of a row come by 16-byte loads and
// the ray components of the token's S rows and S columns are formed once (2 S
// IEEE divisions instead of 2 per covered pixel; the same quotients): 4
// meshes x 6 views at 512 x 512, s = 4, 16.7 -> 11.2 us.
template <int S>
__global__ void __launch_bounds__(kRasterThreads) raster_pool_kernel(const unsigned long long* __restrict__ zbuf,
                                                                      const geocache_camera* __restrict__ cams,
                                                                      int H, int W, int s, long long n_tok,
                                                                      float* __restrict__ pos,
                                                                      uint8_t* __restrict__ valid) {
    const long long HW = (long long)H * W;
    const int Ws = W * s;
    for (long long p = blockIdx.x * (long long)kRasterThreads + threadIdx.x; p < n_tok;
         p += (long long)gridDim.x * kRasterThreads) {
        const long long map = p / HW;
        const int tok = (int)(p % HW), i = tok % W, j = tok / W;
        const unsigned long long* zmap = zbuf + map * HW * s * s;
        const Cam32 c = load_cam(cams + map, (float)s);
        PoolAcc acc;
        if (S > 0) {
            float d0[S > 0 ? S : 1];
#pragma unroll
            for (int sx = 0; sx < S; ++sx)
                d0[sx] = __fdiv_rn(__fsub_rn(__fadd_rn((float)(i * S + sx), 0.5f), c.cx), c.fx);
#pragma unroll(S > 4 ? 2 : 4)
            for (int sy = 0; sy < S; ++sy) {
                const int J = j * S + sy;
                const ulonglong2* row = reinterpret_cast<const ulonglong2*>(zmap + (size_t)J * Ws + i * S);
                ulonglong2 k2[S > 0 ? S / 2 : 1];
#pragma unroll
                for (int h = 0; h < S / 2; ++h) k2[h] = __ldg(row + h);
                const float d1 = __fdiv_rn(__fsub_rn(__fadd_rn((float)J, 0.5f), c.cy), c.fy);
#pragma unroll
                for (int sx = 0; sx < S; ++sx) {
                    const unsigned long long key = sx & 1 ? k2[sx / 2].y : k2[sx / 2].x;
                    if (key == kEmpty) continue;
                    float X[3];
                    ray_position(c, key, d0[sx], d1, X);
                    acc.add(X);
                }
            }
        } else {
            for (int sy = 0; sy < s; ++sy)
                for (int sx = 0; sx < s; ++sx) {
                    const int I = i * s + sx, J = j * s + sy;
                    const unsigned long long key = __ldg(zmap + (size_t)J * Ws + I);
                    if (key == kEmpty) continue;
                    float X[3];
                    key_position(c, key, I, J, X);
                    acc.add(X);
                }
        }
        acc.store(s, pos, valid, p);
    }
}

// pool of fine maps given by the caller: pos_hi [n_maps, H s, W s, 3],
// valid_hi [n_maps, H s, W s] -> pos [n_maps, H, W, 3], valid [n_maps, H, W].
// HBM-bound.  S: s where it is 2, 4 or 8 and the maps are aligned, 0 otherwise.
// With S a token's row comes as one word of validity and 8- or 16-byte words of
// positions (scalar loads at s = 8 touch each
// 128-byte line 32 times): 96 maps of 512 x 512 to 64 x 64, 63.8 -> 33.2
// us (332 MB, of which the rows without foreground are not read).  Launched while
// the kernel that writes the fine maps may still run, so its loads are coherent
// ones after the wait.
template <int S>
__global__ void __launch_bounds__(kRasterThreads) pool_posmaps_kernel(const float* pos_hi,
                                                                       const uint8_t* valid_hi,
                                                                       int H, int W, int s, long long n_tok,
                                                                       float* __restrict__ pos,
                                                                       uint8_t* __restrict__ valid) {
    pdl_wait();
    const long long HW = (long long)H * W;
    const long long Ws = (long long)W * s;
    for (long long p = blockIdx.x * (long long)kRasterThreads + threadIdx.x; p < n_tok;
         p += (long long)gridDim.x * kRasterThreads) {
        const long long map = p / HW;
        const int tok = (int)(p % HW), i = tok % W, j = tok / W;
        const long long base = map * HW * s * s;
        PoolAcc acc;
        if (S > 0) {
            const long long q0 = base + (long long)j * S * Ws + (long long)i * S;
            uint32_t m[S > 0 ? S : 1][S > 4 ? 2 : 1];  // validity bytes of the token's rows
#pragma unroll
            for (int sy = 0; sy < S; ++sy) {
                const uint8_t* v = valid_hi + q0 + sy * Ws;
                if (S == 8) {
                    const uint2 w = __ldca(reinterpret_cast<const uint2*>(v));
                    m[sy][0] = w.x;
                    m[sy][S > 4 ? 1 : 0] = w.y;
                } else {
                    m[sy][0] = S == 4 ? __ldca(reinterpret_cast<const uint32_t*>(v))
                                      : (uint32_t)__ldca(reinterpret_cast<const unsigned short*>(v));
                }
            }
#pragma unroll
            for (int sy = 0; sy < S; ++sy) {
                const bool any = (m[sy][0] | m[sy][S > 4 ? 1 : 0]) != 0;  // a background row's positions are not read
                float x[3 * (S > 0 ? S : 1)];
                const float* row = pos_hi + 3 * (q0 + sy * Ws);
                if (S == 2) {
#pragma unroll
                    for (int h = 0; h < 3 * S / 2; ++h) {
                        const float2 w = any ? __ldca(reinterpret_cast<const float2*>(row) + h) : make_float2(0.f, 0.f);
                        x[2 * h] = w.x;
                        x[2 * h + 1] = w.y;
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 3 * S / 4; ++h) {
                        const float4 w =
                            any ? __ldca(reinterpret_cast<const float4*>(row) + h) : make_float4(0.f, 0.f, 0.f, 0.f);
                        x[4 * h] = w.x;
                        x[4 * h + 1] = w.y;
                        x[4 * h + 2] = w.z;
                        x[4 * h + 3] = w.w;
                    }
                }
#pragma unroll
                for (int sx = 0; sx < S; ++sx) {
                    if (!((m[sy][sx / 4] >> (8 * (sx % 4))) & 0xffu)) continue;
                    const float X[3] = {x[3 * sx], x[3 * sx + 1], x[3 * sx + 2]};
                    acc.add(X);
                }
            }
        } else {
            for (int sy = 0; sy < s; ++sy)
                for (int sx = 0; sx < s; ++sx) {
                    const long long q = base + ((long long)j * s + sy) * Ws + (long long)i * s + sx;
                    if (!__ldca(valid_hi + q)) continue;
                    const float X[3] = {__ldca(pos_hi + 3 * q), __ldca(pos_hi + 3 * q + 1), __ldca(pos_hi + 3 * q + 2)};
                    acc.add(X);
                }
        }
        acc.store(s, pos, valid, p);
    }
}

}  // namespace

cudaError_t read_raster_error(unsigned int* out, bool clear, cudaStream_t s) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_raster_error, sizeof(unsigned int), 0, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess || !clear || *out == 0) return e;
    static const unsigned int zero = 0;
    e = cudaMemcpyToSymbolAsync(g_raster_error, &zero, sizeof(unsigned int), 0, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

// grid of a grid-stride kernel over n items: at most 16 CTAs per SM
static unsigned stride_grid(long long n) {
    const long long want = (n + kRasterThreads - 1) / kRasterThreads, cap = (long long)sm_count() * 16;
    return (unsigned)(want < cap ? (want > 0 ? want : 1) : cap);
}

// All views and 32 faces per warp where that fills the GPU.  A render of more
// pixels per view than faces per asset is bound by its boxes' pixels: its views
// are split until there are 4 waves of CTAs, then its faces until there are 4
// again or a warp's faces hold about kRasterWarpPixels of a view's pixels.
// One of small faces is bound by loading them, which each CTA does again for
// its views: it fills one wave only.  Calls, us, unsplit and split: one mesh x 6
// views of 1,280 faces at 512 x 512 718 and 38 (views alone 137; 512 and 1024
// pixels a warp 36 and 47, but two such meshes at 160 x 160 19 and 26 against
// 16), of 20,480 at 288 x 288 90 and 35, of 5,120 at 64 x 64 19 and 8; 3 x 8
// views of 81,920 at 296 x 512 278 and 240; one x 6 of 81,920 at 128 x 128 19
// and (views split) 23, so those stay whole.
constexpr long long kRasterWarpPixels = 256;

static RasterSplit raster_split(long long nf, int B, int N, long long n_pix) {
    const long long slots = (long long)kRasterBlocks * sm_count(), gx = (nf + kRasterThreads - 1) / kRasterThreads;
    const bool heavy = n_pix * B > nf;
    long long chunks = heavy ? (4 * slots + gx - 1) / gx : slots / gx;
    chunks = chunks < 1 ? 1 : (chunks > N ? N : chunks);
    RasterSplit split{(int)((N + chunks - 1) / chunks), 32};
    while (heavy && split.views == 1 && split.faces > 1 && n_pix * B / nf * split.faces > kRasterWarpPixels &&
           gx * N * (32 / split.faces) < 4 * slots)
        split.faces /= 2;
    return split;
}

cudaError_t launch_raster(const float* V, long long nv, const int32_t* F, long long nf, const int64_t* face_off,
                          int B, const geocache_camera* cams, int N, int H, int W, int ss, unsigned long long* zbuf,
                          float* pos, uint8_t* valid, cudaStream_t s) {
    const long long n_tok = (long long)B * N * H * W, n_pix = n_tok * ss * ss;
    cudaError_t e = cudaMemsetAsync(zbuf, 0xff, sizeof(unsigned long long) * (size_t)n_pix, s);
    if (e != cudaSuccess) return e;
    if (nf > 0) {
        const RasterSplit split = raster_split(nf, B, N, (long long)H * W * ss * ss);
        const long long per_cta = split.faces * (kRasterThreads / 32), gx = (nf + per_cta - 1) / per_cta;
        if (gx > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        note_launches(1);
        raster_faces_kernel<<<dim3((unsigned)gx, (unsigned)((N + split.views - 1) / split.views)), kRasterThreads, 0, s>>>(
            V, nv, F, nf, face_off, B, cams, N, split, H * ss, W * ss, (float)ss, zbuf);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    note_launches(1);
    if (ss == 1)
        raster_resolve_kernel<<<stride_grid(n_pix), kRasterThreads, 0, s>>>(zbuf, cams, N, H, W, n_pix, pos, valid);
    else {
        // 16-byte loads need a 16-byte aligned z-buffer (every token row then starts on 16 bytes)
        auto kern = raster_pool_kernel<0>;
        if ((uintptr_t)zbuf % 16 == 0) {
            if (ss == 2) kern = raster_pool_kernel<2>;
            else if (ss == 4) kern = raster_pool_kernel<4>;
            else if (ss == 8) kern = raster_pool_kernel<8>;
        }
        kern<<<stride_grid(n_tok), kRasterThreads, 0, s>>>(zbuf, cams, H, W, ss, n_tok, pos, valid);
    }
    return cudaGetLastError();
}

cudaError_t launch_pool_posmaps(const float* pos_hi, const uint8_t* valid_hi, long long n_maps, int H, int W, int ss,
                                float* pos, uint8_t* valid, cudaStream_t s) {
    const long long n_tok = n_maps * H * W;
    if (n_tok == 0) return cudaSuccess;
    // a token's row starts at a multiple of s validity bytes and 12 s position bytes
    auto kern = pool_posmaps_kernel<0>;
    if ((uintptr_t)pos_hi % 16 == 0 && (uintptr_t)valid_hi % 8 == 0) {
        if (ss == 2) kern = pool_posmaps_kernel<2>;
        else if (ss == 4) kern = pool_posmaps_kernel<4>;
        else if (ss == 8) kern = pool_posmaps_kernel<8>;
    }
    return launch_pdl(kern, dim3(stride_grid(n_tok)), kRasterThreads, 0, s, pos_hi, valid_hi, H, W, ss, n_tok, pos, valid);
}

}  // namespace geocache
