// CUDA kernels (sm_103a) of the geometric delta transport (GeoCache,
// Sec. 3.2): tau, the correspondence tables, the fused transport +
// reconstruction step, and the full-step reconstruction.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cooperative_groups.h>

#include <atomic>
#include <cfloat>
#include <cstdint>

#include "geocache_device.cuh"
#include "geocache_internal.h"

namespace geocache {

__host__ __device__ int tiles_per_view(int H, int W) { return (H * W + GEOCACHE_TILE_TOKENS - 1) / GEOCACHE_TILE_TOKENS; }

// Loads: __ldg (ld.global.nc) is for memory that nothing writes while the kernel
// is resident.  A kernel launched early (launch_pdl, phase B) is resident before
// the kernel that writes its inputs has ended, and an in-place step writes rows
// that it reads; those load by __ldca or __ldcs, which are coherent.

// ---------------------------------------------------------------- latents --
__device__ __forceinline__ float lat_load(const float* p, size_t i) { return __ldca(p + i); }
__device__ __forceinline__ float lat_load(const __nv_bfloat16* p, size_t i) {
    return __bfloat162float(p[i]);
}
__device__ __forceinline__ void lat_store(float* p, size_t i, float v) { p[i] = v; }
__device__ __forceinline__ void lat_store(__nv_bfloat16* p, size_t i, float v) {
    p[i] = __float2bfloat16_rn(v);
}

// Sampler conversion of one element (Sec. 3.2, closed-form relations after
// Eq. 1).  Fixed operation sequence (explicit intrinsics) so that the fused
// transport step and the standalone reconstruction agree bit for bit.
__device__ __forceinline__ float recon_one(const ReconCoef& c, float xt, float x0, float& pred) {
    if (c.sampler == GEOCACHE_DDIM) {
        const float eps = __fmul_rn(__fmaf_rn(-c.st, x0, xt), c.inv_s1t);
        pred = (c.pred_kind == GEOCACHE_PRED_V) ? __fmaf_rn(c.st, eps, -__fmul_rn(c.s1t, x0)) : eps;
        return __fmaf_rn(c.sp, x0, __fmul_rn(c.s1p, eps));
    } else {
        const float vel = __fmul_rn(__fsub_rn(xt, x0), c.inv_sigma);
        pred = vel;
        return __fmaf_rn(c.dsigma, vel, xt);
    }
}

// One kept tap's term of an anchor's transported quantity, accumulated in
// tap order: Eq. 1 carries the anchor's change x0_new - x0(t-1); the
// value-copy ablation (Sec. 4.3, "delta -> copy") carries x0_new itself.
__device__ __forceinline__ float tap_term(bool copy, float w, float xn, float xp, float acc) {
    return __fmaf_rn(w, copy ? xn : __fsub_rn(xn, xp), acc);
}

// x0(t) of a covered target from x0(t-1) and the anchor-ordered sum g of its
// n covering anchors' terms: x0 + g/n (Eq. 1, normalised multi-anchor sum),
// or g/n under the value copy.
__device__ __forceinline__ float fold_one(bool copy, float x0, float g, int n) {
    // g / n correctly rounded; for n a power of two that is exactly g * (1 / n)
    const float m = n == 1 ? g
                           : ((n & (n - 1)) == 0 ? __fmul_rn(g, __frcp_rn((float)n)) : __fdiv_rn(g, (float)n));
    return copy ? m : __fadd_rn(x0, m);
}

// -------------------------------------------------------------------- tau --
// One thread-block cluster per asset: CTA r of the cluster reduces the
// componentwise min / max of the foreground texels of slice r of the asset's
// texels (exact and order-free), the cluster combines the partial boxes through
// distributed shared memory, and CTA 0 writes tau = tol_frac * sqrt(diag^2)
// with the squares summed ((d0^2 + d1^2) + d2^2) in binary32.
constexpr int kTauBlocks = 4;

struct Box {
    float lo[3], hi[3];
    int any;
};

__device__ __forceinline__ void box_reduce_warp(Box& x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x.lo[c] = fminf(x.lo[c], __shfl_xor_sync(0xffffffffu, x.lo[c], off));
            x.hi[c] = fmaxf(x.hi[c], __shfl_xor_sync(0xffffffffu, x.hi[c], off));
        }
        x.any |= __shfl_xor_sync(0xffffffffu, x.any, off);
    }
}

__global__ void __launch_bounds__(256, kTauBlocks) tau_kernel(const float* __restrict__ pos, const uint8_t* __restrict__ valid,
                                                     int N, int HW, float tol_frac, int quads, float* __restrict__ tau) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int b = blockIdx.x / cs;
    __shared__ Box s_warp[16];
    __shared__ Box s_part;
    Box x;
#pragma unroll
    for (int c = 0; c < 3; ++c) { x.lo[c] = FLT_MAX; x.hi[c] = -FLT_MAX; }
    x.any = 0;
    // the asset's N views are contiguous: each CTA of the cluster takes one
    // slice of their N * HW texels
    const size_t n = (size_t)N * HW;
    const size_t base = (size_t)b * n;
    if (quads) {  // four texels per load: their 4 validity bytes and 12 position floats
        const size_t nq = n / 4, per = (nq + cs - 1) / cs;
        const size_t q0 = (size_t)rank * per, q1 = q0 + per < nq ? q0 + per : nq;
        const uint32_t* vq = reinterpret_cast<const uint32_t*>(valid + base);
        const float4* pq = reinterpret_cast<const float4*>(pos + 3 * base);
        // four quads per thread and round: their validity words in flight
        // together, then the positions of those with foreground (background
        // quads' positions are not read)
        for (size_t i0 = q0 + threadIdx.x; i0 < q1; i0 += 4 * blockDim.x) {
            uint32_t m[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) m[j] = i0 + j * blockDim.x < q1 ? __ldg(vq + i0 + j * blockDim.x) : 0u;
            float4 f[4][3];
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    f[j][k] = m[j] ? __ldg(pq + 3 * (i0 + j * blockDim.x) + k) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float* p = reinterpret_cast<const float*>(f[j]);
                x.any |= m[j] != 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (!((m[j] >> (8 * k)) & 0xffu)) continue;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        x.lo[c] = fminf(x.lo[c], p[3 * k + c]);
                        x.hi[c] = fmaxf(x.hi[c], p[3 * k + c]);
                    }
                }
            }
        }
    } else {
        const size_t per = (n + cs - 1) / cs;
        const size_t i0 = (size_t)rank * per, i1 = i0 + per < n ? i0 + per : n;
        for (size_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            if (!__ldg(valid + base + i)) continue;
            x.any = 1;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float p = __ldg(pos + 3 * (base + i) + c);
                x.lo[c] = fminf(x.lo[c], p);
                x.hi[c] = fmaxf(x.hi[c], p);
            }
        }
    }
    box_reduce_warp(x);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        if (lane < nw) x = s_warp[lane];
        else {
#pragma unroll
            for (int c = 0; c < 3; ++c) { x.lo[c] = FLT_MAX; x.hi[c] = -FLT_MAX; }
            x.any = 0;
        }
        box_reduce_warp(x);
        if (lane == 0) s_part = x;
    }
    cluster.sync();  // every CTA's partial box is in its shared memory
    if (rank == 0 && threadIdx.x == 0) {
        Box t = s_part;
        for (int r = 1; r < cs; ++r) {
            const Box* o = cluster.map_shared_rank(&s_part, r);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                t.lo[c] = fminf(t.lo[c], o->lo[c]);
                t.hi[c] = fmaxf(t.hi[c], o->hi[c]);
            }
            t.any |= o->any;
        }
        float tv = 0.0f;
        if (t.any) {
            const float d0 = __fsub_rn(t.hi[0], t.lo[0]), d1 = __fsub_rn(t.hi[1], t.lo[1]),
                        d2 = __fsub_rn(t.hi[2], t.lo[2]);
            const float diag2 = __fadd_rn(__fadd_rn(__fmul_rn(d0, d0), __fmul_rn(d1, d1)), __fmul_rn(d2, d2));
            tv = __fmul_rn(tol_frac, __fsqrt_rn(diag2));
        }
        tau[b] = tv;
    }
    cluster.sync();  // the other CTAs' shared memory stays alive until CTA 0 has read it
}

cudaError_t launch_tau(const float* pos, const uint8_t* valid, int B, int N, int H, int W, float tol_frac,
                       float* tau, cudaStream_t s) {
    // a cluster of 8 CTAs (the portable size) per asset, 4 CTAs resident per SM
    // (64 registers: the loads in flight)
    const int cs = 8;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B * cs);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // quads: every view's texels start on a 4-texel boundary with 16-byte aligned positions
    const int quads = (H * W) % 4 == 0 && (uintptr_t)pos % 16 == 0 && (uintptr_t)valid % 4 == 0;
    note_launches(1);
    return cudaLaunchKernelEx(&cfg, tau_kernel, pos, valid, N, H * W, tol_frac, quads, tau);
}

// ------------------------------------------------------- correspondence --
// One CTA per 256 tokens of (asset b, target view v).  The CTA's foreground
// tokens are compacted first (warp ballots), so that thread t takes the t-th
// foreground token and the warps that test taps are full; each such thread
// loops over the source views u with the target's position loaded once.
// Background tokens get empty rows from their own thread.  Writes the keep
// masks and (TABLES, when requested) the idx/w tables of every pair; with
// tile_cnt given, adds the kept rows of each (b, v, u, tile) to its count
// (one atomic per warp: a CTA's 256 tokens lie in one tile).  Without tables
// only the keep masks are formed (no renormalised weights): 581 -> 507 us
// for the build graph of 128 assets.
constexpr int kBuildThreads = 256;
static_assert(GEOCACHE_TILE_TOKENS % kBuildThreads == 0, "a build CTA's tokens lie in one tile");

// A build CTA covers REP slices of kBuildThreads tokens of one view (REP = 1
// or 4): its foreground tokens are compacted across the slices and each
// thread takes up to REP of them in turn, so that fewer lanes idle through
// the source loop (the background is ~60% of a view).  REP = 4 for large
// builds with tables (large builds without take build_keep_kernel), 1 for
// small ones, where the 4x fewer CTAs would not fill the GPU.
template <int K, bool TABLES, int REP, bool SPLIT>
__global__ void __launch_bounds__(kBuildThreads) build_corr_kernel(const float* __restrict__ pos,
                                                         const uint8_t* __restrict__ valid,
                                                         const geocache_camera* __restrict__ cams,
                                                         const float* __restrict__ tau, int N, int H, int W,
                                                         int32_t* __restrict__ idx, float* __restrict__ wout,
                                                         uint8_t* __restrict__ keep, int32_t* __restrict__ tile_cnt,
                                                         int n_split) {
    static_assert(GEOCACHE_TILE_TOKENS % (kBuildThreads * REP) == 0, "a build CTA's tokens lie in one tile");
    const int HW = H * W;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int p_base = blockIdx.x * kBuildThreads * REP;
    // SPLIT: n_split CTAs share the source views of the same tokens
    const int v = SPLIT ? blockIdx.y / n_split : blockIdx.y, b = blockIdx.z;
    const int part = SPLIT ? (int)blockIdx.y - v * n_split : 0;
    const int u_first = SPLIT ? part * N / n_split : 0, u_last = SPLIT ? (part + 1) * N / n_split : N;
    __shared__ geocache_camera s_cam[GEOCACHE_MAX_VIEWS];
    __shared__ int s_fg[kBuildThreads * REP];
    __shared__ int s_wcnt[REP][kBuildThreads / 32];
    for (int i = t; i < N * 16; i += kBuildThreads)
        reinterpret_cast<float*>(s_cam)[i] = __ldg(reinterpret_cast<const float*>(cams + (size_t)b * N) + i);
    const size_t view0 = ((size_t)b * N + v) * HW;
    // compaction of the foreground tokens of the CTA's REP slices, in token order
    bool in_h[REP], fg_h[REP];
    unsigned bal[REP];
#pragma unroll
    for (int h = 0; h < REP; ++h) {
        const int ph = p_base + h * kBuildThreads + t;
        in_h[h] = ph < HW;
        fg_h[h] = in_h[h] && __ldg(valid + view0 + ph);
        bal[h] = __ballot_sync(0xffffffffu, fg_h[h]);
        if (lane == 0) s_wcnt[h][warp] = __popc(bal[h]);
    }
    __syncthreads();
    int n_fg = 0;
#pragma unroll
    for (int h = 0; h < REP; ++h) {
        int before = n_fg, tot = 0;
#pragma unroll
        for (int w = 0; w < kBuildThreads / 32; ++w) {
            before += w < warp ? s_wcnt[h][w] : 0;
            tot += s_wcnt[h][w];
        }
        if (fg_h[h]) s_fg[before + __popc(bal[h] & ((1u << lane) - 1u))] = h * kBuildThreads + t;
        n_fg += tot;
    }
    __syncthreads();
    const int T = tiles_per_view(H, W);
    const float tu = __ldg(tau + b);
    const float tau2 = __fmul_rn(tu, tu);
#pragma unroll 1
    for (int it = 0; it < REP; ++it) {
        const int jw = it * kBuildThreads + t;
        if (it > 0 && it * kBuildThreads >= n_fg) break;  // the same for every thread of the CTA
        const bool work = jw < n_fg;
        const int pw = p_base + (work ? s_fg[jw] : 0);  // this thread's foreground token
        float X0 = 0.f, X1 = 0.f, X2 = 0.f;
        if (work) {
            X0 = __ldg(pos + 3 * (view0 + pw));
            X1 = __ldg(pos + 3 * (view0 + pw) + 1);
            X2 = __ldg(pos + 3 * (view0 + pw) + 2);
        }
        for (int u = u_first; u < u_last; ++u) {
            Taps tp;
            taps_clear(tp);
            int mask = 0;
            if (work && u != v) {
                const size_t su = ((size_t)b * N + u) * HW;
                if (TABLES) {
                    compute_taps<K>(s_cam[u], pos + 3 * su, valid + su, H, W, X0, X1, X2, tau2, tp, &mask);
                } else {
                    Footprint fp;
                    if (footprint<K>(s_cam[u], X0, X1, X2, H, W, fp))
                        mask = tap_mask<K>(fp, pos + 3 * su, valid + su, H, W, X0, X1, X2, tau2);
                }
            }
            if (tile_cnt) {
                const unsigned kept = __ballot_sync(0xffffffffu, mask != 0);
                if (lane == 0 && kept)
                    atomicAdd(tile_cnt + (((size_t)b * N + v) * N + u) * T + p_base / GEOCACHE_TILE_TOKENS,
                              __popc(kept));
            }
            const size_t row0 = (((size_t)b * N + v) * N + u) * HW;
            if (keep) {
                if (it == 0) {
#pragma unroll
                    for (int h = 0; h < REP; ++h)
                        if (in_h[h] && !fg_h[h]) keep[row0 + p_base + h * kBuildThreads + t] = 0;
                }
                if (work) keep[row0 + pw] = (uint8_t)mask;
            }
            if (!TABLES || !idx) continue;
            if (it == 0) {
#pragma unroll
                for (int h = 0; h < REP; ++h) {
                    if (!(in_h[h] && !fg_h[h])) continue;
                    const size_t e = row0 + p_base + h * kBuildThreads + t;
                    if (K == 4) {
                        reinterpret_cast<int4*>(idx)[e] = make_int4(-1, -1, -1, -1);
                        reinterpret_cast<float4*>(wout)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                    } else {
                        idx[e] = -1;
                        wout[e] = 0.0f;
                    }
                }
            }
            if (work) {
                if (K == 4) {
                    reinterpret_cast<int4*>(idx)[row0 + pw] = make_int4(tp.q[0], tp.q[1], tp.q[2], tp.q[3]);
                    reinterpret_cast<float4*>(wout)[row0 + pw] = make_float4(tp.w[0], tp.w[1], tp.w[2], tp.w[3]);
                } else {
                    idx[row0 + pw] = tp.q[0];
                    wout[row0 + pw] = tp.w[0];
                }
            }
        }
    }
}

// ---- large builds without tables: keep masks with an occlusion test first --
// Most (token, source view) pairs keep no tap because the token's point X is
// hidden in the source view: the surface there is nearer than X by more than
// the tolerance.  source_depth_kernel therefore stores, for each block of 8 x 8
// texels of every view, a camera depth that no kept tap's target exceeds, and
// build_keep_kernel tests taps only for the pairs that pass (17% of the pairs
// of a 6-view batch keep a tap, 25% pass; with blocks of 4 and 16: 23%, 28%).
//
// The bound: a kept tap's texel P lies within tau of X (to 1e-6 relative in
// binary32), so the depths z = R2 . x + t2 of P and X differ by at most
// |R2| tau, plus the rounding of both, at most 4 * 2^-24 S each with
// S = |R2| . |x| + |t2| summed by component.  A block's value is the largest
// z + 1e-6 S of its foreground texels plus |R2| tau (1 + 1e-5) and the change of
// S over a distance tau; -inf without foreground.  It covers 9 x 9 texels: the
// block and the column and row after it, so that one value serves every
// footprint whose top-left tap lies in the block.  A NaN never rejects, and
// nothing is rejected where a square underflows: with tau^2 or |R2|^2 below
// 1e-30 the tap test's distances (then of few or no bits) or |R2| say nothing
// about the depths.
//
// The values lie in the keep masks' diagonal rows (u = v), which hold no masks
// and are cleared after the build, so that no scratch is needed.
constexpr int kDepthBlock = 8;
__host__ __device__ inline int depth_blocks(int n) { return (n + kDepthBlock - 1) / kDepthBlock; }

__device__ __forceinline__ float* depth_row(uint8_t* keep, size_t view, int v, int N, size_t HW) {
    const uintptr_t p = reinterpret_cast<uintptr_t>(keep + (view * N + v) * HW);
    return reinterpret_cast<float*>((p + 3) & ~(uintptr_t)3);
}

// the 16-byte chunk `i` of the address range [p, p + n), cleared; i runs from 0
// to n / 16 + 1 (an unaligned range has a part of a chunk at either end)
__device__ __forceinline__ void clear_chunk(uint8_t* p, int n, int i) {
    const intptr_t lo = 16 * (intptr_t)i - (reinterpret_cast<uintptr_t>(p) & 15);
    if (lo >= 0 && lo + 16 <= n) {
        *reinterpret_cast<uint4*>(p + lo) = make_uint4(0, 0, 0, 0);
    } else {
        for (intptr_t k = lo < 0 ? 0 : lo; k < lo + 16 && k < n; ++k) p[k] = 0;
    }
}

// One warp per 4 blocks of a row of blocks: lane l reads column l of their 9
// texel rows (coalesced; a warp per block, 9 texels a row, took 27 us against
// 15 at 64 assets x 6 views of 128 x 128, bound by the L1's wavefronts), and 9
// lanes the column after them.
__global__ void __launch_bounds__(256) source_depth_kernel(const float* __restrict__ pos,
                                                           const uint8_t* __restrict__ valid,
                                                           const geocache_camera* __restrict__ cams,
                                                           const float* __restrict__ tau, int N, int H, int W,
                                                           uint8_t* keep) {
    constexpr int kRows = kDepthBlock + 1;
    const int nbx = depth_blocks(W), n_strips = (nbx + 3) / 4;
    const int lane = threadIdx.x & 31, strip = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (strip >= n_strips * depth_blocks(H)) return;
    const int v = blockIdx.y, b = blockIdx.z;
    const size_t view = (size_t)b * N + v, HW = (size_t)H * W;
    const float* cam = reinterpret_cast<const float*>(cams + view);
    const float r0 = __ldg(cam + 6), r1 = __ldg(cam + 7), r2 = __ldg(cam + 8), t2 = __ldg(cam + 11);
    const int by = strip / n_strips, y0 = by * kDepthBlock, x0 = (strip - by * n_strips) * 4 * kDepthBlock;
    const uint8_t* valid_v = valid + view * HW;
    const float* pos_v = pos + 3 * view * HW;
    bool fg[kRows + 1];
    float p[kRows + 1][3];
#pragma unroll
    for (int k = 0; k <= kRows; ++k) {  // the last round: lane l's texel is row l of the next strip's first column
        const int y = k < kRows ? y0 + k : y0 + lane, x = k < kRows ? x0 + lane : x0 + 4 * kDepthBlock;
        const size_t q = (size_t)y * W + x;
        fg[k] = y < H && x < W && (k < kRows || lane < kRows);
        fg[k] = fg[k] && __ldg(valid_v + q);
#pragma unroll
        for (int c = 0; c < 3; ++c) p[k][c] = fg[k] ? __ldg(pos_v + 3 * q + c) : 0.0f;
    }
    float z = -INFINITY, z_next = -INFINITY;
#pragma unroll
    for (int k = 0; k <= kRows; ++k) {
        const float s = fabsf(r0 * p[k][0]) + fabsf(r1 * p[k][1]) + fabsf(r2 * p[k][2]) + fabsf(t2);
        float far = r0 * p[k][0] + r1 * p[k][1] + r2 * p[k][2] + t2 + 1e-6f * s;
        far = far <= FLT_MAX ? far : INFINITY;  // an overflow or NaN: the block rejects nothing
        if (fg[k]) (k < kRows ? z : z_next) = fmaxf(k < kRows ? z : z_next, far);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) z_next = fmaxf(z_next, __shfl_xor_sync(0xffffffffu, z_next, off));
    float block = z;  // over the block's 8 columns, then the next block's first
#pragma unroll
    for (int off = 1; off < kDepthBlock; off <<= 1) block = fmaxf(block, __shfl_xor_sync(0xffffffffu, block, off));
    const float after = __shfl_down_sync(0xffffffffu, z, kDepthBlock);
    block = fmaxf(block, lane < 32 - kDepthBlock ? after : z_next);
    const int bx = (x0 + lane) / kDepthBlock;
    if (lane % kDepthBlock == 0 && bx < nbx) {
        const float t = __ldg(tau + b);
        const float sq = r0 * r0 + r1 * r1 + r2 * r2, norm2 = sqrtf(sq), norm1 = fabsf(r0) + fabsf(r1) + fabsf(r2);
        const bool bounded = t * t >= 1e-30f && sq >= 1e-30f;
        depth_row(keep, view, v, N, HW)[by * nbx + bx] =
            bounded ? block + t * (1.00001f * norm2 + 1e-6f * norm1) : INFINITY;
    }
}

// One CTA per tile (asset b, target view v, GEOCACHE_TILE_TOKENS tokens).  Its
// foreground tokens are compacted with their positions; each thread then
// projects a token into every source view, and the pairs that pass the depth
// test are queued per warp and their taps tested 32 at a time, so that the
// gathers of a warp are full.  The tile's rows of the masks are cleared first
// and only kept masks written; the CTA's counts are the tile's.
//
// 64 assets x 6 views at 128 x 128: 140 -> 87 us (and 15 us for the depths).
// With the taps of every pair tested (16 scalar gathers each) the L1's
// wavefronts were 71% and the issue slots 67% busy; here the slots are 78% busy
// with the projections (78 M instructions against 105 M), the wavefronts 56%.
// 6 resident CTAs per SM (40 registers); 7 or 8 spill and take 116 us.
struct PairQueue {
    uint32_t what[64];  // compacted token | source view << 10 | taps of weight 0 << 16
    uint32_t at[64];    // footprint corner: (i0 + 1) | (j0 + 1) << 16
};

template <int K>
__global__ void __launch_bounds__(kBuildThreads) build_keep_kernel(const float* __restrict__ pos,
                                                                   const uint8_t* __restrict__ valid,
                                                                   const geocache_camera* __restrict__ cams,
                                                                   const float* __restrict__ tau, int N, int H, int W,
                                                                   uint8_t* keep, int32_t* __restrict__ tile_cnt) {
    constexpr int kReps = GEOCACHE_TILE_TOKENS / kBuildThreads, kWarps = kBuildThreads / 32;
    __shared__ geocache_camera s_cam[GEOCACHE_MAX_VIEWS];
    __shared__ float4 s_tok[GEOCACHE_TILE_TOKENS];  // foreground tokens: position, token
    __shared__ PairQueue s_queue[kWarps];
    __shared__ int s_wcnt[kReps][kWarps];
    __shared__ int s_cnt[GEOCACHE_MAX_VIEWS];
    const int HW = H * W, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int p_base = blockIdx.x * GEOCACHE_TILE_TOKENS, v = blockIdx.y, b = blockIdx.z;
    const int n_tok = min(GEOCACHE_TILE_TOKENS, HW - p_base);
    for (int i = t; i < N * 16; i += kBuildThreads)
        reinterpret_cast<float*>(s_cam)[i] = __ldg(reinterpret_cast<const float*>(cams + (size_t)b * N) + i);
    if (t < N) s_cnt[t] = 0;
    const size_t view = (size_t)b * N + v, view0 = view * HW;
    // compaction of the foreground tokens, in token order
    unsigned bal[kReps];
    bool fg[kReps];
#pragma unroll
    for (int h = 0; h < kReps; ++h) {
        const int i = h * kBuildThreads + t;
        fg[h] = i < n_tok && __ldg(valid + view0 + p_base + i);
        bal[h] = __ballot_sync(0xffffffffu, fg[h]);
        if (lane == 0) s_wcnt[h][warp] = __popc(bal[h]);
    }
    // the tile's mask rows of the other views, cleared
    uint8_t* const rows = keep + view * N * HW + p_base;
    if (((reinterpret_cast<uintptr_t>(rows) | (uintptr_t)HW | (uintptr_t)n_tok) & 15) == 0) {
        for (int i = t; i < N * 64; i += kBuildThreads) {
            const int u = i >> 6, c = i & 63;
            if (u != v && 16 * c < n_tok) reinterpret_cast<uint4*>(rows + (size_t)u * HW)[c] = make_uint4(0, 0, 0, 0);
        }
    } else {
        for (int i = t; i < N * 128; i += kBuildThreads) {  // at most 65 chunks a row
            const int u = i >> 7, c = i & 127;
            if (u != v && c <= n_tok / 16 + 1) clear_chunk(rows + (size_t)u * HW, n_tok, c);
        }
    }
    __syncthreads();
    int n_fg = 0;
#pragma unroll
    for (int h = 0; h < kReps; ++h) {
        int before = n_fg, tot = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            before += w < warp ? s_wcnt[h][w] : 0;
            tot += s_wcnt[h][w];
        }
        if (fg[h]) {
            const int p = p_base + h * kBuildThreads + t;
            const float* q = pos + 3 * (view0 + p);
            s_tok[before + __popc(bal[h] & ((1u << lane) - 1u))] =
                make_float4(__ldg(q), __ldg(q + 1), __ldg(q + 2), __int_as_float(p));
        }
        n_fg += tot;
    }
    __syncthreads();
    const float tu = __ldg(tau + b), tau2 = __fmul_rn(tu, tu);
    const int nbx = depth_blocks(W);
    PairQueue& q = s_queue[warp];
    const uint32_t below = (1u << lane) - 1u;
    int head = 0, queued = 0;
    auto test_taps = [&]() {  // the queue's pair `head + lane`
        const uint32_t what = q.what[(head + lane) & 63], at = q.at[(head + lane) & 63];
        const int u = (int)((what >> 10) & 63u), i0 = (int)(at & 0xffffu) - 1, j0 = (int)(at >> 16) - 1;
        const float4 X = s_tok[what & 1023u];
        const uint8_t* valid_u = valid + ((size_t)b * N + u) * HW;
        const float* pos_u = pos + 3 * ((size_t)b * N + u) * HW;
        int mask = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int col = i0 + (k & 1), row = j0 + (k >> 1);
            if ((unsigned)col >= (unsigned)W || (unsigned)row >= (unsigned)H || ((what >> (16 + k)) & 1u)) continue;
            const int tap = row * W + col;
            const int ok = __ldg(valid_u + tap) != 0;
            const int near = sqdist(pos_u + 3 * (size_t)tap, X.x, X.y, X.z) <= tau2;
            mask |= (ok & near) << k;
        }
        if (mask) {
            keep[(view * N + u) * HW + __float_as_int(X.w)] = (uint8_t)mask;
            atomicAdd(&s_cnt[u], 1);
        }
    };
#pragma unroll 1
    for (int j0 = 0; j0 < n_fg; j0 += kBuildThreads) {
        const int j = j0 + t;
        const bool work = j < n_fg;
        const float4 X = s_tok[work ? j : 0];
        for (int u = 0; u < N; ++u) {
            if (u == v) continue;
            bool pass = false;
            uint32_t what = 0, at = 0;
            Footprint f;
            float depth;
            if (work && footprint<K>(s_cam[u], X.x, X.y, X.z, H, W, f, depth)) {
                const float* far = depth_row(keep, (size_t)b * N + u, u, N, HW);
                const int blk = max(f.j0, 0) / kDepthBlock * nbx + max(f.i0, 0) / kDepthBlock;
                pass = !(depth > far[blk]);
                uint32_t dead = 0;  // taps of weight 0
                if (K == 4)
                    dead = (f.ax[0] == 0.0f ? 5u : 0u) | (f.ax[1] == 0.0f ? 10u : 0u) | (f.ay[0] == 0.0f ? 3u : 0u) |
                           (f.ay[1] == 0.0f ? 12u : 0u);
                what = (uint32_t)j | ((uint32_t)u << 10) | (dead << 16);
                at = (uint32_t)(f.i0 + 1) | ((uint32_t)(f.j0 + 1) << 16);
            }
            const uint32_t passed = __ballot_sync(0xffffffffu, pass);
            if (pass) {
                const int e = (head + queued + __popc(passed & below)) & 63;
                q.what[e] = what;
                q.at[e] = at;
            }
            queued += __popc(passed);
            if (queued >= 32) {
                __syncwarp();
                test_taps();
                __syncwarp();  // its entries are rewritten by later pairs
                head += 32;
                queued -= 32;
            }
        }
    }
    __syncwarp();
    if (lane < queued) test_taps();
    if (tile_cnt) {
        __syncthreads();
        if (t < N) tile_cnt[(view * N + t) * gridDim.x + blockIdx.x] = s_cnt[t];
    }
}

// the diagonal rows, cleared of the depths
__global__ void __launch_bounds__(256) clear_diagonal_kernel(uint8_t* keep, int N, int HW) {
    uint8_t* row = keep + ((size_t)blockIdx.z * N + blockIdx.y) * N * HW + (size_t)blockIdx.y * HW;
    clear_chunk(row, HW, blockIdx.x * 256 + threadIdx.x);
}

// CTAs from which a build's CTAs take all source views of their tokens.  With
// fewer, a CTA's views in sequence are the time of the kernel: one asset of 6
// views at 64 x 64 (96 CTAs) 7.5 us, with its views split over 576 CTAs 4.3; 4
// views at 96 x 96 (144) 5.4 and 4.0, 8 at 64 x 64 (128) 9.5 and 5.7.  From 384 CTAs (6 views at 128 x 128)
// on the split gains nothing (8.6 and 8.3), beyond 608 (4 per SM) it loses.
constexpr long long kBuildCtas = 608;

template <int K, bool TABLES, int REP>
static void launch_build_corr_rep(const geocache_corr& c, int32_t* cnt, cudaStream_t s) {
    const int HW = c.H * c.W, gx = (HW + kBuildThreads * REP - 1) / (kBuildThreads * REP);
    const long long ctas = (long long)gx * c.N * c.B, want = (kBuildCtas + ctas - 1) / ctas;
    const int n_split = (int)(want < c.N ? want : c.N);
    note_launches(1);
    if (REP == 1 && n_split > 1)
        build_corr_kernel<K, TABLES, 1, true><<<dim3(gx, c.N * n_split, c.B), kBuildThreads, 0, s>>>(
            c.pos, c.valid, c.cams, c.tau, c.N, c.H, c.W, c.idx, c.w, c.keep, cnt, n_split);
    else
        build_corr_kernel<K, TABLES, REP, false><<<dim3(gx, c.N, c.B), kBuildThreads, 0, s>>>(
            c.pos, c.valid, c.cams, c.tau, c.N, c.H, c.W, c.idx, c.w, c.keep, cnt, 1);
}

// Whether a build without tables tests depths first: where its fewer, larger CTAs
// and two extra launches pay.  That takes tiles that are mostly full, or many views
// to project into, and more tiles for single taps, which have less to skip, and for
// masks whose rows are not 16-byte aligned, which are cleared in pieces.  tau,
// masks and offsets without and with it, us: 6 views of 128 x 128: 384 tiles 26.4
// and 28.6, 672 36.1 and 32.8, 5,952 175 and 121; of 64 x 64: 696 tiles 34.0 and 37.6,
// 1,008 41.9 and 40.9; K = 1: 128 x 128 960 tiles 31.4 and 32.2, 1,440 39.7 and 39.0; 75 x
// 53: 1,392 tiles 58.9 and 61.7, 1,992 82.0 and 81.4, K = 1 3,000 83.3 and 88.2, 6,000 156
// and 158; 16 x 16: 6 views 6,000 tiles 95.7 and 117, 24 views 696 tiles 50.3 and 45.6.
static bool depth_test_pays(const geocache_corr& c, long long tiles) {
    const int HW = c.H * c.W;
    if (HW < GEOCACHE_TILE_TOKENS && !(c.N >= 24 && c.K == 4)) return false;
    return tiles >= (HW % 16 == 0 ? 700 : 1700) * (c.K == 4 ? 1 : 2);
}

cudaError_t launch_build_corr(const geocache_corr& c, cudaStream_t s) {
    const int HW = c.H * c.W, T = tiles_per_view(c.H, c.W);
    const long long tiles = (long long)T * c.N * c.B;
    const long long nb = (long long)depth_blocks(c.H) * depth_blocks(c.W);
    // the depths of a view fit its diagonal row (with 3 bytes to align them)
    if (!c.idx && c.keep && depth_test_pays(c, tiles) && 4 * nb + 3 <= HW) {
        const long long strips = (long long)((depth_blocks(c.W) + 3) / 4) * depth_blocks(c.H);
        source_depth_kernel<<<dim3((unsigned)((strips + 7) / 8), c.N, c.B), 256, 0, s>>>(c.pos, c.valid, c.cams, c.tau, c.N,
                                                                                   c.H, c.W, c.keep);
        if (c.K == 4)
            build_keep_kernel<4><<<dim3(T, c.N, c.B), kBuildThreads, 0, s>>>(c.pos, c.valid, c.cams, c.tau, c.N, c.H,
                                                                             c.W, c.keep, c.tile_ptr);
        else
            build_keep_kernel<1><<<dim3(T, c.N, c.B), kBuildThreads, 0, s>>>(c.pos, c.valid, c.cams, c.tau, c.N, c.H,
                                                                             c.W, c.keep, c.tile_ptr);
        const int chunks = HW / 16 + 2;  // of a row that starts anywhere in a 16-byte word (clear_chunk)
        clear_diagonal_kernel<<<dim3((unsigned)((chunks + 255) / 256), c.N, c.B), 256, 0, s>>>(c.keep, c.N, HW);
        note_launches(3);
        return cudaGetLastError();
    }
    int32_t* cnt = nullptr;
    if (c.tile_ptr) {
        const size_t n = (size_t)c.B * c.N * c.N * T + 1;
        cudaError_t e = cudaMemsetAsync(c.tile_ptr, 0, n * sizeof(int32_t), s);
        if (e != cudaSuccess) return e;
        cnt = c.tile_ptr;
    }
    if (!c.idx)
        c.K == 4 ? launch_build_corr_rep<4, false, 1>(c, cnt, s) : launch_build_corr_rep<1, false, 1>(c, cnt, s);
    else if (tiles >= 4096)  // 4 slices per CTA once the build has at least 4096 CTAs of 1024 tokens
        c.K == 4 ? launch_build_corr_rep<4, true, 4>(c, cnt, s) : launch_build_corr_rep<1, true, 4>(c, cnt, s);
    else
        c.K == 4 ? launch_build_corr_rep<4, true, 1>(c, cnt, s) : launch_build_corr_rep<1, true, 1>(c, cnt, s);
    return cudaGetLastError();
}

// Device status word (the library's only device-resident state): bit 0 = a
// bounded wait gave up, bit 1 = the sparse form did not fit max_records,
// bit 2 = a record permutation entry was out of range, bit 4 = a table index
// was outside [-1, H*W) (bit 3 is the rasteriser's word's bad face index).
// Read and cleared by geocache_device_status().
__device__ unsigned int g_device_error = 0;

// ---------------------------------------------------- sparse operator --
// G_{u->v} in tile-CSR form: for each (asset b, target view v, source view u,
// tile of GEOCACHE_TILE_TOKENS tokens) the records of its kept rows, in token
// order; tile_ptr holds the exclusive prefix sum of the per-tile counts.
__device__ __forceinline__ int tiles_per_view_dev(int H, int W) {
    return (H * W + GEOCACHE_TILE_TOKENS - 1) / GEOCACHE_TILE_TOKENS;
}

// In-place exclusive prefix sum of n counts by one cluster of CTAs; a[n] =
// total, or -1 when the total does not fit an int32.  Rounds of (cluster
// size x 1024 x kScanPer) consecutive counts: each thread loads its kScanPer
// counts (16-byte loads when aligned), each CTA scans its threads' sums, the
// CTAs add the sums of those before them (through distributed shared memory)
// and each thread rewrites its counts as offsets from the running total of
// the earlier rounds.  Bound by the latency of a round (load, two barriers,
// store), so the 8 CTAs take 131,072 counts in one round where one took
// 16,384: 36,864 counts (64 assets x 6 views at 128 x 128) 10.9 -> 6.7 us.
constexpr int kScanPer = 16;
constexpr int kScanCtas = 8;

template <int CTAS>
__global__ void __launch_bounds__(1024) exclusive_scan_kernel(int32_t* a, long long n) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = CTAS > 1 ? (int)cluster.block_rank() : 0;
    __shared__ long long s_warp[32];
    __shared__ long long s_total[2];  // this CTA's sum, by parity of the round
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool vec = (reinterpret_cast<uintptr_t>(a) & 15) == 0;
    long long carry = 0;  // sum of the counts of the earlier rounds
    int par = 0;
    for (long long c0 = 0; c0 < n; c0 += 1024LL * kScanPer * CTAS, par ^= 1) {
        const long long lo = c0 + ((long long)rank * 1024 + t) * kScanPer;
        int x[kScanPer];
        if (vec && lo + kScanPer <= n) {
#pragma unroll
            for (int i = 0; i < kScanPer; i += 4) {
                const int4 q = *reinterpret_cast<const int4*>(a + lo + i);
                x[i] = q.x; x[i + 1] = q.y; x[i + 2] = q.z; x[i + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < kScanPer; ++i) x[i] = lo + i < n ? a[lo + i] : 0;
        }
        long long sum = 0;
#pragma unroll
        for (int i = 0; i < kScanPer; ++i) sum += x[i];
        long long incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            long long w = s_warp[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += y;
            }
            s_warp[lane] = w;
            if (lane == 31) s_total[par] = w;
        }
        long long before = 0, round = 0;
        if (CTAS > 1) {
            cluster.sync();  // every CTA's sum is in its shared memory
#pragma unroll
            for (int r = 0; r < CTAS; ++r) {
                const long long y = *cluster.map_shared_rank(s_total + par, r);
                before += r < rank ? y : 0;
                round += y;
            }
        } else {
            __syncthreads();
            round = s_total[par];
        }
        long long run = carry + before + (warp ? s_warp[warp - 1] : 0) + incl - sum;
#pragma unroll
        for (int i = 0; i < kScanPer; ++i) {  // counts -> offsets
            const int c = x[i];
            x[i] = run > 0x7fffffffLL ? -1 : (int32_t)run;
            run += c;
        }
        if (vec && lo + kScanPer <= n) {
#pragma unroll
            for (int i = 0; i < kScanPer; i += 4)
                *reinterpret_cast<int4*>(a + lo + i) = make_int4(x[i], x[i + 1], x[i + 2], x[i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < kScanPer; ++i)
                if (lo + i < n) a[lo + i] = x[i];
        }
        carry += round;
        __syncthreads();  // s_warp is rewritten by the next round; s_total alternates
    }
    if (CTAS > 1) cluster.sync();  // the others' shared memory stays alive until every CTA has read it
    if (rank == 0 && t == 0) {
        a[n] = carry > 0x7fffffffLL ? -1 : (int32_t)carry;
        if (carry > 0x7fffffffLL) atomicOr(&g_device_error, 2u);  // more records than int32 offsets index
    }
}

static cudaError_t launch_scan(int32_t* a, long long n, cudaStream_t s) {
    note_launches(1);
    if (n <= 1024LL * kScanPer) {  // one round of one CTA, whose barrier is cheaper than the cluster's
        exclusive_scan_kernel<1><<<1, 1024, 0, s>>>(a, n);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kScanCtas);
    cfg.blockDim = dim3(1024);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kScanCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, exclusive_scan_kernel<kScanCtas>, a, n);
}

// tile_ptr holds the per-tile counts written by build_corr_kernel; turn them
// into offsets
cudaError_t launch_tile_ptr(const geocache_corr& c, cudaStream_t s) {
    const int T = tiles_per_view(c.H, c.W);
    return launch_scan(c.tile_ptr, (long long)c.B * c.N * c.N * T, s);
}

// Records of one (b, v, u, tile): kept rows in token order, each with its
// footprint's top-left tap and fractions (recomputed with the same device
// functions as the tables, so the taps and weights they give are identical).
// The tile's offsets and keep masks are loaded together, and the kept
// targets' positions are in flight while the CTA scans its counts; the kept
// rows are then compacted (with their positions) in shared memory, so that
// each thread forms about the same number of footprints (one thread per
// quad with 0 to 4 kept rows left most lanes idle: 464 -> 427 us for the
// build graph of 128 assets).  Eight
// resident CTAs per SM (32 registers, a few spilled) hide more of that
// latency than the unbounded 43-register build (build graph of 128 assets:
// 620 vs 641 us).
template <int K>
__global__ void __launch_bounds__(256, 8) fill_records_cta_kernel(const float* __restrict__ pos,
                                                           const geocache_camera* __restrict__ cams,
                                                           const uint8_t* __restrict__ keep,
                                                           const int32_t* __restrict__ tile_ptr, int N, int H,
                                                           int W, int T, geocache_tap_record* __restrict__ rec,
                                                           long long max_records) {
    // blockIdx.y runs over the N (N - 1) off-diagonal pairs (diagonal pairs
    // have no records): v = y / (N - 1), and u the (y mod (N - 1))-th view
    // other than v
    const int tile = blockIdx.x, b = blockIdx.z;
    const int v = (int)blockIdx.y / (N - 1), up = (int)blockIdx.y - v * (N - 1);
    const int u = up + (up >= v);
    const int vu = v * N + u;
    const int HW = H * W;
    const int t = threadIdx.x;
    const size_t ti = ((size_t)b * N * N + vu) * T + tile;
    const int r_first = __ldg(tile_ptr + ti), r_next = __ldg(tile_ptr + ti + 1);
    const int p0 = tile * GEOCACHE_TILE_TOKENS + 4 * t;
    const uint8_t* row = keep + ((size_t)b * N * N + vu) * HW;
    uint32_t m4 = 0;  // keep masks of tokens p0 .. p0 + 3, one byte each
    if (p0 + 3 < HW && (reinterpret_cast<uintptr_t>(row + p0) & 3) == 0) {
        m4 = __ldg(reinterpret_cast<const uint32_t*>(row + p0));
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (p0 + i < HW) m4 |= (uint32_t)__ldg(row + p0 + i) << (8 * i);
    }
    // a tile without records has nothing to write; < 0: offsets overflowed (flagged by the scan)
    if (r_next == r_first || r_first < 0) return;
    __shared__ geocache_camera s_cam;
    __shared__ int s_warp[8];
    __shared__ int s_kept[GEOCACHE_TILE_TOKENS];
    __shared__ float s_X[GEOCACHE_TILE_TOKENS][3];
    if (t < 16) reinterpret_cast<float*>(&s_cam)[t] = __ldg(reinterpret_cast<const float*>(cams + (size_t)b * N + u) + t);
    const size_t tv0 = ((size_t)b * N + v) * HW;
    float X[4][3];
    int mine = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        X[i][0] = X[i][1] = X[i][2] = 0.0f;
        if ((m4 >> (8 * i)) & 0xffu) {
            const float* q = pos + 3 * (tv0 + p0 + i);
            X[i][0] = __ldg(q);
            X[i][1] = __ldg(q + 1);
            X[i][2] = __ldg(q + 2);
            ++mine;
        }
    }
    // exclusive scan over the CTA (token order)
    const int lane = t & 31, warp = t >> 5;
    int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int base = 0, n_kept = 0;
    for (int w = 0; w < 8; ++w) {
        base += w < warp ? s_warp[w] : 0;
        n_kept += s_warp[w];
    }
    // the kept rows, compacted in token order (= record order) with their
    // target positions, so that the footprints spread evenly over the threads
    int k = base + incl - mine;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t m = (m4 >> (8 * i)) & 0xffu;
        if (!m) continue;
        s_kept[k] = (p0 + i) | (int)(m << 28);
        s_X[k][0] = X[i][0];
        s_X[k][1] = X[i][1];
        s_X[k][2] = X[i][2];
        ++k;
    }
    __syncthreads();
    for (int j = t; j < n_kept; j += 256) {
        const int tm = s_kept[j];
        Footprint f;
        footprint<K>(s_cam, s_X[j][0], s_X[j][1], s_X[j][2], H, W, f);
        geocache_tap_record out;
        out.token_mask = tm;
        out.q_tl = f.j0 * W + f.i0;
        out.fx = K == 4 ? f.ax[1] : 0.0f;
        out.fy = K == 4 ? f.ay[1] : 0.0f;
        const long long r = (long long)r_first + j;
        if (r < max_records)
            reinterpret_cast<int4*>(rec)[r] = *reinterpret_cast<const int4*>(&out);
        else
            atomicOr(&g_device_error, 2u);  // records beyond the capacity are dropped
    }
}

// The same for large builds, with one warp per tile: it reads the tile's masks
// 4 tokens per lane and round, appends the kept ones (ranked by ballots) to a
// list in shared memory and forms the records of a round (at most 128) with
// their positions in flight together.  A tile without records costs a few
// instructions, and no footprint runs in a partly filled warp but a tile's
// last: what a round leaves below 32 waits for the next.
//
// 64 assets x 6 views at 128 x 128 (30,720 tiles of a pair): 48 -> 33.5 us.
// The CTA per tile had 79% of its issue slots busy with the tiles' set-up (44 M
// instructions against 18 M here); what bounds this one is the memory
// latency of the dense tiles' rounds (42% of the slots busy), so small builds,
// whose tiles all fit on the GPU at once, keep the CTA per tile: 480 tiles
// 2.9 against 5.6 us, 7,680 tiles 14.2 against 16.2, 8,448 tiles (12 views)
// 17.6 against 16.3.
constexpr long long kFillWarpTiles = 8192;
constexpr int kFillWarps = 4;  // per CTA: a CTA stays resident until its densest tile is done (8: 4 us slower)
constexpr int kFillAhead = 4;  // positions in flight per lane

template <int K>
__global__ void __launch_bounds__(32 * kFillWarps) fill_records_kernel(const float* __restrict__ pos,
                                                           const geocache_camera* __restrict__ cams,
                                                           const uint8_t* __restrict__ keep,
                                                           const int32_t* __restrict__ tile_ptr, int N, int H,
                                                           int W, int T, geocache_tap_record* __restrict__ rec,
                                                           long long max_records) {
    constexpr int kRounds = GEOCACHE_TILE_TOKENS / 128;
    __shared__ int s_list[kFillWarps][160];
    __shared__ uint32_t s_mask[kFillWarps][kRounds][32];  // masks of tokens 128 k + 4 lane .. + 3, one byte each
    __shared__ geocache_camera s_cam[kFillWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the asset's warps run over the tiles of its N (N - 1) off-diagonal pairs
    // (diagonal pairs have no records): pair y has v = y / (N - 1), and u the
    // (y mod (N - 1))-th view other than v
    const int i_tile = (int)(blockIdx.x * kFillWarps + warp), b = blockIdx.y, y = i_tile / T;
    if (y >= N * (N - 1)) return;
    const int tile = i_tile - y * T, v = y / (N - 1), up = y - v * (N - 1);
    const int u = up + (up >= v);
    const int HW = H * W;
    const size_t vu = (size_t)b * N * N + v * N + u;
    const int r_first = __ldg(tile_ptr + vu * T + tile), r_next = __ldg(tile_ptr + vu * T + tile + 1);
    // a tile without records has nothing to write; < 0: offsets overflowed (flagged by the scan)
    if (r_next == r_first || r_first < 0) return;
    const int p_base = tile * GEOCACHE_TILE_TOKENS;
    const uint8_t* row = keep + vu * HW + p_base;
    const bool words = (reinterpret_cast<uintptr_t>(row) & 3) == 0;
#pragma unroll
    for (int k = 0; k < kRounds; ++k) {
        const int i = 128 * k + 4 * lane;
        uint32_t m = 0;
        if (words && p_base + i + 3 < HW) {
            m = __ldg(reinterpret_cast<const uint32_t*>(row + i));
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (p_base + i + e < HW) m |= (uint32_t)__ldg(row + i + e) << (8 * e);
        }
        s_mask[warp][k][lane] = m;
    }
    if (lane < 16)
        reinterpret_cast<float*>(s_cam + warp)[lane] = __ldg(reinterpret_cast<const float*>(cams + (size_t)b * N + u) + lane);
    int* list = s_list[warp];
    const float* pos_v = pos + 3 * ((size_t)b * N + v) * HW;
    const uint32_t below = (1u << lane) - 1u;
    long long r = r_first;  // record of list[0]
    int listed = 0;
#pragma unroll 1
    for (int k = 0; k < kRounds; ++k) {
        const uint32_t m = s_mask[warp][k][lane];
        const bool last = k == kRounds - 1;
        if (!__any_sync(0xffffffffu, m) && !last) continue;
        int at = listed;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t kept = __ballot_sync(0xffffffffu, (m >> (8 * e)) & 0xffu);
            at += __popc(kept & below);
            listed += __popc(kept);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t mask = (m >> (8 * e)) & 0xffu;
            if (mask) list[at++] = (p_base + 128 * k + 4 * lane + e) | (int)(mask << 28);
        }
        __syncwarp();
        const int n = last ? listed : listed & ~31;
#pragma unroll 1
        for (int j0 = 0; j0 < n; j0 += 32 * kFillAhead) {
            int tm[kFillAhead];
            float X[kFillAhead][3];
#pragma unroll
            for (int g = 0; g < kFillAhead; ++g) {
                const int j = j0 + 32 * g + lane;
                tm[g] = list[j < n ? j : 0];
                const float* x = pos_v + 3 * (size_t)(tm[g] & 0x0fffffff);
#pragma unroll
                for (int c = 0; c < 3; ++c) X[g][c] = j < n ? __ldg(x + c) : 0.0f;
            }
#pragma unroll
            for (int g = 0; g < kFillAhead; ++g) {
                const int j = j0 + 32 * g + lane;
                if (j >= n) break;
                Footprint f;
                footprint<K>(s_cam[warp], X[g][0], X[g][1], X[g][2], H, W, f);
                if (r + j < max_records)
                    reinterpret_cast<int4*>(rec)[r + j] =
                        make_int4(tm[g], f.j0 * W + f.i0, __float_as_int(K == 4 ? f.ax[1] : 0.0f),
                                  __float_as_int(K == 4 ? f.ay[1] : 0.0f));
                else
                    atomicOr(&g_device_error, 2u);  // records beyond the capacity are dropped
            }
        }
        int rest = 0;
        if (n + lane < listed) rest = list[n + lane];
        __syncwarp();
        if (n + lane < listed) list[lane] = rest;
        r += n;
        listed -= n;
    }
}

template <int K>
static void launch_fill_records_k(const geocache_corr& c, cudaStream_t s) {
    const int T = tiles_per_view(c.H, c.W);
    const long long tiles = (long long)T * c.N * (c.N - 1);  // per asset
    note_launches(1);
    if (tiles * c.B >= kFillWarpTiles)
        fill_records_kernel<K><<<dim3((unsigned)((tiles + kFillWarps - 1) / kFillWarps), c.B), 32 * kFillWarps, 0, s>>>(
            c.pos, c.cams, c.keep, c.tile_ptr, c.N, c.H, c.W, T, c.records, c.max_records);
    else
        fill_records_cta_kernel<K><<<dim3(T, c.N * (c.N - 1), c.B), 256, 0, s>>>(
            c.pos, c.cams, c.keep, c.tile_ptr, c.N, c.H, c.W, T, c.records, c.max_records);
}

cudaError_t launch_fill_records(const geocache_corr& c, cudaStream_t s) {
    if (c.K == 4) launch_fill_records_k<4>(c, s);
    else launch_fill_records_k<1>(c, s);
    return cudaGetLastError();
}

// Source index of the sparse form: the records grouped by (asset b, source
// view u, source tile st), st = the tile of the record's first kept tap, so
// that a step can apply the records per source tile with the anchor's tile
// staged in shared memory.  Entries are (record index, target view).  Two
// passes over the records: a count per group, then (after the exclusive scan
// of the counts into src_ptr) a scatter that advances src_ptr[g] by one per
// entry, which leaves src_ptr[g] = the end of group g (its start is
// src_ptr[g - 1], 0 for g = 0).  The order within a group is that of the
// atomics; nothing depends on it (each record's increment is computed on its
// own).
template <int K>
__device__ __forceinline__ int first_kept_tap(int mask, int q_tl, int W) {
    if (K == 1) return q_tl;
    const int k = __ffs(mask) - 1;  // the lowest kept tap: TL, TR, BL, BR
    return q_tl + (k & 1) + (k >> 1) * W;
}

template <int K, bool SCATTER>
__global__ void __launch_bounds__(256) src_index_kernel(const int32_t* __restrict__ tile_ptr,
                                                        const geocache_tap_record* __restrict__ rec,
                                                        long long max_records, int N, int W, int T,
                                                        int32_t* __restrict__ src_ptr, int2* __restrict__ src_rec) {
    const int tile = blockIdx.x, vu = blockIdx.y, b = blockIdx.z;
    const int v = vu / N, u = vu % N;
    if (u == v) return;
    const size_t ti = ((size_t)b * N * N + vu) * T + tile;
    const long long x0 = __ldg(tile_ptr + ti), x1 = __ldg(tile_ptr + ti + 1);
    const int r0 = (int)(x0 < 0 ? 0 : (x0 < max_records ? x0 : max_records));
    const int r1 = (int)(x1 < 0 ? 0 : (x1 < max_records ? x1 : max_records));
    for (int r = r0 + threadIdx.x; r < r1; r += 256) {
        const int4 x = __ldg(reinterpret_cast<const int4*>(rec) + r);
        const int q = first_kept_tap<K>((int)((uint32_t)x.x >> 28), x.y, W);
        const size_t g = ((size_t)b * N + u) * T + q / GEOCACHE_TILE_TOKENS;
        if (!SCATTER) atomicAdd(src_ptr + g, 1);
        else src_rec[atomicAdd(src_ptr + g, 1)] = make_int2(r, v);
    }
}

cudaError_t launch_src_index(const geocache_corr& c, cudaStream_t s) {
    const int T = tiles_per_view(c.H, c.W);
    const long long groups = (long long)c.B * c.N * T;
    cudaError_t e = cudaMemsetAsync(c.src_ptr, 0, (groups + 1) * sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    const dim3 grid(T, c.N * c.N, c.B);
    int2* out = reinterpret_cast<int2*>(c.src_rec);
    note_launches(2);  // the counts and the scatter
    if (c.K == 4)
        src_index_kernel<4, false><<<grid, 256, 0, s>>>(c.tile_ptr, c.records, c.max_records, c.N, c.W, T, c.src_ptr, out);
    else
        src_index_kernel<1, false><<<grid, 256, 0, s>>>(c.tile_ptr, c.records, c.max_records, c.N, c.W, T, c.src_ptr, out);
    e = launch_scan(c.src_ptr, groups, s);
    if (e != cudaSuccess) return e;
    if (c.K == 4)
        src_index_kernel<4, true><<<grid, 256, 0, s>>>(c.tile_ptr, c.records, c.max_records, c.N, c.W, T, c.src_ptr, out);
    else
        src_index_kernel<1, true><<<grid, 256, 0, s>>>(c.tile_ptr, c.records, c.max_records, c.N, c.W, T, c.src_ptr, out);
    return cudaGetLastError();
}

// ------------------------------------------------- fused transport step --
// MASK, TABLE and GEOMETRY steps in one kernel each: a CTA streams the rows of
// its tokens (x0: the anchor's fresh x0, or x0(t-1); x_t), for views outside the
// anchor set adds to each covered token the mean over the covering anchors of
// the tap-weighted anchor increments (Eq. 1 with the multi-anchor aggregation
// of Sec. 3.2; uncovered tokens keep x0(t-1)), and stores x0(t) and the sampler
// reconstruction of every token.
// Taps come from the keep masks (MASK: projection and weights recomputed only
// for covered (token, anchor) pairs), from the full per-tap tests (GEOMETRY) or
// from the tables (TABLE); all three are bit-identical.  Rows that only stream
// use evict-first hints so that the anchors' rows, which the gathers re-read,
// stay in L2.
constexpr int kThreads = 256;

template <typename T>
struct Lat4;
template <>
struct Lat4<float> {
    using Raw = float4;
    __device__ static Raw load_raw(const float* p, size_t e, int cnt, bool vec) {
        if (vec) return __ldcs(reinterpret_cast<const float4*>(p + e));
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (cnt > 0) r.x = __ldcs(p + e);
        if (cnt > 1) r.y = __ldcs(p + e + 1);
        if (cnt > 2) r.z = __ldcs(p + e + 2);
        if (cnt > 3) r.w = __ldcs(p + e + 3);
        return r;
    }
    __device__ static void unpack(const Raw& x, float (&r)[4]) { r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w; }
    __device__ static void load(const float* p, size_t e, int cnt, bool vec, float (&r)[4]) {
        if (vec) {
            const float4 x = __ldcs(reinterpret_cast<const float4*>(p + e));
            r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) r[i] = i < cnt ? __ldcs(p + e + i) : 0.0f;
        }
    }
    __device__ static void store(float* p, size_t e, int cnt, bool vec, const float (&r)[4]) {
        if (vec) {
            __stcs(reinterpret_cast<float4*>(p + e), make_float4(r[0], r[1], r[2], r[3]));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < cnt) __stcs(p + e + i, r[i]);
        }
    }
};
template <>
struct Lat4<__nv_bfloat16> {
    using Raw = uint2;
    __device__ static Raw load_raw(const __nv_bfloat16* p, size_t e, int cnt, bool vec) {
        if (vec) return __ldcs(reinterpret_cast<const uint2*>(p + e));
        const unsigned short* q = reinterpret_cast<const unsigned short*>(p + e);
        uint32_t h[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < cnt) h[i] = q[i];
        return make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
    }
    __device__ static void unpack(const Raw& x, float (&r)[4]) {
        r[0] = __uint_as_float(x.x << 16);
        r[1] = __uint_as_float(x.x & 0xffff0000u);
        r[2] = __uint_as_float(x.y << 16);
        r[3] = __uint_as_float(x.y & 0xffff0000u);
    }
    __device__ static void load(const __nv_bfloat16* p, size_t e, int cnt, bool vec, float (&r)[4]) {
        if (vec) {
            const uint2 x = __ldcs(reinterpret_cast<const uint2*>(p + e));
            const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&x.x);
            const __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162*>(&x.y);
            r[0] = __low2float(lo); r[1] = __high2float(lo); r[2] = __low2float(hi); r[3] = __high2float(hi);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) r[i] = i < cnt ? __bfloat162float(p[e + i]) : 0.0f;
        }
    }
    __device__ static void store(__nv_bfloat16* p, size_t e, int cnt, bool vec, const float (&r)[4]) {
        if (vec) {
            __nv_bfloat162 lo = __floats2bfloat162_rn(r[0], r[1]);
            __nv_bfloat162 hi = __floats2bfloat162_rn(r[2], r[3]);
            uint2 x;
            x.x = *reinterpret_cast<uint32_t*>(&lo);
            x.y = *reinterpret_cast<uint32_t*>(&hi);
            __stcs(reinterpret_cast<uint2*>(p + e), x);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < cnt) p[e + i] = __float2bfloat16_rn(r[i]);
        }
    }
};

// Eight consecutive elements: 32-byte accesses of f32 (sm_100 and later) and 16-byte ones of bf16, not kept
// in the L1
__device__ __forceinline__ void load8(const float* p, float (&r)[8]) {
    asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "l"(p));
}
__device__ __forceinline__ void store8(float* p, const float (&r)[8]) {
    asm volatile("st.global.L1::no_allocate.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(r[0]), "f"(r[1]),
                 "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7])
                 : "memory");
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&r)[8]) {
    const uint4 x = __ldcs(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        r[2 * i] = __uint_as_float(w[i] << 16);
        r[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&r)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(r[2 * i], r[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    __stcs(reinterpret_cast<uint4*>(p), make_uint4(w[0], w[1], w[2], w[3]));
}

// the anchors' rows stay cached (they are re-read by the gathers)
__device__ __forceinline__ void f4_load_keep(const float* p, size_t e, int cnt, bool vec, float (&r)[4]) {
    if (vec) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(p + e));
        r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) r[i] = i < cnt ? __ldg(p + e + i) : 0.0f;
    }
}

// Keep masks of the quad's tokens for source view u, one byte per token.
__device__ __forceinline__ uint32_t quad_masks(const uint8_t* row, int cnt, bool vec) {
    if (vec) return __ldg(reinterpret_cast<const uint32_t*>(row));
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (i < cnt) m |= (uint32_t)__ldg(row + i) << (8 * i);
    return m;
}

// Large MASK steps, and large TABLE and GEOMETRY steps with one anchor (see
// launch_tiles): a persistent kernel whose CTAs loop over work units
// (asset b, view v, tile of kTileTokens tokens, group of 4 channels).
//  * Streaming: one thread arms the unit's mbarrier and issues TMA bulk
//    copies (cp.async.bulk) of the unit's rows of x0 (the anchor's fresh x0,
//    or x0(t-1)) and of x_t into a two-stage shared-memory ring, one unit
//    ahead, so the next unit's rows are in flight while the current unit's
//    increments are formed.
//  * Increments (views outside the anchor set): the (token, anchor) pairs
//    with a kept tap (MASK; in the other modes every candidate pair) are
//    compacted into a work list (block prefix sum, token order) and processed one
//    per thread, so the dependent loads of many tokens overlap (MASK: keep masks
//    -> target position -> projection and weights -> gathers of the anchor
//    increments x0_new - x0(t-1) at the kept taps).  Per-anchor sums are
//    combined in anchor order (Eq. 1 with the multi-anchor aggregation of Sec.
//    3.2: the mean over covering anchors; a token without a kept tap keeps
//    x0(t-1)).
//  * Every token is stored (x0(t)) and reconstructed (x_{t-1}) from the
//    staged rows with 16-byte stores.
constexpr int kTileTokens = 4 * kThreads;
static_assert(kTileTokens == GEOCACHE_TILE_TOKENS, "tile of the sparse form");
constexpr int kChunk = 4;                        // anchors per work-list round
constexpr int kPairCap = kChunk * kTileTokens;   // (token, anchor) work items of one round
constexpr int kStages = 2;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // default limit of a bounded mbarrier wait: 2 s

// Test hook of the failure handling (geocache_debug_set_wait): the limit of
// the bounded waits, and a one-shot request that the next staged transport
// launch arm none of its first unit's copies, so that wait runs out.
static std::atomic<unsigned long long> g_wait_limit_ns{kWaitLimitNs};
static std::atomic<int> g_drop_first_copy{0};

void set_debug_wait(unsigned long long limit_ns, int drop_first_copy) {
    g_wait_limit_ns.store(limit_ns ? limit_ns : kWaitLimitNs);
    g_drop_first_copy.store(drop_first_copy ? 1 : 0);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Wait for the phase with the given parity; false after limit_ns.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, unsigned long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    while (!mbar_try_wait(bar, parity))
        if (globaltimer() - t0 > limit_ns) return false;
    return true;
}

// exclusive prefix sum over the CTA (deterministic); returns the total
__device__ __forceinline__ int block_exclusive_scan(int x, int& total, int* s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < kThreads / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        if (lane < kThreads / 32) s_warp[lane] = w;  // inclusive warp totals
    }
    __syncthreads();
    total = s_warp[kThreads / 32 - 1];
    const int base = warp ? s_warp[warp - 1] : 0;
    return base + incl - x;
}

struct FusedShared {
    float acc[kTileTokens][4];        // per token: sum over covering anchors (anchor order), channel group
    uint32_t pair[kPairCap];          // work items: token | anchor << 10 | keep mask << 16
    uint8_t n[kTileTokens];           // per token: number of covering anchors
    geocache_camera cam[kChunk];
    int warp[kThreads / 32];
    uint64_t bar[kStages];
};

// Taps of work item (token p of view v, anchor slot s2) in the given mode.
template <int K, int MODE>
__device__ __forceinline__ void item_taps(const TransportArgs& args, const geocache_camera& cam, int b, int v,
                                          int s2, int p, int m, size_t tv0, size_t plane, float tau2, Taps& tp) {
    const int N = args.N;
    const int u = args.anchors[s2];
    if (MODE == GEOCACHE_CORR_TABLE) {
        const size_t row = (((size_t)b * N + v) * N + u) * plane + p;
        tp.kept = 0;
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
            int q = __ldca(args.idx + row * K + kk);
            float wq = __ldca(args.w + row * K + kk);
            if (q < -1 || q >= (int)plane) {  // a caller's table with an index outside the view: dropped, reported
                atomicOr(&g_device_error, 16u);
                q = -1;
                wq = 0.0f;
            }
            tp.q[kk] = q;
            tp.w[kk] = wq;
            tp.kept += q >= 0;
        }
        return;
    }
    const float X0 = __ldca(args.pos + 3 * (tv0 + p));
    const float X1 = __ldca(args.pos + 3 * (tv0 + p) + 1);
    const float X2 = __ldca(args.pos + 3 * (tv0 + p) + 2);
    if (MODE == GEOCACHE_CORR_MASK) {
        Footprint f;
        footprint<K>(cam, X0, X1, X2, args.H, args.W, f);
        taps_from_mask<K>(f, m, args.W, tp);
    } else {
        const size_t su = ((size_t)b * N + u) * plane;
        compute_taps<K>(cam, args.pos + 3 * su, args.valid + su, args.H, args.W, X0, X1, X2, tau2, tp);
    }
}

// Tap-weighted increment of one anchor at one token, channels [cg, cg+cn).
template <int K>
__device__ __forceinline__ void item_increment(const TransportArgs& args, const Taps& tp, int b, int s2, int cg,
                                               int cn, size_t plane, float (&g)[4]) {
    const int N = args.N, C = args.C, a = args.a;
    const float* xn = args.x0_new + (((size_t)b * a + s2) * C + cg) * plane;
    const float* xp = args.x0_prev + (((size_t)b * N + args.anchors[s2]) * C + cg) * plane;
    const bool copy = args.update == GEOCACHE_UPDATE_COPY;
    float dn[K][4], dp[K][4];
#pragma unroll
    for (int kk = 0; kk < K; ++kk)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            dn[kk][c] = 0.0f;
            dp[kk][c] = 0.0f;
            if (tp.q[kk] >= 0 && c < cn) {
                const size_t e = (size_t)c * plane + tp.q[kk];
                dn[kk][c] = __ldca(xn + e);
                dp[kk][c] = __ldca(xp + e);
            }
        }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float acc = 0.0f;
#pragma unroll
        for (int kk = 0; kk < K; ++kk)
            if (tp.q[kk] >= 0) acc = tap_term(copy, tp.w[kk], dn[kk][c], dp[kk][c], acc);
        g[c] = acc;
    }
}

struct UnitCoord {
    int b, v, tile, cg;
};

__device__ __forceinline__ UnitCoord unit_coord(long long u, int n_tiles, int n_cg, int N) {
    UnitCoord c;
    c.cg = (int)(u % n_cg) * 4;
    u /= n_cg;
    c.tile = (int)(u % n_tiles);
    u /= n_tiles;
    c.v = (int)(u % N);
    c.b = (int)(u / N);
    return c;
}

// Increments of the tile's covered tokens (views outside the anchor set),
// left in sh.acc / sh.n for the tile's tokens.
template <int K, int MODE, bool VEC>
__device__ __forceinline__ void tile_increments(const TransportArgs& args, FusedShared& sh, int b, int v, int tile0,
                                                int cg, int cn) {
    const int HW = args.H * args.W;
    const int t = threadIdx.x;
    const int p0 = tile0 + 4 * t;
    const int cnt = p0 < HW ? (HW - p0 < 4 ? HW - p0 : 4) : 0;
    const int N = args.N, a = args.a;
    const size_t plane = (size_t)HW;
    const size_t tv0 = ((size_t)b * N + v) * plane;
    float tau2 = 0.0f;
    uint32_t fg = 0;  // GEOMETRY: validity bytes of the thread's tokens
    if (MODE == GEOCACHE_CORR_GEOMETRY) {
        const float tu = __ldg(args.tau + b);
        tau2 = __fmul_rn(tu, tu);
        if (cnt > 0) fg = quad_masks(args.valid + tv0 + p0, cnt, VEC);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float4*>(sh.acc[4 * t + i]) = make_float4(0.f, 0.f, 0.f, 0.f);
        sh.n[4 * t + i] = 0;
    }
    for (int ac = 0; ac < a; ac += kChunk) {
        const int na = a - ac < kChunk ? a - ac : kChunk;
        if (MODE != GEOCACHE_CORR_TABLE)
            for (int i = t; i < na * 16; i += kThreads)
                reinterpret_cast<float*>(sh.cam)[i] = __ldg(
                    reinterpret_cast<const float*>(args.cams + (size_t)b * N + args.anchors[ac + (i >> 4)]) + (i & 15));
        // (token, anchor) work items of this anchor chunk
        uint32_t m4[4] = {0, 0, 0, 0};  // per own token: 4 bits per anchor of the chunk
        if (cnt > 0 && MODE != GEOCACHE_CORR_MASK) {  // every anchor is a candidate of a (foreground) token
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (MODE == GEOCACHE_CORR_TABLE ? i < cnt : ((fg >> (8 * i)) & 0xffu) != 0) m4[i] = (1u << (4 * na)) - 1u;
        } else if (cnt > 0) {
            const uint8_t* krow = args.keep + ((size_t)b * N + v) * N * plane + p0;
            uint32_t q[kChunk];
#pragma unroll
            for (int s2 = 0; s2 < kChunk; ++s2)  // the chunk's masks in flight together
                q[s2] = s2 < na ? quad_masks(krow + (size_t)args.anchors[ac + s2] * plane, cnt, VEC) : 0u;
#pragma unroll
            for (int s2 = 0; s2 < kChunk; ++s2)
#pragma unroll
                for (int i = 0; i < 4; ++i) m4[i] |= ((q[s2] >> (8 * i)) & 15u) << (4 * s2);
        }
        int mine = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int s2 = 0; s2 < kChunk; ++s2) mine += (m4[i] >> (4 * s2)) & 15u ? 1 : 0;
        int n_items;
        int k = block_exclusive_scan(mine, n_items, sh.warp);  // barriers inside
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int s2 = 0; s2 < kChunk; ++s2) {
                const uint32_t m = (m4[i] >> (4 * s2)) & 15u;
                if (m) sh.pair[k++] = (uint32_t)(4 * t + i) | ((uint32_t)s2 << 10) | (m << 16);
            }
        __syncthreads();
        for (int r0 = 0; r0 < n_items; r0 += kThreads) {
            const int j = r0 + t;
            float g[4] = {0.f, 0.f, 0.f, 0.f};
            int s_mine = -1, lp = 0;
            if (j < n_items) {
                const uint32_t it = sh.pair[j];
                lp = (int)(it & 1023u);
                const int s_loc = (int)((it >> 10) & 63u);
                const int m = (int)((it >> 16) & 15u);
                Taps tp;
                item_taps<K, MODE>(args, sh.cam[s_loc], b, v, ac + s_loc, tile0 + lp, m, tv0, plane, tau2, tp);
                if (tp.kept) {
                    item_increment<K>(args, tp, b, ac + s_loc, cg, cn, plane, g);
                    s_mine = s_loc;
                }
            }
            // combine in anchor order (deterministic): anchor s_loc adds in pass s_loc
            for (int s2 = 0; s2 < na; ++s2) {
                if (s_mine == s2) {
                    float4* dst = reinterpret_cast<float4*>(sh.acc[lp]);
                    float4 cur = *dst;
                    cur.x = __fadd_rn(cur.x, g[0]);
                    cur.y = __fadd_rn(cur.y, g[1]);
                    cur.z = __fadd_rn(cur.z, g[2]);
                    cur.w = __fadd_rn(cur.w, g[3]);
                    *dst = cur;
                    sh.n[lp] += 1;
                }
                __syncthreads();
            }
        }
    }
}

template <typename T, int K, int MODE>
__global__ void __launch_bounds__(kThreads) transport_fused_kernel(const TransportArgs args, int n_tiles, int n_cg,
                                                                   long long n_units) {
    __shared__ FusedShared sh;
    extern __shared__ __align__(128) unsigned char dyn[];  // [stage]: x0 rows [4][tile] f32, x_t rows [4][tile] T
    constexpr size_t kStageBytes = 4 * kTileTokens * (sizeof(float) + sizeof(T));
    const int t = threadIdx.x;
    const int HW = args.H * args.W;
    const int N = args.N, C = args.C, a = args.a;
    const size_t plane = (size_t)HW;
    const bool recon = args.coef.enabled;
    const T* xt_p = static_cast<const T*>(args.x_t);
    T* xn_p = static_cast<T*>(args.x_next);

    // issue the bulk copies of unit u into stage st (thread 0)
    auto issue = [&](long long u, int st) {
        if (args.drop_first_copy && u == 0) return;  // test hook: this unit's wait runs out
        const UnitCoord c = unit_coord(u, n_tiles, n_cg, N);
        const int tile0 = c.tile * kTileTokens;
        const int tile_n = HW - tile0 < kTileTokens ? HW - tile0 : kTileTokens;
        const int cn = C - c.cg < 4 ? C - c.cg : 4;
        const int slot = args.slot_of[c.v];
        const float* src = slot >= 0 ? args.x0_new + ((size_t)c.b * a + slot) * C * plane
                                     : args.x0_prev + ((size_t)c.b * N + c.v) * C * plane;
        float* s_x0 = reinterpret_cast<float*>(dyn + st * kStageBytes);
        T* s_xt = reinterpret_cast<T*>(dyn + st * kStageBytes + 4 * kTileTokens * sizeof(float));
        const uint32_t rx = (uint32_t)tile_n * sizeof(float), rt = (uint32_t)tile_n * sizeof(T);
        mbar_arrive_expect_tx(&sh.bar[st], cn * (rx + (recon ? rt : 0)));
        for (int cc = 0; cc < cn; ++cc) {
            bulk_g2s(s_x0 + cc * kTileTokens, src + (size_t)(c.cg + cc) * plane + tile0, rx, &sh.bar[st]);
            if (recon)
                bulk_g2s(s_xt + cc * kTileTokens, xt_p + (((size_t)c.b * N + c.v) * C + c.cg + cc) * plane + tile0, rt,
                         &sh.bar[st]);
        }
    };

    if (t == 0) {
        for (int st = 0; st < kStages; ++st) mbar_init(&sh.bar[st], 1);
        fence_mbar_init();
        if ((long long)blockIdx.x < n_units) issue(blockIdx.x, 0);
    }
    __syncthreads();
    uint32_t parity[kStages] = {0, 0};
    int st = 0;
    for (long long u = blockIdx.x; u < n_units; u += gridDim.x) {
        const long long un = u + gridDim.x;
        if (t == 0 && un < n_units) {
            fence_proxy_async();  // the previous unit's shared-memory reads of this stage come first
            issue(un, st ^ 1);
        }
        const UnitCoord c = unit_coord(u, n_tiles, n_cg, N);
        const int tile0 = c.tile * kTileTokens;
        const int p0 = tile0 + 4 * t;
        const int cnt = p0 < HW ? (HW - p0 < 4 ? HW - p0 : 4) : 0;
        const int cn = C - c.cg < 4 ? C - c.cg : 4;
        const int slot = args.slot_of[c.v];
        if (slot < 0) tile_increments<K, MODE, true>(args, sh, c.b, c.v, tile0, c.cg, cn);

        const bool ok = mbar_wait_bounded(&sh.bar[st], parity[st], args.wait_limit_ns);
        if (__syncthreads_or(!ok)) {  // the whole CTA gives up together
            if (t == 0) atomicOr(&g_device_error, 1u);
            for (int s2 = 0; s2 < kStages; ++s2)  // copies in flight
                mbar_wait_bounded(&sh.bar[s2], parity[s2], args.wait_limit_ns);
            return;
        }
        parity[st] ^= 1u;
        if (cnt > 0) {
            const float* s_x0 = reinterpret_cast<const float*>(dyn + st * kStageBytes);
            const T* s_xt = reinterpret_cast<const T*>(dyn + st * kStageBytes + 4 * kTileTokens * sizeof(float));
            const size_t view_base = ((size_t)c.b * N + c.v) * C * plane + p0;
            float x0[4][4];
            typename Lat4<T>::Raw xt[4];
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                if (cc >= cn) break;
                const float4 q = *reinterpret_cast<const float4*>(s_x0 + cc * kTileTokens + 4 * t);
                x0[cc][0] = q.x; x0[cc][1] = q.y; x0[cc][2] = q.z; x0[cc][3] = q.w;
                if (recon) xt[cc] = *reinterpret_cast<const typename Lat4<T>::Raw*>(s_xt + cc * kTileTokens + 4 * t);
            }
            if (slot < 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int n = sh.n[4 * t + i];
                    if (!n) continue;
                    const float4 g = *reinterpret_cast<const float4*>(sh.acc[4 * t + i]);
                    const float gg[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
                        x0[cc][i] = fold_one(args.update == GEOCACHE_UPDATE_COPY, x0[cc][i], gg[cc], n);
                }
            }
            if (slot < 0 || args.write_anchor_rows) {
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    if (cc >= cn) break;
                    Lat4<float>::store(args.x0_out, view_base + (size_t)(c.cg + cc) * plane, cnt, true, x0[cc]);
                }
            }
            if (recon) {
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    if (cc >= cn) break;
                    float x[4], y[4], pr[4];
                    Lat4<T>::unpack(xt[cc], x);
#pragma unroll
                    for (int i = 0; i < 4; ++i) y[i] = recon_one(args.coef, x[i], x0[cc][i], pr[i]);
                    const size_t e = view_base + (size_t)(c.cg + cc) * plane;
                    Lat4<T>::store(xn_p, e, cnt, true, y);
                    if (args.pred_out) Lat4<float>::store(args.pred_out, e, cnt, true, pr);
                }
            }
        }
        __syncthreads();  // stage st and the sums are reused by later units
        st ^= 1;
    }
}

// General path (sizes the bulk copies cannot serve: H*W not a multiple of 8
// or buffers not 16-byte aligned): one CTA per unit, registers instead of
// the shared-memory ring.
template <typename T, int K, int MODE, bool VEC>
__global__ void __launch_bounds__(kThreads) transport_simple_kernel(const TransportArgs args, int n_tiles, int n_cg) {
    __shared__ FusedShared sh;
    const int t = threadIdx.x;
    const int HW = args.H * args.W;
    const int N = args.N, C = args.C, a = args.a;
    const size_t plane = (size_t)HW;
    const bool recon = args.coef.enabled;
    const T* xt_p = static_cast<const T*>(args.x_t);
    T* xn_p = static_cast<T*>(args.x_next);
    const UnitCoord c = unit_coord(blockIdx.x, n_tiles, n_cg, N);
    const int tile0 = c.tile * kTileTokens;
    const int p0 = tile0 + 4 * t;
    const int cnt = p0 < HW ? (HW - p0 < 4 ? HW - p0 : 4) : 0;
    const int cn = C - c.cg < 4 ? C - c.cg : 4;
    const int slot = args.slot_of[c.v];
    const size_t view_base = ((size_t)c.b * N + c.v) * C * plane + p0;
    const float* src = slot >= 0 ? args.x0_new + ((size_t)c.b * a + slot) * C * plane + p0
                                 : args.x0_prev + ((size_t)c.b * N + c.v) * C * plane + p0;
    float x0[4][4];
    typename Lat4<T>::Raw xt[4];
    if (cnt > 0) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            if (cc >= cn) break;
            if (slot >= 0)
                f4_load_keep(src, (size_t)(c.cg + cc) * plane, cnt, VEC, x0[cc]);
            else
                Lat4<float>::load(src, (size_t)(c.cg + cc) * plane, cnt, VEC, x0[cc]);
            if (recon) xt[cc] = Lat4<T>::load_raw(xt_p, view_base + (size_t)(c.cg + cc) * plane, cnt, VEC);
        }
    }
    if (slot < 0) tile_increments<K, MODE, VEC>(args, sh, c.b, c.v, tile0, c.cg, cn);
    if (cnt <= 0) return;
    if (slot < 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int n = sh.n[4 * t + i];
            if (!n) continue;
            const float4 g = *reinterpret_cast<const float4*>(sh.acc[4 * t + i]);
            const float gg[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
            for (int cc = 0; cc < 4; ++cc)
                x0[cc][i] = fold_one(args.update == GEOCACHE_UPDATE_COPY, x0[cc][i], gg[cc], n);
        }
    }
    if (slot < 0 || args.write_anchor_rows) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            if (cc >= cn) break;
            Lat4<float>::store(args.x0_out, view_base + (size_t)(c.cg + cc) * plane, cnt, VEC, x0[cc]);
        }
    }
    if (recon) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            if (cc >= cn) break;
            float x[4], y[4], pr[4];
            Lat4<T>::unpack(xt[cc], x);
#pragma unroll
            for (int i = 0; i < 4; ++i) y[i] = recon_one(args.coef, x[i], x0[cc][i], pr[i]);
            const size_t e = view_base + (size_t)(c.cg + cc) * plane;
            Lat4<T>::store(xn_p, e, cnt, VEC, y);
            if (args.pred_out) Lat4<float>::store(args.pred_out, e, cnt, VEC, pr);
        }
    }
}

// Quotient by a divisor fixed for a launch, as a multiply-high and a shift
// (Granlund and Montgomery, division by invariant integers using
// multiplication): with l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1,
// n / d = (umulhi(m, n) + n) >> l for 0 <= n < 2^31.  The CTAs of a launch
// split their block index into (asset, view, tile, channel group, ...) with
// these instead of integer divisions.
struct FastDiv {
    uint32_t d, m, l;
    __device__ __forceinline__ uint32_t quo(uint32_t n) const { return (__umulhi(m, n) + n) >> l; }
};
static FastDiv make_fastdiv(uint32_t d) {
    FastDiv f{d, 0u, 0u};
    while ((1ull << f.l) < d) ++f.l;
    f.m = (uint32_t)(((1ull << 32) * ((1ull << f.l) - d)) / d + 1);
    return f;
}

// Tile offset i of the sparse form clamped to the records that exist, [0,
// cap]: a build whose records overflowed the capacity or the int32 offsets
// is flagged in the status word, and the transport then reads only records
// that exist.  (An offset beyond int32 is -1, so the tile before it may end
// before it begins: its count is taken as 0.)
__device__ __forceinline__ int record_offset(const int32_t* __restrict__ tile_ptr, size_t i, long long cap) {
    const long long x = __ldca(tile_ptr + i);
    return (int)(x < 0 ? 0 : (x < cap ? x : cap));
}

// Most TABLE and GEOMETRY steps, and MASK and SPARSE steps of few units: one CTA
// per 256 tokens of a view and group of 4 channels, one token per thread, any
// alignment.
// The two kernels above take a tile of 1024 tokens per CTA, whose work items
// (token, anchor; up to 4 per token and round of anchors) go 256 at a time
// through a chain of dependent loads with a barrier per anchor; where their
// units do not fill the GPU several times over, the chains of a covered tile
// are the time of the call.  Here the items of a CTA are a quarter as many, and
// each writes its increment to the slot of its (anchor, token), so that no
// barrier orders them: every thread then sums its token's slots in anchor
// order (the same additions).  8 assets x 6 views of 96 x 96 x 4 bf16, 3 anchors,
// against those kernels: masks 19.7 -> 12.0 us, tables (every token an item)
// 50.4 -> 19.1, geometry 48.8 -> 17.9; 64 assets: tables 215 -> 144, geometry
// 199 -> 137.
constexpr int kTokenAnchors = 4;  // anchors per round
// resident CTAs per SM: 3 (80 registers, a few spilled) or 2, whichever was
// faster: 8 assets, masks 12.0 / 12.2, geometry 17.9 / 17.9 (64 assets 137 / 155),
// tables 20.4 / 19.1, f32 masks 9.2 / 8.1 (4 assets); 4 were slower
template <typename T, int MODE>
constexpr int kTokenBlocks = MODE == GEOCACHE_CORR_TABLE || (MODE == GEOCACHE_CORR_MASK && sizeof(T) == 4) ? 2 : 3;

template <typename T, int K, int MODE>
__global__ void __launch_bounds__(kThreads, (kTokenBlocks<T, MODE>)) transport_token_kernel(const TransportArgs args, FastDiv n_cg) {
    __shared__ float4 s_g[kTokenAnchors][kThreads];     // increments of the round's (anchor, token)s
    __shared__ uint8_t s_has[kTokenAnchors][kThreads];  // whether the anchor covers the token
    __shared__ uint32_t s_item[kTokenAnchors * kThreads];  // token | anchor << 10 | keep mask << 16
    __shared__ geocache_camera s_cam[kTokenAnchors];
    __shared__ int s_wcnt[kThreads / 32];
    __shared__ int s_r0[kTokenAnchors], s_rn[kTokenAnchors];  // SPARSE: the tile's records of the round's anchors
    pdl_wait();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int HW = args.H * args.W, N = args.N, C = args.C, a = args.a;
    const size_t plane = (size_t)HW;
    const int tile = (int)n_cg.quo(blockIdx.x), cg = ((int)blockIdx.x - tile * (int)n_cg.d) * 4;
    const int v = blockIdx.y, b = blockIdx.z;
    const int p0 = tile * kThreads, p = p0 + t;
    const bool in = p < HW;
    const int cn = C - cg < 4 ? C - cg : 4;
    const int slot = args.slot_of[v];
    const bool recon = args.coef.enabled;
    const size_t base = (((size_t)b * N + v) * C + cg) * plane + p;
    const float* src = slot >= 0 ? args.x0_new + (((size_t)b * a + slot) * C + cg) * plane + p : args.x0_prev + base;
    const T* xt_p = static_cast<const T*>(args.x_t);
    float x0[4], xt[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        x0[c] = in && c < cn ? __ldca(src + (size_t)c * plane) : 0.0f;
        xt[c] = in && c < cn && recon ? lat_load(xt_p, base + (size_t)c * plane) : 0.0f;
    }
    if (slot < 0) {
        const size_t tv0 = ((size_t)b * N + v) * plane;
        float tau2 = 0.0f;
        if (MODE == GEOCACHE_CORR_GEOMETRY) {
            const float tu = __ldca(args.tau + b);
            tau2 = __fmul_rn(tu, tu);
        }
        const bool fg = in && (MODE != GEOCACHE_CORR_GEOMETRY || __ldca(args.valid + tv0 + p) != 0);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        int n = 0;
        for (int ac = 0; ac < a; ac += kTokenAnchors) {
            const int na = a - ac < kTokenAnchors ? a - ac : kTokenAnchors;
            if (MODE == GEOCACHE_CORR_SPARSE) {
                // the records of the 1024-token tile around the CTA's tokens; they are in token order, so a
                // warp's are mostly all its CTA's or all another's
                if (t < kTokenAnchors) {
                    int r0 = 0, r1 = 0;
                    if (t < na) {
                        const size_t i = (((size_t)b * N + v) * N + args.anchors[ac + t]) * tiles_per_view_dev(args.H, args.W) +
                                         p0 / kTileTokens;
                        r0 = record_offset(args.tile_ptr, i, args.max_records);
                        r1 = record_offset(args.tile_ptr, i + 1, args.max_records);
                    }
                    s_r0[t] = r0;
                    s_rn[t] = max(r1 - r0, 0);
                }
#pragma unroll
                for (int s2 = 0; s2 < kTokenAnchors; ++s2) s_has[s2][t] = 0;
                __syncthreads();
                int total = 0;
#pragma unroll
                for (int s2 = 0; s2 < kTokenAnchors; ++s2) total += s_rn[s2];
                for (int j = t; j < total; j += kThreads) {
                    int s2 = 0, jj = j;
                    while (jj >= s_rn[s2]) jj -= s_rn[s2++];
                    const int4 rec = __ldca(reinterpret_cast<const int4*>(args.records) + s_r0[s2] + jj);
                    const int lp = (rec.x & 0x0fffffff) - p0;
                    if ((unsigned)lp >= (unsigned)kThreads) continue;
                    Taps tp;
                    taps_from_record<K>((int)((uint32_t)rec.x >> 28), rec.y, __int_as_float(rec.z),
                                        __int_as_float(rec.w), args.W, tp);
                    float g[4];
                    item_increment<K>(args, tp, b, ac + s2, cg, cn, plane, g);
                    s_g[s2][lp] = make_float4(g[0], g[1], g[2], g[3]);
                    s_has[s2][lp] = 1;
                }
                __syncthreads();
            } else {
                if (MODE != GEOCACHE_CORR_TABLE && t < na * 16)
                    reinterpret_cast<float*>(s_cam)[t] = __ldca(
                        reinterpret_cast<const float*>(args.cams + (size_t)b * N + args.anchors[ac + (t >> 4)]) + (t & 15));
                // the round's candidate (anchor, token)s, listed by warp
                uint32_t m[kTokenAnchors], kept[kTokenAnchors];
                int mine = 0;
#pragma unroll
                for (int s2 = 0; s2 < kTokenAnchors; ++s2) {
                    m[s2] = 0;
                    if (s2 < na && fg)
                        m[s2] = MODE == GEOCACHE_CORR_MASK
                                    ? __ldca(args.keep + (((size_t)b * N + v) * N + args.anchors[ac + s2]) * plane + p)
                                    : 15u;
                }
#pragma unroll
                for (int s2 = 0; s2 < kTokenAnchors; ++s2) {
                    kept[s2] = __ballot_sync(0xffffffffu, m[s2] & 15u);
                    mine += __popc(kept[s2]);
                    s_has[s2][t] = 0;
                }
                if (lane == 0) s_wcnt[warp] = mine;
                __syncthreads();
                int at = 0, n_items = 0;
#pragma unroll
                for (int w = 0; w < kThreads / 32; ++w) {
                    at += w < warp ? s_wcnt[w] : 0;
                    n_items += s_wcnt[w];
                }
#pragma unroll
                for (int s2 = 0; s2 < kTokenAnchors; ++s2) {
                    if (m[s2] & 15u)
                        s_item[at + __popc(kept[s2] & ((1u << lane) - 1u))] =
                            (uint32_t)t | ((uint32_t)s2 << 10) | ((m[s2] & 15u) << 16);
                    at += __popc(kept[s2]);
                }
                __syncthreads();
                for (int j = t; j < n_items; j += kThreads) {
                    const uint32_t it = s_item[j];
                    const int lp = (int)(it & 1023u), s2 = (int)((it >> 10) & 63u);
                    Taps tp;
                    item_taps<K, MODE>(args, s_cam[s2], b, v, ac + s2, p0 + lp, (int)(it >> 16), tv0, plane, tau2, tp);
                    if (tp.kept) {
                        float g[4];
                        item_increment<K>(args, tp, b, ac + s2, cg, cn, plane, g);
                        s_g[s2][lp] = make_float4(g[0], g[1], g[2], g[3]);
                        s_has[s2][lp] = 1;
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int s2 = 0; s2 < kTokenAnchors; ++s2) {
                if (!s_has[s2][t]) continue;
                const float4 g = s_g[s2][t];
                acc[0] = __fadd_rn(acc[0], g.x);
                acc[1] = __fadd_rn(acc[1], g.y);
                acc[2] = __fadd_rn(acc[2], g.z);
                acc[3] = __fadd_rn(acc[3], g.w);
                ++n;
            }
            // the next round clears a thread's own flags and writes the slots two barriers later
        }
        if (n) {
#pragma unroll
            for (int c = 0; c < 4; ++c) x0[c] = fold_one(args.update == GEOCACHE_UPDATE_COPY, x0[c], acc[c], n);
        }
    }
    if (!in) return;
    T* xn_p = static_cast<T*>(args.x_next);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (c >= cn) break;
        const size_t e = base + (size_t)c * plane;
        if (slot < 0 || args.write_anchor_rows) args.x0_out[e] = x0[c];
        if (recon) {
            float pr;
            lat_store(xn_p, e, recon_one(args.coef, xt[c], x0[c], pr));
            if (args.pred_out) args.pred_out[e] = pr;
        }
    }
}

// Sparse mode.  A cached step is two kernels:
//  phase A: (i) the records of the step's pairs (v outside the anchor set,
//    anchor u) applied record-parallel: for each record the kept taps and
//    weights, then sum_k w_k (x0_new - x0(t-1))[q_k] for every channel,
//    written to workspace[r * C + c];  (ii) the anchor views streamed
//    (x0(t) = the denoiser's x0, reconstruction).  The two kinds of CTA are
//    interleaved in launch order so that the latency-bound gathers overlap
//    the bandwidth-bound streaming and both read the anchors' fresh x0 while
//    it is in L2.  For an in-place cache update the anchor rows are written
//    by phase B instead (the gathers read x0(t-1) of the anchors).
//  phase B: the other views streamed; each CTA folds its tile's record
//    increments in anchor order (deterministic: the mean over covering
//    anchors of Eq. 1 with the aggregation of Sec. 3.2; tokens without a
//    record keep x0(t-1)), then stores and reconstructs every token.
// Phase B becomes resident while phase A drains and reads tile_ptr and its
// streamed rows (x0(t-1), x_t) before it waits; CTAs of tiles without records
// never wait.  Phase A writes none of these, and it is launched in stream
// order, after everything before it has completed, so they are written and
// visible before either phase starts.  (Phase A launched early too, with all of
// phase B waiting: 128 assets 112.3 us against 111.1, 8 assets of 12 views x 16
// channels 77.8 against 78.3.)
// Wide latents (C >= 8) with room in the workspace take another phase A:
// the anchor views streamed while their increments are written once as a
// plane (4 channels per 16-byte word), from which phase B forms each
// record's increment itself (sparse_phase_a_plane_kernel below).  Without
// that room, phase A applies the records per source tile when the corr has
// a source index (sparse_phase_a_src_kernel), else record-parallel.

// The thread's four tokens of a tile: with VEC consecutive ones, moved by one
// vector access; without (rows that are not 16-byte aligned) ones kThreads
// apart, so that a warp's scalar accesses are consecutive (four consecutive
// tokens per thread made each of its sectors four accesses: a step of
// 60 assets x 6 views of 75 x 53 x 4 28.3 -> 22.2 us, of 30 of 75 x 53 x 16 54.0 -> 43.3).
template <bool VEC>
__device__ __forceinline__ int tile_token(int i) {
    return VEC ? 4 * (int)threadIdx.x + i : i * kThreads + (int)threadIdx.x;
}
template <typename T, bool VEC>
struct Tile4 {
    using Raw = typename Lat4<T>::Raw;
    // p: the tile's row; left: its tokens
    __device__ static __forceinline__ void load(const T* p, int left, float (&r)[4]) {
        if (VEC) {
            Lat4<T>::load(p, 4 * threadIdx.x, 4, true, r);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) r[i] = tile_token<VEC>(i) < left ? __ldcs(p + tile_token<VEC>(i)) : 0.0f;
        }
    }
    __device__ static __forceinline__ Raw load_raw(const T* p, int left) {
        if (VEC) return Lat4<T>::load_raw(p, 4 * threadIdx.x, 4, true);
        return load_apart(p, left);
    }
    __device__ static __forceinline__ float4 load_apart(const float* p, int left) {
        float r[4];
        Tile4<float, VEC>::load(p, left, r);
        return make_float4(r[0], r[1], r[2], r[3]);
    }
    __device__ static __forceinline__ uint2 load_apart(const __nv_bfloat16* p, int left) {
        const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
        uint32_t h[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = tile_token<VEC>(i) < left ? (uint32_t)q[tile_token<VEC>(i)] : 0u;
        return make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
    }
    __device__ static __forceinline__ void store(T* p, int left, const float (&r)[4]) {
        if (VEC) {
            Lat4<T>::store(p, 4 * threadIdx.x, 4, true, r);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (tile_token<VEC>(i) < left) lat_store(p, tile_token<VEC>(i), r[i]);
        }
    }
};

// Streamed rows of the thread's four tokens of a tile (of `left` tokens from
// tile0) of view v of asset b, channel group cg: x0 (the anchor's fresh x0 or
// x0(t-1)) and x_t.  Threads without a token (tile_token(0) >= left) do not call.
template <typename T, bool VEC>
struct QuadRows {
    float x0[4][4];
    typename Lat4<T>::Raw xt[4];

    __device__ __forceinline__ void load(const TransportArgs& args, int b, int v, int slot, int tile0, int left, int cg,
                                         int cn) {
        const size_t plane = (size_t)args.H * args.W;
        const int N = args.N, C = args.C, a = args.a;
        const float* x0_src = slot >= 0 ? args.x0_new + ((size_t)b * a + slot) * C * plane + tile0
                                        : args.x0_prev + ((size_t)b * N + v) * C * plane + tile0;
        const T* xt_p = static_cast<const T*>(args.x_t) + ((size_t)b * N + v) * C * plane + tile0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (c >= cn) break;
            const float* row = x0_src + (size_t)(cg + c) * plane;
            if (slot < 0) {
                Tile4<float, VEC>::load(row, left, x0[c]);
            } else if (VEC) {  // the anchors' rows stay cached for the gathers
                f4_load_keep(row, 4 * threadIdx.x, 4, true, x0[c]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) x0[c][i] = tile_token<VEC>(i) < left ? __ldg(row + tile_token<VEC>(i)) : 0.0f;
            }
            if (args.coef.enabled) xt[c] = Tile4<T, VEC>::load_raw(xt_p + (size_t)(cg + c) * plane, left);
        }
    }

    // add the folded increments of the thread's tokens (the mean over their
    // covering anchors, Eq. 1 with the aggregation of Sec. 3.2): s_n holds the
    // tile's anchor counts, a byte per token; g / n is a multiplication
    // for n a power of two (exact) and a division otherwise
    template <bool COPY>
    __device__ __forceinline__ void fold4(const float (*s_acc)[4], const uint8_t* s_n) {
        uint32_t n4 = 0;
        if (VEC) {
            n4 = *reinterpret_cast<const uint32_t*>(s_n + 4 * threadIdx.x);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) n4 |= (uint32_t)s_n[tile_token<VEC>(i)] << (8 * i);
        }
        if (!n4) return;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int n = (int)((n4 >> (8 * i)) & 0xffu);
            if (!n) continue;
            const float4 gq = *reinterpret_cast<const float4*>(s_acc[tile_token<VEC>(i)]);
            const float gg[4] = {gq.x, gq.y, gq.z, gq.w};
            float m[4];
            if (n == 1) {
#pragma unroll
                for (int c = 0; c < 4; ++c) m[c] = gg[c];
            } else if ((n & (n - 1)) == 0) {
                const float rn = __frcp_rn((float)n);
#pragma unroll
                for (int c = 0; c < 4; ++c) m[c] = __fmul_rn(gg[c], rn);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) m[c] = __fdiv_rn(gg[c], (float)n);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) x0[c][i] = COPY ? m[c] : __fadd_rn(x0[c][i], m[c]);
        }
    }

    // store x0(t) and the reconstruction
    __device__ __forceinline__ void store(const TransportArgs& args, int b, int v, int tile0, int left, int cg, int cn) {
        const size_t plane = (size_t)args.H * args.W;
        const size_t view_base = ((size_t)b * args.N + v) * args.C * plane + tile0;
        T* xn_p = static_cast<T*>(args.x_next);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (c >= cn) break;
            const size_t e = view_base + (size_t)(cg + c) * plane;
            Tile4<float, VEC>::store(args.x0_out + e, left, x0[c]);
            if (args.coef.enabled) {
                float x[4], yv[4], pr[4];
                Lat4<T>::unpack(xt[c], x);
#pragma unroll
                for (int i = 0; i < 4; ++i) yv[i] = recon_one(args.coef, x[i], x0[c][i], pr[i]);
                Tile4<T, VEC>::store(xn_p + e, left, yv);
                if (args.pred_out) Tile4<float, VEC>::store(args.pred_out + e, left, pr);
            }
        }
    }
};

// Grid shape of a sparse step's launches and the divisors that split it.
struct SparseGrid {
    int n_cg, n_tiles, n_slices, n_stream, n_total;
    int small;  // n_total * n_stream < 2^31: the interleave's quotients in 32 bits
    FastDiv cg, tiles, a, na, slices, total;
};

// Records of one pair applied by one CTA slice (grid-stride over the pair's
// records), channels [cg, cg + 4).  COPY: the value-copy ablation (no x0(t-1)
// gathers).
template <int K, bool COPY>
__device__ __forceinline__ void apply_records(const TransportArgs& args, const SparseGrid& g, int pair_id, int slice,
                                              int cg) {
    const int N = args.N, C = args.C, a = args.a;
    const int HW = args.H * args.W;
    const int T = g.n_tiles;
    const int n_slices = g.n_slices;
    const int pa = (int)g.a.quo((uint32_t)pair_id);
    const int s2 = pair_id - pa * a;
    const int b = (int)g.na.quo((uint32_t)pa);
    const int vi = pa - b * (N - a);
    const int v = args.others[vi];
    const int u = args.anchors[s2];
    const size_t pair = ((size_t)b * N + v) * N + u;
    const long long cap = args.max_records;
    const int r0 = record_offset(args.tile_ptr, pair * T, cap);
    const int r1 = record_offset(args.tile_ptr, pair * T + T, cap);
    const size_t plane = (size_t)HW;
    const float* xn = args.x0_new + ((size_t)b * a + s2) * C * plane;
    const float* xp = args.x0_prev + ((size_t)b * N + u) * C * plane;
    for (int r = r0 + slice * kThreads + threadIdx.x; r < r1; r += n_slices * kThreads) {
        const int4 rec = __ldg(reinterpret_cast<const int4*>(args.records) + r);
        Taps tp;
        taps_from_record<K>((int)((uint32_t)rec.x >> 28), rec.y, __int_as_float(rec.z), __int_as_float(rec.w),
                            args.W, tp);
        float* out = args.workspace + (size_t)r * C;
        {
            const int cn = C - cg < 4 ? C - cg : 4;
            float dn[K][4], dp[K][4];
#pragma unroll
            for (int kk = 0; kk < K; ++kk)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    dn[kk][c] = 0.0f;
                    dp[kk][c] = 0.0f;
                    if (tp.q[kk] >= 0 && c < cn) {
                        const size_t e = (size_t)(cg + c) * plane + tp.q[kk];
                        dn[kk][c] = __ldg(xn + e);
                        if (!COPY) dp[kk][c] = __ldg(xp + e);
                    }
                }
            float g[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float acc = 0.0f;
#pragma unroll
                for (int kk = 0; kk < K; ++kk)
                    if (tp.q[kk] >= 0) acc = tap_term(COPY, tp.w[kk], dn[kk][c], dp[kk][c], acc);
                g[c] = acc;
            }
            if (cn == 4 && C % 4 == 0) {
                *reinterpret_cast<float4*>(out + cg) = make_float4(g[0], g[1], g[2], g[3]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (c < cn) out[cg + c] = g[c];
            }
        }
    }
}

// Phase A: n_apply record-slice CTAs and n_stream anchor-view CTAs (tiles of
// kTileTokens tokens), each for one group of 4 channels, interleaved evenly in
// block order.
// Resident CTAs per SM the phases are compiled for, by latent type: with
// bf16 latents 6 (phase A, at most 40 registers) and 5 (phase B) put more
// gathers and streamed rows in flight than the few spilled registers cost
// (measured: unbounded, 62 / 56 registers, was 2-3 us slower per step); f32
// latents need more registers per quad and are left unbounded.
template <typename T>
constexpr int kPhaseABlocks = sizeof(T) == 2 ? 6 : 1;
template <typename T>
constexpr int kPhaseBBlocks = sizeof(T) == 2 ? 5 : 1;
// The increment-plane kernels (wide latents): phase A at 4 resident CTAs per
// SM (62 registers; at 5 or 6 its spills cost more than the residency
// gains), phase B at 5 (45 registers for 4 taps of bf16: it loads its streamed rows
// after the fold, so they are not held across the gathers; 4 or 6 resident
// CTAs, or the rows prefetched into the L2 before the wait, were slower).
constexpr int kPlaneABlocks = 4;
constexpr int kPlaneBBlocks = 5;

template <typename T, int K, bool VEC, bool COPY>
__global__ void __launch_bounds__(kThreads, kPhaseABlocks<T>) sparse_phase_a_kernel(const TransportArgs args,
                                                                                    const SparseGrid g) {
    pdl_launch_dependents();
    const uint32_t k = blockIdx.x;
    int s_before, s_next;
    if (g.small) {
        s_before = (int)g.total.quo(k * (uint32_t)g.n_stream);
        s_next = (int)g.total.quo((k + 1) * (uint32_t)g.n_stream);
    } else {
        s_before = (int)((long long)k * g.n_stream / g.n_total);
        s_next = (int)(((long long)k + 1) * g.n_stream / g.n_total);
    }
    if (s_next == s_before) {  // a record-apply CTA
        const int ai = (int)k - s_before;
        const int aj = (int)g.cg.quo((uint32_t)ai);
        const int pair = (int)g.slices.quo((uint32_t)aj);
        apply_records<K, COPY>(args, g, pair, aj - pair * g.n_slices, (ai - aj * g.n_cg) * 4);
        return;
    }
    const int q1 = (int)g.cg.quo((uint32_t)s_before);
    const int cg = (s_before - q1 * g.n_cg) * 4;
    const int q2 = (int)g.tiles.quo((uint32_t)q1);
    const int tile = q1 - q2 * g.n_tiles;
    const int b = (int)g.a.quo((uint32_t)q2);
    const int slot = q2 - b * args.a;
    const int v = args.anchors[slot];
    const int HW = args.H * args.W;
    const int tile0 = tile * kTileTokens;
    const int left = min(kTileTokens, HW - tile0);
    if (tile_token<VEC>(0) >= left) return;
    const int cn = args.C - cg < 4 ? args.C - cg : 4;
    QuadRows<T, VEC> q;
    q.load(args, b, v, slot, tile0, left, cg, cn);
    q.store(args, b, v, tile0, left, cg, cn);
}

// Phase B: one CTA per (tile, group of 4 channels) of a view; blockIdx.y <
// N - a: views outside the anchor set (fold the tile's increments);
// blockIdx.y >= N - a: anchor views (only for an in-place cache update, see
// phase A).  PK = 0: each record's increment is its workspace row, written
// by phase A's apply; PK = K: it is formed here from the anchors' increment
// plane, sum_k w_k increment[q_k] in tap order (the same terms in the same
// order as the applies, so the same bits).
template <typename T, bool VEC, bool COPY, int PK>
__global__ void __launch_bounds__(kThreads, PK ? kPlaneBBlocks : kPhaseBBlocks<T>) sparse_phase_b_kernel(const TransportArgs args, const SparseGrid g) {
    __shared__ float s_acc[kTileTokens][4];
    __shared__ __align__(4) uint8_t s_n[kTileTokens];
    __shared__ int s_r0[GEOCACHE_MAX_VIEWS], s_cnt[GEOCACHE_MAX_VIEWS];
    const int HW = args.H * args.W;
    const int T_tiles = tiles_per_view_dev(args.H, args.W);
    const int n_cg = g.n_cg;
    const int tile = (int)g.cg.quo(blockIdx.x), cg = ((int)blockIdx.x - tile * n_cg) * 4, b = blockIdx.z;
    const int N = args.N, C = args.C, a = args.a;
    const int cn = C - cg < 4 ? C - cg : 4;
    const int tile0 = tile * kTileTokens;
    const int t = threadIdx.x;
    const int left = min(kTileTokens, HW - tile0);
    const bool mine = tile_token<VEC>(0) < left;  // the thread has tokens of the tile
    if ((int)blockIdx.y >= N - a) {  // anchor view, in-place update: after phase A's gathers
        const int slot = blockIdx.y - (N - a);
        pdl_wait();
        if (!mine) return;
        QuadRows<T, VEC> q;
        q.load(args, b, args.anchors[slot], slot, tile0, left, cg, cn);
        q.store(args, b, args.anchors[slot], tile0, left, cg, cn);
        return;
    }
    const int v = args.others[blockIdx.y];
    // streamed rows first (phase A writes none of them), tile offsets next;
    // with the plane (PK) the rows are loaded after the fold instead, which
    // keeps the fold's registers free for more resident CTAs
    QuadRows<T, VEC> q;
    if (!PK && mine) q.load(args, b, v, -1, tile0, left, cg, cn);
    if (t < a) {
        const size_t i = (((size_t)b * N + v) * N + args.anchors[t]) * T_tiles + tile;
        // ranges clamped to the records that exist (an overflow is reported by the build)
        const int r0 = record_offset(args.tile_ptr, i, args.max_records);
        s_r0[t] = r0;
        s_cnt[t] = max(record_offset(args.tile_ptr, i + 1, args.max_records) - r0, 0);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // the sums, cleared before the wait
        *reinterpret_cast<float4*>(s_acc[4 * t + i]) = make_float4(0.f, 0.f, 0.f, 0.f);
        s_n[4 * t + i] = 0;
    }
    __syncthreads();
    int total = 0;
    for (int s2 = 0; s2 < a; ++s2) total += s_cnt[s2];
    // a tile without records keeps x0(t-1) and reads and writes nothing phase A
    // touches (rows of views outside the anchor set), so it is stored without
    // waiting for phase A; the first CTA always waits, so that this grid
    // completes only after phase A
    const bool first = blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
    if (total == 0 && !first) {
        if (mine) {
            if (PK) q.load(args, b, v, -1, tile0, left, cg, cn);
            q.store(args, b, v, tile0, left, cg, cn);
        }
        return;
    }
    pdl_wait();  // phase A's workspace writes are complete and visible
    if (total == 0) {  // no record in the tile: every token keeps x0(t-1), nothing to fold
        if (mine) {
            if (PK) q.load(args, b, v, -1, tile0, left, cg, cn);
            q.store(args, b, v, tile0, left, cg, cn);
        }
        return;
    }
    for (int j0 = 0; j0 < total; j0 += kThreads) {
        const int j = j0 + t;
        int s_mine = -1, lp = 0;
        float g[4] = {0.f, 0.f, 0.f, 0.f};
        if (j < total) {
            int s2 = 0, jj = j;
            while (jj >= s_cnt[s2]) jj -= s_cnt[s2++];
            const int r = s_r0[s2] + jj;
            if (PK) {  // sum_k w_k increment[q_k] in tap order, from the anchor's increment plane
                const int4 rec = __ldg(reinterpret_cast<const int4*>(args.records) + r);
                lp = (rec.x & 0x0fffffff) - tile0;
                Taps tp;
                taps_from_record<PK ? PK : 1>((int)((uint32_t)rec.x >> 28), rec.y, __int_as_float(rec.z),
                                              __int_as_float(rec.w), args.W, tp);
                const float4* d = reinterpret_cast<const float4*>(args.workspace) +
                                  (((size_t)b * a + s2) * n_cg + cg / 4) * (size_t)HW;
                float4 dq[PK ? PK : 1];
#pragma unroll
                for (int kk = 0; kk < (PK ? PK : 1); ++kk)
                    dq[kk] = tp.q[kk] >= 0 ? __ldca(d + tp.q[kk]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int kk = 0; kk < (PK ? PK : 1); ++kk) {
                    if (tp.q[kk] < 0) continue;
                    g[0] = __fmaf_rn(tp.w[kk], dq[kk].x, g[0]);
                    g[1] = __fmaf_rn(tp.w[kk], dq[kk].y, g[1]);
                    g[2] = __fmaf_rn(tp.w[kk], dq[kk].z, g[2]);
                    g[3] = __fmaf_rn(tp.w[kk], dq[kk].w, g[3]);
                }
            } else {
                lp = (__ldg(&args.records[r].token_mask) & 0x0fffffff) - tile0;
                const float* w = args.workspace + (size_t)r * C + cg;
                if (cn == 4 && C % 4 == 0) {
                    const float4 wq = *reinterpret_cast<const float4*>(w);
                    g[0] = wq.x; g[1] = wq.y; g[2] = wq.z; g[3] = wq.w;
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (c < cn) g[c] = w[c];
                }
            }
            s_mine = s2;
        }
        // combine in anchor order (deterministic): anchor s2 adds in pass s2; the
        // records are in anchor order, so only the anchors of this round pass
        int s_lo = 0, c_lo = 0;
        while (c_lo + s_cnt[s_lo] <= j0) c_lo += s_cnt[s_lo++];
        const int j_last = (j0 + kThreads < total ? j0 + kThreads : total) - 1;
        int s_hi = s_lo, c_hi = c_lo;
        while (c_hi + s_cnt[s_hi] <= j_last) c_hi += s_cnt[s_hi++];
        for (int s2 = s_lo; s2 <= s_hi; ++s2) {
            if (s_mine == s2) {
                float4* dst = reinterpret_cast<float4*>(s_acc[lp]);
                float4 cur = *dst;
                cur.x = __fadd_rn(cur.x, g[0]);
                cur.y = __fadd_rn(cur.y, g[1]);
                cur.z = __fadd_rn(cur.z, g[2]);
                cur.w = __fadd_rn(cur.w, g[3]);
                *dst = cur;
                s_n[lp] += 1;
            }
            __syncthreads();
        }
    }
    if (mine) {
        if (PK) q.load(args, b, v, -1, tile0, left, cg, cn);
        q.template fold4<COPY>(s_acc, s_n);
        q.store(args, b, v, tile0, left, cg, cn);
    }
}

// Phase A with the anchors' increment plane (wide latents): one CTA per
// (asset, anchor slot, tile, group of 4 channels) streams the anchor tile
// (x0(t) = x0_new and the reconstruction) and writes the tile's increment
// x0_new - x0(t-1) (x0_new itself under the value copy) to the plane
// [b][slot][channel group][token] x 4 channels in the workspace, where phase
// B gathers it at the records' taps.  Each element is read before the same
// thread writes it, so the stream is also correct for an in-place update.
template <typename T, bool VEC, bool COPY>
__global__ void __launch_bounds__(kThreads, kPlaneABlocks) sparse_phase_a_plane_kernel(const TransportArgs args,
                                                                                         const SparseGrid g) {
    pdl_launch_dependents();
    const int HW = args.H * args.W;
    const int n_cg = g.n_cg;
    const int q1 = (int)g.cg.quo(blockIdx.x);
    const int cgi = (int)blockIdx.x - q1 * n_cg;
    const int q2 = (int)g.tiles.quo((uint32_t)q1);
    const int tile = q1 - q2 * g.n_tiles;
    const int b = (int)g.a.quo((uint32_t)q2);
    const int slot = q2 - b * args.a;
    const int tile0 = tile * kTileTokens, left = min(kTileTokens, HW - tile0);
    if (tile_token<VEC>(0) >= left) return;
    const int cg = cgi * 4;
    const int cn = args.C - cg < 4 ? args.C - cg : 4;
    const size_t plane = (size_t)HW;
    const int u = args.anchors[slot];
    const float* xn = args.x0_new + ((size_t)b * args.a + slot) * args.C * plane;
    const float* xp = args.x0_prev + ((size_t)b * args.N + u) * args.C * plane;
    const size_t view_base = ((size_t)b * args.N + u) * args.C * plane;
    const T* xt_p = static_cast<const T*>(args.x_t);
    T* xn_p = static_cast<T*>(args.x_next);
    float dn[4][4], pv[4][4];
    typename Lat4<T>::Raw xr[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (c >= cn) break;
        const size_t e = (size_t)(cg + c) * plane + tile0;
        Tile4<float, VEC>::load(xn + e, left, dn[c]);
        if (!COPY) Tile4<float, VEC>::load(xp + e, left, pv[c]);
        if (args.coef.enabled) xr[c] = Tile4<T, VEC>::load_raw(xt_p + view_base + e, left);
    }
    float dd[4][4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) dd[c][i] = c < cn ? (COPY ? dn[c][i] : __fsub_rn(dn[c][i], pv[c][i])) : 0.0f;
    float4* d = reinterpret_cast<float4*>(args.workspace) + (((size_t)b * args.a + slot) * n_cg + cgi) * plane + tile0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (tile_token<VEC>(i) < left) d[tile_token<VEC>(i)] = make_float4(dd[0][i], dd[1][i], dd[2][i], dd[3][i]);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (c >= cn) break;
        const size_t e = view_base + (size_t)(cg + c) * plane + tile0;
        Tile4<float, VEC>::store(args.x0_out + e, left, dn[c]);
        if (args.coef.enabled) {
            float x[4], yv[4], pr[4];
            Lat4<T>::unpack(xr[c], x);
#pragma unroll
            for (int i = 0; i < 4; ++i) yv[i] = recon_one(args.coef, x[i], dn[c][i], pr[i]);
            Tile4<T, VEC>::store(xn_p + e, left, yv);
            if (args.pred_out) Tile4<float, VEC>::store(args.pred_out + e, left, pr);
        }
    }
}

// Phase A by source tile (wide latents): one CTA per (asset, anchor slot,
// source tile, group of 4 channels).  It stages the anchor's increment
// x0_new - x0(t-1) (x0_new itself for the value copy) of the tile and of the
// W + 1 tokens after it in shared memory ([token][4 channels]: every tap of a
// record whose first kept tap lies in the tile), streams the anchor tile
// itself (x0(t) and the reconstruction) unless the update is in place (both in
// 16-byte words with vec_rows, where every row starts on one), and then applies
// the tile's group of the source index: for each record whose target view is
// outside the anchor set, sum_k w_k increment[q_k] in tap order, read from
// shared memory, into its workspace row.  The scattered per-channel gathers of
// the record-parallel apply become one coalesced read of the anchor tile.
template <typename T, int K, bool COPY>
__global__ void __launch_bounds__(kThreads, kPhaseABlocks<T>) sparse_phase_a_src_kernel(const TransportArgs args,
                                                                                       const SparseGrid g, bool stream,
                                                                                       bool vec_rows) {
    pdl_launch_dependents();
    extern __shared__ __align__(16) float4 s_d[];  // [kTileTokens + W + 1] tokens x 4 channels
    const int HW = args.H * args.W, W = args.W;
    const int N = args.N, C = args.C, a = args.a;
    const int n_tiles = g.n_tiles;
    const int q1 = (int)g.cg.quo(blockIdx.x);
    const int cg = ((int)blockIdx.x - q1 * g.n_cg) * 4;
    const int q2 = (int)g.tiles.quo((uint32_t)q1);
    const int st = q1 - q2 * n_tiles;
    const int b = (int)g.a.quo((uint32_t)q2);
    const int slot = q2 - b * a;
    const int u = args.anchors[slot];
    const int cn = C - cg < 4 ? C - cg : 4;
    const size_t plane = (size_t)HW;
    const int tile0 = st * kTileTokens;
    const int span = min(kTileTokens + W + 1, HW - tile0);  // staged tokens
    const float* xn = args.x0_new + ((size_t)b * a + slot) * C * plane;
    const float* xp = args.x0_prev + ((size_t)b * N + u) * C * plane;
    const size_t view_base = ((size_t)b * N + u) * C * plane;
    const T* xt_p = static_cast<const T*>(args.x_t);
    T* xn_p = static_cast<T*>(args.x_next);
    for (int q = threadIdx.x; 4 * q < span; q += kThreads) {
        const int p0 = tile0 + 4 * q;
        const int cnt = min(4, span - 4 * q);
        const bool vec = vec_rows && cnt == 4;
        float dd[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
#pragma unroll
            for (int i = 0; i < 4; ++i) dd[c][i] = 0.0f;
            if (c >= cn) continue;
            float dn[4];
            f4_load_keep(xn, (size_t)(cg + c) * plane + p0, cnt, vec, dn);
            if (!COPY) {
                float pv[4];
                f4_load_keep(xp, (size_t)(cg + c) * plane + p0, cnt, vec, pv);
#pragma unroll
                for (int i = 0; i < 4; ++i) dd[c][i] = __fsub_rn(dn[i], pv[i]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) dd[c][i] = dn[i];
            }
            if (stream && 4 * q < kTileTokens) {  // the anchor tile itself: x0(t) and the reconstruction
                const size_t e = view_base + (size_t)(cg + c) * plane + p0;
                Lat4<float>::store(args.x0_out, e, cnt, vec, dn);
                if (args.coef.enabled) {
                    float x[4], yv[4], pr[4];
                    Lat4<T>::load(xt_p, e, cnt, vec, x);
#pragma unroll
                    for (int i = 0; i < 4; ++i) yv[i] = recon_one(args.coef, x[i], dn[i], pr[i]);
                    Lat4<T>::store(xn_p, e, cnt, vec, yv);
                    if (args.pred_out) Lat4<float>::store(args.pred_out, e, cnt, vec, pr);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < cnt) s_d[4 * q + i] = make_float4(dd[0][i], dd[1][i], dd[2][i], dd[3][i]);
    }
    __syncthreads();
    const size_t grp = ((size_t)b * N + u) * n_tiles + st;  // group ends: see src_index_kernel
    const int lo = grp ? __ldg(args.src_ptr + grp - 1) : 0, hi = __ldg(args.src_ptr + grp);
    const int2* src_rec = reinterpret_cast<const int2*>(args.src_rec);
    for (int e0 = lo + threadIdx.x; e0 < hi; e0 += 2 * kThreads) {
        // two entries per thread, their loads in flight together
        int2 ent[2];
        int4 rec[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int e = e0 + m * kThreads;
            ent[m] = e < hi ? __ldg(src_rec + e) : make_int2(-1, 0);
            if (ent[m].x >= 0 && args.slot_of[ent[m].y] >= 0) ent[m].x = -1;  // target view is an anchor
            rec[m] = ent[m].x >= 0 ? __ldg(reinterpret_cast<const int4*>(args.records) + ent[m].x)
                                   : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            if (ent[m].x < 0) continue;
            Taps tp;
            taps_from_record<K>((int)((uint32_t)rec[m].x >> 28), rec[m].y, __int_as_float(rec[m].z),
                                __int_as_float(rec[m].w), W, tp);
            float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < K; ++kk) {
                if (tp.q[kk] < 0) continue;
                const float4 d = s_d[tp.q[kk] - tile0];
                g[0] = __fmaf_rn(tp.w[kk], d.x, g[0]);
                g[1] = __fmaf_rn(tp.w[kk], d.y, g[1]);
                g[2] = __fmaf_rn(tp.w[kk], d.z, g[2]);
                g[3] = __fmaf_rn(tp.w[kk], d.w, g[3]);
            }
            float* out = args.workspace + (size_t)ent[m].x * C + cg;
            if (cn == 4 && C % 4 == 0) {
                *reinterpret_cast<float4*>(out) = make_float4(g[0], g[1], g[2], g[3]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (c < cn) out[c] = g[c];
            }
        }
    }
}

// The source-tile apply serves wide latents (at least kSrcMinChannels
// channels) whose workspace has no room for the increment plane, where the
// record-parallel apply's per-channel gathers dominate phase A; with few
// channels it is slower (it reads the anchors' whole x0(t-1) rows instead of
// the tapped tokens).
constexpr int kSrcMinChannels = 8;
// Record-parallel apply: CTAs per (pair, channel group) sized for about this
// many records each, from the mean records per ordered view pair.
constexpr long long kApplyRecords = 384;

template <typename T, int K, int MODE>
static cudaError_t launch_token(const TransportArgs& t, cudaStream_t s);

// A sparse step that is not in place takes one token per thread from the records,
// in one launch instead of two and without the workspace, up to kTokenUnitsSparse
// units (tiles of 1024 tokens x channel groups; in place the anchors' rows wait
// for every gather, so a second launch is needed anyway).  Its cost grows with
// the units of the target views, whose CTAs each read the records of the whole
// tile around their 256 tokens, so those have a lower limit of their own, by what
// the two launches would do: gather from the increment plane, or apply the
// records into rows, or that with unaligned rows.  Device us of the two launches
// and the one (bf16; a anchors of 6 views unless said):
//   plane     64 x 64 x 8, a = 1: 80 target units 5.6 and 4.0, 160 5.8 and 6.3, 240 6.3
//             and 7.7; a = 4: 96 9.9 and 7.5, 128 10.2 and 8.8; 24 views of 32 x 32 x 8,
//             a = 4: 120 8.4 and 9.5
//   rows      64 x 64 x 4, a = 2: 160 8.0 and 7.3, 192 8.2 and 8.1, 256 8.4 and 9.9; 12
//             views, a = 4: 192 15.9 and 12.3
//   unaligned 75 x 53 x 4: a = 1, 240: 9.7 and 8.1, 320 10.5 and 10.0, 480 11.1 and 13.6
// Over 760 steps of up to 384 units (6 to 64 views of 16 x 16 to 128 x 128, 1 to 48
// anchors) the limits choose within 1% of the faster on average, 23% at worst;
// 384 units alone 7% and 86%.
constexpr long long kTokenUnitsSparse = 384, kTokenTargetsPlane = 144, kTokenTargetsRows = 256, kTokenTargetsUnaligned = 320;

template <typename T, int K>
static cudaError_t launch_sparse(const TransportArgs& t, cudaStream_t s) {
    const int HW = t.H * t.W;
    const int n_tiles = (HW + kTileTokens - 1) / kTileTokens;
    const int n_cg = (t.C + 3) / 4;
    const uintptr_t al = (uintptr_t)t.x0_new | (uintptr_t)t.x0_prev | (uintptr_t)t.x0_out | (uintptr_t)t.x_t |
                         (uintptr_t)t.x_next | (uintptr_t)t.pred_out;
    const bool vec = (HW % 4 == 0) && (al % 16 == 0);
    const bool in_place = t.x0_out == t.x0_prev;
    const bool copy = t.update == GEOCACHE_UPDATE_COPY;
    // wide latents: the anchors' increment plane when the workspace holds it
    // beside max_records * C floats, else phase A by source tile when the
    // corr has a source index and the staged span (tile + W + 1 tokens)
    // fits, else the record-parallel apply
    SparseGrid sg{};
    sg.n_cg = n_cg;
    sg.n_tiles = n_tiles;
    sg.cg = make_fastdiv((uint32_t)n_cg);
    sg.tiles = make_fastdiv((uint32_t)n_tiles);
    sg.a = make_fastdiv((uint32_t)t.a);
    sg.na = make_fastdiv((uint32_t)(t.N > t.a ? t.N - t.a : 1));
    const long long n_plane = plane_floats(t.B, t.a, t.C, HW);
    const bool by_plane = t.a < t.N && t.C >= kPlaneMinChannels && t.workspace &&
                          t.workspace_floats >= t.max_records * (long long)t.C + n_plane;
    const bool by_source = !by_plane && t.a < t.N && t.src_ptr && t.src_rec && t.C >= kSrcMinChannels &&
                           t.W + 1 <= kTileTokens;
    const long long per_view = (long long)t.B * n_tiles * n_cg;
    if (!in_place && t.a < t.N && per_view * t.N <= kTokenUnitsSparse &&
        per_view * (t.N - t.a) <= (!vec ? kTokenTargetsUnaligned : (by_plane ? kTokenTargetsPlane : kTokenTargetsRows)))
        return launch_token<T, K, GEOCACHE_CORR_SPARSE>(t, s);
    bool phase_a = false;
    if (by_plane) {
        const long long g = (long long)t.B * t.a * n_tiles * n_cg;
        if (g > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        if (vec && !copy) sparse_phase_a_plane_kernel<T, true, false><<<(unsigned)g, kThreads, 0, s>>>(t, sg);
        else if (vec) sparse_phase_a_plane_kernel<T, true, true><<<(unsigned)g, kThreads, 0, s>>>(t, sg);
        else if (!copy) sparse_phase_a_plane_kernel<T, false, false><<<(unsigned)g, kThreads, 0, s>>>(t, sg);
        else sparse_phase_a_plane_kernel<T, false, true><<<(unsigned)g, kThreads, 0, s>>>(t, sg);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        phase_a = true;
    } else if (by_source) {
        const long long g = (long long)t.B * t.a * n_tiles * n_cg;
        if (g > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        const size_t dyn = (size_t)(kTileTokens + t.W + 1) * sizeof(float4);
        if (!copy)
            sparse_phase_a_src_kernel<T, K, false><<<(unsigned)g, kThreads, dyn, s>>>(t, sg, !in_place, vec);
        else
            sparse_phase_a_src_kernel<T, K, true><<<(unsigned)g, kThreads, dyn, s>>>(t, sg, !in_place, vec);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        phase_a = true;
    } else {
        // apply CTAs per (pair, channel group): about kApplyRecords records each
        const long long pairs = (long long)t.B * t.N * (t.N - 1);
        const long long per_pair = (t.max_records + pairs - 1) / pairs;
        long long n_slices = (per_pair + kApplyRecords - 1) / kApplyRecords;
        n_slices = n_slices < 1 ? 1 : (n_slices > 64 ? 64 : n_slices);
        const long long n_apply = t.a < t.N ? (long long)t.B * (t.N - t.a) * t.a * n_slices * n_cg : 0;
        const long long n_stream = in_place ? 0 : (long long)t.B * t.a * n_tiles * n_cg;
        if (n_apply + n_stream > 0) {
            if (n_apply + n_stream > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
            const unsigned g = (unsigned)(n_apply + n_stream);
            sg.n_slices = (int)n_slices;
            sg.slices = make_fastdiv((uint32_t)n_slices);
            sg.n_stream = (int)n_stream;
            sg.n_total = (int)g;
            sg.total = make_fastdiv(g);
            sg.small = (long long)g * n_stream < 0x80000000LL;
            if (vec && !copy)
                sparse_phase_a_kernel<T, K, true, false><<<g, kThreads, 0, s>>>(t, sg);
            else if (vec)
                sparse_phase_a_kernel<T, K, true, true><<<g, kThreads, 0, s>>>(t, sg);
            else if (!copy)
                sparse_phase_a_kernel<T, K, false, false><<<g, kThreads, 0, s>>>(t, sg);
            else
                sparse_phase_a_kernel<T, K, false, true><<<g, kThreads, 0, s>>>(t, sg);
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            phase_a = true;
        }
    }
    if (phase_a) note_launches(1);
    // an in-place update streams the anchor views after the wait, except with
    // the plane (its phase A reads each anchor element before writing it)
    const int gy = (t.N - t.a) + (in_place && !by_plane ? t.a : 0);
    if (gy > 0) {
        if ((long long)n_tiles * n_cg > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(n_tiles * n_cg), gy, t.B);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = phase_a ? 1 : 0;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e;
        if (by_plane) {
            if (vec && !copy) e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, true, false, K>, t, sg);
            else if (vec) e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, true, true, K>, t, sg);
            else if (!copy) e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, false, false, K>, t, sg);
            else e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, false, true, K>, t, sg);
        } else {
            if (vec && !copy) e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, true, false, 0>, t, sg);
            else if (vec) e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, true, true, 0>, t, sg);
            else if (!copy) e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, false, false, 0>, t, sg);
            else e = cudaLaunchKernelEx(&cfg, sparse_phase_b_kernel<T, false, true, 0>, t, sg);
        }
        if (e != cudaSuccess) return e;
        note_launches(1);
    }
    return cudaGetLastError();
}

// Persistent grid size of an instantiation: resident CTAs per SM x SMs.
template <typename Kern>
static int persistent_grid(Kern kern, size_t dyn_smem) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, dyn_smem) != cudaSuccess) return 0;
    return sms * (per_sm > 0 ? per_sm : 1);
}

// Units (tiles of 1024 tokens x channel groups) up to which a MASK step takes
// one token per thread.  With 16-byte aligned rows, against the staged kernel
// (us; 96 x 96 x 4 bf16, 6 views, 3 anchors): 24 units 8.3 and 4.6, 432 18.7 and
// 12.7, 1,728 49.1 and 53.9; between 512 and 1,024 units it is the faster for
// assets of many tokens, with few anchors later (768 units: 6 views of 32 x 32 x 4,
// 2 anchors 16.0 and 21.2; 12 of 64 x 64 x 4, 4 anchors 37.4 and 26.3).  Otherwise
// against one CTA per tile (75 x 53 x 4): 96 units 8.2 and 5.1, 384 11.9 and 11.1,
// 960 23.7 and 29.2.
static long long mask_token_units(const TransportArgs& t, bool staged) {
    if (!staged) return 384;
    const long long asset = (long long)t.N * t.H * t.W;
    return asset >= (t.a <= 2 ? 98304 : 24576) ? 1024 : 512;
}

template <typename T, int K, int MODE>
static cudaError_t launch_token(const TransportArgs& t, cudaStream_t s) {
    const int HW = t.H * t.W, n_cg = (t.C + 3) / 4;
    const dim3 grid((unsigned)((HW + kThreads - 1) / kThreads * n_cg), t.N, t.B);
    return launch_pdl(transport_token_kernel<T, K, MODE>, grid, kThreads, 0, s, t, make_fastdiv((uint32_t)n_cg));
}

// TABLE and GEOMETRY steps of at least this many units with one anchor (for
// GEOMETRY on unaligned rows and f32 latents, two) keep the kernels with a tile of
// 1024 tokens per CTA: the steps are then bound by their streams, which those
// move in 16-byte words, and one item per token leaves no chain to shorten.
// Token kernel and these (us; 6 views of 128 x 128, bf16): 1 anchor, 6,144 units of
// C = 4: geometry 247 and 225, tables 226 and 198; of C = 16: 234 and 165, 217 and 171;
// 1,056 units of C = 4: 34 and 41, 35 and 36; 2 anchors, 6,144 units of C = 4: 263 and 314, 281
// and 289 (of C = 16: 252 and 223, 267 and 251, but 12 views of 64 x 64: 1.1 to 1.4
// times faster by token).  With aligned rows, tables of single taps read a word per
// item and are faster by token at every size (3,072 units of C = 4: 72 and 88), those
// of f32 latents as fast.
constexpr long long kTileUnitsItems = 1280;
template <typename T, int K>
static bool items_by_tile(const TransportArgs& t, bool staged, long long n_units) {
    if (n_units < kTileUnitsItems) return false;
    if (t.mode == GEOCACHE_CORR_TABLE) return t.a == 1 && !(staged && (K == 1 || sizeof(T) == 4));
    return t.a == 1 || (t.a == 2 && !staged && sizeof(T) == 4);
}

template <typename T, int K, int MODE>
static cudaError_t launch_tiles(const TransportArgs& t, cudaStream_t s) {
    const int HW = t.H * t.W;
    const uintptr_t al = (uintptr_t)t.x0_new | (uintptr_t)t.x0_prev | (uintptr_t)t.x0_out | (uintptr_t)t.x_t |
                         (uintptr_t)t.x_next | (uintptr_t)t.pred_out | (uintptr_t)t.keep | (uintptr_t)t.valid;
    const bool vec = (HW % 4 == 0) && (al % 16 == 0);
    const int n_tiles = (HW + kTileTokens - 1) / kTileTokens;
    const int n_cg = (t.C + 3) / 4;
    const long long n_units = (long long)t.B * t.N * n_tiles * n_cg;
    const bool staged = vec && HW % 8 == 0;
    if (MODE == GEOCACHE_CORR_MASK) {
        // (a pending request of the test hook is for the staged kernel)
        if (n_units <= mask_token_units(t, staged) && !(staged && g_drop_first_copy.load()))
            return launch_token<T, K, MODE>(t, s);
    } else if (!items_by_tile<T, K>(t, staged, n_units)) {
        return launch_token<T, K, MODE>(t, s);
    }
    // TMA bulk rows need 16-byte aligned starts and sizes: HW % 8 == 0 covers bf16 rows
    if (staged) {
        TransportArgs ta = t;
        ta.wait_limit_ns = g_wait_limit_ns.load();
        ta.drop_first_copy = g_drop_first_copy.exchange(0);
        const size_t dyn = kStages * 4 * kTileTokens * (sizeof(float) + sizeof(T));
        auto kern = transport_fused_kernel<T, K, MODE>;
        static int grid = 0;  // per instantiation and process (one device per process)
        if (!grid) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
            if (e != cudaSuccess) return e;
            grid = persistent_grid(kern, dyn);
            if (!grid) return cudaErrorInvalidConfiguration;
        }
        const long long g = n_units < grid ? n_units : grid;
        note_launches(1);
        kern<<<(unsigned)g, kThreads, dyn, s>>>(ta, n_tiles, n_cg, n_units);
        return cudaGetLastError();
    }
    if (n_units > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    note_launches(1);
    if (vec)
        transport_simple_kernel<T, K, MODE, true><<<(unsigned)n_units, kThreads, 0, s>>>(t, n_tiles, n_cg);
    else
        transport_simple_kernel<T, K, MODE, false><<<(unsigned)n_units, kThreads, 0, s>>>(t, n_tiles, n_cg);
    return cudaGetLastError();
}

template <typename T, int K>
static cudaError_t launch_transport_t(const TransportArgs& t, cudaStream_t s) {
    switch (t.mode) {
        case GEOCACHE_CORR_SPARSE: return launch_sparse<T, K>(t, s);
        case GEOCACHE_CORR_MASK: return launch_tiles<T, K, GEOCACHE_CORR_MASK>(t, s);
        case GEOCACHE_CORR_TABLE: return launch_tiles<T, K, GEOCACHE_CORR_TABLE>(t, s);
        default: return launch_tiles<T, K, GEOCACHE_CORR_GEOMETRY>(t, s);
    }
}

cudaError_t launch_transport(const TransportArgs& t, cudaStream_t s) {
    if (t.lat_dtype == GEOCACHE_BF16)
        return t.K == 4 ? launch_transport_t<__nv_bfloat16, 4>(t, s) : launch_transport_t<__nv_bfloat16, 1>(t, s);
    return t.K == 4 ? launch_transport_t<float, 4>(t, s) : launch_transport_t<float, 1>(t, s);
}

// Anchors' rows of an in-place cache update, written after the gathers.
__global__ void copy_anchor_rows_kernel(const TransportArgs args) {
    const size_t HW = (size_t)args.H * args.W;
    const size_t per = (size_t)args.cn * HW;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int s = blockIdx.y, b = blockIdx.z;
    if (i >= per) return;
    const int u = args.anchors[s];
    args.x0_out[(((size_t)b * args.N + u) * args.C + args.c0) * HW + i] =
        args.x0_new[(((size_t)b * args.a + s) * args.C + args.c0) * HW + i];
}

cudaError_t launch_copy_anchor_rows(const TransportArgs& t, cudaStream_t s) {
    const size_t per = (size_t)t.cn * t.H * t.W;
    dim3 grid((unsigned)((per + 255) / 256), t.a, t.B);
    note_launches(1);
    copy_anchor_rows_kernel<<<grid, 256, 0, s>>>(t);
    return cudaGetLastError();
}

// ------------------------------------------------- anchor-row pack / unpack --
// Gather (pack) of the anchor views' rows of a per-view tensor [B, N, row]
// into [B, a, row] in anchor order, and the scatter back (unpack): the batch
// slicing around the denoiser's anchor-only forward (Sec. 3.2).  Rows are
// copied as raw bytes, 16 bytes per thread when sizes and addresses allow.
template <int VB>
__global__ void __launch_bounds__(256) copy_rows_kernel(const uint8_t* __restrict__ src, uint8_t* __restrict__ dst,
                                                        long long row_bytes, int N, int a, RowAnchors anc, int pack) {
    const int s = blockIdx.y, b = blockIdx.z;
    const int u = anc.v[s];
    const long long src_row = pack ? (long long)b * N + u : (long long)b * a + s;
    const long long dst_row = pack ? (long long)b * a + s : (long long)b * N + u;
    const uint8_t* sp = src + src_row * row_bytes;
    uint8_t* dp = dst + dst_row * row_bytes;
    const long long n = row_bytes / VB;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (VB == 16)
            __stcs(reinterpret_cast<uint4*>(dp) + i, __ldcs(reinterpret_cast<const uint4*>(sp) + i));
        else if (VB == 4)
            __stcs(reinterpret_cast<uint32_t*>(dp) + i, __ldcs(reinterpret_cast<const uint32_t*>(sp) + i));
        else
            dp[i] = sp[i];
    }
}

// ---------------------------------------------------- shuffled records --
// The shuffled-correspondence ablation (Sec. 4.3, "corr -> shuffled"): record
// r keeps its target token and takes the taps (keep mask, top-left tap,
// fractions) of record perm[r].  An entry outside [0, n) sets bit 2 of the
// status word and leaves the record as it was.
__global__ void __launch_bounds__(256) permute_records_kernel(const int4* __restrict__ src,
                                                              const int32_t* __restrict__ perm, int4* __restrict__ dst,
                                                              long long n) {
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x) {
        const int4 own = __ldg(src + r);
        const int p = __ldg(perm + r);
        if (p < 0 || p >= n) {
            atomicOr(&g_device_error, 4u);
            dst[r] = own;
            continue;
        }
        const int4 o = __ldg(src + p);
        dst[r] = make_int4((int)(((uint32_t)own.x & 0x0fffffffu) | ((uint32_t)o.x & 0xf0000000u)), o.y, o.z, o.w);
    }
}

cudaError_t launch_permute_records(const geocache_tap_record* src, const int32_t* perm, geocache_tap_record* dst,
                                   long long n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const long long blocks = (n + 255) / 256;
    note_launches(1);
    permute_records_kernel<<<(unsigned)(blocks < 65535 * 8 ? blocks : 65535 * 8), 256, 0, s>>>(
        reinterpret_cast<const int4*>(src), perm, reinterpret_cast<int4*>(dst), n);
    return cudaGetLastError();
}

cudaError_t launch_copy_rows(const void* src, void* dst, long long row_bytes, int B, int N, int a,
                             const RowAnchors& anc, bool pack, cudaStream_t s) {
    if (row_bytes == 0 || B == 0 || a == 0) return cudaSuccess;
    const uintptr_t al = (uintptr_t)src | (uintptr_t)dst | (uintptr_t)row_bytes;
    const int vb = al % 16 == 0 ? 16 : (al % 4 == 0 ? 4 : 1);
    const long long n = row_bytes / vb;
    long long gx = (n + 255) / 256;
    if (gx > 1024) gx = 1024;
    dim3 grid((unsigned)gx, a, B);
    const uint8_t* sp = static_cast<const uint8_t*>(src);
    uint8_t* dp = static_cast<uint8_t*>(dst);
    note_launches(1);
    if (vb == 16)
        copy_rows_kernel<16><<<grid, 256, 0, s>>>(sp, dp, row_bytes, N, a, anc, pack);
    else if (vb == 4)
        copy_rows_kernel<4><<<grid, 256, 0, s>>>(sp, dp, row_bytes, N, a, anc, pack);
    else
        copy_rows_kernel<1><<<grid, 256, 0, s>>>(sp, dp, row_bytes, N, a, anc, pack);
    return cudaGetLastError();
}

// ---------------------------------------------------- full-step recon --
// Elementwise x_t, x0 -> x_next (and optionally pred, a copy of x0), four
// consecutive elements per thread with 16-byte accesses when every pointer
// is 16-byte aligned; grid-stride over groups of four.
template <typename T, bool VEC>
__global__ void __launch_bounds__(256) reconstruct_kernel(const T* xt, const float* x0, T* xn, int64_t n,
                                                          const ReconCoef coef, float* pred_out, float* x0_store) {
    const int64_t groups = (n + 3) / 4;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < groups;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = 4 * g;
        const int cnt = n - e < 4 ? (int)(n - e) : 4;
        const bool vec = VEC && cnt == 4;
        float a[4], x[4], y[4], pr[4];
        Lat4<float>::load(x0, e, cnt, vec, a);
        Lat4<T>::load(xt, e, cnt, vec, x);
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = recon_one(coef, x[i], a[i], pr[i]);
        Lat4<T>::store(xn, e, cnt, vec, y);
        if (pred_out) Lat4<float>::store(pred_out, e, cnt, vec, pr);
        if (x0_store) Lat4<float>::store(x0_store, e, cnt, vec, a);
    }
}

// The same with eight consecutive elements per thread and no loop, for f32
// pointers on 32 bytes and bf16 ones on 16: half the memory instructions, and a
// CTA's loads all issue at once.  64 assets x 6 views at 128 x 128 x 4, bf16, x0
// stored (302 MB): 48.1 -> 44.5 us, 6.78 TB/s (the copy rate); grid-stride
// over 16 or 32 CTAs per SM 45.8 and 45.2; 128 assets without the store 61.6 ->
// 56.8, f32 62.5 -> 59.3.
template <typename T>
__global__ void __launch_bounds__(256) reconstruct8_kernel(const T* xt, const float* x0, T* xn, int64_t n,
                                                           const ReconCoef coef, float* pred_out, float* x0_store) {
    pdl_wait();
    const int64_t e = 8 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (e + 8 <= n) {
        float a[8], x[8], y[8], pr[8];
        load8(x0 + e, a);
        load8(xt + e, x);
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = recon_one(coef, x[i], a[i], pr[i]);
        store8(xn + e, y);
        if (pred_out) store8(pred_out + e, pr);
        if (x0_store) store8(x0_store + e, a);
        return;
    }
    for (int64_t i = e; i < n; ++i) {  // the last n % 8 elements
        const float a = x0[i];
        float pr;
        lat_store(xn, i, recon_one(coef, lat_load(xt, i), a, pr));
        if (pred_out) pred_out[i] = pr;
        if (x0_store) x0_store[i] = a;
    }
}

template <typename T>
static cudaError_t launch_reconstruct_t(const void* x_t, const float* x0, void* x_next, int64_t n,
                                        const ReconCoef& coef, float* pred_out, float* x0_store, cudaStream_t s) {
    int64_t blocks = ((n + 3) / 4 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    const uintptr_t al = (uintptr_t)x_t | (uintptr_t)x0 | (uintptr_t)x_next | (uintptr_t)pred_out | (uintptr_t)x0_store;
    const T* xt = static_cast<const T*>(x_t);
    T* xn = static_cast<T*>(x_next);
    const uintptr_t f32s = (uintptr_t)x0 | (uintptr_t)pred_out | (uintptr_t)x0_store, lats = (uintptr_t)x_t | (uintptr_t)x_next;
    const int64_t blocks8 = (n + 2047) / 2048;
    if (f32s % 32 == 0 && lats % (8 * sizeof(T)) == 0 && blocks8 <= 0x7fffffffLL)
        return launch_pdl(reconstruct8_kernel<T>, dim3((unsigned)blocks8), 256, 0, s, xt, x0, xn, n, coef, pred_out, x0_store);
    note_launches(1);
    if (al % 16 == 0)
        reconstruct_kernel<T, true><<<(unsigned)blocks, 256, 0, s>>>(xt, x0, xn, n, coef, pred_out, x0_store);
    else
        reconstruct_kernel<T, false><<<(unsigned)blocks, 256, 0, s>>>(xt, x0, xn, n, coef, pred_out, x0_store);
    return cudaGetLastError();
}

cudaError_t launch_reconstruct(const void* x_t, const float* x0, void* x_next, int lat_dtype, int64_t n,
                               const ReconCoef& coef, float* pred_out, float* x0_store, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (lat_dtype == GEOCACHE_BF16)
        return launch_reconstruct_t<__nv_bfloat16>(x_t, x0, x_next, n, coef, pred_out, x0_store, s);
    return launch_reconstruct_t<float>(x_t, x0, x_next, n, coef, pred_out, x0_store, s);
}

cudaError_t read_device_error(unsigned int* out, bool clear, cudaStream_t s) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_device_error, sizeof(unsigned int), 0, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess || !clear || *out == 0) return e;
    static const unsigned int zero = 0;
    e = cudaMemcpyToSymbolAsync(g_device_error, &zero, sizeof(unsigned int), 0, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

}  // namespace geocache
