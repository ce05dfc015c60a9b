// O(N^2) direct-summation product u = M f of the wall-corrected RPY blob
// mobility (Section 2.1.1; Section 5 evaluates it by direct summation on a
// GPU).
//
// Work decomposition: targets are cut into blocks of NT * TPT blobs (one CTA,
// TPT targets per thread) and sources into S chunks; a persistent grid of one
// wave of CTAs walks the (target block, source chunk) items.  Each CTA stages
// NT sources at a time in shared memory (coalesced float4 loads; every thread
// then reads the same source, a shared-memory broadcast) and accumulates the
// tile in FP32 registers, folding each tile sum into a Kahan-compensated
// accumulator.  Chunk partials go to an FP64 buffer that a second kernel sums
// in a fixed order, so results are deterministic.  The symmetric kernels (each
// unordered pair evaluated once for both blobs) add to u with FP64 atomics
// instead: their results agree to FP64 rounding from call to call.
//
// FP32 positions carry a hi/lo split: d = (hi_i - hi_j) + (lo_i - lo_j); the
// hi difference is exact for nearby blobs (Sterbenz), so near pairs keep full
// FP32 accuracy even at |x| of several hundred.
#include <algorithm>
#include <mutex>

#include <cooperative_groups.h>

#include "mb_internal.cuh"
#include "pair_tiles.cuh"
#include "rpy_wall.cuh"

namespace mb {
namespace {

#ifndef MB_PAIR_NT
#define MB_PAIR_NT 256
#endif
#ifndef MB_PAIR_TPT
#define MB_PAIR_TPT 1
#endif
constexpr int kNT = MB_PAIR_NT;   // threads per CTA = sources per shared tile
constexpr double kPi = 3.14159265358979323846;

// Coordinates as unsigned integers in the order of the floats (for min/max).
__device__ __forceinline__ unsigned float_order(float x)
{
    const unsigned u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float order_float(unsigned u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Block-wide min of v[0..2] and max of v[3..5] (up to 32 warps; red holds
// 6 x 32) into out[0..5]; every thread of the block must call it.
__device__ __forceinline__ void minmax_block(unsigned (&v)[6], unsigned *red, unsigned *out)
{
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned t = __shfl_xor_sync(0xffffffffu, v[c], o);
            v[c] = c < 3 ? min(v[c], t) : max(v[c], t);
        }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int c = 0; c < 6; ++c) red[6 * (threadIdx.x >> 5) + c] = v[c];
    __syncthreads();
    if (threadIdx.x < 6) {
        const int c = threadIdx.x;
        unsigned r = red[c];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            r = c < 3 ? min(r, red[6 * w + c]) : max(r, red[6 * w + c]);
        out[c] = r;
    }
    __syncthreads();
}

// Positions split into FP32 hi and lo parts.  BOX: also the CTA's bounding
// box of the hi parts (ordered integers: min x, y, z, max x, y, z) into
// part[6 blockIdx.x ..], for the spatial order.
template <bool BOX>
__global__ void __launch_bounds__(256) pack_hilo_kernel(const double *__restrict__ r, int64_t n,
                                                        float4 *__restrict__ hi,
                                                        float4 *__restrict__ lo,
                                                        unsigned *__restrict__ part)
{
    unsigned v[6] = {~0u, ~0u, ~0u, 0u, 0u, 0u};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double x = r[3 * i], y = r[3 * i + 1], z = r[3 * i + 2];
        const float xh = (float)x, yh = (float)y, zh = (float)z;
        hi[i] = make_float4(xh, yh, zh, 0.f);
        lo[i] = make_float4((float)(x - (double)xh), (float)(y - (double)yh),
                            (float)(z - (double)zh), 0.f);
        if (BOX) {
            const unsigned o[3] = {float_order(xh), float_order(yh), float_order(zh)};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[c] = min(v[c], o[c]);
                v[3 + c] = max(v[3 + c], o[c]);
            }
        }
    }
    if (BOX) {
        __shared__ unsigned red[6 * 32], box[6];
        minmax_block(v, red, box);
        if (threadIdx.x < 6) part[6 * blockIdx.x + threadIdx.x] = box[threadIdx.x];
    }
}

template <bool WALL, int TPT>
__global__ void __launch_bounds__(kNT) pair_f32_kernel(
    const float4 *__restrict__ hi, const float4 *__restrict__ lo, const double *__restrict__ f,
    int64_t n, int64_t chunk, int n_tblocks, int64_t n_items, MobConsts<float> k,
    double *__restrict__ out, double scale, int direct)
{
    __shared__ float4 sA[kNT];  // (x_hi, y_hi, z_hi, f_x)
    __shared__ float4 sB[kNT];  // (x_lo, y_lo, z_lo, f_y)
    __shared__ float sC[kNT];   // f_z

    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int tb = (int)(item % n_tblocks);
        const int64_t sc = item / n_tblocks;
        float xh[TPT], yh[TPT], zh[TPT], xl[TPT], yl[TPT], zl[TPT];
        float sx[TPT], sy[TPT], sz[TPT], cx[TPT], cy[TPT], cz[TPT];
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            int64_t i = (int64_t)tb * kNT * TPT + t * kNT + threadIdx.x;
            i = i < n ? i : n - 1;
            const float4 h = hi[i], l = lo[i];
            xh[t] = h.x; yh[t] = h.y; zh[t] = h.z;
            xl[t] = l.x; yl[t] = l.y; zl[t] = l.z;
            sx[t] = sy[t] = sz[t] = cx[t] = cy[t] = cz[t] = 0.f;
        }
        const int64_t j_begin = sc * chunk;
        const int64_t j_end = j_begin + chunk < n ? j_begin + chunk : n;
        for (int64_t jt = j_begin; jt < j_end; jt += kNT) {
            __syncthreads();
            {
                const int64_t j = jt + threadIdx.x;
                const bool valid = j < j_end;
                const int64_t jc = valid ? j : j_begin;
                const float4 h = hi[jc], l = lo[jc];
                const float fx = valid ? (float)f[3 * jc] : 0.f;
                const float fy = valid ? (float)f[3 * jc + 1] : 0.f;
                const float fz = valid ? (float)f[3 * jc + 2] : 0.f;
                sA[threadIdx.x] = make_float4(h.x, h.y, h.z, fx);
                sB[threadIdx.x] = make_float4(l.x, l.y, l.z, fy);
                sC[threadIdx.x] = fz;
            }
            __syncthreads();
            float ax[TPT], ay[TPT], az[TPT];
#pragma unroll
            for (int t = 0; t < TPT; ++t) ax[t] = ay[t] = az[t] = 0.f;
#pragma unroll 4
            for (int s = 0; s < kNT; ++s) {
                const float4 A = sA[s];
                const float4 B = sB[s];
                const float fz = sC[s];
#pragma unroll
                for (int t = 0; t < TPT; ++t) {
                    const float dx = (xh[t] - A.x) + (xl[t] - B.x);
                    const float dy = (yh[t] - A.y) + (yl[t] - B.y);
                    const float dz = (zh[t] - A.z) + (zl[t] - B.z);
                    const Mob<float> m = mob_coefs<WALL>(dx, dy, dz, zh[t], A.z, k);
                    mob_apply<WALL>(m, dx, dy, dz, A.w, B.w, fz, ax[t], ay[t], az[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < TPT; ++t) {
                kahan_add(sx[t], cx[t], ax[t]);
                kahan_add(sy[t], cy[t], ay[t]);
                kahan_add(sz[t], cz[t], az[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            const int64_t i = (int64_t)tb * kNT * TPT + t * kNT + threadIdx.x;
            if (i < n) {
                const double vx = (double)sx[t] - (double)cx[t];
                const double vy = (double)sy[t] - (double)cy[t];
                const double vz = (double)sz[t] - (double)cz[t];
                double *o = direct ? out + 3 * i : out + 3 * (sc * n + i);
                const double m = direct ? scale : 1.0;
                o[0] = m * vx;
                o[1] = m * vy;
                o[2] = m * vz;
            }
        }
    }
}

// Packed FP32 kernel (paired f32x2 arithmetic, 2*NP targets per thread): a
// persistent loop over (target block, source chunk) items; see x2_item.
template <bool WALL, int NP, int NT = kNT>
__global__ void __launch_bounds__(NT, NT == kNT ? (NP == 1 ? 3 : 2) : 16) pair_f32x2_kernel(
    const float4 *__restrict__ hi, const float4 *__restrict__ lo, const double *__restrict__ f,
    int64_t n, int64_t chunk, int n_tblocks, int64_t n_items, MobConsts2 k,
    double *__restrict__ out, double scale, int direct)
{
    __shared__ float4 sP[kX2SmemFloat4PerSource * NT];
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int tb = (int)(item % n_tblocks);
        const int64_t sc = item / n_tblocks;
        const int64_t j_begin = sc * chunk;
        const int64_t j_end = j_begin + chunk < n ? j_begin + chunk : n;
        x2_item<WALL, NP, NT>(sP, hi, lo, n, hi, lo, f, tb, j_begin, j_end, k,
                              direct ? out : out + 3 * sc * n, direct ? scale : 1.0);
    }
}

// Symmetric packed kernel over the upper-triangular pairs of blocks of 2 NT
// blobs; an item is block I against half of block J (x2sym_item), one CTA
// each.  Bound by the FMA pipe once every SM has work, so the items are cut to
// leave no SM idle: smaller blocks for fewer blobs, and more items than fit at
// once, dealt out by the hardware as CTAs end (a persistent grid that strides
// over them ends 6-9% later: items differ by a factor of 1.3 in length).
// Times (us) of a product with the wall, NT = 32 / 64 / 128 / 256:
//    1,000 blobs  21 / 25 / 34 / 74        9,003   142 / 136 / 144 / 183
//    3,000        31 / 31 / 43 / 74       20,011   625 / 590 / 591 / 621
//    7,000        94 / 93 / 102 / 129     65,536  8290 / 5376 / 5207 / 5235
// (blocks of 512 in a persistent grid, the form before: 242 us at 9,003 blobs
// and 5,555 at 65,536).
//
// box (optional): the bounding box of every kBoxBlobs sorted blobs, (min x, y,
// z, max x, y, z), and grid->far2, the squared distance beyond which a block
// pair is far (see x2sym_item); such pairs take the kFar instance, and the
// kVeryFar one from kVeryFarRadii radii on.
// Blocks of 64 and 128 blobs fold their FP32 sums every 16 steps, and all but those
// of 128 with the wall round each term once (x2sym_item): they stand where packed
// kernels summed chunks of 16 to 32 sources, and whole blocks' sums were up to 1.6
// times as far off.  Relative L2 error of 6,480 blobs in shells of 162, whole /
// folded (the packed kernel): 2.4e-7 / 1.8e-7 (1.9e-7) with the wall, 2.3e-7 /
// 1.3e-7 (1.4e-7) without; 2,100 blobs in shells of 42 without 1.35e-7 / 1.15e-7
// (1.25e-7).  9,003 blobs 134 -> 136 us with the wall, 76 -> 87 without.
constexpr int kBoxBlobs = 256;
constexpr int kSymBoxNT = kBoxBlobs / 2;  // the only blocks that come sorted: one a box
constexpr int64_t kSymNT64MinN = 4096, kSymNT128MinN = 12000;

struct SortGrid {
    float lo[3], inv_h[3];  // cell of x: (x - lo) * inv_h per axis
    int bits[3];            // bits of the cell index per axis (nbits in all)
    float far2;             // squared box distance of a far block pair
};

template <bool WALL, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) pair_sym_kernel(
    const float4 *__restrict__ hi, const float4 *__restrict__ lo, const double *__restrict__ f,
    int64_t n, int64_t n_items, MobConsts2 k, double *__restrict__ u, double scale,
    const float *__restrict__ box, const SortGrid *__restrict__ grid)
{
    __shared__ float4 sP[kX2SmemFloat4PerSource * NT];
    __shared__ float sRev[3 * NT * (NT / 32)];
    float far2 = 0.f, vfar2 = 0.f;
    if (NT == kSymBoxNT && box) {
        far2 = fmaxf(grid->far2, 1.5625f * k.four_a2);
        vfar2 = 0.25f * kVeryFarRadii * kVeryFarRadii * k.four_a2;
    }
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        int64_t I, J;
        triangle_pair(item >> 1, I, J);
        const int half = (int)(item & 1);
        if constexpr (NT == kSymBoxNT) {
            int level = kNear;  // the same in every thread
            if (box && I != J) {
                const float *bi = box + 6 * I, *bj = box + 6 * J;
                float d2 = 0.f;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float g = fmaxf(fmaxf(bj[c] - bi[3 + c], bi[c] - bj[3 + c]), 0.f);
                    d2 = fmaf(g, g, d2);
                }
                if (d2 > far2) level = d2 > vfar2 ? kVeryFar : kFar;
            }
            if (level == kVeryFar) {
                x2sym_item<WALL, NT, kVeryFar>(sP, sRev, hi, lo, f, n, I, J, k, u, scale, half);
                continue;
            }
            if (level == kFar) {
                x2sym_item<WALL, NT, kFar>(sP, sRev, hi, lo, f, n, I, J, k, u, scale, half);
                continue;
            }
        }
        x2sym_item<WALL, NT, kNear>(sP, sRev, hi, lo, f, n, I, J, k, u, scale, half);
    }
}

// A whole FP32 product of a few hundred blobs in one launch: a cluster of
// kSmallCluster CTAs per block of 64 targets, each of its warps taking a share
// of the sources (at most 32) straight from the caller's FP64 arrays, and the
// warps' sums meeting in distributed shared memory.  Such a product is bound by
// its launches, not by arithmetic: packed positions, one-warp CTAs and a
// reduction were three (336 blobs, a pass: 32.6 -> 29.4 us).  u must not
// overlap r or f.
constexpr int kSmallCluster = 8, kSmallWarps = 4;
constexpr int64_t kSmallMaxN = 32 * kSmallCluster * kSmallWarps;

template <bool WALL>
__global__ void __cluster_dims__(kSmallCluster, 1, 1) __launch_bounds__(32 * kSmallWarps)
    pair_small_kernel(const double *__restrict__ r, const double *__restrict__ f, int n, MobConsts2 k,
                      double *__restrict__ u, double scale)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ float4 sP[kSmallWarps][kX2SmemFloat4PerSource * 32];
    __shared__ float part[kSmallWarps][3 * 64];
    __shared__ double tot[3 * 64];
    const int rank = (int)cluster.block_rank(), tb = blockIdx.x / kSmallCluster;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chunk = (n + kSmallCluster * kSmallWarps - 1) / (kSmallCluster * kSmallWarps);
    const int j0 = (rank * kSmallWarps + warp) * chunk, cnt = max(0, min(chunk, n - j0));
    auto split = [&](int i, float4 &h, float4 &l) {
        const double x = r[3 * i], y = r[3 * i + 1], z = r[3 * i + 2];
        h = make_float4((float)x, (float)y, (float)z, 0.f);
        l = make_float4((float)(x - (double)h.x), (float)(y - (double)h.y), (float)(z - (double)h.z), 0.f);
    };
    float4 h[2], l[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) split(min(64 * tb + 32 * t + lane, n - 1), h[t], l[t]);
    if (lane < cnt) {
        float4 hj, lj;
        const int j = j0 + lane;
        split(j, hj, lj);
        stage_x2(sP[warp] + kX2SmemFloat4PerSource * lane, hj, lj, (float)f[3 * j],
                 (float)f[3 * j + 1], (float)f[3 * j + 2]);
    }
    __syncwarp();
    const float2 xh = make_float2(h[0].x, h[1].x), xl = make_float2(l[0].x, l[1].x);
    const float2 yh = make_float2(h[0].y, h[1].y), yl = make_float2(l[0].y, l[1].y);
    const float2 zh = make_float2(h[0].z, h[1].z), zl = make_float2(l[0].z, l[1].z);
    float2 ax = make_float2(0.f, 0.f), ay = ax, az = ax;
#pragma unroll 2
    for (int s = 0; s < cnt; ++s) {
        const float4 *Q = sP[warp] + kX2SmemFloat4PerSource * s;
        const float4 P0 = Q[0], P1 = Q[1], P2 = Q[2], P3 = Q[3], P4 = Q[4];
        const float2 zj = make_float2(P1.x, P1.y);
        const float2 dx = add2(add2(xh, make_float2(P0.x, P0.y)), add2(xl, make_float2(P2.x, P2.y)));
        const float2 dy = add2(add2(yh, make_float2(P0.z, P0.w)), add2(yl, make_float2(P2.z, P2.w)));
        const float2 dz = add2(fma2(zj, k.m1, zh), add2(zl, make_float2(P3.x, P3.y)));
        const float2 dxy2 = fma2(dy, dy, fma2(dx, dx, k.tiny));
        const Mob<float2> m = mob_coefs2<WALL, kNear>(dz, dxy2, zh, zj, make_float2(P1.z, P1.w), k);
        mob_apply2<WALL, false, true>(m, dx, dy, dz, make_float2(P3.z, P3.w),
                                      make_float2(P4.x, P4.y), make_float2(P4.z, P4.w), ax, ay, az);
    }
    const float2 a[3] = {ax, ay, az};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        part[warp][3 * lane + c] = a[c].x;
        part[warp][3 * (32 + lane) + c] = a[c].y;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * 64; e += blockDim.x) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < kSmallWarps; ++w) v += (double)part[w][e];
        tot[e] = v;
    }
    cluster.sync();
    constexpr int kShare = 3 * 64 / kSmallCluster;
    const int e = rank * kShare + threadIdx.x;
    if (threadIdx.x < kShare && 64 * tb + e / 3 < n) {
        double v = 0.0;
#pragma unroll
        for (int b = 0; b < kSmallCluster; ++b) v += cluster.map_shared_rank(tot, b)[e];
        u[3 * 64 * (int64_t)tb + e] = scale * v;
    }
    cluster.sync();  // no CTA ends while another reads its sums
}

template <bool WALL>
void launch_small(const double *r, const double *f, int64_t n, double a, double *u, double scale,
                  cudaStream_t s)
{
    pair_small_kernel<WALL><<<(unsigned)(kSmallCluster * ceil_div(n, 64)), 32 * kSmallWarps, 0, s>>>(
        r, f, (int)n, MobConsts2::make(a), u, scale);
    count_launch();
}

// FP64 kernel: one warp per CTA and item, an item being a block of 32
// targets against C sources of a block at or after it (f64sym_item).  The
// FP64 pipe (one instruction per ~19 cycles and SM) is the only resource in
// use, so a warp or two per scheduler keep it busy and what matters is that
// every scheduler gets the same number of pair steps: the items are far more
// than the warps in flight and the hardware deals them out as CTAs end.
// launch_f64sym picks C.  2,730 blobs: 1,274 -> 619 us against every ordered
// pair once in one-warp CTAs; 16,384 blobs: 28.3 -> 20.6 ms against 256-thread
// symmetric items of the ungrouped formula (1.41 TFLOP/s in the method's 108
// flop per ordered pair, of 1.06 measured: each pair is evaluated once).
// u: S arrays of 3 n (f64_sums), block J's items adding to the targets in array
// J mod S and block I's to the sources in array I mod S.
template <bool WALL, int C>
__global__ void __launch_bounds__(32) pair_f64sym_kernel(
    const double *__restrict__ r, const double *__restrict__ f, int64_t n, int64_t n_items,
    MobConsts<double> k, double *u, int S, double scale)
{
    __shared__ double sm[6 * C];
    constexpr int kParts = 32 / C;
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int64_t t = item / kParts;
        int64_t I, J;
        triangle_pair(t, I, J);
        const int64_t j0 = J * 32 + (item - t * kParts) * C;
        if (j0 < n)
            f64sym_item<WALL, C>(sm, r, f, n, I, j0, I == J, k, u + 3 * n * (J % S),
                                 u + 3 * n * (I % S), scale);
        __syncwarp();  // the item is done with sm
    }
}

// Flow evaluation at points other than the blobs (targets != sources): one
// packed FP32 (2 NT targets) or FP64 (32 targets, one warp) item of a target
// block against a source chunk per CTA, partials reduced like the matvec's.
// The targets are tracers of the blob radius a (Appendix B renders flows with
// small blobs of radius a').  Bound by the FMA or the FP64 pipe; the chunks
// (eval_plan) give every SM several items whatever the number of points, where
// chunks of 512 sources and blocks of 512 or 256 points left most idle.
// With the wall (us): 3,072 points and 6,720 blobs 135 -> 78 in FP32 and 6,360
// -> 2,890 in FP64, 100 points 133 -> 26 and 3,180 -> 145, 65,536 points and
// blobs 11,200 -> 10,270 in FP32.
template <bool WALL, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) eval_f32x2_kernel(
    const float4 *__restrict__ thi, const float4 *__restrict__ tlo, int64_t nt,
    const float4 *__restrict__ hi, const float4 *__restrict__ lo, const double *__restrict__ f,
    int64_t ns, int64_t chunk, int n_tblocks, int64_t n_items, MobConsts2 k,
    double *__restrict__ out, double scale, int direct)
{
    __shared__ float4 sP[kX2SmemFloat4PerSource * NT];
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int tb = (int)(item % n_tblocks);
        const int64_t sc = item / n_tblocks;
        const int64_t j_begin = sc * chunk;
        const int64_t j_end = j_begin + chunk < ns ? j_begin + chunk : ns;
        x2_item<WALL, 1, NT>(sP, thi, tlo, nt, hi, lo, f, tb, j_begin, j_end, k,
                             direct ? out : out + 3 * sc * nt, direct ? scale : 1.0);
    }
}

template <bool WALL>
__global__ void __launch_bounds__(32) eval_f64_kernel(
    const double *__restrict__ x, int64_t nt, const double *__restrict__ r,
    const double *__restrict__ f, int64_t ns, int64_t chunk, int n_tblocks, int64_t n_items,
    MobConsts<double> k, double *__restrict__ out, double scale, int direct)
{
    __shared__ double sm[6 * 32];
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int tb = (int)(item % n_tblocks);
        const int64_t sc = item / n_tblocks;
        const int64_t j_begin = sc * chunk;
        const int64_t j_end = j_begin + chunk < ns ? j_begin + chunk : ns;
        f64_item<WALL, 32>(sm, x, nt, r, f, tb, j_begin, j_end, k,
                           direct ? out : out + 3 * sc * nt, direct ? scale : 1.0);
    }
}

// Appendix B: each blob i becomes n_sub blobs at r_i + off_k carrying
// lambda_i / n_sub each (k fastest).
__global__ void refine_blobs_kernel(const double *__restrict__ r, const double *__restrict__ lam,
                                    int64_t n, const double *__restrict__ off, int n_sub,
                                    double *__restrict__ rs, double *__restrict__ ls)
{
    const double w = 1.0 / n_sub;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * n_sub;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / n_sub;
        const int k = (int)(e % n_sub);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            rs[3 * e + c] = r[3 * i + c] + off[3 * k + c];
            ls[3 * e + c] = lam[3 * i + c] * w;
        }
    }
}

// Double-float, forward only, for the smallest problems: 32 targets (one per
// lane) against source chunks of 16, two sources at once in the halves of the
// packed arithmetic, every ordered pair evaluated; the chunk's sums are added
// to u (zeroed) with FP64 atomics.  Twice the pair evaluations of the symmetric
// kernel, in several times as many one-warp CTAs with a quarter of the steps.
constexpr int kDfxChunk = 16;

template <bool WALL>
__global__ void __launch_bounds__(32) pair_dfx_kernel(
    const float4 *__restrict__ hi, const float4 *__restrict__ lo, const double *__restrict__ f,
    int64_t n, MobConstsDf k, double *__restrict__ u, double scale)
{
    // source pair p: x, y, z, fx, fy, fz, -2 z^2, each (hi, hi', lo, lo')
    __shared__ float4 sD[7 * kDfxChunk / 2];
    const int lane = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane, ic = i < n ? i : n - 1;
    const int64_t j0 = (int64_t)blockIdx.y * kDfxChunk;
    const float4 th = hi[ic], tl = lo[ic];
    const dfl2 xi(dfl(th.x, tl.x)), yi(dfl(th.y, tl.y)), zi(dfl(th.z, tl.z));
    if (lane < kDfxChunk) {
        const int64_t j = j0 + lane, jc = j < n ? j : n - 1;
        const float4 h = hi[jc], l = lo[jc];
        const double z = (double)h.z + (double)l.z;
        const dfl v[7] = {dfl(h.x, l.x), dfl(h.y, l.y), dfl(h.z, l.z),
                          j < n ? dfl(f[3 * jc]) : dfl(), j < n ? dfl(f[3 * jc + 1]) : dfl(),
                          j < n ? dfl(f[3 * jc + 2]) : dfl(), dfl(-2.0 * z * z)};
        float *d = (float *)sD + 4 * 7 * (lane >> 1) + (lane & 1);
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            d[4 * c] = v[c].hi;
            d[4 * c + 2] = v[c].lo;
        }
    }
    __syncwarp();
    auto src = [&](int p, int c) {
        const float4 q = sD[7 * p + c];
        return dfl2(make_float2(q.x, q.y), make_float2(q.z, q.w));
    };
    dfl2 ux, uy, uz;
#pragma unroll 1
    for (int p = 0; p < kDfxChunk / 2; ++p) {
        const dfl2 zj = src(p, 2);
        const dfl2 dx = xi - src(p, 0), dy = yi - src(p, 1), dz = zi - zj;
        const Mob<dfl2> m = mob_coefs_df<WALL, false>(dx, dy, dz, zi, zj, src(p, 6), k);
        mob_apply_df<WALL>(m, dx, dy, dz, src(p, 3), src(p, 4), src(p, 5), ux, uy, uz);
    }
    if (i < n) {
        atomicAdd(u + 3 * i, scale * sum_halves(ux));
        atomicAdd(u + 3 * i + 1, scale * sum_halves(uy));
        atomicAdd(u + 3 * i + 2, scale * sum_halves(uz));
    }
}

// Double-float kernel: symmetric over the upper-triangular pairs of blocks of
// 2 NT blobs, an item being block I against half of block J (dfsym_item), one
// CTA each as in pair_sym_kernel.  Bound by the FMA pipe (a pair takes about
// 600 FP32 operations): packed two targets to an instruction it no longer
// waits for the issue of instructions as the scalar form did, and twelve warps
// an SM (168 registers a thread) are enough.
// Times (us) of a product with the wall, forward only / NT = 32 / NT = 128,
// and of the scalar form before:
//    336 blobs  20 / 43 / 127, 23       9,003   - / 823 / 895, 1,222
//    1,000      37 / 45 / 125, 39      20,011   - / 3,771 / 3,830, 5,287
//    1,400      53 / 43 / 124, 50      65,536   - / 38,600 / 38,100, 50,050
constexpr int64_t kDfxMaxN = 1100;       // up to this the product is forward only
constexpr int64_t kDfNT128MinN = 24000;

// box (optional, spatial order): the bounding boxes of every kBoxBlobs sorted
// blobs; block pairs whose boxes are 64 a or more apart take the FAR instance
// of the item.
template <bool WALL, int NT>
__global__ void __launch_bounds__(NT, 384 / NT) pair_df_kernel(
    const float4 *__restrict__ hi, const float4 *__restrict__ lo, const double *__restrict__ f,
    int64_t n, int64_t n_items, MobConstsDf k, double *__restrict__ u, double scale,
    const float *__restrict__ box, float far2)
{
    __shared__ float4 sD[7 * NT];
    __shared__ double sRev[3 * NT * (NT / 32)];
    constexpr int kPer = kBoxBlobs / (2 * NT);  // this kernel's blocks per box
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        int64_t I, J;
        triangle_pair(item >> 1, I, J);
        bool far = false;
        if (box && I / kPer != J / kPer) {
            const float *bi = box + 6 * (I / kPer), *bj = box + 6 * (J / kPer);
            float d2 = 0.f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float g = fmaxf(fmaxf(bj[c] - bi[3 + c], bi[c] - bj[3 + c]), 0.f);
                d2 = fmaf(g, g, d2);
            }
            far = d2 > far2;  // the same in every thread
        }
        const int half = (int)(item & 1);
        if (far) dfsym_item<WALL, NT, true>(sD, sRev, hi, lo, f, n, I, J, half, k, u, scale);
        else dfsym_item<WALL, NT, false>(sD, sRev, hi, lo, f, n, I, J, half, k, u, scale);
        __syncthreads();  // the item is done with sRev
    }
}

// u_i = scale * sum_s partial[s][i] in a fixed order: 32 entries a CTA, eight
// warps summing every eighth chunk of them, then one adding the eight sums (a
// thread that walked all chunks by itself would wait for each load in turn).
constexpr int kReduceWarps = 8;

__global__ void __launch_bounds__(32 * kReduceWarps) reduce_partials_kernel(
    const double *__restrict__ partial, int64_t n, int S, double scale, double *__restrict__ u)
{
    __shared__ double sum[kReduceWarps][32];
    const int64_t m = 3 * n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t e0 = blockIdx.x * (int64_t)32; e0 < m; e0 += (int64_t)gridDim.x * 32) {
        double acc = 0.0;
        if (e0 + lane < m)
#pragma unroll 4
            for (int s = warp; s < S; s += kReduceWarps) acc += partial[s * m + e0 + lane];
        sum[warp][lane] = acc;
        __syncthreads();
        if (warp == 0 && e0 + lane < m) {
#pragma unroll
            for (int w = 1; w < kReduceWarps; ++w) acc += sum[w][lane];
            u[e0 + lane] = scale * acc;
        }
        __syncthreads();
    }
}

void launch_reduce_partials(const double *partial, int64_t n, int S, double scale, double *u,
                            cudaStream_t s)
{
    reduce_partials_kernel<<<(int)std::min<int64_t>(ceil_div(3 * n, 32), 65535), 32 * kReduceWarps, 0,
                             s>>>(partial, n, S, scale, u);
    count_launch();
}

struct Plan {
    int n_tblocks = 0;
    int S = 1;
    int64_t chunk = 0;
    int64_t items = 0;
    int grid = 0;
};

// Split sources into S chunks so that the items fill whole waves of the
// resident grid as evenly as possible, with chunks of at least two tiles.
Plan make_plan(int64_t n, int targets_per_cta, int resident, int64_t s_cap = 64, int tile = kNT,
               int64_t min_chunk = 2 * kNT)
{
    const int64_t ns = n;
    Plan p;
    p.n_tblocks = (int)ceil_div(n, targets_per_cta);
    const int64_t max_s = std::max<int64_t>(1, std::min<int64_t>(s_cap, ceil_div(ns, min_chunk)));
    double best = -1.0;
    for (int64_t s = 1; s <= max_s; ++s) {
        const int64_t chunk = ceil_div(ceil_div(ns, s), tile) * tile;
        const int64_t s_eff = ceil_div(ns, chunk);
        const int64_t items = (int64_t)p.n_tblocks * s_eff;
        const int64_t waves = ceil_div(items, resident);
        double eff = (double)items / (double)(waves * resident);
        // a small preference for fewer chunks (less partial traffic)
        eff -= 1e-3 * (double)s_eff / 64.0;
        if (items < resident) eff *= (double)items / resident;
        if (eff > best + 1e-9) {
            best = eff;
            p.S = (int)s_eff;
            p.chunk = chunk;
        }
    }
    p.items = (int64_t)p.n_tblocks * p.S;
    p.grid = (int)std::min<int64_t>(p.items, resident);
    return p;
}

template <typename K>
int resident_ctas(mb_context *ctx, K kernel, int threads = kNT)
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, 0) != cudaSuccess ||
        occ < 1)
        occ = 1;
    return occ * ctx->sm_count;
}

constexpr int kTPT = MB_PAIR_TPT;  // targets per thread

}  // namespace

// ---------------------------------------------------------------------------
// FP32 variants.
//   0: scalar kernel, kTPT targets per thread
//   1: packed f32x2 kernel, 2 targets per thread
//   2: packed f32x2 kernel, 4 targets per thread
//   3: symmetric packed kernel (each unordered pair once)
//   4: packed f32x2 kernel in one-warp CTAs, 2 targets per thread
constexpr int kSmallNT = 32;        // CTA size of the small-problem kernels

int f32_targets_per_cta(int v)
{
    return v == 0 ? kNT * kTPT : (v == 2 ? 4 * kNT : (v == 4 ? 2 * kSmallNT : 2 * kNT));
}

template <bool WALL, int NT>
void launch_sym_nt(const float4 *hi, const float4 *lo, const double *f, int64_t n, double a,
                   double *u, double scale, const float *box, const SortGrid *sg, cudaStream_t s)
{
    const int64_t nb = ceil_div(n, 2 * NT), items = nb * (nb + 1);
    pair_sym_kernel<WALL, NT><<<(unsigned)std::min<int64_t>(items, 1 << 30), NT, 0, s>>>(
        hi, lo, f, n, items, MobConsts2::make(a), u, scale, box, sg);
}

template <bool WALL>
void launch_sym(const float4 *hi, const float4 *lo, const double *f, int64_t n, double a,
                double *u, double scale, const float *box, const SortGrid *sg, cudaStream_t s)
{
    if (n < kSymNT64MinN) launch_sym_nt<WALL, 32>(hi, lo, f, n, a, u, scale, box, sg, s);
    else if (n < kSymNT128MinN) launch_sym_nt<WALL, 64>(hi, lo, f, n, a, u, scale, box, sg, s);
    else launch_sym_nt<WALL, 128>(hi, lo, f, n, a, u, scale, box, sg, s);
}

// Variant 4: 64-target blocks, source chunks of 16 or more (half a tile: one
// warp per CTA walks fewer sources, more CTAs share the work).
Plan small_plan(int64_t n, int resident)
{
    return make_plan(n, f32_targets_per_cta(4), resident, 1024, kSmallNT / 2, kSmallNT / 2);
}

template <bool WALL>
int f32_resident(mb_context *ctx, int v)
{
    if (v == 0) return resident_ctas(ctx, pair_f32_kernel<WALL, kTPT>);
    if (v == 1) return resident_ctas(ctx, pair_f32x2_kernel<WALL, 1>);
    if (v == 4) return resident_ctas(ctx, pair_f32x2_kernel<WALL, 1, kSmallNT>, kSmallNT);
    return resident_ctas(ctx, pair_f32x2_kernel<WALL, 2>);
}

template <bool WALL>
void f32_launch(int v, const Plan &p, cudaStream_t s, const float4 *hi, const float4 *lo,
                const double *f, int64_t n, double a, double *out, double scale, int direct)
{
    if (v == 0) {
        pair_f32_kernel<WALL, kTPT><<<p.grid, kNT, 0, s>>>(
            hi, lo, f, n, p.chunk, p.n_tblocks, p.items, MobConsts<float>::make(a), out, scale,
            direct);
    } else if (v == 1) {
        pair_f32x2_kernel<WALL, 1><<<p.grid, kNT, 0, s>>>(
            hi, lo, f, n, p.chunk, p.n_tblocks, p.items, MobConsts2::make(a), out, scale, direct);
    } else if (v == 4) {
        pair_f32x2_kernel<WALL, 1, kSmallNT><<<p.grid, kSmallNT, 0, s>>>(
            hi, lo, f, n, p.chunk, p.n_tblocks, p.items, MobConsts2::make(a), out, scale, direct);
    } else {
        pair_f32x2_kernel<WALL, 2><<<p.grid, kNT, 0, s>>>(
            hi, lo, f, n, p.chunk, p.n_tblocks, p.items, MobConsts2::make(a), out, scale, direct);
    }
}

// ---------------------------------------------------------------------------
// Spatial order for the symmetric FP32 kernel (N >= kSortMinN).  The blobs are
// sorted by cell of a grid over their bounding box, cells in Morton order
// (kSortBits bits, dealt to the axes in proportion to their extents), by a
// counting sort; the kernel's blocks of consecutive sorted blobs are then
// compact, and the block pairs far apart take the FAR instance of the
// pair item.  Each matvec gathers f into the sorted order and scatters u back.
// The sort is stable (the blobs of a cell keep their index order), so the
// order, and with it the FP32 rounding of every pair sum, is the same on
// every call: a tile of consecutive blobs per CTA counts its keys in shared
// memory, the counts are scanned over tiles and buckets, and one warp per
// tile deals its blobs out in index order.  The grid has about N / 8 cells
// (2^10 .. 2^kSortBits): blocks of 512 blobs span a few dozen cells, and the
// per-tile count tables stay small.
constexpr int64_t kSortMinN = 16384;
static_assert(kSortMinN >= kSymNT128MinN, "sorted blobs come in blocks of kSymBoxNT");
constexpr int kSortBits = 15;         // most cell bits
constexpr int kSortKeysSmem = 16384;  // keys staged per round of the scatter

int sort_bits(int64_t n)
{
    int b = 10;  // at least 1,024 buckets (sort_scan_kernel's granule)
    while (b < kSortBits && ((int64_t)8 << b) < n) ++b;
    return b;
}

// The grid from the bounding box (ordered integers, as pack_hilo_kernel's
// partials): bits per axis by repeatedly halving the longest cell side, and
// the far distance, separations beyond 2^18 ulp of the largest coordinate.
__device__ void sort_grid_from_box(const unsigned *box, int nbits, SortGrid &g)
{
    float lo[3], ext[3], big = 0.f;
    for (int c = 0; c < 3; ++c) {
        lo[c] = order_float(box[c]);
        const float hi = order_float(box[3 + c]);
        ext[c] = fmaxf(hi - lo[c], 1e-30f);
        big = fmaxf(big, fmaxf(fabsf(lo[c]), fabsf(hi)));
    }
    int bits[3] = {0, 0, 0};
    for (int t = 0; t < nbits; ++t) {
        int a = 0;
        float best = -1.f;
        for (int c = 0; c < 3; ++c) {
            const float side = ldexpf(ext[c], -bits[c]);
            if (side > best) { best = side; a = c; }
        }
        ++bits[a];
    }
    for (int c = 0; c < 3; ++c) {
        g.lo[c] = lo[c];
        g.inv_h[c] = ldexpf(1.f, bits[c]) / ext[c];
        g.bits[c] = bits[c];
    }
    const float d = ldexpf(big, -23 + 18);
    g.far2 = d * d;
}

__device__ __forceinline__ unsigned sort_key(float4 h, const SortGrid &g)
{
    int q[3];
    const float x[3] = {h.x, h.y, h.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int top = (1 << g.bits[c]) - 1;
        q[c] = min(max((int)((x[c] - g.lo[c]) * g.inv_h[c]), 0), top);
    }
    unsigned key = 0;
    for (int l = kSortBits - 1; l >= 0; --l)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (g.bits[c] > l) key = (key << 1) | ((q[c] >> l) & 1);
    return key;
}

// tile b = blobs b T .. min(n, (b + 1) T) - 1: keys, and their counts per bucket
// (B = 2^nbits) in row b of H.  Every CTA first reduces the nparts
// bounding-box partials and forms the grid (CTA 0 also stores it for the
// pair kernel).
__global__ void __launch_bounds__(1024) sort_hist_kernel(const float4 *__restrict__ hi, int64_t n,
                                                         int64_t T, const unsigned *__restrict__ part,
                                                         int nparts, int nbits,
                                                         SortGrid *__restrict__ grid,
                                                         unsigned *__restrict__ key,
                                                         int *__restrict__ H)
{
    extern __shared__ int hist[];
    __shared__ unsigned red[6 * 32], box[6];
    __shared__ SortGrid gs;
    const int B = 1 << nbits;
    unsigned v[6] = {~0u, ~0u, ~0u, 0u, 0u, 0u};
    for (int b = threadIdx.x; b < nparts; b += blockDim.x)
#pragma unroll
        for (int c = 0; c < 6; ++c)
            v[c] = c < 3 ? min(v[c], part[6 * b + c]) : max(v[c], part[6 * b + c]);
    minmax_block(v, red, box);
    if (threadIdx.x == 0) {
        sort_grid_from_box(box, nbits, gs);
        if (blockIdx.x == 0) *grid = gs;
    }
    for (int c = threadIdx.x; c < B; c += blockDim.x) hist[c] = 0;
    __syncthreads();
    const SortGrid g = gs;
    const int64_t i0 = blockIdx.x * T, i1 = min(n, i0 + T);
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const unsigned k = sort_key(hi[i], g);
        key[i] = k;
        atomicAdd(hist + k, 1);
    }
    __syncthreads();
    int *row = H + blockIdx.x * (int64_t)B;
    for (int c = threadIdx.x; c < B; c += blockDim.x) row[c] = hist[c];
}

// per bucket (one thread each): rows 0..tiles-1 of H become the exclusive
// prefix over tiles, row `tiles` the bucket's total (the loads of up to 32
// tiles in flight at once)
__global__ void __launch_bounds__(256) sort_tile_scan_kernel(int *__restrict__ H, int tiles, int B)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= B) return;
    int run = 0;
    for (int b0 = 0; b0 < tiles; b0 += 32) {
        int t[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) t[u] = b0 + u < tiles ? H[(b0 + u) * (int64_t)B + c] : 0;
#pragma unroll
        for (int u = 0; u < 32; ++u)
            if (b0 + u < tiles) {
                H[(b0 + u) * (int64_t)B + c] = run;
                run += t[u];
            }
    }
    H[tiles * (int64_t)B + c] = run;
}

// exclusive scan of the B counters in one CTA of 1024 threads: the counters
// staged in shared memory (coalesced; one pad word per 32 so that thread t's
// run of B / 1024 consecutive counters is free of bank conflicts), a
// sequential sum per thread, a scan of the 1024 sums, the prefixes written
// back through shared memory
__device__ __forceinline__ int scan_pad(int e) { return e + (e >> 5); }

__global__ void __launch_bounds__(1024) sort_scan_kernel(int *__restrict__ count, int B)
{
    extern __shared__ int sc[];
    __shared__ int wsum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = B >> 10;  // B is a power of two >= 1024
    for (int e = threadIdx.x; e < B; e += 1024) sc[scan_pad(e)] = count[e];
    __syncthreads();
    const int e0 = threadIdx.x * per;
    int tot = 0;
    for (int k = 0; k < per; ++k) tot += sc[scan_pad(e0 + k)];
    int x = tot;  // inclusive scan of the per-thread sums
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int y = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += t;
        }
        wsum[lane] = y;
    }
    __syncthreads();
    int run = (warp > 0 ? wsum[warp - 1] : 0) + x - tot;
    for (int k = 0; k < per; ++k) {
        const int v = sc[scan_pad(e0 + k)];
        sc[scan_pad(e0 + k)] = run;
        run += v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < B; e += 1024) count[e] = sc[scan_pad(e)];
}

// perm[position] = blob.  Tile b's first position in bucket k is start[k] +
// H[b][k]; warp 0 takes the tile's keys 32 at a time in index order, ranks
// equal keys among its lanes (match), and advances the bucket's offset in
// shared memory once per group.
__global__ void __launch_bounds__(1024) sort_scatter_kernel(const unsigned *__restrict__ key,
                                                            int64_t n, int64_t T,
                                                            const int *__restrict__ H, int tiles,
                                                            int B, int *__restrict__ perm)
{
    extern __shared__ int off[];
    unsigned *sk = (unsigned *)(off + B);
    const int *row = H + blockIdx.x * (int64_t)B;
    const int *start = H + tiles * (int64_t)B;
    for (int c = threadIdx.x; c < B; c += blockDim.x) off[c] = start[c] + row[c];
    const int64_t i0 = blockIdx.x * T, i1 = min(n, i0 + T);
    for (int64_t c0 = i0; c0 < i1; c0 += kSortKeysSmem) {
        const int m = (int)min((int64_t)kSortKeysSmem, i1 - c0);
        __syncthreads();  // offsets written; warp 0 done with the previous round's keys
        for (int e = threadIdx.x; e < m; e += blockDim.x) sk[e] = key[c0 + e];
        __syncthreads();
        if (threadIdx.x < 32) {
            // the leader of each group of equal keys reads and advances the
            // bucket's offset and hands the base to its group; the next
            // chunk's key is loaded one round ahead
            const unsigned lane = threadIdx.x;
            unsigned k_next = (int)lane < m ? sk[lane] : 0xffffffffu;  // no bucket has this key
            for (int e0 = 0; e0 < m; e0 += 32) {
                const int e = e0 + (int)lane;
                const bool ok = e < m;
                const unsigned k = k_next;
                k_next = e + 32 < m ? sk[e + 32] : 0xffffffffu;
                const unsigned same = __match_any_sync(0xffffffffu, k);
                const int leader = __ffs(same) - 1;
                int base = 0;
                if (ok && (int)lane == leader) {
                    base = off[k];
                    off[k] = base + __popc(same);
                }
                base = __shfl_sync(0xffffffffu, base, leader);
                if (ok) perm[base + __popc(same & ((1u << lane) - 1u))] = (int)(c0 + e);
                __syncwarp();  // this round's offsets before the next round's reads
            }
        }
    }
}

// Sorted positions b kBoxBlobs .. + kBoxBlobs - 1, one CTA each: the packed
// positions in the sorted order, and their bounding box (min x, y, z, max x,
// y, z).
__global__ void __launch_bounds__(256) sort_pack_box_kernel(const int *__restrict__ perm, int64_t n,
                                                            const float4 *__restrict__ hi,
                                                            const float4 *__restrict__ lo,
                                                            float4 *__restrict__ shi,
                                                            float4 *__restrict__ slo,
                                                            float *__restrict__ box)
{
    __shared__ float red[32][6];
    const int64_t b = blockIdx.x;
    float v[6] = {3e38f, 3e38f, 3e38f, -3e38f, -3e38f, -3e38f};
    for (int64_t i = b * kBoxBlobs + threadIdx.x; i < n && i < (b + 1) * kBoxBlobs;
         i += blockDim.x) {
        const int j = perm[i];
        const float4 h = hi[j];
        shi[i] = h;
        slo[i] = lo[j];
        v[0] = fminf(v[0], h.x); v[1] = fminf(v[1], h.y); v[2] = fminf(v[2], h.z);
        v[3] = fmaxf(v[3], h.x); v[4] = fmaxf(v[4], h.y); v[5] = fmaxf(v[5], h.z);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float t = __shfl_xor_sync(0xffffffffu, v[c], o);
            v[c] = c < 3 ? fminf(v[c], t) : fmaxf(v[c], t);
        }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int c = 0; c < 6; ++c) red[threadIdx.x >> 5][c] = v[c];
    __syncthreads();
    if (threadIdx.x < 6) {
        float r = red[0][threadIdx.x];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            r = threadIdx.x < 3 ? fminf(r, red[w][threadIdx.x]) : fmaxf(r, red[w][threadIdx.x]);
        box[6 * b + threadIdx.x] = r;
    }
}

// f into the sorted order, and the sorted velocities zeroed (the pair
// kernel adds into them)
__global__ void __launch_bounds__(256) sort_gather_kernel(const int *__restrict__ perm, int64_t n,
                                                          const double *__restrict__ f,
                                                          double *__restrict__ fs,
                                                          double *__restrict__ us)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = perm[i];
        fs[3 * i] = f[3 * j];
        fs[3 * i + 1] = f[3 * j + 1];
        fs[3 * i + 2] = f[3 * j + 2];
        us[3 * i] = 0.0;
        us[3 * i + 1] = 0.0;
        us[3 * i + 2] = 0.0;
    }
}

__global__ void __launch_bounds__(256) sort_scatter_u_kernel(const int *__restrict__ perm,
                                                             int64_t n,
                                                             const double *__restrict__ us,
                                                             double *__restrict__ u)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = perm[i];
        u[3 * j] = us[3 * i];
        u[3 * j + 1] = us[3 * i + 1];
        u[3 * j + 2] = us[3 * i + 2];
    }
}

// Arrays of a spatial order of n blobs.
struct SortBufs {
    const float4 *hi, *lo;  // packed positions
    SortGrid *grid;         // followed by pack_hilo_kernel's bounding-box partials
    unsigned *key;          // n
    int *perm;              // n
    int *H;                 // 2^sort_bits(n) (sort_tiles(n) + 1)
    float4 *shi, *slo;      // n, sorted
    float *box;             // 6 per kBoxBlobs
};

// Tiles of at least 1,024 blobs, at most one per SM.
int sort_tiles(int64_t n, int sms) { return (int)std::min<int64_t>(ceil_div(n, 1024), sms); }

unsigned *sort_parts(SortGrid *grid) { return (unsigned *)((char *)grid + sizeof(SortGrid)); }

// The order of the packed positions, for N >= kSortMinN: pack_hilo_kernel
// has left nparts bounding-box partials after the SortGrid.
cudaError_t sort_launch(const SortBufs &b, int64_t n, int nparts, int sms, cudaStream_t s)
{
    const int tiles = sort_tiles(n, sms);
    const int64_t T = ceil_div(n, tiles);
    const int nbits = sort_bits(n), B = 1 << nbits;
    const size_t hist_smem = sizeof(int) * (size_t)B;
    const size_t scan_smem = sizeof(int) * (size_t)(B + B / 32);
    const size_t scatter_smem = hist_smem + sizeof(unsigned) * kSortKeysSmem;
    cudaError_t e = cudaFuncSetAttribute(sort_hist_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hist_smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(sort_scan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)scan_smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(sort_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)scatter_smem);
    if (e != cudaSuccess) return e;
    sort_hist_kernel<<<tiles, 1024, hist_smem, s>>>(b.hi, n, T, sort_parts(b.grid), nparts, nbits,
                                                    b.grid, b.key, b.H);
    sort_tile_scan_kernel<<<(B + 255) / 256, 256, 0, s>>>(b.H, tiles, B);
    sort_scan_kernel<<<1, 1024, scan_smem, s>>>(b.H + tiles * (int64_t)B, B);
    sort_scatter_kernel<<<tiles, 1024, scatter_smem, s>>>(b.key, n, T, b.H, tiles, B, b.perm);
    sort_pack_box_kernel<<<(int)ceil_div(n, kBoxBlobs), 256, 0, s>>>(b.perm, n, b.hi, b.lo, b.shi,
                                                                     b.slo, b.box);
    count_launch(5);
    return cudaGetLastError();
}

mb_status sort_positions(mb_context *ctx, int64_t n, int nparts, cudaStream_t s)
{
    const int64_t nb = ceil_div(n, kBoxBlobs);
    MB_TRY(ensure(ctx, ctx->sort_perm, sizeof(int) * (size_t)n, "spatial order"));
    MB_TRY(ensure(ctx, ctx->sort_key, sizeof(unsigned) * (size_t)n, "spatial order"));
    MB_TRY(ensure(ctx, ctx->sort_count,
                  (sizeof(int) << sort_bits(n)) * (size_t)(sort_tiles(n, ctx->sm_count) + 1),
                  "spatial order"));
    MB_TRY(ensure(ctx, ctx->sort_hi, sizeof(float4) * (size_t)n, "spatial order"));
    MB_TRY(ensure(ctx, ctx->sort_lo, sizeof(float4) * (size_t)n, "spatial order"));
    MB_TRY(ensure(ctx, ctx->sort_box, sizeof(float) * 6 * (size_t)nb, "spatial order"));
    const SortBufs b{(const float4 *)ctx->pos_hi.ptr, (const float4 *)ctx->pos_lo.ptr,
                     (SortGrid *)ctx->sort_grid.ptr,  (unsigned *)ctx->sort_key.ptr,
                     (int *)ctx->sort_perm.ptr,       (int *)ctx->sort_count.ptr,
                     (float4 *)ctx->sort_hi.ptr,      (float4 *)ctx->sort_lo.ptr,
                     (float *)ctx->sort_box.ptr};
    MB_CUDA_TRY(ctx, sort_launch(b, n, nparts, ctx->sm_count, s));
    ctx->sorted_n = n;
    return MB_OK;
}

// One FP32 matvec with variant v (pair kernel + chunk reduction).
mb_status f32_run(mb_context *ctx, int v, const double *f, int64_t n, double a, int wall,
                  double scale, double *u, cudaStream_t s, bool profile,
                  MatvecPartials *defer = nullptr)
{
    const int res = v == 3 ? 0 : wall ? f32_resident<true>(ctx, v) : f32_resident<false>(ctx, v);
    if (v == 4) {
        const Plan p = small_plan(n, res);
        double *out = u;
        const int direct = p.S == 1;
        if (!direct) {
            MB_TRY(ensure(ctx, ctx->partial, sizeof(double) * 3 * (size_t)n * p.S, "matvec partials"));
            out = (double *)ctx->partial.ptr;
        }
        auto *ev = profile ? profile_begin(ctx, s) : nullptr;
        const float4 *hi = (const float4 *)ctx->pos_hi.ptr;
        const float4 *lo = (const float4 *)ctx->pos_lo.ptr;
        if (wall)
            f32_launch<true>(4, p, s, hi, lo, f, n, a, out, scale, direct);
        else
            f32_launch<false>(4, p, s, hi, lo, f, n, a, out, scale, direct);
        profile_end(ev, s);
        count_launch();
        MB_CUDA_TRY(ctx, cudaGetLastError());
        if (!direct) {
            if (defer) {
                *defer = MatvecPartials{out, p.S, scale};
                return MB_OK;
            }
            launch_reduce_partials(out, n, p.S, scale, u, s);
            MB_CUDA_TRY(ctx, cudaGetLastError());
        }
        return MB_OK;
    }
    if (v == 3) {
        // symmetric: zero u (or, deferred, the one partial sum the caller
        // scales), then one launch over the block-pair triangle; in the
        // spatial order when the packing made one (f gathered, u scattered
        // back)
        if (defer) {
            MB_TRY(ensure(ctx, ctx->partial, sizeof(double) * 3 * (size_t)n, "matvec partials"));
            u = (double *)ctx->partial.ptr;
            *defer = MatvecPartials{u, 1, scale};
            scale = 1.0;
        }
        const bool sorted = ctx->sorted_n == n;
        const float4 *hi = (const float4 *)(sorted ? ctx->sort_hi.ptr : ctx->pos_hi.ptr);
        const float4 *lo = (const float4 *)(sorted ? ctx->sort_lo.ptr : ctx->pos_lo.ptr);
        const float *box = sorted ? (const float *)ctx->sort_box.ptr : nullptr;
        const SortGrid *sg = sorted ? (const SortGrid *)ctx->sort_grid.ptr : nullptr;
        const double *fk = f;
        double *uk = u;
        const int gv = (int)std::min<int64_t>(ceil_div(n, 256), 8 * (int64_t)ctx->sm_count);
        if (sorted) {
            MB_TRY(ensure(ctx, ctx->sort_f, sizeof(double) * 3 * (size_t)n, "sorted forces"));
            MB_TRY(ensure(ctx, ctx->sort_u, sizeof(double) * 3 * (size_t)n, "sorted velocities"));
            sort_gather_kernel<<<gv, 256, 0, s>>>((const int *)ctx->sort_perm.ptr, n, f,
                                                  (double *)ctx->sort_f.ptr,
                                                  (double *)ctx->sort_u.ptr);
            count_launch();
            fk = (const double *)ctx->sort_f.ptr;
            uk = (double *)ctx->sort_u.ptr;
        } else {
            MB_CUDA_TRY(ctx, cudaMemsetAsync(uk, 0, sizeof(double) * 3 * (size_t)n, s));
        }
        auto *ev = profile ? profile_begin(ctx, s) : nullptr;
        if (wall) launch_sym<true>(hi, lo, fk, n, a, uk, scale, box, sg, s);
        else launch_sym<false>(hi, lo, fk, n, a, uk, scale, box, sg, s);
        profile_end(ev, s);
        count_launch();
        if (sorted) {
            sort_scatter_u_kernel<<<gv, 256, 0, s>>>((const int *)ctx->sort_perm.ptr, n, uk, u);
            count_launch();
        }
        MB_CUDA_TRY(ctx, cudaGetLastError());
        return MB_OK;
    }
    const Plan p = make_plan(n, f32_targets_per_cta(v), res);
    double *out = u;
    const int direct = p.S == 1;
    if (!direct) {
        MB_TRY(ensure(ctx, ctx->partial, sizeof(double) * 3 * (size_t)n * p.S, "matvec partials"));
        out = (double *)ctx->partial.ptr;
    }
    auto *ev = profile ? profile_begin(ctx, s) : nullptr;
    const float4 *hi = (const float4 *)ctx->pos_hi.ptr;
    const float4 *lo = (const float4 *)ctx->pos_lo.ptr;
    if (wall)
        f32_launch<true>(v, p, s, hi, lo, f, n, a, out, scale, direct);
    else
        f32_launch<false>(v, p, s, hi, lo, f, n, a, out, scale, direct);
    profile_end(ev, s);
    count_launch();
    MB_CUDA_TRY(ctx, cudaGetLastError());
    if (!direct && defer) {
        *defer = MatvecPartials{out, p.S, scale};
        return MB_OK;
    }
    if (!direct) {
        launch_reduce_partials(out, n, p.S, scale, u, s);
        MB_CUDA_TRY(ctx, cudaGetLastError());
    }
    return MB_OK;
}

// The symmetric kernel from kSymMinN blobs on; below, one-warp CTAs that evaluate
// every ordered pair in a solver's steps, and the one-launch kernel for a product.
// A mixed solve (us) of 336 / 504 / 672 / 1,344 / 2,688 blobs takes 944 / 962 /
// 1,180 / 1,730 / 3,920 with every ordered pair and 982 / 995 / 1,149 / 1,370 /
// 2,310 with the symmetric kernel: zeroing the sums and the atomics cost two to
// three microseconds a step, and few pairs save less.
constexpr int64_t kSymMinN = 600;
static_assert(kSymMinN <= kSmallMaxN, "a product below kSymMinN takes the one-launch kernel");

int f32_variant(int64_t n) { return n < kSymMinN ? 4 : 3; }

// Size class of a matvec (mb_context_pair_variant): wall flag and half-octaves of N.
int size_class(int64_t n, int wall)
{
    int b = 0;
    for (int64_t m = n; m > 1; m >>= 1) ++b;
    const int half = (n >= 3 * ((int64_t)1 << (b > 0 ? b - 1 : 0))) ? 1 : 0;
    return (2 * b + half) * 2 + (wall ? 1 : 0);
}

mb_status matvec_f32(mb_context *ctx, const double *f, int64_t n, double a, int wall,
                     double scale, double *u, cudaStream_t s, MatvecPartials *defer)
{
    int v = ctx->pair_variant;
    if (v < 0) {
        v = f32_variant(n);
        ctx->chosen[size_class(n, wall)] = true;
    }
    return f32_run(ctx, v, f, n, a, wall, scale, u, s, true, defer);
}

mb_status matvec_pack_positions(mb_context *ctx, const double *r, int64_t n, cudaStream_t s,
                                bool order)
{
    MB_TRY(ensure(ctx, ctx->pos_hi, sizeof(float4) * (size_t)n, "packed positions"));
    MB_TRY(ensure(ctx, ctx->pos_lo, sizeof(float4) * (size_t)n, "packed positions"));
    ctx->sorted_n = 0;
    const int grid = (int)std::min<int64_t>(ceil_div(n, 256), 8 * (int64_t)ctx->sm_count);
    const bool sort = order && n >= kSortMinN;
    if (sort) {
        MB_TRY(ensure(ctx, ctx->sort_grid, sizeof(SortGrid) + sizeof(unsigned) * 6 * (size_t)grid,
                      "spatial order"));
        pack_hilo_kernel<true><<<grid, 256, 0, s>>>(
            r, n, (float4 *)ctx->pos_hi.ptr, (float4 *)ctx->pos_lo.ptr,
            sort_parts((SortGrid *)ctx->sort_grid.ptr));
    } else {
        pack_hilo_kernel<false><<<grid, 256, 0, s>>>(r, n, (float4 *)ctx->pos_hi.ptr,
                                                     (float4 *)ctx->pos_lo.ptr, nullptr);
    }
    count_launch();
    MB_CUDA_TRY(ctx, cudaGetLastError());
    if (sort) MB_TRY(sort_positions(ctx, n, grid, s));
    return MB_OK;
}

// Sources per item of the FP64 kernel: 32 unless that leaves fewer than
// kF64ItemsPerWarp items for each of an SM's four schedulers, then 16, 8 or 4.
// Every scheduler takes a whole number of items, so with m items each about
// 1/(2 m) of the time is lost to the last one; smaller items cost more
// reductions and atomics (C = 4: 12% of the FP64 instructions).
constexpr int kF64ItemsPerWarp = 16;

// Arrays that the sums of an FP64 product are spread over.  Every addition to
// an array is rounded at the size that the array's sum has by then, and a blob
// takes n / 32 + n / C of them, so the error grows with the square root of
// n / S.  Relative L2 error of the product against 113-bit values, S = 1, 8 and
// 16, and of chunk sums in a fixed order or blocks of 256 blobs (with the wall, in
// 1e-16): 336 blobs 3.3, 2.8, 2.7, 3.3; 1,000 6.2, 3.7, 3.5, 5.4; 8,191 6.7,
// 4.6, 4.4, 8.4; 16,384 8.5, 4.9, 4.7, 6.2; 65,536 16.7, 7.3, 5.9, 8.4.  Adding
// the arrays is a launch more: 336 blobs 21.6 -> 25.8 us, 2,730 614 -> 620.
constexpr int64_t kF64SumsMinN = 400;

int f64_sums(int64_t n) { return n < kF64SumsMinN ? 1 : n < 32768 ? 8 : 16; }

// One where the arrays don't fit the budget, or in a capture of the caller's
// where they would have to be allocated or, from kF64HeldMaxN blobs on, at all:
// products of that size hold no workspace, which a later call may move, so that
// their graphs stay valid.  (Graphs of smaller ones hold it, as those of FP32
// products do; the solver's own are dropped when workspace moves.)
constexpr int64_t kF64HeldMaxN = 8192;

int f64_sums_held(mb_context *ctx, int64_t n, cudaStream_t s)
{
    const int S = f64_sums(n);
    const size_t bytes = sizeof(double) * 3 * (size_t)n * S;
    const bool held = ctx->partial.bytes >= bytes;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (S > 1 && s != ctx->cap_stream && cudaStreamIsCapturing(s, &st) != cudaSuccess)
        cudaGetLastError();
    if (st != cudaStreamCaptureStatusNone) return held && n < kF64HeldMaxN ? S : 1;
    return held || ensure_room(ctx, ctx->partial) >= bytes ? S : 1;
}

template <bool WALL, int C>
void launch_f64sym_c(const double *r, const double *f, int64_t n, int64_t pairs, double a,
                     double *u, int S, double scale, cudaStream_t s)
{
    const int64_t items = pairs * (32 / C);
    pair_f64sym_kernel<WALL, C><<<(unsigned)std::min<int64_t>(items, 1 << 30), 32, 0, s>>>(
        r, f, n, items, MobConsts<double>::make(a), u, S, scale);
}

template <bool WALL>
void launch_f64sym(mb_context *ctx, const double *r, const double *f, int64_t n, double a,
                   double *u, int S, double scale, cudaStream_t s)
{
    const int64_t nb = ceil_div(n, 32), pairs = nb * (nb + 1) / 2;
    const int64_t want = (int64_t)kF64ItemsPerWarp * 4 * ctx->sm_count;
    if (pairs >= want) launch_f64sym_c<WALL, 32>(r, f, n, pairs, a, u, S, scale, s);
    else if (2 * pairs >= want) launch_f64sym_c<WALL, 16>(r, f, n, pairs, a, u, S, scale, s);
    else if (4 * pairs >= want) launch_f64sym_c<WALL, 8>(r, f, n, pairs, a, u, S, scale, s);
    else launch_f64sym_c<WALL, 4>(r, f, n, pairs, a, u, S, scale, s);
}

template <bool WALL, int NT>
void launch_df_nt(const float4 *hi, const float4 *lo, const double *f, int64_t n, double a,
                  double *u, double scale, const float *box, cudaStream_t s)
{
    const int64_t nb = ceil_div(n, 2 * NT), items = nb * (nb + 1);
    const float dfar = (float)(64.0 * a);
    pair_df_kernel<WALL, NT><<<(unsigned)std::min<int64_t>(items, 1 << 30), NT, 0, s>>>(
        hi, lo, f, n, items, MobConstsDf::make(a), u, scale, box, dfar * dfar);
}

template <bool WALL>
void launch_df(const float4 *hi, const float4 *lo, const double *f, int64_t n, double a, double *u,
               double scale, const float *box, cudaStream_t s)
{
    if (n <= kDfxMaxN)
        pair_dfx_kernel<WALL><<<dim3((unsigned)ceil_div(n, 32), (unsigned)ceil_div(n, kDfxChunk)),
                                32, 0, s>>>(hi, lo, f, n, MobConstsDf::make(a), u, scale);
    else if (n < kDfNT128MinN) launch_df_nt<WALL, 32>(hi, lo, f, n, a, u, scale, box, s);
    else launch_df_nt<WALL, 128>(hi, lo, f, n, a, u, scale, box, s);
}

mb_status matvec_packed(mb_context *ctx, const double *r, const double *f, int64_t n, double a,
                        double eta, int wall, mb_precision prec, double *u, cudaStream_t s,
                        MatvecPartials *defer)
{
    const double scale = 1.0 / (6.0 * kPi * eta * a);
    if (defer) *defer = MatvecPartials{};
    if (prec == MB_FP32_KAHAN) return matvec_f32(ctx, f, n, a, wall, scale, u, s, defer);
    if (prec == MB_DF64) {
        // zero u, then one launch; in the spatial order when the packing made
        // one (f gathered, u scattered back)
        const bool sorted = ctx->sorted_n == n;
        const float4 *hi = (const float4 *)(sorted ? ctx->sort_hi.ptr : ctx->pos_hi.ptr);
        const float4 *lo = (const float4 *)(sorted ? ctx->sort_lo.ptr : ctx->pos_lo.ptr);
        const float *box = sorted ? (const float *)ctx->sort_box.ptr : nullptr;
        const double *fk = f;
        double *uk = u;
        const int gv = (int)std::min<int64_t>(ceil_div(n, 256), 8 * (int64_t)ctx->sm_count);
        if (sorted) {
            MB_TRY(ensure(ctx, ctx->sort_f, sizeof(double) * 3 * (size_t)n, "sorted forces"));
            MB_TRY(ensure(ctx, ctx->sort_u, sizeof(double) * 3 * (size_t)n, "sorted velocities"));
            sort_gather_kernel<<<gv, 256, 0, s>>>((const int *)ctx->sort_perm.ptr, n, f,
                                                  (double *)ctx->sort_f.ptr,
                                                  (double *)ctx->sort_u.ptr);
            count_launch();
            fk = (const double *)ctx->sort_f.ptr;
            uk = (double *)ctx->sort_u.ptr;
        } else {
            MB_CUDA_TRY(ctx, cudaMemsetAsync(u, 0, sizeof(double) * 3 * (size_t)n, s));
        }
        auto *ev = profile_begin(ctx, s);
        if (wall) launch_df<true>(hi, lo, fk, n, a, uk, scale, box, s);
        else launch_df<false>(hi, lo, fk, n, a, uk, scale, box, s);
        profile_end(ev, s);
        count_launch();
        if (sorted) {
            sort_scatter_u_kernel<<<gv, 256, 0, s>>>((const int *)ctx->sort_perm.ptr, n, uk, u);
            count_launch();
        }
        MB_CUDA_TRY(ctx, cudaGetLastError());
        return MB_OK;
    }
    // FP64: u (or, of several sums or deferred, the sums that a launch or the
    // caller adds and scales) zeroed, then one launch over the block-pair triangle
    int S = f64_sums_held(ctx, n, s);
    const size_t one = sizeof(double) * 3 * (size_t)n;
    if (S > 1 && ensure(ctx, ctx->partial, S * one, "matvec partials") != MB_OK) {
        ctx->err.clear();  // the device has less left than the budget: one array does
        S = 1;
    }
    const bool sums = defer || S > 1;
    const size_t bytes = S * one;
    if (sums) MB_TRY(ensure(ctx, ctx->partial, bytes, "matvec partials"));
    double *uk = sums ? (double *)ctx->partial.ptr : u;
    const double sk = sums ? 1.0 : scale;
    MB_CUDA_TRY(ctx, cudaMemsetAsync(uk, 0, bytes, s));
    auto *ev = profile_begin(ctx, s);
    if (wall) launch_f64sym<true>(ctx, r, f, n, a, uk, S, sk, s);
    else launch_f64sym<false>(ctx, r, f, n, a, uk, S, sk, s);
    profile_end(ev, s);
    count_launch();
    if (defer) *defer = MatvecPartials{uk, S, scale};
    else if (sums) launch_reduce_partials(uk, n, S, scale, u, s);
    MB_CUDA_TRY(ctx, cudaGetLastError());
    return MB_OK;
}

// Whether two arrays of n blob vectors share memory.
bool overlap(const double *x, const double *y, int64_t n)
{
    return x < y + 3 * n && y < x + 3 * n;
}

mb_status matvec_device(mb_context *ctx, const double *r, const double *f, int64_t n, double a,
                        double eta, int wall, mb_precision prec, double *u, cudaStream_t s)
{
    // The symmetric kernels zero u and add to it while they read f (FP64: and
    // r), and the small one writes it, so a product in place works on copies.
    const bool small = prec == MB_FP32_KAHAN && ctx->pair_variant < 0 && n < kSymMinN;
    const size_t bytes = sizeof(double) * 3 * (size_t)n;
    if (overlap(u, f, n)) {
        MB_TRY(ensure(ctx, ctx->stage_f, bytes, "in-place product"));
        MB_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->stage_f.ptr, f, bytes, cudaMemcpyDeviceToDevice, s));
        f = (const double *)ctx->stage_f.ptr;
    }
    if ((prec == MB_FP64 || small) && overlap(u, r, n)) {
        MB_TRY(ensure(ctx, ctx->stage_r, bytes, "in-place product"));
        MB_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->stage_r.ptr, r, bytes, cudaMemcpyDeviceToDevice, s));
        r = (const double *)ctx->stage_r.ptr;
    }
    if (small) {
        const double scale = 1.0 / (6.0 * kPi * eta * a);
        ctx->chosen[size_class(n, wall)] = true;
        auto *ev = profile_begin(ctx, s);
        if (wall) launch_small<true>(r, f, n, a, u, scale, s);
        else launch_small<false>(r, f, n, a, u, scale, s);
        profile_end(ev, s);
        MB_CUDA_TRY(ctx, cudaGetLastError());
        return MB_OK;
    }
    if (prec != MB_FP64) MB_TRY(matvec_pack_positions(ctx, r, n, s));
    return matvec_packed(ctx, r, f, n, a, eta, wall, prec, u, s);
}

// Target blocks of `block` points against source chunks (whole tiles of
// `tile` sources, or a single chunk of 16 or more below one tile) so that there
// are about `want` items.  Splitting costs a reduction launch and 24 B a point
// and chunk, so chunks are shorter than 64 sources only as far as every
// scheduler needs an item at all.  The context's budget has to hold the chunks'
// partial sums, else there are fewer, down to one.
Plan eval_plan(const mb_context *ctx, int64_t nt, int64_t ns, int block, int64_t want, int tile,
               int64_t shortest)
{
    Plan p;
    p.n_tblocks = (int)ceil_div(nt, block);
    const int64_t fits = (int64_t)(ensure_room(ctx, ctx->partial) / (sizeof(double) * 3)) / nt;
    const int64_t need = std::min<int64_t>(4 * ctx->sm_count / p.n_tblocks, ceil_div(ns, shortest));
    const int64_t good = std::min(ceil_div(want, p.n_tblocks), ceil_div(ns, 4 * shortest));
    const int64_t s = std::max<int64_t>(1, std::min(std::max(need, good), fits));
    p.chunk = ceil_div(ns, s);
    if (p.chunk > tile / 2) p.chunk = ceil_div(p.chunk, tile) * tile;
    p.S = (int)ceil_div(ns, p.chunk);
    p.items = (int64_t)p.n_tblocks * p.S;
    p.grid = (int)std::min<int64_t>(p.items, 1 << 30);
    return p;
}

template <bool WALL, int NT>
void launch_eval_f32(const Plan &p, const float4 *thi, const float4 *tlo, int64_t nt,
                     const float4 *hi, const float4 *lo, const double *f, int64_t ns, double a,
                     double *out, double scale, int direct, cudaStream_t s)
{
    eval_f32x2_kernel<WALL, NT><<<p.grid, NT, 0, s>>>(thi, tlo, nt, hi, lo, f, ns, p.chunk,
                                                      p.n_tblocks, p.items, MobConsts2::make(a),
                                                      out, scale, direct);
}

mb_status matvec_eval(mb_context *ctx, const double *x, int64_t nt, const double *r,
                      const double *f, int64_t ns, double a, double eta, int wall,
                      mb_precision prec, double *u, cudaStream_t s)
{
    const double scale = 1.0 / (6.0 * kPi * eta * a);
    if (prec != MB_FP64 && prec != MB_FP32_KAHAN)
        return set_err(ctx, MB_EINVAL, "flow evaluation supports MB_FP32_KAHAN and MB_FP64");
    if (prec == MB_FP32_KAHAN) {
        // sources packed into the context's position buffers, targets into the eval ones
        MB_TRY(matvec_pack_positions(ctx, r, ns, s, false));
        MB_TRY(ensure(ctx, ctx->eval_hi, sizeof(float4) * (size_t)nt, "packed targets"));
        MB_TRY(ensure(ctx, ctx->eval_lo, sizeof(float4) * (size_t)nt, "packed targets"));
        const int grid = (int)std::min<int64_t>(ceil_div(nt, 256), 8 * (int64_t)ctx->sm_count);
        pack_hilo_kernel<false><<<grid, 256, 0, s>>>(x, nt, (float4 *)ctx->eval_hi.ptr,
                                                     (float4 *)ctx->eval_lo.ptr, nullptr);
        count_launch();
    }
    // FP32: kEvalItems items a resident warp slot, in one-warp CTAs unless
    // blocks of 256 points give as many; FP64 as the product's items
    constexpr int kEvalItems = 4;
    const int64_t slots = 16 * (int64_t)ctx->sm_count;
    const bool wide = ceil_div(nt, 256) * ceil_div(ns, 128) >= kEvalItems * slots / 4;
    const Plan p = prec == MB_FP64
                       ? eval_plan(ctx, nt, ns, 32, (int64_t)kF64ItemsPerWarp * 4 * ctx->sm_count, 4, 4)
                   : wide ? eval_plan(ctx, nt, ns, 256, kEvalItems * slots / 4, 128, 128)
                          : eval_plan(ctx, nt, ns, 64, kEvalItems * slots, 32, 16);
    double *out = u;
    const int direct = p.S == 1;
    if (!direct) {
        MB_TRY(ensure(ctx, ctx->partial, sizeof(double) * 3 * (size_t)nt * p.S, "eval partials"));
        out = (double *)ctx->partial.ptr;
    }
    if (prec == MB_FP64) {
        const MobConsts<double> k = MobConsts<double>::make(a);
        if (wall)
            eval_f64_kernel<true><<<p.grid, 32, 0, s>>>(x, nt, r, f, ns, p.chunk, p.n_tblocks,
                                                        p.items, k, out, scale, direct);
        else
            eval_f64_kernel<false><<<p.grid, 32, 0, s>>>(x, nt, r, f, ns, p.chunk, p.n_tblocks,
                                                         p.items, k, out, scale, direct);
    } else {
        const float4 *thi = (const float4 *)ctx->eval_hi.ptr, *tlo = (const float4 *)ctx->eval_lo.ptr;
        const float4 *hi = (const float4 *)ctx->pos_hi.ptr, *lo = (const float4 *)ctx->pos_lo.ptr;
        const auto launch = wide ? (wall ? launch_eval_f32<true, 128> : launch_eval_f32<false, 128>)
                                 : (wall ? launch_eval_f32<true, 32> : launch_eval_f32<false, 32>);
        launch(p, thi, tlo, nt, hi, lo, f, ns, a, out, scale, direct, s);
    }
    count_launch();
    MB_CUDA_TRY(ctx, cudaGetLastError());
    if (!direct) {
        launch_reduce_partials(out, nt, p.S, scale, u, s);
        MB_CUDA_TRY(ctx, cudaGetLastError());
    }
    return MB_OK;
}

mb_status render_flow(mb_context *ctx, const double *x, int64_t nt, const double *r,
                      const double *lam, int64_t n, const double *off, int n_sub, double a_sub,
                      double eta, int wall, mb_precision prec, double *v, cudaStream_t s)
{
    const int64_t ns = n * (int64_t)n_sub;
    MB_TRY(ensure(ctx, ctx->render_r, sizeof(double) * 3 * (size_t)ns, "refined blobs"));
    MB_TRY(ensure(ctx, ctx->render_f, sizeof(double) * 3 * (size_t)ns, "refined blob forces"));
    const int grid = (int)std::min<int64_t>(ceil_div(ns, 256), 8 * (int64_t)ctx->sm_count);
    refine_blobs_kernel<<<grid, 256, 0, s>>>(r, lam, n, off, n_sub, (double *)ctx->render_r.ptr,
                                             (double *)ctx->render_f.ptr);
    count_launch();
    MB_CUDA_TRY(ctx, cudaGetLastError());
    return matvec_eval(ctx, x, nt, (const double *)ctx->render_r.ptr,
                       (const double *)ctx->render_f.ptr, ns, a_sub, eta, wall, prec, v, s);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the FP32 matvec (mb_mobility_matvec_noalloc).
//
// For callers that must not allocate device memory: host applications whose
// framework owns the whole device-memory budget (a caching allocator has
// reserved it, so a cudaMalloc would fail or fragment it) and code on
// latency-critical paths that cannot take cudaMalloc's implicit device
// synchronisation.  The scratch that mb_mobility_matvec keeps in its context
// lives here in one file-scope device array instead, laid out for
// MB_NOALLOC_MAX_BLOBS blobs.  Every GPU that loads the library holds the
// array until the process exits.  All calls share it: calls whose work
// overlaps on the GPU race on it.  Each call writes every element it later
// reads, so nothing needs clearing between calls.
//
// The kernels and the rule by size are mb_mobility_matvec's: the one-launch
// kernel below kSymMinN, the symmetric kernel above, in the spatial
// order from kSortMinN on.  A scalar kernel for every ordered pair ran at every
// size: 5,003 blobs 121 -> 64 us, 65,536 13.1 -> 5.2 ms with the wall, 20,011
// 705 -> 323 us and 65,536 6.0 -> 2.8 ms without.
namespace {

constexpr int64_t kNoallocMaxBlobs = MB_NOALLOC_MAX_BLOBS;
constexpr int kNoallocPackCtas = 256;
constexpr int kNoallocBits = 13;      // sort_bits(kNoallocMaxBlobs)
constexpr int kNoallocMaxTiles = 64;  // sort_tiles(kNoallocMaxBlobs, any)
static_assert(kNoallocMaxBlobs <= ((int64_t)8 << kNoallocBits) &&
                  kNoallocMaxBlobs <= 1024 * (int64_t)kNoallocMaxTiles &&
                  kNoallocMaxBlobs <= 256 * (int64_t)kNoallocPackCtas,
              "the scratch holds the largest order");

struct NoallocScratch {
    float4 hi[kNoallocMaxBlobs], lo[kNoallocMaxBlobs];
    float4 shi[kNoallocMaxBlobs], slo[kNoallocMaxBlobs];
    double f[3 * kNoallocMaxBlobs], u[3 * kNoallocMaxBlobs];  // sorted, or copies for a product
                                                              // in place
    unsigned key[kNoallocMaxBlobs];
    int perm[kNoallocMaxBlobs];
    int H[(kNoallocMaxTiles + 1) << kNoallocBits];
    float box[6 * ((kNoallocMaxBlobs + kBoxBlobs - 1) / kBoxBlobs)];
    struct {
        SortGrid grid;
        unsigned parts[6 * kNoallocPackCtas];
    } sort;
};

static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoallocScratch)];

struct NoallocDevice {
    bool ready = false;
    NoallocScratch *scratch = nullptr;  // device address of g_noalloc_scratch
    int sms = 0;
};
constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mu;
NoallocDevice g_noalloc_dev[kNoallocMaxDevices];

// First call on a device: look up the array's device address (host code may
// not use the symbol itself) and the SM count.  No allocation.
mb_status noalloc_setup(int dev, NoallocDevice **out)
{
    if (dev < 0 || dev >= kNoallocMaxDevices) return MB_EINVAL;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoallocDevice &d = g_noalloc_dev[dev];
    if (!d.ready) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            set_thread_err("cudaGetSymbolAddress of the allocation-free scratch failed");
            return MB_ECUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            set_thread_err("device query failed in the allocation-free matvec set-up");
            return MB_ECUDA;
        }
        d.scratch = (NoallocScratch *)ptr;
        d.sms = sms;
        d.ready = true;
    }
    *out = &d;
    return MB_OK;
}

cudaError_t noalloc_run(const NoallocDevice &d, const double *r, const double *f, int64_t n,
                        double a, double eta, int wall, double *u, cudaStream_t s)
{
    NoallocScratch *w = d.scratch;
    const double scale = 1.0 / (6.0 * kPi * eta * a);
    if (n < kSymMinN) {
        const size_t bytes = sizeof(double) * 3 * (size_t)n;
        cudaError_t e = cudaSuccess;
        if (overlap(u, f, n)) {
            e = cudaMemcpyAsync(w->f, f, bytes, cudaMemcpyDeviceToDevice, s);
            f = w->f;
        }
        if (e == cudaSuccess && overlap(u, r, n)) {
            e = cudaMemcpyAsync(w->u, r, bytes, cudaMemcpyDeviceToDevice, s);
            r = w->u;
        }
        if (e != cudaSuccess) return e;
        if (wall) launch_small<true>(r, f, n, a, u, scale, s);
        else launch_small<false>(r, f, n, a, u, scale, s);
        return cudaGetLastError();
    }
    const int pack = (int)std::min<int64_t>(ceil_div(n, 256), kNoallocPackCtas);
    const bool sorted = n >= kSortMinN;
    if (sorted) pack_hilo_kernel<true><<<pack, 256, 0, s>>>(r, n, w->hi, w->lo, w->sort.parts);
    else pack_hilo_kernel<false><<<pack, 256, 0, s>>>(r, n, w->hi, w->lo, nullptr);
    count_launch();
    cudaError_t e = cudaSuccess;
    double *us = u;
    const SortGrid *sg = nullptr;
    if (sorted) {
        const SortBufs b{w->hi, w->lo, &w->sort.grid, w->key, w->perm, w->H, w->shi, w->slo, w->box};
        e = sort_launch(b, n, pack, d.sms, s);
        if (e != cudaSuccess) return e;
        us = w->u;
        sg = b.grid;
        sort_gather_kernel<<<pack, 256, 0, s>>>(w->perm, n, f, w->f, us);
        count_launch();
        f = w->f;
    } else {
        if (overlap(u, f, n)) {  // u is zeroed and added to while f is read
            e = cudaMemcpyAsync(w->f, f, sizeof(double) * 3 * (size_t)n, cudaMemcpyDeviceToDevice, s);
            if (e != cudaSuccess) return e;
            f = w->f;
        }
        e = cudaMemsetAsync(u, 0, sizeof(double) * 3 * (size_t)n, s);
        if (e != cudaSuccess) return e;
    }
    const float4 *hi = sorted ? w->shi : w->hi, *lo = sorted ? w->slo : w->lo;
    const float *box = sorted ? w->box : nullptr;
    if (wall) launch_sym<true>(hi, lo, f, n, a, us, scale, box, sg, s);
    else launch_sym<false>(hi, lo, f, n, a, us, scale, box, sg, s);
    count_launch();
    if (sorted) {
        sort_scatter_u_kernel<<<pack, 256, 0, s>>>(w->perm, n, us, u);
        count_launch();
    }
    return cudaGetLastError();
}

// Device memory of device `dev` (the one whose scratch array the call uses),
// or managed memory.  Memory of another GPU would reach the kernel as a peer
// pointer, so it is refused on the host instead.
bool on_device(const void *p, int dev)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (at.type == cudaMemoryTypeDevice && at.device == dev) ||
           at.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace mb

extern "C" mb_status mb_mobility_matvec_noalloc(const double *r, const double *f, int64_t n,
                                                double a, double eta, int wall, double *u,
                                                void *stream)
{
    using namespace mb;
    set_thread_err("");
    if (n < 0 || n > kNoallocMaxBlobs) {
        set_thread_err("N must be in [0, MB_NOALLOC_MAX_BLOBS]");
        return MB_EINVAL;
    }
    if (!(a > 0.0) || !(eta > 0.0)) {
        set_thread_err("a and eta must be positive");
        return MB_EINVAL;
    }
    if (n == 0) return MB_OK;
    if (!r || !f || !u) {
        set_thread_err("r, f and u must be device pointers");
        return MB_EINVAL;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        set_thread_err("cudaGetDevice failed");
        return MB_ECUDA;
    }
    if (!on_device(r, dev) || !on_device(f, dev) || !on_device(u, dev)) {
        set_thread_err("r, f and u must be device pointers on the current device");
        return MB_EINVAL;
    }
    NoallocDevice *d = nullptr;
    mb_status st = noalloc_setup(dev, &d);
    if (st != MB_OK) return st;
    cudaError_t e = noalloc_run(*d, r, f, n, a, eta, wall, u, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_thread_err(cudaGetErrorString(e));
        return MB_ECUDA;
    }
    return MB_OK;
}
