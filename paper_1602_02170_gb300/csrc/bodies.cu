// Rigid-body geometry and kinematics on the blobs.
//   blob build:  r_i = q_p + R(theta_p) rho_i                    (Section 2.1)
//   K:           v_i = U_p + Omega_p x (r_i - q_p)               (Eq. noslip_rigid)
//   K^T:         (sum_i lambda_i, sum_i (r_i - q_p) x lambda_i)  (Eq. rigidSystem)
// The gathers go by tiles of consecutive blobs whose bodies are found once a
// tile, one warp or half a warp per body does the segmented reduction of K^T.
//
// With one FP64 warp instruction per ~19 cycles and SM, FP64 instructions and
// not the 48 B a blob moves through HBM bound these kernels: 663,552 blobs
// take 1.3 us for every FP64 instruction a blob costs.  So the rotation matrix
// is formed once per body and tile instead of the quaternion product per blob
// (12 FP64 instructions a blob for 39), K's factor alpha goes into the body's
// velocities, and K^T's sums are exchanged so that a butterfly adds 8 values
// instead of 30.  4,096 bodies of 162 blobs (ncu): blob build 53 -> 25 us, K
// 29 -> 20 us, K^T 43 -> 23 us, of which 15, 11 and 17 are FP64 instructions.
#include <algorithm>

#include "mb_internal.cuh"

namespace mb {
namespace {

// A tile of kTileThreads * PER consecutive blobs from i0 on: their bodies
// (p0 .. p0 + nb_tile - 1) and offsets in shared memory, when there are at
// most kTileBodies of them (empty bodies count); every thread of the CTA must
// call tile_bodies.
constexpr int kTileThreads = 256;
constexpr int kTileBodies = 64;

struct TileBodies {
    int64_t first, last;          // bodies of the tile's first and last blob
    int64_t start[kTileBodies];   // first blob of body first + k
};

__device__ __forceinline__ bool tile_bodies(const int64_t *__restrict__ start, int64_t nb,
                                            int64_t i0, int64_t i1, TileBodies &tb)
{
    if (threadIdx.x == 0) tb.first = body_of(start, nb, i0);
    if (threadIdx.x == 32) tb.last = body_of(start, nb, i1 - 1);
    __syncthreads();
    const int64_t cnt = tb.last - tb.first + 1;
    if (cnt < 1 || cnt > kTileBodies) return false;
    for (int k = threadIdx.x; k < cnt; k += kTileThreads) tb.start[k] = start[tb.first + k];
    return true;
}

// Index in the tile of blob i's body.
__device__ __forceinline__ int tile_body_of(const TileBodies &tb, int64_t i)
{
    int lo = 0, hi = (int)(tb.last - tb.first) + 1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (tb.start[mid] <= i) lo = mid;
        else hi = mid;
    }
    return lo;
}

// 1 / d in FP64 for 1e-30 < d < 1e30: the FP32 reciprocal and one step of third
// order y (1 + e + e^2), e = 1 - d y (|e| < 2^-22).
__device__ __forceinline__ double rcp_mid(double d)
{
    const double y = (double)(1.0f / (float)d);
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// R = (s^2 - v.v) I + 2 v v^T + 2 s [v]_x of the normalised quaternion:
// with t = 2 / |theta|^2, (t s^2 - 1) I + t (v v^T + s [v]_x); R row-major,
// then q, in m[0..11].  Quaternions far from unit length, whose t may be out of
// range, are normalised first.
__device__ __forceinline__ void body_frame(const double *__restrict__ th,
                                           const double *__restrict__ q, double *m)
{
    double s = th[0], x = th[1], y = th[2], z = th[3], t = 2.0;
    const double n2 = fma(s, s, fma(x, x, fma(y, y, z * z)));
    if (n2 > 1e-30 && n2 < 1e30) {
        t *= rcp_mid(n2);
    } else {
        const double inv = rsqrt(n2);
        s *= inv;
        x *= inv;
        y *= inv;
        z *= inv;
    }
    const double ts = t * s, tx = t * x, ty = t * y, tz = t * z, d = fma(ts, s, -1.0);
    m[0] = fma(tx, x, d);
    m[1] = fma(tx, y, -ts * z);
    m[2] = fma(tx, z, ts * y);
    m[3] = fma(tx, y, ts * z);
    m[4] = fma(ty, y, d);
    m[5] = fma(ty, z, -ts * x);
    m[6] = fma(tx, z, -ts * y);
    m[7] = fma(ty, z, ts * x);
    m[8] = fma(tz, z, d);
    m[9] = q[0];
    m[10] = q[1];
    m[11] = q[2];
}

__device__ __forceinline__ double rotate_row(const double *m, int c, double a, double b, double e)
{
    // q last: one rounding at its size, which may be hundreds of body radii
    return fma(m[3 * c], a, fma(m[3 * c + 1], b, m[3 * c + 2] * e)) + m[9 + c];
}

template <int PER>
__global__ void __launch_bounds__(kTileThreads) blob_positions_kernel(
    int64_t nb, int64_t n, const double *__restrict__ q, const double *__restrict__ theta,
    const int64_t *__restrict__ start, const double *__restrict__ rho, double *__restrict__ r)
{
    __shared__ TileBodies tb;
    __shared__ double frame[kTileBodies][12];
    __shared__ double v[3 * kTileThreads];
    const int64_t i0 = blockIdx.x * (int64_t)(kTileThreads * PER);
    const int64_t i1 = i0 + kTileThreads * PER < n ? i0 + kTileThreads * PER : n;
    if (!tile_bodies(start, nb, i0, i1, tb)) {  // many tiny or empty bodies: blob by blob
        for (int64_t i = i0 + threadIdx.x; i < i1; i += kTileThreads) {
            const int64_t p = body_of(start, nb, i);
            double m[12];
            body_frame(theta + 4 * p, q + 3 * p, m);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                r[3 * i + c] = rotate_row(m, c, rho[3 * i], rho[3 * i + 1], rho[3 * i + 2]);
        }
        return;
    }
    const int cnt = (int)(tb.last - tb.first) + 1;
    if ((int)threadIdx.x < cnt)
        body_frame(theta + 4 * (tb.first + threadIdx.x), q + 3 * (tb.first + threadIdx.x),
                   frame[threadIdx.x]);
    __syncthreads();
    // rounds of 32 blobs per warp; rho and r pass through shared memory, so
    // that both are read and written in whole lines
    const int lane = threadIdx.x & 31;
    double *vw = v + 96 * (threadIdx.x >> 5), *w = vw + 3 * lane;
    for (int64_t b = i0 + threadIdx.x - lane; b < i1; b += kTileThreads) {
        const int len = 3 * (int)(i1 - b < 32 ? i1 - b : 32);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (lane + 32 * k < len) vw[lane + 32 * k] = rho[3 * b + lane + 32 * k];
        __syncwarp();
        if (3 * lane < len) {
            const double *m = frame[tile_body_of(tb, b + lane)];
            const double a = w[0], e1 = w[1], e2 = w[2];
#pragma unroll
            for (int c = 0; c < 3; ++c) w[c] = rotate_row(m, c, a, e1, e2);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (lane + 32 * k < len) r[3 * b + lane + 32 * k] = vw[lane + 32 * k];
        __syncwarp();
    }
}

// v = alpha K UO + beta v (ADD), or alpha K UO (v is not read).
template <int PER, bool ADD>
__global__ void __launch_bounds__(kTileThreads) K_apply_kernel(
    int64_t nb, int64_t n, const double *__restrict__ r, const double *__restrict__ q,
    const int64_t *__restrict__ start, const double *__restrict__ UO, double *__restrict__ v,
    double alpha, double beta)
{
    __shared__ TileBodies tb;
    __shared__ double body[kTileBodies][9];  // alpha U, alpha Omega, q
    __shared__ double sh[3 * kTileThreads];
    const int64_t i0 = blockIdx.x * (int64_t)(kTileThreads * PER);
    const int64_t i1 = i0 + kTileThreads * PER < n ? i0 + kTileThreads * PER : n;
    const bool tile = tile_bodies(start, nb, i0, i1, tb);
    if (tile) {
        const int cnt = (int)(tb.last - tb.first) + 1;
        for (int e = threadIdx.x; e < 9 * cnt; e += kTileThreads) {
            const int k = e / 9, c = e % 9;
            body[k][c] = c < 6 ? alpha * UO[6 * (tb.first + k) + c] : q[3 * (tb.first + k) + c - 6];
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    double *vw = sh + 96 * (threadIdx.x >> 5), *x = vw + 3 * lane;
    for (int64_t b = i0 + threadIdx.x - lane; b < i1; b += kTileThreads) {
        const int len = 3 * (int)(i1 - b < 32 ? i1 - b : 32);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (lane + 32 * k < len) vw[lane + 32 * k] = r[3 * b + lane + 32 * k];
        __syncwarp();
        if (3 * lane < len) {
            double w[9];
            if (tile) {
                const double *m = body[tile_body_of(tb, b + lane)];
#pragma unroll
                for (int c = 0; c < 9; ++c) w[c] = m[c];
            } else {  // many tiny or empty bodies
                const int64_t p = body_of(start, nb, b + lane);
#pragma unroll
                for (int c = 0; c < 9; ++c) w[c] = c < 6 ? alpha * UO[6 * p + c] : q[3 * p + c - 6];
            }
            const double dx = x[0] - w[6], dy = x[1] - w[7], dz = x[2] - w[8];
            x[0] = fma(w[4], dz, fma(-w[5], dy, w[0]));
            x[1] = fma(w[5], dx, fma(-w[3], dz, w[1]));
            x[2] = fma(w[3], dy, fma(-w[4], dx, w[2]));
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (lane + 32 * k < len) {
                const int64_t e = 3 * b + lane + 32 * k;
                v[e] = ADD ? fma(beta, v[e], vw[lane + 32 * k]) : vw[lane + 32 * k];
            }
        __syncwarp();
    }
}

// FT = alpha K^T lambda, G lanes per body (16 or 32).
template <int G>
__global__ void __launch_bounds__(256) KT_apply_kernel(int64_t nb, const double *__restrict__ r,
                                                       const double *__restrict__ q,
                                                       const int64_t *__restrict__ start,
                                                       const double *__restrict__ lam,
                                                       double *__restrict__ FT, double alpha)
{
    const int lane = threadIdx.x & (G - 1);
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
    // all groups of a warp take the same number of rounds (shuffles)
    for (int64_t p0 = blockIdx.x * (int64_t)(blockDim.x / G); p0 < nb; p0 += groups) {
        const int64_t p = p0 + threadIdx.x / G;
        double a[6] = {0, 0, 0, 0, 0, 0};
        if (p < nb) {
            const double qx = q[3 * p], qy = q[3 * p + 1], qz = q[3 * p + 2];
            const int64_t end = start[p + 1];
            for (int64_t i = start[p] + lane; i < end; i += G) {
                const double lx = lam[3 * i], ly = lam[3 * i + 1], lz = lam[3 * i + 2];
                const double dx = r[3 * i] - qx, dy = r[3 * i + 1] - qy, dz = r[3 * i + 2] - qz;
                a[0] += lx;
                a[1] += ly;
                a[2] += lz;
                a[3] = fma(dy, lz, fma(-dz, ly, a[3]));
                a[4] = fma(dz, lx, fma(-dx, lz, a[4]));
                a[5] = fma(dx, ly, fma(-dy, lx, a[5]));
            }
        }
        // each exchange halves the values a lane holds: forces or torques,
        // then components {0, 1} or {2}, then 0 or 1
        const unsigned all = 0xffffffffu;
        const bool hi = lane & (G / 2), mid = lane & (G / 4), low = lane & (G / 8);
        double b[3], c[2], d;
#pragma unroll
        for (int k = 0; k < 3; ++k)
            b[k] = (hi ? a[3 + k] : a[k]) + __shfl_xor_sync(all, hi ? a[k] : a[3 + k], G / 2);
        c[0] = (mid ? b[2] : b[0]) + __shfl_xor_sync(all, mid ? b[0] : b[2], G / 4);
        c[1] = (mid ? 0.0 : b[1]) + __shfl_xor_sync(all, mid ? b[1] : 0.0, G / 4);
        d = (low ? c[1] : c[0]) + __shfl_xor_sync(all, low ? c[0] : c[1], G / 8);
#pragma unroll
        for (int o = G / 16; o > 0; o >>= 1) d += __shfl_xor_sync(all, d, o);
        if (p < nb && (lane & (G / 8 - 1)) == 0 && !(mid && low))
            FT[6 * p + (hi ? 3 : 0) + (mid ? 2 : low ? 1 : 0)] = alpha * d;
    }
}

// The same sum with one CTA per body, for few bodies (the warp-per-body form
// would leave most SMs idle and run each body's blobs serially in one warp).
constexpr int64_t kKTBlockBodies = 256;

__global__ void __launch_bounds__(256) KT_apply_block_kernel(
    int64_t nb, const double *__restrict__ r, const double *__restrict__ q,
    const int64_t *__restrict__ start, const double *__restrict__ lam, double *__restrict__ FT,
    double alpha)
{
    __shared__ double red[8][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t p = blockIdx.x; p < nb; p += gridDim.x) {
        double acc[6] = {0, 0, 0, 0, 0, 0};
        const double qx = q[3 * p], qy = q[3 * p + 1], qz = q[3 * p + 2];
        for (int64_t i = start[p] + threadIdx.x; i < start[p + 1]; i += blockDim.x) {
            const double lx = lam[3 * i], ly = lam[3 * i + 1], lz = lam[3 * i + 2];
            const double dx = r[3 * i] - qx, dy = r[3 * i + 1] - qy, dz = r[3 * i + 2] - qz;
            acc[0] += lx;
            acc[1] += ly;
            acc[2] += lz;
            acc[3] += dy * lz - dz * ly;
            acc[4] += dz * lx - dx * lz;
            acc[5] += dx * ly - dy * lx;
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        }
        __syncthreads();
        if (lane == 0) {
#pragma unroll
            for (int c = 0; c < 6; ++c) red[warp][c] = acc[c];
        }
        __syncthreads();
        if (threadIdx.x < 6) {
            double v = 0.0;
            for (int w8 = 0; w8 < 8; ++w8) v += red[w8][threadIdx.x];
            FT[6 * p + threadIdx.x] = alpha * v;
        }
    }
}

static_assert(kSaddleRowsMaxBodies == kKTBlockBodies,
              "saddle_rows_kernel reduces K^T lambda with one CTA per body");

// The saddle operator's rows around M lambda in one launch (Eq. saddle_M),
// from the pair kernel's chunk partials; x = [lambda; U].  Blocks below
// blob_blocks take blobs, one thread per blob:
//   y_i = scale * sum_s partial[s][i] - (K U)_i
// (the sums of reduce_partials_kernel, then K_apply_kernel with alpha = -1,
// beta = 1); the other blocks take bodies, one CTA per body:
//   y_(3N + 6p + c) = -(K^T lambda)_p,c
// (the reduction of KT_apply_block_kernel).  All threads of a block take the
// same branch, so the barriers of the body branch are uniform.  Blocks are
// small (kSaddleThreads): the per-thread work is a short serial chain of FP64
// instructions, which issue slowly on this chip, so spreading the warps over
// more SMs shortens the launch; for bodies of up to 64 blobs the body sums
// round as with one CTA of 256 threads.
constexpr int kSaddleThreads = 64;

__global__ void __launch_bounds__(kSaddleThreads) saddle_rows_kernel(
    const double *__restrict__ partial, int S, double scale, int64_t n, int64_t nb,
    const double *__restrict__ r, const double *__restrict__ q, const int64_t *__restrict__ start,
    const double *__restrict__ x, double *__restrict__ y, int blob_blocks)
{
    const int64_t m = 3 * n;
    if ((int)blockIdx.x < blob_blocks) {
        const double *UO = x + m;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
             i += (int64_t)blob_blocks * blockDim.x) {
            double acc[3] = {0.0, 0.0, 0.0};
            for (int sc = 0; sc < S; ++sc) {
                const double *ps = partial + sc * m + 3 * i;
                acc[0] += ps[0];
                acc[1] += ps[1];
                acc[2] += ps[2];
            }
            const int64_t p = body_of(start, nb, i);
            const double dx = r[3 * i] - q[3 * p], dy = r[3 * i + 1] - q[3 * p + 1],
                         dz = r[3 * i + 2] - q[3 * p + 2];
            const double *u = UO + 6 * p;
            const double vx = u[0] + (u[4] * dz - u[5] * dy);
            const double vy = u[1] + (u[5] * dx - u[3] * dz);
            const double vz = u[2] + (u[3] * dy - u[4] * dx);
            // rounded as the two-kernel sequence: u = scale * acc, then u - v
            y[3 * i] = __dsub_rn(__dmul_rn(scale, acc[0]), vx);
            y[3 * i + 1] = __dsub_rn(__dmul_rn(scale, acc[1]), vy);
            y[3 * i + 2] = __dsub_rn(__dmul_rn(scale, acc[2]), vz);
        }
        return;
    }
    constexpr int kWarps = kSaddleThreads / 32;
    __shared__ double red[kWarps][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int body_blocks = (int)gridDim.x - blob_blocks;
    for (int64_t p = (int)blockIdx.x - blob_blocks; p < nb; p += body_blocks) {
        double acc[6] = {0, 0, 0, 0, 0, 0};
        const double qx = q[3 * p], qy = q[3 * p + 1], qz = q[3 * p + 2];
        for (int64_t i = start[p] + threadIdx.x; i < start[p + 1]; i += blockDim.x) {
            const double lx = x[3 * i], ly = x[3 * i + 1], lz = x[3 * i + 2];
            const double dx = r[3 * i] - qx, dy = r[3 * i + 1] - qy, dz = r[3 * i + 2] - qz;
            acc[0] += lx;
            acc[1] += ly;
            acc[2] += lz;
            acc[3] += dy * lz - dz * ly;
            acc[4] += dz * lx - dx * lz;
            acc[5] += dx * ly - dy * lx;
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        }
        __syncthreads();
        if (lane == 0) {
#pragma unroll
            for (int c = 0; c < 6; ++c) red[warp][c] = acc[c];
        }
        __syncthreads();
        if (threadIdx.x < 6) {
            double v = 0.0;
            for (int w8 = 0; w8 < kWarps; ++w8) v += red[w8][threadIdx.x];
            y[m + 6 * p + threadIdx.x] = -v;
        }
    }
}

int grid_for(int64_t work, int threads)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(work, threads), 4096));
}

// Tiles of two rounds from here on: the body frames of a tile cost as much as
// three rounds' blobs of one warp, and fewer tiles than this leave SMs idle.
constexpr int kTilePer = 2;
constexpr int64_t kTileLargeN = 1 << 18;

int tile_grid(int64_t n, int per) { return (int)ceil_div(n, (int64_t)kTileThreads * per); }

// Half a warp per body once that still gives every scheduler two warps: bodies
// of 162 and 42 blobs fill 92% and 88% of its lanes, against 84% and 66%.
constexpr int64_t kKTHalfWarpBodies = 2048;

}  // namespace

mb_status blob_positions(mb_context *ctx, int64_t nb, int64_t n, const double *q,
                         const double *theta, const int64_t *blob_start, const double *rho,
                         double *r, cudaStream_t s)
{
    if (n == 0) return MB_OK;
    if (n >= kTileLargeN)
        blob_positions_kernel<kTilePer><<<tile_grid(n, kTilePer), kTileThreads, 0, s>>>(
            nb, n, q, theta, blob_start, rho, r);
    else
        blob_positions_kernel<1><<<tile_grid(n, 1), kTileThreads, 0, s>>>(nb, n, q, theta,
                                                                         blob_start, rho, r);
    count_launch();
    MB_CUDA_TRY(ctx, cudaGetLastError());
    return MB_OK;
}

void launch_K_apply(int64_t nb, int64_t n, const double *r, const double *q,
                    const int64_t *blob_start, const double *UO, double *v, double alpha,
                    double beta, cudaStream_t s)
{
    if (n == 0) return;
    const bool add = beta != 0.0, large = n >= kTileLargeN;
    const int grid = tile_grid(n, large ? kTilePer : 1);
    if (add && large)
        K_apply_kernel<kTilePer, true><<<grid, kTileThreads, 0, s>>>(nb, n, r, q, blob_start, UO, v,
                                                                     alpha, beta);
    else if (add)
        K_apply_kernel<1, true><<<grid, kTileThreads, 0, s>>>(nb, n, r, q, blob_start, UO, v, alpha,
                                                             beta);
    else if (large)
        K_apply_kernel<kTilePer, false><<<grid, kTileThreads, 0, s>>>(nb, n, r, q, blob_start, UO,
                                                                      v, alpha, beta);
    else
        K_apply_kernel<1, false><<<grid, kTileThreads, 0, s>>>(nb, n, r, q, blob_start, UO, v,
                                                              alpha, beta);
    count_launch();
}

void launch_saddle_rows(const MatvecPartials &mp, int64_t n, int64_t nb, const double *r,
                        const double *q, const int64_t *blob_start, const double *x, double *y,
                        cudaStream_t s)
{
    const int blob_blocks =
        (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, kSaddleThreads), 4096));
    saddle_rows_kernel<<<blob_blocks + (int)nb, kSaddleThreads, 0, s>>>(
        mp.partial, mp.S, mp.scale, n, nb, r, q, blob_start, x, y, blob_blocks);
    count_launch();
}

// S_p[a][b] = sum_{i in p} lambda_i,a (r_i - q_p)_b: the first moment of the
// blob forces, whose symmetric traceless part is the body's stresslet
// (Section 4.1).  One warp per body.
__global__ void moments_kernel(int64_t nb, const double *__restrict__ r,
                               const double *__restrict__ q, const int64_t *__restrict__ start,
                               const double *__restrict__ lam, double *__restrict__ S)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t p = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); p < nb;
         p += warps) {
        double acc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        const double qx = q[3 * p], qy = q[3 * p + 1], qz = q[3 * p + 2];
        for (int64_t i = start[p] + lane; i < start[p + 1]; i += 32) {
            const double d[3] = {r[3 * i] - qx, r[3 * i + 1] - qy, r[3 * i + 2] - qz};
#pragma unroll
            for (int al = 0; al < 3; ++al)
#pragma unroll
                for (int be = 0; be < 3; ++be) acc[3 * al + be] += lam[3 * i + al] * d[be];
        }
#pragma unroll
        for (int c = 0; c < 9; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        }
        if (lane < 9) {
            double v = acc[0];
#pragma unroll
            for (int c = 1; c < 9; ++c)
                if (lane == c) v = acc[c];
            S[9 * p + lane] = v;
        }
    }
}

void launch_moments(int64_t nb, const double *r, const double *q, const int64_t *blob_start,
                    const double *lambda, double *S, cudaStream_t s)
{
    if (nb == 0) return;
    moments_kernel<<<grid_for(nb * 32, 256), 256, 0, s>>>(nb, r, q, blob_start, lambda, S);
    count_launch();
}

void launch_KT_apply(int64_t nb, const double *r, const double *q, const int64_t *blob_start,
                     const double *lambda, double *FT, double alpha, cudaStream_t s)
{
    if (nb == 0) return;
    if (nb <= kKTBlockBodies)
        KT_apply_block_kernel<<<(int)nb, 256, 0, s>>>(nb, r, q, blob_start, lambda, FT, alpha);
    else if (nb >= kKTHalfWarpBodies)
        KT_apply_kernel<16><<<grid_for(nb * 16, 256), 256, 0, s>>>(nb, r, q, blob_start, lambda, FT,
                                                                   alpha);
    else
        KT_apply_kernel<32><<<grid_for(nb * 32, 256), 256, 0, s>>>(nb, r, q, blob_start, lambda, FT,
                                                                   alpha);
    count_launch();
}

}  // namespace mb
