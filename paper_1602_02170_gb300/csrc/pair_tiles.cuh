// Source-tile loops of the pair kernels, shared by the single-problem
// kernels (pair_matvec.cu) and the batched ones (batch.cu).
//
// One call processes one work item: the targets of target block `tb` of one
// problem against that problem's sources [j_begin, j_end).  Pointers are
// already offset to the problem; `out` receives the item's velocities at
// out + 3 i (i = target index within the problem) multiplied by `m`.  The
// non-symmetric items take the targets (n of them) from their own arrays,
// which are the source arrays themselves for a matvec and other points when
// a flow is evaluated away from the blobs.
#pragma once

#include "df32.cuh"
#include "rpy_wall.cuh"

namespace mb {

__device__ __forceinline__ void kahan_add(float &sum, float &comp, float x)
{
    const float y = x - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// Shared-memory floats per source in the packed kernel (5 float4).
constexpr int kX2SmemFloat4PerSource = 5;

// Pair t = J (J + 1) / 2 + I of the triangle I <= J.
__device__ __forceinline__ void triangle_pair(int64_t t, int64_t &I, int64_t &J)
{
    J = (int64_t)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while (J * (J + 1) / 2 > t) --J;
    while ((J + 1) * (J + 2) / 2 <= t) ++J;
    I = t - J * (J + 1) / 2;
}

__device__ __forceinline__ void stage_x2(float4 *d, float4 h, float4 l, float fx, float fy, float fz)
{
    const float zz = -2.f * h.z * h.z;
    d[0] = make_float4(-h.x, -h.x, -h.y, -h.y);
    d[1] = make_float4(h.z, h.z, zz, zz);
    d[2] = make_float4(-l.x, -l.x, -l.y, -l.y);
    d[3] = make_float4(-l.z, -l.z, fx, fx);
    d[4] = make_float4(fy, fy, fz, fz);
}

// Packed FP32 item: each thread owns 2*NP targets, held as NP float2 pairs;
// target of pair q, half h: tb*NT*2*NP + (2q + h)*NT + threadIdx.x.
// Sources are staged once per tile as duplicated float2 operands:
//   sP[5s+0] = (-x_hi, -x_hi, -y_hi, -y_hi)   sP[5s+1] = (z_hi, z_hi, zz, zz), zz = -2 z_hi^2
//   sP[5s+2] = (-x_lo, -x_lo, -y_lo, -y_lo)   sP[5s+3] = (-z_lo, -z_lo, f_x, f_x)
//   sP[5s+4] = (f_y, f_y, f_z, f_z)
template <bool WALL, int NP, int NT>
__device__ __forceinline__ void x2_item(float4 *__restrict__ sP, const float4 *__restrict__ thi,
                                        const float4 *__restrict__ tlo, int64_t n,
                                        const float4 *__restrict__ hi,
                                        const float4 *__restrict__ lo,
                                        const double *__restrict__ f, int tb,
                                        int64_t j_begin, int64_t j_end, const MobConsts2 &k,
                                        double *__restrict__ out, double m)
{
    float2 xh[NP], yh[NP], zh[NP], xl[NP], yl[NP], zl[NP];
    float sum[2 * NP][3], comp[2 * NP][3];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        float4 h[2], l[2];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            int64_t i = (int64_t)tb * NT * 2 * NP + (2 * q + hh) * NT + threadIdx.x;
            i = i < n ? i : n - 1;
            h[hh] = thi[i];
            l[hh] = tlo[i];
        }
        xh[q] = make_float2(h[0].x, h[1].x);
        yh[q] = make_float2(h[0].y, h[1].y);
        zh[q] = make_float2(h[0].z, h[1].z);
        xl[q] = make_float2(l[0].x, l[1].x);
        yl[q] = make_float2(l[0].y, l[1].y);
        zl[q] = make_float2(l[0].z, l[1].z);
    }
#pragma unroll
    for (int t = 0; t < 2 * NP; ++t)
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[t][c] = comp[t][c] = 0.f;
    for (int64_t jt = j_begin; jt < j_end; jt += NT) {
        __syncthreads();
        {
            const int64_t j = jt + threadIdx.x;
            const bool valid = j < j_end;
            const int64_t jc = valid ? j : j_begin;
            const float4 h = hi[jc], l = lo[jc];
            const float fx = valid ? (float)f[3 * jc] : 0.f;
            const float fy = valid ? (float)f[3 * jc + 1] : 0.f;
            const float fz = valid ? (float)f[3 * jc + 2] : 0.f;
            stage_x2(sP + kX2SmemFloat4PerSource * threadIdx.x, h, l, fx, fy, fz);
        }
        __syncthreads();
        float2 ax[NP], ay[NP], az[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) ax[q] = ay[q] = az[q] = make_float2(0.f, 0.f);
        // the staged sources of this tile (chunks may be shorter than NT)
        const int cnt = j_end - jt < NT ? (int)(j_end - jt) : NT;
#pragma unroll 2
        for (int s = 0; s < cnt; ++s) {
            const float4 *P = sP + kX2SmemFloat4PerSource * s;
            const float4 P0 = P[0], P1 = P[1], P2 = P[2], P3 = P[3], P4 = P[4];
            const float2 nxh = make_float2(P0.x, P0.y), nyh = make_float2(P0.z, P0.w);
            const float2 zj = make_float2(P1.x, P1.y), zz = make_float2(P1.z, P1.w);
            const float2 nxl = make_float2(P2.x, P2.y), nyl = make_float2(P2.z, P2.w);
            const float2 nzl = make_float2(P3.x, P3.y), fx = make_float2(P3.z, P3.w);
            const float2 fy = make_float2(P4.x, P4.y), fz = make_float2(P4.z, P4.w);
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const float2 dx = add2(add2(xh[q], nxh), add2(xl[q], nxl));
                const float2 dy = add2(add2(yh[q], nyh), add2(yl[q], nyl));
                const float2 dz = add2(fma2(zj, k.m1, zh[q]), add2(zl[q], nzl));
                const float2 dxy2 = fma2(dy, dy, fma2(dx, dx, k.tiny));
                const Mob<float2> m = mob_coefs2<WALL, kNear>(dz, dxy2, zh[q], zj, zz, k);
                mob_apply2<WALL>(m, dx, dy, dz, fx, fy, fz, ax[q], ay[q], az[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            kahan_add(sum[2 * q][0], comp[2 * q][0], ax[q].x);
            kahan_add(sum[2 * q][1], comp[2 * q][1], ay[q].x);
            kahan_add(sum[2 * q][2], comp[2 * q][2], az[q].x);
            kahan_add(sum[2 * q + 1][0], comp[2 * q + 1][0], ax[q].y);
            kahan_add(sum[2 * q + 1][1], comp[2 * q + 1][1], ay[q].y);
            kahan_add(sum[2 * q + 1][2], comp[2 * q + 1][2], az[q].y);
        }
    }
#pragma unroll
    for (int t = 0; t < 2 * NP; ++t) {
        const int64_t i = (int64_t)tb * NT * 2 * NP + t * NT + threadIdx.x;
        if (i < n) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                out[3 * i + c] = m * ((double)sum[t][c] - (double)comp[t][c]);
        }
    }
}

// FP64 item: one target per thread, sources staged as six double arrays.
template <bool WALL, int NT>
__device__ __forceinline__ void f64_item(double *__restrict__ sm, const double *__restrict__ tr,
                                         int64_t n, const double *__restrict__ r,
                                         const double *__restrict__ f, int tb,
                                         int64_t j_begin, int64_t j_end,
                                         const MobConsts<double> &k, double *__restrict__ out,
                                         double m)
{
    double *sx = sm, *sy = sm + NT, *sz = sm + 2 * NT, *sfx = sm + 3 * NT, *sfy = sm + 4 * NT,
           *sfz = sm + 5 * NT;
    const int64_t i = (int64_t)tb * NT + threadIdx.x;
    const int64_t ic = i < n ? i : n - 1;
    const double xi = tr[3 * ic], yi = tr[3 * ic + 1], zi = tr[3 * ic + 2];
    double ux = 0.0, uy = 0.0, uz = 0.0;
    for (int64_t jt = j_begin; jt < j_end; jt += NT) {
        __syncthreads();
        {
            const int64_t j = jt + threadIdx.x;
            const bool valid = j < j_end;
            const int64_t jc = valid ? j : j_begin;
            sx[threadIdx.x] = r[3 * jc];
            sy[threadIdx.x] = r[3 * jc + 1];
            sz[threadIdx.x] = r[3 * jc + 2];
            sfx[threadIdx.x] = valid ? f[3 * jc] : 0.0;
            sfy[threadIdx.x] = valid ? f[3 * jc + 1] : 0.0;
            sfz[threadIdx.x] = valid ? f[3 * jc + 2] : 0.0;
        }
        __syncthreads();
        // the staged sources of this tile (chunks may be shorter than NT)
        const int cnt = j_end - jt < NT ? (int)(j_end - jt) : NT;
#pragma unroll 2
        for (int s = 0; s < cnt; ++s) {
            const double dx = xi - sx[s], dy = yi - sy[s], dz = zi - sz[s];
            const Mob<double> m = mob_coefs<WALL>(dx, dy, dz, zi, sz[s], k);
            mob_apply<WALL>(m, dx, dy, dz, sfx[s], sfy[s], sfz[s], ux, uy, uz);
        }
    }
    if (i < n) {
        out[3 * i] = m * ux;
        out[3 * i + 1] = m * uy;
        out[3 * i + 2] = m * uz;
    }
}

// A source of the symmetric item, every operand in both halves of a float2.
struct SrcX2 {
    float2 nx, ny, z, fx, fy, fz;  // -x, -y, z (hi parts), force
    float2 nxl, nyl, nzl;          // - lo parts (kNear only)
    float2 zz;                     // -2 z^2 (wall only)
};

// With the wall the sources are staged duplicated, as in x2_item: the FMA pipe
// bounds the item and every register move would add to the issue.  Without it
// an item does less than half the arithmetic, and its rotated shared-memory
// reads (four wavefronts per float4, all warps of the SM in turn) and shuffles
// bound it instead: three float4 a source,
//   (-x_hi, -y_hi, z_hi, f_x)  (f_y, f_z, -, -)  (-x_lo, -y_lo, -z_lo, -),
// of which a far item reads one and a half, and moves to duplicate them.
// Without the wall: 20,011 blobs 338 -> 323 us, 65,536 2.93 -> 2.77 ms.
template <bool WALL>
__device__ __forceinline__ void stage_sym(float4 *sP, int slot, float4 h, float4 l, float fx, float fy,
                                          float fz)
{
    if (WALL) {
        stage_x2(sP + kX2SmemFloat4PerSource * slot, h, l, fx, fy, fz);
        return;
    }
    float4 *d = sP + 3 * slot;
    d[0] = make_float4(-h.x, -h.y, h.z, fx);
    d[1] = make_float4(fy, fz, 0.f, 0.f);
    d[2] = make_float4(-l.x, -l.y, -l.z, 0.f);
}

template <bool WALL, bool LO>
__device__ __forceinline__ SrcX2 load_sym(const float4 *sP, int slot)
{
    SrcX2 q;
    if (WALL) {
        const float4 *P = sP + kX2SmemFloat4PerSource * slot;
        const float4 P0 = P[0], P1 = P[1], P3 = P[3], P4 = P[4];
        q.nx = make_float2(P0.x, P0.y);
        q.ny = make_float2(P0.z, P0.w);
        q.z = make_float2(P1.x, P1.y);
        q.zz = make_float2(P1.z, P1.w);
        q.fx = make_float2(P3.z, P3.w);
        q.fy = make_float2(P4.x, P4.y);
        q.fz = make_float2(P4.z, P4.w);
        if (LO) {
            const float4 P2 = P[2];
            q.nxl = make_float2(P2.x, P2.y);
            q.nyl = make_float2(P2.z, P2.w);
            q.nzl = make_float2(P3.x, P3.y);
        }
    } else {
        const float4 *P = sP + 3 * slot;
        const float4 A = P[0];
        const float2 B = *(const float2 *)(P + 1);
        q.nx = splat2(A.x);
        q.ny = splat2(A.y);
        q.z = splat2(A.z);
        q.fx = splat2(A.w);
        q.fy = splat2(B.x);
        q.fz = splat2(B.y);
        if (LO) {
            const float4 D = P[2];
            q.nxl = splat2(D.x);
            q.nyl = splat2(D.y);
            q.nzl = splat2(D.z);
        }
    }
    return q;
}

// Symmetric packed item over half of block pair (I, J), I <= J, blocks of 2*NT
// blobs (two targets per thread, as in x2_item with NP = 1; NT sources).  Each unordered pair
// is evaluated once.  Forward contributions accumulate in the thread's
// registers (tile sums folded Kahan-style).  Reverse contributions use a
// rotating schedule inside each group of 32 staged sources: at step t lane l
// pairs its targets with source (l + t) mod 32, adds the reverse term into a
// packed accumulator, and passes that accumulator to lane l - 1; after 32
// steps lane l holds source l's sum over the warp's 64 targets (no per-source
// reduction).  The warps' sums are added in a fixed order in shared memory
// and then to u with FP64 atomics.  Diagonal items (I == J) run forward only
// over all ordered pairs.  u must be zeroed beforehand and receives
// scale * M f.
//
// LEVEL: how far apart the blocks' bounding boxes are known to be (mob_coefs2).
// From kFar on the separations take the hi parts alone, whose rounding then
// moves a separation by at most 2^-18 of itself.
template <bool WALL, int NT, int LEVEL = kNear>
__device__ __forceinline__ void x2sym_item(float4 *__restrict__ sP, float *__restrict__ sRev,
                                           const float4 *__restrict__ hi,
                                           const float4 *__restrict__ lo,
                                           const double *__restrict__ f, int64_t n, int64_t I,
                                           int64_t J, const MobConsts2 &k,
                                           double *__restrict__ u, double scale, int half)
{
    const int64_t j0 = J * 2 * NT + half * NT;
    if (j0 >= n) return;
    constexpr int NW = NT / 32;
    // Blocks of 64 and 128 blobs: FP32 sums over 16 steps instead of 32 to 64,
    // and but for blocks of 128 with the wall one rounding a term
    // (mob_apply2).  These sizes replace kernels whose sums held 16 to 32 terms.
    constexpr bool FINE = NT <= 64, ONCE = NT == 32 || (NT == 64 && !WALL);
    constexpr int kRun = FINE ? 16 : 32;  // steps between folds within a group
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool diag = I == J;
    const int64_t ia = I * 2 * NT + threadIdx.x, ib = ia + NT;
    float2 xh, yh, zh, xl, yl, zl, fix, fiy, fiz;
    {
        const int64_t ca = ia < n ? ia : n - 1, cb = ib < n ? ib : n - 1;
        const float4 ha = hi[ca], hb = hi[cb], la = lo[ca], lb = lo[cb];
        xh = make_float2(ha.x, hb.x); yh = make_float2(ha.y, hb.y); zh = make_float2(ha.z, hb.z);
        xl = make_float2(la.x, lb.x); yl = make_float2(la.y, lb.y); zl = make_float2(la.z, lb.z);
        // padding targets carry no force, so their reverse contributions vanish
        fix = make_float2(ia < n ? (float)f[3 * ia] : 0.f, ib < n ? (float)f[3 * ib] : 0.f);
        fiy = make_float2(ia < n ? (float)f[3 * ia + 1] : 0.f, ib < n ? (float)f[3 * ib + 1] : 0.f);
        fiz = make_float2(ia < n ? (float)f[3 * ia + 2] : 0.f, ib < n ? (float)f[3 * ib + 2] : 0.f);
    }
    float sum[2][3], comp[2][3];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[t][c] = comp[t][c] = 0.f;
    __syncthreads();
    {
        const int64_t j = j0 + threadIdx.x;
        const bool valid = j < n;
        const int64_t jc = valid ? j : j0;
        const float4 h = hi[jc], l = lo[jc];
        const float fx = valid ? (float)f[3 * jc] : 0.f;
        const float fy = valid ? (float)f[3 * jc + 1] : 0.f;
        const float fz = valid ? (float)f[3 * jc + 2] : 0.f;
        stage_sym<WALL>(sP, threadIdx.x, h, l, fx, fy, fz);
    }
    __syncthreads();
    float2 ax = make_float2(0.f, 0.f), ay = ax, az = ax;
    auto fold = [&]() {
        kahan_add(sum[0][0], comp[0][0], ax.x);
        kahan_add(sum[0][1], comp[0][1], ay.x);
        kahan_add(sum[0][2], comp[0][2], az.x);
        kahan_add(sum[1][0], comp[1][0], ax.y);
        kahan_add(sum[1][1], comp[1][1], ay.y);
        kahan_add(sum[1][2], comp[1][2], az.y);
        ax = ay = az = make_float2(0.f, 0.f);
    };
    if (diag) {
        for (int s0 = 0; s0 < NT; s0 += FINE ? kRun : NT) {
#pragma unroll 2
            for (int s = s0; s < s0 + (FINE ? kRun : NT); ++s) {
                const SrcX2 q = load_sym<WALL, true>(sP, s);
                const float2 dx = add2(add2(xh, q.nx), add2(xl, q.nxl));
                const float2 dy = add2(add2(yh, q.ny), add2(yl, q.nyl));
                const float2 dz = add2(fma2(q.z, k.m1, zh), add2(zl, q.nzl));
                const float2 dxy2 = fma2(dy, dy, fma2(dx, dx, k.tiny));
                const Mob<float2> m = mob_coefs2<WALL, kNear>(dz, dxy2, zh, q.z, q.zz, k);
                mob_apply2<WALL, false, ONCE>(m, dx, dy, dz, q.fx, q.fy, q.fz, ax, ay, az);
            }
            if (FINE) fold();
        }
    } else {
        for (int g = 0; g < NT / 32; ++g) {
            float2 rx = make_float2(0.f, 0.f), ry = rx, rz = rx;
            float run[3] = {0.f, 0.f, 0.f};  // FINE: sums of the first run of steps
            for (int t0 = 0; t0 < 32; t0 += kRun) {
#pragma unroll 2
                for (int t = t0; t < t0 + kRun; ++t) {
                    const int s = g * 32 + ((lane + t) & 31);
                    const SrcX2 q = load_sym<WALL, LEVEL == kNear>(sP, s);
                    float2 dx = add2(xh, q.nx);
                    float2 dy = add2(yh, q.ny);
                    float2 dz = fma2(q.z, k.m1, zh);
                    if (LEVEL == kNear) {
                        dx = add2(dx, add2(xl, q.nxl));
                        dy = add2(dy, add2(yl, q.nyl));
                        dz = add2(dz, add2(zl, q.nzl));
                    }
                    const float2 dxy2 = fma2(dy, dy, LEVEL == kNear ? fma2(dx, dx, k.tiny)
                                                                    : mul2(dx, dx));
                    const Mob<float2> m = mob_coefs2<WALL, LEVEL>(dz, dxy2, zh, q.z, q.zz, k);
                    mob_apply2<WALL, false, ONCE>(m, dx, dy, dz, q.fx, q.fy, q.fz, ax, ay, az);
                    mob_apply2<WALL, true, ONCE>(m, dx, dy, dz, fix, fiy, fiz, rx, ry, rz);
                    // hand the accumulator to lane - 1, which meets this source next step
                    const int from = (lane + 1) & 31;
                    rx.x = __shfl_sync(0xffffffffu, rx.x, from);
                    rx.y = __shfl_sync(0xffffffffu, rx.y, from);
                    ry.x = __shfl_sync(0xffffffffu, ry.x, from);
                    ry.y = __shfl_sync(0xffffffffu, ry.y, from);
                    rz.x = __shfl_sync(0xffffffffu, rz.x, from);
                    rz.y = __shfl_sync(0xffffffffu, rz.y, from);
                }
                if (FINE) fold();
                if (FINE && t0 == 0) {
                    run[0] = rx.x + rx.y;
                    run[1] = ry.x + ry.y;
                    run[2] = rz.x + rz.y;
                    rx = ry = rz = make_float2(0.f, 0.f);
                }
            }
            float *o3 = sRev + 3 * (warp * NT + g * 32 + lane);
            const float2 rev[3] = {rx, ry, rz};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o3[c] = rev[c].x + rev[c].y;
                // after half a round lane l held the sums of source l + 16
                if (FINE) o3[c] += __shfl_xor_sync(0xffffffffu, run[c], 16);
            }
        }
    }
    if (!FINE) fold();
    if (!diag) {
        __syncthreads();
        const int64_t j = j0 + threadIdx.x;
        if (j < n) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float acc = 0.f;
#pragma unroll
                for (int w = 0; w < NW; ++w) acc += sRev[3 * (w * NT + threadIdx.x) + c];
                atomicAdd(u + 3 * j + c, scale * (double)acc);
            }
        }
    }
    if (ia < n)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            atomicAdd(u + 3 * ia + c, scale * ((double)sum[0][c] - (double)comp[0][c]));
    if (ib < n)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            atomicAdd(u + 3 * ib + c, scale * ((double)sum[1][c] - (double)comp[1][c]));
}

// Symmetric double-float item over half of block pair (I, J), I <= J, blocks
// of 2 NT blobs: the scheme of x2sym_item (two targets per thread, rotating
// reverse sums) in packed double-float.  Sources are staged as seven float4
// (x, y, z, fx, fy, fz, -2 z^2, each hi, hi, lo, lo; the 112-byte stride keeps
// the rotated reads conflict-free) of NT sources in sD; sRev holds
// 3 NT (NT / 32) doubles, one sum per warp, source and component.  u must be
// zeroed and receives scale * M f.
template <bool WALL, int NT, bool FAR = false>
__device__ __forceinline__ void dfsym_item(float4 *__restrict__ sD, double *__restrict__ sRev,
                                           const float4 *__restrict__ hi,
                                           const float4 *__restrict__ lo,
                                           const double *__restrict__ f, int64_t n, int64_t I,
                                           int64_t J, int half, const MobConstsDf &k,
                                           double *__restrict__ u, double scale)
{
    const int64_t j0 = J * 2 * NT + half * NT;
    if (j0 >= n) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool diag = I == J;
    const int64_t ia = I * 2 * NT + threadIdx.x, ib = ia + NT;
    dfl2 xi, yi, zi, gx, gy, gz, ux, uy, uz;
    {
        const int64_t ca = ia < n ? ia : n - 1, cb = ib < n ? ib : n - 1;
        const float4 ha = hi[ca], hb = hi[cb], la = lo[ca], lb = lo[cb];
        xi = dfl2(make_float2(ha.x, hb.x), make_float2(la.x, lb.x));
        yi = dfl2(make_float2(ha.y, hb.y), make_float2(la.y, lb.y));
        zi = dfl2(make_float2(ha.z, hb.z), make_float2(la.z, lb.z));
        // padding targets carry no force, so their reverse contributions vanish
        dfl g[2][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            g[0][c] = ia < n ? dfl(f[3 * ia + c]) : dfl();
            g[1][c] = ib < n ? dfl(f[3 * ib + c]) : dfl();
        }
        gx = dfl2(make_float2(g[0][0].hi, g[1][0].hi), make_float2(g[0][0].lo, g[1][0].lo));
        gy = dfl2(make_float2(g[0][1].hi, g[1][1].hi), make_float2(g[0][1].lo, g[1][1].lo));
        gz = dfl2(make_float2(g[0][2].hi, g[1][2].hi), make_float2(g[0][2].lo, g[1][2].lo));
    }
    __syncthreads();
    {
        const int64_t j = j0 + threadIdx.x;
        const bool valid = j < n;
        const int64_t jc = valid ? j : j0;
        const float4 h = hi[jc], l = lo[jc];
        const double z = (double)h.z + (double)l.z;
        const dfl v[7] = {dfl(h.x, l.x), dfl(h.y, l.y), dfl(h.z, l.z),
                          valid ? dfl(f[3 * jc]) : dfl(), valid ? dfl(f[3 * jc + 1]) : dfl(),
                          valid ? dfl(f[3 * jc + 2]) : dfl(), dfl(-2.0 * z * z)};
#pragma unroll
        for (int c = 0; c < 7; ++c)
            sD[7 * threadIdx.x + c] = make_float4(v[c].hi, v[c].hi, v[c].lo, v[c].lo);
    }
    __syncthreads();
    auto src = [&](int s, int c) {
        const float4 q = sD[7 * s + c];
        return dfl2(make_float2(q.x, q.y), make_float2(q.z, q.w));
    };
    if (diag) {
#pragma unroll 1
        for (int s = 0; s < NT; ++s) {
            const dfl2 zj = src(s, 2);
            const dfl2 dx = xi - src(s, 0), dy = yi - src(s, 1), dz = zi - zj;
            const Mob<dfl2> m = mob_coefs_df<WALL, false>(dx, dy, dz, zi, zj, src(s, 6), k);
            mob_apply_df<WALL>(m, dx, dy, dz, src(s, 3), src(s, 4), src(s, 5), ux, uy, uz);
            if ((s & 31) == 31) {
                renorm(ux);
                renorm(uy);
                renorm(uz);
            }
        }
    } else {
        const int from = (lane + 1) & 31;
        auto pass = [&](dfl2 &v) {
            v.hi.x = __shfl_sync(0xffffffffu, v.hi.x, from);
            v.hi.y = __shfl_sync(0xffffffffu, v.hi.y, from);
            v.lo.x = __shfl_sync(0xffffffffu, v.lo.x, from);
            v.lo.y = __shfl_sync(0xffffffffu, v.lo.y, from);
        };
        for (int g = 0; g < NT / 32; ++g) {
            dfl2 vx, vy, vz;
#pragma unroll 1
            for (int t = 0; t < 32; ++t) {
                const int s = g * 32 + ((lane + t) & 31);
                const dfl2 zj = src(s, 2);
                const dfl2 dx = xi - src(s, 0), dy = yi - src(s, 1), dz = zi - zj;
                const Mob<dfl2> m = mob_coefs_df<WALL, FAR>(dx, dy, dz, zi, zj, src(s, 6), k);
                mob_apply_df<WALL>(m, dx, dy, dz, src(s, 3), src(s, 4), src(s, 5), ux, uy, uz);
                mob_apply_df<WALL, true>(m, dx, dy, dz, gx, gy, gz, vx, vy, vz);
                pass(vx);
                pass(vy);
                pass(vz);
            }
            double *o3 = sRev + 3 * (warp * NT + g * 32 + lane);
            o3[0] = sum_halves(vx);
            o3[1] = sum_halves(vy);
            o3[2] = sum_halves(vz);
            // the sums are unnormalised: renormalised every 32 terms
            renorm(ux);
            renorm(uy);
            renorm(uz);
        }
        __syncthreads();
        const int64_t j = j0 + threadIdx.x;
        if (j < n) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double acc = 0.0;
#pragma unroll
                for (int w = 0; w < NT / 32; ++w) acc += sRev[3 * (w * NT + threadIdx.x) + c];
                atomicAdd(u + 3 * j + c, scale * acc);
            }
        }
    }
    const dfl2 acc[3] = {ux, uy, uz};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (ia < n)
            atomicAdd(u + 3 * ia + c, scale * ((double)acc[c].hi.x + (double)acc[c].lo.x));
        if (ib < n)
            atomicAdd(u + 3 * ib + c, scale * ((double)acc[c].hi.y + (double)acc[c].lo.y));
    }
}

// FP64 symmetric item of one warp: blob block I (32 targets, one per lane)
// against C sources (C divides 32) starting at j0, a part of block J >= I.
// Sources are staged as six FP64 arrays in sm (6 C).  Each unordered pair is
// evaluated once for both blobs: at step t lane l meets source (l + t) mod C,
// and the reverse sums move to lane l - 1 within the groups of C lanes after
// each step, so that after C steps lane l holds source (l mod C)'s sum over
// its group's targets; the groups are then added.  The targets' sums are added
// to u and the sources' to v with FP64 atomics; both must be zeroed beforehand,
// and may be the same array.  A diagonal item (I == J) runs forward only over
// all ordered pairs.
template <bool WALL, int C>
__device__ __forceinline__ void f64sym_item(double *__restrict__ sm, const double *__restrict__ r,
                                            const double *__restrict__ f, int64_t n, int64_t I,
                                            int64_t j0, bool diag, const MobConsts<double> &k,
                                            double *u, double *v, double scale)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = I * 32 + lane, ic = i < n ? i : n - 1;
    const double xi = r[3 * ic], yi = r[3 * ic + 1], zi = r[3 * ic + 2];
    // padding targets and sources carry no force, so they add nothing
    const double gx = i < n ? f[3 * i] : 0.0, gy = i < n ? f[3 * i + 1] : 0.0,
                 gz = i < n ? f[3 * i + 2] : 0.0;
    if (lane < C) {
        const int64_t j = j0 + lane, jc = j < n ? j : j0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sm[c * C + lane] = r[3 * jc + c];
            sm[(3 + c) * C + lane] = j < n ? f[3 * jc + c] : 0.0;
        }
    }
    __syncwarp();
    double ux = 0.0, uy = 0.0, uz = 0.0;
    if (diag) {
#pragma unroll 1
        for (int s = 0; s < C; ++s) {
            const double dx = xi - sm[s], dy = yi - sm[C + s], zj = sm[2 * C + s], dz = zi - zj;
            const Mob<double> m = mob_coefs<WALL>(dx, dy, dz, zi, zj, k);
            mob_apply<WALL>(m, dx, dy, dz, sm[3 * C + s], sm[4 * C + s], sm[5 * C + s], ux, uy, uz);
        }
    } else {
        double vx = 0.0, vy = 0.0, vz = 0.0;
        const int from = (lane & ~(C - 1)) | ((lane + 1) & (C - 1));
#pragma unroll 1
        for (int t = 0; t < C; ++t) {
            const int s = (lane + t) & (C - 1);
            const double dx = xi - sm[s], dy = yi - sm[C + s], zj = sm[2 * C + s], dz = zi - zj;
            const Mob<double> m = mob_coefs<WALL>(dx, dy, dz, zi, zj, k);
            mob_apply<WALL>(m, dx, dy, dz, sm[3 * C + s], sm[4 * C + s], sm[5 * C + s], ux, uy, uz);
            mob_apply<WALL, true>(m, dx, dy, dz, gx, gy, gz, vx, vy, vz);
            vx = __shfl_sync(0xffffffffu, vx, from);
            vy = __shfl_sync(0xffffffffu, vy, from);
            vz = __shfl_sync(0xffffffffu, vz, from);
        }
#pragma unroll
        for (int o = C; o < 32; o <<= 1) {
            vx += __shfl_xor_sync(0xffffffffu, vx, o);
            vy += __shfl_xor_sync(0xffffffffu, vy, o);
            vz += __shfl_xor_sync(0xffffffffu, vz, o);
        }
        const int64_t j = j0 + lane;
        if (lane < C && j < n) {
            atomicAdd(v + 3 * j, scale * vx);
            atomicAdd(v + 3 * j + 1, scale * vy);
            atomicAdd(v + 3 * j + 2, scale * vz);
        }
    }
    if (i < n) {
        atomicAdd(u + 3 * i, scale * ux);
        atomicAdd(u + 3 * i + 1, scale * uy);
        atomicAdd(u + 3 * i + 2, scale * uz);
    }
}

}  // namespace mb
