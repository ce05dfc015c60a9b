// Device-side blob-blob mobility of the wall-corrected RPY tensor.
//
// Everything here is in units of (6 pi eta a)^-1; callers scale at the end.
//
// Free space (Eq. RPYTensor), with d = r_i - r_j, r = |d|:
//   r >  2a: C I + D' d d^T,  C = (3a/4)/r + (a^3/2)/r^3,
//                             D' = (3a/4)/r^3 - (3a^3/2)/r^5
//   r <= 2a: C = 1 - 9r/(32a), D' = (3/(32a))/r
// (D' is C2/r^2 or C4/r^2, so that D' (d.f) d = C2 (dhat.f) dhat.)
//
// Single no-slip wall at z = 0 (Section 2.1.1): the image part of Blake's
// Green's function with the Faxen operator (1 + a^2/6 Lap) applied at both
// blobs.  Writing R = r_i - (x_j, y_j, -z_j), rho = |R|, e = R/rho,
// hs = z_j/rho, ht = z_i/rho, e3 = hs + ht, E = e3^2, p = hs*ht,
// t2 = a^2/rho^2, t4 = t2^2, that correction is, for unit viscosity,
//   8 pi rho W_ab = f1 d_ab + f2 e_a e_b + f3 e_a d_b3 + f4 d_a3 e_b + f5 d_a3 d_b3
// with (a = velocity component, b = force component)
//   f1 = -1 - 2p + t2 (2E - 2/3)  + t4 (2/3 - 10E/3)
//   f2 = -1 + 6p + t2 (2 - 10E)   + t4 (70E/3 - 10/3)
//   f3 = 2hs + e3 [t2 (20E - 4) + t4 (40/3 - 140E/3) - 12p]
//   f4 = 2hs - (20/3) e3 t4
//   f5 = -4hs^2 - 4E t2 + t4 (20E - 8/3)
// (derived by hand from the two Faxen operators acting on Blake's image
// system; the self term i = j reduces to the Rotne-Prager-Blake self
// mobilities).  In units of (6 pi eta a)^-1 the prefactor 1/(8 pi rho)
// becomes (3a/4)/rho.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "df32.cuh"

namespace mb {

// The regrouped form of the same interaction.  With u = 1/rho, w = u^2,
// X = a^2 w, Q = X^2 / 3, E = R3^2 w, S = X E + Q and c = zi zj w + X / 3, the
// polynomials f1..f5 of the header are
//   f1 / 2     = -1/2 + d1,  d1 = S - 5 E Q - c
//   f2 / 2     = -1/2 + 3 c - 5 S + 35 E Q
//   f3 rho / 2 = t3 = zj - R3 (2 (f2/2) + 1 - 10 Q)
//   f4 rho / 2 = t4 = zj - R3 10 Q
//   f5 / 2     = -2 zj^2 w - 2 S - 2 Q + 30 E Q
// Every coefficient but 1/3 is a small integer or a half, exact in any
// precision, and hs, ht, e3 (three products by 1/rho) are not formed.  The
// block M_ij then has five entries of its own,
//   M_ab = Cx d_ab + H d_a d_b (a, b in x, y),  M_az = Bf d_a,  M_zb = Bb d_b,
//   M_zz = Z,
// with s = (3a/2) u, sw = s w, A2 = sw f2/2:
//   Cx = (3a/4) (1/r - u) + (a^3/2) / r^3 + s d1     H = D' + A2
//   Bf = D' d_z + A2 R3 + sw t3                      Bb = D' d_z + A2 R3 + sw t4
//   Z  = Cx + s f5/2 + D' d_z^2 + R3 (A2 R3 + sw (t3 + t4))
// The Oseen parts of the free and wall terms, which nearly cancel for pairs
// far apart along the wall, meet in 1/r - u before anything is rounded at
// their size.  The transpose (M_ji = M_ij^T) exchanges Bf and Bb.  Both
// directions of a pair take 74 multiplications and additions besides the two
// reciprocal square roots; the formula of the header takes 100.
template <typename T>
struct MobConsts {
    T a2;       // a^2
    T third;    // 1/3
    T d1, s2;   // 3a/4, 3a/2
    T c2, c4;   // far C = d1 inv + c2 inv^3, D' = inv^3 (d1 + c4 inv^2)
    T four_a2;  // 4 a^2: r^2 below this takes the overlap branch
    T k1, k2;   // near C = 1 - k1 r, D' = k2 inv
    T tiny;     // floor on r^2 (coincident blobs, including i = j)

    __host__ static MobConsts make(double a)
    {
        MobConsts k;
        k.a2 = T(a * a);
        k.third = T(1.0 / 3.0);
        k.d1 = T(0.75 * a);
        k.s2 = T(1.5 * a);
        k.c2 = T(0.5 * a * a * a);
        k.c4 = T(-1.5 * a * a * a);
        k.four_a2 = T(4.0 * a * a);
        k.k1 = T(9.0 / (32.0 * a));
        k.k2 = T(3.0 / (32.0 * a));
        k.tiny = std::is_same<T, double>::value ? T(1e-300) : T(1e-30);
        return k;
    }
};

// 1/sqrt(x) in FP64 for x > 0.  FP64 instructions are what the FP64 kernels
// wait for (one per ~19 cycles and SM), conversions between FP32 and FP64
// among them, so the FP32 estimate is taken from x's truncated bits and
// returned to FP64 by integer operations (both exact), and one cubic step
// (Householder's iteration of third order) y + y e (1/2 + 3/8 e),
// e = 1 - x y^2, finishes it in five FP64 instructions: |e| <= 2^-21.4 leaves
// a truncation error of (5/16) e^3 < 2^-65.  x outside the FP32 range (and
// NaN, infinities, zero) takes rsqrt().
__device__ __forceinline__ double rsqrt_pos(double x)
{
    const int h = __double2hiint(x);
    if ((unsigned)(h - 0x38100000) >= 0x47e00000u - 0x38100000u) return rsqrt(x);
    const float xf =
        __int_as_float(((h - 0x38000000) << 3) | (int)((unsigned)__double2loint(x) >> 29));
    const int b = __float_as_int(rsqrt_ftz(xf));
    const double y = __hiloint2double((b >> 3) + 0x38000000, b << 29);
    const double e = fma(-x, y * y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// x < bound for x >= 0 on the bit patterns: an FP64 comparison is an FP64
// instruction.
__device__ __forceinline__ bool below(double x, double bound)
{
    return __double_as_longlong(x) < __double_as_longlong(bound);
}

// Without the wall only Cx = C and H = D' are set.
template <typename T>
struct Mob {
    T Cx, H, Bf, Bb, Z;
};

// Coefficients of one pair at separation d = r_i - r_j, heights zi, zj.
template <bool WALL>
__device__ __forceinline__ Mob<double> mob_coefs(double dx, double dy, double dz, double zi,
                                                 double zj, const MobConsts<double> &k)
{
    Mob<double> m;
    const double dxy2 = fma(dx, dx, dy * dy);
    const double r2 = fma(dz, dz, dxy2);
    double inv = rsqrt_pos(r2);
    const double inv2 = inv * inv, inv3 = inv * inv2;
    double C = k.c2 * inv3, D = inv3 * fma(k.c4, inv2, k.d1);
    if (below(r2, k.four_a2)) {  // overlapping blobs (rare): regularised branch
        const double rr = fmax(r2, k.tiny), ir = rsqrt(rr);
        C = fma(-k.k1, rr * ir, 1.0);
        D = k.k2 * ir;
        inv = 0.0;
    }
    if (!WALL) {
        m.Cx = fma(k.d1, inv, C);
        m.H = D;
        return m;
    }
    const double R3 = zi + zj;
    const double u = rsqrt_pos(fma(R3, R3, dxy2)), w = u * u;
    const double X = k.a2 * w, Q = (X * k.third) * X, E = (R3 * R3) * w;
    const double c = fma(zi * zj, w, X * k.third);
    const double EQ = E * Q, S = fma(X, E, Q);
    const double s = k.s2 * u, sw = s * w;
    m.Cx = fma(k.d1, inv - u, fma(s, fma(-5.0, EQ, S) - c, C));
    const double f2 = fma(35.0, EQ, fma(-5.0, S, fma(3.0, c, -0.5)));
    const double t3 = fma(R3, fma(-2.0, f2, fma(10.0, Q, -1.0)), zj), t4 = fma(R3 * Q, -10.0, zj);
    const double f5 = fma(30.0, EQ, -2.0 * fma(zj * zj, w, S + Q));
    const double A2 = sw * f2, AR = A2 * R3, Dz = D * dz, K = Dz + AR;
    m.H = D + A2;
    m.Bf = fma(sw, t3, K);
    m.Bb = fma(sw, t4, K);
    m.Z = fma(R3, fma(sw, t3 + t4, AR), fma(dz, Dz, fma(s, f5, m.Cx)));
    return m;
}

// The same in FP32.
template <bool WALL>
__device__ __forceinline__ Mob<float> mob_coefs(float dx, float dy, float dz, float zi, float zj,
                                                const MobConsts<float> &k)
{
    Mob<float> m;
    const float dxy2 = fmaf(dx, dx, fmaf(dy, dy, k.tiny));
    const float r2 = fmaf(dz, dz, dxy2);
    float inv = rsqrt_ftz(r2);
    const float inv2 = inv * inv, inv3 = inv * inv2;
    float C = k.c2 * inv3, D = inv3 * fmaf(k.c4, inv2, k.d1);
    if (r2 < k.four_a2) {
        C = fmaf(-k.k1, r2 * inv, 1.f);
        D = k.k2 * inv;
        inv = 0.f;
    }
    if (!WALL) {
        m.Cx = fmaf(k.d1, inv, C);
        m.H = D;
        return m;
    }
    const float R3 = zi + zj;
    const float u = rsqrt_ftz(fmaf(R3, R3, dxy2)), w = u * u;
    const float X = k.a2 * w, X3 = X * k.third, Q = X3 * X, E = (R3 * R3) * w;
    const float c = fmaf(zi * zj, w, X3);
    const float EQ = E * Q, S = fmaf(X, E, Q);
    const float s = k.s2 * u, sw = s * w;
    m.Cx = fmaf(k.d1, inv - u, fmaf(s, fmaf(-5.f, EQ, S) - c, C));
    const float f2 = fmaf(35.f, EQ, fmaf(-5.f, S, fmaf(3.f, c, -0.5f)));
    const float t3 = fmaf(R3, fmaf(-2.f, f2, fmaf(10.f, Q, -1.f)), zj), t4 = fmaf(R3 * Q, -10.f, zj);
    const float f5 = fmaf(30.f, EQ, -2.f * fmaf(zj * zj, w, S + Q));
    const float A2 = sw * f2, AR = A2 * R3, Dz = D * dz, K = Dz + AR;
    m.H = D + A2;
    m.Bf = fmaf(sw, t3, K);
    m.Bb = fmaf(sw, t4, K);
    m.Z = fmaf(R3, fmaf(sw, t3 + t4, AR), fmaf(dz, Dz, fmaf(s, f5, m.Cx)));
    return m;
}

// u += M f from the coefficients; TRANS: u += M^T f.
template <bool WALL, bool TRANS = false, typename T>
__device__ __forceinline__ void mob_apply(const Mob<T> &m, T dx, T dy, T dz, T fx, T fy, T fz,
                                          T &ux, T &uy, T &uz)
{
    const T rf = fma(dx, fx, dy * fy);
    const T G = WALL ? fma(m.H, rf, (TRANS ? m.Bb : m.Bf) * fz) : m.H * fma(dz, fz, rf);
    if (std::is_same<T, float>::value) {
        // one rounding at the size of the sum instead of two (sums of up to
        // 256 terms: error of a 20,011-blob product 4.1e-7 -> 3.0e-7)
        ux += fma(m.Cx, fx, G * dx);
        uy += fma(m.Cx, fy, G * dy);
        uz += WALL ? fma(m.Z, fz, (TRANS ? m.Bf : m.Bb) * rf) : fma(m.Cx, fz, G * dz);
        return;
    }
    ux = fma(m.Cx, fx, fma(G, dx, ux));
    uy = fma(m.Cx, fy, fma(G, dy, uy));
    uz = WALL ? fma(m.Z, fz, fma(TRANS ? m.Bf : m.Bb, rf, uz)) : fma(m.Cx, fz, fma(G, dz, uz));
}

// Full 3x3 block M_ij in FP64, row-major m[3*alpha + beta] (alpha = velocity
// component of i, beta = force component of j).  Used to assemble the
// per-body blocks of the preconditioner.
template <bool WALL>
__device__ __forceinline__ void block_f64(const double *ri, const double *rj,
                                          const MobConsts<double> &k, double m[9])
{
    const double dx = ri[0] - rj[0], dy = ri[1] - rj[1], dz = ri[2] - rj[2];
    const Mob<double> c = mob_coefs<WALL>(dx, dy, dz, ri[2], rj[2], k);
    const double hx = c.H * dx, hy = c.H * dy, hz = c.H * dz;
    m[0] = fma(hx, dx, c.Cx);
    m[1] = m[3] = hx * dy;
    m[4] = fma(hy, dy, c.Cx);
    m[2] = dx * (WALL ? c.Bf : hz);
    m[5] = dy * (WALL ? c.Bf : hz);
    m[6] = dx * (WALL ? c.Bb : hz);
    m[7] = dy * (WALL ? c.Bb : hz);
    m[8] = WALL ? c.Z : fma(hz, dz, c.Cx);
}

// ---------------------------------------------------------------------------
// Packed variant: the same pair interaction for two targets at once, one in
// each half of a float2, with Blackwell's paired FP32 instructions
// (fma/add/mul .f32x2).  Every source operand arrives duplicated in both
// halves.
struct MobConsts2 {
    float2 a2, third, d1, s2, c2, c4, tiny;
    float four_a2, k1, k2;
    // small integers and halves of the wall polynomials
    float2 m1, mhalf, m2, p3, m5, p10, m10, p30, p35;

    __host__ static MobConsts2 make(double a)
    {
        auto d = [](double v) { return make_float2((float)v, (float)v); };
        MobConsts2 k;
        k.a2 = d(a * a);
        k.third = d(1.0 / 3.0);
        k.d1 = d(0.75 * a);
        k.s2 = d(1.5 * a);
        k.c2 = d(0.5 * a * a * a);
        k.c4 = d(-1.5 * a * a * a);
        k.tiny = d(1e-30);
        k.four_a2 = (float)(4.0 * a * a);
        k.k1 = (float)(9.0 / (32.0 * a));
        k.k2 = (float)(3.0 / (32.0 * a));
        k.m1 = d(-1.0); k.mhalf = d(-0.5); k.m2 = d(-2.0); k.p3 = d(3.0); k.m5 = d(-5.0);
        k.p10 = d(10.0); k.m10 = d(-10.0); k.p30 = d(30.0); k.p35 = d(35.0);
        return k;
    }
};

__device__ __forceinline__ float2 rsqrt2(float2 a)
{
    return make_float2(rsqrt_ftz(a.x), rsqrt_ftz(a.y));
}

// How far the targets and sources of an item are known to be apart:
//   kNear     nothing is known: overlap test (a warp vote), hi and lo parts of
//             the separations
//   kFar      beyond 2 a and 2^18 ulp of the largest coordinate: no overlap
//             test, and the caller forms the separations from the hi parts
//   kVeryFar  beyond kVeryFarRadii radii as well: X < 2^-15, so the terms in
//             X^2 (at most 35/3 X^2 of f2/2 = -1/2 + ...) are below 2^-26 and
//             are left out
enum { kNear = 0, kFar = 1, kVeryFar = 2 };
constexpr float kVeryFarRadii = 192.f;

// Coefficients for the two targets in the halves, one source: heights zt, zj
// and zz = -2 zj^2; dxy2 = dx^2 + dy^2 already includes the tiny floor at
// kNear (it keeps r^2 > 0 for i = j).
template <bool WALL, int LEVEL>
__device__ __forceinline__ Mob<float2> mob_coefs2(float2 dz, float2 dxy2, float2 zt, float2 zj,
                                                  float2 zz, const MobConsts2 &k)
{
    Mob<float2> m;
    const float2 r2 = fma2(dz, dz, dxy2);
    float2 inv = rsqrt2(r2);
    const float2 inv2 = mul2(inv, inv), inv3 = mul2(inv, inv2);
    float2 C = mul2(k.c2, inv3), D = mul2(inv3, fma2(k.c4, inv2, k.d1));
    if (LEVEL == kNear && __any_sync(0xffffffffu, (r2.x < k.four_a2) | (r2.y < k.four_a2))) {
        // overlapping blobs (rare): regularised branch, lane by lane
        if (r2.x < k.four_a2) {
            C.x = 1.f - k.k1 * (r2.x * inv.x);
            D.x = k.k2 * inv.x;
            inv.x = 0.f;
        }
        if (r2.y < k.four_a2) {
            C.y = 1.f - k.k1 * (r2.y * inv.y);
            D.y = k.k2 * inv.y;
            inv.y = 0.f;
        }
    }
    if (!WALL) {
        m.Cx = fma2(k.d1, inv, C);
        m.H = D;
        return m;
    }
    const float2 R3 = add2(zt, zj);
    const float2 u = rsqrt2(fma2(R3, R3, dxy2)), w = mul2(u, u);
    const float2 X = mul2(k.a2, w), X3 = mul2(X, k.third), E = mul2(mul2(R3, R3), w);
    const float2 c = fma2(mul2(zt, zj), w, X3);
    const float2 s = mul2(k.s2, u), sw = mul2(s, w);
    const float2 f2c = fma2(c, k.p3, k.mhalf), zw = mul2(zz, w);
    float2 d1, f2, f5, t3, t4;
    if (LEVEL == kVeryFar) {
        const float2 S = mul2(X, E);
        d1 = fma2(c, k.m1, S);
        f2 = fma2(k.m5, S, f2c);
        f5 = fma2(k.m2, S, zw);
        t3 = fma2(R3, fma2(k.m2, f2, k.m1), zj);
        t4 = zj;
    } else {
        const float2 Q = mul2(X3, X), EQ = mul2(E, Q), S = fma2(X, E, Q);
        d1 = fma2(c, k.m1, fma2(k.m5, EQ, S));
        f2 = fma2(k.p35, EQ, fma2(k.m5, S, f2c));
        f5 = fma2(k.p30, EQ, fma2(k.m2, S, fma2(k.m2, Q, zw)));
        t3 = fma2(R3, fma2(k.m2, f2, fma2(k.p10, Q, k.m1)), zj);
        t4 = fma2(mul2(R3, Q), k.m10, zj);
    }
    m.Cx = fma2(k.d1, fma2(u, k.m1, inv), fma2(s, d1, C));
    const float2 A2 = mul2(sw, f2), AR = mul2(A2, R3), Dz = mul2(D, dz), K = add2(Dz, AR);
    m.H = add2(D, A2);
    m.Bf = fma2(sw, t3, K);
    m.Bb = fma2(sw, t4, K);
    m.Z = fma2(R3, fma2(sw, add2(t3, t4), AR), fma2(dz, Dz, fma2(s, f5, m.Cx)));
    return m;
}

// Double-float, two pairs at once.
struct MobConstsDf {
    dfl2 a2, third, d1, s2, c2, c4, four_a2, k1, k2;

    __host__ static MobConstsDf make(double a)
    {
        MobConstsDf k;
        k.a2 = dfl(a * a);
        k.third = dfl(1.0 / 3.0);
        k.d1 = dfl(0.75 * a);
        k.s2 = dfl(1.5 * a);
        k.c2 = dfl(0.5 * a * a * a);
        k.c4 = dfl(-1.5 * a * a * a);
        k.four_a2 = dfl(4.0 * a * a);
        k.k1 = dfl(-9.0 / (32.0 * a));
        k.k2 = dfl(3.0 / (32.0 * a));
        return k;
    }
};

// The overlap branch, half by half (rare).
__device__ __forceinline__ void overlap_df(dfl2 r2, const MobConstsDf &k, dfl2 &inv, dfl2 &C, dfl2 &D)
{
    dfl2 x = r2;
    if (!(x.hi.x > 1e-30f)) { x.hi.x = 1e-30f; x.lo.x = 0.f; }
    if (!(x.hi.y > 1e-30f)) { x.hi.y = 1e-30f; x.lo.y = 0.f; }
    const dfl2 ir = rsqrt_df(x), Cn = addf(k.k1 * (x * ir), 1.f), Dn = k.k2 * ir;
    const float2 g = add2(sub2(r2.hi, k.four_a2.hi), sub2(r2.lo, k.four_a2.lo));
    if (g.x < 0.f) {
        C.hi.x = Cn.hi.x; C.lo.x = Cn.lo.x;
        D.hi.x = Dn.hi.x; D.lo.x = Dn.lo.x;
        inv.hi.x = inv.lo.x = 0.f;
    }
    if (g.y < 0.f) {
        C.hi.y = Cn.hi.y; C.lo.y = Cn.lo.y;
        D.hi.y = Dn.hi.y; D.lo.y = Dn.lo.y;
        inv.hi.y = inv.lo.y = 0.f;
    }
}

// Coefficients in double-float, zz = -2 zj^2.  FAR (every pair 64 a or more
// apart, so that X < 2^-12 and no pair overlaps): the terms carrying
// X^2 = 3 Q < 2^-24 are summed in FP32 and added to the lo parts; their
// rounding is below 2^-24 X^2 of the polynomials, under the double-float
// rounding of the other terms.
template <bool WALL, bool FAR>
__device__ __forceinline__ Mob<dfl2> mob_coefs_df(dfl2 dx, dfl2 dy, dfl2 dz, dfl2 zi, dfl2 zj,
                                                  dfl2 zz, const MobConstsDf &k)
{
    Mob<dfl2> m;
    const dfl2 dxy2 = dx * dx + dy * dy;
    const dfl2 r2 = dz * dz + dxy2;
    dfl2 inv = rsqrt_df(r2);
    const dfl2 inv2 = inv * inv;
    dfl2 inv3 = inv * inv2;
    renorm(inv3);  // inv3, w and f2 enter most products: their lo parts kept short
    // 3a/4 exceeds (3a^3/2) / r^2 wherever this is used (r > 2a)
    dfl2 C = k.c2 * inv3, D = inv3 * add_ordered(k.d1, k.c4 * inv2);
    if (!FAR) {
        const float2 g = add2(sub2(r2.hi, k.four_a2.hi), sub2(r2.lo, k.four_a2.lo));
        if (g.x < 0.f || g.y < 0.f) overlap_df(r2, k, inv, C, D);
    }
    if (!WALL) {
        m.Cx = k.d1 * inv + C;
        m.H = D;
        return m;
    }
    const dfl2 R3 = zi + zj, H2 = R3 * R3;
    const dfl2 u = rsqrt_df(H2 + dxy2);
    dfl2 w = u * u;
    renorm(w);
    const dfl2 X = k.a2 * w, E = H2 * w, X3 = X * k.third, V = X * E;
    const dfl2 c = (zi * zj) * w + X3, zw = zz * w;
    dfl2 d1, f2, br, t4, f5;
    if (FAR) {
        const float2 Q = mul2(X3.hi, X.hi), EQ = mul2(E.hi, Q);
        d1 = add_lo(V + (-c), fma2(splat2(-5.f), EQ, Q));
        f2 = add_lo(addf(mulf(c, 3.f), -0.5f) + mulf(V, -5.f),
                    fma2(splat2(35.f), EQ, mul2(splat2(-5.f), Q)));
        br = add_lo(addf(mul_pow2(f2, -2.f), -1.f), mul2(splat2(10.f), Q));
        t4 = add_lo(zj, mul2(mul2(splat2(-10.f), Q), R3.hi));
        f5 = add_lo(zw + mul_pow2(V, -2.f), fma2(splat2(30.f), EQ, mul2(splat2(-4.f), Q)));
    } else {
        const dfl2 Q = X3 * X, EQ = E * Q, S = V + Q;
        d1 = (S + mulf(EQ, -5.f)) + (-c);
        f2 = (addf(mulf(c, 3.f), -0.5f) + mulf(S, -5.f)) + mulf(EQ, 35.f);
        br = addf(mul_pow2(f2, -2.f), -1.f) + mulf(Q, 10.f);
        t4 = zj + mulf(R3 * Q, -10.f);
        f5 = (zw + mul_pow2(S + Q, -2.f)) + mulf(EQ, 30.f);
    }
    renorm(f2);
    const dfl2 t3 = R3 * br + zj;
    const dfl2 s = k.s2 * u, sw = s * w;
    m.Cx = (k.d1 * (inv + (-u)) + s * d1) + C;
    const dfl2 A2 = sw * f2, AR = A2 * R3, Dz = D * dz, K = Dz + AR;
    m.H = D + A2;
    m.Bf = sw * t3 + K;
    m.Bb = sw * t4 + K;
    m.Z = ((sw * (t3 + t4) + AR) * R3 + Dz * dz) + (s * f5 + m.Cx);
    return m;
}

// u += M f (TRANS: M^T f), unnormalised sums.
template <bool WALL, bool TRANS = false>
__device__ __forceinline__ void mob_apply_df(const Mob<dfl2> &m, dfl2 dx, dfl2 dy, dfl2 dz,
                                             dfl2 fx, dfl2 fy, dfl2 fz, dfl2 &ux, dfl2 &uy,
                                             dfl2 &uz)
{
    const dfl2 rf = dx * fx + dy * fy;
    const dfl2 G = WALL ? m.H * rf + (TRANS ? m.Bb : m.Bf) * fz : m.H * (rf + dz * fz);
    ux = ux + (m.Cx * fx + G * dx);
    uy = uy + (m.Cx * fy + G * dy);
    uz = uz + (WALL ? m.Z * fz + (TRANS ? m.Bf : m.Bb) * rf : m.Cx * fz + G * dz);
}

// u += M f (TRANS: M^T f) for the two targets in the halves.  ONCE: one
// rounding at the size of the sum instead of two (six instructions more for
// both directions), where there is nothing else to round: sums of a few terms
// that go on in FP64.
template <bool WALL, bool TRANS = false, bool ONCE = false>
__device__ __forceinline__ void mob_apply2(const Mob<float2> &m, float2 dx, float2 dy, float2 dz,
                                           float2 fx, float2 fy, float2 fz, float2 &ux, float2 &uy,
                                           float2 &uz)
{
    const float2 rf = fma2(dx, fx, mul2(dy, fy));
    const float2 G = WALL ? fma2(m.H, rf, mul2(TRANS ? m.Bb : m.Bf, fz))
                          : mul2(m.H, fma2(dz, fz, rf));
    if (ONCE) {
        ux = add2(ux, fma2(m.Cx, fx, mul2(G, dx)));
        uy = add2(uy, fma2(m.Cx, fy, mul2(G, dy)));
        uz = add2(uz, WALL ? fma2(m.Z, fz, mul2(TRANS ? m.Bf : m.Bb, rf))
                           : fma2(m.Cx, fz, mul2(G, dz)));
        return;
    }
    ux = fma2(m.Cx, fx, fma2(G, dx, ux));
    uy = fma2(m.Cx, fy, fma2(G, dy, uy));
    uz = WALL ? fma2(m.Z, fz, fma2(TRANS ? m.Bf : m.Bb, rf, uz))
              : fma2(m.Cx, fz, fma2(G, dz, uz));
}

}  // namespace mb
