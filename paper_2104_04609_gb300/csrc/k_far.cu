// k_far.cu -- matrix-free FP32 far-field apply of the permuted PMCHWT
// operator (Sec. 2.7) for all triangle pairs that share no vertex, with the
// 6-point degree-4 triangle rule (Strang & Fix / Dunavant) on both triangles.
//
// Structure of one apply y = B_far x:
//   1. far_prep_kernel   (per source rule point)  densities at the 6 source
//      points and the surface-curl vector of the phi density, FP32;
//   2. far_kernel        (per test triangle)       N-body sum over all source
//      points staged through shared memory in tiles of triangles; both
//      wavenumbers are evaluated from one distance; the source range is split
//      over gridDim.y so that the grid fills every SM; partial sums per test
//      point (u1, u2) and per test triangle (curl term) go to d_part, d_partA
//      (no atomics);
//   3. gather_kernel     (a group of lanes per vertex)  sums the partials of
//      the test points of the incident triangles with the test weights (FP64)
//      and adds the near-field CSR product (touching pairs, Sauter-Schwab
//      values).
//
// Kernel identities (G = e^{ikr}/(4 pi r), d = x - y, r = |d|):
//   dG/dn_y = H (y - x).n_y,  dG/dn_x = H (x - y).n_x,
//   H = e^{ikr} (ikr - 1) / (4 pi r^3);
//   D (Maue form) = G [curl phi_i . curl phi_j - k^2 (n_x.n_y) phi_i phi_j].
// Because every source point of a flat triangle lies in its plane,
// (x - y).n_y = x.n_y - n_y.P0 is constant over the triangle's six points,
// and so is n_x.n_y; the surface curl of the P1 density is constant per
// triangle.  These per-triangle factors are applied once per (test point,
// source triangle), not per point pair.
#include <algorithm>

#include "osrc_internal.cuh"

namespace {

// 6-point symmetric rule: barycentric (1-2a, a, a) and permutations.
constexpr double kQa1 = 0.445948490915965;
constexpr double kQw1 = 0.223381589678011;
constexpr double kQa2 = 0.091576213509771;
constexpr double kQw2 = 0.109951743655322;

__host__ __device__ inline void rule_point(int q, double bary[3], double &w) {
    const double a = q < 3 ? kQa1 : kQa2;
    w = q < 3 ? kQw1 : kQw2;
    const int i = q % 3;
    for (int j = 0; j < 3; ++j) bary[j] = (j == i) ? 1.0 - 2.0 * a : a;
}

constexpr int FAR_THREADS = 128;
// resident blocks per SM the one-right-hand-side kernel is compiled for
// (registers per thread = 65536 / (FAR_THREADS x FAR_MIN_BLOCKS))
#ifndef OSRC_FAR_MIN_BLOCKS
#define OSRC_FAR_MIN_BLOCKS 2
#endif
// largest k_max x (bounding-box diagonal) for the plain (FP32 k r) variant
constexpr double FAR_PLAIN_MAX_PHASE = 32.0 * 3.14159265358979323846;
constexpr int FAR_TS = 64;  // source triangles per shared-memory tile
#ifndef OSRC_FAR_QUNROLL
#define OSRC_FAR_QUNROLL 3
#endif
#ifndef OSRC_FAR_HUNROLL
#define OSRC_FAR_HUNROLL 2
#endif
constexpr int FAR_QUNROLL = OSRC_FAR_QUNROLL, FAR_HUNROLL = OSRC_FAR_HUNROLL;  // unrolls of the rule-point loops
constexpr int FAR_MIN_TPS = 16;  // fewest source triangles per split
// test triangles per block: 32 below FAR_TRIS32_NT triangles, 64 below
// FAR_TRIS64_NT, else FAR_THREADS (128).  Measured: 5136 triangles on four
// objects 2.136 ms with 128, 2.145 with 64, 2.256 with 32; 296 triangles
// 38 us with 32 sharing the sources between four warps, 46 us without
constexpr int FAR_TRIS32_NT = 2048;
constexpr int FAR_TRIS64_NT = 4096;
constexpr int FAR_MAX_NS = 64;   // most source splits
// lanes of the gather per vertex: a block up to GATHER_BLOCK_NV vertices, a
// warp up to GATHER_WARP_NV, then 8 (150 vertices: block 38 us an apply, warp
// 41; 642: warp 10.28 ms a solve, block 10.38, 8 lanes 10.60; 2568: 8 lanes
// 2.140 ms an apply, warp 2.145)
constexpr int GATHER_BLOCK_NV = 400;
constexpr int GATHER_WARP_NV = 1500;

__global__ void far_geom_kernel(const double *__restrict__ verts, const int *__restrict__ tris,
                                int nt, float4 *__restrict__ pt, float4 *__restrict__ poff,
                                float4 *__restrict__ cen, float4 *__restrict__ tn,
                                int4 *__restrict__ tv, double *__restrict__ tgeo) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    double P[3][3];
    int v[3];
    for (int a = 0; a < 3; ++a) {
        v[a] = tris[3 * t + a];
        for (int j = 0; j < 3; ++j) P[a][j] = verts[3 * v[a] + j];
    }
    double e1[3], e2[3], c[3];
    for (int j = 0; j < 3; ++j) {
        e1[j] = P[1][j] - P[0][j];
        e2[j] = P[2][j] - P[0][j];
    }
    c[0] = e1[1] * e2[2] - e1[2] * e2[1];
    c[1] = e1[2] * e2[0] - e1[0] * e2[2];
    c[2] = e1[0] * e2[1] - e1[1] * e2[0];
    const double len = sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
    const double area = 0.5 * len;
    double n[3] = {c[0] / len, c[1] / len, c[2] / len};
    double cc[3];
    for (int j = 0; j < 3; ++j) cc[j] = (P[0][j] + P[1][j] + P[2][j]) / 3.0;
    for (int q = 0; q < 6; ++q) {
        double b[3], w;
        rule_point(q, b, w);
        double x[3];
        for (int j = 0; j < 3; ++j) x[j] = b[0] * P[0][j] + b[1] * P[1][j] + b[2] * P[2][j];
        pt[6 * t + q] = make_float4((float)x[0], (float)x[1], (float)x[2], (float)(w * area));
        poff[6 * t + q] = make_float4((float)(x[0] - cc[0]), (float)(x[1] - cc[1]),
                                      (float)(x[2] - cc[2]), (float)(w * area));
    }
    // centroid as an unevaluated float pair (hi + lo), about 48 significant bits
    float hi[3], lo[3];
    for (int j = 0; j < 3; ++j) {
        hi[j] = (float)cc[j];
        lo[j] = (float)(cc[j] - (double)hi[j]);
    }
    cen[2 * t] = make_float4(hi[0], hi[1], hi[2], 0.f);
    cen[2 * t + 1] = make_float4(lo[0], lo[1], lo[2], 0.f);
    const double h = n[0] * P[0][0] + n[1] * P[0][1] + n[2] * P[0][2];
    tn[t] = make_float4((float)n[0], (float)n[1], (float)n[2], (float)h);
    // w: bits of n.(P0 - x_0) with the FP32 normal and the FP32 first rule
    // point x_0, the distance of x_0 from the plane that its rounding made
    {
        const double x0 = (1.0 - 2.0 * kQa1) * P[0][0] + kQa1 * (P[1][0] + P[2][0]);
        const double x1 = (1.0 - 2.0 * kQa1) * P[0][1] + kQa1 * (P[1][1] + P[2][1]);
        const double x2 = (1.0 - 2.0 * kQa1) * P[0][2] + kQa1 * (P[1][2] + P[2][2]);
        const double off = (double)(float)n[0] * (P[0][0] - (double)(float)x0) +
                           (double)(float)n[1] * (P[0][1] - (double)(float)x1) +
                           (double)(float)n[2] * (P[0][2] - (double)(float)x2);
        tv[t] = make_int4(v[0], v[1], v[2], __float_as_int((float)off));
    }
    double *g = tgeo + 16 * (size_t)t;
    g[0] = area;
    g[1] = n[0];
    g[2] = n[1];
    g[3] = n[2];
    // curl phi_a = n x grad phi_a = (P_{a+1} - P_{a+2}) / (2 area)
    for (int a = 0; a < 3; ++a)
        for (int j = 0; j < 3; ++j)
            g[4 + 3 * a + j] = (P[(a + 1) % 3][j] - P[(a + 2) % 3][j]) / (2.0 * area);
    g[13] = g[14] = g[15] = 0.0;
}

// Source data of one apply, duplicated into (value, value) pairs, the values
// that enter with both signs stored with both, so that the far kernel's
// packed FP32 instructions (two test points per pair of lanes) take every
// operand of a complex multiply-add straight from shared memory, without
// moves or negations:
//   sP[4k]   = (-y.x, -y.x, -y.y, -y.y)     sP[4k+1] = (-y.z, -y.z, psi.re, psi.re)
//   sP[4k+2] = (psi.im, psi.im, -psi.im, -psi.im)
//   sP[4k+3] = (phi.re, phi.re, phi.im, phi.im)    sP5[k] = (-phi.im, -phi.im)
// with psi_q = w_q |s| sum_b lambda_b(q) psi_b (the same for phi); per
// triangle c_s = |s| sum_b phi_b curl phi_b as
//   sC[2t] = (cx.re, cx.im, cy.re, cy.im)   sC[2t+1] = (cz.re, cz.im, 0, 0)
// One thread per rule point (FP64 is slow here and its chains are short this
// way: the 150-vertex hull's densities took 11 us with a thread per
// triangle); threads q < 3 also form component q of c_s.
__global__ void far_prep_kernel(const double2 *__restrict__ x, int nv, int nt,
                                const int *__restrict__ tris, const float4 *__restrict__ pt,
                                const double *__restrict__ tgeo, float4 *__restrict__ sP,
                                float2 *__restrict__ sP5, float4 *__restrict__ sC) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 6 * nt) return;
    const int t = k / 6, q = k - 6 * (k / 6);
    double2 ps[3], ph[3];
    for (int a = 0; a < 3; ++a) {
        const int v = tris[3 * t + a];
        ps[a] = x[v];
        ph[a] = x[nv + v];
    }
    const double *g = tgeo + 16 * (size_t)t;
    const double area = g[0];
    double b[3], w;
    rule_point(q, b, w);
    const double W = w * area;
    double2 s = cd(0, 0), f = cd(0, 0);
    for (int a = 0; a < 3; ++a) {
        s = cadd(s, cscale(ps[a], b[a]));
        f = cadd(f, cscale(ph[a], b[a]));
    }
    const float4 p = pt[k];
    const float psr = (float)(W * s.x), psi = (float)(W * s.y);
    const float phr = (float)(W * f.x), phi = (float)(W * f.y);
    float4 *d = sP + 4 * (size_t)k;
    d[0] = make_float4(-p.x, -p.x, -p.y, -p.y);
    d[1] = make_float4(-p.z, -p.z, psr, psr);
    d[2] = make_float4(psi, psi, -psi, -psi);
    d[3] = make_float4(phr, phr, phi, phi);
    sP5[k] = make_float2(-phi, -phi);
    if (q < 3) {
        double2 cv = cd(0, 0);
        for (int a = 0; a < 3; ++a) cv = cadd(cv, cscale(ph[a], g[4 + 3 * a + q]));
        float2 *c = reinterpret_cast<float2 *>(sC + 2 * (size_t)t);
        c[q] = make_float2((float)(cv.x * area), (float)(cv.y * area));
        if (q == 0) c[3] = make_float2(0.f, 0.f);
    }
}

typedef float2 f2;
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ f2 hi2(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ f2 dup2(float a) { return make_float2(a, a); }

// Constants as (value, value) pairs for the packed instructions.  The D
// normal term k0^2 G0 + (k1^2/rho) G1 is evaluated as dks (G0 + dk1 G1):
// dk0 holds the scale dks (applied once per source triangle) and dk1 the
// ratio (k1^2/rho) / dks.
struct FarConst2 {
    f2 k0, k1, nk0, nk1, rho, irho, dk0, dk1;
};

// Accumulators of two test points, packed (point a, point b): tile sums of
// u1, u2 (complex) and the per-source-triangle sums T1n = -sum_q Hs phi_q,
// U = sum_q Gk phi_q.
struct PairAcc {
    f2 u1r, u1i, u2r, u2i;
    f2 t1r, t1i, ur, ui;
};

// Unweighted sums of G0 and G1 over the pairs of a thread and the source
// points of one weight class (lane x: test points 0..2, lane y: 3..5).
struct CurlAcc {
    f2 g0r, g0i, g1r, g1i;
};

// Per (test triangle, source triangle) data of the centred (large k r)
// variant: D = c_x - c_y (centroid difference, FP32 rounding of a
// float-float value), r_c = |D| and the phase k r_c as a fraction of a
// revolution in [-1/2, 1/2], from float-float arithmetic (about 48 bits).
struct CenterPair {
    f2 Dx, Dy, Dz, rc, b0, b1;
    float lx, ly, lz;  // low parts of D
};

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float v = s - a;
    e = (a - (s - v)) + (b - v);
}

// s + e += v exactly up to the rounding of e
__device__ __forceinline__ void comp_add(float &s, float &e, float v) {
    float t, d;
    two_sum(s, v, t, d);
    s = t;
    e += d;
}

// the same with Dekker's FastTwoSum (exact for |s| >= |v|, else the error
// term misses at most a rounding of v: sums whose terms rarely exceed them)
__device__ __forceinline__ void comp_add_fast(float &s, float &e, float v) {
    const float t = s + v;
    e += v - (t - s);
    s = t;
}

// a - b for float-float a = (ah, al), b = (bh, bl); result (h, l)
__device__ __forceinline__ void ff_sub(float ah, float al, float bh, float bl, float &h, float &l) {
    float s, e;
    two_sum(ah, -bh, s, e);
    e += al - bl;
    h = s + e;
    l = e - (h - s);
}

// frac(r (kh + kl)) in revolutions for float-float r = (rh, rl)
__device__ __forceinline__ float ff_phase_rev(float rh, float rl, float kh, float kl) {
    const float p = rh * kh;
    const float pe = fmaf(rh, kh, -p) + fmaf(rh, kl, rl * kh);
    const float n = rintf(p);
    return (p - n) + pe;
}

// 1/x to about one ulp (PTX rcp.approx), used where the result scales a
// small quantity
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ CenterPair center_pair(const float4 &cth, const float4 &ctl,
                                                  const float4 &csh, const float4 &csl,
                                                  float k0h, float k0l, float k1h, float k1l) {
    float dh[3], dl[3];
    ff_sub(cth.x, ctl.x, csh.x, csl.x, dh[0], dl[0]);
    ff_sub(cth.y, ctl.y, csh.y, csl.y, dh[1], dl[1]);
    ff_sub(cth.z, ctl.z, csh.z, csl.z, dh[2], dl[2]);
    // |D|^2 as float-float: exact squares of the high parts plus cross terms
    float sh = 0.f, sl = 0.f;
    for (int i = 0; i < 3; ++i) {
        const float p = dh[i] * dh[i];
        const float e = fmaf(dh[i], dh[i], -p) + 2.f * dh[i] * dl[i];
        float s, t;
        two_sum(sh, p, s, t);
        sh = s;
        sl += t + e;
    }
    // square root with one Newton correction (the correction only needs a
    // few significant bits of 1/(2 sqrt(sh)), so approximate rsqrt suffices)
    const float y = rsqrtf(sh);
    const float rs = sh * y;
    const float corr = (fmaf(-rs, rs, sh) + sl) * (0.5f * y);
    const float rh = rs + corr;
    const float rl = corr - (rh - rs);
    CenterPair c;
    c.Dx = dup2(dh[0]);
    c.Dy = dup2(dh[1]);
    c.Dz = dup2(dh[2]);
    c.lx = dl[0];
    c.ly = dl[1];
    c.lz = dl[2];
    c.rc = dup2(rh);
    // reduced centroid phases in radians (in [-pi, pi])
    c.b0 = dup2(6.28318530717958647692f * ff_phase_rev(rh, rl, k0h, k0l));
    c.b1 = dup2(6.28318530717958647692f * ff_phase_rev(rh, rl, k1h, k1l));
    return c;
}

// One source point against the six test points of a triangle (three pairs),
// both wavenumbers, packed FP32 arithmetic.  P0..P3, P5 hold the signed
// duplicated source data; (y - x).n_x is the same for every test point (they
// lie in the triangle's plane) and is formed once: from the first test point,
// corrected by pdn = n.(P0 - x_0) for the distance that rounding moved it off
// the plane, or (centred) from the centroid, pdn = D.n_x.  Each
// step is written for the three pairs together, so that neighbouring
// instructions share their source operand (the register reuse cache) and none
// waits for its predecessor.  Plain variant: (X, Y, Z) are the test points
// and the source coordinates absolute; the MUFU sine / cosine take k r
// directly (their own argument scaling has the same FP32 rounding as an
// explicit reduction).  CENTRED variant (large k r): coordinates are offsets
// from the triangle centroids, x - y = D + delta, and the phase is
// k r = k r_c + k (2 D.delta + delta.delta) / (r + r_c) with k r_c reduced in
// float-float arithmetic once per triangle pair.
// MULTI: m1 multiplies the interior terms (0: source on another object, -1:
// Mueller); k1i / dk1i: imaginary parts of k1 and k1^2 / rho (attenuation).
struct Diff2 {
    f2 dx, dy, dz;     // x - y
    f2 ddx, ddy, ddz;  // centred: difference of the offsets
};

template <bool CENTRED>
__device__ __forceinline__ Diff2 far_diff(f2 X, f2 Y, f2 Z, const float4 &P0, const float4 &P1, const CenterPair &cp) {
    Diff2 d;
    if (CENTRED) {
        d.ddx = add2(X, lo2(P0));  // delta = a - b
        d.ddy = add2(Y, hi2(P0));
        d.ddz = add2(Z, lo2(P1));
        d.dx = add2(d.ddx, cp.Dx);
        d.dy = add2(d.ddy, cp.Dy);
        d.dz = add2(d.ddz, cp.Dz);
    } else {
        d.dx = add2(X, lo2(P0));  // x - y
        d.dy = add2(Y, hi2(P0));
        d.dz = add2(Z, lo2(P1));
    }
    return d;
}

template <bool CENTRED, bool MULTI, bool ABSORB>
__device__ __forceinline__ void far_tri(const f2 (&X)[3], const f2 (&Y)[3], const f2 (&Z)[3], const float4 &n4,
                                        float pdn, const float4 &P0, const float4 &P1, const float4 &P2, const float4 &P3,
                                        const f2 &P5, const FarConst2 &c, const CenterPair &cp, f2 m1, f2 k1i,
                                        f2 dk1i, PairAcc (&A)[3], CurlAcc &B) {
#define F3 _Pragma("unroll") for (int p = 0; p < 3; ++p)
    Diff2 d[3];
    F3 d[p] = far_diff<CENTRED>(X[p], Y[p], Z[p], P0, P1, cp);
    const f2 dnxn = CENTRED ? dup2(-fmaf(P0.x, n4.x, fmaf(P0.z, n4.y, fmaf(P1.x, n4.z, pdn))))
                            : dup2(-fmaf(d[0].dz.x, n4.z, fmaf(d[0].dy.x, n4.y, fmaf(d[0].dx.x, n4.x, -pdn))));
    f2 r2[3], ri[3], r[3], ri2[3], s0[3], c0[3], s1[3], c1[3];
    F3 r2[p] = mul2(d[p].dx, d[p].dx);
    F3 r2[p] = fma2(d[p].dy, d[p].dy, r2[p]);
    F3 r2[p] = fma2(d[p].dz, d[p].dz, r2[p]);
    F3 ri[p] = make_float2(rsqrtf(r2[p].x), rsqrtf(r2[p].y));
    F3 r[p] = mul2(r2[p], ri[p]);
    F3 ri2[p] = mul2(ri[p], ri[p]);
    if (CENTRED) {
        f2 num[3], dd[3];
        F3 num[p] = mul2(d[p].ddx, d[p].ddx);
        F3 num[p] = fma2(d[p].ddy, d[p].ddy, num[p]);
        F3 num[p] = fma2(d[p].ddz, d[p].ddz, num[p]);
        F3 dd[p] = mul2(d[p].ddx, cp.Dx);
        F3 dd[p] = fma2(d[p].ddy, cp.Dy, dd[p]);
        F3 dd[p] = fma2(d[p].ddz, cp.Dz, dd[p]);
        F3 num[p] = fma2(dd[p], dup2(2.f), num[p]);  // r^2 - r_c^2
        F3 {
            const f2 den = add2(r[p], cp.rc);
            const f2 dlt = mul2(num[p], make_float2(rcp_approx(den.x), rcp_approx(den.y)));  // r - r_c
            const f2 ph0 = fma2(c.k0, dlt, cp.b0), ph1 = fma2(c.k1, dlt, cp.b1);
            __sincosf(ph0.x, &s0[p].x, &c0[p].x);
            __sincosf(ph0.y, &s0[p].y, &c0[p].y);
            __sincosf(ph1.x, &s1[p].x, &c1[p].x);
            __sincosf(ph1.y, &s1[p].y, &c1[p].y);
        }
    } else {
        F3 {
            const f2 kr0 = mul2(r[p], c.k0), kr1 = mul2(r[p], c.k1);
            __sincosf(kr0.x, &s0[p].x, &c0[p].x);
            __sincosf(kr0.y, &s0[p].y, &c0[p].y);
            __sincosf(kr1.x, &s1[p].x, &c1[p].x);
            __sincosf(kr1.y, &s1[p].y, &c1[p].y);
        }
    }
    constexpr bool absorb = MULTI && ABSORB;
    if (MULTI) {  // e^{i k1 r} with k1 = k1r + i k1i: damping e^{-k1i r}, and m1
        F3 {
            f2 damp = m1;
            if (absorb) {
                const f2 br = mul2(r[p], k1i);
                damp = mul2(m1, make_float2(__expf(-br.x), __expf(-br.y)));
            }
            c1[p] = mul2(c1[p], damp);
            s1[p] = mul2(s1[p], damp);
        }
    }
    const f2 psr = hi2(P1), psi = lo2(P2), mpsi = hi2(P2), phr = lo2(P3), phi = hi2(P3), mphi = P5;
    // cos and sin scaled by 1/r once: G = (c + i s)/r for every kernel below
    f2 c0r[3], s0r[3], c1r[3], s1r[3], ga[3], gb[3], hp[3], hq[3];
    F3 c0r[p] = mul2(c0[p], ri[p]);
    F3 s0r[p] = mul2(s0[p], ri[p]);
    F3 c1r[p] = mul2(c1[p], ri[p]);
    F3 s1r[p] = mul2(s1[p], ri[p]);
    // -(H0 + H1) r^2, H = e^{ikr} (i k r - 1) / r^3, with the scaled c, s:
    //   re = c0/r + c1/r + k0 s0 + k1 s1,  im = s0/r + s1/r - k0 c0 - k1 c1
    F3 hp[p] = add2(c0r[p], c1r[p]);
    F3 hq[p] = add2(s0r[p], s1r[p]);
    F3 hp[p] = fma2(c.k0, s0[p], hp[p]);
    F3 hp[p] = fma2(c.k1, s1[p], hp[p]);
    F3 hq[p] = fma2(c.nk0, c0[p], hq[p]);
    F3 hq[p] = fma2(c.nk1, c1[p], hq[p]);
    if (absorb) {  // (i k1 r - 1) with Im k1: + k1i r (c1, s1) / r
        F3 hp[p] = fma2(k1i, c1[p], hp[p]);
        F3 hq[p] = fma2(k1i, s1[p], hq[p]);
    }
    // D curl term: sums of G0 and G1, weighted and combined by the caller
    F3 B.g0r = add2(B.g0r, c0r[p]);
    F3 B.g0i = add2(B.g0i, s0r[p]);
    F3 B.g1r = add2(B.g1r, c1r[p]);
    F3 B.g1i = add2(B.g1i, s1r[p]);
    // V block (G0 + rho G1) psi, without 1/(4 pi)
    F3 ga[p] = fma2(c.rho, c1r[p], c0r[p]);
    F3 gb[p] = fma2(c.rho, s1r[p], s0r[p]);
    F3 A[p].u1r = fma2(gb[p], mpsi, A[p].u1r);
    F3 A[p].u1i = fma2(gb[p], psr, A[p].u1i);
    F3 A[p].u1r = fma2(ga[p], psr, A[p].u1r);
    F3 A[p].u1i = fma2(ga[p], psi, A[p].u1i);
    // D normal term (k0^2 G0 + k1^2/rho G1) phi, as (G0 + dk1 G1) phi; the
    // scale dks is applied per source triangle
    F3 ga[p] = fma2(c.dk1, c1r[p], c0r[p]);
    F3 gb[p] = fma2(c.dk1, s1r[p], s0r[p]);
    if (absorb) {  // complex k1^2 / (rho dks)
        F3 ga[p] = fma2(mul2(dk1i, s1r[p]), dup2(-1.f), ga[p]);
        F3 gb[p] = fma2(dk1i, c1r[p], gb[p]);
    }
    F3 A[p].ur = fma2(gb[p], mphi, A[p].ur);
    F3 A[p].ui = fma2(gb[p], phr, A[p].ui);
    F3 A[p].ur = fma2(ga[p], phr, A[p].ur);
    F3 A[p].ui = fma2(ga[p], phi, A[p].ui);
    // T1n = -sum Hs phi
    F3 hp[p] = mul2(hp[p], ri2[p]);
    F3 hq[p] = mul2(hq[p], ri2[p]);
    F3 A[p].t1r = fma2(hq[p], mphi, A[p].t1r);
    F3 A[p].t1i = fma2(hq[p], phr, A[p].t1i);
    F3 A[p].t1r = fma2(hp[p], phr, A[p].t1r);
    F3 A[p].t1i = fma2(hp[p], phi, A[p].t1i);
    // T block: (H0 + H1)(x - y).n_x psi = (-(H0 + H1)) (y - x).n_x psi
    F3 hp[p] = mul2(hp[p], dnxn);
    F3 hq[p] = mul2(hq[p], dnxn);
    F3 A[p].u2r = fma2(hq[p], mpsi, A[p].u2r);
    F3 A[p].u2i = fma2(hq[p], psr, A[p].u2i);
    F3 A[p].u2r = fma2(hp[p], psr, A[p].u2r);
    F3 A[p].u2i = fma2(hp[p], psi, A[p].u2i);
#undef F3
}

// One thread per test triangle: its six points are three pairs (p, p + 3)
// packed into the two lanes of FP32x2 instructions (a lane holds the points
// of one rule weight).  Outputs per source split
//   part[(split * 4 + c) * npts + p], c = u1 (re, im), u2 (re, im):
//     u1 = sum [ (G0 + rho G1) psi_q + (x.n_y - h_y)(H0 + H1) phi_q ]
//     u2 = sum [ (H0 + H1)(x - y).n_x psi_q - (n_x.n_y)(k0^2 G0 + k1^2/rho G1) phi_q ]
//   partA[(split * 6 + c) * nt + t], c = A (x re, x im, y re, y im, z re, z im):
//     A  = sum_s (sum_p w_p sum_q w_q (G0 + G1/rho)) c_s
// with G, H here without the factor 1/(4 pi) (applied in the gather).  Sums
// run per 64-triangle tile, then tile sums are added to running sums kept in
// the outputs.
// The kernel is bound by the FP32 pipe (packed FMA at 2.5 to 3.3 cycles a
// warp instruction with three distinct register pairs, packed add and
// multiply at 2).  A thread holds the whole triangle so that what is common
// to its points is done once: (y - x).n_x per source point (8 of about 154
// pipe cycles per pair of test points before), the curl term summed over test
// and source points by plain adds, weighted per class and multiplied into c_s
// once per triangle pair (10 cycles), the source
// loads from shared memory (a third), and the centroid phases of the centred
// variant (a third).  An apply at 10242 vertices: 25.9 ms (29.1 where a
// thread held one pair of points), 20000 vertices centred 124 ms (147), four
// objects of 642 vertices 2.19 ms (3.27).  255 registers and two blocks per
// SM measured 1 to 4 % better than 168 and three.
// Small meshes give a block 32 or 64 test triangles and split each source
// tile between its warps, whose sums are added in shared memory: more warps
// in flight for the same number of partial sums (see far_setup_geometry).
// CENTRED: pt holds offsets from the test-triangle centroid and cen the
// float-float centroids (see far_tri).
// MULTI: disjoint objects (Sec. 2.2) or the Mueller formulation; the interior
// constants are the test triangle's object's, interior terms vanish for
// sources on other objects and change sign for Mueller.  ABSORB (with MULTI):
// complex interior wavenumbers (attenuation).
template <bool CENTRED, bool MULTI, bool ABSORB>
__global__ void __launch_bounds__(FAR_THREADS, OSRC_FAR_MIN_BLOCKS)
far_kernel(const float4 *__restrict__ pt, const float4 *__restrict__ cen,
           const float4 *__restrict__ tn, const int4 *__restrict__ tv,
           const float4 *__restrict__ sP, const float2 *__restrict__ sP5,
           const float4 *__restrict__ sC, int nt, int npts, int tris_per_split, int block_tris, FarConst2 c0,
           float4 kff0, const int *__restrict__ tcomp, const FarObj *__restrict__ fobj,
           float *__restrict__ part, float *__restrict__ partA) {
    __shared__ float4 shP[FAR_TS * 6 * 4];
    __shared__ float2 shP5[FAR_TS * 6];
    __shared__ float4 shN[FAR_TS];
    __shared__ float4 shC[FAR_TS * 2];
    __shared__ int4 shV[FAR_TS];
    __shared__ float4 shCen[CENTRED ? 2 * FAR_TS : 1];
    __shared__ int shComp[MULTI ? FAR_TS : 1];

    // block_tris test triangles x FAR_THREADS / block_tris source groups (whole
    // warps); a group takes every ngrp-th source triangle of a tile
    const int tx = threadIdx.x % block_tris, grp = threadIdx.x / block_tris, ngrp = FAR_THREADS / block_tris;
    const int j = blockIdx.x * block_tris + tx;
    const int split = blockIdx.y;
    const int s_begin = min(nt, split * tris_per_split);
    const int s_end = min(nt, s_begin + tris_per_split);
    const bool active = j < nt;
    const int tau = active ? j : 0;
    f2 X[3], Y[3], Z[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const float4 xa = pt[6 * tau + p], xb = pt[6 * tau + p + 3];
        X[p] = make_float2(xa.x, xb.x);
        Y[p] = make_float2(xa.y, xb.y);
        Z[p] = make_float2(xa.z, xb.z);
    }
    const float4 n4 = tn[tau];
    const int4 vt = tv[tau];
    constexpr float W1 = (float)kQw1, W2 = (float)kQw2;
    FarConst2 c = c0;
    float4 kff = kff0;
    int ct = 0;
    float sgn = 1.f;  // sign of the interior terms (-1: Mueller)
    f2 k1i = make_float2(0.f, 0.f), dk1i = k1i;
    if (MULTI) {
        ct = tcomp[tau];
        const FarObj o = fobj[ct];
        c.k1 = dup2(o.k1);
        c.nk1 = dup2(o.nk1);
        c.rho = dup2(o.rho);
        c.irho = dup2(o.irho);
        c.dk1 = dup2(o.dk1);
        kff.z = o.k1h;
        kff.w = o.k1l;
        sgn = o.sgn;
        k1i = dup2(o.k1i);
        dk1i = dup2(o.dk1i);
    }
    float4 cth = make_float4(0.f, 0.f, 0.f, 0.f), ctl = cth;
    if (CENTRED) {
        cth = cen[2 * tau];
        ctl = cen[2 * tau + 1];
    }
    // curl-term sums of the whole split, rounding errors carried along: one sum per triangle stands for the six points' sums, whose
    // independent rounding errors the test weights would have averaged
    float ar[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, ae[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const size_t o1 = (size_t)split * 4 * npts + 6 * (size_t)tau, oA = (size_t)split * 6 * nt + tau;

    for (int t0 = s_begin; t0 < s_end; t0 += FAR_TS) {
        const int cnt = min(FAR_TS, s_end - t0);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt * 24; i += blockDim.x) shP[i] = sP[24 * (size_t)t0 + i];
        for (int i = threadIdx.x; i < cnt * 6; i += blockDim.x) shP5[i] = sP5[6 * (size_t)t0 + i];
        for (int i = threadIdx.x; i < cnt * 2; i += blockDim.x) shC[i] = sC[2 * (size_t)t0 + i];
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
            const float4 ns = tn[t0 + i];
            shN[i] = make_float4(-ns.x, -ns.y, -ns.z, ns.w);
            shV[i] = tv[t0 + i];
        }
        if (CENTRED)
            for (int i = threadIdx.x; i < 2 * cnt; i += blockDim.x) shCen[i] = cen[2 * (size_t)t0 + i];
        if (MULTI)
            for (int i = threadIdx.x; i < cnt; i += blockDim.x) shComp[i] = tcomp[t0 + i];
        __syncthreads();

        PairAcc A[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) A[p].u1r = A[p].u1i = A[p].u2r = A[p].u2i = make_float2(0.f, 0.f);
        for (int s = grp; s < cnt; s += ngrp) {
            const int4 vs = shV[s];
            const bool touch = (vs.x == vt.x) | (vs.x == vt.y) | (vs.x == vt.z) |
                               (vs.y == vt.x) | (vs.y == vt.y) | (vs.y == vt.z) |
                               (vs.z == vt.x) | (vs.z == vt.y) | (vs.z == vt.z);
            if (touch) continue;
            CenterPair cp;
            float pdn = __int_as_float(vt.w);
            if (CENTRED) {
                cp = center_pair(cth, ctl, shCen[2 * s], shCen[2 * s + 1], kff.x, kff.y, kff.z, kff.w);
                pdn = fmaf(cp.Dx.x, n4.x, fmaf(cp.Dy.x, n4.y, cp.Dz.x * n4.z)) +
                      fmaf(cp.lx, n4.x, fmaf(cp.ly, n4.y, cp.lz * n4.z));
            }
#pragma unroll
            for (int p = 0; p < 3; ++p)
                A[p].t1r = A[p].t1i = A[p].ur = A[p].ui = make_float2(0.f, 0.f);
            f2 t3r = make_float2(0.f, 0.f), t3i = t3r;  // sum_q w_q (G0 + G1/rho), lanes summed over their points
            const f2 m1 = dup2(MULTI ? (shComp[s] != ct ? 0.f : sgn) : 1.f);
#pragma unroll FAR_HUNROLL
            for (int h = 0; h < 2; ++h) {  // the two weight classes of the source points
                CurlAcc Bs;
                Bs.g0r = Bs.g0i = Bs.g1r = Bs.g1i = make_float2(0.f, 0.f);
#pragma unroll FAR_QUNROLL
                for (int q = 3 * h; q < 3 * h + 3; ++q) {
                    const float4 *P = &shP[24 * s + 4 * q];
                    const float4 P0 = P[0], P1 = P[1], P2 = P[2], P3 = P[3];
                    const f2 P5 = shP5[6 * s + q];
                    far_tri<CENTRED, MULTI, ABSORB>(X, Y, Z, n4, pdn, P0, P1, P2, P3, P5, c, cp, m1, k1i, dk1i, A, Bs);
                }
                const f2 wh = dup2(h ? W2 : W1);
                t3r = fma2(wh, fma2(c.irho, Bs.g1r, Bs.g0r), t3r);
                t3i = fma2(wh, fma2(c.irho, Bs.g1i, Bs.g0i), t3i);
            }
            const float4 mns = shN[s];  // (-n_y, n_y.P0)
            float dn = mns.w;           // -(x - y).n_y, constant over the source triangle
            // centred: (x - y).n_y = (c_x - c_y + a).n_y since c_y lies in the source plane
            if (CENTRED) dn = cp.Dx.x * mns.x + cp.Dy.x * mns.y + cp.Dz.x * mns.z;
            const float nxnyn = n4.x * mns.x + n4.y * mns.y + n4.z * mns.z;  // -n_x.n_y
            const f2 nn = dup2(nxnyn * c.dk0.x);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                // u1 += (x - y).n_y T1 = (-(x - y).n_y)(-T1);  u2 += (-n_x.n_y) U
                const f2 xnyn = fma2(Z[p], dup2(mns.z), fma2(Y[p], dup2(mns.y), fma2(X[p], dup2(mns.x), dup2(dn))));
                A[p].u1r = fma2(xnyn, A[p].t1r, A[p].u1r);
                A[p].u1i = fma2(xnyn, A[p].t1i, A[p].u1i);
                A[p].u2r = fma2(nn, A[p].ur, A[p].u2r);
                A[p].u2i = fma2(nn, A[p].ui, A[p].u2i);
            }
            // A += (sum_p w_p T3_p) c_s
            const float wr = fmaf(W1, t3r.x, W2 * t3r.y), wi = fmaf(W1, t3i.x, W2 * t3i.y);
            const float4 C0 = shC[2 * s], C1 = shC[2 * s + 1];
            const float cr[3] = {C0.x, C0.z, C1.x}, ci[3] = {C0.y, C0.w, C1.y};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                comp_add_fast(ar[2 * i], ae[2 * i], fmaf(wr, cr[i], -(wi * ci[i])));
                comp_add_fast(ar[2 * i + 1], ae[2 * i + 1], fmaf(wr, ci[i], wi * cr[i]));
            }
        }
        if (ngrp > 1) {  // add the groups' sums through shared memory (the tile is done with)
            float *red = reinterpret_cast<float *>(shP);
            const int rs = (ngrp - 1) * block_tris;
            __syncthreads();
            if (grp > 0) {
                float *o = red + (grp - 1) * block_tris + tx;
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    const f2 v[4] = {A[p].u1r, A[p].u1i, A[p].u2r, A[p].u2i};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        o[(8 * p + 2 * i) * rs] = v[i].x;
                        o[(8 * p + 2 * i + 1) * rs] = v[i].y;
                    }
                }
            }
            __syncthreads();
            if (grp == 0)
                for (int g = 0; g < ngrp - 1; ++g) {
                    const float *o = red + g * block_tris + tx;
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        f2 *v[4] = {&A[p].u1r, &A[p].u1i, &A[p].u2r, &A[p].u2i};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            *v[i] = add2(*v[i], make_float2(o[(8 * p + 2 * i) * rs], o[(8 * p + 2 * i + 1) * rs]));
                    }
                }
        }
        // running sums of u live in the outputs: the first tile stores, later
        // tiles add (the thread's own entries; registers stay free for the
        // pair loop)
        if (active && grp == 0) {
            const bool first = t0 == s_begin;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                const f2 v[4] = {A[p].u1r, A[p].u1i, A[p].u2r, A[p].u2i};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const size_t o = o1 + (size_t)i * npts + p;
                    part[o] = first ? v[i].x : part[o] + v[i].x;
                    part[o + 3] = first ? v[i].y : part[o + 3] + v[i].y;
                }
            }
        }
    }
    if (ngrp > 1) {  // the groups' curl sums
        float *red = reinterpret_cast<float *>(shP);
        const int rs = (ngrp - 1) * block_tris;
        __syncthreads();
        if (grp > 0)
#pragma unroll
            for (int i = 0; i < 6; ++i) red[i * rs + (grp - 1) * block_tris + tx] = ar[i] + ae[i];
        __syncthreads();
        if (grp == 0)
            for (int g = 0; g < ngrp - 1; ++g)
#pragma unroll
                for (int i = 0; i < 6; ++i) comp_add(ar[i], ae[i], red[i * rs + g * block_tris + tx]);
    }
    if (active && grp == 0)
#pragma unroll
        for (int i = 0; i < 6; ++i) partA[oA + (size_t)i * nt] = ar[i] + ae[i];
    if (active && grp == 0 && s_begin >= s_end) {  // empty split: zero sums
#pragma unroll
        for (int i = 0; i < 4; ++i)
            for (int p = 0; p < 6; ++p) part[o1 + (size_t)i * npts + p] = 0.f;
    }
}

// ---------------------------------------------------------------------------
// Gather: L lanes per (vertex, right-hand side).  Far field, over the
// incident (triangle t, local index a):
//   y1_v = (1/4pi) sum |t| sum_q w_q lambda_a(q) u1(t,q)
//   y2_v = (1/4pi) sum |t| [sum_q w_q lambda_a(q) u2(t,q) + curl_a . A(t)]
// plus the near-field CSR rows (2x2 complex blocks) applied to x.  Partial
// sums as far_kernel and farm_kernel leave them: part [ns][R][4][npts],
// partA [ns][R][6][nt].
// The lanes share the (triangle, point) items and the CSR entries.  The
// source splits are added in FP32 with their rounding errors carried along
// (Knuth's TwoSum: the sum to about 48 bits), because FP64 issues at 1/64 of
// the FP32 rate on this part; the rest is FP64.  One thread per vertex with
// FP64 sums took 215 us on the 150-vertex hull and 0.24 ms on the
// 10242-vertex sphere.  Small meshes, where the splits are many and the
// vertices too few to fill the GPU, take a block per vertex (L = 32, W = 4:
// the splits shared by its four warps); larger ones a warp, then L = 8 where
// lanes would idle.
// ---------------------------------------------------------------------------
constexpr int FARM_MAX_R = 8;

struct VecPtrs {
    const double2 *p[FARM_MAX_R];
};
struct OutPtrs {
    double2 *p[FARM_MAX_R];
};

constexpr int GATHER_THREADS = 128;

// value of a compensated sum; an infinite or NaN sum stands alone (its error
// term is not a number)
__device__ __forceinline__ double comp_value(float s, float e) {
    return isfinite(s) ? (double)s + (double)e : (double)s;
}

template <int L, int W>
__global__ void __launch_bounds__(GATHER_THREADS)
gather_kernel(int nv, int nt, int npts, int ns, int R, const int *__restrict__ vt_ptr,
              const int *__restrict__ vt_idx, const double *__restrict__ tgeo, const float *__restrict__ part,
              const float *__restrict__ partA, int use_far, const int *__restrict__ nr_ptr,
              const int *__restrict__ nr_col, const double2 *__restrict__ nr_val, int use_near,
              const __grid_constant__ VecPtrs x, const __grid_constant__ OutPtrs y) {
    static_assert(W == 1 || L == 32, "split groups are warps");
    __shared__ double2 red[W > 1 ? W : 1][2];
    const int lane = threadIdx.x % L;
    const int wg = W > 1 ? threadIdx.x / L % W : 0;  // split group
    const int v = blockIdx.x * (GATHER_THREADS / (L * W)) + threadIdx.x / (L * W);
    const int rr = blockIdx.y;
    const bool valid = v < nv;  // every lane takes part in the shuffles below
    double2 y1 = cd(0, 0), y2 = cd(0, 0);
    if (valid && use_far) {
        const int e0 = vt_ptr[v], items = 6 * (vt_ptr[v + 1] - e0);
        const size_t su = (size_t)R * 4 * npts, sa = (size_t)R * 6 * nt;
        for (int it = lane; it < items; it += L) {
            const int e = it / 6, q = it - 6 * e;
            const int ta = vt_idx[e0 + e], t = ta / 3, a = ta - 3 * t;
            const double *g = tgeo + 16 * (size_t)t;
            const float *P = part + (size_t)rr * 4 * npts + 6 * (size_t)t + q;
            const float *PA = partA + ((size_t)rr * 6 + q) * nt + t;
            float s[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, c[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int sp = wg; sp < ns; sp += W) {
#pragma unroll
                for (int i = 0; i < 4; ++i) comp_add(s[i], c[i], P[sp * su + (size_t)i * npts]);
                comp_add(s[4], c[4], PA[sp * sa]);
            }
            const double al = q < 3 ? kQa1 : kQa2, w = q < 3 ? kQw1 : kQw2;
            const double wl = w * (a == (q < 3 ? q : q - 3) ? 1.0 - 2.0 * al : al) * g[0], wa = g[4 + 3 * a + (q >> 1)] * g[0];
            y1 = cadd(y1, cd(wl * comp_value(s[0], c[0]), wl * comp_value(s[1], c[1])));
            y2 = cadd(y2, cd(wl * comp_value(s[2], c[2]), wl * comp_value(s[3], c[3])));
            const double av = wa * comp_value(s[4], c[4]);  // component q / 2 of curl_a . A, re or im
            if (q & 1) y2.y += av;
            else y2.x += av;
        }
        const double inv4pi = 0.079577471545947667884;
        y1 = cscale(y1, inv4pi);
        y2 = cscale(y2, inv4pi);
    }
    if (valid && use_near) {
        const double2 *xr = x.p[rr];
        for (int e = nr_ptr[v] + wg * L + lane; e < nr_ptr[v + 1]; e += L * W) {
            const int jc = nr_col[e];
            const double2 xa = xr[jc], xb = xr[nv + jc];
            const double2 *Bk = nr_val + 4 * (size_t)e;
            y1 = cadd(y1, cadd(cmul(Bk[0], xa), cmul(Bk[1], xb)));
            y2 = cadd(y2, cadd(cmul(Bk[2], xa), cmul(Bk[3], xb)));
        }
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
        y1.x += __shfl_xor_sync(0xffffffffu, y1.x, o);
        y1.y += __shfl_xor_sync(0xffffffffu, y1.y, o);
        y2.x += __shfl_xor_sync(0xffffffffu, y2.x, o);
        y2.y += __shfl_xor_sync(0xffffffffu, y2.y, o);
    }
    if (W > 1) {  // a block per vertex: its warps' sums in warp order
        if (lane == 0) {
            red[wg][0] = y1;
            red[wg][1] = y2;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 1; w < W; ++w) {
                y1 = cadd(y1, red[w][0]);
                y2 = cadd(y2, red[w][1]);
            }
    }
    if (valid && lane == 0 && wg == 0) {
        y.p[rr][v] = y1;
        y.p[rr][nv + v] = y2;
    }
}

// ---------------------------------------------------------------------------
// Multi-right-hand-side far field: one launch applies B_far to R vectors.
// Everything that depends only on the point pair (distance, 1/r, the four
// sine / cosine values, the kernel combinations) is computed once and shared
// by the R right-hand sides; only the accumulations scale with R.  To keep
// per-right-hand-side state small, the per-source-triangle factors of the
// K and D-normal terms ((x - y).n_y and n_x.n_y) are folded into the pair's
// kernel values, so each right-hand side has just the two complex sums
//   u1 = sum [ (G0 + rho G1) psi_q + (x - y).n_y (H0 + H1) phi_q ]
//   u2 = sum [ (H0 + H1)(x - y).n_x psi_q - (n_x.n_y)(k0^2 G0 + k1^2/rho G1) phi_q ]
// per test point, kept in registers over the whole source range.  The D
// curl term A = sum_s (sum_q w_q (G0 + G1/rho)) c_s needs only
// W(tau, s) = sum_p w_p sum_q w_q (G0 + G1/rho), which does not depend on the
// right-hand side: each thread's share of it goes to shared memory per
// source triangle, and after each tile the three threads of a test triangle
// contract it with the right-hand sides' curl sources c_s (each thread a
// third of the right-hand sides).
//
// Block: FARM_THREADS = 384 threads = 128 test triangles, thread j holds test
// points 2 (j mod 3), 2 (j mod 3) + 1 of triangle j / 3 packed in FP32x2
// lanes.  Source data (per point, duplicated pairs for the packed lanes):
//   sG [6nt][2]   (-y.x, -y.x, -y.y, -y.y), (-y.z, -y.z, w_q, w_q)   (static)
//   sD [nt][6][R][2]  (psi.re, psi.re, psi.im, psi.im), (phi.re, ..., phi.im)
//   sCm [nt][R][3]    c_s components (complex)
// Outputs (no atomics; gridDim.y splits the source range):
//   part  [ns][R][4][npts]  u1 (re, im), u2 (re, im) per test point
//   partA [ns][R][6][nt]    sum_p w_p A(x_p) per test triangle (x, y, z; re, im)
// ---------------------------------------------------------------------------
// 384 threads = 12 warps, 3 on each of the SM's four schedulers (a block
// whose warps spread unevenly over the schedulers waits at every tile
// barrier for its most crowded scheduler); one block per SM at <= 170
// registers per thread
#ifndef OSRC_FARM_THREADS
#define OSRC_FARM_THREADS 384
#endif
constexpr int FARM_THREADS = OSRC_FARM_THREADS;
#ifndef OSRC_FARM_MIN_BLOCKS
#define OSRC_FARM_MIN_BLOCKS 1
#endif
#ifndef OSRC_FARM_QUNROLL
#define OSRC_FARM_QUNROLL 2
#endif
constexpr int FARM_QUNROLL = OSRC_FARM_QUNROLL;  // unroll of the rule-point loop
constexpr int FARM_TRIS = FARM_THREADS / 3;  // test triangles per block
constexpr int FARM_TS = 16;                  // source triangles per shared-memory tile
// one shared-memory tile buffer: sG, sD, sCm, normals, vertex ids, centroids
constexpr size_t farm_buf_bytes(int R, bool centred) {
    return (size_t)FARM_TS * (12 * 16 + 12 * 16 * R + 24 * R + 16 + 16 + (centred ? 32 : 0));
}

size_t farm_smem_bytes(int R, bool centred) {
    return 2 * farm_buf_bytes(R, centred) + (size_t)FARM_TS * FARM_THREADS * sizeof(float2) + 2 * sizeof(uint64_t);
}

constexpr unsigned long long FARM_TIMEOUT_NS = 2000000000ULL;

__device__ __forceinline__ uint32_t farm_saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long farm_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// waits for phase `parity` of the mbarrier, at most FARM_TIMEOUT_NS of global time
__device__ __forceinline__ bool farm_wait(uint64_t *bar, uint32_t parity) {
    const unsigned long long t0 = farm_ns();
    while (true) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(farm_saddr(bar)), "r"(parity)
            : "memory");
        if (done) return true;
        if (farm_ns() - t0 > FARM_TIMEOUT_NS) return false;
    }
}

// 1-D bulk copy global -> shared (16-byte aligned addresses, size a multiple
// of 16), completion counted on the mbarrier
__device__ __forceinline__ void farm_bulk(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            farm_saddr(dst)),
        "l"((uint64_t)src), "r"(bytes), "r"(farm_saddr(bar))
        : "memory");
}

// static source geometry of the multi kernel: coordinates (absolute, or
// offsets from the triangle centroid for the centred variant) negated and
// duplicated, and the rule weight w_q
__global__ void farm_geom_kernel(const float4 *__restrict__ pts, int npts, float4 *__restrict__ sG) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npts) return;
    const float4 p = pts[k];
    const int q = k % 6;
    const float w = (float)(q < 3 ? kQw1 : kQw2);
    sG[2 * (size_t)k] = make_float4(-p.x, -p.x, -p.y, -p.y);
    sG[2 * (size_t)k + 1] = make_float4(-p.z, -p.z, w, w);
}

// densities of R right-hand sides at the source rule points and the curl
// sources c_s, one thread per (source triangle, right-hand side)
__global__ void farm_prep_kernel(VecPtrs x, int R, int nv, int nt, const int *__restrict__ tris,
                                 const double *__restrict__ tgeo, float4 *__restrict__ sD,
                                 float2 *__restrict__ sCm) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (t >= nt || r >= R) return;
    const double2 *xr = x.p[r];
    double2 ps[3], ph[3];
    for (int a = 0; a < 3; ++a) {
        const int v = tris[3 * t + a];
        ps[a] = xr[v];
        ph[a] = xr[nv + v];
    }
    const double *g = tgeo + 16 * (size_t)t;
    const double area = g[0];
    for (int q = 0; q < 6; ++q) {
        double b[3], w;
        rule_point(q, b, w);
        const double W = w * area;
        double2 sv = cd(0, 0), fv = cd(0, 0);
        for (int a = 0; a < 3; ++a) {
            sv = cadd(sv, cscale(ps[a], b[a]));
            fv = cadd(fv, cscale(ph[a], b[a]));
        }
        const float psr = (float)(W * sv.x), psi = (float)(W * sv.y);
        const float phr = (float)(W * fv.x), phi = (float)(W * fv.y);
        float4 *d = sD + 2 * ((6 * (size_t)t + q) * R + r);
        d[0] = make_float4(psr, psr, psi, psi);
        d[1] = make_float4(phr, phr, phi, phi);
    }
    for (int j = 0; j < 3; ++j) {
        double2 cv = cd(0, 0);
        for (int a = 0; a < 3; ++a) cv = cadd(cv, cscale(ph[a], g[4 + 3 * a + j]));
        sCm[3 * ((size_t)t * R + r) + j] = make_float2((float)(cv.x * area), (float)(cv.y * area));
    }
}

// One source point against the thread's two test points, R right-hand sides.
template <int R, bool CENTRED>
__device__ __forceinline__ void farm_pair(f2 X, f2 Y, f2 Z, const float4 G0, const float4 G1,
                                          const float4 *__restrict__ D, f2 mnx, f2 mny, f2 mnz, f2 xnyn,
                                          f2 nn, const FarConst2 &c, const CenterPair &cp, f2 &t3r,
                                          f2 &t3i, f2 (&u1r)[R], f2 (&u1i)[R], f2 (&u2r)[R],
                                          f2 (&u2i)[R]) {
    f2 dx, dy, dz, ddx, ddy, ddz;
    if (CENTRED) {
        ddx = add2(X, lo2(G0));
        ddy = add2(Y, hi2(G0));
        ddz = add2(Z, lo2(G1));
        dx = add2(ddx, cp.Dx);
        dy = add2(ddy, cp.Dy);
        dz = add2(ddz, cp.Dz);
    } else {
        dx = add2(X, lo2(G0));
        dy = add2(Y, hi2(G0));
        dz = add2(Z, lo2(G1));
    }
    f2 r2 = mul2(dx, dx);
    r2 = fma2(dy, dy, r2);
    r2 = fma2(dz, dz, r2);
    const f2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
    const f2 r = mul2(r2, ri);
    const f2 ri2 = mul2(ri, ri);
    f2 dnxn = mul2(dx, mnx);  // (y - x).n_x
    dnxn = fma2(dy, mny, dnxn);
    dnxn = fma2(dz, mnz, dnxn);
    f2 s0, c0, s1, c1;
    if (CENTRED) {
        f2 num = mul2(ddx, ddx);
        num = fma2(ddy, ddy, num);
        num = fma2(ddz, ddz, num);
        f2 dd = mul2(ddx, cp.Dx);
        dd = fma2(ddy, cp.Dy, dd);
        dd = fma2(ddz, cp.Dz, dd);
        num = fma2(dd, dup2(2.f), num);
        const f2 den = add2(r, cp.rc);
        const f2 dlt = mul2(num, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
        const f2 ph0 = fma2(c.k0, dlt, cp.b0);
        const f2 ph1 = fma2(c.k1, dlt, cp.b1);
        __sincosf(ph0.x, &s0.x, &c0.x);
        __sincosf(ph0.y, &s0.y, &c0.y);
        __sincosf(ph1.x, &s1.x, &c1.x);
        __sincosf(ph1.y, &s1.y, &c1.y);
    } else {
        const f2 kr0 = mul2(r, c.k0), kr1 = mul2(r, c.k1);
        __sincosf(kr0.x, &s0.x, &c0.x);
        __sincosf(kr0.y, &s0.y, &c0.y);
        __sincosf(kr1.x, &s1.x, &c1.x);
        __sincosf(kr1.y, &s1.y, &c1.y);
    }
    const f2 c0r = mul2(c0, ri), s0r = mul2(s0, ri), c1r = mul2(c1, ri), s1r = mul2(s1, ri);
    // V: G0 + rho G1
    const f2 gpr = fma2(c.rho, c1r, c0r), gpi = fma2(c.rho, s1r, s0r);
    // D normal: (-n_x.n_y) dks (G0 + dk1 G1), nn = -n_x.n_y dks
    const f2 gkr = mul2(nn, fma2(c.dk1, c1r, c0r)), gki = mul2(nn, fma2(c.dk1, s1r, s0r));
    // D curl weight: sum_q w_q (G0 + G1/rho)
    const f2 wq = hi2(G1);
    t3r = fma2(fma2(c.irho, c1r, c0r), wq, t3r);
    t3i = fma2(fma2(c.irho, s1r, s0r), wq, t3i);
    // -(H0 + H1) with the scaled c, s (see far_tri)
    const f2 hp = mul2(fma2(c.k1, s1, fma2(c.k0, s0, add2(c0r, c1r))), ri2);
    const f2 hq = mul2(fma2(c.nk1, c1, fma2(c.nk0, c0, add2(s0r, s1r))), ri2);
    // K: (x - y).n_y (H0 + H1) = (-(x - y).n_y)(-(H0 + H1));  T: (H0 + H1)(x - y).n_x
    const f2 kr = mul2(xnyn, hp), ki = mul2(xnyn, hq);
    const f2 tr = mul2(dnxn, hp), ti = mul2(dnxn, hq);
    const f2 m1 = dup2(-1.f);
    const f2 ngpi = mul2(gpi, m1), nki = mul2(ki, m1), nti = mul2(ti, m1), ngki = mul2(gki, m1);
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
        const float4 Ps = D[2 * rr], Ph = D[2 * rr + 1];
        const f2 psr = lo2(Ps), psi = hi2(Ps), phr = lo2(Ph), phi = hi2(Ph);
        u1r[rr] = fma2(gpr, psr, fma2(ngpi, psi, fma2(kr, phr, fma2(nki, phi, u1r[rr]))));
        u1i[rr] = fma2(gpr, psi, fma2(gpi, psr, fma2(kr, phi, fma2(ki, phr, u1i[rr]))));
        u2r[rr] = fma2(tr, psr, fma2(nti, psi, fma2(gkr, phr, fma2(ngki, phi, u2r[rr]))));
        u2i[rr] = fma2(tr, psi, fma2(ti, psr, fma2(gkr, phi, fma2(gki, phr, u2i[rr]))));
    }
}

template <int R, bool CENTRED>
struct FarmBuf {
    float4 *G;   // [TS*6][2]
    float4 *D;   // [TS*6][R][2]
    float2 *C;   // [TS][R][3]
    float4 *N;   // [TS] normal, plane offset
    int4 *V;     // [TS] vertex ids
    float4 *Cen; // [2 TS] (centred)
    __device__ FarmBuf(unsigned char *base) {
        G = reinterpret_cast<float4 *>(base);
        D = G + FARM_TS * 12;
        C = reinterpret_cast<float2 *>(D + FARM_TS * 12 * R);
        N = reinterpret_cast<float4 *>(C + FARM_TS * 3 * R);
        V = reinterpret_cast<int4 *>(N + FARM_TS);
        Cen = reinterpret_cast<float4 *>(V + FARM_TS);
    }
};

// Source tiles are staged by 1-D TMA bulk copies (cp.async.bulk) into a
// two-buffer shared-memory ring: thread 0 issues tile k + 1 while every
// thread computes tile k, and an mbarrier per buffer counts the bytes in.
// Every wait is bounded (FARM_TIMEOUT_NS of global time); a thread that
// gives up sets *err, stops waiting, and writes NaN instead of its sums, and
// thread 0 waits (bounded) for the copies it issued before the block exits.
template <int R, bool CENTRED>
__global__ void __launch_bounds__(FARM_THREADS, OSRC_FARM_MIN_BLOCKS)
farm_kernel(const float4 *__restrict__ pt, const float4 *__restrict__ cen, const float4 *__restrict__ tn,
            const int4 *__restrict__ tv, const float4 *__restrict__ sG, const float4 *__restrict__ sD,
            const float2 *__restrict__ sCm, int nt, int npts, int tris_per_split, FarConst2 c,
            float4 kff, float *__restrict__ part, float *__restrict__ partA, int *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char farm_smem[];
    constexpr size_t BUF = farm_buf_bytes(R, CENTRED);
    float2 *shW = reinterpret_cast<float2 *>(farm_smem + 2 * BUF);  // [TS][threads]
    uint64_t *bar = reinterpret_cast<uint64_t *>(shW + FARM_TS * FARM_THREADS);

    const int j = threadIdx.x;
    const int lt = j / 3, sub = j - 3 * (j / 3);
    const int tau_raw = blockIdx.x * FARM_TRIS + lt;
    const bool active = tau_raw < nt;
    const int tau = active ? tau_raw : 0;
    const int p0 = 6 * tau + 2 * sub;
    const int split = blockIdx.y;
    const int s_begin = split * tris_per_split;
    const int s_end = min(nt, s_begin + tris_per_split);
    const int ntiles = s_end > s_begin ? (s_end - s_begin + FARM_TS - 1) / FARM_TS : 0;
    const float4 xa = pt[p0], xb = pt[p0 + 1];
    const f2 X = make_float2(xa.x, xb.x), Y = make_float2(xa.y, xb.y), Z = make_float2(xa.z, xb.z);
    const float4 n4 = tn[tau];
    const int4 vt = tv[tau];
    const f2 mnx = dup2(-n4.x), mny = dup2(-n4.y), mnz = dup2(-n4.z);
    const float wa = (float)(2 * sub < 3 ? kQw1 : kQw2), wb = (float)(2 * sub + 1 < 3 ? kQw1 : kQw2);
    float4 cth = make_float4(0.f, 0.f, 0.f, 0.f), ctl = cth;
    if (CENTRED) {
        cth = cen[2 * tau];
        ctl = cen[2 * tau + 1];
    }
    f2 u1r[R], u1i[R], u2r[R], u2i[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) u1r[rr] = u1i[rr] = u2r[rr] = u2i[rr] = make_float2(0.f, 0.f);

    // thread 0: the copies of tile k into buffer k & 1
    auto issue = [&](int k) {
        const int t0 = s_begin + k * FARM_TS;
        const int cnt = min(FARM_TS, s_end - t0);
        FarmBuf<R, CENTRED> fb(farm_smem + (k & 1) * BUF);
        uint64_t *mb = &bar[k & 1];
        const uint32_t bytes = (uint32_t)cnt * (12 * 16 + 12 * 16 * R + 24 * R + 16 + 16 + (CENTRED ? 32 : 0));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(farm_saddr(mb)), "r"(bytes)
                     : "memory");
        farm_bulk(fb.G, sG + 12 * (size_t)t0, (uint32_t)cnt * 12 * 16, mb);
        farm_bulk(fb.D, sD + 12 * (size_t)R * t0, (uint32_t)cnt * 12 * 16 * R, mb);
        farm_bulk(fb.C, sCm + 3 * (size_t)R * t0, (uint32_t)cnt * 24 * R, mb);
        farm_bulk(fb.N, tn + t0, (uint32_t)cnt * 16, mb);
        farm_bulk(fb.V, tv + t0, (uint32_t)cnt * 16, mb);
        if (CENTRED) farm_bulk(fb.Cen, cen + 2 * (size_t)t0, (uint32_t)cnt * 32, mb);
    };
    if (j == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(farm_saddr(&bar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(farm_saddr(&bar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (j == 0 && ntiles > 0) issue(0);
    bool dead = false;      // a bounded wait gave up
    int issued = ntiles > 0 ? 1 : 0;  // tiles issued (thread 0)

    for (int k = 0; k < ntiles; ++k) {
        const int t0 = s_begin + k * FARM_TS;
        const int cnt = min(FARM_TS, s_end - t0);
        FarmBuf<R, CENTRED> fb(farm_smem + (k & 1) * BUF);
        if (!dead && !farm_wait(&bar[k & 1], (uint32_t)(k >> 1) & 1u)) {
            dead = true;
            atomicExch(err, 1);
        }
        // the other buffer held tile k - 1, released by the barrier that ended it
        if (j == 0 && !dead && k + 1 < ntiles) {
            issue(k + 1);
            issued = k + 2;
        }
        for (int s = 0; s < cnt; ++s) {
            const int4 vs = fb.V[s];
            const bool touch = (vs.x == vt.x) | (vs.x == vt.y) | (vs.x == vt.z) |
                               (vs.y == vt.x) | (vs.y == vt.y) | (vs.y == vt.z) |
                               (vs.z == vt.x) | (vs.z == vt.y) | (vs.z == vt.z);
            if (touch) {
                shW[s * FARM_THREADS + j] = make_float2(0.f, 0.f);
                continue;
            }
            const float4 ns = fb.N[s];
            const float4 mns = make_float4(-ns.x, -ns.y, -ns.z, ns.w);
            CenterPair cp;
            f2 xnyn;
            if (CENTRED) {
                cp = center_pair(cth, ctl, fb.Cen[2 * s], fb.Cen[2 * s + 1], kff.x, kff.y, kff.z, kff.w);
                const float dn = cp.Dx.x * mns.x + cp.Dy.x * mns.y + cp.Dz.x * mns.z;
                xnyn = fma2(Z, dup2(mns.z), fma2(Y, dup2(mns.y), fma2(X, dup2(mns.x), dup2(dn))));
            } else {
                xnyn = fma2(Z, dup2(mns.z), fma2(Y, dup2(mns.y), fma2(X, dup2(mns.x), dup2(mns.w))));
            }
            const f2 nn = dup2((n4.x * mns.x + n4.y * mns.y + n4.z * mns.z) * c.dk0.x);
            f2 t3r = make_float2(0.f, 0.f), t3i = t3r;
#pragma unroll FARM_QUNROLL
            for (int q = 0; q < 6; ++q)
                farm_pair<R, CENTRED>(X, Y, Z, fb.G[12 * s + 2 * q], fb.G[12 * s + 2 * q + 1],
                                      &fb.D[2 * R * (6 * s + q)], mnx, mny, mnz, xnyn, nn, c, cp, t3r,
                                      t3i, u1r, u1i, u2r, u2i);
            shW[s * FARM_THREADS + j] = make_float2(wa * t3r.x + wb * t3r.y, wa * t3i.x + wb * t3i.y);
        }
        __syncthreads();
        // curl term of this tile: thread (lt, sub) takes right-hand sides sub, sub + 3, ...
        if (active) {
            for (int rr = sub; rr < R; rr += 3) {
                float ar[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int s = 0; s < cnt; ++s) {
                    const float2 *w3 = shW + s * FARM_THREADS + 3 * lt;
                    const float wr = w3[0].x + w3[1].x + w3[2].x, wi = w3[0].y + w3[1].y + w3[2].y;
                    const float2 *cc = fb.C + 3 * (s * R + rr);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float2 cv = cc[d];
                        ar[2 * d] += wr * cv.x - wi * cv.y;
                        ar[2 * d + 1] += wr * cv.y + wi * cv.x;
                    }
                }
                float *pa = partA + (((size_t)split * R + rr) * 6) * nt + tau;
#pragma unroll
                for (int d = 0; d < 6; ++d) pa[(size_t)d * nt] = k == 0 ? ar[d] : pa[(size_t)d * nt] + ar[d];
            }
        }
        __syncthreads();
    }
    if (j == 0 && dead) {  // copies still in flight land before the block exits: the
                           // last tile issued into each buffer
        for (int k = max(0, issued - 2); k < issued; ++k)
            if (!farm_wait(&bar[k & 1], (uint32_t)(k >> 1) & 1u)) break;
    }
    if (active) {
        f2 *pp = reinterpret_cast<f2 *>(part);
        const f2 nan2 = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
            const size_t base = (((size_t)split * R + rr) * 4) * npts + p0;
            pp[base / 2] = dead ? nan2 : u1r[rr];
            pp[(base + (size_t)npts) / 2] = dead ? nan2 : u1i[rr];
            pp[(base + 2 * (size_t)npts) / 2] = dead ? nan2 : u2r[rr];
            pp[(base + 3 * (size_t)npts) / 2] = dead ? nan2 : u2i[rr];
        }
        if (ntiles == 0)  // empty split: zero curl sums
            for (int rr = sub; rr < R; rr += 3)
                for (int d = 0; d < 6; ++d) partA[(((size_t)split * R + rr) * 6 + d) * nt + tau] = 0.f;
    }
}

}  // namespace

int far_setup_geometry(osrc_problem *pb, cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt;
    OSRC_TRY(pb->d_pt.alloc(m->ctx, 6 * (size_t)nt));
    OSRC_TRY(pb->d_poff.alloc(m->ctx, 6 * (size_t)nt));
    OSRC_TRY(pb->d_cen.alloc(m->ctx, 2 * (size_t)nt));
    OSRC_TRY(pb->d_tn.alloc(m->ctx, nt));
    OSRC_TRY(pb->d_tv.alloc(m->ctx, nt));
    OSRC_TRY(pb->d_tgeo.alloc(m->ctx, 16 * (size_t)nt));
    OSRC_TRY(pb->d_sP.alloc(m->ctx, 24 * (size_t)nt));
    OSRC_TRY(pb->d_sP5.alloc(m->ctx, 6 * (size_t)nt));
    OSRC_TRY(pb->d_sC.alloc(m->ctx, 2 * (size_t)nt));
    far_geom_kernel<<<(nt + 127) / 128, 128, 0, st>>>(m->d_verts.p, m->d_tris.p, nt, pb->d_pt.p,
                                                      pb->d_poff.p, pb->d_cen.p, pb->d_tn.p,
                                                      pb->d_tv.p, pb->d_tgeo.p);
    pb->launches++;
    OSRC_CK(cudaGetLastError());
    // largest phase k r over the mesh (bounding-box diagonal): beyond
    // FAR_PLAIN_MAX_PHASE radians the centred variant with float-float
    // phases is used.  The plain variant's FP32 phase error grows linearly
    // with k r: measured 1.04e-5 relative (operator apply) at
    // k_max x diagonal = 63 pi, so the switch sits at 32 pi (about 5e-6)
    {
        double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
        for (int i = 0; i < m->nv; ++i)
            for (int d = 0; d < 3; ++d) {
                lo[d] = fmin(lo[d], m->verts[3 * i + d]);
                hi[d] = fmax(hi[d], m->verts[3 * i + d]);
            }
        const double diag = sqrt((hi[0] - lo[0]) * (hi[0] - lo[0]) + (hi[1] - lo[1]) * (hi[1] - lo[1]) +
                                 (hi[2] - lo[2]) * (hi[2] - lo[2]));
        double kmax = fmax(pb->p.k_ext, pb->p.k_int);
        for (const ObjMat &o : pb->obj) kmax = fmax(kmax, o.k1);
        pb->far_reduce = kmax * diag > FAR_PLAIN_MAX_PHASE;
    }
    // Test triangles per block and source splits.  Small meshes take few test
    // triangles per block (the block's warps then share the sources); the
    // splits, at least FAR_MIN_TPS source triangles each so that summing the
    // partial sums stays small beside the pair work, fill the resident blocks
    // four times over, and near that number the one with the fullest last
    // wave is taken.
    int dev = m->ctx->device, sms = 0;
    OSRC_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    pb->far_tris = nt < FAR_TRIS32_NT ? 32 : nt < FAR_TRIS64_NT ? 64 : FAR_THREADS;
    const int slots = sms * OSRC_FAR_MIN_BLOCKS;
    const int bx = (nt + pb->far_tris - 1) / pb->far_tris;
    const int max_ns = std::max(1, std::min(FAR_MAX_NS, nt / FAR_MIN_TPS));
    const int ns0 = std::min(max_ns, std::max(1, (4 * slots + bx - 1) / bx));
    int ns = ns0;
    double best = -1.0;
    for (int cand = std::max(1, ns0 / 2); cand <= std::min(max_ns, 2 * ns0); ++cand) {
        const long long blocks = (long long)bx * cand;
        const long long waves = (blocks + slots - 1) / slots;
        const double eff = (double)blocks / (double)(waves * slots);
        if (eff > best + 1e-9) {
            best = eff;
            ns = cand;
        }
    }
    pb->nsplit = ns;
    OSRC_TRY(pb->d_part.alloc(m->ctx, (size_t)ns * 4 * pb->npts));
    OSRC_TRY(pb->d_partA1.alloc(m->ctx, (size_t)ns * 6 * nt));
    return OSRC_OK;
}

// Adds the duration of the last timed far-kernel launch to the statistics.
int far_prof_collect(osrc_problem *pb) {
    if (!pb->prof_pending) return OSRC_OK;
    OSRC_CK(cudaEventSynchronize(pb->prof_ev[1]));
    float ms = 0.f;
    OSRC_CK(cudaEventElapsedTime(&ms, pb->prof_ev[0], pb->prof_ev[1]));
    pb->prof_ms += ms;
    pb->prof_launches++;
    pb->prof_rhs += pb->prof_rhs_pending;
    pb->prof_rhs_pending = 1;
    pb->prof_pending = false;
    return OSRC_OK;
}

static int gather_launch(osrc_problem *pb, int ns, int R, const float *part, const float *partA, int use_far,
                         int use_near, const VecPtrs &x, const OutPtrs &y, cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nv = pb->nv;
    const int per = nv <= GATHER_BLOCK_NV ? 1 : nv <= GATHER_WARP_NV ? GATHER_THREADS / 32 : GATHER_THREADS / 8;
    const dim3 grid((nv + per - 1) / per, R);
#define OSRC_GATHER_LAUNCH(LL, WW)                                                                             \
    gather_kernel<LL, WW><<<grid, GATHER_THREADS, 0, st>>>(nv, pb->nt, pb->npts, ns, R, m->d_vt_ptr.p, m->d_vt_idx.p, \
                                                       pb->d_tgeo.p, part, partA, use_far, pb->d_nr_ptr.p,       \
                                                       pb->d_nr_col.p, pb->d_nr_val.p, use_near, x, y)
    if (nv <= GATHER_BLOCK_NV) OSRC_GATHER_LAUNCH(32, 4);
    else if (nv <= GATHER_WARP_NV) OSRC_GATHER_LAUNCH(32, 1);
    else OSRC_GATHER_LAUNCH(8, 1);
#undef OSRC_GATHER_LAUNCH
    pb->launches++;
    OSRC_CK(cudaGetLastError());
    return OSRC_OK;
}

int far_apply(osrc_problem *pb, const double2 *x, double2 *y, int part, cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt, nv = pb->nv, npts = pb->npts;
    const int use_far = (part & OSRC_PART_FAR) ? 1 : 0;
    const int use_near = (part & OSRC_PART_NEAR) ? 1 : 0;
    if (use_far) {
        const float4 *src_pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
        far_prep_kernel<<<(npts + 127) / 128, 128, 0, st>>>(x, nv, nt, m->d_tris.p, src_pts,
                                                          pb->d_tgeo.p, pb->d_sP.p, pb->d_sP5.p,
                                                          pb->d_sC.p);
        pb->launches++;
        const double k0 = pb->p.k_ext, k1 = pb->p.k_int, rho = pb->p.rho_ratio;
        const double inv2pi = 0.15915494309189533577;
        auto d2 = [](double v) { return make_float2((float)v, (float)v); };
        FarConst2 c;
        c.k0 = d2(k0);
        c.k1 = d2(k1);
        c.nk0 = d2(-k0);
        c.nk1 = d2(-k1);
        c.rho = d2(rho);
        c.irho = d2(1.0 / rho);
        c.dk0 = d2(pb->far_dks);
        c.dk1 = d2(k1 * k1 / rho / pb->far_dks);
        // k / (2 pi) as float pairs (hi, lo) for the float-float phases
        const double q0 = k0 * inv2pi, q1 = k1 * inv2pi;
        const float q0h = (float)q0, q1h = (float)q1;
        const float4 kff = make_float4(q0h, (float)(q0 - (double)q0h), q1h, (float)(q1 - (double)q1h));
        const int ns = pb->nsplit;
        const int tps = (nt + ns - 1) / ns;
        dim3 grid((nt + pb->far_tris - 1) / pb->far_tris, ns);
        if (pb->prof_on) {
            OSRC_TRY(far_prof_collect(pb));
            OSRC_CK(cudaEventRecord(pb->prof_ev[0], st));
        }
        const float4 *pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
        const int *tc = m->d_tcomp.p;
        const FarObj *fo = pb->d_fobj.p;
        float *prt = pb->d_part.p;
        const bool ab = pb->absorb;
#define OSRC_FAR_LAUNCH(C, M, A)                                                                               \
    far_kernel<C, M, A><<<grid, FAR_THREADS, 0, st>>>(pts, pb->d_cen.p, pb->d_tn.p, pb->d_tv.p, pb->d_sP.p,  \
                                                          pb->d_sP5.p, pb->d_sC.p, nt, npts, tps, pb->far_tris, c, kff, tc, fo, \
                                                          prt, pb->d_partA1.p)
        if (pb->far_reduce && pb->far_obj && ab) OSRC_FAR_LAUNCH(true, true, true);
        else if (pb->far_reduce && pb->far_obj) OSRC_FAR_LAUNCH(true, true, false);
        else if (pb->far_reduce) OSRC_FAR_LAUNCH(true, false, false);
        else if (pb->far_obj && ab) OSRC_FAR_LAUNCH(false, true, true);
        else if (pb->far_obj) OSRC_FAR_LAUNCH(false, true, false);
        else OSRC_FAR_LAUNCH(false, false, false);
#undef OSRC_FAR_LAUNCH
        pb->launches++;
        if (pb->prof_on) {
            OSRC_CK(cudaEventRecord(pb->prof_ev[1], st));
            pb->prof_pending = true;
        }
    }
    VecPtrs xp{};
    OutPtrs yp{};
    xp.p[0] = x;
    yp.p[0] = y;
    return gather_launch(pb, pb->nsplit, 1, pb->d_part.p, pb->d_partA1.p, use_far, use_near, xp, yp, st);
}

// ---------------------------------------------------------------------------
// multi-right-hand-side apply: y_r = B_far x_r (+ near) for r < nrhs, in
// launches of up to FARM_MAX_R right-hand sides (chunks of 8, then 4, 2;
// a last single vector takes the one-right-hand-side kernel)
// ---------------------------------------------------------------------------
template <int R, bool C>
static int farm_setup_kernel_attr(size_t smem) {
    OSRC_CK(cudaFuncSetAttribute(farm_kernel<R, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return OSRC_OK;
}

static PerDeviceOnce g_farm_once;

static int farm_prepare(osrc_problem *pb, int rmax, cudaStream_t st) {
    OSRC_TRY(per_device_once(g_farm_once, [](int) {
        int s = OSRC_OK;
        if (!s) s = farm_setup_kernel_attr<2, false>(farm_smem_bytes(2, false));
        if (!s) s = farm_setup_kernel_attr<4, false>(farm_smem_bytes(4, false));
        if (!s) s = farm_setup_kernel_attr<8, false>(farm_smem_bytes(8, false));
        if (!s) s = farm_setup_kernel_attr<2, true>(farm_smem_bytes(2, true));
        if (!s) s = farm_setup_kernel_attr<4, true>(farm_smem_bytes(4, true));
        if (!s) s = farm_setup_kernel_attr<8, true>(farm_smem_bytes(8, true));
        return s;
    }));
    osrc_ctx *ctx = pb->mesh->ctx;
    const int nt = pb->nt, npts = pb->npts;
    if (!pb->d_sG.p) {
        OSRC_TRY(pb->d_sG.alloc(ctx, 2 * (size_t)npts));
        const float4 *pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
        farm_geom_kernel<<<(npts + 127) / 128, 128, 0, st>>>(pts, npts, pb->d_sG.p);
        pb->launches++;
        OSRC_CK(cudaGetLastError());
    }
    if (pb->farm_cap < rmax) {
        int dev = ctx->device, sms = 0, per_sm = 0;
        OSRC_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const size_t sm8 = farm_smem_bytes(8, pb->far_reduce);
        if (pb->far_reduce)
            OSRC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, farm_kernel<8, true>, FARM_THREADS, sm8));
        else
            OSRC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, farm_kernel<8, false>, FARM_THREADS, sm8));
        if (per_sm < 1) per_sm = 1;
        // source splits: at least four blocks per resident slot, and among
        // the counts up to twice that, the one whose last wave is fullest
        const int bx = (nt + FARM_TRIS - 1) / FARM_TRIS;
        const int slots = sms * per_sm;
        const int max_ns = std::max(1, (nt + 4 * FARM_TS - 1) / (4 * FARM_TS));
        int ns0 = std::min(max_ns, std::max(1, (4 * slots + bx - 1) / bx));
        int ns = ns0;
        double best = -1.0;
        for (int cand = ns0; cand <= std::min(max_ns, 2 * ns0); ++cand) {
            const long long blocks = (long long)bx * cand;
            const long long waves = (blocks + slots - 1) / slots;
            const double eff = (double)blocks / (double)(waves * slots);
            if (eff > best + 1e-9) {
                best = eff;
                ns = cand;
            }
        }
        pb->farm_ns = ns;
        pb->d_sD.release();
        pb->d_sCm.release();
        pb->d_partm.release();
        pb->d_partA.release();
        OSRC_TRY(pb->d_sD.alloc(ctx, 12 * (size_t)nt * FARM_MAX_R));
        OSRC_TRY(pb->d_sCm.alloc(ctx, 3 * (size_t)nt * FARM_MAX_R));
        OSRC_TRY(pb->d_partm.alloc(ctx, (size_t)ns * FARM_MAX_R * 4 * npts));
        OSRC_TRY(pb->d_partA.alloc(ctx, (size_t)ns * FARM_MAX_R * 6 * nt));
        if (!pb->d_farm_err.p) {
            OSRC_TRY(pb->d_farm_err.alloc(ctx, 1));
            OSRC_CK(cudaMemsetAsync(pb->d_farm_err.p, 0, sizeof(int), st));
        }
        pb->farm_cap = FARM_MAX_R;
    }
    return OSRC_OK;
}

static int farm_launch(osrc_problem *pb, const double2 *const *xs, double2 *const *ys, int R, int part,
                       cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt, nv = pb->nv, npts = pb->npts;
    const int use_far = (part & OSRC_PART_FAR) ? 1 : 0;
    const int use_near = (part & OSRC_PART_NEAR) ? 1 : 0;
    VecPtrs xp{};
    OutPtrs yp{};
    for (int r = 0; r < R; ++r) {
        xp.p[r] = xs[r];
        yp.p[r] = ys[r];
    }
    const int ns = pb->farm_ns;
    if (use_far) {
        farm_prep_kernel<<<dim3((nt + 127) / 128, R), 128, 0, st>>>(xp, R, nv, nt, m->d_tris.p, pb->d_tgeo.p,
                                                                   pb->d_sD.p, pb->d_sCm.p);
        pb->launches++;
        const double k0 = pb->p.k_ext, k1 = pb->p.k_int, rho = pb->p.rho_ratio;
        const double inv2pi = 0.15915494309189533577;
        auto d2 = [](double v) { return make_float2((float)v, (float)v); };
        FarConst2 c;
        c.k0 = d2(k0);
        c.k1 = d2(k1);
        c.nk0 = d2(-k0);
        c.nk1 = d2(-k1);
        c.rho = d2(rho);
        c.irho = d2(1.0 / rho);
        c.dk0 = d2(pb->far_dks);
        c.dk1 = d2(k1 * k1 / rho / pb->far_dks);
        const double q0 = k0 * inv2pi, q1 = k1 * inv2pi;
        const float q0h = (float)q0, q1h = (float)q1;
        const float4 kff = make_float4(q0h, (float)(q0 - (double)q0h), q1h, (float)(q1 - (double)q1h));
        const int tps = (nt + ns - 1) / ns;
        dim3 grid((nt + FARM_TRIS - 1) / FARM_TRIS, ns);
        const float4 *pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
        const size_t smem = farm_smem_bytes(R, pb->far_reduce);
        if (pb->prof_on) {
            OSRC_TRY(far_prof_collect(pb));
            OSRC_CK(cudaEventRecord(pb->prof_ev[0], st));
        }
#define OSRC_FARM_LAUNCH(RR, C)                                                                          \
    farm_kernel<RR, C><<<grid, FARM_THREADS, smem, st>>>(pts, pb->d_cen.p, pb->d_tn.p, pb->d_tv.p, pb->d_sG.p, \
                                                         pb->d_sD.p, pb->d_sCm.p, nt, npts, tps, c, kff,    \
                                                         pb->d_partm.p, pb->d_partA.p, pb->d_farm_err.p)
        if (pb->far_reduce) {
            if (R == 8) OSRC_FARM_LAUNCH(8, true);
            else if (R == 4) OSRC_FARM_LAUNCH(4, true);
            else OSRC_FARM_LAUNCH(2, true);
        } else {
            if (R == 8) OSRC_FARM_LAUNCH(8, false);
            else if (R == 4) OSRC_FARM_LAUNCH(4, false);
            else OSRC_FARM_LAUNCH(2, false);
        }
#undef OSRC_FARM_LAUNCH
        pb->launches++;
        OSRC_CK(cudaGetLastError());
        if (pb->prof_on) {
            OSRC_CK(cudaEventRecord(pb->prof_ev[1], st));
            pb->prof_pending = true;
            pb->prof_rhs_pending = R;
        }
    }
    return gather_launch(pb, ns, R, pb->d_partm.p, pb->d_partA.p, use_far, use_near, xp, yp, st);
}

// OSRC_TIMEOUT if a several-right-hand-side far kernel gave up a bounded
// wait since the last check (the flag is cleared); synchronises the stream
int far_multi_check(osrc_problem *pb, cudaStream_t st) {
    if (!pb->d_farm_err.p) return OSRC_OK;
    int h = 0;
    OSRC_CK(cudaMemcpyAsync(&h, pb->d_farm_err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    OSRC_CK(cudaStreamSynchronize(st));
    if (h) {
        OSRC_CK(cudaMemsetAsync(pb->d_farm_err.p, 0, sizeof(int), st));
        osrc_set_error("far kernel: a bounded wait for a staged source tile gave up");
        return OSRC_TIMEOUT;
    }
    return OSRC_OK;
}

bool far_multi_supported(const osrc_problem *pb) {
    return pb->p.precision == OSRC_FP32_MATFREE && !pb->far_obj;
}

int far_apply_multi(osrc_problem *pb, const double2 *const *xs, double2 *const *ys, int nrhs, int part,
                    cudaStream_t st) {
    if (nrhs < 1) return OSRC_INVALID_ARG;
    if (nrhs == 1 || !far_multi_supported(pb) || !(part & OSRC_PART_FAR)) {
        for (int r = 0; r < nrhs; ++r) OSRC_TRY(far_apply(pb, xs[r], ys[r], part, st));
        return OSRC_OK;
    }
    OSRC_TRY(farm_prepare(pb, FARM_MAX_R, st));
    int r0 = 0;
    while (r0 < nrhs) {
        const int left = nrhs - r0;
        const int R = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        if (R == 1) OSRC_TRY(far_apply(pb, xs[r0], ys[r0], part, st));
        else OSRC_TRY(farm_launch(pb, xs + r0, ys + r0, R, part, st));
        r0 += R;
    }
    return OSRC_OK;
}
