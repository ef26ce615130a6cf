// k_far.cu -- matrix-free FP32 far-field apply of the permuted PMCHWT
// operator (Sec. 2.7) for all triangle pairs that share no vertex, with the
// 6-point degree-4 triangle rule (Strang & Fix / Dunavant) on both triangles.
//
// Structure of one apply y = B_far x:
//   1. far_prep_kernel   (per source rule point)  densities at the 6 source
//      points and the surface-curl vector of the phi density, FP32;
//   2. below SYM_MIN_NT triangles far_kernel (per test triangle), N-body sum
//      over all source points staged through shared memory in tiles of triangles; both
//      wavenumbers are evaluated from one distance; the source range is split
//      over gridDim.y so that the grid fills every SM; partial sums per test
//      point (u1, u2) and per test triangle (curl term) go to d_part, d_partA1
//      (no atomics); from SYM_MIN_NT on sym_kernel, which evaluates each pair of
//      triangles once, as element matrices, for both directions, and takes
//      several right-hand sides (farm_kernel: the same one-sided, for several
//      right-hand sides on small meshes and more than SYM_MAX_R);
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

// Scale of the weights in the element matrices of one vector, chosen so that all
// four (weight times barycentric coordinate, of both classes) are FP32 numbers to
// 4e-10: rounded as they are, they scale every value by 1 + 3.7e-8 and the corners'
// shares by up to 1.4e-7 (1 % of an apply's error).
constexpr double kElemScale = 0.982727956;

constexpr int FAR_THREADS = 128;
// resident blocks per SM the one-right-hand-side kernel is compiled for
// (registers per thread = 65536 / (FAR_THREADS x FAR_MIN_BLOCKS))
constexpr int FAR_MIN_BLOCKS = 2;
// largest k_max x (bounding-box diagonal) for the plain (FP32 k r) variant
constexpr double FAR_PLAIN_MAX_PHASE = 32.0 * 3.14159265358979323846;
constexpr int FAR_TS = 64;  // source triangles per shared-memory tile
constexpr int FAR_MIN_TPS = 16;  // fewest source triangles per split
// test triangles per block: 32 below FAR_TRIS32_NT triangles, 64 below
// FAR_TRIS64_NT, else FAR_THREADS (128).  far_kernel (meshes below SYM_MIN_NT) has
// 32: 296 triangles 52 us an apply with 32 sharing the sources between four warps,
// 54 with 64, 64 with 128.  64 and 128 are farm_kernel's (6 and more vectors there);
// 8 vectors take, with 32 / 64 / 128, at 1796 triangles 509 / 564 / 535 us, 2048:
// 622 / 600 / 609, 4094: 2.22 / 2.14 / 2.13 ms, 7996: 8.24 / 7.88 / 7.92, 11996:
// 18.4 / 17.7 / 17.5, 19996: 51.3 / 49.4 / 48.9
constexpr int FAR_TRIS32_NT = 2048;
constexpr int FAR_TRIS64_NT = 4096;
constexpr int FAR_MAX_NS = 64;   // most source splits
// sym_kernel from this many triangles on (far_kernel / sym_kernel at 796
// triangles 73 / 97 us, 1280: 144 / 145, 2048: 299 / 276, 2996: 618 / 506, 3996:
// 1062 / 940, 20480: 25.9 / 17.4 ms; its work comes in tiles of 128 x 32
// triangles, too few of them for small meshes)
constexpr int SYM_MIN_NT = 2048;
constexpr int SYM_MAX_SLOTS = 104;  // most partial sums of an apply (R = 1): 104 x 18 floats a triangle
                                    // (70 or 200 measure the same within 1 %)
// right-hand sides of a sym_kernel launch: what two blocks per SM have shared
// memory for (8 as 5 + 3 would take 55.1 ms at 10242 vertices, farm_kernel 49.0)
constexpr int SYM_MAX_R = 5;
constexpr int SYM_MULTI_SLOTS = 96; // partial sums, times right-hand sides, of several-right-hand-side launches
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

// Kernel values of one source point at the six test points (three pairs):
// c / r and s / r of both wavenumbers, -(H0 + H1) r^2 = hp + i hq, 1 / r^2, and
// (y - x).n_x.
struct FarVals {
    f2 c0r[3], s0r[3], c1r[3], s1r[3], hp[3], hq[3], ri2[3], dnxn;
};

#define F3 _Pragma("unroll") for (int p = 0; p < 3; ++p)
template <bool CENTRED, bool MULTI, bool ABSORB>
__device__ __forceinline__ FarVals far_vals(const f2 (&X)[3], const f2 (&Y)[3], const f2 (&Z)[3], const float4 &n4,
                                            float pdn, const float4 &P0, const float4 &P1, const FarConst2 &c,
                                            const CenterPair &cp, f2 m1, f2 k1i) {
    FarVals v;
    Diff2 d[3];
    F3 d[p] = far_diff<CENTRED>(X[p], Y[p], Z[p], P0, P1, cp);
    v.dnxn = CENTRED ? dup2(-fmaf(P0.x, n4.x, fmaf(P0.z, n4.y, fmaf(P1.x, n4.z, pdn))))
                     : dup2(-fmaf(d[0].dz.x, n4.z, fmaf(d[0].dy.x, n4.y, fmaf(d[0].dx.x, n4.x, pdn))));
    f2 r2[3], ri[3], r[3], s0[3], c0[3], s1[3], c1[3];
    F3 r2[p] = mul2(d[p].dx, d[p].dx);
    F3 r2[p] = fma2(d[p].dy, d[p].dy, r2[p]);
    F3 r2[p] = fma2(d[p].dz, d[p].dz, r2[p]);
    F3 ri[p] = make_float2(rsqrtf(r2[p].x), rsqrtf(r2[p].y));
    F3 r[p] = mul2(r2[p], ri[p]);
    F3 v.ri2[p] = mul2(ri[p], ri[p]);
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
    // cos and sin scaled by 1/r once: G = (c + i s)/r for every kernel below
    F3 v.c0r[p] = mul2(c0[p], ri[p]);
    F3 v.s0r[p] = mul2(s0[p], ri[p]);
    F3 v.c1r[p] = mul2(c1[p], ri[p]);
    F3 v.s1r[p] = mul2(s1[p], ri[p]);
    // -(H0 + H1) r^2, H = e^{ikr} (i k r - 1) / r^3, with the scaled c, s:
    //   re = c0/r + c1/r + k0 s0 + k1 s1,  im = s0/r + s1/r - k0 c0 - k1 c1
    F3 v.hp[p] = add2(v.c0r[p], v.c1r[p]);
    F3 v.hq[p] = add2(v.s0r[p], v.s1r[p]);
    F3 v.hp[p] = fma2(c.k0, s0[p], v.hp[p]);
    F3 v.hp[p] = fma2(c.k1, s1[p], v.hp[p]);
    F3 v.hq[p] = fma2(c.nk0, c0[p], v.hq[p]);
    F3 v.hq[p] = fma2(c.nk1, c1[p], v.hq[p]);
    if (absorb) {  // (i k1 r - 1) with Im k1: + k1i r (c1, s1) / r
        F3 v.hp[p] = fma2(k1i, c1[p], v.hp[p]);
        F3 v.hq[p] = fma2(k1i, s1[p], v.hq[p]);
    }
    return v;
}

template <bool CENTRED, bool MULTI, bool ABSORB>
__device__ __forceinline__ void far_tri(const f2 (&X)[3], const f2 (&Y)[3], const f2 (&Z)[3], const float4 &n4,
                                        float pdn, const float4 &P0, const float4 &P1, const float4 &P2, const float4 &P3,
                                        const f2 &P5, const FarConst2 &c, const CenterPair &cp, f2 m1, f2 k1i,
                                        f2 dk1i, PairAcc (&A)[3], CurlAcc &B) {
    constexpr bool absorb = MULTI && ABSORB;
    FarVals v = far_vals<CENTRED, MULTI, ABSORB>(X, Y, Z, n4, pdn, P0, P1, c, cp, m1, k1i);
    const f2 psr = hi2(P1), psi = lo2(P2), mpsi = hi2(P2), phr = lo2(P3), phi = hi2(P3), mphi = P5;
    f2 ga[3], gb[3];
    // D curl term: sums of G0 and G1, weighted and combined by the caller
    F3 B.g0r = add2(B.g0r, v.c0r[p]);
    F3 B.g0i = add2(B.g0i, v.s0r[p]);
    F3 B.g1r = add2(B.g1r, v.c1r[p]);
    F3 B.g1i = add2(B.g1i, v.s1r[p]);
    // V block (G0 + rho G1) psi, without 1/(4 pi)
    F3 ga[p] = fma2(c.rho, v.c1r[p], v.c0r[p]);
    F3 gb[p] = fma2(c.rho, v.s1r[p], v.s0r[p]);
    F3 A[p].u1r = fma2(gb[p], mpsi, A[p].u1r);
    F3 A[p].u1i = fma2(gb[p], psr, A[p].u1i);
    F3 A[p].u1r = fma2(ga[p], psr, A[p].u1r);
    F3 A[p].u1i = fma2(ga[p], psi, A[p].u1i);
    // D normal term (k0^2 G0 + k1^2/rho G1) phi, as (G0 + dk1 G1) phi; the
    // scale dks is applied per source triangle
    F3 ga[p] = fma2(c.dk1, v.c1r[p], v.c0r[p]);
    F3 gb[p] = fma2(c.dk1, v.s1r[p], v.s0r[p]);
    if (absorb) {  // complex k1^2 / (rho dks)
        F3 ga[p] = fma2(mul2(dk1i, v.s1r[p]), dup2(-1.f), ga[p]);
        F3 gb[p] = fma2(dk1i, v.c1r[p], gb[p]);
    }
    F3 A[p].ur = fma2(gb[p], mphi, A[p].ur);
    F3 A[p].ui = fma2(gb[p], phr, A[p].ui);
    F3 A[p].ur = fma2(ga[p], phr, A[p].ur);
    F3 A[p].ui = fma2(ga[p], phi, A[p].ui);
    // T1n = -sum Hs phi
    F3 v.hp[p] = mul2(v.hp[p], v.ri2[p]);
    F3 v.hq[p] = mul2(v.hq[p], v.ri2[p]);
    F3 A[p].t1r = fma2(v.hq[p], mphi, A[p].t1r);
    F3 A[p].t1i = fma2(v.hq[p], phr, A[p].t1i);
    F3 A[p].t1r = fma2(v.hp[p], phr, A[p].t1r);
    F3 A[p].t1i = fma2(v.hp[p], phi, A[p].t1i);
    // T block: (H0 + H1)(x - y).n_x psi = (-(H0 + H1)) (y - x).n_x psi
    F3 v.hp[p] = mul2(v.hp[p], v.dnxn);
    F3 v.hq[p] = mul2(v.hq[p], v.dnxn);
    F3 A[p].u2r = fma2(v.hq[p], mpsi, A[p].u2r);
    F3 A[p].u2i = fma2(v.hq[p], psr, A[p].u2i);
    F3 A[p].u2r = fma2(v.hp[p], psr, A[p].u2r);
    F3 A[p].u2i = fma2(v.hp[p], psi, A[p].u2i);
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
// variant (a third).  642 vertices: 0.144 ms an apply, 1.67 ms at 2562 (0.16 and
// 1.85 where a thread held one pair of points; sym_kernel 0.145 and 1.31).  255
// registers and two blocks per SM measured 1 to 4 % better than 168 and three.
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
__global__ void __launch_bounds__(FAR_THREADS, FAR_MIN_BLOCKS)
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
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // the two weight classes of the source points
                CurlAcc Bs;
                Bs.g0r = Bs.g0i = Bs.g1r = Bs.g1i = make_float2(0.f, 0.f);
#pragma unroll
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
// incident (triangle t, local index a), from far_kernel's sums:
//   y1_v = (1/4pi) sum |t| sum_q w_q lambda_a(q) u1(t,q)
//   y2_v = (1/4pi) sum |t| [sum_q w_q lambda_a(q) u2(t,q) + curl_a . A(t)]
// or from farm_kernel's (E), which hold the test weights already:
//   y1_v = (1/4pi) sum |t| E1(t,a),  y2_v = (1/4pi) sum |t| [E2(t,a) + curl_a . A(t)]
// plus the near-field CSR rows (2x2 complex blocks) applied to x.  Partial
// sums: part [ns][R][4][npts] and partA [ns][R][6][nt], or (E) part
// [ns][R][18][nt], u1 (re, im) and u2 (re, im) of the corners 0, 1, 2, then A.
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

template <int L, int W, bool E>
__global__ void __launch_bounds__(GATHER_THREADS)
gather_kernel(int nv, int nt, int npts, int ns, int R, const int *__restrict__ vt_ptr,
              const int *__restrict__ vt_idx, const double *__restrict__ tgeo, const float *__restrict__ part,
              const float *__restrict__ partA, int use_far, const int *__restrict__ nr_ptr,
              const int *__restrict__ nr_col, const double2 *__restrict__ nr_val, int use_near, double escale,
              const __grid_constant__ VecPtrs x, const __grid_constant__ OutPtrs y) {
    static_assert(W == 1 || L == 32, "split groups are warps");
    __shared__ double2 red[W > 1 ? W : 1][2];
    const int lane = threadIdx.x % L;
    const int wg = W > 1 ? threadIdx.x / L % W : 0;  // split group
    const int v = blockIdx.x * (GATHER_THREADS / (L * W)) + threadIdx.x / (L * W);
    const int rr = blockIdx.y;
    const bool valid = v < nv;  // every lane takes part in the shuffles below
    double2 y1 = cd(0, 0), y2 = cd(0, 0);
    if (E && valid && use_far) {
        const int e0 = vt_ptr[v], items = 5 * (vt_ptr[v + 1] - e0);
        const size_t su = (size_t)R * 18 * nt;
        for (int it = lane; it < items; it += L) {
            const int e = it / 5, q = it - 5 * e;  // q: u1, u2, A.x, A.y, A.z (complex)
            const int ta = vt_idx[e0 + e], t = ta / 3, a = ta - 3 * t;
            const double *g = tgeo + 16 * (size_t)t;
            const float *P = part + ((size_t)rr * 18 + (q < 2 ? 4 * a + 2 * q : 8 + 2 * q)) * nt + t;
            float s[2] = {0.f, 0.f}, c[2] = {0.f, 0.f};
#pragma unroll 4
            for (int sp = wg; sp < ns; sp += W) {
                comp_add(s[0], c[0], P[sp * su]);
                comp_add(s[1], c[1], P[sp * su + nt]);
            }
            const double w = escale * g[0] * (q < 2 ? 1.0 : g[4 + 3 * a + (q - 2)]);
            const double2 val = cd(w * comp_value(s[0], c[0]), w * comp_value(s[1], c[1]));
            if (q == 0) y1 = cadd(y1, val);
            else y2 = cadd(y2, val);
        }
    } else if (valid && use_far) {
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
        // (a constant here: the same factor as an argument took the loads in flight
        // from 125 registers' worth to 96, and an apply at 150 vertices from 36.5 to
        // 42.5 us)
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
// The densities are linear on a triangle and the test functions its three hat
// functions, so what a pair of triangles contributes is, for any number of
// right-hand sides, four complex 3 x 3 matrices [test corner b][source corner a]:
//   S = sum_pq w_p w_q L_b(x_p) L_a(y_q) (G0 + rho G1),   K: (x - y).n_y (H0 + H1),
//   T: (H0 + H1)(x - y).n_x,   N: -(n_x.n_y)(k0^2 G0 + k1^2/rho G1)
// and the scalar W = sum_pq w_p w_q (G0 + G1/rho) of the curl term.  A pair of
// points costs its kernel values and their share of the matrices; a
// right-hand side costs 4 multiply-adds a point pair (144 a triangle pair,
// u1_b += S psi + K phi, u2_b += T psi + N phi) instead of the 16 of sums point
// by point.  The matrices come from sums M0, M1 of G0 and G1 (S, N and W are
// combinations of them, formed once per triangle pair), and the rule's two
// classes of three points with barycentric (alpha, beta, beta) give
// sum_q v_q L_a(y_q) = beta sum_q v_q + (alpha - beta) v_a per class.
//
// Source data (the points duplicated into pairs for the packed lanes):
//   sG [6nt][2]   (-y.x, -y.x, -y.y, -y.y), (-y.z, -y.z, 0, 0)   (static)
//   sD [R][5][nt] corner a: |s| (psi_a, phi_a); then c_s (three complex, 0, 0)
// Output (no atomics; gridDim.y splits the source range):
//   part [ns][R][18][nt]  u1 (re, im), u2 (re, im) of corners 0, 1, 2; then
//                         A = sum_s W c_s (x, y, z; re, im)
// ---------------------------------------------------------------------------
constexpr int FARM_TS = 32;  // source triangles per shared-memory tile
constexpr int FARM_MIN_BLOCKS = 2;

constexpr size_t farm_smem_bytes(int R) {
    return (size_t)FARM_TS * (12 * 16 + 5 * 16 * R + 16 + 16 + 32) + (size_t)FAR_THREADS * 72 * R;
}

// static source geometry of the multi kernel: coordinates (absolute, or
// offsets from the triangle centroid for the centred variant) negated and
// duplicated
__global__ void farm_geom_kernel(const float4 *__restrict__ pts, int npts, float4 *__restrict__ sG) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npts) return;
    const float4 p = pts[k];
    sG[2 * (size_t)k] = make_float4(-p.x, -p.x, -p.y, -p.y);
    sG[2 * (size_t)k + 1] = make_float4(-p.z, -p.z, 0.f, 0.f);
}

// corner densities of R right-hand sides times the triangle's area and the
// curl sources c_s, one thread per (source triangle, right-hand side)
__global__ void farm_prep_kernel(VecPtrs x, int R, int nv, int nt, const int *__restrict__ tris,
                                 const double *__restrict__ tgeo, float4 *__restrict__ sD) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (t >= nt || r >= R) return;
    const double2 *xr = x.p[r];
    const double *g = tgeo + 16 * (size_t)t;
    const double area = g[0];
    float4 *d = sD + 5 * (size_t)r * nt + t;
    double2 cv[3] = {cd(0, 0), cd(0, 0), cd(0, 0)};
    for (int a = 0; a < 3; ++a) {
        const int v = tris[3 * t + a];
        const double2 ps = cscale(xr[v], area), ph = cscale(xr[nv + v], area);
        d[a * (size_t)nt] = make_float4((float)ps.x, (float)ps.y, (float)ph.x, (float)ph.y);
        for (int j = 0; j < 3; ++j) cv[j] = cadd(cv[j], cscale(ph, g[4 + 3 * a + j]));
    }
    d[3 * (size_t)nt] = make_float4((float)cv[0].x, (float)cv[0].y, (float)cv[1].x, (float)cv[1].y);
    d[4 * (size_t)nt] = make_float4((float)cv[2].x, (float)cv[2].y, 0.f, 0.f);
}

// The matrices of one triangle pair, [re, im of S, N, T, K][b][a], and W; SCALED:
// all times kElemScale^2 (the gather divides by it).
struct ElemMat {
    float E[8][3][3];
    float wr, wi;
};

// mns = (-n_y, .), my0 = -y_0, dn: -(x - y).n_y = (X - y_0).mns + dn (centred:
// X.mns + dn); load(q, P0, P1) gives source point q as duplicated pairs; m1, k1i, dk1i as in far_vals (MULTI, ABSORB).
template <bool CENTRED, bool MULTI, bool ABSORB, bool SCALED, typename L>
__device__ __forceinline__ void elem_matrices(const f2 (&X)[3], const f2 (&Y)[3], const f2 (&Z)[3], const float4 &n4,
                                              float pdn, const float4 &mns, const float4 &my0, float dn, const L &load,
                                              const FarConst2 &c, const CenterPair &cp, f2 m1, f2 k1i, float dk1i,
                                              ElemMat &M) {
    // the rule's classes: weights times beta, and times alpha - beta
    constexpr double sc = SCALED ? kElemScale : 1.0;
    constexpr float WB1 = (float)(sc * kQw1 * kQa1), WB2 = (float)(sc * kQw2 * kQa2);
    constexpr float WG1 = (float)(sc * kQw1 * (1.0 - 3.0 * kQa1)), WG2 = (float)(sc * kQw2 * (1.0 - 3.0 * kQa2));
    const f2 wb = make_float2(WB1, WB2), wg = make_float2(WG1, WG2);
    f2 kb[3], kg[3];  // the test weights times -(x - y).n_y
    F3 {
        const f2 dx = CENTRED ? X[p] : add2(X[p], dup2(my0.x)), dy = CENTRED ? Y[p] : add2(Y[p], dup2(my0.y)),
                 dz = CENTRED ? Z[p] : add2(Z[p], dup2(my0.z));
        const f2 xnyn = fma2(dz, dup2(mns.z), fma2(dy, dup2(mns.y), fma2(dx, dup2(mns.x), dup2(dn))));
        kb[p] = mul2(wb, xnyn);
        kg[p] = mul2(wg, xnyn);
    }
    // first M0, M1 (G0, G1), T, K; class 0 stores, class 1 adds; bs: the beta parts
    float(&E)[8][3][3] = M.E;
    float bs[8][3];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        float4 P0, P1;
        load(q, P0, P1);
        FarVals v = far_vals<CENTRED, MULTI, ABSORB>(X, Y, Z, n4, pdn, P0, P1, c, cp, m1, k1i);
        F3 v.hp[p] = mul2(v.hp[p], v.ri2[p]);
        F3 v.hq[p] = mul2(v.hq[p], v.ri2[p]);
        const float wgq = q < 3 ? WG1 : WG2, wbq = q < 3 ? WB1 : WB2;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const f2(&u)[3] = i == 0 ? v.c0r : i == 1 ? v.s0r : i == 2 ? v.c1r : i == 3 ? v.s1r : (i & 1) ? v.hq : v.hp;
            const f2 sum = i < 6 ? mul2(wb, add2(add2(u[0], u[1]), u[2]))
                                 : fma2(kb[2], u[2], fma2(kb[1], u[1], mul2(kb[0], u[0])));
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const f2 tb = fma2(i < 6 ? wg : kg[b], u[b], sum);
                float t = tb.x + tb.y;
                if (i == 4 || i == 5) t *= v.dnxn.x;  // T: (y - x).n_x is the source point's alone
                E[i][b][q % 3] = q < 3 ? wgq * t : fmaf(wgq, t, E[i][b][q % 3]);
                bs[i][b] = q == 0 ? wbq * t : fmaf(wbq, t, bs[i][b]);
            }
        }
    }
    float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f;
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#pragma unroll
            for (int i = 0; i < 8; ++i) E[i][b][a] += bs[i][b];
            w0 += E[0][b][a];
            w1 += E[1][b][a];
            w2 += E[2][b][a];
            w3 += E[3][b][a];
        }
    M.wr = fmaf(c.irho.x, w2, w0);
    M.wi = fmaf(c.irho.x, w3, w1);
    const float nn = (n4.x * mns.x + n4.y * mns.y + n4.z * mns.z) * c.dk0.x;  // -(n_x.n_y) dks
    // M0, M1 -> S and N
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float g0 = E[0][b][a], g1 = E[1][b][a], g2 = E[2][b][a], g3 = E[3][b][a];
            E[0][b][a] = fmaf(c.rho.x, g2, g0);
            E[1][b][a] = fmaf(c.rho.x, g3, g1);
            float nr = fmaf(c.dk1.x, g2, g0), ni = fmaf(c.dk1.x, g3, g1);
            if (MULTI && ABSORB) {
                nr = fmaf(-dk1i, g3, nr);
                ni = fmaf(dk1i, g2, ni);
            }
            E[2][b][a] = nn * nr;
            E[3][b][a] = nn * ni;
        }
}

// u[b FAR_THREADS] (u1 re, im, u2 re, im) += the matrices on the corner densities
// d[a stride] (psi, phi).  REV: the pair seen from the source triangle.  S and N are symmetric;
// the normals change places and x - y its sign, so K becomes -T^T and T -K^T.
// PAIR: a pair's 12 products are summed before they meet the tile's sums, which
// then round once a pair: a third less error of an apply where coordinates and
// phases do not hide it (four spheres of 642 vertices 1.48e-7 -> 1.02e-7, bumpy
// ellipsoid of 3001 1.32 -> 0.89; far_kernel 1.34, 1.28) for 0.3 % of the time at
// R = 1.  Several vectors are as accurate as point-by-point sums without it, and it
// would take 1.8 % at R = 8.  The tile's sums are loaded after the products (before
// them they cost 11 registers and 8 % of the centred kernel's time).
template <bool REV, bool PAIR>
__device__ __forceinline__ void elem_apply(const ElemMat &M, const float4 *d, size_t stride, float4 *u) {
    float4 s[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) s[b] = PAIR ? make_float4(0.f, 0.f, 0.f, 0.f) : u[b * FAR_THREADS];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float4 da = d[a * stride];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int i = REV ? a : b, j = REV ? b : a;
            const float sr = M.E[0][i][j], si = M.E[1][i][j], nr = M.E[2][i][j], ni = M.E[3][i][j];
            const float tr = REV ? -M.E[6][i][j] : M.E[4][i][j], ti = REV ? -M.E[7][i][j] : M.E[5][i][j];
            const float kr = REV ? -M.E[4][i][j] : M.E[6][i][j], ki = REV ? -M.E[5][i][j] : M.E[7][i][j];
            s[b].x = fmaf(sr, da.x, fmaf(-si, da.y, fmaf(kr, da.z, fmaf(-ki, da.w, s[b].x))));
            s[b].y = fmaf(sr, da.y, fmaf(si, da.x, fmaf(kr, da.w, fmaf(ki, da.z, s[b].y))));
            s[b].z = fmaf(tr, da.x, fmaf(-ti, da.y, fmaf(nr, da.z, fmaf(-ni, da.w, s[b].z))));
            s[b].w = fmaf(tr, da.y, fmaf(ti, da.x, fmaf(nr, da.w, fmaf(ni, da.z, s[b].w))));
        }
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (PAIR) {
            const float4 v = u[b * FAR_THREADS];
            s[b] = make_float4(v.x + s[b].x, v.y + s[b].y, v.z + s[b].z, v.w + s[b].w);
        }
        u[b * FAR_THREADS] = s[b];
    }
}

// A += W c; with COMP the sums' rounding errors are carried along in *e4, *e2
template <bool COMP>
__device__ __forceinline__ void elem_curl(const ElemMat &M, float4 C0, float4 C1, float4 *a4, float2 *a2, float4 *e4, float2 *e2) {
    float4 A = *a4;
    float2 Z = *a2;
    if (COMP) {
        float4 E = *e4;
        float2 F = *e2;
        comp_add_fast(A.x, E.x, fmaf(M.wr, C0.x, -M.wi * C0.y));
        comp_add_fast(A.y, E.y, fmaf(M.wr, C0.y, M.wi * C0.x));
        comp_add_fast(A.z, E.z, fmaf(M.wr, C0.z, -M.wi * C0.w));
        comp_add_fast(A.w, E.w, fmaf(M.wr, C0.w, M.wi * C0.z));
        comp_add_fast(Z.x, F.x, fmaf(M.wr, C1.x, -M.wi * C1.y));
        comp_add_fast(Z.y, F.y, fmaf(M.wr, C1.y, M.wi * C1.x));
        *e4 = E;
        *e2 = F;
    } else {
        A.x = fmaf(M.wr, C0.x, fmaf(-M.wi, C0.y, A.x));
        A.y = fmaf(M.wr, C0.y, fmaf(M.wi, C0.x, A.y));
        A.z = fmaf(M.wr, C0.z, fmaf(-M.wi, C0.w, A.z));
        A.w = fmaf(M.wr, C0.w, fmaf(M.wi, C0.z, A.w));
        Z.x = fmaf(M.wr, C1.x, fmaf(-M.wi, C1.y, Z.x));
        Z.y = fmaf(M.wr, C1.y, fmaf(M.wi, C1.x, Z.y));
    }
    *a4 = A;
    *a2 = Z;
}

// One thread per test triangle, on far_kernel's grid (blocks of block_tris test
// triangles, the warps of a block sharing its source tiles when that is less
// than FAR_THREADS).  The matrices stay in registers (72, and 24 sums; 255
// registers, two blocks per SM); the right-hand sides' sums, 18 floats each,
// are in shared memory, a thread's own column, so R costs no registers and one
// kernel takes every R up to FARM_MAX_R.  After each tile they move to part:
// short sums keep their rounding errors (1.2 to 2 times less than without on
// 3000 to 5000 vertices) for 2 % of the time, the old values of an entry's 18
// being loaded together.
// Bound by the FP32 pipe: an apply at 10242 vertices is 27.1 ms of kernel
// values and matrices and 2.7 ms a right-hand side (R 8: 49.0 ms), where
// point-by-point sums took 24 + 9.9 (102.7).  Tensor cores do not help: TF32
// pieces with the kernel values as an operand took 64.7 ms at R 2 and 80.8 at
// 8, mma.sync and packed FMA not overlapping.
template <bool CENTRED>
__global__ void __launch_bounds__(FAR_THREADS, FARM_MIN_BLOCKS)
farm_kernel(const float4 *__restrict__ pt, const float4 *__restrict__ cen, const float4 *__restrict__ tn,
            const int4 *__restrict__ tv, const float4 *__restrict__ sG, const float4 *__restrict__ sD, int R,
            int nt, int tris_per_split, int block_tris, FarConst2 c, float4 kff, float *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char farm_smem[];
    float4 *acc4 = reinterpret_cast<float4 *>(farm_smem);                            // [R][4][threads]
    float2 *acc2 = reinterpret_cast<float2 *>(acc4 + (size_t)R * 4 * FAR_THREADS);   // [R][threads]
    float4 *shG = reinterpret_cast<float4 *>(acc2 + (size_t)R * FAR_THREADS);        // [TS][6][2]
    float4 *shD = shG + FARM_TS * 12;                                                // [R][5][TS]
    float4 *shN = shD + FARM_TS * 5 * R;                                             // [TS] (-n, n.P0)
    int4 *shV = reinterpret_cast<int4 *>(shN + FARM_TS);                             // [TS]
    float4 *shCen = reinterpret_cast<float4 *>(shV + FARM_TS);                       // [TS][2] (centred)

    const int tx = threadIdx.x % block_tris, grp = threadIdx.x / block_tris, ngrp = FAR_THREADS / block_tris;
    const int j = blockIdx.x * block_tris + tx;
    const int split = blockIdx.y;
    const int s_begin = min(nt, split * tris_per_split);
    const int s_end = min(nt, s_begin + tris_per_split);
    const int tau = j < nt ? j : 0;
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
    float4 cth = make_float4(0.f, 0.f, 0.f, 0.f), ctl = cth;
    if (CENTRED) {
        cth = cen[2 * tau];
        ctl = cen[2 * tau + 1];
    }
    float *const out = part + (size_t)split * R * 18 * nt;
    for (int i = threadIdx.x; i < R * 18 * FAR_THREADS; i += FAR_THREADS) reinterpret_cast<float *>(acc4)[i] = 0.f;

    for (int t0 = s_begin; t0 < s_end; t0 += FARM_TS) {
        const int cnt = min(FARM_TS, s_end - t0);
        for (int i = threadIdx.x; i < cnt * 12; i += FAR_THREADS) shG[i] = sG[12 * (size_t)t0 + i];
#pragma unroll 1  // an unrolled copy's addresses would stay in registers the pair loop needs
        for (int i = threadIdx.x; i < 5 * R * FARM_TS; i += FAR_THREADS) {
            const int si = i % FARM_TS, k = i / FARM_TS;
            if (si < cnt) shD[i] = sD[(size_t)k * nt + t0 + si];
        }
        for (int i = threadIdx.x; i < cnt; i += FAR_THREADS) {
            const float4 ns = tn[t0 + i];
            shN[i] = make_float4(-ns.x, -ns.y, -ns.z, ns.w);
            shV[i] = tv[t0 + i];
        }
        if (CENTRED)
            for (int i = threadIdx.x; i < 2 * cnt; i += FAR_THREADS) shCen[i] = cen[2 * (size_t)t0 + i];
        __syncthreads();

        for (int s = grp; s < cnt; s += ngrp) {
            const int4 vs = shV[s];
            const bool touch = (vs.x == vt.x) | (vs.x == vt.y) | (vs.x == vt.z) |
                               (vs.y == vt.x) | (vs.y == vt.y) | (vs.y == vt.z) |
                               (vs.z == vt.x) | (vs.z == vt.y) | (vs.z == vt.z);
            if (touch) continue;
            CenterPair cp;
            float pdn = __int_as_float(vt.w);
            const float4 mns = shN[s];
            const float4 g0 = shG[12 * s], g1 = shG[12 * s + 1], my0 = make_float4(g0.x, g0.z, g1.x, 0.f);
            float dn = __int_as_float(vs.w);  // n_y.(P0 - y_0), see far_geom_kernel
            if (CENTRED) {
                cp = center_pair(cth, ctl, shCen[2 * s], shCen[2 * s + 1], kff.x, kff.y, kff.z, kff.w);
                pdn = fmaf(cp.Dx.x, n4.x, fmaf(cp.Dy.x, n4.y, cp.Dz.x * n4.z)) +
                      fmaf(cp.lx, n4.x, fmaf(cp.ly, n4.y, cp.lz * n4.z));
                dn = cp.Dx.x * mns.x + cp.Dy.x * mns.y + cp.Dz.x * mns.z;
            }
            ElemMat M;
            elem_matrices<CENTRED, false, false, false>(
                X, Y, Z, n4, pdn, mns, my0, dn, [&](int q, float4 &P0, float4 &P1) {
                    P0 = shG[12 * s + 2 * q];
                    P1 = shG[12 * s + 2 * q + 1];
                },
                c, cp, dup2(1.f), dup2(0.f), 0.f, M);
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const float4 *D = shD + 5 * r * FARM_TS + s;
                float4 *o4 = acc4 + (size_t)r * 4 * FAR_THREADS + threadIdx.x;
                elem_apply<false, false>(M, D, FARM_TS, o4);
                elem_curl<false>(M, D[3 * FARM_TS], D[4 * FARM_TS], o4 + 3 * FAR_THREADS,
                                 acc2 + (size_t)r * FAR_THREADS + threadIdx.x, nullptr, nullptr);
            }
        }
        __syncthreads();
        // the tile's sums of all groups to part (the first tile stores, later
        // ones add; the same thread has the same entries each time)
        const bool first = t0 == s_begin;
        for (int i = threadIdx.x; i < R * block_tris; i += FAR_THREADS) {
            const int r = i / block_tris, jj = i - r * block_tris, jt = blockIdx.x * block_tris + jj;
            float *o = out + (size_t)r * 18 * nt + jt;
            float v[18];
#pragma unroll
            for (int e = 0; e < 18; ++e) v[e] = first || jt >= nt ? 0.f : o[(size_t)e * nt];
            for (int g = 0; g < ngrp; ++g) {
                const int th = g * block_tris + jj;
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    float4 *a = acc4 + ((size_t)r * 4 + f) * FAR_THREADS + th;
                    const float4 w = *a;
                    v[4 * f] += w.x;
                    v[4 * f + 1] += w.y;
                    v[4 * f + 2] += w.z;
                    v[4 * f + 3] += w.w;
                    *a = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                float2 *a = acc2 + (size_t)r * FAR_THREADS + th;
                v[16] += a->x;
                v[17] += a->y;
                *a = make_float2(0.f, 0.f);
            }
            if (jt < nt)
#pragma unroll
                for (int e = 0; e < 18; ++e) o[(size_t)e * nt] = v[e];
        }
        __syncthreads();
    }
    if (s_begin >= s_end)  // empty split: zero sums
        for (int i = threadIdx.x; i < R * 18 * block_tris; i += FAR_THREADS) {
            const int k = i / block_tris, jt = blockIdx.x * block_tris + i - k * block_tris;
            if (jt < nt) out[(size_t)k * nt + jt] = 0.f;
        }
}
// ---------------------------------------------------------------------------
// The same with each pair of triangles evaluated once for both directions
// (elem_apply<true>): the kernel values and matrices, most of the work of few
// right-hand sides, are halved.  The triangles are cut into N groups of 128; a
// block takes test group I (a thread per triangle) against groups I + d mod N,
// d = 0 (its own, every ordered pair, test side only) and d = 1 .. N/2 (for
// even N the last only from I < N/2), which meets every two groups once.
//
// A source group is staged 32 triangles at a time.  At step i lane l of a warp
// takes source triangle (i + l) mod 32, so the lanes' source-side sums, in
// shared memory, a set per warp, never meet; after the 32 steps the four
// warps' sums are added and leave for the slot of d (source side), the test
// side's for the block's split.  A launch covers nsrc values of d, so no two
// blocks write one entry; further launches add to it.  Everything is added in
// a fixed order.
//   part [ntst + nsrc][R][18][nt]  as farm_kernel's
// One vector's curl sums carry their rounding errors along, its pairs are summed
// first and its weights scaled (COMP; several vectors are as accurate as
// point-by-point sums without).  Bound by the FP32
// pipe at 8 warps per SM: an apply at 10242 vertices 17.4 ms (far_kernel 25.9),
// 20000 vertices centred 79.6 (124), four objects of 642 vertices 1.71 (2.19);
// R = 2: 20.0, 3: 23.1, 4: 28.4, 5: 32.0 (farm_kernel 32.5, 35.3, 38.0, 40.6).
// ---------------------------------------------------------------------------
constexpr int SYM_U = 32;  // source triangles per tile (one step each per lane)
constexpr size_t sym_smem_bytes(int R, bool centred) {
    return (size_t)R * (2 * 72 * FAR_THREADS + 80 * SYM_U) + (R == 1 ? 2 * 24 * FAR_THREADS : 0) +
           (size_t)SYM_U * (96 + 16 + 16 + (centred ? 32 : 0) + 16);
}

template <bool CENTRED, bool MULTI, bool ABSORB, bool COMP>
__global__ void __launch_bounds__(FAR_THREADS, FARM_MIN_BLOCKS)
sym_kernel(const float4 *__restrict__ pt, const float4 *__restrict__ cen, const float4 *__restrict__ tn,
           const int4 *__restrict__ tv, const float4 *__restrict__ sD, int R, int nt, int d_first, int d_count,
           int units_per_split, int ntst, int accumulate, FarConst2 c0, float4 kff0, const int *__restrict__ tcomp,
           const FarObj *__restrict__ fobj, float *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char sym_smem[];
    float4 *acc4 = reinterpret_cast<float4 *>(sym_smem);           // [R][4][threads] test side
    float4 *src4 = acc4 + (size_t)R * 4 * FAR_THREADS;             // [R][4][warp][32] source side
    float2 *acc2 = reinterpret_cast<float2 *>(src4 + (size_t)R * 4 * FAR_THREADS);
    float2 *src2 = acc2 + (size_t)R * FAR_THREADS;
    // errors of the curl sums (COMP): [test, source][threads]
    float4 *err4 = reinterpret_cast<float4 *>(src2 + (size_t)R * FAR_THREADS);
    float2 *err2 = reinterpret_cast<float2 *>(err4 + (COMP ? 2 * FAR_THREADS : 0));
    float4 *shP = reinterpret_cast<float4 *>(err2 + (COMP ? 2 * FAR_THREADS : 0));  // [6][32] -y
    float4 *shD = shP + 6 * SYM_U;                                 // [R][5][32]
    float4 *shN = shD + (size_t)5 * R * SYM_U;                     // [32] -n
    int4 *shV = reinterpret_cast<int4 *>(shN + SYM_U);             // [32]
    int *shComp = reinterpret_cast<int *>(shV + SYM_U);            // [32] (16 bytes each reserved)
    float4 *shCen = reinterpret_cast<float4 *>(shV + 2 * SYM_U);   // [2][32] (centred)

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = (nt + FAR_THREADS - 1) / FAR_THREADS, I = blockIdx.x;
    const int j = I * FAR_THREADS + threadIdx.x;
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
    FarConst2 c = c0;
    float4 kff = kff0;
    int ct = 0;
    float sgn = 1.f, dk1i = 0.f;
    f2 k1i = make_float2(0.f, 0.f);
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
        dk1i = o.dk1i;
    }
    float4 cth = make_float4(0.f, 0.f, 0.f, 0.f), ctl = cth;
    if (CENTRED) {
        cth = cen[2 * tau];
        ctl = cen[2 * tau + 1];
    }
    // both sides' sums: acc4 to err2 are contiguous
    for (int i = threadIdx.x; i < (R * 36 + (COMP ? 12 : 0)) * FAR_THREADS; i += FAR_THREADS) reinterpret_cast<float *>(acc4)[i] = 0.f;

    float *const tout = part + (size_t)blockIdx.y * R * 18 * nt + j;
    const int u0 = blockIdx.y * units_per_split, u1 = min(4 * d_count, u0 + units_per_split);
    bool stored = accumulate != 0, any = false;
    for (int u = u0; u < u1; ++u) {
        const int d = d_first + u / 4;
        if (2 * d == N && I >= d) break;  // the other group of the pair has it
        const int J = I + d < N ? I + d : I + d - N;
        const int t0 = J * FAR_THREADS + (u % 4) * SYM_U, cnt = min(SYM_U, nt - t0);
        if (cnt <= 0) continue;
        const bool both = d != 0;
        __syncthreads();
        for (int i = threadIdx.x; i < 6 * SYM_U; i += FAR_THREADS) {
            const int si = i / 6, q = i - 6 * si;
            if (si < cnt) {
                const float4 y = pt[6 * (size_t)t0 + i];
                shP[q * SYM_U + si] = make_float4(-y.x, -y.y, -y.z, 0.f);
            }
        }
        for (int i = threadIdx.x; i < 5 * R * SYM_U; i += FAR_THREADS) {
            const int si = i % SYM_U, k = i / SYM_U;
            if (si < cnt) shD[i] = sD[(size_t)k * nt + t0 + si];
        }
        if (threadIdx.x < cnt) {
            const float4 ns = tn[t0 + threadIdx.x];
            shN[threadIdx.x] = make_float4(-ns.x, -ns.y, -ns.z, ns.w);
            shV[threadIdx.x] = tv[t0 + threadIdx.x];
            if (MULTI) shComp[threadIdx.x] = tcomp[t0 + threadIdx.x];
            if (CENTRED) {
                shCen[threadIdx.x] = cen[2 * (size_t)(t0 + threadIdx.x)];
                shCen[SYM_U + threadIdx.x] = cen[2 * (size_t)(t0 + threadIdx.x) + 1];
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int st = 0; st < SYM_U; ++st) {
            const int s = (st + lane) & (SYM_U - 1);
            const int4 vs = shV[s];
            const bool touch = (vs.x == vt.x) | (vs.x == vt.y) | (vs.x == vt.z) |
                               (vs.y == vt.x) | (vs.y == vt.y) | (vs.y == vt.z) |
                               (vs.z == vt.x) | (vs.z == vt.y) | (vs.z == vt.z);
            if (active && s < cnt && !touch) {
                CenterPair cp;
                float pdn = __int_as_float(vt.w);
                const float4 mns = shN[s];
                float dn;
                if (CENTRED) {
                    cp = center_pair(cth, ctl, shCen[s], shCen[SYM_U + s], kff.x, kff.y, kff.z, kff.w);
                    pdn = fmaf(cp.Dx.x, n4.x, fmaf(cp.Dy.x, n4.y, cp.Dz.x * n4.z)) +
                          fmaf(cp.lx, n4.x, fmaf(cp.ly, n4.y, cp.lz * n4.z));
                    dn = fmaf(cp.Dx.x, mns.x, fmaf(cp.Dy.x, mns.y, cp.Dz.x * mns.z)) +
                         fmaf(cp.lx, mns.x, fmaf(cp.ly, mns.y, cp.lz * mns.z));
                } else {
                    dn = __int_as_float(vs.w);  // n_y.(P0 - y_0), see far_geom_kernel
                }
                const f2 m1 = dup2(MULTI ? (shComp[s] != ct ? 0.f : sgn) : 1.f);
                ElemMat M;
                elem_matrices<CENTRED, MULTI, ABSORB, COMP>(
                    X, Y, Z, n4, pdn, mns, shP[s], dn, [&](int q, float4 &P0, float4 &P1) {
                        const float4 y = shP[q * SYM_U + s];
                        P0 = make_float4(y.x, y.x, y.y, y.y);
                        P1 = make_float4(y.z, y.z, 0.f, 0.f);
                    },
                    c, cp, m1, k1i, dk1i, M);
#pragma unroll 1
                for (int r = 0; r < R; ++r) {
                    const float4 *D = shD + 5 * r * SYM_U + s;
                    float4 *o4 = acc4 + (size_t)r * 4 * FAR_THREADS + threadIdx.x;
                    float2 *o2 = acc2 + (size_t)r * FAR_THREADS + threadIdx.x;
                    elem_apply<false, COMP>(M, D, SYM_U, o4);
                    elem_curl<COMP>(M, D[3 * SYM_U], D[4 * SYM_U], o4 + 3 * FAR_THREADS, o2, err4 + threadIdx.x, err2 + threadIdx.x);
                    if (both) {
                        const float4 *T = sD + 5 * (size_t)r * nt + tau;
                        o4 = src4 + (size_t)r * 4 * FAR_THREADS + warp * 32 + s;
                        o2 = src2 + (size_t)r * FAR_THREADS + warp * 32 + s;
                        elem_apply<true, COMP>(M, T, nt, o4);
                        elem_curl<COMP>(M, T[3 * (size_t)nt], T[4 * (size_t)nt], o4 + 3 * FAR_THREADS, o2,
                                        err4 + FAR_THREADS + warp * 32 + s, err2 + FAR_THREADS + warp * 32 + s);
                    }
                }
            }
            __syncwarp();
        }
        __syncthreads();
        // test side: the thread's own sums (the first tile stores, later ones
        // add; compensated curl sums stay until the last)
        constexpr int TE = COMP ? 12 : 18;
        for (int r = 0; r < R; ++r) {
            float *o = tout + (size_t)r * 18 * nt;
            float v[TE];
#pragma unroll
            for (int e = 0; e < TE; ++e) v[e] = stored && active ? o[(size_t)e * nt] : 0.f;
#pragma unroll
            for (int f = 0; f < TE / 4; ++f) {
                float4 *a = acc4 + ((size_t)r * 4 + f) * FAR_THREADS + threadIdx.x;
                const float4 w = *a;
                v[4 * f] += w.x;
                v[4 * f + 1] += w.y;
                v[4 * f + 2] += w.z;
                v[4 * f + 3] += w.w;
                *a = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if (!COMP) {
                float2 *a = acc2 + (size_t)r * FAR_THREADS + threadIdx.x;
                v[TE - 2] += a->x;
                v[TE - 1] += a->y;
                *a = make_float2(0.f, 0.f);
            }
            if (active)
#pragma unroll
                for (int e = 0; e < TE; ++e) o[(size_t)e * nt] = v[e];
        }
        stored = any = true;
        // source side: the four warps' sums, in their order, to the slot of d
        if (both) {
            const int slot = ntst + (d - max(d_first, 1));
#pragma unroll 1
            for (int i = threadIdx.x; i < R * 5 * SYM_U; i += FAR_THREADS) {
                const int si = i % SYM_U, k = i / SYM_U, r = k / 5, f = k - 5 * r;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f), ve = v;
                for (int w = 0; w < FAR_THREADS / 32; ++w) {
                    if (f < 4) {
                        float4 *a = src4 + ((size_t)r * 4 + f) * FAR_THREADS + w * 32 + si;
                        comp_add(v.x, ve.x, a->x);
                        comp_add(v.y, ve.y, a->y);
                        comp_add(v.z, ve.z, a->z);
                        comp_add(v.w, ve.w, a->w);
                        *a = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (COMP && f == 3) {
                            a = err4 + FAR_THREADS + w * 32 + si;
                            ve.x += a->x;
                            ve.y += a->y;
                            ve.z += a->z;
                            ve.w += a->w;
                            *a = make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    } else {
                        float2 *a = src2 + (size_t)r * FAR_THREADS + w * 32 + si;
                        comp_add(v.x, ve.x, a->x);
                        comp_add(v.y, ve.y, a->y);
                        *a = make_float2(0.f, 0.f);
                        if (COMP) {
                            a = err2 + FAR_THREADS + w * 32 + si;
                            ve.x += a->x;
                            ve.y += a->y;
                            *a = make_float2(0.f, 0.f);
                        }
                    }
                }
                if (si < cnt) {
                    float *o = part + (((size_t)slot * R + r) * 18 + 4 * f) * nt + t0 + si;
                    const float w4[4] = {v.x + ve.x, v.y + ve.y, v.z + ve.z, v.w + ve.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (f < 4 || e < 2) o[(size_t)e * nt] = accumulate ? o[(size_t)e * nt] + w4[e] : w4[e];
                }
            }
        }
    }
    if (!stored && active)  // no tile: zero sums
        for (int i = 0; i < R * 18; ++i) tout[(size_t)i * nt] = 0.f;
    // (without a tile the sums have not met a barrier since they were cleared)
    if (COMP && any && active) {
        const float4 A = acc4[3 * FAR_THREADS + threadIdx.x], Ae = err4[threadIdx.x];
        const float2 Az = acc2[threadIdx.x], Aze = err2[threadIdx.x];
        const float v[6] = {A.x + Ae.x, A.y + Ae.y, A.z + Ae.z, A.w + Ae.w, Az.x + Aze.x, Az.y + Aze.y};
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            float *o = tout + (size_t)(12 + e) * nt;
            *o = accumulate ? *o + v[e] : v[e];
        }
    }
}
#undef F3

}  // namespace

// Work split of sym_kernel: cuts the N / 2 offsets into launches of nsrc and a
// launch's 32-triangle tiles over ntst blocks per test group, such that the
// launches' waves of blocks, times the tiles of a block, are fewest, within
// max_slots partial sums.
static PerDeviceOnce g_sym_once;

static FarSymPlan sym_plan(int nt, int sms, int max_slots) {
    const int N = (nt + FAR_THREADS - 1) / FAR_THREADS, half = N / 2;
    const long long slots = (long long)sms * FARM_MIN_BLOCKS;
    FarSymPlan best;
    double cost = -1.0;
    for (int nsrc = half ? 1 : 0; nsrc <= std::min(half, max_slots - 1); ++nsrc) {
        const int units = 4 * (nsrc + 1), launches = nsrc ? (half + nsrc - 1) / nsrc : 1;
        for (int ups = 1; ups <= units; ++ups) {
            const int ntst = (units + ups - 1) / ups;
            if (ntst + nsrc > max_slots) continue;
            const double c = launches * ((double)((N * (long long)ntst + slots - 1) / slots) * ups + 1.0);
            if (cost < 0.0 || c < cost) {
                cost = c;
                best.nsrc = nsrc;
                best.ntst = ntst;
                best.ups = ups;
            }
        }
    }
    return best;
}

// partial sums times right-hand sides of the several-right-hand-side launches
static size_t farm_slots(const osrc_problem *pb) {
    const int s = pb->nsplit * FARM_MAX_R;
    return pb->far_sym && !pb->mesh->ctx->budget ? std::max(s, SYM_MULTI_SLOTS) : std::max(s, 2 * FARM_MAX_R);
}

// every buffer of the one-vector apply's path is there
static bool far_workspace_made(const osrc_problem *pb) {
    return pb->far_sym ? pb->d_sD.p && pb->d_part.p
                       : pb->d_sP.p && pb->d_sP5.p && pb->d_sC.p && pb->d_part.p && pb->d_partA1.p;
}

int far_workspace(osrc_problem *pb) {
    osrc_ctx *ctx = pb->mesh->ctx;
    const size_t nt = pb->nt;
    if (pb->far_sym) {
        int s = pb->d_sD.alloc(ctx, 5 * nt);
        if (!s) s = pb->d_part.alloc(ctx, (size_t)(pb->sym[1].ntst + pb->sym[1].nsrc) * 18 * nt);
        if (s != OSRC_OUT_OF_MEMORY) return s;
        pb->d_sD.release();  // no room: the one-sided kernels' buffers may fit
        pb->d_part.release();
        pb->far_sym = false;
    }
    OSRC_TRY(pb->d_sP.alloc(ctx, 24 * nt));
    OSRC_TRY(pb->d_sP5.alloc(ctx, 6 * nt));
    OSRC_TRY(pb->d_sC.alloc(ctx, 2 * nt));
    OSRC_TRY(pb->d_part.alloc(ctx, (size_t)pb->nsplit * 4 * pb->npts));
    return pb->d_partA1.alloc(ctx, (size_t)pb->nsplit * 6 * nt);
}

int far_setup_geometry(osrc_problem *pb, cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt;
    OSRC_TRY(pb->d_pt.alloc(m->ctx, 6 * (size_t)nt));
    OSRC_TRY(pb->d_poff.alloc(m->ctx, 6 * (size_t)nt));
    OSRC_TRY(pb->d_cen.alloc(m->ctx, 2 * (size_t)nt));
    OSRC_TRY(pb->d_tn.alloc(m->ctx, nt));
    OSRC_TRY(pb->d_tv.alloc(m->ctx, nt));
    OSRC_TRY(pb->d_tgeo.alloc(m->ctx, 16 * (size_t)nt));
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
    int dev = m->ctx->device;
    int &sms = pb->sms;
    OSRC_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    pb->far_tris = nt < FAR_TRIS32_NT ? 32 : nt < FAR_TRIS64_NT ? 64 : FAR_THREADS;
    const int slots = sms * FAR_MIN_BLOCKS;  // farm_kernel runs on the same grid
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
    pb->far_sym = nt >= SYM_MIN_NT;
    static_assert(SYM_MAX_R < sizeof(pb->sym) / sizeof(pb->sym[0]), "a plan for every R");
    // on a context with a memory budget no more than far_kernel's buffers
    const int one = m->ctx->budget ? std::max(2, std::min(SYM_MAX_SLOTS, (30 * ns + 96) / 18)) : SYM_MAX_SLOTS;
    if (pb->far_sym)
        for (int r = 1; r <= SYM_MAX_R; ++r)
            pb->sym[r] = sym_plan(nt, sms, r == 1 ? one : (int)farm_slots(pb) / r);
    OSRC_TRY(per_device_once(g_sym_once, [](int) {
        const int sp = (int)sym_smem_bytes(SYM_MAX_R, false), sc = (int)sym_smem_bytes(SYM_MAX_R, true);
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        OSRC_CK(cudaFuncSetAttribute(sym_kernel<false, false, false, false>, attr, sp));
        OSRC_CK(cudaFuncSetAttribute(sym_kernel<true, false, false, false>, attr, sc));
        return OSRC_OK;
    }));
    return far_workspace(pb);
}

int far_prof_collect(osrc_problem *pb);

static FarConst2 far_consts(const osrc_problem *pb, float4 &kff) {
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
    kff = make_float4(q0h, (float)(q0 - (double)q0h), q1h, (float)(q1 - (double)q1h));
    return c;
}

// sD from the vectors and the launches of sym_kernel over all offsets
static int sym_launch(osrc_problem *pb, const VecPtrs &xp, int R, const FarSymPlan &pl, float4 *sD, float *part,
                      cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt, N = (nt + FAR_THREADS - 1) / FAR_THREADS, half = N / 2;
    farm_prep_kernel<<<dim3((nt + 127) / 128, R), 128, 0, st>>>(xp, R, pb->nv, nt, m->d_tris.p, pb->d_tgeo.p, sD);
    pb->launches++;
    float4 kff;
    const FarConst2 c = far_consts(pb, kff);
    const size_t smem = sym_smem_bytes(R, pb->far_reduce);
    const float4 *pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
    if (pb->prof_on) {
        OSRC_TRY(far_prof_collect(pb));
        OSRC_CK(cudaEventRecord(pb->prof_ev[0], st));
    }
    // even N in one launch: the lower half of the groups has no sums of the last offset
    if (half && 2 * half == N && pl.nsrc >= half)
        OSRC_CK(cudaMemsetAsync(part + (size_t)(pl.ntst + half - 1) * R * 18 * nt, 0, (size_t)R * 18 * nt * sizeof(float), st));
    for (int d = 0; d <= half; d += d ? pl.nsrc : pl.nsrc + 1) {
        const int count = d ? std::min(pl.nsrc, half + 1 - d) : pl.nsrc + 1;
        const dim3 grid(N, (4 * count + pl.ups - 1) / pl.ups);
#define OSRC_SYM_LAUNCH(C, M, A, E)                                                                                \
    sym_kernel<C, M, A, E><<<grid, FAR_THREADS, smem, st>>>(pts, pb->d_cen.p, pb->d_tn.p, pb->d_tv.p, sD, R, \
                                                            nt, d, count, pl.ups, pl.ntst, d ? 1 : 0, c, kff,       \
                                                            m->d_tcomp.p, pb->d_fobj.p, part)
        if (pb->far_reduce && pb->far_obj && pb->absorb) OSRC_SYM_LAUNCH(true, true, true, true);
        else if (pb->far_reduce && pb->far_obj) OSRC_SYM_LAUNCH(true, true, false, true);
        else if (pb->far_reduce && R == 1) OSRC_SYM_LAUNCH(true, false, false, true);
        else if (pb->far_reduce) OSRC_SYM_LAUNCH(true, false, false, false);
        else if (pb->far_obj && pb->absorb) OSRC_SYM_LAUNCH(false, true, true, true);
        else if (pb->far_obj) OSRC_SYM_LAUNCH(false, true, false, true);
        else if (R == 1) OSRC_SYM_LAUNCH(false, false, false, true);
        else OSRC_SYM_LAUNCH(false, false, false, false);
#undef OSRC_SYM_LAUNCH
        pb->launches++;
        OSRC_CK(cudaGetLastError());
    }
    if (pb->prof_on) {
        OSRC_CK(cudaEventRecord(pb->prof_ev[1], st));
        pb->prof_pending = pb->prof_sym_pending = true;
        pb->prof_rhs_pending = R;
    }
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
    pb->prof_sym += pb->prof_sym_pending;
    pb->prof_rhs_pending = 1;
    pb->prof_sym_pending = pb->prof_pending = false;
    return OSRC_OK;
}

// es: scale of the element matrices' weights (with part alone)
static int gather_launch(osrc_problem *pb, int ns, int R, const float *part, const float *partA, int use_far,
                         int use_near, double es, const VecPtrs &x, const OutPtrs &y, cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const double escale = 0.079577471545947667884 / (es * es);  // 1 / (4 pi)
    const int nv = pb->nv;
    const int per = nv <= GATHER_BLOCK_NV ? 1 : nv <= GATHER_WARP_NV ? GATHER_THREADS / 32 : GATHER_THREADS / 8;
    const dim3 grid((nv + per - 1) / per, R);
#define OSRC_GATHER_LAUNCH(LL, WW)                                                                             \
    (partA ? gather_kernel<LL, WW, false> : gather_kernel<LL, WW, true>)<<<grid, GATHER_THREADS, 0, st>>>(nv, pb->nt, pb->npts, ns, R, m->d_vt_ptr.p, m->d_vt_idx.p, \
                                                       pb->d_tgeo.p, part, partA, use_far, pb->d_nr_ptr.p,       \
                                                       pb->d_nr_col.p, pb->d_nr_val.p, use_near, escale, x, y)
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
    VecPtrs xp{};
    OutPtrs yp{};
    xp.p[0] = x;
    yp.p[0] = y;
    if (use_far && !far_workspace_made(pb)) OSRC_TRY(far_workspace(pb));  // a clone made without it
    if (use_far && pb->far_sym) {
        OSRC_TRY(sym_launch(pb, xp, 1, pb->sym[1], pb->d_sD.p, pb->d_part.p, st));
        return gather_launch(pb, pb->sym[1].ntst + pb->sym[1].nsrc, 1, pb->d_part.p, nullptr, use_far, use_near, kElemScale,
                             xp, yp, st);
    }
    if (use_far) {
        const float4 *src_pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
        far_prep_kernel<<<(npts + 127) / 128, 128, 0, st>>>(x, nv, nt, m->d_tris.p, src_pts,
                                                          pb->d_tgeo.p, pb->d_sP.p, pb->d_sP5.p,
                                                          pb->d_sC.p);
        pb->launches++;
        float4 kff;
        const FarConst2 c = far_consts(pb, kff);
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
    return gather_launch(pb, pb->nsplit, 1, pb->d_part.p, pb->d_partA1.p, use_far, use_near, 1.0, xp, yp, st);
}

// ---------------------------------------------------------------------------
// multi-right-hand-side apply: y_r = B_far x_r (+ near) for r < nrhs, in
// launches of up to FARM_MAX_R right-hand sides (a last single vector takes
// the one-right-hand-side kernel)
// ---------------------------------------------------------------------------
static PerDeviceOnce g_farm_once;

static int farm_prepare(osrc_problem *pb, cudaStream_t st) {
    OSRC_TRY(per_device_once(g_farm_once, [](int) {
        const int smem = (int)farm_smem_bytes(FARM_MAX_R);
        OSRC_CK(cudaFuncSetAttribute(farm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        OSRC_CK(cudaFuncSetAttribute(farm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        return OSRC_OK;
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
    // buffers of its own: one-vector applies, also captured ones and those on
    // another stream, keep d_sD and d_part whatever happens here
    if (!pb->d_sDm.p) OSRC_TRY(pb->d_sDm.alloc(ctx, 5 * (size_t)nt * FARM_MAX_R));
    if (!pb->d_partm.p) OSRC_TRY(pb->d_partm.alloc(ctx, farm_slots(pb) * 18 * nt));
    return OSRC_OK;
}

static int farm_launch(osrc_problem *pb, const double2 *const *xs, double2 *const *ys, int R, int part,
                       cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt, nv = pb->nv;
    const int use_far = (part & OSRC_PART_FAR) ? 1 : 0;
    const int use_near = (part & OSRC_PART_NEAR) ? 1 : 0;
    VecPtrs xp{};
    OutPtrs yp{};
    for (int r = 0; r < R; ++r) {
        xp.p[r] = xs[r];
        yp.p[r] = ys[r];
    }
    const int ns = pb->nsplit;
    if (use_far && pb->far_sym && R <= SYM_MAX_R) {
        const FarSymPlan pl = pb->sym[R];
        OSRC_TRY(sym_launch(pb, xp, R, pl, pb->d_sDm.p, pb->d_partm.p, st));
        return gather_launch(pb, pl.ntst + pl.nsrc, R, pb->d_partm.p, nullptr, use_far, use_near, 1.0, xp, yp, st);
    }
    if (use_far) {
        farm_prep_kernel<<<dim3((nt + 127) / 128, R), 128, 0, st>>>(xp, R, nv, nt, m->d_tris.p, pb->d_tgeo.p,
                                                                   pb->d_sDm.p);
        pb->launches++;
        float4 kff;
        const FarConst2 c = far_consts(pb, kff);
        const int tps = (nt + ns - 1) / ns;
        dim3 grid((nt + pb->far_tris - 1) / pb->far_tris, ns);
        const float4 *pts = pb->far_reduce ? pb->d_poff.p : pb->d_pt.p;
        const size_t smem = farm_smem_bytes(R);
        if (pb->prof_on) {
            OSRC_TRY(far_prof_collect(pb));
            OSRC_CK(cudaEventRecord(pb->prof_ev[0], st));
        }
#define OSRC_FARM_LAUNCH(C)                                                                                    \
    farm_kernel<C><<<grid, FAR_THREADS, smem, st>>>(pts, pb->d_cen.p, pb->d_tn.p, pb->d_tv.p, pb->d_sG.p,      \
                                                    pb->d_sDm.p, R, nt, tps, pb->far_tris, c, kff, pb->d_partm.p)
        if (pb->far_reduce) OSRC_FARM_LAUNCH(true);
        else OSRC_FARM_LAUNCH(false);
#undef OSRC_FARM_LAUNCH
        pb->launches++;
        OSRC_CK(cudaGetLastError());
        if (pb->prof_on) {
            OSRC_CK(cudaEventRecord(pb->prof_ev[1], st));
            pb->prof_pending = true;
            pb->prof_rhs_pending = R;
        }
    }
    return gather_launch(pb, ns, R, pb->d_partm.p, nullptr, use_far, use_near, 1.0, xp, yp, st);
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
    OSRC_TRY(farm_prepare(pb, st));
    int r0 = 0;
    while (r0 < nrhs) {
        const int left = nrhs - r0;
        const int R = std::min(left, FARM_MAX_R);
        if (R == 1) OSRC_TRY(far_apply(pb, xs[r0], ys[r0], part, st));
        else OSRC_TRY(farm_launch(pb, xs + r0, ys + r0, R, part, st));
        r0 += R;
    }
    return OSRC_OK;
}
