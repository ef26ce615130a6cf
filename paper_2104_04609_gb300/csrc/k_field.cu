// k_field.cu -- total pressure at points off the surface from a solution of
// the permuted PMCHWT system (Sec. 2.2, representation formulas; the paper
// measures its accuracy this way on a grid through the object, Sec. 3.2).
//
// With psi = exterior normal derivative and phi = trace of the total field
// (outward normal), rho = rho_int / rho_ext:
//   outside: u = u_inc + DLP_0 phi - SLP_0 psi
//   inside:  u = rho SLP_1 psi - DLP_1 phi
//   SLP_k psi(x) = int G_k(x, y) psi(y) dy,  DLP_k phi(x) = int dG_k/dn_y phi(y) dy,
// each integral by the 6-point rule per triangle with the P1 densities
// interpolated at the rule points.  A point's region comes from the Laplace
// double layer of the constant 1 (Gauss: 1 inside, 0 outside), so each
// target needs one wavenumber only and a warp never diverges in the pair loop.
// Disjoint objects (Sec. 2.2): source points are stored object by object;
// a point inside object m (region m + 1) takes the interior representation
// over that object's surface with its own material.
// Pass 1 (region) runs in FP32; pass 2 (field) in FP64.  Both split the source
// points over gridDim.y, so that a few thousand targets fill every SM, and add
// the splits' sums in order (10201 targets in 80 blocks of 128 left 72 of 152
// SMs idle).
#include <algorithm>

#include "osrc_internal.cuh"

namespace {

constexpr double kFa1 = 0.445948490915965, kFw1 = 0.223381589678011;
constexpr double kFa2 = 0.091576213509771, kFw2 = 0.109951743655322;
constexpr double kFInv4Pi = 0.079577471545947667884;
constexpr int FT = 128;          // targets per block; source points per tile of the region pass
constexpr int FTT = 16;          // source triangles per tile of the field pass
constexpr int FIELD_TAB = 512;   // entries of the e^{i theta} table per turn
constexpr int FIELD_MAX_SPLIT = 64;
// most doubles of splits' sums (256 MB); beyond it, and where the memory is not
// there, both passes run unsplit, which takes none (targets enough to reach it
// fill the SMs without splits)
constexpr size_t FIELD_MAX_SCRATCH = (size_t)1 << 25;

// Source data per rule point (6 per triangle): {y, w |tau|}, {n, 0} and
// {w psi_q re, im, w phi_q re, im} with w including the area.
__global__ void field_src_kernel(int nt, int nv, const int *__restrict__ tris, const double *__restrict__ verts,
                                 const double *__restrict__ tgeo, const int *__restrict__ order,
                                 const double2 *__restrict__ x, double4 *__restrict__ src) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 6 * nt) return;
    const int t = order[idx / 6], q = idx % 6;
    const double al = q < 3 ? kFa1 : kFa2, w = q < 3 ? kFw1 : kFw2;
    double bc[3] = {al, al, al};
    bc[q % 3] = 1.0 - 2.0 * al;
    double y[3] = {0, 0, 0};
    double2 ps = cd(0, 0), ph = cd(0, 0);
    for (int a = 0; a < 3; ++a) {
        const int v = tris[3 * t + a];
        for (int j = 0; j < 3; ++j) y[j] += bc[a] * verts[3 * v + j];
        ps = cadd(ps, cscale(x[v], bc[a]));
        ph = cadd(ph, cscale(x[nv + v], bc[a]));
    }
    const double *g = tgeo + 16 * (size_t)t;
    const double W = w * g[0];
    src[3 * (size_t)idx] = make_double4(y[0], y[1], y[2], W);
    src[3 * (size_t)idx + 1] = make_double4(g[1], g[2], g[3], 0.0);
    src[3 * (size_t)idx + 2] = make_double4(W * ps.x, W * ps.y, W * ph.x, W * ph.y);
}

// rtot[(split * nobj + m) * npts + i]: the split's share of the solid angle of
// object m's surface at point i, sum_q w_q (y_q - x).n_q / r^3.  obeg:
// [nobj + 1] source-point ranges of the objects.  One split (rtot null): the
// regions themselves (see field_region).
__global__ void __launch_bounds__(FT)
field_region_kernel(int npts, const double *__restrict__ pts, int nobj, const int *__restrict__ obeg,
                    const double4 *__restrict__ src, double *__restrict__ rtot, int *__restrict__ region) {
    __shared__ float4 sy[FT], sn[FT];
    const int i = blockIdx.x * FT + threadIdx.x;
    const bool valid = i < npts;
    const float x0 = valid ? (float)pts[3 * (size_t)i] : 0.f, x1 = valid ? (float)pts[3 * (size_t)i + 1] : 0.f,
                x2 = valid ? (float)pts[3 * (size_t)i + 2] : 0.f;
    int reg = 0;
    for (int m = 0; m < nobj; ++m) {
        const int b0 = obeg[m], b1 = obeg[m + 1];
        const long long tiles = (b1 - b0 + FT - 1) / FT;
        const int t0 = (int)(tiles * blockIdx.y / gridDim.y), t1 = (int)(tiles * (blockIdx.y + 1) / gridDim.y);
        double total = 0.0;
        for (int base = b0 + t0 * FT; base < min(b1, b0 + t1 * FT); base += FT) {
            const int j = base + threadIdx.x;
            if (j < b1) {
                const double4 a = src[3 * (size_t)j], b = src[3 * (size_t)j + 1];
                sy[threadIdx.x] = make_float4((float)a.x, (float)a.y, (float)a.z, (float)a.w);
                sn[threadIdx.x] = make_float4((float)b.x, (float)b.y, (float)b.z, 0.f);
            }
            __syncthreads();
            const int jn = min(FT, b1 - base);
            float acc = 0.f;
            for (int jj = 0; jj < jn; ++jj) {
                const float4 y = sy[jj], n = sn[jj];
                const float d0 = y.x - x0, d1 = y.y - x1, d2 = y.z - x2;
                const float ri = rsqrtf(d0 * d0 + d1 * d1 + d2 * d2);
                acc += y.w * (d0 * n.x + d1 * n.y + d2 * n.z) * ri * ri * ri;
            }
            total += (double)acc;
            __syncthreads();
        }
        if (!rtot) {
            if (total * kFInv4Pi > 0.5) reg = m + 1;
        } else if (valid) {
            rtot[((size_t)blockIdx.y * nobj + m) * npts + i] = total;
        }
    }
    if (!rtot && valid) region[i] = reg;
}

// region of target i: the last object whose surface has a solid angle of more
// than half a turn there (inside), m + 1, else 0
__device__ __forceinline__ int field_region(int i, int npts, int nobj, int nsplit, const double *__restrict__ rtot) {
    int reg = 0;
    for (int m = 0; m < nobj; ++m) {
        double total = 0.0;
        for (int s = 0; s < nsplit; ++s) total += rtot[((size_t)s * nobj + m) * npts + i];
        if (total * kFInv4Pi > 0.5) reg = m + 1;
    }
    return reg;
}

struct FieldConst {
    double k0;
    int inc_kind;  // 0 none, 1 plane wave (s = direction), 2 point source (s = position)
    double s0, s1, s2;
};

// One split's sum at each target, part[split * npts + i] = D - S outside,
// rho S - D inside (without 1/(4 pi)).  Bound by the FP64 pipe, 2 operations a
// cycle and SM on this part, so the pair's operations are what counts, 43
// here: 97 ms for 101^2 targets x 122880 points (307 ms with sincos(), rsqrt()
// and the normal product per point, 154 issue slots a pair, and with blocks
// for half of the SMs):
//  - (y - x).n is constant over a flat triangle: once per six points;
//  - 1/r from the hardware's approximation (rsqrt.approx.ftz.f64, about 2^-20)
//    and one third-order step of the binomial series of (1 - e)^(-1/2),
//    e = 1 - r^2 y^2;
//  - e^{i k r} from a table of 512 angles per turn and short Taylor series of
//    the rest (|delta| <= pi / 512: delta^5 / 120 and delta^4 / 24 are the last
//    terms above 1e-16); the turn fraction r k / 2 pi - integer is formed by
//    fused multiply-adds with k / 2 pi as a pair, so no rounding of k r enters;
//  - densities carry the weights, 1/(4 pi) is applied at the end.
template <bool ABSORB>
__global__ void __launch_bounds__(FT)
field_kernel(int npts, const double *__restrict__ pts, int nt, int nobj, const int *__restrict__ obeg,
             const ObjMat *__restrict__ obj, const double4 *__restrict__ src, const double *__restrict__ rtot, int nrs,
             int *__restrict__ region, FieldConst c, double2 *__restrict__ part) {
    __shared__ double2 tab[FIELD_TAB];
    __shared__ double sy[FTT * 6][3];
    __shared__ double4 sd[FTT * 6];
    __shared__ double sn[FTT][3];
    const int i = blockIdx.x * FT + threadIdx.x;
    const bool valid = i < npts;
    for (int j = threadIdx.x; j < FIELD_TAB; j += FT) sincospi(j * (2.0 / FIELD_TAB), &tab[j].y, &tab[j].x);
    const double x0 = valid ? pts[3 * (size_t)i] : 0.0, x1 = valid ? pts[3 * (size_t)i + 1] : 0.0,
                 x2 = valid ? pts[3 * (size_t)i + 2] : 0.0;
    const int ins = !valid ? 0 : rtot ? field_region(i, npts, nobj, nrs, rtot) : region[i];
    if (valid && rtot && blockIdx.y == 0) region[i] = ins;
    // outside: every source point, k0; inside object m: its own points, k_m
    const double k = ins ? obj[ins - 1].k1 : c.k0;
    const double ki = ins ? obj[ins - 1].k1i : 0.0;  // attenuation inside
    const int lo = ins ? obeg[ins - 1] / 6 : 0, hi = ins ? obeg[ins] / 6 : nt;  // triangles
    // k FIELD_TAB / (2 pi) as hi + lo, 1 / (2 pi) a pair itself
    const double i2p = 0.15915494309189535, i2pl = -9.839338337591243e-18;
    const double ch = k * (FIELD_TAB * i2p), cl = fma(k, FIELD_TAB * i2p, -ch) + k * (FIELD_TAB * i2pl);
    const double magic = 6755399441055744.0;  // 1.5 * 2^52: rounds to an integer in the low bits
    const double e = 6.283185307179586 / FIELD_TAB;
    const double a1 = e, a3 = -e * e * e / 6.0, a5 = e * e * e * e * e / 120.0, b2 = -e * e / 2.0,
                 b4 = e * e * e * e / 24.0;
    double2 S = cd(0, 0), D = cd(0, 0);
    const int t_begin = (int)((long long)nt * blockIdx.y / gridDim.y),
              t_end = (int)((long long)nt * (blockIdx.y + 1) / gridDim.y);
    for (int base = t_begin; base < t_end; base += FTT) {
        const int cnt = min(FTT, t_end - base);
        __syncthreads();
        for (int j = threadIdx.x; j < cnt * 6; j += FT) {
            const double4 a = src[3 * (6 * (size_t)base + j)];
            sy[j][0] = a.x;
            sy[j][1] = a.y;
            sy[j][2] = a.z;
            sd[j] = src[3 * (6 * (size_t)base + j) + 2];
        }
        for (int j = threadIdx.x; j < cnt; j += FT) {
            const double4 b = src[18 * ((size_t)base + j) + 1];
            sn[j][0] = b.x;
            sn[j][1] = b.y;
            sn[j][2] = b.z;
        }
        __syncthreads();
        const int j0 = max(0, lo - base), j1 = min(cnt, hi - base);
        for (int jj = j0; jj < j1; ++jj) {
            double dn = 0.0;
            double2 T = cd(0, 0);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const double *y = sy[6 * jj + q];
                const double4 dv = sd[6 * jj + q];
                const double d0 = y[0] - x0, d1 = y[1] - x1, d2 = y[2] - x2;  // y - x
                if (q == 0) dn = fma(d2, sn[jj][2], fma(d1, sn[jj][1], d0 * sn[jj][0]));
                const double r2 = fma(d2, d2, fma(d1, d1, d0 * d0));
                double y0;
                asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(r2));
                const double er = fma(-(r2 * y0), y0, 1.0);
                const double ri = fma(y0 * er, fma(0.375, er, 0.5), y0);
                const double r = r2 * ri;
                const double qd = fma(r, ch, magic), qn = qd - magic;
                const double f = fma(r, cl, fma(r, ch, -qn)), t = f * f;
                const double2 E = tab[__double2loint(qd) & (FIELD_TAB - 1)];
                const double sp = f * fma(t, fma(t, a5, a3), a1), cm = t * fma(t, b4, b2);
                double gr = fma(E.x, cm, fma(-E.y, sp, E.x)) * ri, gi = fma(E.y, cm, fma(E.x, sp, E.y)) * ri;
                if (ABSORB) {
                    const double damp = ki != 0.0 ? exp(-ki * r) : 1.0;
                    gr *= damp;
                    gi *= damp;
                }
                S.x = fma(gr, dv.x, fma(-gi, dv.y, S.x));  // w G psi_q
                S.y = fma(gr, dv.y, fma(gi, dv.x, S.y));
                // w dG/dn_y r^2 / ((y - x).n) = G (i k r - 1) [- k_i r]
                const double kr = k * r;
                double hr = -fma(kr, gi, gr), hi_ = fma(kr, gr, -gi);
                if (ABSORB) {
                    hr = fma(-ki * r, gr, hr);
                    hi_ = fma(-ki * r, gi, hi_);
                }
                const double ri2 = ri * ri;
                hr *= ri2;
                hi_ *= ri2;
                T.x = fma(hr, dv.z, fma(-hi_, dv.w, T.x));
                T.y = fma(hr, dv.w, fma(hi_, dv.z, T.y));
            }
            D.x = fma(dn, T.x, D.x);
            D.y = fma(dn, T.y, D.y);
        }
    }
    if (valid) part[(size_t)blockIdx.y * npts + i] = ins ? csub(cscale(S, obj[ins - 1].rho), D) : csub(D, S);
}

// u = sum of the splits / (4 pi), plus the incident field outside; a single
// split's sums are in u already (part = u)
__global__ void field_finish_kernel(int npts, const double *__restrict__ pts, int nsplit, const double2 *part,
                                    const int *__restrict__ region, FieldConst c, double2 *u) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npts) return;
    double2 out = cd(0, 0);
    for (int s = 0; s < nsplit; ++s) out = cadd(out, part[(size_t)s * npts + i]);
    out = cscale(out, kFInv4Pi);
    if (!region[i] && c.inc_kind) {
        const double x0 = pts[3 * (size_t)i], x1 = pts[3 * (size_t)i + 1], x2 = pts[3 * (size_t)i + 2];
        double sn_, cs_;
        if (c.inc_kind == 1) {
            sincos(c.k0 * (c.s0 * x0 + c.s1 * x1 + c.s2 * x2), &sn_, &cs_);
            out = cadd(out, cd(cs_, sn_));
        } else {
            const double e0 = x0 - c.s0, e1 = x1 - c.s1, e2 = x2 - c.s2;
            const double R = sqrt(e0 * e0 + e1 * e1 + e2 * e2);
            sincos(c.k0 * R, &sn_, &cs_);
            out = cadd(out, cd(cs_ * kFInv4Pi / R, sn_ * kFInv4Pi / R));
        }
    }
    u[i] = out;
}

// splits of `tiles` source tiles for nb target blocks: about `waves` times
// `slots` blocks in all, the count with the fullest last wave
int field_splits(int nb, int tiles, int slots, int waves) {
    const int cap = std::max(1, std::min(FIELD_MAX_SPLIT, tiles));
    const int s0 = std::max(1, std::min(cap, (waves * slots + nb - 1) / nb));
    int best = s0;
    double eff = -1.0;
    for (int s = std::max(1, s0 / 2); s <= std::min(cap, 2 * s0); ++s) {
        const long long blocks = (long long)nb * s, w = (blocks + slots - 1) / slots;
        const double f = (double)blocks / (double)(w * slots);
        if (f > eff + 1e-9) {
            eff = f;
            best = s;
        }
    }
    return best;
}

}  // namespace

extern "C" int osrc_field_eval(osrc_problem *pb, const void *x, const double *pts, int npts, int inc_kind,
                               const double *inc_param, void *u, int *region, void *stream) {
    if (!pb || !x || npts < 0 || inc_kind < 0 || inc_kind > 2 || (inc_kind && !inc_param))
        return OSRC_INVALID_ARG;
    if (npts == 0) return OSRC_OK;
    if (!pts || !u) return OSRC_INVALID_ARG;
    OSRC_CK(cudaSetDevice(pb->mesh->ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    osrc_mesh *m = pb->mesh;
    const int nt = pb->nt, ns = 6 * nt;
    if (pb->d_fsrc.n < 3 * (size_t)ns) OSRC_TRY(pb->d_fsrc.alloc(m->ctx, 3 * (size_t)ns));
    int *reg = region;
    if (!reg) {
        if (pb->d_freg.n < (size_t)npts) OSRC_TRY(pb->d_freg.alloc(m->ctx, npts));
        reg = pb->d_freg.p;
    }
    if (pb->d_fobeg.n < (size_t)m->ncomp + 1) {
        OSRC_TRY(pb->d_fobeg.alloc(m->ctx, m->ncomp + 1));
        std::vector<int> ob(m->ncomp + 1);
        for (int c = 0; c <= m->ncomp; ++c) ob[c] = 6 * m->comp_tbeg[c];
        OSRC_CK(cudaMemcpy(pb->d_fobeg.p, ob.data(), ob.size() * sizeof(int), cudaMemcpyHostToDevice));
    }
    field_src_kernel<<<(ns + 255) / 256, 256, 0, st>>>(nt, pb->nv, m->d_tris.p, m->d_verts.p, pb->d_tgeo.p,
                                                       m->d_tri_order.p, (const double2 *)x, pb->d_fsrc.p);
    const int nb = (npts + FT - 1) / FT;
    int sms = 0, per_r = 0, per_f = 0;
    OSRC_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->ctx->device));
    auto fk = pb->absorb ? field_kernel<true> : field_kernel<false>;
    OSRC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_r, field_region_kernel, FT, 0));
    OSRC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_f, fk, FT, 0));
    int nrs = field_splits(nb, (ns / m->ncomp + FT - 1) / FT, sms * std::max(1, per_r), 1);
    int nfs = field_splits(nb, (nt + FTT - 1) / FTT, sms * std::max(1, per_f), 3);
    // splits' sums: region [nrs][objects][npts], field [nfs][npts] complex
    const size_t nr = nrs > 1 ? (size_t)nrs * m->ncomp * npts : 0;
    const size_t np = nr + (nr & 1) + (nfs > 1 ? 2 * (size_t)nfs * npts : 0);
    bool split = np <= FIELD_MAX_SCRATCH;
    if (split && pb->d_fpart.n < np) {
        const int s = pb->d_fpart.alloc(m->ctx, np);
        if (s != OSRC_OK && s != OSRC_OUT_OF_MEMORY) return s;
        split = s == OSRC_OK;
    }
    if (!split) nrs = nfs = 1;
    double *rtot = nrs > 1 ? pb->d_fpart.p : nullptr;
    double2 *part = nfs > 1 ? (double2 *)(pb->d_fpart.p + nr + (nr & 1)) : (double2 *)u;
    field_region_kernel<<<dim3(nb, nrs), FT, 0, st>>>(npts, pts, m->ncomp, pb->d_fobeg.p, pb->d_fsrc.p, rtot, reg);
    FieldConst c{pb->p.k_ext, inc_kind, 0.0, 0.0, 0.0};
    if (inc_kind) {
        c.s0 = inc_param[0];
        c.s1 = inc_param[1];
        c.s2 = inc_param[2];
    }
    fk<<<dim3(nb, nfs), FT, 0, st>>>(npts, pts, nt, m->ncomp, pb->d_fobeg.p, pb->d_obj.p, pb->d_fsrc.p, rtot, nrs, reg,
                                     c, part);
    field_finish_kernel<<<(npts + 127) / 128, 128, 0, st>>>(npts, pts, nfs, part, reg, c, (double2 *)u);
    pb->launches += 4;
    OSRC_CK(cudaGetLastError());
    return OSRC_OK;
}
