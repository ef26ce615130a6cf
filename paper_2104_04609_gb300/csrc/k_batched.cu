// k_batched.cu -- kernels of the batched mixed-precision solve of the
// assembled system (the dense path for blocks of right-hand sides):
//   - packing of the FP64 dense system into the BF16 real embedding used by
//     the tensor-core GEMM (far-field entries only: the touching-pair blocks
//     stay exact in the near-field CSR);
//   - packing / unpacking of blocks of right-hand sides around the GEMM,
//     fused with the near-field CSR product;
//   - an FP32 multi-right-hand-side CG / COCG for the fused OSRC
//     preconditioner (Sec. 2.6, 2.7), one thread-block cluster per (system,
//     group of 8 right-hand sides), and the explicit BF16 preconditioner
//     matrix built from it;
//   - FP32 batched Arnoldi helpers (projections, updates, norms, Givens;
//     one classical Gram-Schmidt pass per iteration);
//   - the residual product R = B - A X of the outer refinement in
//     float-float arithmetic (about 48 significant bits) on the FP32 pipes.
// Block vectors of the inner solver are stored [row][rhs] (right-hand sides
// fastest, complex FP32), so every row access is coalesced across the block.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <memory>

#include "osrc_internal.cuh"

namespace cg = cooperative_groups;

namespace {

__device__ __forceinline__ float2 f2c(float r, float i) { return make_float2(r, i); }
__device__ __forceinline__ float2 fadd(float2 a, float2 b) { return f2c(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 fsub(float2 a, float2 b) { return f2c(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 fmulc(float2 a, float2 b) {
    return f2c(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 fscale(float2 a, float s) { return f2c(a.x * s, a.y * s); }
__device__ __forceinline__ float fabs2(float2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ float2 fdivc(float2 a, float2 b) {
    const float d = b.x * b.x + b.y * b.y;
    return f2c((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

// A_cat[m][k] = Re A[m][k] (k < n2), Im A[m][k - n2] (n2 <= k < 2 n2), 0 else.
__global__ void pack_a_kernel(int n2, int Mp, int Kp, const double2 *__restrict__ A,
                              __nv_bfloat16 *__restrict__ Acat) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)Mp * Kp) return;
    const int m = (int)(idx / Kp), k = (int)(idx % Kp);
    float v = 0.f;
    if (m < n2) {
        if (k < n2) v = (float)A[(size_t)m * n2 + k].x;
        else if (k < 2 * n2) v = (float)A[(size_t)m * n2 + (k - n2)].y;
    }
    Acat[idx] = __float2bfloat16_rn(v);
}

// At the vertex pairs of the near-field CSR the BF16 matrix keeps only the
// far-field part: A - (touching-pair blocks), which are applied exactly in
// FP32 from the CSR (a vertex pair can receive both touching and
// non-touching triangle-pair contributions).
__global__ void far_part_near_kernel(int nv, int Kp, const int *__restrict__ ptr, const int *__restrict__ col,
                                     const double2 *__restrict__ val, const double2 *__restrict__ A,
                                     __nv_bfloat16 *__restrict__ Acat) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nv) return;
    const int n2 = 2 * nv;
    for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
        const int j = col[e];
        const int rows[2] = {i, nv + i}, cols[2] = {j, nv + j};
        for (int a = 0; a < 2; ++a)
            for (int b = 0; b < 2; ++b) {
                const double2 f = csub(A[(size_t)rows[a] * n2 + cols[b]], val[4 * (size_t)e + 2 * a + b]);
                Acat[(size_t)rows[a] * Kp + cols[b]] = __float2bfloat16_rn((float)f.x);
                Acat[(size_t)rows[a] * Kp + n2 + cols[b]] = __float2bfloat16_rn((float)f.y);
            }
    }
}

// B_cat rows r < R: [Re X_r | -Im X_r]; rows R + r: [Im X_r | Re X_r];
// X given [row][rhs] complex FP32 (R right-hand sides, n2 rows).  With V, X is
// first divided by nrm[r] (0 where the column is done or nrm is 0) and stored
// there: the new basis vector, packed for the next product in the same pass.
__global__ void pack_b_kernel(int n2, int R, int Kp, const float2 *__restrict__ X, const float *__restrict__ nrm,
                              const int *__restrict__ done, float2 *__restrict__ V,
                              __nv_bfloat16 *__restrict__ Bcat) {
    __shared__ float2 tile[32][33];
    const int k0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    float sc = 1.f;
    if (V && r0 + tx < R) {
        const float s = nrm[r0 + tx];
        sc = (done[r0 + tx] || !(s > 0.f)) ? 0.f : 1.f / s;
    }
    for (int j = ty; j < 32; j += 8) {
        const int k = k0 + j, r = r0 + tx;
        float2 v = f2c(0.f, 0.f);
        if (k < n2 && r < R) {
            v = X[(size_t)k * R + r];
            if (V) {
                v = sc == 0.f ? f2c(0.f, 0.f) : fscale(v, sc);
                V[(size_t)k * R + r] = v;
            }
        }
        tile[j][tx] = v;
    }
    __syncthreads();
    for (int j = ty; j < 32; j += 8) {
        const int r = r0 + j, k = k0 + tx;
        if (r >= R || k >= n2) continue;
        const float2 v = tile[tx][j];
        Bcat[(size_t)r * Kp + k] = __float2bfloat16_rn(v.x);
        Bcat[(size_t)r * Kp + n2 + k] = __float2bfloat16_rn(-v.y);
        Bcat[(size_t)(R + r) * Kp + k] = __float2bfloat16_rn(v.y);
        Bcat[(size_t)(R + r) * Kp + n2 + k] = __float2bfloat16_rn(v.x);
    }
}

// y[m][r] = (C[m][r], C[m][R + r]) + (near CSR product)[m][r]
__global__ void unpack_near_kernel(int nv, int R, int ldc, const float *__restrict__ C,
                                   const int *__restrict__ ptr, const int *__restrict__ col,
                                   const float2 *__restrict__ val, const float2 *__restrict__ X,
                                   float2 *__restrict__ Y) {
    const int i = blockIdx.x;  // vertex
    const int r = threadIdx.x;
    if (i >= nv || r >= R) return;
    float2 y1 = f2c(C[(size_t)i * ldc + r], C[(size_t)i * ldc + R + r]);
    float2 y2 = f2c(C[(size_t)(nv + i) * ldc + r], C[(size_t)(nv + i) * ldc + R + r]);
    for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
        const int j = col[e];
        const float2 *b = val + 4 * (size_t)e;
        const float2 xa = X[(size_t)j * R + r], xb = X[(size_t)(nv + j) * R + r];
        const float2 b0 = b[0], b1 = b[1], b2 = b[2], b3 = b[3];
        y1 = fadd(y1, fadd(fmulc(b0, xa), fmulc(b1, xb)));
        y2 = fadd(y2, fadd(fmulc(b2, xa), fmulc(b3, xb)));
    }
    Y[(size_t)i * R + r] = y1;
    Y[(size_t)(nv + i) * R + r] = y2;
}

// Y[m][c] = 1 if m == k0 + c else 0 (a block of R identity columns)
__global__ void identity_block_kernel(int n2, int R, int k0, float2 *__restrict__ Y) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n2 * R) return;
    const int m = (int)(idx / R), c = (int)(idx % R);
    Y[idx] = f2c(m == k0 + c ? 1.f : 0.f, 0.f);
}

// Columns k0 .. k0 + R - 1 of the packed preconditioner matrix from the
// block Z = P M^-1 [e_k0 .. e_k0+R-1]: Pcat[m][k] = Re, Pcat[m][n2 + k] = Im.
__global__ void pack_p_block_kernel(int n2, int R, int k0, int Kp, const float2 *__restrict__ Z,
                                    __nv_bfloat16 *__restrict__ Pcat) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n2 * R) return;
    const int m = (int)(idx / R), c = (int)(idx % R);
    if (k0 + c >= n2) return;
    const float2 z = Z[idx];
    Pcat[(size_t)m * Kp + k0 + c] = __float2bfloat16_rn(z.x);
    Pcat[(size_t)m * Kp + n2 + k0 + c] = __float2bfloat16_rn(z.y);
}

// Y[m][r] = (C[m][r], C[m][R + r]) for the complex product of a packed matrix
__global__ void unpack_plain_kernel(int n2, int R, int ldc, const float *__restrict__ C, float2 *__restrict__ Y) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n2 * R) return;
    const int m = (int)(idx / R), r = (int)(idx % R);
    Y[idx] = f2c(C[(size_t)m * ldc + r], C[(size_t)m * ldc + R + r]);
}

// ---------------------------------------------------------------------------
// FP32 multi-right-hand-side CG / COCG: one CTA per (system, group of 8
// right-hand sides).  System s: (M + beta_s S) w = f, rows n = nv, input f
// is block row `half` of the block vector F ([2nv][R]), solution into W_s
// ([nv][R]).  Jacobi preconditioning, stop per right-hand side at
// |r| <= tol |f| (converged columns freeze), bounded by maxit.
// ---------------------------------------------------------------------------
constexpr int K32_THREADS = 512;
constexpr int K32_G = 8;

struct Kry32Sys {
    float2 beta;
    int half;    // 0: rows [0, nv), 1: rows [nv, 2nv) of F
    int conj;    // 1: Hermitian CG, 0: COCG
    int scaled;  // disjoint objects: row i uses beta * bscale[vcomp[i]]
};

struct Kry32Batch {
    int nsys;
    const int *vcomp;      // object of each row
    const float2 *bscale;  // per object (1 / k_eps^2 of the object)
    Kry32Sys s[34];
};

__device__ __forceinline__ float2 kry32_beta(const Kry32Batch &b, const Kry32Sys &s, int i) {
    return s.scaled ? fmulc(s.beta, b.bscale[b.vcomp[i]]) : s.beta;
}

__device__ float2 dotf(float2 a, float2 b, int conj) {
    return conj ? f2c(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x) : fmulc(a, b);
}

// Jacobi inverse diagonal of every system: dinv[s][i] = 1 / (M_ii + beta_s S_ii)
__global__ void kry32_diag_kernel(Kry32Batch batch, int nv, const int *__restrict__ ptr,
                                  const int *__restrict__ col, const float *__restrict__ Mv,
                                  const float *__restrict__ Sv, float2 *__restrict__ dinv) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int sid = blockIdx.y;
    if (i >= nv) return;
    float md = 0.f, sd = 0.f;
    for (int e = ptr[i]; e < ptr[i + 1]; ++e)
        if (col[e] == i) {
            md = Mv[e];
            sd = Sv[e];
        }
    const float2 be = kry32_beta(batch, batch.s[sid], i);
    dinv[(size_t)sid * nv + i] = fdivc(f2c(1.f, 0.f), f2c(md + be.x * sd, be.y * sd));
}

// One cluster of CS CTAs per (system, group of 8 right-hand sides); each CTA
// owns a contiguous block of rows.  Search directions of other CTAs are read
// with L2-only loads after the cluster barrier; per-right-hand-side dot
// products are reduced over the cluster through distributed shared memory
// and summed in rank order, so every CTA takes the same decisions.
__global__ void __launch_bounds__(K32_THREADS)
kry32_kernel(Kry32Batch batch, int nv, int R, int ngroups, const int *__restrict__ ptr,
             const int *__restrict__ col, const float *__restrict__ Mv, const float *__restrict__ Sv,
             const float2 *__restrict__ F, const float2 *__restrict__ dinv, float2 *__restrict__ W,
             float2 *__restrict__ work, float tol, int maxit, int *__restrict__ its_out) {
    __shared__ float red[K32_THREADS / 32][K32_G][3];
    __shared__ float slotA[K32_G][3], slotB[K32_G][3], slotC[K32_G][3];
    __shared__ float gath[16][K32_G][3];
    __shared__ float sums[K32_G][3];
    __shared__ float2 sc_rho[K32_G], sc_al[K32_G], sc_be[K32_G];
    __shared__ float sc_bb[K32_G];
    __shared__ int active[K32_G], stepped[K32_G];
    cg::cluster_group cl = cg::this_cluster();
    const unsigned cs = cl.num_blocks(), rank = cl.block_rank();
    const int cid = blockIdx.x / cs;
    const int sid = cid / ngroups, grp = cid % ngroups;
    const int g0 = grp * K32_G;
    const Kry32Sys sy = batch.s[sid];
    const int gl = threadIdx.x % K32_G, rl = threadIdx.x / K32_G;
    const int nrl = K32_THREADS / K32_G;
    const int rows = (nv + (int)cs - 1) / (int)cs;
    const int r0 = min(nv, (int)rank * rows), r1 = min(nv, r0 + rows);
    const int r = g0 + gl;
    const bool rv = r < R;
    const size_t plane = (size_t)nv * R;
    float2 *rr = work + ((size_t)sid * 3 + 0) * plane;
    float2 *pp = work + ((size_t)sid * 3 + 1) * plane;
    float2 *qq = work + ((size_t)sid * 3 + 2) * plane;
    float2 *x = W + (size_t)sid * plane;
    const float2 *f = F + (size_t)sy.half * plane;
    const int cj = sy.conj;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // sums[g][0..2] = cluster-wide sums of (a, b, c) for right-hand side g
    auto reduce3 = [&](float a, float b, float c, float (*slot)[3]) {
        for (int o = 16; o >= K32_G; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (lane < K32_G) {
            red[warp][lane][0] = a;
            red[warp][lane][1] = b;
            red[warp][lane][2] = c;
        }
        __syncthreads();
        if (threadIdx.x < K32_G) {
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
            for (int w = 0; w < K32_THREADS / 32; ++w) {
                s0 += red[w][threadIdx.x][0];
                s1 += red[w][threadIdx.x][1];
                s2 += red[w][threadIdx.x][2];
            }
            slot[threadIdx.x][0] = s0;
            slot[threadIdx.x][1] = s1;
            slot[threadIdx.x][2] = s2;
        }
        cl.sync();
        if (threadIdx.x < cs * K32_G) {
            const int rk = threadIdx.x / K32_G, g = threadIdx.x % K32_G;
            const float *rem = cl.map_shared_rank(&slot[0][0], rk);
            gath[rk][g][0] = rem[3 * g];
            gath[rk][g][1] = rem[3 * g + 1];
            gath[rk][g][2] = rem[3 * g + 2];
        }
        __syncthreads();
        if (threadIdx.x < K32_G) {
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
            for (unsigned rk = 0; rk < cs; ++rk) {
                s0 += gath[rk][threadIdx.x][0];
                s1 += gath[rk][threadIdx.x][1];
                s2 += gath[rk][threadIdx.x][2];
            }
            sums[threadIdx.x][0] = s0;
            sums[threadIdx.x][1] = s1;
            sums[threadIdx.x][2] = s2;
        }
        __syncthreads();
    };

    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
    if (rv)
        for (int i = r0 + rl; i < r1; i += nrl) {
            const float2 di = dinv[(size_t)sid * nv + i];
            const size_t k = (size_t)i * R + r;
            const float2 b = f[k];
            x[k] = f2c(0.f, 0.f);
            rr[k] = b;
            const float2 zi = fmulc(di, b);
            pp[k] = zi;
            const float2 t = dotf(b, zi, cj);
            a0 += t.x;
            a1 += t.y;
            a2 += fabs2(b);
        }
    reduce3(a0, a1, a2, slotA);
    if (threadIdx.x < K32_G) {
        sc_rho[threadIdx.x] = f2c(sums[threadIdx.x][0], sums[threadIdx.x][1]);
        sc_bb[threadIdx.x] = sums[threadIdx.x][2];
        active[threadIdx.x] = (g0 + (int)threadIdx.x < R && sums[threadIdx.x][2] > 0.f) ? 1 : 0;
        if (rank == 0 && its_out && g0 + (int)threadIdx.x < R) its_out[sid * R + g0 + threadIdx.x] = 0;
    }
    cl.sync();  // p complete everywhere
    for (int it = 1; it <= maxit; ++it) {
        int any = 0;
        for (int g = 0; g < K32_G; ++g) any |= active[g];
        if (!any) break;
        // q = A p on own rows, (p, q)
        const bool act = rv && active[gl];
        float w0 = 0.f, w1 = 0.f;
        if (act)
            for (int i = r0 + rl; i < r1; i += nrl) {
                float2 mp = f2c(0.f, 0.f), sp = f2c(0.f, 0.f), pi = f2c(0.f, 0.f);
                for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
                    const int j = col[e];
                    const float2 pj = __ldcg(&pp[(size_t)j * R + r]);
                    if (j == i) pi = pj;
                    mp = fadd(mp, fscale(pj, Mv[e]));
                    sp = fadd(sp, fscale(pj, Sv[e]));
                }
                const float2 acc = fadd(mp, fmulc(kry32_beta(batch, sy, i), sp));
                qq[(size_t)i * R + r] = acc;
                const float2 t = dotf(pi, acc, cj);
                w0 += t.x;
                w1 += t.y;
            }
        reduce3(w0, w1, 0.f, slotB);
        if (threadIdx.x < K32_G) {
            const float2 pq = f2c(sums[threadIdx.x][0], sums[threadIdx.x][1]);
            if (active[threadIdx.x] && !(fabs2(pq) > 0.f)) active[threadIdx.x] = 0;  // breakdown: freeze
            stepped[threadIdx.x] = active[threadIdx.x];
            sc_al[threadIdx.x] = active[threadIdx.x] ? fdivc(sc_rho[threadIdx.x], pq) : f2c(0.f, 0.f);
        }
        __syncthreads();
        // r -= alpha q, z = D^-1 r, (r, z), |r|^2
        const bool act2 = rv && stepped[gl];
        const float2 al = sc_al[gl];
        float u0 = 0.f, u1 = 0.f, u2 = 0.f;
        if (act2)
            for (int i = r0 + rl; i < r1; i += nrl) {
                const size_t k = (size_t)i * R + r;
                const float2 ri = fsub(rr[k], fmulc(al, qq[k]));
                rr[k] = ri;
                const float2 zi = fmulc(dinv[(size_t)sid * nv + i], ri);
                const float2 t = dotf(ri, zi, cj);
                u0 += t.x;
                u1 += t.y;
                u2 += fabs2(ri);
            }
        reduce3(u0, u1, u2, slotC);
        if (threadIdx.x < K32_G) {
            const int g = threadIdx.x;
            if (active[g]) {
                const float2 rn = f2c(sums[g][0], sums[g][1]);
                if (rank == 0 && its_out) its_out[sid * R + g0 + g] = it;
                if (sums[g][2] <= tol * tol * sc_bb[g] || !(fabs2(sc_rho[g]) > 0.f)) {
                    active[g] = 0;
                    sc_be[g] = f2c(0.f, 0.f);
                } else {
                    sc_be[g] = fdivc(rn, sc_rho[g]);
                    sc_rho[g] = rn;
                }
            }
        }
        __syncthreads();
        // x += alpha p_old (every column that stepped); p = z + beta p_old (columns still active)
        const bool act3 = rv && active[gl];
        const float2 be = sc_be[gl];
        if (act2)
            for (int i = r0 + rl; i < r1; i += nrl) {
                const size_t k = (size_t)i * R + r;
                const float2 po = pp[k];
                x[k] = fadd(x[k], fmulc(al, po));
                if (act3) pp[k] = fadd(fmulc(dinv[(size_t)sid * nv + i], rr[k]), fmulc(be, po));
            }
        cl.sync();
    }
    cl.sync();  // shared memory of every CTA stays alive until all have read it
}

struct OsrcComb32 {
    int np;
    float2 ik, iik, cu, g0;
    float2 a[16], g[16];
    const float2 *ik_obj;  // disjoint objects: i k of each object (else ik)
    const int *vcomp;
};

// z1 = i k [cu u1 - sum_j a_j v_j],  z2 = [g0 v'_0 + sum_j g_j v'_j] / (i k)
__global__ void osrc_combine32_kernel(int nv, int R, OsrcComb32 c, const float2 *__restrict__ W,
                                      float2 *__restrict__ Z) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t plane = (size_t)nv * R;
    if (k >= plane) return;
    float2 a = fmulc(c.cu, W[k]);
    for (int j = 0; j < c.np; ++j) a = fsub(a, fmulc(c.a[j], W[(size_t)(1 + j) * plane + k]));
    float2 b = fmulc(c.g0, W[(size_t)(c.np + 1) * plane + k]);
    for (int j = 0; j < c.np; ++j) b = fadd(b, fmulc(c.g[j], W[(size_t)(c.np + 2 + j) * plane + k]));
    float2 ik = c.ik, iik = c.iik;
    if (c.ik_obj) {
        ik = c.ik_obj[c.vcomp[k / R]];
        iik = fdivc(f2c(1.f, 0.f), ik);
    }
    Z[k] = fmulc(ik, a);
    Z[plane + k] = fmulc(iik, b);
}

// M and S values in FP32
__global__ void d2f2_kernel(size_t n, const double2 *__restrict__ a, float2 *__restrict__ b) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = make_float2((float)a[i].x, (float)a[i].y);
}

__global__ void d2f_kernel(int n, const double *__restrict__ a, float *__restrict__ b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}

// ---------------------------------------------------------------------------
// FP32 batched Arnoldi: block vectors [n2][R]
// ---------------------------------------------------------------------------
// Column dot products out[i][r] = sum_m conj(V_i[m][r]) w[m][r], i < nvec, in
// two deterministic stages.  Stage 1: block (c, group of BD_VEC vectors) sums
// row chunk c into part[i][c][r]; a thread holds two neighbouring columns
// (16-byte loads) and BD_VEC vectors, so that w is read once for all of them
// and BD_VEC + 1 loads are in flight per row.  Stage 2 adds the chunks in
// order.  One vector a block with 8-byte loads streamed at 60 % of this.
constexpr int BD_THREADS = 256;
constexpr int BD_MAX_CHUNK = 64;
constexpr int BD_VEC = 4;

__device__ __forceinline__ void cdot_acc(float4 &s, const float4 &a, const float4 &b) {  // s += conj(a) b, two columns
    s.x += a.x * b.x + a.y * b.y;
    s.y += a.x * b.y - a.y * b.x;
    s.z += a.z * b.z + a.w * b.w;
    s.w += a.z * b.w - a.w * b.z;
}

__global__ void __launch_bounds__(BD_THREADS)
bdots_part_kernel(const float2 *__restrict__ V, size_t ldv, int nvec, const float2 *__restrict__ w, int n2, int R,
                  int nchunk, float2 *__restrict__ part) {
    __shared__ float4 acc[BD_THREADS];
    const int c = blockIdx.x, i0 = blockIdx.y * BD_VEC, R2 = R / 2;
    const int r = threadIdx.x % R2, rl = threadIdx.x / R2, nrl = BD_THREADS / R2;
    const int rows = (n2 + nchunk - 1) / nchunk;
    const int m0 = c * rows, m1 = min(n2, m0 + rows);
    const float4 *v[BD_VEC];
#pragma unroll
    for (int a = 0; a < BD_VEC; ++a) v[a] = reinterpret_cast<const float4 *>(V + ldv * min(i0 + a, nvec - 1));
    const float4 *w4 = reinterpret_cast<const float4 *>(w);
    float4 s[BD_VEC];
#pragma unroll
    for (int a = 0; a < BD_VEC; ++a) s[a] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rl < nrl) {
#pragma unroll 2
        for (int m = m0 + rl; m < m1; m += nrl) {
            const size_t k = (size_t)m * R2 + r;
            const float4 b = w4[k];
#pragma unroll
            for (int a = 0; a < BD_VEC; ++a) cdot_acc(s[a], v[a][k], b);
        }
    }
#pragma unroll
    for (int a = 0; a < BD_VEC; ++a) {
        if (i0 + a >= nvec) break;
        __syncthreads();
        acc[threadIdx.x] = s[a];
        __syncthreads();
        if (threadIdx.x < R2) {
            float4 t = acc[threadIdx.x];
            for (int l = 1; l < nrl; ++l) {
                const float4 o = acc[l * R2 + threadIdx.x];
                t.x += o.x;
                t.y += o.y;
                t.z += o.z;
                t.w += o.w;
            }
            reinterpret_cast<float4 *>(part + ((size_t)(i0 + a) * nchunk + c) * R)[threadIdx.x] = t;
        }
    }
}

// out[i][r] = sum_c part[i][c][r], four lanes per entry; with nrm != NULL (one
// vector, V = w) nrm[r] = sqrt(Re out[0][r]) instead
__global__ void bdots_fin_kernel(const float2 *__restrict__ part, int nvec, int nchunk, int R,
                                 float2 *__restrict__ out, float *__restrict__ nrm) {
    // thread = (entry group of 8, lane of 4, entry): eight neighbouring columns a quarter warp
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = idx / 32 * 8 + (idx & 7), q = (idx >> 3) & 3;
    const bool ok = k < nvec * R;
    const int i = ok ? k / R : 0, r = ok ? k % R : 0;
    float2 t = f2c(0.f, 0.f);
#pragma unroll 8
    for (int c = q; c < nchunk; c += 4) t = fadd(t, part[((size_t)i * nchunk + c) * R + r]);
    for (int o = 8; o < 32; o <<= 1) {
        t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
        t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
    if (!ok || q) return;
    if (nrm)
        nrm[r] = sqrtf(fmaxf(t.x, 0.f));
    else
        out[k] = t;
}

// w[m][r] -= sum_i h[i][r] V_i[m][r], and part[c][r] = sum over the block's row
// chunk of |w[m][r]|^2 (the columns' norms cost no pass of their own).  Block c
// takes rows [c rows, (c + 1) rows); a thread holds two neighbouring columns
// (16-byte loads), eight vectors ahead.
constexpr int BU_THREADS = 256;
__global__ void __launch_bounds__(BU_THREADS)
bupdate_kernel(const float2 *__restrict__ V, size_t ldv, int nvec, const float2 *__restrict__ h,
               float2 *__restrict__ w, int n2, int R, int rows, float *__restrict__ part) {
    __shared__ float2 acc[BU_THREADS];
    const int R2 = R / 2, r = threadIdx.x % R2, rl = threadIdx.x / R2, nrl = BU_THREADS / R2;
    const int m0 = blockIdx.x * rows, m1 = min(n2, m0 + rows);
    const float4 *V4 = reinterpret_cast<const float4 *>(V), *h4 = reinterpret_cast<const float4 *>(h);
    float4 *w4 = reinterpret_cast<float4 *>(w);
    float2 a = f2c(0.f, 0.f);
    if (rl < nrl)
        for (int m = m0 + rl; m < m1; m += nrl) {
            const size_t k = (size_t)m * R2 + r;
            float4 s = w4[k];
#pragma unroll 8
            for (int i = 0; i < nvec; ++i) {
                const float4 v = V4[ldv / 2 * i + k], g = h4[(size_t)i * R2 + r];
                s.x -= g.x * v.x - g.y * v.y;
                s.y -= g.x * v.y + g.y * v.x;
                s.z -= g.z * v.z - g.w * v.w;
                s.w -= g.z * v.w + g.w * v.z;
            }
            w4[k] = s;
            a.x += s.x * s.x + s.y * s.y;
            a.y += s.z * s.z + s.w * s.w;
        }
    acc[threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.x < R2) {
        float2 t = acc[threadIdx.x];
        for (int l = 1; l < nrl; ++l) t = fadd(t, acc[l * R2 + threadIdx.x]);
        reinterpret_cast<float2 *>(part + (size_t)blockIdx.x * R)[threadIdx.x] = t;
    }
}

// Per right-hand side r (BG_LANES lanes each): the column norm from its nc row
// chunks' shares, the new Hessenberg column H[.][j][r] (h from the projections,
// h_{j+1} = |w_r|), earlier Givens rotations, the new rotation, g update,
// residual estimate; columns that have converged keep their state (done[r] = 1,
// iteration count fixed).  The rotations are a serial chain per column: a warp
// stages their operands in shared memory, BG_TILE at a time, and one lane walks
// it (through global memory step by step it took 27 us at 25 iterations).
constexpr int BG_LANES = 32, BG_COLS = 4, BG_TILE = 64;
__global__ void bgivens_kernel(int j, int ldh, int R, const float2 *__restrict__ hcol,
                               const float *__restrict__ part, int nc, float *__restrict__ nrm,
                               float2 *__restrict__ H, float *__restrict__ cs, float2 *__restrict__ sn,
                               float2 *__restrict__ g, const float *__restrict__ beta, float tol,
                               int *__restrict__ done, int *__restrict__ its, float *__restrict__ res) {
    __shared__ float sc[BG_COLS][BG_TILE];
    __shared__ float2 ss[BG_COLS][BG_TILE], sh[BG_COLS][BG_TILE];
    const int lane = threadIdx.x % BG_LANES, col = threadIdx.x / BG_LANES, r = blockIdx.x * BG_COLS + col;
    if (r >= R) return;  // whole warps
    float t = 0.f;
    for (int c = lane; c < nc; c += BG_LANES) t += part[(size_t)c * R + r];
    for (int o = BG_LANES / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    const float wn = sqrtf(fmaxf(t, 0.f));
    if (lane == 0) nrm[r] = wn;
    if (done[r]) return;
    float2 *h = H + ((size_t)j * ldh) * R;  // h[i] at h[i * R + r]
    float2 hi = hcol[r];
    for (int i0 = 0; i0 < j; i0 += BG_TILE) {
        const int m = min(BG_TILE, j - i0);
        for (int a = lane; a < m; a += BG_LANES) {
            sc[col][a] = cs[(size_t)(i0 + a) * R + r];
            ss[col][a] = sn[(size_t)(i0 + a) * R + r];
            sh[col][a] = hcol[(size_t)(i0 + a + 1) * R + r];
        }
        __syncwarp();
        if (lane == 0)
            for (int a = 0; a < m; ++a) {
                const float c = sc[col][a];
                const float2 s = ss[col][a], h1 = sh[col][a];
                sh[col][a] = fadd(fscale(hi, c), fmulc(s, h1));
                hi = fadd(fscale(fmulc(f2c(s.x, -s.y), hi), -1.f), fscale(h1, c));
            }
        __syncwarp();
        for (int a = lane; a < m; a += BG_LANES) h[(size_t)(i0 + a) * R + r] = sh[col][a];
        __syncwarp();
    }
    if (lane != 0) return;
    const float2 a = hi, b = f2c(wn, 0.f);
    const float aa = sqrtf(fabs2(a)), bb = sqrtf(fabs2(b));
    const float nu = hypotf(aa, bb);
    float c;
    float2 s;
    if (aa == 0.f) {
        c = 0.f;
        s = f2c(1.f, 0.f);
    } else {
        c = aa / nu;
        s = fscale(fmulc(fscale(a, 1.f / aa), f2c(b.x, -b.y)), 1.f / nu);
    }
    cs[(size_t)j * R + r] = c;
    sn[(size_t)j * R + r] = s;
    h[(size_t)j * R + r] = fadd(fscale(a, c), fmulc(s, b));
    h[(size_t)(j + 1) * R + r] = f2c(0.f, 0.f);
    const float2 gj = g[(size_t)j * R + r];
    const float2 gn = fscale(fmulc(f2c(s.x, -s.y), gj), -1.f);
    g[(size_t)(j + 1) * R + r] = gn;
    g[(size_t)j * R + r] = fscale(gj, c);
    const float rel = sqrtf(fabs2(gn)) / beta[r];
    res[r] = rel;
    its[r] = j + 1;
    if (rel <= tol || !(nu > 0.f)) done[r] = 1;
}

// y_r = H_r^-1 g_r (its[r] x its[r] upper triangular) by columns: BS_COLS
// right-hand sides a block, BS_LANES threads each; y_i is final once the columns
// behind it have been subtracted from the right-hand side, and all lanes subtract
// column i together (row by row, a thread per right-hand side took 2.7 ms at 117
// iterations).
constexpr int BS_COLS = 8, BS_LANES = 32;
__global__ void __launch_bounds__(BS_COLS *BS_LANES)
bbacksub_kernel(int ldh, int R, const float2 *__restrict__ H, const float2 *__restrict__ g,
                const int *__restrict__ its, float2 *y) {
    __shared__ float2 yi[2][BS_COLS];
    const int cl = threadIdx.x % BS_COLS, ln = threadIdx.x / BS_COLS, r = blockIdx.x * BS_COLS + cl;
    const int m = r < R ? its[r] : 0;
    int mx = 0;
    for (int c = 0; c < BS_COLS; ++c)
        if (blockIdx.x * BS_COLS + c < R) mx = max(mx, its[blockIdx.x * BS_COLS + c]);
    for (int i = ln; i < m; i += BS_LANES) y[(size_t)i * R + r] = g[(size_t)i * R + r];
    for (int i = mx - 1; i >= 0; --i) {
        __syncthreads();
        if (ln == i % BS_LANES && i < m) {  // the lane that owns row i
            const float2 v = fdivc(y[(size_t)i * R + r], H[((size_t)i * ldh + i) * R + r]);
            y[(size_t)i * R + r] = v;
            yi[i & 1][cl] = v;
        }
        __syncthreads();
        if (i < m) {
            const float2 v = yi[i & 1][cl];
            for (int k = ln; k < i; k += BS_LANES)
                y[(size_t)k * R + r] = fsub(y[(size_t)k * R + r], fmulc(H[((size_t)i * ldh + k) * R + r], v));
        }
    }
}

// x[m][r] = sum_{i < its[r]} y[i][r] V_i[m][r]
__global__ void bcombine_kernel(const float2 *__restrict__ V, size_t ldv, int maxm, const float2 *__restrict__ y,
                                const int *__restrict__ its, float2 *__restrict__ x, int n2, int R) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (size_t)n2 * R) return;
    const int r = (int)(k % R);
    const int m = min(its[r], maxm);
    float2 s = f2c(0.f, 0.f);
    for (int i = 0; i < m; ++i) s = fadd(s, fmulc(y[(size_t)i * R + r], V[ldv * i + k]));
    x[k] = s;
}

// beta[r] = |c[:, r]| and V_0 = c / beta, g_0 = beta
__global__ void binit_kernel(int R, const float *__restrict__ nrm, float *__restrict__ beta,
                             float2 *__restrict__ g, int *__restrict__ done, int *__restrict__ its) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    beta[r] = nrm[r];
    g[r] = f2c(nrm[r], 0.f);
    done[r] = nrm[r] > 0.f ? 0 : 1;
    its[r] = 0;
}

// ---------------------------------------------------------------------------
// Residual of the outer refinement in float-float arithmetic on the FP32
// pipes (this part's FP64 rate is 1/64 of its FP32 rate).  Every real value
// is an unevaluated sum hi + lo of two floats (Dekker 1971): products by
// TwoProd with an FMA (exact), accumulation by Knuth's TwoSum (exact) with
// the rounding errors and cross terms carried in the low word, about 48
// significant bits.  A is split once (AFF: {Re hi, Im hi, Re lo, Im lo} per
// entry); X is split as it is staged.  R[r][m] = B[r][m] - sum_k A[m][k] X[r][k].
// ---------------------------------------------------------------------------
__global__ void split_ff_kernel(size_t n, const double2 *__restrict__ A, float4 *__restrict__ out) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 a = A[i];
    const float rh = (float)a.x, ih = (float)a.y;
    out[i] = make_float4(rh, ih, (float)(a.x - (double)rh), (float)(a.y - (double)ih));
}

// (sh, sl) += (ah + al) (xh + xl)
__device__ __forceinline__ void ff_mac(float &sh, float &sl, float ah, float al, float xh, float xl) {
    const float ph = __fmul_rn(ah, xh);
    float pl = fmaf(ah, xh, -ph);
    pl = fmaf(ah, xl, pl);
    pl = fmaf(al, xh, pl);
    const float t = __fadd_rn(sh, ph);
    const float bb = __fsub_rn(t, sh);
    const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bb)), __fsub_rn(ph, bb));
    sl = __fadd_rn(sl, __fadd_rn(err, pl));
    sh = t;
}

// 64 rows x 8 right-hand sides a block: with 16 a 6000-row, 64-column residual is
// 376 blocks, 2.5 per SM, and the SMs with three set the time
constexpr int FF_TM = 64, FF_TR = 8, FF_TK = 16;

__global__ void __launch_bounds__(256)
resid_ff_kernel(int n2, int nrhs, const float4 *__restrict__ AFF, const double2 *__restrict__ X,
                const double2 *__restrict__ B, double2 *__restrict__ Rr) {
    __shared__ float4 sa[FF_TM][FF_TK + 1];
    __shared__ float4 sx[FF_TR][FF_TK + 1];
    const int m0 = blockIdx.x * FF_TM, r0 = blockIdx.y * FF_TR;
    const int tid = threadIdx.x;
    const int tm = tid % 32, tr = tid / 32;  // rows tm, tm + 32; right-hand side tr
    float acc[2][4];                          // [row][re h, re l, im h, im l]
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = 0.f;
    for (int k0 = 0; k0 < n2; k0 += FF_TK) {
        for (int e = tid; e < FF_TM * FF_TK; e += 256) {
            const int mm = e / FF_TK, kk = e % FF_TK;
            sa[mm][kk] = (m0 + mm < n2 && k0 + kk < n2) ? AFF[(size_t)(m0 + mm) * n2 + k0 + kk]
                                                         : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int e = tid; e < FF_TR * FF_TK; e += 256) {
            const int rr = e / FF_TK, kk = e % FF_TK;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r0 + rr < nrhs && k0 + kk < n2) {
                const double2 x = X[(size_t)(r0 + rr) * n2 + k0 + kk];
                const float rh = (float)x.x, ih = (float)x.y;
                v = make_float4(rh, ih, (float)(x.x - (double)rh), (float)(x.y - (double)ih));
            }
            sx[rr][kk] = v;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < FF_TK; ++kk) {
            const float4 a[2] = {sa[tm][kk], sa[tm + 32][kk]};
            const float4 x = sx[tr][kk];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float *c = acc[i];
                ff_mac(c[0], c[1], a[i].x, a[i].z, x.x, x.z);    // + Re a Re x
                ff_mac(c[2], c[3], a[i].x, a[i].z, x.y, x.w);    // + Re a Im x
                ff_mac(c[0], c[1], -a[i].y, -a[i].w, x.y, x.w);  // - Im a Im x
                ff_mac(c[2], c[3], a[i].y, a[i].w, x.x, x.z);    // + Im a Re x
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = m0 + tm + 32 * i, r = r0 + tr;
        if (m < n2 && r < nrhs) {
            const float *c = acc[i];
            const double2 ax = cd((double)c[0] + (double)c[1], (double)c[2] + (double)c[3]);
            Rr[(size_t)r * n2 + m] = csub(B[(size_t)r * n2 + m], ax);
        }
    }
}

// per right-hand side: nrm[r] = |v[r][:]| (FP64, [nrhs][n2])
__global__ void norm_rows64_kernel(int n2, const double2 *__restrict__ v, double *__restrict__ nrm) {
    __shared__ double acc[256];
    const int r = blockIdx.x;
    double s = 0.0;
    for (int m = threadIdx.x; m < n2; m += blockDim.x) s += cabs2(v[(size_t)r * n2 + m]);
    acc[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) acc[threadIdx.x] += acc[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) nrm[r] = sqrt(acc[0]);
}

// [nrhs][n2] FP64 -> [n2][R] FP32, scaled per right-hand side by 1/scale[r]
__global__ void to_block32_kernel(int n2, int nrhs, int R, const double2 *__restrict__ src,
                                  const double *__restrict__ scale, float2 *__restrict__ dst) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (size_t)n2 * R) return;
    const int m = (int)(k / R), r = (int)(k % R);
    if (r >= nrhs || !(scale[r] > 0.0)) {
        dst[k] = f2c(0.f, 0.f);
        return;
    }
    const double2 v = src[(size_t)r * n2 + m];
    const double s = 1.0 / scale[r];
    dst[k] = f2c((float)(v.x * s), (float)(v.y * s));
}

// x[r][m] = d[m][r] (FP32 block -> FP64 rows)
__global__ void from_block32_kernel(int n2, int nrhs, int R, const float2 *__restrict__ d,
                                    double2 *__restrict__ x) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (size_t)n2 * nrhs) return;
    const int r = (int)(k / n2), m = (int)(k % n2);
    const float2 v = d[(size_t)m * R + r];
    x[k] = cd(v.x, v.y);
}

__global__ void fill1_kernel(double *__restrict__ a, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = 1.0;
}

// x[r][m] += scale[r] * d[m][r]
__global__ void add_block32_kernel(int n2, int nrhs, int R, const float2 *__restrict__ d,
                                   const double *__restrict__ scale, double2 *__restrict__ x) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (size_t)n2 * nrhs) return;
    const int r = (int)(k / n2), m = (int)(k % n2);
    const float2 v = d[(size_t)m * R + r];
    const double s = scale[r];
    x[k] = cadd(x[k], cd(s * v.x, s * v.y));
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int umma_gemm_bf16(const void *A, int M, int K, const void *Bm, int N, float *C, int ldc, float *ws,
                   size_t ws_floats, int *err, cudaStream_t st);
size_t umma_gemm_ws_floats(int M, int N, int K);

struct BatchedState {
    int n2 = 0, Mp = 0, Kp = 0, R = 0;
    DBuf<__nv_bfloat16> Acat, Bcat;
    DBuf<__nv_bfloat16> Pcat;   // explicit preconditioner matrix P M^-1 (packed like Acat), if built
    bool pdense = false;
    DBuf<float> C;
    DBuf<float> gws;            // pieces of the GEMM's split tiles
    DBuf<float> M32, S32;
    DBuf<float4> AFF;           // float-float split of the FP64 system matrix (residuals)
    DBuf<float2> nr32;          // touching-pair CSR values in FP32
    DBuf<float2> obj32;         // [2][objects]: i k_osrc, 1 / k_eps^2 in FP32
    DBuf<int> err;
    DBuf<float2> kwork, kW;     // multi-RHS Krylov work and solutions
    DBuf<float2> kdinv;         // Jacobi inverse diagonals [system][row]
    DBuf<float2> V, w, t1, t2;  // inner GMRES basis and temporaries
    DBuf<float2> H, hcol, g, sn, yv;
    DBuf<float2> part;          // per-chunk partial column dot products
    DBuf<float> cs, nrm, beta, res;
    DBuf<int> done, its, kits;
    DBuf<double2> X64, R64;
    DBuf<double> bn, rn, scl;
    int basis_cap = 0;
    int *hdone = nullptr;       // pinned: convergence flags of two iterations
    cudaEvent_t ev[2] = {nullptr, nullptr};
    ~BatchedState() {
        if (hdone) cudaFreeHost(hdone);
        for (auto &e : ev)
            if (e) cudaEventDestroy(e);
    }
};

void batched_free(BatchedState *s) { delete s; }

int batched_prepare(osrc_problem *pb, int R, int maxit_inner, cudaStream_t st) {
    if (!pb->d_dense.p) return OSRC_UNSUPPORTED;
    osrc_ctx *ctx = pb->mesh->ctx;
    const int nv = pb->nv, n2 = 2 * nv;
    if (!pb->batched) {
        // the problem's only once it is complete (out of memory may end it anywhere)
        std::unique_ptr<BatchedState> bs(new BatchedState);
        bs->n2 = n2;
        bs->Mp = (n2 + 127) / 128 * 128;
        bs->Kp = (2 * n2 + 63) / 64 * 64;
        OSRC_TRY(bs->Acat.alloc(ctx, (size_t)bs->Mp * bs->Kp));
        const size_t tot = (size_t)bs->Mp * bs->Kp;
        pack_a_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n2, bs->Mp, bs->Kp, pb->d_dense.p, bs->Acat.p);
        far_part_near_kernel<<<(nv + 127) / 128, 128, 0, st>>>(nv, bs->Kp, pb->d_nr_ptr.p, pb->d_nr_col.p,
                                                               pb->d_nr_val.p, pb->d_dense.p, bs->Acat.p);
        const size_t nn = (size_t)n2 * n2;
        OSRC_TRY(bs->AFF.alloc(ctx, nn));
        split_ff_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(nn, pb->d_dense.p, bs->AFF.p);
        const size_t nq = 4 * (size_t)pb->near_nnz;
        OSRC_TRY(bs->nr32.alloc(ctx, nq));
        d2f2_kernel<<<(unsigned)((nq + 255) / 256), 256, 0, st>>>(nq, pb->d_nr_val.p, bs->nr32.p);
        {
            const int nc = pb->mesh->ncomp;
            std::vector<float2> o(2 * (size_t)nc);
            for (int m = 0; m < nc; ++m) {
                const ObjMat &om = pb->obj[m];
                const double2 ke2 = cmul(om.k_eps, om.k_eps), inv = cdiv(cd(1.0, 0.0), ke2);
                o[m] = make_float2((float)-om.k_osrc_i, (float)om.k_osrc);
                o[nc + m] = make_float2((float)inv.x, (float)inv.y);
            }
            OSRC_TRY(bs->obj32.alloc(ctx, o.size()));
            OSRC_CK(cudaMemcpy(bs->obj32.p, o.data(), o.size() * sizeof(float2), cudaMemcpyHostToDevice));
        }
        OSRC_TRY(bs->M32.alloc(ctx, pb->ms_nnz));
        OSRC_TRY(bs->S32.alloc(ctx, pb->ms_nnz));
        d2f_kernel<<<(pb->ms_nnz + 255) / 256, 256, 0, st>>>(pb->ms_nnz, pb->d_M.p, bs->M32.p);
        d2f_kernel<<<(pb->ms_nnz + 255) / 256, 256, 0, st>>>(pb->ms_nnz, pb->d_S.p, bs->S32.p);
        OSRC_TRY(bs->err.alloc(ctx, 1));
        OSRC_CK(cudaMemsetAsync(bs->err.p, 0, sizeof(int), st));
        pb->launches += 4;
        OSRC_CK(cudaGetLastError());
        pb->batched = bs.release();
    }
    BatchedState *bs = pb->batched;
    if (bs->R != R || bs->basis_cap < maxit_inner) {
        const size_t plane = (size_t)n2 * R, vplane = (size_t)nv * R;
        const int nsys = 2 * pb->p.n_pade + 2;
        bs->R = bs->basis_cap = 0;  // until all are there
        OSRC_TRY(bs->Bcat.alloc(ctx, (size_t)2 * R * bs->Kp));
        OSRC_CK(cudaMemsetAsync(bs->Bcat.p, 0, (size_t)2 * R * bs->Kp * sizeof(__nv_bfloat16), st));
        OSRC_TRY(bs->C.alloc(ctx, (size_t)bs->Mp * 2 * R));
        OSRC_TRY(bs->gws.alloc(ctx, umma_gemm_ws_floats(bs->Mp, 2 * R, bs->Kp)));
        OSRC_TRY(bs->kwork.alloc(ctx, (size_t)nsys * 3 * vplane));
        OSRC_TRY(bs->kdinv.alloc(ctx, (size_t)nsys * nv));
        OSRC_TRY(bs->kW.alloc(ctx, (size_t)nsys * vplane));
        OSRC_TRY(bs->V.alloc(ctx, (size_t)(maxit_inner + 1) * plane));
        OSRC_TRY(bs->w.alloc(ctx, plane));
        OSRC_TRY(bs->t1.alloc(ctx, plane));
        OSRC_TRY(bs->t2.alloc(ctx, plane));
        OSRC_TRY(bs->H.alloc(ctx, (size_t)(maxit_inner + 1) * (maxit_inner + 1) * R));
        OSRC_TRY(bs->hcol.alloc(ctx, (size_t)(maxit_inner + 1) * R));
        // projections' chunk sums, or the update's row-chunk norms (at most 1216 floats a column)
        OSRC_TRY(bs->part.alloc(ctx, std::max((size_t)(maxit_inner + 1) * BD_MAX_CHUNK, (size_t)640) * R));
        OSRC_TRY(bs->g.alloc(ctx, (size_t)(maxit_inner + 1) * R));
        OSRC_TRY(bs->sn.alloc(ctx, (size_t)(maxit_inner + 1) * R));
        OSRC_TRY(bs->yv.alloc(ctx, (size_t)(maxit_inner + 1) * R));
        OSRC_TRY(bs->cs.alloc(ctx, (size_t)(maxit_inner + 1) * R));
        OSRC_TRY(bs->nrm.alloc(ctx, R));
        OSRC_TRY(bs->beta.alloc(ctx, R));
        OSRC_TRY(bs->res.alloc(ctx, R));
        OSRC_TRY(bs->done.alloc(ctx, R));
        OSRC_TRY(bs->its.alloc(ctx, R));
        OSRC_TRY(bs->kits.alloc(ctx, (size_t)nsys * R));
        OSRC_TRY(bs->bn.alloc(ctx, R));
        OSRC_TRY(bs->rn.alloc(ctx, R));
        OSRC_TRY(bs->scl.alloc(ctx, R));
        bs->R = R;
        bs->basis_cap = maxit_inner;
    }
    return OSRC_OK;
}

// y = A_inner x for a block x ([n2][R] FP32): BF16 tensor-core GEMM of the
// far-field part + exact near-field CSR product
static void batched_pack(osrc_problem *pb, const float2 *x, float2 *v, cudaStream_t st) {
    BatchedState *bs = pb->batched;
    const dim3 gb((bs->n2 + 31) / 32, (bs->R + 31) / 32);
    pack_b_kernel<<<gb, dim3(32, 8), 0, st>>>(bs->n2, bs->R, bs->Kp, x, bs->nrm.p, bs->done.p, v, bs->Bcat.p);
    pb->launches++;
}

// packed: Bcat holds x already
static int batched_matvec(osrc_problem *pb, const float2 *x, float2 *y, bool packed, cudaStream_t st) {
    BatchedState *bs = pb->batched;
    const int R = bs->R, nv = pb->nv;
    if (!packed) batched_pack(pb, x, nullptr, st);
    OSRC_TRY(umma_gemm_bf16(bs->Acat.p, bs->Mp, bs->Kp, bs->Bcat.p, 2 * R, bs->C.p, 2 * R, bs->gws.p,
                            bs->gws.n, bs->err.p, st));
    unpack_near_kernel<<<nv, R, 0, st>>>(nv, R, 2 * R, bs->C.p, pb->d_nr_ptr.p, pb->d_nr_col.p, bs->nr32.p, x,
                                         y);
    pb->launches += 2;
    OSRC_CK(cudaGetLastError());
    return OSRC_OK;
}

// z = P M^-1 y for a block y ([n2][R] FP32), inner tolerance tol
static int batched_precond(osrc_problem *pb, const float2 *y, float2 *z, float tol, int maxit, cudaStream_t st) {
    BatchedState *bs = pb->batched;
    const int nv = pb->nv, R = bs->R, np = pb->p.n_pade;
    const double2 ke2 = cmul(pb->k_eps, pb->k_eps);
    // disjoint objects: 1/k_eps^2 of each row's object through bscale
    const double2 inv = pb->multi ? cd(1.0, 0.0) : cdiv(cd(1.0, 0.0), ke2);
    const int sc = pb->multi ? 1 : 0;
    Kry32Batch b{};
    b.nsys = 2 * np + 2;
    b.vcomp = pb->mesh->d_vcomp.p;
    b.bscale = pb->multi ? bs->obj32.p + pb->mesh->ncomp : nullptr;
    b.s[0] = Kry32Sys{make_float2(0.f, 0.f), 0, 1, 0};
    for (int j = 0; j < np; ++j) {
        const double2 be = cscale(cmul(pb->B[j], inv), -1.0);
        b.s[1 + j] = Kry32Sys{make_float2((float)be.x, (float)be.y), 0, 0, sc};
        b.s[np + 2 + j] = Kry32Sys{make_float2((float)be.x, (float)be.y), 1, 0, sc};
    }
    const double2 be0 = cscale(inv, -1.0);
    b.s[np + 1] = Kry32Sys{make_float2((float)be0.x, (float)be0.y), 1, 0, sc};
    kry32_diag_kernel<<<dim3((nv + 255) / 256, b.nsys), 256, 0, st>>>(b, nv, pb->d_ms_ptr.p, pb->d_ms_col.p,
                                                                        bs->M32.p, bs->S32.p, bs->kdinv.p);
    const int ngroups = (R + K32_G - 1) / K32_G;
    int cs = (nv + 999) / 1000;
    if (cs < 1) cs = 1;
    if (cs > 8) cs = 8;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b.nsys * ngroups * cs, 1, 1);
    cfg.blockDim = dim3(K32_THREADS, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    OSRC_CK(cudaLaunchKernelEx(&cfg, kry32_kernel, b, nv, R, ngroups, (const int *)pb->d_ms_ptr.p,
                               (const int *)pb->d_ms_col.p, (const float *)bs->M32.p, (const float *)bs->S32.p,
                               y, (const float2 *)bs->kdinv.p, bs->kW.p, bs->kwork.p, tol, maxit,
                               bs->kits.p));
    OsrcComb32 c{};
    c.np = np;
    {
        const double2 ik = cd(-pb->k_osrc_i, pb->k_osrc), iik = cdiv(cd(1.0, 0.0), ik);
        c.ik = make_float2((float)ik.x, (float)ik.y);
        c.iik = make_float2((float)iik.x, (float)iik.y);
    }
    double2 cu = pb->C0;
    for (int j = 0; j < np; ++j) {
        const double2 a = cdiv(pb->A[j], pb->B[j]);
        cu = cadd(cu, a);
        c.a[j] = make_float2((float)a.x, (float)a.y);
        c.g[j] = make_float2((float)pb->g[j].x, (float)pb->g[j].y);
    }
    c.cu = make_float2((float)cu.x, (float)cu.y);
    c.g0 = make_float2((float)pb->g0.x, (float)pb->g0.y);
    c.ik_obj = pb->multi ? bs->obj32.p : nullptr;
    c.vcomp = pb->mesh->d_vcomp.p;
    const size_t plane = (size_t)nv * R;
    osrc_combine32_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, st>>>(nv, R, c, bs->kW.p, z);
    pb->launches += 3;
    OSRC_CK(cudaGetLastError());
    return OSRC_OK;
}

// z = P M^-1 y through the explicit BF16 preconditioner matrix (one
// tensor-core GEMM); used once osrc_dense_precond_build has run
static int batched_precond_dense(osrc_problem *pb, const float2 *y, float2 *z, cudaStream_t st) {
    BatchedState *bs = pb->batched;
    const int n2 = bs->n2, R = bs->R;
    batched_pack(pb, y, nullptr, st);
    OSRC_TRY(umma_gemm_bf16(bs->Pcat.p, bs->Mp, bs->Kp, bs->Bcat.p, 2 * R, bs->C.p, 2 * R, bs->gws.p,
                            bs->gws.n, bs->err.p, st));
    const size_t plane = (size_t)n2 * R;
    unpack_plain_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, st>>>(n2, R, 2 * R, bs->C.p, z);
    pb->launches += 2;
    OSRC_CK(cudaGetLastError());
    return OSRC_OK;
}

static int batched_apply_precond(osrc_problem *pb, const float2 *y, float2 *z, float ptol, int pmaxit,
                                 cudaStream_t st) {
    return pb->batched->pdense ? batched_precond_dense(pb, y, z, st) : batched_precond(pb, y, z, ptol, pmaxit, st);
}

// Inner solve: GMRES (FP32, classical Gram-Schmidt) on P M^-1 A_inner d = P M^-1 c
// for a block c ([n2][R]); d returned in bs->t1.  Returns the largest
// iteration count.
static int batched_inner_gmres(osrc_problem *pb, const float2 *c, float tol, int maxit, float ptol,
                               int pmaxit, int *iters_out, cudaStream_t st) {
    BatchedState *bs = pb->batched;
    const int n2 = bs->n2, R = bs->R;
    const size_t plane = (size_t)n2 * R;
    const int ldh = maxit + 1;
    const unsigned gp = (unsigned)((plane + 255) / 256);
    const int nchunk = std::max(1, std::min(BD_MAX_CHUNK, n2 / 64));
    if (!bs->hdone) OSRC_CK(cudaMallocHost((void **)&bs->hdone, 2 * 128 * sizeof(int)));
    for (auto &e : bs->ev)
        if (!e) OSRC_CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    auto dots = [&](int nvec, const float2 *w, float2 *out) {
        bdots_part_kernel<<<dim3(nchunk, (nvec + BD_VEC - 1) / BD_VEC), BD_THREADS, 0, st>>>(bs->V.p, plane, nvec, w,
                                                                                              n2, R, nchunk, bs->part.p);
        bdots_fin_kernel<<<(nvec * R * 4 + 255) / 256, 256, 0, st>>>(bs->part.p, nvec, nchunk, R, out, nullptr);
    };
    auto norm = [&](const float2 *w) {
        bdots_part_kernel<<<dim3(nchunk, 1), BD_THREADS, 0, st>>>(w, plane, 1, w, n2, R, nchunk, bs->part.p);
        bdots_fin_kernel<<<(R * 4 + 255) / 256, 256, 0, st>>>(bs->part.p, 1, nchunk, R, nullptr, bs->nrm.p);
    };
    // rhs of the preconditioned system
    OSRC_TRY(batched_apply_precond(pb, c, bs->w.p, ptol, pmaxit, st));
    norm(bs->w.p);
    binit_kernel<<<(R + 127) / 128, 128, 0, st>>>(R, bs->nrm.p, bs->beta.p, bs->g.p, bs->done.p, bs->its.p);
    OSRC_CK(cudaMemsetAsync(bs->g.p + R, 0, (size_t)maxit * R * sizeof(float2), st));
    batched_pack(pb, bs->w.p, bs->V.p, st);
    // row chunks of the update: as many as bs->part has room for
    const int unrl = 2 * BU_THREADS / R;  // rows a block takes at a time
    const int urows = ((n2 + 1215) / 1216 + unrl - 1) / unrl * unrl, uchunk = (n2 + urows - 1) / urows;
    // The host reads the convergence flags of iteration j while the device
    // runs iteration j + 1 (an iteration too many, on columns that are all
    // frozen, when j was the last): it waited 60 to 90 us for them otherwise.
    int *hdone[2] = {bs->hdone, bs->hdone + R};
    int j = 0, its = 0;
    for (j = 0; j < maxit; ++j) {
        float2 *vj = bs->V.p + (size_t)j * plane;
        OSRC_TRY(batched_matvec(pb, vj, bs->t2.p, true, st));
        OSRC_TRY(batched_apply_precond(pb, bs->t2.p, bs->w.p, ptol, pmaxit, st));
        // one classical Gram-Schmidt pass: the inner solve only reduces the
        // residual by inner_tol (>= 1e-3 in use), far above where FP32 CGS
        // loses orthogonality, and the outer refinement corrects the rest
        // (a second pass cost 25 % more time for 2 % fewer iterations)
        dots(j + 1, bs->w.p, bs->hcol.p);
        bupdate_kernel<<<uchunk, BU_THREADS, 0, st>>>(bs->V.p, plane, j + 1, bs->hcol.p, bs->w.p, n2, R, urows,
                                                      (float *)bs->part.p);
        bgivens_kernel<<<(R + BG_COLS - 1) / BG_COLS, BG_COLS * BG_LANES, 0, st>>>(j, ldh, R, bs->hcol.p, (const float *)bs->part.p,
                                                                   uchunk, bs->nrm.p, bs->H.p, bs->cs.p, bs->sn.p,
                                                                   bs->g.p, bs->beta.p, tol, bs->done.p, bs->its.p,
                                                                   bs->res.p);
        batched_pack(pb, bs->w.p, bs->V.p + (size_t)(j + 1) * plane, st);
        pb->launches += 4;
        OSRC_CK(cudaMemcpyAsync(hdone[j & 1], bs->done.p, R * sizeof(int), cudaMemcpyDeviceToHost, st));
        OSRC_CK(cudaEventRecord(bs->ev[j & 1], st));
        its = j + 1;
        if (j > 0) {
            OSRC_CK(cudaEventSynchronize(bs->ev[(j - 1) & 1]));
            bool all = true;
            for (int r = 0; r < R; ++r) all = all && hdone[(j - 1) & 1][r];
            if (all) {
                its = j;
                break;
            }
        }
    }
    // the flags' last copies land before the buffers are used again
    OSRC_CK(cudaStreamSynchronize(st));
    j = its;
    bbacksub_kernel<<<(R + BS_COLS - 1) / BS_COLS, BS_COLS * BS_LANES, 0, st>>>(ldh, R, bs->H.p, bs->g.p, bs->its.p, bs->yv.p);
    bcombine_kernel<<<gp, 256, 0, st>>>(bs->V.p, plane, maxit, bs->yv.p, bs->its.p, bs->t1.p, n2, R);
    pb->launches += 2;
    OSRC_CK(cudaGetLastError());
    *iters_out = j;
    return OSRC_OK;
}

// ---------------------------------------------------------------------------
// outer FP64 iterative refinement
// ---------------------------------------------------------------------------
extern "C" int osrc_dense_batched_solve(osrc_problem *pb, const void *b, void *x, int nrhs, double tol,
                                        int max_refine, double inner_tol, int inner_maxit, double precond_tol,
                                        osrc_batched_info *info_out, void *stream) {
    if (!pb || !b || !x || nrhs < 1 || nrhs > 128 || !(tol > 0.0) || max_refine < 1 || !(inner_tol > 0.0) ||
        inner_tol >= 1.0 || inner_maxit < 1 || inner_maxit > 1000 || !(precond_tol < 1.0))
        return OSRC_INVALID_ARG;
    if (pb->p.precision != OSRC_FP64_DENSE) {
        osrc_set_error("osrc_dense_batched_solve needs a problem created with OSRC_FP64_DENSE");
        return OSRC_UNSUPPORTED;
    }
    OSRC_CK(cudaSetDevice(pb->mesh->ctx->device));
    const auto t0 = std::chrono::steady_clock::now();
    cudaStream_t st = (cudaStream_t)stream;
    const int R = (nrhs + 7) / 8 * 8;
    OSRC_TRY(batched_prepare(pb, R, inner_maxit, st));
    BatchedState *bs = pb->batched;
    osrc_ctx *ctx = pb->mesh->ctx;
    const int n2 = bs->n2;
    if (bs->R64.n < (size_t)nrhs * n2) OSRC_TRY(bs->R64.alloc(ctx, (size_t)nrhs * n2));
    const double2 *B = (const double2 *)b;
    double2 *X = (double2 *)x;
    osrc_batched_info info{};
    OSRC_CK(cudaMemsetAsync(X, 0, (size_t)nrhs * n2 * sizeof(double2), st));
    OSRC_CK(cudaMemcpyAsync(bs->R64.p, B, (size_t)nrhs * n2 * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    OSRC_CK(cudaMemsetAsync(bs->rn.p, 0, R * sizeof(double), st));
    norm_rows64_kernel<<<nrhs, 256, 0, st>>>(n2, B, bs->bn.p);
    std::vector<double> hb(nrhs), hr(nrhs);
    OSRC_CK(cudaMemcpyAsync(hb.data(), bs->bn.p, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
    OSRC_CK(cudaStreamSynchronize(st));
    const size_t plane = (size_t)n2 * R;
    const unsigned gp = (unsigned)((plane + 255) / 256);
    const unsigned gx = (unsigned)(((size_t)nrhs * n2 + 255) / 256);
    double worst = 1.0;
    int refine = 0;
    for (refine = 0; refine <= max_refine; ++refine) {
        norm_rows64_kernel<<<nrhs, 256, 0, st>>>(n2, bs->R64.p, bs->rn.p);
        OSRC_CK(cudaMemcpyAsync(hr.data(), bs->rn.p, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
        OSRC_CK(cudaStreamSynchronize(st));
        worst = 0.0;
        for (int r = 0; r < nrhs; ++r) worst = fmax(worst, hb[r] > 0 ? hr[r] / hb[r] : 0.0);
        if (!std::isfinite(worst)) return OSRC_BREAKDOWN;
        if (worst <= tol || refine == max_refine) break;
        // scaled residual block: c = R64 / |R64_r|
        OSRC_CK(cudaMemcpyAsync(bs->scl.p, bs->rn.p, nrhs * sizeof(double), cudaMemcpyDeviceToDevice, st));
        to_block32_kernel<<<gp, 256, 0, st>>>(n2, nrhs, R, bs->R64.p, bs->scl.p, bs->t2.p);
        OSRC_CK(cudaMemcpyAsync(bs->w.p, bs->t2.p, plane * sizeof(float2), cudaMemcpyDeviceToDevice, st));
        int its = 0;
        const double ptol = precond_tol > 0.0 ? precond_tol : std::min(1e-3, std::max(1e-6, 0.1 * inner_tol));
        OSRC_TRY(batched_inner_gmres(pb, bs->w.p, (float)inner_tol, inner_maxit, (float)ptol, 500, &its, st));
        info.inner_iterations += its;
        add_block32_kernel<<<gx, 256, 0, st>>>(n2, nrhs, R, bs->t1.p, bs->scl.p, X);
        dim3 grid((n2 + FF_TM - 1) / FF_TM, (nrhs + FF_TR - 1) / FF_TR);
        resid_ff_kernel<<<grid, 256, 0, st>>>(n2, nrhs, bs->AFF.p, X, B, bs->R64.p);
        pb->launches += 3;
        OSRC_CK(cudaGetLastError());
    }
    int err = 0;
    OSRC_CK(cudaMemcpyAsync(&err, bs->err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    OSRC_CK(cudaStreamSynchronize(st));
    info.refinements = refine;
    info.residual = worst;
    info.ms_total = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    if (info_out) *info_out = info;
    if (err) {
        osrc_set_error("tensor-core GEMM: a bounded wait gave up");
        return OSRC_TIMEOUT;
    }
    return worst <= tol ? OSRC_OK : OSRC_NOT_CONVERGED;
}

extern "C" int osrc_dense_batched_apply_ex(osrc_problem *pb, const void *x, void *y, int nrhs, int what,
                                           double ptol, int pmaxit, int *pits_max, void *stream) {
    if (!pb || !x || !y || nrhs < 1 || nrhs > 128 || what < 0 || what > 3) return OSRC_INVALID_ARG;
    if (!(ptol > 0.0) || pmaxit < 1) return OSRC_INVALID_ARG;
    if (pb->p.precision != OSRC_FP64_DENSE) return OSRC_UNSUPPORTED;
    OSRC_CK(cudaSetDevice(pb->mesh->ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    const int R = (nrhs + 7) / 8 * 8;
    OSRC_TRY(batched_prepare(pb, R, 8, st));
    BatchedState *bs = pb->batched;
    const int n2 = bs->n2;
    const size_t plane = (size_t)n2 * R;
    fill1_kernel<<<(R + 127) / 128, 128, 0, st>>>(bs->scl.p, R);
    to_block32_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, st>>>(n2, nrhs, R, (const double2 *)x,
                                                                      bs->scl.p, bs->t2.p);
    float2 *out = bs->t2.p;
    if (what == 3) {
        if (!bs->pdense) {
            osrc_set_error("no explicit preconditioner matrix: call osrc_dense_precond_build first");
            return OSRC_UNSUPPORTED;
        }
        OSRC_TRY(batched_precond_dense(pb, bs->t2.p, bs->t1.p, st));
        out = bs->t1.p;
    }
    if (what == 0 || what == 2) {
        OSRC_TRY(batched_matvec(pb, bs->t2.p, bs->w.p, false, st));
        out = bs->w.p;
    }
    if (what == 1 || what == 2) {
        OSRC_TRY(batched_precond(pb, out, bs->t1.p, (float)ptol, pmaxit, st));
        out = bs->t1.p;
        if (pits_max) {
            const int ns = 2 * pb->p.n_pade + 2;
            std::vector<int> k((size_t)ns * R);
            OSRC_CK(cudaMemcpyAsync(k.data(), bs->kits.p, k.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
            OSRC_CK(cudaStreamSynchronize(st));
            int mx = 0;
            for (int v : k) mx = v > mx ? v : mx;
            *pits_max = mx;
        }
    }
    from_block32_kernel<<<(unsigned)(((size_t)n2 * nrhs + 255) / 256), 256, 0, st>>>(n2, nrhs, R, out,
                                                                                     (double2 *)y);
    OSRC_CK(cudaGetLastError());
    int err = 0;
    OSRC_CK(cudaMemcpyAsync(&err, bs->err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    OSRC_CK(cudaStreamSynchronize(st));
    return err ? OSRC_TIMEOUT : OSRC_OK;
}

// y = op(x) with the inner (mixed-precision) pieces, for tests: what 0 the
// BF16 far + exact near operator, 1 the FP32 preconditioner P M^-1, 2 both.
extern "C" int osrc_dense_batched_apply(osrc_problem *pb, const void *x, void *y, int nrhs, int what,
                                        void *stream) {
    return osrc_dense_batched_apply_ex(pb, x, y, nrhs, what, 1e-6, 1000, nullptr, stream);
}

extern "C" int osrc_dense_precond_build(osrc_problem *pb, double tol, int maxit, void *stream) {
    if (!pb || !(tol > 0.0) || !(tol < 1.0) || maxit < 1 || maxit > 1000) return OSRC_INVALID_ARG;
    if (pb->p.precision != OSRC_FP64_DENSE) {
        osrc_set_error("osrc_dense_precond_build needs a problem created with OSRC_FP64_DENSE");
        return OSRC_UNSUPPORTED;
    }
    OSRC_CK(cudaSetDevice(pb->mesh->ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    const int R = 128;
    OSRC_TRY(batched_prepare(pb, R, pb->batched ? std::max(8, pb->batched->basis_cap) : 8, st));
    BatchedState *bs = pb->batched;
    const int n2 = bs->n2;
    bs->pdense = false;
    if (!bs->Pcat.p) OSRC_TRY(bs->Pcat.alloc(pb->mesh->ctx, (size_t)bs->Mp * bs->Kp));
    OSRC_CK(cudaMemsetAsync(bs->Pcat.p, 0, (size_t)bs->Mp * bs->Kp * sizeof(__nv_bfloat16), st));
    const size_t plane = (size_t)n2 * R;
    const unsigned gp = (unsigned)((plane + 255) / 256);
    for (int k0 = 0; k0 < n2; k0 += R) {
        identity_block_kernel<<<gp, 256, 0, st>>>(n2, R, k0, bs->t2.p);
        OSRC_TRY(batched_precond(pb, bs->t2.p, bs->t1.p, (float)tol, maxit, st));
        pack_p_block_kernel<<<gp, 256, 0, st>>>(n2, R, k0, bs->Kp, bs->t1.p, bs->Pcat.p);
        pb->launches += 2;
    }
    OSRC_CK(cudaGetLastError());
    OSRC_CK(cudaStreamSynchronize(st));
    bs->pdense = true;
    return OSRC_OK;
}

extern "C" int osrc_dense_precond_drop(osrc_problem *pb) {
    if (!pb) return OSRC_INVALID_ARG;
    if (pb->batched) {
        OSRC_CK(cudaSetDevice(pb->mesh->ctx->device));
        pb->batched->pdense = false;
        pb->batched->Pcat.release();
    }
    return OSRC_OK;
}

// Device bytes the batched solve of a problem with nv vertices adds for R
// right-hand sides (rounded up to 8) and an inner cap maxit: packed BF16
// system and preconditioner matrices, the float-float split of the system,
// the inner basis and block vectors, the FP32 shifted-solve work.
size_t estimate_batched_bytes(int nv, int n_pade, int nrhs, int maxit) {
    const size_t R = (size_t)((nrhs + 7) / 8 * 8), n2 = 2 * (size_t)nv;
    const size_t Mp = (n2 + 127) / 128 * 128, Kp = (2 * n2 + 63) / 64 * 64;
    const size_t nsys = 2 * (size_t)n_pade + 2;
    size_t b = 2 * Mp * Kp * 2 + n2 * n2 * 16;                 // Acat, Pcat, AFF
    b += (size_t)(maxit + 1) * n2 * R * 8;                      // inner basis
    b += (size_t)(maxit + 1) * (maxit + 1) * R * 8;             // Hessenberg
    b += (size_t)(maxit + 1) * 64 * R * 8 + 8 * (size_t)(maxit + 1) * R * 8;
    b += 4 * n2 * R * 8 + Mp * 2 * R * 4 + 2 * R * Kp * 2;     // block vectors, GEMM in/out
    b += umma_gemm_ws_floats((int)Mp, (int)(2 * R), (int)Kp) * 4;  // GEMM split-tile pieces
    b += nsys * (4 * (size_t)nv * R + nv) * 8;                  // shifted solves
    b += (size_t)nrhs * n2 * 16;                                // FP64 residual block
    return b;
}
