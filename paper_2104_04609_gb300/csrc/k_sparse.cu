// k_sparse.cu -- P1 mass M and Laplace-Beltrami stiffness S (CSR, FP64), the
// mass preconditioner M^-1 (Sec. 2.4) and the OSRC preconditioner (Sec. 2.6,
// 2.7) by batched Krylov solves.
//
// Every inner system has the form (alpha M + beta S) w = f on the shared
// vertex-graph pattern.  One thread-block cluster (up to 8 CTAs) solves one
// system: each CTA owns a contiguous block of rows, the SpMV reads the search
// direction of the other CTAs from global memory after a cluster barrier,
// and dot products are reduced over the cluster through distributed shared
// memory, so a solve needs no host round trip and no grid-wide barrier.
// Rows owned by other CTAs are read with L2-only loads (__ldcg) after the
// cluster barrier, so no stale L1 line of an earlier iteration is used.
// Systems with real SPD matrices (M) use Hermitian CG; the complex-symmetric
// shifted OSRC systems use COCG (conjugate orthogonal CG, van der Vorst &
// Melissen 1990) with the unconjugated bilinear form x^T y.  Both are
// Jacobi-preconditioned and stop at |r| <= tol |f|.  All loops are bounded by
// the iteration cap; every CTA of a cluster takes the same branch because
// the decisions are made from cluster-reduced values summed in rank order.
// Two kernels: kmix_kernel (FP32 inner solves refined in FP64, used whenever
// a CTA's rows fit its registers; its vectors cross the cluster through
// distributed shared memory) and kry_kernel (all FP64, the layout above:
// larger meshes, in-place systems, the allocation-free entry).
#include <cooperative_groups.h>
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "bounded_wait.cuh"
#include "osrc_internal.cuh"

namespace cg = cooperative_groups;

namespace {

__global__ void ms_element_kernel(int nt, const double *__restrict__ tgeo,
                                  const double *__restrict__ verts, const int *__restrict__ tris,
                                  double *__restrict__ bm, double *__restrict__ bs) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    const double *g = tgeo + 16 * (size_t)t;
    const double area = g[0];
    // grad phi_a = curl phi_a x n has the same length, and grad.grad = curl.curl
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
            const double *ca = g + 4 + 3 * a, *cb = g + 4 + 3 * b;
            bm[9 * (size_t)t + 3 * a + b] = area / 12.0 * (a == b ? 2.0 : 1.0);
            bs[9 * (size_t)t + 3 * a + b] = area * (ca[0] * cb[0] + ca[1] * cb[1] + ca[2] * cb[2]);
        }
}

__global__ void csr_sum_kernel(int nnz, const int *__restrict__ cptr, const int *__restrict__ cidx,
                               const double *__restrict__ bm, const double *__restrict__ bs,
                               double *__restrict__ M, double *__restrict__ S) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nnz) return;
    double m = 0.0, s = 0.0;
    for (int k = cptr[e]; k < cptr[e + 1]; ++k) {
        m += bm[cidx[k]];
        s += bs[cidx[k]];
    }
    M[e] = m;
    S[e] = s;
}

constexpr int KRY_THREADS = 256;
constexpr int KRY_MAX_SYS = 128;  // systems per launch
constexpr int KRY_STAT = 40;      // status words of one problem (2 * 16 + 2 systems at most)

struct KrySys {
    double2 alpha, beta;  // system matrix alpha M + beta S
    const double2 *f;     // right-hand side
    double2 *x;           // solution
    int conj;             // 1: Hermitian CG, 0: COCG
    // disjoint objects: row i uses beta * bscale[vcomp[i]] (S has no entries
    // between objects, so the matrix stays complex symmetric); null: beta
    const double2 *bscale;
    int *stat;    // kmix_kernel: iteration count / status and relative residual
    double *res;
};

struct KryBatch {
    int nsys;
    const int *vcomp;  // object of each row (with KrySys::bscale)
    KrySys s[KRY_MAX_SYS];
};

__device__ __forceinline__ double2 dot_term(double2 a, double2 b, int conj) {
    // conj: conj(a) b, else a b
    return conj ? cd(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x) : cmul(a, b);
}

// Cluster-wide sum of three doubles.  Each warp reduces with shuffles, warp
// leaders write to `red`, thread 0 adds the warps and publishes the CTA sum
// in `slot`; after a cluster barrier lanes 0..cs-1 of warp 0 fetch the
// CTA sums of every rank through distributed shared memory and thread 0 adds
// them in rank order (the same order in every CTA, so all CTAs hold
// bit-identical sums).  The result is left in out[0..2] (shared memory),
// valid for every thread of the CTA after the final __syncthreads.
__device__ void cluster_sum3(cg::cluster_group &cl, double v0, double v1, double v2, double *red,
                             double *slot, double *gath, double *out) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
        v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    }
    if (lane == 0) {
        red[3 * wid] = v0;
        red[3 * wid + 1] = v1;
        red[3 * wid + 2] = v2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0, c = 0.0;
        for (int w = 0; w < nw; ++w) {
            a += red[3 * w];
            b += red[3 * w + 1];
            c += red[3 * w + 2];
        }
        slot[0] = a;
        slot[1] = b;
        slot[2] = c;
    }
    cl.sync();
    const unsigned cs = cl.num_blocks();
    if (threadIdx.x < cs) {
        const double *rem = cl.map_shared_rank(slot, threadIdx.x);
        gath[3 * threadIdx.x] = rem[0];
        gath[3 * threadIdx.x + 1] = rem[1];
        gath[3 * threadIdx.x + 2] = rem[2];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0, c = 0.0;
        for (unsigned r = 0; r < cs; ++r) {
            a += gath[3 * r];
            b += gath[3 * r + 1];
            c += gath[3 * r + 2];
        }
        out[0] = a;
        out[1] = b;
        out[2] = c;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(KRY_THREADS)
kry_kernel(const __grid_constant__ KryBatch batch, int n, const int *__restrict__ ptr, const int *__restrict__ col,
           const double *__restrict__ M, const double *__restrict__ S, double2 *__restrict__ work,
           double tol, int maxit, int *__restrict__ stat, double *__restrict__ res_out) {
    __shared__ double red[3 * 32];
    __shared__ double slotA[4], slotB[4], slotC[4];
    __shared__ double gath[3 * 16];
    __shared__ double sums[4];
    __shared__ double2 scal[2];  // alpha, beta of the current iteration
    __shared__ int flag;         // 0 continue, 1 converged, 2 breakdown
    cg::cluster_group cl = cg::this_cluster();
    const unsigned cs = cl.num_blocks();
    const unsigned rank = cl.block_rank();
    const int sid = blockIdx.x / cs;
    const KrySys sy = batch.s[sid];
    const int rows = (n + cs - 1) / cs;
    const int r0 = min(n, (int)rank * rows), r1 = min(n, r0 + rows);
    double2 *r = work + (5 * (size_t)sid + 0) * n;
    double2 *z = work + (5 * (size_t)sid + 1) * n;
    double2 *p = work + (5 * (size_t)sid + 2) * n;
    double2 *q = work + (5 * (size_t)sid + 3) * n;
    double2 *dinv = work + (5 * (size_t)sid + 4) * n;
    double2 *x = sy.x;
    const int cj = sy.conj;

    double v0 = 0.0, v1 = 0.0, v2 = 0.0;
    for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
        double md = 0.0, sd = 0.0;
        for (int e = ptr[i]; e < ptr[i + 1]; ++e)
            if (col[e] == i) { md = M[e]; sd = S[e]; }
        const double2 bi = sy.bscale ? cmul(sy.beta, sy.bscale[batch.vcomp[i]]) : sy.beta;
        const double2 d = cadd(cscale(sy.alpha, md), cscale(bi, sd));
        const double2 di = cdiv(cd(1.0, 0.0), d);
        const double2 b = sy.f[i];
        dinv[i] = di;
        x[i] = cd(0.0, 0.0);
        r[i] = b;
        const double2 zi = cmul(di, b);
        z[i] = zi;
        p[i] = zi;
        const double2 t = dot_term(b, zi, cj);
        v0 += t.x;
        v1 += t.y;
        v2 += cabs2(b);
    }
    cluster_sum3(cl, v0, v1, v2, red, slotA, gath, sums);
    double2 rho = cd(sums[0], sums[1]);
    const double bb = sums[2];
    double rr = bb;
    int its = 0, status = 0;  // 0 converged, 1 not converged, 2 breakdown
    if (bb > 0.0) {
        cl.sync();  // p complete everywhere
        status = 1;
        for (int it = 1; it <= maxit; ++it) {
            double w0 = 0.0, w1 = 0.0;
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
                double2 mp = cd(0.0, 0.0), sp = cd(0.0, 0.0);
                for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
                    const double2 pj = __ldcg(&p[col[e]]);
                    const double me = M[e], se = S[e];
                    mp.x += me * pj.x;
                    mp.y += me * pj.y;
                    sp.x += se * pj.x;
                    sp.y += se * pj.y;
                }
                const double2 bi = sy.bscale ? cmul(sy.beta, sy.bscale[batch.vcomp[i]]) : sy.beta;
                const double2 acc = cadd(cmul(sy.alpha, mp), cmul(bi, sp));
                q[i] = acc;
                const double2 t = dot_term(p[i], acc, cj);
                w0 += t.x;
                w1 += t.y;
            }
            cluster_sum3(cl, w0, w1, 0.0, red, slotB, gath, sums);
            if (threadIdx.x == 0) {
                const double2 pq = cd(sums[0], sums[1]);
                flag = (cabs2(pq) > 0.0) ? 0 : 2;
                scal[0] = flag ? cd(0.0, 0.0) : cdiv(rho, pq);
            }
            __syncthreads();
            if (flag) { status = 2; its = it; break; }
            const double2 al = scal[0];
            double u0 = 0.0, u1 = 0.0, u2 = 0.0;
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
                x[i] = cadd(x[i], cmul(al, p[i]));
                const double2 ri = csub(r[i], cmul(al, q[i]));
                r[i] = ri;
                const double2 zi = cmul(dinv[i], ri);
                z[i] = zi;
                const double2 t = dot_term(ri, zi, cj);
                u0 += t.x;
                u1 += t.y;
                u2 += cabs2(ri);
            }
            cluster_sum3(cl, u0, u1, u2, red, slotC, gath, sums);
            rr = sums[2];
            its = it;
            if (rr <= tol * tol * bb) { status = 0; break; }
            if (threadIdx.x == 0) {
                const double2 rn = cd(sums[0], sums[1]);
                flag = (cabs2(rho) > 0.0) ? 0 : 2;
                scal[1] = flag ? cd(0.0, 0.0) : cdiv(rn, rho);
                scal[0] = rn;
            }
            __syncthreads();
            if (flag) { status = 2; break; }
            const double2 be = scal[1];
            rho = scal[0];
            for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) p[i] = cadd(z[i], cmul(be, p[i]));
            cl.sync();
        }
    } else {
        rr = 0.0;
    }
    cl.sync();  // keep shared memory alive until every CTA has read it
    if (rank == 0 && threadIdx.x == 0) {
        stat[sid] = status == 0 ? its : (status == 1 ? -its : -1000000 - its);
        res_out[sid] = bb > 0.0 ? sqrt(rr / bb) : 0.0;
    }
}

// ---- mixed-precision refinement ---------------------------------------------
// The same systems (alpha M + beta S) w = f, solved by iterative refinement:
// an FP32 Jacobi-CG/COCG solve of A d = r, with r scaled to unit norm, reduces
// the residual by up to 2e-6; then the FP64 solution is updated, x += d,
// and the FP64 residual r = f - A x decides: stop when |r| <= tol |f| (the
// criterion of kry_kernel, here on the true residual), else refine again.
// Most arithmetic runs on the FP32 pipe, which on this part issues 64 times
// the FP64 rate; a refinement costs one FP64 product.  Refinement converges
// while cond(D^-1 A) * 2^-24 stays well below one (the OSRC and mass systems
// sit near cond 10..100); a refinement that fails to halve the residual norm
// ends the solve as not converged.
//
// An iteration is latency: about 15 flops per matrix entry between
// cluster-wide sums.  So a thread keeps one row (RPT rows) of A in registers,
// every CTA holds z = D^-1 r of the rows that its columns name in its own
// shared memory, and an iteration has two waits, those of its two sums: z is
// sent with the sum (r, z), and after it q = A p follows from A z and the
// recurrences p = z + beta p, q = A z + beta q, so the search direction is
// never sent.  What crosses between CTAs (z of the rows that another CTA's
// columns name, the CTAs' sums) goes by st.async, whose bytes the receiver's
// mbarrier counts: no fence and no cluster barrier in the iteration (a release
// at cluster scope cost 1000 to 2000 cycles a sum).  Rows are numbered by
// reverse Cuthill-McKee (d_ms_perm), so that a CTA's columns lie mostly in
// itself and its neighbours.  A system that fits one CTA needs no cluster.
// One preconditioner apply (10 systems; before: three cluster barriers an
// iteration, the search direction in L2, entries in shared memory): Fibonacci
// spheres of 10242 vertices 0.40 ms (0.76), 2562 0.28 (0.71), 642 0.26 (0.56), 150
// 0.10 (0.17).
// most threads with one row each (80 registers; in a cluster 180 bytes of spill
// stores and 124 of loads, alone none) and with two (96; 452 and 336, alone 200 and
// 148)
constexpr int KMIX_THREADS1 = 768, KMIX_THREADS2 = 640;
constexpr float KMIX_MIN_TOL = 2e-6f;      // most a FP32 solve reduces the residual by
constexpr int KMIX_MAX_REFINE = 40;
constexpr int KMIX_MAX_N = 25600;          // rows (below 2^16: the column places are 16 bits)
constexpr int KMIX_SMEM_MAX = 224 * 1024;  // bytes of z and of the long rows' entries

// Sum of NV <= 4 values over the warp by halving (each exchange hands half of
// the values to the other lane: 6 shuffles for 3 or 4 values instead of 5 per
// value): lane l < 4 ends with value kmix_slot(l).
__device__ __forceinline__ int kmix_slot(int lane) { return 2 * (lane & 1) + ((lane >> 1) & 1); }

template <typename T, int NV>
__device__ __forceinline__ T kmix_wsum(const T (&v)[NV], int lane) {
    const T v0 = v[0], v1 = NV > 1 ? v[NV > 1 ? 1 : 0] : T(0), v2 = NV > 2 ? v[NV > 2 ? 2 : 0] : T(0);
    T a;
    if (NV > 2) {  // lane bit 0: values {2, 3} (3 is zero), else {0, 1}
        const bool o = lane & 1, h = lane & 2;
        const T k0 = (o ? v2 : v0) + __shfl_xor_sync(0xffffffffu, o ? v0 : v2, 1);
        const T k1 = (o ? T(0) : v1) + __shfl_xor_sync(0xffffffffu, o ? v1 : T(0), 1);
        a = (h ? k1 : k0) + __shfl_xor_sync(0xffffffffu, h ? k0 : k1, 2);
    } else if (NV == 2) {  // lane bit 1: value 1
        const bool h = lane & 2;
        a = (h ? v1 : v0) + __shfl_xor_sync(0xffffffffu, h ? v0 : v1, 2);
        a += __shfl_xor_sync(0xffffffffu, a, 1);
    } else {
        a = v0 + __shfl_xor_sync(0xffffffffu, v0, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
    }
    a += __shfl_xor_sync(0xffffffffu, a, 4);
    a += __shfl_xor_sync(0xffffffffu, a, 8);
    a += __shfl_xor_sync(0xffffffffu, a, 16);
    return a;
}

// One cluster-wide sum's mailbox: warp 0 of every CTA sends the CTA's sums to
// slot[.][its rank] of each CTA of the cluster (st.async, counted in bytes by
// that CTA's mbarrier); every thread waits for its own CTA's mbarrier, whose
// one arrival is thread 0's with the bytes expected.  A box is used again only
// after another box's sum, which every CTA enters after it has read this one.
template <typename T, int NV>
struct KmixBox {
    uint64_t bar;
    T slot[NV][16];
    T wred[NV][32];  // the CTA's warp sums
};

#ifndef OSRC_KMIX_TIMEOUT_NS  // (tests of the give-up path set a short one)
#define OSRC_KMIX_TIMEOUT_NS 2000000000ULL
#endif
constexpr unsigned long long KMIX_TIMEOUT_NS = OSRC_KMIX_TIMEOUT_NS;
constexpr unsigned long long KMIX_DRAIN_NS = 1000000ULL;

__device__ __forceinline__ unsigned long long kmix_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// the CTA's threads that have given up the present wait
struct KmixCount {
    int *p;
    __device__ int load() const { return *(volatile int *)p; }
    __device__ void add() const { atomicAdd(p, 1); }
    __device__ bool cas(int e, int v) const { return atomicCAS(p, e, v) == e; }
};

// waits for phase `parity`, at most KMIX_TIMEOUT_NS of global time; the same
// result in every thread of the CTA
__device__ __forceinline__ bool kmix_wait(uint32_t bar, uint32_t parity, int *gave) {
    return bounded_wait(
        [&] {
            uint32_t done;
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(done)
                : "r"(bar), "r"(parity)
                : "memory");
            return done != 0;
        },
        kmix_ns, KmixCount{gave}, blockDim.x, KMIX_TIMEOUT_NS);
}

// store to the cluster's shared memory, its bytes counted by the mbarrier bar
// of the same CTA
__device__ __forceinline__ void kmix_send(uint32_t a, uint32_t bar, float v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
                 "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void kmix_send(uint32_t a, uint32_t bar, double v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void kmix_send(uint32_t a, uint32_t bar, float2 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(a),
                 "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ uint32_t kmix_mapa(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// Sums of NV values over the cluster (CL) or CTA, identical in every thread of
// every CTA: the warps' sums meet in shared memory, warp 0 (CL; else every
// warp) adds them, and the ranks' sums are added in the same order everywhere.
// parity: phase of the box's next use, flipped here; extra: bytes that other
// CTAs send with this sum besides the sums.  False, in every thread of the CTA,
// when the wait gave up: v is not a sum then, and the CTA goes to kmix_meet.
template <bool CL, typename T, int NV>
__device__ __forceinline__ bool kmix_csum(unsigned cs, unsigned rank, T (&v)[NV], KmixBox<T, NV> *box, uint32_t &parity,
                                          uint32_t extra, int *gave) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int k = kmix_slot(lane);
    T a = kmix_wsum<T, NV>(v, lane);
    if (lane < 4 && k < NV) box->wred[k][wid] = a;
    __syncthreads();
    if (!CL || wid == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = lane < nw ? box->wred[i][lane] : T(0);
        a = kmix_wsum<T, NV>(v, lane);
    }
    if (CL) {
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&box->bar);
        if (wid == 0) {
            if (lane == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                             "r"((uint32_t)(cs * NV * sizeof(T)) + extra)
                             : "memory");
            const uint32_t to = min((unsigned)lane, cs - 1);
            const uint32_t rbar = kmix_mapa(bar, to);
            const uint32_t rslot = kmix_mapa((uint32_t)__cvta_generic_to_shared(&box->slot[0][rank]), to);
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const T w = __shfl_sync(0xffffffffu, a, (i >> 1) | ((i & 1) << 1));
#ifdef OSRC_KMIX_MUTE  // tests: sums that a rank leaves out
                if (OSRC_KMIX_MUTE(rank, to, i)) continue;
#endif
                if ((unsigned)lane < cs) kmix_send(rslot + (uint32_t)(i * 16 * sizeof(T)), rbar, w);
            }
        }
        const bool here = kmix_wait(bar, parity, gave);
        __syncwarp();
        if (!here) return false;
        parity ^= 1u;
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = (unsigned)lane < cs ? box->slot[i][lane] : T(0);
        a = kmix_wsum<T, NV>(v, lane);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = __shfl_sync(0xffffffffu, a, (i >> 1) | ((i & 1) << 1));
    return true;
}

// A cluster barrier, the nth of this kernel, at which CTAs that go on (lost
// false) learn of those that gave up a wait (lost true): true when any has.  The
// latter leave n in every CTA's word `lost_at` before they arrive.  A CTA that
// gives up has no further barrier before this one, and whichever the others come
// to next (x published, the end; a CTA that waits for the lost one's sums gives
// up itself) is the same nth, so all of them leave together, none writes to a CTA
// that is gone, and a word written for a later barrier (n + 1 by a CTA that has
// gone on already) is not taken for this one's.  Copies still on their way have
// been issued by then: they get KMIX_DRAIN_NS, a thousand times a copy's latency,
// to land before the CTAs exit.
__device__ __forceinline__ bool kmix_meet(cg::cluster_group &cl, unsigned cs, int n, bool lost, int *lost_at) {
    if (lost && threadIdx.x < cs) *(volatile int *)cl.map_shared_rank(lost_at, threadIdx.x) = n;
    cl.sync();
    const int at = *(volatile int *)lost_at;
    if (at == 0 || at > n) return false;
    for (const unsigned long long t0 = kmix_ns(); kmix_ns() - t0 < KMIX_DRAIN_NS;) {}
    return true;
}

__device__ __forceinline__ float2 f2mul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 f2dot(float2 a, float2 b, int conj) {
    return conj ? make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x) : f2mul(a, b);
}
// a / b with an approximate reciprocal (PTX rcp.approx, 1 ulp: the same bits in
// every CTA).  It serves an iteration's scalars, which steer the search and enter
// x and r alike: a preconditioner apply's error against a direct FP64 solve is
// 5e-11 at 10242 vertices and 2.6e-10 at 642, with divisions the same to the
// iteration (7e-11, 2.4e-10), but every warp forms them, and with `/` an apply on
// 642 rows takes 288 us instead of 273.
__device__ __forceinline__ float2 f2div(float2 a, float2 b) {
    float ri;
    asm("rcp.approx.f32 %0, %1;" : "=f"(ri) : "f"(b.x * b.x + b.y * b.y));
    return make_float2((a.x * b.x + a.y * b.y) * ri, (a.y * b.x - a.x * b.y) * ri);
}
// 1 / a to about 48 bits, one Newton step from the FP32 reciprocal (where that is
// within its range; beyond it the iteration's FP32 products leave theirs as well):
// an FP64 division per row, or a branch to one, takes 8 us of a 270 us apply on
// 642 rows
__device__ __forceinline__ double kmix_rcp(double a) {
    const double r = 1.0f / (float)a;
    return a > 1e-36 && a < 1e36 ? fma(r, fma(-a, r, 1.0), r) : r;
}
// an entry m + beta s: formed in FP64 and rounded once (the terms cancel where a
// shifted system comes near singular: with entries 1e-6 of their terms' size 2
// refinements reach 1e-10, from terms rounded to FP32 6).  The systems that come
// here have alpha 1 (launch_kry): a factor tested in the kernel takes 12 us of a
// 270 us apply on 642 rows.
__device__ __forceinline__ double2 kmix_entry(double2 beta, double m, double s) {
    return cd(fma(beta.x, s, m), beta.y * s);
}
// a b + c
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}

// One cluster (CL) or CTA per system; CTA rank r owns the rows perm[r rows ..
// (r + 1) rows).  Dynamic shared memory: z by row number (the CTA's own rows
// and those its columns name), then the entries of its rows past the KMIX_E
// that a thread holds, and their columns' places (long_cap of each).  One such
// row sets an iteration's time: a preconditioner apply on a UV sphere with poles
// of degree 64 (1986 vertices) takes 1.58 ms with them in shared memory and took
// 3.33 when each iteration read them from the FP64 matrices, a Menger sponge with
// 40 % rows of 9 to 11 entries (896 vertices) 0.32 and 0.47.
// sy.x holds the published FP64 solution.  Status and residual as kry_kernel; the
// iteration count is the number of FP32 iterations over all refinements.
template <int RPT, bool CL>
__global__ void __launch_bounds__(RPT == 1 ? KMIX_THREADS1 : KMIX_THREADS2, 1)
kmix_kernel(const __grid_constant__ KryBatch batch, int n, const int *__restrict__ ptr, const int *__restrict__ col,
            const double *__restrict__ M, const double *__restrict__ S, const int *__restrict__ perm,
            const int *__restrict__ inv, int long_cap, double tol, int maxit) {
    extern __shared__ __align__(16) float2 zs[];
    float2 *la = zs + n;
    uint16_t *lc = reinterpret_cast<uint16_t *>(la + long_cap);
    // the sums of an iteration, of a refinement's start, of its end and of the
    // start: boxes of their own, so that none is written before the barrier
    // after its last reading
    __shared__ KmixBox<float, 2> boxP;
    __shared__ KmixBox<float, 3> boxR, boxI;
    __shared__ KmixBox<double, 1> boxD, boxB;
    __shared__ int s_gave, s_lost, s_cnt, s_long;
    uint32_t phP = 0, phR = 0, phI = 0, phD = 0, phB = 0;
    cg::cluster_group cl = cg::this_cluster();
    const unsigned cs = CL ? cl.num_blocks() : 1u, rank = CL ? cl.block_rank() : 0u;
    const KrySys &sy = batch.s[blockIdx.x / cs];
    const int rows = (n + (int)cs - 1) / (int)cs;
    const int r0 = min(n, (int)rank * rows), r1 = min(n, r0 + rows);
    double2 *xg = sy.x;
    const int cj = sy.conj;
    if (threadIdx.x == 0) {
        s_gave = s_lost = s_long = 0;
        if (CL) {
            uint64_t *bars[5] = {&boxP.bar, &boxR.bar, &boxI.bar, &boxD.bar, &boxB.bar};
            for (uint64_t *b : bars)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(b)),
                             "r"(1));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    if (CL) cl.sync();  // every CTA of the cluster runs, its barriers initialised
    else __syncthreads();
    const uint32_t zbase = (uint32_t)__cvta_generic_to_shared(zs);
    const uint32_t barR = (uint32_t)__cvta_generic_to_shared(&boxR.bar);
    const uint32_t barI = (uint32_t)__cvta_generic_to_shared(&boxI.bar);

    // per row: the FP64 residual, the FP32 state and the row of A with the
    // places of its columns' z (the FP64 solution lives in sy.x, the right-hand
    // side is read again when needed); who: the other ranks that need its z,
    // which are the owners of its columns (the pattern is symmetric)
    int row[RPT], nlong[RPT], at[RPT];  // entries past KMIX_E, the first one's place in la, lc
    uint32_t who[RPT];
    bool ok[RPT];
    double2 r64[RPT];
    float2 a[RPT][KMIX_E];
    uint16_t ad[RPT][KMIX_E];
    float2 dinv[RPT], d[RPT], r[RPT], z[RPT], p[RPT], q[RPT];
    for (int i = threadIdx.x; i < n; i += blockDim.x) zs[i] = make_float2(0.f, 0.f);
    __syncthreads();
    double bb = 0.0;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        const int li = threadIdx.x + k * blockDim.x, i = r0 + li;
        ok[k] = i < r1;
        row[k] = ok[k] ? perm[i] : 0;
        nlong[k] = at[k] = 0;
        r64[k] = cd(0.0, 0.0);
        dinv[k] = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < KMIX_E; ++e) {
            a[k][e] = make_float2(0.f, 0.f);
            ad[k][e] = 0;
        }
        who[k] = 0;
        if (ok[k]) {
            const double2 b64 = sy.bscale ? cmul(sy.beta, sy.bscale[batch.vcomp[row[k]]]) : sy.beta;
            const int p0 = ptr[row[k]], deg = ptr[row[k] + 1] - p0;
            double2 dg = cd(0.0, 0.0);
#pragma unroll
            for (int e = 0; e < KMIX_E; ++e)
                if (e < deg) {
                    const int c = col[p0 + e];
                    const double2 ae = kmix_entry(b64, M[p0 + e], S[p0 + e]);
                    a[k][e] = make_float2((float)ae.x, (float)ae.y);
                    const int ci = inv[c];
                    ad[k][e] = (uint16_t)ci;
                    who[k] |= 1u << (ci / rows);
                    if (CL && ci / rows != (int)rank) zs[ci].x = 1.f;  // mark: sent by its owner
                    if (c == row[k]) dg = ae;
                }
            if (deg > KMIX_E) {
                nlong[k] = deg - KMIX_E;
                at[k] = atomicAdd(&s_long, nlong[k]);
                for (int e = 0; e < nlong[k]; ++e) {
                    const int pe = p0 + KMIX_E + e, ci = inv[col[pe]];
                    const double2 ae = kmix_entry(b64, M[pe], S[pe]);
                    la[at[k] + e] = make_float2((float)ae.x, (float)ae.y);
                    lc[at[k] + e] = (uint16_t)ci;
                    who[k] |= 1u << (ci / rows);
                    if (CL && ci / rows != (int)rank) zs[ci].x = 1.f;
                    if (col[pe] == row[k]) dg = ae;
                }
            }
            who[k] &= ~(1u << rank);
            const double ri = kmix_rcp(cabs2(dg));
            dinv[k] = make_float2((float)(dg.x * ri), (float)(-dg.y * ri));
            r64[k] = sy.f[row[k]];
            bb += cabs2(r64[k]);
        }
    }
    // bytes of z that the other CTAs send with each sum (r, z)
    uint32_t zbytes = 0;
    if (CL) {
        __syncthreads();
        int cnt = 0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            cnt += zs[i].x != 0.f;
            zs[i] = make_float2(0.f, 0.f);
        }
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();
        if (cnt) atomicAdd(&s_cnt, cnt);
        __syncthreads();
        zbytes = 8u * (uint32_t)s_cnt;
    }
    // z of row k to the CTA's own copy and to the CTAs that need it
    auto publish = [&](int k, uint32_t bar) {
        const int ci = r0 + threadIdx.x + k * blockDim.x;
        zs[ci] = z[k];
        if (CL)
            for (uint32_t w = who[k]; w; w &= w - 1) {
                const uint32_t to = __ffs(w) - 1;
                kmix_send(kmix_mapa(zbase + 8u * (uint32_t)ci, to), kmix_mapa(bar, to), z[k]);
            }
    };
    bool lost = false, left = false;  // a wait gave up, here or (left) anywhere; both the same in the whole CTA
    int meets = 0;
    {   // its wait also ends the other CTAs' clearing of their copies
        double v[1] = {bb};
        lost = !kmix_csum<CL, double, 1>(cs, rank, v, &boxB, phB, 0u, &s_gave);
        bb = v[0];
    }
    double rr = bb;
    int its = 0, status = 0;  // 0 converged, 1 not converged, 2 breakdown
    if (!lost && bb > 0.0) {
        status = 1;
        for (int ref = 0; ref < KMIX_MAX_REFINE && its < maxit; ++ref) {
            // FP32 solve of A d = r / |r|
            const double sc = 1.0 / sqrt(rr);
            // the reduction still needed, taken in one solve where FP32 can
            // reach it (with a margin, so that the FP64 residual passes), else
            // split evenly between this solve and the next
            const double need = tol * sqrt(bb) * sc;
            const float itol = (float)(need >= 1e-5 ? fmin(0.3 * need, 0.5) : fmax((double)KMIX_MIN_TOL, 0.5 * sqrt(need)));
            float v3[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
                r[k] = make_float2((float)(r64[k].x * sc), (float)(r64[k].y * sc));
                z[k] = f2mul(dinv[k], r[k]);
                p[k] = q[k] = d[k] = make_float2(0.f, 0.f);
                if (ok[k]) {
                    publish(k, barI);
                    const float2 t = f2dot(r[k], z[k], cj);
                    v3[0] += t.x;
                    v3[1] += t.y;
                    v3[2] += r[k].x * r[k].x + r[k].y * r[k].y;
                }
            }
            lost = !kmix_csum<CL, float, 3>(cs, rank, v3, &boxI, phI, zbytes, &s_gave);  // also publishes z
            if (lost) break;
            float2 rho = make_float2(v3[0], v3[1]), be = make_float2(0.f, 0.f);
            const float rr0 = v3[2];
            bool brk = false;
            while (its < maxit) {
                // p = z + beta p, q = A z + beta q
                float v2[2] = {0.f, 0.f};
#pragma unroll
                for (int k = 0; k < RPT; ++k) {
                    p[k] = f2fma(be, p[k], z[k]);
                    float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
                    for (int e = 0; e < KMIX_E; e += 2) {
                        s0 = f2fma(a[k][e], zs[ad[k][e]], s0);
                        s1 = f2fma(a[k][e + 1], zs[ad[k][e + 1]], s1);
                    }
#pragma unroll 4
                    for (int e = 0; e < nlong[k]; ++e) s0 = f2fma(la[at[k] + e], zs[lc[at[k] + e]], s0);
                    q[k] = f2fma(be, q[k], make_float2(s0.x + s1.x, s0.y + s1.y));
                    if (ok[k]) {
                        const float2 t = f2dot(p[k], q[k], cj);
                        v2[0] += t.x;
                        v2[1] += t.y;
                    }
                }
                lost = !kmix_csum<CL, float, 2>(cs, rank, v2, &boxP, phP, 0u, &s_gave);  // every CTA has read its columns
                if (lost) break;
                const float2 pq = make_float2(v2[0], v2[1]);
                if (!(pq.x * pq.x + pq.y * pq.y > 0.f)) { brk = true; break; }
                const float2 al = f2div(rho, pq), mal = make_float2(-al.x, -al.y);
                float w3[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < RPT; ++k) {
                    d[k] = f2fma(al, p[k], d[k]);
                    r[k] = f2fma(mal, q[k], r[k]);
                    z[k] = f2mul(dinv[k], r[k]);
                    if (ok[k]) {
                        publish(k, barR);
                        const float2 t = f2dot(r[k], z[k], cj);
                        w3[0] += t.x;
                        w3[1] += t.y;
                        w3[2] += r[k].x * r[k].x + r[k].y * r[k].y;
                    }
                }
                lost = !kmix_csum<CL, float, 3>(cs, rank, w3, &boxR, phR, zbytes, &s_gave);
                if (lost) break;
                ++its;
                if (w3[2] <= itol * itol * rr0) break;
                if (!(rho.x * rho.x + rho.y * rho.y > 0.f)) { brk = true; break; }
                const float2 rz = make_float2(w3[0], w3[1]);
                be = f2div(rz, rho);
                rho = rz;
            }
            if (lost) break;
            if (brk) { status = 2; break; }
            // FP64 update and residual
            const double back = sqrt(rr);
#pragma unroll
            for (int k = 0; k < RPT; ++k)
                if (ok[k]) {
                    const double2 dx = cd((double)d[k].x * back, (double)d[k].y * back);
                    xg[row[k]] = ref ? cadd(xg[row[k]], dx) : dx;
                }
            if (!CL) __syncthreads();
            else if ((left = kmix_meet(cl, cs, ++meets, false, &s_lost))) break;  // x published
            double rn = 0.0;
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
                if (!ok[k]) continue;
                const int i = row[k];
                double2 mx = cd(0.0, 0.0), sx = cd(0.0, 0.0);
                for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
                    const double2 xj = __ldcg(&xg[col[e]]);
                    const double me = M[e], se = S[e];
                    mx.x += me * xj.x;
                    mx.y += me * xj.y;
                    sx.x += se * xj.x;
                    sx.y += se * xj.y;
                }
                const double2 bi = sy.bscale ? cmul(sy.beta, sy.bscale[batch.vcomp[i]]) : sy.beta;
                r64[k] = csub(sy.f[i], cadd(mx, cmul(bi, sx)));
                rn += cabs2(r64[k]);
            }
            double v[1] = {rn};
            lost = !kmix_csum<CL, double, 1>(cs, rank, v, &boxD, phD, 0u, &s_gave);
            if (lost) break;
            const double rprev = rr;
            rr = v[0];
            if (rr <= tol * tol * bb) { status = 0; break; }
            if (!(rr <= 0.25 * rprev)) break;  // refinement stagnates (or NaN): not converged
        }
    } else if (!lost) {
        rr = 0.0;
#pragma unroll
        for (int k = 0; k < RPT; ++k)
            if (ok[k]) xg[row[k]] = cd(0.0, 0.0);
    }
    // the end: shared memory stays until every CTA has read it
    if (CL && !left) left = kmix_meet(cl, cs, ++meets, lost, &s_lost);
    if (rank == 0 && threadIdx.x == 0) {
        *sy.stat = left ? KRY_LOST : status == 0 ? its : (status == 1 ? -its : -1000000 - its);
        *sy.res = bb > 0.0 ? sqrt(rr / bb) : 0.0;
    }
}

// y = M u on both block rows (turns a strong-form vector into the weak one)
__global__ void mass_spmv_kernel(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                                 const double *__restrict__ M, const double2 *__restrict__ u,
                                 double2 *__restrict__ y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 a = cd(0, 0), b = cd(0, 0);
    for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
        const int j = col[e];
        a = cadd(a, cscale(u[j], M[e]));
        b = cadd(b, cscale(u[n + j], M[e]));
    }
    y[i] = a;
    y[n + i] = b;
}

struct OsrcComb {
    int np;
    double2 ik, iik;  // i k and 1/(i k)
    const double2 *ik_obj;  // disjoint objects: i k of each object (else ik)
    const int *vcomp;
    double2 cu;       // C0 + sum_j A_j / B_j
    double2 g0;
    double2 a[16];    // A_j / B_j
    double2 g[16];
};

constexpr int OSRC_COMB_RUNS = 16;  // workspaces per launch
struct OsrcCombRuns {
    const double2 *sol[OSRC_COMB_RUNS];
    double2 *z[OSRC_COMB_RUNS];
};

// sol[0] = u1 = M^-1 y1, sol[1..np] = v_j, sol[np+1] = v'_0, sol[np+2..2np+1] = v'_j:
//   z1 = i k [(C0 + sum_j A_j/B_j) u1 - sum_j (A_j/B_j) v_j]   (blockIdx.y 0)
//   z2 = [g0 v'_0 + sum_j g_j v'_j] / (i k)                   (blockIdx.y 1)
// One thread per entry and block row, small blocks: FP64 chains are slow on
// this part, and a thread with both block rows in blocks of 256 took 8.4 us
// on 642 vertices.
__global__ void osrc_combine_kernel(int n, const __grid_constant__ OsrcComb c, const __grid_constant__ OsrcCombRuns v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 *sol = v.sol[blockIdx.z];
    double2 *z = v.z[blockIdx.z];
    const double2 ik = c.ik_obj ? c.ik_obj[c.vcomp[i]] : c.ik;
    if (blockIdx.y == 0) {
        double2 a = cmul(c.cu, sol[i]);
        for (int j = 0; j < c.np; ++j) a = csub(a, cmul(c.a[j], sol[(size_t)(1 + j) * n + i]));
        z[i] = cmul(ik, a);
    } else {
        const double2 iik = c.ik_obj ? cdiv(cd(1.0, 0.0), ik) : c.iik;
        double2 b = cmul(c.g0, sol[(size_t)(c.np + 1) * n + i]);
        for (int j = 0; j < c.np; ++j) b = cadd(b, cmul(c.g[j], sol[(size_t)(c.np + 2 + j) * n + i]));
        z[n + i] = cmul(iik, b);
    }
}

// Largest cluster the kernels may use on each device: 16 CTAs (a
// non-portable size that the kernel opts into) if the device can schedule
// it, else 8; 0 until kry_opt_in has run on that device.
int g_kry_max_cluster[OSRC_MAX_DEVICES] = {};

int kry_opt_in() {
    static PerDeviceOnce once;
    return per_device_once(once, [](int dev) -> int {
        g_kry_max_cluster[dev] = 8;
        if (cudaFuncSetAttribute(kry_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            (void)cudaGetLastError();
            return (int)OSRC_OK;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16, 1, 1);
        cfg.blockDim = dim3(KRY_THREADS, 1, 1);
        int size = 0;
        if (cudaOccupancyMaxPotentialClusterSize(&size, kry_kernel, &cfg) == cudaSuccess && size >= 16)
            g_kry_max_cluster[dev] = 16;
        (void)cudaGetLastError();
        return (int)OSRC_OK;
    });
}

// CTAs per system: about 640 rows each, at most the device's largest
// cluster (call after kry_opt_in).
int cluster_size_for(int n) {
    int dev = 0;
    const int mx = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < OSRC_MAX_DEVICES &&
                           g_kry_max_cluster[dev] > 0
                       ? g_kry_max_cluster[dev]
                       : 8;
    int cs = (n + 639) / 640;
    if (cs < 1) cs = 1;
    if (cs > mx) cs = mx;
    return cs;
}

// Launch shape of kmix_kernel for nsys systems of n rows: cluster size, rows
// per thread, threads; cs = 0: not usable (too many rows, or no cluster of that
// shape fits the device).  Among the cluster sizes the one with the smallest
// estimate is taken: the time of an iteration, measured as 0.85 us (one CTA) or
// 1.85 us (cluster) of sums plus 1.3 ns per row of a CTA, times the load of the
// device beyond one wave (the average system takes about 0.6 of the hardest
// one's iterations and the hardest start first).
// Shared memory holds z and, where the mesh has rows of more than KMIX_E
// entries, what a CTA's rows have beyond them.
struct KmixPlan {
    int nsys = 0, cs = 0, rpt = 0, threads = 0, long_cap = 0;
};

size_t kmix_smem(int n, int long_cap) {
    return (size_t)n * sizeof(float2) + (size_t)long_cap * (sizeof(float2) + sizeof(uint16_t));
}

template <int RPT, bool CL>
int kmix_active_clusters(size_t smem, int cs, int threads, int *count) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    if (!CL) {
        int per_sm = 0, dev = 0, sms = 0;
        OSRC_CK(cudaGetDevice(&dev));
        OSRC_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        OSRC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kmix_kernel<RPT, CL>, threads,
                                                              cfg.dynamicSmemBytes));
        *count = per_sm * sms;
        return OSRC_OK;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(count, kmix_kernel<RPT, CL>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        *count = 0;
    }
    return OSRC_OK;
}

int kmix_plan(osrc_problem *pb, int nsys, KmixPlan *out) {
    *out = KmixPlan{};
    const int n = pb->nv;
    if (!pb->d_ms_perm.p || n > KMIX_MAX_N) return OSRC_OK;
    for (const auto &q : pb->kmix_plans)
        if (q[0] == nsys) {
            out->nsys = q[0];
            out->cs = q[1];
            out->rpt = q[2];
            out->threads = q[3];
            out->long_cap = q[4];
            return OSRC_OK;
        }
    static PerDeviceOnce once;
    static int max_cluster[OSRC_MAX_DEVICES] = {};
    OSRC_TRY(per_device_once(once, [](int dev) -> int {
        max_cluster[dev] = 8;
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        OSRC_CK(cudaFuncSetAttribute(kmix_kernel<1, false>, attr, KMIX_SMEM_MAX));
        OSRC_CK(cudaFuncSetAttribute(kmix_kernel<2, false>, attr, KMIX_SMEM_MAX));
        OSRC_CK(cudaFuncSetAttribute(kmix_kernel<1, true>, attr, KMIX_SMEM_MAX));
        OSRC_CK(cudaFuncSetAttribute(kmix_kernel<2, true>, attr, KMIX_SMEM_MAX));
        if (cudaFuncSetAttribute(kmix_kernel<1, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaFuncSetAttribute(kmix_kernel<2, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
            max_cluster[dev] = 16;
        (void)cudaGetLastError();
        return (int)OSRC_OK;
    }));
    int dev = 0;
    OSRC_CK(cudaGetDevice(&dev));
    KmixPlan best;
    best.nsys = nsys;
    double cost = 1e300;
    for (int cs = 1; cs <= max_cluster[dev]; ++cs) {
        const int rows = (n + cs - 1) / cs;
        const int rpt = rows <= KMIX_THREADS1 ? 1 : 2;
        const int threads = ((rows + rpt - 1) / rpt + 31) / 32 * 32;
        if (rpt == 2 && threads > KMIX_THREADS2) continue;
        int long_cap = 0;
        if (!pb->ms_long.empty())
            for (int r = 0; r < n; r += rows)
                long_cap = std::max(long_cap, pb->ms_long[std::min(n, r + rows)] - pb->ms_long[r]);
        const size_t smem = kmix_smem(n, long_cap);
        if (smem > (size_t)KMIX_SMEM_MAX) continue;
        int count = 0;
        auto active = cs == 1 ? (rpt == 1 ? kmix_active_clusters<1, false> : kmix_active_clusters<2, false>)
                              : (rpt == 1 ? kmix_active_clusters<1, true> : kmix_active_clusters<2, true>);
        OSRC_TRY(active(smem, cs, threads, &count));
        if (count < 1) continue;
        const double load = std::max(1.0, 0.6 * nsys / count);
        const double t = load * ((cs == 1 ? 0.85 : 1.85) + 1.3e-3 * rows);
        if (t < cost * (1.0 - 1e-9)) {
            cost = t;
            best.cs = cs;
            best.rpt = rpt;
            best.threads = threads;
            best.long_cap = long_cap;
        }
    }
    if (pb->kmix_plans.size() < 16) pb->kmix_plans.push_back({best.nsys, best.cs, best.rpt, best.threads, best.long_cap});
    *out = best;
    return OSRC_OK;
}

template <int RPT, bool CL>
int kmix_launch(osrc_problem *pb, const KryBatch &batch, const KmixPlan &pl, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(batch.nsys * pl.cs, 1, 1);
    cfg.blockDim = dim3(pl.threads, 1, 1);
    cfg.dynamicSmemBytes = kmix_smem(pb->nv, pl.long_cap);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = pl.cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CL ? 1 : 0;
    OSRC_CK(cudaLaunchKernelEx(&cfg, kmix_kernel<RPT, CL>, batch, pb->nv, (const int *)pb->d_ms_ptr.p,
                               (const int *)pb->d_ms_col.p, (const double *)pb->d_M.p, (const double *)pb->d_S.p,
                               (const int *)pb->d_ms_perm.p, (const int *)(pb->d_ms_perm.p + pb->nv), pl.long_cap,
                               pb->p.inner_tol, pb->p.inner_maxit));
    pb->launches++;
    return OSRC_OK;
}

static bool ranges_overlap(const double2 *a, const double2 *b, int n) {
    return a < b + n && b < a + n;
}

// One launch for the batch.  kmix_kernel starts the hardest systems (largest
// |beta|: closest to the stiffness matrix) first; kry_kernel, whose status
// words go by system number, takes the systems of one workspace in order.
int launch_kry(osrc_problem *pb, KryBatch &batch, cudaStream_t st) {
    const int n = pb->nv;
    KmixPlan pl;
    OSRC_TRY(kmix_plan(pb, batch.nsys, &pl));
    bool mix = pl.cs > 0;
    for (int k = 0; k < batch.nsys && mix; ++k)  // in-place systems (and alpha other than 1) stay on the FP64 kernel
        if (ranges_overlap(batch.s[k].f, batch.s[k].x, n) || batch.s[k].alpha.x != 1.0 || batch.s[k].alpha.y != 0.0)
            mix = false;
    if (mix) {
        std::stable_sort(batch.s, batch.s + batch.nsys,
                         [](const KrySys &a, const KrySys &c) { return cabs2(a.beta) > cabs2(c.beta); });
        if (pl.cs == 1) return pl.rpt == 1 ? kmix_launch<1, false>(pb, batch, pl, st) : kmix_launch<2, false>(pb, batch, pl, st);
        return pl.rpt == 1 ? kmix_launch<1, true>(pb, batch, pl, st) : kmix_launch<2, true>(pb, batch, pl, st);
    }
    OSRC_TRY(kry_opt_in());
    const int cs = cluster_size_for(n);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(batch.nsys * cs, 1, 1);
    cfg.blockDim = dim3(KRY_THREADS, 1, 1);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    OSRC_CK(cudaLaunchKernelEx(&cfg, kry_kernel, batch, n, (const int *)pb->d_ms_ptr.p,
                               (const int *)pb->d_ms_col.p, (const double *)pb->d_M.p,
                               (const double *)pb->d_S.p, pb->d_kry.p, pb->p.inner_tol,
                               pb->p.inner_maxit, batch.s[0].stat, batch.s[0].res));
    pb->launches++;
    return OSRC_OK;
}

// Reads back the inner solver status (one small copy; the caller's stream is
// synchronised) and turns non-convergence into a status code.
int check_kry(osrc_problem *pb, int nsys, cudaStream_t st) {
    int stat[KRY_STAT];
    OSRC_CK(cudaMemcpyAsync(stat, pb->d_kry_stat.p, nsys * sizeof(int), cudaMemcpyDeviceToHost, st));
    OSRC_CK(cudaStreamSynchronize(st));
    return kry_status_host(pb, stat, nsys);
}

}  // namespace

int ms_build(osrc_problem *pb, const std::vector<int> &cptr, const std::vector<int> &cidx,
             cudaStream_t st) {
    osrc_mesh *m = pb->mesh;
    osrc_ctx *ctx = m->ctx;
    const int nt = pb->nt, nnz = pb->ms_nnz;
    DBuf<double> bm, bs;
    DBuf<int> d_cptr, d_cidx;
    OSRC_TRY(bm.alloc(ctx, 9 * (size_t)nt));
    OSRC_TRY(bs.alloc(ctx, 9 * (size_t)nt));
    OSRC_TRY(d_cptr.alloc(ctx, cptr.size()));
    OSRC_TRY(d_cidx.alloc(ctx, cidx.size()));
    OSRC_TRY(pb->d_M.alloc(ctx, nnz));
    OSRC_TRY(pb->d_S.alloc(ctx, nnz));
    OSRC_CK(cudaMemcpyAsync(d_cptr.p, cptr.data(), cptr.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    OSRC_CK(cudaMemcpyAsync(d_cidx.p, cidx.data(), cidx.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    ms_element_kernel<<<(nt + 127) / 128, 128, 0, st>>>(nt, pb->d_tgeo.p, m->d_verts.p, m->d_tris.p,
                                                        bm.p, bs.p);
    csr_sum_kernel<<<(nnz + 255) / 256, 256, 0, st>>>(nnz, d_cptr.p, d_cidx.p, bm.p, bs.p, pb->d_M.p,
                                                      pb->d_S.p);
    pb->launches += 2;
    OSRC_CK(cudaGetLastError());
    // inner solver workspace: 2 N_Pade + 2 systems of 5 vectors, plus the
    // weak-form input and the solutions
    const int nsys = 2 * pb->p.n_pade + 2;
    OSRC_TRY(pb->d_kry.alloc(ctx, 5 * (size_t)nsys * pb->nv));
    OSRC_TRY(pb->d_kry_rhs.alloc(ctx, (size_t)(2 + nsys) * pb->nv));
    OSRC_TRY(pb->d_kry_stat.alloc(ctx, KRY_STAT));
    OSRC_TRY(pb->d_kry_res.alloc(ctx, KRY_STAT));
    OSRC_CK(cudaStreamSynchronize(st));
    return OSRC_OK;
}

static int mass_solve_async(osrc_problem *pb, const double2 *y, double2 *z, bool swap, int word, cudaStream_t st);

int mass_solve(osrc_problem *pb, const double2 *x, double2 *y, cudaStream_t st) {
    OSRC_TRY(mass_solve_async(pb, x, y, false, 0, st));
    return check_kry(pb, 2, st);
}

// z = P M^-1 y for a weak-form vector y = [y1; y2] (Sec. 2.4, 2.6, 2.7).
// With u = M^-1 y and X = -M^-1 S / k_eps^2 the Pade terms are rewritten so
// that no system waits for another:
//   X (1 + B_j X)^-1 u1 = (u1 - v_j) / B_j,  (M - B_j S / k_eps^2) v_j = y1
//   (1 + B X)^-1 u2 = (M - B S / k_eps^2)^-1 y2
// so the mass solve of row 1 and all 2 N_Pade + 1 shifted systems run as one
// batched launch (row 2 needs no mass solve at all).
int osrc_precond_nsys(const osrc_problem *pb) {
    // (Calderon: two mass solves of two systems each)
    return pb->p.precond == OSRC_PRECOND_OSRC ? 2 * pb->p.n_pade + 2 : pb->p.precond == OSRC_PRECOND_CALDERON ? 4 : 2;
}

// both block rows of M^-1 y; rows swapped in the output when swap is set; word:
// the first's status word
static void mass_systems(osrc_problem *pb, const double2 *y, double2 *z, bool swap, int word, KryBatch &b) {
    const int n = pb->nv;
    for (int k = 0; k < 2; ++k) {
        KrySys &s = b.s[b.nsys++];
        s = KrySys{};
        s.alpha = cd(1.0, 0.0);
        s.beta = cd(0.0, 0.0);
        s.f = y + (size_t)k * n;
        s.x = z + (size_t)(swap ? 1 - k : k) * n;
        s.conj = 1;
        s.stat = pb->d_kry_stat.p + word + k;
        s.res = pb->d_kry_res.p + word + k;
    }
}

static int mass_solve_async(osrc_problem *pb, const double2 *y, double2 *z, bool swap, int word, cudaStream_t st) {
    KryBatch b{};
    mass_systems(pb, y, z, swap, word, b);
    return launch_kry(pb, b, st);
}

int kry_status_host(osrc_problem *pb, const int *stat, int nsys) {
    int worst = 0;
    const int s = kry_stat_code(stat, nsys, &worst);
    if (s == OSRC_TIMEOUT) osrc_set_error("inner solve: a bounded wait gave up");
    if (s == OSRC_OK && worst > pb->inner_last_max) pb->inner_last_max = worst;
    return s;
}

int osrc_precond_fused(osrc_problem *pb, const double2 *y, double2 *z, cudaStream_t st) {
    OSRC_TRY(osrc_precond_fused_async(pb, y, z, st));
    return check_kry(pb, osrc_precond_nsys(pb), st);
}

// the 2 N_Pade + 2 systems of P M^-1 y, solutions after the weak-form input in
// d_kry_rhs
static void osrc_systems(osrc_problem *pb, const double2 *y, KryBatch &b) {
    const int n = pb->nv, np = pb->p.n_pade;
    const double2 ke2 = cmul(pb->k_eps, pb->k_eps);
    // disjoint objects: 1/k_eps^2 of each row's object via KrySys::bscale
    const double2 inv_ke2 = pb->multi ? cd(1.0, 0.0) : cdiv(cd(1.0, 0.0), ke2);
    const double2 *bscale = pb->multi ? pb->d_obj_ike.p + pb->mesh->ncomp : nullptr;
    double2 *sol = pb->d_kry_rhs.p + 2 * (size_t)n;
    const double2 *y1 = y, *y2 = y + n;
    b.vcomp = pb->mesh->d_vcomp.p;
    // solution k: 0 M u1 = y1 (Hermitian CG); 1..np DtN (M - B_j S / k_eps^2) v_j = y1;
    // np + 1 NtD (M - S / k_eps^2) v'_0 = y2; then NtD (M - B_j S / k_eps^2) v'_j = y2
    for (int k = 0; k < 2 * np + 2; ++k) {
        KrySys &s = b.s[b.nsys++];
        s = KrySys{};
        s.alpha = cd(1.0, 0.0);
        const int j = k <= np ? k - 1 : k - np - 2;  // Pade term (-1: none)
        s.beta = k == 0 ? cd(0.0, 0.0) : cscale(j < 0 ? inv_ke2 : cmul(pb->B[j], inv_ke2), -1.0);
        s.bscale = k == 0 ? nullptr : bscale;
        s.f = k <= np ? y1 : y2;
        s.x = sol + (size_t)k * n;
        s.conj = k == 0 ? 1 : 0;
        s.stat = pb->d_kry_stat.p + k;
        s.res = pb->d_kry_res.p + k;
    }
}

// z_r = P M^-1 y_r for nrun workspaces (the problem itself or clones of one
// problem): the systems of all of them in as few launches as they fit
// (KRY_MAX_SYS), so that the lockstep solve's right-hand sides fill the GPU
// together instead of one after the other.
int osrc_precond_fused_multi(osrc_problem *const *pbs, const double2 *const *ys, double2 *const *zs, int nrun,
                             cudaStream_t st) {
    osrc_problem *pb = pbs[0];
    const int n = pb->nv, np = pb->p.n_pade;
    if (pb->p.precond == OSRC_PRECOND_CALDERON) {
        // z = M^-1 B Pi M^-1 y: the first mass solve writes its rows swapped
        for (int r = 0; r < nrun; ++r) {
            osrc_problem *q = pbs[r];
            double2 *t = q->d_kry_rhs.p + 2 * (size_t)n, *w = q->d_tmp2.p + 2 * (size_t)n;
            OSRC_TRY(mass_solve_async(q, ys[r], t, true, 0, st));
            if (q->p.precision == OSRC_FP64_DENSE) OSRC_TRY(dense_apply(q, t, w, st));
            else OSRC_TRY(far_apply(q, t, w, OSRC_PART_ALL, st));
            OSRC_TRY(mass_solve_async(q, w, zs[r], false, 2, st));
        }
        return OSRC_OK;
    }
    const bool mass = pb->p.precond == OSRC_PRECOND_MASS;
    const int per = mass ? 2 : 2 * np + 2;
    int group = std::max(1, std::min(nrun, KRY_MAX_SYS / per));
    if (group > 1) {  // only the mixed kernel takes systems of several workspaces
        KmixPlan pl;
        OSRC_TRY(kmix_plan(pb, per * group, &pl));
        if (pl.cs == 0) group = 1;
    }
    for (int r0 = 0; r0 < nrun; r0 += group) {
        const int R = std::min(group, nrun - r0);
        KryBatch b{};
        for (int r = 0; r < R; ++r) {
            if (mass) mass_systems(pbs[r0 + r], ys[r0 + r], zs[r0 + r], false, 0, b);
            else osrc_systems(pbs[r0 + r], ys[r0 + r], b);
        }
        OSRC_TRY(launch_kry(pbs[r0], b, st));
    }
    if (mass) return OSRC_OK;
    OsrcComb c{};
    c.np = np;
    c.ik = cd(-pb->k_osrc_i, pb->k_osrc);  // i k_osrc (complex with attenuation)
    c.iik = cdiv(cd(1.0, 0.0), c.ik);
    c.ik_obj = pb->multi ? pb->d_obj_ike.p : nullptr;
    c.vcomp = pb->mesh->d_vcomp.p;
    double2 cu = pb->C0;
    for (int j = 0; j < np; ++j) {
        c.a[j] = cdiv(pb->A[j], pb->B[j]);
        cu = cadd(cu, c.a[j]);
        c.g[j] = pb->g[j];
    }
    c.cu = cu;
    c.g0 = pb->g0;
    for (int r0 = 0; r0 < nrun; r0 += OSRC_COMB_RUNS) {
        const int R = std::min((int)OSRC_COMB_RUNS, nrun - r0);
        OsrcCombRuns v{};
        for (int r = 0; r < R; ++r) {
            v.sol[r] = pbs[r0 + r]->d_kry_rhs.p + 2 * (size_t)n;
            v.z[r] = zs[r0 + r];
        }
        osrc_combine_kernel<<<dim3((n + 63) / 64, 2, R), 64, 0, st>>>(n, c, v);
        pbs[r0]->launches++;
        OSRC_CK(cudaGetLastError());
    }
    return OSRC_OK;
}

int osrc_precond_fused_async(osrc_problem *pb, const double2 *y, double2 *z, cudaStream_t st) {
    return osrc_precond_fused_multi(&pb, &y, &z, 1, st);
}

// P x for a strong-form vector x: P x = P M^-1 (M x).
int osrc_precond(osrc_problem *pb, const double2 *x, double2 *y, cudaStream_t st) {
    const int n = pb->nv;
    double2 *mx = pb->d_kry_rhs.p;
    mass_spmv_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, pb->d_ms_ptr.p, pb->d_ms_col.p, pb->d_M.p, x,
                                                      mx);
    pb->launches++;
    OSRC_CK(cudaGetLastError());
    return osrc_precond_fused(pb, mx, y, st);
}

// ---------------------------------------------------------------------------
// Allocation-free batched shifted solve.
//
// Some callers cannot call cudaMalloc at the point where they need a solve:
// code that runs while a stream is being captured into a CUDA graph (an
// allocation there breaks or invalidates the capture), real-time or
// callback-driven hosts that forbid allocation after start-up, and
// frameworks whose device memory is owned by their own pool allocator.
// osrc_shifted_solve_noalloc serves them: it runs the same cluster-batched
// CG / COCG kernel as the library's mass and OSRC solves, but its Krylov
// workspace is the file-scope array below instead of memory from
// cudaMalloc, so the call allocates nothing.  The caller owns every input
// and output buffer.
//
// The array holds NOALLOC_MAX_ENTRIES complex entries per Krylov vector
// (5 vectors, 10 MiB in total) on every GPU that loads this library, until
// the process exits.  Every call on a device shares it, and it keeps the
// last call's contents; the kernel writes each scratch entry before reading
// it, so only the per-system status words need clearing, which every call
// does.  Calls whose kernels overlap on the GPU (two streams, or two host
// threads) race on the array: serialise them.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t NOALLOC_MAX_ENTRIES = 131072;  // nsys * n complex values per vector
constexpr int NOALLOC_MAX_SYS = 16;

static __device__ __align__(256) double2 g_noalloc_work[5 * NOALLOC_MAX_ENTRIES];
static __device__ __align__(256) int g_noalloc_stat[NOALLOC_MAX_SYS];
static __device__ __align__(256) double g_noalloc_res[NOALLOC_MAX_SYS];

struct NoAllocScratch {
    double2 *work = nullptr;
    int *stat = nullptr;
    double *res = nullptr;
    unsigned long long ctx_id = 0;  // context the addresses belong to
    bool ready = false;
};

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;
NoAllocScratch g_noalloc[NOALLOC_MAX_DEVICES];

// Unique id of the context current on this host thread (driver entry
// points reached through the runtime, so no link against libcuda).  Ids are
// never reused, so a device reset, which replaces the primary context and
// with it the array's address, shows up as a new id.
typedef CUresult (*PfnCtxGetCurrent)(CUcontext *);
typedef CUresult (*PfnCtxGetId)(CUcontext, unsigned long long *);
int current_ctx_id(unsigned long long &id) {
    static PfnCtxGetCurrent get_cur = nullptr;
    static PfnCtxGetId get_id = nullptr;
    if (!get_cur || !get_id) {
        cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
        OSRC_CK(cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", (void **)&get_cur, 12000,
                                                 cudaEnableDefault, &q1));
        OSRC_CK(cudaGetDriverEntryPointByVersion("cuCtxGetId", (void **)&get_id, 12000,
                                                 cudaEnableDefault, &q2));
        if (q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !get_cur || !get_id) {
            osrc_set_error("driver entry points cuCtxGetCurrent / cuCtxGetId not found");
            return OSRC_UNSUPPORTED;
        }
    }
    CUcontext c = nullptr;
    if (get_cur(&c) != CUDA_SUCCESS || !c || get_id(c, &id) != CUDA_SUCCESS) {
        osrc_set_error("no current CUDA context");
        return OSRC_CUDA_ERROR;
    }
    return OSRC_OK;
}

// Device address of the scratch array on the current device.  Looked up
// with cudaGetSymbolAddress (that device current) on the first call on a
// device and again whenever the device's context has changed since (after
// cudaDeviceReset), so a kernel is never given an address of a context that
// no longer exists.
int noalloc_scratch(int dev, NoAllocScratch &out) {
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return OSRC_UNSUPPORTED;
    // makes the device's primary context current (created if needed)
    OSRC_CK(cudaSetDevice(dev));
    unsigned long long id = 0;
    OSRC_TRY(current_ctx_id(id));
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocScratch &s = g_noalloc[dev];
    if (!s.ready || s.ctx_id != id) {
        s.ready = false;
        OSRC_CK(cudaGetSymbolAddress((void **)&s.work, g_noalloc_work));
        OSRC_CK(cudaGetSymbolAddress((void **)&s.stat, g_noalloc_stat));
        OSRC_CK(cudaGetSymbolAddress((void **)&s.res, g_noalloc_res));
        s.ctx_id = id;
        s.ready = true;
    }
    out = s;
    return OSRC_OK;
}

}  // namespace

extern "C" int osrc_shifted_solve_noalloc(int n, const int32_t *row_ptr, const int32_t *col_idx,
                                          const double *M_vals, const double *S_vals, int nsys,
                                          const double *alpha, const double *beta, const void *f,
                                          void *w, double tol, int maxit, int conj,
                                          int *iters_out, void *stream) {
    if (n < 1 || nsys < 1 || nsys > NOALLOC_MAX_SYS || !row_ptr || !col_idx || !M_vals ||
        !S_vals || !alpha || !beta || !f || !w || !(tol > 0.0) || tol > 1e-4 || maxit < 1 ||
        (conj != 0 && conj != 1)) {
        osrc_set_error("osrc_shifted_solve_noalloc: invalid argument");
        return OSRC_INVALID_ARG;
    }
    if ((size_t)n * (size_t)nsys > NOALLOC_MAX_ENTRIES) {
        osrc_set_error("osrc_shifted_solve_noalloc: nsys * n exceeds the static scratch "
                       "capacity of 131072 complex entries");
        return OSRC_INVALID_ARG;
    }
    int dev = 0;
    OSRC_CK(cudaGetDevice(&dev));
    NoAllocScratch sc;
    OSRC_TRY(noalloc_scratch(dev, sc));
    cudaStream_t st = (cudaStream_t)stream;
    KryBatch b{};
    b.nsys = nsys;
    for (int s = 0; s < nsys; ++s) {
        b.s[s].alpha = cd(alpha[2 * s], alpha[2 * s + 1]);
        b.s[s].beta = cd(beta[2 * s], beta[2 * s + 1]);
        b.s[s].f = (const double2 *)f + (size_t)s * n;
        b.s[s].x = (double2 *)w + (size_t)s * n;
        b.s[s].conj = conj;
    }
    OSRC_TRY(kry_opt_in());
    // status words start as "not written" so that a failed launch is seen
    OSRC_CK(cudaMemsetAsync(sc.stat, 0x80, nsys * sizeof(int), st));
    const int cs = cluster_size_for(n);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nsys * cs, 1, 1);
    cfg.blockDim = dim3(KRY_THREADS, 1, 1);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    OSRC_CK(cudaLaunchKernelEx(&cfg, kry_kernel, b, n, (const int *)row_ptr, (const int *)col_idx,
                               M_vals, S_vals, sc.work, tol, maxit, sc.stat, sc.res));
    if (!iters_out) return OSRC_OK;
    OSRC_CK(cudaMemcpyAsync(iters_out, sc.stat, nsys * sizeof(int), cudaMemcpyDeviceToHost, st));
    OSRC_CK(cudaStreamSynchronize(st));
    int status = OSRC_OK;
    for (int s = 0; s < nsys; ++s) {
        if (iters_out[s] <= -1000000) status = OSRC_BREAKDOWN;
        else if (iters_out[s] < 0 && status == OSRC_OK) status = OSRC_NOT_CONVERGED;
    }
    return status;
}
