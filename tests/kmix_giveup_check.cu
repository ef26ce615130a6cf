// GPU check of the inner solver's give-up path: the library's kernel, compiled
// here with a wait limit of 5 ms and a rank that can be told to leave out sums
// that it owes the other blocks of its cluster.  Every sum of a solve is left out
// in turn, to all ranks, to one and to the rank itself, once or from then on: the
// kernel ends within its limits, reports the wait that gave up (never a converged
// system), and the next cluster's system and the next launch are undisturbed.
// Prints "ok <cases>" and exits 0, or reports the first violation and exits 1.
#include <chrono>
#include <cstdio>
#include <vector>

#define OSRC_KMIX_TIMEOUT_NS 5000000ULL
#define OSRC_KMIX_MUTE(rank, to, i) kmix_mute(rank, to, i)

static __device__ int g_rank, g_after, g_once, g_sums;
static __device__ unsigned g_to;

// called by warp 0 of every block for value i of a sum about to go to rank `to`
static __device__ bool kmix_mute(unsigned rank, unsigned to, int i) {
    unsigned cs;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cs));
    if (blockIdx.x / cs != 0 || (int)rank != g_rank) return false;
    int c = 0;
    if (threadIdx.x == 0) c = i == 0 ? atomicAdd(&g_sums, 1) : *(volatile int *)&g_sums - 1;
    c = __shfl_sync(0xffffffffu, c, 0);
    return (g_once ? c == g_after : c >= g_after) && (g_to >> to & 1);
}

#include "../paper_2104_04609_gb300/csrc/k_sparse.cu"

// what the library's other files hold
void osrc_set_error(const std::string &) {}
int ctx_alloc(osrc_ctx *, void **p, size_t) {
    *p = nullptr;
    return OSRC_OUT_OF_MEMORY;
}
void ctx_free(osrc_ctx *, void *, size_t) {}
int far_apply(osrc_problem *, const double2 *, double2 *, int, cudaStream_t) { return OSRC_UNSUPPORTED; }
int dense_apply(osrc_problem *, const double2 *, double2 *, cudaStream_t) { return OSRC_UNSUPPORTED; }

#define CK(c)                                                                              \
    do {                                                                                   \
        cudaError_t e_ = (c);                                                              \
        if (e_ != cudaSuccess) {                                                           \
            std::printf("FAIL line %d: %s: %s\n", __LINE__, #c, cudaGetErrorString(e_)); \
            return 1;                                                                      \
        }                                                                                  \
    } while (0)

template <class T>
static T *upload(const std::vector<T> &h) {
    T *d = nullptr;
    if (cudaMalloc(&d, h.size() * sizeof(T)) != cudaSuccess) return nullptr;
    cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}

// two systems M x = f, M a ring (2 on the diagonal, 0.45 beside it), n rows on cs CTAs
template <int RPT>
static int check(int n, int cs, int *cases, double *worst) {
    const int rows = (n + cs - 1) / cs, threads = ((rows + RPT - 1) / RPT + 31) / 32 * 32;
    std::vector<int> ptr(n + 1), col, id(n);
    std::vector<double> M, S;
    for (int i = 0; i < n; ++i) {
        id[i] = i;
        ptr[i + 1] = ptr[i] + 3;
        int c[3] = {(i + n - 1) % n, i, (i + 1) % n};
        std::sort(c, c + 3);
        for (int k : c) {
            col.push_back(k);
            M.push_back(k == i ? 2.0 : 0.45);
            S.push_back(0.0);
        }
    }
    std::vector<double2> x0(2 * (size_t)n), f(2 * (size_t)n), x(2 * (size_t)n);
    for (size_t i = 0; i < x0.size(); ++i) x0[i] = cd(1.0 + 0.3 * ((i * 7) % 11), 0.2 * ((i * 5) % 13) - 1.0);
    for (int s = 0; s < 2; ++s)
        for (int i = 0; i < n; ++i) {
            double2 v = cd(0, 0);
            for (int e = ptr[i]; e < ptr[i + 1]; ++e) v = cadd(v, cscale(x0[(size_t)s * n + col[e]], M[e]));
            f[(size_t)s * n + i] = v;
        }
    int *dptr = upload(ptr), *dcol = upload(col), *did = upload(id), *dstat = upload(std::vector<int>(2));
    double *dM = upload(M), *dS = upload(S), *dres = upload(std::vector<double>(2));
    double2 *df = upload(f), *dx = upload(x);
    if (!dptr || !dcol || !did || !dstat || !dM || !dS || !dres || !df || !dx) return std::printf("FAIL memory\n"), 1;
    KryBatch b{};
    b.nsys = 2;
    for (int s = 0; s < 2; ++s) {
        b.s[s].alpha = cd(1.0, 0.0);
        b.s[s].f = df + (size_t)s * n;
        b.s[s].x = dx + (size_t)s * n;
        b.s[s].conj = 1;
        b.s[s].stat = dstat + s;
        b.s[s].res = dres + s;
    }
    // stat of both systems, error of the solutions and the launch's time
    auto run = [&](int rank, int after, int once, unsigned to, int *stat, double *err, double *ms, int *sums) -> int {
        const int zero = 0;
        CK(cudaMemcpyToSymbol(g_rank, &rank, sizeof(int)));
        CK(cudaMemcpyToSymbol(g_after, &after, sizeof(int)));
        CK(cudaMemcpyToSymbol(g_once, &once, sizeof(int)));
        CK(cudaMemcpyToSymbol(g_to, &to, sizeof(unsigned)));
        CK(cudaMemcpyToSymbol(g_sums, &zero, sizeof(int)));
        CK(cudaMemset(dx, 0, x.size() * sizeof(double2)));
        CK(cudaDeviceSynchronize());
        const auto t0 = std::chrono::steady_clock::now();
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * cs, 1, 1);
        cfg.blockDim = dim3(threads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)n * sizeof(float2);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        CK(cudaLaunchKernelEx(&cfg, kmix_kernel<RPT, true>, b, n, (const int *)dptr, (const int *)dcol,
                              (const double *)dM, (const double *)dS, (const int *)did, (const int *)did, 0, 1e-10, 500));
        CK(cudaDeviceSynchronize());
        *ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        CK(cudaMemcpy(stat, dstat, 2 * sizeof(int), cudaMemcpyDeviceToHost));
        CK(cudaMemcpy(x.data(), dx, x.size() * sizeof(double2), cudaMemcpyDeviceToHost));
        CK(cudaMemcpyFromSymbol(sums, g_sums, sizeof(int)));
        for (int s = 0; s < 2; ++s) {
            err[s] = 0.0;
            for (int i = 0; i < n; ++i)
                err[s] = std::fmax(err[s], std::sqrt(cabs2(csub(x[(size_t)s * n + i], x0[(size_t)s * n + i]))));
        }
        return 0;
    };
    int stat[2], total = 0, sums;
    double err[2], ms;
    if (run(0, 1 << 30, 0, 0u, stat, err, &ms, &total)) return 1;
    if (stat[0] <= 0 || stat[1] <= 0 || err[0] > 1e-8 || err[1] > 1e-8 || total < 6)
        return std::printf("FAIL n %d: undisturbed solve: status %d %d, errors %g %g, %d sums\n", n, stat[0], stat[1],
                           err[0], err[1], total), 1;
    for (int rank = 0; rank < cs; rank += cs - 1)
        for (int once = 0; once < 2; ++once)
            for (int after = 0; after < total; ++after)
                for (unsigned to : {(1u << cs) - 1, 1u << rank, 1u << (rank + 1) % cs}) {
                    if (run(rank, after, once, to, stat, err, &ms, &sums)) return 1;
                    // a wait of 5 ms, once more where the others notice only then, and the landing time
                    if (stat[0] != KRY_LOST || stat[1] <= 0 || err[1] > 1e-8 || ms > 100.0)
                        return std::printf("FAIL n %d cs %d rank %d sum %d of %d to %x once %d: status %d %d, error %g, %.1f ms\n",
                                           n, cs, rank, after, total, to, once, stat[0], stat[1], err[1], ms), 1;
                    ++*cases;
                    *worst = std::max(*worst, ms);
                }
    if (run(0, 1 << 30, 0, 0u, stat, err, &ms, &sums)) return 1;
    if (stat[0] <= 0 || stat[1] <= 0 || err[0] > 1e-8 || err[1] > 1e-8) return std::printf("FAIL n %d: solve afterwards\n", n), 1;
    for (void *p : {(void *)dptr, (void *)dcol, (void *)did, (void *)dstat, (void *)dM, (void *)dS, (void *)dres, (void *)df, (void *)dx})
        cudaFree(p);
    return 0;
}

int main() {
    int cases = 0;
    double worst = 0.0;
    if (check<1>(60, 4, &cases, &worst) || check<1>(2000, 8, &cases, &worst) || check<2>(1500, 2, &cases, &worst)) return 1;
    std::printf("ok %d cases, longest launch %.1f ms\n", cases, worst);
    return 0;
}
