// GPU check of the mixed inner solver's matrix entries M + beta S where the
// two terms nearly cancel (to 1e-6 of their size): formed in FP64 and rounded
// once they carry FP32's 6e-8, and an FP32 solve reduces the FP64 residual
// accordingly; formed in FP32 they would be a few per cent off, and so would each
// refinement.  A diagonal system takes one FP32 iteration a refinement and two
// refinements to 1e-10 (three are allowed for), also when its rows hold 12 zeros
// and some of the diagonal entries lie past the 8 that a thread keeps.
// Prints "ok" and exits 0, or reports the violation and exits 1.
#include <cstdio>
#include <vector>

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

template <class T>
static T *upload(const std::vector<T> &h) {
    T *d = nullptr;
    if (cudaMalloc(&d, h.size() * sizeof(T)) != cudaSuccess) return nullptr;
    cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}

// half zeros to either side of the diagonal
static int check(int half) {
    const int n = 64, per = 2 * half + 1;
    const double2 alpha = cd(1.0, 0.0), beta = cd(-1.0, 0.0);
    std::vector<int> ptr(n + 1), col, id(n);
    std::vector<double> M, S;
    for (int i = 0; i < n; ++i) {
        id[i] = i;
        ptr[i + 1] = ptr[i] + per;
        std::vector<int> c;
        for (int o = -half; o <= half; ++o) c.push_back((i + o + n) % n);
        std::sort(c.begin(), c.end());
        for (int j : c) {
            const double m = j == i ? (1.0 + 0.01 * ((i + j) % 17)) / 3.0 : 0.0;
            col.push_back(j);
            M.push_back(m);
            S.push_back(j == i ? m - 1e-6 : 0.0);
        }
    }
    std::vector<double2> x0(n), f(n), x(n);
    for (int i = 0; i < n; ++i) x0[i] = cd(1.0 + 0.3 * ((i * 7) % 11), 0.2 * ((i * 5) % 13) - 1.0);
    for (int i = 0; i < n; ++i)
        for (int e = ptr[i]; e < ptr[i + 1]; ++e)
            f[i] = cadd(f[i], cmul(cadd(cscale(alpha, M[e]), cscale(beta, S[e])), x0[col[e]]));
    int *dptr = upload(ptr), *dcol = upload(col), *did = upload(id), *dstat = upload(std::vector<int>(1));
    double *dM = upload(M), *dS = upload(S), *dres = upload(std::vector<double>(1));
    double2 *df = upload(f), *dx = upload(x);
    if (!dptr || !dcol || !did || !dstat || !dM || !dS || !dres || !df || !dx) return std::printf("FAIL memory\n"), 1;
    KryBatch b{};
    b.nsys = 1;
    b.s[0].alpha = alpha;
    b.s[0].beta = beta;
    b.s[0].f = df;
    b.s[0].x = dx;
    b.s[0].stat = dstat;
    b.s[0].res = dres;
    const int cap = n * std::max(0, per - KMIX_E);
    kmix_kernel<1, false><<<1, n, kmix_smem(n, cap)>>>(b, n, dptr, dcol, dM, dS, did, did, cap, 1e-10, 500);
    const cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return std::printf("FAIL %s\n", cudaGetErrorString(e)), 1;
    int stat = 0;
    cudaMemcpy(&stat, dstat, sizeof(int), cudaMemcpyDeviceToHost);
    cudaMemcpy(x.data(), dx, n * sizeof(double2), cudaMemcpyDeviceToHost);
    double err = 0.0;
    for (int i = 0; i < n; ++i) err = std::fmax(err, std::sqrt(cabs2(csub(x[i], x0[i]))));
    std::printf("%d entries a row: status %d, error %.1e\n", per, stat, err);
    for (void *p : {(void *)dptr, (void *)dcol, (void *)did, (void *)dstat, (void *)dM, (void *)dS, (void *)dres, (void *)df, (void *)dx})
        cudaFree(p);
    // the FP64 entries themselves are 1e-16 / 1e-6 off, beside a residual of 1e-10
    return stat < 1 || stat > 3 || err > 1e-8 ? std::printf("FAIL\n"), 1 : 0;
}

int main() {
    if (check(0) || check(6)) return 1;
    std::printf("ok\n");
    return 0;
}
