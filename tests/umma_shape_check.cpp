// Host check of the GEMM's MMA shapes (umma_shape.cuh): for every N that the GEMM
// takes the instruction exists (kind::f16: 128 rows with one CTA and N a multiple
// of 16, 256 rows with two and N a multiple of 32, at most 256), the CTAs' B rows
// cover the columns, a B tile is whole 1024-byte swizzle atoms, and two
// accumulators fit tensor memory, an epilogue read of 32 columns included.
// Prints "ok <cases>" and exits 0, or reports the first violation and exits 1.
#include <cstdio>

#include "../paper_2104_04609_gb300/csrc/umma_shape.cuh"

int main() {
    int cases = 0;
    for (int n = 16; n <= 256; n += 16) {
        const int cg = umma_ctas(n), m = umma_cols(n), b = umma_b_rows(n), acc = umma_acc_cols(n);
        const bool shape = cg == 1 ? m % 16 == 0 && m >= 16 : cg == 2 && m % 32 == 0 && m >= 32;
        const bool cover = m >= n && m <= 256 && b * cg == m && (cg - 1) * b < n;  // each CTA's box meets B
        const bool tile = b % 8 == 0 && b <= 256;
        const bool tmem = (acc & (acc - 1)) == 0 && 2 * acc <= 512 && acc >= m && (n + 31) / 32 * 32 <= acc;
        if (!shape || !cover || !tile || !tmem) {
            std::printf("FAIL N %d: %d CTAs, %d columns, %d B rows each, accumulator %d\n", n, cg, m, b, acc);
            return 1;
        }
        ++cases;
    }
    std::printf("ok %d\n", cases);
    return 0;
}
