// One iteration of the diagnostic's power iteration whose column kernel has more
// blocks than run at once, with the iteration's end (max_iters = 1) written by
// its first block: every block of that launch still does its share, and the two
// kernels queued behind it change nothing but hand its end on.  Prints "OK" or
// the first violation.
#include <cmath>
#include <cstdio>
#include <vector>

#include "rikfad_diag_kernels.cuh"

using namespace rikfad;

template <typename T>
static T *device(const std::vector<T> &v)
{
    T *p = nullptr;
    if (cudaMalloc(&p, v.size() * sizeof(T)) != cudaSuccess ||
        cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
        std::printf("FAIL allocation\n");
    return p;
}

int main()
{
    const int64_t m = 2048, n = 16384;
    DiagParams d{};
    d.td.rows = m;
    d.td.cols = n;
    d.td.spart_cnt = 1;
    d.nblk = (int)diag_row_blocks(m, n);
    d.wpr = diag_warps_per_row(m);
    d.ncb = diag_col_blocks(n);
    d.cpb = diag_cols_per_block(n);
    d.max_iters = 1;
    std::vector<float> xi(m * n), R(m, 1.f / m), C(n, 1.f), spart(1, 1.f), v(n, NAN), wpart((size_t)d.nblk * n, NAN);
    for (int64_t i = 0; i < m * n; ++i)
        xi[i] = 1.f + 1e-3f * (float)(i % 97);
    d.xi = device(xi);
    d.R = device(R);
    d.C = device(C);
    d.spart = device(spart);
    d.v = device(v);
    d.wpart = device(wpart);
    d.upart = device(std::vector<double>(d.nblk, NAN));
    d.npart = device(std::vector<double>(2 * d.nblk, NAN));
    d.v2part = device(std::vector<double>(2 * d.ncb, NAN));
    DiagState *const states = device(std::vector<DiagState>(2));
    d.host = device(std::vector<DiagState>(1));
    DiagState st[3];
    std::vector<float> after(n);
    for (int it = 0; it < 3; ++it) {
        d.parity = it & 1;
        d.st = states + d.parity;
        d.st_next = states + (d.parity ^ 1);
        if (it == 0)
            diag_rows_kernel<true>(n)<<<d.nblk, kThreads>>>(d);
        else
            diag_rows_kernel<false>(n)<<<d.nblk, kThreads>>>(d);
        rikfad_diag_cols_kernel<<<d.ncb, diag_col_threads(d.nblk)>>>(d);
        if (cudaDeviceSynchronize() != cudaSuccess) {
            std::printf("FAIL %s\n", cudaGetErrorString(cudaGetLastError()));
            return 1;
        }
        cudaMemcpy(it == 0 ? v.data() : after.data(), d.v, n * sizeof(float), cudaMemcpyDeviceToHost);
        cudaMemcpy(&st[it], d.st_next, sizeof(DiagState), cudaMemcpyDeviceToHost);
    }
    for (int64_t j = 0; j < n; ++j)
        if (!std::isfinite(v[j]) || v[j] != after[j]) {
            std::printf("FAIL column %lld of %lld: %g, then %g\n", (long long)j, (long long)n, v[j], after[j]);
            return 1;
        }
    std::vector<double> v2(2 * d.ncb);
    cudaMemcpy(v2.data(), d.v2part, v2.size() * sizeof(double), cudaMemcpyDeviceToHost);
    for (int b = 0; b < d.ncb; ++b)
        if (!(v2[d.ncb + b] > 0.0)) {
            std::printf("FAIL block %d of %d\n", b, d.ncb);
            return 1;
        }
    if (st[0].done != 1 || st[0].it != 1 || st[1].done != 1 || st[2].done != 1) {
        std::printf("FAIL state\n");
        return 1;
    }
    std::printf("OK\n");
    return 0;
}
