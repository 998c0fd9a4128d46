// The bounded wait of the FP64 dense solve (csrc/dense.cu): a solution block that never appears.  The solve
// of two blocks of 32 is launched with its first CTA alone, so that the backward wait for the second block's
// part runs out (within seconds), or ends at the next look when the error word is already set; the kernel
// returns, the error word says why and the device works on.  With both CTAs the solution is complete.
#include "dense.cu"

#include <cstdio>
#include <vector>

int main() {
    using namespace ot;
    const int n = 2 * kB;
    double *A, *Linv, *D, *b, *z, *x;
    int *err;
    if (cudaMalloc(&A, 8 * n * n) || cudaMalloc(&Linv, 8 * n * kB) || cudaMalloc(&D, 8 * n) || cudaMalloc(&b, 8 * n) ||
        cudaMalloc(&z, 8 * n) || cudaMalloc(&x, 8 * n) || cudaMalloc(&err, 4))
        return 2;
    // L = I (its diagonal blocks' inverses too), D = 4: x = b / 4
    std::vector<double> hLinv(n * kB, 0.0), hD(n, 4.0), hb(n), hx(n);
    for (int i = 0; i < n; ++i) { hLinv[(size_t)(i % kB) * n + i] = 1.0; hb[i] = i + 1; }
    cudaMemset(A, 0, 8 * n * n);
    cudaMemcpy(Linv, hLinv.data(), 8 * n * kB, cudaMemcpyHostToDevice);
    cudaMemcpy(D, hD.data(), 8 * n, cudaMemcpyHostToDevice);
    cudaMemcpy(b, hb.data(), 8 * n, cudaMemcpyHostToDevice);
    int bad = 0;
    for (int run = 0; run < 3; ++run) {
        // 0: the wait runs out; 1: an error is there before; 2: complete
        int e = run == 1 ? (int)OT_ERR_NUMERIC : 0;
        cudaMemset(z, 0xff, 8 * n);
        cudaMemset(x, 0xff, 8 * n);
        cudaMemcpy(err, &e, 4, cudaMemcpyHostToDevice);
        if (run < 2) {
            dense_solve_kernel<<<1, kST>>>(n, A, Linv, D, b, z, x, err);
        } else {
            int nn = n;
            const double *cA = A, *cL = Linv, *cD = D, *cb = b;
            void *args[] = {&nn, &cA, &cL, &cD, &cb, &z, &x, &err};
            if (cudaLaunchCooperativeKernel((void *)dense_solve_kernel, dim3(2), dim3(kST), args, 0, 0) != cudaSuccess) return 2;
        }
        if (cudaDeviceSynchronize() != cudaSuccess) return 2;
        cudaMemcpy(&e, err, 4, cudaMemcpyDeviceToHost);
        cudaMemcpy(hx.data(), x, 8 * n, cudaMemcpyDeviceToHost);
        bool done = true;
        for (int i = 0; i < n; ++i) done = done && hx[i] == hb[i] / 4.0;
        printf("run %d: error %d, complete %d\n", run, e, (int)done);
        if (e != (run == 0 ? (int)OT_ERR_TIMEOUT : run == 1 ? (int)OT_ERR_NUMERIC : 0) || done != (run == 2)) ++bad;
    }
    if (bad) return 1;
    printf("OK\n");
    return 0;
}
