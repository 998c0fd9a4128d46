// Dense LDL^T of the assembled Schur complement S_M (Section 4.2's direct solve) for moderate n.
//
// When the support is still large, the exact factor of S_M is a sizeable fraction of dense
// (a quarter of n^2 on 64x64 images), and a sparse factorisation then only adds dependency-chain
// latency.  This path factors the dense matrix (column-major, FP64) with a blocked right-looking
// LDL^T: per panel of kB columns
//   (1) panel: every CTA eliminates the kB x kB diagonal block and its own 32 rows below together
//       (pivots keeping less than eps of their original diagonal become +infinity: the column is
//       zeroed, Section 4.2), which yields L21 and LD = L21 D1 without a separate block inverse;
//   (2) the trailing update A22 -= LD L21^T on tiles of the lower triangle; one CTA more inverts
//       the panel's unit block for the solves.
// What bounds it here: a warp's FP64 multiply-add occupies its scheduler for 64 cycles (measured;
// 1.7 per cycle and SM in all), a division for 650, so the work goes to as many SMs as there are
// and nothing is computed twice on the chain except the small diagonal block.
// Solves run in one cooperative launch, one CTA per block row: each waits for the blocks of the
// solution it needs as they appear, so a panel costs one block product and one hand-over instead
// of two grid barriers.
#include "chol.cuh"
#include "primitives.cuh"

#include <cmath>

namespace ot {
namespace {

constexpr int kB = 32;      // panel width
constexpr int kT = 256;

#define GSD(var, count) \
    for (int64_t var = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; var < (count); var += (int64_t)gridDim.x * blockDim.x)

inline unsigned gridd(int64_t work) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(4096, ceil_div(work, kT)));
}

// one warp per row
__global__ void dense_scatter_kernel(int n, const int32_t *__restrict__ Ap, const int32_t *__restrict__ Aj,
                                     const double *__restrict__ Ax, const double *__restrict__ Adiag,
                                     double *__restrict__ A, double *__restrict__ d0) {
    const int lane = threadIdx.x & 31;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        // the values of row r, at (r, column): the matrix is symmetric, so they fill column r
        for (int e = Ap[r] + lane; e < Ap[r + 1]; e += 32) A[r * n + Aj[e]] = Ax[e];
        if (lane == 0) {
            A[r * n + r] = Adiag[r];
            d0[r] = Adiag[r];
        }
    }
}

// (1) Panel [k, k + bs): warps 0-3 hold the diagonal block's rows, warps 4-7 the CTA's 32 rows below
// (one row per lane, columns w, w + 4, ... of warp w in registers).  Step j: the owners of column j
// publish it, then every row takes l = a_rj / d_j (quotient) and a_rc -= l a_cj for its later columns.
// CTA 0 writes D and the block's L.  32 steps of about 500 cycles; the substitution with one thread
// per row that it replaced took 350 us per 64 columns at n = 961 (and the diagonal block 210 us).
__global__ void __launch_bounds__(kT)
dense_panel_kernel(int n, int k, int bs, double *__restrict__ A, double *__restrict__ D,
                   const double *__restrict__ d0, double eps, double *__restrict__ LD) {
    __shared__ double col[2][2][kB];
    __shared__ double thr[kB];
    const int lane = threadIdx.x & 31, half = threadIdx.x >> 7, w = (threadIdx.x >> 5) & 3;
    const int r = half ? k + bs + (int)blockIdx.x * 32 + lane : k + lane;
    const bool live = r < n && (half || lane < bs);
    if (threadIdx.x < kB) thr[threadIdx.x] = (int)threadIdx.x < bs ? eps * d0[k + threadIdx.x] : 0.0;
    double a[kB / 4];
#pragma unroll
    for (int q = 0; q < kB / 4; ++q) {
        const int c = w + 4 * q;
        a[q] = live && c < bs ? A[(int64_t)(k + c) * n + r] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < kB; ++j) {
        if (j >= bs) break;
        double (*cj)[kB] = col[j & 1];
        if (w == (j & 3)) cj[half][lane] = a[j >> 2];
        __syncthreads();
        const double d = cj[0][j], v = cj[half][lane];
        const bool inf = !(d > thr[j]);
        const double l = inf ? 0.0 : quotient(v, d);
#pragma unroll
        for (int q = 0; q < kB / 4; ++q)
            if (w + 4 * q > j) a[q] = fma(-l, cj[0][w + 4 * q], a[q]);
        if (w == (j & 3) && live) {
            if (half) {
                A[(int64_t)(k + j) * n + r] = l;
                LD[(int64_t)j * n + r] = inf ? 0.0 : v;
            } else if (blockIdx.x == 0) {
                a[j >> 2] = l;   // stored after the other CTAs' reads: see below
                if (lane == 0) D[k + j] = inf ? INFINITY : d;
            }
        }
    }
    // the block's L goes to LD's rows of the block (the other CTAs read A's block unscaled);
    // dense_update_kernel's last CTA moves it to A
    if (!half && blockIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < kB / 4; ++q) {
            const int c = w + 4 * q;
            if (c < bs && lane < bs) LD[(int64_t)c * n + k + lane] = lane > c ? a[q] : 0.0;
        }
    }
}

// X = L11^-1 of panel k (unit lower, from LD's rows of the block), written to Linv, and L11 to A.
// One CTA of kT threads: lane = column of X, warp w the rows w, w + 8, ...; step j publishes row j.
__device__ void dense_invert_block(int n, int k, int bs, double *__restrict__ A, const double *__restrict__ LD,
                                   double *__restrict__ Linv, double (*L)[kB + 1], double (*row)[kB]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < kB * kB; t += kT) {
        const int i = t % kB, j = t / kB;
        const double l = i < bs && j < bs && i > j ? LD[(int64_t)j * n + k + i] : 0.0;
        L[i][j] = l;
        if (i < bs && j < bs && i > j) A[(int64_t)(k + j) * n + k + i] = l;
    }
    double x[kB / 8];
#pragma unroll
    for (int q = 0; q < kB / 8; ++q) x[q] = w + 8 * q == lane ? 1.0 : 0.0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kB; ++j) {
        if (w == (j & 7)) row[j & 1][lane] = x[j >> 3];
        __syncthreads();
        const double xj = row[j & 1][lane];
#pragma unroll
        for (int q = 0; q < kB / 8; ++q)
            if (w + 8 * q > j) x[q] = fma(-L[w + 8 * q][j], xj, x[q]);
    }
#pragma unroll
    for (int q = 0; q < kB / 8; ++q)
        if (w + 8 * q < bs && lane < bs) Linv[(int64_t)lane * n + k + w + 8 * q] = x[q];
}

// (2) A22(r, c) -= sum_l LD(r, l) L21(c, l) on the lower triangle in T x T tiles (64: 4 x 4 per
// thread; 32 while fewer than four tiles of 64 per SM are left: 2 x 2 per thread).  The last CTA
// inverts the panel's block.
template <int T>
__global__ void __launch_bounds__(kT)
dense_update_kernel(int n, int k, int bs, double *__restrict__ A, const double *__restrict__ LD,
                    double *__restrict__ Linv) {
    __shared__ double sm[2 * kB * T > kB * (kB + 1) + 2 * kB ? 2 * kB * T : kB * (kB + 1) + 2 * kB];
    if (blockIdx.x == gridDim.x - 1) {
        dense_invert_block(n, k, bs, A, LD, Linv, (double (*)[kB + 1])sm, (double (*)[kB])(sm + kB * (kB + 1)));
        return;
    }
    constexpr int Q = T / 16;
    double (*Ls)[T] = (double (*)[T])sm, (*Rs)[T] = (double (*)[T])(sm + kB * T);   // [depth][row], [depth][column]
    const int base = k + bs;
    // tile index -> (ti, tj) with ti >= tj
    const int idx = blockIdx.x;
    int ti = (int)((sqrtf(8.0f * idx + 1.0f) - 1.0f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= idx) ++ti;
    while (ti * (ti + 1) / 2 > idx) --ti;
    const int tj = idx - ti * (ti + 1) / 2;
    const int r0 = base + ti * T, c0 = base + tj * T;
    for (int q = threadIdx.x; q < kB * T; q += kT) {
        const int l = q / T, rr = q % T;
        Ls[l][rr] = r0 + rr < n ? LD[(int64_t)l * n + r0 + rr] : 0.0;
        Rs[l][rr] = c0 + rr < n ? A[(int64_t)(k + l) * n + c0 + rr] : 0.0;
    }
    const int tr = (threadIdx.x % 16) * Q, tc = (threadIdx.x / 16) * Q;
    // the products are summed by themselves and subtracted once (an accumulator started from A would
    // round every term at A's magnitude)
    double acc[Q][Q], old[Q][Q];
#pragma unroll
    for (int w = 0; w < Q; ++w)
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const int r = r0 + tr + u, c = c0 + tc + w;
            acc[u][w] = 0.0;
            old[u][w] = r < n && c < n && r >= c ? A[(int64_t)c * n + r] : 0.0;
        }
    __syncthreads();
    for (int l = 0; l < kB; ++l) {   // (a panel with rows below it is full)
        double a[Q], b[Q];
#pragma unroll
        for (int u = 0; u < Q; ++u) { a[u] = Ls[l][tr + u]; b[u] = Rs[l][tc + u]; }
#pragma unroll
        for (int u = 0; u < Q; ++u)
#pragma unroll
            for (int w = 0; w < Q; ++w) acc[u][w] = fma(a[u], b[w], acc[u][w]);
    }
#pragma unroll
    for (int w = 0; w < Q; ++w)
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const int r = r0 + tr + u, c = c0 + tc + w;
            if (r < n && c < n && r >= c) A[(int64_t)c * n + r] = old[u][w] - acc[u][w];
        }
}

// ------------------------------------------------------------------------ solves
// Forward L z = b, y = D^-1 z, backward L^T x = y.  CTA i owns block row i (kB rows, four warps: warp
// g takes depths 8 g .. 8 g + 7 of every block product); the blocks of L that it will need are loaded
// ahead of the wait.  z and x are preset to an all-ones pattern that no result has; a value that
// differs is complete, so data and flag arrive in one load.  Every wait is bounded.
constexpr int kST = 128;
constexpr unsigned long long kUnset = ~0ull;

__device__ __forceinline__ void publish(double *p, double v) {
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b == kUnset) b = 0x7ff8000000000000ull;   // a NaN from the caller's data stays a NaN
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(b) : "memory");
}

// this lane's value of p[0 .. 7] (lane & 7; entries at or beyond `valid` are zero) once all are set;
// false when the wait gave up
__device__ __forceinline__ bool await8(const double *p, int valid, double &v, int *err) {
    const int q = threadIdx.x & 7;
    unsigned long long b = q < valid ? kUnset : 0ull;
    for (unsigned spin = 0;; ++spin) {
        if (b == kUnset) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(b) : "l"(p + q) : "memory");
        if (__all_sync(0xffffffffu, b != kUnset)) break;
        // (one decision for the warp: a lane that left alone would leave the others in the votes)
        if ((spin & 63u) == 63u && __any_sync(0xffffffffu, spin > kSpinLimit || *(volatile int *)err != 0)) {
            atomicCAS(err, 0, (int)OT_ERR_TIMEOUT);
            return false;
        }
    }
    v = __longlong_as_double((long long)b);
    return true;
}

__global__ void __launch_bounds__(kST)
dense_solve_kernel(int n, const double *__restrict__ A, const double *__restrict__ Linv,
                   const double *__restrict__ D, const double *__restrict__ b, double *z, double *x, int *err) {
    __shared__ double red[4][kB];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, nb = (n + kB - 1) / kB;
    const int i = (int)blockIdx.x, k = i * kB, bs = min(kB, n - k);
    const bool live = lane < bs;
    // the inverse block: row `lane`, columns 8 g .. (forward), column `lane`, rows 8 g .. (backward)
    double Fi[8], Bi[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int c = 8 * g + q;
        Fi[q] = live && c < bs ? Linv[(int64_t)c * n + k + lane] : 0.0;
        Bi[q] = live && c < bs ? Linv[(int64_t)lane * n + k + c] : 0.0;
    }
    const double bv = live ? b[k + lane] : 0.0, dv = live ? D[k + lane] : 1.0;
    auto reduce = [&](double v) {   // the four warps' parts, in every warp
        red[g][lane] = v;
        __syncthreads();
        const double s = (red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane]);
        __syncthreads();
        return s;
    };
    bool ok = true;
    // ---- forward: z_i = L_ii^-1 (b_i - sum_{j < i} L_ij z_j)
    double acc = 0.0, cur[8], nxt[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) nxt[q] = live && i > 0 ? A[(int64_t)(8 * g + q) * n + k + lane] : 0.0;
    for (int j = 0; j < i; ++j) {
#pragma unroll
        for (int q = 0; q < 8; ++q) cur[q] = nxt[q];
        if (j + 1 < i)
#pragma unroll
            for (int q = 0; q < 8; ++q) nxt[q] = live ? A[(int64_t)((j + 1) * kB + 8 * g + q) * n + k + lane] : 0.0;
        double zv = 0.0;
        ok = ok && await8(z + j * kB + 8 * g, 8, zv, err);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc = fma(cur[q], __shfl_sync(0xffffffffu, zv, q), acc);
    }
    double t = bv - reduce(acc);
    acc = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) acc = fma(Fi[q], __shfl_sync(0xffffffffu, t, 8 * g + q), acc);
    t = reduce(acc);
    if (__syncthreads_or(!ok)) return;
    if (g == 0 && live) publish(z + k + lane, t);
    // ---- backward: x_i = L_ii^-T (D_i^-1 z_i - sum_{j > i} L_ji^T x_j)
    const double y = isinf(dv) ? 0.0 : t / dv;
    acc = 0.0;
    const double *Ai = A + (int64_t)(k + lane) * n;   // column k + lane
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int r = (nb - 1) * kB + 8 * g + q;
        nxt[q] = live && i < nb - 1 && r < n ? Ai[r] : 0.0;
    }
    for (int j = nb - 1; j > i; --j) {
#pragma unroll
        for (int q = 0; q < 8; ++q) cur[q] = nxt[q];
        if (j - 1 > i)
#pragma unroll
            for (int q = 0; q < 8; ++q) nxt[q] = live ? Ai[(j - 1) * kB + 8 * g + q] : 0.0;
        double xv = 0.0;
        ok = ok && await8(x + j * kB + 8 * g, n - (j * kB + 8 * g), xv, err);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc = fma(cur[q], __shfl_sync(0xffffffffu, xv, q), acc);
    }
    t = y - reduce(acc);
    acc = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) acc = fma(Bi[q], __shfl_sync(0xffffffffu, t, 8 * g + q), acc);
    t = reduce(acc);
    if (__syncthreads_or(!ok)) return;
    if (g == 0 && live) publish(x + k + lane, t);
}

}  // namespace

Error dense_alloc(DenseLDL &M, int32_t n) {
    M.n = n;
    OT_CUDA(cudaMalloc((void **)&M.A, sizeof(double) * (size_t)n * n));
    OT_CUDA(cudaMalloc((void **)&M.LD, sizeof(double) * (size_t)n * kB));
    OT_CUDA(cudaMalloc((void **)&M.Linv, sizeof(double) * (size_t)n * kB));
    OT_CUDA(cudaMalloc((void **)&M.D, sizeof(double) * n));
    OT_CUDA(cudaMalloc((void **)&M.d0, sizeof(double) * n));
    OT_CUDA(cudaMalloc((void **)&M.z, sizeof(double) * n));
    OT_CUDA(cudaMalloc((void **)&M.err, sizeof(int)));
    return ok();
}

void dense_free(DenseLDL &M) {
    for (void *p : {(void *)M.A, (void *)M.LD, (void *)M.Linv, (void *)M.D, (void *)M.d0, (void *)M.z, (void *)M.err})
        if (p) cudaFree(p);
    M = DenseLDL();
}

Error dense_factor(DenseLDL &M, const Chol &C, double eps, cudaStream_t st) {
    const int n = M.n;
    int dev = 0, sms = 0;
    OT_CUDA(cudaGetDevice(&dev));
    OT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    OT_CUDA(cudaMemsetAsync(M.A, 0, sizeof(double) * (size_t)n * n, st));
    dense_scatter_kernel<<<gridd(32LL * n), kT, 0, st>>>(n, C.Ap, C.Aj, C.Ax, C.Adiag, M.A, M.d0);
    OT_LAUNCHED();
    ktimer_begin(KT_LDL_NUMERIC, st);
    for (int k = 0; k < n; k += kB) {
        const int bs = std::min(kB, n - k), rest = n - k - bs;
        dense_panel_kernel<<<(unsigned)std::max<int64_t>(1, ceil_div(rest, 32)), kT, 0, st>>>(n, k, bs, M.A, M.D, M.d0,
                                                                                             eps, M.LD);
        OT_LAUNCHED();
        const int64_t t = ceil_div(rest, 64), t2 = ceil_div(rest, 32);
        if (t * (t + 1) / 2 >= 4LL * sms)
            dense_update_kernel<64><<<(unsigned)(t * (t + 1) / 2 + 1), kT, 0, st>>>(n, k, bs, M.A, M.LD, M.Linv);
        else
            dense_update_kernel<32><<<(unsigned)(t2 * (t2 + 1) / 2 + 1), kT, 0, st>>>(n, k, bs, M.A, M.LD, M.Linv);
        OT_LAUNCHED();
    }
    ktimer_end(KT_LDL_NUMERIC, st);
    ktimer_add_work(KT_LDL_NUMERIC, (double)n * n * n / 3.0);  // L D L^T: n^3/3 flops
    return ok();
}

Error dense_solve(DenseLDL &M, const double *b, double *x, cudaStream_t st) {
    int n = M.n;
    OT_CUDA(cudaMemsetAsync(M.z, 0xff, sizeof(double) * n, st));
    OT_CUDA(cudaMemsetAsync(x, 0xff, sizeof(double) * n, st));
    const double *A = M.A, *Li = M.Linv, *D = M.D;
    double *z = M.z;
    int *err = M.err;
    void *args[] = {&n, &A, &Li, &D, &b, &z, &x, &err};
    ktimer_begin(KT_LDL_SOLVE, st);
    OT_CUDA(cudaLaunchCooperativeKernel((void *)dense_solve_kernel, dim3((unsigned)ceil_div(n, kB)), dim3(kST), args, 0,
                                        st));
    OT_LAUNCHED();
    ktimer_end(KT_LDL_SOLVE, st);
    ktimer_add_work(KT_LDL_SOLVE, 8.0 * (double)n * n);  // reads L twice
    return ok();
}

}  // namespace ot
