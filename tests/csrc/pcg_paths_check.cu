// The grid PCG (csrc/newton.cu) by where a block keeps its share: its columns' vectors and its pairs in shared
// memory, the vectors only, the pairs only, neither.  Which one applies depends on the share, so systems of
// one size are solved with one block (everything is beyond 160 KB), a few and many.  Every solution's
// residual is recomputed on the host in FP64 from the operator itself.
//
// Bars: the iteration stops when its own residual is at tol |b|; the true one differs by rounding, at most
// about eps cond(S_M) iterations-growth of |b|: cond is below 1e4 here (grids with theta within a decade,
// chains of 40), so 1e-12 .. 1e-11 in FP64 against tol = 1e-9, and 1e-3 in FP32 against tol = 1e-3.  Twice
// tol bounds both.  All shares run the same arithmetic up to the order of sums: iterations within 10 %.
#include "newton.cu"

#include <cstdio>
#include <random>
#include <vector>

namespace {

using namespace ot;

struct Sys {
    int n;
    std::vector<int32_t> I, J, lab;   // pairs by (i, j); component of each column
    std::vector<double> th, b;
};

// k x k grid, pairs within squared distance r2; or (r2 < 0) chains i - i, i - (i + 1) of 40 points
Sys make(int k, int r2, unsigned seed) {
    Sys s;
    s.n = k * k;
    s.lab.assign(s.n, 0);
    std::mt19937 rng(seed);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    for (int i = 0; i < s.n; ++i)
        for (int j = 0; j < s.n; ++j) {
            const int dx = i % k - j % k, dy = i / k - j / k;
            const bool in = r2 >= 0 ? dx * dx + dy * dy <= r2 : i == j || (j == i + 1 && j % 40 != 0);
            if (!in) continue;
            s.I.push_back(i);
            s.J.push_back(j);
            s.th.push_back(std::pow(10.0, U(rng) - 0.5));
        }
    if (r2 < 0)
        for (int j = 0; j < s.n; ++j) s.lab[j] = j / 40;
    s.b.resize(s.n);
    for (double &x : s.b) x = U(rng) - 0.5;
    std::vector<double> sum(s.n, 0.0), cnt(s.n, 0.0);
    for (int j = 0; j < s.n; ++j) { sum[s.lab[j]] += s.b[j]; cnt[s.lab[j]] += 1.0; }
    for (int j = 0; j < s.n; ++j) s.b[j] -= sum[s.lab[j]] / cnt[s.lab[j]];
    return s;
}

template <typename T>
double relres(const Sys &s, const std::vector<T> &x) {
    std::vector<double> M(s.n, 0.0), w(s.n, 0.0), r = s.b;
    for (size_t e = 0; e < s.th.size(); ++e) { M[s.I[e]] += s.th[e]; w[s.I[e]] += s.th[e] * (double)x[s.J[e]]; }
    for (size_t e = 0; e < s.th.size(); ++e) r[s.J[e]] -= s.th[e] * ((double)x[s.J[e]] - w[s.I[e]] / M[s.I[e]]);
    double a = 0, b = 0;
    for (int j = 0; j < s.n; ++j) { a += r[j] * r[j]; b += s.b[j] * s.b[j]; }
    return std::sqrt(a / b);
}

#define TRY(expr)                                                            \
    do {                                                                     \
        const Error e_ = (expr);                                             \
        if (e_.code != OT_OK) { printf("%s: %s\n", #expr, e_.msg.c_str()); return 2; } \
    } while (0)

template <typename T>
T *up(const std::vector<T> &v) {
    T *p = nullptr;
    if (cudaMalloc(&p, sizeof(T) * v.size()) != cudaSuccess) return nullptr;
    cudaMemcpy(p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice);
    return p;
}

int run(const Sys &sys, const char *name, std::initializer_list<int> blocks) {
    const int n = sys.n;
    const int64_t psi = (int64_t)sys.th.size();
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    Newton W;
    TRY(newton_alloc(W, n, n, psi, sms));
    Support S;
    S.psi = S.cap = psi;
    S.i = up(sys.I);
    S.j = up(sys.J);
    S.p = up(sys.th);
    S.s = up(std::vector<double>(psi, 1.0));
    S.row_ptr = up(std::vector<int32_t>(n + 1));
    S.col_ptr = up(std::vector<int32_t>(n + 1));
    S.col_perm = up(std::vector<int32_t>(psi));
    S.col_row = up(std::vector<int32_t>(psi));
    TRY(rebuild_views(S, n, n, 0));
    TRY(schur_setup(W, S, 0));
    cudaMemcpy(W.rhs, sys.b.data(), sizeof(double) * n, cudaMemcpyHostToDevice);
    cudaMemcpy(W.b32, std::vector<float>(sys.b.begin(), sys.b.end()).data(), sizeof(float) * n, cudaMemcpyHostToDevice);
    W.pcg_cluster = 0;   // the grid kernel at every size
    int bad = 0;
    for (int fp32 = 0; fp32 < 2; ++fp32) {
        int most = 0, least = 1 << 30;
        for (int G : blocks) {
            W.pcg_grid = G;
            const double tol = fp32 ? 1e-3 : 1e-9;
            if (fp32)
                TRY(launch_pcg<float>(W, S, W.theta32, W.theta32_col, W.Minv32, W.Dinv32, W.b32, W.x32, W.r32, W.q32, W.w32,
                                      tol, 5000, 0));
            else
                TRY(launch_pcg<double>(W, S, W.theta, W.theta_col, W.Minv, W.Dinv, W.rhs, W.x64, W.r64, W.q64, W.w64, tol,
                                       5000, 0));
            double hs[SC_COUNT];
            TRY(read_scalars(W, hs, 0));
            int err = 0;
            cudaMemcpy(&err, W.err, sizeof(int), cudaMemcpyDeviceToHost);
            std::vector<double> x(n);
            std::vector<float> x32(n);
            double rel;
            if (fp32) {
                cudaMemcpy(x32.data(), W.x32, sizeof(float) * n, cudaMemcpyDeviceToHost);
                rel = relres(sys, x32);
            } else {
                cudaMemcpy(x.data(), W.x64, sizeof(double) * n, cudaMemcpyDeviceToHost);
                rel = relres(sys, x);
            }
            // (the first block's share, had all the same)
            const size_t t = fp32 ? 4 : 8, c = (n + G - 1) / G, vec = c * 10 * t + (2 * c + 2) * 4, e = 2 * ((psi + G - 1) / G) * (t + 4);
            const bool v_in = vec + 16 <= (size_t)kPcgSmem, p_in = (v_in ? vec + 16 : 0) + e <= (size_t)kPcgSmem;
            const int its = (int)hs[SC_PCG_ITERS];
            printf("%s n %d %s %d blocks (vectors %s, pairs %s): %d iterations, residual %.2e\n", name, n, fp32 ? "FP32" : "FP64",
                   G, v_in ? "in" : "out", p_in ? "in" : "out", its, rel);
            most = std::max(most, its);
            least = std::min(least, its);
            if (err || !(rel <= 2 * tol)) ++bad;
        }
        if (most > 1.1 * least + 1) ++bad;
    }
    newton_free(W);
    for (void *p : {(void *)S.i, (void *)S.j, (void *)S.p, (void *)S.s, (void *)S.row_ptr, (void *)S.col_ptr,
                    (void *)S.col_perm, (void *)S.col_row})
        cudaFree(p);
    return bad;
}

}  // namespace

int main() {
    int bad = run(make(31, 9, 1), "grid", {1, 2, 9, 40});
    bad += run(make(47, 5, 2), "grid", {1, 2, 4, 20, 100});
    bad += run(make(64, 2, 3), "grid", {1, 2, 7, 60, 152});
    bad += run(make(63, -1, 4), "chains", {1, 2, 40});
    if (bad) return 1;
    printf("OK\n");
    return 0;
}
