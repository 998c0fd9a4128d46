// FP32 dense LDL^T of S_M with the explicit inverse of its unit lower factor (dense32.cuh).
//
// Per 64-column panel k (column-major, leading dimension ld):
//   colsum  sums of the panel's columns below its diagonal block (the rows not yet eliminated);
//   diag    one CTA factors the 64x64 diagonal block in shared memory, each pivot being minus the
//           sum of its column's remaining off-diagonal entries (in the block, plus the below-block
//           sum updated as columns are eliminated), and writes the inverse of the unit block;
//   step    L21 = A21 L11^-T D1^-1 through the inverse block (a product of non-positive entries
//           with non-negative ones: no cancellation), LD = L21 D1; block row k of X = L^-1: X_kj =
//           L11^-1 B_kj (B: the updates accumulated in X); the part of both updates that the next
//           panel needs;
//   update  the rest of both rank-64 updates beside the chain, the trailing lower triangle
//           A22 -= LD L21^T and the rows of X below the panel, B -= L21 X_k: FP32 128x128 tiles, or two
//           panels at once on the tensor cores.
// The sequence depends on n only, so it is captured once into a CUDA graph.
#include "dense32.cuh"
#include "primitives.cuh"
#include "tc05.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace ot {
namespace {

constexpr int kP = 64;       // panel width
constexpr int kMaxN = 65536;  // largest n
constexpr int kSlice = 16384; // rows per assembly block (a column slice of 64-bit sums in shared memory)
constexpr int kTT = 256;     // threads per CTA
constexpr int kTile = 128;   // update tile (rows and columns)
constexpr int kKc = 16;      // depth of one staged slice of the update tiles

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return x;
}

// One CTA per column j: S_jj' = -sum_i theta_ij theta_ij' / M_i over the sources i shared by j and
// j', accumulated in fixed point (2^62 / N_j per unit: each |S_jj'| <= N_j, and so is their sum).
// Above kSlice rows, block (j, y) keeps only the rows [y kSlice, (y + 1) kSlice) of column j and
// adds its part of the diagonal's sum to tot[j] (an integer sum: the same in any order).
__global__ void __launch_bounds__(kTT)
d32_assemble_kernel(int n, int ld, const int32_t *__restrict__ col_ptr, const int32_t *__restrict__ col_row,
                    const double *__restrict__ theta_col, const int32_t *__restrict__ row_ptr,
                    const int32_t *__restrict__ sj, const double *__restrict__ theta,
                    const double *__restrict__ Minv, const double *__restrict__ Nc, float *__restrict__ A,
                    float *__restrict__ d0, unsigned long long *__restrict__ tot) {
    extern __shared__ unsigned long long acc[];
    __shared__ unsigned long long red[kTT / 32];
    const int j = blockIdx.x;
    const int lo = blockIdx.y * kSlice, hi = min(n, lo + kSlice), len = hi - lo;
    for (int t = threadIdx.x; t < len; t += blockDim.x) acc[t] = 0ull;
    __syncthreads();
    const double Nj = Nc[j];
    const double scale = Nj > 0 ? 4611686018427387904.0 / Nj : 0.0;  // 2^62 / N_j
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (scale > 0) {
        for (int k = col_ptr[j] + warp; k < col_ptr[j + 1]; k += nw) {
            const int i = col_row[k];
            const double f = theta_col[k] * Minv[i] * scale;
            for (int e = row_ptr[i] + lane; e < row_ptr[i + 1]; e += 32) {
                const int jp = sj[e];
                if (jp != j && jp >= lo && jp < hi)
                    atomicAdd(&acc[jp - lo], (unsigned long long)__double2ull_rn(f * theta[e]));
            }
        }
    }
    __syncthreads();
    unsigned long long s = 0;
    for (int t = threadIdx.x; t < len; t += blockDim.x) s += acc[t];
    s = warp_sum_u64(s);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < nw; ++w) t += red[w];
        if (tot) atomicAdd(&tot[j], t);
        else d0[j] = scale > 0 ? (float)((double)t / scale) : 0.f;
    }
    const double inv = scale > 0 ? 1.0 / scale : 0.0;
    // a column shares sources with a few dozen others: 32 rows of zeros (most are) skip the three FP64
    // instructions of the scaling, of which a scheduler takes one per 64 clocks (n =
    // 4096: 101 -> 62 us, n = 16,384: 1415 -> 985)
    for (int r0 = lo + ((max(j + 1, lo) - lo) & ~31); r0 < hi; r0 += blockDim.x) {
        const int r = r0 + (int)threadIdx.x;
        const bool in = r > j && r < hi;
        const unsigned long long a = in ? acc[r - lo] : 0ull;
        if (__any_sync(0xffffffffu, a != 0ull)) {
            if (in) A[(size_t)j * ld + r] = -(float)((double)a * inv);
        } else if (in) {
            A[(size_t)j * ld + r] = -0.f;
        }
    }
}

// the diagonal from the slices' integer sums (the same scaling as the single-block case)
__global__ void d32_diag_total_kernel(int n, const double *__restrict__ Nc, const unsigned long long *__restrict__ tot,
                                      float *__restrict__ d0) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const double Nj = Nc[j];
        const double scale = Nj > 0 ? 4611686018427387904.0 / Nj : 0.0;
        d0[j] = scale > 0 ? (float)((double)tot[j] / scale) : 0.f;
    }
}

// csum[l] = sum of column l over the rows [bs, n) (first panel; later panels receive these sums
// from the previous update's epilogue)
__global__ void __launch_bounds__(kTT)
d32_colsum_kernel(int n, int ld, int bs, const float *__restrict__ A, float *__restrict__ csum) {
    __shared__ double sh[kTT / 32];
    const int l = blockIdx.x;
    const float *col = A + (size_t)l * ld;
    double s = 0.0;
    for (int r = bs + threadIdx.x; r < n; r += blockDim.x) s += (double)col[r];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) csum[l] = (float)s;
}

// One CTA factors the diagonal block in micro-panels of 8 columns.  Warp 0 eliminates a
// micro-panel with its 64 rows in registers (lane q: rows q and q+32; shuffles only): each pivot
// is minus the sum of the column's remaining entries plus its below-block sum (np fixed-order
// partials in csum[p * kP + l]), kept as sums of same-sign terms by a recurrence over the
// micro-panel's own 8 x 8 block (the warp-wide sums are taken once per micro-panel).  Meanwhile the
// other warps apply the micro-panel before's rank-8 update to the rest of the block (one barrier per
// micro-panel) and carry the inverse of the unit block on.  Columns stay unscaled in shared memory
// (l_ij = S_ij / d_j on the way out).
constexpr int kMp = 8;   // micro-panel width
static_assert(kTT == 4 * kP, "warp 0, three threads per column, one warp");

// Warp 0's elimination of one micro-panel (columns c0 .. c0 + nc - 1) with the block's 64 rows in
// registers (lane q: rows q and q + 32).  prev >= 0: the micro-panel's columns first receive the
// rank-8 update of the micro-panel starting at prev (eliminated by this warp just before), in the
// same order as the other warps apply it to the later columns.  kFull: nc == kMp known at compile
// time, so the whole micro-panel is one straight-line block.
template <bool kFull>
__device__ __forceinline__ void d32_micro_panel(int lane, int k, int c0, int nc, int prev, float (*S)[kP + 1],
                                                float *g, const float *thr, float *ids, float *D) {
    const unsigned full = 0xffffffffu;
    const int ncc = kFull ? kMp : nc;
    __syncwarp();
    float v0[kMp], v1[kMp], gm[kMp], tl[kMp], dv[kMp], iv[kMp];
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj) {
        v0[jj] = jj < ncc ? S[lane][c0 + jj] : 0.f;
        v1[jj] = jj < ncc ? S[lane + 32][c0 + jj] : 0.f;
        gm[jj] = jj < ncc ? g[c0 + jj] : 0.f;
        tl[jj] = jj < ncc ? thr[c0 + jj] : 0.f;
    }
    if (prev >= 0) {
        float a0[kMp], a1[kMp], gp[kMp], ip[kMp];
#pragma unroll
        for (int q = 0; q < kMp; ++q) {
            a0[q] = S[lane][prev + q];
            a1[q] = S[lane + 32][prev + q];
            gp[q] = g[prev + q];
            ip[q] = ids[prev + q];
        }
#pragma unroll
        for (int jj = 0; jj < kMp; ++jj) {
            if (jj < ncc) {
                const int l = c0 + jj;
                float s0 = 0.f, s1 = 0.f, sg = 0.f;
#pragma unroll
                for (int q = 0; q < kMp; ++q) {
                    const float f = S[l][prev + q] * ip[q];
                    s0 += a0[q] * f;
                    s1 += a1[q] * f;
                    sg += f * gp[q];
                }
                if (lane > l) v0[jj] -= s0;
                if (lane + 32 > l) v1[jj] -= s1;
                gm[jj] -= sg;
            }
        }
    }
    // The pivots without a warp reduction on their chain.  With W_c the sum of column c's entries in
    // the rows from c0 + 8 on (in the block, and below it through g) and B the micro-panel's own
    // 8 x 8 lower part, eliminating column c changes, for every later column j of the micro-panel,
    //   B[r][j] -= B[r][c] l_jc  (r > j),   W_j -= W_c l_jc,   g_j -= g_c l_jc,   l_jc = B[j][c] / d_c,
    // and d_j = -(sum_{r > j} B[r][j] + W_j).  Every W and every B entry below the diagonal stays a
    // sum of non-positive terms (an M-matrix's Schur complements), so the pivots keep the
    // cancellation-free form.  The 8 initial W sums are reduced together, B is broadcast once,
    // and the 8-step recurrence runs on scalars in every lane.
    const bool lo_half = c0 < 32;   // the micro-panel's rows c0 .. c0 + 7 sit in one half
    float W[kMp], B[kMp][kMp];
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj) {
        W[jj] = (lane >= c0 + kMp ? v0[jj] : 0.f) + (lane + 32 >= c0 + kMp ? v1[jj] : 0.f);
#pragma unroll
        for (int r = 0; r < kMp; ++r) B[r][jj] = 0.f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int jj = 0; jj < kMp; ++jj) W[jj] += __shfl_xor_sync(full, W[jj], o);
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj) {
        W[jj] += gm[jj];
#pragma unroll
        for (int r = jj + 1; r < kMp; ++r) B[r][jj] = __shfl_sync(full, lo_half ? v0[jj] : v1[jj], (c0 + r) & 31);
    }
    float L[kMp][kMp];   // L[j][c] = l_jc of the micro-panel (j > c)
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj)
#pragma unroll
        for (int c = 0; c < kMp; ++c) L[jj][c] = 0.f;
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj) {
        dv[jj] = INFINITY;
        iv[jj] = 0.f;
        if (jj < ncc) {
            float sum = W[jj];
#pragma unroll
            for (int r = jj + 1; r < kMp; ++r) sum += B[r][jj];
            const float d = -sum;
            const bool inf = !(d > tl[jj]);
            const float id = inf ? 0.f : 1.f / d;
#pragma unroll
            for (int j2 = jj + 1; j2 < kMp; ++j2) {
                const float l = B[j2][jj] * id;
                L[j2][jj] = l;
#pragma unroll
                for (int r = j2 + 1; r < kMp; ++r) B[r][j2] -= B[r][jj] * l;
                W[j2] -= W[jj] * l;
                gm[j2] -= gm[jj] * l;
            }
            dv[jj] = inf ? INFINITY : d;
            iv[jj] = id;
        }
    }
    // each lane's own rows, in the same order: S_ij -= S_ic l_jc for c < j, rows below j only
#pragma unroll
    for (int jj = 1; jj < kMp; ++jj) {
        const int j = c0 + jj;
#pragma unroll
        for (int c = 0; c < jj; ++c) {
            if (lane > j) v0[jj] -= v0[c] * L[jj][c];
            if (lane + 32 > j) v1[jj] -= v1[c] * L[jj][c];
        }
    }
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj) {
        if (dv[jj] == INFINITY) {   // a grounded column: its entries no longer enter anything
            v0[jj] = 0.f;
            v1[jj] = 0.f;
        }
    }
#pragma unroll
    for (int jj = 0; jj < kMp; ++jj) {
        if (jj < ncc) {
            S[lane][c0 + jj] = v0[jj];
            S[lane + 32][c0 + jj] = v1[jj];
            if (lane == jj) {
                g[c0 + jj] = gm[jj];
                D[k + c0 + jj] = dv[jj];
                ids[c0 + jj] = iv[jj];
            }
        }
    }
}

// shared memory of one diagonal-block factorisation (kDiagSmem bytes when carved from a buffer)
struct DiagSmem {
    float (*S)[kP + 1];
    float (*Xs)[kP + 1];
    float (*red)[kP];
    float *g, *thr, *ids;
};
constexpr int kDiagSmem = (2 * kP * (kP + 1) + 4 * kP + 3 * kP) * 4;

__device__ __forceinline__ DiagSmem diag_smem(float *buf) {
    DiagSmem m;
    m.S = (float (*)[kP + 1])buf;
    m.Xs = (float (*)[kP + 1])(buf + kP * (kP + 1));
    m.red = (float (*)[kP])(buf + 2 * kP * (kP + 1));
    m.g = buf + 2 * kP * (kP + 1) + 4 * kP;
    m.thr = m.g + kP;
    m.ids = m.thr + kP;
    return m;
}

// The diagonal block at k (bs columns) by one CTA of kTT threads.  The block and the partial sums
// are read through L2 (__ldcg).  The partial column sums below the block come as np strips of
// `per` rows each (per = 2: the step kernel's two half-strip CTAs), added in a fixed order.
__device__ __forceinline__ void d32_diag_block(const DiagSmem &m, int ld, int k, int bs, float *__restrict__ A,
                                               float *__restrict__ D, const float *__restrict__ d0,
                                               const float *__restrict__ csum, int np, int per, float eps,
                                               float *__restrict__ Linv) {
    float (*S)[kP + 1] = m.S;
    float (*Xs)[kP + 1] = m.Xs;
    float *g = m.g, *thr = m.thr, *ids = m.ids;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // every global load of the block, of the first kP rows of partial sums and of the diagonal
    // is issued before the first of them is used (kTT = 4 kP threads: 16 block entries each)
    constexpr int kPer = kP * kP / kTT;
    const int nq0 = min(kP, np);
    float sv[kPer], cv[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int t = (int)threadIdx.x + q * kTT, i = t % kP, j = t / kP;
        sv[q] = (i > j && i < bs) ? __ldcg(A + (size_t)(k + j) * ld + (k + i)) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        // strip t / kP's sum: its per (1 or 2) partial rows added in order
        const int t = (int)threadIdx.x + q * kTT, row = t / kP, col = t % kP;
        float v = 0.f;
        if (t < nq0 * kP) {
            v = __ldcg(csum + (size_t)(row * per) * kP + col);
            if (per == 2) v += __ldcg(csum + (size_t)(row * per + 1) * kP + col);
        }
        cv[q] = v;
    }
    const float d0v = (int)threadIdx.x < bs ? d0[k + threadIdx.x] : 0.f;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int t = (int)threadIdx.x + q * kTT;
        S[t % kP][t / kP] = sv[q];
        Xs[t / kP][t % kP] = cv[q];
    }
    __syncthreads();
    // each column's partials: four threads take every fourth row (those beyond kP, for n above 4096,
    // straight from memory), then one adds the four in order
    float gs = 0.f;
    {
        const int c = threadIdx.x % kP, h = threadIdx.x / kP;
        float part = 0.f;
        for (int q = h; q < nq0; q += kTT / kP) part += Xs[q][c];
#pragma unroll 16
        for (int q = kP + h; q < np; q += kTT / kP) {
            float v = __ldcg(csum + (size_t)(q * per) * kP + c);
            if (per == 2) v += __ldcg(csum + (size_t)(q * per + 1) * kP + c);
            part += v;
        }
        m.red[h][c] = part;
        __syncthreads();
        if ((int)threadIdx.x < bs) gs = m.red[0][c] + m.red[1][c] + m.red[2][c] + m.red[3][c];
    }
    if (threadIdx.x < kP) {
        g[threadIdx.x] = gs;
        thr[threadIdx.x] = eps * d0v;
        ids[threadIdx.x] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int t = (int)threadIdx.x + q * kTT;
        Xs[t / kP][t % kP] = t / kP == t % kP ? 1.f : 0.f;
    }
    __syncthreads();
    // micro-panel 0, then per step: warp 0 updates and eliminates the next micro-panel while the
    // other warps apply the current one's rank-8 update to the columns after it, carry the inverse X =
    // L^-1 on by its 8 rows, and write those and the micro-panel's columns of L out.  X starts as the
    // identity: X_I = L_II^-1 X_I (a thread per column, the 8 values in registers), then X_r -= L_rI X_I
    // for the rows r below.  L <= 0 below the diagonal and X >= 0, so every sum has terms of one sign.
    // Done after the elimination (scaling, then an inverse by recursive doubling) this made a factorisation
    // of n = 1024 take 550 us instead of 519; warp 0's chain hides most but not all of it.
    if (warp == 0) {
        if (bs >= kMp) d32_micro_panel<true>(lane, k, 0, kMp, -1, S, g, thr, ids, D);
        else d32_micro_panel<false>(lane, k, 0, bs, -1, S, g, thr, ids, D);
    }
    __syncthreads();
    for (int c0 = 0; c0 < bs; c0 += kMp) {
        const int c1 = c0 + kMp, nc1 = min(kMp, bs - c1);   // micro-panel c0 is full when c1 < bs
        if (warp == 0) {
            if (nc1 == kMp) d32_micro_panel<true>(lane, k, c1, kMp, c0, S, g, thr, ids, D);
            else if (nc1 > 0) d32_micro_panel<false>(lane, k, c1, nc1, c0, S, g, thr, ids, D);
        } else {
            // rank-8 update of the columns l >= lo: S[i][l] -= sum_jj S[i][c] S[l][c] / d_c (i > l),
            // and of their below-block sums: g[l] -= sum_jj (S[l][c] / d_c) g[c].  Thread (ty, tx):
            // the columns la = lo + tx and lb = la + 32 with their 8 factors in registers, the rows
            // lo + ty, +7, ... (each row's 8 entries read once for both columns)
            const int lo = c1 + max(nc1, 0);
            if (lo < bs) {
                const int tx = lane, ty = warp - 1;
                const int la = lo + tx, lb = la + 32;
                float fa[kMp], fb[kMp];
#pragma unroll
                for (int jj = 0; jj < kMp; ++jj) {
                    fa[jj] = (la < bs) ? S[la][c0 + jj] * ids[c0 + jj] : 0.f;
                    fb[jj] = (lb < bs) ? S[lb][c0 + jj] * ids[c0 + jj] : 0.f;
                }
                for (int i = lo + ty; i < bs; i += kTT / 32 - 1) {
                    if (i <= la) continue;
                    float sa = 0.f, sb = 0.f;
#pragma unroll
                    for (int jj = 0; jj < kMp; ++jj) {
                        const float x = S[i][c0 + jj];
                        sa += x * fa[jj];
                        sb += x * fb[jj];
                    }
                    S[i][la] -= sa;
                    if (i > lb) S[i][lb] -= sb;
                }
                if (ty == 0) {
                    float ga = 0.f, gb = 0.f;
#pragma unroll
                    for (int jj = 0; jj < kMp; ++jj) {
                        ga += fa[jj] * g[c0 + jj];
                        gb += fb[jj] * g[c0 + jj];
                    }
                    if (la < bs) g[la] -= ga;
                    if (lb < bs) g[lb] -= gb;
                }
            }
            if (warp == kTT / 32 - 1) {
                // L = S D^-1 (grounded columns are zero) of this micro-panel, back to A
#pragma unroll
                for (int q = 0; q < kMp; ++q) {
                    const int j = c0 + q;
                    const float id = ids[j];
#pragma unroll
                    for (int i = lane; i < kP; i += 32)
                        if (i > j && i < bs) A[(size_t)(k + j) * ld + (k + i)] = S[i][j] * id;
                }
            } else {
                const int c = (int)(threadIdx.x - 32) % kP, part = (int)(threadIdx.x - 32) / kP;   // 3 threads per column
                float x[kMp], xd[kMp];   // X_I, D^-1 X_I
#pragma unroll
                for (int q = 0; q < kMp; ++q) x[q] = Xs[c0 + q][c];
#pragma unroll
                for (int q = 0; q < kMp; ++q) {
#pragma unroll
                    for (int e = 0; e < q; ++e) x[q] -= S[c0 + q][c0 + e] * xd[e];
                    xd[q] = x[q] * ids[c0 + q];
                }
                if (part == 0 && c < bs) {
#pragma unroll
                    for (int q = 0; q < kMp; ++q)
                        if (c0 + q < bs) Linv[(size_t)c * ld + (k + c0 + q)] = x[q];
                }
                if (c < c1) {
#pragma unroll 4
                    for (int r = c1 + part; r < bs; r += 3) {
                        float v = S[r][c0] * xd[0], w = S[r][c0 + 1] * xd[1];
#pragma unroll
                        for (int q = 2; q < kMp; q += 2) {
                            v += S[r][c0 + q] * xd[q];
                            w += S[r][c0 + q + 1] * xd[q + 1];
                        }
                        Xs[r][c] -= v + w;
                    }
                }
            }
        }
        __syncthreads();
    }
}

// L0 != NULL: first the rows [k, k + bs) of the previous panel's L21 (kept in L0 by the step
// kernel, whose other CTAs read those rows of A unscaled) go to A
__global__ void __launch_bounds__(kTT)
d32_diag_kernel(int ld, int k, int bs, float *__restrict__ A, float *__restrict__ D, const float *__restrict__ d0,
                const float *__restrict__ csum, int np, int per, float eps, float *__restrict__ Linv,
                const float *__restrict__ L0) {
    __shared__ __align__(16) float buf[kDiagSmem / 4];
    if (L0)
        for (int t = threadIdx.x; t < kP * kP; t += blockDim.x) {
            const int r = t % kP, j = t / kP;
            if (r < bs) A[(size_t)(k - kP + j) * ld + k + r] = L0[j * kP + r];
        }
    d32_diag_block(diag_smem(buf), ld, k, bs, A, D, d0, csum, np, per, eps, Linv);
}

// block row k of X = L^-1 for the columns [c0, c0+64) of [0, k+bs); 4 rows x 4 columns per thread
__global__ void __launch_bounds__(kTT)
d32_invrow_kernel(int ld, int k, int bs, float *__restrict__ X, const float *__restrict__ Linv) {
    __shared__ __align__(16) float Lt[kP][kP];   // Lt[l][i] = (L11^-1)_il
    __shared__ __align__(16) float B[kP][kP];    // B[l][c] = X(k + l, c0 + c)
    const int c0 = blockIdx.x * kP;
    const int base = k + bs;
    for (int t = threadIdx.x; t < kP * kP; t += blockDim.x) {
        const int i = t % kP, l = t / kP;
        Lt[l][i] = (i < bs && l < bs) ? Linv[(size_t)l * ld + (k + i)] : 0.f;
    }
    for (int t = threadIdx.x; t < kP * kP; t += blockDim.x) {
        const int l = t % kP, c = t / kP;
        B[l][c] = (l < bs && c0 + c < k) ? X[(size_t)(c0 + c) * ld + (k + l)] : 0.f;
    }
    __syncthreads();
    const int ti = threadIdx.x & 15, tcc = threadIdx.x >> 4;  // rows ti*4.., columns tcc*4..
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) acc[u][w] = 0.f;
    if (c0 < k) {
#pragma unroll 16
        for (int l = 0; l < kP; ++l) {
            const float4 a = *(const float4 *)&Lt[l][ti * 4];
            const float4 b = *(const float4 *)&B[l][tcc * 4];
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int w = 0; w < 4; ++w) acc[u][w] += av[u] * bv[w];
        }
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int c = c0 + tcc * 4 + w;
        if (c >= base) continue;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = ti * 4 + u;
            if (i >= bs) continue;
            X[(size_t)c * ld + (k + i)] = c < k ? acc[u][w] : Lt[c - k][i];
        }
    }
}

// The two rank-64 updates of panel k (trailing triangle A22 -= LD L21^T, rows of L^-1 below the
// panel B -= L21 X_k): d32_step_kernel covers the blocks that the chain needs next, d32_update_kernel
// (128x128 tiles, 8x8 per thread) or, two panels at once, d32_tc_update_kernel the rest.
__device__ __forceinline__ void tri_decode(int idx, int &ti, int &tj) {
    ti = (int)((sqrt(8.0 * idx + 1.0) - 1.0) * 0.5);
    while ((ti + 1) * (ti + 2) / 2 <= idx) ++ti;
    while (ti * (ti + 1) / 2 > idx) --ti;
    tj = idx - ti * (ti + 1) / 2;
}

// the rest of the update of panel k, from base2 = base + 128 on.  Launched with kRestPad bytes of shared
// memory that it does not use, which halves an SM's room beside its CTAs: factorisations of n = 4096 take
// 2737 us instead of 2935 and of n = 6400 7.61 ms instead of 7.81 (50 to 60 KB alike, 84 KB leaves one CTA per
// SM: 3228; n = 2025 takes 1063 us either way).  Registers already keep a third CTA off the SM, and
// asking for the same carve-out without the bytes does not do it (2936), so how it favours the chain is not
// explained.
constexpr int kRestPad = 52 * 1024;
__global__ void __launch_bounds__(kTT, 2)
d32_update_kernel(int n, int ld, int k, float *__restrict__ A, float *__restrict__ X,
                  const float *__restrict__ LD) {
    // two stages: slice s + 1 is fetched into registers while slice s is multiplied
    __shared__ __align__(16) float As[2][kKc][kTile];
    __shared__ __align__(16) float Bs[2][kKc][kTile];
    const int base = k + kP, base2 = base + 2 * kP;
    const int t = (n - base2 + kTile - 1) / kTile;   // row / column tiles from base2 on
    const int tcn = (base + kTile - 1) / kTile;      // column tiles of the rows of L^-1
    const int idx = blockIdx.x;
    const int ntri = t * (t + 1) / 2;                // trailing tiles, diagonal ones included
    const bool tri = idx < ntri;
    int ti, tj;
    if (tri) {
        tri_decode(idx, ti, tj);
    } else {
        const int q = idx - ntri;
        ti = q / tcn;
        tj = q % tcn;
    }
    const int r0 = base2 + ti * kTile;
    const int c0 = tri ? base2 + tj * kTile : tj * kTile;
    const int climit = tri ? n : base;
    // A operand (l, r) = Pa[l * ld + r]; B operand (l, c) = Pb[l * ld + c] (trailing) or
    // X[c * ld + k + l] (inverse)
    const float *Pa = tri ? LD : A + (size_t)k * ld;
    const float *Pb = A + (size_t)k * ld;
    const int tr = threadIdx.x & 15, tc = threadIdx.x >> 4;
    float acc[8][8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int w = 0; w < 8; ++w) acc[u][w] = 0.f;
    float ra[8], rb[8];
    const int fl = threadIdx.x >> 4, fq = (threadIdx.x & 15) * 8;       // A (and trailing B) slot
    const int xc = threadIdx.x & (kTile - 1), xh = threadIdx.x >> 7;      // inverse B slot
    const float *pa0 = Pa + (size_t)fl * ld + r0 + fq, *pb0 = Pb + (size_t)fl * ld + c0 + fq;
    auto fetch = [&](int l0) {
        const float *src = pa0 + (size_t)l0 * ld;
        if (r0 + fq + 8 <= n) {
            const float4 v0 = *(const float4 *)src, v1 = *(const float4 *)(src + 4);
            ra[0] = v0.x; ra[1] = v0.y; ra[2] = v0.z; ra[3] = v0.w;
            ra[4] = v1.x; ra[5] = v1.y; ra[6] = v1.z; ra[7] = v1.w;
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) ra[u] = (r0 + fq + u < n) ? src[u] : 0.f;
        }
        if (tri) {
            const float *sb = pb0 + (size_t)l0 * ld;
            if (c0 + fq + 8 <= climit) {
                const float4 v0 = *(const float4 *)sb, v1 = *(const float4 *)(sb + 4);
                rb[0] = v0.x; rb[1] = v0.y; rb[2] = v0.z; rb[3] = v0.w;
                rb[4] = v1.x; rb[5] = v1.y; rb[6] = v1.z; rb[7] = v1.w;
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) rb[u] = (c0 + fq + u < climit) ? sb[u] : 0.f;
            }
        } else if (c0 + xc < climit) {
            const float *sx = X + (size_t)(c0 + xc) * ld + k + l0 + xh * 8;
            const float4 v0 = *(const float4 *)sx, v1 = *(const float4 *)(sx + 4);
            rb[0] = v0.x; rb[1] = v0.y; rb[2] = v0.z; rb[3] = v0.w;
            rb[4] = v1.x; rb[5] = v1.y; rb[6] = v1.z; rb[7] = v1.w;
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) rb[u] = 0.f;
        }
    };
    auto stash = [&](int b) {
        *(float4 *)&As[b][fl][fq] = make_float4(ra[0], ra[1], ra[2], ra[3]);
        *(float4 *)&As[b][fl][fq + 4] = make_float4(ra[4], ra[5], ra[6], ra[7]);
        if (tri) {
            *(float4 *)&Bs[b][fl][fq] = make_float4(rb[0], rb[1], rb[2], rb[3]);
            *(float4 *)&Bs[b][fl][fq + 4] = make_float4(rb[4], rb[5], rb[6], rb[7]);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) Bs[b][xh * 8 + u][xc] = rb[u];
        }
    };
    fetch(0);
    int buf = 0;
    for (int l0 = 0; l0 < kP; l0 += kKc) {
        stash(buf);
        __syncthreads();
        if (l0 + kKc < kP) fetch(l0 + kKc);
#pragma unroll
        for (int l = 0; l < kKc; ++l) {
            const float4 a0 = *(const float4 *)&As[buf][l][tr * 8], a1 = *(const float4 *)&As[buf][l][tr * 8 + 4];
            const float4 b0 = *(const float4 *)&Bs[buf][l][tc * 8], b1 = *(const float4 *)&Bs[buf][l][tc * 8 + 4];
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int w = 0; w < 8; ++w) acc[u][w] += a[u] * b[w];
        }
        buf ^= 1;
    }
    float *C = tri ? A : X;
    const bool full = r0 + kTile <= n && c0 + kTile <= climit && (!tri || r0 > c0);
    if (full) {
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            float *dst = C + (size_t)(c0 + tc * 8 + w) * ld + r0 + tr * 8;
            float4 v0 = *(float4 *)dst, v1 = *(float4 *)(dst + 4);
            v0.x -= acc[0][w]; v0.y -= acc[1][w]; v0.z -= acc[2][w]; v0.w -= acc[3][w];
            v1.x -= acc[4][w]; v1.y -= acc[5][w]; v1.z -= acc[6][w]; v1.w -= acc[7][w];
            *(float4 *)dst = v0;
            *(float4 *)(dst + 4) = v1;
        }
    } else {
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int c = c0 + tc * 8 + w;
            if (c >= climit) continue;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = r0 + tr * 8 + u;
                if (r < n && (!tri || r > c)) C[(size_t)c * ld + r] -= acc[u][w];
            }
        }
    }
}

// ------------------------------------------------------------------ fused panel step
// One launch per panel k (bs = 64, base = k + 64 < n) does what the next diagonal block waits for,
// so the panel-to-panel chain is two kernels (this one and the next diagonal block).  Its units are
// 64-row strips and 64-column blocks, each split over two CTAs (CTA 2 s + h takes half h of unit s),
// so that a CTA's dependent products are 2.5 instead of 4 64x64x64 ones and about 130 CTAs share the
// SMs instead of 65:
//   strip s (rows R = base + 64 s ..), half rows R_h = R[32 h, 32 h + 32): LD[R_h] = A21[R_h] L11^-T
//     and L21[R_h] = LD[R_h] D1^-1 (the panel), then the next panel's 64 columns A22[R_h, R0] -=
//     LD[R_h] L21[R0]^T (R0 = the next panel's rows; L21[R0] recomputed in every CTA from the
//     unscaled A21[R0]) together with the update of the same columns by the npv previous panels that
//     the rest-updates have left to it, -= LD'[R_h] L21'[R0]^T, and the fixed-order partial column sums below the next diagonal block (one row of
//     csum per half: row 2 s + h);
//   X block s - ts (columns C = 64 (s - ts) .. of block row k of L^-1), half columns C_h:
//     X[k, C_h] = L11^-1 B[k, C_h] (the block row), then X[R0, C_h] -= L21[R0] X[k, C_h] +
//     L21'[R0] X[k - 64, C_h] (+ the one before, likewise);
// L21[R0] goes to A with the next diagonal block's kernel (the other CTAs read A21[R0] unscaled).
// What remains of both updates is the rest-update's: d32_update_kernel takes one panel's from base +
// 128 on (npv = 1), d32_tc_update_kernel that of panels p and p + 1 (p even) from block p + 4 on, so
// that block p + 3 gets its part of panel p with step p + 2: npv = 2 for even panels, 1 for odd ones.
constexpr int kHalf = kP / 2;
constexpr int step_smem(int npv) { return ((5 + 3 * npv) * kP * kP / 2 + kP) * 4; }

// acc[u][w] += sum_l a[l][tr * 4 + u] b[l][tc * 4 + w] (64 x 64 operands, [depth][index])
__device__ __forceinline__ void mm64(const float *__restrict__ a, const float *__restrict__ b, float (&acc)[4][4],
                                     int tr, int tc) {
#pragma unroll 16
    for (int l = 0; l < kP; ++l) {
        const float4 x = *(const float4 *)(a + l * kP + tr * 4);
        const float4 y = *(const float4 *)(b + l * kP + tc * 4);
        const float av[4] = {x.x, x.y, x.z, x.w}, bv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w) acc[u][w] += av[u] * bv[w];
    }
}

// 32 x 64 outputs: acc[u][w] += sum_l a[l][tr * 2 + u] b[l][tc * 4 + w] (a's rows SA apart)
template <int SA>
__device__ __forceinline__ void mm_r32(const float *__restrict__ a, const float *__restrict__ b, float (&acc)[2][4],
                                       int tr, int tc) {
#pragma unroll 16
    for (int l = 0; l < kP; ++l) {
        const float2 x = *(const float2 *)(a + l * SA + tr * 2);
        const float4 y = *(const float4 *)(b + l * kP + tc * 4);
        const float av[2] = {x.x, x.y}, bv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w) acc[u][w] += av[u] * bv[w];
    }
}

// 64 x 32 outputs: acc[u][w] += sum_l a[l][tr * 4 + u] b[l][tc * 2 + w] (b: 64 x 32)
__device__ __forceinline__ void mm_c32(const float *__restrict__ a, const float *__restrict__ b, float (&acc)[4][2],
                                       int tr, int tc) {
#pragma unroll 16
    for (int l = 0; l < kP; ++l) {
        const float4 x = *(const float4 *)(a + l * kP + tr * 4);
        const float2 y = *(const float2 *)(b + l * kHalf + tc * 2);
        const float av[4] = {x.x, x.y, x.z, x.w}, bv[2] = {y.x, y.y};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 2; ++w) acc[u][w] += av[u] * bv[w];
    }
}

// tile[l][r] = G[(col0 + l) ld + row0 + r] for r < R and row0 + r < rlim, else 0 (row0 a multiple
// of 4; depth 64, tile stride R)
template <int R>
__device__ __forceinline__ void load_cm(float *__restrict__ tile, const float *__restrict__ G, int ld, int col0,
                                        int row0, int rlim) {
    for (int t = threadIdx.x; t < kP * (R / 4); t += blockDim.x) {
        const int l = t / (R / 4), q = (t % (R / 4)) * 4;
        const float *src = G + (size_t)(col0 + l) * ld + row0 + q;
        float4 v;
        if (row0 + q + 4 <= rlim) v = *(const float4 *)src;
        else {
            v.x = row0 + q < rlim ? src[0] : 0.f;
            v.y = row0 + q + 1 < rlim ? src[1] : 0.f;
            v.z = row0 + q + 2 < rlim ? src[2] : 0.f;
            v.w = row0 + q + 3 < rlim ? src[3] : 0.f;
        }
        *(float4 *)(tile + l * R + q) = v;
    }
}

// tile[l][c] = X(row0 + l, c0 + c) = X[(c0 + c) ld + row0 + l] for c < C and c0 + c < climit, else
// 0 (depth 64, tile stride C)
template <int C>
__device__ __forceinline__ void load_rows_of_x(float *__restrict__ tile, const float *__restrict__ X, int ld,
                                               int row0, int c0, int climit) {
    for (int t = threadIdx.x; t < C * (kP / 4); t += blockDim.x) {
        const int c = t % C, lq = (t / C) * 4;
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c0 + c < climit) w = *(const float4 *)(X + (size_t)(c0 + c) * ld + row0 + lq);
        tile[(lq + 0) * C + c] = w.x;
        tile[(lq + 1) * C + c] = w.y;
        tile[(lq + 2) * C + c] = w.z;
        tile[(lq + 3) * C + c] = w.w;
    }
}

__global__ void __launch_bounds__(kTT)
d32_step_kernel(int n, int ld, int k, int npv, float *__restrict__ A, float *__restrict__ X,
                const float *__restrict__ D, const float *__restrict__ Linv, float *__restrict__ LDc,
                const float *__restrict__ LDprev, const float *__restrict__ LDprev2, float *__restrict__ L0buf,
                float *__restrict__ csum) {
    extern __shared__ __align__(16) float sm[];
    float *idv = sm, *Lt = sm + kP, *T1 = Lt + kP * kP, *T2 = T1 + kP * kHalf;   // T1: 64 x 32
    // per previous panel a 64 x 64 tile and a 64 x 32 one
    float *T4 = T2 + kP * kP, *T3 = T4 + kP * kP, *T6 = T3 + kP * kHalf, *T5 = T6 + kP * kP;
    const int base = k + kP;
    const int ts = (n - base + kP - 1) / kP;
    const int unit = (int)blockIdx.x >> 1, h = (int)blockIdx.x & 1;
    const bool strip = unit < ts;
    const bool prev = npv > 0, prev2 = npv > 1;
    const int tr = threadIdx.x & 15, tc = threadIdx.x >> 4;
    // Lt[l][j] = (L11^-1)_jl; idv = D1^+ (0 for grounded pivots)
    for (int t = threadIdx.x; t < kP * kP; t += blockDim.x) {
        const int j = t % kP, l = t / kP;
        Lt[l * kP + j] = Linv[(size_t)l * ld + (k + j)];
    }
    if (threadIdx.x < kP) {
        const float dj = D[k + threadIdx.x];
        idv[threadIdx.x] = isinf(dj) ? 0.f : 1.f / dj;
    }
    if (strip) {
        const int rb = unit, rh = base + rb * kP + h * kHalf;   // this half's first row
        float acc[2][4], acc2[4][4], acc3[2][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                acc2[u][w] = 0.f;
                if (u < 2) acc[u][w] = acc3[u][w] = 0.f;
            }
        // the A22[R_h, R0] entries this thread updates, loaded with the operands (no other CTA of
        // this launch, and no rest-update running beside it, writes them)
        float cur[2][4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int c = base + tc * 4 + w;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int r = rh + tr * 2 + u;
                cur[u][w] = (c < n && r < n && r > c) ? A[(size_t)c * ld + r] : 0.f;
            }
        }
        if (rb > 0) load_cm<kHalf>(T1, A, ld, k, rh, n);       // A21[R_h]     [l][r], r < 32
        load_cm<kP>(T2, A, ld, k, base, n);                     // A21[R0]      [l][c]
        if (prev) {
            load_cm<kHalf>(T3, LDprev, ld, 0, rh, n);           // LD'[R_h]     [j][r]
            load_cm<kP>(T4, A, ld, k - kP, base, n);            // L21'[R0]     [j][c]
        }
        if (prev2) {
            load_cm<kHalf>(T5, LDprev2, ld, 0, rh, n);
            load_cm<kP>(T6, A, ld, k - 2 * kP, base, n);
        }
        __syncthreads();
        // LD(R_h row tr*2+u, j = tc*4+w) (the first strip's rows are R0's: read from T2)
        if (rb > 0) mm_r32<kHalf>(T1, Lt, acc, tr, tc);
        else mm_r32<kP>(T2 + h * kHalf, Lt, acc, tr, tc);
        mm64(T2, Lt, acc2, tr, tc);                             // LD(R0 row tr*4+u, j = tc*4+w)
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int j = tc * 4 + w;
            const float id = idv[j];
            const bool inf = id == 0.f;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int rr = tr * 2 + u, r = rh + rr;
                const float ldv = inf ? 0.f : acc[u][w];
                if (r < n) {
                    LDc[(size_t)j * ld + r] = ldv;
                    if (rb == 0) L0buf[j * kP + h * kHalf + rr] = acc[u][w] * id;
                    else A[(size_t)(k + j) * ld + r] = acc[u][w] * id;
                }
                T1[j * kHalf + rr] = ldv;                                   // A operand [j][r]
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) T2[j * kP + tr * 4 + u] = acc2[u][w] * id;   // B operand [j][c]
        }
        __syncthreads();
        mm_r32<kHalf>(T1, T2, acc3, tr, tc);
        if (prev) mm_r32<kHalf>(T3, T4, acc3, tr, tc);
        if (prev2) mm_r32<kHalf>(T5, T6, acc3, tr, tc);
        // A22[R_h, R0] -= acc3 below the diagonal; column sums of the rows below the next block
        float cs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int c = base + tc * 4 + w;
            if (c >= n) continue;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int r = rh + tr * 2 + u;
                if (r < n && r > c) {
                    const float v = cur[u][w] - acc3[u][w];
                    A[(size_t)c * ld + r] = v;
                    if (r >= base + kP) cs[w] += v;
                }
            }
        }
        // the 16 threads with this tc are one half-warp (lanes tr = 0..15)
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            float v = cs[w];
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (tr == 0) csum[(size_t)(2 * rb + h) * kP + tc * 4 + w] = v;
        }
    } else {
        const int cb = unit - ts, c0 = cb * kP, ch = c0 + h * kHalf;   // this half's first column
        const bool before = c0 < k;                           // columns left of the diagonal block
        float acc[4][2], acc2[4][4], acc3[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                acc2[u][w] = 0.f;
                if (w < 2) acc[u][w] = acc3[u][w] = 0.f;
            }
        // the X[R0, C_h] entries this thread updates, loaded with the operands
        float cur[4][2];
#pragma unroll
        for (int w = 0; w < 2; ++w)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = base + tr * 4 + u;
                cur[u][w] = r < n ? X[(size_t)(ch + tc * 2 + w) * ld + r] : 0.f;
            }
        if (before) load_rows_of_x<kHalf>(T1, X, ld, k, ch, k);     // B[k, C_h]      [l][c], c < 32
        load_cm<kP>(T2, A, ld, k, base, n);                          // A21[R0]        [l][r]
        if (prev && before) {
            load_cm<kP>(T4, A, ld, k - kP, base, n);                 // L21'[R0]       [j][r]
            load_rows_of_x<kHalf>(T3, X, ld, k - kP, ch, k);         // X[k - 64, C_h] [j][c]
        }
        if (prev2 && before) {
            load_cm<kP>(T6, A, ld, k - 2 * kP, base, n);
            load_rows_of_x<kHalf>(T5, X, ld, k - 2 * kP, ch, k - kP);
        }
        __syncthreads();
        if (before) mm_c32(Lt, T1, acc, tr, tc);              // X(k + i, c), i = tr*4+u, c = tc*2+w
        mm64(T2, Lt, acc2, tr, tc);                           // LD(R0_r, j), r = tr*4+u, j = tc*4+w
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const int i = tr * 4 + u, c = tc * 2 + w;
                const float x = before ? acc[u][w] : Lt[(h * kHalf + c) * kP + i];
                X[(size_t)(ch + c) * ld + (k + i)] = x;
                T1[i * kHalf + c] = x;                                       // B operand [i][c]
            }
#pragma unroll
            for (int w = 0; w < 4; ++w)
                T2[(tc * 4 + w) * kP + tr * 4 + u] = acc2[u][w] * idv[tc * 4 + w];  // A operand [j][r]
        }
        __syncthreads();
        mm_c32(T2, T1, acc3, tr, tc);
        if (prev && before) mm_c32(T4, T3, acc3, tr, tc);
        if (prev2 && before) mm_c32(T6, T5, acc3, tr, tc);
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int c = ch + tc * 2 + w;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = base + tr * 4 + u;
                if (r < n) X[(size_t)c * ld + r] = cur[u][w] - acc3[u][w];
            }
        }
    }
}

// ------------------------------------------------------------------ tensor-core bulk update
// The rest-update C -= A_op B_op^T of two panels (depth 128) on the fifth-generation tensor cores, each
// FP32 operand as the sum of three BF16 pieces (8 + 8 + 8 bits: exact) a = a1 + a2 + a3 and C -= a1 b1 +
// (a1 b2 + a2 b1 + a1 b3 + a3 b1 + a2 b2) (what is left out is 2^-24 of a b and below).  The tensor cores
// truncate a sum that they add to, and here all terms have one sign, so every MMA into an accumulator
// costs it a part of its last place.  So the five small products of both panels go to one accumulator
// before anything large does, a1 b1 of the first panel to another and a1 b1 of the second, last, on top of the
// small ones: four MMAs into a large sum.  Relative
// error of X = L^-1 against FP64 at n = 8281 (RMS, largest): 6.5e-7, 3.2e-6; 1.2e-6, 4.8e-6 with all of a1 b1
// in one accumulator; 1.5e-6, 4.4e-6 with two TF32 pieces, one panel, and 24 MMAs into one (2.5e-6, 7.5e-6 for
// two panels).  The FP32 SIMT update has 2.4e-7, 2.2e-6 and stays below n = 8192, where it was the choice
// before; from there on it takes 15.6 ms against 7.4.
// Once per panel the operands are split and written in the MMA's shared-memory layout (K-major,
// no swizzle: core matrices of 8 rows x 8 depths (16 bytes), (row / 8, k / 8) of a 128-row piece of 16
// depths at byte ((k / 8) 16 + row / 8) 128, row row % 8 at 16-byte steps), the three pieces of 16 depths
// together, so that a stage is two bulk copies completing on one mbarrier.
constexpr int kTcM = 128;                             // tile rows and columns
constexpr int kTcK = 16, kTcStages = 4;               // depth of a stage, stages of the ring
constexpr int kTcPiece = kTcM * kTcK * 2;             // one BF16 piece of a stage: 4 KB
constexpr int kTcOperand = 3 * kTcPiece;              // one operand of a stage
constexpr int kTcStage = 2 * kTcOperand;
constexpr int kTcBlock = kP / kTcK * kTcOperand;      // 128 rows of one panel's operand: 48 KB
constexpr int kTcPer = 2 * kP / kTcK;                 // stages of a tile: two panels
constexpr int kTcSmem = 116 * 1024;   // 96 KB used; more than half an SM's, so that a CTA cannot start beside
                                      // another one that holds all of the tensor memory
static_assert(kTcSmem >= kTcStages * kTcStage + 128 && 2 * kTcSmem > 228 * 1024, "stages and barriers");
static_assert(kTcPer == 2 * kTcStages, "the ring holds a panel");
constexpr int kTcAutoN = 8192;    // tc_mode 0: the tensor-core update from this n on
constexpr uint32_t kTcIdesc = tc_idesc(kTcM, kTcM);   // BF16, both K-major

// Split operands of one panel in blocks of 128 rows: LD rows (A of the trailing tiles), panel rows (their
// B, and A of the inverse's tiles), rows of L^-1 by column (B of the inverse's)
struct TcOps { unsigned char *LDs, *Ps, *Xs; };
__host__ __device__ __forceinline__ size_t tc_op_bytes(int n) { return (size_t)ceil_div(n, kTcM) * kTcBlock; }
__host__ __device__ __forceinline__ size_t tc_per_panel(int n) { return 3 * tc_op_bytes(n); }
__host__ __device__ __forceinline__ TcOps tc_ops(unsigned char *buf, int n) {
    return {buf, buf + tc_op_bytes(n), buf + 2 * tc_op_bytes(n)};
}

// depths 8 kg .. 8 kg + 7 of row r, split into its three pieces
__device__ __forceinline__ void tc_put(unsigned char *op, int r, int kg, const float (&v)[8]) {
    uint32_t w[3][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        float x = v[q];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const __nv_bfloat16 b = __float2bfloat16(x);
            x -= __bfloat162float(b);
            const uint32_t u = __bfloat16_as_ushort(b);
            w[e][q >> 1] = q & 1 ? w[e][q >> 1] | (u << 16) : u;
        }
    }
    unsigned char *at = op + (size_t)(r / kTcM) * kTcBlock + (kg >> 1) * kTcOperand + ((kg & 1) * 16 + (r % kTcM) / 8) * 128 +
                        (r & 7) * 16;
#pragma unroll
    for (int e = 0; e < 3; ++e) *(uint4 *)(at + e * kTcPiece) = make_uint4(w[e][0], w[e][1], w[e][2], w[e][3]);
}

// The split operands of panels k0 and k0 + 64 (blockIdx.y) for the rest-update from base2 on, 128 rows per
// CTA: first the rows of LD and of the panel (T blocks; rows at or beyond n are zero), then the columns
// of the panel's block row of L^-1 (zero from the panel's end on).
__global__ void __launch_bounds__(kTT)
d32_tc_split_kernel(int n, int ld, int k0, int base2, int T, const float *__restrict__ A, const float *__restrict__ X,
                    const float *__restrict__ LD0, const float *__restrict__ LD1, unsigned char *__restrict__ buf) {
    const int k = k0 + (int)blockIdx.y * kP, base = k + kP;
    const float *LD = blockIdx.y ? LD1 : LD0, *P = A + (size_t)k * ld;
    const TcOps o = tc_ops(buf + blockIdx.y * tc_per_panel(n), n);
    const bool rows = (int)blockIdx.x < T;
    const int b0 = ((int)blockIdx.x - (rows ? 0 : T)) * kTcM;
    float v[8];
    if (rows) {
        for (int t = threadIdx.x; t < kTcM * (kP / 8); t += kTT) {
            const int r = b0 + t % kTcM, kg = t / kTcM, row = base2 + r;
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = row < n ? P[(size_t)(kg * 8 + q) * ld + row] : 0.f;
            tc_put(o.Ps, r, kg, v);
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = row < n ? LD[(size_t)(kg * 8 + q) * ld + row] : 0.f;
            tc_put(o.LDs, r, kg, v);
        }
    } else {
        // a warp takes 8 columns by 32 rows at a time: 128-byte reads, 128-byte writes
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int t = warp; t < kTcM / 8 * (kP / 32); t += kTT / 32) {
            const int r = b0 + (t / (kP / 32)) * 8 + (lane & 7), kg = (t % (kP / 32)) * 4 + (lane >> 3);
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
            if (r < base) {
                const float4 *src = (const float4 *)(X + (size_t)r * ld + k + kg * 8);
                x = src[0];
                y = src[1];
            }
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
            tc_put(o.Xs, r, kg, v);
        }
    }
}

// Tile t of a rest-update: T (T + 1) / 2 tiles of the trailing triangle from base2, then T x tcx tiles of the
// rows of L^-1 (C = X, columns below base)
struct TcTile { bool tri; int ti, tj, r0, c0, climit; };
__device__ __forceinline__ TcTile tc_tile(int t, int n, int base, int base2, int T, int tcx) {
    TcTile q;
    const int ntri = T * (T + 1) / 2;
    q.tri = t < ntri;
    if (q.tri) {
        int ti = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
        while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
        while (ti * (ti + 1) / 2 > t) --ti;
        q.ti = ti;
        q.tj = t - ti * (ti + 1) / 2;
    } else {
        q.ti = (t - ntri) / tcx;
        q.tj = (t - ntri) % tcx;
    }
    q.r0 = base2 + q.ti * kTcM;
    q.c0 = q.tri ? base2 + q.tj * kTcM : q.tj * kTcM;
    q.climit = q.tri ? n : base;
    return q;
}

// Persistent CTAs (one per SM), each taking tiles gridDim.x apart, warp-specialised.  One lane of warp 17
// brings the operands through a ring of four stages of 16 depths (two bulk copies on the stage's "load"
// mbarrier); one lane of warp 16 issues the MMAs into one of two pairs of accumulators, committing a
// stage's last to its "free" mbarrier and a tile's last to the pair's "full"; warps 0-15 wait for that,
// subtract the pair's sum from C and arrive on its "empty".  So the next tile's copies and MMAs run while a
// tile's epilogue does, and each epilogue warp requests its 32 columns of the next tile's C as soon as it has
// written this one's.
// Every wait is bounded: one that gives up records the failure in *err and the CTA winds down (its own
// copies and MMAs waited for once more) before it releases the tensor memory.
// What bounds it is C, 64 KB read and 64 KB written per tile, in bursts.  n = 16,384, whole factorisation: 74 ms
// with four epilogue warps (16 KB of C in flight per SM), one panel per pass and TF32 (66 of them in this
// kernel, 2.7 TB/s of C); 47 with sixteen warps; 34.8 with two panels per pass; 34.0 so.  n = 8281: 14.1 ->
// 7.4 ms; with a third of the panels done, 50 us per two panels, DRAM at 44 %, the tensor pipe at 41 %.
// Bringing and storing C by bulk copies instead was slower (49 and 60 ms: 512-byte copies take about 60
// clocks each), and so was keeping A in shared memory along a tile row (47 ms: no room for the accumulators'
// second pair).
constexpr int kTcEpi = 16, kTcThreads = (kTcEpi + 2) * 32;
constexpr int kTcCols = kTcM / (kTcEpi / 4);   // columns of one epilogue warp

__global__ void __launch_bounds__(kTcThreads, 1)
d32_tc_update_kernel(int n, int ld, int base, int base2, int T, unsigned char *__restrict__ ops, float *__restrict__ A,
                     float *__restrict__ X, int *__restrict__ err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tcx = (int)ceil_div(base, kTcM), ntiles = T * (T + 1) / 2 + T * tcx, step = (int)gridDim.x;
    // load, free (kTcStages each), full, empty (one per pair of accumulators each)
    uint64_t *mbs = (uint64_t *)(smem + kTcStages * kTcStage);
    uint32_t *tslot = (uint32_t *)(mbs + 2 * kTcStages + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) tc_alloc(tslot, 4 * kTcM);
    const uint32_t sbase = tc_smem_u32(smem), mload = tc_smem_u32(mbs), mfree = mload + 8 * kTcStages;
    const uint32_t mfull = mfree + 8 * kTcStages, mempty = mfull + 16;
    if (threadIdx.x == 0) {
        for (int q = 0; q < 2 * kTcStages + 2; ++q) tc_mbar_init(mload + 8 * q, 1);
        for (int q = 0; q < 2; ++q) tc_mbar_init(mempty + 8 * q, kTcEpi);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    auto copy = [](uint32_t dst, const void *src, uint32_t bytes, uint32_t mb) {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     :: "r"(dst), "l"(src), "r"(bytes), "r"(mb) : "memory");
    };
    auto expect = [](uint32_t mb, uint32_t bytes) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mb), "r"(bytes) : "memory");
    };
    if (warp == kTcEpi) {
        if (lane == 0) {
            const uint64_t d0 = tc_desc(sbase, (kTcM / 8) * 128);
            constexpr uint32_t kPieceD = kTcPiece >> 4, kStageD = kTcStage >> 4;   // in the descriptor's address units
            bool ok = true;
            int g = 0, i = 0;   // stages whose last MMA is committed, tiles
            for (int t = (int)blockIdx.x; t < ntiles && ok; t += step, ++i) {
                const int bsel = i & 1;
                const uint32_t first = tmem + (uint32_t)(bsel * 2 * kTcM), second = first + kTcM;
                // the accumulators are free once the epilogue of tile i - 2 is done
                if (i >= 2 && !tc_wait(mempty + 8 * bsel, (uint32_t)(((i - 2) >> 1) & 1))) { ok = false; break; }
#pragma unroll
                for (int q = 0; q < kTcPer + kTcStages; ++q) {
                    // stages of panel 0, of panel 1 without a1 b1, then a1 b1 of panel 1
                    const int slot = q % kTcStages;
                    const uint64_t a0 = d0 + slot * kStageD, a1 = a0 + kPieceD, a2 = a1 + kPieceD;
                    const uint64_t b0 = a2 + kPieceD, b1 = b0 + kPieceD, b2 = b1 + kPieceD;
                    if (q < kTcPer) {
                        if (!tc_wait(mload + 8 * slot, (uint32_t)((2 * i + q / kTcStages) & 1))) { ok = false; break; }
                        tc_fence_after();
                        tc_mma(second, a0, b2, kTcIdesc, q > 0);
                        tc_mma(second, a2, b0, kTcIdesc, true);
                        tc_mma(second, a1, b1, kTcIdesc, true);
                        tc_mma(second, a0, b1, kTcIdesc, true);
                        tc_mma(second, a1, b0, kTcIdesc, true);
                    }
                    if (q < kTcStages) tc_mma(first, a0, b0, kTcIdesc, q > 0);
                    if (q >= kTcPer) tc_mma(second, a0, b0, kTcIdesc, true);
                    if (q < kTcStages || q >= kTcPer) {
                        tc_commit(mfree + 8 * slot);
                        ++g;
                    }
                }
                if (ok) tc_commit(mfull + 8 * bsel);
            }
            if (!ok) {
                atomicExch(err, 1);
                tc_commit(mfree + 8 * (g % kTcStages));   // the MMAs issued since the last commit
                ++g;
            }
            // before the CTA ends: the last MMAs (bounded)
            if (g > 0) tc_wait(mfree + 8 * ((g - 1) % kTcStages), (uint32_t)(((g - 1) / kTcStages) & 1));
        }
    } else if (warp == kTcEpi + 1) {
        if (lane == 0) {
            bool ok = true;
            int g = 0;   // stages requested
            for (int t = (int)blockIdx.x; t < ntiles && ok; t += step) {
                const TcTile q = tc_tile(t, n, base, base2, T, tcx);
                for (int p = 0; p < 2 && ok; ++p) {
                    const TcOps o = tc_ops(ops + p * tc_per_panel(n), n);
                    const unsigned char *pa = (q.tri ? o.LDs : o.Ps) + (size_t)q.ti * kTcBlock;
                    const unsigned char *pb = (q.tri ? o.Ps : o.Xs) + (size_t)q.tj * kTcBlock;
                    for (int e = 0; e < kP / kTcK; ++e, ++g) {
                        const uint32_t slot = (uint32_t)(g % kTcStages), mb = mload + 8 * slot;
                        if (g >= kTcStages && !tc_wait(mfree + 8 * slot, (uint32_t)((g / kTcStages - 1) & 1))) { ok = false; break; }
                        expect(mb, (uint32_t)kTcStage);
                        copy(sbase + slot * kTcStage, pa + e * kTcOperand, (uint32_t)kTcOperand, mb);
                        copy(sbase + slot * kTcStage + kTcOperand, pb + e * kTcOperand, (uint32_t)kTcOperand, mb);
                    }
                }
            }
            if (!ok) atomicExch(err, 1);
            // before the CTA ends: its copies in flight (bounded)
            for (int q = max(0, g - kTcStages); q < g; ++q) tc_wait(mload + 8 * (q % kTcStages), (uint32_t)((q / kTcStages) & 1));
        }
    } else {
        // epilogue warps: warp w owns tensor-memory lanes (tile rows) 32 (w % 4) .. + 31 and columns
        // kTcCols (w / 4) .. + kTcCols - 1
        const int wrow = (warp & 3) * 32, wcol = (warp >> 2) * kTcCols;
        float cv[kTcCols];
        // this warp's part of a tile: first entry of row r and the columns it has an entry in
        auto place = [&](int t, float *&C, int &live) {
            const TcTile q = tc_tile(t, n, base, base2, T, tcx);
            const int r = q.r0 + wrow + lane, c0 = q.c0 + wcol;
            C = (q.tri ? A : X) + (size_t)c0 * ld + r;
            live = r < n ? (q.tri ? min(q.climit, r) : q.climit) - c0 : 0;
        };
        auto fetch = [&](const float *C, int live, int j0) {
#pragma unroll
            for (int j = j0; j < j0 + 16; ++j) cv[j] = j < live ? C[(size_t)j * ld] : 0.f;
        };
        float *C = nullptr, *Cn = nullptr;
        int live = 0, liven = 0, i = 0;
        if ((int)blockIdx.x < ntiles) place((int)blockIdx.x, C, live);
        fetch(C, live, 0);
        fetch(C, live, 16);
        for (int t = (int)blockIdx.x; t < ntiles; t += step, ++i) {
            const int bsel = i & 1;
            liven = 0;
            if (t + step < ntiles) place(t + step, Cn, liven);
            if (!__all_sync(0xffffffffu, tc_wait(mfull + 8 * bsel, (uint32_t)((i >> 1) & 1)))) {
                if (lane == 0) atomicExch(err, 1);
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + ((uint32_t)wrow << 16) + (uint32_t)(bsel * 2 * kTcM + wcol);
#pragma unroll
            for (int j0 = 0; j0 < kTcCols; j0 += 16) {
                float u[16];
                tc_ld16x2(acc + (uint32_t)j0, kTcM, u);   // first + second
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j0 + j < live) C[(size_t)(j0 + j) * ld] = cv[j0 + j] - u[j];
                fetch(Cn, liven, j0);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) tc_arrive(mempty + 8 * bsel);
            C = Cn;
            live = liven;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tc_dealloc(tmem, 4 * kTcM);
}

// partial sums of y = X r: CTA (rb, cb) covers rows [rb*256, +256) (four per thread, float4 loads)
// and columns [cb*64, +64) for the lower-triangle tiles only (rows beyond n read the zero padding);
// the tile's 64 columns are split over four thread groups of 16 columns, reduced in shared memory
constexpr int kFr = 256, kFc = 64;
__global__ void __launch_bounds__(kFr)
d32_fwd_kernel(int n, int ld, int ncb, const float *__restrict__ X, const double *__restrict__ r,
               float *__restrict__ part) {
    __shared__ float rs[kFc];
    __shared__ float4 red[3][kFr / 4];
    // tile index -> (rb, cb) with cb*kFc < (rb+1)*kFr
    const int per = kFr / kFc;
    int idx = blockIdx.x, rb = 0;
    while (idx >= min(ncb, (rb + 1) * per)) { idx -= min(ncb, (rb + 1) * per); ++rb; }
    const int cb = idx;
    const int rq = threadIdx.x & (kFr / 4 - 1), cg = threadIdx.x / (kFr / 4);
    const int c0 = cb * kFc, i = rb * kFr + rq * 4;
    if (threadIdx.x < kFc) rs[threadIdx.x] = c0 + (int)threadIdx.x < n ? (float)r[c0 + threadIdx.x] : 0.f;
    __syncthreads();
    const bool live = i < n && i + 3 >= c0;
    const int jn = min(kFc, n - c0);
    const int jlo = cg * (kFc / 4), jhi = min(jlo + kFc / 4, jn);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) {
        const float *col = X + (size_t)c0 * ld + i;
        if (i >= c0 + kFc - 1) {
#pragma unroll 16
            for (int jj = jlo; jj < jhi; ++jj) {
                const float4 v = *(const float4 *)(col + (size_t)jj * ld);
                const float rj = rs[jj];
                acc.x += v.x * rj; acc.y += v.y * rj; acc.z += v.z * rj; acc.w += v.w * rj;
            }
        } else {
            for (int jj = jlo; jj < jhi; ++jj) {
                const int j = c0 + jj;
                const float4 v = *(const float4 *)(col + (size_t)jj * ld);
                const float rj = rs[jj];
                if (j <= i) acc.x += v.x * rj;
                if (j <= i + 1) acc.y += v.y * rj;
                if (j <= i + 2) acc.z += v.z * rj;
                if (j <= i + 3) acc.w += v.w * rj;
            }
        }
    }
    if (cg > 0) red[cg - 1][rq] = acc;
    __syncthreads();
    if (cg == 0 && live) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 o = red[q][rq];
            acc.x += o.x; acc.y += o.y; acc.z += o.z; acc.w += o.w;
        }
        *(float4 *)(part + (size_t)cb * ld + i) = acc;
    }
}

// w = D^+ y, y_i = sum of the partials of row i (fixed order)
__global__ void d32_mid_kernel(int n, int ld, const float *__restrict__ part, const float *__restrict__ D,
                               float *__restrict__ w) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int last = i / kFc;
    float y = 0.f;
    for (int cb = 0; cb <= last; ++cb) y += part[(size_t)cb * ld + i];
    const float d = D[i];
    w[i] = isinf(d) ? 0.f : y / d;
}

// z_j = sum_{i >= j} X_ij w_i, one warp per column, float4 per lane
__global__ void __launch_bounds__(kTT)
d32_bwd_kernel(int n, int ld, const float *__restrict__ X, const float *__restrict__ w, double *__restrict__ z) {
    const int j = blockIdx.x * (kTT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= n) return;
    const float *col = X + (size_t)j * ld;
    float acc = 0.f;
    const int i0 = j & ~3;
#pragma unroll 4
    for (int i = i0 + lane * 4; i < n; i += 128) {
        const float4 v = *(const float4 *)(col + i);
        if (i >= j && i + 3 < n) {
            acc += v.x * w[i] + v.y * w[i + 1] + v.z * w[i + 2] + v.w * w[i + 3];
        } else {
            if (i >= j && i < n) acc += v.x * w[i];
            if (i + 1 >= j && i + 1 < n) acc += v.y * w[i + 1];
            if (i + 2 >= j && i + 2 < n) acc += v.z * w[i + 2];
            if (i + 3 >= j && i + 3 < n) acc += v.w * w[i + 3];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) z[j] = (double)acc;
}

}  // namespace

Error d32_alloc(Dense32 &F, int32_t n) {
    F.n = n;
    F.ld = (n + 31) / 32 * 32;
    const size_t big = sizeof(float) * (size_t)F.ld * n;
    OT_CUDA(cudaMalloc((void **)&F.A, big));
    OT_CUDA(cudaMalloc((void **)&F.X, big));
    OT_CUDA(cudaMalloc((void **)&F.LD, 3 * sizeof(float) * (size_t)F.ld * kP));
    OT_CUDA(cudaMalloc((void **)&F.Linv, sizeof(float) * (size_t)F.ld * kP));
    OT_CUDA(cudaMalloc((void **)&F.D, sizeof(float) * n));
    OT_CUDA(cudaMalloc((void **)&F.d0, sizeof(float) * n));
    // partial column sums: up to two rows (one per half strip) per 64-row strip
    OT_CUDA(cudaMalloc((void **)&F.csum, sizeof(float) * 2 * kP * (size_t)ceil_div(n, kP)));
    OT_CUDA(cudaMalloc((void **)&F.L0, sizeof(float) * kP * kP));
    OT_CUDA(cudaMalloc((void **)&F.w, sizeof(float) * n));
    OT_CUDA(cudaMalloc((void **)&F.part, sizeof(float) * (size_t)F.ld * (size_t)ceil_div(n, kFc)));
    // lower bound of the unwritten upper parts, so that nothing uninitialised is ever read
    OT_CUDA(cudaMemset(F.A, 0, big));
    OT_CUDA(cudaMemset(F.LD, 0, 3 * sizeof(float) * (size_t)F.ld * kP));
    OT_CUDA(cudaMemset(F.Linv, 0, sizeof(float) * (size_t)F.ld * kP));
    // the largest limits any n of this path needs (a per-n value set by one handle could undercut
    // another handle's launch on another thread), for the current device
    OT_CUDA(cudaFuncSetAttribute(d32_assemble_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(unsigned long long) * kSlice)));
    OT_CUDA(cudaFuncSetAttribute(d32_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRestPad));
    OT_CUDA(cudaFuncSetAttribute(d32_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, step_smem(2)));
    if (n > kMaxN) return fail(OT_ERR_ARG, "dense32: n above the supported size");
    return ok();
}

void d32_free(Dense32 &F) {
    if (F.graph) cudaGraphExecDestroy(F.graph);
    for (void *p : {(void *)F.A, (void *)F.X, (void *)F.LD, (void *)F.Linv, (void *)F.D, (void *)F.d0, (void *)F.csum,
                    (void *)F.L0, (void *)F.w, (void *)F.part, (void *)F.tc, (void *)F.tc_err})
        if (p) cudaFree(p);
    if (F.tc_err_host) cudaFreeHost(F.tc_err_host);
    F = Dense32();
}

Error d32_assemble(Dense32 &F, const Newton &W, const Support &S, cudaStream_t st) {
    const int n = F.n;
    const int slices = (int)ceil_div(n, kSlice);
    const size_t smem = sizeof(unsigned long long) * std::min(n, kSlice);
    if (slices == 1) {
        d32_assemble_kernel<<<n, kTT, smem, st>>>(n, F.ld, S.col_ptr, S.col_row, W.theta_col, S.row_ptr, S.j,
                                                   W.theta, W.Minv, W.N, F.A, F.d0, nullptr);
        OT_LAUNCHED();
        return ok();
    }
    DevTemp<unsigned long long> tot;
    OT_TRY(tot.alloc(n, st));
    OT_CUDA(cudaMemsetAsync(tot.p, 0, sizeof(unsigned long long) * n, st));
    d32_assemble_kernel<<<dim3(n, slices), kTT, smem, st>>>(n, F.ld, S.col_ptr, S.col_row, W.theta_col, S.row_ptr,
                                                             S.j, W.theta, W.Minv, W.N, F.A, F.d0, tot.p);
    OT_LAUNCHED();
    d32_diag_total_kernel<<<(unsigned)ceil_div(n, kTT), kTT, 0, st>>>(n, W.N, tot.p, F.d0);
    OT_LAUNCHED();
    return ok();
}

// The factorisation's launch sequence for this n as an explicit CUDA graph: a chain of kernel
// nodes built with the graph API (no stream capture, so nothing another host thread does, such as
// a device-synchronising cudaFree, can invalidate it).
namespace {
struct Dag {
    cudaGraph_t g = nullptr;
    int64_t nodes = 0;
    cudaError_t err = cudaSuccess;
    template <typename... Args>
    cudaGraphNode_t kernel_grid(std::vector<cudaGraphNode_t> deps, void (*fn)(Args...), dim3 grid, unsigned block,
                                unsigned smem, Args... args) {
        cudaGraphNode_t node = nullptr;
        if (err != cudaSuccess) return node;
        void *ptrs[] = {(void *)&args...};
        cudaKernelNodeParams kp = {};
        kp.func = (void *)fn;
        kp.gridDim = grid;
        kp.blockDim = dim3(block);
        kp.sharedMemBytes = smem;
        kp.kernelParams = ptrs;
        kp.extra = nullptr;
        deps.erase(std::remove(deps.begin(), deps.end(), nullptr), deps.end());
        err = cudaGraphAddKernelNode(&node, g, deps.data(), deps.size(), &kp);
        if (err == cudaSuccess) ++nodes;
        return node;
    }
    template <typename... Args>
    cudaGraphNode_t kernel(std::vector<cudaGraphNode_t> deps, void (*fn)(Args...), unsigned grid, unsigned block,
                           Args... args) {
        return kernel_grid(deps, fn, dim3(grid), block, 0u, args...);
    }
    // launch priority of a kernel node (stream-priority scale: lower values run first)
    void priority(cudaGraphNode_t node, int value) {
        if (err != cudaSuccess || !node) return;
        cudaKernelNodeAttrValue v = {};
        v.priority = value;
        err = cudaGraphKernelNodeSetAttribute(node, cudaKernelNodeAttributePriority, &v);
    }
    cudaGraphNode_t memset0(float *dst, size_t count, std::vector<cudaGraphNode_t> deps) {
        cudaGraphNode_t node = nullptr;
        if (err != cudaSuccess) return node;
        cudaMemsetParams mp = {};
        mp.dst = dst;
        mp.value = 0;
        mp.elementSize = sizeof(float);
        mp.width = count;
        mp.height = 1;
        mp.pitch = 0;
        err = cudaGraphAddMemsetNode(&node, g, deps.data(), deps.size(), &mp);
        if (err == cudaSuccess) ++nodes;
        return node;
    }
    cudaGraphNode_t join(std::vector<cudaGraphNode_t> deps) {
        cudaGraphNode_t node = nullptr;
        if (err != cudaSuccess) return node;
        deps.erase(std::remove(deps.begin(), deps.end(), nullptr), deps.end());
        err = cudaGraphAddEmptyNode(&node, g, deps.data(), deps.size());
        return node;
    }
};
}  // namespace

static Error d32_build(Dense32 &F, float eps, cudaGraph_t g, int64_t *nodes) {
    const int n = F.n, ld = F.ld;
    Dag c;
    c.g = g;
    cudaGraphNode_t prev = c.memset0(F.X, (size_t)ld * n, {});
    int lo_prio = 0, hi_prio = 0;
    if (cudaDeviceGetStreamPriorityRange(&lo_prio, &hi_prio) != cudaSuccess) lo_prio = hi_prio = 0;
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 1;
    // The first diagonal block, then one fused step and the next diagonal block per panel on the chain,
    // the rest of the updates beside it and in order.  SIMT: one rest-update per panel, which the
    // step two panels on waits for (it covered its columns).  Tensor cores: one per two panels p, p + 1
    // (p even), from block p + 4 on, which step p + 3 waits for; their operands are split behind step
    // p + 1 into buffers that alternate (the rest-update before may still read the other).  Three LD
    // buffers: a rest-update (or split) still reads its panels' while the next steps write theirs.
    const int bs0 = std::min(kP, n);
    prev = c.kernel({prev}, d32_colsum_kernel, (unsigned)bs0, kTT, n, ld, bs0, (const float *)F.A, F.csum);
    cudaGraphNode_t chain = c.kernel({prev}, d32_diag_kernel, 1u, kTT, ld, 0, bs0, F.A, F.D, (const float *)F.d0,
                                     (const float *)F.csum, 1, 1, eps, F.Linv, (const float *)nullptr);
    c.priority(chain, hi_prio);
    cudaGraphNode_t rest1 = nullptr, rest2 = nullptr;   // the newest rest-update and the one before
    int k = 0, p = 0;
    for (; k + kP < n; k += kP, ++p) {
        const int base = k + kP;
        const int ts = (int)ceil_div(n - base, kP), tx = (int)ceil_div(base, kP);
        float *LDc = F.LD + (size_t)(p % 3) * ld * kP;
        float *LDprev = F.LD + (size_t)((p + 2) % 3) * ld * kP, *LDprev2 = F.LD + (size_t)((p + 1) % 3) * ld * kP;
        const int npv = std::min(p, F.use_tc && p % 2 == 0 ? 2 : 1);
        // the rest-update that covered this step's columns last
        const cudaGraphNode_t wait = !F.use_tc ? rest2 : p % 2 == 1 ? rest1 : nullptr;
        const cudaGraphNode_t sn =
            c.kernel_grid({chain, wait}, d32_step_kernel, dim3(2 * (ts + tx)), kTT, (unsigned)step_smem(npv), n, ld,
                          k, npv, F.A, F.X, (const float *)F.D, (const float *)F.Linv, LDc, (const float *)LDprev,
                          (const float *)LDprev2, F.L0, F.csum);
        c.priority(sn, hi_prio);
        const cudaGraphNode_t dn =
            c.kernel({sn}, d32_diag_kernel, 1u, kTT, ld, base, std::min(kP, n - base), F.A, F.D,
                     (const float *)F.d0, (const float *)F.csum, ts, 2, eps, F.Linv, (const float *)F.L0);
        c.priority(dn, hi_prio);
        const int b2 = base + 2 * kP;
        cudaGraphNode_t rest = nullptr;
        if (F.use_tc) {
            if (p % 2 == 1 && b2 < n) {
                const int T = (int)ceil_div(n - b2, kTcM), nx = (int)ceil_div(base, kTcM);
                unsigned char *buf = F.tc + (size_t)((p / 2) & 1) * 2 * tc_per_panel(n);
                const cudaGraphNode_t sp =
                    c.kernel_grid({sn}, d32_tc_split_kernel, dim3(T + nx, 2), kTT, 0u, n, ld, k - kP, b2, T,
                                  (const float *)F.A, (const float *)F.X, (const float *)LDprev, (const float *)LDc, buf);
                c.priority(sp, lo_prio);
                const int tiles = T * (T + 1) / 2 + T * nx;   // persistent CTAs: one per SM at most
                rest = c.kernel_grid({sp, rest1}, d32_tc_update_kernel, dim3(std::min(tiles, sms)), kTcThreads,
                                     (unsigned)kTcSmem, n, ld, base, b2, T, buf, F.A, F.X, F.tc_err);
                c.priority(rest, lo_prio);
                rest1 = rest;
            }
        } else {
            const int t2 = b2 < n ? (int)ceil_div(n - b2, kTile) : 0, tcn = (int)ceil_div(base, kTile);
            const int n2 = t2 * (t2 + 1) / 2 + t2 * tcn;
            if (n2 > 0) {
                rest = c.kernel_grid({sn, rest1}, d32_update_kernel, dim3(n2), kTT, (unsigned)kRestPad, n, ld, k, F.A, F.X,
                                     (const float *)LDc);
                c.priority(rest, lo_prio);
            } else {
                rest = c.join({sn, rest1});
            }
            rest2 = rest1;
            rest1 = rest;
        }
        chain = dn;
    }
    // the last panel: its diagonal block came with the last step (or is the first block); its
    // block row of L^-1, then the end of the graph after all writes
    const int bs = n - k;
    const cudaGraphNode_t ir = c.kernel({chain}, d32_invrow_kernel, (unsigned)ceil_div(n, kP), kTT, ld, k, bs,
                                        F.X, (const float *)F.Linv);
    c.priority(ir, hi_prio);
    c.join({ir, rest1, rest2});
    if (c.err != cudaSuccess) return fail(OT_ERR_CUDA, cudaGetErrorString(c.err));
    *nodes = c.nodes;
    return ok();
}

Error d32_factor(Dense32 &F, float eps, cudaStream_t st) {
    if (F.tc_err_host && *F.tc_err_host)
        return fail(OT_ERR_TIMEOUT, "dense32: a bounded wait of the tensor-core update gave up");
    if (!F.graph || F.eps != eps) {
        const bool want_tc = F.tc_mode > 0 || (F.tc_mode == 0 && F.n >= kTcAutoN);
        if (want_tc && !F.tc) {
            OT_CUDA(cudaMalloc((void **)&F.tc, 4 * tc_per_panel(F.n)));
            OT_CUDA(cudaMalloc((void **)&F.tc_err, sizeof(int)));
            OT_CUDA(cudaMemset(F.tc_err, 0, sizeof(int)));
            OT_CUDA(cudaMallocHost((void **)&F.tc_err_host, sizeof(int)));
            *F.tc_err_host = 0;
            OT_CUDA(cudaFuncSetAttribute(d32_tc_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem));
        }
        F.use_tc = want_tc;
        if (F.graph) {
            cudaGraphExecDestroy(F.graph);
            F.graph = nullptr;
        }
        cudaGraph_t g = nullptr;
        OT_CUDA(cudaGraphCreate(&g, 0));
        int64_t nodes = 0;
        Error e = d32_build(F, eps, g, &nodes);
        if (e.code == OT_OK && cudaGraphInstantiate(&F.graph, g, 0) != cudaSuccess) {
            F.graph = nullptr;
            e = fail(OT_ERR_CUDA, "dense32: graph instantiation failed");
        }
        cudaGraphDestroy(g);
        cudaGetLastError();
        OT_TRY(e);
        F.graph_nodes = nodes;
        F.eps = eps;
    }
    ktimer_begin(KT_D32_FACTOR, st);
    OT_CUDA(cudaGraphLaunch(F.graph, st));
    g_launches.fetch_add(F.graph_nodes, std::memory_order_relaxed);
    ktimer_end(KT_D32_FACTOR, st);
    if (F.use_tc) OT_CUDA(cudaMemcpyAsync(F.tc_err_host, F.tc_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    // FP32 flops: n^3/3 for L D L^T (n^3/6 multiply-adds) plus n^3/3 for the unit triangular inverse
    ktimer_add_work(KT_D32_FACTOR, 2.0 * (double)F.n * F.n * F.n / 3.0);
    return ok();
}

Error d32_apply(Dense32 &F, const double *r, double *z, cudaStream_t st) {
    const int n = F.n, ld = F.ld;
    const int ncb = (int)ceil_div(n, kFc), nrb = (int)ceil_div(n, kFr);
    int tiles = 0;
    for (int rb = 0; rb < nrb; ++rb) tiles += std::min(ncb, (rb + 1) * (kFr / kFc));
    ktimer_begin(KT_D32_APPLY, st);
    d32_fwd_kernel<<<(unsigned)tiles, kFr, 0, st>>>(n, ld, ncb, F.X, r, F.part);
    OT_LAUNCHED();
    d32_mid_kernel<<<(unsigned)ceil_div(n, kTT), kTT, 0, st>>>(n, ld, F.part, F.D, F.w);
    OT_LAUNCHED();
    d32_bwd_kernel<<<(unsigned)ceil_div(n, kTT / 32), kTT, 0, st>>>(n, ld, F.X, F.w, z);
    OT_LAUNCHED();
    ktimer_end(KT_D32_APPLY, st);
    // bytes: the lower triangle of L^-1 read twice
    ktimer_add_work(KT_D32_APPLY, 4.0 * (double)n * n);
    return ok();
}

}  // namespace ot
