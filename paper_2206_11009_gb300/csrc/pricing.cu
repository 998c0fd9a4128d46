// Pricing: reduced costs d_ij = c_ij - u_i - v_j over all m*n pairs (Section 3.4), costs
// evaluated on the fly from integer point coordinates (never stored) -- the squared Euclidean
// distance, or the L1, Euclidean and L-infinity distances of Section 5.1 -- or read from an
// explicit matrix, and the exact selection of the at most kmax most negative pairs outside the
// support (Section 3.2).  Optionally the scan covers only the listed pairs of the heuristic set
// J = {(i, j) : c_ij < C_max} of Section 3.4.
//
// Pipeline (one host synchronisation, at its end):
//   bounds   bounding box of the points (skipped when the caller knows it);
//   cells,   the points in Morton order of up to 64 x 64 cells (counting sort), in their FP32 forms:
//   prep     squared cost: rows (A_i, X_i, Y_i), cols (B_j, x_j, y_j) with A_i = |x_i|^2 - u_i,
//            X_i = -2 x_i (coordinates shifted to a common origin); other distances: rows
//            (u_i, x_i, y_i), cols (v_j, x_j, y_j); plus the magnitudes that bound the FP32 rounding
//            error, and from them (last block) E >= |d_fp32 - d| for every pair (a priori analysis);
//   tiles    boxes and largest duals of groups of rows and of 256 columns; the pairs of groups
//            whose least possible reduced cost is at most 2E form the tile list (the others hold
//            no pair with d_fp32 <= E);
//   pass 1   one warp per tile: histogram of d < E over 4096 magnitude bins + [0, E], minimum of
//            the tile; further blocks of the same launch take the histogram of the support's pairs;
//   thresh   T = edge of the bin holding the kmax-th smallest key outside the support; gather
//            threshold Tg = min(T + 2E, E): every pair of the exact selection has d_fp32 <= Tg;
//   pass 2   rescan only tiles whose minimum is <= Tg, append (i, j) with d_fp32 <= Tg;
//   select   FP64 d = (c - u) - v (no fusion), support membership by binary search in the CSR
//            rows, sort by (d, jlin), keep the first kmax.
// The candidate buffer has a fixed capacity (spec_capacity), so nothing waits for the host to learn
// how many pairs pass 2 gathers: tiles of kSelT candidates are rechecked and sorted in shared memory,
// one CTA each, and every candidate's final position is its place in its own tile plus the number
// of smaller candidates in the other tiles (binary searches).  When the host finds at the end that
// more pairs were gathered, pass 2 and the selection are redone with an exact-size buffer and a
// stable LSD radix sort.  With a J list the passes go over the list instead of the tiles.
// In the FP64 variant the scan covers all pairs in tiles of TI rows x kPT * RJ columns, computes d
// exactly, keys are float(d) (monotone), E = 0.  An explicit cost matrix always takes it.
#include "pricing.cuh"
#include "primitives.cuh"

#include <cfloat>
#include <cmath>
#include <type_traits>

namespace ot {
namespace {

constexpr int kBins = 4097;       // bins 0..4095: d < 0 by magnitude (large first); 4096: [0, E]
constexpr int kPT = 256;          // threads per scan CTA
// Columns held in registers per thread, kPT * RJ of them per tile: 8, or 2 where n <= kNarrowN (a
// 2048-column tile would be mostly padding: the FP64 scan of 256 x 256 pairs took 25 us with 8).
constexpr int kRJ = 8, kRJNarrow = 2;
constexpr int kNarrowN = 1024;
// above this many pairs inside the FP32 gather window the selection is redone with the FP64 scan
constexpr unsigned long long kMaxWindowPairs = 1ull << 27;

struct Geo {
    unsigned box[4];                             // order-preserving keys of max x, max y, max ~x, max ~y
    unsigned done, done2;                        // blocks of cells_kernel / prep_kernel that are through
    unsigned long long umax_bits, vmax_bits;     // max |u|, max |v| (nonneg double bit patterns)
    int xs_max, ys_max, xt_max, yt_max;          // max |shifted coordinate|
    unsigned long long x2s_max, x2t_max;         // max |x|^2 (integers)
    float E;                                     // FP32 error window
    float Tg;                                    // gather threshold (inclusive)
    unsigned long long gather_bound;             // upper bound of pairs with key <= Tg
    unsigned int ntile;                          // tiles of the FP32 passes
    unsigned int ncand;                          // gathered pairs
    unsigned int nvalid;                         // rechecked candidates
};

// Magnitude bins of d <= 0: 64 octaves from 2^-30 up, 64 bins each (larger and smaller magnitudes in
// the first and last bin).  The kmax-th key's bin is gathered whole: with 16 bins an octave it held
// more pairs than kmax itself at 256x256.
constexpr int kBinBase = (127 - 30) << 6;
__device__ __forceinline__ int bin_of_neg(float d) {
    const int b = (int)(__float_as_uint(-d) >> 17) - kBinBase;   // exponent and 6 mantissa bits
    return 4095 - min(max(b, 0), 4095);                          // larger magnitude -> smaller bin
}
__device__ __forceinline__ float bin_edge(int bin) {             // the least magnitude in the bin
    const int b = 4095 - bin;
    return b > 0 ? __uint_as_float((unsigned)(b + kBinBase) << 17) : 0.f;
}

// ------------------------------------------------------------------------ cost evaluation
// Kinds are the ot_cost_kind values.  FP64 costs follow the oracle's definitions exactly: the
// coordinate differences are integers, the squared distance is an exact integer, and the
// Euclidean distance is its correctly rounded square root.
enum : int { K_SQ = OT_COST_SQEUCLID, K_EU = OT_COST_EUCLID, K_L1 = OT_COST_L1, K_LI = OT_COST_LINF,
             K_DN = OT_COST_DENSE };

// v >= 0 as a double: 2^52 + v is exact in the bit pattern, so one FP64 addition converts it (the
// FP64 pipe is the bound of the FP64 scan and a conversion instruction takes it for longer).
__device__ __forceinline__ double uint_to_f64(int v) {
    return __dsub_rn(__hiloint2double(0x43300000, v), 4503599627370496.0);
}

template <int K>
__device__ __forceinline__ double cost64(int dx, int dy) {
    if (K == K_SQ) return uint_to_f64(dx * dx + dy * dy);
    if (K == K_EU) return __dsqrt_rn(uint_to_f64(dx * dx + dy * dy));
    if (K == K_L1) return uint_to_f64(abs(dx) + abs(dy));
    return uint_to_f64(max(abs(dx), abs(dy)));
}

__device__ __forceinline__ double cost64_rt(int kind, int dx, int dy) {
    switch (kind) {
    case K_SQ: return cost64<K_SQ>(dx, dy);
    case K_EU: return cost64<K_EU>(dx, dy);
    case K_L1: return cost64<K_L1>(dx, dy);
    default: return cost64<K_LI>(dx, dy);
    }
}

// Integer key ordered like the cost (the J test c_ij < C_max is key < jlim, exact).
__device__ __forceinline__ long long cost_key(int kind, int dx, int dy) {
    if (kind == K_L1) return (long long)abs(dx) + abs(dy);
    if (kind == K_LI) return (long long)max(abs(dx), abs(dy));
    return (long long)dx * dx + (long long)dy * dy;  // squared and Euclidean distances
}

// FP32 key of one pair.  Squared cost: the alpha/beta form (2 FMA + 1 add) on the packed rows
// (A_i, X_i, Y_i) and columns (B_j, x_j, y_j).  Other distances, direct form on (u_i, x_i, y_i)
// and (v_j, x_j, y_j): dx, dy exact; L1 / L-infinity exact; Euclidean sqrt(fma(dx, dx, dy*dy));
// then d = (c - u_i) - v_j.
template <int K>
__device__ __forceinline__ float key32(const float4 &R, float cB, float cx, float cy) {
    if (K == K_SQ) {
        const float t1 = __fadd_rn(R.x, cB);
        const float t2 = __fmaf_rn(R.z, cy, t1);
        return __fmaf_rn(R.y, cx, t2);
    }
    const float dx = __fsub_rn(R.y, cx), dy = __fsub_rn(R.z, cy);
    float c;
    if (K == K_L1) c = __fadd_rn(fabsf(dx), fabsf(dy));
    else if (K == K_LI) c = fmaxf(fabsf(dx), fabsf(dy));
    else c = __fsqrt_rn(__fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
    return __fsub_rn(__fsub_rn(c, R.x), cB);
}

// Order-preserving signed key of a double's high word (the low word only refines it), shifted so that
// -infinity is the least: the quiet NaNs with the sign bit set, below it before, wrap to the top, next to
// the others (as the least key of a thread's part of a tile, one of them hid the pairs there from pass 2).
constexpr int kKeyShift = 0xfffff;
__device__ __forceinline__ int hi_key(double d) {
    const int h = __double2hiint(d);
    return (int)((unsigned)(h ^ ((h >> 31) & 0x7fffffff)) - kKeyShift);
}
// A float at or below every double whose hi_key is k.
__device__ __forceinline__ float hi_key_floor(int k) {
    k = (int)((unsigned)k + kKeyShift);
    const int h = k ^ ((k >> 31) & 0x7fffffff);
    return __double2float_rd(__hiloint2double(h, h < 0 && h != (int)0xfff00000 ? -1 : 0));   // (-infinity has no low bits)
}

// --------------------------------------------------------------------------------- prep
// Block-wide maxima: a warp tree, then one value per warp through shared memory; thread 0 gets it.
template <typename T>
__device__ __forceinline__ T block_max(T x, T *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = max(x, __shfl_down_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) x = max(x, sh[w]);
    __syncthreads();
    return x;
}

constexpr int kPrepPer = 4;   // points per thread of the passes below (one atomic per block and maximum)

// Bounding box of all points: max over x, y and over ~x, ~y (~x = -x - 1 is decreasing and never
// overflows) as unsigned keys, so that zero is below every value and idle threads add nothing.
__global__ void __launch_bounds__(256)
bounds_kernel(int m, int n, const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
              const int32_t *__restrict__ tx, const int32_t *__restrict__ ty, Geo *geo) {
    __shared__ unsigned sh[8];
    unsigned k[4] = {0u, 0u, 0u, 0u};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)m + n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int x = i < m ? sx[i] : tx[i - m], y = i < m ? sy[i] : ty[i - m];
        k[0] = max(k[0], (unsigned)x ^ 0x80000000u);
        k[1] = max(k[1], (unsigned)y ^ 0x80000000u);
        k[2] = max(k[2], (unsigned)~x ^ 0x80000000u);
        k[3] = max(k[3], (unsigned)~y ^ 0x80000000u);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned v = block_max(k[q], sh);
        if (threadIdx.x == 0) atomicMax(&geo->box[q], v);
    }
}

// The same from a box that the caller knows.
__global__ void box_kernel(int xlo, int ylo, int xhi, int yhi, Geo *geo) {
    if (threadIdx.x == 0) {
        geo->box[0] = (unsigned)xhi ^ 0x80000000u;
        geo->box[1] = (unsigned)yhi ^ 0x80000000u;
        geo->box[2] = (unsigned)~xlo ^ 0x80000000u;
        geo->box[3] = (unsigned)~ylo ^ 0x80000000u;
    }
}

// Midpoint of the bounding box along axis q (0: x, 1: y).
__device__ __forceinline__ int box_origin(const Geo *geo, int q) {
    const int hi = (int)(geo->box[q] ^ 0x80000000u), lo = ~(int)(geo->box[q + 2] ^ 0x80000000u);
    return (int)(((long long)lo + (long long)hi) / 2);
}

// A priori bound of |d_fp32 - d|.  Every rounding contributes at most 2^-24 times the magnitude
// of the value it rounds; each magnitude is bounded from the maxima gathered by prep.
//  squared cost, evaluation order
//    A = fl(fl(|x_i|^2) - fl(u_i)), B = fl(fl(|x_j|^2) - fl(v_j)),
//    t1 = fl(A + B), t2 = fma(Y_i, y_j, t1), d~ = fma(X_i, x_j, t2)
//  (products of integers are exact inside the FMA);
//  other distances, d~ = fl(fl(c~ - fl(u_i)) - fl(v_j)) with c~ exact for L1 and L-infinity and
//  |c~ - c| <= 2.001 * 2^-24 * c for the Euclidean distance (one rounding of dy*dy, one of the
//  FMA, one of the square root; the first two enter the root halved).
__device__ float error_bound(const Geo &geo, int kind) {
    const double uu = 5.9604644775390625e-08;  // 2^-24
    double umax = __longlong_as_double((long long)geo.umax_bits);
    double vmax = __longlong_as_double((long long)geo.vmax_bits);
    double E;
    if (kind == K_SQ) {
        double x2s = (double)geo.x2s_max, x2t = (double)geo.x2t_max;
        double cross = 2.0 * ((double)geo.xs_max * geo.xt_max + (double)geo.ys_max * geo.yt_max);
        double A = (x2s + umax) * (1 + 2 * uu), B = (x2t + vmax) * (1 + 2 * uu);
        double T1 = (A + B) * (1 + uu), T2 = (T1 + cross) * (1 + uu), D = (T2 + cross) * (1 + uu);
        E = uu * (x2s + umax + A + x2t + vmax + B + T1 + T2 + D) * 1.0001 + 1e-30;
    } else {
        const double xs = (double)geo.xs_max + geo.xt_max, ys = (double)geo.ys_max + geo.yt_max;
        double cmax, epsc = 0.0;
        if (kind == K_L1) cmax = xs + ys;
        else if (kind == K_LI) cmax = fmax(xs, ys);
        else { cmax = sqrt(xs * xs + ys * ys) * (1 + 1e-15); epsc = 2.001 * uu * cmax; }
        const double Cp = cmax + epsc, Up = umax * (1 + uu), Vp = vmax * (1 + uu);
        const double T = Cp + Up;            // |c~ - u~|
        const double Dd = T * (1 + uu) + Vp; // |fl(c~ - u~) - v~|
        E = (epsc + uu * (umax + vmax + T + Dd)) * 1.0001 + 1e-30;
    }
    const float Ef = __double2float_ru(E);
    return isfinite(Ef) ? Ef : FLT_MAX;
}

// ---- spatial order.  Cells of 2^s x 2^s coordinate units, s the least with at most 64 x 64 cells over
// the bounding box, numbered in Morton order: consecutive points form compact groups.
constexpr int kCells = 4096;
constexpr int kCG = 256;     // columns per group (32 lanes x 8)

__device__ __forceinline__ int cell_shift(const Geo *geo) {
    unsigned ext = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int hi = (int)(geo->box[q] ^ 0x80000000u), lo = ~(int)(geo->box[q + 2] ^ 0x80000000u);
        ext = max(ext, (unsigned)hi - (unsigned)lo);
    }
    return max(0, 26 - __clz(ext));   // ext >> s < 64
}

__device__ __forceinline__ int cell_of(const Geo *geo, int s, int x, int y) {
    const int xlo = ~(int)(geo->box[2] ^ 0x80000000u), ylo = ~(int)(geo->box[3] ^ 0x80000000u);
    auto spread = [](unsigned v) {   // six bits to the even positions
        v = (v | (v << 4)) & 0x30fu;
        v = (v | (v << 2)) & 0x333u;
        return (v | (v << 1)) & 0x555u;
    };
    return (int)(spread(((unsigned)x - (unsigned)xlo) >> s) | (spread(((unsigned)y - (unsigned)ylo) >> s) << 1));
}

// Points per cell (sources, then targets), each point's place in its cell (any order), and by the
// last block the cells' first positions.
__global__ void __launch_bounds__(256)
cells_kernel(int m, int n, const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
             const int32_t *__restrict__ tx, const int32_t *__restrict__ ty, Geo *geo, unsigned *cells,
             unsigned *__restrict__ place) {
    __shared__ unsigned wsum[8];
    __shared__ int s_last;
    const int s = cell_shift(geo);
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < (int64_t)m + n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const bool src = k < m;
        const int64_t e = src ? k : k - m;
        place[k] = atomicAdd(&cells[(src ? 0 : kCells) + cell_of(geo, s, (src ? sx : tx)[e], (src ? sy : ty)[e])], 1u);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&geo->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int side = 0; side < 2; ++side) {   // exclusive scan, 16 cells per thread
        unsigned *c = cells + side * kCells + threadIdx.x * (kCells / 256);
        unsigned v[kCells / 256], sum = 0;
#pragma unroll
        for (int q = 0; q < kCells / 256; ++q) { v[q] = __ldcg(c + q); }
#pragma unroll
        for (int q = 0; q < kCells / 256; ++q) { const unsigned t = v[q]; v[q] = sum; sum += t; }
        unsigned x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        unsigned first = x - sum;
        for (int w = 0; w < wid; ++w) first += wsum[w];
#pragma unroll
        for (int q = 0; q < kCells / 256; ++q) c[q] = first + v[q];
        __syncthreads();
    }
}

// FP32 forms of the points, in the caller's order (rows, cols) and, with place != NULL, in cell order
// (srt: sources then targets, the point's index in .w; sdual: its dual rounded up), and the error
// bound.  The maxima are reduced per block before the atomics: one atomic per thread on eight words
// took 171 us at m = n = 65536, this takes 11.
template <bool SQ>
__global__ void __launch_bounds__(256)
prep_kernel(int m, int n, int kind, const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
            const int32_t *__restrict__ tx, const int32_t *__restrict__ ty, const double *__restrict__ u,
            const double *__restrict__ v, float4 *__restrict__ rows, float4 *__restrict__ cols,
            const unsigned *__restrict__ cells, const unsigned *__restrict__ place, float4 *__restrict__ srt,
            float *__restrict__ sdual, Geo *geo) {
    __shared__ unsigned long long shl[8];
    __shared__ int shi[8];
    const int ox = box_origin(geo, 0), oy = box_origin(geo, 1), s = cell_shift(geo);
    unsigned long long umax = 0, vmax = 0, x2s = 0, x2t = 0;
    int xsm = 0, ysm = 0, xtm = 0, ytm = 0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < (int64_t)m + n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const bool src = k < m;
        const int64_t e = src ? k : k - m;
        const int x0 = (src ? sx : tx)[e], y0 = (src ? sy : ty)[e], x = x0 - ox, y = y0 - oy;
        const long long x2 = (long long)x * x + (long long)y * y;
        const double dual = (src ? u : v)[e];
        const float df = __double2float_rn(dual), fac = SQ && src ? -2.0f : 1.0f;
        // |dual|: its bit pattern orders like its value (a NaN never compares below E: left out)
        const unsigned long long bits = dual == dual ? (unsigned long long)__double_as_longlong(fabs(dual)) : 0ull;
        const float4 f = make_float4(SQ ? __fsub_rn(__ll2float_rn(x2), df) : df, fac * (float)x, fac * (float)y,
                                     __int_as_float((int)e));
        (src ? rows : cols)[e] = f;
        if (place) {
            const int64_t at = (src ? 0 : m) +
                               (int64_t)cells[(src ? 0 : kCells) + cell_of(geo, s, x0, y0)] + place[k];
            srt[at] = f;
            sdual[at] = __double2float_ru(dual);
        }
        if (src) {
            umax = max(umax, bits);
            xsm = max(xsm, abs(x)); ysm = max(ysm, abs(y)); x2s = max(x2s, (unsigned long long)x2);
        } else {
            vmax = max(vmax, bits);
            xtm = max(xtm, abs(x)); ytm = max(ytm, abs(y)); x2t = max(x2t, (unsigned long long)x2);
        }
    }
    umax = block_max(umax, shl); vmax = block_max(vmax, shl);
    x2s = block_max(x2s, shl); x2t = block_max(x2t, shl);
    xsm = block_max(xsm, shi); ysm = block_max(ysm, shi);
    xtm = block_max(xtm, shi); ytm = block_max(ytm, shi);
    if (threadIdx.x == 0) {
        atomicMax(&geo->umax_bits, umax);
        atomicMax(&geo->vmax_bits, vmax);
        atomicMax(&geo->x2s_max, x2s);
        atomicMax(&geo->x2t_max, x2t);
        atomicMax(&geo->xs_max, xsm); atomicMax(&geo->ys_max, ysm);
        atomicMax(&geo->xt_max, xtm); atomicMax(&geo->yt_max, ytm);
        __threadfence();
        if (atomicAdd(&geo->done2, 1u) == gridDim.x - 1) {   // every block's maxima are in
            __threadfence();
            Geo g;
            volatile Geo *vg = geo;
            g.umax_bits = vg->umax_bits; g.vmax_bits = vg->vmax_bits;
            g.xs_max = vg->xs_max; g.ys_max = vg->ys_max; g.xt_max = vg->xt_max; g.yt_max = vg->yt_max;
            g.x2s_max = vg->x2s_max; g.x2t_max = vg->x2t_max;
            geo->E = error_bound(g, kind);
        }
    }
}

// Box and largest dual of each group: G consecutive sources, or kCG targets, in cell order.  One warp
// per group, sources' groups first.
struct Group { float xlo, xhi, ylo, yhi, dual; };

__global__ void __launch_bounds__(256)
groups_kernel(int m, int n, int G, int nrg, int ncg, float row_fac, const float4 *__restrict__ srt,
              const float *__restrict__ sdual, Group *__restrict__ grp) {
    const int lane = threadIdx.x & 31;
    for (int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); w < (int64_t)nrg + ncg; w += (int64_t)gridDim.x * 8) {
        const bool src = w < nrg;
        const int64_t lo = src ? w * G : m + (w - nrg) * kCG;
        const int64_t hi = src ? min(lo + G, (int64_t)m) : min(lo + kCG, (int64_t)m + n);
        Group g{INFINITY, -INFINITY, INFINITY, -INFINITY, -INFINITY};
        for (int64_t k = lo + lane; k < hi; k += 32) {
            const float4 f = srt[k];
            const float fac = src ? row_fac : 1.0f;   // -1/2 undoes the squared form's -2 (exact)
            const float x = fac * f.y, y = fac * f.z;
            g.xlo = fminf(g.xlo, x); g.xhi = fmaxf(g.xhi, x);
            g.ylo = fminf(g.ylo, y); g.yhi = fmaxf(g.yhi, y);
            g.dual = fmaxf(g.dual, sdual[k]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            g.xlo = fminf(g.xlo, __shfl_xor_sync(0xffffffffu, g.xlo, o));
            g.xhi = fmaxf(g.xhi, __shfl_xor_sync(0xffffffffu, g.xhi, o));
            g.ylo = fminf(g.ylo, __shfl_xor_sync(0xffffffffu, g.ylo, o));
            g.yhi = fmaxf(g.yhi, __shfl_xor_sync(0xffffffffu, g.yhi, o));
            g.dual = fmaxf(g.dual, __shfl_xor_sync(0xffffffffu, g.dual, o));
        }
        if (lane == 0) grp[w] = g;
    }
}

// The tile list: pairs of groups (column group h, row group g -> h nrg + g) that can hold a pair with
// d_fp32 <= E.  Every d there is at least the cost of the boxes' gap minus the largest duals (all
// rounded down), d_fp32 >= d - E: groups with that bound above 2E are left out.  At 256x256, duals of
// slope 6 per pixel, 4 % of the pairs remain.
template <int K>
__global__ void __launch_bounds__(256)
tiles_kernel(int nrg, int64_t total, const Group *__restrict__ grp, Geo *geo, unsigned *__restrict__ list) {
    const float lim = 2.0f * geo->E;
    const int lane = threadIdx.x & 31;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < total;
         t0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = t0 + lane;
        bool keep = false;
        if (t < total) {
            const Group a = grp[t % nrg], b = grp[nrg + t / nrg];
            const float gx = fmaxf(0.f, fmaxf(a.xlo - b.xhi, b.xlo - a.xhi));   // integers: exact
            const float gy = fmaxf(0.f, fmaxf(a.ylo - b.yhi, b.ylo - a.yhi));
            float c;
            if (K == K_L1) c = __fadd_rd(gx, gy);
            else if (K == K_LI) c = fmaxf(gx, gy);
            else {
                c = __fadd_rd(__fmul_rd(gx, gx), __fmul_rd(gy, gy));
                if (K == K_EU) c = __fsqrt_rd(c);
            }
            keep = !(__fsub_rd(__fsub_rd(c, a.dual), b.dual) > lim);   // (kept where it is not a number)
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (!bal) continue;
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&geo->ntile, (unsigned)__popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (keep) list[at + __popc(bal & ((1u << lane) - 1u))] = (unsigned)t;
    }
}

// One key into the histogram (pass 1) or the candidate list (pass 2).
// Padding columns (j >= n) carry key +inf and never qualify; the gather also checks j < n.
template <bool FP64, bool GATHER>
__device__ __forceinline__ void take_key(float d, bool neg64, float E, float Tg, unsigned *sh_hist, int i, int j,
                                         int n, int32_t *ci, int32_t *cj, unsigned long long cap, unsigned *ncand) {
    const bool neg = FP64 ? neg64 : (d < 0.f);
    if (!GATHER) {
        if (neg) atomicAdd(&sh_hist[bin_of_neg(d)], 1u);
        else if (!FP64 && d <= E) atomicAdd(&sh_hist[4096], 1u);
    } else {
        const bool take = (FP64 ? (neg && d <= Tg) : (d <= Tg)) && j < n;
        if (take) {
            const unsigned pos = atomicAdd(ncand, 1u);
            if (pos < cap) { ci[pos] = i; cj[pos] = j; }
        }
    }
}

// Pass 2 has nothing to do when its bound exceeds the buffer: the host redoes it with a larger one, or in
// FP64 (evaluating and counting the 151M pairs of a flooded FP32 window took 3.0 ms; 0.01 so).
__device__ __forceinline__ bool gather_in_vain(const Geo *geo, unsigned long long cap) {
    return geo->gather_bound > cap;
}

// The support pairs entered the histogram too (the scan does not test membership): their own
// histogram, with the same arithmetic as the scan so that every key lands in the same bin, by the
// blocks `part` of `parts` of the histogram launch (shared-memory counts first: global atomics on
// the few occupied bins took 91 us for 588k pairs).  With a J list only the support pairs inside J
// were scanned: jlim > 0 (integer cost key < jlim) or, for an explicit matrix, jcmax > 0
// (c_ij < jcmax) selects them.
struct SupArgs {
    const int32_t *si, *sj;
    int64_t psi;
    long long jlim;
    double jcmax;
    int first;                   // blocks from this one on take the support
    unsigned long long *hist;
};

template <int K, bool FP64>
__device__ __forceinline__ void support_hist(const SupArgs &S, int n, const float4 *__restrict__ rows,
                                             const float4 *__restrict__ cols, const int32_t *__restrict__ sx,
                                             const int32_t *__restrict__ sy, const int32_t *__restrict__ tx,
                                             const int32_t *__restrict__ ty, const double *__restrict__ u,
                                             const double *__restrict__ v, const double *__restrict__ C, float E,
                                             unsigned *sh_hist) {
    const int part = (int)blockIdx.x - S.first, parts = (int)gridDim.x - S.first;
    for (int64_t e = (int64_t)part * kPT + threadIdx.x; e < S.psi; e += (int64_t)parts * kPT) {
        const int i = S.si[e], j = S.sj[e];
        if (K == K_DN) {
            if (S.jcmax > 0.0 && !(C[(int64_t)i * n + j] < S.jcmax)) continue;
        } else if (S.jlim > 0 && cost_key(K, sx[i] - tx[j], sy[i] - ty[j]) >= S.jlim) {
            continue;
        }
        if (FP64) {
            const double cc = K == K_DN ? C[(int64_t)i * n + j] : cost64<K>(sx[i] - tx[j], sy[i] - ty[j]);
            const double d = __dsub_rn(__dsub_rn(cc, u[i]), v[j]);
            if (d < 0.0) atomicAdd(&sh_hist[bin_of_neg(__double2float_rn(d))], 1u);
        } else {
            const float4 R = rows[i], Q = cols[j];
            const float d = key32<K>(R, Q.x, Q.y, Q.z);
            if (d < 0.f) atomicAdd(&sh_hist[bin_of_neg(d)], 1u);
            else if (d <= E) atomicAdd(&sh_hist[4096], 1u);
        }
    }
}

// ------------------------------------------------------------------------------- FP32 scan
// One warp per tile of the list: 8 columns per lane in registers, the tile's rows staged through the
// warp's shared memory 64 at a time, keys in groups of 4 rows x 8 columns with one branch per group.
// Bound by the issue of the FP32 pipes: one add, two FMAs and one minimum per pair (squared cost).
// Packed f32x2 arithmetic on two columns was 1.6 times slower, three-input minima no faster
// (256x256, all pairs: 565 us scalar, 925 packed, 579 with three-input minima).
constexpr int kStage = 64;

template <int K, bool GATHER>
__global__ void __launch_bounds__(kPT)
tile_scan_kernel(int m, int n, int G, int nrg, SupArgs S, const float4 *__restrict__ rows,
                 const float4 *__restrict__ cols, const float4 *__restrict__ srt, const int32_t *__restrict__ sx,
                 const int32_t *__restrict__ sy, const int32_t *__restrict__ tx, const int32_t *__restrict__ ty,
                 const double *__restrict__ u, const double *__restrict__ v, const Geo *__restrict__ geo,
                 const unsigned *__restrict__ list, float *__restrict__ tile_min,
                 unsigned long long *__restrict__ hist, int32_t *__restrict__ ci, int32_t *__restrict__ cj,
                 unsigned long long cap, unsigned int *__restrict__ ncand) {
    __shared__ float4 srow[kPT / 32][kStage];
    __shared__ unsigned sh_hist[GATHER ? 1 : kBins];
    if (GATHER && gather_in_vain(geo, cap)) return;
    if (!GATHER) {
        for (int b = threadIdx.x; b < kBins; b += kPT) sh_hist[b] = 0;
        __syncthreads();
    }
    const float E = geo->E, Tg = geo->Tg, thr = GATHER ? Tg : E;
    const bool support = !GATHER && (int)blockIdx.x >= S.first;
    if constexpr (!GATHER) {
        if (support) support_hist<K, false>(S, n, rows, cols, sx, sy, tx, ty, u, v, nullptr, E, sh_hist);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned ntile = support ? 0u : geo->ntile;
    for (unsigned t = (blockIdx.x * (kPT / 32) + warp); t < ntile; t += S.first * (kPT / 32)) {
        if (GATHER && tile_min[t] > Tg) continue;   // uniform over the warp
        const unsigned id = list[t];
        const int64_t c0 = (int64_t)(id / nrg) * kCG + lane;
        const int r0 = (int)(id % nrg) * G, nr = min(G, m - r0);
        // padding columns get key +inf: cB = +inf in the squared form (d = ... + B_j), -inf in the
        // direct form (d = ... - v_j)
        float cB[8], cx[8], cy[8];
        int jj[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 q = c0 + 32 * c < n ? srt[m + c0 + 32 * c]
                                             : make_float4(K == K_SQ ? INFINITY : -INFINITY, 0.f, 0.f, __int_as_float(n));
            cB[c] = q.x; cx[c] = q.y; cy[c] = q.z; jj[c] = __float_as_int(q.w);
        }
        float tmin = INFINITY;
        for (int b0 = 0; b0 < nr; b0 += kStage) {
            const int nb = min(kStage, nr - b0);
            __syncwarp();
            for (int k = lane; k < nb; k += 32) srow[warp][k] = srt[r0 + b0 + k];
            __syncwarp();
            for (int g0 = 0; g0 < nb; g0 += 4) {
                float d[4][8], mq[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    // (a ragged last group repeats its last row: the same keys, never taken twice)
                    const float4 R = srow[warp][min(g0 + q, nb - 1)];
                    mq[q] = INFINITY;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        d[q][c] = key32<K>(R, cB[c], cx[c], cy[c]);
                        mq[q] = fminf(mq[q], d[q][c]);
                    }
                }
                const float dmin = fminf(fminf(mq[0], mq[1]), fminf(mq[2], mq[3]));
                tmin = fminf(tmin, dmin);
                if (dmin <= thr) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (g0 + q >= nb || mq[q] > thr) continue;
                        const int i = GATHER ? __float_as_int(srow[warp][g0 + q].w) : 0;
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            take_key<false, GATHER>(d[q][c], false, E, Tg, sh_hist, i, jj[c], n, ci, cj, cap, ncand);
                    }
                }
            }
        }
        if (!GATHER) {   // the tile's minimum (for skipping it in pass 2)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tmin = fminf(tmin, __shfl_down_sync(0xffffffffu, tmin, o));
            if (lane == 0) tile_min[t] = tmin;
        }
    }
    if (!GATHER) {
        __syncthreads();
        unsigned long long *out = support ? S.hist : hist;
        for (int b = threadIdx.x; b < kBins; b += kPT)
            if (sh_hist[b]) atomicAdd(&out[b], (unsigned long long)sh_hist[b]);
    }
}

// ------------------------------------------------------------------------------- FP64 scan
// Tiles of TI source rows x kPT * RJ target columns; RJ columns per thread in registers, rows from
// shared memory.  Bound by the FP64 pipe: only the three FP64 operations of the definition per pair,
// the minima and the sign on the high words.
template <int K, bool GATHER, int RJ>
__global__ void __launch_bounds__(kPT)
scan64_kernel(int m, int n, int TI, int ncb, int64_t ntiles, SupArgs S,
              const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
              const int32_t *__restrict__ tx, const int32_t *__restrict__ ty,
              const double *__restrict__ u, const double *__restrict__ v, const double *__restrict__ C,
              const Geo *__restrict__ geo, float *__restrict__ tile_min,
              unsigned long long *__restrict__ hist, int32_t *__restrict__ ci,
              int32_t *__restrict__ cj, unsigned long long cap, unsigned int *__restrict__ ncand) {
    constexpr int TJ = kPT * RJ;
    __shared__ int2 srowi[256];
    __shared__ double srowu[256];
    __shared__ unsigned sh_hist[GATHER ? 1 : kBins];
    __shared__ float sred[kPT / 32];
    if (GATHER && gather_in_vain(geo, cap)) return;
    if (!GATHER) {
        for (int b = threadIdx.x; b < kBins; b += kPT) sh_hist[b] = 0;
        __syncthreads();
    }
    const float Tg = geo->Tg;
    const bool support = !GATHER && (int)blockIdx.x >= S.first;
    if constexpr (!GATHER) {
        if (support) support_hist<K, true>(S, n, nullptr, nullptr, sx, sy, tx, ty, u, v, C, 0.f, sh_hist);
    }
    for (int64_t t = support ? ntiles : blockIdx.x; t < ntiles; t += S.first) {
        const int rb = (int)(t / ncb), cb = (int)(t % ncb);
        if (GATHER && tile_min[t] > Tg) continue;  // uniform over the block
        const int i0 = rb * TI;
        const int nrows = min(TI, m - i0);
        __syncthreads();
        if (threadIdx.x < nrows) {
            const int i = i0 + threadIdx.x;
            if (K != K_DN) srowi[threadIdx.x] = make_int2(sx[i], sy[i]);
            srowu[threadIdx.x] = u[i];
        }
        const int j0 = cb * TJ + (int)threadIdx.x;   // this thread's columns: j0 + c * kPT
        int ix[RJ], iy[RJ];
        double dv[RJ];
#pragma unroll
        for (int c = 0; c < RJ; ++c) {
            const int j = j0 + c * kPT;
            ix[c] = 0; iy[c] = 0; dv[c] = -INFINITY;   // padding: d = +inf
            if (j < n) { if (K != K_DN) { ix[c] = tx[j]; iy[c] = ty[j]; } dv[c] = v[j]; }
        }
        __syncthreads();
        // Tg <= 0 here.  A pair is taken when float(d) <= Tg (d < 0 in the histogram pass): its high
        // word's key is then at most one above Tg's (the rounding to float)
        const int kthr = GATHER ? hi_key((double)Tg) + 1 : hi_key(-0.0);
        int kmin = INT_MAX;
        for (int r = 0; r < nrows; ++r) {
            double dd[RJ];
            int kq = INT_MAX;
            const double ur = srowu[r];
            const int2 R = K != K_DN ? srowi[r] : make_int2(0, 0);
#pragma unroll
            for (int c = 0; c < RJ; ++c) {
                double cc;
                if (K == K_DN) {
                    const int j = j0 + c * kPT;
                    cc = j < n ? C[(int64_t)(i0 + r) * n + j] : 0.0;
                } else {
                    cc = cost64<K>(R.x - ix[c], R.y - iy[c]);
                }
                dd[c] = __dsub_rn(__dsub_rn(cc, ur), dv[c]);
                kq = min(kq, hi_key(dd[c]));
            }
            kmin = min(kmin, kq);
            if (kq <= kthr) {
#pragma unroll
                for (int c = 0; c < RJ; ++c)
                    take_key<true, GATHER>(__double2float_rn(dd[c]), dd[c] < 0.0, 0.f, Tg, sh_hist, i0 + r,
                                           j0 + c * kPT, n, ci, cj, cap, ncand);
            }
        }
        if (!GATHER) {
            // tile minimum (for skipping tiles in pass 2)
            float w = kmin != INT_MAX ? hi_key_floor(kmin) : INFINITY;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w = fminf(w, __shfl_down_sync(0xffffffffu, w, o));
            if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = w;
            __syncthreads();
            if (threadIdx.x == 0) {
                float b = sred[0];
                for (int k = 1; k < kPT / 32; ++k) b = fminf(b, sred[k]);
                tile_min[t] = b;
            }
        }
    }
    if (!GATHER) {
        __syncthreads();
        unsigned long long *out = support ? S.hist : hist;
        for (int b = threadIdx.x; b < kBins; b += kPT)
            if (sh_hist[b]) atomicAdd(&out[b], (unsigned long long)sh_hist[b]);
    }
}

// ------------------------------------------------------------------------ J-list scan
// Section 3.4's heuristic: only the pairs of J (listed, sorted by (i, j)) are priced.  Tiles of
// kJT consecutive list entries; each thread takes kJE entries kPT apart (coalesced list reads;
// the row and column data come from L2).
constexpr int kJE = 16;
constexpr int kJT = kPT * kJE;

template <int K, bool FP64, bool GATHER>
__global__ void __launch_bounds__(kPT)
jscan_kernel(int n, int64_t jn, int64_t ntiles, SupArgs S, const int32_t *__restrict__ ji,
             const int32_t *__restrict__ jj,
             const float4 *__restrict__ rows, const float4 *__restrict__ cols,
             const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
             const int32_t *__restrict__ tx, const int32_t *__restrict__ ty,
             const double *__restrict__ u, const double *__restrict__ v, const double *__restrict__ C,
             const Geo *__restrict__ geo, float *__restrict__ tile_min,
             unsigned long long *__restrict__ hist, int32_t *__restrict__ ci,
             int32_t *__restrict__ cj, unsigned long long cap, unsigned int *__restrict__ ncand) {
    __shared__ unsigned sh_hist[GATHER ? 1 : kBins];
    __shared__ float sred[kPT / 32];
    if (GATHER && gather_in_vain(geo, cap)) return;
    if (!GATHER) {
        for (int b = threadIdx.x; b < kBins; b += kPT) sh_hist[b] = 0;
        __syncthreads();
    }
    const float E = geo->E;
    const float Tg = geo->Tg;
    const bool support = !GATHER && (int)blockIdx.x >= S.first;
    if constexpr (!GATHER) {
        if (support) support_hist<K, FP64>(S, n, rows, cols, sx, sy, tx, ty, u, v, C, E, sh_hist);
    }
    for (int64_t t = support ? ntiles : blockIdx.x; t < ntiles; t += S.first) {
        if (GATHER && tile_min[t] > Tg) continue;  // uniform over the block
        float tmin = INFINITY;
#pragma unroll 4
        for (int k = 0; k < kJE; ++k) {
            const int64_t e = t * kJT + (int64_t)k * kPT + threadIdx.x;
            if (e >= jn) break;
            const int i = ji[e], j = jj[e];
            float d;
            bool neg64 = false;
            if (FP64) {
                double cc;
                if (K == K_DN) cc = C[(int64_t)i * n + j];
                else cc = cost64<K>(sx[i] - tx[j], sy[i] - ty[j]);
                const double dd = __dsub_rn(__dsub_rn(cc, u[i]), v[j]);
                d = __double2float_rn(dd);
                neg64 = dd < 0.0;
            } else {
                const float4 R = rows[i], Q = cols[j];
                d = key32<K>(R, Q.x, Q.y, Q.z);
            }
            tmin = fminf(tmin, d);
            if (d <= (GATHER ? Tg : E))
                take_key<FP64, GATHER>(d, neg64, E, Tg, sh_hist, i, j, n, ci, cj, cap, ncand);
        }
        if (!GATHER) {
            float w = tmin;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w = fminf(w, __shfl_down_sync(0xffffffffu, w, o));
            __syncthreads();
            if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = w;
            __syncthreads();
            if (threadIdx.x == 0) {
                float b = sred[0];
                for (int q = 1; q < kPT / 32; ++q) b = fminf(b, sred[q]);
                tile_min[t] = b;
            }
        }
    }
    if (!GATHER) {
        __syncthreads();
        unsigned long long *out = support ? S.hist : hist;
        for (int b = threadIdx.x; b < kBins; b += kPT)
            if (sh_hist[b]) atomicAdd(&out[b], (unsigned long long)sh_hist[b]);
    }
}

// One block: find the bin holding the kmax-th smallest key outside the support, the gather
// threshold Tg and an upper bound on the number of pairs (support included) pass 2 will append.
// Thread t holds bins 4 t .. 4 t + 3 (the last one also bin 4096).
__global__ void __launch_bounds__(1024)
threshold_kernel(const unsigned long long *__restrict__ hist_all, const unsigned long long *__restrict__ hist_sup,
                 int kmax, int fp64, Geo *geo) {
    __shared__ unsigned long long wsum[32];
    __shared__ int s_bstar;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    unsigned long long all[5], ns[5], loc = 0;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const bool have = k < 4 || t == 1023;
        all[k] = have ? hist_all[4 * t + k] : 0ull;
        ns[k] = have ? all[k] - hist_sup[4 * t + k] : 0ull;
        loc += ns[k];
    }
    if (t == 0) s_bstar = -1;
    unsigned long long x = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    unsigned long long before = x - loc;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    if (before < (unsigned long long)kmax && before + loc >= (unsigned long long)kmax) {
        unsigned long long acc = before;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            acc += ns[k];
            if (acc >= (unsigned long long)kmax) { s_bstar = 4 * t + k; break; }
        }
    }
    __syncthreads();
    const int bstar = s_bstar;
    const float E = geo->E;
    float Tg;
    if (bstar < 0 || bstar == 4096) {
        Tg = fp64 ? 0.0f : E;                 // take every candidate
    } else {
        const float T = -bin_edge(bstar);     // every key in bins <= bstar is <= T
        if (fp64) Tg = T;
        else Tg = fminf(__fadd_ru(T, __fmul_ru(2.0f, E)), E);
    }
    // bins that can hold keys <= Tg
    const int bg = Tg < 0.f ? bin_of_neg(Tg) : (fp64 ? 4095 : 4096);
    unsigned long long take = 0;
#pragma unroll
    for (int k = 0; k < 5; ++k) take += 4 * t + k <= bg ? all[k] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) take += __shfl_down_sync(0xffffffffu, take, o);
    if (lane == 0) wsum[wid] = take;
    __syncthreads();
    if (t == 0) {
        for (int w = 1; w < 32; ++w) take += wsum[w];
        geo->Tg = Tg;
        geo->gather_bound = take;
    }
}

// FP64 reduced cost of pair (i, j) and whether it is a candidate (d < 0 outside the support)
__device__ __forceinline__ bool recheck_pair(int i, int j, int n, int kind, const int32_t *__restrict__ sx,
                                             const int32_t *__restrict__ sy, const int32_t *__restrict__ tx,
                                             const int32_t *__restrict__ ty, const double *__restrict__ u,
                                             const double *__restrict__ v, const double *__restrict__ C,
                                             const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ sup_j,
                                             double &d) {
    const int end = row_ptr[i + 1];
    int lo = row_ptr[i], hi = end;
    while (lo < hi) {  // lower_bound of j in the sorted columns of row i
        const int mid = (lo + hi) >> 1;
        if (sup_j[mid] < j) lo = mid + 1; else hi = mid;
    }
    const bool member = lo < end && sup_j[lo] == j;
    const double cc = kind == K_DN ? C[(int64_t)i * n + j] : cost64_rt(kind, sx[i] - tx[j], sy[i] - ty[j]);
    d = __dsub_rn(__dsub_rn(cc, u[i]), v[j]);
    return !member && d < 0.0;
}

// ------------------------------------------------------------------------ selection
// Candidates in tiles of kSelT: each CTA rechecks its tile in FP64 and sorts it by (d, jlin) with a
// bitonic network -- two elements per thread, distances up to 32 in registers by shuffles, the
// others through shared memory (10 of the 55 steps).  Pairs that are no candidates get the largest
// key.  Latency-bound; it replaced two radix sorts (11 passes of three launches, 350 us at 12k).
constexpr int kSelT = 1024;

__device__ __forceinline__ bool key_less(unsigned long long ka, unsigned ja, unsigned long long kb, unsigned jb) {
    return ka < kb || (ka == kb && ja < jb);
}

__global__ void __launch_bounds__(kSelT / 2)
select_sort_kernel(int m, int n, int kind, unsigned cap, const int32_t *__restrict__ ci,
                   const int32_t *__restrict__ cj, const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
                   const int32_t *__restrict__ tx, const int32_t *__restrict__ ty, const double *__restrict__ u,
                   const double *__restrict__ v, const double *__restrict__ C, const int32_t *__restrict__ row_ptr,
                   const int32_t *__restrict__ sup_j, Geo *geo, unsigned long long *__restrict__ skey,
                   unsigned *__restrict__ sjl) {
    __shared__ unsigned long long sk[kSelT];
    __shared__ unsigned sj[kSelT];
    const unsigned count = geo->ncand, base = blockIdx.x * kSelT;
    if (geo->gather_bound > cap || base >= count) return;   // uniform over the block
    const int lane = threadIdx.x & 31, p0 = (threadIdx.x >> 5) * 64 + lane;   // positions p0 and p0 + 32
    unsigned long long k[2];
    unsigned l[2];
    int nv = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const unsigned e = base + p0 + 32 * h;
        k[h] = ~0ull;
        l[h] = ~0u;
        bool ok = false;
        if (e < count) {
            const int i = ci[e], j = cj[e];
            double d;
            ok = recheck_pair(i, j, n, kind, sx, sy, tx, ty, u, v, C, row_ptr, sup_j, d);
            if (ok) {
                k[h] = f64_key(d);
                l[h] = (unsigned)i + (unsigned)j * (unsigned)m;   // jlin < m n <= 2^32
            }
        }
        nv += __syncthreads_count(ok);
    }
    if (threadIdx.x == 0 && nv) atomicAdd(&geo->nvalid, (unsigned)nv);
    auto keep = [&](int h, unsigned long long ok, unsigned ol, int pos, int dist, int size) {
        // position pos meets pos ^ dist: the lower position keeps the smaller when ascending
        const bool lower = (pos & dist) == 0, asc = (pos & size) == 0;
        const bool less = key_less(ok, ol, k[h], l[h]);
        if (less == (lower == asc)) { k[h] = ok; l[h] = ol; }
    };
    for (int size = 2; size <= kSelT; size <<= 1) {
        int dist = size >> 1;
        for (; dist >= 64; dist >>= 1) {
            __syncthreads();
            sk[p0] = k[0]; sj[p0] = l[0];
            sk[p0 + 32] = k[1]; sj[p0 + 32] = l[1];
            __syncthreads();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int pos = p0 + 32 * h;
                keep(h, sk[pos ^ dist], sj[pos ^ dist], pos, dist, size);
            }
        }
        if (dist == 32) {
            const bool asc = (p0 & size) == 0;
            if (key_less(k[1], l[1], k[0], l[0]) == asc) {
                const unsigned long long tk = k[0]; k[0] = k[1]; k[1] = tk;
                const unsigned tl = l[0]; l[0] = l[1]; l[1] = tl;
            }
            dist = 16;
        }
        for (; dist > 0; dist >>= 1)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned long long ok = __shfl_xor_sync(0xffffffffu, k[h], dist);
                const unsigned ol = __shfl_xor_sync(0xffffffffu, l[h], dist);
                keep(h, ok, ol, p0 + 32 * h, dist, size);
            }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        skey[base + p0 + 32 * h] = k[h];
        sjl[base + p0 + 32 * h] = l[h];
    }
}

// Final position of every candidate: its place in its own tile plus, for every other tile, the
// number of smaller keys there.  Four lanes per candidate share the tiles, each lane two binary
// searches at a time (the chain of probes is the cost); neighbouring candidates search for
// neighbouring keys, so their probes share cache lines.  The keys are distinct.
__global__ void __launch_bounds__(256)
select_rank_kernel(int m, int kmax, unsigned cap, const unsigned long long *__restrict__ skey,
                   const unsigned *__restrict__ sjl, const Geo *__restrict__ geo, int32_t *__restrict__ out_i,
                   int32_t *__restrict__ out_j, double *__restrict__ out_d, int32_t *__restrict__ out_count) {
    if (geo->gather_bound > cap) return;   // redone by the host with an exact-size buffer
    const unsigned e = blockIdx.x * 64 + (threadIdx.x >> 2), part = threadIdx.x & 3;
    if (blockIdx.x == 0 && threadIdx.x == 0) *out_count = (int)min((unsigned)kmax, geo->nvalid);
    const int ntiles = (int)((geo->ncand + kSelT - 1) / kSelT), own = (int)(e / kSelT);
    if (own >= ntiles) return;             // uniform over the block (64 candidates of one tile)
    const unsigned long long k = skey[e];
    const unsigned l = sjl[e];
    unsigned rank = part == 0 ? e % kSelT : 0u;
    auto probe = [&](unsigned at) { return key_less(skey[at], sjl[at], k, l); };
    for (int t = (int)part; k != ~0ull && t < ntiles && rank < (unsigned)kmax; t += 8) {
        const int t2 = t + 4;
        const unsigned ba = (unsigned)t * kSelT, bb = (unsigned)min(t2, ntiles - 1) * kSelT;
        unsigned a = 0, b = 0;
#pragma unroll
        for (int s = kSelT / 2; s > 0; s >>= 1) {
            if (probe(ba + a + s - 1)) a += s;
            if (probe(bb + b + s - 1)) b += s;
        }
        if (a == kSelT - 1 && probe(ba + a)) ++a;
        if (b == kSelT - 1 && probe(bb + b)) ++b;
        if (t != own) rank += a;
        if (t2 < ntiles && t2 != own) rank += b;
    }
    rank += __shfl_xor_sync(0xffffffffu, rank, 1);
    rank += __shfl_xor_sync(0xffffffffu, rank, 2);
    if (part == 0 && k != ~0ull && rank < (unsigned)kmax) {
        out_i[rank] = (int32_t)(l % (unsigned)m);
        out_j[rank] = (int32_t)(l / (unsigned)m);
        if (out_d) out_d[rank] = f64_from_key(k);
    }
}

// The same for candidate sets beyond the fixed capacity: keys for a stable radix sort by (d, jlin)
__global__ void recheck_kernel(int m, int n, int kind, unsigned long long count, const int32_t *__restrict__ ci,
                               const int32_t *__restrict__ cj, const int32_t *__restrict__ sx,
                               const int32_t *__restrict__ sy, const int32_t *__restrict__ tx,
                               const int32_t *__restrict__ ty, const double *__restrict__ u,
                               const double *__restrict__ v, const double *__restrict__ C,
                               const int32_t *__restrict__ row_ptr,
                               const int32_t *__restrict__ sup_j, Geo *geo,
                               uint64_t *__restrict__ key, uint32_t *__restrict__ val,
                               uint64_t *__restrict__ dkey) {
    const unsigned ncand = geo->ncand;
    for (unsigned long long g = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; g < count;
         g += (unsigned long long)gridDim.x * blockDim.x) {
        uint64_t kj = ~0ull, kd = ~0ull;
        if (g < ncand) {
            const int i = ci[g], j = cj[g];
            double d;
            kj = (uint64_t)i + (uint64_t)j * (uint64_t)m;
            if (recheck_pair(i, j, n, kind, sx, sy, tx, ty, u, v, C, row_ptr, sup_j, d)) {
                kd = f64_key(d);
                atomicAdd(&geo->nvalid, 1u);
            }
        }
        key[g] = kj;
        val[g] = (uint32_t)g;
        dkey[g] = kd;
    }
}

__global__ void rekey_kernel(unsigned long long count, const uint32_t *__restrict__ val,
                             const uint64_t *__restrict__ dkey, uint64_t *__restrict__ key) {
    for (unsigned long long g = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; g < count;
         g += (unsigned long long)gridDim.x * blockDim.x)
        key[g] = dkey[val[g]];
}

// (key: the reduced costs' keys, sorted)
__global__ void finalize_kernel(int kmax, const uint32_t *__restrict__ val, const int32_t *__restrict__ ci,
                                const int32_t *__restrict__ cj, const uint64_t *__restrict__ key,
                                const Geo *__restrict__ geo, int32_t *__restrict__ out_i,
                                int32_t *__restrict__ out_j, double *__restrict__ out_d,
                                int32_t *__restrict__ out_count) {
    const int cnt = (int)min((unsigned)kmax, geo->nvalid);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        const uint32_t g = val[k];
        out_i[k] = ci[g];
        out_j[k] = cj[g];
        if (out_d) out_d[k] = f64_from_key(key[k]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *out_count = cnt;
}

// rp[r] = first entry of row >= r: entry e fills the rows after its predecessor's up to its own (the
// last one the rest).  A warp's lanes with longer gaps are served by the whole warp in turn.
__global__ void row_ptr_kernel(const int32_t *__restrict__ sup_i, int64_t psi, int m, int32_t *__restrict__ rp) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; e0 <= psi; e0 += stride) {
        const int64_t e = e0 + lane;
        int lo = 0, hi = -1;   // rows lo .. hi get e
        if (e <= psi) {
            lo = e > 0 ? sup_i[e - 1] + 1 : 0;
            hi = e < psi ? sup_i[e] : m;
        }
        if (lo == hi) rp[lo] = (int32_t)e;
        unsigned wide = __ballot_sync(0xffffffffu, lo < hi);
        while (wide) {
            const int q = __ffs(wide) - 1;
            wide &= wide - 1;
            const int a = __shfl_sync(0xffffffffu, lo, q), b = __shfl_sync(0xffffffffu, hi, q);
            for (int r = a + lane; r <= b; r += 32) rp[r] = (int32_t)(e0 + q);
        }
    }
}

// J list (Section 3.4): the pairs with c_ij < C_max, sorted by (i, j).  One block per (row,
// chunk of kJC columns): count, then (after an exclusive scan over the counts) fill in order.
constexpr int kJC = 2048;

__device__ __forceinline__ bool in_jset(int kind, int i, int j, int n, const int32_t *sx, const int32_t *sy,
                                        const int32_t *tx, const int32_t *ty, const double *C, long long jlim,
                                        double jcmax) {
    if (kind == K_DN) return C[(int64_t)i * n + j] < jcmax;
    return cost_key(kind, sx[i] - tx[j], sy[i] - ty[j]) < jlim;
}

__global__ void jcount_kernel(int m, int n, int kind, const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
                              const int32_t *__restrict__ tx, const int32_t *__restrict__ ty,
                              const double *__restrict__ C, long long jlim, double jcmax,
                              uint32_t *__restrict__ counts, unsigned long long *__restrict__ total) {
    __shared__ int sh[kPT / 32];
    const int nch = (int)ceil_div(n, kJC);
    const int64_t blk = blockIdx.x;
    const int i = (int)(blk / nch), c0 = (int)(blk % nch) * kJC;
    int cnt = 0;
    for (int j = c0 + threadIdx.x; j < min(n, c0 + kJC); j += kPT)
        cnt += in_jset(kind, i, j, n, sx, sy, tx, ty, C, jlim, jcmax) ? 1 : 0;
    cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < kPT / 32; ++w) s += sh[w];
        counts[blk] = (uint32_t)s;
        atomicAdd(total, (unsigned long long)s);
    }
}

__global__ void jfill_kernel(int m, int n, int kind, const int32_t *__restrict__ sx, const int32_t *__restrict__ sy,
                             const int32_t *__restrict__ tx, const int32_t *__restrict__ ty,
                             const double *__restrict__ C, long long jlim, double jcmax,
                             const uint32_t *__restrict__ offs, int32_t *__restrict__ ji, int32_t *__restrict__ jj) {
    __shared__ int wtot[kPT / 32];
    const int nch = (int)ceil_div(n, kJC);
    const int64_t blk = blockIdx.x;
    const int i = (int)(blk / nch), c0 = (int)(blk % nch) * kJC;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t base = offs[blk];
    for (int r = 0; r < kJC / kPT; ++r) {
        const int j = c0 + r * kPT + threadIdx.x;
        const bool f = j < n && in_jset(kind, i, j, n, sx, sy, tx, ty, C, jlim, jcmax);
        const unsigned bal = __ballot_sync(0xffffffffu, f);
        if (lane == 0) wtot[wid] = __popc(bal);
        __syncthreads();
        int before = 0, all = 0;
        for (int w = 0; w < kPT / 32; ++w) { if (w < wid) before += wtot[w]; all += wtot[w]; }
        if (f) {
            const int64_t pos = base + before + __popc(bal & ((1u << lane) - 1u));
            ji[pos] = i;
            jj[pos] = j;
        }
        base += all;
        __syncthreads();
    }
}

}  // namespace

Error build_row_ptr(const int32_t *sup_i, int64_t psi, int32_t m, int32_t *row_ptr, cudaStream_t st) {
    row_ptr_kernel<<<(unsigned)std::min<int64_t>(ceil_div(psi + 1, 256), 4096), 256, 0, st>>>(sup_i, psi, m, row_ptr);
    OT_LAUNCHED();
    return ok();
}

long long jset_limit(int kind, double cmax) {
    if (!(cmax > 0)) return 0;
    // smallest integer key D whose cost is >= cmax (costs are nondecreasing in the key)
    long long lo = 0, hi = 1LL << 33;
    while (lo < hi) {
        const long long mid = lo + (hi - lo) / 2;
        const double c = kind == K_EU ? std::sqrt((double)mid) : (double)mid;
        if (c >= cmax) hi = mid; else lo = mid + 1;
    }
    return lo;
}

void jset_free(JSet &J) {
    if (J.i) cudaFree(J.i);
    if (J.j) cudaFree(J.j);
    J = JSet();
}

Error jset_build(int kind, int32_t m, int32_t n, const int32_t *sx, const int32_t *sy, const int32_t *tx,
                 const int32_t *ty, const double *C, double cmax, JSet *out, cudaStream_t st) {
    jset_free(*out);
    if (m <= 0 || n <= 0 || !(cmax > 0)) return fail(OT_ERR_ARG, "J set: sizes or C_max out of range");
    if (kind == K_DN ? !C : (!sx || !sy || !tx || !ty)) return fail(OT_ERR_ARG, "J set: missing cost data");
    const long long lim = kind == K_DN ? 0 : jset_limit(kind, cmax);
    const int64_t nch = ceil_div(n, kJC), nblk = (int64_t)m * nch;
    if (nblk > 0x7fffffffLL) return fail(OT_ERR_ARG, "J set: too many row chunks");
    DevTemp<uint32_t> counts;
    DevTemp<unsigned long long> total;
    OT_TRY(counts.alloc(nblk, st));
    OT_TRY(total.alloc(1, st));
    OT_CUDA(cudaMemsetAsync(total.p, 0, sizeof(unsigned long long), st));
    jcount_kernel<<<(unsigned)nblk, kPT, 0, st>>>(m, n, kind, sx, sy, tx, ty, C, lim, cmax, counts.p, total.p);
    OT_LAUNCHED();
    unsigned long long tot = 0;
    OT_CUDA(cudaMemcpyAsync(&tot, total.p, sizeof(tot), cudaMemcpyDeviceToHost, st));
    OT_CUDA(cudaStreamSynchronize(st));
    if (tot > 0x7fffffffull) return fail(OT_ERR_ARG, "J set: more than 2^31 pairs (lower C_max)");
    JSet J;
    J.n = (int64_t)tot;
    J.lim = lim;
    J.cmax = cmax;
    OT_CUDA(cudaMalloc((void **)&J.i, sizeof(int32_t) * std::max<int64_t>(J.n, 1)));
    Error e = [&]() -> Error {
        OT_CUDA(cudaMalloc((void **)&J.j, sizeof(int32_t) * std::max<int64_t>(J.n, 1)));
        OT_TRY(scan_exclusive_u32(counts.p, counts.p, nblk, nullptr, st));
        jfill_kernel<<<(unsigned)nblk, kPT, 0, st>>>(m, n, kind, sx, sy, tx, ty, C, lim, cmax, counts.p, J.i, J.j);
        OT_LAUNCHED();
        OT_CUDA(cudaStreamSynchronize(st));
        return ok();
    }();
    if (e.code != OT_OK) { jset_free(J); return e; }
    *out = J;
    return ok();
}

namespace {

// What the passes read: FP32 points in the caller's order and in cell order, the tile list.
struct ScanData {
    bool fp64 = false, narrow = false;
    int TI = 0, ncb = 0;          // FP64 scan
    int64_t ntiles = 0;           // FP64 tiles or J-list tiles
    int G = 0, nrg = 0, ncg = 0;  // FP32 tiles: rows per group, row and column groups
    float4 *rows = nullptr, *cols = nullptr, *srt = nullptr;
    float *sdual = nullptr;
    Group *grp = nullptr;
    unsigned *list = nullptr, *cells = nullptr, *place = nullptr;
    float *tmin = nullptr;
    Geo *geo = nullptr;
    unsigned long long *hist = nullptr;
};

// One scan pass for cost kind K.  S.first tile blocks; the histogram pass has sup_blocks more for the
// support.
template <int K>
Error scan_pass(const PriceInput &in, const ScanData &D, bool gather, const SupArgs &S, int sup_blocks, int32_t *ci,
                int32_t *cj, unsigned long long cap, cudaStream_t st) {
    const int grid = S.first + (gather ? 0 : sup_blocks);
    unsigned *ncand = &D.geo->ncand;
    auto scan = [&](auto ga) {
        constexpr bool G = decltype(ga)::value;
        if (in.jn >= 0) {
            auto j = [&](auto fp) {
                jscan_kernel<K, decltype(fp)::value, G><<<grid, kPT, 0, st>>>(
                    in.n, in.jn, D.ntiles, S, in.ji, in.jj, D.rows, D.cols, in.sx, in.sy, in.tx, in.ty, in.u, in.v,
                    in.C, D.geo, D.tmin, D.hist, ci, cj, cap, ncand);
            };
            if constexpr (K == K_DN) j(std::true_type());
            else D.fp64 ? j(std::true_type()) : j(std::false_type());
            return;
        }
        if constexpr (K != K_DN) {
            if (!D.fp64) {
                tile_scan_kernel<K, G><<<grid, kPT, 0, st>>>(in.m, in.n, D.G, D.nrg, S, D.rows, D.cols, D.srt, in.sx,
                                                            in.sy, in.tx, in.ty, in.u, in.v, D.geo, D.list, D.tmin,
                                                            D.hist, ci, cj, cap, ncand);
                return;
            }
        }
        auto f = [&](auto rj) {
            scan64_kernel<K, G, decltype(rj)::value><<<grid, kPT, 0, st>>>(
                in.m, in.n, D.TI, D.ncb, D.ntiles, S, in.sx, in.sy, in.tx, in.ty, in.u, in.v, in.C, D.geo, D.tmin,
                D.hist, ci, cj, cap, ncand);
        };
        D.narrow ? f(std::integral_constant<int, kRJNarrow>()) : f(std::integral_constant<int, kRJ>());
    };
    gather ? scan(std::true_type()) : scan(std::false_type());
    OT_LAUNCHED();
    return ok();
}

// FP32 forms, error bound and tile list.
template <int K>
Error prepare_tiles(const PriceInput &in, const ScanData &D, int sms, cudaStream_t st) {
    const int m = in.m, n = in.n;
    const int pb = (int)std::min<int64_t>(4 * sms, ceil_div((int64_t)m + n, 256 * kPrepPer));
    const bool sort = in.jn < 0;
    if (in.have_box) {
        box_kernel<<<1, 32, 0, st>>>(in.box_lo[0], in.box_lo[1], in.box_hi[0], in.box_hi[1], D.geo);
    } else {
        bounds_kernel<<<pb, 256, 0, st>>>(m, n, in.sx, in.sy, in.tx, in.ty, D.geo);
    }
    OT_LAUNCHED();
    if (sort) {
        cells_kernel<<<pb, 256, 0, st>>>(m, n, in.sx, in.sy, in.tx, in.ty, D.geo, D.cells, D.place);
        OT_LAUNCHED();
    }
    prep_kernel<K == K_SQ><<<pb, 256, 0, st>>>(m, n, K, in.sx, in.sy, in.tx, in.ty, in.u, in.v, D.rows, D.cols,
                                               D.cells, sort ? D.place : nullptr, D.srt, D.sdual, D.geo);
    OT_LAUNCHED();
    if (sort) {
        const int64_t total = (int64_t)D.nrg * D.ncg;
        groups_kernel<<<(unsigned)std::min<int64_t>(ceil_div((int64_t)D.nrg + D.ncg, 8), 8LL * sms), 256, 0, st>>>(
            m, n, D.G, D.nrg, D.ncg, K == K_SQ ? -0.5f : 1.0f, D.srt, D.sdual, D.grp);
        OT_LAUNCHED();
        tiles_kernel<K><<<(unsigned)std::min<int64_t>(ceil_div(total, 256), 8LL * sms), 256, 0, st>>>(
            D.nrg, total, D.grp, D.geo, D.list);
        OT_LAUNCHED();
    }
    return ok();
}

template <typename F>
Error by_kind(int kind, F &&f) {
    switch (kind) {
    case K_SQ: return f(std::integral_constant<int, K_SQ>());
    case K_EU: return f(std::integral_constant<int, K_EU>());
    case K_L1: return f(std::integral_constant<int, K_L1>());
    case K_LI: return f(std::integral_constant<int, K_LI>());
    case K_DN: return f(std::integral_constant<int, K_DN>());
    default: return fail(OT_ERR_ARG, "price_topk: unknown cost kind");
    }
}

// Capacity of the candidate buffer that needs no host round trip (a multiple of kSelT): four times
// kmax, at least 8 and at most 128 tiles (the rank searches grow with tiles per candidate).
unsigned spec_capacity(int32_t kmax) {
    const int64_t want = ceil_div(4LL * kmax, kSelT) * kSelT;
    return (unsigned)std::max<int64_t>(8 * kSelT, std::min<int64_t>(want, 128 * kSelT));
}

PriceStats stats_of(const Geo &g, int32_t kmax) {
    PriceStats s;
    s.gathered = g.ncand;
    s.valid = g.nvalid;
    s.selected = std::min<uint32_t>((uint32_t)kmax, g.nvalid);
    s.err_bound = g.E;
    return s;
}

}  // namespace

Error price_topk(const PriceInput &in, int32_t *out_i, int32_t *out_j, double *out_d,
                 int32_t *out_count, PriceStats *stats, cudaStream_t st) {
    const int m = in.m, n = in.n;
    if (m <= 0 || n <= 0 || in.kmax < 0) return fail(OT_ERR_ARG, "price_topk: bad sizes");
    if ((uint64_t)m * (uint64_t)n > (1ull << 32)) return fail(OT_ERR_ARG, "price_topk: m*n > 2^32");
    const int kind = in.kind;
    if (kind < K_SQ || kind > K_DN) return fail(OT_ERR_ARG, "price_topk: unknown cost kind");
    if (kind == K_DN ? !in.C : (!in.sx || !in.sy || !in.tx || !in.ty))
        return fail(OT_ERR_ARG, "price_topk: missing coordinates or cost matrix");
    const bool jmode = in.jn >= 0;
    if (jmode && in.jn > 0 && (!in.ji || !in.jj)) return fail(OT_ERR_ARG, "price_topk: J list missing");
    const bool fp64 = in.precision == 0 || kind == K_DN;
    int sms = in.num_sms;
    if (sms <= 0) {
        int dev;
        OT_CUDA(cudaGetDevice(&dev));
        OT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    }
    // FP64 tiles: TI rows x kPT * RJ columns (aim for >= 4 tiles per SM); J list: kJT entries; FP32
    // tiles: G rows x 256 columns, one per warp (aim for >= 16 per SM before pruning)
    ScanData D;
    D.fp64 = fp64;
    const bool tiled32 = !fp64 && !jmode;
    D.narrow = n <= kNarrowN;
    D.ncb = (int)ceil_div(n, kPT * (D.narrow ? kRJNarrow : kRJ));
    D.TI = kPT;
    while (D.TI > (D.narrow ? 4 : 8) && ceil_div(m, D.TI) * (int64_t)D.ncb < 4LL * sms) D.TI >>= 1;
    D.ncg = (int)ceil_div(n, kCG);
    D.G = 64;
    while (D.G > 16 && ceil_div(m, D.G) * (int64_t)D.ncg < 16LL * sms) D.G >>= 1;
    if (in.rows > 0) D.TI = D.G = std::max(8, std::min(kPT, in.rows));
    D.nrg = (int)ceil_div(m, D.G);
    D.ntiles = jmode ? ceil_div(in.jn, kJT) : (int64_t)ceil_div(m, D.TI) * D.ncb;
    const int64_t ntiles = tiled32 ? (int64_t)D.nrg * D.ncg : D.ntiles;

    // one workspace: Geo, the two histograms (all pairs, the support's), FP32 points, tiles
    DevTemp<char> ws;
    size_t need = 0;
    auto take = [&](size_t bytes) { const size_t at = need; need += (bytes + 255) & ~(size_t)255; return at; };
    const size_t pts = (size_t)m + n;
    const size_t o_geo = take(sizeof(Geo)), o_hist = take(sizeof(unsigned long long) * 2 * kBins);
    const size_t o_cells = take(tiled32 ? sizeof(unsigned) * 2 * kCells : 0), zeroed = need;
    const size_t o_rows = take(fp64 ? 0 : sizeof(float4) * m), o_cols = take(fp64 ? 0 : sizeof(float4) * n);
    const size_t o_srt = take(tiled32 ? sizeof(float4) * pts : 0), o_dual = take(tiled32 ? sizeof(float) * pts : 0);
    const size_t o_place = take(tiled32 ? sizeof(unsigned) * pts : 0);
    const size_t o_grp = take(tiled32 ? sizeof(Group) * ((size_t)D.nrg + D.ncg) : 0);
    const size_t o_list = take(tiled32 ? sizeof(unsigned) * ntiles : 0);
    const size_t o_tmin = take(sizeof(float) * std::max<int64_t>(ntiles, 1));
    const size_t o_rp = take(in.row_ptr ? 0 : sizeof(int32_t) * ((size_t)m + 1));
    OT_TRY(ws.alloc((int64_t)need, st));
    Geo *geo = D.geo = (Geo *)(ws.p + o_geo);
    unsigned long long *hist = D.hist = (unsigned long long *)(ws.p + o_hist), *hist_sup = hist + kBins;
    D.tmin = (float *)(ws.p + o_tmin);
    if (!fp64) {
        D.rows = (float4 *)(ws.p + o_rows);
        D.cols = (float4 *)(ws.p + o_cols);
    }
    if (tiled32) {
        D.cells = (unsigned *)(ws.p + o_cells);
        D.srt = (float4 *)(ws.p + o_srt);
        D.sdual = (float *)(ws.p + o_dual);
        D.place = (unsigned *)(ws.p + o_place);
        D.grp = (Group *)(ws.p + o_grp);
        D.list = (unsigned *)(ws.p + o_list);
    }
    OT_CUDA(cudaMemsetAsync(ws.p, 0, zeroed, st));

    const int32_t *rp = in.row_ptr;   // support membership needs CSR rows
    if (!rp) {
        int32_t *own = (int32_t *)(ws.p + o_rp);
        OT_TRY(build_row_ptr(in.sup_i, in.psi, m, own, st));
        rp = own;
    }
    if (!fp64)   // (E stays 0 in the FP64 variant)
        OT_TRY(by_kind(kind, [&](auto kc) -> Error {
            if constexpr (decltype(kc)::value == K_DN) return ok();
            else return prepare_tiles<decltype(kc)::value>(in, D, sms, st);
        }));

    SupArgs S{in.sup_i, in.sup_j, in.psi, jmode ? in.jlim : 0, jmode ? in.jcmax : 0.0, 0, hist_sup};
    S.first = (int)std::max<int64_t>(1, tiled32 ? std::min<int64_t>(ceil_div(ntiles, kPT / 32), 3LL * sms)
                                                : std::min<int64_t>(ntiles, 8LL * sms));
    const int sup_blocks = (int)std::min<int64_t>(2 * sms, ceil_div(in.psi, 4 * kPT));
    auto pass = [&](bool gather, int32_t *ci, int32_t *cj, unsigned long long cap) -> Error {
        ktimer_begin(gather ? KT_SCAN_GATHER : KT_SCAN_HIST, st);
        OT_TRY(by_kind(kind, [&](auto kc) {
            return scan_pass<decltype(kc)::value>(in, D, gather, S, sup_blocks, ci, cj, cap, st);
        }));
        ktimer_end(gather ? KT_SCAN_GATHER : KT_SCAN_HIST, st);
        return ok();
    };
    if (ntiles > 0) OT_TRY(pass(false, nullptr, nullptr, 0));   // (an empty J list holds no support pair either)
    threshold_kernel<<<1, 1024, 0, st>>>(hist, hist_sup, std::max(in.kmax, 1), fp64 ? 1 : 0, geo);
    OT_LAUNCHED();
    Geo hg;
    {
        // the gathered set rarely passes a few times kmax (its last bin is a sixty-fourth of an octave of
        // |d|, plus the support's pairs and the FP32 window)
        const unsigned cap = spec_capacity(in.kmax);
        DevTemp<char> cand;
        OT_TRY(cand.alloc((int64_t)cap * (2 * sizeof(int32_t) + sizeof(unsigned long long) + sizeof(unsigned)), st));
        unsigned long long *skey = (unsigned long long *)cand.p;
        unsigned *sjl = (unsigned *)(skey + cap);
        int32_t *ci = (int32_t *)(sjl + cap), *cj = ci + cap;
        if (ntiles > 0) OT_TRY(pass(true, ci, cj, cap));
        ktimer_begin(KT_RECHECK, st);
        select_sort_kernel<<<cap / kSelT, kSelT / 2, 0, st>>>(m, n, kind, cap, ci, cj, in.sx, in.sy, in.tx, in.ty, in.u,
                                                              in.v, in.C, rp, in.sup_j, geo, skey, sjl);
        OT_LAUNCHED();
        ktimer_end(KT_RECHECK, st);
        select_rank_kernel<<<cap / 64, 256, 0, st>>>(m, in.kmax, cap, skey, sjl, geo, out_i, out_j, out_d, out_count);
        OT_LAUNCHED();
        OT_CUDA(cudaMemcpyAsync(&hg, geo, sizeof(Geo), cudaMemcpyDeviceToHost, st));
        OT_CUDA(cudaStreamSynchronize(st));
        // the pairs that pass 1 evaluated, in FP32 operations
        const double per_pair = kind == K_SQ ? 4.0 : (kind == K_EU ? 8.0 : 6.0);
        ktimer_add_work(KT_SCAN_HIST, per_pair * (jmode ? (double)in.jn
                                                  : tiled32 ? (double)hg.ntile * D.G * kCG : (double)m * (double)n));
        if (hg.gather_bound <= cap) {
            if (stats) *stats = stats_of(hg, in.kmax);
            return ok();
        }
    }
    const unsigned long long cap = hg.gather_bound;
    if (!fp64 && cap > kMaxWindowPairs) {
        // fewer negative keys than kmax and a flood of pairs inside the FP32 window [0, E] (duals
        // near a degenerate optimum): the exact FP64 scan gathers only the pairs with d < 0
        PriceInput in64 = in;
        in64.precision = 0;
        return price_topk(in64, out_i, out_j, out_d, out_count, stats, st);
    }
    if (cap > 0x7fffffffull) return fail(OT_ERR_OOM, "price_topk: candidate set exceeds 2^31 pairs");

    // beyond the fixed capacity: pass 2 again into buffers of the exact size, then stable radix sorts
    const int64_t cnt = (int64_t)cap;
    DevTemp<int32_t> ci, cj;
    OT_TRY(ci.alloc(cnt, st));
    OT_TRY(cj.alloc(cnt, st));
    OT_CUDA(cudaMemsetAsync(&geo->ncand, 0, sizeof(unsigned), st));
    OT_CUDA(cudaMemsetAsync(&geo->nvalid, 0, sizeof(unsigned), st));
    OT_TRY(pass(true, ci.p, cj.p, cap));
    DevTemp<uint64_t> key, dkey;
    DevTemp<uint32_t> val;
    OT_TRY(key.alloc(cnt, st));
    OT_TRY(dkey.alloc(cnt, st));
    OT_TRY(val.alloc(cnt, st));
    const int rb = (int)std::min<int64_t>(8 * sms, ceil_div(cnt, 256));
    ktimer_begin(KT_RECHECK, st);
    recheck_kernel<<<rb, 256, 0, st>>>(m, n, kind, cap, ci.p, cj.p, in.sx, in.sy, in.tx, in.ty, in.u, in.v, in.C, rp,
                                       in.sup_j, geo, key.p, val.p, dkey.p);
    OT_LAUNCHED();
    ktimer_end(KT_RECHECK, st);
    int jbits = 1;
    while (jbits < 64 && ((uint64_t)m * (uint64_t)n - 1) >> jbits) ++jbits;
    OT_TRY(radix_sort_pairs(key.p, val.p, cnt, jbits, st));
    rekey_kernel<<<rb, 256, 0, st>>>(cap, val.p, dkey.p, key.p);
    OT_LAUNCHED();
    OT_TRY(radix_sort_pairs(key.p, val.p, cnt, 64, st));
    finalize_kernel<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(in.kmax, 256), 4 * sms)), 256, 0, st>>>(
        in.kmax, val.p, ci.p, cj.p, key.p, geo, out_i, out_j, out_d, out_count);
    OT_LAUNCHED();
    OT_CUDA(cudaMemcpyAsync(&hg, geo, sizeof(Geo), cudaMemcpyDeviceToHost, st));
    OT_CUDA(cudaStreamSynchronize(st));
    if (stats) *stats = stats_of(hg, in.kmax);
    return ok();
}

}  // namespace ot
