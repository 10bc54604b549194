// FP64 kernels of the outer flexible GMRES (dot products, classical Gram-Schmidt, gauge
// projection) and of the coarsest-grid exact solve (dense operator, Gauss-Jordan inverse,
// pseudo-inverse apply).  All reductions use a fixed block count and a fixed reduction tree,
// so results are bitwise reproducible run to run.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "sib_internal.h"

namespace cg = cooperative_groups;

namespace sib {

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) ws[wid] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? ws[threadIdx.x] : 0.0;
    if (wid == 0)
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;   // valid in thread 0
}

__global__ void k_dot_partials(const double* __restrict__ x, const double* __restrict__ y, int64_t n,
                               double* __restrict__ partials) {
    pdl_entry();
    double s = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        s += x[k] * y[k];
    s = block_sum(s);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}
void launch_dot_partials(const double* x, const double* y, int64_t n, double* partials, int nblk, cudaStream_t s) {
    launch_pdl(k_dot_partials, nblk, 256, 0, s, x, y, n, partials);
}

// partials[i * nblk + b] = sum over block b's slice of V_i . w, for i < k
__global__ void k_multidot(const double* __restrict__ V, int64_t ld, const double* __restrict__ w, int64_t n,
                           double* __restrict__ partials) {
    pdl_entry();
    const int i = blockIdx.y;
    const double* v = V + (int64_t)i * ld;
    double s = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        s += v[k] * w[k];
    s = block_sum(s);
    if (threadIdx.x == 0) partials[(int64_t)i * gridDim.x + blockIdx.x] = s;
}
void launch_multidot(const double* V, int64_t ld, int k, const double* w, int64_t n, double* partials, int nblk,
                     cudaStream_t s) {
    launch_pdl(k_multidot, dim3(nblk, k), 256, 0, s, V, ld, w, n, partials);
}

__global__ void k_reduce_partials(const double* __restrict__ partials, int nblk, double* __restrict__ out) {
    pdl_entry();
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += partials[(int64_t)blockIdx.x * nblk + b];
    s = block_sum(s);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}
void launch_reduce_partials(const double* partials, int k, int nblk, double* out, cudaStream_t s) {
    launch_pdl(k_reduce_partials, k, 256, 0, s, partials, nblk, out);
}

// y += sign * sum_{i<k} coef[i] V_i
__global__ void k_multi_axpy(const double* __restrict__ V, int64_t ld, int k, const double* __restrict__ coef,
                             double sign, double* __restrict__ y, int64_t n) {
    pdl_entry();
    __shared__ double c[128];
    for (int t = threadIdx.x; t < k; t += blockDim.x) c[t] = sign * coef[t];
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double acc = y[e];
        for (int i = 0; i < k; ++i) acc += c[i] * V[(int64_t)i * ld + e];
        y[e] = acc;
    }
}
void launch_multi_axpy(const double* V, int64_t ld, int k, const double* coef, double sign, double* y, int64_t n,
                       cudaStream_t s) {
    launch_pdl(k_multi_axpy, num_blocks_for(n), 256, 0, s, V, ld, k, coef, sign, y, n);
}

// x *= 1 / sqrt(vals[idx])   (normalisation of the next Arnoldi vector)
__global__ void k_scale_rsqrt(double* __restrict__ x, const double* __restrict__ vals, int idx, int64_t n) {
    pdl_entry();
    const double nrm = sqrt(vals[idx]);
    const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        x[k] *= inv;
}
void launch_scale(double* x, const double* vals, int idx, int64_t n, cudaStream_t s) {
    launch_pdl(k_scale_rsqrt, num_blocks_for(n), 256, 0, s, x, vals, idx, n);
}

// gauge projection: means of the u, v, p blocks and their removal (mask bit b = block b)
__global__ void k_block_means(const double* __restrict__ x, int64_t n, double* __restrict__ partials) {
    pdl_entry();
    const double* xb = x + blockIdx.y * n;
    double s = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        s += xb[k];
    s = block_sum(s);
    if (threadIdx.x == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = s;
}
void launch_block_means(const double* x, int N, int nblocks_vec, double* partials, int nblk, cudaStream_t s) {
    launch_pdl(k_block_means, dim3(nblk, nblocks_vec), 256, 0, s, x, (int64_t)N * N, partials);
}
__global__ void k_subtract_means(double* __restrict__ x, int64_t n, const double* __restrict__ partials, int nblk,
                                 int mask) {
    pdl_entry();
    __shared__ double mean[3];
    if (threadIdx.x < 32) {
        for (int b = 0; b < 3; ++b) {
            double s = 0.0;
            for (int q = threadIdx.x; q < nblk; q += 32) s += partials[b * nblk + q];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (threadIdx.x == 0) mean[b] = ((mask >> b) & 1) ? s / (double)n : 0.0;
        }
    }
    __syncthreads();
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < 3 * n; k += (int64_t)gridDim.x * blockDim.x)
        x[k] -= mean[k / n];
}
void launch_subtract_means(double* x, int N, const double* partials, int nblk, int mask, cudaStream_t s) {
    const int64_t n = (int64_t)N * N;
    launch_pdl(k_subtract_means, num_blocks_for(3 * n), 256, 0, s, x, n, partials, nblk, mask);
}

// ------------------------------------------------------------------------------------------
// Coarsest level: dense L^0 + Z Z^T (Z = orthonormal kernel basis: the constant pressure, and
// the constant velocity components when rho = 0), augmented with the identity: Aug = [L0+ZZ^T | I].
// One thread per entry: momentum rows hold A = a0 I - mu Lap (5-point, periodic), + G and - dt [SKJ]^0;
// pressure rows hold - D.  Coincident periodic neighbours add up (counted per offset).
__global__ void k_assemble_L0(int N, double rho, double mu, double dt, const double* __restrict__ B,
                              double* __restrict__ Aug) {
    pdl_entry();
    const int n0 = N * N, n = 3 * n0, mk = N - 1;
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= (int64_t)n * 2 * n) return;
    const int r = (int)(q / (2 * n)), col = (int)(q % (2 * n));
    if (col >= n) {
        Aug[q] = (col - n == r) ? 1.0 : 0.0;
        return;
    }
    const double h = 1.0 / N, ih = (double)N;
    const double a0 = rho / dt + 4.0 * mu / (h * h), cc = mu / (h * h);
    const int br = r / n0, f = r % n0, i = f % N, j = f / N;
    const int bc = col / n0, gcell = col % n0;
    double v = 0.0;
    if (br < 2) {
        if (bc == br) {
            if (gcell == f) v += a0;
            if (gcell == j * N + ((i + 1) & mk)) v -= cc;
            if (gcell == j * N + ((i - 1) & mk)) v -= cc;
            if (gcell == ((j + 1) & mk) * N + i) v -= cc;
            if (gcell == ((j - 1) & mk) * N + i) v -= cc;
            v -= dt * B[(int64_t)br * n0 * n0 + (int64_t)f * n0 + gcell];
        } else if (bc == 2) {   // G p: (p_ij - p_{i-1,j})/h on u faces, (p_ij - p_{i,j-1})/h on v faces
            if (gcell == f) v += ih;
            if (gcell == (br == 0 ? j * N + ((i - 1) & mk) : ((j - 1) & mk) * N + i)) v -= ih;
        }
    } else if (bc < 2) {        // - D u
        if (bc == 0) {
            if (gcell == f) v += ih;
            if (gcell == j * N + ((i + 1) & mk)) v -= ih;
        } else {
            if (gcell == f) v += ih;
            if (gcell == ((j + 1) & mk) * N + i) v -= ih;
        }
    }
    if (bc == br && (rho == 0.0 || br == 2)) v += 1.0 / (double)n0;
    Aug[q] = v;
}
void launch_assemble_L0(int N0, double rho, double mu, double dt, const double* B, double* Aug, cudaStream_t s) {
    const int64_t tot = (int64_t)3 * N0 * N0 * 6 * N0 * N0;
    launch_pdl(k_assemble_L0, (int)((tot + 255) / 256), 256, 0, s, N0, rho, mu, dt, B, Aug);
}

// Blocked Gauss-Jordan inversion with partial pivoting of Aug = [A | I] (n x 2n, row-major), in
// panels of GJ_B columns.  For the panel Q = columns [c0, c0 + GJ_B):
//   1. one block selects the panel's pivot rows P by partial pivoting on a working copy of the
//      panel's candidate rows (largest |a| among rows not yet pivots, ties to the lower row, the
//      copy eliminated as unblocked elimination would), and inverts the pivot block A_PQ in FP64
//      with its pivots on the diagonal in selection order.  The working copy only chooses rows --
//      the result is computed from the FP64 panel and A_PQ^{-1} -- so it is kept in FP32: one SM's
//      FP64 rate made an FP64 copy cost ~120 us a panel, and FP32 can change a choice only between
//      candidates equal to rounding, which partial pivoting leaves free;
//   2. column slabs form the new pivot rows  W = A_PQ^{-1} A_P  on the columns right of Q;
//   3. every other row r becomes  A_r - A_rQ W  there (A_rQ: its panel entries before the panel's
//      elimination), and its panel entries 0 (the pivot rows' panel entries become unit vectors).
// Rows are never swapped: piv[k] is the pivot row of column k and row k of A^{-1} is
// Aug[piv[k]][n:].  A zero *info (the caller clears it, once for a series of inversions that share the word) becomes
// k + 1 for the first pivot column without a nonzero candidate.
// The panel steps are sequential but tiny; the O(n^3) work of step 3 spreads over the GPU, whose
// FP64 rate is low per SM.
constexpr int GJ_B = 16;

struct GjWork {
    double* Q0;   // n x GJ_B: the panel before its elimination
    double* G;    // GJ_B x GJ_B: A_PQ^{-1}
    double* W;    // GJ_B x 2n: the new pivot rows
    int* used;    // n: row already a pivot
    int* prow;    // GJ_B: the panel's pivot rows in selection order
};
static GjWork gj_work(void* base, int n) {
    GjWork w;
    double* d = static_cast<double*>(base);
    w.Q0 = d;
    w.G = w.Q0 + (size_t)n * GJ_B;
    w.W = w.G + GJ_B * GJ_B;
    w.used = reinterpret_cast<int*>(w.W + (size_t)GJ_B * 2 * n);
    w.prow = w.used + n;
    return w;
}
size_t gauss_jordan_work_bytes(int n) {
    return sizeof(double) * ((size_t)n * GJ_B + GJ_B * GJ_B + (size_t)GJ_B * 2 * n) + sizeof(int) * (size_t)(n + GJ_B);
}

// The end of a panel: G = A_PQ^{-1} for the chosen rows pS, by the whole block (at least GJ_B^2 threads)
__device__ __forceinline__ void gj_pivot_block(int c0, GjWork w, const int* pS, int* piv, int* info) {
    __shared__ double colv[2][GJ_B], rowv[2][GJ_B], rcp[2];
    const int r = threadIdx.x;
    // Gauss-Jordan in place in FP64 with the pivots on the diagonal; entry (s, u) of column u < t already belongs
    // to the inverse, whose column t appears at step t as a unit vector
    const int s = r / GJ_B, u = r % GJ_B;
    const bool in = r < GJ_B * GJ_B;
    double m = in ? w.Q0[(size_t)pS[s] * GJ_B + u] : 0.0;
    auto next_pivot = [&](int t) {
        if (!(m != 0.0) && *info == 0) *info = c0 + t + 1;
        rcp[t & 1] = m != 0.0 ? 1.0 / m : 0.0;
    };
    if (r == 0) next_pivot(0);
    for (int t = 0; t < GJ_B; ++t) {
        const int b = t & 1;
        if (in && u == t) colv[b][s] = m;
        if (in && s == t) rowv[b][u] = u == t ? 1.0 : m;
        __syncthreads();
        if (!in) continue;
        const double ipv = rcp[b], rv = rowv[b][u];
        if (s == t) {
            m = rv * ipv;
        } else {
            const double f = colv[b][s] * ipv;
            m = (u == t ? 0.0 : m) - f * rv;
        }
        if (s == t + 1 && u == s) next_pivot(t + 1);
    }
    if (in) w.G[r] = m;
    if (r < GJ_B) {
        w.prow[r] = pS[r];
        piv[c0 + r] = pS[r];
    }
}

// One block, one candidate row per thread, its panel entries in registers.  The panels are the serial chain of
// the inversion, a latency each: a pivot search is two warp-wide maxima with one barrier between them, every
// warp's best row waiting in shared memory so that the winner's needs no second trip, and the pivot block is
// inverted in place, one entry per thread, its reciprocal formed by the one thread that updates it (a division
// in every warp cost the FP64 pipe more than the step's updates).  192 rows: 42 us a panel with the working
// copy in shared memory, 16.5 us so (the whole inversion of 192 x 192: 575 -> 330 us).
constexpr int GJ_MAXN = 768;   // 3 * 16^2, the largest coarsest grid
__global__ void __launch_bounds__(GJ_MAXN) k_gj_panel(const double* __restrict__ A, int n, int c0, GjWork w,
                                                      int* __restrict__ piv, int* __restrict__ info) {
    pdl_entry();
    __shared__ float cand[2][32][GJ_B];   // every warp's best row, its size and index (two steps in turn)
    __shared__ unsigned ckey[2][32];
    __shared__ int crow[2][32];
    __shared__ int pS[GJ_B];
    const int r = threadIdx.x, lane = r & 31, wid = r >> 5, nw = blockDim.x >> 5;
    float a[GJ_B] = {};
    bool used = true;
    if (r < n) {
        used = c0 != 0 && w.used[r];
        const double2* row = reinterpret_cast<const double2*>(A + (size_t)r * 2 * n + c0);
        double2* q0 = reinterpret_cast<double2*>(w.Q0 + (size_t)r * GJ_B);
        double2 v[GJ_B / 2];
#pragma unroll
        for (int q = 0; q < GJ_B / 2; ++q) v[q] = row[q];
#pragma unroll
        for (int q = 0; q < GJ_B / 2; ++q) {
            q0[q] = v[q];
            a[2 * q] = (float)v[q].x;
            a[2 * q + 1] = (float)v[q].y;
        }
    }
#pragma unroll
    for (int t = 0; t < GJ_B; ++t) {
        const int b = t & 1;
        // magnitudes order as their bits do; 0: no candidate, 1: a zero (or not a number)
        const float m = fabsf(a[t]);
        const unsigned key = used ? 0u : (m >= 0.0f ? __float_as_uint(m) + 1u : 1u);
        const unsigned wbest = __reduce_max_sync(0xffffffffu, key);
        const int src = __ffs(__ballot_sync(0xffffffffu, key == wbest)) - 1;   // ties to the lower row
        if (lane == src) {
            ckey[b][wid] = key;
            crow[b][wid] = r;
#pragma unroll
            for (int q = t; q < GJ_B; ++q) cand[b][wid][q] = a[q];
        }
        __syncthreads();
        const unsigned k = lane < nw ? ckey[b][lane] : 0u;
        const unsigned best = __reduce_max_sync(0xffffffffu, k);
        const int ww = __ffs(__ballot_sync(0xffffffffu, k == best)) - 1;
        const int p = crow[b][ww];
        if (r == 0) pS[t] = p;
        used = used || r == p;
        const float pv = cand[b][ww][t];
        const float ipv = pv != 0.0f ? 1.0f / pv : 0.0f;
        const float f = a[t] * ipv;
        if (!used && f != 0.0f) {
#pragma unroll
            for (int q = t + 1; q < GJ_B; ++q) a[q] -= f * cand[b][ww][q];
        }
    }
    __syncthreads();
    gj_pivot_block(c0, w, pS, piv, info);
    if (r < n) w.used[r] = used;
}

// The same with the working copy in shared memory, for more rows than a block has registers for.
__global__ void __launch_bounds__(512) k_gj_panel_wide(const double* __restrict__ A, int n, int c0, GjWork w,
                                                       int* __restrict__ piv, int* __restrict__ info) {
    pdl_entry();
    extern __shared__ float smf[];
    float* Wp = smf;                                      // n x GJ_B working copy of the panel
    float* fac = Wp + (size_t)n * GJ_B;                   // n: column t before the pivot's elimination
    int* usedS = reinterpret_cast<int*>(fac + n);         // n
    __shared__ float prowv[GJ_B];
    __shared__ unsigned wv[32];
    __shared__ int wi[32];
    __shared__ int pS[GJ_B];
    const int ld = 2 * n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int q = threadIdx.x; q < n * GJ_B; q += blockDim.x) {
        const double v = A[(size_t)(q / GJ_B) * ld + c0 + (q % GJ_B)];
        Wp[q] = (float)v;
        w.Q0[q] = v;
    }
    for (int r = threadIdx.x; r < n; r += blockDim.x) usedS[r] = c0 == 0 ? 0 : w.used[r];
    __syncthreads();
    for (int t = 0; t < GJ_B; ++t) {
        // magnitudes order as their bits do; 0: no candidate, 1: a zero (or not a number), so that a row of the matrix is
        // chosen whatever its values
        unsigned best = 0u;
        int bi = n;
        auto take = [&](unsigned key, int row) {   // ties to the lower row
            if (key > best || (key == best && row < bi)) {
                best = key;
                bi = row;
            }
        };
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            if (usedS[r]) continue;
            const float m = fabsf(Wp[r * GJ_B + t]);
            take(m >= 0.0f ? __float_as_uint(m) + 1u : 1u, r);
        }
        for (int o = 16; o > 0; o >>= 1) take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, bi, o));
        if (lane == 0) {
            wv[wid] = best;
            wi[wid] = bi;
        }
        __syncthreads();
        if (wid == 0) {
            best = lane < nw ? wv[lane] : 0u;
            bi = lane < nw ? wi[lane] : n;
            for (int o = 16; o > 0; o >>= 1)
                take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, bi, o));
            if (lane == 0) {
                pS[t] = bi;
                usedS[bi] = 1;
            }
        }
        __syncthreads();
        const int p = pS[t];
        for (int r = threadIdx.x; r < n; r += blockDim.x) fac[r] = Wp[r * GJ_B + t];
        if (threadIdx.x < GJ_B) prowv[threadIdx.x] = Wp[p * GJ_B + threadIdx.x];
        __syncthreads();
        const float pv = prowv[t];
        const float ipv = pv != 0.0f ? 1.0f / pv : 0.0f;
        for (int q = threadIdx.x; q < n * GJ_B; q += blockDim.x) {   // candidate rows only
            const int r = q / GJ_B, tt = q % GJ_B;
            if (tt <= t || usedS[r]) continue;
            const float f = fac[r] * ipv;
            if (f != 0.0f) Wp[q] -= f * prowv[tt];
        }
        __syncthreads();
    }
    gj_pivot_block(c0, w, pS, piv, info);
    for (int r = threadIdx.x; r < n; r += blockDim.x) w.used[r] = usedS[r];
}

// W = A_PQ^{-1} A_P on columns c >= c0 + GJ_B, written to the work array and into the pivot rows;
// block (16 x 16): a slab of 16 columns, thread (x, y) = (column, pivot t)
__global__ void __launch_bounds__(GJ_B * 16) k_gj_w(double* __restrict__ A, int n, int c0, GjWork w) {
    pdl_entry();
    __shared__ double ap[GJ_B][16];
    __shared__ double g[GJ_B][GJ_B];
    const int ld = 2 * n;
    const int c = c0 + GJ_B + blockIdx.x * 16 + threadIdx.x;
    const int t = threadIdx.y;
    g[t][threadIdx.x] = w.G[t * GJ_B + threadIdx.x];
    ap[t][threadIdx.x] = c < ld ? A[(size_t)w.prow[t] * ld + c] : 0.0;
    __syncthreads();
    if (c >= ld) return;
    double acc = 0.0;
#pragma unroll
    for (int u = 0; u < GJ_B; ++u) acc += g[t][u] * ap[u][threadIdx.x];
    w.W[(size_t)t * ld + c] = acc;
    A[(size_t)w.prow[t] * ld + c] = acc;
}

// Other rows: A_r -= A_rQ W on columns right of the panel, and their panel entries 0;
// the pivot rows' panel entries become unit vectors.  Block (row r, slab of 128 columns from c0).
__global__ void __launch_bounds__(128) k_gj_rows(double* __restrict__ A, int n, int c0, GjWork w) {
    pdl_entry();
    __shared__ double m[GJ_B];
    __shared__ int piv_t;
    const int ld = 2 * n, r = blockIdx.x;
    const int c = c0 + blockIdx.y * 128 + threadIdx.x;
    if (threadIdx.x == 0) {
        int pt = -1;
        for (int t = 0; t < GJ_B; ++t)
            if (w.prow[t] == r) pt = t;
        piv_t = pt;
    }
    if (threadIdx.x < GJ_B) m[threadIdx.x] = w.Q0[(size_t)r * GJ_B + threadIdx.x];
    __syncthreads();
    if (c >= ld) return;
    const int pt = piv_t;
    if (c < c0 + GJ_B) {
        A[(size_t)r * ld + c] = (pt >= 0 && c - c0 == pt) ? 1.0 : 0.0;
        return;
    }
    if (pt >= 0) return;   // pivot rows: written by k_gj_w
    double acc = A[(size_t)r * ld + c];
#pragma unroll
    for (int u = 0; u < GJ_B; ++u) acc -= m[u] * w.W[(size_t)u * ld + c];
    A[(size_t)r * ld + c] = acc;
}

void launch_gauss_jordan(double* Aug, int n, int* info, int* piv, void* work, cudaStream_t s) {
    const GjWork w = gj_work(work, n);
    const size_t smem = sizeof(float) * ((size_t)n * GJ_B + n) + sizeof(int) * (size_t)n;
    const bool wide = n > GJ_MAXN;   // the box smoothers' largest subdomains
    if (wide) allow_smem(k_gj_panel_wide, smem);
    const int ld = 2 * n;
    for (int c0 = 0; c0 < n; c0 += GJ_B) {
        if (wide)
            launch_pdl(k_gj_panel_wide, 1, 512, smem, s, (const double*)Aug, n, c0, w, piv, info);
        else
            launch_pdl(k_gj_panel, 1, std::max(GJ_B * GJ_B, (n + 31) / 32 * 32), 0, s, (const double*)Aug, n, c0, w, piv,
                       info);
        const int R = ld - c0 - GJ_B;
        launch_pdl(k_gj_w, dim3((R + 15) / 16), dim3(16, GJ_B), 0, s, Aug, n, c0, w);
        launch_pdl(k_gj_rows, dim3(n, (ld - c0 + 127) / 128), dim3(128), 0, s, Aug, n, c0, w);
    }
}

// Pinv = (L0 + Z Z^T)^{-1} - Z Z^T, the pseudo-inverse of the symmetric L0 whose kernel is span Z;
// row r of the inverse is the right half of Aug's pivot row piv[r].
__global__ void k_extract_pinv(const double* __restrict__ Aug, const int* __restrict__ piv, int n, int N0, double rho,
                               double* __restrict__ P) {
    pdl_entry();
    const int r = blockIdx.y;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const int n0 = N0 * N0;
    double v = Aug[(int64_t)piv[r] * 2 * n + n + c];
    const int br = r / n0, bc = c / n0;
    if (br == bc && (rho == 0.0 || br == 2)) v -= 1.0 / (double)n0;
    P[(int64_t)r * n + c] = v;
}
void launch_extract_pinv(const double* Aug, const int* piv, int n, int N0, double rho, double* Pinv, cudaStream_t s) {
    launch_pdl(k_extract_pinv, dim3((n + 127) / 128, n), 128, 0, s, Aug, piv, n, N0, rho, Pinv);
}

// x = Pinv b, one warp per row, FP64 accumulation for both precisions
template <typename T>
__global__ void k_coarse_apply(const double* __restrict__ P, int n, const T* __restrict__ b, T* __restrict__ x) {
    pdl_entry();
    const int lane = threadIdx.x & 31;
    const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= n) return;
    const double* row = P + (int64_t)r * n;
    double s = 0.0;
    for (int c = lane; c < n; c += 32) s += row[c] * (double)b[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) x[r] = (T)s;
}
template <typename T>
void launch_coarse_apply(const double* Pinv, int n, const T* b, T* x, cudaStream_t s) {
    launch_pdl(k_coarse_apply<T>, (n + 7) / 8, 256, 0, s, Pinv, n, b, x);
}
template void launch_coarse_apply<float>(const double*, int, const float*, float*, cudaStream_t);
template void launch_coarse_apply<double>(const double*, int, const double*, double*, cudaStream_t);

// xo = x + omega P r, one warp per row, FP64 accumulation (x == nullptr: 0)
template <typename T>
__global__ void k_dense_correct(const double* __restrict__ P, int n, const T* __restrict__ r, const T* x, T omega,
                                T* xo) {
    pdl_entry();
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= n) return;
    const double* pr = P + (int64_t)row * n;
    double s = 0.0;
    for (int c = lane; c < n; c += 32) s += pr[c] * (double)r[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) xo[row] = (T)((x ? (double)x[row] : 0.0) + (double)omega * s);
}
template <typename T>
void launch_dense_correct(const double* P, int n, const T* r, const T* x, T omega, T* xo, cudaStream_t s) {
    launch_pdl(k_dense_correct<T>, (n + 7) / 8, 256, 0, s, P, n, r, x, omega, xo);
}
template void launch_dense_correct<float>(const double*, int, const float*, const float*, float, float*, cudaStream_t);
template void launch_dense_correct<double>(const double*, int, const double*, const double*, double, double*,
                                           cudaStream_t);

__global__ void k_check_finite(const double* __restrict__ x, int64_t n, int* __restrict__ flag) {
    pdl_entry();
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        if (!isfinite(x[k])) *flag = 1;
}
void launch_check_finite(const double* x, int64_t n, int* flag, cudaStream_t s) {
    if (n == 0) return;
    launch_pdl(k_check_finite, num_blocks_for(n), 256, 0, s, x, n, flag);
}


// ------------------------------------------------------------------------------------------
// Flexible GMRES cycle on the device (the same recurrence as the host loop: CGS2 Arnoldi,
// Givens rotations, stop at ||r|| <= tol, at the cycle length or at the iteration cap).
__global__ void k_fg_init(FgDev* st, double beta, int m, int max_it, double tol) {
    pdl_entry();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    st->j = 0;
    st->jn = 0;
    st->its = 0;
    st->k = 0;
    st->converged = 0;
    st->m = m;
    st->max_it = max_it;
    st->tol = tol;
    st->est = beta;
    st->beta = beta;
    st->inv_hn = 0.0;
    for (int i = 0; i <= FG_MAXM; ++i) st->g[i] = 0.0;
    st->g[0] = beta;
    st->hist[0] = beta;
}
void launch_fg_init(FgDev* st, double beta, int m, int max_it, double tol, cudaStream_t s) {
    launch_pdl(k_fg_init, 1, 1, 0, s, st, beta, m, max_it, tol);
}

// Start of Arnoldi step j = st->jn: for j > 0 the new basis vector V_j = w / h_{j,j-1} (w, the
// orthogonalised product of the previous step, and 1/h from its norm) is stored; V_j, cast to
// the V-cycle precision, becomes the finest level's right-hand side.
template <typename T>
__global__ void k_fg_prep(double* __restrict__ V, const double* __restrict__ w, int64_t n, FgDev* st,
                          T* __restrict__ dst) {
    pdl_entry();
    const int j = st->jn;
    double* v = V + (int64_t)j * n;
    const double inv = st->inv_hn;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double x;
        if (j == 0) {
            x = v[e];
        } else {
            x = w[e] * inv;
            v[e] = x;
        }
        dst[e] = (T)x;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->j = j;
}
template <typename T>
void launch_fg_prep(double* V, const double* w, int64_t n, FgDev* st, T* dst, cudaStream_t s) {
    launch_pdl(k_fg_prep<T>, num_blocks_for(n), 256, 0, s, V, w, n, st, dst);
}

template <typename T>
__global__ void k_fg_zstore(const T* __restrict__ src, double* __restrict__ Z, int64_t n, const FgDev* st,
                            double* __restrict__ zcur) {
    pdl_entry();
    double* z = Z + (int64_t)st->j * n;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const double v = (double)src[e];
        z[e] = v;
        zcur[e] = v;
    }
}
template <typename T>
void launch_fg_zstore(const T* src, double* Z, int64_t n, const FgDev* st, double* zcur, cudaStream_t s) {
    launch_pdl(k_fg_zstore<T>, num_blocks_for(n), 256, 0, s, src, Z, n, st, zcur);
}
template void launch_fg_prep<float>(double*, const double*, int64_t, FgDev*, float*, cudaStream_t);
template void launch_fg_prep<double>(double*, const double*, int64_t, FgDev*, double*, cudaStream_t);
template void launch_fg_zstore<float>(const float*, double*, int64_t, const FgDev*, double*, cudaStream_t);
template void launch_fg_zstore<double>(const double*, double*, int64_t, const FgDev*, double*, cudaStream_t);

// partials[i * S + s] = slice s of V_i . w for all i <= j.  The j + 1 vectors go in groups of up to MD_G, and
// a block takes one slice for one group: w is read once per group, a thread has MD_G + 1 independent 16-byte loads
// in flight, and the block's MD_G sums are transposed while they are added (9 FP64 additions a warp for the eight
// sums instead of 40, which a short slice would wait for: the FP64 pipe takes a warp's addition in 16 clocks).
// As many slices as MD_BLOCKS leaves a group, at least 1024 elements each.
// Large vectors take one wave of exactly three blocks an SM: each block reserves a third of the shared memory, so
// that those of the next kernel, which wait beside them, come one for one in their places; placed as registers
// allow, they crowd some SMs.  Small ones let the next kernel come only when their sums are done, for the same reason.
// The step's two products and two updates at 1024^2, 32 and 64 vectors: 1030 and 2020 us with a warp per vector
// and slice (ten warps an SM; products of 328 and 649 us), 820 and 1480 us so, where the FP64 pipe needs 700 and
// 1390; with the next kernel's blocks placed freely 1310 and 2560.
constexpr int GS_BLOCKS = 3 * 152;        // also k_gs_update_dev's
constexpr int GS_RESERVE = 72 * 1024;
constexpr int MD_BLOCKS = GS_BLOCKS, MD_SLICE = 1024, MD_G = 8;
__device__ __forceinline__ int md_groups(int k) { return (k + MD_G - 1) / MD_G; }
__device__ __forceinline__ int md_slices(int k, int64_t n) {
    return (int)min((int64_t)(MD_BLOCKS / md_groups(k)), (n + MD_SLICE - 1) / MD_SLICE);
}
static_assert(MD_BLOCKS * MD_G <= MD_MAXPART && MD_BLOCKS / ((FG_MAXM + MD_G - 1) / MD_G) >= 1, "partials, slices");
__global__ void __launch_bounds__(256) k_multidot_dev(const double* __restrict__ V, int64_t ld,
                                                      const double* __restrict__ w, int64_t n,
                                                      double* __restrict__ partials, const FgDev* st, bool wave) {
    pdl_wait();
    if (wave) pdl_launch();
    __shared__ double ws[8][MD_G];
    const int k = st->j + 1, groups = md_groups(k), S = md_slices(k, n);
    if ((int)blockIdx.x >= groups * S) return;
    const int g = blockIdx.x / S, sl = blockIdx.x - g * S, per = (k + groups - 1) / groups;
    const int i0 = g * per, cnt = min(per, k - i0), lane = threadIdx.x & 31;
    const int64_t n2 = n / 2, len = (n2 + S - 1) / S, e1 = min((sl + 1) * len, n2);   // n = 3 N^2 is even
    const double2* w2 = reinterpret_cast<const double2*>(w);
    const double2* v2 = reinterpret_cast<const double2*>(V + (int64_t)i0 * ld);
    double acc[MD_G] = {};
    auto dots = [&](auto m) {   // m vectors, U elements at a time: eight loads or so in flight
        constexpr int M = decltype(m)::value, U = M <= 4 ? MD_G / M : 1;
        int64_t e = sl * len + threadIdx.x;
        for (; e + 256 * (U - 1) < e1; e += 256 * U) {
            double2 x[U], v[U][M];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = w2[e + 256 * u];
#pragma unroll
                for (int q = 0; q < M; ++q) v[u][q] = v2[q * (ld / 2) + e + 256 * u];
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < M; ++q) acc[q] = fma(v[u][q].y, x[u].y, fma(v[u][q].x, x[u].x, acc[q]));
        }
        for (; e < e1; e += 256) {
            const double2 x = w2[e];
#pragma unroll
            for (int q = 0; q < M; ++q) {
                const double2 v = v2[q * (ld / 2) + e];
                acc[q] = fma(v.y, x.y, fma(v.x, x.x, acc[q]));
            }
        }
    };
    switch (cnt) {
        case 1: dots(std::integral_constant<int, 1>()); break;
        case 2: dots(std::integral_constant<int, 2>()); break;
        case 3: dots(std::integral_constant<int, 3>()); break;
        case 4: dots(std::integral_constant<int, 4>()); break;
        case 5: dots(std::integral_constant<int, 5>()); break;
        case 6: dots(std::integral_constant<int, 6>()); break;
        case 7: dots(std::integral_constant<int, 7>()); break;
        default: dots(std::integral_constant<int, MD_G>()); break;
    }
    if (!wave) pdl_launch();
    // each step halves the values a lane carries and doubles the lanes they are sums of
#pragma unroll
    for (int o = 16, h = MD_G / 2; o >= 4; o >>= 1, h >>= 1) {
        const bool hi = lane & o;
#pragma unroll
        for (int q = 0; q < MD_G / 2; ++q)
            if (q < h) {
                const double give = hi ? acc[q] : acc[q + h], keep = hi ? acc[q + h] : acc[q];
                acc[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 3) == 0) ws[threadIdx.x >> 5][(lane & 16 ? 4 : 0) + (lane & 8 ? 2 : 0) + (lane & 4 ? 1 : 0)] = acc[0];
    __syncthreads();
    if ((int)threadIdx.x < cnt) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) s += ws[q][threadIdx.x];
        partials[(int64_t)(i0 + threadIdx.x) * S + sl] = s;
    }
}
void launch_multidot_dev(const double* V, int64_t ld, const double* w, int64_t n, double* partials,
                         const FgDev* st, cudaStream_t s) {
    const int64_t nb = (FG_MAXM + MD_G - 1) / MD_G * ((n + MD_SLICE - 1) / MD_SLICE);
    const bool wave = n >= (int64_t)MD_SLICE * MD_BLOCKS;
    if (wave) allow_smem(k_multidot_dev, GS_RESERVE);
    launch_pdl(k_multidot_dev, (int)std::min<int64_t>(MD_BLOCKS, nb), 256, wave ? GS_RESERVE : 0, s, V, ld, w, n, partials,
               st, wave);
}
// y += sum_{i < k} coef[i] V_i with k = st->k
__global__ void k_multi_axpy_dev(const double* __restrict__ V, int64_t ld, const double* __restrict__ coef,
                                 double* __restrict__ y, int64_t n, const FgDev* st) {
    pdl_entry();
    __shared__ double c[FG_MAXM + 1];
    const int k = st->k;
    for (int t = threadIdx.x; t < k; t += blockDim.x) c[t] = coef[t];
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double acc = y[e];
        for (int i = 0; i < k; ++i) acc += c[i] * V[(int64_t)i * ld + e];
        y[e] = acc;
    }
}
void launch_multi_axpy_dev(const double* V, int64_t ld, const double* coef, double* y, int64_t n, const FgDev* st,
                           cudaStream_t s) {
    launch_pdl(k_multi_axpy_dev, num_blocks_for(n), 256, 0, s, V, ld, coef, y, n, st);
}

// A Gram-Schmidt update, y -= sum_{i <= j} h_i V_i, with h_i summed here from the slices' partials of
// k_multidot_dev (block 0 leaves them in `h`); NORM: and the block partials of ||y||^2.
// Every block sums the partials for itself, as many lanes per vector as the block has (up to 20 FP64
// instructions a warp): cheaper than a launch for the sums between two launches that wait for each other.  At most
// three blocks per SM repeat it (GS_BLOCKS).
// With the norm's sum in k_fg_arnoldi three of the 13 launches outside the V-cycle go.
template <bool NORM>
__global__ void __launch_bounds__(256) k_gs_update_dev(const double* __restrict__ V, int64_t ld,
                                                       const double* __restrict__ dots, double* __restrict__ h,
                                                       double* __restrict__ y, int64_t n, const FgDev* st,
                                                       double* __restrict__ partials, bool wave) {
    pdl_wait();
    if (wave) pdl_launch();
    __shared__ double c[FG_MAXM + 1];
    const int k = st->j + 1, S = md_slices(k, n);
    int lg = 5;
    while (lg > 0 && (k << lg) > (int)blockDim.x) --lg;   // k <= FG_MAXM vectors, 2^lg lanes each
    const int g = 1 << lg, i = threadIdx.x >> lg, sub = threadIdx.x & (g - 1);
    double s = 0.0;
    if (i < k) {
#pragma unroll 4
        for (int b = sub; b < S; b += g) s += dots[(int64_t)i * S + b];
    }
    for (int o = 1; o < g; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (i < k && sub == 0) {
        c[i] = -s;
        if (blockIdx.x == 0) h[i] = s;
    }
    __syncthreads();
    double ss = 0.0;
    double2* y2 = reinterpret_cast<double2*>(y);   // n = 3 N^2 is even
    const double2* v2 = reinterpret_cast<const double2*>(V);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n / 2; e += (int64_t)gridDim.x * blockDim.x) {
        double2 acc = y2[e];
#pragma unroll 8
        for (int q = 0; q < k; ++q) {
            const double2 v = v2[q * (ld / 2) + e];
            acc.x = fma(c[q], v.x, acc.x);
            acc.y = fma(c[q], v.y, acc.y);
        }
        y2[e] = acc;
        if (NORM) ss += acc.x * acc.x + acc.y * acc.y;
    }
    if (!wave) pdl_launch();
    if (!NORM) return;
    ss = block_sum(ss);
    if (threadIdx.x == 0) partials[blockIdx.x] = ss;
}
int launch_gs_update_dev(const double* V, int64_t ld, const double* dots, double* h, double* y, int64_t n,
                         const FgDev* st, double* partials, cudaStream_t s) {
    const int nb = std::min(num_blocks_for(n / 2), GS_BLOCKS);
    const bool wave = n >= (int64_t)MD_SLICE * MD_BLOCKS;   // as k_multidot_dev
    auto kern = partials ? k_gs_update_dev<true> : k_gs_update_dev<false>;
    if (wave) allow_smem(kern, GS_RESERVE);
    launch_pdl(kern, nb, 256, wave ? GS_RESERVE : 0, s, V, ld, dots, h, y, n, st, partials, wave);
    return nb;
}

// One block: ||w||^2 from its nb block partials, then (one thread) Hessenberg column j from the two
// Gram-Schmidt passes, previous and new Givens rotation, residual estimate, and the loop decision (always
// terminates: the iteration cap and the cycle length bound it, and a non-finite estimate or a zero new norm stops
// it).  The rotations are a serial chain; their operands are fetched by the whole block beforehand.
__global__ void __launch_bounds__(128) k_fg_arnoldi(FgDev* st, const double* __restrict__ h1,
                                                    const double* __restrict__ h2, const double* __restrict__ nrm,
                                                    int nb, cudaGraphConditionalHandle handle) {
    pdl_entry();
    __shared__ double hs[FG_MAXM + 1], cs[FG_MAXM], sn[FG_MAXM];
    const int j = st->j, t = threadIdx.x;
    double nn = 0.0;
    for (int b = t; b < nb; b += 128) nn += nrm[b];
    for (int i = t; i <= j; i += 128) hs[i] = h1[i] + h2[i];
    for (int i = t; i < j; i += 128) {
        cs[i] = st->cs[i];
        sn[i] = st->sn[i];
    }
    nn = block_sum(nn);   // also the barrier for the copies above
    if (t != 0) return;
    double* Hj = st->H + (size_t)j * (FG_MAXM + 1);
    const double hn = sqrt(nn);
    double a = hs[0];
    for (int i = 0; i < j; ++i) {
        const double b = hs[i + 1];
        Hj[i] = cs[i] * a + sn[i] * b;
        a = -sn[i] * a + cs[i] * b;
    }
    const double d = hypot(a, hn);
    st->cs[j] = a / d;
    st->sn[j] = hn / d;
    Hj[j] = d;
    Hj[j + 1] = 0.0;
    st->g[j + 1] = -st->sn[j] * st->g[j];
    st->g[j] = st->cs[j] * st->g[j];
    const double est = fabs(st->g[j + 1]);
    st->its += 1;
    st->est = est;
    st->hist[j + 1] = est;
    const bool conv = est <= st->tol;
    const bool stop = conv || !(hn > 0.0) || !isfinite(est) || !isfinite(d) || st->its >= st->max_it || j + 1 >= st->m;
    st->inv_hn = hn > 0.0 ? 1.0 / hn : 0.0;
    st->jn = j + 1;
    if (stop) {
        st->k = j + 1;
        st->converged = (conv || hn == 0.0) ? 1 : 0;   // a zero new direction: the solution is exact
    }
    cudaGraphSetConditional(handle, stop ? 0u : 1u);
}
void launch_fg_arnoldi(FgDev* st, const double* h1, const double* h2, const double* nrm, int nb,
                       cudaGraphConditionalHandle handle, cudaStream_t s) {
    launch_pdl(k_fg_arnoldi, 1, 128, 0, s, st, h1, h2, nrm, nb, handle);
}

// y = H^{-1} g on the k x k upper triangle, column by column: thread q carries entry q of the right-hand side and
// has its entry of the next column at hand.  (One thread walking the rows: 23 us for 19 columns.)
__global__ void __launch_bounds__(128) k_fg_backsolve(FgDev* st) {
    pdl_entry();
    __shared__ double ys[2];
    const int k = st->k, q = threadIdx.x;
    double acc = q < k ? st->g[q] : 0.0;
    double h = q < k ? st->H[(size_t)(k - 1) * (FG_MAXM + 1) + q] : 0.0;
    for (int i = k - 1; i >= 0; --i) {
        const double next = i > 0 && q < i ? st->H[(size_t)(i - 1) * (FG_MAXM + 1) + q] : 0.0;
        if (q == i) ys[i & 1] = st->y[i] = acc / h;
        __syncthreads();
        if (q < i) acc -= h * ys[i & 1];
        h = next;
    }
}
void launch_fg_backsolve(FgDev* st, cudaStream_t s) { launch_pdl(k_fg_backsolve, 1, 128, 0, s, st); }

}  // namespace sib
