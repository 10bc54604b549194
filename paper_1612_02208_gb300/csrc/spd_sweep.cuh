// In-place inversion of a symmetric positive definite matrix by one thread block (FP64, shared memory).
#pragma once

namespace sib {

// start of row i of a packed lower triangle
__device__ __forceinline__ int tri(int i) { return i * (i + 1) / 2; }

// 1 / x by Newton's iteration r <- r + r (1 - x r) from the FP32 quotient (23 bits, then 46, then rounding): four
// dependent FP64 operations, where the division takes an order more and stands in every step's critical path
__device__ __forceinline__ double sweep_recip(double x) {
    const float f = (float)x;
    if (!(f > 1e-30f && f < 1e30f)) return 1.0 / x;
    double r = (double)(1.0f / f);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// A (lower triangle, packed rows, n x n) <- -A^{-1} by symmetric sweeps: at step k, with d = 1 / A_kk and
// v = column k, A_ij -= v_i v_j d for i, j != k, A_ik = v_i d, A_kk = -d.  No pivoting: a pivot that is not
// positive sets bit 1 of *info and voids the result.  v, vd: n values each.  Rows i and n - 1 - i are swept as
// one row of n + 1 entries, so that the warps' lanes stay full.  Bound by the FP64 pipe (n^2 / 2 multiply-adds a
// step, two per clock) and, for small n, by a step's latency.  The next pivot's reciprocal is formed by the one
// thread that updates it, beside the other warps' updates: a division costs the FP64 pipe as much as forty
// multiply-adds.
__device__ inline void spd_sweep(double* A, double* v, double* vd, int n, int* info) {
    __shared__ double rcp[2];   // 1 / A_kk of this step and of the next
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, pairs = (n + 1) / 2;
    if (threadIdx.x == 0) {
        if (!(A[0] > 0.0)) atomicOr(info, 2);
        rcp[0] = sweep_recip(A[0]);
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        const double d = rcp[k & 1];
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const double x = i >= k ? A[tri(i) + k] : A[tri(k) + i];
            v[i] = x;
            vd[i] = x * d;
        }
        __syncthreads();
        for (int p = wid; p < pairs; p += nw) {
            const int i1 = p, i2 = n - 1 - p;             // i1 <= i2; equal in the middle of an odd n
            const int len = i1 == i2 ? i1 + 1 : n + 1;
            for (int t = lane; t < len; t += 32) {
                const int i = t <= i1 ? i1 : i2, j = t <= i1 ? t : t - i1 - 1;
                double* a = A + tri(i) + j;
                double x = *a - v[i] * vd[j];
                if (i == k || j == k) x = i == j ? -d : vd[i == k ? j : i];
                *a = x;
                if (i == k + 1 && j == i) {
                    if (!(x > 0.0)) atomicOr(info, 2);
                    rcp[(k + 1) & 1] = sweep_recip(x);
                }
            }
        }
        __syncthreads();
    }
}

// The same inversion with the triangle in registers, for n small enough that a step's latency counts: thread t
// owns the entries t, t + T, ... of the triangle (T = blockDim.x, at most E each), a step's column passes through
// shared memory, and the E updates of a thread are independent.  get(i, j) gives an entry (i >= j); put(i, j, x)
// receives that of A^{-1}.  col: 2 n values of shared memory.  64 x 64 in one block of 256: 140 us.
template <int E, typename Get, typename Put>
__device__ __forceinline__ void spd_sweep_regs(int n, double* col, int* info, Get get, Put put) {
    __shared__ double rcp[2];
    double a[E];
    int ij[E];   // i << 16 | j; -1: none
    double* v = col;
    double* vd = col + n;
    const int total = tri(n), T = blockDim.x;
#pragma unroll
    for (int u = 0; u < E; ++u) {
        const int e = threadIdx.x + u * T;
        int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        while (tri(i + 1) <= e) ++i;
        while (tri(i) > e) --i;
        const int j = e - tri(i);
        const bool own = e < total;
        ij[u] = own ? (i << 16 | j) : -1;
        a[u] = own ? get(i, j) : 0.0;
        if (own && i == 0) {
            if (!(a[u] > 0.0)) atomicOr(info, 2);
            rcp[0] = sweep_recip(a[u]);
        }
    }
    for (int k = 0; k < n; ++k) {
#pragma unroll
        for (int u = 0; u < E; ++u) {   // column k to shared memory
            if (ij[u] < 0) continue;
            const int i = ij[u] >> 16, j = ij[u] & 0xffff;
            if (j == k) v[i] = a[u];
            else if (i == k) v[j] = a[u];
        }
        __syncthreads();
        const double d = rcp[k & 1];
        for (int i = threadIdx.x; i < n; i += T) vd[i] = v[i] * d;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < E; ++u) {
            if (ij[u] < 0) continue;
            const int i = ij[u] >> 16, j = ij[u] & 0xffff;
            double x = a[u] - v[i] * vd[j];
            if (i == k || j == k) x = i == j ? -d : vd[i == k ? j : i];
            a[u] = x;
            if (i == k + 1 && j == i) {
                if (!(x > 0.0)) atomicOr(info, 2);
                rcp[(k + 1) & 1] = sweep_recip(x);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < E; ++u)
        if (ij[u] >= 0) put(ij[u] >> 16, ij[u] & 0xffff, -a[u]);
}

}  // namespace sib
