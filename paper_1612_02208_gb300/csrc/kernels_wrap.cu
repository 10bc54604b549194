// Kernels of the Krylov-wrapped smoothing step (Sec. 3.3): a pre- or post-smoothing stage of nu
// sweeps becomes nu iterations of flexible GMRES on the level's residual equation, each
// preconditioned by one undamped sweep of the basic smoother.  The level vectors are in the
// V-cycle's precision T.  Inner products are formed per thread over 16-byte vectors of T (products
// of one vector summed in T), accumulated in FP64, reduced per block, and the block partials are
// summed by one block per product in block order: a fixed order, so results do not depend on
// timing.  The classical Gram-Schmidt update of each pass is fused with the inner products that
// follow it (the second pass's coefficients, or the norm).  The small Hessenberg least-squares
// problem is solved in FP64 by one thread.
#include <cooperative_groups.h>

#include "sib_internal.h"

namespace cg = cooperative_groups;

namespace sib {

namespace {

template <typename T>
struct WVec;
template <>
struct WVec<float> {
    using type = float4;
    static constexpr int n = 4;
};
template <>
struct WVec<double> {
    using type = double2;
    static constexpr int n = 2;
};
template <typename T>
__device__ __forceinline__ T wv(const typename WVec<T>::type& v, int c);
template <>
__device__ __forceinline__ float wv<float>(const float4& v, int c) {
    return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w;
}
template <>
__device__ __forceinline__ double wv<double>(const double2& v, int c) {
    return c == 0 ? v.x : v.y;
}
template <typename T>
__device__ __forceinline__ void wset(typename WVec<T>::type& v, int c, T x);
template <>
__device__ __forceinline__ void wset<float>(float4& v, int c, float x) {
    if (c == 0) v.x = x;
    else if (c == 1) v.y = x;
    else if (c == 2) v.z = x;
    else v.w = x;
}
template <>
__device__ __forceinline__ void wset<double>(double2& v, int c, double x) {
    if (c == 0) v.x = x;
    else v.y = x;
}

constexpr int WT = 256;           // threads per block
constexpr int WW = WT / 32;       // warps per block

// Block sums of acc[i], i < cnt, written to partials[i * gridDim.x + blockIdx.x]: warp shuffles,
// then the warps' values in warp order.
template <int KC>
__device__ __forceinline__ void block_partials(double (&acc)[KC], int cnt, double* __restrict__ partials) {
    __shared__ double ws[KC][WW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < KC; ++i) {
        if (i < cnt) {
            double v = acc[i];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) ws[i][wid] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < cnt) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < WW; ++q) s += ws[threadIdx.x][q];
        partials[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = s;
    }
}

// partials of V_i . w, i < cnt (cnt <= KC <= WRAP_MAXK + 1)
template <typename T, int KC>
__global__ void __launch_bounds__(WT) k_wdots(const T* __restrict__ V, int64_t ld, int cnt, const T* __restrict__ w,
                                              int64_t n, double* __restrict__ partials) {
    using VT = typename WVec<T>::type;
    constexpr int VN = WVec<T>::n;
    pdl_entry();
    double acc[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) acc[i] = 0.0;
    const int64_t nv = n / VN;
    for (int64_t e = blockIdx.x * (int64_t)WT + threadIdx.x; e < nv; e += (int64_t)gridDim.x * WT) {
        const VT we = reinterpret_cast<const VT*>(w)[e];
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            if (i < cnt) {
                const VT vi = reinterpret_cast<const VT*>(V + (int64_t)i * ld)[e];
                T s = T(0);
#pragma unroll
                for (int c = 0; c < VN; ++c) s = fma(wv<T>(vi, c), wv<T>(we, c), s);
                acc[i] += (double)s;
            }
        }
    }
    for (int64_t e = nv * VN + blockIdx.x * (int64_t)WT + threadIdx.x; e < n; e += (int64_t)gridDim.x * WT)
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < cnt) acc[i] += (double)V[(int64_t)i * ld + e] * (double)w[e];
    block_partials(acc, cnt, partials);
}

// wout = win - sum_{i < cnt} coef[i] V_i, and then (MODE 1) partials of V_i . wout, i < cnt, or
// (MODE 2) the partial of wout . wout; cnt <= KC
template <typename T, int MODE, int KC>
__global__ void __launch_bounds__(WT) k_wgs(const T* __restrict__ V, int64_t ld, int cnt,
                                            const double* __restrict__ coef, const T* win, T* wout, int64_t n,
                                            double* __restrict__ partials) {
    using VT = typename WVec<T>::type;
    constexpr int VN = WVec<T>::n;
    pdl_entry();
    T cf[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) cf[i] = i < cnt ? (T)coef[i] : T(0);
    double acc[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) acc[i] = 0.0;
    const int64_t nv = n / VN;
    for (int64_t e = blockIdx.x * (int64_t)WT + threadIdx.x; e < nv; e += (int64_t)gridDim.x * WT) {
        VT y = reinterpret_cast<const VT*>(win)[e];
        VT vi[KC];
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < cnt) vi[i] = reinterpret_cast<const VT*>(V + (int64_t)i * ld)[e];
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < cnt)
#pragma unroll
                for (int c = 0; c < VN; ++c) wset<T>(y, c, fma(-cf[i], wv<T>(vi[i], c), wv<T>(y, c)));
        reinterpret_cast<VT*>(wout)[e] = y;
        if (MODE == 1) {
#pragma unroll
            for (int i = 0; i < KC; ++i) {
                if (i < cnt) {
                    T s = T(0);
#pragma unroll
                    for (int c = 0; c < VN; ++c) s = fma(wv<T>(vi[i], c), wv<T>(y, c), s);
                    acc[i] += (double)s;
                }
            }
        } else if (MODE == 2) {
            T s = T(0);
#pragma unroll
            for (int c = 0; c < VN; ++c) s = fma(wv<T>(y, c), wv<T>(y, c), s);
            acc[0] += (double)s;
        }
    }
    for (int64_t e = nv * VN + blockIdx.x * (int64_t)WT + threadIdx.x; e < n; e += (int64_t)gridDim.x * WT) {
        T y = win[e];
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < cnt) y = fma(-cf[i], V[(int64_t)i * ld + e], y);
        wout[e] = y;
        if (MODE == 1) {
#pragma unroll
            for (int i = 0; i < KC; ++i)
                if (i < cnt) acc[i] += (double)V[(int64_t)i * ld + e] * (double)y;
        } else if (MODE == 2) {
            acc[0] += (double)y * (double)y;
        }
    }
    if (MODE == 1) block_partials(acc, cnt, partials);
    else if (MODE == 2) block_partials(acc, 1, partials);
}

// out[i] = sum over the nblk block partials of product i, in block order; one block per product
__global__ void __launch_bounds__(WT) k_wreduce(const double* __restrict__ partials, int nblk, double* __restrict__ out) {
    pdl_entry();
    __shared__ double ws[WW];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += WT) s += partials[(int64_t)blockIdx.x * nblk + b];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ws[wid] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < WW; ++q) t += ws[q];
        out[blockIdx.x] = t;
    }
}

// yout = yin + sign * sum_{i < cnt} coef[i] V_i   (yin == nullptr: 0); cnt <= KC
template <typename T, int KC>
__global__ void __launch_bounds__(WT) k_wmaxpy(const T* __restrict__ V, int64_t ld, int cnt,
                                               const double* __restrict__ coef, double sign, const T* yin, T* yout,
                                               int64_t n) {
    using VT = typename WVec<T>::type;
    constexpr int VN = WVec<T>::n;
    pdl_entry();
    T cf[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) cf[i] = i < cnt ? (T)(sign * coef[i]) : T(0);
    const int64_t nv = n / VN;
    for (int64_t e = blockIdx.x * (int64_t)WT + threadIdx.x; e < nv; e += (int64_t)gridDim.x * WT) {
        VT y;
        if (yin) {
            y = reinterpret_cast<const VT*>(yin)[e];
        } else {
#pragma unroll
            for (int c = 0; c < VN; ++c) wset<T>(y, c, T(0));
        }
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            if (i < cnt) {
                const VT vi = reinterpret_cast<const VT*>(V + (int64_t)i * ld)[e];
#pragma unroll
                for (int c = 0; c < VN; ++c) wset<T>(y, c, fma(cf[i], wv<T>(vi, c), wv<T>(y, c)));
            }
        }
        reinterpret_cast<VT*>(yout)[e] = y;
    }
    for (int64_t e = nv * VN + blockIdx.x * (int64_t)WT + threadIdx.x; e < n; e += (int64_t)gridDim.x * WT) {
        T y = yin ? yin[e] : T(0);
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < cnt) y = fma(cf[i], V[(int64_t)i * ld + e], y);
        yout[e] = y;
    }
}

// v = w / sqrt(nrm2[0]), or 0 when the norm is zero (a vanished Arnoldi vector); the scale is
// formed once in FP64 and applied in T
template <typename T>
__global__ void __launch_bounds__(WT) k_wscale(const T* __restrict__ w, const double* __restrict__ nrm2,
                                               T* __restrict__ v, int64_t n) {
    using VT = typename WVec<T>::type;
    constexpr int VN = WVec<T>::n;
    pdl_entry();
    const T s = (T)(nrm2[0] > 0.0 ? 1.0 / sqrt(nrm2[0]) : 0.0);
    const int64_t nv = n / VN;
    for (int64_t e = blockIdx.x * (int64_t)WT + threadIdx.x; e < nv; e += (int64_t)gridDim.x * WT) {
        VT y = reinterpret_cast<const VT*>(w)[e];
#pragma unroll
        for (int c = 0; c < VN; ++c) wset<T>(y, c, wv<T>(y, c) * s);
        reinterpret_cast<VT*>(v)[e] = y;
    }
    for (int64_t e = nv * VN + blockIdx.x * (int64_t)WT + threadIdx.x; e < n; e += (int64_t)gridDim.x * WT)
        v[e] = w[e] * s;
}

// y = argmin || beta e1 - H y || for the (m + 1) x m Hessenberg matrix of the step (Givens
// rotations, back substitution).  H(i, j) = hA[j][i] + hB[j][i] for i <= j (the two Gram-Schmidt
// passes), H(j + 1, j) = sqrt(nr[j]); m stops at the first vanished subdiagonal entry.  y[m..k) = 0.
// One thread.  The loops run to a compile-time bound KM >= k, predicated on k and m, so that H stays in
// registers and every entry is loaded at once.
template <int KM>
__device__ void wlsq_solve_t(const double* __restrict__ hA, const double* __restrict__ hB,
                             const double* __restrict__ nr, const double* __restrict__ beta2, int k,
                             double* __restrict__ y) {
    double H[KM + 1][KM];
    double g[KM + 1], yv[KM];
#pragma unroll
    for (int j = 0; j < KM; ++j) {
        yv[j] = 0.0;
#pragma unroll
        for (int i = 0; i <= KM; ++i) H[i][j] = 0.0;
        if (j < k) {
#pragma unroll
            for (int i = 0; i <= j; ++i) H[i][j] = hA[j * (WRAP_MAXK + 1) + i] + hB[j * (WRAP_MAXK + 1) + i];
            H[j + 1][j] = sqrt(nr[j]);
        }
    }
    const double beta = sqrt(beta2[0]);
    int m = k;
#pragma unroll
    for (int j = KM - 1; j >= 0; --j)
        if (j < k && !(H[j + 1][j] > 0.0)) m = j + 1;
    if (beta > 0.0) {
#pragma unroll
        for (int i = 0; i <= KM; ++i) g[i] = i == 0 ? beta : 0.0;
#pragma unroll
        for (int j = 0; j < KM; ++j) {   // rotate H(j, j), H(j + 1, j) to (r, 0)
            if (j < m) {
                const double a = H[j][j], b = H[j + 1][j];
                const double d = hypot(a, b);
                const double cs = d > 0.0 ? a / d : 1.0, sn = d > 0.0 ? b / d : 0.0;
#pragma unroll
                for (int q = j; q < KM; ++q) {
                    if (q < m) {
                        const double u = H[j][q], v = H[j + 1][q];
                        H[j][q] = cs * u + sn * v;
                        H[j + 1][q] = -sn * u + cs * v;
                    }
                }
                const double gu = g[j], gv = g[j + 1];
                g[j] = cs * gu + sn * gv;
                g[j + 1] = -sn * gu + cs * gv;
            }
        }
#pragma unroll
        for (int i = KM - 1; i >= 0; --i) {
            if (i < m) {
                double acc = g[i];
#pragma unroll
                for (int q = i + 1; q < KM; ++q)
                    if (q < m) acc -= H[i][q] * yv[q];
                yv[i] = H[i][i] != 0.0 ? acc / H[i][i] : 0.0;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < KM; ++j)
        if (j < k) y[j] = yv[j];
}
__device__ void wlsq_solve(const double* __restrict__ hA, const double* __restrict__ hB,
                           const double* __restrict__ nr, const double* __restrict__ beta2, int k,
                           double* __restrict__ y) {
    if (k <= 2)
        wlsq_solve_t<2>(hA, hB, nr, beta2, k, y);
    else if (k <= 4)
        wlsq_solve_t<4>(hA, hB, nr, beta2, k, y);
    else
        wlsq_solve_t<WRAP_MAXK>(hA, hB, nr, beta2, k, y);
}

// The stage's last norm, out = sum of the nblk partials (as k_wreduce with one product), then the
// stage's least-squares solve into y by the thread that wrote it
__global__ void __launch_bounds__(WT) k_wreduce_lsq(const double* __restrict__ partials, int nblk, double* out,
                                                    const double* __restrict__ hA, const double* __restrict__ hB,
                                                    const double* nrAll, const double* __restrict__ beta2, int k,
                                                    double* __restrict__ y) {
    pdl_entry();
    __shared__ double ws[WW];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += WT) s += partials[b];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ws[wid] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < WW; ++q) t += ws[q];
        out[0] = t;
        wlsq_solve(hA, hB, nrAll, beta2, k, y);
    }
}

// Levels of up to wrap_cluster_max values: a whole orthogonalisation step in one cluster of eight blocks.  w stays
// in registers (E vectors of 16 bytes a thread); the two Gram-Schmidt passes h = V^T w, w -= V h and the norm each
// end with every block's sums in every block's shared memory and one cluster barrier; then Vnext = w / |w|
// (Vnext != nullptr) and, on the stage's last step (lsq_k > 0), its least-squares solve into y.  cnt = 0: the norm
// alone, of the stage's residual.  Bound by latency: seven launches of 2.5 us each did a step (three on levels
// of up to 32^2, in one block).  Solves with wrapped Schur-complement sweeps, disk, FP32: 32^2 2.35 -> 2.27 ms,
// 128^2 6.49 -> 6.20, 256^2 11.75 -> 11.38.  FP64 levels take it up to 32^2 (3.67 -> 3.35): above, eight SMs' FP64 pipes
// are slower than the launches (128^2: 10.6 against 11.0 ms with it).
constexpr int WC = 8;
template <typename T, int KC, int E>
__global__ void __launch_bounds__(WT) k_wstep_cluster(const T* __restrict__ V, int64_t n, int cnt, const T* __restrict__ w,
                                                      double* hA, double* hB, double* nr, T* __restrict__ Vnext,
                                                      int lsq_k, const double* hAll, const double* hBll,
                                                      const double* nrAll, const double* beta2, double* y) {
    using VT = typename WVec<T>::type;
    constexpr int VN = WVec<T>::n;
    __shared__ double part[3][WC][KC], ws[KC][WW], sum[KC];
    __shared__ T scale;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nv = (int)(n / VN), e0 = rank * WT + tid;   // n = 3 N^2 is a multiple of VN
    pdl_entry();
    cl.sync();   // every block has started: its shared memory may be written
    VT x[E];
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int e = e0 + q * WC * WT;
        if (e < nv) {
            x[q] = reinterpret_cast<const VT*>(w)[e];
        } else {
#pragma unroll
            for (int c = 0; c < VN; ++c) wset<T>(x[q], c, T(0));
        }
    }
    // sums over the cluster of acc[i], i < m, into sum[] (every block, in rank order)
    auto reduce = [&](double (&acc)[KC], int m, int slot) {
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < m) {
                double v = acc[i];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) ws[i][wid] = v;
            }
        __syncthreads();
        if (tid < m) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < WW; ++q) v += ws[tid][q];
            for (int r = 0; r < WC; ++r) *cl.map_shared_rank(&part[slot][rank][tid], r) = v;
        }
        cl.sync();
        if (tid < m) {
            double v = 0.0;
#pragma unroll
            for (int r = 0; r < WC; ++r) v += part[slot][r][tid];
            sum[tid] = v;
        }
        __syncthreads();
    };
    if (cnt > 0) {
        for (int pass = 0; pass < 2; ++pass) {
            double acc[KC] = {};
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int e = e0 + q * WC * WT;
#pragma unroll
                for (int i = 0; i < KC; ++i)
                    if (i < cnt && e < nv) {
                        const VT v = reinterpret_cast<const VT*>(V + (int64_t)i * n)[e];
                        T s = T(0);
#pragma unroll
                        for (int c = 0; c < VN; ++c) s = fma(wv<T>(v, c), wv<T>(x[q], c), s);
                        acc[i] += (double)s;
                    }
            }
            reduce(acc, cnt, pass);
            if (rank == 0 && tid < cnt) (pass == 0 ? hA : hB)[tid] = sum[tid];
            T cf[KC];
#pragma unroll
            for (int i = 0; i < KC; ++i) cf[i] = i < cnt ? (T)sum[i] : T(0);
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int e = e0 + q * WC * WT;
#pragma unroll
                for (int i = 0; i < KC; ++i)
                    if (i < cnt && e < nv) {
                        const VT v = reinterpret_cast<const VT*>(V + (int64_t)i * n)[e];
#pragma unroll
                        for (int c = 0; c < VN; ++c) wset<T>(x[q], c, fma(-cf[i], wv<T>(v, c), wv<T>(x[q], c)));
                    }
            }
            __syncthreads();   // sum[] is read
        }
    }
    double acc[KC] = {};
#pragma unroll
    for (int q = 0; q < E; ++q) {
        T s = T(0);
#pragma unroll
        for (int c = 0; c < VN; ++c) s = fma(wv<T>(x[q], c), wv<T>(x[q], c), s);
        acc[0] += (double)s;
    }
    reduce(acc, 1, 2);
    if (rank == 0 && tid == 0) {
        nr[0] = sum[0];
        if (lsq_k > 0) wlsq_solve(hAll, hBll, nrAll, beta2, lsq_k, y);
    }
    if (!Vnext) return;
    if (tid == 0) scale = (T)(sum[0] > 0.0 ? 1.0 / sqrt(sum[0]) : 0.0);
    __syncthreads();
    const T sc = scale;
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int e = e0 + q * WC * WT;
        if (e < nv) {
#pragma unroll
            for (int c = 0; c < VN; ++c) wset<T>(x[q], c, wv<T>(x[q], c) * sc);
            reinterpret_cast<VT*>(Vnext)[e] = x[q];
        }
    }
}

}  // namespace

// blocks of the inner-product and update kernels for n values: one 16-byte vector per thread and
// pass, at most WRAP_BLK blocks (8 per SM)
template <typename T>
int wrap_blocks(int64_t n) {
    const int64_t per = (int64_t)WT * WVec<T>::n;
    const int64_t b = (n + per - 1) / per;
    return (int)(b < 1 ? 1 : (b > WRAP_BLK ? WRAP_BLK : b));
}

// the kernels hold their cnt coefficients and sums in registers, sized by a compile-time bound
#define SIB_WRAP_KC(cnt, CALL) \
    do {                       \
        if ((cnt) <= 2) {      \
            constexpr int KC = 2; \
            CALL;              \
        } else if ((cnt) <= 4) { \
            constexpr int KC = 4; \
            CALL;              \
        } else {               \
            constexpr int KC = WRAP_MAXK + 1; \
            CALL;              \
        }                      \
    } while (0)

template <typename T>
int launch_wdots(const T* V, int64_t ld, int cnt, const T* w, int64_t n, double* partials, cudaStream_t s) {
    const int nb = wrap_blocks<T>(n);
    SIB_WRAP_KC(cnt, launch_pdl(k_wdots<T, KC>, nb, WT, 0, s, V, ld, cnt, w, n, partials));
    return nb;
}
template <typename T>
int launch_wgs(const T* V, int64_t ld, int cnt, const double* coef, const T* win, T* wout, int64_t n, int mode,
               double* partials, cudaStream_t s) {
    const int nb = wrap_blocks<T>(n);
    if (mode == 1)
        SIB_WRAP_KC(cnt, launch_pdl(k_wgs<T, 1, KC>, nb, WT, 0, s, V, ld, cnt, coef, win, wout, n, partials));
    else
        SIB_WRAP_KC(cnt, launch_pdl(k_wgs<T, 2, KC>, nb, WT, 0, s, V, ld, cnt, coef, win, wout, n, partials));
    return nb;
}
template <typename T>
void launch_wstep_cluster(const T* V, int64_t n, int cnt, const T* w, double* hA, double* hB, double* nr, T* Vnext,
                          int lsq_k, const double* hAll, const double* hBll, const double* nrAll, const double* beta2,
                          double* y, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(WC);
    cfg.blockDim = dim3(WT);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = WC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    // vectors of 16 bytes a thread for levels of up to 32^2, and for the largest
    constexpr int VN = WVec<T>::n, ESMALL = 4 / VN, ELARGE = (int)(wrap_cluster_max<T> / VN / (WC * WT));
    if constexpr (ELARGE > ESMALL) {
        if (n > (int64_t)ESMALL * VN * WC * WT) {
            SIB_WRAP_KC(cnt, cudaLaunchKernelEx(&cfg, k_wstep_cluster<T, KC, ELARGE>, V, n, cnt, w, hA, hB, nr, Vnext,
                                                lsq_k, hAll, hBll, nrAll, beta2, y));
            return;
        }
    }
    SIB_WRAP_KC(cnt, cudaLaunchKernelEx(&cfg, k_wstep_cluster<T, KC, ESMALL>, V, n, cnt, w, hA, hB, nr, Vnext, lsq_k,
                                        hAll, hBll, nrAll, beta2, y));
}
void launch_wreduce(const double* partials, int cnt, int nblk, double* out, cudaStream_t s) {
    launch_pdl(k_wreduce, cnt, WT, 0, s, partials, nblk, out);
}
template <typename T>
void launch_wmaxpy(const T* V, int64_t ld, int cnt, const double* coef, double sign, const T* yin, T* yout, int64_t n,
                   cudaStream_t s) {
    SIB_WRAP_KC(cnt, launch_pdl(k_wmaxpy<T, KC>, wrap_blocks<T>(n), WT, 0, s, V, ld, cnt, coef, sign, yin, yout, n));
}
template <typename T>
void launch_wscale(const T* w, const double* nrm2, T* v, int64_t n, cudaStream_t s) {
    launch_pdl(k_wscale<T>, wrap_blocks<T>(n), WT, 0, s, w, nrm2, v, n);
}
void launch_wreduce_lsq(const double* partials, int nblk, double* out, const double* hA, const double* hB,
                        const double* nrAll, const double* beta2, int k, double* y, cudaStream_t s) {
    launch_pdl(k_wreduce_lsq, 1, WT, 0, s, partials, nblk, out, hA, hB, nrAll, beta2, k, y);
}

#define SIB_WRAP_INST(T)                                                                                    \
    template int launch_wdots<T>(const T*, int64_t, int, const T*, int64_t, double*, cudaStream_t);           \
    template int launch_wgs<T>(const T*, int64_t, int, const double*, const T*, T*, int64_t, int, double*,     \
                               cudaStream_t);                                                               \
    template void launch_wmaxpy<T>(const T*, int64_t, int, const double*, double, const T*, T*, int64_t,      \
                                   cudaStream_t);                                                           \
    template void launch_wscale<T>(const T*, const double*, T*, int64_t, cudaStream_t); \
    template void launch_wstep_cluster<T>(const T*, int64_t, int, const T*, double*, double*, double*, T*, int, \
                                          const double*, const double*, const double*, const double*, double*, \
                                          cudaStream_t);
SIB_WRAP_INST(float)
SIB_WRAP_INST(double)

}  // namespace sib
